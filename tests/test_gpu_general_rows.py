"""General meshes whose rows are long or whose slices are ragged, against the
FP64 oracle: the rows are stored in slices of 32 nodes, read in chunks, with
one byte for a node's degree.

Tolerance: 1e-12 relative L2 in FP64 (reordered sums only).  The states start
with a flow and a density step, so no field is zero.
"""
import numpy as np
import pytest

from conftest import rel_l2
from oracle.oracle import Oracle, Params
from paper_1608_01906_gb300 import configs, felbm, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1608_01906_gb300 import build

    build.build()
    felbm.load()


def fan(per_side):
    """A square fanned from its centre: one node of degree 4 per_side, the
    others of degree 3."""
    t = np.arange(per_side) / per_side
    o, z = np.ones(per_side), np.zeros(per_side)
    ring = np.concatenate([np.stack([t, z], 1), np.stack([o, t], 1), np.stack([1 - t, o], 1), np.stack([z, 1 - t], 1)])
    xy = np.concatenate([[[0.5, 0.5]], ring]) * 16.0
    k = np.arange(len(ring))
    tri = np.stack([np.zeros_like(k), 1 + k, 1 + (k + 1) % len(ring)], 1).astype(np.int32)
    return xy, tri, np.zeros(2), np.zeros(len(xy), dtype=np.uint8)


def case(name):
    if name.startswith("fan"):
        return fan(int(name[4:])), 0.01
    nx, ny = (int(v) for v in name.split("x"))
    return inputs.jittered_delaunay_mesh(nx, ny, 0.25, seed=nx), 0.4


# degrees 2 chunks (8), 9, and beyond one byte; node counts around a slice, a
# patch, and three patches of which the last has one node
@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("name", ["fan_2", "fan_3", "fan_63", "fan_64", "fan_80", "5x5", "11x5", "16x16", "27x19"])
def test_rows(name, split):
    (xy, tri, box, tag), dt = case(name)
    pr = configs.params(dt=dt)
    rng = np.random.default_rng(11)
    n = len(xy)
    rho0 = 0.1 + 0.9 * rng.uniform(0.2, 0.8, size=n)
    u0, p0 = rng.uniform(-0.02, 0.02, size=(n, 2)), rng.uniform(0.0, 0.01, size=n)
    mesh = felbm.Mesh(xy, tri, box, tag, general=True, split_step=split)
    st = felbm.State(mesh, felbm.make_params(precision="fp64", **pr), rho0, u0, p0)
    st.step(3)
    m = st.moments()
    o = Oracle(xy, tri, box, tag, Params(**pr))
    o.init(rho0, u0, p0)
    o.step(3)
    st.close()
    mesh.close()
    assert rel_l2(m["rho"], o.rho) <= 1e-12
    assert rel_l2(m["u"], np.stack([o.ux, o.uy], 1)) <= 1e-12
    assert rel_l2(m["p"], o.p) <= 1e-12
