"""Patch step of meshes with a node of very many neighbours, whose patches have
more rows than a block stages: against the four-launch step, bit for bit, and
that such a mesh still takes it."""
import numpy as np
import pytest
from scipy.spatial import Delaunay

from paper_1608_01906_gb300 import configs, felbm
from test_gpu_general_rows import fan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1608_01906_gb300 import build

    build.build()
    felbm.load()


def hub(side, degree):
    """A jittered square whose middle is one node joined to a ring of others."""
    rng = np.random.default_rng(3)
    xy = np.stack(np.meshgrid(np.arange(side), np.arange(side)), -1).reshape(-1, 2).astype(float)
    inner = ((xy > 0) & (xy < side - 1)).all(1)
    xy[inner] += rng.uniform(-0.2, 0.2, xy.shape)[inner]
    r, c = degree / (2 * np.pi), side / 2.0
    t = 2 * np.pi * np.arange(degree) / degree
    xy = xy[np.hypot(*(xy - c).T) > r + 0.7]
    xy = np.concatenate([xy, c + r * np.stack([np.cos(t), np.sin(t)], 1), [[c, c]]])
    tri = Delaunay(xy).simplices.astype(np.int32)
    e = xy[tri[:, 1:]] - xy[tri[:, :1]]
    flip = np.linalg.det(e) < 0
    tri[flip] = tri[flip][:, [0, 2, 1]]
    return xy, tri, np.zeros(2), np.zeros(len(xy), dtype=np.uint8)


# every patch with the long row; some patches with it, staged and not
@pytest.mark.parametrize("precision, lap_fp64", [("fp32", False), ("fp32", True), ("fp64", False)])
@pytest.mark.parametrize("name, dt", [("fan_400", 0.0005), ("hub_120_100", 0.01), ("hub_150_420", 0.01)])
def test_long_rows_bitwise(name, dt, precision, lap_fp64):
    kind, *size = name.split("_")
    mesh_args = (fan if kind == "fan" else hub)(*map(int, size))
    n = len(mesh_args[0])
    rng = np.random.default_rng(11)
    rho0 = 0.1 + 0.9 * rng.uniform(0.2, 0.8, size=n)
    u0, p0 = rng.uniform(-0.02, 0.02, size=(n, 2)), rng.uniform(0.0, 0.01, size=n)
    out = []
    for split in (False, True):
        mesh = felbm.Mesh(*mesh_args, general=True, split_step=split)
        st = felbm.State(mesh, felbm.make_params(precision=precision, lap_fp64=lap_fp64, **configs.params(dt=dt)),
                         rho0, u0, p0)
        st.profile_enable(True)
        st.step(3)
        assert st.profile_read()["k_patch_step"][2] == (0 if split else 3)
        out.append((*(st.moments()[k] for k in ("rho", "u", "p", "totals")), *st.export()))
        st.close()
        mesh.close()
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(a, b)
