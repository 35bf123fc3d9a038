"""Device memory of general meshes: the rows of a precision are uploaded for
the first state that reads them and serve all later ones.  Entry counts: a
Delaunay mesh has 6 neighbours a node, up to 8 entries with the slices'
padding (24 B in FP32, 48 B in FP64, 32 B of them for the FP64 Laplacian), and
about 14 in the patch rows (10 B in FP32, 18 B in FP64, 26 B for the Laplacian);
mass, order and slices take less than 45 B.  Jittered tetrahedra: 14
neighbours, up to 17 entries (40 and 80 B)."""
import threading

import numpy as np
import pytest

from paper_1608_01906_gb300 import configs, felbm, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1608_01906_gb300 import build

    build.build()
    felbm.load()


KINDS = [("fp32", False), ("fp64", False), ("fp32", True)]


def state(mesh, args, precision, lap):
    n, dim = args[0].shape
    rng = np.random.default_rng(4)
    prm = {**configs.params(dt=0.4), "gravity": (0.0,) * 3}
    return felbm.State(mesh, felbm.make_params(precision=precision, lap_fp64=lap, **prm),
                       0.1 + 0.9 * rng.uniform(0.3, 0.7, size=n), rng.uniform(-0.02, 0.02, size=(n, dim)),
                       rng.uniform(0.0, 0.01, size=n))


def grown(args, kinds):
    """Bytes a node after the states of the given kinds, one after the other."""
    mesh = felbm.Mesh(*args)
    out, keep = [], []
    for precision, lap in kinds:
        keep += [state(mesh, args, precision, lap)]
        out.append(mesh.info()["device_bytes"] / len(args[0]))
    for s in keep:
        s.close()
    mesh.close()
    return out


def test_bytes_of_triangle_meshes():
    args = inputs.jittered_delaunay_mesh(120, 100, 0.25, seed=2)
    once, twice = grown(args, [KINDS[0], KINDS[0]])
    assert once == twice <= 8 * 24 + 14 * 10 + 45
    assert grown(args, [KINDS[1]])[0] <= 8 * 48 + 14 * 18 + 45
    assert grown(args, [KINDS[2]])[0] <= 8 * (24 + 32) + 14 * 26 + 45
    assert len({grown(args, k)[-1] for k in (KINDS, KINDS[::-1])}) == 1  # whatever the order


def test_bytes_of_tetrahedra():
    args = inputs.jittered_tet_mesh(12, 11, 10, 0.1, 5)[:3]
    assert grown(args, [KINDS[0]])[0] <= 17 * 40 + 45
    assert grown(args, [KINDS[1]])[0] <= 17 * 80 + 45


def advanced(st):
    st.step(5)
    m = st.moments()
    st.close()
    return m


@pytest.mark.parametrize("dim", [2, 3])
def test_states_made_by_threads(dim):
    """States of every kind made at once on one mesh, each by its own thread,
    as on meshes of their own."""
    args = inputs.jittered_delaunay_mesh(70, 60, 0.25, seed=2) if dim == 2 else inputs.jittered_tet_mesh(9, 8, 7, 0.1, 5)[:3]
    kinds = (KINDS if dim == 2 else KINDS[:2]) * 2
    ref = []
    for k in kinds:
        mesh = felbm.Mesh(*args)
        ref.append(advanced(state(mesh, args, *k)))
        mesh.close()
    mesh = felbm.Mesh(*args)
    got = [None] * len(kinds)

    def make(q):
        got[q] = state(mesh, args, *kinds[q])

    threads = [threading.Thread(target=make, args=(q,)) for q in range(len(kinds))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s, r in zip(got, ref):
        m = advanced(s)
        for name in ("rho", "u", "p"):
            assert np.array_equal(m[name], r[name]), name
    mesh.close()
