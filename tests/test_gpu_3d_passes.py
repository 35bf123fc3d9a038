"""The passes of the 3-D step at the sizes where their forms change: columns
that end in the lattice's last planes, planes that are no multiple of a
block, wall layers within a column, blocks of few nodes, rows longer than
the entries a thread holds at once.

FP64 against the oracle: sums in another order only, 1e-12.  FP32 against the
FP64 run of the same mesh: a step rounds each population about twice, 2^-24
of its size, so ten steps keep rho within 20 x 2^-24 = 1.2e-6 (bound 2e-6)
and u, carried by differences of populations of the size of p + rho u, within
1e-5."""
import numpy as np
import pytest

from conftest import rel_l2
from oracle.oracle3d import Oracle3, Params3
from paper_1608_01906_gb300 import felbm, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1608_01906_gb300 import build

    build.build()
    felbm.load()


def params(xi=4.0, gravity=(0.0, 0.0, 0.0)):
    return dict(rho_l=1.0, rho_v=0.2, sigma=0.01, xi=xi, tau_l=0.6, tau_v=0.5, dt=0.4, gravity=gravity)


def fields(xyz, seed=7):
    """Smooth density and flow of several wave lengths on any set of nodes."""
    s = np.ptp(xyz, axis=0) + 1.0
    rng = np.random.default_rng(seed)
    ph = rng.uniform(0, 2 * np.pi, (5, 3))
    w = 2 * np.pi * xyz / s
    f = [np.sin(w + ph[k]).prod(axis=1) for k in range(5)]
    return 0.6 + 0.3 * f[0], 0.04 * np.stack(f[1:4], 1), 0.01 + 0.002 * f[4]


def run(mesh_args, prm, precision, steps, kind):
    mesh = felbm.Mesh(*mesh_args)
    assert mesh.info()["kind"] == kind
    rho0, u0, p0 = fields(mesh_args[0])
    st = felbm.State(mesh, felbm.make_params(precision=precision, **prm), rho0, u0, p0)
    st.step(steps)
    m = st.moments()
    st.close()
    mesh.close()
    return m


def check_oracle(mesh_args, prm, steps, kind):
    m = run(mesh_args, prm, "fp64", steps, kind)
    o = Oracle3(*mesh_args, Params3(**prm))
    o.init(*fields(mesh_args[0]))
    o.step(steps)
    for name, ref in (("rho", o.rho), ("u", o.u), ("p", o.p)):
        assert rel_l2(m[name], ref) <= 1e-12, (name, rel_l2(m[name], ref))


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("size", [(3, 3, 3), (5, 7, 4), (9, 8, 13), (31, 9, 5)])
def test_fp64_lattice_sizes(size, walls):
    xyz, tet, box, tag = inputs.structured_tet_mesh(*size, periodic_z=not walls)
    prm = params(gravity=(1e-5, -2e-5, 0.0)) if walls else params()
    check_oracle((xyz, tet, box, tag if walls else None), prm, 6, 3)


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("size", [(3, 4, 3), (31, 9, 5), (33, 33, 31), (61, 47, 33), (64, 40, 35), (75, 41, 65)])
def test_fp32_lattice_sizes(size, walls):
    xyz, tet, box, tag = inputs.structured_tet_mesh(*size, periodic_z=not walls)
    prm = params(gravity=(1e-5, -2e-5, 0.0)) if walls else params()
    args = (xyz, tet, box, tag if walls else None)
    a, b = (run(args, prm, precision, 10, 3) for precision in ("fp32", "fp64"))
    assert rel_l2(a["rho"], b["rho"]) <= 2e-6, rel_l2(a["rho"], b["rho"])
    assert rel_l2(a["u"], b["u"]) <= 1e-5, rel_l2(a["u"], b["u"])


@pytest.mark.parametrize("size", [(5, 4, 3), (4, 4, 4), (7, 5, 9)])
def test_fp64_general_sizes(size):
    xyz, tet, box, _ = inputs.jittered_tet_mesh(*size, 0.1, 5)
    check_oracle((xyz, tet, box, None), params(), 6, 2)


def hub_mesh(n):
    """A cube whose surface nodes all share tetrahedra with its centre: a row
    of 6 n^2 + 2 entries, the others with at most 9."""
    grid = {}
    xyz = [(n / 2.0, n / 2.0, n / 2.0)]

    def node(p):
        if p not in grid:
            grid[p] = len(xyz)
            xyz.append(tuple(float(v) for v in p))
        return grid[p]

    tet = []
    for c in range(3):
        for side in (0, n):
            for a in range(n):
                for b in range(n):
                    q = []
                    for da, db in ((0, 0), (1, 0), (1, 1), (0, 1)):
                        p = [0, 0, 0]
                        p[c], p[(c + 1) % 3], p[(c + 2) % 3] = side, a + da, b + db
                        q.append(node(tuple(p)))
                    tet += [[0, q[0], q[1], q[2]], [0, q[0], q[2], q[3]]]
    xyz, tet = np.array(xyz), np.array(tet, dtype=np.int32)
    e = xyz[tet[:, 1:]] - xyz[tet[:, :1]]
    flip = np.linalg.det(e) < 0
    tet[flip] = tet[flip][:, [0, 2, 1, 3]]
    return xyz, tet, np.zeros(3)


@pytest.mark.parametrize("n", [2, 4])
def test_fp64_long_rows(n):
    xyz, tet, box = hub_mesh(n)
    check_oracle((xyz, tet, box, None), {**params(), "dt": 0.1}, 3, 2)
