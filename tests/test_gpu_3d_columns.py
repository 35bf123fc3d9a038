"""The scalar passes of the 3-D lattice where their columns lie unevenly on the
threads: blocks that hold several planes or end within one, columns of two
nodes (from 2^18 nodes on, FP32) of which the last is cut by an odd height or
reaches a wall layer; and the passes with a thread per node (from 2^16 nodes
on) in FP64.

FP64 against the oracle: sums in another order only, 1e-12.  FP32 against the
FP64 run of the same mesh: a step rounds each population about twice, 2^-24
of its size, so ten steps keep rho within 20 x 2^-24 = 1.2e-6 (bound 2e-6)
and u, carried by differences of populations of the size of p + rho u, within
1e-5."""
import pytest

from conftest import rel_l2
from paper_1608_01906_gb300 import felbm, inputs
from test_gpu_3d_passes import check_oracle, params, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1608_01906_gb300 import build

    build.build()
    felbm.load()


def lattice(size, walls):
    xyz, tet, box, tag = inputs.structured_tet_mesh(*size, periodic_z=not walls)
    prm = params(gravity=(1e-5, -2e-5, 0.0)) if walls else params()
    return (xyz, tet, box, tag if walls else None), prm


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("size", [(3, 3, 157), (3, 5, 300), (17, 16, 9)])
def test_fp64_planes_and_blocks(size, walls):
    check_oracle(*lattice(size, walls), 4, 3)


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("size", [(3, 3, 29999)])
def test_fp32_two_node_columns(size, walls):
    args, prm = lattice(size, walls)
    a, b = (run(args, prm, precision, 10, 3) for precision in ("fp32", "fp64"))
    assert rel_l2(a["rho"], b["rho"]) <= 2e-6, rel_l2(a["rho"], b["rho"])
    assert rel_l2(a["u"], b["u"]) <= 1e-5, rel_l2(a["u"], b["u"])


# (planes that are no multiple of a block, and an odd height: the last column
# of a periodic lattice has one node, the first and last of a walled one mix a
# wall layer with an inner one)
@pytest.mark.parametrize("walls", [False, True])
def test_fp32_two_node_columns_odd_height(walls):
    args, prm = lattice((67, 61, 65), walls)
    a, b = (run(args, prm, precision, 10, 3) for precision in ("fp32", "fp64"))
    assert rel_l2(a["rho"], b["rho"]) <= 2e-6, rel_l2(a["rho"], b["rho"])
    assert rel_l2(a["u"], b["u"]) <= 1e-5, rel_l2(a["u"], b["u"])


@pytest.mark.parametrize("walls", [False, True])
def test_fp64_thread_per_node(walls):
    check_oracle(*lattice((43, 41, 39), walls), 3, 3)  # 68,757 nodes
