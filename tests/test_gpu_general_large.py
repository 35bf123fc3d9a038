"""General meshes of more patches than are resident at once (two per SM, 77,824
nodes), whose kernels have their own register bounds: the patch step against
the four-launch step, bit for bit, and which of the two a state takes by
itself."""
import numpy as np
import pytest

from paper_1608_01906_gb300 import configs, felbm, inputs

pytestmark = pytest.mark.gpu

NX, NY, STEPS = 301, 277, 8  # 83,377 nodes, the last patch with 177


@pytest.fixture(scope="module")
def mesh_args():
    from paper_1608_01906_gb300 import build

    build.build()
    felbm.load()
    return inputs.jittered_delaunay_mesh(NX, NY, 0.25, seed=3)


def run(mesh_args, precision, lap_fp64, **step):
    xy, _, box, _ = mesh_args
    rho0, u0, p0 = inputs.droplet_fields(xy, box, (150, 138), 60.0, 1.0, 0.1, 6.0, u0=(0.02, 0.01))
    mesh = felbm.Mesh(*mesh_args, general=True, **step)
    st = felbm.State(mesh, felbm.make_params(precision=precision, lap_fp64=lap_fp64, **configs.params(dt=0.4)),
                     rho0, u0, p0)
    st.profile_enable(True)
    st.step(STEPS)
    launches = st.profile_read()["k_patch_step"][2]
    got = (*(st.moments()[k] for k in ("rho", "C", "u", "p", "totals")), *st.export())
    st.close()
    mesh.close()
    return got, launches


@pytest.mark.parametrize("precision, lap_fp64, default", [("fp32", False, STEPS), ("fp32", True, STEPS), ("fp64", False, 0)])
def test_patch_and_four_launch_step_bitwise(mesh_args, precision, lap_fp64, default):
    a, na = run(mesh_args, precision, lap_fp64, patch_step=True)
    b, nb = run(mesh_args, precision, lap_fp64, split_step=True)
    c, nc = run(mesh_args, precision, lap_fp64)
    assert (na, nb, nc) == (STEPS, 0, default)
    for x, y, z in zip(a, b, c):
        assert np.array_equal(x, y) and np.array_equal(x, z)
