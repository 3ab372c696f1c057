"""Resident solves of small velocities, mixed precision.

With velocities of 2^-50 and 2^-56 the squares of the pressure residual's entries are
around the smallest normal float32 values and 1 / <r, M r> is beyond the largest: the
scalars of the Krylov iterations must not have float32's range.  The separate kernels
hold them in float64 and set the pace.  Some of the products in the sums underflow, so
the counts are compared loosely: within a factor of two, and two refinement sweeps
(a breakdown in every sweep shows as several times the iterations, a sweep for each).
"""
import numpy as np
import pytest

from workloads import problems as WP
from workloads import meshes as WM

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_03643_gb300 import build
    build.build()
    torch.cuda.init()


def box(scale):
    mesh = WM.jitter_interior(WM.box_mesh_3d(12, 12, 12), 0.15, 1.0 / 12, 3)
    X = 2 * np.pi * mesh.dof_coords() - np.pi
    return WP._held_problem("box", mesh, 1e-3, 1e-3, np.zeros(3), scale * WP.tg3d_u(X), scale ** 2 * WP.tg3d_p(X), 2,
                            1e-8, mesh.boundary_dofs["all"])


@pytest.mark.parametrize("update", [0, 1])
@pytest.mark.parametrize("pc", [0, 1])
@pytest.mark.parametrize("power", [0, 50, 56])
def test_small_velocities(power, pc, update):
    from paper_1602_03643_gb300.driver import IPCSRun
    st = []
    for forced in (0, 1):
        run = IPCSRun(box(2.0 ** -power), precision=1, rtol_u=1e-8, rtol_p=1e-8, use_graph=1, guess=1, pressure_pc=pc,
                      velocity_update=update, bicg_variant=forced, spmv_variant=forced, max_it_p=4000)
        try:
            st.append(run.step(2))
        finally:
            run.close()
    a, b = st
    assert a.status == 0 and b.status == 0
    assert a.sweeps_p <= b.sweeps_p + 2 and a.sweeps_u <= b.sweeps_u + 2
    assert a.it_p <= 2 * b.it_p + 10 and a.it_m <= 2 * b.it_m + 10
    assert all(x <= 2 * y + 10 for x, y in zip(a.it_u, b.it_u))
