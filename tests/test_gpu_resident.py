"""Solves that run as one launch (resident) against the same solves as separate kernels.

Forcing a product shape (bicg_variant, spmv_variant) selects the separate kernels, so a run
with and one without agree to the solvers' tolerances: the bounds are those between the
batched and the unbatched solve (test_gpu_parity.py).  Sizes: fewer rows than a block takes,
each number of lanes per row (8, 4, 2 and 1: up to 9,728, 19,456 and 38,912 rows on 152 SMs,
then more), and matrices too large for shared memory (from ~165,000 rows mixed, ~80,000
float64).
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


def relerr(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-300))


def box3(nx, ny, nz, ordering="natural"):
    mesh = WM.jitter_interior(WM.box_mesh_3d(nx, ny, nz), 0.15, 1.0 / max(nx, ny, nz), 3)
    X = 2 * np.pi * mesh.dof_coords() - np.pi
    pb = WP._held_problem("box", mesh, 1e-3, 1e-3, np.zeros(3), WP.tg3d_u(X), WP.tg3d_p(X), 2, 1e-8,
                          mesh.boundary_dofs["all"])
    if ordering == "random":
        pb.perm = WM.random_permutation(mesh.n_dofs, 5)
    return pb


CASES = {
    "box_3x2x2": (lambda: box3(3, 2, 2), 0),
    "box_5x4x3": (lambda: box3(5, 4, 3), 0),
    "channel_8x7x6": (lambda: WP.channel(nx=8, ny=7, nz=6), 1),
    "square_97": (lambda: WP.taylor_green_2d(97), 1),
    "square_190": (lambda: WP.taylor_green_2d(190), 1),
    "box_20": (lambda: box3(20, 20, 20), 1),
    "box_22_random": (lambda: box3(22, 23, 22, "random"), 1),
    "box_30": (lambda: box3(30, 30, 31), 1),
    "box_44": (lambda: box3(44, 43, 45), 1),
    "box_56": (lambda: box3(56, 56, 57), 0),
}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_resident_equals_separate_kernels(name, precision):
    from paper_1602_03643_gb300.driver import IPCSRun
    make, amg = CASES[name]
    pb = make()
    rtol = 1e-12 if precision == 0 else 1e-9
    out = []
    for forced in (0, 1):
        # the smallest and largest meshes with Jacobi, the others with multigrid
        run = IPCSRun(pb, precision=precision, rtol_u=rtol, rtol_p=rtol, use_graph=1, pressure_pc=amg, guess=1,
                      bicg_variant=forced, spmv_variant=forced)
        try:
            st = run.step(2)
            assert st.status == 0
            assert max(st.res_u) <= rtol and st.res_p <= rtol
            out.append((run.fields(), st))
        finally:
            run.close()
    (a, sa), (b, sb) = out
    assert relerr(a[0], b[0]) < (1e-10 if precision == 0 else 1e-7)
    assert relerr(a[1], b[1]) < (1e-9 if precision == 0 else 1e-6)
    # the same method: iteration counts differ by rounding only
    assert abs(sa.it_p - sb.it_p) <= 2 + sb.it_p // 10 and abs(sa.it_u[0] - sb.it_u[0]) <= 3


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("opts", [dict(batch_rhs=0), dict(velocity_update=1), dict(scalars=2)])
def test_resident_options(precision, opts):
    """One component at a time, the consistent-mass update, passive scalars."""
    from paper_1602_03643_gb300.driver import IPCSRun
    opts = dict(opts)
    pb = box3(14, 13, 12)
    if opts.pop("scalars", 0):
        pb = WP.with_scalars(pb, ns=2)
    rtol = 1e-12 if precision == 0 else 1e-9
    out = []
    for forced in (0, 1):
        run = IPCSRun(pb, precision=precision, rtol_u=rtol, rtol_p=rtol, use_graph=1, pressure_pc=1,
                      bicg_variant=forced, spmv_variant=forced, **opts)
        try:
            st = run.step(3)
            assert st.status == 0
            out.append(list(run.fields()[:2]) + ([run.scalar_fields()] if run.ns else []))
        finally:
            run.close()
    for x, y in zip(*out):
        assert relerr(x, y) < (1e-9 if precision == 0 else 1e-6)


@pytest.mark.parametrize("pc", [0, 1])
def test_resident_graph_equals_eager_bitwise(pc):
    from paper_1602_03643_gb300.driver import IPCSRun
    out = []
    for g in (0, 1):
        run = IPCSRun(box3(9, 8, 10), rtol_u=1e-9, rtol_p=1e-9, use_graph=g, precision=1, pressure_pc=pc, guess=1)
        try:
            run.step(3)
            out.append(run.fields())
        finally:
            run.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


def test_resident_solvers_on_two_streams():
    """Two threads step solvers of their own on streams of their own (graph and eager):
    launches that each need every SM take turns, and each solver gets the bits it gets alone."""
    import threading
    import torch
    from paper_1602_03643_gb300.driver import IPCSRun

    def make(k):
        pb = box3(24, 23, 25) if k == 0 else WP.taylor_green_2d(60)
        return IPCSRun(pb, rtol_u=1e-9, rtol_p=1e-9, use_graph=1 - k, precision=1, pressure_pc=1, guess=1,
                       stream=torch.cuda.Stream())

    def go(run, out, k):
        run.step(25)
        out[k] = run.fields()

    alone, both = [None, None], [None, None]
    for k in (0, 1):
        run = make(k)
        go(run, alone, k)
        run.close()
    runs = [make(0), make(1)]
    threads = [threading.Thread(target=go, args=(runs[k], both, k)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for run in runs:
        run.close()
    for k in (0, 1):
        for a, b in zip(alone[k], both[k]):
            np.testing.assert_array_equal(a, b)
