"""Rounding errors of the stand-alone products with the library's own shape (lanes = 0).

Measured against sums in extended precision, over a mesh with ~15 entries per row, beside
16 lanes per row (one entry per lane and a tree of four additions, every product rounded).
A lane of the library's shape takes eight entries: it must not round more than that.  Over
68,921 rows the root mean square of the errors is known to better than a percent; 2 % are
allowed for it.  Infinities and NaN in the operand come out as in the plain sum.
"""
import numpy as np
import pytest

from test_gpu_resident import _lib  # noqa: F401
from workloads import meshes as WM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["rcm", "random"])
def test_own_shape_rounds_no_more_than_16_lanes(order):
    import torch
    from paper_1602_03643_gb300 import capi as c
    m = WM.jitter_interior(WM.box_mesh_3d(40, 40, 40), 0.15, 1 / 40, 3)
    perm = WM.rcm_permutation(m) if order == "rcm" else WM.random_permutation(m.n_dofs, 8)
    h = c.oasis_mesh_create(m.dim, m.coords, m.cells, m.dof_of_vertex, m.n_dofs, perm)
    try:
        c.oasis_assemble_constant(h)
        rp, col = c.oasis_mesh_get_pattern(h)
        x = np.random.default_rng(2).normal(size=m.n_dofs)
        for dt, spmv in ((np.float64, c.oasis_spmv_f64), (np.float32, c.oasis_spmv_f32)):
            xi = np.empty(m.n_dofs, dt)
            xi[perm] = x.astype(dt)
            X = torch.from_numpy(xi).cuda()
            wide = np.longdouble if dt is np.float64 else np.float64
            for which in (c.OASIS_MAT_M, c.OASIS_MAT_K, c.OASIS_MAT_G0):
                v = c.oasis_mesh_get_matrix(h, which).astype(dt).astype(wide)
                want = np.add.reduceat(v * x.astype(dt).astype(wide)[col], rp[:-1])
                rms = []
                for lanes in (0, 16):
                    Y = torch.empty_like(X)
                    spmv(h, which, X, Y, lanes)
                    torch.cuda.synchronize()
                    rms.append(float(np.sqrt(np.mean((Y.cpu().numpy()[perm].astype(wide) - want) ** 2))))
                assert rms[0] <= 1.02 * rms[1], (which, dt, rms)
        # the columns of one row reach its neighbours: infinities and NaN as in the plain sum
        for bad in (np.inf, -np.inf, np.nan):
            xb = x.astype(np.float32)
            xb[1234] = bad
            xi = np.empty_like(xb)
            xi[perm] = xb
            X = torch.from_numpy(xi).cuda()
            Y = [torch.empty_like(X) for _ in range(2)]
            for y, lanes in zip(Y, (0, 16)):
                c.oasis_spmv_f32(h, c.OASIS_MAT_M, X, y, lanes)
            torch.cuda.synchronize()
            a, b = (y.cpu().numpy() for y in Y)
            hit = ~np.isfinite(b)
            assert hit.any()
            np.testing.assert_array_equal(a[hit], b[hit])
            assert np.isfinite(a[~hit]).all()
    finally:
        c.oasis_mesh_destroy(h)


@pytest.mark.parametrize("side,f64_own,f32_own", [(3, False, False), (24, False, False), (26, True, False),
                                                  (37, True, True)])
def test_small_products_take_16_lanes(side, f64_own, f32_own):
    """Rows up to which the library's choice is 16 lanes per row: 16,384 float64, 50,000 float32
    (the same bits as with lanes = 16; above, sums in another order)."""
    import torch
    from paper_1602_03643_gb300 import capi as c
    m = WM.jitter_interior(WM.box_mesh_3d(side, side, side), 0.15, 1 / side, 3)
    h = c.oasis_mesh_create(m.dim, m.coords, m.cells, m.dof_of_vertex, m.n_dofs, None)
    try:
        c.oasis_assemble_constant(h)
        for dt, spmv, own in ((torch.float64, c.oasis_spmv_f64, f64_own), (torch.float32, c.oasis_spmv_f32, f32_own)):
            x = torch.randn(m.n_dofs, dtype=dt, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
            y = [torch.empty_like(x) for _ in range(2)]
            for out, lanes in zip(y, (0, 16)):
                spmv(h, c.OASIS_MAT_K, x, out, lanes)
            torch.cuda.synchronize()
            assert torch.equal(y[0], y[1]) != own
    finally:
        c.oasis_mesh_destroy(h)


@pytest.mark.parametrize("side", [1, 2, 5, 24, 25, 40, 66])
@pytest.mark.parametrize("order", ["natural", "random"])
def test_dot_shapes(side, order):
    """The dot form's shapes by rows (up to 16,384, above), with 16-bit columns and
    without (random order from 33 per side on), down to fewer rows than a warp takes; scratch
    for every block, of the mesh and of the form that allocates nothing."""
    import torch
    from paper_1602_03643_gb300 import capi as c
    m = WM.box_mesh_3d(side, side, side)
    perm = WM.random_permutation(m.n_dofs, 8) if order == "random" else np.arange(m.n_dofs, dtype=np.int32)
    h = c.oasis_mesh_create(m.dim, m.coords, m.cells, m.dof_of_vertex, m.n_dofs, perm)
    try:
        c.oasis_assemble_constant(h)
        rp, col = c.oasis_mesh_get_pattern(h)
        v = c.oasis_mesh_get_matrix(h, c.OASIS_MAT_M)
        x = np.random.default_rng(4).normal(size=m.n_dofs)
        want = np.add.reduceat(v * x[col], rp[:-1])
        xi = np.empty_like(x)
        xi[perm] = x
        X = torch.from_numpy(xi).cuda()
        for call in (c.oasis_spmv_dot_f64, c.oasis_spmv_dot_f64_noalloc):
            Y, d = torch.empty_like(X), torch.zeros(1, dtype=torch.float64, device="cuda")
            for _ in range(2):                    # the ticket is left ready for the next call
                call(h, c.OASIS_MAT_M, X, Y, d)
            torch.cuda.synchronize()
            # float64 sums of up to 15 positive and negative terms, and of all rows
            assert np.abs(Y.cpu().numpy()[perm] - want).max() <= 1e-14 * np.abs(v).max() * np.abs(x).max() * 15
            assert abs(float(d) - float(x @ want)) <= 1e-12 * float(np.abs(x) @ np.abs(want))
    finally:
        c.oasis_mesh_destroy(h)
