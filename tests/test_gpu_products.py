"""The stand-alone products with the library's own choice of shape (lanes = 0) and the
training kernels at sizes where they can go wrong: fewer rows than a warp takes at once,
ragged ends, periodic neighbours behind 16-bit offsets, and an order whose offsets need 32
bits.  Tolerances: those of the other product and gradient tests (test_gpu_parity.py,
test_gpu_net.py).
"""
import numpy as np
import pytest

from oracle import net as ON
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


MESHES = {
    "box_1x1x1": lambda: (WM.box_mesh_3d(1, 1, 1), None),
    "box_7x5x9": lambda: (WM.jitter_interior(WM.box_mesh_3d(7, 5, 9), 0.15, 1 / 9, 3), None),
    "periodic_6x5x7": lambda: (WM.box_mesh_3d(6, 5, 7, periodic=(True, False, True)), None),
    "square_33x31": lambda: (WM.box_mesh_2d(33, 31), None),
    "box_41_random": lambda: (lambda m: (m, WM.random_permutation(m.n_dofs, 8)))(WM.box_mesh_3d(41, 41, 41)),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_products_own_shape(name):
    import torch
    from paper_1602_03643_gb300 import capi as c
    m, perm = MESHES[name]()
    h = c.oasis_mesh_create(m.dim, m.coords, m.cells, m.dof_of_vertex, m.n_dofs, perm)
    try:
        c.oasis_assemble_constant(h)
        rp, col = c.oasis_mesh_get_pattern(h)
        at = np.arange(m.n_dofs) if perm is None else perm     # internal index of caller dof d
        rng = np.random.default_rng(2)
        x = rng.normal(size=m.n_dofs)
        xi = np.empty_like(x)
        xi[at] = x
        for which in (c.OASIS_MAT_M, c.OASIS_MAT_K, c.OASIS_MAT_G0):
            v = c.oasis_mesh_get_matrix(h, which)
            want = np.add.reduceat(v * x[col], rp[:-1])
            X = torch.from_numpy(xi).cuda()
            Y, Z, dot = torch.empty_like(X), torch.empty_like(X), torch.zeros(1, dtype=torch.float64, device="cuda")
            c.oasis_spmv_f64(h, which, X, Y, 0)
            c.oasis_spmv_dot_f64(h, which, X, Z, dot)
            F = X.float()
            G = torch.empty_like(F)
            c.oasis_spmv_f32(h, which, F, G, 0)
            torch.cuda.synchronize()
            scale = np.abs(want).max()
            np.testing.assert_allclose(Y.cpu().numpy()[at], want, rtol=0, atol=1e-13 * scale)
            np.testing.assert_allclose(Z.cpu().numpy()[at], want, rtol=0, atol=1e-13 * scale)
            assert np.linalg.norm(G.cpu().numpy()[at] - want) < 2e-6 * np.linalg.norm(want)
            assert abs(dot.item() - x @ want) <= 1e-12 * (np.abs(x) @ np.abs(want))
    finally:
        c.oasis_mesh_destroy(h)


@pytest.mark.parametrize("name", ["box_1x1x1", "box_7x5x9", "periodic_6x5x7", "square_33x31"])
def test_gradient_at_ragged_sizes(name):
    import torch
    from paper_1602_03643_gb300 import capi as c
    from paper_1602_03643_gb300.guess import GuessNet
    m, _ = MESHES[name]()
    h = c.oasis_mesh_create(m.dim, m.coords, m.cells, m.dof_of_vertex, m.n_dofs)
    c.oasis_assemble_constant(h)
    rng = np.random.default_rng(4)
    p = ON.round_bf16(ON.init_params(6) + 0.1 * rng.normal(size=ON.init_params(6).size))
    net = GuessNet(h, m.n_dofs, params=p)
    try:
        x = rng.normal(0, 1, (m.n_dofs, 3)).astype(np.float32)
        t = rng.normal(0, 1, m.n_dofs).astype(np.float32)
        loss, grad = net.loss_and_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
        Am = ON.mean_operator(*c.oasis_mesh_get_pattern(h))
        L_ref, g_ref, _ = ON.loss_and_grad(p, x.astype(np.float64), t.astype(np.float64), Am)
        assert abs(float(loss.item()) - L_ref) <= 1e-5 * L_ref
        np.testing.assert_allclose(grad.cpu().numpy(), g_ref, rtol=0, atol=1e-4 * np.abs(g_ref).max())
    finally:
        net.close()
        c.oasis_mesh_destroy(h)
