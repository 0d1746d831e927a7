"""Training GEMMs and the solid at the edges of their tiles: batches around one
and two row tiles and the split of the weight gradients, element counts around a
CTA's sixteen."""
import numpy as np
import pytest

import test_gpu_mlp as mlp_case
import test_gpu_solid as solid_case
from test_gpu_mlp import fsi  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


# A hidden value within FP32 rounding of a BF16 boundary may round the other way in the
# oracle: about one in four rows, and then it moves an output by 2^-9 of one of 256
# terms, 1e-4 of it; with few rows nothing averages that, hence 1e-3 here, and 1e-2
# for the gradients, which pass through it twice.
@pytest.mark.parametrize("B", [1, 2, 63, 65, 127, 128, 129, 2049])
def test_training_at_tile_edges(fsi, B):
    import torch
    from oracle import mlp as om
    rng = np.random.default_rng(B)
    p = om.init_params(3)
    for k in p:
        if k.startswith("b"):
            p[k] = rng.normal(scale=0.1, size=p[k].shape)
    theta = om.flatten(p).astype(np.float32).astype(np.float64)
    p = om.unflatten(theta)
    X = rng.normal(size=(B, om.N_IN)).astype(np.float32).astype(np.float64)
    Y = rng.normal(size=(B, om.N_OUT)).astype(np.float32).astype(np.float64)
    h = fsi.Mlp(2048 + 1)
    P, Xd, Yd = (mlp_case.T(a, torch.float32) for a in (theta, X, Y))
    out = torch.empty((B, 4), dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    grad, grad2 = torch.empty_like(P), torch.empty_like(P)
    fsi.fsi_mlp_forward(h, P, Xd, out)
    fsi.fsi_mlp_loss_grad(h, P, Xd, Yd, loss, grad)
    for _ in range(5):
        fsi.fsi_mlp_loss_grad(h, P, Xd, Yd, loss, grad2)
    h.check()
    assert torch.equal(grad, grad2)
    O_b, _ = om.forward(p, X, bf16=True)
    l_b, g_b = om.loss_and_grad(p, X, Y, bf16=True)
    assert mlp_case.rel(mlp_case.H(out), O_b) < 1e-3
    assert abs(float(loss.item()) - l_b) < 1e-3 * l_b
    g = om.unflatten(mlp_case.H(grad))
    for name, _ in om.param_shapes():
        assert mlp_case.rel(g[name], g_b[name]) < 1e-2, name


@pytest.mark.parametrize("n", [(1, 1, 1), (5, 3, 1), (4, 2, 2), (17, 1, 1), (7, 5, 3)])
def test_solid_by_element_count(fsi, n):
    import torch
    from oracle import solid as so
    T, H, MAT = solid_case.T, solid_case.H, solid_case.MAT
    mesh = fsi.Mesh(8, rho=MAT["rho_f"], mu=0.05, dt=0.01, rho_inf=0.5, device=0)
    m = solid_case.body_mesh(n=n, amp=0.003)
    b = solid_case.make_solid(fsi, mesh, m)
    rng = np.random.default_rng(sum(n))
    u, u_n = 0.002 * rng.normal(size=(m.ns, 3)), 0.002 * rng.normal(size=(m.ns, 3))
    v, a, x = (rng.normal(size=(m.ns, 3)) for _ in range(3))
    g = (0.0, -9.81, 0.5)
    R = torch.empty((m.ns, 3), dtype=torch.float64, device="cuda")
    fsi.fsi_solid_residual(b, T(u), T(v), T(a), T(u_n), g, R)
    torch.cuda.synchronize()
    assert solid_case.rel(H(R), so.residual(m, u, v, a, u_n, MAT, 0.05, g)) < 1e-12
    ca, cu, cv = so.chain(0.01)
    J = torch.empty_like(R)
    fsi.fsi_solid_tangent_apply(b, fsi.FSI_F64, T(u), T(u_n), T(x), J)
    torch.cuda.synchronize()
    assert solid_case.rel(H(J), so.tangent_apply(m, u, u_n, x, MAT, 0.05, ca, cu, cv)) < 1e-12
    b.close()
