"""The Krylov solver's parts that change with a size: the Gram-Schmidt update
by the number of basis vectors, the V-cycle's coarse levels by their shape."""
import numpy as np
import pytest

import test_gpu_newton as newton_case
import test_gpu_precond as precond_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2601_08266_gb300 as pkg
    return pkg


# basis lengths at the edges of 8 (one group of dots), 16 (the vectors an FP32
# update holds) and beyond; with block Jacobi the solves use the whole restart
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("restart", [7, 8, 9, 16, 17, 40])
def test_newton_step_by_restart_length(fsi, oracle, mixed, restart):
    """Every solve reaches the residual reduction that was planned for it, so
    the step converges in as many Newton iterations as with a long basis."""
    mesh, st, dev, P, y0 = newton_case.setup(fsi, oracle, N=6, m=200, seed=3)
    code, rep = fsi.fsi_newton_step(mesh, st, mixed=mixed, restart=restart, max_newton=12,
                                    max_krylov=4000, newton_rtol=1e-8, krylov_rtol=1e-3, precond=0)
    assert code == 0 and rep["converged"] == 1
    assert rep["krylov_iters"] > restart, rep
    r = np.linalg.norm(P.residual(newton_case.H(dev["y"])))
    assert r <= 1.01e-8 * rep["r_ref"], (r, rep)
    mesh2, st2, _, _, _ = newton_case.setup(fsi, oracle, N=6, m=200, seed=3)
    _, full = fsi.fsi_newton_step(mesh2, st2, mixed=mixed, restart=150, max_newton=12,
                                  max_krylov=4000, newton_rtol=1e-8, krylov_rtol=1e-3, precond=0)
    assert rep["newton_iters"] <= full["newton_iters"] + 1, (rep, full)


# first coarse levels of 1,331 nodes (split, 2 planes a slab), 729 (not split),
# a wide flat one (33 x 33 x 3), a long thin one (3 x 3 x 129), unequal planes per
# slab (13 planes), and a dense level too large for shared memory (9 x 9 x 5)
@pytest.mark.parametrize("faces", precond_case.FACES)
@pytest.mark.parametrize("N", [(20, 20, 20), (16, 16, 16), (64, 64, 4), (4, 4, 256), (24, 24, 24),
                               (48, 40, 24), (32, 32, 16)])
def test_f32_vcycle_coarse_level_shapes(fsi, N, faces):
    import torch
    mesh, mg = precond_case.setup(fsi, N, None, faces)
    n = mg.levels[0].n
    b = np.random.default_rng(11).normal(size=n).astype(np.float32).astype(np.float64)
    x = torch.empty(n, dtype=torch.float32, device="cuda")
    fsi.fsi_pressure_vcycle(mesh, precond_case.T(b, torch.float32), x)
    x2 = torch.empty_like(x)
    fsi.fsi_pressure_vcycle(mesh, precond_case.T(b, torch.float32), x2)
    torch.cuda.synchronize()
    assert torch.equal(x, x2)
    assert precond_case.rel(precond_case.H(x), mg.vcycle(b)) < 2e-5, N


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("N", [(8, 8, 8), (33, 20, 12), (48, 40, 24)])
def test_vcycle_repeats_and_under_capture(fsi, prec, N):
    """The V-cycle's launches overlap: back-to-back cycles on changing inputs,
    eager and replayed from a CUDA graph, give the bits of a cycle by itself."""
    import torch
    mesh, mg = precond_case.setup(fsi, N, None)
    n = mg.levels[0].n
    dt = precond_case.dtype_of(prec)
    rng = np.random.default_rng(5)
    bs = [precond_case.T(rng.normal(size=n), dt) for _ in range(3)]
    alone = []
    for b in bs:
        x = torch.empty(n, dtype=dt, device="cuda")
        torch.cuda.synchronize()
        fsi.fsi_pressure_vcycle(mesh, b, x)
        torch.cuda.synchronize()
        alone.append(x.clone())
    xs = [torch.empty(n, dtype=dt, device="cuda") for _ in range(30)]
    for q, x in enumerate(xs):
        fsi.fsi_pressure_vcycle(mesh, bs[q % 3], x)
    torch.cuda.synchronize()
    assert all(torch.equal(x, alone[q % 3]) for q, x in enumerate(xs))
    side = torch.cuda.Stream()
    mesh2 = fsi.Mesh(N, device=0, stream=side.cuda_stream)
    x = torch.empty(n, dtype=dt, device="cuda")
    y = torch.empty(n, dtype=dt, device="cuda")
    with torch.cuda.stream(side):
        fsi.fsi_pressure_vcycle(mesh2, bs[0], x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        fsi.fsi_pressure_vcycle(mesh2, bs[0], x)
        fsi.fsi_pressure_vcycle(mesh2, bs[1], y)
    for _ in range(3):
        x.zero_()
        y.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(x, alone[0]) and torch.equal(y, alone[1])


# 45^3 and 35^3 nodes: more records than the one-launch orthogonalisation holds, so the
# passes of long vectors run (8 vectors and fewer, then up to 16)
@pytest.mark.parametrize("mixed,N", [(True, 44), (False, 34)])
def test_newton_step_on_long_vectors(fsi, mixed, N):
    import torch
    from paper_2601_08266_gb300 import inputs
    n, m = (N + 1) ** 3, 20000
    rng = np.random.default_rng(2)
    ax = np.arange(N + 1) / N
    Z, Y, X = np.meshgrid(ax, ax, ax, indexing="ij")
    X, Y, Z = X.ravel(), Y.ravel(), Z.ravel()
    wall = (Y < 1e-12) | (Y > 1 - 1e-12) | (Z < 1e-12) | (Z > 1 - 1e-12)
    inflow = (X < 1e-12) & ~wall
    mask = np.zeros((n, 4), dtype=np.uint8)
    mask[wall | inflow, :3] = 1
    prof = 16 * Y * (1 - Y) * Z * (1 - Z)
    Vn = np.zeros((n, 4))
    Vn[:, 0] = prof
    Vn[:, :3] += 0.05 * rng.normal(size=(n, 3))
    Vn[mask[:, 0].astype(bool), :3] = 0
    Vn[inflow, 0] = prof[inflow]
    f64 = lambda a: precond_case.T(a, torch.float64)
    mesh = fsi.Mesh(N, rho=1.0, mu=1e-3, dt=1e-3, rho_inf=0.5, device=0)
    e = torch.empty(m, dtype=torch.int32, device="cuda")
    xi = torch.empty((m, 3), dtype=torch.float64, device="cuda")
    cs = torch.empty(N ** 3 + 1, dtype=torch.int32, device="cuda")
    pm = torch.empty(m, dtype=torch.int32, device="cuda")
    fsi.fsi_locate(mesh, f64(inputs.leaflet_points(m, seed=5)), e, xi, cs, pm)
    y = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    keep = [f64(Vn), f64(np.zeros((n, 4))), precond_case.T(mask, torch.uint8),
            f64(np.zeros((n, 4))), torch.full((m,), 0.024 / m, dtype=torch.float64, device="cuda")]
    st = fsi.StepState(y, keep[0], keep[1], mask=keep[2], yD=keep[3], elem=e, xi=xi, cell_start=cs,
                       perm=pm, w=keep[4], drho_s=0.5)
    code, rep = fsi.fsi_newton_step(mesh, st, mixed=mixed, restart=50, max_newton=10, max_krylov=400,
                                    newton_rtol=1e-8, krylov_rtol=1e-3, precond=fsi.PRECOND_SCHUR)
    assert code == 0 and rep["converged"] == 1
    assert rep["krylov_iters"] <= 20 * rep["newton_iters"], rep  # ~10 a solve; no stagnation
    R = torch.empty_like(y)
    fsi.fsi_coupled_residual(mesh, st, R)
    torch.cuda.synchronize()
    assert R.norm().item() <= 1.01e-8 * rep["r_ref"]
    mesh.close()
