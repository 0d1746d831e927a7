"""The VMS kernels under every kind of brick schedule: single elements, columns
taller than the grid, bricks wider than a CTA has lanes for, bricks whose shared
memory has to be halved, partial warps, and the default schedule of grids from
one element to several bricks.  Bars as in test_gpu_parity.py."""
import numpy as np
import pytest

import parity

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5, "df64": 1e-11}
BRICKS = [None, (1, 1, 1, 32), (1, 1, 64, 32), (97, 1, 1, 256), (8, 8, 6, 256), (3, 5, 2, 64),
          (16, 16, 1, 256), (2, 1, 100, 32)]


@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("N", [(1, 1, 1), (1, 2, 17), (9, 1, 2), (13, 10, 9), (33, 5, 4)])
def test_brick_schedules(oracle, prec, N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2601_08266_gb300 as fsi
    P = {"f64": fsi.FSI_F64, "f32": fsi.FSI_F32, "df64": fsi.FSI_DF64}[prec]
    dt = torch.float32 if prec == "f32" else torch.float64
    h, x0 = (0.07, 0.11, 0.09), (0.2, -0.1, 0.4)
    p = dict(rho=1.3, mu=0.02, dt=0.01, rho_inf=0.3, has_s=True)
    grid = oracle.core.Grid(N, x0=x0, h=h)
    mesh = fsi.Mesh(N, x0=x0, h=h, **p, device=0)
    rng = np.random.default_rng(17)
    n = mesh.n_nodes
    U, A, f, x = (rng.uniform(-1, 1, (n, 4)) for _ in range(4))
    A[:, 3] = rng.uniform(1.0, 30.0, n)
    if prec == "f32":
        U, A, f, x = (a.astype(np.float32).astype(np.float64) for a in (U, A, f, x))
    c_a, c_v = oracle.timeint.chain_factors(p["rho_inf"], p["dt"])
    Rref = oracle.core.residual(grid, p, U, A, f=f)
    Jref = oracle.core.jacobian_apply(grid, p, U, A, x, c_a, c_v, f=f)
    Ud, Ad, fd, xd = (torch.as_tensor(a, device="cuda").to(dt) for a in (U, A, f, x))
    for b in BRICKS:
        if b:
            for op in (0, 1, 2):
                fsi.fsi_mesh_set_brick(mesh, op, P, *b)
        R1, J1, R2, J2 = (torch.full_like(Ud, float("nan")) for _ in range(4))
        fsi.fsi_residual(mesh, P, Ud, Ad, fd, R1)
        fsi.fsi_jacobian_apply(mesh, P, Ud, Ad, fd, xd, J1)
        fsi.fsi_residual_jacobian_apply(mesh, P, Ud, Ad, fd, xd, R2, J2)
        for got, ref in ((R1, Rref), (J1, Jref), (R2, Rref), (J2, Jref)):
            e = parity.rel_local(got.double().cpu().numpy(), ref, N)
            assert e < TOL[prec], (b, e)
    mesh.close()


# as include/fsi.h states them
@pytest.mark.parametrize("prec,op,most", [("f64", 0, 800), ("f64", 2, 400), ("df64", 1, 800),
                                          ("df64", 2, 400), ("f32", 1, 1600), ("f32", 2, 800)])
def test_brick_size_limit(prec, op, most):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2601_08266_gb300 as fsi
    P = {"f64": fsi.FSI_F64, "f32": fsi.FSI_F32, "df64": fsi.FSI_DF64}[prec]
    mesh = fsi.Mesh((3, 2, 2), device=0)
    for b in [(most // 8, 4, 2), (1, 1, most), (20, most // 20, 1)]:
        fsi.fsi_mesh_set_brick(mesh, op, P, *b, 128)
    for b in [(most // 8, 4, 3), (1, 1, most + 1), (2 ** 20, 2 ** 20, 2 ** 20), (2 ** 30, 4, 1)]:
        with pytest.raises(fsi.FsiError, match=f"more than {most} elements"):
            fsi.fsi_mesh_set_brick(mesh, op, P, *b, 128)
    mesh.close()
