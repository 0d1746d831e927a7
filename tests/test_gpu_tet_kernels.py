"""Tetrahedral kernels at the sizes where their route or their launch shape
changes: the VMS operators by element count, the location by point count."""
import numpy as np
import pytest

import test_gpu_tet as case
from test_gpu_tet import fsi, tet  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


# 9,984 | 10,032 elements (FP32 and FP64: lanes | a thread per element) and 24,480 |
# 25,920 (double-float); the last CTA is ragged
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
@pytest.mark.parametrize("N", [(8, 13, 16), (19, 11, 8), (17, 16, 15), (16, 15, 18)])
def test_tet_vms_by_element_count(fsi, tet, oracle, prec, N):
    mesh, X, Tt, p = case.make(fsi, N, seed=sum(N), rho=1.3, mu=0.02, dt=0.01, rho_inf=0.3,
                               has_s=sum(N) % 2 == 0)
    n = mesh.n_nodes
    rng = np.random.default_rng(sum(N) + 1)
    U = rng.uniform(-2, 2, (n, 4))
    U[rng.random(n) < 0.1] = 0.0
    A = rng.uniform(-1, 1, (n, 4))
    A[:, 3] = rng.uniform(1.0, 50.0, n)
    f, x = rng.normal(size=(n, 4)), rng.normal(size=(n, 4))
    U, A, f, x = (case.cast(prec, a) for a in (U, A, f, x))
    R, Jx = case.vms(fsi, mesh, prec, U, A, f, x)
    om = tet.TetMesh(case.cast(prec, X), Tt)
    c_a, c_v = oracle.timeint.chain_factors(p["rho_inf"], p["dt"])
    assert case.rel(R, tet.residual(om, p, U, A, f=f)) < case.TOL[prec]
    assert case.rel(Jx, tet.jacobian_apply(om, p, U, A, x, c_a, c_v, f=f)) < case.TOL[prec]
    mesh.close()


@pytest.mark.parametrize("m", [1, 3, 5, 129, 12_001, 40_003])
def test_tet_locate_by_point_count(fsi, tet, m):
    """Elements, coordinates and the table bit for bit, with 4, 8 and 16 points a
    warp; a tenth of the points on nodes (many holders), a tenth outside."""
    mesh, X, Tt, _ = case.make(fsi, (5, 4, 3), seed=7, perturb=0.25)
    om = tet.TetMesh(X, Tt)
    rng = np.random.default_rng(m)
    P = rng.uniform(0.0, 1.0, (m, 3))
    k = m // 10
    P[:k] = X[rng.integers(0, len(X), k)]
    P[k:2 * k] += 1.5
    P = P[rng.permutation(m)]
    e, l3, cs, perm, nout, _ = case.locate_gpu(fsi, mesh, P)
    eo, lo, nouto = tet.locate(om, P)
    assert nout == nouto
    assert np.array_equal(e, eo) and np.array_equal(l3, lo)
    cso, permo = tet.cell_hash(om, eo)
    assert np.array_equal(cs, cso) and np.array_equal(perm, permo)
    mesh.close()
