"""Spreading and location where their launch shapes change: grids whose cell segments
outnumber the resident CTAs, elements with few and many points a lane, more points than
the tetrahedral location has warps for.  Bars as in test_gpu_parity.py."""
import numpy as np
import pytest

import test_gpu_tet as case
from test_gpu_tet import fsi, tet  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


# 172,032 cells (21,504 segments: more than 64 CTAs of two warps, or 32 of four, per SM
# take at once) with a few points, and with more than a point per segment
@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("m", [3, 21_503, 21_504, 60_000])
def test_structured_spread_on_a_large_grid(fsi, oracle, prec, m):
    import torch
    N = (64, 56, 48)
    mesh, grid = fsi.Mesh(N, device=0), oracle.core.Grid(N)
    rng = np.random.default_rng(m)
    X = rng.uniform(0.02, 0.98, (m, 3))
    e = torch.empty(m, dtype=torch.int32, device="cuda")
    xi = torch.empty((m, 3), dtype=torch.float64, device="cuda")
    cs = torch.empty(mesh.n_elems + 1, dtype=torch.int32, device="cuda")
    pm = torch.empty(m, dtype=torch.int32, device="cuda")
    fsi.fsi_locate(mesh, case.T(X), e, xi, cs, pm)
    dt = case.dtype_of(prec)
    lam = case.cast(prec, rng.uniform(0.5, 1.5, (m, 3)))
    F = torch.zeros((mesh.n_nodes, 4), dtype=dt, device="cuda")
    fsi.fsi_dlm_spread(mesh, case.PREC(fsi, prec), e, xi.to(dt), cs, pm, case.T(lam, dt), None, F, False)
    torch.cuda.synchronize()
    Fo = oracle.core.spread(grid, e.cpu().numpy(), case.cast(prec, case.H(xi)), lam)
    assert case.rel(case.H(F)[:, :3], Fo[:, :3]) < case.TOL[prec]
    mesh.close()


# six elements: lanes (a quarter of an element's points) with none, one, two, three and
# many points, with and without weights
@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("m", [1, 4, 20, 50, 90, 1000])
def test_tet_spread_by_points_per_element(fsi, tet, prec, m):
    import torch
    mesh, X, Tt, _ = case.make(fsi, (1, 1, 1), seed=2, perturb=0.0)
    om = tet.TetMesh(X, Tt)
    rng = np.random.default_rng(m)
    e, l3, _, _, _, (ed, ld, csd, pmd) = case.locate_gpu(fsi, mesh, rng.uniform(0.05, 0.95, (m, 3)))
    dt = case.dtype_of(prec)
    lv, w = (case.cast(prec, rng.uniform(0.5, 1.5, s)) for s in ((m, 3), m))
    for wt in (None, w):
        F = torch.zeros((om.n_nodes, 4), dtype=dt, device="cuda")
        fsi.fsi_tet_spread(mesh, case.PREC(fsi, prec), ed, ld.to(dt), csd, pmd, case.T(lv, dt),
                           None if wt is None else case.T(wt, dt), F, False)
        torch.cuda.synchronize()
        Fo = tet.spread(om, e, case.cast(prec, l3), lv, w=wt)
        assert case.rel(case.H(F)[:, :3], Fo[:, :3]) < case.TOL[prec]
    mesh.close()


def test_tet_locate_more_points_than_warps(fsi):
    """A point's element and coordinates do not depend on the other points: one call
    with warps that take several groups of points has the bits of calls with fewer."""
    mesh, _, _, _ = case.make(fsi, (5, 4, 3), seed=7, perturb=0.25)
    P = np.random.default_rng(0).uniform(-0.05, 1.05, (330_001, 3))
    e, l3, cs, pm, nout, _ = case.locate_gpu(fsi, mesh, P)
    parts = [case.locate_gpu(fsi, mesh, q) for q in np.array_split(P, 11)]
    assert np.array_equal(e, np.concatenate([p[0] for p in parts]))
    assert np.array_equal(l3, np.concatenate([p[1] for p in parts]))
    assert nout == sum(p[4] for p in parts)
    mesh.close()
