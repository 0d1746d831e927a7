"""The Krylov solver's parts that change with a size: the V-cycle's coarse levels
by their shape."""
import numpy as np
import pytest

import test_gpu_precond as precond_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2601_08266_gb300 as pkg
    return pkg


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
