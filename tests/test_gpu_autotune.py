"""The autotuners start from the schedule that the handle has: it is the first
candidate, so a call never leaves a slower one behind."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2601_08266_gb300 as pkg
    return pkg


# a schedule outside the fixed list; one of the list, asked for with more threads than
# run; one whose shared memory is too large in FP64 with both operators, halved
@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("op", [0, 1, 2])
@pytest.mark.parametrize("brick,runs", [((3, 5, 2, 64), (3, 5, 2, 64)),
                                        ((4, 4, 4, 256), (4, 4, 4, 64)),
                                        ((1, 1, 100, 32), None)])
def test_mesh_autotune_starts_from_the_present_brick(fsi, op, prec, brick, runs):
    P = {"f64": fsi.FSI_F64, "f32": fsi.FSI_F32, "df64": fsi.FSI_DF64}[prec]
    mesh = fsi.Mesh((8, 8, 8), device=0)
    fsi.fsi_mesh_set_brick(mesh, op, P, *brick)
    t = fsi.fsi_mesh_autotune(mesh, op, P, reps=2)
    c = t["candidates"]
    if runs:
        assert (c[0][0], c[0][1]) == (runs[:3], runs[3])
    else:
        assert c[0][0][:2] == brick[:2] and c[0][1] == 32
    assert len({(b, n) for b, n, _ in c}) == len(c) == 10   # no launch timed twice
    assert all(n <= 128 for _, n, _ in c)                   # the threads that run
    assert t["seconds"] <= c[0][2]
    # the default or the choice of an earlier call is the next one's first candidate
    again = fsi.fsi_mesh_autotune(mesh, op, P, reps=2)["candidates"][0]
    assert (again[0], again[1]) == (t["brick"], t["threads"])
    mesh.close()


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_batch_autotune_starts_from_the_present_schedule(fsi, prec):
    import torch
    P, dt = (fsi.FSI_F64, torch.float64) if prec == "f64" else (fsi.FSI_F32, torch.float32)
    s = torch.cuda.Stream()
    meshes, items = [], []
    for N in [(3, 5, 2), (6, 2, 7), (5, 5, 5)]:
        mesh = fsi.Mesh(N, device=0, stream=s.cuda_stream)
        nodal = lambda: torch.rand((mesh.n_nodes, 4), dtype=dt, device="cuda")
        it = {k: nodal() for k in ("U", "A", "x", "R", "Jx", "F")}
        it["cell_start"] = torch.zeros(mesh.n_elems + 1, dtype=torch.int32, device="cuda")
        meshes.append(mesh)
        items.append(it)
    torch.cuda.synchronize()
    b = fsi.Batch(meshes, items, P, s.cuda_stream)
    t = b.autotune(reps=2)
    c = t["candidates"]
    # grids this small start with bricks of their own size, which the fixed list
    # (at least 4 x 4 x 4) does not hold
    assert c[0][0] * c[0][1] * c[0][2] < 64 and c[0][3] == 4
    assert len({k[:4] for k in c}) == len(c)
    assert t["seconds"] <= c[0][4]
    again = b.autotune(reps=2)["candidates"][0]
    assert (again[:3], again[3]) == (t["brick"], t["ctas_per_sm"])
    b.close()
    for m in meshes:
        m.close()
