"""Kernels of a chain overlap the end of the one before.  Back-to-back calls on
changing inputs, without a synchronisation, on arrays that share memory sectors,
and replayed from a CUDA graph, give the bits of each call by itself on arrays of
its own."""
import numpy as np
import pytest

import test_gpu_tet as tet_case
from test_gpu_tet import fsi  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

K = 4  # different inputs


class Pack:
    """Arrays in one allocation, each right behind the one before (8-byte steps)."""

    def __init__(self, nbytes):
        import torch
        self.buf, self.at = torch.zeros(nbytes, dtype=torch.uint8, device="cuda"), 0

    def __call__(self, shape, dtype):
        import torch
        size = int(np.prod(shape)) * torch.empty(0, dtype=dtype).element_size()
        t = self.buf[self.at:self.at + size].view(dtype).view(shape)
        self.at += (size + 7) // 8 * 8
        return t


def own(shape, dtype):
    import torch
    return torch.zeros(shape, dtype=dtype, device="cuda")


def replayed(fn, stream, outs, want):
    """fn(stream) captured once and replayed gives the tensors `want` in `outs`."""
    import torch
    fn()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        fn()
    for _ in range(3):
        for o in outs:
            o.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(o, w) for o, w in zip(outs, want))


# m = 5, 101: the rank pass is the cell table's last kernel, and a caller's kernel follows
# it; the odd counts leave neighbouring arrays in one sector
@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("N,m", [((2, 2, 2), 5), ((5, 4, 3), 101), ((13, 9, 7), 3001),
                                 ((24, 24, 24), 60001)])
def test_coupling_chain(fsi, prec, N, m):
    import torch
    P, dt = tet_case.PREC(fsi, prec), tet_case.dtype_of(prec)
    rng = np.random.default_rng(m)
    side = torch.cuda.Stream()
    mesh = fsi.Mesh(N, device=0, stream=side.cuda_stream)
    n, E = mesh.n_nodes, mesh.n_elems
    X = [tet_case.T(rng.uniform(-0.02, 1.02, (m, 3))) for _ in range(K)]
    U = [tet_case.T(rng.normal(size=(n, 4)), dt) for _ in range(K)]
    A = [tet_case.T(np.abs(rng.normal(size=(n, 4))) + 1.0, dt) for _ in range(K)]

    def arrays(new):
        # xi in FP64 as located; the FP32 operators take coordinates of their own below
        i32 = torch.int32
        return dict(R=own((n, 4), dt), elem=new((m,), i32), xi=new((m, 3), torch.float64),
                    elem2=new((m,), i32), xi2=new((m, 3), torch.float64),
                    cs=new((E + 1,), i32), perm=new((m,), i32), u=new((m, 3), dt),
                    F=own((n, 4), dt))

    xi32 = [tet_case.T(rng.uniform(-1, 1, (m, 3)), dt) for _ in range(K)]

    def chain(q, a, sync):
        """residual; location; table; u = C^T R; F = C u"""
        done = torch.cuda.synchronize if sync else (lambda: None)
        fsi.fsi_residual(mesh, P, U[q], A[q], None, a["R"])
        done()
        fsi.fsi_locate(mesh, X[q], a["elem2"], a["xi2"], want_outside=False)
        done()
        fsi.fsi_dlm_interp(mesh, P, a["elem2"], xi32[q] if prec == "f32" else a["xi2"], U[q], a["u"])
        done()
        fsi.fsi_locate(mesh, X[q], a["elem"], a["xi"], a["cs"], a["perm"], want_outside=False)
        done()
        xi = xi32[q] if prec == "f32" else a["xi"]
        fsi.fsi_dlm_spread(mesh, P, a["elem"], xi, a["cs"], a["perm"], a["u"], None, a["F"], False)
        done()
        fsi.fsi_dlm_interp(mesh, P, a["elem"], xi, a["R"], a["u"])
        done()
        fsi.fsi_dlm_spread(mesh, P, a["elem"], xi, a["cs"], a["perm"], a["u"], None, a["F"], True)
        done()

    alone = [arrays(own) for _ in range(K)]
    torch.cuda.synchronize()
    for q in range(K):
        chain(q, alone[q], True)
    size = sum(v.numel() * v.element_size() + 8 for v in alone[0].values())
    sets = [arrays(Pack(size)) for _ in range(6 * K)]
    torch.cuda.synchronize()
    for k, a in enumerate(sets):
        chain(k % K, a, False)
    torch.cuda.synchronize()
    for k, a in enumerate(sets):
        for name, w in alone[k % K].items():
            assert torch.equal(a[name], w), (k, name)

    def both():
        chain(0, sets[0], False)
        chain(1, sets[1], False)
    replayed(both, side, [s[v] for s in sets[:2] for v in s],
             [alone[q][v] for q in (0, 1) for v in alone[q]])
    mesh.close()


@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("N", [(3, 2, 2), (19, 16, 15)])
def test_tetrahedral_chain(fsi, prec, N):
    import torch
    P, dt = tet_case.PREC(fsi, prec), tet_case.dtype_of(prec)
    mesh, X, Tt, _ = tet_case.make(fsi, N, seed=3)
    side = torch.cuda.Stream()
    meshes = [mesh, fsi.TetMesh(tet_case.T(X), tet_case.T(Tt), device=0, stream=side.cuda_stream)]
    n, E, m = X.shape[0], Tt.shape[0], 2001
    rng = np.random.default_rng(4)
    U = [tet_case.T(rng.normal(size=(n, 4)), dt) for _ in range(K)]
    A = [tet_case.T(np.abs(rng.normal(size=(n, 4))) + 1.0, dt) for _ in range(K)]
    Q = [tet_case.T(rng.uniform(0, 1, (m, 3))) for _ in range(K)]
    lam = [tet_case.T(rng.uniform(0, 0.3, (m, 3)), dt) for _ in range(K)]

    def arrays():
        i32 = torch.int32
        return dict(R=own((n, 4), dt), J=own((n, 4), dt), elem=own((m,), i32),
                    l3=own((m, 3), torch.float64), cs=own((E + 1,), i32), perm=own((m,), i32),
                    F=own((n, 4), dt))

    def chain(q, a, sync, mm):
        done = torch.cuda.synchronize if sync else (lambda: None)
        fsi.fsi_tet_residual(mm, P, U[q], A[q], None, a["R"])
        done()
        fsi.fsi_tet_jacobian_apply(mm, P, a["R"], A[q], None, U[q], a["J"])
        done()
        fsi.fsi_tet_locate(mm, Q[q], a["elem"], a["l3"], a["cs"], a["perm"], want_outside=False)
        done()
        fsi.fsi_tet_spread(mm, P, a["elem"], lam[q], a["cs"], a["perm"], lam[(q + 1) % K], None,
                           a["F"], False)
        done()

    alone = [arrays() for _ in range(K)]
    for q in range(K):
        chain(q, alone[q], True, mesh)
    sets = [arrays() for _ in range(6 * K)]
    torch.cuda.synchronize()
    for k, a in enumerate(sets):
        chain(k % K, a, False, mesh)
    torch.cuda.synchronize()
    for k, a in enumerate(sets):
        for name, w in alone[k % K].items():
            assert torch.equal(a[name], w), (k, name)

    def both():
        chain(0, sets[0], False, meshes[1])
        chain(1, sets[1], False, meshes[1])
    replayed(both, side, [s[v] for s in sets[:2] for v in s],
             [alone[q][v] for q in (0, 1) for v in alone[q]])


@pytest.mark.parametrize("B", [3, 129, 1000])
def test_training_chain(fsi, B):
    import torch
    from oracle import mlp as om
    rng = np.random.default_rng(B)
    f32 = torch.float32
    theta = tet_case.T(om.flatten(om.init_params(3)), f32)
    X = [tet_case.T(rng.normal(size=(B, om.N_IN)), f32) for _ in range(K)]
    Y = [tet_case.T(rng.normal(size=(B, om.N_OUT)), f32) for _ in range(K)]
    side = torch.cuda.Stream()
    h = fsi.Mlp(1024, stream=side.cuda_stream)

    def train(a, sync):
        for q in range(2 * K):
            fsi.fsi_mlp_loss_grad(h, a["p"], X[q % K], Y[q % K], a["loss"], a["g"])
            if sync:
                torch.cuda.synchronize()
            fsi.fsi_mlp_adam(h, a["p"], a["g"], a["m"], a["v"], q + 1)
            if sync:
                torch.cuda.synchronize()
        fsi.fsi_mlp_forward(h, a["p"], X[0], a["out"])

    def arrays(new):
        a = {k: new((theta.numel(),), f32) for k in ("p", "g", "m", "v")}
        a["loss"], a["out"] = new((1,), f32), new((B, om.N_OUT), f32)
        a["p"].copy_(theta)
        return a

    alone = arrays(own)
    torch.cuda.synchronize()
    train(alone, True)
    torch.cuda.synchronize()
    for _ in range(3):
        a = arrays(Pack(4 * (4 * theta.numel() + 4 * B) + 64))
        torch.cuda.synchronize()
        train(a, False)
        torch.cuda.synchronize()
        for name, w in alone.items():
            assert torch.equal(a[name], w), name

    def restart():
        a["p"].copy_(theta)
        a["m"].zero_()
        a["v"].zero_()
        train(a, False)
    with torch.cuda.stream(side):
        replayed(restart, side, list(a.values()), list(alone.values()))
    h.check()
