"""The work that users of this framework have it do, as cases to be timed.

Every case goes through the public entry points of ``paper_2601_08266_gb300``
with the default schedules (nothing autotuned).  Kinds of cases:

* ``step``    one operator step on a uniform grid: generalized-alpha stage, VMS
              residual and/or Jacobian apply, location of the solid points with the
              cell table, interpolation, spreading, in one of the precisions.
* ``newton``  one implicit step of a channel flow with three immersed leaflets
              (point masses, or the hyperelastic body), Schur preconditioner.
* ``coupled`` what a caller's own nonlinear solver asks for on a mapped grid:
              location, coupled residual, one coupled Jacobian apply.
* ``tet``     the operator step on an unstructured tetrahedral mesh.
* ``batch``   one batched step of an ensemble of uneven instances (CUDA graph).
* ``train``   one training iteration of the initial-guess network.
* ``predict`` the network's Newton predictor on a whole grid.

``exact`` states the same results in 64-bit torch from the definitions: element
loops as einsums over explicit shape-function tables, the Jacobian apply as the
forward-mode derivative of the residual.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2601_08266_gb300 as fsi
from paper_2601_08266_gb300 import inputs

DEV = torch.device("cuda:0")
F64 = torch.float64
PREC = {"f64": fsi.FSI_F64, "df64": fsi.FSI_DF64, "f32": fsi.FSI_F32}
DT, RHO_INF = 1e-3, 0.5
AM = 0.5 * (3.0 - RHO_INF) / (1.0 + RHO_INF)
AF = 1.0 / (1.0 + RHO_INF)
GAM = 0.5 + AM - AF


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: the 8^3 grid of the smoke test with its 500 ball points
        dict(name="step_f64_8", kind="step", prec="f64", op="both", nx=8, ny=8, nz=8, m=500,
             points="ball", extras=False),
        # the benchmark's step: 64^3, 200 k leaflet points, native FP64
        dict(name="step_f64_64", kind="step", prec="f64", op="both", nx=64, ny=64, nz=64,
             m=200_000, points="leaflets", extras=False),
        # FP64-accurate double-float on a ragged grid, with the interface
        # scaling s and a body force
        dict(name="step_df64_ragged", kind="step", prec="df64", op="both", nx=47, ny=61, nz=38,
             m=60_001, points="leaflets", extras=True),
        # the Krylov operator of the mixed solver at the size of its largest
        # runs: FP32 Jacobian apply and coupling, 128^3 with 1 M points
        dict(name="step_f32_128", kind="step", prec="f32", op="jac", nx=128, ny=128, nz=128,
             m=1_000_000, points="leaflets", extras=False),
        # an implicit step of an ordinary small run, where launches count
        dict(name="newton_mixed_32", kind="newton", mixed=True, n=32, m=25_000, body=False),
        # the largest implicit step: 128^3 channel, 8.6 M unknowns, 1 M points
        dict(name="newton_mixed_128", kind="newton", mixed=True, n=128, m=1_000_000, body=False),
        # the plain FP64 solver with the hyperelastic leaflets, as in validation runs
        dict(name="newton_f64_body_24", kind="newton", mixed=False, n=24, m=0, body=True),
        # a user's own solver on a mapped grid with ragged extents
        dict(name="coupled_mapped", kind="coupled", nx=52, ny=45, nz=48, m=75_000),
        # unstructured background mesh, FP64-accurate operators
        dict(name="tet_df64", kind="tet", prec="df64", nx=36, ny=36, nz=36, m=50_000),
        # the ensemble of the benchmark: 64 uneven instances, FP32, one graph
        dict(name="batch_f32_64", kind="batch", prec="f32", count=64, lo=16, hi=48),
        # one training iteration at the training batch size
        dict(name="train_4096", kind="train", rows=4096),
        # the predictor of the largest implicit step
        dict(name="predict_128", kind="predict", nx=128, ny=128, nz=128),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "newton", "coupled", "tet", "batch", "train",
                       "predict"])
    if kind == "step":
        prec = rng.choice(["f64", "df64", "f32"])
        cap = {"f64": 64 ** 3, "df64": 96 ** 3, "f32": 128 ** 3}[prec]
        n = [_logint(rng, 6, 128) for _ in range(3)]
        while n[0] * n[1] * n[2] > cap:
            k = n.index(max(n))
            n[k] = max(6, int(n[k] * 0.8))
        E = n[0] * n[1] * n[2]
        m = _logint(rng, 300, max(600, min(1_000_000, E)))
        return dict(kind="step", prec=prec, op=rng.choice(["both", "jac", "res"]), nx=n[0],
                    ny=n[1], nz=n[2], m=m, points=rng.choice(["ball", "leaflets"]),
                    extras=rng.random() < 0.5)
    if kind == "newton":
        mixed = rng.random() < 0.7
        return dict(kind="newton", mixed=mixed, n=_logint(rng, 12, 72 if mixed else 24),
                    m=_logint(rng, 1000, 200_000), body=rng.random() < 0.3)
    if kind == "coupled":
        return dict(kind="coupled", nx=_logint(rng, 12, 64), ny=_logint(rng, 12, 64),
                    nz=_logint(rng, 12, 64), m=_logint(rng, 1000, 200_000))
    if kind == "tet":
        return dict(kind="tet", prec=rng.choice(["f64", "df64", "f32"]), nx=_logint(rng, 6, 36),
                    ny=_logint(rng, 6, 36), nz=_logint(rng, 6, 36), m=_logint(rng, 500, 50_000))
    if kind == "batch":
        lo = rng.randint(8, 24)
        return dict(kind="batch", prec=rng.choice(["f32", "f32", "f64"]),
                    count=_logint(rng, 4, 64), lo=lo, hi=lo + rng.randint(4, 20))
    if kind == "train":
        return dict(kind="train", rows=_logint(rng, 256, 16384))
    return dict(kind="predict", nx=_logint(rng, 16, 128), ny=_logint(rng, 16, 128),
                nz=_logint(rng, 16, 128))


# ------------------------------------------------------------------ inputs
class Gen:
    """Draws on the GPU from one seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 1)

    def normal(self, *shape, dtype=F64):
        return torch.randn(shape, dtype=dtype, device=DEV, generator=self.g)

    def uniform(self, lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, dtype=F64, device=DEV, generator=self.g)

    def fourier(self, N, ncomp=4, noise=0.01):
        """Smooth nodal field: separable sinusoids of wavenumbers 1..8, max 1."""
        k = torch.arange(1, 9, dtype=F64, device=DEV)
        out = torch.empty(((N[0] + 1) * (N[1] + 1) * (N[2] + 1), ncomp), dtype=F64, device=DEV)
        for c in range(ncomp):
            S = []
            for d in range(3):
                t = torch.arange(N[d] + 1, dtype=F64, device=DEV) / N[d]
                S.append(torch.sin(2 * math.pi * t[None, :] * k[:, None]
                                   + self.uniform(0, 2 * math.pi, 8, 1)))
            amp = self.normal(8, 8, 8) / (1 + k[:, None, None] ** 2 + k[None, :, None] ** 2
                                          + k[None, None, :] ** 2)
            f = torch.einsum("abc,xa,yb,zc->zyx", amp, S[0].T, S[1].T, S[2].T)
            f = f / f.abs().max() + noise * self.normal(*f.shape)
            out[:, c] = f.reshape(-1)
        return out

    def points(self, m, kind):
        """m points in a ball, or in three thin leaflets (cylindrical sectors)."""
        if kind == "ball":
            d = self.normal(m, 3)
            d = d / d.norm(dim=1, keepdim=True)
            return 0.5 + 0.3 * self.uniform(0, 1, m, 1) ** (1 / 3) * d
        th0 = self.uniform(0, 2 * math.pi, 1)
        which = torch.randint(0, 3, (m,), device=DEV, generator=self.g)
        half = 0.5 * 0.5 / 0.3
        r = torch.sqrt(self.uniform(0.29 ** 2, 0.31 ** 2, m))
        th = th0 + which * (2 * math.pi / 3) + self.uniform(-half, half, m)
        x = self.uniform(0.1, 0.9, m)
        return torch.stack([x, 0.5 + r * torch.cos(th), 0.5 + r * torch.sin(th)], 1).contiguous()


def _dims(c):
    return (c["nx"], c["ny"], c["nz"])


def _nodes(N):
    """Coordinates [n, 3] of the nodes of the unit box, x fastest."""
    ax = [torch.arange(N[d] + 1, dtype=F64, device=DEV) / N[d] for d in range(3)]
    Z, Y, X = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    return torch.stack([X.reshape(-1), Y.reshape(-1), Z.reshape(-1)], 1).contiguous()


def _i32(n):
    return torch.zeros(n, dtype=torch.int32, device=DEV)


def _step_inputs(c, seed):
    N, g = _dims(c), Gen(seed)
    d = dict(y=g.fourier(N), Vn=g.fourier(N), An=g.fourier(N))
    n = d["y"].shape[0]
    d["x"] = g.uniform(-1, 1, n, 4)
    d["X"] = g.points(c["m"], c["points"])
    d["lam"] = g.normal(c["m"], 3)
    d["s"] = d["f"] = None
    if c["extras"]:
        # s = 100 around the solid, 1 elsewhere (what fsi_interface_scaling makes)
        r = (_nodes(N)[:, 1:] - 0.5).norm(dim=1)
        d["s"] = torch.where((r - 0.3).abs() < 0.03, 100.0, 1.0).to(F64).contiguous()
        d["f"] = g.fourier(N)
    if c["prec"] == "f32":
        d = {k: v if v is None or k == "X" else v.float() for k, v in d.items()}
    return d


def _channel(N, seed):
    """Channel on the unit cube: inflow at x = 0, no-slip walls, free outflow."""
    g = Gen(seed)
    P = _nodes(N)
    X, Y, Z = P[:, 0], P[:, 1], P[:, 2]
    prof = 16 * Y * (1 - Y) * Z * (1 - Z)
    wall = (Y < 1e-12) | (Y > 1 - 1e-12) | (Z < 1e-12) | (Z > 1 - 1e-12)
    inflow = (X < 1e-12) & ~wall
    fixed = wall | inflow
    Vn = torch.zeros((P.shape[0], 4), dtype=F64, device=DEV)
    Vn[:, 0] = prof
    Vn[:, :3] += 0.01 * g.fourier(N, 3, 0.0)
    Vn[fixed, :3] = 0.0
    # the inflow ramps up by half a per cent in this step
    Vn[inflow, 0] = prof[inflow]
    gD = torch.zeros((P.shape[0], 3), dtype=F64, device=DEV)
    gD[inflow, 0] = 1.005 * prof[inflow]
    yD = torch.zeros_like(Vn)
    yD[:, :3] = (gD - Vn[:, :3]) / (GAM * DT)
    mask = torch.zeros(Vn.shape, dtype=torch.uint8, device=DEV)
    mask[fixed, :3] = 1
    y0 = torch.where(mask.bool(), yD, torch.zeros_like(yD))
    return g, dict(Vn=Vn, An=torch.zeros_like(Vn), yD=yD, mask=mask, y0=y0)


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def _prepare_step(c, seed):
    N, d = _dims(c), _step_inputs(c, seed)
    mesh = fsi.Mesh(N, rho=1.0, mu=0.01, dt=DT, rho_inf=RHO_INF, has_s=c["extras"])
    o = {k: torch.zeros_like(d["y"]) for k in ("U", "A", "R", "Jx", "F")}
    xi = torch.zeros((c["m"], 3), dtype=F64, device=DEV)
    o.update(elem=_i32(c["m"]), xi=xi, cs=_i32(mesh.n_elems + 1), perm=_i32(c["m"]),
             u=torch.zeros_like(d["lam"]))
    return dict(kind="step", c=c, mesh=mesh, d=d, o=o)


def _prepare_newton(c, seed):
    N = (c["n"],) * 3
    g, d = _channel(N, seed)
    mesh = fsi.Mesh(N, rho=1.0, mu=1e-3, dt=DT, rho_inf=RHO_INF)
    kw = {}
    body = None
    if c["body"]:
        X, conn = inputs.leaflet_hex_mesh(2, 2 * c["n"], 3 * c["n"], seed=int(seed) % (1 << 31))
        P = torch.as_tensor(X, device=DEV)
        body = fsi.Solid(mesh, P, torch.as_tensor(conn, device=DEV), 1.2, 50.0, 500.0)
        z = [torch.zeros_like(P) for _ in range(3)]
        kw = dict(body=body, us=z[0], vs=z[1], as_=z[2], g_s=(0.0, 0.0, -1.0))
    else:
        P = g.points(c["m"], "leaflets")
        kw = dict(w=torch.full((c["m"],), 0.024 / c["m"], dtype=F64, device=DEV), drho_s=0.5)
    m = P.shape[0]
    e, xi, cs, pm = (_i32(m), torch.zeros((m, 3), dtype=F64, device=DEV),
                     _i32(mesh.n_elems + 1), _i32(m))
    fsi.fsi_locate(mesh, P, e, xi, cs, pm)
    y = torch.empty_like(d["y0"])
    st = fsi.StepState(y, d["Vn"], d["An"], mask=d["mask"], yD=d["yD"], elem=e, xi=xi,
                       cell_start=cs, perm=pm, **kw)
    return dict(kind="newton", c=c, mesh=mesh, body=body, st=st, y=y, y0=d["y0"])


def _coupled_inputs(c, seed):
    N = _dims(c)
    g, d = _channel(N, seed)
    P = _nodes(N)
    b = torch.sin(2 * math.pi * P[:, 0]) * torch.sin(2 * math.pi * P[:, 1]) * torch.sin(
        2 * math.pi * P[:, 2])
    d["coords"] = (P + 0.02 * b[:, None] * torch.tensor([1.0, -0.7, 0.4], dtype=F64,
                                                        device=DEV)).contiguous()
    # the points at leaflet positions of the parent box, through the trilinear map
    t = g.points(c["m"], "leaflets")
    h = torch.tensor([1.0 / v for v in N], dtype=F64, device=DEV)
    e3 = torch.minimum((t / h).floor(), torch.tensor([v - 1.0 for v in N], dtype=F64, device=DEV))
    # off the faces of the elements, so that each point has one element
    d["xi"] = (2 * (t / h - e3) - 1).clamp(-0.999, 0.999)
    e3 = e3.long()
    d["elem"] = e3[:, 0] + N[0] * (e3[:, 1] + N[1] * e3[:, 2])
    Nq = _shape8(d["xi"])
    d["X"] = torch.einsum("ba,bai->bi", Nq, d["coords"][_conn8(N)[d["elem"]]]).contiguous()
    n = P.shape[0]
    d["y"] = torch.where(d["mask"].bool(), d["yD"], 0.1 * g.fourier(N, 4, 0.0))
    d["An"] = 0.1 * g.fourier(N, 4, 0.0)
    d["f"] = g.fourier(N, 4, 0.0)
    d["x32"] = g.uniform(-1, 1, n, 4).float()
    d["w"] = torch.full((c["m"],), 0.024 / c["m"], dtype=F64, device=DEV)
    return d


def _prepare_coupled(c, seed):
    N, d = _dims(c), _coupled_inputs(c, seed)
    mesh = fsi.Mesh(N, rho=1.0, mu=1e-3, dt=DT, rho_inf=RHO_INF)
    mesh.set_coordinates(d["coords"])
    m = c["m"]
    o = dict(elem=_i32(m), xi=torch.zeros((m, 3), dtype=F64, device=DEV),
             cs=_i32(mesh.n_elems + 1), perm=_i32(m), R=torch.zeros_like(d["y"]),
             Jx=torch.zeros_like(d["x32"]))
    st = fsi.StepState(d["y"], d["Vn"], d["An"], f=d["f"], mask=d["mask"], yD=d["yD"],
                       elem=o["elem"], xi=o["xi"], cell_start=o["cs"], perm=o["perm"], w=d["w"],
                       drho_s=0.5, k_s=10.0, g_s=(0.0, 0.0, -1.0))
    return dict(kind="coupled", c=c, mesh=mesh, d=d, st=st, o=o)


def _tet_inputs(c, seed):
    g = Gen(seed)
    X, T = inputs.tet_box_mesh(_dims(c), seed=int(seed) % (1 << 31), perturb=0.2)
    n = X.shape[0]
    d = dict(Xn=torch.as_tensor(X, device=DEV), T=torch.as_tensor(T, device=DEV))
    d.update({k: 0.5 * g.normal(n, 4) for k in ("U", "A")}, x=g.normal(n, 4),
             lam=g.normal(c["m"], 3))
    if c["prec"] == "f32":
        d.update({k: d[k].float() for k in ("U", "A", "x", "lam")})
    d["P"] = g.points(c["m"], "leaflets")
    return d


def _prepare_tet(c, seed):
    d = _tet_inputs(c, seed)
    mesh = fsi.TetMesh(d["Xn"], d["T"], rho=1.0, mu=1e-3, dt=DT, rho_inf=RHO_INF)
    m = c["m"]
    o = {k: torch.zeros_like(d["U"]) for k in ("R", "Jx", "F")}
    o.update(elem=_i32(m), xi=torch.zeros((m, 3), dtype=F64, device=DEV),
             cs=_i32(mesh.n_elems + 1), perm=_i32(m), u=torch.zeros_like(d["lam"]))
    return dict(kind="tet", c=c, mesh=mesh, d=d, o=o)


def _batch_inputs(c, seed):
    """Per-instance sizes from the case alone (so that another seed is the same
    work), values from the seed; each array of all instances in one tensor."""
    r = np.random.default_rng(1000 * c["count"] + 50 * c["lo"] + c["hi"])
    Ns = [int(v) for v in r.integers(c["lo"], c["hi"] + 1, size=c["count"])]
    mus = np.exp(r.uniform(math.log(1e-3), math.log(1e-1), size=c["count"]))
    ms = [int(v) for v in r.integers(10_000, 150_001, size=c["count"])]
    g = Gen(seed)
    dt = torch.float32 if c["prec"] == "f32" else F64

    def pads(sizes):  # starts of the instances, 256-byte aligned rows
        return np.concatenate([[0], np.cumsum([-(-s // 64) * 64 for s in sizes])]).astype(int)

    on, om, oc = (pads([(N + 1) ** 3 for N in Ns]), pads(ms), pads([N ** 3 + 1 for N in Ns]))
    big = {k: g.uniform(-1, 1, int(on[-1]), 4).to(dt) for k in ("U", "A", "x")}
    big["lam"] = g.normal(int(om[-1]), 3).to(dt)
    X = torch.zeros((int(om[-1]), 3), dtype=F64, device=DEV)
    for i, m in enumerate(ms):
        X[om[i]:om[i] + m] = g.points(m, "leaflets")
    big["X"] = X
    return Ns, mus, ms, on, om, oc, big, dt


def _prepare_batch(c, seed):
    Ns, mus, ms, on, om, oc, big, dt = _batch_inputs(c, seed)
    out = {k: torch.zeros((int(on[-1]), 4), dtype=dt, device=DEV) for k in ("R", "Jx", "F")}
    out.update(u=torch.zeros((int(om[-1]), 3), dtype=dt, device=DEV),
               xi=torch.zeros((int(om[-1]), 3), dtype=dt, device=DEV), elem=_i32(int(om[-1])),
               perm=_i32(int(om[-1])), cell_start=_i32(int(oc[-1])))
    stream = torch.cuda.Stream()
    meshes, items = [], []
    for i, N in enumerate(Ns):
        meshes.append(fsi.Mesh(N, rho=1.0, mu=float(mus[i]), dt=DT, rho_inf=RHO_INF,
                               stream=stream.cuda_stream))
        n, m = (N + 1) ** 3, ms[i]
        it = {k: big[k][on[i]:on[i] + n] for k in ("U", "A", "x")}
        it.update({k: out[k][on[i]:on[i] + n] for k in ("R", "Jx", "F")})
        it.update({k: big[k][om[i]:om[i] + m] for k in ("lam", "X")})
        it.update({k: out[k][om[i]:om[i] + m] for k in ("u", "xi", "elem", "perm")})
        it["cell_start"] = out["cell_start"][oc[i]:oc[i] + N ** 3 + 1]
        items.append(it)
    torch.cuda.synchronize()
    b = fsi.Batch(meshes, items, PREC[c["prec"]], stream.cuda_stream)
    return dict(kind="batch", c=c, batch=b, stream=stream, big=big, out=out)


def _params(g):
    """He-initialised network parameters, W1 b1 W2 b2 W3 b3, small biases."""
    parts = []
    for fan, size in ((112, 112 * 256), (0, 256), (256, 256 * 256), (0, 256), (256, 1024), (0, 4)):
        parts.append(g.normal(size) * (math.sqrt(2.0 / fan) if fan else 0.02))
    return torch.cat(parts).float().contiguous()


def _train_inputs(c, seed):
    g = Gen(seed)
    P = _params(g)
    d = dict(P=P, X=g.normal(c["rows"], 112).float(), T=g.normal(c["rows"], 4).float())
    # the optimiser's state some hundred steps into the training
    d["m"] = (1e-3 * g.normal(P.numel())).float()
    d["v"] = (1e-5 + 1e-4 * g.uniform(0, 1, P.numel())).float()
    return d


def _prepare_train(c, seed):
    d = _train_inputs(c, seed)
    return dict(kind="train", c=c, d=d, mlp=fsi.Mlp(c["rows"]), G=torch.zeros_like(d["P"]),
                loss=torch.zeros(1, device=DEV))


def _predict_inputs(c, seed):
    N, g = _dims(c), Gen(seed)
    # velocities of order 1; increments of the acceleration-pressure unknown
    d = dict(Vn=g.fourier(N, 4, 0.0), y=g.fourier(N, 4, 0.0), d1=0.1 * g.fourier(N, 4, 0.0))
    d["d2"] = d["d1"] + 0.02 * g.fourier(N, 4, 0.0)
    d["P"] = _params(g)
    d["im"] = (0.05 * g.normal(112)).float()
    d["isd"] = g.uniform(0.2, 0.4, 112).float()
    d["isd"][108:] *= 0.2
    d["om"] = (0.001 * g.normal(4)).float()
    d["osd"] = g.uniform(0.005, 0.02, 4).float()
    return d


def _prepare_predict(c, seed):
    N, d = _dims(c), _predict_inputs(c, seed)
    return dict(kind="predict", c=c, d=d, mesh=fsi.Mesh(N, rho=1.0, mu=1e-3, dt=DT),
                mlp=fsi.Mlp(1024), y0=torch.zeros_like(d["y"]))


# ------------------------------------------------------------------ run
def run(state):
    return globals()["_run_" + state["kind"]](state)


def _run_step(s):
    c, mesh, d, o = s["c"], s["mesh"], s["d"], s["o"]
    p = PREC[c["prec"]]
    fsi.fsi_stage(mesh, fsi.FSI_F32 if c["prec"] == "f32" else fsi.FSI_F64, d["y"], d["Vn"],
                  d["An"], d["s"], o["U"], o["A"])
    if c["op"] == "both":
        fsi.fsi_residual_jacobian_apply(mesh, p, o["U"], o["A"], d["f"], d["x"], o["R"], o["Jx"])
    elif c["op"] == "jac":
        fsi.fsi_jacobian_apply(mesh, p, o["U"], o["A"], d["f"], d["x"], o["Jx"])
    else:
        fsi.fsi_residual(mesh, p, o["U"], o["A"], d["f"], o["R"])
    fsi.fsi_locate(mesh, d["X"], o["elem"], o["xi"], o["cs"], o["perm"], want_outside=False)
    xi = o["xi"].float() if c["prec"] == "f32" else o["xi"]
    fsi.fsi_dlm_interp(mesh, p, o["elem"], xi, o["U"], o["u"])
    fsi.fsi_dlm_spread(mesh, p, o["elem"], xi, o["cs"], o["perm"], d["lam"], None, o["F"], False)
    out = {k: o[k] for k in ("U", "A", "elem", "xi", "cs", "perm", "u", "F")}
    if c["op"] != "jac":
        out["R"] = o["R"]
    if c["op"] != "res":
        out["Jx"] = o["Jx"]
    return out


def _run_newton(s):
    # one decade below the benchmark's 1e-8, so that y itself is settled to ~1e-10
    s["y"].copy_(s["y0"])
    fsi.fsi_newton_step(s["mesh"], s["st"], mixed=s["c"]["mixed"], newton_rtol=1e-9,
                        krylov_rtol=1e-3, restart=50, max_krylov=4000,
                        residual_prec=fsi.FSI_DF64 if s["c"]["mixed"] else fsi.FSI_F64)
    return {"y": s["y"]}


def _run_coupled(s):
    mesh, d, o = s["mesh"], s["d"], s["o"]
    fsi.fsi_locate(mesh, d["X"], o["elem"], o["xi"], o["cs"], o["perm"], want_outside=False)
    fsi.fsi_coupled_residual(mesh, s["st"], o["R"], prec=fsi.FSI_DF64)
    fsi.fsi_coupled_jacobian_apply(mesh, fsi.FSI_F32, s["st"], d["x32"], o["Jx"])
    return dict(o)


def _run_tet(s):
    c, mesh, d, o = s["c"], s["mesh"], s["d"], s["o"]
    p = PREC[c["prec"]]
    fsi.fsi_tet_residual(mesh, p, d["U"], d["A"], None, o["R"])
    fsi.fsi_tet_jacobian_apply(mesh, p, d["U"], d["A"], None, d["x"], o["Jx"])
    fsi.fsi_tet_locate(mesh, d["P"], o["elem"], o["xi"], o["cs"], o["perm"], want_outside=False)
    xi = o["xi"].float() if c["prec"] == "f32" else o["xi"]
    fsi.fsi_tet_interp(mesh, p, o["elem"], xi, d["U"], o["u"])
    fsi.fsi_tet_spread(mesh, p, o["elem"], xi, o["cs"], o["perm"], d["lam"], None, o["F"], False)
    return dict(o)


def _run_batch(s):
    s["batch"].run(fsi.FSI_BATCH_GRAPH)
    return dict(s["out"])


def _run_train(s):
    d = s["d"]
    fsi.fsi_mlp_loss_grad(s["mlp"], d["P"], d["X"], d["T"], s["loss"], s["G"])
    fsi.fsi_mlp_adam(s["mlp"], d["P"], s["G"], d["m"], d["v"], 100, lr=1e-3)
    return dict(loss=s["loss"], G=s["G"], P=d["P"], m=d["m"], v=d["v"])


def _run_predict(s):
    d = s["d"]
    fsi.fsi_mlp_predict(s["mlp"], s["mesh"], d["P"], d["im"], d["isd"], d["om"], d["osd"],
                        d["Vn"], d["y"], d["d1"], d["d2"], s["y0"])
    return {"y0": s["y0"]}


# ------------------------------------------------------------------ work
# operations per element, common subexpressions counted once: residual,
# Jacobian apply, both at one state; a tetrahedron has half the points and
# half the nodes of a hexahedron
FLOPS = {"res": 5834, "jac": 8248, "both": 12524}


def work(case):
    c, k = case, case["kind"]
    if k in ("step", "coupled", "predict"):
        N = _dims(c)
        n, E = (N[0] + 1) * (N[1] + 1) * (N[2] + 1), N[0] * N[1] * N[2]
    if k == "step":
        b, m = 4 if c["prec"] == "f32" else 8, c["m"]
        fields = 5 + {"res": 0, "jac": 1, "both": 1}[c["op"]]       # y Vn An -> U A (+ x)
        fields += {"res": 1, "jac": 1, "both": 2}[c["op"]] + 0.75 + 1.25 * c["extras"]
        return {"bytes": 4 * b * n * fields + m * (24 + 24 + 8 + 6 * b) + 4 * E,
                "flops": FLOPS[c["op"]] * E + 144.0 * m}
    if k == "newton":
        n, E = (c["n"] + 1) ** 3, c["n"] ** 3
        its = 40  # GMRES iterations of a step, in two or three Newton iterations
        b = 4 if c["mixed"] else 8
        m = c["m"] if not c["body"] else 0
        # per iteration: U, A, x -> Jx, the preconditioner's blocks and
        # vectors, the basis read twice over its mean length
        return {"bytes": its * (n * b * 4 * (4 + 3 + 2 + 14) + m * (16 + 3 * b)) + 40.0 * n * 8,
                "flops": its * E * FLOPS["jac"] + 3.0 * E * FLOPS["res"]}
    if k == "coupled":
        # the mapped geometry is read once per operator
        return {"bytes": n * (8 * 4 * 6 + 4 * 4 * 2) + E * 144 * 4.0 + c["m"] * 120.0,
                "flops": (FLOPS["res"] + FLOPS["jac"]) * E * 1.3 + 800.0 * c["m"]}
    if k == "tet":
        N, b = _dims(c), 4 if c["prec"] == "f32" else 8
        n, E = (N[0] + 1) * (N[1] + 1) * (N[2] + 1), 6 * N[0] * N[1] * N[2]
        return {"bytes": n * 4 * b * 5.75 + E * (16 * 3 + 4) + c["m"] * (56 + 6 * b),
                "flops": E * (FLOPS["res"] + FLOPS["jac"]) / 4 + 300.0 * c["m"]}
    if k == "batch":
        r = np.random.default_rng(1000 * c["count"] + 50 * c["lo"] + c["hi"])
        Ns = r.integers(c["lo"], c["hi"] + 1, size=c["count"]).astype(float)
        r.uniform(math.log(1e-3), math.log(1e-1), size=c["count"])
        m = float(r.integers(10_000, 150_001, size=c["count"]).sum())
        b = 4 if c["prec"] == "f32" else 8
        return {"bytes": 4 * b * 5.75 * float(((Ns + 1) ** 3).sum()) + m * (32 + 9 * b)
                + 4 * float((Ns ** 3).sum()),
                "flops": FLOPS["both"] * float((Ns ** 3).sum()) + 144.0 * m}
    net = 112 * 256 + 256 * 256 + 256 * 4
    if k == "train":
        return {"bytes": c["rows"] * 464 + (net + 516) * 4 * 8.0,
                "flops": 2.0 * c["rows"] * (3 * net - 112 * 256)}
    return {"bytes": n * 32.0 * 5, "flops": 2.0 * n * net}


# ------------------------------------------------------------------ exact
def _shape8(xi):
    """N [.., 8] of the trilinear hexahedron, corner a = ax + 2 ay + 4 az."""
    s = torch.tensor([[2.0 * ((a >> k) & 1) - 1 for k in range(3)] for a in range(8)], dtype=F64,
                     device=xi.device)
    return (0.5 * (1 + s * xi[..., None, :])).prod(-1)


def _dshape8(xi):
    s = torch.tensor([[2.0 * ((a >> k) & 1) - 1 for k in range(3)] for a in range(8)], dtype=F64,
                     device=xi.device)
    f = 0.5 * (1 + s * xi[..., None, :])
    return torch.stack([0.5 * s[:, k] * f[..., (k + 1) % 3] * f[..., (k + 2) % 3]
                        for k in range(3)], -1)


def _conn8(N):
    i = torch.arange(N[0], device=DEV)
    j = torch.arange(N[1], device=DEV)
    k = torch.arange(N[2], device=DEV)
    base = (i[None, None, :] + (N[0] + 1) * (j[None, :, None] + (N[1] + 1) * k[:, None, None]))
    off = torch.tensor([(a & 1) + (N[0] + 1) * (((a >> 1) & 1) + (N[1] + 1) * ((a >> 2) & 1))
                        for a in range(8)], device=DEV)
    return base.reshape(-1, 1) + off


def _geometry(conn, coords):
    """Shape values N [g, a], gradients dN [e, g, a, 3], weights w [e, g] and the
    metric G [e, g, 3, 3] of hexahedra (2x2x2 Gauss) or linear tetrahedra."""
    if conn.shape[1] == 8:
        q = 1 / math.sqrt(3.0)
        xi = torch.tensor([[q * (2 * ((a >> k) & 1) - 1) for k in range(3)] for a in range(8)],
                          dtype=F64, device=DEV)
        Nq, dq = _shape8(xi), _dshape8(xi)
        scale = 1.0
    else:
        a, b = 0.25 + 0.15 * math.sqrt(5.0), 0.25 - 0.05 * math.sqrt(5.0)
        lam = torch.full((4, 4), b, dtype=F64, device=DEV)
        lam.fill_diagonal_(a)
        Nq = lam
        d1 = torch.tensor([[-1.0, -1, -1], [1, 0, 0], [0, 1, 0], [0, 0, 1]], dtype=F64, device=DEV)
        dq = d1.expand(4, 4, 3)
        scale = 1.0 / 24
    J = torch.einsum("gak,eai->egik", dq, coords[conn])
    Ji = torch.linalg.inv(J)                                  # [e, g, k, i] = dxi_k / dx_i
    dN = torch.einsum("gak,egki->egai", dq, Ji)
    return Nq, dN, scale * torch.linalg.det(J).abs(), Ji.transpose(-1, -2) @ Ji


def _element_residual(Ue, Ae, fe, geo, ph):
    Nq, dN, w, G = geo
    rho, mu, dt = 1.0, ph["mu"], DT
    u = torch.einsum("ga,eac->egc", Nq, Ue)
    gu = torch.einsum("egaj,eac->egcj", dN, Ue)
    A = torch.einsum("ga,eac->egc", Nq, Ae)
    v, p, gv, gp = u[..., :3], u[..., 3], gu[..., :3, :], gu[..., 3, :]
    a = A[..., :3] if fe is None else A[..., :3] - torch.einsum("ga,eac->egc", Nq, fe)[..., :3]
    s = A[..., 3] if ph["has_s"] else 1.0
    conv = torch.einsum("egij,egj->egi", gv, v)
    rM = rho * (a + conv) + gp
    rC = gv.diagonal(dim1=-2, dim2=-1).sum(-1)
    q = (4.0 / dt ** 2 + torch.einsum("egi,egij,egj->eg", v, G, v)
         + 36.0 * (mu / rho) ** 2 * (G * G).sum((-1, -2)))
    tM = (s * q) ** -0.5
    tC = 1.0 / (tM * G.diagonal(dim1=-2, dim2=-1).sum(-1))
    up = -(tM / rho)[..., None] * rM
    pp = -rho * tC * rC
    X = rho * (a + conv + torch.einsum("egij,egj->egi", gv, up))
    Y = mu * (gv + gv.transpose(-1, -2)) - rho * up[..., :, None] * (v + up)[..., None, :]
    Y = Y - (p + pp)[..., None, None] * torch.eye(3, dtype=F64, device=DEV)
    X = torch.cat([X, rC[..., None]], -1) * w[..., None]
    Y = torch.cat([Y, -up[..., None, :]], -2) * w[..., None, None]
    return torch.einsum("ga,egc->eac", Nq, X) + torch.einsum("egaj,egcj->eac", dN, Y)


def _vms(conn, coords, U, A, f, x, ph, want=("R", "Jx"), chunk=32768):
    """Residual and Jacobian apply; f and x may be None."""
    U, A = U.double(), A.double()
    f = None if f is None else f.double()
    R, J = torch.zeros_like(U), torch.zeros_like(U)
    if x is not None:
        x = x.double()
        dU = torch.cat([AF * GAM * DT * x[:, :3], x[:, 3:]], 1)
        dA = torch.cat([AM * x[:, :3], torch.zeros_like(x[:, 3:])], 1)
    for i in range(0, conn.shape[0], chunk):
        c = conn[i:i + chunk]
        geo = _geometry(c, coords)
        fe = None if f is None else f[c]
        if x is None or "Jx" not in want:
            r, j = _element_residual(U[c], A[c], fe, geo, ph), None
        else:
            r, j = torch.func.jvp(lambda p, q: _element_residual(p, q, fe, geo, ph), (U[c], A[c]),
                                  (dU[c], dA[c]))
            J.index_add_(0, c.reshape(-1), j.reshape(-1, 4))
        R.index_add_(0, c.reshape(-1), r.reshape(-1, 4))
    return R, J


def _spread(conn, elem, Nq, lam, n, w=None):
    F = torch.zeros((n, 4), dtype=F64, device=DEV)
    lam = lam.double() if w is None else lam.double() * w[:, None]
    for i in range(0, elem.shape[0], 1 << 18):
        k = slice(i, i + (1 << 18))
        c = Nq[k][:, :, None] * lam[k][:, None, :]
        F[:, :3].index_add_(0, conn[elem[k]].reshape(-1), c.reshape(-1, 3))
    return F


def _interp(conn, elem, Nq, U):
    return torch.cat([torch.einsum("ba,bac->bc", Nq[i:i + (1 << 18)],
                                   U.double()[:, :3][conn[elem[i:i + (1 << 18)]]])
                      for i in range(0, elem.shape[0], 1 << 18)])


def _locate(N, X):
    """Element and xi of points of the unit box (all inside)."""
    h = torch.tensor([1.0 / v for v in N], dtype=F64, device=DEV)
    t = X / h
    e = torch.minimum(t.floor(), torch.tensor([v - 1.0 for v in N], dtype=F64, device=DEV))
    xi = 2 * (t - e) - 1
    e = e.long()
    return e[:, 0] + N[0] * (e[:, 1] + N[1] * e[:, 2]), xi


def _stage(y, Vn, An, s):
    y, Vn, An = y.double(), Vn.double(), An.double()
    V1 = Vn + DT * An + GAM * DT * (y - An)
    U, A = Vn + AF * (V1 - Vn), An + AM * (y - An)
    U[:, 3] = y[:, 3]
    A[:, 3] = 1.0 if s is None else s.double()
    return U, A


def exact(case, seed):
    f = globals().get("_exact_" + case["kind"])
    return None if f is None else f(case, seed)


def _exact_step(c, seed):
    N, d = _dims(c), _step_inputs(c, seed)
    conn = _conn8(N)
    U, A = _stage(d["y"], d["Vn"], d["An"], d["s"])
    ph = dict(mu=0.01, has_s=c["extras"])
    R, J = _vms(conn, _nodes(N), U, A, d["f"], d["x"], ph, ("R", "Jx") if c["op"] != "res" else "R")
    elem, xi = _locate(N, d["X"])
    Nq = _shape8(xi)
    out = dict(U=U, A=A, elem=None, xi=xi, cs=None, perm=None, u=_interp(conn, elem, Nq, U),
               F=_spread(conn, elem, Nq, d["lam"], U.shape[0]))
    if c["op"] != "jac":
        out["R"] = R
    if c["op"] != "res":
        out["Jx"] = J
    return out


def _exact_coupled(c, seed):
    N, d = _dims(c), _coupled_inputs(c, seed)
    conn, elem, Nq = _conn8(N), d["elem"], _shape8(d["xi"])
    U, A = _stage(d["y"], d["Vn"], d["An"], None)
    ph = dict(mu=1e-3, has_s=False)
    R, J = _vms(conn, d["coords"], U, A, d["f"], d["x32"], ph)
    n = U.shape[0]
    V1 = d["Vn"] + DT * d["An"] + GAM * DT * (d["y"] - d["An"])
    g = torch.tensor([0.0, 0.0, -1.0], dtype=F64, device=DEV)
    rs = 0.5 * (_interp(conn, elem, Nq, d["y"]) - g) + 10.0 * DT * _interp(conn, elem, Nq, V1)
    R = R + _spread(conn, elem, Nq, rs, n, d["w"])
    x = d["x32"].double()
    J = J + _spread(conn, elem, Nq, (0.5 + 10.0 * GAM * DT ** 2) * _interp(conn, elem, Nq, x), n,
                    d["w"])
    mask = d["mask"].bool()
    return dict(elem=None, xi=d["xi"], cs=None, perm=None,
                R=torch.where(mask, d["y"] - d["yD"], R), Jx=torch.where(mask, x, J))


def _exact_tet(c, seed):
    d = _tet_inputs(c, seed)
    conn = d["T"].long()
    R, J = _vms(conn, d["Xn"], d["U"], d["A"], None, d["x"], dict(mu=1e-3, has_s=False),
                chunk=65536)
    # elem and barycentric coordinates by the definition need the mesh's search:
    # only the fields are stated here
    return dict(R=R, Jx=J, F=None, elem=None, xi=None, cs=None, perm=None, u=None)


def _exact_batch(c, seed):
    Ns, mus, ms, on, om, oc, big, dt = _batch_inputs(c, seed)
    out = {k: torch.zeros((int(on[-1]), 4), dtype=F64, device=DEV) for k in ("R", "Jx", "F")}
    out.update({k: torch.zeros((int(om[-1]), 3), dtype=F64, device=DEV) for k in ("u", "xi")})
    for i, N in enumerate(Ns):
        D, n, m = (N,) * 3, (N + 1) ** 3, ms[i]
        ns, mm = slice(on[i], on[i] + n), slice(om[i], om[i] + m)
        conn = _conn8(D)
        out["R"][ns], out["Jx"][ns] = _vms(conn, _nodes(D), big["U"][ns], big["A"][ns], None,
                                           big["x"][ns], dict(mu=float(mus[i]), has_s=False))
        elem, xi = _locate(D, big["X"][mm])
        Nq = _shape8(xi)
        out["xi"][mm] = xi
        out["u"][mm] = _interp(conn, elem, Nq, big["U"][ns])
        out["F"][ns] = _spread(conn, elem, Nq, big["lam"][mm], n)
    return dict(out, elem=None, perm=None, cell_start=None)


def _weights(P):
    P, k, out = P.double(), 0, []
    for shp in ((112, 256), (256,), (256, 256), (256,), (256, 4), (4,)):
        size = math.prod(shp)
        out.append(P[k:k + size].reshape(shp))
        k += size
    return out


def _exact_train(c, seed):
    d = _train_inputs(c, seed)
    P = d["P"].double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = _weights(P)
    h = torch.relu(torch.relu(d["X"].double() @ W1 + b1) @ W2 + b2) @ W3 + b3
    loss = 0.5 * ((h - d["T"].double()) ** 2).sum() / c["rows"]
    G, = torch.autograd.grad(loss, P)
    m = 0.9 * d["m"].double() + 0.1 * G
    v = 0.999 * d["v"].double() + 0.001 * G * G
    new = P.detach() - 1e-3 * (m / (1 - 0.9 ** 100)) / ((v / (1 - 0.999 ** 100)).sqrt() + 1e-8)
    return dict(loss=loss.detach().reshape(1), G=G, P=new, m=m, v=v)


def _exact_predict(c, seed):
    N, d = _dims(c), _predict_inputs(c, seed)
    W1, b1, W2, b2, W3, b3 = _weights(d["P"])
    f = d["Vn"].clone()
    f[:, 3] = d["y"][:, 3]
    shape = (N[2] + 1, N[1] + 1, N[0] + 1)
    pad = torch.nn.functional.pad(f.reshape(*shape, 4), (0, 0, 1, 1, 1, 1, 1, 1))
    e = 2 * d["d1"] - d["d2"]
    im, isd = d["im"].double(), d["isd"].double()
    out = torch.empty_like(f)
    plane = shape[1] * shape[2]
    for k in range(shape[0]):
        cols = [pad[k + dz:k + dz + 1, dy:dy + shape[1], dx:dx + shape[2]].reshape(-1, 4)
                for dz in range(3) for dy in range(3) for dx in range(3)]
        sl = slice(k * plane, (k + 1) * plane)
        X = (torch.cat(cols + [e[sl]], 1) - im) / isd
        out[sl] = torch.relu(torch.relu(X @ W1 + b1) @ W2 + b2) @ W3 + b3
    return {"y0": d["y"] + e + d["om"].double() + d["osd"].double() * out}
