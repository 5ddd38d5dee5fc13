"""Performance cases of the TPFA pressure solver: what its users run, through the
public entry points of ``paper_2408_03452_gb300`` (tpfa.py, transient.py).

Kinds of case
  apply     one application of the matrix-free operator A p (tpfa_apply,
            tpfa_apply_bf16): what any Krylov method or check built on it calls
  setup     a new permeability field arrives: coefficient records, right-hand
            side and the FP64 residual of a start vector
  solve     pressure solve with Dirichlet ends (cg_solve / cg_solve_bf16)
  step      one backward-Euler time step with a well pair (transient.run)
  ensemble  many realizations of uneven sizes in one batch (cg_solve_batch)
  conv      one convolution layer of the preconditioner network, forward
  convgrad  input and weight gradient of one such layer (training)
  unet      one application of the preconditioner network
  learned   one time step solved by flexible CG with that network (fcg_solve)

Solves run to a tolerance at which the answer itself is determined to about
ten digits, so that the result does not depend on the path of the iteration.
"""
import math

import torch

from paper_2408_03452_gb300 import tpfa, transient

# the sizes the batched workload draws from (synth.ENSEMBLE_SIZES)
ENSEMBLE_SIZES = ((48, 48, 24), (64, 64, 32), (96, 96, 48), (128, 128, 64))
CONV_SHAPES = ((16, 16), (16, 32), (32, 16), (32, 64), (64, 32))
NET_LAYERS = ((2, 16), (16, 32), (32, 64), (64, 32), (32, 16), (16, 16), (16, 1))


def listed():
    return [
        # the smallest call: the operator on the 32^3 grid of the plain method's
        # small workload, with the fused p'Ap a hand-written CG would ask for
        dict(name="apply_32", kind="apply", nx=32, ny=32, nz=32, sigma=1.0, records="f32", dot=True),
        # half of the paper's Table III mesh (750 x 994 x 922) per axis: odd
        # extents, rows that are not a multiple of 16 bytes
        dict(name="apply_odd", kind="apply", nx=375, ny=497, nz=461, sigma=1.5, records="f32",
             dot=False),
        # a new field on the 256^3 grid of the mixed-precision and learned workloads
        dict(name="setup_256", kind="setup", nx=256, ny=256, nz=256, sigma=1.5),
        # the plain method's small workload, plain CG
        dict(name="solve_32", kind="solve", nx=32, ny=32, nz=32, sigma=1.0, channels=False,
             records="f32", precond=0, tol=1e-12),
        # one realization of the training set of the learned preconditioner
        dict(name="solve_64", kind="solve", nx=64, ny=64, nz=64, sigma=1.5, channels=False,
             records="f32", precond=0, tol=1e-12),
        # the mixed-precision workload (channels 1e4 times more permeable, BF16
        # records, Jacobi) at half its extent
        dict(name="solve_channels", kind="solve", nx=128, ny=128, nz=128, sigma=2.0, channels=True,
             records="bf16", precond=1, tol=1e-13),
        # the paper-scale grid: one time step of the layered field with a well pair
        dict(name="step_1024", kind="step", nx=1024, ny=1024, nz=256, sigma=1.5, layer=8, d=16.0,
             precond=0, tol=1e-10),
        # a third of the 96-instance ensemble, Jacobi as its fastest plain solver
        dict(name="ensemble_32", kind="ensemble", n_inst=32, mix=0, sigma=2.5, precond=1, tol=1e-12),
        # the network's widest-volume layer on the 64^3 grid it runs on for 256^3 fields
        dict(name="conv_16_16", kind="conv", nx=64, ny=64, nz=64, ns=1, cin=16, cout=16),
        # training: gradients of the second layer for a batch of 16 samples
        dict(name="convgrad_16_32", kind="convgrad", nx=32, ny=32, nz=32, ns=16, cin=16, cout=32),
        # the whole network on that 64^3 grid
        dict(name="unet_64", kind="unet", nx=64, ny=64, nz=64, ns=1),
        # the learned workload's grid: flexible CG, network on the 4x coarser grid
        dict(name="learned_256", kind="learned", nx=256, ny=256, nz=256, sigma=1.5, levels=2,
             d=0.1, m=2, tol=1e-12),
    ]


def _extent(rng, lo, hi, step=1):
    """An extent in [lo, hi], spread over its logarithm, a multiple of step."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(("apply", "apply", "setup", "solve", "solve", "step", "ensemble", "conv",
                       "convgrad", "unet", "learned"))
    if kind == "apply":
        return dict(kind=kind, nx=_extent(rng, 16, 768), ny=_extent(rng, 16, 512),
                    nz=_extent(rng, 8, 460), sigma=round(rng.uniform(0.5, 2.5), 2),
                    records=rng.choice(("f32", "f32", "bf16")), dot=rng.random() < 0.5)
    if kind == "setup":
        return dict(kind=kind, nx=_extent(rng, 16, 320), ny=_extent(rng, 16, 320),
                    nz=_extent(rng, 8, 256), sigma=round(rng.uniform(0.5, 2.5), 2))
    if kind == "solve":
        channels = rng.random() < 0.3
        return dict(kind=kind, nx=_extent(rng, 16, 128), ny=_extent(rng, 12, 128),
                    nz=_extent(rng, 12, 128),
                    sigma=round(rng.uniform(0.5, 2.0 if channels else 1.5), 2), channels=channels,
                    records=rng.choice(("f32", "f32", "bf16")),
                    precond=1 if channels else rng.choice((0, 1)),
                    tol=1e-13 if channels else 1e-12)
    if kind == "step":
        return dict(kind=kind, nx=_extent(rng, 24, 512), ny=_extent(rng, 24, 512),
                    nz=_extent(rng, 16, 256), sigma=1.5, layer=rng.choice((1, 8)),
                    d=rng.choice((4.0, 16.0)), precond=rng.choice((0, 1)), tol=1e-10)
    if kind == "ensemble":
        precond = rng.choice((0, 1, 1))
        return dict(kind=kind, n_inst=_extent(rng, 2, 40), mix=rng.randrange(1, 1000),
                    sigma=2.5 if precond else 1.5, precond=precond, tol=1e-12)
    if kind in ("conv", "convgrad"):
        cin, cout = rng.choice(CONV_SHAPES)
        ns = rng.choice((1, 1, 2, 5, 16))
        top = {1: 96, 2: 72, 5: 48, 16: 32}[ns]
        return dict(kind=kind, nx=_extent(rng, 6, top), ny=_extent(rng, 6, top),
                    nz=_extent(rng, 4, top), ns=ns, cin=cin, cout=cout)
    if kind == "unet":
        ns = rng.choice((1, 1, 3, 16))
        top = {1: 96, 3: 64, 16: 32}[ns]
        return dict(kind=kind, nx=_extent(rng, 8, top, 4), ny=_extent(rng, 8, top, 4),
                    nz=_extent(rng, 8, top, 4), ns=ns)
    return dict(kind=kind, nx=_extent(rng, 48, 256, 16), ny=_extent(rng, 48, 256, 16),
                nz=_extent(rng, 32, 256, 16), sigma=round(rng.uniform(0.5, 2.0), 2), levels=2,
                d=rng.choice((0.1, 1.0)), m=rng.choice((2, 2, 4)), tol=1e-12)


# ---------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(shape, g):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _uniform(shape, g):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _field(nx, ny, nz, sigma, g, layer=1):
    """Lognormal permeability [nz, ny, nx]; constant over runs of `layer` planes."""
    K = (_normal((-(-nz // layer), ny, nx), g) * sigma).exp_()
    return K if layer == 1 else K.repeat_interleave(layer, 0)[:nz].contiguous()


def _channels(K, g, contrast=1e4):
    """Eight sinusoidal channels 4 cells wide and 8 layers thick (clipped to small grids)."""
    nz, ny, nx = K.shape
    u = _uniform((8, 3), g).cpu()
    x = torch.arange(nx, device="cuda", dtype=torch.float64)
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
    inside = torch.zeros((nz, ny, nx), device="cuda", dtype=torch.bool)
    for c in range(8):
        z0 = int(u[c, 1] * max(nz - 8, 1))
        mid = float(u[c, 0]) * ny + 16.0 * torch.sin(2 * math.pi * (x / 128.0 + float(u[c, 2])))
        inside[z0:z0 + 8] |= ((y - mid).abs() < 2.0)
    return torch.where(inside, K * contrast, K)


def _ends(nx, ny, nz, axis=2, hi=1.0):
    """Dirichlet mask and values on the end layers of one axis of [nz, ny, nx]."""
    mask = torch.zeros((nz, ny, nx), device="cuda", dtype=torch.uint8)
    pD = torch.zeros((nz, ny, nx), device="cuda", dtype=torch.float64)
    mask.select(axis, 0).fill_(1)
    mask.select(axis, -1).fill_(1)
    pD.select(axis, 0).fill_(hi)
    return mask, pD


def _problem(case, seed):
    """One pressure problem: K, Dirichlet mask and values, accumulation
    diagonal, well pair, previous pressure (None where there is none)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    g = _gen(seed)
    P = dict(mask=None, pD=None, d=0.0, wells=None, p0=None)
    P["K"] = _field(nx, ny, nz, case["sigma"], g, case.get("layer", 1))
    if case.get("channels"):
        P["K"] = _channels(P["K"], g)
    if case["kind"] in ("solve", "setup"):
        P["mask"], P["pD"] = _ends(nx, ny, nz)
    else:
        P["d"] = case["d"]
        P["wells"] = (torch.tensor([0, nx * ny * nz - 1], device="cuda"),
                      torch.tensor([1.0, -1.0], device="cuda", dtype=torch.float64))
        P["p0"] = _uniform((nz, ny, nx), g)
    if case["kind"] == "setup":
        P["p0"] = _uniform((nz, ny, nx), g)
    return P


def _ensemble(case, seed):
    """Grids from `mix` (so that a case's sizes do not change with the seed),
    sigma in [0.5, case sigma], Dirichlet ends on a drawn axis, p in [0.5, 2]."""
    pick = torch.Generator().manual_seed(7 + case["mix"])
    u = torch.rand((case["n_inst"], 3), generator=pick, dtype=torch.float64)
    g, out = _gen(seed), []
    for i in range(case["n_inst"]):
        nx, ny, nz = ENSEMBLE_SIZES[min(int(u[i, 0] * 4), 3)]
        K = _field(nx, ny, nz, 0.5 + (case["sigma"] - 0.5) * float(u[i, 1]), g)
        mask, pD = _ends(nx, ny, nz, min(int(u[i, 2] * 3), 2), 0.5 + 1.5 * float(_uniform((1,), g)))
        out.append(dict(K=K, mask=mask, pD=pD, d=0.0, wells=None, p0=None))
    return out


def _volume(shape, c, g, relu):
    """A haloed channels-last BF16 volume [ns, nz+2, ny+2, nx+2, c] with a zero halo."""
    nx, ny, nz, ns = shape
    v = torch.zeros((ns, nz + 2, ny + 2, nx + 2, c), device="cuda", dtype=torch.bfloat16)
    x = _normal((ns, nz, ny, nx, c), g)
    v[:, 1:-1, 1:-1, 1:-1] = (x.clamp_(min=0) if relu else x).bfloat16()
    return v


def _conv_inputs(case, seed):
    shape = (case["nx"], case["ny"], case["nz"], case["ns"])
    cin, cout = case["cin"], case["cout"]
    g = _gen(seed)
    S = dict(shape=shape, cin=cin, cout=cout)
    S["x"] = _volume(shape, cin, g, True)
    S["w"] = (_normal((27, cout, cin), g) * math.sqrt(2.0 / (27 * cin))).bfloat16()
    S["bias"] = (_normal((cout,), g) * 0.1).float()
    if case["kind"] == "convgrad":
        S["dy"] = _volume(shape, cout, g, False)
        # gradient kernel: taps flipped, each tap's matrix transposed
        S["wt"] = S["w"].flip(0).transpose(1, 2).contiguous()
    return S


def _net_params(seed):
    """He-style weights and small biases in the library's flat layout."""
    g, flat = _gen(seed + 17), []
    for cin, cout in NET_LAYERS:
        flat += [_normal((27 * cout * cin,), g) * math.sqrt(2.0 / (27 * cin)), _normal((cout,), g) * 0.05]
    return torch.cat(flat).float()


def _net_inputs(case, seed):
    g = _gen(seed)
    shape = (case["ns"], case["nz"], case["ny"], case["nx"])
    return _normal(shape, g).float(), (1.5 * _normal(shape, g)).exp_()


# ---------------------------------------------------------------------------
# what a program has in hand before the call
# ---------------------------------------------------------------------------
def _flat(t):
    return None if t is None else t.reshape(-1)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("conv", "convgrad"):
        S = _conv_inputs(case, seed)
        if kind == "conv":
            S["y"] = torch.zeros(S["x"].shape[:-1] + (S["cout"],), device="cuda", dtype=torch.bfloat16)
        else:
            S["dx"] = torch.zeros_like(S["x"])
            S["dw"] = torch.empty((27, S["cout"], S["cin"]), device="cuda", dtype=torch.float32)
        return S | dict(kind=kind)
    if kind == "unet":
        r, K = _net_inputs(case, seed)
        net = tpfa.UNet(case["nx"], case["ny"], case["nz"], ns=case["ns"])
        net.set_params(_net_params(seed))
        return dict(kind=kind, net=net, r=_flat(r), lnk=tpfa.log_perm(_flat(K)))
    if kind == "ensemble":
        parts = _ensemble(case, seed)
        bc = tpfa.BatchContext([tuple(reversed(p["K"].shape)) for p in parts])
        bc.set_option("precond", case["precond"])
        K, mask, pD = (torch.cat([_flat(p[k]) for p in parts]) for k in ("K", "mask", "pD"))
        coef, coef64 = bc.build_trans(K, mask)
        return dict(kind=kind, bc=bc, coef=coef, coef64=coef64, b=bc.build_rhs(K, mask, pD=pD),
                    tol=case["tol"])
    ctx = tpfa.Context(case["nx"], case["ny"], case["nz"])
    S = dict(kind=kind, ctx=ctx)
    if kind == "apply":
        g = _gen(seed)
        K = _flat(_field(case["nx"], case["ny"], case["nz"], case["sigma"], g))
        S["p"] = (2.0 * _uniform((ctx.n,), g) - 1.0).float()
        S["records"] = case["records"]
        S["coef"] = ctx.build_trans_bf16(K, d_uniform=1e-3) if case["records"] == "bf16" else \
            ctx.build_trans(K, d_uniform=1e-3, coef64=False)[0]
        S["pAp"] = torch.zeros(1, device="cuda", dtype=torch.float64) if case["dot"] else None
        return S
    P = _problem(case, seed)
    S |= {k: _flat(P[k]) for k in ("K", "mask", "pD", "p0")}
    if kind == "setup":
        return S
    S["tol"], S["d"], S["wells"] = case["tol"], P["d"], P["wells"]
    S["coef"], S["coef64"] = ctx.build_trans(S["K"], S["mask"], d_uniform=P["d"])
    if kind == "solve":
        S["b"] = ctx.build_rhs(S["K"], S["mask"], pD=S["pD"])
        if case["records"] == "bf16":
            S["coef"] = ctx.build_trans_bf16(S["K"], S["mask"])
        del S["K"], S["mask"], S["pD"], S["p0"]
    if kind == "learned":
        f = 1 << case["levels"]
        S["net"] = tpfa.UNet(case["nx"] // f, case["ny"] // f, case["nz"] // f)
        S["net"].set_params(_net_params(seed))
        S["lnk"] = tpfa.log_perm(S["K"])
        S["b"] = ctx.build_rhs_transient(S["K"], S["p0"], src_idx=P["wells"][0], src_val=P["wells"][1],
                                         d_uniform=P["d"])
        ctx.set_option("fcg_m", case["m"])
        del S["K"], S["p0"]
    else:
        ctx.set_option("precond", case["precond"])
    return S


def run(S):
    kind = S["kind"]
    if kind == "apply":
        f = S["ctx"].apply_bf16 if S["records"] == "bf16" else S["ctx"].apply
        q = f(S["coef"], S["p"], pAp=S["pAp"])
        return [q] if S["pAp"] is None else [q, S["pAp"]]
    if kind == "setup":
        ctx = S["ctx"]
        coef, coef64 = ctx.build_trans(S["K"], S["mask"])
        b = ctx.build_rhs(S["K"], S["mask"], pD=S["pD"])
        return [coef, coef64, b, ctx.residual64(coef64, b, S["p0"])]
    if kind == "solve":
        return S["ctx"].cg_solve(S["coef"], S["coef64"], S["b"], tol=S["tol"])[0]
    if kind == "step":
        return transient.run(S["ctx"], S["coef"], S["coef64"], S["K"], S["p0"], 1, d_uniform=S["d"],
                             src_idx=S["wells"][0], src_val=S["wells"][1], tol=S["tol"])[0][0]
    if kind == "ensemble":
        return S["bc"].cg_solve(S["coef"], S["coef64"], S["b"], tol=S["tol"])[0]
    if kind == "conv":
        return tpfa.conv3d_bf16(S["x"], S["w"], S["y"], S["shape"], S["cin"], S["cout"],
                                bias=S["bias"], flags=tpfa.CONV_RELU)
    if kind == "convgrad":
        # the layer's input x is its predecessor's ReLU output, so x masks dx
        tpfa.conv3d_bf16(S["dy"], S["wt"], S["dx"], S["shape"], S["cout"], S["cin"], mask=S["x"],
                         flags=tpfa.CONV_MASK)
        tpfa.conv3d_wgrad_bf16(S["x"], S["dy"], S["dw"], S["shape"], S["cin"], S["cout"])
        return [S["dx"], S["dw"]]
    if kind == "unet":
        return S["net"].forward(S["r"], S["lnk"])
    return S["ctx"].fcg_solve(S["coef"], S["coef64"], S["b"], net=S["net"], lnk=S["lnk"],
                              tol=S["tol"])[0]


def work(case):
    """Inputs read once, outputs written once, and the operations of the direct
    kinds.  How often a solve has to iterate depends on its inputs: only its
    inputs, its outputs and one iteration's operations are counted."""
    kind = case["kind"]
    if kind == "ensemble":
        pick = torch.Generator().manual_seed(7 + case["mix"])
        u = torch.rand((case["n_inst"], 3), generator=pick, dtype=torch.float64)
        n = sum(math.prod(ENSEMBLE_SIZES[min(int(v * 4), 3)]) for v in u[:, 0])
        return {"bytes": n * (16 + 32 + 8 + 8), "flops": 25 * n}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "apply":
        return {"bytes": n * (16 if case["records"] == "bf16" else 24), "flops": 13 * n}
    if kind == "setup":  # K, mask, p^D, start vector; FP32 and FP64 records, b, residual
        return {"bytes": n * (8 + 1 + 8 + 8 + 16 + 32 + 8 + 8), "flops": 45 * n}
    if kind == "solve":
        return {"bytes": n * ((8 if case["records"] == "bf16" else 16) + 32 + 8 + 8), "flops": 25 * n}
    if kind == "step":
        return {"bytes": n * (16 + 32 + 8 + 8), "flops": 25 * n}
    if kind == "learned":
        return {"bytes": n * (16 + 32 + 4 + 8 + 8), "flops": 25 * n}
    n *= case["ns"]
    if kind == "unet":
        f = sum(54 * a * b * (1.0, 1 / 8, 1 / 64, 1 / 64, 1 / 8, 1.0, 1.0)[i]
                for i, (a, b) in enumerate(NET_LAYERS))
        return {"bytes": 12 * n + 4 * sum(27 * a * b + b for a, b in NET_LAYERS), "flops": f * n}
    cin, cout = case["cin"], case["cout"]
    flops = 54 * cin * cout * n
    if kind == "conv":
        return {"bytes": 2 * n * (cin + cout) + 54 * cin * cout, "flops": flops}
    return {"bytes": 2 * n * (2 * cin + cout) + 162 * cin * cout, "flops": 2 * flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, with plain torch
# ---------------------------------------------------------------------------
def _faces(P):
    """Face transmissibilities (unit cells, mu = 1), the accumulation diagonal
    plus Dirichlet couplings E, the lifted Dirichlet values and the mask; faces
    of Dirichlet cells are taken out."""
    K = P["K"]
    T, E = [], torch.full_like(K, P["d"])
    lift = torch.zeros_like(K)
    m = None if P["mask"] is None else P["mask"].bool()
    for axis in (2, 1, 0):
        n = K.shape[axis]
        if n == 1:
            T.append(None)
            continue
        a, b = K.narrow(axis, 0, n - 1), K.narrow(axis, 1, n - 1)
        t = 1.0 / (1.0 / (2.0 * a) + 1.0 / (2.0 * b))
        if m is not None:
            ma, mb = m.narrow(axis, 0, n - 1), m.narrow(axis, 1, n - 1)
            E.narrow(axis, 0, n - 1).add_(t * mb)
            E.narrow(axis, 1, n - 1).add_(t * ma)
            pa, pb = P["pD"].narrow(axis, 0, n - 1), P["pD"].narrow(axis, 1, n - 1)
            lift.narrow(axis, 0, n - 1).add_(t * mb * pb)
            lift.narrow(axis, 1, n - 1).add_(t * ma * pa)
            t = torch.where(ma | mb, torch.zeros_like(t), t)
        T.append(t)
    if m is not None:
        E = torch.where(m, torch.ones_like(E), E)
    return T, E, lift, m


def _diag(T, E):
    D = E.clone()
    for t, axis in zip(T, (2, 1, 0)):
        if t is not None:
            D.narrow(axis, 0, t.shape[axis]).add_(t)
            D.narrow(axis, 1, t.shape[axis]).add_(t)
    return D


def _matvec(T, D, p):
    q = D * p
    for t, axis in zip(T, (2, 1, 0)):
        if t is not None:
            n = t.shape[axis]
            q.narrow(axis, 0, n).addcmul_(t, p.narrow(axis, 1, n), value=-1.0)
            q.narrow(axis, 1, n).addcmul_(t, p.narrow(axis, 0, n), value=-1.0)
    return q


def _rhs(P, lift, m):
    b = lift if P["p0"] is None else lift + P["d"] * P["p0"]
    if P["wells"] is not None:
        b.view(-1).index_add_(0, *P["wells"])
    return b if m is None else torch.where(m, P["pD"], b)


def _pcg(T, D, b, tol=1e-14, maxit=60000):
    """Jacobi-preconditioned CG, restarted once from the true residual."""
    x = torch.zeros_like(b)
    stop = float((b * b).sum()) * tol * tol
    for _ in range(3):
        r = b - _matvec(T, D, x)
        z = r / D
        p = z.clone()
        rz = (r * z).sum()
        for it in range(maxit):
            if it % 20 == 0 and float((r * r).sum()) <= stop:
                break
            q = _matvec(T, D, p)
            alpha = rz / (p * q).sum()
            x.addcmul_(p, alpha.expand_as(p))
            r.addcmul_(q, alpha.expand_as(q), value=-1.0)
            torch.div(r, D, out=z)
            new = (r * z).sum()
            p.mul_(new / rz).add_(z)
            rz = new
        if it == 0:
            break
    return x


def _solution(P):
    T, E, lift, m = _faces(P)
    b = _rhs(P, lift, m)
    D = _diag(T, E)
    if m is not None:
        D = torch.where(m, torch.ones_like(D), D)
    return _pcg(T, D, b).reshape(-1)


def _records(T, D):
    out = torch.zeros(D.shape + (4,), device="cuda", dtype=torch.float64)
    for c, (t, axis) in enumerate(zip(T, (2, 1, 0))):
        if t is not None:
            out[..., c].narrow(axis, 0, t.shape[axis]).copy_(t)
    out[..., 3] = D
    return out.reshape(-1, 4)


def _conv64(x, w, bias=None):
    """3x3x3 convolution of [ns, nz+2, ny+2, nx+2, cin] with a halo, w [27, cout, cin]."""
    nz, ny, nx = (s - 2 for s in x.shape[1:4])
    y = torch.zeros(x.shape[:1] + (nz, ny, nx, w.shape[1]), device="cuda", dtype=torch.float64)
    for t in range(27):
        a, b, c = t // 9, t // 3 % 3, t % 3
        y += x[:, a:a + nz, b:b + ny, c:c + nx] @ w[t].T
    return y if bias is None else y + bias


def _halo(v):
    return torch.nn.functional.pad(v, (0, 0, 1, 1, 1, 1, 1, 1))


def _net64(r, lnk, params):
    P, at, W = params.double(), 0, []
    for cin, cout in NET_LAYERS:
        n = 27 * cin * cout
        W.append((P[at:at + n].view(27, cout, cin), P[at + n:at + n + cout]))
        at += n + cout

    def conv(x, i, relu=True):
        y = _conv64(_halo(x), *W[i])
        return y.clamp_(min=0) if relu else y

    def pool(x):
        s, c, b, a, ch = x.shape
        return x.view(s, c // 2, 2, b // 2, 2, a // 2, 2, ch).mean((2, 4, 6))

    def up(x):
        for axis in (1, 2, 3):
            x = x.repeat_interleave(2, axis)
        return x

    r = r.double()
    rms = (r * r).mean((1, 2, 3), keepdim=True).sqrt()
    e0 = conv(torch.stack((r / rms, lnk.double()), -1), 0)
    e1 = conv(pool(e0), 1)
    d2 = conv(conv(pool(e1), 2), 3)
    d1 = conv(up(d2) + e1, 4)
    d0 = conv(up(d1) + e0, 5)
    return (rms * conv(d0, 6, False)[..., 0]).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        g = _gen(seed)
        K = _field(case["nx"], case["ny"], case["nz"], case["sigma"], g)
        p = (2.0 * _uniform((K.numel(),), g) - 1.0).float().double().view_as(K)
        T, E, _, _ = _faces(dict(K=K, mask=None, pD=None, d=1e-3))
        if case["records"] == "bf16":
            T = [None if t is None else t.bfloat16().double() for t in T]
            D = _diag(T, E.bfloat16().double())
        else:
            D = _diag(T, E).float().double()
            T = [None if t is None else t.float().double() for t in T]
        q = _matvec(T, D, p)
        return [q.reshape(-1), (p * q).sum().reshape(1)] if case["dot"] else [q.reshape(-1)]
    if kind == "setup":
        P = _problem(case, seed)
        p0, P["p0"] = P["p0"], None
        T, E, lift, m = _faces(P)
        D = torch.where(m, torch.ones_like(E), _diag(T, E))
        b = _rhs(P, lift, m)
        rec = _records(T, D)
        return [rec, rec, b.reshape(-1), (b - _matvec(T, D, p0)).reshape(-1)]
    if kind in ("solve", "step", "learned"):
        return _solution(_problem(case, seed))
    if kind == "ensemble":
        return torch.cat([_solution(P) for P in _ensemble(case, seed)])
    if kind == "unet":
        r, K = _net_inputs(case, seed)
        return _net64(r, K.log().float(), _net_params(seed))
    S = _conv_inputs(case, seed)
    x, w = S["x"].double(), S["w"].double()
    if kind == "conv":
        return _halo(_conv64(x, w, S["bias"].double()).clamp_(min=0))
    dy = S["dy"].double()
    dx = _conv64(dy, S["wt"].double()) * (x[:, 1:-1, 1:-1, 1:-1] > 0)
    nx, ny, nz, _ = S["shape"]
    flat = dy[:, 1:-1, 1:-1, 1:-1].reshape(-1, S["cout"])
    dw = torch.stack([flat.T @ x[:, t // 9:t // 9 + nz, t // 3 % 3:t // 3 % 3 + ny,
                                 t % 3:t % 3 + nx].reshape(-1, S["cin"]) for t in range(27)])
    return [_halo(dx), dw]
