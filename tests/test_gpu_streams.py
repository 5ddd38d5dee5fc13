"""First calls on a side stream while the default stream has work queued: what a
call clears or copies for itself is ordered with the caller's stream, whatever
another stream is doing."""
import numpy as np
import pytest
import torch

from paper_2408_03452_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_03452_gb300 import build, tpfa
    build.build()
    return tpfa


def _busy():
    """About 0.1 s of ordinary work on the default stream."""
    a = torch.ones(1 << 28, device="cuda")
    for _ in range(300):
        a.mul_(1.0)
    return a


def _system(tp, shape, seed):
    nx, ny, nz = shape
    K = torch.from_numpy(synth.lognormal_field(nx, ny, nz, 1.0, seed)).cuda()
    mask, pD = (torch.from_numpy(v).cuda() for v in synth.dirichlet_faces(nx, ny, nz, "x", 1.0, 0.0))
    with tp.Context(*shape) as ctx:
        coef, coef64 = ctx.build_trans(K, mask, None, 0.0)
        b = ctx.build_rhs(K, mask, None, pD)
    return coef, coef64, b


@pytest.mark.parametrize("precond", [0, 1])
@pytest.mark.parametrize("shape", [(33, 17, 9), (128, 128, 80)])
def test_first_solve_on_a_side_stream(tp, shape, precond):
    """Low and tall bricks of the resident solve."""
    coef, coef64, b = _system(tp, shape, 21)
    side = torch.cuda.Stream()
    xs = []
    for busy in (False, True):
        with tp.Context(*shape) as ctx:
            ctx.set_option("precond", precond)
            x = torch.zeros_like(b)
            torch.cuda.synchronize()
            keep = _busy() if busy else None
            with torch.cuda.stream(side):
                _, info = ctx.cg_solve(coef, coef64, b, x=x, tol=1e-8, maxit=20000, check=False)
            torch.cuda.synchronize()
            del keep
            assert info["code"] == 0, info
            xs.append(x.cpu().numpy())
    assert np.array_equal(*xs)


def test_first_batched_solve_on_a_side_stream(tp):
    grids = [(33, 17, 9), (48, 48, 24), (20, 40, 12)]
    parts = [_system(tp, g, 31 + i) for i, g in enumerate(grids)]
    coef, coef64, b = (torch.cat([p[k] for p in parts]) for k in range(3))
    side = torch.cuda.Stream()
    xs = []
    for busy in (False, True):
        with tp.BatchContext(grids) as bc:
            x = torch.zeros_like(b)
            torch.cuda.synchronize()
            keep = _busy() if busy else None
            with torch.cuda.stream(side):
                _, _, tot = bc.cg_solve(coef, coef64, b, x=x, tol=1e-8, maxit=20000, check=False)
            torch.cuda.synchronize()
            del keep
            assert tot["code"] == 0, tot
            xs.append(x.cpu().numpy())
    assert np.array_equal(*xs)


def test_new_network_on_a_side_stream(tp):
    """Created while the default stream is busy: the clears of its buffers do not
    land in the weights or between the layers."""
    from paper_2408_03452_gb300 import learned
    n = 32
    g = torch.Generator(device="cuda").manual_seed(5)
    r, lnk = (torch.randn(n ** 3, generator=g, device="cuda") for _ in range(2))
    P = learned.init_params(3).cuda()
    side = torch.cuda.Stream()
    zs = []
    for busy in (False, True):
        torch.cuda.synchronize()
        keep = _busy() if busy else None
        net = tp.UNet(n, n, n, 1)
        with torch.cuda.stream(side):
            net.set_params(P)
            z = net.forward(r, lnk)
        torch.cuda.synchronize()
        del keep
        zs.append(z.cpu().numpy())
    assert np.isfinite(zs[0]).all() and np.abs(zs[0]).max() > 0
    assert np.array_equal(*zs)


def test_batched_sweeps_and_flexible_cg_on_a_side_stream(tp):
    """A batch created, and a flexible-CG solve made, while the default stream is busy."""
    grids = [(24, 20, 12), (33, 17, 9)]
    parts = [_system(tp, g, 41 + i) for i, g in enumerate(grids)]
    coef, coef64, b = (torch.cat([p[k] for p in parts]) for k in range(3))
    side = torch.cuda.Stream()
    xs, es = [], []
    for busy in (False, True):
        x, e = torch.zeros_like(b), torch.zeros_like(parts[0][2])
        with tp.Context(*grids[0]) as ctx:
            ctx.set_option("fcg_m", 2)
            torch.cuda.synchronize()
            keep = _busy() if busy else None
            with torch.cuda.stream(side):
                _, info = ctx.fcg_solve(*parts[0], x=e, tol=1e-8,
                                        maxit=5000, check=False)
            torch.cuda.synchronize()
            del keep
        keep = _busy() if busy else None
        with tp.BatchContext(grids) as bc:
            bc.set_option("tma_tile", 1)
            with torch.cuda.stream(side):
                _, _, tot = bc.cg_solve(coef, coef64, b, x=x, tol=1e-8, maxit=20000, check=False)
            torch.cuda.synchronize()
        del keep
        assert info["code"] == 0 and tot["code"] == 0, (info, tot)
        xs.append(x.cpu().numpy())
        es.append(e.cpu().numpy())
    assert np.array_equal(*xs) and np.array_equal(*es)


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("shape", [(24, 20, 12), (64, 33, 40)])
def test_operator_beside_another_stream(tp, shape, bf16):
    """The operator on a vector rewritten before each call, quiet and beside traffic
    that fills the load pipes: bit for bit the same (a stage of the ring is refilled
    only when every lane has read it)."""
    nx, ny, nz = shape
    n = nx * ny * nz
    K = torch.from_numpy(synth.lognormal_field(nx, ny, nz, 1.0, 51)).cuda()
    g = torch.Generator(device="cuda").manual_seed(3)
    ps = [torch.randn(n, generator=g, device="cuda") for _ in range(150)]
    work = torch.empty(n, device="cuda")
    side = torch.cuda.Stream()
    with tp.Context(*shape) as ctx:
        coef = ctx.build_trans_bf16(K, None, None, 1e-3) if bf16 else ctx.build_trans(K, None, None, 1e-3)[0]
        op = ctx.apply_bf16 if bf16 else ctx.apply
        out = [[torch.empty(n, device="cuda") for _ in ps] for _ in range(2)]
        torch.cuda.synchronize()
        for p, y in zip(ps, out[0]):
            work.copy_(p)
            op(coef, work, y)
        for _ in range(6):
            torch.cuda.synchronize()
            keep = _busy()
            with torch.cuda.stream(side):
                for p, y in zip(ps, out[1]):
                    work.copy_(p)
                    op(coef, work, y)
            torch.cuda.synchronize()
            del keep
            assert all(torch.equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("levels", [0, 1, 2])
def test_learned_solve_beside_another_stream(tp, levels):
    """Flexible CG with a network, whose operator also forms the dot products (levels 1
    and 2: of the network's coarser output), quiet and beside another stream."""
    from paper_2408_03452_gb300 import learned
    n = 32
    coef, coef64, b = _system(tp, (n, n, n), 52)
    lnk = tp.log_perm(torch.from_numpy(synth.lognormal_field(n, n, n, 1.0, 52)).cuda())
    net = tp.UNet(*(3 * [n >> levels]))
    net.set_params(learned.init_params(4).cuda())
    side = torch.cuda.Stream()
    xs = []
    with tp.Context(n, n, n) as ctx:
        ctx.set_option("fcg_m", 2)
        for busy in (False, True, True, True):
            x = torch.zeros_like(b)
            torch.cuda.synchronize()
            keep = _busy() if busy else None
            with torch.cuda.stream(side):
                _, info = ctx.fcg_solve(coef, coef64, b, net=net, lnk=lnk, x=x, tol=1e-8, maxit=3000,
                                        check=False)
            torch.cuda.synchronize()
            del keep
            xs.append((x.cpu().numpy(), info["iters"], info["code"]))
    assert xs[0][2] == 0
    for x, it, _ in xs[1:]:
        assert it == xs[0][1] and np.array_equal(x, xs[0][0])
