"""The resident batch's scheduler: instances that queue for SMs."""
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


def _insts(shapes, seed):
    out = []
    for i, (nx, ny, nz) in enumerate(shapes):
        K = synth.lognormal_field(nx, ny, nz, 1.0 + 0.2 * (i % 4), seed + i)
        mask, pD = synth.dirichlet_faces(nx, ny, nz, "xyz"[i % 3], 1.0, 0.0)
        out.append(dict(shape=(nx, ny, nz), K=K, mask=mask, pD=pD))
    return out


def _system(ctx, insts):
    K, mask, pD = (torch.from_numpy(np.concatenate([w[k] for w in insts])).cuda()
                   for k in ("K", "mask", "pD"))
    coef, coef64 = ctx.build_trans(K, mask, None, 0.0)
    return coef, coef64, ctx.build_rhs(K, mask, None, pD)


def test_idle_blocks_stay_while_another_team_runs(tp):
    """Two instances that need most of the chip each: the blocks that the first
    leaves idle wait for the second through a solve many times as long as their
    limit of looks without progress (about 2 ms here; 64 iterations of the running
    team take 0.4)."""
    insts = _insts([(128, 128, 64)] * 2, 61)
    xs = []
    with tp.BatchContext([w["shape"] for w in insts]) as bc:
        coef, coef64, b = _system(bc, insts)
        for looks in (0, 2000):
            assert tp.lib().tpfa_resident_wait_limits(None, bc._h, 0, looks) == tp.OK
            x, per, tot = bc.cg_solve(coef, coef64, b, tol=1e-10, check=False)
            assert tot["code"] == 0, tot
            assert sum(p["iters"] for p in per) > 1500
            xs.append(x.cpu().numpy())
    assert np.array_equal(*xs)


@pytest.mark.parametrize("precond", [0, 1])
def test_queue_of_instances(tp, oracle_mod, precond):
    """Several times as many bricks as SMs, at all three brick heights and of unlike
    sizes: teams wait, blocks are returned and serve again.  Every instance equals its
    solve alone bit for bit, in two solves of the same batch."""
    O = oracle_mod
    shapes = [(128, 128, 64), (48, 48, 24), (96, 96, 48), (24, 20, 12), (128, 128, 64), (33, 17, 9),
              (64, 64, 32), (100, 60, 70), (48, 48, 24), (128, 100, 60), (7, 5, 3), (96, 96, 48),
              (64, 64, 32), (1, 1, 1), (96, 90, 48), (48, 48, 24), (32, 16, 4), (70, 50, 16)]
    insts = _insts(shapes, 400)
    with tp.BatchContext([w["shape"] for w in insts]) as bc:
        bc.set_option("precond", precond)
        coef, coef64, b = _system(bc, insts)
        x, per, tot = bc.cg_solve(coef, coef64, b, tol=1e-9)
        again, per2, _ = bc.cg_solve(coef, coef64, b, tol=1e-9)
        assert tot["code"] == 0, (tot, per)
        assert torch.equal(x, again) and [p["iters"] for p in per] == [p["iters"] for p in per2]
        xs = [x[bc.offsets[i]:bc.offsets[i + 1]].cpu().numpy() for i in range(len(insts))]
        runs = bc.zc
    for i, w in enumerate(insts):
        assert O.rel_residual(O.Grid(*w["shape"]), w["K"], w["mask"], 0.0, None, w["pD"],
                              xs[i]) <= 1e-9 * 1.01
        with tp.Context(*w["shape"]) as ctx:
            ctx.set_option("tile_zc", runs[i])
            ctx.set_option("precond", precond)
            x1, info = ctx.cg_solve(*_system(ctx, [w]), tol=1e-9)
            assert np.array_equal(xs[i], x1.cpu().numpy()) and per[i]["iters"] == info["iters"], i


# ---- waits that run out ------------------------------------------------------
@pytest.mark.parametrize("precond", [0, 1])
@pytest.mark.parametrize("shape", [(33, 17, 9), (64, 64, 64), (128, 128, 64), (100, 100, 100),
                                   (128, 128, 120)])
def test_a_wait_that_runs_out_is_reported(tp, shape, precond):
    """Waits of a single look (in hundreds of exchanges some block's word is not there
    yet at the first): the solve ends by itself with TPFA_EINTERNAL, and the next one on
    the same context is what it would have been."""
    (w,) = _insts([shape], 500)
    with tp.Context(*shape) as ctx:
        ctx.set_option("precond", precond)
        coef, coef64, b = _system(ctx, [w])
        want, info = ctx.cg_solve(coef, coef64, b, tol=1e-9, check=False)
        assert info["code"] == 0
        for _ in range(2):
            assert tp.lib().tpfa_resident_wait_limits(ctx._h, None, 1, 0) == tp.OK
            _, info = ctx.cg_solve(coef, coef64, b, tol=1e-9, check=False)
            assert info["code"] == tp.EINTERNAL, info
            assert tp.lib().tpfa_resident_wait_limits(ctx._h, None, 0, 0) == tp.OK
            x, info = ctx.cg_solve(coef, coef64, b, tol=1e-9, check=False)
            assert info["code"] == 0 and torch.equal(x, want), info


def test_a_wait_that_runs_out_in_a_batch_is_reported(tp):
    insts = _insts([(128, 128, 64), (48, 48, 24), (128, 128, 64), (96, 96, 48), (640, 130, 2)], 510)
    with tp.BatchContext([w["shape"] for w in insts]) as bc:
        coef, coef64, b = _system(bc, insts)
        want, _, tot = bc.cg_solve(coef, coef64, b, tol=1e-8, check=False)
        assert tot["code"] == 0
        for _ in range(2):
            assert tp.lib().tpfa_resident_wait_limits(None, bc._h, 1, 0) == tp.OK
            _, per, tot = bc.cg_solve(coef, coef64, b, tol=1e-8, check=False)
            assert tot["code"] == tp.EINTERNAL and per[0]["status"] == tp.EINTERNAL, per
            assert per[4]["status"] == 0  # the instance in the sweeps is not concerned
            assert tp.lib().tpfa_resident_wait_limits(None, bc._h, 0, 0) == tp.OK
            x, per, tot = bc.cg_solve(coef, coef64, b, tol=1e-8, check=False)
            assert tot["code"] == 0 and torch.equal(x, want), per


def test_wait_limits_are_bounded(tp):
    with tp.Context(4, 4, 4) as ctx:
        L = tp.lib()
        assert L.tpfa_resident_wait_limits(ctx._h, None, (1 << 23) + 1, 0) == tp.EINVAL
        assert L.tpfa_resident_wait_limits(ctx._h, None, 1 << 23, 0) == tp.OK
