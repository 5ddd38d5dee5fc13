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
