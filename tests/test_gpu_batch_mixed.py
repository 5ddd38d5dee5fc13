"""Batches in which only some instances fit on the chip: those run resident, the
others in the TMA-staged batched sweep (default tile, plain and Jacobi), and every
instance is bit-identical to the same problem solved alone with its z-run."""
import numpy as np
import pytest
import torch

from paper_2408_03452_gb300 import synth

pytestmark = pytest.mark.gpu

# one brick column per SM at most: 20 x 9 columns of 32 x 16 cells do not fit
SHAPES = [(33, 17, 9), (640, 130, 2), (24, 20, 12), (637, 140, 3), (96, 96, 48)]


@pytest.fixture(scope="module")
def tp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_03452_gb300 import build, tpfa
    build.build()
    return tpfa


def _insts():
    out = []
    for i, (nx, ny, nz) in enumerate(SHAPES):
        K = synth.lognormal_field(nx, ny, nz, 0.8 + 0.2 * i, 300 + i)
        mask, pD = synth.dirichlet_faces(nx, ny, nz, "xyxyz"[i], 1.0, 0.0)
        out.append(dict(shape=(nx, ny, nz), K=K, mask=mask, pD=pD))
    return out


def _system(ctx, insts):
    K, mask, pD = (torch.from_numpy(np.concatenate([w[k] for w in insts])).cuda()
                   for k in ("K", "mask", "pD"))
    coef, coef64 = ctx.build_trans(K, mask, None, 0.0)
    return coef, coef64, ctx.build_rhs(K, mask, None, pD)


@pytest.mark.parametrize("zc", [None, [3, 2, 4, 1, 8]], ids=["auto", "explicit"])
@pytest.mark.parametrize("precond", [0, 1])
def test_mixed_batch_matches_oracle_and_single_solves(tp, oracle_mod, precond, zc):
    O = oracle_mod
    insts = _insts()
    with tp.BatchContext([w["shape"] for w in insts], zc=zc) as bc:
        bc.set_option("precond", precond)
        coef, coef64, b = _system(bc, insts)
        x, per, tot = bc.cg_solve(coef, coef64, b, tol=1e-8)
        again, _, _ = bc.cg_solve(coef, coef64, b, tol=1e-8)
        assert tot["code"] == 0, (tot, per)
        assert torch.equal(x, again)
        xs = [x[bc.offsets[i]:bc.offsets[i + 1]].cpu().numpy() for i in range(len(insts))]
        runs = bc.zc
    for i, w in enumerate(insts):
        assert O.rel_residual(O.Grid(*w["shape"]), w["K"], w["mask"], 0.0, None, w["pD"],
                              xs[i]) <= 1e-8 * 1.001
        with tp.Context(*w["shape"]) as ctx:
            ctx.set_option("tile_zc", runs[i])
            ctx.set_option("precond", precond)
            x1, info = ctx.cg_solve(*_system(ctx, [w]), tol=1e-8)
            fits = info["kernel_launches"] <= 2 * info["outer"] + 2
            assert fits == (w["shape"][0] < 600), info
            assert np.array_equal(xs[i], x1.cpu().numpy()), i
            assert per[i]["iters"] == info["iters"], i
