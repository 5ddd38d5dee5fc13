"""The loops of the sweeps (graph while node, host-polled chunks), asked for by
TPFA_OPT_SWEEP: solves of grids that fit on the chip take neither by default."""
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


@pytest.mark.parametrize("b16,precond", [(False, 0), (False, 1), (True, 0), (True, 1)],
                         ids=["f32", "f32-jacobi", "bf16", "bf16-jacobi"])
@pytest.mark.parametrize("shape", [(33, 17, 9), (40, 24, 16), (64, 9, 17), (1, 1, 40)])
@pytest.mark.parametrize("sweep", [1, 2], ids=["cpasync", "tma"])
def test_loop_modes_agree_bitwise(tp, oracle_mod, sweep, shape, b16, precond):
    if sweep == 2 and b16 and shape[0] % (4 if precond else 2):
        pytest.skip("the copy engine needs rows of whole 16-byte pieces")
    O = oracle_mod
    nx, ny, nz = shape
    K = synth.lognormal_field(nx, ny, nz, 1.5, 90, layer=2)
    q = synth.dense_sources(nx * ny * nz, *synth.well_pair(nx, ny, nz))
    Kd, qd = torch.from_numpy(K).cuda(), torch.from_numpy(q).cuda()
    xs = []
    for loop, chunk in ((0, 32), (1, 32), (1, 7)):
        with tp.Context(*shape) as ctx:
            for k, v in dict(sweep=sweep, precond=precond, loop=loop, chunk=chunk).items():
                ctx.set_option(k, v)
            coef, coef64 = ctx.build_trans(Kd, None, None, 1e-3)
            inner = ctx.build_trans_bf16(Kd, None, None, 1e-3) if b16 else coef
            b = ctx.build_rhs(Kd, None, qd, None)
            x, info = ctx.cg_solve(inner, coef64, b, tol=1e-8, maxit=100000)
            assert info["code"] == 0 and info["kernel_launches"] > info["iters"], info
            xs.append((x.cpu().numpy(), info["iters"]))
    assert O.rel_residual(O.Grid(*shape), K, None, 1e-3, q, None, xs[0][0]) <= 1e-8 * 1.001
    for x, it in xs[1:]:
        assert it == xs[0][1] and np.array_equal(x, xs[0][0])
