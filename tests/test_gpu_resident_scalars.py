"""Precision of the resident CG: scalars over the whole FP32 range, iterations of the
sweep on high-contrast fields."""
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


def _inner(tp, shape, precond, sweep):
    nx, ny, nz = shape
    K = torch.from_numpy(synth.lognormal_field(nx, ny, nz, 1.0, 5)).cuda()
    q = torch.from_numpy(synth.dense_sources(nx * ny * nz, *synth.well_pair(nx, ny, nz))).cuda()
    with tp.Context(*shape) as ctx:
        for k, v in dict(precond=precond, sweep=sweep, max_outer=1, inner_rtol=1e-20).items():
            ctx.set_option(k, v)
        coef, coef64 = ctx.build_trans(K, None, None, 1e-3)
        b = ctx.build_rhs(K, None, q, None)
        x, info = ctx.cg_solve(coef, coef64, b, tol=1e-30, maxit=20000, check=False)
        torch.cuda.synchronize()
        assert torch.isfinite(x).all()
        return info


@pytest.mark.parametrize("precond", [0, 1])
@pytest.mark.parametrize("shape", [(33, 17, 9), (40, 20, 12), (64, 64, 40)])
def test_inner_tolerance_of_1e20(tp, shape, precond):
    """The recurrence's r'r and p'Ap fall by forty orders of magnitude, below the
    normal range of FP32.  The resident solve goes on as the sweep does: iterations
    within a tenth, the same attainable residual (to a factor of two)."""
    a, s = (_inner(tp, shape, precond, sweep) for sweep in (0, 1))
    assert a["code"] == s["code"] == tp.NOTCONV, (a, s)
    assert a["rel_res_inner"] <= 1.01e-20
    assert abs(a["iters"] - s["iters"]) <= 0.1 * s["iters"], (a, s)
    assert a["rel_res_fp64"] <= 2 * s["rel_res_fp64"], (a, s)


@pytest.mark.parametrize("b16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("shape", [(100, 100, 100), (128, 128, 80), (128, 128, 120)])
def test_jacobi_iterations_of_tall_bricks(tp, shape, b16):
    """High-contrast fields (channels 1e4 times more permeable) over bricks of 24 and 32
    planes: the operator of the inner solve is that of the records, so the resident
    Jacobi solve takes the iterations of the sweep, to 3 % over four fields."""
    nx, ny, nz = shape
    total = [0, 0]
    for seed in range(4):
        K = torch.from_numpy(synth.channelized_field(nx, ny, nz, 2.0, 60 + seed)).cuda()
        mask, pD = (torch.from_numpy(v).cuda() for v in synth.dirichlet_faces(nx, ny, nz, "x", 1.0, 0.0))
        for sweep in (0, 1):
            with tp.Context(*shape) as ctx:
                ctx.set_option("precond", 1)
                ctx.set_option("sweep", sweep)
                coef, coef64 = ctx.build_trans(K, mask, None, 0.0)
                inner = ctx.build_trans_bf16(K, mask, None, 0.0) if b16 else coef
                b = ctx.build_rhs(K, mask, None, pD)
                _, info = ctx.cg_solve(inner, coef64, b, tol=1e-12, maxit=100000, check=False)
                assert info["code"] == 0, info
                total[sweep] += info["iters"]
    assert abs(total[0] - total[1]) <= 0.03 * total[1], total
