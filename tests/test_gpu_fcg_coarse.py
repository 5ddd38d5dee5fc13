"""Flexible CG with a network on a coarser grid: the operator that reads the
network's output from that grid, against the separate passes (prolongation,
operator, dot products).

One iteration from the same start: both apply the same operator to the same
network output, so the directions differ by the rounding of the blend weight
alone.  Its sums run over FP32 products with compensated or FP64 totals, 2^-22 of
the sums of magnitudes; the weight is a difference, for which a factor of 100 is
allowed, and the step length another sum of the same kind: 1e-4.  A wrong
ancestor or halo value changes the weight by a part of order one."""
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


@pytest.mark.parametrize("shape,f", [((32, 16, 24), 2), ((40, 24, 40), 2), ((72, 56, 8), 2),
                                     ((48, 48, 16), 4), ((80, 16, 144), 4), ((96, 32, 64), 8),
                                     ((160, 96, 32), 8)])
@pytest.mark.parametrize("steps", [1, 3])
def test_coarse_operator_equals_passes(tp, shape, f, steps):
    from test_gpu_unet import params_case
    K = synth.lognormal_field(*shape, 1.0, 3)
    mask, pD = synth.dirichlet_faces(*shape, "x", 1.0, 0.0)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    out = []
    for sweep in (0, 1):
        with tp.Context(*shape) as ctx:
            ctx.set_option("sweep", sweep)
            coef, coef64 = ctx.build_trans(dev(K), dev(mask))
            b = ctx.build_rhs(dev(K), dev(mask), pD=dev(pD))
            net = tp.UNet(*(d // f for d in shape))
            net.set_params(dev(params_case(9)[1]))
            lnk = dev(np.log(K).astype(np.float32))
            x, info = ctx.fcg_solve(coef, coef64, b, net=net, lnk=lnk, tol=1e-14, maxit=steps,
                                    check=False)
            assert info["iters"] == steps and torch.isfinite(x).all()
            out.append(x.cpu().numpy())
    if steps == 1:
        assert np.linalg.norm(out[0] - out[1]) <= 1e-4 * np.linalg.norm(out[1])
    else:  # the network's BF16 roundings may differ from the second iteration on: 2^-8 each
        assert np.linalg.norm(out[0] - out[1]) <= 2.0 ** -6 * np.linalg.norm(out[1])
