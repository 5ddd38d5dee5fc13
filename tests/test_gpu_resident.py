"""The resident CG kernel (inner solves of grids that fit on the chip) against
the cp.async sweep, which does the same per-cell arithmetic, and the oracle.

Shapes: one cell, single brick columns and planes, bricks with ragged edges on
every axis, several bricks along every axis, every brick height (1 to 32
planes), the largest grid that fits one brick per SM and the first that does
not (which keeps the sweeps)."""
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


def _case(shape, seed, kind, kscale=1.0, sigma=1.0):
    nx, ny, nz = shape
    n = nx * ny * nz
    K = synth.lognormal_field(nx, ny, nz, sigma, seed) * kscale
    if kind == "dirx":
        mask, pD = synth.dirichlet_faces(nx, ny, nz, "x", 1.0, 0.0)
        return dict(K=K, mask=mask, pD=pD, d=0.0, q=None)
    q = synth.dense_sources(n, *synth.well_pair(nx, ny, nz))
    return dict(K=K, mask=None, pD=None, d=1e-3 * kscale, q=q)


def _solve(tp, shape, c, tol, maxit, opts, b16=False):
    dev = lambda a: None if a is None else torch.from_numpy(a).cuda()  # noqa: E731
    with tp.Context(*shape) as ctx:
        for k, v in opts.items():
            ctx.set_option(k, v)
        K, mask = dev(c["K"]), dev(c["mask"])
        coef, coef64 = ctx.build_trans(K, mask, None, c["d"])
        inner = ctx.build_trans_bf16(K, mask, None, c["d"]) if b16 else coef
        b = ctx.build_rhs(K, mask, dev(c["q"]), dev(c["pD"]))
        x, info = ctx.cg_solve(inner, coef64, b, tol=tol, maxit=maxit, check=False)
        torch.cuda.synchronize()
        return x.cpu().numpy(), info


# a resident inner solve is one launch: residual + solve + residual per step
def _resident(info):
    return info["kernel_launches"] <= 2 * info["outer"] + 2


SHAPES = [((1, 1, 1), "wells"), ((5, 3, 2), "wells"), ((32, 16, 1), "wells"), ((33, 17, 9), "dirx"),
          ((31, 15, 40), "wells"), ((64, 1, 300), "wells"), ((1, 200, 7), "wells"),
          ((100, 30, 41), "wells"), ((65, 47, 90), "dirx"), ((48, 24, 200), "wells"),
          ((96, 96, 48), "dirx"), ((128, 128, 64), "wells"), ((65, 33, 300), "dirx"),
          ((128, 128, 128), "wells")]


@pytest.mark.parametrize("b16,jac", [(False, 0), (False, 1), (True, 0), (True, 1)],
                         ids=["f32", "f32-jacobi", "bf16", "bf16-jacobi"])
@pytest.mark.parametrize("shape,kind", SHAPES)
def test_resident_iterates_and_solution(tp, oracle_mod, shape, kind, b16, jac):
    """Iterates 1 and 3 agree with the sweep's (1e-5 of the norm; by iterate 8
    FP32 CG itself is up to 2e-4 off the FP64 iterates on the well cases, so
    later iterates say nothing), and the refined solve meets its tolerance by
    the oracle's FP64 residual."""
    O = oracle_mod
    c = _case(shape, 11, kind)
    n = shape[0] * shape[1] * shape[2]
    for k in [k for k in (1, 3) if k < n]:
        x0, i0 = _solve(tp, shape, c, 1e-30, k, {"precond": jac, "max_outer": 1}, b16)
        x1, i1 = _solve(tp, shape, c, 1e-30, k, {"precond": jac, "max_outer": 1, "sweep": 1}, b16)
        assert i0["iters"] == i1["iters"] == k and _resident(i0) and not _resident(i1)
        assert np.linalg.norm(x0 - x1) <= 1e-5 * np.linalg.norm(x1), k
    tol = 1e-9
    x, info = _solve(tp, shape, c, tol, 400000, {"precond": jac}, b16)
    assert info["code"] == 0 and _resident(info), info
    g = O.Grid(*shape)
    assert O.rel_residual(g, c["K"], c["mask"], c["d"], c["q"], c["pD"], x) <= tol * 1.01
    x2, _ = _solve(tp, shape, c, tol, 400000, {"precond": jac}, b16)
    assert np.array_equal(x, x2)  # fixed-order sums


def test_grid_beyond_the_chip_keeps_the_sweeps(tp):
    c = _case((192, 160, 96), 12, "wells")
    _, info = _solve(tp, (192, 160, 96), c, 1e-4, 1000, {"precond": 1})
    assert info["code"] == 0 and not _resident(info)


@pytest.mark.parametrize("kscale", [1e-22, 1e14])
def test_resident_scale_of_the_permeability(tp, oracle_mod, kscale):
    """Permeabilities far from one (an m^2 field, a huge one): the iteration
    works on the operator scaled by a power of two."""
    O = oracle_mod
    shape = (40, 20, 12)
    c = _case(shape, 13, "wells", kscale)
    x, info = _solve(tp, shape, c, 1e-9, 400000, {})
    assert info["code"] == 0 and _resident(info), info
    g = O.Grid(*shape)
    assert O.rel_residual(g, c["K"], None, c["d"], c["q"], None, x) <= 1e-9 * 1.01


def test_resident_reports_nonfinite_and_limits(tp):
    shape = (40, 20, 12)
    c = _case(shape, 14, "wells")
    x, info = _solve(tp, shape, c, 1e-9, 7, {})
    assert info["code"] == 1 and info["iters"] == 7 and np.isfinite(x).all()
    c["K"] = c["K"].copy()
    c["K"][1234] = np.nan
    _, info = _solve(tp, shape, c, 1e-9, 100, {})
    assert info["code"] == tp.ENONFINITE
