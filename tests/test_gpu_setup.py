"""Coefficient records and right-hand sides over the whole FP64 range: quotients
formed in integer arithmetic and those that fall back to the operator (zeros,
subnormals, infinities, negative values, quotients out of range) against NumPy's,
bit for bit, on tiles with ragged edges, several z-runs and thin grids."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_03452_gb300 import build, tpfa
    build.build()
    return tpfa


def _K(kind, n, rng):
    if kind == "plain":
        return rng.lognormal(0.0, 2.0, n)
    if kind == "fractions":  # leading or trailing runs of ones and zeros
        f = rng.integers(0, 1 << 52, n, dtype=np.uint64)
        s = rng.integers(0, 52, n, dtype=np.uint64)
        low = (np.uint64(1) << s) - np.uint64(1)
        f = np.where(rng.random(n) < 0.5, f | low, f & ~low) & np.uint64((1 << 52) - 1)
        return (f | np.uint64(1023 << 52)).view(np.float64)
    K = np.exp2(rng.uniform(-1070.0, 1020.0, n))
    special = np.array([0.0, -0.0, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308, np.inf,
                        -1.0, -3.5])
    pick = rng.random(n) < 0.1
    return np.where(pick, special[rng.integers(0, len(special), n)], K)


def _shift(a, axis, step, fill=0.0):
    """a of the neighbour at +-1 along the axis (0: x, 1: y, 2: z); a has shape (nz, ny, nx)."""
    ax, out = 2 - axis, np.full_like(a, fill)
    src = [slice(None)] * 3
    dst = [slice(None)] * 3
    src[ax], dst[ax] = (slice(1, None), slice(None, -1)) if step > 0 else (slice(None, -1), slice(1, None))
    out[tuple(dst)] = a[tuple(src)]
    return out


def _reference(shape, geom, K, mask, q, pD):
    nx, ny, nz = shape
    K, q, pD = (a.reshape(nz, ny, nx) for a in (K, q, pD))
    m = mask.reshape(nz, ny, nx) != 0
    h = [geom["dx"], geom["dy"], geom["dz"]]
    area = [h[1] * h[2] / geom["mu"], h[0] * h[2] / geom["mu"], h[0] * h[1] / geom["mu"]]
    D, b, T = np.zeros_like(K), q.copy(), []
    for a in range(3):
        half = 0.5 * h[a] / K
        face = area[a] / (half + _shift(half, a, 1))
        inside = _shift(np.ones_like(K), a, 1) != 0
        face = np.where(inside, face, 0.0)
        dn, dp = _shift(m, a, -1, False), _shift(m, a, 1, False)
        for s, dir_, at in ((_shift(face, a, -1), dn, -1), (face, dp, 1)):
            D = D + s
            with np.errstate(invalid="ignore"):
                b = np.where(dir_, b + s * _shift(pD, a, at), b)
        T.append(np.where(m | dp, 0.0, face))
    coef = np.stack([*T, np.where(m, 1.0, D + 1e-3)], axis=-1).reshape(-1, 4)
    return coef, np.where(m, pD, b).reshape(-1)


@pytest.mark.parametrize("kind", ["plain", "fractions", "range"])
@pytest.mark.parametrize("geom", [dict(dx=1.0, dy=1.0, dz=1.0, mu=1.0),
                                  dict(dx=0.7, dy=2.0, dz=1.3, mu=0.3)], ids=["equal", "unequal"])
@pytest.mark.parametrize("shape", [(32, 8, 17), (33, 9, 40), (65, 23, 5), (31, 7, 3), (3, 200, 9),
                                   (200, 2, 4), (1, 1, 1)])
def test_setup_bits(tp, shape, geom, kind):
    n = shape[0] * shape[1] * shape[2]
    rng = np.random.default_rng([n, len(kind)])
    K, q = _K(kind, n, rng), rng.standard_normal(n)
    mask = (rng.random(n) < 0.15).astype(np.uint8)
    # powers of two: T p^D is exact, so one rounding or two make no difference
    pD = np.where(mask != 0, np.exp2(rng.integers(-2, 3, n).astype(np.float64)), 0.0)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    with tp.Context(*shape, **geom) as ctx:
        coef, coef64 = ctx.build_trans(dev(K), dev(mask), None, 1e-3)
        b = ctx.build_rhs(dev(K), dev(mask), dev(q), dev(pD)).cpu().numpy()
    with np.errstate(all="ignore"):
        ref, ref_b = _reference(shape, geom, K, mask, q, pD)
        np.testing.assert_array_equal(coef64.cpu().numpy(), ref)
        np.testing.assert_array_equal(coef.cpu().numpy(), ref.astype(np.float32))
        np.testing.assert_array_equal(b, ref_b)
