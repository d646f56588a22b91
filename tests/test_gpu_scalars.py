"""The scalar pieces that stand in for the division operator, log and square
root in the kernels: against extended precision, at random, at the edges of
their ranges and of their rounding, and on special values."""
import numpy as np
import pytest

import paper_2605_13736_gb300 as m
from gpu_util import dev, make_ctx, torch_cuda

pytestmark = pytest.mark.gpu
LD = np.longdouble
RCP, DIV, LOGSUM, ADAM, RSQRT = range(5)
needs_quad = pytest.mark.skipif(np.finfo(LD).nmant < 100, reason="the host's long double is too short to judge by")


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    m.mdsip_ctx_destroy(c)


def _run(ctx, op, a, b=None, per=1, count=None):
    torch = torch_cuda()
    n = len(a) if count is None else count
    out = torch.zeros(per * n, dtype=torch.float64, device="cuda")
    m.mdsip_debug_scalar(ctx, op, n, dev(a), dev(b) if b is not None else None, out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _mantissas(rng, n):
    """Random ones, 1, all ones, both neighbours, and few-bit ones."""
    k = rng.integers(0, 2 ** 52, n)
    edge = np.concatenate([[0, 1, 2, 2 ** 52 - 1, 2 ** 52 - 2, 2 ** 51, 2 ** 51 - 1, 2 ** 51 + 1, 2 ** 29 - 1, 2 ** 29,
                            2 ** 52 - 2 ** 29, 2 ** 52 - 2 ** 28], 2 ** np.arange(52), 2 ** 52 - 2 ** np.arange(1, 52)])
    return np.concatenate([k, edge]).astype(np.int64)


def _doubles(rng, n, lo, hi):
    """Doubles of biased exponent lo .. hi (each edge with the edge mantissas), either sign."""
    k = _mantissas(rng, n)
    e = rng.integers(lo, hi + 1, len(k))
    k = np.concatenate([k, _mantissas(rng, 0), _mantissas(rng, 0)])
    e = np.concatenate([e, np.full(len(_mantissas(rng, 0)), lo), np.full(len(_mantissas(rng, 0)), hi)])
    s = rng.integers(0, 2, len(k))
    return np.where(s, -1.0, 1.0) * ((e.astype(np.int64) << 52) | k).view(np.float64)


def _ulps(got, want):
    """|got - want| in units in the last place of want."""
    want = want.astype(LD)
    _, e = np.frexp(want)
    return np.abs(got.astype(LD) - want) / np.ldexp(LD(1.0), e - 53)


@needs_quad
@pytest.mark.parametrize("lo,hi", [(1, 2046), (100, 1946), (99, 100), (1946, 1947), (1022, 1024)])
def test_reciprocal(ctx, lo, hi):
    d = _doubles(np.random.default_rng(lo), 200000, lo, hi)
    want = LD(1.0) / d.astype(LD)
    got = _run(ctx, RCP, d)
    ok = np.abs(want) >= LD(2.0) ** -1022      # (a subnormal quotient has coarser units)
    assert (_ulps(got[ok], want[ok]) <= 0.51).all(), float(_ulps(got[ok], want[ok]).max())
    np.testing.assert_array_equal(got[~ok], (1.0 / d[~ok]))


def test_reciprocal_of_special_values(ctx):
    d = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, -1e-310])
    with np.errstate(all="ignore"):
        want = np.where(d == 0.0, 0.0, 1.0 / d)
    np.testing.assert_array_equal(_run(ctx, RCP, d), want)


@needs_quad
@pytest.mark.parametrize("lo,hi", [(523, 1523), (1000, 1046), (522, 523), (1523, 1524)])
def test_quotient(ctx, lo, hi):
    rng = np.random.default_rng(lo)
    a, b = _doubles(rng, 200000, lo, hi), _doubles(rng, 200000, lo, hi)
    rng.shuffle(b)
    want = a.astype(LD) / b.astype(LD)
    assert (_ulps(_run(ctx, DIV, a, b), want) <= 0.51).all(), float(_ulps(_run(ctx, DIV, a, b), want).max())


def test_quotient_of_special_values(ctx):
    v = np.array([0.0, -0.0, 1.0, -3.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, 1e308, -1e308, 1e-300, 2.0 ** -500,
                  2.0 ** 500, 2.0 ** 501, 2.0 ** -501])
    a, b = (x.ravel() for x in np.meshgrid(v, v))
    with np.errstate(all="ignore"):
        want = a / b
    np.testing.assert_array_equal(_run(ctx, DIV, a, b), want)   # short quotients: every form is exact or rounds alike


@needs_quad
@pytest.mark.parametrize("lo,hi", [(1, 2046), (1010, 1036), (1022, 1023)])
def test_sum_of_logarithms(ctx, lo, hi):
    rng = np.random.default_rng(lo)
    a = np.abs(_doubles(rng, 160000, lo, hi))
    a = a[:len(a) // 16 * 16]
    got = _run(ctx, LOGSUM, a, count=len(a) // 16)
    logs = np.log(a.astype(LD)).reshape(-1, 16)
    want = logs.sum(axis=1)
    # sixteen rounded products (2^-53 each), the exponent times a rounded log 2 (2^-54
    # relative), one logarithm and two roundings of the total
    e = np.abs(logs).sum(axis=1) / np.log(LD(2.0)) + 16
    tol = 16 * LD(2.0) ** -53 + e * LD(2.0) ** -55 + 3 * LD(2.0) ** -53 * (np.abs(want) + 1)
    assert (np.abs(got.astype(LD) - want) <= tol).all(), float((np.abs(got.astype(LD) - want) / tol).max())


def test_sum_of_logarithms_of_special_values(ctx):
    rows = np.ones((6, 16))
    rows[0, 3], rows[1, 0], rows[2, 15], rows[3, 7] = 0.0, -1.0, np.inf, np.nan
    rows[4, 2] = 1e-310
    rows[5] = 2.0 ** 1000
    got = _run(ctx, LOGSUM, rows.ravel(), count=6)
    assert got[0] == -np.inf and np.isnan(got[1]) and got[2] == np.inf and np.isnan(got[3])
    np.testing.assert_allclose(got[4:], [np.log(1e-310), 16000 * np.log(2.0)], rtol=2.0 ** -51)


def test_adam_quotient(ctx):
    """The branch-free form within two units of the operators' (each of its two
    quotient steps and its root is within one of a rounded operation), NaN outside
    its range only."""
    rng = np.random.default_rng(0)
    mm = np.concatenate([rng.standard_normal(200000) * 10.0 ** rng.uniform(-12, 3, 200000), [0.0, 0.0, 1.0, 1e-30]])
    v = np.concatenate([10.0 ** rng.uniform(-24, 6, 200000), [0.0, 1.0, 0.0, 1e-36]])
    out = _run(ctx, ADAM, mm, v, per=2).reshape(-1, 2)
    assert not np.isnan(out[:200003]).any()
    fast, ref = out[:200000, 0].astype(np.float32), out[:200000, 1].astype(np.float32)
    assert (np.abs(fast - ref) <= 2 * np.spacing(np.abs(ref))).all()
    # bit for bit but for a few: both are the rounded quotient of nearly always the same operands
    assert (fast != ref).mean() < 0.25
    far = _run(ctx, ADAM, np.array([1.0, 1.0, 1.0]), np.array([1e30, 1e-35, 3e37]), per=2).reshape(-1, 2)
    assert np.isnan(far[:, 0]).all() and np.isfinite(far[:, 1]).all()
    assert far[2, 1] == 0.0                     # v / (1 - beta2^t) overflows: no step, as with the operators

@needs_quad
@pytest.mark.parametrize("lo,hi", [(30, 2010), (1022, 1024)])
def test_reciprocal_root(ctx, lo, hi):
    w = np.abs(_doubles(np.random.default_rng(hi), 200000, lo, hi))
    out = _run(ctx, RSQRT, w, per=3).reshape(-1, 3)
    got = np.ldexp(out[:, 0].astype(LD) * LD(2.0) ** 32 + out[:, 1].astype(LD), out[:, 2].astype(int) - 63)
    want = 1 / np.sqrt(w.astype(LD))
    # 64 bits, one Newton correction of a value good to 2^-52: 2^-62 from the integer, 2^-63 beside it
    assert (np.abs(got / want - 1) <= LD(2.0) ** -61).all(), float(np.abs(got / want - 1).max() * LD(2.0) ** 61)
