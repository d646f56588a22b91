"""The FP64 condensation product on columns whose entries span many binary
orders: every entry of C to the error of an FP64 sum of its own terms,
(m + 4) 2^-53 sum_i |a_ip a_iq| / w_i, wherever the spread lies (fixed point
per column would lose the small entries)."""
import numpy as np
import pytest

import paper_2605_13736_gb300 as m
from gpu_util import dev, make_ctx, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    m.mdsip_ctx_destroy(c)


def _check(ctx, A, w, beta, pairs):
    torch = torch_cuda()
    mm, n = A.shape
    C0 = np.random.default_rng(1).standard_normal((n, n))
    C = dev(C0.T.copy())
    m.mdsip_syrk_scaled(ctx, mm, n, dev(A), n, dev(w), beta, C, n)
    torch.cuda.synchronize()
    got = C.cpu().numpy().T
    ld = np.longdouble
    for p, q in pairs:
        t = A[:, p].astype(ld) * A[:, q].astype(ld) / w.astype(ld)
        want = t.sum() + beta * ld(C0[p, q])
        # one more rounding each for 1 / w, a / w and the addition to C, and one to spare
        tol = 2.0 ** -53 * ((mm + 4) * np.abs(t).sum() + abs(beta * ld(C0[p, q])))
        assert abs(ld(got[p, q]) - want) <= tol, (p, q, float(abs(ld(got[p, q]) - want) / np.abs(t).sum()))


PAIRS = [(131, 5), (131, 131), (5, 5), (140, 131), (140, 5), (199, 0)]


@pytest.mark.parametrize("k", [5, 8, 12, 20, 40, 60])
@pytest.mark.parametrize("beta", [0.0, 1.0])
def test_one_large_entry(ctx, k, beta):
    """Row 0 of column 131 is 2^k above the rest and meets zeros elsewhere."""
    rng = np.random.default_rng(k)
    mm, n = 600, 200
    A = rng.standard_normal((mm, n))
    A[0] = 0.0
    A[0, 131] = 2.0 ** k
    _check(ctx, A, np.ones(mm), beta, PAIRS)


@pytest.mark.parametrize("k", [20, 40, 60])
def test_row_blocks_of_different_scales(ctx, k):
    """[2^k X 0; Y Z]: the large rows of the left columns meet zeros of the right ones."""
    rng = np.random.default_rng(k)
    mm, n = 800, 200
    A = rng.standard_normal((mm, n))
    A[:mm // 2, :100] *= 2.0 ** k
    A[:mm // 2, 100:] = 0.0
    _check(ctx, A, np.ones(mm), 1.0, PAIRS)


@pytest.mark.parametrize("row", [0, 32767, 39999])
def test_spread_from_the_weights_in_any_chunk(ctx, row):
    """A weight of 2^-60 in one row, in whichever range of rows it falls, with C kept until then."""
    rng = np.random.default_rng(row)
    mm, n = 40000, 72
    A = rng.standard_normal((mm, n))
    A[row, ::2] = 0.0
    w = np.ones(mm)
    w[row] = 2.0 ** -60
    _check(ctx, A, w, 1.0, [(71, 0), (70, 2), (71, 1), (33, 33), (40, 31)])
