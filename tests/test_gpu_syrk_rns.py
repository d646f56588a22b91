"""The FP64 condensation product by residue numbers (tensor cores) at the sizes
where it can go wrong, element by element against extended precision, and the
operands outside its range, which take the DFMA kernel instead."""
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


def _product(ctx, A, w, beta=0.0, C0=None):
    torch = torch_cuda()
    mm, n = A.shape
    lda = n + (n & 1)
    Ap = np.full((mm, lda), np.nan)      # the padding column is never used
    Ap[:, :n] = A
    C = dev(np.zeros((n, n)) if C0 is None else C0.T.copy())
    m.mdsip_syrk_scaled(ctx, mm, n, dev(Ap), lda, dev(w), beta, C, n)
    torch.cuda.synchronize()
    return C.cpu().numpy().T


def _case(kind, rng, mm, n):
    A = rng.standard_normal((mm, n))
    w = 10.0 ** rng.uniform(-4, 1, mm)
    if kind == "wide":                   # weights and columns over many binades
        w = 10.0 ** rng.uniform(-8, 8, mm)
        A *= 10.0 ** rng.uniform(-30, 30, n)
    elif kind == "constant":             # equal rows: the accumulators reach their bound 256^3
        A = np.repeat(rng.standard_normal((1, n)), mm, axis=0)
        w = np.ones(mm)
    elif kind == "sparse":               # zero columns and mostly-zero rows
        A *= rng.random((mm, n)) < 0.05
        A[:, n // 2] = 0.0
    return A, w


# orders around the 128/256 tile edges and below one box; rows around the
# 64-row slab, the 256-row fold and the 32768-row chunk; 5003 x 1500 takes
# several chunks, splits and both tile parities
@pytest.mark.parametrize("mm,n,kind", [
    (257, 250, "mild"), (320, 256, "constant"), (1000, 129, "wide"), (4099, 65, "sparse"), (5003, 1500, "mild"),
    (32768, 70, "constant"), (33000, 97, "wide"), (20000, 383, "sparse"), (300, 257, "constant")])
def test_residue_product(ctx, mm, n, kind):
    rng = np.random.default_rng(mm + n)
    A, w = _case(kind, rng, mm, n)
    C0 = rng.standard_normal((n, n)) if kind != "wide" else np.zeros((n, n))
    got = _product(ctx, A, w, 1.0, C0)
    up = np.triu_indices(n, 1)
    np.testing.assert_array_equal(got[up], C0[up])
    ld = np.longdouble
    S = A.astype(ld) / np.sqrt(w.astype(ld))[:, None]
    big, tot = np.abs(S).max(axis=0), np.abs(S).sum(axis=0)
    P = np.concatenate([rng.integers(0, n, 150), [0, n - 1, n - 1]])
    Q = np.concatenate([rng.integers(0, n, 150), [0, n - 1, 0]])
    P, Q = np.maximum(P, Q), np.minimum(P, Q)
    P[:20] = Q[:20]
    for p, q in zip(P, Q):
        want = (S[:, p] * S[:, q]).sum() + C0[p, q]
        # each entry is rounded once to a multiple of its column's unit, at most
        # 4 max|s| 2^-53 in a chunk: half a unit per factor, the square of units
        # below that, and FP64 roundings of the sums added to C (<= 16 chunks)
        tol = 2.0 ** -52 * (big[p] * tot[q] + big[q] * tot[p]) + 16 * 2.0 ** -53 * (
            abs(C0[p, q]) + (np.abs(S[:, p] * S[:, q])).sum())
        assert abs(ld(got[p, q]) - want) <= tol, (p, q)


@pytest.mark.parametrize("kind", ["negative", "zero_w", "nan", "inf", "subnormal", "tiny_w"])
def test_operands_outside_the_residue_range(ctx, kind):
    """They keep the DFMA kernel's results: bit for bit those of the definition
    where it is exact (dyadic values), non-finite where it is not finite."""
    rng = np.random.default_rng(7)
    mm, n = 400, 200
    A = rng.integers(-8, 9, (mm, n)).astype(float)
    w = 2.0 ** rng.integers(-2, 3, mm)
    if kind == "negative":
        w[5] = -w[5]
    elif kind == "zero_w":
        w[5] = 0.0
        A[5] = 1.0
    elif kind == "nan":
        A[17, 30] = np.nan
    elif kind == "inf":
        A[17, 30] = np.inf
    elif kind == "subnormal":
        A[:, 30] = 0.0
        A[17, 30] = 2.0 ** -1060
    else:
        w[:] = 2.0 ** -1010
        A *= 2.0 ** -500
    with np.errstate(all="ignore"):
        want = np.einsum("ip,iq->pq", A / w[:, None], A)
    got = _product(ctx, A, w)
    low = np.tril_indices(n)
    fin = np.isfinite(want[low])
    np.testing.assert_array_equal(np.isnan(got[low]), np.isnan(want[low]))
    np.testing.assert_array_equal(got[low][fin], want[low][fin])
