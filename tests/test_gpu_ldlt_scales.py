"""The persistent FP64 LDL^T far from scale 1: whole matrices near the ends of
its range and blocks of very different scales in one matrix, entry-wise
against the reconstruction in extended precision."""
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


def _factor(ctx, K, zero_tol):
    torch = torch_cuda()
    N = K.shape[0]
    S = dev(np.tril(K).T.copy())                              # column-major lower triangle
    L = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    Dd, Doff = (torch.zeros(N, dtype=torch.float64, device="cuda") for _ in range(2))
    perm, kind = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    inr = torch.zeros(3, dtype=torch.int32, device="cuda")
    m.mdsip_ldlt_factor(ctx, N, S, N, zero_tol, L, Dd, Doff, perm, kind, inr)
    torch.cuda.synchronize()
    ld = np.longdouble
    Lh, d, o = np.tril(L.cpu().numpy().T).astype(ld), Dd.cpu().numpy().astype(ld), Doff.cpu().numpy().astype(ld)
    p = perm.cpu().numpy()
    W = Lh * d                                                # L D, D tridiagonal by 2x2 blocks
    W[:, :-1] += Lh[:, 1:] * o[:-1]
    W[:, 1:] += Lh[:, :-1] * o[:-1]
    R = np.abs(K.astype(ld)[np.ix_(p, p)] - W @ Lh.T)
    b = (np.abs(Lh) * np.abs(W)).sum(axis=1)                  # sum_j |l_ij| |w_ij|
    return R, b, tuple(inr.cpu().numpy()), m.mdsip_ldlt_panel_counts(ctx), d


def _convex(rng, N):
    g = rng.standard_normal((N, N)) / np.sqrt(N)
    return g @ g.T + np.diag(rng.uniform(1.0, 3.0, N))


@pytest.mark.parametrize("N", [16, 48, 161])
@pytest.mark.parametrize("e", [-890, -700, -540, -520, 520, 900])
def test_scaled_matrix(ctx, N, e):
    """A power of two on the whole matrix changes no bit of L and only the exponents of D."""
    K = _convex(np.random.default_rng(N), N)
    R, b, inertia, counts, d = _factor(ctx, K * 2.0 ** e, 1e-14)
    assert inertia == (N, 0, 0)
    assert counts == ((N + 63) // 64, 0)                      # the no-interchange form holds this range
    # as at scale 1: 2 N 2^-52 sqrt(b_i b_j)
    tol = 2 * N * np.longdouble(2.0) ** -52 * np.sqrt(np.outer(b, b))
    assert (R <= tol).all(), float((R / tol).max())
    np.testing.assert_array_equal((d * np.longdouble(2.0) ** -e), _factor(ctx, K, 1e-14)[4])


@pytest.mark.parametrize("n1,n2", [(8, 8), (16, 16), (20, 45), (33, 64)])
@pytest.mark.parametrize("e", [-560, -800])
def test_blocks_of_different_scales(ctx, n1, n2, e):
    """A block at scale 1 beside one at 2^e: no threshold on max|S| can tell."""
    rng = np.random.default_rng(n1 + n2)
    N = n1 + n2
    K = np.zeros((N, N))
    K[:n1, :n1] = _convex(rng, n1)
    K[n1:, n1:] = _convex(rng, n2) * 2.0 ** e
    R, b, inertia, _, _ = _factor(ctx, K, 0.0)
    assert inertia == (N, 0, 0)
    tol = 2 * N * np.longdouble(2.0) ** -52 * np.sqrt(np.outer(b, b))
    assert (R <= tol).all(), float((R / np.where(tol > 0, tol, 1)).max())


@pytest.mark.parametrize("i,j", [(3, 9), (31, 40), (5, 70)])
def test_pivots_below_the_integer_form(ctx, i, j):
    """Without a zero tolerance a pivot below 2^-1000 is a pivot like any other:
    its column's update counts although |d|^-1/2 is outside the integer form."""
    N = 96
    K = np.eye(N)
    t = 2.0 ** -1010
    K[i, i], K[j, j] = 4 * t, 3 * t
    K[i, j] = K[j, i] = 2 * t                                 # d_j = 3 t - (2 t)^2 / 4 t = 2 t
    R, _, inertia, _, d = _factor(ctx, K, 0.0)
    assert inertia == (N, 0, 0)
    assert not R.any()                                        # powers of two: exact
    want = np.ones(N)
    want[i], want[j] = 4 * t, 2 * t
    np.testing.assert_array_equal(np.sort(d.astype(float)), np.sort(want))


@pytest.mark.parametrize("N", [40, 100, 300, 1000])
def test_fp32_updates_keep_the_matrix_in_fp64(ctx, N):
    """Below order 2048, without MDSIP_LDLT_PERSISTENT, FP32 enters through the
    updates only: the first column of L, which takes none, is an FP64 quotient."""
    torch = torch_cuda()
    K = _convex(np.random.default_rng(N), N)
    S = dev(np.tril(K).T.copy())
    L = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    Dd, Doff = (torch.zeros(N, dtype=torch.float64, device="cuda") for _ in range(2))
    perm, kind = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    inr = torch.zeros(3, dtype=torch.int32, device="cuda")
    m.mdsip_ldlt_factor_ex(ctx, N, S, N, 1e-14, m.MDSIP_LDLT_FP32_UPDATES, L, Dd, Doff, perm, kind, inr)
    torch.cuda.synchronize()
    assert tuple(inr.cpu().numpy()) == (N, 0, 0)
    d0, col = float(Dd[0]), L[0].cpu().numpy()
    assert d0 == K[0, 0]
    # a reciprocal and a product: two roundings
    np.testing.assert_allclose(col[1:], K[1:, 0] / K[0, 0], rtol=2.0 ** -51, atol=0)
