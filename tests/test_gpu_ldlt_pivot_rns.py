"""Pivoting FP64 panels with tensor-core trailing updates: remainders of the
31-column panels and of the 128-row tiles, rows over many decades, scales near
both ends of the range (below 2^-900 the update runs term by term), against
the reconstruction P K P^T = L D L^T in extended precision."""
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


@pytest.mark.parametrize("N", [33, 62, 64, 65, 96, 159, 190, 289, 418])
@pytest.mark.parametrize("kind,scale", [("zero_diag", 1.0), ("saddle", 1.0), ("graded", 1.0), ("zero_diag", 2.0 ** -950),
                                        ("saddle", 2.0 ** 900)])
def test_reconstruction(ctx, N, kind, scale):
    torch = torch_cuda()
    rng = np.random.default_rng(N)
    K = rng.standard_normal((N, N))
    K = K + K.T
    if kind == "zero_diag":
        np.fill_diagonal(K, 0.0)
    elif kind == "saddle":
        k = N // 2
        K[k:, k:] = 0.0
    else:                                      # rows over ten decades, zero diagonal: pivots of all sizes
        np.fill_diagonal(K, 0.0)
        s = 10.0 ** np.linspace(5, -5, N)
        K = s[:, None] * K * s[None, :]
    K = K * scale
    S = dev(np.tril(K).T.copy())
    L = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    Dd, Doff = (torch.zeros(N, dtype=torch.float64, device="cuda") for _ in range(2))
    perm, kd = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    inr = torch.zeros(3, dtype=torch.int32, device="cuda")
    m.mdsip_ldlt_factor_ex(ctx, N, S, N, 0.0, 2, L, Dd, Doff, perm, kd, inr)   # 2: every panel pivots
    torch.cuda.synchronize()
    assert int(inr.sum()) == N
    Lh = np.tril(L.cpu().numpy().T).astype(np.longdouble)
    d, o = (t.cpu().numpy().astype(np.longdouble) for t in (Dd, Doff))
    p = perm.cpu().numpy()
    W = Lh * d                                 # L D, D tridiagonal by 2x2 blocks
    W[:, :-1] += Lh[:, 1:] * o[:-1]
    W[:, 1:] += Lh[:, :-1] * o[:-1]
    R = np.abs(K.astype(np.longdouble)[np.ix_(p, p)] - W @ Lh.T)
    # each panel rounds a row of L and of W to 4 2^-55 of its largest balanced entry,
    # 32 terms each way, on top of the FP64 roundings of the panels: with the
    # balanced magnitudes b_i = sum_t |l_it| |w_it| of a row, 2 N 2^-52 sqrt(b_i b_j)
    h = np.zeros(N, dtype=np.longdouble)
    for t in range(N):
        q = max(abs(d[t]), abs(o[t]), abs(o[t - 1]) if t else 0.0)
        h[t] = np.sqrt(q) if q > 0 else 1.0
    b = ((np.abs(Lh) * h) ** 2).sum(axis=1) + ((np.abs(W) / h) ** 2).sum(axis=1)
    tol = 2 * N * np.longdouble(2.0) ** -52 * np.sqrt(np.outer(b, b))
    assert (R <= tol).all(), float((R / tol).max())


@pytest.mark.parametrize("N,spots", [(300, (70,)), (705, (333,)), (1036, (500,)), (1036, (100, 431, 800)), (417, (64, 380))])
def test_persistent_form_resumes_after_an_interchange(ctx, N, spots):
    """A convex matrix with a few zero diagonals that only an interchange (a 2x2
    pivot) gets past: the persistent kernel goes on behind each pivoting panel,
    from whatever column that ends at."""
    torch = torch_cuda()
    rng = np.random.default_rng(N + len(spots))
    g = rng.standard_normal((N, N)) / np.sqrt(N)
    K = 0.1 * (g + g.T) / np.sqrt(N) + np.diag(rng.uniform(1.0, 2.0, N))
    for j in spots:                            # [[0, 3], [3, 0]] coupled weakly to the rest
        K[j, j] = K[j + 5, j + 5] = 0.0
        K[j, j + 5] = K[j + 5, j] = 3.0
    S = dev(np.tril(K).T.copy())
    L = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    Dd, Doff = (torch.zeros(N, dtype=torch.float64, device="cuda") for _ in range(2))
    perm, kd = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    inr = torch.zeros(3, dtype=torch.int32, device="cuda")
    m.mdsip_ldlt_factor(ctx, N, S, N, 1e-14, L, Dd, Doff, perm, kd, inr)
    torch.cuda.synchronize()
    assert tuple(inr.cpu().numpy()) == (N - len(spots), len(spots), 0)
    assert int((kd == 2).sum()) == len(spots)
    # all but two panels of 64 columns per interchange stay with the persistent kernel
    assert m.mdsip_ldlt_panel_counts(ctx)[0] >= N // 64 - 2 * len(spots) - 1
    Lh = np.tril(L.cpu().numpy().T)
    d, o = Dd.cpu().numpy(), Doff.cpu().numpy()
    p = perm.cpu().numpy()
    R = K[np.ix_(p, p)] - Lh @ (np.diag(d) + np.diag(o[:-1], -1) + np.diag(o[:-1], 1)) @ Lh.T
    assert np.abs(R).max() <= 1e-13 * N        # N 2^-53 times entries of at most 3 and a few roundings each
