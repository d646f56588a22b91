"""Small FP64 factorizations through the default entry, across its rules: the
first column's test (orders up to 128), pivoting panels that follow without a
read-back (up to 96) and the resumed form above, for matrices that pivot at
once, half way and never; against the reconstruction."""
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


def _matrix(kind, N):
    rng = np.random.default_rng(N)
    g = rng.standard_normal((N, N)) / np.sqrt(N)
    if kind == "zero_diag":
        K = g + g.T
        np.fill_diagonal(K, 0.0)
        return K
    K = 0.1 * (g + g.T) / np.sqrt(N) + np.diag(rng.uniform(1.0, 2.0, N))
    if kind == "half_way" and N >= 2:
        j = (N - 1) // 2
        K[j, j] = K[j + 1, j + 1] = 0.0
        K[j, j + 1] = K[j + 1, j] = 3.0
    return K


@pytest.mark.parametrize("kind", ["zero_diag", "half_way", "convex"])
@pytest.mark.parametrize("N", [1, 2, 3, 8, 16, 17, 31, 32, 33, 63, 64, 65, 95, 96, 97, 114, 128, 129, 160])
def test_reconstruction(ctx, kind, N):
    torch = torch_cuda()
    K = _matrix(kind, N)
    S = dev(np.tril(K).T.copy())
    L = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    Dd, Doff = (torch.zeros(N, dtype=torch.float64, device="cuda") for _ in range(2))
    perm, kd = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    inr = torch.zeros(3, dtype=torch.int32, device="cuda")
    m.mdsip_ldlt_factor(ctx, N, S, N, 1e-14, L, Dd, Doff, perm, kd, inr)
    torch.cuda.synchronize()
    w = np.linalg.eigvalsh(K)
    assert tuple(inr.cpu().numpy()) == (int((w > 1e-13).sum()), int((w < -1e-13).sum()), int((abs(w) <= 1e-13).sum()))
    Lh, d, o, p = np.tril(L.cpu().numpy().T), Dd.cpu().numpy(), Doff.cpu().numpy(), perm.cpu().numpy()
    W = Lh * d
    W[:, :-1] += Lh[:, 1:] * o[:-1]
    W[:, 1:] += Lh[:, :-1] * o[:-1]
    R = np.abs(K[np.ix_(p, p)] - W @ Lh.T)
    b = np.abs(W) @ np.abs(Lh).T                # sum_j |w_ij| |l_kj|
    assert (R <= 4 * (N + 4) * 2.0 ** -53 * np.maximum(b, b.T).max()).all()


@pytest.mark.parametrize("N,spots", [(20, ()), (20, (9,)), (80, (40,)), (300, (70,)), (1036, (100, 431, 800))])
def test_panels_handed_over_are_counted(ctx, N, spots):
    """mdsip_ldlt_panel_counts: one hand-over per interchange that stands alone, none without."""
    torch = torch_cuda()
    K = _matrix("convex", N)
    for j in spots:                             # [[0, 3], [3, 0]], which only a 2x2 pivot gets past
        K[j, j] = K[j + 1, j + 1] = 0.0
        K[j, j + 1] = K[j + 1, j] = 3.0
    S = dev(np.tril(K).T.copy())
    L = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    Dd, Doff = (torch.zeros(N, dtype=torch.float64, device="cuda") for _ in range(2))
    perm, kd = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    inr = torch.zeros(3, dtype=torch.int32, device="cuda")
    m.mdsip_ldlt_factor(ctx, N, S, N, 1e-14, L, Dd, Doff, perm, kd, inr)
    torch.cuda.synchronize()
    assert int((kd == 2).sum()) == len(spots)
    assert m.mdsip_ldlt_panel_counts(ctx)[1] == len(spots)
    m.mdsip_ldlt_factor(ctx, N, dev(np.tril(K * 2.0 ** -950).T.copy()), N, 1e-14, L, Dd, Doff, perm, kd, inr)
    torch.cuda.synchronize()
    assert m.mdsip_ldlt_panel_counts(ctx) == (0, 1)   # below the persistent kernel's range: handed over whole


def test_pivots_round_a_few_times(ctx):
    """An element of the persistent kernel's panel rounds at its own magnitude once
    after the first sixteen columns, once when its four columns are due and up to
    three times within them, not once per column: the diagonal of the
    reconstruction, with the product by l of the stored row once more."""
    torch = torch_cuda()
    N, worst = 32, []
    for seed in range(40):
        rng = np.random.default_rng(seed)
        g = rng.standard_normal((N, N)) / np.sqrt(N)
        K = g @ g.T + np.diag(rng.uniform(1.0, 3.0, N))
        S = dev(np.tril(K).T.copy())
        L = torch.zeros((N, N), dtype=torch.float64, device="cuda")
        Dd, Doff = (torch.zeros(N, dtype=torch.float64, device="cuda") for _ in range(2))
        perm, kd = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
        inr = torch.zeros(3, dtype=torch.int32, device="cuda")
        m.mdsip_ldlt_factor(ctx, N, S, N, 1e-14, L, Dd, Doff, perm, kd, inr)
        torch.cuda.synchronize()
        assert m.mdsip_ldlt_panel_counts(ctx) == (1, 0)
        Lh, d = np.tril(L.cpu().numpy().T).astype(np.longdouble), Dd.cpu().numpy().astype(np.longdouble)
        diag = ((Lh * d) * Lh).sum(axis=1)
        worst.append(((diag - np.diag(K)) / np.diag(K))[16:])
    rms = float(np.sqrt((np.array(worst) ** 2).mean()))
    # a rounding is 2^-52 sqrt(1 / 24) rms relative to a value of random mantissa; six of them 1.11e-16
    assert rms <= np.sqrt(6 / 24) * 2.0 ** -52, rms
