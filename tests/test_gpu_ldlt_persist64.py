"""The persistent FP64 LDL^T (exact integer trailing updates on the tensor
cores) at the edges of its panels and tiles and on matrices whose rows span
many orders of magnitude: entry-wise reconstruction."""
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


# one panel (16- and 32-column sub-panels), one trailing tile and its edges,
# several 128-row tiles, a single column left over
@pytest.mark.parametrize("N", [15, 17, 32, 33, 48, 63, 161, 289, 417, 705])
@pytest.mark.parametrize("decades", [0, 10])
def test_reconstruction_entrywise(ctx, N, decades):
    torch = torch_cuda()
    rng = np.random.default_rng(N + decades)
    mi = N // 4
    nd = N - mi
    g = rng.standard_normal((nd, nd)) / np.sqrt(nd)
    K = np.zeros((N, N))
    K[:nd, :nd] = g @ g.T + np.diag(rng.uniform(1.0, 3.0, nd))
    K[nd:, :nd] = 0.1 * rng.standard_normal((mi, nd))
    K[:nd, nd:] = K[nd:, :nd].T
    K[nd:, nd:] = -np.diag(rng.uniform(0.5, 2.0, mi))
    s = 10.0 ** np.linspace(decades / 2, -decades / 2, N)     # descending: every diagonal pivot is kept
    K = s[:, None] * K * s[None, :]
    S = dev(np.tril(K).T.copy())                              # column-major lower triangle
    L = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    Dd, Doff = (torch.zeros(N, dtype=torch.float64, device="cuda") for _ in range(2))
    perm, kind = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
    inr = torch.zeros(3, dtype=torch.int32, device="cuda")
    m.mdsip_ldlt_factor(ctx, N, S, N, 1e-30, L, Dd, Doff, perm, kind, inr)
    torch.cuda.synchronize()
    assert m.mdsip_ldlt_panel_counts(ctx) == ((N + 63) // 64, 0)
    assert tuple(inr.cpu().numpy()) == (nd, mi, 0)
    np.testing.assert_array_equal(perm.cpu().numpy(), np.arange(N))
    np.testing.assert_array_equal(kind.cpu().numpy(), np.ones(N))
    assert not Doff.cpu().numpy().any()
    Lh, d = np.tril(L.cpu().numpy().T).astype(np.longdouble), Dd.cpu().numpy().astype(np.longdouble)
    R = np.abs(np.tril(K) - np.tril((Lh * d) @ Lh.T))
    b = (np.abs(Lh) ** 2 * np.abs(d)).sum(axis=1)             # sum_j l_ij^2 |d_j|
    # per panel each factor is rounded to at most 4 max 2^-55 of its row, 32
    # terms each way, plus the FP64 roundings of the chain and of the updates
    tol = 2 * N * 2.0 ** -52 * np.sqrt(np.outer(b, b))
    assert (R <= tol).all(), (R / tol).max()
