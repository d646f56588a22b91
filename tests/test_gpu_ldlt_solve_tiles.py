"""The solve's tile kernel at the edges of a diagonal block (64) and of a
warp's half of it (32): a given unit lower L with entries of size 1/sqrt(N), a
diagonal D and the identity permutation against forward and backward
substitution on the host.  Bound: gamma_3N = 4e-14 at N = 129 times the
condition of the two triangles (below 100 for such L) is under 1e-11."""
import numpy as np
import pytest
from scipy.linalg import solve_triangular

import paper_2605_13736_gb300 as m
from gpu_util import dev, make_ctx, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    m.mdsip_ctx_destroy(c)


@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 63, 64, 65, 95, 96, 97, 128, 129])
def test_solve_at_block_edges(ctx, N):
    torch = torch_cuda()
    rng = np.random.default_rng(N)
    L = np.tril(rng.uniform(-1, 1, (N, N)) / np.sqrt(N), -1) + np.eye(N)
    D = rng.uniform(1, 2, N) * rng.choice([-1.0, 1.0], N)
    b = rng.standard_normal(N)
    y = solve_triangular(L, b, lower=True, unit_diagonal=True)
    want = solve_triangular(L.T, y / D, lower=False, unit_diagonal=True)
    Ld, x = dev(L.T.copy()), dev(b)                       # column-major
    m.mdsip_ldlt_solve(ctx, N, Ld, dev(D), dev(np.zeros(N)), dev(np.arange(N, dtype=np.int32)), 1, x, N)
    torch.cuda.synchronize()
    assert np.abs(x.cpu().numpy() - want).max() <= 1e-11 * np.abs(want).max()


@pytest.mark.parametrize("N,nrhs", [(65, 7), (1033, 9), (700, 4)])
def test_solve_several_right_hand_sides(ctx, N, nrhs):
    """Columns solved side by side equal the same columns solved one at a time, bit for bit."""
    torch = torch_cuda()
    rng = np.random.default_rng(N)
    L = np.tril(rng.uniform(-1, 1, (N, N)) / np.sqrt(N), -1) + np.eye(N)
    D = rng.uniform(1, 2, N) * rng.choice([-1.0, 1.0], N)
    Ld, Dd, off = dev(L.T.copy()), dev(D), dev(np.zeros(N))
    perm = dev(np.arange(N, dtype=np.int32))
    b = rng.standard_normal((nrhs, N))
    X = dev(b)
    m.mdsip_ldlt_solve(ctx, N, Ld, Dd, off, perm, nrhs, X, N)
    for k in range(nrhs):
        x = dev(b[k])
        m.mdsip_ldlt_solve(ctx, N, Ld, Dd, off, perm, 1, x, N)
        torch.cuda.synchronize()
        assert torch.equal(x, X[k])
