"""The warm-start network's fused output layer and training step, and the GEMM's
column-tile form with several row chunks, at the edges of their tiles."""
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


# 131 hidden units: rows of W3 that are not whole 16-byte units, the update without TMA
@pytest.mark.parametrize("batch,nh", [(1, 136), (17, 136), (129, 136), (257, 136), (600, 136), (129, 131)])
def test_out_layer_ragged_batches(ctx, batch, nh):
    """The fused output layer (scaling, loss, targets by index) and the training
    step's fused Adam at batches around the 16-row, 128-row and 256-row edges
    of its tiles: the loss and the updated output weights from the kernel's own
    prediction and gradient."""
    torch = torch_cuda()
    rng = np.random.default_rng(batch)
    n_in, n_out = 5, 391
    mlp = m.mdsip_mlp_create(ctx, n_in, nh, n_out)
    try:
        off = m.mdsip_mlp_param_offsets(mlp)
        nP = m.mdsip_mlp_num_params(mlp)
        p0 = (rng.standard_normal(nP) * 0.1).astype(np.float32)
        m.mdsip_mlp_set_params(mlp, p0, ctx=ctx)
        mean = rng.standard_normal(n_out).astype(np.float32)
        sd = (10.0 ** rng.uniform(-3, 2, n_out)).astype(np.float32)
        m.mdsip_mlp_set_scaling(mlp, out_mean=mean, out_std=sd, ctx=ctx)
        X = rng.standard_normal((batch + 3, n_in))
        Y = rng.standard_normal((batch + 3, n_out)) * sd + mean
        Y[0, :40] = 0.0
        Y[1, :40] = 10.0 ** rng.uniform(-40, -20, 40)      # parts below the FP32 range
        Y[2, :40] = mean[:40]
        idx = rng.permutation(batch + 3)[:batch].astype(np.int32)
        Xd, Yd, idxd = dev(X), dev(Y), dev(idx)
        pred = torch.zeros((batch + 3, n_out), dtype=torch.float32, device="cuda")
        m.mdsip_mlp_forward(mlp, Xd, n_in, batch + 3, pred, n_out, ctx=ctx)
        yn = (pred.cpu().numpy().astype(float)[idx] - mean) / sd
        tn = (Y[idx] - mean) / sd
        grad = torch.zeros(nP, dtype=torch.float32, device="cuda")
        loss = m.mdsip_mlp_gradient(mlp, Xd, n_in, Yd, n_out, idxd, batch, grad, ctx=ctx)
        want = np.mean((yn - tn) ** 2)
        # yn is recovered from the FP32 prediction (rounded at |mean| / std), tn is rounded to FP32
        tol = 2.0 ** -22 * np.mean(np.abs(yn - tn) * (np.abs(yn) + np.abs(tn) + np.abs(mean / sd) + 1))
        assert abs(loss - want) <= 2 * tol + 1e-7 * want
        g = grad.cpu().numpy()
        # db3 = column sums of the BF16-rounded dL/dyn: 2^-9 per term, FP32 sums below that
        dy = 2.0 * (yn - tn) / (batch * n_out)
        np.testing.assert_allclose(g[off[5]:off[5] + n_out], dy.sum(0), rtol=0,
                                   atol=float((2.0 ** -8 * np.abs(dy)).sum(0).max()
                                              + 2.0 ** -20 * np.abs(mean / sd).max() / n_out))
        l2 = m.mdsip_mlp_train_step(mlp, Xd, n_in, Yd, n_out, idxd, batch, 1e-2, ctx=ctx)
        assert l2 == loss
        p1 = np.zeros(nP, np.float32)
        m.mdsip_mlp_get_params(mlp, p1, ctx=ctx)
        step = 1e-2 * g / (np.abs(g) + 1e-8)               # first Adam step from zero moments
        # FP32 roundings of the moments, the corrections, the quotient and the weight
        tolw = 2.0 ** -23 * np.abs(p0) + 1e-2 * (2.0 ** -19)
        for a, b in ((off[4], n_out * nh), (off[5], n_out), (off[0], nh * n_in), (off[2], nh * nh)):
            s_ = slice(a, a + b)
            assert np.all(np.abs(p1[s_] - (p0[s_] - step[s_])) <= tolw[s_])
    finally:
        m.mdsip_mlp_destroy(mlp)


def test_gemm_wide_more_than_one_row_chunk(ctx):
    """The column-tile GEMM with several 256-row chunks of A, ragged."""
    torch = torch_cuda()
    M, N, K = 515, 128 * 152 + 40, 72
    g = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    B = torch.randn(N, K, generator=g, device="cuda").to(torch.bfloat16)
    C = torch.zeros(M, N, device="cuda")
    m.mdsip_gemm_bf16(ctx, M, N, K, A, K, B, K, C, N)
    want = A.double() @ B.double().T
    bound = K * 2.0 ** -23 * (A.double().abs() @ B.double().abs().T)
    assert bool(((C.double() - want).abs() <= bound).all())
