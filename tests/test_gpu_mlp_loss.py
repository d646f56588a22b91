"""The training loss as an FP64 sum: with a network whose output is zero it is
the mean square of the standardised targets, here FP32 numbers, so only the
summation rounds."""
import numpy as np
import pytest

import paper_2605_13736_gb300 as m
from gpu_util import make_ctx, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,n_out,seed", [(256, 180937, 0), (256, 180937, 1), (256, 180937, 2), (200, 50003, 0), (1, 999, 0), (300, 130, 0)])
def test_loss_is_an_fp64_sum(batch, n_out, seed):
    torch = torch_cuda()
    ctx = make_ctx()
    mlp = m.mdsip_mlp_create(ctx, 8, 16, n_out)
    try:
        m.mdsip_mlp_set_params(mlp, torch.zeros(m.mdsip_mlp_num_params(mlp), device="cuda"), m.MDSIP_MEM_DEVICE, ctx)
        g = torch.Generator(device="cuda").manual_seed(seed)
        X = torch.zeros(batch, 8, dtype=torch.float64, device="cuda")
        Y = torch.randn(batch, n_out, generator=g, device="cuda").double()
        loss = m.mdsip_mlp_train_step(mlp, X, 8, Y, n_out, None, batch, 0.0, ctx=ctx)
        rows = (Y * Y).sum(dim=1).cpu().numpy().astype(np.longdouble)   # squares of FP32 numbers are exact in FP64
        want = rows.sum() / (batch * n_out)
        # sums of some hundred terms a level in FP64: a few 2^-53, here 2^-49
        assert abs(loss - want) <= 2.0 ** -49 * want, float((loss - want) / want)
    finally:
        m.mdsip_mlp_destroy(mlp)
        m.mdsip_ctx_destroy(ctx)


def test_a_step_on_overflowing_moments():
    """Gradients so large that the second moment overflows move nothing: m / inf."""
    torch = torch_cuda()
    ctx = make_ctx()
    mlp = m.mdsip_mlp_create(ctx, 8, 16, 200)
    try:
        n = m.mdsip_mlp_num_params(mlp)
        P = torch.zeros(n, device="cuda")
        m.mdsip_mlp_set_params(mlp, P, m.MDSIP_MEM_DEVICE, ctx)
        X = torch.zeros(4, 8, dtype=torch.float64, device="cuda")
        Y = torch.full((4, 200), 1e22, dtype=torch.float64, device="cuda")
        for _ in range(3):                      # db3 = -1e20: v = 1e37, v / (1 - beta2^t) = inf
            m.mdsip_mlp_train_step(mlp, X, 8, Y, 200, None, 4, 1e-3, ctx=ctx)
        m.mdsip_mlp_get_params(mlp, P, m.MDSIP_MEM_DEVICE, ctx)
        assert bool(torch.isfinite(P).all())
    finally:
        m.mdsip_mlp_destroy(mlp)
        m.mdsip_ctx_destroy(ctx)
