"""What mdsip_syrk_scaled, which returns before its kernels have run, reports of
a device wait that expires in them: NaN in C, DEVICE from the next call, once."""
import numpy as np
import pytest

import paper_2605_13736_gb300 as m
from gpu_util import dev, make_ctx, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mm,n", [(1000, 130), (40000, 70)])
def test_expired_wait_is_reported(mm, n):
    torch = torch_cuda()
    ctx = make_ctx()
    try:
        A = dev(np.random.default_rng(0).integers(-4, 5, (mm, n)).astype(float))
        w = dev(np.ones(mm))
        C = dev(np.zeros((n, n)))
        m.mdsip_debug_expire_wait(ctx)
        m.mdsip_syrk_scaled(ctx, mm, n, A, n, w, 0.0, C, n)
        torch.cuda.synchronize()
        low = torch.tril(torch.ones(n, n, dtype=torch.bool, device="cuda")).T
        assert bool(torch.isnan(C[low]).all())
        with pytest.raises(m.MdsipError) as ei:
            m.mdsip_syrk_scaled(ctx, mm, n, A, n, w, 0.0, C, n)
        assert ei.value.status == 11                       # MDSIP_ERR_DEVICE
        assert "mdsip_syrk_scaled" in m.mdsip_ctx_last_error(ctx)
        m.mdsip_syrk_scaled(ctx, mm, n, A, n, w, 0.0, C, n)   # reported once; the context goes on
        torch.cuda.synchronize()
        np.testing.assert_array_equal(C[low].cpu().numpy(), (A.T @ A)[low].cpu().numpy())
    finally:
        m.mdsip_ctx_destroy(ctx)
