"""The 256 x 256 form of the tensor-core product at the edges of its blocks:
widths just above its lower limit, with a last block of one, 128, 129 and 256
columns, and row counts of one slab to many splits.  Bound as for the narrow
form: the operand type's rounding (BF16 2^-8, TF32 2^-10 per product) relative
to sum_i |A_ip A_iq| / w_i."""
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


@pytest.mark.parametrize("prec", [m.MDSIP_PREC_BF16, m.MDSIP_PREC_TF32])
@pytest.mark.parametrize("mrows,n", [(1, 1025), (100, 1152), (2000, 1153), (5001, 1280), (9000, 2000), (70, 4095)])
def test_wide_product_matches_definition(ctx, prec, mrows, n):
    torch = torch_cuda()
    rng = np.random.default_rng(mrows + n + prec)
    A = rng.standard_normal((mrows, n)) * 0.1
    w = rng.uniform(0.05, 4.0, mrows)
    C0 = rng.standard_normal((n, n))
    want = A.T @ (A / w[:, None]) + C0
    scale = np.abs(A).T @ (np.abs(A) / w[:, None])
    Cd = dev(C0.T.copy())
    m.mdsip_syrk_scaled_tc(ctx, mrows, n, dev(A), n, dev(w), 1.0, Cd, n, prec)
    torch.cuda.synchronize()
    got = Cd.cpu().numpy().T
    low = np.tril_indices(n)
    rel = np.abs(got[low] - want[low]) / scale[low]
    assert rel.max() <= (2.0 ** -7 if prec == m.MDSIP_PREC_BF16 else 2.0 ** -9)
    up = np.triu_indices(n, 1)
    np.testing.assert_array_equal(got[up], C0[up])
