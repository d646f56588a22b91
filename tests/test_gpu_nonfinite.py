"""Infinities and NaN that reach a direction: the mixed path (whose sweeps form
the refinement's sums in FP32 pairs) ends with a non-finite direction, as the
FP64 path does, and neither hangs nor reports a device error."""
import math

import numpy as np
import pytest

import paper_2605_13736_gb300 as m
import synth
from gpu_util import make_ctx, make_problem, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [m.MDSIP_PREC_FP64, m.MDSIP_PREC_TF32, m.MDSIP_PREC_BF16])
@pytest.mark.parametrize("n_d", [40, 300])          # four and eight columns a thread of the sweep
@pytest.mark.parametrize("what", ["zl_nan", "yg_inf", "x_huge", "x_on_bound"])
def test_direction_from_nonfinite_data(precision, n_d, what):
    torch = torch_cuda()
    ctx = make_ctx()
    inst = synth.make_instance(n_d=n_d, m_E=10 * n_d, m_I=4, sigma_a=0.01, seed=5)
    it = synth.random_iterate(inst, 5)
    prob = make_problem(ctx, inst)
    try:
        m.mdsip_set_option_int(prob, "precision", precision, ctx)
        p = np.concatenate([it["x"], it["d"], it["yg"], it["yh"], it["zl"], it["zu"], it["vl"], it["vu"]])
        n, mE, mI = len(it["x"]), len(it["yg"]), len(it["d"])
        if what == "zl_nan":
            p[n + mI + mE + mI + 5] = math.nan
        elif what == "yg_inf":
            p[n + mI + 7] = math.inf
        elif what == "x_huge":
            p[3] = 1e120
        else:
            p[3] = float(inst.xu[3])
        out = torch.zeros(len(p), dtype=torch.float64, device="cuda")
        m.mdsip_debug_direction(prob, torch.as_tensor(p).cuda(), 0.05, 0.0, 0.0, out, mem=m.MDSIP_MEM_DEVICE, ctx=ctx)
        assert int((~torch.isfinite(out)).sum()) > 0
    finally:
        m.mdsip_problem_destroy(prob)
        m.mdsip_ctx_destroy(ctx)
