"""One-pass refinement sweeps at the edges of their row groups (widths 128, 256,
512, 1024, 2048, 4096 and one more), with batches that end ragged, CTAs of one
short batch and of more than 256 rows a thread: the refined direction against
the FP64 path's from the same iterate.  Each path is held to 1e-10 of the exact
direction by the oracle tests, so the two differ by at most 2e-10."""
import numpy as np
import pytest

import paper_2605_13736_gb300 as m
import synth
from gpu_util import make_ctx, make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    m.mdsip_ctx_destroy(c)


@pytest.mark.parametrize("prec", [m.MDSIP_PREC_BF16, m.MDSIP_PREC_TF32])
@pytest.mark.parametrize("n_d,m_E,m_I", [(1, 3, 1), (31, 64, 2), (128, 65, 3), (129, 2000, 9), (256, 4865, 1),
                                         (257, 17, 5), (513, 1001, 40), (1025, 39001, 2), (2048, 1217, 33),
                                         (2049, 39001, 3), (4096, 305, 7), (4097, 305, 7)])
def test_refined_direction_equals_fp64(ctx, n_d, m_E, m_I, prec):
    inst = synth.make_instance(n_d, m_E, m_I, 0.1 / np.sqrt(n_d), seed=n_d + 3)
    it = synth.random_iterate(inst, n_d)
    packed = np.concatenate([it[k] for k in ("x", "d", "yg", "yh", "zl", "zu", "vl", "vu")])
    prob = make_problem(ctx, inst, m.MDSIP_PATH_P2)
    try:
        want, out = (np.zeros(m.mdsip_packed_size(prob)) for _ in range(2))
        i64 = m.mdsip_debug_direction(prob, packed, 0.05, 1e-4, 1e-9, want, ctx=ctx)
        m.mdsip_set_option_int(prob, "precision", prec, ctx)
        itc = m.mdsip_debug_direction(prob, packed, 0.05, 1e-4, 1e-9, out, refine=40, ctx=ctx)
    finally:
        m.mdsip_problem_destroy(prob)
    assert i64 == itc
    assert np.linalg.norm(out - want) <= 2e-10 * np.linalg.norm(want)
