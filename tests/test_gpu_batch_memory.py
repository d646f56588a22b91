"""A batch starts its worker threads anew on every call: none of them may leave
host memory behind."""
import pytest

import paper_2605_13736_gb300 as m
import synth
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def _rss_kb():
    with open("/proc/self/status") as fh:
        return int(next(line for line in fh if line.startswith("VmRSS")).split()[1])


def test_batches_leave_no_host_memory():
    torch = torch_cuda()
    m.build()
    streams = [torch.cuda.Stream() for _ in range(32)]
    ctxs = [m.mdsip_ctx_create(0, s.cuda_stream) for s in streams]
    probs = [m.mdsip_problem_create_synthetic(c, **m.synth_arrays(synth.make_instance(
        n_d=8, m_E=20, m_I=1, sigma_a=0.1, seed=i))) for i, c in enumerate(ctxs)]
    try:
        for p, c in zip(probs, ctxs):
            m.mdsip_set_option_int(p, "max_iter", 1, c)
        for _ in range(5):
            m.mdsip_batch_solve(probs)
        before = _rss_kb()
        for _ in range(200):                     # 6400 worker threads
            m.mdsip_batch_solve(probs)
        assert _rss_kb() - before < 4096         # 12 MB with two pinned words lost a thread
    finally:
        for p in probs:
            m.mdsip_problem_destroy(p)
        for c in ctxs:
            m.mdsip_ctx_destroy(c)
