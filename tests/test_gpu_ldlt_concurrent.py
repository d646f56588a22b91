"""Several FP64 factorizations at once, one context, stream and thread each, of
uneven orders that pivot at once, half way and never: the bits of the same
factorizations one after the other."""
import threading

import numpy as np
import pytest

import paper_2605_13736_gb300 as m
from gpu_util import dev, torch_cuda

pytestmark = pytest.mark.gpu

JOBS = [(33, "never"), (64, "once"), (97, "half"), (161, "never"), (300, "half"), (417, "once"), (705, "half"),
        (1036, "never"), (128, "once"), (350, "never")]


def _matrix(N, kind):
    rng = np.random.default_rng(N)
    g = rng.standard_normal((N, N)) / np.sqrt(N)
    if kind == "once":
        K = g + g.T
        np.fill_diagonal(K, 0.0)
        return K
    K = 0.1 * (g + g.T) / np.sqrt(N) + np.diag(rng.uniform(1.0, 2.0, N))
    if kind == "half":
        j = N // 2
        K[j, j] = K[j + 3, j + 3] = 0.0
        K[j, j + 3] = K[j + 3, j] = 3.0
    return K


class _Job:
    def __init__(self, torch, N, kind):
        self.N = N
        self.stream = torch.cuda.Stream()
        self.ctx = m.mdsip_ctx_create(0, self.stream.cuda_stream)
        self.S0 = dev(np.tril(_matrix(N, kind)).T.copy())
        self.S = torch.empty_like(self.S0)
        self.out = [torch.zeros(N, N, dtype=torch.float64, device="cuda")]
        self.out += [torch.zeros(N, dtype=torch.float64, device="cuda") for _ in range(2)]
        self.out += [torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2)]
        self.out += [torch.zeros(3, dtype=torch.int32, device="cuda")]
        self.error = None

    def run(self, torch, reps):
        try:
            with torch.cuda.stream(self.stream):
                for _ in range(reps):
                    self.S.copy_(self.S0)
                    m.mdsip_ldlt_factor(self.ctx, self.N, self.S, self.N, 1e-14, *self.out)
        except Exception as e:      # reported by the test's thread
            self.error = e

    def result(self):
        return [t.cpu().numpy().copy() for t in self.out]


def test_factorizations_at_once():
    torch = torch_cuda()
    m.build()
    jobs = [_Job(torch, N, kind) for N, kind in JOBS]
    try:
        torch.cuda.synchronize()
        want = []
        for j in jobs:
            j.run(torch, 1)
            torch.cuda.synchronize()
            want.append(j.result())
            for t in j.out:
                t.zero_()
        torch.cuda.synchronize()
        threads = [threading.Thread(target=j.run, args=(torch, 6)) for j in jobs]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        for j, w, (N, kind) in zip(jobs, want, JOBS):
            assert j.error is None, (N, kind, j.error)
            for a, b in zip(j.result(), w):
                np.testing.assert_array_equal(a, b, err_msg=f"{N} {kind}")
    finally:
        for j in jobs:
            m.mdsip_ctx_destroy(j.ctx)
