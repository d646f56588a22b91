"""A call that fails for want of memory leaves nothing half made: the next one,
with memory again, gives the result of an undisturbed run."""
import numpy as np
import pytest

import paper_2605_13736_gb300 as m
import synth
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


class _Failing:
    """Hooks over torch's caching allocator; the allocation numbered `at` from now on fails."""

    def __init__(self):
        self.torch = torch_cuda()
        self.at = None
        self.hooks = m.mdsip_alloc_hooks(m.ALLOC_FN(self.alloc), m.FREE_FN(self.free), None)

    def alloc(self, nbytes, stream, user):
        if self.at is not None:
            self.at -= 1
            if self.at < 0:
                return None
        return self.torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))

    def free(self, ptr, nbytes, stream, user):
        self.torch.cuda.caching_allocator_delete(int(ptr))


def _context():
    torch = torch_cuda()
    m.build()
    rec = _Failing()
    return rec, m.mdsip_ctx_create(0, torch.cuda.current_stream().cuda_stream, allocator=rec.hooks)


def _oom(rec, at, call):
    """Whether the call ran out of memory with its allocation `at` refused."""
    rec.at = at
    try:
        call()
        return False
    except m.MdsipError as e:
        assert e.status == 3, e                 # MDSIP_ERR_OOM
        return True
    finally:
        rec.at = None


def test_network_buffers():
    torch = torch_cuda()
    rec, ctx = _context()
    mlp = m.mdsip_mlp_create(ctx, 8, 32, 100)
    try:
        g = torch.Generator(device="cuda").manual_seed(0)
        n = m.mdsip_mlp_num_params(mlp)
        P = torch.randn(n, generator=g, device="cuda")
        X = torch.randn(500, 8, generator=g, device="cuda", dtype=torch.float64)
        Y = torch.randn(500, 100, generator=g, device="cuda", dtype=torch.float64)
        small = torch.zeros(40, 100, device="cuda")

        def forward(out, rows):
            m.mdsip_mlp_forward(mlp, X, 8, rows, out, 100, ctx=ctx)

        def gradient(rows):
            grad = torch.zeros(n, device="cuda")
            m.mdsip_mlp_gradient(mlp, X, 8, Y, 100, None, rows, grad, ctx=ctx)
            return grad.cpu().numpy()

        m.mdsip_mlp_set_params(mlp, P, m.MDSIP_MEM_DEVICE, ctx)
        forward(small, 40)
        want, want_g = small.cpu().numpy().copy(), gradient(40)
        large = torch.zeros(500, 100, device="cuda")
        at = 0
        while _oom(rec, at, lambda: forward(large, 500) or gradient(500)):
            small.zero_()
            forward(small, 40)
            np.testing.assert_array_equal(small.cpu().numpy(), want)
            np.testing.assert_array_equal(gradient(40), want_g)
            at += 1
            # a fresh network, so that the large call allocates again
            m.mdsip_mlp_destroy(mlp)
            mlp = m.mdsip_mlp_create(ctx, 8, 32, 100)
            m.mdsip_mlp_set_params(mlp, P, m.MDSIP_MEM_DEVICE, ctx)
            forward(small, 40)
            gradient(40)
        assert at >= 5
    finally:
        m.mdsip_mlp_destroy(mlp)
        m.mdsip_ctx_destroy(ctx)


@pytest.mark.parametrize("precision", [m.MDSIP_PREC_FP64, m.MDSIP_PREC_BF16])
def test_problem_buffers(precision):
    torch = torch_cuda()
    inst = synth.make_instance(n_d=60, m_E=3000, m_I=4, sigma_a=0.01, seed=9)
    want, at = None, -1
    while True:
        rec, ctx = _context()
        prob = m.mdsip_problem_create_synthetic(ctx, **m.synth_arrays(inst))
        try:
            m.mdsip_set_option_int(prob, "precision", precision, ctx)
            if precision != m.MDSIP_PREC_FP64:
                m.mdsip_set_option_int(prob, "direction_check", 1, ctx)
            out = torch.zeros(m.mdsip_packed_size(prob), dtype=torch.float64, device="cuda")
            failed = at >= 0 and _oom(rec, at, lambda: m.mdsip_solve(prob, ctx))
            assert m.STATUS[m.mdsip_solve(prob, ctx)] == "OK"
            m.mdsip_get_iterate(prob, out, m.MDSIP_MEM_DEVICE, ctx)
            got = out.cpu().numpy()
            if want is None:
                want = got
            np.testing.assert_array_equal(got, want)
            if at >= 0 and not failed:
                break
            at += 1
        finally:
            m.mdsip_problem_destroy(prob)
            m.mdsip_ctx_destroy(ctx)
    assert at >= 15
