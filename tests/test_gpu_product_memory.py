"""Memory of the FP64 condensation product: a solve holds its workspace only
while it runs, and where the memory for the large form is not to be had it
takes smaller ones, with the same solution."""
import numpy as np
import pytest

import paper_2605_13736_gb300 as m
import synth
from gpu_util import dev, torch_cuda

pytestmark = pytest.mark.gpu
MB = 1 << 20


class _Limited:
    """Hooks over torch's caching allocator; allocations above `limit` bytes fail."""

    def __init__(self):
        self.torch = torch_cuda()
        self.limit = None
        self.live, self.sizes, self.refused = {}, [], 0
        self.hooks = m.mdsip_alloc_hooks(m.ALLOC_FN(self.alloc), m.FREE_FN(self.free), None)

    def alloc(self, nbytes, stream, user):
        if self.limit is not None and nbytes > self.limit:
            self.refused += 1
            return None
        p = self.torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))
        self.live[p] = int(nbytes)
        self.sizes.append(int(nbytes))
        return p

    def free(self, ptr, nbytes, stream, user):
        assert self.live.pop(ptr) == int(nbytes)
        self.torch.cuda.caching_allocator_delete(int(ptr))


def _solve(limit, allocator=None):
    """One FP64 solve with allocations above `limit` refused from its first on."""
    torch = torch_cuda()
    m.build()
    rec = _Limited()
    ctx = m.mdsip_ctx_create(0, torch.cuda.current_stream().cuda_stream, allocator=allocator or rec.hooks)
    try:
        prob = m.mdsip_problem_create_synthetic(ctx, **m.synth_arrays(synth.make_instance(
            n_d=200, m_E=10000, m_I=8, sigma_a=0.01, seed=3)))
        try:
            made = len(rec.sizes)
            rec.limit = limit
            st = m.mdsip_solve(prob, ctx)
            held = sorted(rec.live.values())
            x = torch.zeros(m.mdsip_packed_size(prob), dtype=torch.float64, device="cuda")
            m.mdsip_get_iterate(prob, x, m.MDSIP_MEM_DEVICE, ctx)
            return m.STATUS[st], m.mdsip_get_stats(prob)["iters"], x.cpu().numpy(), rec.sizes[made:], held, rec.refused
        finally:
            m.mdsip_problem_destroy(prob)
    finally:
        m.mdsip_ctx_destroy(ctx)
        assert not rec.live


def test_a_solve_gives_its_product_workspace_back():
    st, _, _, sizes, held, _ = _solve(None)
    assert st == "OK"
    assert max(sizes) > 32 * MB                 # the residues of 10000 x 200 at 28 bytes an entry
    assert max(held) <= 16 * MB                 # A: 10000 x 200 doubles


# 32 MB of residues at a time; none (the FP64 pipe, whose split sums
# take 17 MB at most, or none at all)
@pytest.mark.parametrize("limit", [50, 24, 4])
def test_less_memory_takes_smaller_forms(limit):
    ref = _solve(None)
    got = _solve(limit * MB)
    assert got[5] > 0 and max(got[3]) <= limit * MB
    assert got[:2] == ref[:2]
    # the product's roundings differ; both solutions have KKT errors of at most 1e-8
    assert np.linalg.norm(got[2] - ref[2]) <= 1e-6 * np.linalg.norm(ref[2])


def test_without_hooks():
    ref = _solve(None)
    got = _solve(None, allocator="cuda")
    assert got[:2] == ref[:2]
    np.testing.assert_array_equal(got[2], ref[2])


@pytest.mark.parametrize("limit", [60, 12, 1])
def test_product_entry_with_less_memory(limit):
    torch = torch_cuda()
    m.build()
    rec = _Limited()
    ctx = m.mdsip_ctx_create(0, torch.cuda.current_stream().cuda_stream, allocator=rec.hooks)
    rec.limit = limit * MB
    try:
        mm, n = 40000, 150
        A = dev(np.random.default_rng(0).integers(-8, 9, (mm, n)).astype(float))
        C = dev(np.ones((n, n)))
        m.mdsip_syrk_scaled(ctx, mm, n, A, n, dev(np.full(mm, 0.25)), 1.0, C, n)
        torch.cuda.synchronize()
        want = 4 * (A.T @ A) + 1
        np.testing.assert_array_equal(torch.triu(C).cpu().numpy(), torch.triu(want).cpu().numpy())
        assert rec.refused > 0 and max(rec.sizes) <= rec.limit
    finally:
        m.mdsip_ctx_destroy(ctx)
    assert not rec.live
