"""Edges of the step's vector kernels: A^T u with one, two or four columns per
thread and with several rows of a block per column, J_dh^T y by groups of 32
columns, and the reductions' grids from a single block up, each through a
direction from the same iterate as the oracle's two-stage solve (1e-10
relative, the bound of the other direction tests) with equal inertia."""
import numpy as np
import pytest

import paper_2605_13736_gb300 as m
import synth
from oracle import ipm
from oracle.model import SynthModel
from gpu_util import make_ctx, make_problem, pack_dir

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    m.mdsip_ctx_destroy(c)


@pytest.mark.parametrize("n_d,m_E,m_I", [(1, 1, 1), (31, 65, 9), (33, 127, 3), (256, 129, 17), (257, 305, 8),
                                         (512, 77, 1), (513, 2433, 33), (1030, 40, 40)])
def test_direction_at_kernel_edges(ctx, n_d, m_E, m_I):
    inst = synth.make_instance(n_d, m_E, m_I, 0.05, seed=n_d + m_E)
    model = SynthModel(inst)
    it = synth.random_iterate(inst, n_d + 7)
    pt = ipm.Point(it["x"], it["d"], it["yg"], it["yh"], it["zl"], it["zu"], it["vl"], it["vu"])
    want = ipm.direction_at(model, pt, 0.05, 1e-4, 0.0, "p2")
    prob = make_problem(ctx, inst, m.MDSIP_PATH_P2)
    try:
        out = np.zeros(m.mdsip_packed_size(prob))
        inertia = m.mdsip_debug_direction(prob, pt.packed(), 0.05, 1e-4, 0.0, out, ctx=ctx)
    finally:
        m.mdsip_problem_destroy(prob)
    assert inertia == tuple(want["inertia"])
    ref = pack_dir(want)
    assert np.linalg.norm(out - ref) <= 1e-10 * np.linalg.norm(ref)
