"""The work that users of mdsip have it do, as measurable cases.

A case is a dict of plain values; its `kind` names the entry points it goes through:

  solve      mdsip_solve from the problem's x0 to E_0 <= tol, iterate read back
  batch      mdsip_batch_solve of uneven instances, one context and stream each
  direction  one Newton direction at a given iterate (mdsip_debug_direction)
  syrk       the FP64 condensation product on its own (mdsip_syrk_scaled)
  ldlt       Bunch-Kaufman factorization and solve (mdsip_ldlt_factor, mdsip_ldlt_solve)
  train      one Adam step of the warm-start network, parameters read back
  predict    warm-start predictions for a batch of family members

Instances follow the benchmark family of `synth` (n_s = 2 m_E, identity-pair
J_sg, dense A, quadratic inequalities on disjoint subsets of x_d), drawn on the
GPU from the case's seed.
"""
from __future__ import annotations

import math

import torch

import paper_2605_13736_gb300 as m

DEV = "cuda:0"
F64 = torch.float64
PREC = {"fp64": m.MDSIP_PREC_FP64, "tf32": m.MDSIP_PREC_TF32, "bf16": m.MDSIP_PREC_BF16}
MU = 0.05          # barrier parameter of the direction cases
LR = 1e-3          # learning rate of the training case
ADAM_EPS = 1e-8
N_P = 64           # parameters of the warm-start family
HIDDEN = 512


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest NLP of the benchmark, solved whole: launches, host round trips and small
        # factorizations are all there is
        dict(name="solve fp64 n32", kind="solve", n_d=32, m_E=1000, m_I=1, sigma_a=0.1, precision="fp64"),
        # one member of the warm-start family: what data generation and the judged solves run thousands of times
        dict(name="solve bf16 n512", kind="solve", n_d=512, m_E=25600, m_I=50, sigma_a=0.01, precision="bf16"),
        # a contingency screening step: many instances of uneven size at once
        dict(name="batch bf16 24 uneven", kind="batch", count=24, lo=64, hi=300, m_I=50, precision="bf16"),
        # inequalities with a sparse block: the one-stage path, whose matrix keeps all equality rows
        dict(name="direction p1 n32", kind="direction", n_d=32, m_E=1000, m_I=4, sigma_a=0.1, jsh=5, precision="fp64"),
        # a batch-sized instance in plain FP64, ragged sizes
        dict(name="direction fp64 n301", kind="direction", n_d=301, m_E=15053, m_I=50, sigma_a=0.01, jsh=0,
             precision="fp64"),
        # the headline: a plain FP64 Newton direction of the OPF-sized instance
        dict(name="direction fp64 n2000", kind="direction", n_d=2000, m_E=100000, m_I=50, sigma_a=0.01, jsh=0,
             precision="fp64"),
        # the same direction from the refined tensor-core path
        dict(name="direction bf16 n2000", kind="direction", n_d=2000, m_E=100000, m_I=50, sigma_a=0.01, jsh=0,
             precision="bf16"),
        # the mixed-precision scale of the benchmark, TF32 operands
        dict(name="direction tf32 n4000", kind="direction", n_d=4000, m_E=200000, m_I=50, sigma_a=0.01, jsh=0,
             precision="tf32"),
        # the condensation product called by itself, odd sizes (a leading dimension wider than the row)
        dict(name="syrk fp64 30011x771", kind="syrk", m=30011, n=771),
        # a dense indefinite matrix of the paper's order sweep (N = 2k + 3) that needs interchanges, four right-hand sides
        dict(name="ldlt kkt 2003", kind="ldlt", k=1000, matrix="kkt", nrhs=4),
        # training the warm-start network on a batch of members
        dict(name="train b256", kind="train", n_out=180937, batch=256),
        # starting points for all held-out members in one forward pass
        dict(name="predict b1024", kind="predict", n_out=180937, batch=1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "batch", "direction", "direction", "direction", "p1", "syrk", "ldlt", "train",
                       "predict"])
    if kind == "solve":
        prec = rng.choice(["fp64", "bf16", "tf32"])
        n_d = _log_int(rng, 32, 512)
        return dict(kind="solve", n_d=n_d, m_E=n_d * rng.randint(30, 50) + rng.randint(0, 7),
                    m_I=rng.choice([1, 8, min(50, n_d)]), sigma_a=0.01 if n_d > 48 else 0.1, precision=prec)
    if kind == "batch":
        lo = rng.randint(64, 128)
        return dict(kind="batch", count=rng.randint(8, 32), lo=lo, hi=lo + rng.randint(40, 200), m_I=50,
                    precision=rng.choice(["bf16", "tf32"]))
    if kind == "direction":
        prec = rng.choice(["fp64", "bf16", "tf32"])
        n_d = _log_int(rng, 64, 1900 if prec == "fp64" else 3900)
        return dict(kind="direction", n_d=n_d, m_E=n_d * rng.randint(35, 50) + rng.randint(0, 9),
                    m_I=rng.choice([1, 8, 50]), sigma_a=0.01, jsh=0, precision=prec)
    if kind == "p1":
        return dict(kind="direction", n_d=rng.randint(8, 64), m_E=_log_int(rng, 150, 1500), m_I=rng.randint(1, 8),
                    sigma_a=0.1, jsh=rng.randint(2, 9), precision="fp64")
    if kind == "syrk":
        n = _log_int(rng, 64, 1500)
        return dict(kind="syrk", m=n * rng.randint(20, 50) + rng.randint(0, 63), n=n)
    if kind == "ldlt":
        return dict(kind="ldlt", k=_log_int(rng, 50, 1300), matrix=rng.choice(["kkt", "ipm"]), nrhs=rng.randint(1, 4))
    n_out = 3 * (101 * rng.randint(100, 590)) + rng.randint(1, 800)
    if kind == "train":
        return dict(kind="train", n_out=n_out, batch=rng.choice([64, 128, 200, 256]))
    return dict(kind="predict", n_out=n_out, batch=_log_int(rng, 1, 1024))


# ---------------------------------------------------------------------------
# inputs (drawn on the GPU from the seed alone)
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rand(g, n, lo, hi):
    return torch.rand(n, generator=g, device=DEV, dtype=F64) * (hi - lo) + lo


def _instance(n_d, m_E, m_I, sigma_a, seed, jsh=0):
    """Arguments of mdsip_problem_create_synthetic for one benchmark-family instance (device tensors)."""
    g = _gen(seed)
    n_s = 2 * m_E
    n = n_s + n_d
    G = torch.randn(n_d, n_d, generator=g, device=DEV, dtype=F64)
    Q = G.T @ G / n_d
    Q = 0.5 * (Q + Q.T) + 0.1 * torch.eye(n_d, device=DEV, dtype=F64)
    c = _rand(g, n, -1.0, 1.0)
    A = torch.randn(m_E, n_d, generator=g, device=DEV, dtype=F64).mul_(sigma_a)
    gE = _rand(g, m_E, -0.5, 0.5)
    i = torch.arange(m_E, device=DEV, dtype=torch.int32)
    h_set = torch.full((n_d,), -1, device=DEV, dtype=torch.int32)
    if m_I == 1:
        h_set.zero_()
        hu = torch.full((1,), 4.0, device=DEV, dtype=F64)
    else:
        chunk = n_d // m_I
        perm = torch.randperm(n_d, generator=g, device=DEV)[:chunk * m_I]
        h_set[perm] = torch.arange(m_I, device=DEV, dtype=torch.int32).repeat_interleave(chunk)
        hu = torch.ones(m_I, device=DEV, dtype=F64)
    inf = math.inf
    one = torch.ones(n_s, device=DEV, dtype=F64)
    free = torch.full((n_d,), inf, device=DEV, dtype=F64)
    d = dict(n_d=n_d, n_s=n_s, m_E=m_E, m_I=m_I, Q=Q.contiguous(), c=c, A=A, gE=gE,
             Jsg_rows=torch.cat([i, i]), Jsg_cols=torch.cat([i, i + m_E]),
             Jsg_vals=torch.cat([torch.ones(m_E, device=DEV, dtype=F64), -torch.ones(m_E, device=DEV, dtype=F64)]),
             h_set=h_set, hl=torch.full((m_I,), -inf, device=DEV, dtype=F64), hu=hu,
             xl=torch.cat([-one, -free]), xu=torch.cat([one, free]), x0=torch.zeros(n, device=DEV, dtype=F64))
    if jsh:
        cols = torch.stack([torch.randperm(n_s, generator=g, device=DEV)[:jsh] for _ in range(m_I)])
        d.update(Jsh_rows=torch.arange(m_I, device=DEV, dtype=torch.int32).repeat_interleave(jsh),
                 Jsh_cols=cols.reshape(-1).to(torch.int32).contiguous(), Jsh_vals=_rand(g, m_I * jsh, -0.5, 0.5))
    return d


def _iterate(d, seed):
    """A strictly interior primal-dual point, as blocks of the packed layout."""
    g = _gen(seed * 7 + 3)
    n, m_E, m_I = d["n_s"] + d["n_d"], d["m_E"], d["m_I"]
    x = torch.cat([_rand(g, d["n_s"], -0.9, 0.9), _rand(g, d["n_d"], -0.3, 0.3)])
    bounded = torch.isfinite(d["xu"])
    zero = torch.zeros(n, device=DEV, dtype=F64)
    zl = torch.where(bounded, torch.exp(_rand(g, n, -1.0, 1.0)), zero)
    zu = torch.where(bounded, torch.exp(_rand(g, n, -1.0, 1.0)), zero)
    slack = torch.exp(_rand(g, m_I, -1.0, 0.0))
    return dict(x=x, d=d["hu"] - slack, yg=_rand(g, m_E, -1.0, 1.0), yh=_rand(g, m_I, 0.0, 1.0), zl=zl, zu=zu,
                vl=torch.zeros(m_I, device=DEV, dtype=F64), vu=torch.exp(_rand(g, m_I, -1.0, 1.0)))


PACKED = ("x", "d", "yg", "yh", "zl", "zu", "vl", "vu")


def _syrk_inputs(c, seed):
    g = _gen(seed)
    lda = c["n"] + c["n"] % 2
    A = torch.randn(c["m"], lda, generator=g, device=DEV, dtype=F64).mul_(0.01)
    w = torch.pow(10.0, _rand(g, c["m"], -4.0, 1.0))   # the spread of J Q_s^-1 J^T in mid-solve
    return A, lda, w


def _ldlt_inputs(c, seed):
    """[[H, J^T], [J, -R]] of order 2k + 3: `kkt` needs interchanges, `ipm` is the convex Newton-step shape."""
    g = _gen(seed)
    k, mm = c["k"], c["k"] + 3
    G = torch.randn(k, k, generator=g, device=DEV, dtype=F64)
    H = G @ G.T / k
    J = torch.randn(mm, k, generator=g, device=DEV, dtype=F64)
    if c["matrix"] == "ipm":
        H = H + torch.diag(_rand(g, k, 1.0, 3.0))
        J = 0.1 * J
        R = torch.diag(_rand(g, mm, 0.5, 2.0))
    else:
        H = H + 0.1 * torch.eye(k, device=DEV, dtype=F64)
        R = torch.eye(mm, device=DEV, dtype=F64)
    K = torch.cat([torch.cat([H, J.T], 1), torch.cat([J, -R], 1)])
    B = torch.randn(c["nrhs"], k + mm, generator=g, device=DEV, dtype=F64)   # right-hand sides by row
    return (0.5 * (K + K.T)).contiguous(), B


def _mlp_inputs(c, seed):
    """Network weights (He-uniform hidden layers, small output layer), members and targets around a common point."""
    g = _gen(seed)
    n_out, B = c["n_out"], c["batch"]
    u = lambda r, k, s: ((torch.rand(r, k, generator=g, device=DEV) * 2 - 1) * s)
    P = dict(W1=u(HIDDEN, N_P, math.sqrt(6 / N_P)), b1=torch.zeros(HIDDEN, device=DEV),
             W2=u(HIDDEN, HIDDEN, math.sqrt(6 / HIDDEN)), b2=torch.zeros(HIDDEN, device=DEV),
             W3=u(n_out, HIDDEN, 0.1 * math.sqrt(3 / HIDDEN)), b3=torch.zeros(n_out, device=DEV))
    rows = 2 * B if c["kind"] == "train" else B
    X = _rand(g, (rows, N_P), -1.0, 1.0)
    mean, sd = _rand(g, n_out, -1.0, 1.0).float(), torch.exp(_rand(g, n_out, -3.0, 0.0)).float()
    Y = idx = None
    if c["kind"] == "train":
        Y = torch.randn(rows, n_out, generator=g, device=DEV, dtype=F64).mul_(sd).add_(mean)
        idx = torch.randperm(rows, generator=g, device=DEV)[:B].to(torch.int32)
    return P, X, Y, idx, mean, sd


# ---------------------------------------------------------------------------
# states
# ---------------------------------------------------------------------------
class State:
    """Handles and buffers of a user's program; destroys its handles with itself."""

    def __init__(self, case):
        self.case = case
        self.ctxs, self.probs, self.mlp = [], [], None

    def context(self, stream=None):
        s = stream if stream is not None else torch.cuda.current_stream()
        ctx = m.mdsip_ctx_create(0, s.cuda_stream)
        self.ctxs.append(ctx)
        return ctx

    def problem(self, ctx, d, precision):
        p = m.mdsip_problem_create_synthetic(ctx, mem=m.MDSIP_MEM_DEVICE, **d)
        self.probs.append(p)
        m.mdsip_set_option_int(p, "precision", PREC[precision], ctx)
        return p

    def __del__(self):
        for p in self.probs:
            m.mdsip_problem_destroy(p)
        if self.mlp:
            m.mdsip_mlp_destroy(self.mlp)
        for c in self.ctxs:
            m.mdsip_ctx_destroy(c)


def _batch_sizes(c):
    """Uneven n_d spread over [lo, hi]."""
    span, k = c["hi"] - c["lo"], c["count"]
    return [c["lo"] + (span * ((7 * i) % k)) // max(1, k - 1) for i in range(k)]


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind in ("solve", "direction"):
        d = _instance(case["n_d"], case["m_E"], case["m_I"], case["sigma_a"], seed, case.get("jsh", 0))
        s.ctx = s.context()
        s.prob = s.problem(s.ctx, d, case["precision"])
        s.out = torch.zeros(m.mdsip_packed_size(s.prob), device=DEV, dtype=F64)
        if kind == "direction":
            s.point = torch.cat([_iterate(d, seed)[k] for k in PACKED])
    elif kind == "batch":
        data = [_instance(n, 50 * n, case["m_I"], 0.01, seed * 64 + i) for i, n in enumerate(_batch_sizes(case))]
        s.streams = [torch.cuda.Stream() for _ in data]
        torch.cuda.synchronize()
        for st, d in zip(s.streams, data):
            s.problem(s.context(st), d, case["precision"])
        s.outs = [torch.zeros(m.mdsip_packed_size(p), device=DEV, dtype=F64) for p in s.probs]
    elif kind == "syrk":
        s.ctx = s.context()
        s.A, s.lda, s.w = _syrk_inputs(case, seed)
        s.C = torch.zeros(case["n"], case["n"], device=DEV, dtype=F64)
    elif kind == "ldlt":
        s.ctx = s.context()
        s.K, s.B = _ldlt_inputs(case, seed)
        N = s.K.shape[0]
        s.S, s.L = torch.empty_like(s.K), torch.zeros_like(s.K)
        s.X = torch.empty_like(s.B)
        s.Dd, s.Doff = torch.zeros(N, device=DEV, dtype=F64), torch.zeros(N, device=DEV, dtype=F64)
        s.perm, s.piv = (torch.zeros(N, device=DEV, dtype=torch.int32) for _ in range(2))
        s.inertia = torch.zeros(3, device=DEV, dtype=torch.int32)
    else:
        P, s.Xin, s.Y, s.idx, mean, sd = _mlp_inputs(case, seed)
        s.ctx = s.context()
        s.mlp = m.mdsip_mlp_create(s.ctx, N_P, HIDDEN, case["n_out"])
        flat = torch.zeros(m.mdsip_mlp_num_params(s.mlp), device=DEV)
        for o, v in zip(m.mdsip_mlp_param_offsets(s.mlp), P.values()):
            flat[o:o + v.numel()] = v.reshape(-1)
        m.mdsip_mlp_set_params(s.mlp, flat, m.MDSIP_MEM_DEVICE, s.ctx)
        m.mdsip_mlp_set_scaling(s.mlp, out_mean=mean, out_std=sd, mem=m.MDSIP_MEM_DEVICE, ctx=s.ctx)
        s.out = flat if kind == "train" else torch.empty(case["batch"], case["n_out"], device=DEV)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "solve":
        status = m.mdsip_solve(s.prob, s.ctx)
        m.mdsip_get_iterate(s.prob, s.out, m.MDSIP_MEM_DEVICE, s.ctx)
        return dict(iterate=s.out, iters=m.mdsip_get_stats(s.prob)["iters"], status=status)
    if kind == "batch":
        status = m.mdsip_batch_solve(s.probs)
        for p, ctx, o in zip(s.probs, s.ctxs, s.outs):
            m.mdsip_get_iterate(p, o, m.MDSIP_MEM_DEVICE, ctx)
        iters = torch.tensor([m.mdsip_get_stats(p)["iters"] for p in s.probs])
        return dict(iterates=s.outs, iters=iters, status=torch.tensor(status))
    if kind == "direction":
        inertia = m.mdsip_debug_direction(s.prob, s.point, MU, 0.0, 0.0, s.out, mem=m.MDSIP_MEM_DEVICE, ctx=s.ctx)
        return dict(direction=s.out, inertia=torch.tensor(inertia))
    if kind == "syrk":
        m.mdsip_syrk_scaled(s.ctx, c["m"], c["n"], s.A, s.lda, s.w, 0.0, s.C, c["n"])
        return s.C
    if kind == "ldlt":
        N = s.K.shape[0]
        s.S.copy_(s.K)     # the factorization overwrites its input
        s.X.copy_(s.B)
        m.mdsip_ldlt_factor(s.ctx, N, s.S, N, 1e-14, s.L, s.Dd, s.Doff, s.perm, s.piv, s.inertia)
        m.mdsip_ldlt_solve(s.ctx, N, s.L, s.Dd, s.Doff, s.perm, c["nrhs"], s.X, N)
        return dict(L=s.L, Dd=s.Dd, Doff=s.Doff, perm=s.perm, kind=s.piv, inertia=s.inertia, X=s.X)
    if kind == "train":
        loss = m.mdsip_mlp_train_step(s.mlp, s.Xin, N_P, s.Y, c["n_out"], s.idx, c["batch"], LR, ctx=s.ctx)
        m.mdsip_mlp_get_params(s.mlp, s.out, m.MDSIP_MEM_DEVICE, s.ctx)
        return dict(params=s.out, loss=loss)
    return m.mdsip_mlp_forward(s.mlp, s.Xin, N_P, c["batch"], s.out, c["n_out"], ctx=s.ctx)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
SOLVE_STEPS = 15   # Newton steps of a solve of this family to 1e-8


def _step_work(n_d, m_E, m_I, p1=False):
    N = n_d + m_I + (m_E if p1 else 0)
    flops = N ** 3 / 3 + 8.0 * m_E * n_d + (0 if p1 else n_d * (n_d + 1.0) * m_E)
    return 8.0 * (m_E * n_d + n_d * n_d + 16 * (2 * m_E + n_d)), flops


def work(c):
    kind = c["kind"]
    if kind in ("solve", "direction"):
        b, f = _step_work(c["n_d"], c["m_E"], c["m_I"], bool(c.get("jsh")))
        return dict(bytes=b, flops=f * (SOLVE_STEPS if kind == "solve" else 1))
    if kind == "batch":
        each = [_step_work(n, 50 * n, c["m_I"]) for n in _batch_sizes(c)]
        return dict(bytes=sum(b for b, _ in each), flops=SOLVE_STEPS * sum(f for _, f in each))
    if kind == "syrk":
        mm, n = c["m"], c["n"]
        return dict(bytes=8.0 * (mm * n + mm + n * (n + 1) / 2), flops=n * (n + 1.0) * mm)
    if kind == "ldlt":
        N = 2 * c["k"] + 3
        return dict(bytes=8.0 * (N * N + 2 * N * c["nrhs"]), flops=N ** 3 / 3 + 2.0 * N * N * c["nrhs"])
    B, O = c["batch"], c["n_out"]
    params = O * (HIDDEN + 1.0) + HIDDEN * (HIDDEN + N_P + 2.0)
    if kind == "predict":
        return dict(bytes=4 * params + 8.0 * B * N_P + 4.0 * B * O, flops=2 * params * B)
    # parameters and both moments read and written, the parameters read back, the targets read
    return dict(bytes=28 * params + 8.0 * B * (O + N_P), flops=6 * params * B)


# ---------------------------------------------------------------------------
# the same in plain 64-bit torch
# ---------------------------------------------------------------------------
def _exact_direction(d, it, mu):
    """Newton direction of the primal-dual system by dense elimination of x_s (and, without J_sh, of y_g)."""
    n_s, n_d, m_E, m_I = d["n_s"], d["n_d"], d["m_E"], d["m_I"]
    A, c = d["A"], d["c"]
    x, xs, xd = it["x"], it["x"][:n_s], it["x"][n_s:]
    sub = d["h_set"].long()
    E = torch.zeros(m_I, n_d, device=DEV, dtype=F64)
    k = torch.nonzero(sub >= 0).reshape(-1)
    E[sub[k], k] = 1.0
    Jsh = torch.zeros(m_I, n_s, device=DEV, dtype=F64)
    if "Jsh_vals" in d:
        Jsh[d["Jsh_rows"].long(), d["Jsh_cols"].long()] = d["Jsh_vals"]
    Jdh = 2.0 * E * xd
    sgT = lambda y: torch.cat([y, -y])                       # J_sg^T y
    sg = lambda v: v[:m_E] - v[m_E:]                         # J_sg v
    # barrier terms (x_d is free, the inequalities have upper bounds only)
    sl, su = xs + 1.0, 1.0 - xs
    zl, zu = it["zl"][:n_s], it["zu"][:n_s]
    sv = d["hu"] - it["d"]
    sig_d = it["vu"] / sv
    grad = torch.cat([xs ** 3, d["Q"] @ xd]) + c
    gs = grad[:n_s] + sgT(it["yg"]) + Jsh.T @ it["yh"]
    gd = grad[n_s:] + A.T @ it["yg"] + Jdh.T @ it["yh"]
    b_s = -(gs - mu / sl + mu / su)
    b_d = -gd
    b_g = -(sg(xs) + A @ xd - d["gE"])
    r_h = E @ (xd * xd) + Jsh @ xs - it["d"]
    r_d = -it["yh"] + mu / sv
    b_h = -(r_h + r_d / sig_d)
    q = 3.0 * xs ** 2 + zl / sl + zu / su
    Hdd = d["Q"] + torch.diag(2.0 * (E.T @ it["yh"]))
    D = torch.diag(1.0 / sig_d)
    if "Jsh_vals" not in d:
        w = 1.0 / q[:m_E] + 1.0 / q[m_E:]
        bt = b_g - sg(b_s / q)
        S = torch.cat([torch.cat([Hdd + A.T @ (A / w[:, None]), Jdh.T], 1), torch.cat([Jdh, -D], 1)])
        sol = torch.linalg.solve(S, torch.cat([b_d + A.T @ (bt / w), b_h]))
        dxd, dyh = sol[:n_d], sol[n_d:]
        dyg = (A @ dxd - bt) / w
    else:
        Js = torch.cat([torch.cat([torch.eye(m_E, device=DEV, dtype=F64), -torch.eye(m_E, device=DEV, dtype=F64)], 1), Jsh])
        Jd = torch.cat([A, Jdh])
        M = torch.cat([torch.cat([Hdd, Jd.T], 1), torch.cat([Jd, -(Js / q) @ Js.T], 1)])
        i = torch.arange(m_I, device=DEV) + n_d + m_E
        M[i, i] -= 1.0 / sig_d
        sol = torch.linalg.solve(M, torch.cat([b_d, torch.cat([b_g, b_h]) - Js @ (b_s / q)]))
        dxd, dyg, dyh = sol[:n_d], sol[n_d:n_d + m_E], sol[n_d + m_E:]
    dxs = (b_s - sgT(dyg) - Jsh.T @ dyh) / q
    dd = (dyh - r_d) / sig_d
    zero = torch.zeros(n_d, device=DEV, dtype=F64)
    dzl = torch.cat([mu / sl - zl - zl / sl * dxs, zero])
    dzu = torch.cat([mu / su - zu + zu / su * dxs, zero])
    dvu = mu / sv - it["vu"] + sig_d * dd
    return torch.cat([dxs, dxd, dd, dyg, dyh, dzl, dzu, torch.zeros(m_I, device=DEV, dtype=F64), dvu])


def exact(case, seed):
    kind = case["kind"]
    if kind == "direction":
        d = _instance(case["n_d"], case["m_E"], case["m_I"], case["sigma_a"], seed, case["jsh"])
        return dict(direction=_exact_direction(d, _iterate(d, seed), MU), inertia=None)
    if kind == "syrk":
        A, _, w = _syrk_inputs(case, seed)
        A = A[:, :case["n"]]
        return torch.triu(A.T @ (A / w[:, None]))   # column-major lower triangle
    if kind == "ldlt":
        K, B = _ldlt_inputs(case, seed)
        return dict(L=None, Dd=None, Doff=None, perm=None, kind=None, inertia=None,
                    X=torch.linalg.solve(K, B.T).T.contiguous())
    if kind in ("train", "predict"):
        P, X, Y, idx, mean, sd = _mlp_inputs(case, seed)
        P = {k: v.double() for k, v in P.items()}
        mean, sd = mean.double(), sd.double()
        if kind == "train":
            X, T = X[idx.long()], (Y[idx.long()] - mean) / sd
        z1 = X @ P["W1"].T + P["b1"]
        h1 = torch.relu(z1)
        z2 = h1 @ P["W2"].T + P["b2"]
        h2 = torch.relu(z2)
        yn = h2 @ P["W3"].T + P["b3"]
        if kind == "predict":
            return yn * sd + mean
        e = yn - T
        loss = float((e * e).mean())
        dy = 2.0 * e / e.numel()
        dz2 = (dy @ P["W3"]) * (z2 > 0)
        dz1 = (dz2 @ P["W2"]) * (z1 > 0)
        grads = dict(W1=dz1.T @ X, b1=dz1.sum(0), W2=dz2.T @ h1, b2=dz2.sum(0), W3=dy.T @ h2, b3=dy.sum(0))
        flat = []
        for k, p in P.items():                      # first Adam step: lr g / (|g| + eps)
            v = (p - LR * grads[k] / (grads[k].abs() + ADAM_EPS)).reshape(-1)
            flat += [v, torch.zeros(-v.numel() % 4, device=DEV, dtype=F64)]
        return dict(params=torch.cat(flat), loss=loss)
    return None
