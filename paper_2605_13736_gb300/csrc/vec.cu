// Fused vector kernels of one Newton step (Section 2.3, kernel classes K1 and
// K2) and the evaluation of the benchmark model family (Section 2 problem
// class).  All FP64.  Reductions are deterministic: every reduction kernel
// runs on at most kRedBlocks blocks, one element per thread where there are
// fewer, and its last block combines the blocks' partials in order.
#include "internal.cuh"
#include "vec.cuh"

namespace mdsip {

namespace {

constexpr int NT = kRedThreads;

// ---------------------------------------------------------------------------
// Model: f and grad f.  f = 1/2 x_d^T Q x_d + sum 1/4 x_s^4 + c^T x
// ---------------------------------------------------------------------------
template <int NT>
__global__ void __launch_bounds__(NT) k_eval_f(Dims D, ModelView M, const double *__restrict__ x,
                                               double *__restrict__ grad, RedOut red) {
    double acc = 0.0;
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * NT;
    for (int64_t i = gtid; i < D.n_s; i += gsz) {
        const double v = x[i];
        const double v2 = v * v;
        acc += 0.25 * v2 * v2 + M.c[i] * v;
        if (grad) grad[i] = v2 * v + M.c[i];
    }
    // x_d part: one warp per row of Q
    const int lane = threadIdx.x & 31;
    const int64_t gw = gtid >> 5, nw = gsz >> 5;
    const double *xd = x + D.n_s;
    for (int64_t p = gw; p < D.n_d; p += nw) {
        const double *row = M.Q + p * D.n_d;
        double s = 0.0;
        for (int64_t k = lane; k < D.n_d; k += 32) s += row[k] * xd[k];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) {
            const double cp = M.c[D.n_s + p];
            acc += 0.5 * xd[p] * s + cp * xd[p];
            if (grad) grad[D.n_s + p] = s + cp;
        }
    }
    double v[1] = {acc};
    reduce_finish<NT, R_SUM>(v, red);
}

// ---------------------------------------------------------------------------
// Model: constraint residuals cg = g(x) - g_E (warp per row: sparse part plus
// the dense row of A), ch = h(x) - d.  Reductions: sum |c|, max |c|.
// ---------------------------------------------------------------------------
template <int NT>
__global__ void __launch_bounds__(NT) k_eval_cons(Dims D, ModelView M, const double *__restrict__ x,
                                                  const double *__restrict__ Axd, const double *__restrict__ d,
                                                  double *__restrict__ cg, double *__restrict__ ch, double alpha,
                                                  const double *__restrict__ dAx, double *__restrict__ Ax_out,
                                                  RedOut red) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * NT + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * NT) >> 5;
    const double *xd = x + D.n_s;
    double s1 = 0.0, mx = 0.0;
    // equalities: the dense part A x_d comes from the row-block pass (Axd)
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < D.m_E; i += (int64_t)gridDim.x * NT) {
        double s = Axd[i];
        if (dAx) {   // a step of alpha from where Axd was formed
            s = fma(alpha, dAx[i], s);
            Ax_out[i] = s;
        }
        for (int e = M.csr_ptr[i]; e < M.csr_ptr[i + 1]; ++e) s += M.csr_val[e] * x[M.csr_col[e]];
        const double r = s - M.gE[i];
        cg[i] = r;
        s1 += fabs(r);
        mx = fmax(mx, fabs(r));
    }
    for (int64_t j = gw; j < D.m_I; j += nw) {
        double s = 0.0;
        for (int64_t k = lane; k < D.n_d; k += 32)
            if (M.h_set[k] == j) s += xd[k] * xd[k];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) {
            if (M.hsr_ptr)   // the sparse x_s part of the inequality (J_sh x_s)_j
                for (int e = M.hsr_ptr[j]; e < M.hsr_ptr[j + 1]; ++e) s += M.hsr_val[e] * x[M.hsr_col[e]];
            const double r = s - d[j];
            ch[j] = r;
            s1 += fabs(r);
            mx = fmax(mx, fabs(r));
        }
    }
    double v[2] = {s1, mx};
    reduce_finish<NT, R_SUM, R_MAX>(v, red);
}

// Jacobian of h (dense m_I x n_d row-major) and the Hessian blocks:
// Hss = 3 x_s^2 (diagonal), Hdd = Q + 2 diag(y_h[h_set[k]]).
__global__ void k_jac_hess(Dims D, ModelView M, const double *__restrict__ x,
                           const double *__restrict__ yh, double *__restrict__ Jdh,
                           double *__restrict__ Hss, double *__restrict__ Hdd) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * blockDim.x;
    const double *xd = x + D.n_s;
    for (int64_t i = gtid; i < D.n_s; i += gsz) Hss[i] = 3.0 * x[i] * x[i];
    for (int64_t e = gtid; e < D.m_I * D.n_d; e += gsz) {
        const int64_t j = e / D.n_d, k = e % D.n_d;
        Jdh[e] = M.h_set[k] == j ? 2.0 * xd[k] : 0.0;
    }
    for (int64_t e = gtid; e < D.n_d * D.n_d; e += gsz) {
        const int64_t p = e / D.n_d, q = e % D.n_d;
        double v = M.Q[e];
        if (p == q && M.h_set[p] >= 0) v += 2.0 * yh[M.h_set[p]];
        Hdd[e] = v;
    }
}

// ---------------------------------------------------------------------------
// A passes
// ---------------------------------------------------------------------------
// out = A v: two threads per row, v staged in shared memory.  The pair reads
// alternate 16-byte chunks of its row, so each warp load fills 16 whole
// 32-byte sectors; each thread keeps eight independent FP64 accumulators and
// loads the next group of its row before using the current one (a pass over A
// is bound by memory latency at the ~20 rows per SM that one-thread-per-row
// occupancy gives, and on GB300 by the DFMA rate next: 2 flop per 8 bytes).
__global__ void __launch_bounds__(NT) k_gemv_rows(const double *__restrict__ A, int64_t m, int64_t n,
                                                  int64_t lda, const double *__restrict__ v,
                                                  double *__restrict__ out) {
    extern __shared__ double vs[];   // n rounded up to a multiple of 16, zero padded
    const int64_t n16 = (n + 15) / 16 * 16;
    for (int64_t k = threadIdx.x; k < n16; k += NT) vs[k] = k < n ? v[k] : 0.0;
    __syncthreads();
    const int64_t gt = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int64_t i = gt >> 1;
    const int h = (int)(gt & 1);
    const bool live = i < m;
    const double2 *r = reinterpret_cast<const double2 *>(A + (live ? i : 0) * lda);
    const double2 *x2 = reinterpret_cast<const double2 *>(vs);
    double acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = 0.0;
    const int64_t full = live ? n / 16 : 0;   // groups of 16 columns (8 chunks; 4 per thread)
    double2 cur[4], nxt[4] = {};
    if (full > 0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) cur[u] = __ldg(r + h + 2 * u);
    }
    for (int64_t g = 0; g < full; ++g) {
        if (g + 1 < full) {
#pragma unroll
            for (int u = 0; u < 4; ++u) nxt[u] = __ldg(r + 8 * (g + 1) + h + 2 * u);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const double2 b = x2[8 * g + h + 2 * u];
            acc[2 * u] = fma(cur[u].x, b.x, acc[2 * u]);
            acc[2 * u + 1] = fma(cur[u].y, b.y, acc[2 * u + 1]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) cur[u] = nxt[u];
    }
    if (live && h == 0) {
        const double *rd = A + i * lda;
#pragma unroll
        for (int t = 0; t < 16; ++t) {   // ragged tail (fewer than 16 columns)
            const int64_t c = 16 * full + t;
            if (c < n) acc[t & 7] = fma(rd[c], vs[c], acc[t & 7]);
        }
    }
    double sum = ((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7]));
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);   // the pair's halves (every lane reaches this)
    if (live && h == 0) out[i] = sum;
}

// partial[b][p] = sum over the rows of block b of A[i][p] u[i].  tc threads (a
// power of two) take the columns, C each, and the block's NT / tc groups its
// rows, U in flight: 8 to 12 loads a thread cover the memory's latency (m =
// 15053, n = 301: 54 us with one row pair in flight and 8 columns per thread of
// which two were used, 20 us so; m = 1000, n = 32: 8 -> 6 us).  Above 1024
// columns eight a thread stay: bound by the FP64 pipe, fewer columns repeat the
// row's addresses (m = 100000, n = 2000: 363 us, with four columns 467).
template <int C, int U>
__global__ void __launch_bounds__(NT) k_gemv_t(const double *__restrict__ A, int64_t m, int64_t n,
                                               int64_t lda, const double *__restrict__ u, int tc,
                                               double *__restrict__ partial) {
    __shared__ double sh[NT];
    const int col = threadIdx.x & (tc - 1), g = threadIdx.x / tc, G = NT / tc;
    const int64_t rows_per = (m + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = (int64_t)blockIdx.x * rows_per;
    const int64_t r1 = min(m, r0 + rows_per);
    for (int64_t c0 = 0; c0 < n; c0 += (int64_t)tc * C) {
        double acc[C];
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] = 0.0;
        int64_t i = r0 + g;
        if constexpr (C <= 2)                  // few rows a thread: the last batch stays whole
            for (; i < r1; i += (int64_t)U * G) {
                double a[U][C], ui[U];
#pragma unroll
                for (int x = 0; x < U; ++x) {
                    const int64_t r = i + (int64_t)x * G;
                    ui[x] = r < r1 ? __ldg(u + r) : 0.0;
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        const int64_t p = c0 + col + (int64_t)c * tc;
                        a[x][c] = r < r1 && p < n ? __ldg(A + r * lda + p) : 0.0;
                    }
                }
#pragma unroll
                for (int x = 0; x < U; ++x)
                    if (i + (int64_t)x * G < r1)
#pragma unroll
                        for (int c = 0; c < C; ++c) acc[c] = fma(a[x][c], ui[x], acc[c]);
            }
        for (; i + (int64_t)(U - 1) * G < r1; i += (int64_t)U * G) {
            double a[U][C], ui[U];
#pragma unroll
            for (int x = 0; x < U; ++x) {
                const double *row = A + (i + (int64_t)x * G) * lda;
                ui[x] = __ldg(u + i + (int64_t)x * G);
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int64_t p = c0 + col + (int64_t)c * tc;
                    a[x][c] = p < n ? __ldg(row + p) : 0.0;
                }
            }
#pragma unroll
            for (int x = 0; x < U; ++x)
#pragma unroll
                for (int c = 0; c < C; ++c) acc[c] = fma(a[x][c], ui[x], acc[c]);
        }
        for (; i < r1; i += G) {
            const double *row = A + i * lda;
            const double ui = __ldg(u + i);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int64_t p = c0 + col + (int64_t)c * tc;
                if (p < n) acc[c] = fma(__ldg(row + p), ui, acc[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int64_t p = c0 + col + (int64_t)c * tc;
            double v = acc[c];
            if (G > 1) {                       // tc < NT: one pass, one column per thread
                sh[threadIdx.x] = v;
                __syncthreads();
                for (int x = 1; x < G; ++x)
                    if (g == 0) v += sh[x * tc + col];
            }
            if (g == 0 && p < n) partial[(size_t)blockIdx.x * n + p] = v;
        }
    }
}

// out[p] = sum_b partial[b][p]: a block per 32 columns, warp w summing the
// partials b = w, w + 8, ... in order (coalesced 32-column rows, eight rows in
// flight per warp), then the eight warp sums in order (deterministic).
__global__ void __launch_bounds__(256) k_colsum(const double *__restrict__ partial, int nparts, int64_t n,
                                                double *__restrict__ out) {
    __shared__ double sp[8][33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * 32 + lane;
    double s = 0.0;
    if (p < n) {
        int b = wid;
        for (; b + 24 < nparts; b += 32) {
            const double a0 = partial[(size_t)b * n + p], a1 = partial[(size_t)(b + 8) * n + p];
            const double a2 = partial[(size_t)(b + 16) * n + p], a3 = partial[(size_t)(b + 24) * n + p];
            s += a0;
            s += a1;
            s += a2;
            s += a3;
        }
        for (; b < nparts; b += 8) s += partial[(size_t)b * n + p];
    }
    sp[wid][lane] = s;
    __syncthreads();
    if (wid == 0 && p < n) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += sp[w][lane];
        out[p] = t;
    }
}

// ---------------------------------------------------------------------------
// Gradient of the Lagrangian: gl = grad f + J_g^T y_g + J_h^T y_h
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(NT) k_lagrangian_grad(Dims D, ModelView M, const double *__restrict__ grad,
                                  const double *__restrict__ yg, const double *__restrict__ yh,
                                  const double *__restrict__ Jdh, const double *__restrict__ ATy,
                                  double *__restrict__ gl) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = gtid; i < D.n_s; i += gsz) {
        double s = grad[i];
        for (int e = M.csc_ptr[i]; e < M.csc_ptr[i + 1]; ++e) s += M.csc_val[e] * yg[M.csc_row[e]];
        if (M.hsc_ptr)
            for (int e = M.hsc_ptr[i]; e < M.hsc_ptr[i + 1]; ++e) s += M.hsc_val[e] * yh[M.hsc_row[e]];
        gl[i] = s;
    }
    __shared__ double sp[NT / 32][33];
    for (int64_t k0 = (int64_t)blockIdx.x * 32; k0 < D.n_d; k0 += (int64_t)gridDim.x * 32) {
        const double jt = colgroup_dot<NT>(Jdh, D.m_I, D.n_d, k0, yh, sp);
        const int64_t k = k0 + threadIdx.x;
        if (threadIdx.x < 32 && k < D.n_d) gl[D.n_s + k] = grad[D.n_s + k] + ATy[k] + jt;
    }
}

// ---------------------------------------------------------------------------
// Optimality error components (W&B scaled KKT error) and the log-barrier sum.
// quantities: 0 max|dual| (max), 1 max|c| (max), 2 max s*z (max),
//             3 min s*z (min), 4 ||y||_1 (sum), 5 ||z||_1 (sum), 6 sum log s (sum)
// ---------------------------------------------------------------------------
template <int NT>
__global__ void __launch_bounds__(NT) k_errors(Dims D, ModelView M, IterView I,
                                               const double *__restrict__ gl,
                                               const double *__restrict__ cg,
                                               const double *__restrict__ ch, RedOut red) {
    unsigned long long du = 0, pr = 0;
    MinMax comp;
    LogSum lg;
    double y1 = 0.0, z1 = 0.0;
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * NT;
    for (int64_t i = gtid; i < D.n; i += gsz) {
        const double xi = I.x[i];
        max_abs(du, gl[i] - I.zl[i] + I.zu[i]);
        if (fin(M.xl[i])) {
            const double s = xi - M.xl[i];
            comp.add(s * I.zl[i]);
            z1 += fabs(I.zl[i]);
            lg.add(s);
        }
        if (fin(M.xu[i])) {
            const double s = M.xu[i] - xi;
            comp.add(s * I.zu[i]);
            z1 += fabs(I.zu[i]);
            lg.add(s);
        }
    }
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        max_abs(du, -I.yh[j] - I.vl[j] + I.vu[j]);
        max_abs(pr, ch[j]);
        y1 += fabs(I.yh[j]);
        const double dj = I.d[j];
        if (fin(M.hl[j])) {
            const double s = dj - M.hl[j];
            comp.add(s * I.vl[j]);
            z1 += fabs(I.vl[j]);
            lg.add(s);
        }
        if (fin(M.hu[j])) {
            const double s = M.hu[j] - dj;
            comp.add(s * I.vu[j]);
            z1 += fabs(I.vu[j]);
            lg.add(s);
        }
    }
    for (int64_t i = gtid; i < D.m_E; i += gsz) {
        max_abs(pr, cg[i]);
        y1 += fabs(I.yg[i]);
    }
    double v[7] = {__longlong_as_double((long long)du), __longlong_as_double((long long)pr), MinMax::value(comp.hi),
                   MinMax::value(comp.lo), y1, z1, lg.value()};
    reduce_finish<NT, R_MAX, R_MAX, R_MAX, R_MIN, R_SUM, R_SUM, R_SUM>(v, red);
}

// ---------------------------------------------------------------------------
// Diagonal scaling (Section 2.1 barrier diagonals) and the diagonal W of the
// two-stage elimination.  q = H_ss + Sigma_xs + dw; Sigma_d; w = J_sg^2 q^-1 + dc.
// quantities: 0..2 inertia of Q_s (pos, neg, zero), 3..5 inertia of -W.
// ---------------------------------------------------------------------------
// sign of a value by its bit pattern (NaN counts nowhere)
__device__ __forceinline__ void count_sign(double v, unsigned &pos, unsigned &neg, unsigned &zero) {
    const long long b = __double_as_longlong(v), m = b & 0x7fffffffffffffffLL;
    if (m > 0x7ff0000000000000LL) return;
    zero += m == 0;
    pos += m != 0 && b > 0;
    neg += m != 0 && b < 0;
}

__device__ __forceinline__ double sigma_x(const ModelView &M, const IterView &I, int64_t i) {
    double s = 0.0;
    if (fin(M.xl[i])) s += ddiv(I.zl[i], I.x[i] - M.xl[i]);
    if (fin(M.xu[i])) s += ddiv(I.zu[i], M.xu[i] - I.x[i]);
    return s;
}

template <int NT>
__global__ void __launch_bounds__(NT) k_newton_diag(Dims D, ModelView M, IterView I,
                                                    const double *__restrict__ Hss, double dw,
                                                    double dc, int want_w, double *__restrict__ sig_x,
                                                    double *__restrict__ q, double *__restrict__ sig_d,
                                                    double *__restrict__ w, RedOut red) {
    unsigned c6[6] = {0, 0, 0, 0, 0, 0};   // In(Q_s), In(-W): positive, negative, zero
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * NT;
    for (int64_t i = gtid; i < D.n; i += gsz) {
        const double s = sigma_x(M, I, i);
        sig_x[i] = s;
        if (i < D.n_s) {
            const double qi = Hss[i] + s + dw;
            q[i] = qi;
            count_sign(qi, c6[0], c6[1], c6[2]);
        }
    }
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        double s = 0.0;
        if (fin(M.hl[j])) s += ddiv(I.vl[j], I.d[j] - M.hl[j]);
        if (fin(M.hu[j])) s += ddiv(I.vu[j], M.hu[j] - I.d[j]);
        sig_d[j] = s;
    }
    if (want_w) {
        for (int64_t i = gtid; i < D.m_E; i += gsz) {
            double s = dc;
            for (int e = M.csr_ptr[i]; e < M.csr_ptr[i + 1]; ++e) {
                const int64_t c = M.csr_col[e];
                const double qc = Hss[c] + sigma_x(M, I, c) + dw;
                s += ddiv(M.csr_val[e] * M.csr_val[e], qc);
            }
            w[i] = s;
            count_sign(s, c6[4], c6[3], c6[5]);   // of -W
        }
    }
    count_finish<NT>(c6, red);
}

// barrier gradient of the Lagrangian at x: rN_i = gl_i - mu/s_l + mu/s_u
__device__ __forceinline__ double rN_x(const ModelView &M, const IterView &I, const double *gl,
                                       double mu, int64_t i) {
    double r = gl[i];
    if (fin(M.xl[i])) r -= ddiv(mu, I.x[i] - M.xl[i]);
    if (fin(M.xu[i])) r += ddiv(mu, M.xu[i] - I.x[i]);
    return r;
}

// r_d = grad_d phi - y_h = -mu/(d - hl) + mu/(hu - d) - y_h
__device__ __forceinline__ double r_dslack(const ModelView &M, const IterView &I, double mu,
                                           int64_t j) {
    double r = -I.yh[j];
    if (fin(M.hl[j])) r -= ddiv(mu, I.d[j] - M.hl[j]);
    if (fin(M.hu[j])) r += ddiv(mu, M.hu[j] - I.d[j]);
    return r;
}

// ---------------------------------------------------------------------------
// Right-hand sides.  b = -[rN_x; c_g; c_h + Dh^-1 r_d] (Eq. (linsys4x4) rows).
// Path P2: bt_g = b_g - J_sg (b_s / q);  u = bt_g / w;  rhs_S = [b_d + A^T u; b_h]
// Path P1: rhs_M = [b_d; b_y - J_s (b_s / q)]
// ---------------------------------------------------------------------------
__global__ void k_rhs_y(Dims D, ModelView M, IterView I, const double *__restrict__ gl,
                        const double *__restrict__ cg, const double *__restrict__ q,
                        const double *__restrict__ w, double mu, double *__restrict__ bt_g,
                        double *__restrict__ u) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = gtid; i < D.m_E; i += gsz) {
        double s = -cg[i];
        for (int e = M.csr_ptr[i]; e < M.csr_ptr[i + 1]; ++e) {
            const int64_t c = M.csr_col[e];
            s += ddiv(M.csr_val[e] * rN_x(M, I, gl, mu, c), q[c]);   // -J_sg (b_s/q), b_s = -rN_s
        }
        bt_g[i] = s;
        if (u) u[i] = ddiv(s, w[i]);
    }
}

// P2: rhs_S[0:n_d] = -rN_xd + ATu ; rhs_S[n_d + j] = -(ch + r_d / Dh)
// P1: rhs_M[0:n_d] = -rN_xd ; rhs_M[n_d + i] = bt_g[i] ; rhs_M[n_d + m_E + j] = -(ch + r_d/Dh)
// (with J_sh != 0, P1's h rows also take -J_sh (b_s / q))
__global__ void k_rhs_reduced(Dims D, ModelView M, IterView I, const double *__restrict__ gl,
                              const double *__restrict__ ch, const double *__restrict__ sig_d,
                              const double *__restrict__ ATu, const double *__restrict__ bt_g,
                              const double *__restrict__ q, double mu, double dw, int p1,
                              double *__restrict__ rhs) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = gtid; k < D.n_d; k += gsz) {
        double r = -rN_x(M, I, gl, mu, D.n_s + k);
        if (!p1) r += ATu[k];
        rhs[k] = r;
    }
    const int64_t off_h = p1 ? D.n_d + D.m_E : D.n_d;
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        double r = -(ch[j] + ddiv(r_dslack(M, I, mu, j), sig_d[j] + dw));
        if (p1 && M.hsr_ptr)
            for (int e = M.hsr_ptr[j]; e < M.hsr_ptr[j + 1]; ++e) {
                const int64_t c = M.hsr_col[e];
                r += ddiv(M.hsr_val[e] * rN_x(M, I, gl, mu, c), q[c]);   // -J_sh (b_s/q), b_s = -rN_s
            }
        rhs[off_h + j] = r;
    }
    if (p1)
        for (int64_t i = gtid; i < D.m_E; i += gsz) rhs[D.n_d + i] = bt_g[i];
}

// P2: dy_g = (A dx_d - bt_g) / w
__global__ void k_dyg_p2(int64_t m_E, const double *__restrict__ Adx, const double *__restrict__ bt_g,
                         const double *__restrict__ w, double *__restrict__ dyg) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m_E;
         i += (int64_t)gridDim.x * blockDim.x)
        dyg[i] = ddiv(Adx[i] - bt_g[i], w[i]);
}

// Common back-substitution: dx_s = (b_s - J_sg^T dy_g)/q, dx_d, dy_h from the
// reduced solution, dd = (dy_h - r_d)/Dh, and the bound-multiplier steps
// dz = mu/s - z - (z/s) ds (W&B eq. (11)).
__global__ void k_backsub(Dims D, ModelView M, IterView I, DirView Dir, const double *__restrict__ gl,
                          const double *__restrict__ q, const double *__restrict__ sig_d,
                          const double *__restrict__ sol_dxd, const double *__restrict__ sol_dyh,
                          double mu, double dw) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = gtid; i < D.n; i += gsz) {
        double dx;
        if (i < D.n_s) {
            double s = -rN_x(M, I, gl, mu, i);
            for (int e = M.csc_ptr[i]; e < M.csc_ptr[i + 1]; ++e)
                s -= M.csc_val[e] * Dir.dyg[M.csc_row[e]];
            if (M.hsc_ptr)   // J_sh^T dy_h (dy_h from the reduced solution: Dir.dyh is written below)
                for (int e = M.hsc_ptr[i]; e < M.hsc_ptr[i + 1]; ++e) s -= M.hsc_val[e] * sol_dyh[M.hsc_row[e]];
            dx = ddiv(s, q[i]);
        } else {
            dx = sol_dxd[i - D.n_s];
        }
        Dir.dx[i] = dx;
        const double xi = I.x[i];
        if (fin(M.xl[i])) {
            const double s = xi - M.xl[i];
            Dir.dzl[i] = ddiv(mu, s) - I.zl[i] - ddiv(I.zl[i], s) * dx;
        } else {
            Dir.dzl[i] = 0.0;
        }
        if (fin(M.xu[i])) {
            const double s = M.xu[i] - xi;
            Dir.dzu[i] = ddiv(mu, s) - I.zu[i] + ddiv(I.zu[i], s) * dx;
        } else {
            Dir.dzu[i] = 0.0;
        }
    }
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        const double dyh = sol_dyh[j];
        Dir.dyh[j] = dyh;
        const double dd = ddiv(dyh - r_dslack(M, I, mu, j), sig_d[j] + dw);
        Dir.dd[j] = dd;
        const double dj = I.d[j];
        if (fin(M.hl[j])) {
            const double s = dj - M.hl[j];
            Dir.dvl[j] = ddiv(mu, s) - I.vl[j] - ddiv(I.vl[j], s) * dd;
        } else {
            Dir.dvl[j] = 0.0;
        }
        if (fin(M.hu[j])) {
            const double s = M.hu[j] - dj;
            Dir.dvu[j] = ddiv(mu, s) - I.vu[j] + ddiv(I.vu[j], s) * dd;
        } else {
            Dir.dvu[j] = 0.0;
        }
    }
}

// Distance between two packed directions: quantities 0 = sum (a - b)^2,
// 1 = sum b^2 over the eight blocks (dx, dd, dyg, dyh, dzl, dzu, dvl, dvu).
__global__ void __launch_bounds__(NT) k_dir_diff(Dims D, DirView a, DirView b, RedOut red) {
    const double *pa[8] = {a.dx, a.dd, a.dyg, a.dyh, a.dzl, a.dzu, a.dvl, a.dvu};
    const double *pb[8] = {b.dx, b.dd, b.dyg, b.dyh, b.dzl, b.dzu, b.dvl, b.dvu};
    const int64_t len[8] = {D.n, D.m_I, D.m_E, D.m_I, D.n, D.n, D.m_I, D.m_I};
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * NT;
    double dd = 0.0, bb = 0.0;
    for (int k = 0; k < 8; ++k)
        for (int64_t i = gtid; i < len[k]; i += gsz) {
            const double y = pb[k][i], e = pa[k][i] - y;
            dd += e * e;
            bb += y * y;
        }
    double v[2] = {dd, bb};
    reduce_finish<NT, R_SUM, R_SUM>(v, red);
}

__global__ void k_copy(const double *__restrict__ src, double *__restrict__ dst, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[i];
}

// ---------------------------------------------------------------------------
// Line-search scalars: fraction-to-boundary (Section 2.1: the search starts at
// the farthest bound-feasible point) and grad phi^T d.
// quantities: 0 alpha_max (min), 1 alpha_z (min), 2 gphi (sum)
// ---------------------------------------------------------------------------
// alpha such that v + alpha dv = (1 - tau) v, where that is below 1 (larger ones
// do not bind: the caller caps alpha at 1)
__device__ __forceinline__ double ftb(double v, double dv, double tau) {
    const double t = tau * v;
    return -dv > t ? ddiv(-t, dv) : INFINITY;
}

template <int NT>
__global__ void __launch_bounds__(NT) k_step_scalars(Dims D, ModelView M, IterView I, DirView Dir,
                                                     const double *__restrict__ grad, double tau,
                                                     double mu, RedOut red) {
    double ap = INFINITY, az = INFINITY, gp = 0.0;
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * NT;
    for (int64_t i = gtid; i < D.n; i += gsz) {
        const double dx = Dir.dx[i];
        double g = grad[i];
        if (fin(M.xl[i])) {
            const double s = I.x[i] - M.xl[i];
            ap = fmin(ap, ftb(s, dx, tau));
            az = fmin(az, ftb(I.zl[i], Dir.dzl[i], tau));
            g -= ddiv(mu, s);
        }
        if (fin(M.xu[i])) {
            const double s = M.xu[i] - I.x[i];
            ap = fmin(ap, ftb(s, -dx, tau));
            az = fmin(az, ftb(I.zu[i], Dir.dzu[i], tau));
            g += ddiv(mu, s);
        }
        gp += g * dx;
    }
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        const double dd = Dir.dd[j];
        double g = 0.0;
        if (fin(M.hl[j])) {
            const double s = I.d[j] - M.hl[j];
            ap = fmin(ap, ftb(s, dd, tau));
            az = fmin(az, ftb(I.vl[j], Dir.dvl[j], tau));
            g -= ddiv(mu, s);
        }
        if (fin(M.hu[j])) {
            const double s = M.hu[j] - I.d[j];
            ap = fmin(ap, ftb(s, -dd, tau));
            az = fmin(az, ftb(I.vu[j], Dir.dvu[j], tau));
            g += ddiv(mu, s);
        }
        gp += g * dd;
    }
    double v[3] = {ap, az, gp};
    reduce_finish<NT, R_MIN, R_MIN, R_SUM>(v, red);
}

// Trial point x_t = x + alpha dx, d_t = d + alpha dd; sum of log slacks and
// "strictly inside" count at the trial point.
// quantities: 0 sum log s (sum), 1 number of non-positive slacks (sum)
template <int NT>
__global__ void __launch_bounds__(NT) k_trial(Dims D, ModelView M, IterView I, DirView Dir,
                                              double alpha, double *__restrict__ xt,
                                              double *__restrict__ dt, RedOut red) {
    LogSum lg;
    unsigned bad = 0;
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * NT;
    for (int64_t i = gtid; i < D.n; i += gsz) {
        const double v = I.x[i] + alpha * Dir.dx[i];
        xt[i] = v;
        if (fin(M.xl[i])) {
            const double s = v - M.xl[i];
            if (s > 0.0) lg.add(s); else ++bad;
        }
        if (fin(M.xu[i])) {
            const double s = M.xu[i] - v;
            if (s > 0.0) lg.add(s); else ++bad;
        }
    }
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        const double v = I.d[j] + alpha * Dir.dd[j];
        dt[j] = v;
        if (fin(M.hl[j])) {
            const double s = v - M.hl[j];
            if (s > 0.0) lg.add(s); else ++bad;
        }
        if (fin(M.hu[j])) {
            const double s = M.hu[j] - v;
            if (s > 0.0) lg.add(s); else ++bad;
        }
    }
    double v[2] = {lg.value(), (double)bad};
    reduce_finish<NT, R_SUM, R_SUM>(v, red);
}

// Accept: y += alpha dy, z += alpha_z dz, then the kappa_Sigma safeguard
// (W&B eq. (16)) against the new slacks (x, d already hold the new point).
__global__ void k_accept(Dims D, ModelView M, IterView I, DirView Dir, double alpha,
                         double alpha_z, double mu, double ks, double *__restrict__ ATy,
                         const double *__restrict__ dATy) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * blockDim.x;
    auto guard = [&](double z, double s) { return fmax(fmin(z, ddiv(ks * mu, s)), ddiv(mu, ks * s)); };
    for (int64_t i = gtid; i < D.m_E; i += gsz) I.yg[i] += alpha * Dir.dyg[i];
    if (dATy)   // A^T y_g follows y_g
        for (int64_t k = gtid; k < D.n_d; k += gsz) ATy[k] = fma(alpha, dATy[k], ATy[k]);
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        I.yh[j] += alpha * Dir.dyh[j];
        const double dj = I.d[j];
        if (fin(M.hl[j])) I.vl[j] = guard(I.vl[j] + alpha_z * Dir.dvl[j], dj - M.hl[j]);
        if (fin(M.hu[j])) I.vu[j] = guard(I.vu[j] + alpha_z * Dir.dvu[j], M.hu[j] - dj);
    }
    for (int64_t i = gtid; i < D.n; i += gsz) {
        const double xi = I.x[i];
        if (fin(M.xl[i])) I.zl[i] = guard(I.zl[i] + alpha_z * Dir.dzl[i], xi - M.xl[i]);
        if (fin(M.xu[i])) I.zu[i] = guard(I.zu[i] + alpha_z * Dir.dzu[i], M.xu[i] - xi);
    }
}

// W&B Section 3.6 starting point: push x0 (and d0 = h(x0)) inside the bounds;
// multipliers of finite bounds 1, y = 0.
__device__ double push_inside(double v, double lo, double hi, double k1, double k2) {
    const bool hl = fin(lo), hu = fin(hi);
    const double width = (hl && hu) ? hi - lo : INFINITY;
    if (hl) {
        const double pl = fmin(k1 * fmax(1.0, fabs(lo)), k2 * width);
        v = fmax(v, lo + pl);
    }
    if (hu) {
        const double pu = fmin(k1 * fmax(1.0, fabs(hi)), k2 * width);
        v = fmin(v, hi - pu);
    }
    return v;
}

__global__ void k_init_x(Dims D, ModelView M, const double *__restrict__ x0, double k1, double k2,
                         IterView I) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = gtid; i < D.n; i += gsz) {
        I.x[i] = push_inside(x0 ? x0[i] : 0.0, M.xl[i], M.xu[i], k1, k2);
        I.zl[i] = fin(M.xl[i]) ? 1.0 : 0.0;
        I.zu[i] = fin(M.xu[i]) ? 1.0 : 0.0;
    }
    for (int64_t i = gtid; i < D.m_E; i += gsz) I.yg[i] = 0.0;
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        I.yh[j] = 0.0;
        I.d[j] = 0.0;
        I.vl[j] = fin(M.hl[j]) ? 1.0 : 0.0;
        I.vu[j] = fin(M.hu[j]) ? 1.0 : 0.0;
    }
}

// d0 = push(h(x0)); ch currently holds h(x0) - 0
__global__ void k_init_d(Dims D, ModelView M, const double *__restrict__ ch, double k1, double k2,
                         IterView I) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < D.m_I;
         j += (int64_t)gridDim.x * blockDim.x)
        I.d[j] = push_inside(ch[j], M.hl[j], M.hu[j], k1, k2);
}

// Warm start from a prediction in the packed layout [x | d | y_g | y_h | z_l |
// z_u | v_l | v_u]: primal values pushed inside the bounds (the Section 3.6
// rule of W&B with kappa_1 = kappa_2 = push), each finite-bound multiplier
// raised to at least mu0 / (its slack), so that every complementarity
// product is at least mu0; multipliers of infinite bounds are 0.
__global__ void k_start_predicted(Dims D, ModelView M, const float *__restrict__ pred, double push, double mu0,
                                  IterView I) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * blockDim.x;
    const int64_t o_d = D.n, o_yg = o_d + D.m_I, o_yh = o_yg + D.m_E, o_zl = o_yh + D.m_I, o_zu = o_zl + D.n,
                  o_vl = o_zu + D.n, o_vu = o_vl + D.m_I;
    for (int64_t i = gtid; i < D.n; i += gsz) {
        const double lo = M.xl[i], hi = M.xu[i];
        const double x = push_inside((double)pred[i], lo, hi, push, push);
        I.x[i] = x;
        I.zl[i] = fin(lo) ? fmax((double)pred[o_zl + i], mu0 / (x - lo)) : 0.0;
        I.zu[i] = fin(hi) ? fmax((double)pred[o_zu + i], mu0 / (hi - x)) : 0.0;
    }
    for (int64_t i = gtid; i < D.m_E; i += gsz) I.yg[i] = (double)pred[o_yg + i];
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        const double lo = M.hl[j], hi = M.hu[j];
        const double d = push_inside((double)pred[o_d + j], lo, hi, push, push);
        I.d[j] = d;
        I.yh[j] = (double)pred[o_yh + j];
        I.vl[j] = fin(lo) ? fmax((double)pred[o_vl + j], mu0 / (d - lo)) : 0.0;
        I.vu[j] = fin(hi) ? fmax((double)pred[o_vu + j], mu0 / (hi - d)) : 0.0;
    }
}

__global__ void __launch_bounds__(NT) k_cons_from_values(Dims D, ModelView M, const double *__restrict__ g,
                                                         const double *__restrict__ h, const double *__restrict__ d,
                                                         double *__restrict__ cg, double *__restrict__ ch,
                                                         RedOut red) {
    double s1 = 0.0, mx = 0.0;
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x, gsz = (int64_t)gridDim.x * NT;
    for (int64_t i = gtid; i < D.m_E; i += gsz) {
        const double r = g[i] - M.gE[i];
        cg[i] = r;
        s1 += fabs(r);
        mx = fmax(mx, fabs(r));
    }
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        const double r = h[j] - d[j];
        ch[j] = r;
        s1 += fabs(r);
        mx = fmax(mx, fabs(r));
    }
    double v[2] = {s1, mx};
    reduce_finish<NT, R_SUM, R_MAX>(v, red);
}

__global__ void k_gather(int64_t n, const double *__restrict__ src, const int32_t *__restrict__ idx,
                         double *__restrict__ dst) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[idx[i]];
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// Up to one element per thread of kRedBlocks blocks of 128 a kernel is one chain
// of FP64 instructions per thread, 64 cycles each for a warp alone on its
// sub-partition: such blocks spread them over twice the SMs (2032 variables,
// with the logarithms and maxima above: k_errors 15.6 -> 11.3 us, k_trial 13.5 ->
// 9.9).  Longer vectors keep 256: at 51712 a second round took k_newton_diag
// from 14.7 to 18.6.
constexpr int64_t kSmallLen = (int64_t)128 * kRedBlocks;
#define MDSIP_RED(kern, len, ...)                                                      \
    do {                                                                               \
        const int64_t len_ = (len);                                                    \
        if (len_ <= kSmallLen) kern<128><<<red_grid(len_, 128), 128, 0, st>>>(__VA_ARGS__); \
        else kern<NT><<<red_grid(len_), NT, 0, st>>>(__VA_ARGS__);                     \
        MDSIP_LAUNCHED();                                                              \
    } while (0)

static int elem_grid(int64_t n, int threads = 256) { return std::max(1, std::min(4096, ceil_div(n, threads))); }
static int elem_threads(int64_t n) { return n <= kSmallLen ? 128 : 256; }

// A: rows 16-byte aligned (lda even, A 16-byte aligned); n <= 24560 (v staged in shared memory)
void launch_gemv_rows(cudaStream_t s, const double *A, int64_t m, int64_t n, int64_t lda,
                      const double *v, double *out) {
    if (m <= 0) return;
    MDSIP_REQUIRE((lda & 1) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0, MDSIP_ERR_INVALID_ARG,
                  "gemv: rows of A must be 16-byte aligned");
    const size_t smem = (size_t)((n + 15) / 16) * 16 * sizeof(double);
    MDSIP_REQUIRE(smem <= 192 * 1024, MDSIP_ERR_INVALID_ARG, "gemv: n too large");
    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_gemv_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, 192 * 1024);
    }));
    const int64_t grid = (2 * m + NT - 1) / NT;   // two threads per row
    MDSIP_REQUIRE(grid <= 0x7fffffff, MDSIP_ERR_INVALID_ARG, "gemv: m too large");
    k_gemv_rows<<<(unsigned)grid, NT, smem, s>>>(A, m, n, lda, v, out);
    MDSIP_LAUNCHED();
}

void launch_colsum(cudaStream_t s, const double *partial, int nparts, int64_t n, double *out) {
    if (n <= 0) return;
    k_colsum<<<(unsigned)ceil_div(n, 32), 256, 0, s>>>(partial, nparts, n, out);
    MDSIP_LAUNCHED();
}

void launch_gemv_t(cudaStream_t s, const double *A, int64_t m, int64_t n, int64_t lda,
                   const double *u, double *partial, double *out) {
    if (n <= 0) return;
    if (m <= 0) {
        MDSIP_CUDA(cudaMemsetAsync(out, 0, n * sizeof(double), s));
        return;
    }
    // threads over columns first; with fewer than NT columns the rest of the block takes further rows
    int tc = 32;
    while (tc < NT && tc < n) tc *= 2;
    const int grid = (int)std::min<int64_t>(kRedBlocks, ceil_div(m, (int64_t)8 * (NT / tc)));
    if (n <= NT) k_gemv_t<1, 8><<<grid, NT, 0, s>>>(A, m, n, lda, u, tc, partial);
    else if (n <= 2 * NT) k_gemv_t<2, 6><<<grid, NT, 0, s>>>(A, m, n, lda, u, tc, partial);
    else if (n <= 4 * NT) k_gemv_t<4, 3><<<grid, NT, 0, s>>>(A, m, n, lda, u, tc, partial);
    else k_gemv_t<8, 2><<<grid, NT, 0, s>>>(A, m, n, lda, u, tc, partial);
    MDSIP_LAUNCHED();
    k_colsum<<<(unsigned)ceil_div(n, 32), 256, 0, s>>>(partial, grid, n, out);
    MDSIP_LAUNCHED();
}

void VecOps::eval_f(const double *x, double *grad, double *out_scalar) {
    MDSIP_RED(k_eval_f, std::max(D.n_s, 32 * D.n_d), D, M, x, grad, red(out_scalar));
}

void VecOps::eval_cons(const double *x, const double *d, double *cg, double *ch, double *out2) {
    if (D.m_E > 0) {
        if (Ahi) launch_gemv_rows_df(st, Ahi, Alo, D.m_E, D.n_d, D.lda, x + D.n_s, split, rowtmp);
        else launch_gemv_rows(st, M.A, D.m_E, D.n_d, D.lda, x + D.n_s, rowtmp);
    }
    MDSIP_RED(k_eval_cons, std::max(D.m_E, 32 * D.m_I), D, M, x, rowtmp, d, cg, ch, 0.0, nullptr, nullptr, red(out2));
}

void VecOps::eval_cons_ax(const double *x, const double *Ax, const double *d, double *cg, double *ch,
                          double *out2, double alpha, const double *dAx, double *Ax_out) {
    MDSIP_RED(k_eval_cons, std::max(D.m_E, 32 * D.m_I), D, M, x, Ax, d, cg, ch, alpha, dAx, Ax_out, red(out2));
}

void VecOps::jac_hess(const double *x, const double *yh, double *Jdh, double *Hss, double *Hdd) {
    k_jac_hess<<<elem_grid(std::max(D.n_s, D.n_d * D.n_d)), 256, 0, st>>>(D, M, x, yh, Jdh, Hss, Hdd);
    MDSIP_LAUNCHED();
}

void VecOps::lagrangian_grad(const IterView &I, const double *grad, const double *Jdh, double *ATy,
                             double *gl) {
    if (Ahi) launch_gemv_t_df(st, Ahi, Alo, D.m_E, D.n_d, D.lda, I.yg, split, colpart, ATy);
    else launch_gemv_t(st, M.A, D.m_E, D.n_d, D.lda, I.yg, colpart, ATy);
    k_lagrangian_grad<<<elem_grid(std::max(D.n_s, (NT / 32) * D.n_d)), NT, 0, st>>>(D, M, grad, I.yg, I.yh, Jdh,
                                                                         ATy, gl);
    MDSIP_LAUNCHED();
}

void VecOps::both_products(const IterView &I, double *ATy, int *err) {
    launch_gemv_both_df(st, Ahi, Alo, D.m_E, D.n_d, D.lda, I.x + D.n_s, I.yg, split + D.m_E, split, colpart, rowtmp, ATy,
                        err, nullptr);
}
void VecOps::lagrangian_grad_aty(const IterView &I, const double *grad, const double *Jdh, const double *ATy,
                                 double *gl) {
    k_lagrangian_grad<<<elem_grid(std::max(D.n_s, (NT / 32) * D.n_d)), NT, 0, st>>>(D, M, grad, I.yg, I.yh, Jdh,
                                                                         ATy, gl);
    MDSIP_LAUNCHED();
}

void VecOps::errors(const IterView &I, const double *gl, const double *cg, const double *ch,
                    double *out7) {
    MDSIP_RED(k_errors, std::max(D.n, D.m_E), D, M, I, gl, cg, ch, red(out7));
}

void VecOps::newton_diag(const IterView &I, const double *Hss, double dw, double dc, bool want_w,
                         double *sig_x, double *q, double *sig_d, double *w, double *out6) {
    MDSIP_RED(k_newton_diag, std::max(D.n, D.m_E), D, M, I, Hss, dw, dc, want_w ? 1 : 0, sig_x, q, sig_d, w, red(out6));
}

void VecOps::rhs_y(const IterView &I, const double *gl, const double *cg, const double *q,
                   const double *w, double mu, double *bt_g, double *u) {
    k_rhs_y<<<elem_grid(D.m_E, elem_threads(D.m_E)), elem_threads(D.m_E), 0, st>>>(D, M, I, gl, cg, q, w, mu, bt_g, u);
    MDSIP_LAUNCHED();
}

void VecOps::rhs_reduced(const IterView &I, const double *gl, const double *ch, const double *sig_d,
                         const double *ATu, const double *bt_g, const double *q, double mu, double dw, bool p1,
                         double *rhs) {
    k_rhs_reduced<<<elem_grid(std::max(D.n_d, D.m_E), elem_threads(std::max(D.n_d, D.m_E))), elem_threads(std::max(D.n_d, D.m_E)), 0, st>>>(D, M, I, gl, ch, sig_d, ATu, bt_g, q,
                                                                     mu, dw, p1 ? 1 : 0, rhs);
    MDSIP_LAUNCHED();
}

void VecOps::dyg_p2(const double *Adx, const double *bt_g, const double *w, double *dyg) {
    k_dyg_p2<<<elem_grid(D.m_E), 256, 0, st>>>(D.m_E, Adx, bt_g, w, dyg);
    MDSIP_LAUNCHED();
}

void VecOps::copy(const double *src, double *dst, int64_t n) {
    if (n <= 0) return;
    k_copy<<<elem_grid(n), 256, 0, st>>>(src, dst, n);
    MDSIP_LAUNCHED();
}

void VecOps::backsub(const IterView &I, const DirView &Dir, const double *gl, const double *q,
                     const double *sig_d, const double *sol_dxd, const double *sol_dyh, double mu,
                     double dw) {
    k_backsub<<<elem_grid(D.n, elem_threads(D.n)), elem_threads(D.n), 0, st>>>(D, M, I, Dir, gl, q, sig_d, sol_dxd, sol_dyh, mu, dw);
    MDSIP_LAUNCHED();
}

void VecOps::step_scalars(const IterView &I, const DirView &Dir, const double *grad, double tau,
                          double mu, double *out3) {
    MDSIP_RED(k_step_scalars, D.n, D, M, I, Dir, grad, tau, mu, red(out3));
}

void VecOps::trial(const IterView &I, const DirView &Dir, double alpha, double *xt, double *dt,
                   double *out2) {
    MDSIP_RED(k_trial, D.n, D, M, I, Dir, alpha, xt, dt, red(out2));
}

void VecOps::accept(const IterView &I, const DirView &Dir, double alpha, double alpha_z, double mu,
                    double ks, double *ATy, const double *dATy) {
    k_accept<<<elem_grid(std::max(D.n, D.m_E), elem_threads(std::max(D.n, D.m_E))), elem_threads(std::max(D.n, D.m_E)), 0, st>>>(D, M, I, Dir, alpha, alpha_z, mu, ks, ATy, dATy);
    MDSIP_LAUNCHED();
}

void VecOps::init_x(const double *x0, double k1, double k2, const IterView &I) {
    k_init_x<<<elem_grid(std::max(D.n, D.m_E)), 256, 0, st>>>(D, M, x0, k1, k2, I);
    MDSIP_LAUNCHED();
}

void VecOps::init_d(const double *ch, double k1, double k2, const IterView &I) {
    k_init_d<<<elem_grid(D.m_I), 256, 0, st>>>(D, M, ch, k1, k2, I);
    MDSIP_LAUNCHED();
}

void VecOps::start_predicted(const float *pred, double push, double mu0, const IterView &I) {
    k_start_predicted<<<elem_grid(std::max(D.n, D.m_E)), 256, 0, st>>>(D, M, pred, push, mu0, I);
    MDSIP_LAUNCHED();
}

void VecOps::cons_from_values(const double *g, const double *h, const double *d, double *cg, double *ch,
                              double *out2) {
    k_cons_from_values<<<red_grid(D.m_E), NT, 0, st>>>(D, M, g, h, d, cg, ch, red(out2));
    MDSIP_LAUNCHED();
}

void VecOps::dir_diff(const DirView &a, const DirView &b, double *out2) {
    k_dir_diff<<<red_grid(D.n), NT, 0, st>>>(D, a, b, red(out2));
    MDSIP_LAUNCHED();
}

void VecOps::copy_dir(const DirView &src, const DirView &dst) {
    copy(src.dx, dst.dx, D.n);
    copy(src.dd, dst.dd, D.m_I);
    copy(src.dyg, dst.dyg, D.m_E);
    copy(src.dyh, dst.dyh, D.m_I);
    copy(src.dzl, dst.dzl, D.n);
    copy(src.dzu, dst.dzu, D.n);
    copy(src.dvl, dst.dvl, D.m_I);
    copy(src.dvu, dst.dvu, D.m_I);
}

void VecOps::gather(int64_t n, const double *src, const int32_t *idx, double *dst) {
    if (n <= 0) return;
    k_gather<<<elem_grid(n), 256, 0, st>>>(n, src, idx, dst);
    MDSIP_LAUNCHED();
}

}  // namespace mdsip
