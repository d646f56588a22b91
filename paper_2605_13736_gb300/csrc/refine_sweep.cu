// One sweep of the iterative refinement in one read of A (path P2, FP32 tiles
// of a tensor-core factor, n_d <= 4096).
//
// A sweep solves S~ sol = rhs, completes the correction on the eliminated rows
// and columns, adds it to u and forms the residual b - K u and the first half
// of the next approximate solve.  Written out per equality row i (P2: every
// sparse column has at most one row, so all of it is the row's own):
//
//   sol_g,i = ((A_hi sol_d)_i - bt_i) / w_i          FP32 row product
//   u_g,i += sol_g,i
//   u_c   += (r_c - J_ic sol_g,i) / q_c              the row's sparse columns c
//   (A u_d)_i                                        double-float row product
//   bt_i   = b_i + dc u_g,i - sum J_ic u_c - sum J_ic (b_c - q_c u_c - J_ic u_g,i) / q_c - (A u_d)_i
//   A^T u_g                                          double-float column product
//   A_hi^T (bt / w)                                  FP32 column product
//
// Both row products need only sol_d and u_d, known before the pass; both
// column products need the row's own results.  So a batch of rows stays in
// shared memory between its two halves and A_hi, A_lo are read once a sweep, 8
// bytes per entry (12 in the separate passes, with ten small launches more
// around them).  A sweep's passes at m = 100000, n = 2000: 361 + 164 us apart,
// 358 in one; m = 200000, n = 4000: 1275 + 800 + 498 apart, 1360; m = 25600,
// n = 512: 78 + 23 apart, 35.
#include "df.cuh"
#include "internal.cuh"
#include "refine.cuh"
#include "tc.cuh"

namespace mdsip {

namespace {

constexpr int NT = kRedThreads;
constexpr int kSwC = 512;                     // column threads: 16 warps
constexpr int kSwThreads = 640;               // 20 warps, five a sub-partition: 96 registers a thread
constexpr int kSwMaxSlots = 12;
constexpr int KBR = 2;                        // rows of a group in a batch
constexpr size_t kSwSmem = 224 * 1024;        // batches in flight or in use
constexpr size_t kSwMin = 48 * 1024;          // the groups' column sums meet in the ring at the end

struct SweepArgs {
    const float *Ahi, *Alo;
    int64_t m, lda;
    int n, T, S;           // columns, threads per row, batches of the ring
    const float4 *xq;      // per column: u_d split (x, y), fl32(sol_d) (z)
    const double *b_g, *winv;
    const float *wf;
    double *u_g, *bt, *sol_g, *Au;
    double dc;
    const int *csr_ptr, *csr_col;
    const double *csr_val, *b_s, *u_s, *r_s, *q, *qinv;
    int init;              // u = 0 and r = b before this sweep
    double *pu;            // partial sums of A^T u_g, a row per CTA and group (the CTA's in its first)
    float *pv;             // and of A_hi^T (bt / w), a row per CTA
    int *err;
};

// the sparse column's new u_s: the same bits wherever it is formed
__device__ __forceinline__ double new_us(double u, double r, double J, double sol, double qinv) {
    return fma(fma(-J, sol, r), qinv, u);
}

// v = hi + lo to 2^-49, hi to nearest: on the bits for ordinary magnitudes (four
// FP64 conversions and a subtraction otherwise, 64 cycles each)
__device__ __forceinline__ float2 split64(double v) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e < 1023 - 60 || e > 1023 + 100) {
        const float h = (float)v;
        return make_float2(h, (float)(v - (double)h));
    }
    const long long t = (b + 0x10000000LL) & ~0x1fffffffLL;   // the magnitude's upper 24 bits, rounded
    const unsigned sg = (unsigned)(b >> 32) & 0x80000000u;
    const unsigned hi = sg | ((unsigned)(((t & 0x7fffffffffffffffLL) >> 29) - (896LL << 23)));
    const float lo = (float)(int)(b - t) * __uint_as_float(sg | (unsigned)((e - 948) << 23));
    return make_float2(__uint_as_float(hi), lo);
}

// Warps 0 .. 15 compute, warp 16 loads, warps 17 .. 19 finish rows in turn
// (batch b by warp 17 + b mod 3).  T threads (32 .. 512) take a row's columns,
// 4 CH each; the 512 / T groups take KBR rows of a batch each, so a batch is
// 32 (CH = 1) or 64 KB at any width and comes as one bulk copy of A_hi and one
// of A_lo (the rows are contiguous).  Per batch: row products, warp sums to
// shared memory, the finishing warp's scalars in FP64 (some 20 instructions of
// 64 cycles, its gathers a turn ahead), and kLag batches later, with the
// finished rows, the column products.  Only mbarriers; waits are bounded.
// What bounds it is the double-float arithmetic's dependent chains with the
// five warps a sub-partition holds: the FP32 pipe is 49% busy, HBM at 4.7 of
// 6.9 TB/s at n = 4000.  Eight columns and two rows a thread (CH = KBR = 2)
// spread the row sums' shuffles over the most products: m = 100000, n = 2000
// 358 us, with four columns and three batches of lag (whose row and column
// parts interleave) 385, summing the rows in the finishing warps 377; m =
// 200000, n = 4000 1360 us, with one row a batch 1770.
template <int CH, int kLag>
__global__ void __launch_bounds__(kSwThreads, 1) k_sweep(SweepArgs a) {
    extern __shared__ __align__(128) unsigned char sw_smem[];
    constexpr int kVals = KBR * 16;            // (row, warp) sums of a batch: one a lane of the finishing warp
    __shared__ float4 s_y[3][kVals];
    __shared__ float2 s_red[3][kVals];
    __shared__ float s_red2[3][kVals];
    __shared__ __align__(8) uint64_t full[kSwMaxSlots], empty[kSwMaxSlots], rowdone[3], rowready[3];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int T = a.T, W = T / 32, G = kSwC / T, RB = G * KBR, S = a.S;
    const int lda = (int)a.lda;
    const uint32_t slot_bytes = 2u * RB * lda * (uint32_t)sizeof(float);
    const int64_t rows_per = (a.m + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = (int64_t)blockIdx.x * rows_per;
    const int nrow = (int)max((int64_t)0, min(a.m - r0, rows_per));
    const int nbat = (nrow + RB - 1) / RB;
    if (tid == 0) {
        for (int i = 0; i < S; ++i) {
            tc::mbar_init(&full[i], 1);
            tc::mbar_init(&empty[i], 16);
        }
        for (int i = 0; i < 3; ++i) {
            tc::mbar_init(&rowdone[i], 16);
            tc::mbar_init(&rowready[i], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    bool ok = true;
    if (wid < 16) {
        const int g = tid / T, t = tid - g * T;
        float2 xh[2 * CH], xl[2 * CH], xs[2 * CH];
        bool on[CH];
#pragma unroll
        for (int ch = 0; ch < CH; ++ch) {
            const int p0 = 4 * t + ch * 4 * T;
            on[ch] = p0 < a.n;
            float4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = p0 + q < a.n ? __ldg(a.xq + p0 + q) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                xh[2 * ch + h] = make_float2(v[2 * h].x, v[2 * h + 1].x);
                xl[2 * ch + h] = make_float2(v[2 * h].y, v[2 * h + 1].y);
                xs[2 * ch + h] = make_float2(v[2 * h].z, v[2 * h + 1].z);
            }
        }
        // column sums: a double-float pair per 16 rows, added into a second pair,
        // which goes into FP64 every 256 rows (the FP64 pipe: 1/64 of the FP32 rate)
        const float2 z2 = make_float2(0.0f, 0.0f);
        float2 cs[2 * CH], cc[2 * CH], CS[2 * CH], CC[2 * CH], cv[2 * CH];
        bool flushed = false;
#pragma unroll
        for (int j = 0; j < 2 * CH; ++j) cs[j] = cc[j] = CS[j] = CC[j] = cv[j] = z2;
        int cnt = 0, cnt2 = 0;
        int rslot = 0, cslot = 0, rb = 0, cb = 0;   // ring slots, result buffers (b mod 3) of the two halves
        uint32_t rph = 0, cph = 0;
        const uint32_t off = (uint32_t)(g * KBR * lda) * (uint32_t)sizeof(float), lo_off = (uint32_t)(RB * lda) * 4u;
        // columns beyond n read the row's first ones: x is zero there, their sums are not stored
        uint32_t coff[CH];
#pragma unroll
        for (int ch = 0; ch < CH; ++ch) coff[ch] = on[ch] ? (uint32_t)(4 * t + ch * 4 * T) * 4u : 0u;
        float2 ps[KBR][CH], pc[KBR][CH], p2[KBR];
        auto row_part = [&](const unsigned char *base, int k) {
            p2[k] = z2;
#pragma unroll
            for (int ch = 0; ch < CH; ++ch) {
                const unsigned char *at = base + (uint32_t)(k * lda) * 4u + coff[ch];
                const float4 ah = *reinterpret_cast<const float4 *>(at);
                const float4 al = *reinterpret_cast<const float4 *>(at + lo_off);
                const float2 h0 = make_float2(ah.x, ah.y), h1 = make_float2(ah.z, ah.w);
                ps[k][ch] = pc[k][ch] = z2;
                df_acc2(h0, make_float2(al.x, al.y), xh[2 * ch], xl[2 * ch], ps[k][ch], pc[k][ch]);
                df_acc2(h1, make_float2(al.z, al.w), xh[2 * ch + 1], xl[2 * ch + 1], ps[k][ch], pc[k][ch]);
                p2[k] = __ffma2_rn(h0, xs[2 * ch], p2[k]);
                p2[k] = __ffma2_rn(h1, xs[2 * ch + 1], p2[k]);
            }
        };
        auto col_part = [&](const unsigned char *base, int k, float4 y) {
            const float2 yh = make_float2(y.x, y.x), yl = make_float2(y.y, y.y), yv = make_float2(y.z, y.z);
#pragma unroll
            for (int ch = 0; ch < CH; ++ch) {
                const unsigned char *at = base + (uint32_t)(k * lda) * 4u + coff[ch];
                const float4 ah = *reinterpret_cast<const float4 *>(at);
                const float4 al = *reinterpret_cast<const float4 *>(at + lo_off);
                const float2 h0 = make_float2(ah.x, ah.y), h1 = make_float2(ah.z, ah.w);
                df_acc2(h0, make_float2(al.x, al.y), yh, yl, cs[2 * ch], cc[2 * ch]);
                df_acc2(h1, make_float2(al.z, al.w), yh, yl, cs[2 * ch + 1], cc[2 * ch + 1]);
                cv[2 * ch] = __ffma2_rn(h0, yv, cv[2 * ch]);
                cv[2 * ch + 1] = __ffma2_rn(h1, yv, cv[2 * ch + 1]);
            }
        };
        for (int b = 0; b < nbat + kLag; ++b) {
            if (!__all_sync(0xffffffffu, ok)) break;   // a wait ran out: the whole warp stops
            if (b < nbat && !tc::mbar_wait(&full[rslot], rph)) ok = false;
            if (kLag > 1 && b >= kLag && !tc::mbar_wait(&rowready[cb], cph)) ok = false;
            const unsigned char *rbase = sw_smem + rslot * slot_bytes + off;
            const unsigned char *cbase = sw_smem + cslot * slot_bytes + off;
            auto rows = [&]() {
#pragma unroll
                for (int k = 0; k < KBR; ++k) {
                    if (b * RB + g * KBR + k < nrow) {
                        row_part(rbase, k);
                    } else {
                        p2[k] = z2;
#pragma unroll
                        for (int ch = 0; ch < CH; ++ch) ps[k][ch] = pc[k][ch] = z2;
                    }
                }
            };
            auto cols = [&]() {
#pragma unroll
                for (int k = 0; k < KBR; ++k)
                    if ((b - kLag) * RB + g * KBR + k < nrow) col_part(cbase, k, s_y[cb][g * KBR + k]);
            };
            auto release = [&]() {
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&empty[cslot]);
                if (++cslot == S) cslot = 0;
                if (++cb == 3) cb = 0, cph ^= 1;
            };
            if (kLag > 1 && b >= kLag && (b + 1) * RB <= nrow) {   // whole batches: both parts in one stream of instructions
#pragma unroll
                for (int k = 0; k < KBR; ++k) {
                    row_part(rbase, k);
                    col_part(cbase, k, s_y[cb][g * KBR + k]);
                }
            } else {
                rows();
                if (kLag > 1 && b >= kLag) cols();
            }
            if (kLag > 1 && b >= kLag) release();
            if (b < nbat) {   // ---- the rows' sums over the warp: two rows exchange halves, then a butterfly
                float rs[KBR], rc[KBR], r2[KBR];
#pragma unroll
                for (int k = 0; k < KBR; ++k) {
                    float2 s = ps[k][0], c = pc[k][0];
#pragma unroll
                    for (int ch = 1; ch < CH; ++ch) {
                        df_add(s.x, c.x, ps[k][ch].x, pc[k][ch].x);
                        df_add(s.y, c.y, ps[k][ch].y, pc[k][ch].y);
                    }
                    df_add(s.x, c.x, s.y, c.y);
                    rs[k] = s.x;
                    rc[k] = c.x;
                    r2[k] = p2[k].x + p2[k].y;
                }
                if (++rslot == S) rslot = 0, rph ^= 1;
                float s = rs[0], c = rc[0], d = r2[0];
                const bool up = (lane & 16) != 0;
                const int row = g * KBR + (up ? 1 : 0);
                float es = up ? s : rs[1], ec = up ? c : rc[1], ed = up ? d : r2[1];
                s = up ? rs[1] : s;
                c = up ? rc[1] : c;
                d = up ? r2[1] : d;
                es = __shfl_xor_sync(0xffffffffu, es, 16);
                ec = __shfl_xor_sync(0xffffffffu, ec, 16);
                d += __shfl_xor_sync(0xffffffffu, ed, 16);
                df_add(s, c, es, ec);
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) {
                    es = __shfl_xor_sync(0xffffffffu, s, o);
                    ec = __shfl_xor_sync(0xffffffffu, c, o);
                    d += __shfl_xor_sync(0xffffffffu, d, o);
                    df_add(s, c, es, ec);
                }
                if ((lane & 15) == 0) {
                    s_red[rb][row * W + (t >> 5)] = make_float2(s, c);
                    s_red2[rb][row * W + (t >> 5)] = d;
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&rowdone[rb]);
                if (++rb == 3) rb = 0;
            }
            if (b < kLag) continue;
            if (kLag == 1) {
                if (!tc::mbar_wait(&rowready[cb], cph)) ok = false;
                cols();
                release();
            }
            if (++cnt == 16 / KBR) {   // every 16 rows
                cnt = 0;
#pragma unroll
                for (int j = 0; j < 2 * CH; ++j) {
                    df_add(CS[j].x, CC[j].x, cs[j].x, cc[j].x);
                    df_add(CS[j].y, CC[j].y, cs[j].y, cc[j].y);
                    cs[j] = cc[j] = z2;
                }
                if (++cnt2 == 16) {   // every 256 rows
                    cnt2 = 0;
                    // this group's row of sums, its own until the end
#pragma unroll
                    for (int q = 0; q < 4 * CH; ++q) {
                        const int p = 4 * t + (q >> 2) * 4 * T + (q & 3);
                        const float2 A = CS[q >> 1], B = CC[q >> 1];
                        const double v = (double)(q & 1 ? A.y : A.x) + (double)(q & 1 ? B.y : B.x);
                        double *at = a.pu + ((size_t)blockIdx.x * G + g) * a.n + p;
                        if (p < a.n) *at = flushed ? *at + v : v;
                    }
                    flushed = true;
#pragma unroll
                    for (int j = 0; j < 2 * CH; ++j) CS[j] = CC[j] = z2;
                }
            }
        }
        if (!ok) atomicExch(a.err, 1);
#pragma unroll
        for (int j = 0; j < 2 * CH; ++j) {
            df_add(CS[j].x, CC[j].x, cs[j].x, cc[j].x);
            df_add(CS[j].y, CC[j].y, cs[j].y, cc[j].y);
        }
        if (G > 1) {   // the groups' sums meet in shared memory, group 0 adds them up in order
            asm volatile("bar.sync 1, 512;" ::: "memory");   // every warp is through with the ring
            float4 *gp = reinterpret_cast<float4 *>(sw_smem);            // [2 CH][512]: pairs of columns
            float4 *gv = gp + 2 * CH * kSwC;                             // [CH][512]
#pragma unroll
            for (int j = 0; j < 2 * CH; ++j) gp[j * kSwC + tid] = make_float4(CS[j].x, CC[j].x, CS[j].y, CC[j].y);
#pragma unroll
            for (int ch = 0; ch < CH; ++ch)
                gv[ch * kSwC + tid] = make_float4(cv[2 * ch].x, cv[2 * ch].y, cv[2 * ch + 1].x, cv[2 * ch + 1].y);
            asm volatile("bar.sync 1, 512;" ::: "memory");
            if (g == 0)
                for (int x = 1; x < G; ++x) {
                    const int o = x * T + t;
#pragma unroll
                    for (int j = 0; j < 2 * CH; ++j) {
                        const float4 v = gp[j * kSwC + o];
                        df_add(CS[j].x, CC[j].x, v.x, v.y);
                        df_add(CS[j].y, CC[j].y, v.z, v.w);
                    }
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch) {
                        const float4 v = gv[ch * kSwC + o];
                        cv[2 * ch] = make_float2(cv[2 * ch].x + v.x, cv[2 * ch].y + v.y);
                        cv[2 * ch + 1] = make_float2(cv[2 * ch + 1].x + v.z, cv[2 * ch + 1].y + v.w);
                    }
                }
        }
        if (g == 0)
#pragma unroll
            for (int q = 0; q < 4 * CH; ++q) {
                const int p = 4 * t + (q >> 2) * 4 * T + (q & 3);
                if (p >= a.n) continue;
                const float2 A = CS[q >> 1], B = CC[q >> 1], V = cv[q >> 1];
                double v = (double)(q & 1 ? A.y : A.x) + (double)(q & 1 ? B.y : B.x);
                double *at = a.pu + (size_t)blockIdx.x * G * a.n + p;
                if (flushed)
                    for (int x = 0; x < G; ++x) v += at[(size_t)x * a.n];
                *at = v;
                a.pv[(size_t)blockIdx.x * a.n + p] = q & 1 ? V.y : V.x;
            }
    } else if (wid == 16) {
        // ---- loads
        int slot = 0;
        uint32_t ph = 1;   // of the slot's previous use
        int b = 0;
        for (; b < nbat; ++b) {
            if (b >= S) ok = __all_sync(0xffffffffu, tc::mbar_wait(&empty[slot], ph));
            if (!ok) break;
            const uint32_t bytes = (uint32_t)(min(RB, nrow - b * RB) * lda) * (uint32_t)sizeof(float);
            if (lane == 0) tc::mbar_expect_tx(&full[slot], 2 * bytes);
            __syncwarp();
            if (lane < 2)
                tc::bulk_load(sw_smem + slot * slot_bytes + lane * (slot_bytes / 2),
                              (lane ? a.Alo : a.Ahi) + (r0 + (int64_t)b * RB) * lda, bytes, &full[slot]);
            if (++slot == S) slot = 0, ph ^= 1;
        }
        if (!ok && lane == 0) atomicExch(a.err, 1);
        // no copy is in flight when the CTA leaves
        for (int x = max(0, b - S); x < b; ++x) tc::mbar_wait(&full[x % S], (uint32_t)(x / S) & 1);
    } else {
        // ---- finishing warps: lane = (row, warp sum)
        const int me = wid - 17, rho = lane / W, sub = lane - rho * W;
        static_assert(kVals == 32, "a lane a sum");
        const bool lead = sub == 0;
        uint32_t ph = 0;
        int e0 = 0, e1 = 0;
        auto rows_entries = [&](int b) {   // the row's entries, loaded a turn ahead
            const int x = b * RB + rho;
            const bool live = x < nrow && b < nbat;
            e0 = live ? __ldg(a.csr_ptr + r0 + x) : 0;
            e1 = live ? __ldg(a.csr_ptr + r0 + x + 1) : 0;
        };
        rows_entries(me);
        for (int b = me; b < nbat; b += 3) {
            const bool live = b * RB + rho < nrow;
            const int64_t i = r0 + b * RB + rho;
            double ug = 0.0, bt = 0.0, winv = 0.0, bg = 0.0;
            float wf = 0.0f;
            // the row's sparse entries over its lanes; the first one's data now
            const int f0 = e0 + sub, f1 = e1, most = __reduce_max_sync(0xffffffffu, e1 - e0);
            double J = 0.0, bc = 0.0, uc = 0.0, rcv = 0.0, q = 0.0, qi = 0.0;
            auto entry = [&](int e) {
                const int cidx = __ldg(a.csr_col + e);
                J = __ldg(a.csr_val + e);
                bc = __ldg(a.b_s + cidx);
                q = __ldg(a.q + cidx);
                qi = __ldg(a.qinv + cidx);
                uc = a.init ? 0.0 : __ldg(a.u_s + cidx);
                rcv = a.init ? bc : __ldg(a.r_s + cidx);
            };
            if (f0 < f1) entry(f0);
            if (live) {
                bg = __ldg(a.b_g + i);
                winv = __ldg(a.winv + i);
                wf = __ldg(a.wf + i);
                bt = a.bt[i];
                ug = a.init ? 0.0 : a.u_g[i];
            }
            rows_entries(b + 3);
            ok = __all_sync(0xffffffffu, tc::mbar_wait(&rowdone[me], ph));
            if (!ok) break;
            ph ^= 1;
            float s = s_red[me][lane].x, c = s_red[me][lane].y, d = s_red2[me][lane];
            for (int o = 1; o < W; o <<= 1) {
                const float es = __shfl_xor_sync(0xffffffffu, s, o), ec = __shfl_xor_sync(0xffffffffu, c, o);
                d += __shfl_xor_sync(0xffffffffu, d, o);
                df_add(s, c, es, ec);
            }
            const double sol = ((double)d - bt) * winv;
            const double un = ug + sol;
            double part = 0.0;
            for (int e = f0; e < f1; e += W) {
                if (e != f0) entry(e);
                const double us = new_us(uc, rcv, J, sol, qi);
                const double rs = bc - fma(J, un, q * us);
                part = fma(-J, us, part);
                part = fma(-(J * qi), rs, part);
            }
            for (int o = 1; o < W && o < most; o <<= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
            const double Au = (double)s + (double)c;
            const double btn = (fma(a.dc, un, bg) + part) - Au;
            if (lead) {
                const float2 y = split64(un);
                s_y[me][rho] = make_float4(y.x, y.y, (float)btn * wf, 0.0f);
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&rowready[me]);
            if (lead && live) {
                a.u_g[i] = un;
                a.sol_g[i] = sol;
                a.bt[i] = btn;
                a.Au[i] = Au;
            }
        }
        if (!ok && lane == 0) atomicExch(a.err, 1);
    }
}

// bt = b_g - J_sg (b_s / q), u = fl32(bt / w) padded to ldt (first approximate solve); 1 / w
// in FP64 and FP32, 1 / q; the inequalities' part of the first right-hand side
__global__ void k_sweep_start(Dims D, ModelView M, const double *__restrict__ b, const double *__restrict__ q,
                              const double *__restrict__ w, double *__restrict__ bt, float *__restrict__ u,
                              double *__restrict__ winv, float *__restrict__ wf, double *__restrict__ qinv,
                              int64_t ldt, double *__restrict__ rhsS) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, gsz = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = gtid; i < D.m_E; i += gsz) {
        double s = b[D.n + i];
        for (int e = M.csr_ptr[i]; e < M.csr_ptr[i + 1]; ++e) {
            const int c = M.csr_col[e];
            s -= ddiv(M.csr_val[e] * b[c], q[c]);
        }
        bt[i] = s;
        u[i] = (float)ddiv(s, w[i]);
        const double r = ddiv(1.0, w[i]);
        winv[i] = r;
        wf[i] = (float)r;
    }
    for (int64_t i = D.m_E + gtid; i < ldt; i += gsz) u[i] = 0.0f;
    for (int64_t k = gtid; k < D.n_s; k += gsz) qinv[k] = ddiv(1.0, q[k]);
    for (int64_t j = gtid; j < D.m_I; j += gsz) rhsS[D.n_d + j] = b[D.n + D.m_E + j];
}

// x = u_d + sol_d, u_h + sol_h into xnew, x and sol_d as FP32 parts, and
// Hu = [H_dd; J_dh] x, a warp per row with x in shared memory
__global__ void __launch_bounds__(NT) k_sweep_x(int64_t n_d, int64_t m_I, const double *__restrict__ Hdd,
                                                const double *__restrict__ Jdh, const double *__restrict__ ud,
                                                const double *__restrict__ uh, const double *__restrict__ sol, int init,
                                                float4 *__restrict__ xq, double *__restrict__ xnew,
                                                double *__restrict__ Hu) {
    extern __shared__ double xsh[];
    for (int64_t k = threadIdx.x; k < n_d; k += NT) {
        const double d = sol[k], x = init ? d : ud[k] + d;
        xsh[k] = x;
        if (k / NT == blockIdx.x) {   // the grid has a block per NT columns at least
            const float h = (float)x;
            xq[k] = make_float4(h, (float)(x - (double)h), (float)d, 0.0f);
            xnew[k] = x;
        }
    }
    for (int64_t j = (int64_t)blockIdx.x * NT + threadIdx.x; j < m_I; j += (int64_t)gridDim.x * NT)
        xnew[n_d + j] = init ? sol[n_d + j] : uh[j] + sol[n_d + j];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int64_t p = (int64_t)blockIdx.x * (NT / 32) + (threadIdx.x >> 5); p < n_d + m_I; p += (int64_t)gridDim.x * (NT / 32)) {
        const double *row = p < n_d ? Hdd + p * n_d : Jdh + (p - n_d) * n_d;
        double s0 = 0.0, s1 = 0.0;
        int64_t k = lane;
        for (; k + 96 < n_d; k += 128) {
            const double a0 = __ldg(row + k), a1 = __ldg(row + k + 32), a2 = __ldg(row + k + 64), a3 = __ldg(row + k + 96);
            s0 = fma(a0, xsh[k], s0);
            s1 = fma(a1, xsh[k + 32], s1);
            s0 = fma(a2, xsh[k + 64], s0);
            s1 = fma(a3, xsh[k + 96], s1);
        }
        for (; k < n_d; k += 32) s0 = fma(row[k], xsh[k], s0);
        double s = s0 + s1;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) Hu[p] = s;
    }
}

// The rest of the sweep: u_s, u_d, u_h, the residual r = b - K u with its norms
// (||r||, ||b||, ||K u||, ||u|| in the maximum norm), A^T u_g and the next
// right-hand side of the reduced system from the CTAs' partial column sums.
__global__ void __launch_bounds__(NT) k_sweep_residual(
    Dims D, ModelView M, const double *__restrict__ b, double *__restrict__ u, double *__restrict__ r,
    const double *__restrict__ q, const double *__restrict__ qinv, const double *__restrict__ sig_xd,
    const double *__restrict__ sig_d, const double *__restrict__ Jdh, const double *__restrict__ Au,
    const double *__restrict__ sol_g, const double *__restrict__ Hu, const double *__restrict__ xnew,
    const double *__restrict__ pu, const float *__restrict__ pv, int nparts, int pstep, int init, double dw, double dc,
    double *__restrict__ ATu, double *__restrict__ rhsS, RedOut red) {
    __shared__ double su[NT / 32][8], sj[NT / 32][8];
    __shared__ float2 sv[NT / 32][8];
    unsigned long long rm = 0, bm = 0, km = 0, um = 0;
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x, gsz = (int64_t)gridDim.x * NT;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    auto put = [&](int64_t idx, double Ku, double ui) -> double {
        const double bi = b[idx], ri = bi - Ku;
        r[idx] = ri;
        max_abs(rm, ri);
        max_abs(bm, bi);
        max_abs(km, Ku);
        max_abs(um, ui);
        return ri;
    };
    // eight dense columns per block at a time: 32 threads share a column's partial
    // sums (five rows each for 152 CTAs) and its part of J_dh^T u_h
    for (int64_t k0 = (int64_t)blockIdx.x * 8; k0 < D.n_d; k0 += (int64_t)gridDim.x * 8) {
        const int64_t k = k0 + (threadIdx.x & 7);
        double s = 0.0, jt = 0.0;
        float vs = 0.0f, vc = 0.0f;
        if (k < D.n_d) {
#pragma unroll 4
            for (int p = threadIdx.x >> 3; p < nparts; p += NT / 8) {
                s += pu[(size_t)p * pstep * D.n_d + k];
                df_add(vs, vc, pv[(size_t)p * D.n_d + k], 0.0f);
            }
            for (int64_t j = threadIdx.x >> 3; j < D.m_I; j += NT / 8) jt = fma(Jdh[j * D.n_d + k], xnew[D.n_d + j], jt);
        }
#pragma unroll
        for (int o = 8; o < 32; o <<= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            jt += __shfl_xor_sync(0xffffffffu, jt, o);
            const float es = __shfl_xor_sync(0xffffffffu, vs, o), ec = __shfl_xor_sync(0xffffffffu, vc, o);
            df_add(vs, vc, es, ec);
        }
        __syncthreads();   // an earlier group's sums are read
        if (lane < 8) {
            su[wid][lane] = s;
            sj[wid][lane] = jt;
            sv[wid][lane] = make_float2(vs, vc);
        }
        __syncthreads();
        if (threadIdx.x < 8 && k < D.n_d) {
#pragma unroll
            for (int x = 1; x < NT / 32; ++x) {
                s += su[x][lane];
                jt += sj[x][lane];
                df_add(vs, vc, sv[x][lane].x, sv[x][lane].y);
            }
            const double x = xnew[k];
            ATu[k] = s;
            u[D.n_s + k] = x;
            const double ri = put(D.n_s + k, Hu[k] + (sig_xd[k] + dw) * x + s + jt, x);
            rhsS[k] = ri + ((double)vs + (double)vc);
        }
    }
    // equality rows with their sparse columns
    for (int64_t i = gtid; i < D.m_E; i += gsz) {
        const double ug = u[D.n + i], sol = sol_g[i];
        double Kg = Au[i] - dc * ug;
        for (int e = M.csr_ptr[i]; e < M.csr_ptr[i + 1]; ++e) {
            const int c = M.csr_col[e];
            const double J = M.csr_val[e];
            const double us = new_us(init ? 0.0 : u[c], init ? b[c] : r[c], J, sol, qinv[c]);
            u[c] = us;
            put(c, fma(J, ug, q[c] * us), us);
            Kg = fma(J, us, Kg);
        }
        put(D.n + i, Kg, ug);
    }
    for (int64_t k = gtid; k < D.n_s; k += gsz)
        if (M.csc_ptr[k] == M.csc_ptr[k + 1]) {   // a sparse variable of no equality row
            const double us = new_us(init ? 0.0 : u[k], init ? b[k] : r[k], 0.0, 0.0, qinv[k]);
            u[k] = us;
            put(k, q[k] * us, us);
        }
    for (int64_t j = gtid; j < D.m_I; j += gsz) {
        const double uh = xnew[D.n_d + j];
        u[D.n + D.m_E + j] = uh;
        rhsS[D.n_d + j] = put(D.n + D.m_E + j, Hu[D.n_d + j] - (ddiv(1.0, sig_d[j] + dw) + dc) * uh, uh);
    }
    double v[4] = {__longlong_as_double((long long)rm), __longlong_as_double((long long)bm),
                   __longlong_as_double((long long)km), __longlong_as_double((long long)um)};
    reduce_finish<NT, R_MAX, R_MAX, R_MAX, R_MAX>(v, red);
}

int grid_for(int64_t n) { return std::max(1, std::min(4096, ceil_div(std::max<int64_t>(n, 1), 256))); }

struct SweepParts {
    int n, step;       // rows of partial sums, and their distance in rows
    const float *pv;
};

template <int CH, int kLag>
SweepParts launch_sweep_t(cudaStream_t st, int num_sms, SweepArgs a) {
    a.T = 32;
    while (a.T < kSwC && 4 * CH * a.T < a.n) a.T *= 2;
    const int RB = kSwC / a.T * KBR;
    const size_t slot = (size_t)2 * RB * a.lda * sizeof(float);
    a.S = (int)std::min<size_t>(kSwMaxSlots, kSwSmem / slot);
    MDSIP_REQUIRE(a.S > kLag + 1, MDSIP_ERR_INVALID_ARG, "refinement sweep: rows too long");
    // two batches a CTA where there are few: as fast alone, and half the SMs for the other
    // instances of a batch (24 at once 70.5 -> 68.8 ms)
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(num_sms, kRedBlocks / 2), ceil_div(a.m, (int64_t)2 * RB)));
    const size_t groups = (size_t)(kSwC / a.T);
    a.pv = reinterpret_cast<float *>(a.pu + grid * groups * a.n);
    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_sweep<CH, kLag>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSwSmem);
    }));
    k_sweep<CH, kLag><<<grid, kSwThreads, std::max(kSwMin, a.S * slot), st>>>(a);
    MDSIP_LAUNCHED();
    return SweepParts{grid, (int)groups, a.pv};
}

}  // namespace

// doubles of Refiner::colpart that a sweep's partial sums take
int64_t refine_sweep_parts(int64_t n) { return kRedBlocks / 2 * std::max<int64_t>(8192, 2 * n); }

// FP32 tiles of a tensor-core factor with the FP32 pair of A; above 4096
// columns a batch and its predecessor no longer fit the shared memory together
// (the separate passes of refine.cu take those)
bool Refiner::sweep_path() const { return xq && Ahi && solve_fp32 && AfT && D.n_d > 0 && D.n_d <= 4096; }

void Refiner::sweep_start(const double *b) {
    k_sweep_start<<<grid_for(std::max(D.m_E, D.n_s)), 256, 0, st>>>(D, M, b, q, w, bt, vf, winv, wf, qinv, ldt, rhsS);
    MDSIP_LAUNCHED();
    launch_aft_dot_add(st, num_sms, AfT, ldt, D.n_d, vf, b + D.n_s, rhsS);   // b_d + A_hi^T u
}

void Refiner::sweep(const double *b, double *u, double *r, bool init, double dw, double dc, double *out4) {
    launch_ldlt_solve_coop(st, num_sms, N, Dd, Doff, perm, 1, rhsS, N, solve_ws, solve_err, solve_fp32);
    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_sweep_x, cudaFuncAttributeMaxDynamicSharedMemorySize, 4096 * (int)sizeof(double));
    }));
    k_sweep_x<<<std::max(1, std::min(4096, ceil_div(D.n_d + D.m_I, NT / 32))), NT, D.n_d * sizeof(double), st>>>(
        D.n_d, D.m_I, Hdd, Jdh, u + D.n_s, u + D.n + D.m_E, rhsS, init ? 1 : 0, xq, xnew, tmp_nd2);
    MDSIP_LAUNCHED();
    SweepArgs a{};
    a.Ahi = Ahi;
    a.Alo = Alo;
    a.m = D.m_E;
    a.lda = D.lda;
    a.n = (int)D.n_d;
    a.xq = xq;
    a.b_g = b + D.n;
    a.winv = winv;
    a.wf = wf;
    a.u_g = u + D.n;
    a.bt = bt;
    a.sol_g = sol_g;
    a.Au = tmp_m;
    a.dc = dc;
    a.csr_ptr = M.csr_ptr;
    a.csr_col = M.csr_col;
    a.csr_val = M.csr_val;
    a.b_s = b;
    a.u_s = u;
    a.r_s = r;
    a.q = q;
    a.qinv = qinv;
    a.init = init ? 1 : 0;
    a.pu = colpart;
    a.err = solve_err;
    // up to 128 columns a warp of four columns a thread holds a row; wider rows go by eight
    const SweepParts pt = D.n_d <= 128 ? launch_sweep_t<1, 3>(st, num_sms, a) : launch_sweep_t<2, 1>(st, num_sms, a);
    k_sweep_residual<<<red_grid(std::max(std::max(D.n_s, D.m_E), 32 * D.n_d)), NT, 0, st>>>(
        D, M, b, u, r, q, qinv, sig_xd, sig_d, Jdh, tmp_m, sol_g, tmp_nd2, xnew, colpart,
        pt.pv, pt.n, pt.step, init ? 1 : 0, dw, dc, tmp_nd, rhsS,
        RedOut{partial, reinterpret_cast<unsigned *>(partial + kRedBlocks * 8), out4});
    MDSIP_LAUNCHED();
}

}  // namespace mdsip
