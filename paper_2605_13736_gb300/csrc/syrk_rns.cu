// FP64 condensation product on the BF16 tensor cores through residue numbers:
//
//     C[p][q] = beta C[p][q] + sum_i A[i][p] A[i][q] / w_i       (p >= q)
//
// GB300 multiplies FP64 on the SIMT pipe at 1.26 TFLOP/s and BF16 on tcgen05
// at about 1.9 PFLOP/s, so an exact integer product built from 14 BF16
// contractions beats the DFMA kernel by more than an order of magnitude
// wherever the product is large enough to pay for its passes.
//
// For a chunk of rows the scaled entry s_ip = a_ip w_i^-1/2 is rounded once to
// an integer X_ip of at most b bits (b = 53 .. 56) relative to the largest entry
// of its column in the chunk; the integer sums sum_i X_ip X_iq are then formed
// exactly: residues of X modulo 14 pairwise coprime moduli (<= 512, residues
// of magnitude <= 256, exact in BF16), one tensor-core contraction per modulus
// whose FP32 accumulators stay exact over 256 rows (256 * 256^2 = 2^24), the
// accumulators reduced modulo p every 256 rows, and the sum recovered by the
// Chinese remainder theorem in 128-bit integers (the construction published
// as the Ozaki scheme II).  The only roundings are the one of X, the one of a
// chunk's sum to FP64 and the FP64 sum of the chunks.
//
// The operands are in fixed point per column: an entry 2^k below its column's
// largest keeps b - k bits.  An X is off by at most 2^(1 - b) max|s_p| (0 for a
// zero entry), so a chunk's sum by 2^(1 - b) (max|s_p| sum|s_q| + max|s_q|
// sum|s_p|) over the rows where both are nonzero, where a DFMA sum of r rows is
// off by up to r 2^-53 sum|s_p s_q|.  The first is the smaller one as long as a
// column's entries are not far below its largest: where the geometric mean of a
// column's nonzero entries in a chunk is more than 2^kMeanGap below the largest
// entry, the DFMA kernel takes the product.  kMeanGap = 9: N(0, 1) entries have a
// gap of 3.6 to 4.6, at every step of the benchmark family's solves as well
// (whose w_i span nine decades in the end), and 7.1 with weights over five
// decades; one entry 2^8 above the others, or half of the rows 2^15 above the
// other half, is where the bound meets that of a DFMA sum of some 400 rows.
//
// Passes: (1) k_rns_rows: w_i^-1/2 as a 64-bit mantissa and an exponent;
// (2) k_rns_colmax: exponent bound of every column in every chunk; per chunk
// (3) k_rns_residues: residues to HBM (28 bytes per entry of A, integer and
// FP32 arithmetic only: one FP64 instruction per entry costs as much as 64
// FP32 ones); (4) k_rns_mma; (5) k_rns_combine.  Entries the integer form does
// not cover (non-finite or subnormal entries of A; w not positive, finite and
// within 2^+-1000; columns of too wide a spread) raise a device flag in (1), (2)
// or, for the spread in any chunk, the first chunk's (3); the later passes then do
// nothing and the DFMA kernel, gated on the same flag, forms the product.
#include <cuda.h>

#include <algorithm>
#include <climits>

#include "internal.cuh"
#include "rns.cuh"
#include "tc.cuh"

namespace mdsip {

namespace {

using namespace rns;

constexpr int RN = 14;                 // moduli
constexpr int kModBits = 125;          // floor(log2 of their product)

__constant__ Tab<RN> c_tab = make_tab<RN>();

constexpr int T_M = 128, T_N = 256;    // output tile: 128 rows p, 256 columns q
constexpr int SLAB = 64;               // rows of A (K) per pipeline stage
constexpr int STAGES = 4;
constexpr int FOLD = 4;                // stages per exact accumulation (256 rows)
constexpr int BOX_BYTES = (int)tc::kMnBoxBytes;    // one 64-column x 64-row TMA box
constexpr int STAGE_BYTES = (T_M + T_N) / 64 * BOX_BYTES;   // 48 KiB
constexpr int MMA_THREADS = 384;       // warp 0 loads, warp 1 issues, warps 4-11 fold
constexpr size_t kMmaSmem = 1024 + (size_t)STAGES * STAGE_BYTES + 256;

// tile t of the lower triangle: row block P of 128, column block Q of 256, P >= 2 Q
__device__ __forceinline__ void rns_tile(int t, int &P, int &Q) {
    int a = (int)((sqrtf(4.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((a + 1) * (a + 2) <= t) ++a;
    while (a * (a + 1) > t) --a;
    const int r = t - a * (a + 1);
    P = 2 * a + (r > a ? 1 : 0);
    Q = r > a ? r - a - 1 : r;
}

__host__ __device__ inline int rns_tiles(int64_t n) {
    const int64_t np = (n + T_M - 1) / T_M, a = np / 2;
    return (int)(a * (a + 1) + (np & 1 ? a + 1 : 0));
}

constexpr int kMeanGap = 9;            // binary orders (see above)

// of the columns of every chunk: exponent bound, sum and count of the exponents
struct ColStat {
    int *E, *sum, *cnt;
};

// w_i^-1/2 = sm[i] 2^(se[i] - 63)
__global__ void k_rns_rows(int64_t m, const double *__restrict__ w, unsigned long long *__restrict__ sm,
                           int *__restrict__ se, int *__restrict__ flag) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = w[i];
        if (!(v > 0x1p-1000 && v < 0x1p1000)) {
            atomicExch(flag, 1);
            continue;
        }
        rsqrt64(v, sm[i], se[i]);
    }
}

// col[chunk][q]: E = 2 + max_i (exponent of A[i][q] + se[i]) over the chunk's
// rows, |a s| < 2^E, and the sum and count of the exponents of its nonzero
// entries.  32 x 8 threads, 64 columns and `strip` rows per block; HBM-bound (one
// read of A; m = 100000, n = 2000: 269 us, 255 with the maximum alone).
__global__ void __launch_bounds__(256) k_rns_colmax(const double *__restrict__ A, int64_t m, int64_t n, int64_t lda,
                                                    int64_t kc, int strip, int strips_per_chunk,
                                                    const int *__restrict__ se, ColStat col_stat,
                                                    int *__restrict__ flag) {
    __shared__ int red[3][8][64];
    const int64_t col = (int64_t)blockIdx.x * 64 + 2 * threadIdx.x;
    const int64_t chunk = blockIdx.y / strips_per_chunk;
    const int64_t i0 = chunk * kc + (int64_t)(blockIdx.y % strips_per_chunk) * strip;
    const int64_t i1 = min(m, min(i0 + strip, (chunk + 1) * kc));
    // per column and thread: the largest and the sum of kOne + (exponent + kOff) over
    // the nonzero entries (at most 32 rows: the count above the sum, no carry)
    constexpr unsigned kOne = 1u << 18, kOff = 1024u;
    unsigned m0 = 0, m1 = 0, a0 = 0, a1 = 0;
    unsigned bad = 0;
    auto upd = [&](double v, unsigned s, unsigned &mx, unsigned &acc) {
        const unsigned h = (unsigned)__double2hiint(v) << 1, lo = (unsigned)__double2loint(v);
        if (h - 0x200000u < 0xffc00000u) {   // a normal number
            mx = __viaddmax_u32(h >> 21, s, mx);
            acc += (h >> 21) + s;
        } else {
            bad |= h | lo;                   // zeros pass
        }
    };
    if (col < n) {
        const bool two = col + 1 < n;
        const double *a = A + col;
#pragma unroll 8
        for (int64_t i = i0 + threadIdx.y; i < i1; i += 8) {
            const double2 v = __ldg(reinterpret_cast<const double2 *>(a + i * lda));
            const unsigned s = (unsigned)__ldg(se + i) + (kOne + kOff);
            upd(v.x, s, m0, a0);
            if (two) upd(v.y, s, m1, a1);
        }
    }
    if (bad != 0u) atomicExch(flag, 1);
    auto put = [&](int c, unsigned mx, unsigned acc) {
        const int cnt = (int)(acc / kOne);
        red[0][threadIdx.y][c] = mx ? (int)(mx % kOne) - (int)kOff : INT_MIN;
        red[1][threadIdx.y][c] = (int)(acc % kOne) - cnt * (int)kOff;
        red[2][threadIdx.y][c] = cnt;
    };
    put(2 * threadIdx.x, m0, a0);
    put(2 * threadIdx.x + 1, m1, a1);
    __syncthreads();
    const int t = threadIdx.y * 32 + threadIdx.x, u = t & 63, what = t >> 6;   // 64 threads a quantity
    if (what < 3) {
        int r = red[what][0][u];
        for (int y = 1; y < 8; ++y) r = what == 0 ? max(r, red[0][y][u]) : r + red[what][y][u];
        const int64_t q = (int64_t)blockIdx.x * 64 + u, o = chunk * n + q;
        if (q < n) {
            if (what == 0 && r != INT_MIN) atomicMax(col_stat.E + o, r - 1023 + 2);
            if (what == 1 && r != 0) atomicAdd(col_stat.sum + o, r);
            if (what == 2 && r != 0) atomicAdd(col_stat.cnt + o, r);
        }
    }
}

__global__ void k_rns_init(int64_t cnt, ColStat col_stat) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x) {
        col_stat.E[i] = INT_MIN;
        col_stat.sum[i] = col_stat.cnt[i] = 0;
    }
}

// Raises the flag where a column's spread is too wide.  Out of line: inside the
// kernel below it took that from 64 to 104 registers.
__device__ __noinline__ void rns_spread(ColStat cols, int64_t cnt, int *flag) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x)
        if (cols.cnt[i] > 0 && (int64_t)cols.cnt[i] * (cols.E[i] + 1023 - 2 - kMeanGap) > (int64_t)cols.sum[i])
            atomicExch(flag, 1);
}

// R[l][k][q] = BF16 of X mod p_l, X = rint(A[i0 + k][q] s_(i0+k) 2^(b - colE[q])),
// for k < kpad (zero beyond the chunk's rows) and q < ldn (zero beyond n).
// Eight columns per thread: four 16-byte loads of A, one 16-byte store per
// modulus.  X comes from a 64 x 64 -> high 64-bit integer product and one
// rounding shift; its residues from four 14-bit limbs in FP32 (|v| < 2^24,
// exact), the quotient rounded by the 1.5 2^23 trick.  Bound by the 28 bytes
// written per entry.
__global__ void __launch_bounds__(256) k_rns_residues(const double *__restrict__ A, int64_t lda, int64_t n, int64_t i0,
                                                      int rows, int kpad, int ldn, int b,
                                                      const unsigned long long *__restrict__ sm,
                                                      const int *__restrict__ se, const int *__restrict__ colE,
                                                      uint4 *__restrict__ R, int *flag, ColStat all, int64_t check) {
    if (*flag) return;
    if (check) rns_spread(all, check, flag);
    const int groups = ldn / 8;
    const int64_t total = (int64_t)kpad * groups;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(e / groups), g = (int)(e - (int64_t)k * groups);
        const int q0 = 8 * g;
        double v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = 0.0;
        unsigned long long s = 0;
        int es = 0;
        if (k < rows) {
            const double *row = A + (i0 + k) * lda + q0;
            s = __ldg(sm + i0 + k);
            es = __ldg(se + i0 + k);
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                if (q0 + j < n) {   // lda is even: the pair lies inside the row
                    const double2 t = __ldg(reinterpret_cast<const double2 *>(row + j));
                    v[j] = t.x;
                    if (q0 + j + 1 < n) v[j + 1] = t.y;
                }
            }
        }
        Limbs x[8];
        unsigned sgn[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            // (columns beyond n hold zeros; subnormal entries raised the flag)
            x[j] = limbs(v[j] != 0.0 ? scaled_int(v[j], s, es, __ldg(colE + q0 + j), b) : 0ULL);
            if (__double2hiint(v[j]) < 0) sgn[j >> 1] |= 0x8000u << (16 * (j & 1));
        }
        uint4 *out = R + (int64_t)k * groups + g;
#pragma unroll
        for (int l = 0; l < RN; ++l) {
            uint32_t r[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) r[j] = __float_as_uint(residue(c_tab, l, x[j]));
            uint4 o;   // the BF16 of an integer of magnitude <= 256 is the upper half of its FP32
            o.x = __byte_perm(r[0], r[1], 0x7632) ^ sgn[0];
            o.y = __byte_perm(r[2], r[3], 0x7632) ^ sgn[1];
            o.z = __byte_perm(r[4], r[5], 0x7632) ^ sgn[2];
            o.w = __byte_perm(r[6], r[7], 0x7632) ^ sgn[3];
            out[(int64_t)l * total] = o;
        }
    }
}

struct MmaArgs {
    int tile0, ntile;      // tiles of this launch
    int nsplit;            // K splits
    int nslab, slabs_per_split;
    int kpad;
    int16_t *W;            // [l][split][tile][256 q][128 p] residues of the sums
    const int *flag;
    int *err;
};

// One persistent CTA per SM; work item = (modulus, split, tile), tiles fastest
// so that concurrent items share a modulus's residues in L2.  Warp 0 lane 0
// streams 64-row slabs of the two column blocks by TMA into a 4-stage ring,
// warp 1 lane 0 issues 128 x 256 x 16 MMAs (both operands MN-major: the
// residues keep A's row-major order, no transposition anywhere) into one of
// two 256-column TMEM accumulators; after every 256 rows the eight fold warps
// reduce that accumulator modulo p into registers (128 columns per thread)
// while the other fills.  A diagonal tile (P = 2 Q) needs only its first 128
// columns and runs 128 x 128 MMAs.
__global__ void __launch_bounds__(MMA_THREADS, 1) k_rns_mma(const __grid_constant__ CUtensorMap rmap, MmaArgs a) {
    if (*a.flag) return;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + (size_t)STAGES * STAGE_BYTES);
    uint64_t *empty = full + STAGES;
    uint64_t *tfull = empty + STAGES;     // [2] accumulator ready
    uint64_t *tempty = tfull + 2;         // [2] accumulator folded
    uint64_t *done = tempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&tfull[s], 1);
            tc::mbar_init(&tempty[s], 8);   // one arrival per fold warp
        }
        tc::mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&rmap)) : "memory");
    }
    if (warp == 0) tc::tmem_alloc(tmem_slot, 512);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;

    const int per_l = a.nsplit * a.ntile;
    const int items = RN * per_l;
    if (warp == 0 && lane == 0) {
        int it = 0;
        for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
            const int l = w / per_l, sp = (w - l * per_l) / a.ntile, t = w - l * per_l - sp * a.ntile;
            int P, Q;
            rns_tile(a.tile0 + t, P, Q);
            const int nb = P == 2 * Q ? 2 : 4;   // 64-column boxes of the q block
            const int s0 = sp * a.slabs_per_split, s1 = min(a.nslab, s0 + a.slabs_per_split);
            for (int ks = s0; ks < s1; ++ks, ++it) {
                const int st = it % STAGES, rnd = it / STAGES;
                if (!tc::mbar_wait(&empty[st], (rnd & 1) ^ 1)) {
                    ok = false;
                    break;
                }
                tc::mbar_expect_tx(&full[st], (2 + nb) * BOX_BYTES);
                uint8_t *d = smem + (size_t)st * STAGE_BYTES;
                const int y = l * a.kpad + ks * SLAB;
                for (int u = 0; u < 2; ++u) tc::tma_load_2d(d + u * BOX_BYTES, &rmap, &full[st], P * T_M + 64 * u, y);
                for (int u = 0; u < nb; ++u)
                    tc::tma_load_2d(d + (2 + u) * BOX_BYTES, &rmap, &full[st], Q * T_N + 64 * u, y);
            }
        }
        for (int j = max(0, it - STAGES); j < it; ++j)   // no copy is in flight when the CTA leaves
            if (!tc::mbar_wait(&full[j % STAGES], (j / STAGES) & 1)) ok = false;
    } else if (warp == 1 && lane == 0) {
        int it = 0, fold = 0;
        for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
            const int l = w / per_l, sp = (w - l * per_l) / a.ntile, t = w - l * per_l - sp * a.ntile;
            int P, Q;
            rns_tile(a.tile0 + t, P, Q);
            const bool half = P == 2 * Q;
            const int s0 = sp * a.slabs_per_split, s1 = min(a.nslab, s0 + a.slabs_per_split);
            for (int f0 = s0; f0 < s1 && ok; f0 += FOLD, ++fold) {
                const int buf = fold & 1, use = fold >> 1;
                if (!tc::mbar_wait(&tempty[buf], (use & 1) ^ 1)) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                const uint32_t acc = tmem + (uint32_t)(buf * T_N);
                const int f1 = min(s1, f0 + FOLD);
                for (int ks = f0; ks < f1; ++ks, ++it) {
                    const int st = it % STAGES, rnd = it / STAGES;
                    if (!tc::mbar_wait(&full[st], rnd & 1)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after();
                    const uint32_t ab = tc::smem_u32(smem + (size_t)st * STAGE_BYTES), bb = ab + 2 * BOX_BYTES;
#pragma unroll
                    for (int k = 0; k < SLAB / 16; ++k) {
                        const uint64_t da = tc::sw128_mnmajor_desc(ab + 2048 * k), db = tc::sw128_mnmajor_desc(bb + 2048 * k);
                        const uint32_t on = (ks > f0 || k > 0) ? 1u : 0u;
                        if (half)
                            tc::mma<false, tc::instr_desc(false, T_M, 128, true, true)>(acc, da, db, on);
                        else
                            tc::mma<false, tc::instr_desc(false, T_M, 256, true, true)>(acc, da, db, on);
                    }
                    tc::commit(&empty[st]);
                }
                if (!ok) break;
                tc::commit(&tfull[buf]);
            }
        }
        tc::commit(done);   // every MMA this CTA issued has completed when `done` flips
        if (!tc::mbar_wait(done, 0)) ok = false;
    } else if (warp >= 4) {
        const int quad = warp & 3, hc = (warp - 4) >> 2;   // TMEM lanes 32 quad .., columns 128 hc ..
        int fold = 0;
        uint64_t acc[64];
        const uint64_t magic = pk(kMagic, kMagic), nmagic = pk(-kMagic, -kMagic);
        for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
            const int l = w / per_l, sp = (w - l * per_l) / a.ntile, t = w - l * per_l - sp * a.ntile;
            int P, Q;
            rns_tile(a.tile0 + t, P, Q);
            const bool skip = P == 2 * Q && hc == 1;   // the columns above the diagonal
            const int s0 = sp * a.slabs_per_split, s1 = min(a.nslab, s0 + a.slabs_per_split);
            const float pf = c_tab.p[l], pi = c_tab.pinv[l];
            const uint64_t np2 = pk(-pf, -pf), pi2 = pk(pi, pi);
#pragma unroll
            for (int j = 0; j < 64; ++j) acc[j] = 0;
            for (int f0 = s0; f0 < s1; f0 += FOLD, ++fold) {
                const int buf = fold & 1, use = fold >> 1;
                if (!tc::mbar_wait(&tfull[buf], use & 1)) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                if (!skip) {
                    const uint32_t base = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(buf * T_N + 128 * hc);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        uint32_t r[16];
                        tc::tmem_ld16(base + 16 * c, r);
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const uint64_t x = pk(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
                            const uint64_t q = add2(fma2(x, pi2, magic), nmagic);
                            acc[8 * c + j] = add2(acc[8 * c + j], fma2(np2, q, x));
                        }
                    }
                }
                tc::fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&tempty[buf]);
            }
            if (ok && !skip) {
                int16_t *out = a.W + ((size_t)w * T_N + 128 * hc) * T_M + 32 * quad + lane;
#pragma unroll
                for (int j = 0; j < 64; ++j) {
                    const uint64_t q = add2(fma2(acc[j], pi2, magic), nmagic);
                    const float2 v = upk(fma2(np2, q, acc[j]));
                    out[(size_t)(2 * j) * T_M] = (int16_t)v.x;
                    out[(size_t)(2 * j + 1) * T_M] = (int16_t)v.y;
                }
            }
        }
    }
    if (!ok) atomicExch(a.err, 1);
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// C[p][q] = beta C[p][q] + 2^(colE_p + colE_q - 2 b) sum_i X_ip X_iq: the
// residues of the splits added, y_l = r_l (M/p_l)^-1 mod p_l, the sum
// X = sum_l y_l M/p_l - k M with k = rint(sum_l y_l / p_l) (|X| < M / 4, so FP32
// finds k), rounded once to FP64.  A raised err word (a wait that expired in
// k_rns_mma) poisons the result with NaN and is passed on to late_err.  Bound by the latency of its loads: a
// thread loads its next column's 14 residues under the arithmetic of this one,
// whose 14 terms of five 30-bit limbs are seven pairs of four 32-bit ones (n =
// 2000, 72 tiles: 98 us with a column a thread and three splits, 46 so).
__global__ void __launch_bounds__(256) k_rns_combine(int64_t n, int tile0, int ntile, int nsplit, int b,
                                                     const int16_t *__restrict__ W, const int *__restrict__ colE,
                                                     double beta, double *__restrict__ C, int64_t ldc,
                                                     const int *__restrict__ flag, const int *__restrict__ err,
                                                     int *late_err) {
    if (*flag) return;
    const bool poison = *err != 0;
    if (poison && late_err && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0) *(volatile int *)late_err = 1;
    int P, Q;
    rns_tile(tile0 + blockIdx.x, P, Q);
    const int row = threadIdx.x & 127;
    const int64_t p = (int64_t)P * T_M + row;
    const size_t per_item = (size_t)T_M * T_N;
    const size_t ls = (size_t)ntile * per_item;   // one split; nsplit of them per modulus
    const int16_t *wp = W + (size_t)blockIdx.x * per_item + row;
    const int step = gridDim.y * 2;
    const int c0 = blockIdx.y * 2 + (threadIdx.x >> 7);
    // columns this row has: c < T_N, q <= p < n
    const int cend = p < n ? (int)min((int64_t)T_N, p - (int64_t)Q * T_N + 1) : 0;
    int nx[RN];   // the next column's residues of the first split, loaded under this one's arithmetic
    auto fetch = [&](int c) {
        if (c < cend)
#pragma unroll
            for (int l = 0; l < RN; ++l) nx[l] = __ldg(wp + (size_t)(l * nsplit) * ls + (size_t)c * T_M);
    };
    fetch(c0);
    for (int c = c0; c < cend; c += step) {
        const int64_t q = (int64_t)Q * T_N + c;
        int r[RN];
#pragma unroll
        for (int l = 0; l < RN; ++l) r[l] = nx[l];
        double *out = C + p + q * ldc;
        const double old = beta != 0.0 ? *out : 0.0;
        const int e = __ldg(colE + p) + __ldg(colE + q) - 2 * b;
        fetch(c + step);
        for (int s = 1; s < nsplit; ++s) {   // the 14 loads of a split in flight together
#pragma unroll
            for (int l = 0; l < RN; ++l) r[l] += wp[(size_t)(l * nsplit + s) * ls + (size_t)c * T_M];
        }
        // pairs of moduli: z = y_p q + y_q p (exact, |z| < 2^19), X = sum z M/(p q) - k M
        // modulo 2^128 in 32-bit limbs, z + 2^19 against the bias
        unsigned long long acc[4] = {0, 0, 0, 0};
        float frac = 0.0f;
#pragma unroll
        for (int l = 0; l < RN; l += 2) {
            const float y0 = mod((float)r[l] * c_tab.inv[l], c_tab.p[l], c_tab.pinv[l]);   // the product < 2^24
            const float y1 = mod((float)r[l + 1] * c_tab.inv[l + 1], c_tab.p[l + 1], c_tab.pinv[l + 1]);
            frac = fmaf(y0, c_tab.pinv[l], fmaf(y1, c_tab.pinv[l + 1], frac));
            const unsigned z = (unsigned)((int)fmaf(y0, c_tab.p[l + 1], y1 * c_tab.p[l]) + (1 << 19));
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j] += (unsigned long long)z * c_tab.mpair32[l / 2][j];
        }
        const int kq = (int)rintf(frac);
        unsigned __int128 M = 0, B = 0, u = 0;   // X modulo 2^128
#pragma unroll
        for (int j = 3; j >= 0; --j) {
            M = (M << 32) | c_tab.mod32[j];
            B = (B << 32) | c_tab.bias32[j];
            u = (u << 32) + acc[j];
        }
        u -= B + M * (unsigned __int128)(__int128)kq;
        const double val = poison ? (double)NAN : to_double(u, e);
        *out = old + val;
    }
}

static_assert(RN % 2 == 0, "moduli are taken in pairs");

struct RnsPlan {
    int64_t ldn, kc, chunks;
    int tiles, group, nsplit, slabs_per_split;   // tiles, tiles per launch, K splits of a full chunk
};

size_t al1k(size_t b) { return (b + 1023) / 1024 * 1024; }

// cap: bytes of one chunk's residues; half of it for the residues of one launch's sums
RnsPlan rns_plan(int64_t m, int64_t n, int num_sms, size_t cap) {
    RnsPlan pl{};
    pl.ldn = (n + 7) / 8 * 8;
    const int64_t mp = (m + SLAB - 1) / SLAB * SLAB;
    int64_t kc = (int64_t)(cap / (2 * RN * (size_t)pl.ldn)) / (SLAB * FOLD) * (SLAB * FOLD);
    kc = std::min<int64_t>(std::max<int64_t>(kc, SLAB * FOLD), 32768);
    pl.chunks = (mp + kc - 1) / kc;
    // equal chunks
    kc = ((mp + pl.chunks - 1) / pl.chunks + SLAB * FOLD - 1) / (SLAB * FOLD) * (SLAB * FOLD);
    pl.kc = std::min(kc, mp);
    pl.chunks = (m + pl.kc - 1) / pl.kc;
    pl.tiles = rns_tiles(n);
    // K splits so that the items fill whole waves of one CTA per SM, each at
    // least 512 rows: two 256-row folds
    const int nslab = (int)(pl.kc / SLAB);
    // (products at their rate over the fill of the last wave, plus the sums'
    // residues written and read once per split)
    double best = 1e30;
    pl.nsplit = 1;
    const double t0 = 2.0 * pl.tiles * RN * T_M * T_N * (double)pl.kc / 1.35e15;
    for (int s = 1; s <= 16; ++s) {
        if (s > 1 && nslab / s < 2 * FOLD) break;
        const double waves = (double)pl.tiles * RN * s / num_sms;
        const double t = t0 * std::ceil(waves) / waves + 2.0 * s * pl.tiles * RN * T_M * T_N * sizeof(int16_t) / 5e12;
        if (t < 0.99 * best) {
            best = t;
            pl.nsplit = s;
        }
    }
    pl.slabs_per_split = ((nslab + pl.nsplit - 1) / pl.nsplit + FOLD - 1) / FOLD * FOLD;
    pl.nsplit = (nslab + pl.slabs_per_split - 1) / pl.slabs_per_split;
    const size_t per_tile = (size_t)RN * pl.nsplit * T_M * T_N * sizeof(int16_t);
    pl.group = (int)std::min<int64_t>(pl.tiles, std::max<int64_t>(1, (int64_t)(cap / 2 / per_tile)));
    return pl;
}

int ceil_log2(int64_t v) {
    int r = 0;
    while ((1LL << r) < v) ++r;
    return r;
}

}  // namespace

// The rule of the dispatch, both sides measured (us per call, residues /
// DFMA): 1003 x 130 54 / 70, 4000 x 80 59 / 82, 5000 x 100 62 / 181,
// 15053 x 301 141 / 1588, 100000 x 2000 6980 / 336087; below, where the
// residue form's passes and launches cost about 55 us, 2000 x 64 56 / 35,
// 3200 x 64 58 / 35, 1000 x 32 55 / 23 (orders up to 64 use the DFMA kernel's
// 32 x 32 tiles, which spread better).
bool syrk_rns_pays(int64_t m, int64_t n) {
    const double work = (double)m * (double)n * (double)n;
    return m >= 256 && work >= (n > 64 ? 1.5e7 : 3e7) && n <= (1 << 20) && m <= (1 << 23);
}

size_t syrk_rns_workspace_bytes(int64_t m, int64_t n, int num_sms, size_t cap) {
    const RnsPlan pl = rns_plan(m, n, num_sms, cap);
    return 1024 + al1k((size_t)m * 8) + al1k((size_t)m * 4) + 3 * al1k((size_t)pl.chunks * n * 4) +
           al1k((size_t)RN * pl.kc * pl.ldn * 2) +
           al1k((size_t)RN * pl.nsplit * pl.group * T_M * T_N * sizeof(int16_t));
}

// ws: syrk_rns_workspace_bytes(m, n, num_sms, cap), 1024-byte aligned.  Returns the device flag that gates the DFMA kernel: it
// is nonzero after these launches when C still has to be formed.
const int *launch_syrk_rns(cudaStream_t st, int num_sms, const double *A, int64_t m, int64_t n, int64_t lda,
                           const double *w, double beta, double *C, int64_t ldc, void *ws, size_t cap, int *late_err,
                           bool expire) {
    const RnsPlan pl = rns_plan(m, n, num_sms, cap);
    char *base = static_cast<char *>(ws);
    int *flag = reinterpret_cast<int *>(base), *err = flag + 1;
    base += 1024;
    auto *sm = reinterpret_cast<unsigned long long *>(base);
    base += al1k((size_t)m * 8);
    int *se = reinterpret_cast<int *>(base);
    base += al1k((size_t)m * 4);
    ColStat cols{};
    for (int **v : {&cols.E, &cols.sum, &cols.cnt}) {
        *v = reinterpret_cast<int *>(base);
        base += al1k((size_t)pl.chunks * n * 4);
    }
    const int *colE = cols.E;
    uint4 *R = reinterpret_cast<uint4 *>(base);
    base += al1k((size_t)RN * pl.kc * pl.ldn * 2);
    int16_t *W = reinterpret_cast<int16_t *>(base);

    MDSIP_CUDA(cudaMemsetAsync(flag, 0, 2 * sizeof(int), st));
    if (expire) MDSIP_CUDA(cudaMemsetAsync(err, 1, sizeof(int), st));
    k_rns_init<<<std::max(1, std::min(1024, ceil_div(pl.chunks * n, 256))), 256, 0, st>>>(pl.chunks * n, cols);
    MDSIP_LAUNCHED();
    k_rns_rows<<<std::max(1, std::min(4096, ceil_div(m, 256))), 256, 0, st>>>(m, w, sm, se, flag);
    MDSIP_LAUNCHED();
    const int strip = 256, spc = (int)((pl.kc + strip - 1) / strip);
    MDSIP_REQUIRE(pl.chunks * spc <= 65535, MDSIP_ERR_INVALID_ARG, "syrk: m too large");
    const dim3 cg((unsigned)ceil_div(n, 64), (unsigned)(pl.chunks * spc));
    k_rns_colmax<<<cg, dim3(32, 8), 0, st>>>(A, m, n, lda, pl.kc, strip, spc, se, cols, flag);
    MDSIP_LAUNCHED();

    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_rns_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMmaSmem);
    }));
    for (int64_t c = 0; c < pl.chunks; ++c) {
        const int64_t i0 = c * pl.kc;
        const int rows = (int)std::min<int64_t>(pl.kc, m - i0);
        const int kpad = (rows + SLAB - 1) / SLAB * SLAB;
        const int b = std::min(56, (kModBits - 2 - ceil_log2(rows)) / 2);   // |sum| <= rows 2^(2b) < M / 4
        const int64_t total = (int64_t)kpad * (pl.ldn / 8);
        k_rns_residues<<<(int)std::min<int64_t>((int64_t)num_sms * 32, (total + 255) / 256), 256, 0, st>>>(
            A, lda, n, i0, rows, kpad, (int)pl.ldn, b, sm, se, colE + c * n, R, flag, cols, c == 0 ? pl.chunks * n : 0);
        MDSIP_LAUNCHED();
        CUtensorMap rmap;
        tc::encode_2d(&rmap, R, false, (uint64_t)pl.ldn, (uint64_t)RN * kpad, (uint64_t)pl.ldn, 64, SLAB);
        const int nslab = kpad / SLAB;
        const int nsplit = (nslab + pl.slabs_per_split - 1) / pl.slabs_per_split;
        for (int t0 = 0; t0 < pl.tiles; t0 += pl.group) {
            const int nt = std::min(pl.group, pl.tiles - t0);
            MmaArgs a{t0, nt, nsplit, nslab, pl.slabs_per_split, kpad, W, flag, err};
            k_rns_mma<<<std::min(num_sms, RN * nsplit * nt), MMA_THREADS, kMmaSmem, st>>>(rmap, a);
            MDSIP_LAUNCHED();
            // four columns a thread where there are blocks enough, fewer for few tiles
            const int yb = nt >= 32 ? T_N / 8 : nt >= 8 ? T_N / 4 : T_N / 2;
            k_rns_combine<<<dim3((unsigned)nt, (unsigned)yb), 256, 0, st>>>(n, t0, nt, nsplit, b, W, colE + c * n,
                                                                  c == 0 ? beta : 1.0, C, ldc, flag, err, late_err);
            MDSIP_LAUNCHED();
        }
    }
    return flag;
}

}  // namespace mdsip
