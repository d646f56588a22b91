// BF16 GEMM on the 5th-generation tensor cores for the warm-start network:
//
//     C[m][n] = sum_k A[m][k] B[n][k]          (FP32 accumulation)
//
// with A (M x K) and B (N x K) in BF16, C FP32 row-major.  Every layer of the
// network, forward and backward, is this one contraction; either operand may
// be given transposed (stored K x M or K x N, "MN-major"), which the tensor
// core reads directly through its descriptor, so no transposed copies exist.
//
// One CTA computes a 128 x 128 tile over one K range: warp 0 lane 0 streams
// 64-element K slabs of A and B by TMA (128-byte swizzle, out-of-range rows
// and columns read as zero) into a 3-stage ring, warp 1 lane 0 issues
// tcgen05.mma into a 128-column FP32 accumulator in tensor memory, and the
// four warps move the accumulator out with tcgen05.ld.  When the tile grid is
// smaller than the GPU, K is split and the partial tiles are summed in a
// fixed order by a second kernel.  Waits are bounded and raise an error flag.
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.cuh"
#include "mlp.cuh"
#include "tc.cuh"

namespace mdsip {

namespace {

constexpr int G_TILE = 128;
constexpr int G_THREADS = 128;
constexpr int G_STAGES = 3;
constexpr int G_SLAB = 64;                       // BF16 elements (128 bytes) of K per stage
constexpr int G_TILE_BYTES = G_TILE * G_SLAB * 2;
constexpr uint32_t G_TMEM_COLS = 128;
constexpr size_t kGemmSmemBytes = 1024 + 2 * G_STAGES * G_TILE_BYTES + 256;

struct GemmArgs {
    int64_t M, N;
    int total_slabs, slabs_per_split;
    float *out;       // nsplit == 1: C; else partials [split][M][N]
    int64_t ldo;
    int64_t split_stride;
    int *err;
};

// One operand slab (128 rows of the operand x 64 of K) into a stage: one K-major
// box, or two MN-major boxes of 64.
template <bool MN>
__device__ __forceinline__ void load_slab(uint8_t *dst, const CUtensorMap *map, uint64_t *bar, int kx, int r0) {
    if constexpr (MN) {
        tc::tma_load_2d(dst, map, bar, r0, kx);
        tc::tma_load_2d(dst + tc::kMnBoxBytes, map, bar, r0 + 64, kx);
    } else {
        tc::tma_load_2d(dst, map, bar, kx, r0);
    }
}
template <bool MN>
__device__ __forceinline__ uint64_t slab_desc(uint32_t saddr, int k) {   // K step k of 16
    return MN ? tc::sw128_mnmajor_desc(saddr + 2048 * k) : tc::sw128_kmajor_desc(saddr + 32 * k);
}

template <bool AMN, bool BMN>
__global__ void __launch_bounds__(G_THREADS, 2)
    k_gemm_bf16(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap, GemmArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sA = smem;
    uint8_t *sB = smem + G_STAGES * G_TILE_BYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + 2 * G_STAGES * G_TILE_BYTES);
    uint64_t *empty = full + G_STAGES;
    uint64_t *accum = empty + G_STAGES;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(accum + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * G_TILE, m0 = blockIdx.y * G_TILE;
    const int split = blockIdx.z;
    const int s0 = split * a.slabs_per_split;
    const int nslab = max(0, min(a.total_slabs, s0 + a.slabs_per_split) - s0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < G_STAGES; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        tc::mbar_init(accum, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&amap)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&bmap)) : "memory");
    }
    if (warp == 0) tc::tmem_alloc(tmem_slot, G_TMEM_COLS);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        for (int it = 0; it < nslab; ++it) {
            const int st = it % G_STAGES, rnd = it / G_STAGES;
            if (!tc::mbar_wait(&empty[st], (rnd & 1) ^ 1)) {
                atomicExch(a.err, 1);
                break;
            }
            tc::mbar_expect_tx(&full[st], 2 * G_TILE_BYTES);
            const int kx = (s0 + it) * G_SLAB;
            load_slab<AMN>(sA + st * G_TILE_BYTES, &amap, &full[st], kx, m0);
            load_slab<BMN>(sB + st * G_TILE_BYTES, &bmap, &full[st], kx, n0);
        }
    } else if (warp == 1 && lane == 0) {
        for (int it = 0; it < nslab; ++it) {
            const int st = it % G_STAGES, rnd = it / G_STAGES;
            if (!tc::mbar_wait(&full[st], rnd & 1)) {
                atomicExch(a.err, 1);
                break;
            }
            tc::fence_after();
            const uint32_t ab = tc::smem_u32(sA + st * G_TILE_BYTES), bb = tc::smem_u32(sB + st * G_TILE_BYTES);
#pragma unroll
            for (int k = 0; k < 4; ++k)   // four K steps of 16 elements (32 bytes)
                tc::mma<false, tc::instr_desc(false, G_TILE, G_TILE, AMN, BMN)>(
                    tmem, slab_desc<AMN>(ab, k), slab_desc<BMN>(bb, k), (it > 0 || k > 0) ? 1u : 0u);
            tc::commit(&empty[st]);
        }
        tc::commit(accum);
    }
    __syncwarp();
    const bool ok = nslab == 0 || tc::mbar_wait(accum, 0);
    tc::fence_after();
    if (!ok) atomicExch(a.err, 1);
    float *out = a.out + (size_t)split * a.split_stride;
    const int64_t m = m0 + warp * 32 + lane;   // TMEM lane = tile row
    const bool vec = (a.ldo % 4 == 0) && (reinterpret_cast<uintptr_t>(a.out) % 16 == 0);
#pragma unroll 1
    for (int c = 0; c < G_TILE / 32; ++c) {
        const int64_t nb = n0 + 32 * c;
        if (nb >= a.N) break;   // uniform across the CTA
        uint32_t r[32];
        if (ok && nslab > 0) {
            tc::tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(c * 32), r);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) r[j] = 0u;
        }
        if (m >= a.M) continue;
        float *row = out + m * a.ldo + nb;
        if (vec && nb + 32 <= a.N) {
#pragma unroll
            for (int j = 0; j < 32; j += 4)
                *reinterpret_cast<float4 *>(row + j) = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                                                   __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (nb + j < a.N) row[j] = __uint_as_float(r[j]);
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, G_TMEM_COLS);
}

// ---------------------------------------------------------------------------
// Many column tiles (the network's output layer): persistent CTAs, one per
// SM, each walking its 128-column tiles of C.  Per tile and per 256 rows of A
// one tcgen05.mma of shape 128 x 256 per K step computes the transposed tile
// C^T[n][m] = sum_k B[n][k] A[m][k] (B's rows as the instruction's A operand,
// 256 rows of A as its B operand), so every slab of B is read once from HBM
// and A is re-read from L2.  Warp roles: warp 0 lane 0 streams K slabs by TMA
// into a 4-stage ring; warp 1 lane 0 issues the MMAs into one of two
// 256-column TMEM accumulators; warps 4-11 drain the other accumulator (TMEM
// lane = column n of C, so each store of a warp writes 32 consecutive values
// of one row of C; two warps share a lane quarter, 128 rows each) while the
// next tile accumulates.  Waits are bounded and raise the error flag.
//
// What the drain does with a value is the MODE: W_STORE writes C; W_DENORM
// writes the network's output (c + b3_n) std_n + mean_n; W_LOSS forms the
// training loss and its gradient (below).  The separate passes these replace
// wrote and re-read the FP32 C (741 MB for 1024 predictions of 180937
// values: 476 + 449 us, now one kernel of 230 us) and spent the training
// step's largest share, 1344 us, on FP64 divisions and sums; the loss form
// takes 242 us at 256 x 180937, bound by its 2 x 4 drain warps' issue slots.
constexpr int W_THREADS = 384;
constexpr int W_STAGES = 4;
constexpr int W_BN = 128;                          // columns of C per tile (rows of B)
constexpr int W_BM = 256;                          // rows of C (A) per accumulator
constexpr int W_B_BYTES = W_BN * G_SLAB * 2;       // 16 KB
constexpr int W_A_BYTES = W_BM * G_SLAB * 2;       // 32 KB
constexpr uint32_t W_TMEM_COLS = 512;              // two 256-column accumulators
constexpr size_t kGemmWideSmemBytes = 1024 + (size_t)W_STAGES * (W_A_BYTES + W_B_BYTES) + 256;

enum WideMode { W_STORE, W_DENORM, W_LOSS };

struct GemmWideArgs {
    int64_t M, N;
    int ntiles, nslab, mchunks;
    float *C;
    int64_t ldc;
    int *err;
    OutLayer o;
};

// (y - mean) / sd as FP32: the FP64 expression rounded once, formed from FP32
// parts to about 2^-46 before that rounding (a conversion, subtraction and
// division on the FP64 pipe cost about 64 FP32 instructions each here).  y is
// cut into its upper 24 bits, the next 15 and the last 14, each exact in FP32.
// Free of branches, so that a thread's independent values overlap; sets bad
// where a part is not a normal FP32 number: those take the FP64 expression.
__device__ __forceinline__ float standardise(double y, float mean, float sd, float rsd, bool &bad) {
    const int hi = __double2hiint(y);
    const unsigned lo = (unsigned)__double2loint(y);
    const int e = (hi >> 20) & 0x7ff;                    // biased FP64 exponent
    const bool zero = ((hi & 0x7fffffff) | (int)lo) == 0;
    const unsigned sign = (unsigned)hi & 0x80000000u;
    const int ec = min(max(e, 1023 - 70), 1023 + 120);
    float unit = __uint_as_float(sign | ((unsigned)(ec - 896 - 52) << 23));   // the last bit's value
    float yh = __uint_as_float(sign | ((unsigned)(ec - 896) << 23) | (((unsigned)hi & 0xfffffu) << 3) | (lo >> 29));
    unit = zero ? 0.0f : unit;
    yh = zero ? 0.0f : yh;
    const float ym = (float)(lo & 0x1fffc000u) * unit, yl = (float)(lo & 0x3fffu) * unit;
    float h = yh - mean, bb = h - yh;                    // two-sums of yh - mean and ym
    float l = (yh - (h - bb)) + (-mean - bb);
    const float h2 = h + ym;
    bb = h2 - h;
    l += ((h - (h2 - bb)) + (ym - bb)) + yl;
    const float q = h2 * rsd;
    const float r = fmaf(-q, sd, h2) + l;                // remainder of the quotient estimate
    const float t = fmaf(r, rsd, q);
    bad |= (e != ec && !zero) || !isfinite(t);
    return t;
}

template <WideMode MODE>
__global__ void __launch_bounds__(W_THREADS, 1)
    k_gemm_bf16_wide(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
                     GemmWideArgs a) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ int64_t s_off[MODE == W_LOSS ? 8 : 1][128];   // target offsets of each drain warp's rows
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sA = smem;                                  // [stage][256 rows][64 K]
    uint8_t *sB = smem + W_STAGES * W_A_BYTES;           // [stage][128 rows][64 K]
    uint64_t *full = reinterpret_cast<uint64_t *>(sB + W_STAGES * W_B_BYTES);
    uint64_t *empty = full + W_STAGES;
    uint64_t *tfull = empty + W_STAGES;                  // [2]: accumulator ready for the epilogue
    uint64_t *tempty = tfull + 2;                        // [2]: accumulator drained
    uint64_t *done = tempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < W_STAGES; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&tfull[b], 1);
            tc::mbar_init(&tempty[b], 8);   // one arrival per drain warp
        }
        tc::mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&amap)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&bmap)) : "memory");
    }
    if (warp == 0) tc::tmem_alloc(tmem_slot, W_TMEM_COLS);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;

    if (warp == 0 && lane == 0) {   // producer
        int it = 0;
        for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
            for (int mc = 0; mc < a.mchunks && ok; ++mc) {
                for (int ks = 0; ks < a.nslab; ++ks, ++it) {
                    const int st = it % W_STAGES, rnd = it / W_STAGES;
                    if (!tc::mbar_wait(&empty[st], (rnd & 1) ^ 1)) {
                        ok = false;
                        break;
                    }
                    tc::mbar_expect_tx(&full[st], W_A_BYTES + W_B_BYTES);
                    tc::tma_load_2d(sA + st * W_A_BYTES, &amap, &full[st], ks * G_SLAB, mc * W_BM);
                    tc::tma_load_2d(sB + st * W_B_BYTES, &bmap, &full[st], ks * G_SLAB, t * W_BN);
                }
            }
        }
        for (int j = max(0, it - W_STAGES); j < it; ++j)   // no copy is in flight when the CTA leaves
            if (!tc::mbar_wait(&full[j % W_STAGES], (j / W_STAGES) & 1)) ok = false;
    } else if (warp == 1 && lane == 0) {   // MMA issuer
        int it = 0, tl = 0;
        for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
            for (int mc = 0; mc < a.mchunks && ok; ++mc, ++tl) {
                const int b = tl & 1, use = tl >> 1;
                if (!tc::mbar_wait(&tempty[b], (use & 1) ^ 1)) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                const uint32_t acc = tmem + (uint32_t)(b * W_BM);
                for (int ks = 0; ks < a.nslab; ++ks, ++it) {
                    const int st = it % W_STAGES, rnd = it / W_STAGES;
                    if (!tc::mbar_wait(&full[st], rnd & 1)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after();
                    const uint32_t ab = tc::smem_u32(sB + st * W_B_BYTES), bb = tc::smem_u32(sA + st * W_A_BYTES);
#pragma unroll
                    for (int k = 0; k < 4; ++k)   // four K steps of 16 elements (32 bytes)
                        tc::mma<false, tc::instr_desc(false, W_BN, W_BM)>(acc, tc::sw128_kmajor_desc(ab + 32 * k),
                                                                          tc::sw128_kmajor_desc(bb + 32 * k),
                                                                          (ks > 0 || k > 0) ? 1u : 0u);
                    tc::commit(&empty[st]);
                }
                if (ok) tc::commit(&tfull[b]);
            }
        }
        tc::commit(done);   // every MMA this CTA issued has completed when `done` flips
        if (!tc::mbar_wait(done, 0)) ok = false;
    } else if (warp >= 4) {   // drain: TMEM lanes 32 q .. 32 q + 31 = columns n of the tile, rows 128 half ..
        const int q = warp & 3, half = (warp - 4) >> 2;
        int tl = 0;
        // W_LOSS: this thread's sum of squares, in FP64 over the tiles and in FP32 parts
        // within one (128 values): the sum, its rounding errors and those of the squares,
        // the latter over pairs first -- their low bits are those of squares, 0, 1 or 4
        // modulo 8, and adding one after the other rounds with a bias.  Relative error of
        // the loss at 256 x 180937 2e-16, as an FP64 sum; with one low part throughout 9e-15.
        double sum = 0.0;
        float sq = 0.0f, sq_lo = 0.0f, sq_e = 0.0f;
        for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
            const int64_t n = (int64_t)t * W_BN + 32 * q + lane;
            const bool live = n < a.N;
            float b3 = 0.0f, mean = 0.0f, sd = 1.0f, rsd = 1.0f;
            if constexpr (MODE != W_STORE) {
                if (live) {
                    b3 = a.o.b3[n];
                    mean = a.o.mean[n];
                    sd = a.o.sd[n];
                }
                if constexpr (MODE == W_LOSS) rsd = 1.0f / sd;
            }
            for (int mc = 0; mc < a.mchunks; ++mc, ++tl) {
                const int b = tl & 1, use = tl >> 1;
                const int64_t mb = (int64_t)mc * W_BM + 128 * half;
                const int cnt = (int)min((int64_t)128, a.M - mb);   // rows of this half (may be <= 0)
                double y[2][16];   // 16 rows of targets in use, the next 16 in flight
                auto targets = [&](double (&v)[16], int c) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        v[j] = live && c + j < cnt ? __ldg(a.o.Y + s_off[warp - 4][c + j] + n) : 0.0;
                };
                if constexpr (MODE == W_LOSS) {
                    if (a.mchunks > 1 || tl == 0) {   // one set for the whole launch when the batch fits a chunk
                        __syncwarp();
                        for (int r = lane; r < cnt; r += 32)
                            s_off[warp - 4][r] = (a.o.idx ? (int64_t)a.o.idx[mb + r] : mb + r) * a.o.ldy;
                        __syncwarp();
                    }
                    targets(y[0], 0);   // ahead of the wait for the accumulator
                }
                if (!tc::mbar_wait(&tfull[b], use & 1)) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                auto drain = [&](int c, double (&yc)[16], double (&yn2)[16]) {
                    uint32_t r[16];
                    __syncwarp();
                    if constexpr (MODE == W_LOSS) targets(yn2, c + 16);
                    tc::tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * W_BM + 128 * half + c), r);
                    if constexpr (MODE == W_LOSS) {
                        __nv_bfloat16 *gp = a.o.dY + (mb + c) * a.o.ldo + n;
                        float tn[16];
                        bool bad = false;
#pragma unroll
                        for (int j = 0; j < 16; ++j) tn[j] = standardise(yc[j], mean, sd, rsd, bad);
                        if (bad) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) tn[j] = (float)((yc[j] - (double)mean) / (double)sd);
                        }
                        float e2[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            e2[j] = 0.0f;
                            if (live && c + j < cnt) {
                                const float yn = __uint_as_float(r[j]) + b3;
                                const float d = yn - tn[j];
                                // the exact square s2 + e2, s2 added with a two-sum
                                const float s2 = __fmul_rn(d, d);
                                e2[j] = fmaf(d, d, -s2);
                                const float ns = __fadd_rn(sq, s2), bv = __fadd_rn(ns, -sq);
                                sq_lo += (sq - (ns - bv)) + __fadd_rn(s2, -bv);
                                sq = ns;
                                const __nv_bfloat16 g = __float2bfloat16_rn(a.o.scale * d);
                                gp[j * a.o.ldo] = g;
                            }
                        }
#pragma unroll
                        for (int h = 1; h < 16; h *= 2)
#pragma unroll
                            for (int j = 0; j < 16; j += 2 * h) e2[j] += e2[j + h];
                        sq_e += e2[0];
                    } else if (live) {
                        float *cp = a.C + (mb + c) * a.ldc + n;
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (c + j < cnt) {
                                const float v = __uint_as_float(r[j]);
                                cp[j * a.ldc] = MODE == W_DENORM ? (v + b3) * sd + mean : v;
                            }
                    }
                };
#pragma unroll 1
                for (int c = 0; c < cnt; c += 32) {   // uniform across the warp
                    drain(c, y[0], y[1]);
                    if (c + 16 < cnt) drain(c + 16, y[1], y[0]);
                }
                if constexpr (MODE == W_LOSS) {
                    sum += (double)sq + ((double)sq_lo + (double)sq_e);
                    sq = sq_lo = sq_e = 0.0f;
                }
                tc::fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&tempty[b]);
            }
        }
        __syncwarp();
        if constexpr (MODE == W_LOSS) {
            double s = sum;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) a.o.part[blockIdx.x * 8 + (warp - 4)] = s;
        }
    }
    if (!ok) atomicExch(a.err, 1);
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, W_TMEM_COLS);
}

// ---------------------------------------------------------------------------
// Output-layer weight gradient g[o][h] = sum_b dY[b][o] H2[b][h], and the same
// contraction with its Adam step: the gradient goes from the TMEM accumulator
// straight into the update of w, m, v and the BF16 copy of w, so the FP32
// gradient (371 MB at 180937 x 512) is never stored.  HBM-bound: 26 bytes per
// weight (w, m, v in and out, BF16 out).
//
// Work item = 128 outputs x 128 hidden units, computed as the transposed tile
// (TMEM lane = hidden unit, so that a warp's lanes are neighbours in memory);
// both operands MN-major.  Warp 0 lane 0 loads operand slabs, warp 1 lane 0
// issues into one of four 128-column accumulators.  In the Adam form w, m and
// v come and go through shared memory by TMA, 32 outputs x 128 hidden units at
// a time in two buffers: warp 2 lane 0 loads, warps 4-11 update in place (16
// outputs each, immediate addresses), warp 3 lane 0 stores and hands the
// buffer back.  With global loads and stores by the updating threads the
// kernel issued 115 instructions per weight, mostly addresses, and took 668 us
// at that size, this form 411 us (6.1 TB/s); before the fusion gradient GEMM
// 159, Adam 511, BF16 copies 226 us.
constexpr int D_STAGES = 3;
constexpr int D_TILE_BYTES = 128 * G_SLAB * 2;
constexpr int D_ROWS = 32;                              // outputs per update chunk
constexpr int D_F32_BYTES = D_ROWS * 128 * 4;           // one of w, m, v
constexpr int D_BUF_BYTES = 3 * D_F32_BYTES + D_ROWS * 128 * 2;
constexpr size_t kGemmGradSmemBytes = 1024 + (size_t)2 * D_STAGES * D_TILE_BYTES + 256;
constexpr size_t kGemmAdamSmemBytes = kGemmGradSmemBytes + 2 * D_BUF_BYTES;

struct GemmAdamArgs {
    int64_t O, H;
    int nslab, hblocks, items;
    float *g;                // the gradient, row stride H (without ADAM)
    AdamStep s;
    int *err;
};

template <bool ADAM>
__global__ void __launch_bounds__(W_THREADS, 1)
    k_gemm_w3(const __grid_constant__ CUtensorMap hmap, const __grid_constant__ CUtensorMap ymap,
              const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap mmap,
              const __grid_constant__ CUtensorMap vmap, const __grid_constant__ CUtensorMap bmap, GemmAdamArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sH = smem, *sY = smem + D_STAGES * D_TILE_BYTES;
    uint8_t *sC = smem + 2 * D_STAGES * D_TILE_BYTES;                  // update buffers
    uint64_t *full = reinterpret_cast<uint64_t *>(sC + (ADAM ? 2 * D_BUF_BYTES : 0));
    uint64_t *empty = full + D_STAGES;
    uint64_t *tfull = empty + D_STAGES;    // [4] accumulator ready
    uint64_t *tempty = tfull + 4;          // [4] accumulator drained
    uint64_t *cfull = tempty + 4;          // [2] w, m, v loaded
    uint64_t *cdone = cfull + 2;           // [2] updated
    uint64_t *cempty = cdone + 2;          // [2] stored
    uint64_t *done = cempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < D_STAGES; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 4; ++b) {
            tc::mbar_init(&tfull[b], 1);
            tc::mbar_init(&tempty[b], 8);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&cfull[b], 1);
            tc::mbar_init(&cdone[b], 8);
            tc::mbar_init(&cempty[b], 1);
        }
        tc::mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tc::tmem_alloc(tmem_slot, 512);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    // chunks of 32 outputs with any row inside, in an item's 128
    auto chunks = [&](int ot) { return (int)min((int64_t)4, (a.O - (int64_t)ot * 128 + D_ROWS - 1) / D_ROWS); };
    if (warp == 0 && lane == 0) {
        int it = 0;
        for (int w = blockIdx.x; w < a.items && ok; w += gridDim.x) {
            const int ot = w / a.hblocks, hb = w - ot * a.hblocks;
            for (int ks = 0; ks < a.nslab; ++ks, ++it) {
                const int st = it % D_STAGES, rnd = it / D_STAGES;
                if (!tc::mbar_wait(&empty[st], (rnd & 1) ^ 1)) {
                    ok = false;
                    break;
                }
                tc::mbar_expect_tx(&full[st], 2 * D_TILE_BYTES);
                load_slab<true>(sH + st * D_TILE_BYTES, &hmap, &full[st], ks * G_SLAB, hb * 128);
                load_slab<true>(sY + st * D_TILE_BYTES, &ymap, &full[st], ks * G_SLAB, ot * 128);
            }
        }
        for (int j = max(0, it - D_STAGES); j < it; ++j)   // no copy is in flight when the CTA leaves
            if (!tc::mbar_wait(&full[j % D_STAGES], (j / D_STAGES) & 1)) ok = false;
    } else if (warp == 1 && lane == 0) {
        int it = 0, tl = 0;
        for (int w = blockIdx.x; w < a.items && ok; w += gridDim.x, ++tl) {
            const int b = tl & 3, use = tl >> 2;
            if (!tc::mbar_wait(&tempty[b], (use & 1) ^ 1)) {
                ok = false;
                break;
            }
            tc::fence_after();
            for (int ks = 0; ks < a.nslab; ++ks, ++it) {
                const int st = it % D_STAGES, rnd = it / D_STAGES;
                if (!tc::mbar_wait(&full[st], rnd & 1)) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                const uint32_t hbs = tc::smem_u32(sH + st * D_TILE_BYTES), ybs = tc::smem_u32(sY + st * D_TILE_BYTES);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    tc::mma<false, tc::instr_desc(false, 128, 128, true, true)>(
                        tmem + (uint32_t)(b * 128), slab_desc<true>(hbs, k), slab_desc<true>(ybs, k),
                        (ks > 0 || k > 0) ? 1u : 0u);
                tc::commit(&empty[st]);
            }
            if (ok) tc::commit(&tfull[b]);
        }
        tc::commit(done);
        if (!tc::mbar_wait(done, 0)) ok = false;
    } else if (ADAM && warp == 2 && lane == 0) {   // loads of w, m, v
        int it = 0;
        for (int w = blockIdx.x; w < a.items && ok; w += gridDim.x) {
            const int ot = w / a.hblocks, hb = w - ot * a.hblocks, nc = chunks(ot);
            for (int c = 0; c < nc; ++c, ++it) {
                const int b = it & 1, rnd = it >> 1;
                if (!tc::mbar_wait(&cempty[b], (rnd & 1) ^ 1)) {
                    ok = false;
                    break;
                }
                uint8_t *d = sC + b * D_BUF_BYTES;
                tc::mbar_expect_tx(&cfull[b], 3 * D_F32_BYTES);
                tc::tma_load_2d(d, &wmap, &cfull[b], hb * 128, ot * 128 + c * D_ROWS);
                tc::tma_load_2d(d + D_F32_BYTES, &mmap, &cfull[b], hb * 128, ot * 128 + c * D_ROWS);
                tc::tma_load_2d(d + 2 * D_F32_BYTES, &vmap, &cfull[b], hb * 128, ot * 128 + c * D_ROWS);
            }
        }
        for (int j = max(0, it - 2); j < it; ++j)
            if (!tc::mbar_wait(&cfull[j & 1], (j >> 1) & 1)) ok = false;
    } else if (ADAM && warp == 3 && lane == 0) {   // stores
        int it = 0;
        for (int w = blockIdx.x; w < a.items && ok; w += gridDim.x) {
            const int ot = w / a.hblocks, hb = w - ot * a.hblocks, nc = chunks(ot);
            for (int c = 0; c < nc; ++c, ++it) {
                const int b = it & 1, rnd = it >> 1;
                if (!tc::mbar_wait(&cdone[b], rnd & 1)) {
                    ok = false;
                    break;
                }
                const uint8_t *d = sC + b * D_BUF_BYTES;
                tc::tma_store_2d(&wmap, d, hb * 128, ot * 128 + c * D_ROWS);
                tc::tma_store_2d(&mmap, d + D_F32_BYTES, hb * 128, ot * 128 + c * D_ROWS);
                tc::tma_store_2d(&vmap, d + 2 * D_F32_BYTES, hb * 128, ot * 128 + c * D_ROWS);
                tc::tma_store_2d(&bmap, d + 3 * D_F32_BYTES, hb * 128, ot * 128 + c * D_ROWS);
                tc::bulk_commit();
                tc::bulk_wait_read();
                tc::mbar_arrive(&cempty[b]);
            }
        }
        tc::bulk_wait();
    } else if (warp >= 4) {
        const int q = warp & 3, half = (warp - 4) >> 2;
        int tl = 0, it = 0;
        for (int w = blockIdx.x; w < a.items && ok; w += gridDim.x, ++tl) {
            const int ot = w / a.hblocks, hb = w - ot * a.hblocks, nc = chunks(ot);
            const int b = tl & 3, use = tl >> 2;
            if (!tc::mbar_wait(&tfull[b], use & 1)) {
                ok = false;
                break;
            }
            tc::fence_after();
            for (int c = 0; c < nc; ++c, ++it) {
                uint32_t r[16];
                __syncwarp();
                tc::tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * 128 + D_ROWS * c + 16 * half), r);
                if constexpr (ADAM) {
                    if (!tc::mbar_wait(&cfull[it & 1], (it >> 1) & 1)) {
                        ok = false;
                        break;
                    }
                    uint8_t *d = sC + (it & 1) * D_BUF_BYTES;
                    float *wp = reinterpret_cast<float *>(d) + 16 * half * 128 + 32 * q + lane;
                    float *mp = wp + D_F32_BYTES / 4, *vp = mp + D_F32_BYTES / 4;
                    __nv_bfloat16 *bp =
                        reinterpret_cast<__nv_bfloat16 *>(d + 3 * D_F32_BYTES) + 16 * half * 128 + 32 * q + lane;
                    float m[16], v[16], up[16];
                    bool bad = false;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        m[j] = mp[j * 128];
                        v[j] = vp[j * 128];
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) up[j] = adam_moments(a.s, __uint_as_float(r[j]), m[j], v[j], bad);
                    if (bad) {
#pragma unroll 1
                        for (int j = 0; j < 16; ++j) {   // rare: the moments again from the stored ones
                            float mj = mp[j * 128], vj = vp[j * 128], rj = 0.0f;
#pragma unroll
                            for (int t = 0; t < 16; ++t) rj = t == j ? __uint_as_float(r[t]) : rj;
                            adam_ema(a.s, rj, mj, vj);
                            const float uj = adam_quotient(a.s, mj, vj);
#pragma unroll
                            for (int t = 0; t < 16; ++t) up[t] = t == j ? uj : up[t];
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float x = wp[j * 128] - up[j];
                        wp[j * 128] = x;
                        mp[j * 128] = m[j];
                        vp[j * 128] = v[j];
                        bp[j * 128] = __float2bfloat16_rn(x);
                    }
                    tc::fence_async_shared();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&cdone[it & 1]);
                } else {
                    const int64_t h = (int64_t)hb * 128 + 32 * q + lane;
                    const int64_t o0 = (int64_t)ot * 128 + D_ROWS * c + 16 * half;
                    if (h < a.H) {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (o0 + j < a.O) a.g[(o0 + j) * a.H + h] = __uint_as_float(r[j]);
                    }
                }
            }
            tc::fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&tempty[b]);
        }
    }
    if (!ok) atomicExch(a.err, 1);
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// C[m][n] = sum_s part[s][m][n]  (fixed order)
__global__ void k_gemm_reduce(int64_t M, int64_t N, int nsplit, const float *__restrict__ part, float *__restrict__ C,
                              int64_t ldc) {
    const int64_t total = M * N;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        float s = 0.0f;
        for (int k = 0; k < nsplit; ++k) s += part[(size_t)k * total + e];
        C[(e / N) * ldc + e % N] = s;
    }
}

struct GemmPlan {
    int64_t tm, tn;
    int total_slabs, nsplit, slabs_per_split;
};

GemmPlan gemm_plan(int64_t M, int64_t N, int64_t K, int num_sms) {
    GemmPlan p{};
    p.tm = (M + G_TILE - 1) / G_TILE;
    p.tn = (N + G_TILE - 1) / G_TILE;
    p.total_slabs = (int)((K + G_SLAB - 1) / G_SLAB);
    const int64_t tiles = p.tm * p.tn;
    int s = 1;
    if (tiles < 2LL * num_sms && p.total_slabs >= 8)
        s = (int)std::min<int64_t>((2LL * num_sms + tiles - 1) / tiles, p.total_slabs / 4);
    s = std::max(1, s);
    p.slabs_per_split = (p.total_slabs + s - 1) / s;
    p.nsplit = p.slabs_per_split > 0 ? (p.total_slabs + p.slabs_per_split - 1) / p.slabs_per_split : 1;
    p.nsplit = std::max(1, p.nsplit);
    return p;
}

// the persistent column-tile kernel: at least one column tile per SM, K of at
// least one slab
bool gemm_wide(int64_t M, int64_t N, int64_t K, int num_sms) {
    return M <= (1 << 22) && K >= 1 && (N + W_BN - 1) / W_BN >= num_sms && (N + W_BN - 1) / W_BN < (1LL << 31);
}

template <WideMode MODE>
void launch_wide(cudaStream_t s, int num_sms, const __nv_bfloat16 *A, int64_t lda, const __nv_bfloat16 *B, int64_t ldb,
                 int64_t M, int64_t N, int64_t K, GemmWideArgs wa) {
    CUtensorMap amap, bmap;
    tc::encode_2d(&amap, A, false, (uint64_t)K, (uint64_t)M, (uint64_t)std::max<int64_t>(lda, 8), G_SLAB, W_BM);
    tc::encode_2d(&bmap, B, false, (uint64_t)K, (uint64_t)N, (uint64_t)std::max<int64_t>(ldb, 8), G_SLAB, W_BN);
    wa.M = M;
    wa.N = N;
    wa.ntiles = (int)((N + W_BN - 1) / W_BN);
    wa.nslab = (int)((K + G_SLAB - 1) / G_SLAB);
    wa.mchunks = (int)((M + W_BM - 1) / W_BM);
    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_gemm_bf16_wide<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kGemmWideSmemBytes);
    }));
    k_gemm_bf16_wide<MODE><<<std::min(wa.ntiles, num_sms), W_THREADS, kGemmWideSmemBytes, s>>>(amap, bmap, wa);
    MDSIP_LAUNCHED();
}

template <bool AMN, bool BMN>
void launch_tiles(cudaStream_t s, dim3 grid, const CUtensorMap &amap, const CUtensorMap &bmap, const GemmArgs &a) {
    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_gemm_bf16<AMN, BMN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kGemmSmemBytes);
    }));
    k_gemm_bf16<AMN, BMN><<<grid, G_THREADS, kGemmSmemBytes, s>>>(amap, bmap, a);
    MDSIP_LAUNCHED();
}

}  // namespace

size_t gemm_bf16_ws_bytes(int64_t M, int64_t N, int64_t K, int num_sms, bool amn, bool bmn) {
    if (!amn && !bmn && gemm_wide(M, N, K, num_sms)) return 0;
    const GemmPlan p = gemm_plan(M, N, K, num_sms);
    return p.nsplit > 1 ? (size_t)p.nsplit * M * N * sizeof(float) : 0;
}

// C = A B^T.  A: M x K BF16 (row stride lda elements), or K x M with amn; B:
// N x K (ldb), or K x N with bmn; 16-byte aligned with lda, ldb multiples of
// 8.  C: FP32, row stride ldc.  ws: gemm_bf16_ws_bytes of the same arguments.
// err_dev: device int.
void launch_gemm_bf16(cudaStream_t s, int num_sms, const __nv_bfloat16 *A, int64_t lda, const __nv_bfloat16 *B,
                      int64_t ldb, int64_t M, int64_t N, int64_t K, float *C, int64_t ldc, void *ws, int *err_dev,
                      bool amn, bool bmn) {
    if (M <= 0 || N <= 0) return;
    MDSIP_REQUIRE(K >= 0 && lda >= (amn ? M : K) && ldb >= (bmn ? N : K) && ldc >= N, MDSIP_ERR_INVALID_ARG,
                  "gemm: bad leading dimension");
    MDSIP_REQUIRE(M < (1LL << 31) / G_TILE * G_TILE && N < (1LL << 31) / G_TILE * G_TILE, MDSIP_ERR_INVALID_ARG,
                  "gemm: dimension too large");
    const GemmPlan p = gemm_plan(M, N, K, num_sms);
    if (!amn && !bmn && gemm_wide(M, N, K, num_sms)) {
        GemmWideArgs wa{};
        wa.C = C;
        wa.ldc = ldc;
        wa.err = err_dev;
        launch_wide<W_STORE>(s, num_sms, A, lda, B, ldb, M, N, K, wa);
        return;
    }
    MDSIP_REQUIRE(p.tm <= 65535, MDSIP_ERR_INVALID_ARG, "gemm: M too large");
    const uint64_t k1 = (uint64_t)std::max<int64_t>(K, 1);
    CUtensorMap amap, bmap;
    if (amn)
        tc::encode_2d(&amap, A, false, (uint64_t)M, k1, (uint64_t)std::max<int64_t>(lda, 8), 64, G_SLAB);
    else
        tc::encode_2d(&amap, A, false, k1, (uint64_t)M, (uint64_t)std::max<int64_t>(lda, 8), G_SLAB, G_TILE);
    if (bmn)
        tc::encode_2d(&bmap, B, false, (uint64_t)N, k1, (uint64_t)std::max<int64_t>(ldb, 8), 64, G_SLAB);
    else
        tc::encode_2d(&bmap, B, false, k1, (uint64_t)N, (uint64_t)std::max<int64_t>(ldb, 8), G_SLAB, G_TILE);
    GemmArgs a{};
    a.M = M;
    a.N = N;
    a.total_slabs = p.total_slabs;
    a.slabs_per_split = p.slabs_per_split;
    a.err = err_dev;
    if (p.nsplit > 1) {
        MDSIP_REQUIRE(ws != nullptr, MDSIP_ERR_INVALID_ARG, "gemm: missing split workspace");
        a.out = static_cast<float *>(ws);
        a.ldo = N;
        a.split_stride = M * N;
    } else {
        a.out = C;
        a.ldo = ldc;
        a.split_stride = 0;
    }
    const dim3 grid((unsigned)p.tn, (unsigned)p.tm, (unsigned)p.nsplit);
    if (amn && bmn) launch_tiles<true, true>(s, grid, amap, bmap, a);
    else if (amn) launch_tiles<true, false>(s, grid, amap, bmap, a);
    else if (bmn) launch_tiles<false, true>(s, grid, amap, bmap, a);
    else launch_tiles<false, false>(s, grid, amap, bmap, a);
    if (p.nsplit > 1) {
        const int g = (int)std::max<int64_t>(1, std::min<int64_t>(num_sms * 8, ceil_div(M * N, 256)));
        k_gemm_reduce<<<g, 256, 0, s>>>(M, N, p.nsplit, a.out, C, ldc);
        MDSIP_LAUNCHED();
    }
}

// Output layer of the network: A = h2 (batch x K), B = W3 (N x K).  With
// o.Y == nullptr the predictions go to Yout (row stride ldy); otherwise the
// loss partials and dL/dyn (BF16) of o (o.part: 8 values per CTA, the count is
// returned).
int launch_out_layer(cudaStream_t s, int num_sms, const __nv_bfloat16 *A, int64_t lda, const __nv_bfloat16 *B,
                     int64_t ldb, int64_t batch, int64_t N, int64_t K, const OutLayer &o, float *Yout, int64_t ldy,
                     int *err_dev) {
    MDSIP_REQUIRE(N < (1LL << 31) / W_BN * W_BN, MDSIP_ERR_INVALID_ARG, "gemm: dimension too large");
    GemmWideArgs wa{};
    wa.C = Yout;
    wa.ldc = ldy;
    wa.err = err_dev;
    wa.o = o;
    if (o.Y) launch_wide<W_LOSS>(s, num_sms, A, lda, B, ldb, batch, N, K, wa);
    else launch_wide<W_DENORM>(s, num_sms, A, lda, B, ldb, batch, N, K, wa);
    return 8 * std::min((int)((N + W_BN - 1) / W_BN), num_sms);
}

static GemmAdamArgs w3_args(int64_t batch, int64_t O, int64_t H, int *err_dev) {
    GemmAdamArgs a{};
    a.O = O;
    a.H = H;
    a.nslab = (int)((batch + G_SLAB - 1) / G_SLAB);
    a.hblocks = (int)((H + 127) / 128);
    const int64_t items = (O + 127) / 128 * a.hblocks;
    MDSIP_REQUIRE(items < (1LL << 31), MDSIP_ERR_INVALID_ARG, "gemm: dimension too large");
    a.items = (int)items;
    a.err = err_dev;
    return a;
}

// g (O x H) = dY^T H2.  H2: batch x H (row stride ldh), dY: batch x O (ldo).
void launch_gemm_w3_grad(cudaStream_t s, int num_sms, const __nv_bfloat16 *H2, int64_t ldh, const __nv_bfloat16 *dY,
                         int64_t ldo, int64_t batch, int64_t O, int64_t H, float *g, int *err_dev) {
    CUtensorMap hmap, ymap;
    tc::encode_2d(&hmap, H2, false, (uint64_t)H, (uint64_t)batch, (uint64_t)ldh, 64, G_SLAB);
    tc::encode_2d(&ymap, dY, false, (uint64_t)O, (uint64_t)batch, (uint64_t)ldo, 64, G_SLAB);
    GemmAdamArgs a = w3_args(batch, O, H, err_dev);
    a.g = g;
    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_gemm_w3<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kGemmGradSmemBytes);
    }));
    k_gemm_w3<false><<<std::min(a.items, num_sms), W_THREADS, kGemmGradSmemBytes, s>>>(hmap, ymap, hmap, hmap, hmap,
                                                                                     hmap, a);
    MDSIP_LAUNCHED();
}

// One Adam step of w (O x H, with m and v, packed rows, 16-byte aligned) and of
// its BF16 copy wb (row stride ldb) on the gradient dY^T H2, bit for bit
// launch_gemm_w3_grad's.  H must be a multiple of 4 (rows of w on 16 bytes).
void launch_gemm_w3_adam(cudaStream_t s, int num_sms, const __nv_bfloat16 *H2, int64_t ldh, const __nv_bfloat16 *dY,
                         int64_t ldo, int64_t batch, int64_t O, int64_t H, float *w, float *m, float *v,
                         __nv_bfloat16 *wb, int64_t ldb, const AdamStep &st, int *err_dev) {
    CUtensorMap hmap, ymap, wmap, mmap, vmap, bmap;
    tc::encode_2d(&hmap, H2, false, (uint64_t)H, (uint64_t)batch, (uint64_t)ldh, 64, G_SLAB);
    tc::encode_2d(&ymap, dY, false, (uint64_t)O, (uint64_t)batch, (uint64_t)ldo, 64, G_SLAB);
    tc::encode_2d(&wmap, w, true, (uint64_t)H, (uint64_t)O, (uint64_t)H, 128, D_ROWS, 0);
    tc::encode_2d(&mmap, m, true, (uint64_t)H, (uint64_t)O, (uint64_t)H, 128, D_ROWS, 0);
    tc::encode_2d(&vmap, v, true, (uint64_t)H, (uint64_t)O, (uint64_t)H, 128, D_ROWS, 0);
    tc::encode_2d(&bmap, wb, false, (uint64_t)H, (uint64_t)O, (uint64_t)ldb, 128, D_ROWS, 0);
    GemmAdamArgs a = w3_args(batch, O, H, err_dev);
    a.s = st;
    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_gemm_w3<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kGemmAdamSmemBytes);
    }));
    k_gemm_w3<true><<<std::min(a.items, num_sms), W_THREADS, kGemmAdamSmemBytes, s>>>(hmap, ymap, wmap, mmap, vmap,
                                                                                    bmap, a);
    MDSIP_LAUNCHED();
}

}  // namespace mdsip

extern "C" mdsip_status mdsip_gemm_bf16(mdsip_ctx *hctx, int64_t M, int64_t N, int64_t K, const uint16_t *A,
                                        int64_t lda, const uint16_t *B, int64_t ldb, float *C, int64_t ldc) {
    if (!hctx) return MDSIP_ERR_INVALID_ARG;
    mdsip::Ctx *ctx = reinterpret_cast<mdsip::Ctx *>(hctx);
    return mdsip::guarded(ctx, [&] {
        mdsip::DeviceGuard g(ctx->device);
        MDSIP_REQUIRE(M >= 0 && N >= 0 && K >= 0, MDSIP_ERR_INVALID_ARG, "gemm: negative size");
        if (M == 0 || N == 0) return;
        MDSIP_REQUIRE(A && B && C, MDSIP_ERR_INVALID_ARG, "gemm: null pointer");
        MDSIP_REQUIRE(lda % 8 == 0 && ldb % 8 == 0 && reinterpret_cast<uintptr_t>(A) % 16 == 0 &&
                          reinterpret_cast<uintptr_t>(B) % 16 == 0,
                      MDSIP_ERR_INVALID_ARG, "gemm: A and B need 16-byte aligned rows (lda, ldb multiples of 8)");
        const size_t ws = mdsip::gemm_bf16_ws_bytes(M, N, K, ctx->num_sms);
        const size_t wsa = (ws + 255) / 256 * 256;
        char *base = static_cast<char *>(ctx->scratch_at_least(wsa + 256));
        int *err = reinterpret_cast<int *>(base + wsa);
        MDSIP_CUDA(cudaMemsetAsync(err, 0, sizeof(int), ctx->stream));
        mdsip::launch_gemm_bf16(ctx->stream, ctx->num_sms, reinterpret_cast<const __nv_bfloat16 *>(A), lda,
                                reinterpret_cast<const __nv_bfloat16 *>(B), ldb, M, N, K, C, ldc,
                                ws ? base : nullptr, err);
        int herr = 0;
        MDSIP_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        MDSIP_CUDA(cudaStreamSynchronize(ctx->stream));
        MDSIP_REQUIRE(herr == 0, MDSIP_ERR_DEVICE, "gemm: a bounded device wait expired");
    });
}
