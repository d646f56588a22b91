// Solve with the Bunch-Kaufman factor P K P^T = L D L^T (Section 2.3):
//
//     x = L^-1 P b,   w = D^-1 x,   z = L^-T w,   b <- P^T z.
//
// N is a few thousand at most, so the time of a solve is its dependency
// chain, not its 2 N^2 flops.  The layout and schedule are built around that
// chain:
//
//  * once per factorization, L is copied into 64 x 64 tiles (column-major
//    inside a tile, in FP64 or, for the refined mixed-precision path, FP32):
//    F(I, J) = L_IJ for J < I and F(I, I) = inv(L_II) for the forward sweep,
//    and their transposes for the backward sweep, so that every tile
//    product in both sweeps reads its tile with lanes along contiguous rows;
//  * one CTA per 64-row block row (cooperative launch, so all are resident).
//    The CTA of block row I accumulates L_IJ x_J for J < I as soon as block J
//    has published x_J (words tagged with the launch's epoch, no grid-wide
//    barrier), has its tiles in registers before it waits, and finishes with
//    inv(L_II); the backward sweep runs the same way from the last block up;
//  * D^-1 (1x1 and 2x2 blocks) is applied per block row between the sweeps;
//    a 2x2 block that straddles two block rows waits for the neighbour's
//    forward result.
//
// Words hold the epoch of the launch that set them, so no reset is needed
// between solves; the last CTA to finish advances the epoch.  Every wait is
// bounded and sets the error flag on expiry.
#include <algorithm>

#include "internal.cuh"

namespace mdsip {

namespace {

constexpr int kBS = 64;            // block rows and tile edge
constexpr int kThreads = 256;      // 64 rows x 4 column quarters
constexpr int kTile = kBS * kBS;
constexpr int kSolveRhs = 4;       // right-hand sides side by side

__host__ __device__ inline int64_t tile_index(int64_t I, int64_t J) { return I * (I + 1) / 2 + J; }  // J <= I

struct Layout {
    int nblk = 0;
    int64_t ntile = 0;
    size_t off_x = 0, off_z = 0, off_F = 0, off_B = 0, total = 0;
};

Layout layout_for(int64_t N) {
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    Layout l;
    l.nblk = (int)((std::max<int64_t>(N, 1) + kBS - 1) / kBS);
    l.ntile = (int64_t)l.nblk * (l.nblk + 1) / 2;
    size_t o = 256;                                    // epoch, done counter
    l.off_x = o; o += al(kSolveRhs * (size_t)l.nblk * kBS * 2 * sizeof(double));   // two tagged words per value
    l.off_z = o; o += al(kSolveRhs * (size_t)l.nblk * kBS * 2 * sizeof(double));
    l.off_F = o; o += al((size_t)l.ntile * kTile * sizeof(double));
    l.off_B = o; o += al((size_t)l.ntile * kTile * sizeof(double));
    l.total = o;
    return l;
}

// Tiles of one factorization.  Blocks past the diagonal blocks' shares: tile
// t = tile_index(I, J), J < I, copied in both orders.  Before them, diagonal
// block I's inverse of the unit lower triangle.  FP64: kDiagParts thread blocks
// of four columns, a warp per column (lane r holds rows r and r + 32 and the
// entries already known come by shuffle), so that one column's chain of 63
// products is all that is serial; every entry sums its products in the order
// of the column sweep.  (One thread per column did 2016 of them in turn, each
// 64 cycles of the FP64 pipe: 104 us at any order, here 10 at
// N <= 64 and 21 at N = 2003.)
constexpr int kDiagParts = 16;

template <typename T>
__global__ void __launch_bounds__(kThreads) k_solve_tiles(int N, const double *__restrict__ L, T *__restrict__ F,
                                                          T *__restrict__ Bk) {
    __shared__ double s[kBS][kBS + 1];
    constexpr int parts = sizeof(T) == sizeof(double) ? kDiagParts : 1;
    const int nblk = (N + kBS - 1) / kBS, ndiag = nblk * parts;
    int I, J;
    if ((int)blockIdx.x < ndiag) {
        I = J = blockIdx.x / parts;
    } else {
        const int64_t o = (int64_t)blockIdx.x - ndiag;   // I (I - 1) / 2 + J, J < I
        I = (int)((sqrtf(8.0f * (float)o + 1.0f) + 1.0f) * 0.5f);
        while ((int64_t)(I + 1) * I / 2 <= o) ++I;
        while ((int64_t)I * (I - 1) / 2 > o) --I;
        J = (int)(o - (int64_t)I * (I - 1) / 2);
    }
    const int64_t t = (int64_t)I * (I + 1) / 2 + J;
    const int tid = threadIdx.x;
    T *f = F + t * kTile, *bk = Bk + t * kTile;
    if (J < I) {
        // s[r][c] = L[64I + r][64J + c]  (read along r: L is column-major)
        for (int e = tid; e < kTile; e += kThreads) {
            const int r = e & (kBS - 1), c = e >> 6;
            const int64_t gr = (int64_t)I * kBS + r, gc = (int64_t)J * kBS + c;
            const double v = (gr < N && gc < N) ? L[gr + gc * (int64_t)N] : 0.0;
            s[r][c] = v;
            f[c * kBS + r] = (T)v;
        }
        __syncthreads();
        for (int e = tid; e < kTile; e += kThreads) {
            const int r = e & (kBS - 1), c = e >> 6;   // Bk(r = j, c = i) = L[64I + i][64J + j]
            bk[c * kBS + r] = (T)s[c][r];
        }
        return;
    }
    // diagonal block: inverse of the unit lower triangle, column c by forward substitution
    const int jb = I * kBS, bw = min(kBS, N - jb);
    if constexpr (sizeof(T) == sizeof(float)) {
        // FP32 tiles (the refined path's approximate solves): the inverse in FP32 arithmetic,
        // four partial sums per entry.  On the FP64 pipe (1/64 of the FP32 rate) the 2016
        // dependent products of a column made this launch take about 0.1 ms at N = 2050.
        float(*sf)[kBS + 1] = reinterpret_cast<float(*)[kBS + 1]>(&s[0][0]);   // s's storage
        for (int e = tid; e < kTile; e += kThreads) {
            const int r = e & (kBS - 1), c = e >> 6;
            sf[r][c] = (r < bw && c < bw) ? (float)L[(jb + r) + (int64_t)(jb + c) * N] : 0.0f;
        }
        __syncthreads();
        float xf[kBS];
        const int c = tid;
        if (c < kBS) {
#pragma unroll
            for (int i = 0; i < kBS; ++i) {
                float v[4] = {(i == c) ? 1.0f : 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int j = 0; j < i; ++j) v[j & 3] = fmaf(-sf[i][j], xf[j], v[j & 3]);
                xf[i] = i < c ? 0.0f : (v[0] + v[1]) + (v[2] + v[3]);
            }
        }
        __syncthreads();
        if (c < kBS) {
#pragma unroll
            for (int i = 0; i < kBS; ++i) sf[i][c] = (i < bw && c < bw) ? xf[i] : 0.0f;
        }
        __syncthreads();
        for (int e = tid; e < kTile; e += kThreads) {
            const int r = e & (kBS - 1), cc = e >> 6;
            f[cc * kBS + r] = (T)sf[r][cc];    // F(I, I)(r, c) = inv(L_II)[r][c]
            bk[cc * kBS + r] = (T)sf[cc][r];   // B(I, I)(r, c) = inv(L_II)[c][r]
        }
        return;
    }
    for (int e = tid; e < kTile; e += kThreads) {
        const int r = e & (kBS - 1), c = e >> 6;
        s[r][c] = (r < bw && c < bw) ? L[(jb + r) + (int64_t)(jb + c) * N] : 0.0;
    }
    __syncthreads();
    const int lane = tid & 31, c = (int)(blockIdx.x % parts) * (kBS / parts) + (tid >> 5);
    if ((tid >> 5) >= kBS / parts) return;
    double x0 = lane == c ? 1.0 : 0.0, x1 = lane + 32 == c ? 1.0 : 0.0;
    for (int j = c; j < min(bw, 32) - 1; ++j) {
        const double xj = __shfl_sync(0xffffffffu, x0, j);
        if (lane > j) x0 = fma(-s[lane][j], xj, x0);
        if (bw > 32) x1 = fma(-s[lane + 32][j], xj, x1);
    }
    for (int j = max(c, 31); j < bw - 1; ++j) {
        const double xj = __shfl_sync(0xffffffffu, j < 32 ? x0 : x1, j & 31);
        if (lane + 32 > j) x1 = fma(-s[lane + 32][j], xj, x1);
    }
    x0 = lane < bw && c < bw ? x0 : 0.0;
    x1 = lane + 32 < bw && c < bw ? x1 : 0.0;
    f[c * kBS + lane] = (T)x0;                // F(I, I)(r, c) = inv(L_II)[r][c]
    f[c * kBS + lane + 32] = (T)x1;
    bk[lane * kBS + c] = (T)x0;               // B(I, I)(r, c) = inv(L_II)[c][r]
    bk[(lane + 32) * kBS + c] = (T)x1;
}

// partial of (tile * v)[r] over the column quarter q, tile in registers
template <typename T>
__device__ __forceinline__ void load_quarter(const T *tile, int r, int q, T (&reg)[16]) {
    const T *p = tile + (16 * q) * kBS + r;
#pragma unroll
    for (int c = 0; c < 16; ++c) reg[c] = __ldg(p + c * kBS);
}

template <typename T>
__device__ __forceinline__ T dot_quarter(const T (&reg)[16], const T *sv, int q, T acc) {
#pragma unroll
    for (int c = 0; c < 16; ++c) acc = fma(reg[c], sv[16 * q + c], acc);
    return acc;
}

// A block's result travels as 64-bit words (32 bits of a value | epoch << 32; an
// FP64 value takes two), so one load both tests that block J is published and
// delivers x_J: no separate flags, no fences between value and flag.
template <typename T>
struct TagSolve {
    int N, nblk;
    const T *F, *Bk;
    const double *Dd, *Doff;
    const int32_t *perm;
    double *b;
    int64_t ldb;
    unsigned long long *xw, *zw;   // tagged block results, kSolveRhs sets
    unsigned *epoch, *done;
    int *err;
};

__device__ __forceinline__ void tag_store(unsigned long long *w, int64_t i, float v, unsigned e) {
    w[i] = ((unsigned long long)e << 32) | (unsigned long long)__float_as_uint(v);
}
__device__ __forceinline__ void tag_store(unsigned long long *w, int64_t i, double v, unsigned e) {
    const unsigned long long t = (unsigned long long)e << 32;
    *reinterpret_cast<ulonglong2 *>(w + 2 * i) =
        make_ulonglong2(t | (unsigned)__double2loint(v), t | (unsigned)__double2hiint(v));
}
__device__ __forceinline__ bool tag_load(const unsigned long long *w, int64_t i, unsigned e, float &v) {
    const unsigned long long x = *((volatile const unsigned long long *)w + i);
    v = __uint_as_float((unsigned)x);
    return (unsigned)(x >> 32) == e;
}
__device__ __forceinline__ bool tag_load(const unsigned long long *w, int64_t i, unsigned e, double &v) {
    unsigned long long x, y;
    asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(w + 2 * i) : "memory");
    v = __hiloint2double((int)(unsigned)y, (int)(unsigned)x);
    return (unsigned)(x >> 32) == e && (unsigned)(y >> 32) == e;
}

// value i once its words carry epoch e (bounded wait; false on expiry)
template <typename T>
__device__ __forceinline__ bool tag_wait(const unsigned long long *w, int64_t i, unsigned e, int *err, T &v) {
    if (tag_load(w, i, e, v)) return true;
    const long long t0 = clock64();
    while (!tag_load(w, i, e, v))
        if (*((volatile int *)err) != 0 || clock64() - t0 > kBarrierLimitCycles) {
            atomicExch(err, 1);
            return false;
        }
    return true;
}

// Grid: CTAs over block rows (x), right-hand sides (y), each with its own set of
// result words.  What does not depend on the last block to arrive -- the
// diagonal tile, its predecessor's tile, the right-hand side -- is loaded
// before the wait for it: a step of the chain is one exchange through L2, two
// 64 x 64 products and three barriers.  Blocks before the last come kB at a
// time (FP32: a round trip for four tiles; FP64: a product is bound by the FP64
// pipe, so one, with the next tile on its way).  N = 2050: FP32 113 -> 52 us,
// FP64 311 -> 195 (which had a flag, a fence and a second load per block).
template <typename T>
__global__ void __launch_bounds__(kThreads) k_ldlt_solve_tagged(TagSolve<T> p) {
    constexpr int kB = sizeof(T) == sizeof(float) ? 4 : 1;
    constexpr int kW = sizeof(T) / sizeof(float);
    __shared__ T sv[kB][kBS], sy[kBS];
    __shared__ T spart[4][kBS], spart2[4][kBS];
    __shared__ unsigned s_e;
    const int tid = threadIdx.x, r = tid & (kBS - 1), q = tid >> 6;
    const int G = (int)gridDim.x, N = p.N, nblk = p.nblk;
    const int64_t set = (int64_t)blockIdx.y * nblk * kBS * kW;
    unsigned long long *const xw = p.xw + set, *const zw = p.zw + set;
    double *const bvec = p.b + (int64_t)blockIdx.y * p.ldb;
    if (tid == 0) s_e = *((volatile unsigned *)p.epoch) + 1u;
    __syncthreads();
    const unsigned e = s_e;
    bool ok = true;   // the same in every thread: agreed on at a barrier
    T reg[kB][16], lt[16], dg[16];

    // sum over `count` blocks J0, J0 + step, .. of tile(J) v_J, results in words w; the last one's tile in lt
    auto accumulate = [&](auto tile_of, const unsigned long long *w, int J0, int count, int step) {
        T acc = (T)0;
        if (kB == 1 && count > 1) load_quarter(tile_of(J0), r, q, reg[0]);
        for (int j = 0; j < count;) {
            const bool last = j == count - 1;
            const int nbat = last ? 1 : min(kB, count - 1 - j);
            T nx[16];
            if (!last) {
                if (kB > 1) {
#pragma unroll
                    for (int bq = 0; bq < kB; ++bq)
                        if (bq < nbat) load_quarter(tile_of(J0 + (j + bq) * step), r, q, reg[bq]);
                } else if (j + 2 < count) {
                    load_quarter(tile_of(J0 + (j + 1) * step), r, q, nx);
                }
            }
            const int bq = tid >> 6;   // thread t fetches value t % 64 of block t / 64
            bool got = true;
            if (bq < nbat) {
                T v = (T)0;
                got = tag_wait(w, (int64_t)(J0 + (j + bq) * step) * kBS + r, e, p.err, v);
                sv[bq][r] = v;
            }
            ok = __syncthreads_and(got);
            if (!ok) break;
            if (last) {
                acc = dot_quarter(lt, sv[0], q, acc);
                break;   // the caller's barrier follows
            }
#pragma unroll
            for (int bq2 = 0; bq2 < kB; ++bq2)
                if (bq2 < nbat) acc = dot_quarter(reg[bq2], sv[bq2], q, acc);
            __syncthreads();
            if (kB == 1 && j + 2 < count)
#pragma unroll
                for (int c = 0; c < 16; ++c) reg[0][c] = nx[c];
            j += nbat;
        }
        return acc;
    };
    // block row's result from its right-hand side y (threads 0 .. 63) and the sum: inv(L_II) (y - acc)
    auto finish = [&](T y, T acc) -> T {
        spart[q][r] = acc;
        __syncthreads();
        if (tid < kBS) sy[tid] = y - ((spart[0][tid] + spart[1][tid]) + (spart[2][tid] + spart[3][tid]));
        __syncthreads();
        spart2[q][r] = dot_quarter(dg, sy, q, (T)0);
        __syncthreads();
        return tid < kBS ? (spart2[0][tid] + spart2[1][tid]) + (spart2[2][tid] + spart2[3][tid]) : (T)0;
    };

    // ---------------- forward: x_I = inv(L_II) (P b - sum_J<I L_IJ x_J) ----------------
    for (int I = blockIdx.x; I < nblk; I += G) {
        load_quarter(p.F + tile_index(I, I) * kTile, r, q, dg);
        if (I > 0) load_quarter(p.F + tile_index(I, I - 1) * kTile, r, q, lt);
        T y0 = (T)0;
        if (tid < kBS && I * kBS + tid < N) y0 = (T)bvec[p.perm[I * kBS + tid]];
        const T acc = accumulate([&](int J) { return p.F + tile_index(I, J) * kTile; }, xw, 0, I, 1);
        if (!ok) break;
        const T xi = finish(y0, acc);
        if (tid < kBS) tag_store(xw, (int64_t)I * kBS + tid, xi, e);
        __syncthreads();
    }

    // ---------------- w = D^-1 x, then z_I = inv(L_II)^T (w_I - sum_J>I L_JI^T z_J) ----------------
    int first = (int)blockIdx.x;
    while (first + G < nblk) first += G;
    for (int I = first; ok && I >= 0 && (int)blockIdx.x < nblk; I -= G) {
        load_quarter(p.Bk + tile_index(I, I) * kTile, r, q, dg);
        if (I + 1 < nblk) load_quarter(p.Bk + tile_index(I + 1, I) * kTile, r, q, lt);
        T w = (T)0;
        bool got = true;
        if (tid < kBS) {
            const int k = I * kBS + tid;
            if (k < N) {
                // x of rows k and k + 1 (a 2x2 block may straddle into block I + 1)
                auto xval = [&](int kk) {
                    T v = (T)0;
                    got = tag_wait(xw, kk, e, p.err, v) && got;
                    return (double)v;
                };
                const double off = p.Doff[k];
                if (off != 0.0) {
                    const double a = p.Dd[k], c = p.Dd[k + 1];
                    const double u = xval(k), v = xval(k + 1);
                    w = (T)((c * u - off * v) / (a * c - off * off));
                } else if (k > 0 && p.Doff[k - 1] != 0.0) {
                    const double a = p.Dd[k - 1], c = p.Dd[k], o2 = p.Doff[k - 1];
                    const double u = xval(k - 1), v = xval(k);
                    w = (T)((a * v - o2 * u) / (a * c - o2 * o2));
                } else {
                    w = (T)ddiv(xval(k), p.Dd[k]);
                }
            }
        }
        ok = __syncthreads_and(got);
        if (!ok) break;
        const T acc = accumulate([&](int J) { return p.Bk + tile_index(J, I) * kTile; }, zw, nblk - 1, nblk - 1 - I, -1);
        if (!ok) break;
        const T zi = finish(w, acc);
        if (tid < kBS) {
            tag_store(zw, (int64_t)I * kBS + tid, zi, e);
            const int row = I * kBS + tid;
            if (row < N) bvec[p.perm[row]] = (double)zi;
        }
        __syncthreads();
    }

    // the last CTA to finish advances the epoch (every CTA has read it by then:
    // none can finish before all of its right-hand side have published their
    // backward blocks, and the counter waits for every right-hand side)
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const unsigned d = atomicAdd(p.done, 1u);
        if (d == (unsigned)G * gridDim.y - 1u) {
            atomicExch(p.done, 0u);
            __threadfence();
            atomicAdd(p.epoch, 1u);
        }
    }
}

// As many right-hand sides at once as fit the device beside one another: their
// chains run side by side (N = 2003, four: 1208 us one after the other, 189 so).
template <typename T>
void launch_solve_t(cudaStream_t s, int num_sms, int64_t N, const double *Dd, const double *Doff,
                    const int32_t *perm, int64_t nrhs, double *B, int64_t ldb, char *w, int *err_dev) {
    const Layout l = layout_for(N);
    TagSolve<T> p{};
    p.N = (int)N;
    p.nblk = l.nblk;
    p.F = reinterpret_cast<const T *>(w + l.off_F);
    p.Bk = reinterpret_cast<const T *>(w + l.off_B);
    p.Dd = Dd;
    p.Doff = Doff;
    p.perm = perm;
    p.ldb = ldb;
    p.xw = reinterpret_cast<unsigned long long *>(w + l.off_x);
    p.zw = reinterpret_cast<unsigned long long *>(w + l.off_z);
    p.epoch = reinterpret_cast<unsigned *>(w);
    p.done = reinterpret_cast<unsigned *>(w + 4);
    p.err = err_dev;
    int per_sm = 0;
    MDSIP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ldlt_solve_tagged<T>, kThreads, 0));
    MDSIP_REQUIRE(per_sm >= 1, MDSIP_ERR_INVALID_ARG, "ldlt_solve: kernel does not fit on an SM");
    const int64_t room = (int64_t)num_sms * per_sm;
    const int grid = (int)std::min<int64_t>(l.nblk, room);
    const int64_t side = std::min<int64_t>(kSolveRhs, std::max<int64_t>(1, (int64_t)num_sms / grid));
    for (int64_t rr = 0; rr < nrhs; rr += side) {
        p.b = B + rr * ldb;
        void *args[] = {&p};
        MDSIP_CUDA(cudaLaunchCooperativeKernel((const void *)k_ldlt_solve_tagged<T>,
                                               dim3(grid, (unsigned)std::min<int64_t>(side, nrhs - rr)), dim3(kThreads),
                                               args, 0, s));
        count_launch();
    }
}

}  // namespace

size_t ldlt_solve_scratch_bytes(int64_t N) { return layout_for(N).total; }

// Tiles of L (FP64, or FP32 when fp32) and cleared words; once per factorization.
void launch_ldlt_solve_prepare(cudaStream_t s, int64_t N, const double *L, void *scratch, bool fp32) {
    if (N <= 0) return;
    char *w = static_cast<char *>(scratch);
    MDSIP_REQUIRE((reinterpret_cast<uintptr_t>(w) & 255) == 0, MDSIP_ERR_INVALID_ARG,
                  "ldlt_solve: misaligned scratch");
    const Layout l = layout_for(N);
    // epoch, done counter and the tagged results (a stale word must
    // not carry an epoch of the new series)
    MDSIP_CUDA(cudaMemsetAsync(w, 0, l.off_F, s));
    if (fp32)
        k_solve_tiles<float><<<(unsigned)l.ntile, kThreads, 0, s>>>(
            (int)N, L, reinterpret_cast<float *>(w + l.off_F), reinterpret_cast<float *>(w + l.off_B));
    else
        k_solve_tiles<double><<<(unsigned)(l.ntile + (int64_t)l.nblk * (kDiagParts - 1)), kThreads, 0, s>>>(
            (int)N, L, reinterpret_cast<double *>(w + l.off_F), reinterpret_cast<double *>(w + l.off_B));
    MDSIP_LAUNCHED();
}

// b_r <- K^-1 b_r for nrhs right-hand sides (columns of B, ld ldb), with the
// tiles of the last launch_ldlt_solve_prepare (same fp32 flag).  err_dev: set
// to 1 when a bounded wait expires.
void launch_ldlt_solve_coop(cudaStream_t s, int num_sms, int64_t N, const double *Dd, const double *Doff,
                            const int32_t *perm, int64_t nrhs, double *B, int64_t ldb, void *scratch, int *err_dev,
                            bool fp32) {
    if (N <= 0 || nrhs <= 0) return;
    char *w = static_cast<char *>(scratch);
    if (fp32)
        launch_solve_t<float>(s, num_sms, N, Dd, Doff, perm, nrhs, B, ldb, w, err_dev);
    else
        launch_solve_t<double>(s, num_sms, N, Dd, Doff, perm, nrhs, B, ldb, w, err_dev);
}

}  // namespace mdsip
