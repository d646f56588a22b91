// Internal declarations of libmdsip: context, problem state, device helpers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../../include/mdsip.h"

namespace mdsip {

// ---------------------------------------------------------------------------
// Error handling: every CUDA call is checked; failures become statuses.
// ---------------------------------------------------------------------------
struct Error {
    mdsip_status status;
    std::string msg;
};

#define MDSIP_CUDA(call)                                                                   \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess)                                                             \
            throw ::mdsip::Error{e_ == cudaErrorMemoryAllocation ? MDSIP_ERR_OOM           \
                                                                 : MDSIP_ERR_CUDA,         \
                                 std::string(#call) + ": " + cudaGetErrorString(e_)};      \
    } while (0)

#define MDSIP_REQUIRE(cond, st, text)                                                      \
    do {                                                                                   \
        if (!(cond)) throw ::mdsip::Error{st, text};                                       \
    } while (0)

void count_launch();
#define MDSIP_LAUNCHED()                   \
    do {                                   \
        ::mdsip::count_launch();           \
        MDSIP_CUDA(cudaGetLastError());    \
    } while (0)

// ---------------------------------------------------------------------------
// Context
// ---------------------------------------------------------------------------
struct Ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    mdsip_alloc_hooks hooks{};
    bool has_hooks = false;
    int num_sms = 0;
    std::string last_error;
    int32_t ldlt_panels[2] = {0, 0};   // of the last mdsip_ldlt_factor* call
    // 16 pinned words the device can write: [0] nonzero once a wait expired in a call
    // that had returned before (reported by the next call); [2], [3] read back by the
    // factorization
    int *words = nullptr;
    bool debug_expire = false;         // the next FP64 product ends as if a wait had expired
    // grow-only scratch arena for kernel-level calls
    void *scratch = nullptr;
    size_t scratch_bytes = 0;

    void *alloc(size_t bytes);
    void release(void *p, size_t bytes);
    void *scratch_at_least(size_t bytes);
    // memory for the length of one call: through the hooks, or stream-ordered from a pool
    cudaMemPool_t pool = nullptr;
    void *lease(size_t bytes);
    void give_back(void *p, size_t bytes);
};

// Makes `dev` current for the scope of the object.
struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        MDSIP_CUDA(cudaSetDevice(dev));
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

// Runs fn, turning exceptions into a status and the context's last error.
template <class F>
inline mdsip_status guarded(Ctx *ctx, F &&fn) {
    if (ctx && ctx->words && *(volatile int *)ctx->words) {
        *(volatile int *)ctx->words = 0;
        ctx->last_error = "a bounded device wait expired in an earlier mdsip_syrk_scaled (its C is NaN)";
        return MDSIP_ERR_DEVICE;
    }
    try {
        fn();
        return MDSIP_OK;
    } catch (const Error &e) {
        if (ctx) ctx->last_error = e.msg;
        return e.status;
    } catch (const std::bad_alloc &) {
        if (ctx) ctx->last_error = "host allocation failed";
        return MDSIP_ERR_OOM;
    } catch (...) {
        if (ctx) ctx->last_error = "unknown error";
        return MDSIP_ERR_CUDA;
    }
}

// A device buffer owned through the context's allocator.
struct DBuf {
    Ctx *ctx = nullptr;
    void *ptr = nullptr;
    size_t bytes = 0;
    DBuf() = default;
    DBuf(const DBuf &) = delete;
    DBuf &operator=(const DBuf &) = delete;
    ~DBuf() { reset(); }
    void reset() {
        if (ptr && ctx) ctx->release(ptr, bytes);
        ptr = nullptr;
        bytes = 0;
    }
    template <class T>
    T *get(Ctx *c, size_t count) {
        reset();
        ctx = c;
        bytes = count * sizeof(T) > 0 ? count * sizeof(T) : 16;
        ptr = c->alloc(bytes);
        return static_cast<T *>(ptr);
    }
    template <class T>
    T *as() const { return static_cast<T *>(ptr); }
};

// ---------------------------------------------------------------------------
// Options: constants of the method (Section 2.1, with the readings of the
// filter line search and inertia correction it delegates).
// ---------------------------------------------------------------------------
struct Options {
    double tol = 1e-8;
    int64_t max_iter = 200;
    double mu0 = 0.1;
    double kappa_eps = 10.0, kappa_mu = 0.2, theta_mu = 1.5, tau_min = 0.99;
    double s_max = 100.0, kappa_1 = 1e-2, kappa_2 = 1e-2, kappa_sigma = 1e10;
    double gamma_theta = 1e-5, gamma_phi = 1e-8, delta = 1.0, s_theta = 1.1, s_phi = 2.3;
    double eta_phi = 1e-8, gamma_alpha = 0.05;
    double theta_max_fact = 1e4, theta_min_fact = 1e-4;
    int64_t max_ls = 60;
    double dw0 = 1e-4, dw_min = 1e-20, dw_max = 1e40, kw_minus = 1.0 / 3.0, kw_plus = 8.0,
           kw_plus_bar = 100.0, dc_bar = 1e-8, kappa_c = 0.25;
    double zero_tol = 1e-14;
    int64_t path = MDSIP_PATH_AUTO;
    int64_t refine_max = -1;          // -1: 0 for FP64, 30 for tensor-core products
    int64_t precision = MDSIP_PREC_FP64;
    double refine_tol = 1e-14;
    double refine_fallback_tol = 1e-10;
    double time_limit_s = 0.0;
    int64_t graphs = 1;               // 1: replay the factorization phase as a CUDA graph
    int64_t autotune = 1;             // 1: time tile-shape candidates at first use per shape
    int64_t ldlt_spec = 1;            // 1: mixed-precision LDL^T panels try the verified no-interchange path
    int64_t direction_check = 0;      // 1: each mixed-precision step also forms the FP64 direction and logs the gap
};

// ---------------------------------------------------------------------------
// Device views passed to kernels by value.
// ---------------------------------------------------------------------------
struct Dims {
    int64_t n_s, n_d, m_E, m_I, n, m;
    int64_t lda;  // leading dimension of A (row-major, padded to a multiple of 4)
};

struct ModelView {
    const double *Q, *c, *A, *gE, *hl, *hu, *xl, *xu;
    const int32_t *h_set;
    const int32_t *csr_ptr, *csr_col;  // J_sg by rows (m_E + 1, nnz)
    const double *csr_val;
    const int32_t *csc_ptr, *csc_row;  // J_sg by columns (n_s + 1, nnz)
    const double *csc_val;
    // J_sh (the inequalities' sparse block): by rows (m_I + 1) and by columns
    // (n_s + 1); all null when J_sh = 0 (the benchmark family)
    const int32_t *hsr_ptr, *hsr_col;
    const double *hsr_val;
    const int32_t *hsc_ptr, *hsc_row;
    const double *hsc_val;
};

// Number of per-block partial slots used by the reduction kernels.
constexpr int kRedBlocks = 304;
constexpr int kRedThreads = 256;

// Scalars written by reduction kernels and read by the host control.
enum Scalar : int {
    S_F = 0,          // objective
    S_THETA,          // ||c||_1
    S_INF_PR,         // ||c||_inf
    S_INF_DU,         // ||grad L - z||_inf (x and d parts)
    S_COMP_MAX,       // max over finite bounds of s*z
    S_COMP_MIN,       // min over finite bounds of s*z
    S_Y1,             // ||y||_1
    S_Z1,             // ||z||_1 + ||v||_1
    S_LOGSUM,         // sum of log slacks at the current point
    S_GPHI,           // grad phi_mu^T (dx, dd)
    S_AMAX,           // fraction-to-boundary alpha for the primal
    S_AZ,             // fraction-to-boundary alpha for the multipliers
    S_QPOS, S_QNEG, S_QZERO,   // inertia of Q_s
    S_WPOS, S_WNEG, S_WZERO,   // inertia of -W (path P2)
    S_T_F, S_T_THETA, S_T_LOGSUM, S_T_INSIDE, S_T_FINITE,  // trial point
    S_MAXABS,         // max |reduced matrix| (zero-pivot scale)
    S_NONFINITE,      // count of non-finite model values
    S_RES_INF, S_RHS_INF, S_SOL_INF,  // refinement: ||r||_inf, ||rhs||_inf, ||dir||_inf
    S_COUNT
};

// ---------------------------------------------------------------------------
// FP64 scalar pieces.  GB300 issues one FP64 instruction of a warp in 64
// cycles per sub-partition, comparisons included, so the small kernels of a
// step are bound by the number of FP64 instructions on their longest chain:
// tests and maxima work on bit patterns, divisions on the short reciprocal.
// ---------------------------------------------------------------------------
// 1/d by Newton-Raphson iteration x <- x (2 - d x) (0 for d = 0), on FP32 and
// integers alone: hardware reciprocal q of the upper 24 bits of d's mantissa m,
// the residual 1 - m q with all of m, x = q + q (e + e^2) as an integer X of
// units 2^-53, good to about 2^-46; then the second step with M = 2^52 m: E =
// 2^105 - M X fits 64 bits, and X + X E / 2^105 rounded is 1/m to 0.51 units in
// the last place.  An FP64 instruction occupies a warp's pipe for 64 cycles and
// every pivot waits for this value: the two that the second step took, and six
// with conversions, were most of its latency.  d near the ends of the range
// goes through the division operator.
__device__ __forceinline__ double rcp_newton(double d) {
    const int hi = __double2hiint(d);
    const unsigned lo = (unsigned)__double2loint(d);
    const int ef = (hi >> 20) & 0x7ff;
    if (ef < 100 || ef > 1946) return d == 0.0 ? 0.0 : 1.0 / d;
    const float mh = __uint_as_float(0x3f800000u | (((unsigned)hi & 0xfffffu) << 3) | (lo >> 29));
    const float ml = (float)(lo & 0x1fffffffu) * 0x1p-52f;
    float q;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(mh));
    const float e = fmaf(-ml, q, fmaf(-mh, q, 1.0f));
    const float qe = q * e;
    const int c = __float2int_rn(fmaf(qe, e, qe) * 0x1p52f);       // |q e| < 2^-21
    const unsigned qb = __float_as_uint(q);                        // 1/2 <= q <= 1
    const long long X = ((long long)((qb & 0x7fffffu) | 0x800000u) << (29 + (int)(qb >> 23) - 126)) + 2LL * c;
    const unsigned long long M = ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const long long E = -(long long)(M * (unsigned long long)X);   // |E| < 2^60
    const long long t = (long long)(int)(E >> 30) * (long long)(int)(X >> 23);
    const long long Y = X + ((t + (1LL << 51)) >> 52);             // 2^52 <= Y <= 2^53
    const long long y = (1021LL << 52) + Y;                        // as 1022 << 52 plus Y - 2^52
    return __hiloint2double(((int)(y >> 32) - ((ef - 1023) << 20)) | (hi & (int)0x80000000), (int)y);
}

// a / b: reciprocal, product and one residual correction (Markstein 1990), five
// FP64 instructions; magnitudes outside 2^-500 .. 2^500 take the operator
__device__ __forceinline__ double ddiv(double a, double b) {
    const int ha = __double2hiint(a), hb = __double2hiint(b);
    const bool zero = (((unsigned)ha << 1) | (unsigned)__double2loint(a)) == 0u;
    const unsigned ea = (unsigned)((ha >> 20) & 0x7ff) - 523u, eb = (unsigned)((hb >> 20) & 0x7ff) - 523u;
    if ((ea > 1000u && !zero) || eb > 1000u) return a / b;
    const double r = rcp_newton(b);
    const double q = a * r;
    return fma(fma(-q, b, a), r, q);
}

__device__ __forceinline__ bool fin(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

// non-NaN doubles as integers of the same order
__device__ __forceinline__ long long ord64(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

// |v| by its bit pattern into a running maximum (NaN passed over, as fmax does)
__device__ __forceinline__ void max_abs(unsigned long long &m, double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
    if (b > m && b <= 0x7ff0000000000000ULL) m = b;
}

// running maximum and minimum of v as ordered integers (NaN passed over)
struct MinMax {
    long long hi = (long long)0x800fffffffffffffULL, lo = 0x7ff0000000000000LL;   // of -inf and inf
    __device__ __forceinline__ void add(double v) {
        const long long k = ord64(v);
        if (((unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL) > 0x7ff0000000000000ULL) return;
        hi = k > hi ? k : hi;
        lo = k < lo ? k : lo;
    }
    static __device__ __forceinline__ double value(long long k) {
        return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
    }
};

// sum of logarithms of positive values: the mantissas' product and the
// exponents' sum, one logarithm in the end (some 35 FP64 instructions each)
struct LogSum {
    double m = 1.0, rest = 0.0;
    int e = 0;
    __device__ __forceinline__ void add(double v) {
        const long long b = __double_as_longlong(v);
        const int ef = (int)(b >> 52);   // sign included
        if (ef <= 0 || ef >= 0x7ff) {    // not a positive normal number
            rest += log(v);
            return;
        }
        const double p = m * __longlong_as_double((b & 0xfffffffffffffLL) | (1023LL << 52));   // in [1, 4)
        const long long q = __double_as_longlong(p);
        const int ep = (int)(q >> 52) - 1023;
        e += ef - 1023 + ep;
        m = __longlong_as_double(q - ((long long)ep << 52));
    }
    __device__ __forceinline__ double value() const {
        return fma((double)e, 0.69314718055994530942, log(m)) + rest;
    }
};

// ---------------------------------------------------------------------------
// Grid-wide reductions of up to 8 quantities in one kernel (deterministic for
// a fixed launch shape): warps by shuffles, the block's warps by one warp per
// quantity, and the last block to arrive combines the blocks' partials in
// order.  The ticket counter returns to zero by itself, so any grid size may
// follow; the kernels that share one run in turn on a stream.  (A separate
// combining launch per operation took 4 to 8 us each, eleven a Newton step.)
// ---------------------------------------------------------------------------
struct RedOut {
    double *partial;     // kRedBlocks per quantity
    unsigned *ticket;
    double *out;         // one per quantity
};

enum RedOp { R_SUM, R_MAX, R_MIN };

__device__ __forceinline__ double red_identity(RedOp op) {
    return op == R_SUM ? 0.0 : (op == R_MAX ? -INFINITY : INFINITY);
}
__device__ __forceinline__ double red_combine(RedOp op, double a, double b) {
    if (op == R_SUM) return a + b;
    return (op == R_MAX) == (ord64(b) > ord64(a)) ? b : a;
}

// whether this block is the last of the grid to get here (all threads)
__device__ __forceinline__ bool red_last(unsigned *ticket) {
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

template <int NT, RedOp... OPS>
__device__ __forceinline__ void reduce_finish(double (&v)[sizeof...(OPS)], const RedOut &o) {
    constexpr int K = sizeof...(OPS), W = NT / 32;
    constexpr RedOp ops[K] = {OPS...};
    static_assert(W <= 32, "a quantity's warp sums fit a warp");
    __shared__ double sh[K][W];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1)
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = red_combine(ops[k], v[k], __shfl_xor_sync(0xffffffffu, v[k], s));
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) sh[k][wid] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (wid == k % W) {
            double x = lane < W ? sh[k][lane] : red_identity(ops[k]);
#pragma unroll
            for (int s = W / 2; s > 0; s >>= 1) x = red_combine(ops[k], x, __shfl_xor_sync(0xffffffffu, x, s));
            if (lane == 0) *(gridDim.x == 1 ? o.out + k : o.partial + (size_t)k * kRedBlocks + blockIdx.x) = x;
        }
    if (gridDim.x == 1 || !red_last(o.ticket)) return;
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (wid == k % W) {
            double p[(kRedBlocks + 31) / 32];
#pragma unroll
            for (int i = 0; i < (kRedBlocks + 31) / 32; ++i)
                p[i] = lane + 32 * i < (int)gridDim.x ? __ldcg(o.partial + (size_t)k * kRedBlocks + lane + 32 * i)
                                                      : red_identity(ops[k]);
            double x = p[0];
#pragma unroll
            for (int i = 1; i < (kRedBlocks + 31) / 32; ++i)
                if (32 * i < (int)gridDim.x) x = red_combine(ops[k], x, p[i]);
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) x = red_combine(ops[k], x, __shfl_xor_sync(0xffffffffu, x, s));
            if (lane == 0) o.out[k] = x;
        }
}

// the same for K counts (integers; out receives them as doubles)
template <int NT, int K>
__device__ __forceinline__ void count_finish(unsigned (&c)[K], const RedOut &o) {
    constexpr int W = NT / 32;
    __shared__ unsigned sh[K][W];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) c[k] = __reduce_add_sync(0xffffffffu, c[k]);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) sh[k][wid] = c[k];
    __syncthreads();
    unsigned *part = reinterpret_cast<unsigned *>(o.partial);
    for (int k = wid; k < K; k += W) {
        const unsigned x = __reduce_add_sync(0xffffffffu, lane < W ? sh[k][lane] : 0u);
        if (lane == 0) {
            if (gridDim.x == 1) o.out[k] = (double)x;
            else part[(size_t)k * kRedBlocks + blockIdx.x] = x;
        }
    }
    if (gridDim.x == 1 || !red_last(o.ticket)) return;
    for (int k = wid; k < K; k += W) {
        unsigned x = 0;
        for (int i = lane; i < (int)gridDim.x; i += 32) x += __ldcg(part + (size_t)k * kRedBlocks + i);
        x = __reduce_add_sync(0xffffffffu, x);
        if (lane == 0) o.out[k] = (double)x;
    }
}

// (J^T y)_k of 32 columns k0 .. k0 + 31 of a row-major m x n matrix, by a block
// whose warps share the rows: returned to threads 0 .. 31 (every thread calls)
template <int NT>
__device__ __forceinline__ double colgroup_dot(const double *__restrict__ J, int64_t m, int64_t n, int64_t k0,
                                               const double *__restrict__ y, double (*sp)[33]) {
    if (m == 0) return 0.0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t k = k0 + lane;
    double s = 0.0;
    if (k < n)
#pragma unroll 4
        for (int64_t j = wid; j < m; j += NT / 32) s = fma(J[j * n + k], y[j], s);
    __syncthreads();                               // an earlier group's sums are read
    sp[wid][lane] = s;
    __syncthreads();
    double t = 0.0;
    if (wid == 0)
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) t += sp[w][lane];
    return t;
}

// blocks of a reduction kernel over `len` elements or more (one per thread)
inline int red_grid(int64_t len, int threads = kRedThreads) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(kRedBlocks, (len + threads - 1) / threads));
}

// ---------------------------------------------------------------------------
// Grid barrier with a bounded wait.  Used only in cooperative launches (all
// blocks co-resident).  On expiry it raises *err and returns false; callers
// leave their loops at once, so a lost block never hangs the GPU.
// ---------------------------------------------------------------------------
struct GridBar {
    unsigned int *count;
    unsigned int *gen;
    int *err;
};

constexpr long long kBarrierLimitCycles = 4000000000LL;  // ~2 s at 2 GHz

__device__ __forceinline__ bool grid_barrier(const GridBar &b, unsigned int nblocks) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        volatile unsigned int *vgen = b.gen;
        const unsigned int my = *vgen;
        __threadfence();
        const unsigned int arrived = atomicAdd(b.count, 1u);
        if (arrived == nblocks - 1) {
            atomicExch(b.count, 0u);
            __threadfence();
            atomicAdd(b.gen, 1u);
        } else {
            const long long t0 = clock64();
            while (*vgen == my) {
                if (*((volatile int *)b.err) != 0 || clock64() - t0 > kBarrierLimitCycles) {
                    atomicExch(b.err, 1);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

inline int ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

// Runs a configuration call (e.g. a kernel attribute, which is global to the
// kernel on a device) once per device, thread-safely; returns its result.
struct PerDeviceOnce {
    std::mutex mu;
    bool done[64] = {};
    cudaError_t err[64] = {};
    template <class F>
    cudaError_t run(F &&f) {
        int dev = 0;
        const cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return f();
        std::lock_guard<std::mutex> lk(mu);
        if (!done[dev]) {
            err[dev] = f();
            done[dev] = true;
        }
        return err[dev];
    }
};

// ---------------------------------------------------------------------------
// Kernel launchers (defined in the .cu files).
// ---------------------------------------------------------------------------
// probe.cu: blocks x 256 threads, each iters x 8 independent FP64 FMAs; sink
// holds blocks x 256 doubles
void launch_fp64_fma_probe(cudaStream_t s, int blocks, int64_t iters, double *sink);
// as mdsip_debug_scalar
void launch_scalar(cudaStream_t s, int op, int64_t n, const double *a, const double *b, double *out);

// A passes (row-major A, m x n, leading dimension lda)
void launch_gemv_rows(cudaStream_t s, const double *A, int64_t m, int64_t n, int64_t lda,
                      const double *v, double *out);  // out = A v
// out[p] = sum_b partial[b][p] (fixed order); partial: nparts x n
void launch_colsum(cudaStream_t s, const double *partial, int nparts, int64_t n, double *out);
// gemv_df.cu: passes over A = A_hi + A_lo (FP32 pair, m x lda) in double-float
// arithmetic with FP64 accuracy; xs / ys: scratch of n / m float2
void launch_split_matrix(cudaStream_t s, const double *A, int64_t m, int64_t n, int64_t lda, float *hi,
                         float *lo);
void launch_gemv_rows_df(cudaStream_t s, const float *Ahi, const float *Alo, int64_t m, int64_t n, int64_t lda,
                         const double *x, float2 *xs, double *out);
void launch_gemv_t_df(cudaStream_t s, const float *Ahi, const float *Alo, int64_t m, int64_t n, int64_t lda,
                      const double *y, float2 *ys, double *partial, double *out);
// out_rows = A x and out_cols = A^T y from one read of A.  With nx, the same
// read also gives out_v = A_hi^T v, v_i = fl32((cpre_i - (A x)_i) wf_i) with
// the difference in double-float (FP32 products and sums): the first half of
// a refinement's next approximate solve (mdsip_gemv_pair_df_next; the solver's own
// sweeps are in refine_sweep.cu).  cw = cpre as FP32 halves
// (launch_split_vector), wf = fl32(1 / w) (launch_round_vector).  The fused
// form needs the whole row in one slice: gemv_both_fusable(n).
struct BothNextArgs {
    const float2 *cw;   // m
    const float *wf;    // m
    double *out_v;      // n
};
void launch_split_vector(cudaStream_t s, const double *v, int64_t n, float2 *out);   // out = (fl32(v), fl32(v - hi))
void launch_round_vector(cudaStream_t s, const double *v, int64_t n, float *out);    // out = fl32(v)
bool gemv_both_fusable(int64_t n);
void launch_gemv_both_df(cudaStream_t s, const float *Ahi, const float *Alo, int64_t m, int64_t n, int64_t lda,
                         const double *x, const double *y, float2 *xs, float2 *ys, double *partial,
                         double *out_rows, double *out_cols, int *err, const BothNextArgs *nx = nullptr);
// out = A_hi x with FP32 products and sums
void launch_gemv_rows_f32(cudaStream_t s, const float *Ahi, int64_t m, int64_t n, int64_t lda, const double *x,
                          double *out);
void launch_gemv_t(cudaStream_t s, const double *A, int64_t m, int64_t n, int64_t lda,
                   const double *u, double *partial, double *out);  // out = A^T u

// SYRK: C (column-major, ldc) = beta C + A^T diag(1/w) A (lower)
void launch_syrk_fp64(Ctx *ctx, const double *A, int64_t m, int64_t n, int64_t lda, const double *w,
                      double beta, double *C, int64_t ldc);
// what the workspace has room for: residues of one chunk of rows (0: the DFMA
// kernel alone) and the DFMA kernel's split partials, in bytes
struct SyrkRoom {
    size_t rns = 0, part = (size_t)1 << 30;
};
size_t syrk_workspace_bytes(int64_t m, int64_t n, int num_sms, const SyrkRoom &room);
void launch_syrk_fp64_ws(cudaStream_t s, int num_sms, const double *A, int64_t m, int64_t n,
                         int64_t lda, const double *w, double beta, double *C, int64_t ldc,
                         void *ws, const SyrkRoom &room, int bm = 0, int *late_err = nullptr, bool expire = false);
// The same product by residue numbers on the tensor cores (syrk_rns.cu), the
// faster form from syrk_rns_pays on; ws as syrk_rns_workspace_bytes.  The
// returned device flag is nonzero afterwards when the operands were outside
// its range and C is untouched.  late_err: null, or a host word set to 1 when a
// wait expired; expire: as if one had (a test of that path).
bool syrk_rns_pays(int64_t m, int64_t n);
size_t syrk_rns_workspace_bytes(int64_t m, int64_t n, int num_sms, size_t cap);
inline const int *syrk_rns_err(const void *ws) { return static_cast<const int *>(ws) + 1; }   // nonzero: a wait expired
const int *launch_syrk_rns(cudaStream_t s, int num_sms, const double *A, int64_t m, int64_t n, int64_t lda,
                           const double *w, double beta, double *C, int64_t ldc, void *ws, size_t cap,
                           int *late_err = nullptr, bool expire = false);
// Workspace of the product from `get(bytes)`, which throws OOM where that much is
// not to be had: fewer rows of residues at a time then (m = 25600, n = 512: 377 MB
// 266 us, 86 MB 599; m = 15053, n = 301: 140 MB 145 us, 38 MB 232), and only at last
// the DFMA kernel (n = 301 1.6 ms with room for its split partials, 15.8 with none).
template <class F>
void *syrk_workspace(int64_t m, int64_t n, int num_sms, SyrkRoom &room, F &&get) {
    constexpr size_t kMB = (size_t)1 << 20;
    constexpr SyrkRoom rooms[] = {{512 * kMB, 1024 * kMB}, {128 * kMB, 128 * kMB}, {32 * kMB, 32 * kMB},
                                  {0, 1024 * kMB}, {0, 32 * kMB}, {0, 0}};
    size_t last = 0;
    for (const SyrkRoom &r : rooms) {
        if (r.rns && !syrk_rns_pays(m, n)) continue;
        const size_t bytes = syrk_workspace_bytes(m, n, num_sms, r);
        if (last && bytes >= last) continue;   // no less than what was refused
        last = bytes;
        room = r;
        try {
            return get(bytes);
        } catch (const Error &e) {
            if (e.status != MDSIP_ERR_OOM) throw;
        }
    }
    throw Error{MDSIP_ERR_OOM, "no memory for the condensation product"};
}

// Tensor-core SYRK (syrk_tc.cu)
struct TcPlan {
    int tiles, nsplit, slabs_per_split, total_slabs, elems_per_slab;
    int nt, blocks;   // 128-row blocks; 256 x 256 blocks of the lower triangle (wide)
    bool wide;
    int64_t ldt;
    size_t work_floats;
};
int64_t syrk_tc_ld(int64_t m);
void launch_aft_dot(cudaStream_t s, int num_sms, const float *AfT, int64_t ldt, int64_t m, int64_t n,
                    const double *v, float *vf, double *out);
void launch_aft_dot_add(cudaStream_t s, int num_sms, const float *AfT, int64_t ldt, int64_t n, const float *vf,
                        const double *add, double *out);
TcPlan syrk_tc_plan(int64_t m, int64_t n, int num_sms, int precision);
size_t syrk_tc_workspace_bytes(const TcPlan &pl, int64_t n, int precision);
void launch_transpose_f32(cudaStream_t s, const double *A, int64_t m, int64_t n, int64_t lda, float *AfT,
                          int64_t ldt);
void launch_syrk_tc(cudaStream_t s, int num_sms, int precision, const float *AfT, int64_t m, int64_t n,
                    const double *w, double beta, double *C, int64_t ldc, void *ws, int *err_dev);

// Bunch-Kaufman LDL^T
struct LdltOut {
    double *L, *Dd, *Doff;
    int32_t *perm, *kind, *inertia;
    int32_t *panels = nullptr;   // optional: panels taken by the no-interchange path, and handed back
};
size_t ldlt_scratch_bytes(int64_t N);
void launch_ldlt(cudaStream_t s, int num_sms, int64_t N, const double *S, int64_t ld,
                 const double *maxabs_dev, double zero_tol, LdltOut out, void *scratch,
                 int *err_dev, int *host2, bool fp32_update = false, int nb = 0, int spec = 1);
size_t ldlt_blocked_scratch_bytes(int64_t N);
bool ldlt_blocked_available(int64_t N);
// Speculation mode of the blocked factorization: 0 every panel pivots; 1 and 2
// the persistent no-interchange kernel first, then (FP32 updates) no-interchange
// panels; kSpecPanels (FP32 updates) no-interchange panels alone.  Where the persistent kernel stopped is read back into host2, two pinned
// words (synchronises the stream).
constexpr int kSpecPanels = 3;
bool ldlt_persistent_path(int64_t N, int spec);
std::vector<int> ldlt_blocked_widths(int64_t N, bool f32);
void launch_ldlt_blocked(cudaStream_t s, int num_sms, int64_t N, double *S, const double *maxabs_dev,
                         double zero_tol, LdltOut out, void *scratch, bool fp32_update, int nb,
                         int spec, int *err_dev, int *host2);
void launch_ldlt_solve(cudaStream_t s, int64_t N, const double *L, const double *Dd,
                       const double *Doff, const int32_t *perm, int64_t nrhs, double *B,
                       int64_t ldb);
void launch_maxabs_lower(cudaStream_t s, int64_t N, const double *S, int64_t ld, double *out);
size_t ldlt_solve_scratch_bytes(int64_t N);
// tiles of L for the solve (FP64, or FP32 when fp32), into the solve scratch; after each factorization
void launch_ldlt_solve_prepare(cudaStream_t s, int64_t N, const double *L, void *scratch, bool fp32);
// b_r <- K^-1 b_r with the prepared tiles (same fp32 flag)
void launch_ldlt_solve_coop(cudaStream_t s, int num_sms, int64_t N, const double *Dd, const double *Doff,
                            const int32_t *perm, int64_t nrhs, double *B, int64_t ldb, void *scratch, int *err_dev,
                            bool fp32);
// LDL^T with its scratch in a fixed device array (no allocation); N <= the limit.
int64_t ldlt_fixed_scratch_max_n();
void ldlt_factor_fixed_scratch(cudaStream_t s, int device, int num_sms, int64_t N, double *S,
                               int64_t ld, double zero_tol, LdltOut out);

}  // namespace mdsip
