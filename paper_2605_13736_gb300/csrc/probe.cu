// FP64 fused multiply-add throughput probe.
//
// The roofline of the FP64 condensation product and factorization is the rate
// of the SM's FP64 FMA pipe.  This kernel measures that rate on the GPU at
// hand: every thread runs eight independent FMA chains (enough independent
// work per warp scheduler to hide the pipe's latency), so the time of the
// launch is the time the FP64 pipe takes for blocks x 256 x iters x 8 FMAs.
// The result of each chain is written out so that no work can be removed.
//
// And the scalar pieces of the other kernels, element by element, for tests.
#include "internal.cuh"
#include "mlp.cuh"
#include "rns.cuh"

namespace mdsip {

namespace {

constexpr int kProbeThreads = 256;

__global__ void __launch_bounds__(kProbeThreads) k_fp64_fma_probe(int64_t iters, double *sink) {
    const double a = 1.0 + 1e-9 * threadIdx.x, b = 1e-7;
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = 1e-3 * (k + 1) + 1e-6 * blockIdx.x;
    // eight chain steps per loop trip: the loop's own instructions take a
    // negligible share of the issue slots
    int64_t i = 0;
    for (; i + 8 <= iters; i += 8) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = fma(v[k], a, b);
    }
    for (; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = fma(v[k], a, b);
    }
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += v[k];
    sink[(size_t)blockIdx.x * kProbeThreads + threadIdx.x] = s;
}

__global__ void k_scalar(int op, int64_t n, const double *a, const double *b, double *out) {
    const AdamStep st{1e-3f, 0.9f, 0.999f, 1e-8f, 0.19f, 1.999e-3f, 1.0f / 0.19f, 1.0f / 1.999e-3f};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (op == MDSIP_SCALAR_RCP) {
            out[i] = rcp_newton(a[i]);
        } else if (op == MDSIP_SCALAR_DIV) {
            out[i] = ddiv(a[i], b[i]);
        } else if (op == MDSIP_SCALAR_LOGSUM) {
            LogSum s;
            for (int k = 0; k < 16; ++k) s.add(a[16 * i + k]);
            out[i] = s.value();
        } else if (op == MDSIP_SCALAR_ADAM) {
            float m = (float)a[i], v = (float)b[i];
            bool bad = false;
            const float u = adam_moments(st, 0.0f, m, v, bad);
            out[2 * i] = bad ? NAN : u;
            out[2 * i + 1] = adam_quotient(st, m, v);
        } else {
            unsigned long long sm = 0;
            int se = 0;
            rns::rsqrt64(a[i], sm, se);
            out[3 * i] = (double)(sm >> 32);
            out[3 * i + 1] = (double)(sm & 0xffffffffULL);
            out[3 * i + 2] = se;
        }
    }
}

}  // namespace

void launch_scalar(cudaStream_t s, int op, int64_t n, const double *a, const double *b, double *out) {
    k_scalar<<<std::min(1024, ceil_div(n, 256)), 256, 0, s>>>(op, n, a, b, out);
    MDSIP_LAUNCHED();
}

void launch_fp64_fma_probe(cudaStream_t s, int blocks, int64_t iters, double *sink) {
    k_fp64_fma_probe<<<blocks, kProbeThreads, 0, s>>>(iters, sink);
    MDSIP_LAUNCHED();
}

}  // namespace mdsip
