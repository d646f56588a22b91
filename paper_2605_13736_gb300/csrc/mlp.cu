// Warm-start network: a two-hidden-layer ReLU perceptron
//
//     h1 = relu(W1 xn + b1),  h2 = relu(W2 h1 + b2),  yn = W3 h2 + b3
//
// mapping the parameters p of a parametric problem family (xn: p
// standardised per input) to a standardised primal-dual point plus log mu0
// (y = yn * out_std + out_mean).  Training minimises the mean squared error in
// standardised units, L = sum (yn - (y* - out_mean) / out_std)^2 / (B O), with
// Adam.  Every contraction (three forward, five backward) runs on the BF16
// tcgen05 GEMM with FP32 accumulation; parameters, moments and gradients are
// FP32; the bias and ReLU are fused into the kernels that produce the BF16
// operands of the next contraction, the output layer's bias, scaling, loss and
// Adam step into its contractions.  No operand is stored twice: where a
// contraction needs the other orientation the tensor core reads it MN-major.
//
// BF16 operand points (each value rounded to nearest even once): the
// standardised input, W1, W2, W3, h1, h2, the output gradient dL/dyn, and the
// hidden-layer gradients dL/dz2, dL/dz1.  Bias gradients are column sums of
// the rounded BF16 gradients.
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.cuh"
#include "mlp.cuh"

namespace mdsip {

namespace {

using bf16 = __nv_bfloat16;

int64_t r8(int64_t v) { return (std::max<int64_t>(v, 1) + 7) / 8 * 8; }

// Xb[b][i] = bf16((X[row(b)][i] - mean_i) / std_i)
__global__ void k_gather_x(int64_t B, int64_t I, const double *__restrict__ X, int64_t ldx,
                           const int32_t *__restrict__ idx, const float *__restrict__ mean,
                           const float *__restrict__ sd, bf16 *__restrict__ Xb, int64_t ldI) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < B * I; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = e / I, i = e - b * I;
        const int64_t row = idx ? (int64_t)idx[b] : b;
        Xb[b * ldI + i] = __float2bfloat16_rn((float)((X[row * ldx + i] - (double)mean[i]) / (double)sd[i]));
    }
}

// Hh[b][j] = bf16(relu(Z[b][j] + bias[j]))
__global__ void k_bias_relu(int64_t B, int64_t Hn, const float *__restrict__ Z, int64_t ldz,
                            const float *__restrict__ bias, bf16 *__restrict__ Hh, int64_t ldh) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < B * Hn; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = e / Hn, j = e - b * Hn;
        Hh[b * ldh + j] = __float2bfloat16_rn(fmaxf(Z[b * ldz + j] + bias[j], 0.0f));
    }
}

// Sum of the 32 row groups of a block's columns (groups halved pairwise) by
// the threads with threadIdx.y == 0.
__device__ __forceinline__ float group_sum(float s, float (&red)[32][33]) {
    red[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    for (int w = 16; w > 0; w >>= 1) {
        if ((int)threadIdx.y < w) red[threadIdx.y][threadIdx.x] += red[threadIdx.y + w][threadIdx.x];
        __syncthreads();
    }
    return red[0][threadIdx.x];
}

// dZ = bf16(dH * [Hact > 0]) and its column sums (the bias gradient): 32
// columns x 32 row groups per block, fixed order
__global__ void __launch_bounds__(1024) k_relu_back(int64_t B, int64_t Hn, const float *__restrict__ dH, int64_t ldd,
                                                    const bf16 *__restrict__ Hact, int64_t ldh, bf16 *__restrict__ dZ,
                                                    float *__restrict__ db) {
    __shared__ float red[32][33];
    const int64_t j = (int64_t)blockIdx.x * 32 + threadIdx.x;
    float s = 0.0f;
    if (j < Hn) {
#pragma unroll 4
        for (int64_t b = threadIdx.y; b < B; b += 32) {
            const float h = __bfloat162float(Hact[b * ldh + j]);
            const bf16 v = __float2bfloat16_rn(h > 0.0f ? dH[b * ldd + j] : 0.0f);
            dZ[b * ldh + j] = v;
            s += __bfloat162float(v);
        }
    }
    s = group_sum(s, red);
    if (threadIdx.y == 0 && j < Hn) db[j] = s;
}

// out[j] = sum_b T[b][j] in the same order, two columns per thread (ld even);
// HBM / L2-bound, one read of T
__global__ void __launch_bounds__(1024) k_colsum_bf16(int64_t B, int64_t cols, const bf16 *__restrict__ T, int64_t ld,
                                                      float *__restrict__ out) {
    __shared__ float red[2][32][33];
    const int64_t j = (int64_t)blockIdx.x * 64 + 2 * threadIdx.x;
    float s0 = 0.0f, s1 = 0.0f;
    if (j < cols) {
#pragma unroll 8
        for (int64_t b = threadIdx.y; b < B; b += 32) {
            const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(T + b * ld + j));
            s0 += v.x;
            s1 += v.y;
        }
    }
    s0 = group_sum(s0, red[0]);
    s1 = group_sum(s1, red[1]);
    if (threadIdx.y == 0 && j < cols) {
        out[j] = s0;
        if (j + 1 < cols) out[j + 1] = s1;
    }
}

// single-block fixed-order sum of n doubles
__global__ void k_sum_partials(int64_t n, const double *__restrict__ part, double *__restrict__ out) {
    __shared__ double red[256];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

__global__ void k_adam(int64_t n, float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, AdamStep st) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float wi = w[i], mi = m[i], vi = v[i];
        adam_update(st, g[i], wi, mi, vi);
        m[i] = mi;
        v[i] = vi;
        w[i] = wi;
    }
}

// dst[r][c] = bf16(src[r][c])
__global__ void k_cast_bf16(int64_t rows, int64_t cols, const float *__restrict__ src, int64_t lds,
                            bf16 *__restrict__ dst, int64_t ldd) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < rows * cols;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / cols, c = e - r * cols;
        dst[r * ldd + c] = __float2bfloat16_rn(src[r * lds + c]);
    }
}

// Column mean and standard deviation (two passes, FP64, fixed order); a
// standard deviation below 1e-6 max(1, |mean|) is replaced by that floor.
__global__ void k_col_stats(int64_t rows, int64_t cols, const double *__restrict__ Y, int64_t ldy,
                            float *__restrict__ mean, float *__restrict__ sd) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < cols; c += (int64_t)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int64_t r = 0; r < rows; ++r) s += Y[r * ldy + c];
        const double mu = rows > 0 ? s / (double)rows : 0.0;
        double q = 0.0;
        for (int64_t r = 0; r < rows; ++r) {
            const double d = Y[r * ldy + c] - mu;
            q += d * d;
        }
        const double sdev = rows > 0 ? sqrt(q / (double)rows) : 0.0;
        mean[c] = (float)mu;
        sd[c] = (float)fmax(sdev, 1e-6 * fmax(1.0, fabs(mu)));
    }
}

__global__ void k_fill_f32(int64_t n, float *p, float v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

int grid_for(int64_t n, int num_sms) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms * 16, ceil_div(n, 256)));
}

}  // namespace

struct Mlp {
    Ctx *ctx = nullptr;
    int64_t I = 0, H = 0, O = 0;
    int64_t ldI = 8, ldH = 8, ldO = 8;
    int64_t off_W1 = 0, off_b1 = 0, off_W2 = 0, off_b2 = 0, off_W3 = 0, off_b3 = 0, n_params = 0;
    double beta1 = 0.9, beta2 = 0.999, eps = 1e-8;
    int64_t t = 0;  // Adam steps taken
    DBuf params, grads, m1, m2;
    DBuf W1b, W2b, W3b;
    DBuf in_mean, in_std, out_mean, out_std;
    DBuf err, loss;
    // activations, sized for `cap` rows
    int64_t cap = 0, tcap = 0;   // rows of the forward and of the training buffers
    DBuf Xb, H1, H2, Zbuf, gws, dY, dZ2, dZ1, lpart, tws;
    size_t gws_bytes = 0;

    float *P() const { return params.as<float>(); }
    float *G() const { return grads.as<float>(); }

    // buffers for batches of B rows: the forward pass's, and with `train` the
    // backward pass's (a prediction needs no batch x outputs gradient)
    void ensure(int64_t B, bool train) {
        const int sms = ctx->num_sms;
        if (B > cap) {
            const int64_t c = std::max<int64_t>(B, 64);
            cap = 0;   // until all of them are there: an allocation may fail
            Xb.get<bf16>(ctx, c * ldI);
            H1.get<bf16>(ctx, c * ldH);
            H2.get<bf16>(ctx, c * ldH);
            Zbuf.get<float>(ctx, c * ldH);
            gws.get<uint8_t>(ctx, std::max({split_ws(c, H, I, false, false), split_ws(c, H, H, false, false), (size_t)16}));
            cap = c;
        }
        if (train && B > tcap) {
            const int64_t c = std::max<int64_t>(B, 64);
            tcap = 0;
            dY.get<bf16>(ctx, c * ldO);
            dZ2.get<bf16>(ctx, c * ldH);
            dZ1.get<bf16>(ctx, c * ldH);
            lpart.get<double>(ctx, (int64_t)8 * sms);
            tws.get<uint8_t>(ctx, std::max({split_ws(c, H, O, false, true),
                                            split_ws(H, H, c, true, true), split_ws(c, H, H, false, true),
                                            split_ws(H, I, c, true, true), (size_t)16}));
            tcap = c;
        }
    }

    // largest split workspace over batches of up to B rows (the plan's split
    // count is not monotone in the batch): dimensions M, N, K with the batch as
    // M (or as K, for the weight gradients)
    size_t split_ws(int64_t M, int64_t N, int64_t K, bool amn, bool bmn) const {
        const bool batch_k = amn;   // weight gradients contract over the batch
        const int64_t c = batch_k ? K : M;
        size_t best = 0;
        for (int64_t b = 1; b <= c; b = b < c && b + 64 > c ? c : b + 64)
            best = std::max(best, gemm_bf16_ws_bytes(batch_k ? M : std::min(c, (b + 127) / 128 * 128), N,
                                                     batch_k ? b : K, ctx->num_sms, amn, bmn));
        return std::max(best, gemm_bf16_ws_bytes(M, N, K, ctx->num_sms, amn, bmn));
    }

    void gemm(const bf16 *A, int64_t lda, const bf16 *Bm, int64_t ldb, int64_t M, int64_t N, int64_t K, float *C,
              int64_t ldc, void *ws, bool amn = false, bool bmn = false) {
        launch_gemm_bf16(ctx->stream, ctx->num_sms, A, lda, Bm, ldb, M, N, K, C, ldc, ws, err.as<int>(), amn, bmn);
    }

    // BF16 copies of the hidden layers' weights, and of W3 (the training step's
    // fused update writes that one itself)
    void cast_hidden() {
        cudaStream_t s = ctx->stream;
        k_cast_bf16<<<grid_for(H * I, ctx->num_sms), 256, 0, s>>>(H, I, P() + off_W1, I, W1b.as<bf16>(), ldI);
        MDSIP_LAUNCHED();
        k_cast_bf16<<<grid_for(H * H, ctx->num_sms), 256, 0, s>>>(H, H, P() + off_W2, H, W2b.as<bf16>(), ldH);
        MDSIP_LAUNCHED();
    }
    void cast_weights() {
        cast_hidden();
        k_cast_bf16<<<grid_for(O * H, ctx->num_sms), 256, 0, ctx->stream>>>(O, H, P() + off_W3, H, W3b.as<bf16>(), ldH);
        MDSIP_LAUNCHED();
    }

    // forward through h2 (kept for the backward pass)
    void forward(const double *X, int64_t ldx, const int32_t *idx, int64_t B) {
        cudaStream_t s = ctx->stream;
        float *Z = Zbuf.as<float>();
        k_gather_x<<<grid_for(B * I, ctx->num_sms), 256, 0, s>>>(B, I, X, ldx, idx, in_mean.as<float>(),
                                                                 in_std.as<float>(), Xb.as<bf16>(), ldI);
        MDSIP_LAUNCHED();
        gemm(Xb.as<bf16>(), ldI, W1b.as<bf16>(), ldI, B, H, I, Z, ldH, gws.ptr);
        k_bias_relu<<<grid_for(B * H, ctx->num_sms), 256, 0, s>>>(B, H, Z, ldH, P() + off_b1, H1.as<bf16>(), ldH);
        MDSIP_LAUNCHED();
        gemm(H1.as<bf16>(), ldH, W2b.as<bf16>(), ldH, B, H, H, Z, ldH, gws.ptr);
        k_bias_relu<<<grid_for(B * H, ctx->num_sms), 256, 0, s>>>(B, H, Z, ldH, P() + off_b2, H2.as<bf16>(), ldH);
        MDSIP_LAUNCHED();
    }

    OutLayer out_layer() const {
        OutLayer o{};
        o.b3 = params.as<float>() + off_b3;
        o.mean = out_mean.as<float>();
        o.sd = out_std.as<float>();
        return o;
    }

    // loss (device scalar) and gradients into G(); without w3_grad the output
    // layer's weight gradient is left to the fused update
    void backward(const double *Y, int64_t ldy, const int32_t *idx, int64_t B, bool w3_grad) {
        cudaStream_t s = ctx->stream;
        float *Z = Zbuf.as<float>();
        float *G_ = G();
        OutLayer o = out_layer();
        o.Y = Y;
        o.ldy = ldy;
        o.idx = idx;
        o.scale = (float)(2.0 / ((double)B * (double)O));
        o.dY = dY.as<bf16>();
        o.ldo = ldO;
        o.part = lpart.as<double>();
        // yn = W3 h2 + b3, loss partials, dL/dyn and db3
        const int np = launch_out_layer(s, ctx->num_sms, H2.as<bf16>(), ldH, W3b.as<bf16>(), ldH, B, O, H, o, nullptr,
                                        0, err.as<int>());
        k_sum_partials<<<1, 256, 0, s>>>(np, lpart.as<double>(), loss.as<double>());
        MDSIP_LAUNCHED();
        k_colsum_bf16<<<ceil_div(O, 64), dim3(32, 32), 0, s>>>(B, O, dY.as<bf16>(), ldO, G_ + off_b3);
        MDSIP_LAUNCHED();
        // output layer: dW3 = dY^T h2
        if (w3_grad)
            launch_gemm_w3_grad(s, ctx->num_sms, H2.as<bf16>(), ldH, dY.as<bf16>(), ldO, B, O, H, G_ + off_W3,
                                err.as<int>());
        // second hidden layer: dh2 = dY W3, dz2 = dh2 [h2 > 0]
        const int hb = ceil_div(H, 32);
        gemm(dY.as<bf16>(), ldO, W3b.as<bf16>(), ldH, B, H, O, Z, ldH, tws.ptr, false, true);
        k_relu_back<<<hb, dim3(32, 32), 0, s>>>(B, H, Z, ldH, H2.as<bf16>(), ldH, dZ2.as<bf16>(), G_ + off_b2);
        MDSIP_LAUNCHED();
        gemm(dZ2.as<bf16>(), ldH, H1.as<bf16>(), ldH, H, H, B, G_ + off_W2, H, tws.ptr, true, true);
        // first hidden layer: dh1 = dz2 W2, dz1 = dh1 [h1 > 0]
        gemm(dZ2.as<bf16>(), ldH, W2b.as<bf16>(), ldH, B, H, H, Z, ldH, tws.ptr, false, true);
        k_relu_back<<<hb, dim3(32, 32), 0, s>>>(B, H, Z, ldH, H1.as<bf16>(), ldH, dZ1.as<bf16>(), G_ + off_b1);
        MDSIP_LAUNCHED();
        gemm(dZ1.as<bf16>(), ldH, Xb.as<bf16>(), ldI, H, I, B, G_ + off_W1, I, tws.ptr, true, true);
    }

    // the fused update moves rows of W3 by TMA: whole 16-byte units
    bool fused_w3() const { return H % 4 == 0; }

    // one Adam step on the gradients of the last backward pass: W3 from its
    // fused gradient where that applies, the rest from G()
    void adam(const AdamStep &st, int64_t B) {
        cudaStream_t s = ctx->stream;
        auto range = [&](int64_t a, int64_t b) {
            k_adam<<<grid_for(b - a, ctx->num_sms), 256, 0, s>>>(b - a, P() + a, G() + a, m1.as<float>() + a,
                                                                 m2.as<float>() + a, st);
            MDSIP_LAUNCHED();
        };
        if (!fused_w3()) {
            range(0, n_params);
            cast_weights();
            return;
        }
        launch_gemm_w3_adam(s, ctx->num_sms, H2.as<bf16>(), ldH, dY.as<bf16>(), ldO, B, O, H, P() + off_W3,
                            m1.as<float>() + off_W3, m2.as<float>() + off_W3, W3b.as<bf16>(), ldH, st, err.as<int>());
        range(0, off_W3);
        range(off_b3, n_params);
        cast_hidden();
    }

    void check_err() {
        int e = 0;
        MDSIP_CUDA(cudaMemcpyAsync(&e, err.ptr, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        MDSIP_CUDA(cudaStreamSynchronize(ctx->stream));
        MDSIP_REQUIRE(e == 0, MDSIP_ERR_DEVICE, "tensor-core GEMM pipeline wait expired");
    }
};

}  // namespace mdsip

using mdsip::Ctx;
using mdsip::DeviceGuard;
using mdsip::Mlp;
using mdsip::guarded;

static inline Mlp *M_(mdsip_mlp *m) { return reinterpret_cast<Mlp *>(m); }
static inline const Mlp *M_(const mdsip_mlp *m) { return reinterpret_cast<const Mlp *>(m); }

static void copy_in(void *dst, const void *src, size_t bytes, int mem, cudaStream_t s) {
    MDSIP_REQUIRE(src != nullptr || bytes == 0, MDSIP_ERR_INVALID_ARG, "null data pointer");
    MDSIP_REQUIRE(mem == MDSIP_MEM_HOST || mem == MDSIP_MEM_DEVICE, MDSIP_ERR_INVALID_ARG, "bad mem tag");
    if (bytes == 0) return;
    MDSIP_CUDA(cudaMemcpyAsync(dst, src, bytes, mem == MDSIP_MEM_HOST ? cudaMemcpyHostToDevice
                                                                      : cudaMemcpyDeviceToDevice, s));
    MDSIP_CUDA(cudaStreamSynchronize(s));
}

static void copy_out(void *dst, const void *src, size_t bytes, int mem, cudaStream_t s) {
    MDSIP_REQUIRE(dst != nullptr || bytes == 0, MDSIP_ERR_INVALID_ARG, "null output pointer");
    MDSIP_REQUIRE(mem == MDSIP_MEM_HOST || mem == MDSIP_MEM_DEVICE, MDSIP_ERR_INVALID_ARG, "bad mem tag");
    if (bytes == 0) return;
    MDSIP_CUDA(cudaMemcpyAsync(dst, src, bytes, mem == MDSIP_MEM_HOST ? cudaMemcpyDeviceToHost
                                                                      : cudaMemcpyDeviceToDevice, s));
    MDSIP_CUDA(cudaStreamSynchronize(s));
}

extern "C" {

mdsip_status mdsip_mlp_create(mdsip_ctx *hctx, int64_t n_in, int64_t n_hidden, int64_t n_out, mdsip_mlp **out) {
    if (!hctx || !out) return MDSIP_ERR_INVALID_ARG;
    *out = nullptr;
    Ctx *ctx = reinterpret_cast<Ctx *>(hctx);
    return guarded(ctx, [&] {
        MDSIP_REQUIRE(n_in > 0 && n_hidden > 0 && n_out > 0 && n_in <= (1 << 20) && n_hidden <= (1 << 16) &&
                          n_out <= (1LL << 30),
                      MDSIP_ERR_INVALID_ARG, "mlp: sizes out of range");
        DeviceGuard g(ctx->device);
        auto *m = new Mlp();
        try {
            m->ctx = ctx;
            m->I = n_in;
            m->H = n_hidden;
            m->O = n_out;
            m->ldI = mdsip::r8(n_in);
            m->ldH = mdsip::r8(n_hidden);
            m->ldO = mdsip::r8(n_out);
            // parameter layout: W1 (H x I) | b1 (H) | W2 (H x H) | b2 (H) | W3 (O x H) | b3 (O),
            // each block starting on a 16-byte boundary
            auto al4 = [](int64_t v) { return (v + 3) / 4 * 4; };
            int64_t o = 0;
            m->off_W1 = o; o = al4(o + n_hidden * n_in);
            m->off_b1 = o; o = al4(o + n_hidden);
            m->off_W2 = o; o = al4(o + n_hidden * n_hidden);
            m->off_b2 = o; o = al4(o + n_hidden);
            m->off_W3 = o; o = al4(o + n_out * n_hidden);
            m->off_b3 = o; o = al4(o + n_out);
            m->n_params = o;
            cudaStream_t s = ctx->stream;
            for (mdsip::DBuf *b : {&m->params, &m->grads, &m->m1, &m->m2}) {
                b->get<float>(ctx, m->n_params);
                MDSIP_CUDA(cudaMemsetAsync(b->ptr, 0, m->n_params * sizeof(float), s));
            }
            m->W1b.get<__nv_bfloat16>(ctx, n_hidden * m->ldI);
            m->W2b.get<__nv_bfloat16>(ctx, n_hidden * m->ldH);
            m->W3b.get<__nv_bfloat16>(ctx, n_out * m->ldH);
            m->in_mean.get<float>(ctx, n_in);
            m->in_std.get<float>(ctx, n_in);
            m->out_mean.get<float>(ctx, n_out);
            m->out_std.get<float>(ctx, n_out);
            mdsip::k_fill_f32<<<1, 256, 0, s>>>(n_in, m->in_mean.as<float>(), 0.0f);
            MDSIP_LAUNCHED();
            mdsip::k_fill_f32<<<1, 256, 0, s>>>(n_in, m->in_std.as<float>(), 1.0f);
            MDSIP_LAUNCHED();
            mdsip::k_fill_f32<<<mdsip::grid_for(n_out, ctx->num_sms), 256, 0, s>>>(n_out, m->out_mean.as<float>(),
                                                                                     0.0f);
            MDSIP_LAUNCHED();
            mdsip::k_fill_f32<<<mdsip::grid_for(n_out, ctx->num_sms), 256, 0, s>>>(n_out, m->out_std.as<float>(),
                                                                                     1.0f);
            MDSIP_LAUNCHED();
            m->err.get<int>(ctx, 1);
            MDSIP_CUDA(cudaMemsetAsync(m->err.ptr, 0, sizeof(int), s));
            m->loss.get<double>(ctx, 1);
            m->cast_weights();
            MDSIP_CUDA(cudaStreamSynchronize(s));
        } catch (...) {
            delete m;
            throw;
        }
        *out = reinterpret_cast<mdsip_mlp *>(m);
    });
}

void mdsip_mlp_destroy(mdsip_mlp *hm) {
    if (!hm) return;
    Mlp *m = M_(hm);
    try {
        DeviceGuard g(m->ctx->device);
        cudaStreamSynchronize(m->ctx->stream);
        delete m;
    } catch (...) {
    }
}

int64_t mdsip_mlp_num_params(const mdsip_mlp *hm) { return hm ? M_(hm)->n_params : 0; }

mdsip_status mdsip_mlp_param_offsets(const mdsip_mlp *hm, int64_t offsets[6]) {
    if (!hm || !offsets) return MDSIP_ERR_INVALID_ARG;
    const Mlp *m = M_(hm);
    offsets[0] = m->off_W1;
    offsets[1] = m->off_b1;
    offsets[2] = m->off_W2;
    offsets[3] = m->off_b2;
    offsets[4] = m->off_W3;
    offsets[5] = m->off_b3;
    return MDSIP_OK;
}

mdsip_status mdsip_mlp_set_params(mdsip_mlp *hm, const float *params, int mem) {
    if (!hm) return MDSIP_ERR_INVALID_ARG;
    Mlp *m = M_(hm);
    return guarded(m->ctx, [&] {
        DeviceGuard g(m->ctx->device);
        cudaStream_t s = m->ctx->stream;
        copy_in(m->params.ptr, params, m->n_params * sizeof(float), mem, s);
        MDSIP_CUDA(cudaMemsetAsync(m->m1.ptr, 0, m->n_params * sizeof(float), s));
        MDSIP_CUDA(cudaMemsetAsync(m->m2.ptr, 0, m->n_params * sizeof(float), s));
        m->t = 0;
        m->cast_weights();
        MDSIP_CUDA(cudaStreamSynchronize(s));
    });
}

mdsip_status mdsip_mlp_get_params(mdsip_mlp *hm, float *params, int mem) {
    if (!hm) return MDSIP_ERR_INVALID_ARG;
    Mlp *m = M_(hm);
    return guarded(m->ctx, [&] {
        DeviceGuard g(m->ctx->device);
        copy_out(params, m->params.ptr, m->n_params * sizeof(float), mem, m->ctx->stream);
    });
}

mdsip_status mdsip_mlp_set_adam(mdsip_mlp *hm, double beta1, double beta2, double eps) {
    if (!hm) return MDSIP_ERR_INVALID_ARG;
    Mlp *m = M_(hm);
    if (!(beta1 >= 0.0 && beta1 < 1.0 && beta2 >= 0.0 && beta2 < 1.0 && eps > 0.0)) {
        m->ctx->last_error = "mlp: Adam constants out of range";
        return MDSIP_ERR_INVALID_ARG;
    }
    m->beta1 = beta1;
    m->beta2 = beta2;
    m->eps = eps;
    return MDSIP_OK;
}

mdsip_status mdsip_mlp_set_scaling(mdsip_mlp *hm, const float *in_mean, const float *in_std, const float *out_mean,
                                   const float *out_std, int mem) {
    if (!hm) return MDSIP_ERR_INVALID_ARG;
    Mlp *m = M_(hm);
    return guarded(m->ctx, [&] {
        DeviceGuard g(m->ctx->device);
        cudaStream_t s = m->ctx->stream;
        if (mem == MDSIP_MEM_HOST) {
            auto pos = [](const float *v, int64_t n) {
                for (int64_t i = 0; i < n; ++i)
                    if (!(v[i] > 0.0f)) return false;
                return true;
            };
            MDSIP_REQUIRE((!in_std || pos(in_std, m->I)) && (!out_std || pos(out_std, m->O)), MDSIP_ERR_INVALID_ARG,
                          "mlp: scaling standard deviations must be positive");
        }
        if (in_mean) copy_in(m->in_mean.ptr, in_mean, m->I * sizeof(float), mem, s);
        if (in_std) copy_in(m->in_std.ptr, in_std, m->I * sizeof(float), mem, s);
        if (out_mean) copy_in(m->out_mean.ptr, out_mean, m->O * sizeof(float), mem, s);
        if (out_std) copy_in(m->out_std.ptr, out_std, m->O * sizeof(float), mem, s);
    });
}

mdsip_status mdsip_mlp_get_scaling(mdsip_mlp *hm, float *in_mean, float *in_std, float *out_mean, float *out_std,
                                   int mem) {
    if (!hm) return MDSIP_ERR_INVALID_ARG;
    Mlp *m = M_(hm);
    return guarded(m->ctx, [&] {
        DeviceGuard g(m->ctx->device);
        cudaStream_t s = m->ctx->stream;
        if (in_mean) copy_out(in_mean, m->in_mean.ptr, m->I * sizeof(float), mem, s);
        if (in_std) copy_out(in_std, m->in_std.ptr, m->I * sizeof(float), mem, s);
        if (out_mean) copy_out(out_mean, m->out_mean.ptr, m->O * sizeof(float), mem, s);
        if (out_std) copy_out(out_std, m->out_std.ptr, m->O * sizeof(float), mem, s);
    });
}

mdsip_status mdsip_mlp_fit_scaling(mdsip_mlp *hm, const double *X, int64_t ldx, const double *Y, int64_t ldy,
                                   int64_t count) {
    if (!hm) return MDSIP_ERR_INVALID_ARG;
    Mlp *m = M_(hm);
    return guarded(m->ctx, [&] {
        MDSIP_REQUIRE(X && Y && count > 0 && ldx >= m->I && ldy >= m->O, MDSIP_ERR_INVALID_ARG,
                      "mlp: bad training data");
        DeviceGuard g(m->ctx->device);
        cudaStream_t s = m->ctx->stream;
        mdsip::k_col_stats<<<mdsip::grid_for(m->I, m->ctx->num_sms), 256, 0, s>>>(
            count, m->I, X, ldx, m->in_mean.as<float>(), m->in_std.as<float>());
        MDSIP_LAUNCHED();
        mdsip::k_col_stats<<<mdsip::grid_for(m->O, m->ctx->num_sms), 256, 0, s>>>(
            count, m->O, Y, ldy, m->out_mean.as<float>(), m->out_std.as<float>());
        MDSIP_LAUNCHED();
        MDSIP_CUDA(cudaStreamSynchronize(s));
    });
}

mdsip_status mdsip_mlp_forward(mdsip_mlp *hm, const double *X, int64_t ldx, int64_t batch, float *Y, int64_t ldy) {
    if (!hm) return MDSIP_ERR_INVALID_ARG;
    Mlp *m = M_(hm);
    return guarded(m->ctx, [&] {
        MDSIP_REQUIRE(batch >= 0 && ldx >= m->I && ldy >= m->O, MDSIP_ERR_INVALID_ARG, "mlp: bad forward arguments");
        if (batch == 0) return;
        MDSIP_REQUIRE(X && Y, MDSIP_ERR_INVALID_ARG, "mlp: null data pointer");
        DeviceGuard g(m->ctx->device);
        m->ensure(batch, false);
        m->forward(X, ldx, nullptr, batch);
        mdsip::launch_out_layer(m->ctx->stream, m->ctx->num_sms, m->H2.as<__nv_bfloat16>(), m->ldH,
                                m->W3b.as<__nv_bfloat16>(), m->ldH, batch, m->O, m->H, m->out_layer(), Y, ldy,
                                m->err.as<int>());
        m->check_err();
    });
}

static void run_gradient(Mlp *m, const double *X, int64_t ldx, const double *Y, int64_t ldy, const int32_t *idx,
                         int64_t batch, bool w3_grad) {
    MDSIP_REQUIRE(X && Y && batch > 0 && ldx >= m->I && ldy >= m->O, MDSIP_ERR_INVALID_ARG,
                  "mlp: bad training arguments");
    m->ensure(batch, true);
    m->forward(X, ldx, idx, batch);
    m->backward(Y, ldy, idx, batch, w3_grad);
}

mdsip_status mdsip_mlp_gradient(mdsip_mlp *hm, const double *X, int64_t ldx, const double *Y, int64_t ldy,
                                const int32_t *idx, int64_t batch, float *grad, double *loss) {
    if (!hm) return MDSIP_ERR_INVALID_ARG;
    Mlp *m = M_(hm);
    return guarded(m->ctx, [&] {
        DeviceGuard g(m->ctx->device);
        run_gradient(m, X, ldx, Y, ldy, idx, batch, true);
        m->check_err();
        if (grad) copy_out(grad, m->grads.ptr, m->n_params * sizeof(float), MDSIP_MEM_DEVICE, m->ctx->stream);
        if (loss) copy_out(loss, m->loss.ptr, sizeof(double), MDSIP_MEM_HOST, m->ctx->stream);
        if (loss) *loss /= (double)batch * (double)m->O;
    });
}

mdsip_status mdsip_mlp_train_step(mdsip_mlp *hm, const double *X, int64_t ldx, const double *Y, int64_t ldy,
                                  const int32_t *idx, int64_t batch, double lr, double *loss) {
    if (!hm) return MDSIP_ERR_INVALID_ARG;
    Mlp *m = M_(hm);
    return guarded(m->ctx, [&] {
        MDSIP_REQUIRE(lr >= 0.0, MDSIP_ERR_INVALID_ARG, "mlp: negative learning rate");
        DeviceGuard g(m->ctx->device);
        run_gradient(m, X, ldx, Y, ldy, idx, batch, !m->fused_w3());
        m->t += 1;
        // the moments decay with the FP32 rates the kernel uses, so the bias
        // corrections 1 - beta^t take those same rates (Kingma-Ba Algorithm 1);
        // with the FP64 rates 1 - 0.999 and 1 - fl32(0.999) differ by 1.3e-5
        const float b1f = (float)m->beta1, b2f = (float)m->beta2;
        const double bc1 = 1.0 - std::pow((double)b1f, (double)m->t), bc2 = 1.0 - std::pow((double)b2f, (double)m->t);
        m->adam(mdsip::AdamStep{(float)lr, b1f, b2f, (float)m->eps, (float)bc1, (float)bc2, 1.0f / (float)bc1,
                               1.0f / (float)bc2}, batch);
        if (loss) {
            m->check_err();
            copy_out(loss, m->loss.ptr, sizeof(double), MDSIP_MEM_HOST, m->ctx->stream);
            *loss /= (double)batch * (double)m->O;
        }
    });
}

}  // extern "C"
