// Declarations shared by the blocked LDL^T (ldlt_blocked.cu) and its
// persistent FP64 kernel (ldlt_persist64.cu).
#pragma once

#include "internal.cuh"

namespace mdsip {

struct PanelState {
    int k;       // first column of the next panel
    int kb;      // columns factored by the last panel
    int npos, nneg, nzero;
    int spec;    // 1: the last panel was taken by the verified no-interchange path
    int nacc, nrej;   // panels that path accepted / handed to the pivoting panel
    unsigned done;    // k_bk_spec CTAs done with the current panel (reset by the last)
    int nfail;        // columns of the pending panel whose row test k_bk_spec_rows evaluates
    unsigned done2;   // k_bk_spec_rows CTAs done (reset by the last)
};

struct PanelBar {
    unsigned count;   // grid-barrier arrivals of the current launch
    unsigned pad0;
    int err, pad;
};

struct PersistArgs {
    int N;
    double *A;                      // lower triangle, column-major, ld N (trailing part updated in place)
    double *L, *Dd, *Doff;
    int32_t *kind;
    float *Lf, *Wf;                 // FP32-update kernel: L and W of the current panel, ld N
    unsigned long long *cmax;       // [2][64]: per-column maxima of |w| (bit patterns), by panel parity
    PanelState *st;
    PanelBar *bar;
    const double *maxabs;
    double zero_tol;
    long long wait_ns;              // bound of each grid-barrier wait
    float *Af;                      // FP32 copy of the lower triangle, ld N (FP32-update kernel)
    float *Lf2, *Wf2;               // FP32-update kernel: the odd panels' L and W columns (ld N)
    unsigned *colcnt;               // FP32-update kernel: per 64-column block, trailing tiles updated
};

namespace {

// Programmatic dependent launch: the kernels of the panel loop are launched
// with programmatic stream serialization, so a kernel's launch overlaps the
// tail of the one before it.  Each waits for its predecessor's completion (and
// memory) before touching data, then lets its own successor launch.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ unsigned long long absbits64(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
}

__device__ __forceinline__ long long global_ns() {
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier of a cooperative launch (all CTAs co-resident).  The
// arrival counter only grows within a launch (k_bk_init clears it): the
// barrier numbered `epoch` (counted by each CTA's thread 0) completes when
// the counter reaches epoch x gridDim.x, so arriving is one release-add with
// no reply to wait for and nobody resets anything.  Every wait is bounded: a
// CTA that waits longer than wait_ns sets the error word and returns false,
// and so does every CTA that sees the word set.
__device__ bool panel_barrier(PanelBar *b, unsigned &epoch, long long wait_ns) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned target = ++epoch * gridDim.x;
        __threadfence();
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&b->count) : "memory");
        const long long t0 = global_ns();
        for (unsigned it = 0;; ++it) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&b->count) : "memory");
            if ((int)(v - target) >= 0) break;
            if ((it & 63) == 63) {
                if (*(volatile int *)&b->err) {
                    ok = 0;
                    break;
                }
                if (global_ns() - t0 > wait_ns) {
                    atomicExch(&b->err, 1);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        if (*(volatile int *)&b->err) ok = 0;
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// launch with programmatic stream serialization (and a cluster when cluster > 1)
template <typename... KArgs, typename... Args>
void launch_pdl(void (*kern)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, int cluster,
                Args... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at[2];
    int na = 0;
    at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
    if (cluster > 1) {
        at[na].id = cudaLaunchAttributeClusterDimension;
        at[na].val.clusterDim.x = (unsigned)cluster;
        at[na].val.clusterDim.y = 1;
        at[na].val.clusterDim.z = 1;
        ++na;
    }
    c.attrs = at;
    c.numAttrs = na;
    MDSIP_CUDA(cudaLaunchKernelEx(&c, kern, args...));
    count_launch();
}

}  // namespace

// ldlt_persist64.cu: the persistent no-interchange factorization, FP64.  One
// cooperative launch from column pa.st->k on; it stops (st->k) at the first
// panel the rule's column test rejects.  scratch: persist64_scratch_bytes(N).
size_t persist64_scratch_bytes(int64_t N);
void launch_persist64(cudaStream_t s, int num_sms, int64_t N, const PersistArgs &pa, void *scratch);
// and the trailing update after a pivoting FP64 panel of at most 32 columns
void launch_rns_trailing(cudaStream_t s, int num_sms, int64_t N, int64_t rest, int panel, double *A, const double *L,
                         const double *Dd, const double *Doff, const double *Wg, const double *maxabs,
                         const PanelState *st, int *err, void *scratch);

}  // namespace mdsip
