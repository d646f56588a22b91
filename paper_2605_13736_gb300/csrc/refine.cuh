// Iterative refinement of the Newton direction (refine.cu).
#pragma once
#include "vec.cuh"

namespace mdsip {

int64_t refine_sweep_parts(int64_t n);

struct Refiner {
    Dims D;
    ModelView M;
    cudaStream_t st;
    // factor of the reduced matrix
    int64_t N;
    const double *L, *Dd, *Doff;
    const int32_t *perm;
    int num_sms;
    void *solve_ws;   // ldlt_solve_scratch_bytes(N)
    bool solve_fp32;  // the prepared tiles are FP32 (tensor-core factor)
    // FP32 transposed copy of A (n_d x ldt) and an ldt-float scratch: with a
    // tensor-core factor the approximate solve forms its A^T products from it
    const float *AfT;
    int64_t ldt;
    float *vf;
    int *solve_err;
    // Newton quantities of the current attempt
    const double *q, *w, *sig_xd, *sig_d, *Jdh, *Hdd;
    // scratch: bt, tmp_m (m_E), tmp_nd (n_d), tmp_nd2 (n_d + m_I), rhsS (N), colpart, partial
    double *bt, *tmp_m, *tmp_nd, *tmp_nd2, *rhsS, *colpart, *partial;
    double *Au_run;   // A u_d of the current solution, kept as a running sum (m_E)
    // A as an FP32 pair (null: FP64 passes).  With it the approximate solves
    // take FP32 products with A_hi and the residual takes A u_d and A^T u_g
    // from one double-float pass over (A_hi, A_lo)
    const float *Ahi, *Alo;
    float2 *split;    // m_E + n_d float2
    // one-pass sweeps (null xq: not available): the new u_d as FP32 parts with sol_d
    // (n_d), u_d and u_h (n_d + m_I), 1 / q (n_s), 1 / w as FP64 and FP32, sol_g (m_E)
    float4 *xq;
    double *xnew, *qinv, *winv, *sol_g;
    float *wf;

    // b = right-hand side of Eq. (linsys4x4), packed [s | d | g | h]
    void rhs(const IterView &I, const double *gl, const double *cg, const double *ch, const double *sig_d,
             double mu, double dw, double *b);
    // sol = S~^-1-based solve of K sol = b (two-stage elimination with the factor)
    void approx_solve(const double *b, double *sol);
    // after approx_solve: Au_run = A sol_d (init) or Au_run += A sol_d (FP64 passes only)
    void track_Au(bool init);
    // r = b - K u in FP64 (A u_d from Au_run, or from the double-float pass);
    // out4 = (||r||inf, ||b||inf, ||K u||inf, ||u||inf)
    void residual(const double *b, const double *u, double dw, double dc, double *r, double *out4);
    void axpy(int64_t n, const double *x, double *y);
    // The same refinement with approximate solve, update and residual in one
    // step (refine_sweep.cu): rhsS = right-hand side of the first solve, then
    // per sweep u += S~^-1-based solve of K sol = r (u = that of b when init),
    // r = b - K u, out4 as above, rhsS = the next right-hand side; A u_d is left
    // in tmp_m, A^T u_g in tmp_nd
    bool sweep_path() const;
    void sweep_start(const double *b);
    void sweep(const double *b, double *u, double *r, bool init, double dw, double dc, double *out4);
    void rhs_S(const double *b, const double *ATu);   // rhsS = [b_d + A^T u; b_h]
    // full direction (incl. dd and the bound-multiplier steps) from the packed solution
    void direction(const IterView &I, const DirView &Dir, const double *u, double mu, double dw);
};

}  // namespace mdsip
