// Persistent no-interchange LDL^T, FP64 (Section 2.3; the form that runs first
// on the FP64 path): one cooperative launch walks panels of 32 columns; a panel
// is kept when the Bunch-Kaufman rule's column test, evaluated on the computed
// columns, keeps every diagonal pivot, and the first one that is not ends the
// kernel with st->k at its first column (the pivoting panels take over).
//
// GB300 issues an FP64 instruction of a warp in 64 cycles per sub-partition
// (76 with all four busy), whatever its lanes do, and one chain of dependent
// FP64 instructions runs at that same rate.  So the kernel counts FP64 warp
// instructions: element-wise parallel steps spread over the four
// sub-partitions, and the N^3 / 6 multiply-adds of the trailing updates taken
// off that pipe altogether.  Per panel:
//   A  every CTA factors the 32 x 32 diagonal block and its own rows below it
//      in shared memory, in two 16-column sub-panels: the 16 x 16 sub-block one
//      lower-triangle element per thread (one multiply and one FMA per column
//      and warp) with the rows beside it, four threads each, then a rank-16
//      update of the rest; L, D, the column maxima;
//   R  the rows' W scaled by |d|^-1/2 and rounded once to 54-bit integers per
//      row, as residues modulo 13 coprime moduli in BF16 (rns.cuh);
//   B  grid barrier, the column test, the same decision in every CTA;
//   C  the trailing update A -= W D^-1 W^T of a kept panel as 13 exact
//      tensor-core contractions per 128 x 32 tile (bulk copies, tcgen05 into TMEM, the
//      Chinese remainder in 128-bit integers on 16 warps, one rounding to FP64, one FP64
//      subtraction per entry): sum_j sign(d_j) X_ij X_cj <= 32 2^108 in exact
//      integers.  An X is off by at most 2^-53 of its row's largest in the panel, an
//      entry's update by 2^-53 (max|x_i| sum|x_c| + max|x_c| sum|x_i|), at most 2^-49
//      sqrt(b_i b_c) with b_i = sum_j w_ij^2 / |d_j| (a 32-term FP64 dot product by
//      2^-48 sum_j |x_ij x_cj|): the scale of the factorization's other roundings, not
//      entry-wise; grid barrier.
// Against the 64-column form with DFMA trailing tiles (its first panel's tiles
// alone took 215 us): N = 2050 7.90 -> 2.37 ms, 4050 30.6 -> 8.1 ms.  A panel
// takes 30 us at N = 351 to 1036, its pivot chain about 12 of them (32 columns
// of an FP64 multiply and FMA, a reciprocal, an exchange); at N = 2050 37 us, 16
// of them the tiles, whose read-back (13 residues to 128-bit integers per
// entry) is bound by the integer pipes.
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.cuh"
#include "ldlt_panel.cuh"
#include "rns.cuh"
#include "tc.cuh"

namespace mdsip {

namespace {

using bf16 = __nv_bfloat16;

constexpr int RL = 13;                  // moduli: log2 of their product 116.3
constexpr int QB = 54;                  // 2 QB + 5 + 2 <= 116
constexpr int QN = 32;                  // panel width
constexpr int Q_THREADS = 544;          // warps 0-7 factor; 0-15 update, 0-12 issue a modulus each, 16 loads
constexpr int Q_COMP = 256;             // threads of the factorization
constexpr int Q_EPI = 16;               // warps of the trailing update
constexpr int Q_OWN = 96;               // rows below the block staged at a time
constexpr int kFirstTestMax = 128;      // orders whose first column is tested before its panel
constexpr int VP = 33, LP = 33;         // shared-memory row pitches (doubles)
constexpr int QA_BYTES = 128 * 64, QB_BYTES = 32 * 64;   // residues of 128 rows / 32 rows, 32 BF16 each
constexpr int Q_STAGE = QA_BYTES + QB_BYTES;             // one modulus; a tile's 13 are loaded together
constexpr size_t kQSmem = 1024 + (size_t)RL * Q_STAGE + (size_t)(QN + Q_OWN) * (VP + LP) * sizeof(double);

__constant__ rns::Tab<RL> c_tab13 = rns::make_tab<RL>();

struct P64Args {
    PersistArgs p;
    // [modulus][row][32]: X, and sign(d) X (M/p)^-1, modulo p, each 8 rows laid out as
    // the tensor core's 64-byte-swizzled shared-memory atom (16-byte unit c of row r
    // at unit c ^ (r / 2) mod 4), so that a tile's operand is one contiguous copy
    bf16 *RA, *RB;
    int *rowE;           // row exponents
    int npad;
};

__device__ __forceinline__ void bar_comp() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void bar_chain() { asm volatile("bar.sync 2, 128;" ::: "memory"); }

// The 16 x 16 diagonal sub-block at c0 and up to 32 rows below it, together.
// Warps 0 .. 3 hold one element (ei, ej), ej >= 1, of the block's lower
// triangle per lane, 30 lanes each; column j goes through `col` (two buffers of
// 18, one barrier per column); v_it -= (w_i / d) w_t, in that order: w_i w_t
// leaves the range below 2^-511 and above 2^512, and w_i / d is the L that the
// rows below use.  An element gathers what the columns take off it apart until
// its own four columns are due, so that it rounds at its own magnitude four
// times at most, not once a column (reconstruction error at N = 100: 1.1e-16
// rms entry-wise before, 0.67e-16 so; 0.56e-16 with one sum for all columns,
// which costs an addition per column of the chain, 2 us a panel).  Lane 31 of
// each warp also forms the next pivot from its value before the column (col[16],
// col[17]), so that its reciprocal is under way while the column's elements are
// exchanged: a column is a product, an FMA, a reciprocal and two shuffles of
// latency.  Warps 4 .. 7 take the rows on the FP64 pipes that the chain leaves
// idle, four threads each with columns strided by four.  (Chain and rows one
// after the other, with the second Newton step on the FP64 pipe, took 31 of a
// panel's 77 thousand cycles; all four columns unrolled, 0.7 us a panel less.)
__device__ bool q_chain_rows(double *V, double *Ls, double *col, double *s_rc, uint64_t *colbar, uint32_t phase, int c0,
                             int cw, int ei, int ej, int nblk, int nr) {
    bool ok = true;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < 128) {
        const bool elem = lane < 30;
        // y: the element from its own four columns on, what the columns before take off it until then
        const double base = elem && ei < cw ? V[(c0 + ei) * VP + c0 + ej] : 0.0;
        double y = ej < 4 ? base : 0.0;
        double r = rcp_newton(V[c0 * VP + c0]);
        for (int j0 = 0; j0 < cw; j0 += 4) {
            const double add = lane == 31 ? 0.0 : ej >> 2 == (j0 >> 2) + 1 ? base : 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + u;
                if (j >= cw) break;
                double *cb = col + (u & 1) * 18;
                if (j == 0) {
                    if (tid < 16) cb[tid] = V[(c0 + tid) * VP + c0];
                    if (tid == 16) cb[16] = V[(c0 + 1) * VP + c0 + 1];
                } else if (elem && ej == j) {
                    cb[ei] = y;
                    V[(c0 + ei) * VP + c0 + j] = y;
                }
                if (j > 0 && elem && ei == j + 1 && ej == j + 1) {
                    cb[16] = y;
                    if (u == 3) cb[17] = base;
                }
                if (tid == 0) s_rc[c0 + j] = r;
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&colbar[j]);
                bar_chain();
                if (j + 1 < cw) {
                    const bool nd = lane == 31;
                    const double wi = cb[nd ? j + 1 : ei], wt = cb[nd ? j + 1 : ej];
                    double x = fma(-(wi * r), wt, nd ? cb[16] : y);
                    if (u == 3) x += nd ? cb[17] : add;
                    if (ej > j) y = x;
                    r = rcp_newton(__shfl_sync(0xffffffffu, x, 31));
                }
            }
        }
    } else {
        const int q = lane & 3, x = (tid - 128) >> 2, total = min(32, nblk + nr);
        const bool live = x < total;
        const int row = live ? (x < nblk ? c0 + 16 + x : QN + x - nblk) : c0;
        double v[4], y[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            v[s] = live ? V[row * VP + c0 + q + 4 * s] : 0.0;
            y[s] = s == 0 ? v[s] : 0.0;
        }
        const bool any = __any_sync(0xffffffffu, live);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            if (!any || j >= cw) break;
            if (!tc::mbar_wait(&colbar[j], phase)) ok = false;   // column j and its reciprocal are there
            const double l = __shfl_sync(0xffffffffu, y[j >> 2], (lane & ~3) | (j & 3)) * s_rc[c0 + j];
            if (live && (j & 3) == q) Ls[row * LP + c0 + j] = l;
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (4 * s + 3 > j) {
                    const int t = q + 4 * s;
                    y[s] = fma(-l, t > j ? V[(c0 + t) * VP + c0 + j] : 0.0, y[s]);
                    if (4 * s == j + 1) y[s] += v[s];
                }
        }
        if (live) {
#pragma unroll
            for (int s = 0; s < 4; ++s) V[row * VP + c0 + q + 4 * s] = y[s];
        }
    }
    return ok;
}

// Rows x0 .. of those below the sub-block at c0 (nblk block rows from c0 + 16 on,
// then the nr staged own rows): four threads per row, columns strided by four.
__device__ void q_rows(double *V, double *Ls, const double *s_rc, int c0, int first, int nblk, int nr) {
    const int total = nblk + nr;
    const int lane = threadIdx.x & 31, q = lane & 3;
    for (int x0 = first; x0 < total; x0 += Q_COMP / 4) {
        const int x = x0 + (threadIdx.x >> 2);
        const bool live = x < total;
        if (!__any_sync(0xffffffffu, live)) break;   // warp-uniform: no row in this warp
        const int row = live ? (x < nblk ? c0 + 16 + x : QN + x - nblk) : 0;
        double v[4], y[4];   // as above
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            v[s] = live ? V[row * VP + c0 + q + 4 * s] : 0.0;
            y[s] = s == 0 ? v[s] : 0.0;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const double w = __shfl_sync(0xffffffffu, y[j >> 2], (lane & ~3) | (j & 3));
            const double l = w * s_rc[c0 + j];
            if (live && (j & 3) == q) Ls[row * LP + c0 + j] = l;
            if (j < 15) {
#pragma unroll
                for (int s = j >> 2; s < 4; ++s) {
                    if ((j & 3) == 3 && s == (j >> 2)) continue;   // no column of this slot beyond j
                    const int t = q + 4 * s;
                    const double w2 = t > j ? V[(c0 + t) * VP + c0 + j] : 0.0;
                    y[s] = fma(-l, w2, y[s]);
                    if (4 * s == j + 1) y[s] += v[s];
                }
            }
        }
        if (live) {
#pragma unroll
            for (int s = 0; s < 4; ++s) V[row * VP + c0 + q + 4 * s] = y[s];
        }
    }
}

// Rank-16 update of columns 16 .. 31 with the first sub-panel, two columns per
// thread: block rows 16 .. nb - 1 (lower triangle, when blk), own rows.
__device__ void q_rank16(double *V, const double *Ls, int nb, bool blk, int nr) {
    const int nblk = blk ? nb - 16 : 0;
    for (int e = threadIdx.x; e < (nblk + nr) * 8; e += Q_COMP) {
        const int x = e >> 3, c = 16 + 2 * (e & 7);
        const int row = x < nblk ? 16 + x : QN + x - nblk;
        if (x < nblk && c > row) continue;
        double a0 = 0.0, a1 = 0.0;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const double l = Ls[row * LP + j];
            a0 = fma(l, V[c * VP + j], a0);
            a1 = fma(l, V[(c + 1) * VP + j], a1);
        }
        V[row * VP + c] -= a0;
        V[row * VP + c + 1] -= a1;
    }
}

// column maximum of |w| over a warp's rows into s_cmax (bit patterns)
__device__ __forceinline__ void q_colmax(unsigned long long bm, unsigned long long *dst, int lane) {
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(bm >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(bm >> 32) == hi ? (unsigned)bm : 0u);
    if (lane == 0 && (hi | lo)) atomicMax(dst, ((unsigned long long)hi << 32) | lo);
}

// whether the rule keeps a diagonal pivot d against the column's maximum.  (A pivot
// below 2^-1000 has no scaling |d|^-1/2 in the integer form: its panel goes to the
// pivoting kernel, as one that needs an interchange.)
__device__ __forceinline__ bool q_keeps(double d, double colmax, unsigned long long zbits) {
    const double alpha = 0.6403882032022076;   // (1 + sqrt 17) / 8
    constexpr unsigned long long kInf = 0x7ff0000000000000ULL;
    const unsigned long long bd = absbits64(d);
    return bd >= absbits64(alpha * colmax) && bd > zbits && bd < kInf && absbits64(colmax) < kInf;
}

// the panel loop takes over at st->k
__device__ __forceinline__ void q_hand_over(PanelState *st) {
    st->kb = 0;
    st->spec = 0;
    st->nrej += 1;
}

// mbarriers of q_update, and -(bias + k M) modulo 2^128 in s_km (threads 0 .. 15)
__device__ void q_update_init(uint64_t *full, uint64_t *tfull, uint64_t *tempty, uint4 *s_km) {
    const int tid = threadIdx.x;
    if (tid == 0) {
        for (int l = 0; l < RL; ++l) tc::mbar_init(&full[l], 1);
        tc::mbar_init(tfull, RL);
        tc::mbar_init(tempty, Q_EPI);
    }
    if (tid < 16) {
        unsigned __int128 M = 0, B = 0;
        for (int m = 3; m >= 0; --m) {
            M = (M << 32) | c_tab13.mod32[m];
            B = (B << 32) | c_tab13.bias32[m];
        }
        const unsigned __int128 v = (unsigned __int128)0 - B - M * (unsigned __int128)(__int128)(tid - 8);
        s_km[tid] = make_uint4((unsigned)v, (unsigned)(v >> 32), (unsigned)(v >> 64), (unsigned)(v >> 96));
    }
}

// the residues of one row's scaled value (lane = column) at the tensor core's layout
__device__ __forceinline__ int64_t q_at(int64_t row, int lane) {
    return row * QN + ((((lane >> 3) ^ (int)(row >> 1)) & 3) << 3) + (lane & 7);
}

// The trailing update A(i, c) -= sum_t X(i, t) Y(c, t), first <= c <= i < N, from
// residues of X in RA and of Y in RB, by this CTA g of G: tiles of 128 rows from
// `base` (at most 7 below `first`) and tw columns of the lower
// triangle.  tl counts the tiles this warp's role has gone through.
struct QUpdate {
    double *A;
    const bf16 *RA, *RB;
    const int *EA, *EB;   // row exponents
    int N, npad, base, first;
    int off;              // row i's residues are at i - off: a multiple of 8 for base
};

__device__ bool q_update(const QUpdate &u, int G, int g, uint8_t *ring, uint32_t tmem, uint64_t *full, uint64_t *tfull,
                         uint64_t *tempty, const uint4 *s_km, int &tl) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, N = u.N, base = u.base;
    const int nbr = (N - base + 127) / 128;
    // 16 columns a tile when that still is one tile per CTA: half the read-back
    const int tw = 4 * nbr * (nbr + 1) <= G ? 16 : 32, per = 64 / tw;
    const int tiles = per * nbr * (nbr + 1);
            bool ok = true;
            auto tile_at = [&](int t, int &i0, int &c0) {   // false: beyond the last column
                int tr = (int)(sqrtf((float)t / (float)per + 0.25f) - 0.5f);
                while (per * (tr + 1) * (tr + 2) <= t) ++tr;
                while (per * tr * (tr + 1) > t) --tr;
                i0 = base + 128 * tr;
                c0 = base + tw * (t - per * tr * (tr + 1));
                return c0 < N;
            };
            if (wid == Q_EPI) {   // loads: lane l takes modulus l (one thread issuing all 26 copies took 750 cycles each)
                asm volatile("fence.proxy.async;" ::: "memory");
                for (int t = g; t < tiles && ok; t += G) {
                    int i0, c0;
                    if (!tile_at(t, i0, c0)) continue;
                    if (tl > 0 && !tc::mbar_wait(tfull, (tl - 1) & 1)) {   // the previous tile's operands are read
                        ok = false;
                        break;
                    }
                    ++tl;
                    if (lane < RL) {
                        uint8_t *d = ring + lane * Q_STAGE;
                        tc::mbar_expect_tx(&full[lane], QA_BYTES + tw * 64);
                        tc::bulk_load(d, u.RA + ((int64_t)lane * u.npad + i0 - u.off) * QN, QA_BYTES, &full[lane]);
                        tc::bulk_load(d + QA_BYTES, u.RB + ((int64_t)lane * u.npad + c0 - u.off) * QN, tw * 64, &full[lane]);
                    }
                    __syncwarp();
                }
            } else if (wid < Q_EPI) {
                const int quad = wid & 3, quarter = wid >> 2;
                for (int t = g; t < tiles && ok; t += G) {
                    int i0, c0;
                    if (!tile_at(t, i0, c0)) continue;
                    if (wid < RL && lane == 0) {   // this warp's modulus, as soon as it is there
                        if (tc::mbar_wait(tempty, (tl & 1) ^ 1) && tc::mbar_wait(&full[wid], tl & 1)) {
                            tc::fence_after();
                            const uint32_t ab = tc::smem_u32(ring + wid * Q_STAGE), bb = ab + QA_BYTES;
    #pragma unroll
                            for (int s = 0; s < 2; ++s) {
                                const uint64_t da = tc::sw64_kmajor_desc(ab + 32 * s), db = tc::sw64_kmajor_desc(bb + 32 * s);
                                if (tw == 32) tc::mma<false, tc::instr_desc(false, 128, 32)>(tmem + 32 * wid, da, db, s ? 1u : 0u);
                                else tc::mma<false, tc::instr_desc(false, 128, 16)>(tmem + 32 * wid, da, db, s ? 1u : 0u);
                            }
                            tc::commit(tfull);
                        }
                    }
                    __syncwarp();
                    const int i = i0 + 32 * quad + lane, cb = c0 + (tw / 4) * quarter;
                    const int Ei = i < N ? __ldcg(u.EA + i) : 0;
                    const int Ecl = lane < 8 && cb + lane < N ? __ldcg(u.EB + cb + lane) : 0;
                    // two entries of A in use, the next two in flight
                    double old[2], nxt[2];
                    auto fetch = [&](double (&d)[2], int c) {
    #pragma unroll
                        for (int j = 0; j < 2; ++j)
                            d[j] = i < N && c + j <= i && c + j >= u.first ? __ldcg(u.A + i + (int64_t)(c + j) * N) : 0.0;
                    };
                    fetch(nxt, cb);
                    if (!tc::mbar_wait(tfull, tl & 1)) {
                        ok = false;
                        break;
                    }
                    ++tl;
                    tc::fence_after();
                    // parts of the tile above the diagonal or beyond N: nothing to do (warp-uniform)
                    const int nbatch = i0 + 32 * quad < N && cb <= i0 + 32 * quad + 31 ? tw / 8 : 0;
    #pragma unroll 1
                    for (int b = 0; b < nbatch; ++b) {
                        const int c = cb + 2 * b;
    #pragma unroll
                        for (int j = 0; j < 2; ++j) old[j] = nxt[j];
                        if (b + 1 < nbatch) fetch(nxt, c + 2);
                        uint32_t r[RL][2];
                        __syncwarp();
    #pragma unroll
                        for (int l = 0; l < RL; ++l)
                            tc::tmem_ld2_async(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(32 * l + (tw / 4) * quarter + 2 * b), r[l]);
                        tc::tmem_wait_ld();
    #pragma unroll
                        for (int l = 0; l < RL; ++l)   // the values exist only after the wait
                            asm volatile("" : "+r"(r[l][0]), "+r"(r[l][1]));
                        unsigned long long acc[2][4] = {};   // per entry, 32-bit limbs
                        uint64_t yp = 0;                     // the pair's first residues
    #pragma unroll
                        for (int l = 0; l < RL; ++l) {
                            const float pf = c_tab13.p[l], pi = c_tab13.pinv[l];
                            const uint64_t x = rns::pk(__uint_as_float(r[l][0]), __uint_as_float(r[l][1]));
                            const uint64_t qq = rns::add2(rns::fma2(x, rns::pk(pi, pi), rns::pk(rns::kMagic, rns::kMagic)),
                                                          rns::pk(-rns::kMagic, -rns::kMagic));
                            const uint64_t y = rns::fma2(rns::pk(-pf, -pf), qq, x);   // x mod p
                            if (l % 2 == 0 && l + 1 < RL) {
                                yp = y;
                                continue;
                            }
                            // z = y_p q + y_q p (exact); z + 2^19 is the low 23 bits of z + 2^23 + 2^19
                            const uint64_t zb = rns::pk(8912896.0f, 8912896.0f);
                            const float pp = c_tab13.p[l > 0 ? l - 1 : 0];
                            const uint64_t z =
                                l % 2 ? rns::add2(rns::fma2(yp, rns::pk(pf, pf), rns::mul2(y, rns::pk(pp, pp))), zb) : rns::add2(y, zb);
                            const float2 zf = rns::upk(z);
                            const uint32_t u0 = __float_as_uint(zf.x) & 0x7fffffu, u1 = __float_as_uint(zf.y) & 0x7fffffu;
    #pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                acc[0][m] += (unsigned long long)u0 * c_tab13.mpair32[l / 2][m];
                                acc[1][m] += (unsigned long long)u1 * c_tab13.mpair32[l / 2][m];
                            }
                        }
    #pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            // T = sum z M/(p q) + bias; X = T - bias - k M with k = rint((T - bias) / M)
                            unsigned __int128 T = ((unsigned __int128)acc[j][3] << 96) + ((unsigned __int128)acc[j][2] << 64) +
                                                  ((unsigned __int128)acc[j][1] << 32) + acc[j][0];
                            const float f = fmaf((float)(uint32_t)(T >> 96), c_tab13.top, -c_tab13.btop) + rns::kMagic;
                            const uint4 km = s_km[(__float_as_uint(f) + 8u) & 15u];   // kMagic's low bits are zero
                            T += ((unsigned __int128)(((unsigned long long)km.w << 32) | km.z) << 64) |
                                 (((unsigned long long)km.y << 32) | km.x);
                            const int Ec = __shfl_sync(0xffffffffu, Ecl, 2 * b + j);
                            if (i < N && c + j <= i && c + j >= u.first)
                                u.A[i + (int64_t)(c + j) * N] = old[j] - rns::to_double(T, Ei + Ec - 2 * QB);
                        }
                    }
                    tc::fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(tempty);
                }
            }
    return ok;
}

__global__ void __launch_bounds__(Q_THREADS, 1) k_bk_persist64(P64Args q) {
    const PersistArgs &a = q.p;
    extern __shared__ uint8_t psm_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(psm_raw) + 1023) & ~uintptr_t(1023));
    double *V = reinterpret_cast<double *>(ring + RL * Q_STAGE);   // [32 + Q_OWN][VP]: block rows, own rows
    double *Ls = V + (QN + Q_OWN) * VP;                            // [32 + Q_OWN][LP]: L below the 16 x 16 sub-blocks
    __shared__ double s_d[QN], s_rc[QN], s_col[36];
    __shared__ unsigned long long s_cmax[QN], s_sm[QN];
    __shared__ int s_se[QN];
    __shared__ uint4 s_km[16];   // -(bias + k M) modulo 2^128, k = -8 .. 7 at k + 8
    __shared__ __align__(8) uint64_t full[RL], tfull, tempty;   // a modulus loaded, products done, accumulators read
    __shared__ __align__(8) uint64_t colbar[16];   // the chain's columns
    __shared__ uint32_t s_tmem;
    const int N = a.N, G = (int)gridDim.x, g = (int)blockIdx.x, tid = threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
    const double maxabs = __ldg(a.maxabs);
    const unsigned long long zbits = absbits64(fmax(a.zero_tol * maxabs, 0x1p-1000));
    // entries near the subnormal range would lose bits in the integer form: the
    // pivoting panels take such a matrix (st->k stays where it is)
    if (!(maxabs > 0x1p-900)) {
        if (g == 0 && tid == 0) q_hand_over(a.st);
        return;
    }
    // The rule's test on the first column, which takes no update: a small matrix that
    // pivots at once leaves here, the same decision in every CTA (zero diagonal, with
    // the read-back saved below order 96: N = 8 87 -> 67 us, 33 199 -> 160, 64 310 ->
    // 262; at N = 350 the test would cost 9 us of 347 and save 30 of 1680)
    if (N <= kFirstTestMax) {
        if (tid == 0) s_cmax[0] = 0ULL;
        __syncthreads();
        const double *col = a.A + (int64_t)a.st->k * (N + 1);
        unsigned long long bm = 0ULL;
        for (int i = 1 + tid; i < N - a.st->k; i += Q_THREADS) {
            const unsigned long long b = absbits64(__ldcg(col + i));
            bm = b > bm ? b : bm;
        }
        q_colmax(bm, &s_cmax[0], lane);
        __syncthreads();
        const double d = __ldcg(col), colmax = __longlong_as_double((long long)s_cmax[0]);
        if (!q_keeps(d, colmax, zbits)) {
            if (g == 0 && tid == 0) q_hand_over(a.st);
            return;
        }
    }
    if (tid == 0) {
        for (int j = 0; j < 16; ++j) tc::mbar_init(&colbar[j], 4);
    }
    q_update_init(full, &tfull, &tempty, s_km);
    if (tid == 0) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (wid == 0) tc::tmem_alloc(&s_tmem, 512);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = s_tmem;
    int tl = 0;   // tiles this warp's role has gone through
    auto release = [&]() {
        if (wid == Q_EPI && tl > 0 && lane < RL) tc::mbar_wait(&full[lane], (tl - 1) & 1);   // no copy is in flight when the CTA leaves
        __syncwarp();
        tc::fence_before();
        __syncthreads();
        if (wid == 0) tc::tmem_dealloc(tmem, 512);
    };
    // this thread's element of a 16 x 16 lower triangle without its first column
    int ei = 0, ej = 0;
    if (tid < 128 && lane < 30) {
        int e = 30 * wid + lane;
        for (ej = 1; e >= 16 - ej; ++ej) e -= 16 - ej;
        ei = ej + e;
    }

    unsigned epoch = 0;   // grid barriers passed (thread 0)
    uint32_t sub = 0;     // sub-panels gone through
    int p = 0;
    const int kfirst = a.st->k;   // any column: a pivoting panel may have come before
    for (int k = kfirst; k < N; k += QN, ++p) {
        const int nb = min(QN, N - k);
        const int buf = p & 1;
        // own rows: multiples of 8 per CTA
        const int brow = N - k - nb;
        const int R = ((brow + G - 1) / G + 7) / 8 * 8;
        const int r_begin = k + nb + g * R, r_end = min(N, r_begin + R);
        if (wid < 8) {
            for (int cb = r_begin, first = 1; first || cb < r_end; cb += Q_OWN, first = 0) {
                const int nr = max(0, min(Q_OWN, r_end - cb));
                // ---- stage the block (first time) and the own rows
                {
                    double sb[QN * QN / Q_COMP], so[QN / 8];   // every load in flight before the first store
#pragma unroll
                    for (int x = 0; x < QN * QN / Q_COMP; ++x) {
                        const int c = wid + 8 * x;
                        sb[x] = first && lane < nb && c <= lane ? __ldcg(a.A + (int64_t)(k + lane) + (int64_t)(k + c) * N) : 0.0;
                    }
#pragma unroll
                    for (int x = 0; x < QN / 8; ++x) {
                        const int c = wid + 8 * x;
                        so[x] = lane < nr && c < nb ? __ldcg(a.A + (int64_t)(cb + lane) + (int64_t)(k + c) * N) : 0.0;
                    }
                    if (first) {
#pragma unroll
                        for (int x = 0; x < QN * QN / Q_COMP; ++x) V[lane * VP + wid + 8 * x] = sb[x];
                        if (tid < QN) {
                            s_cmax[tid] = 0ULL;
                            s_rc[tid] = 0.0;    // columns beyond a narrow last panel stay zero
                        }
                    }
                    if (lane < nr)
#pragma unroll
                        for (int x = 0; x < QN / 8; ++x) V[(QN + lane) * VP + wid + 8 * x] = so[x];
                }
                for (int c = wid; c < QN; c += 8)
                    for (int r = lane + 32; r < nr; r += 32)
                        V[(QN + r) * VP + c] = c < nb ? __ldcg(a.A + (int64_t)(cb + r) + (int64_t)(k + c) * N) : 0.0;
                bar_comp();
                // ---- factor and solve
                for (int c0 = 0; c0 < nb; c0 += 16) {
                    const int nblk = first ? max(0, nb - c0 - 16) : 0;
                    if (first) {
                        if (!q_chain_rows(V, Ls, s_col, s_rc, colbar, sub & 1, c0, min(16, nb - c0), ei, ej, nblk, nr))
                            atomicExch(&a.bar->err, 1);
                        ++sub;
                        bar_comp();
                    }
                    if (!first || nblk + nr > 32) {
                        q_rows(V, Ls, s_rc, c0, first ? 32 : 0, nblk, nr);
                        bar_comp();
                    }
                    if (c0 == 0 && nb > 16) {
                        q_rank16(V, Ls, nb, first, nr);
                        bar_comp();
                    }
                }
                // ---- pivots and their scaling |d|^-1/2 (warp 0); the block's L and D and the
                // column maxima of its rows, column c by CTA c mod G; the own rows' L and column
                // maxima; a warp per column, lanes over rows
                if (wid == 0) {
                    if (first) {
                        const double d = lane < nb ? V[lane * VP + lane] : 0.0;
                        s_d[lane] = d;
                        unsigned long long m = 0ULL;
                        int e = 0;
                        const double ad = fabs(d);
                        if (ad > 0x1p-1000 && isfinite(ad)) rns::rsqrt64(ad, m, e);   // else the column test rejects the panel
                        s_sm[lane] = m;
                        s_se[lane] = e;
                    }
                } else {
                    for (int c = wid - 1; c < nb; c += 7) {
                        unsigned long long bm = 0ULL;
                        for (int r = lane; r < nr; r += 32) {
                            const double w = V[(QN + r) * VP + c];
                            a.L[(int64_t)(cb + r) + (int64_t)(k + c) * N] = Ls[(QN + r) * LP + c];
                            const unsigned long long bw = absbits64(w);
                            bm = bw > bm ? bw : bm;
                        }
                        if (first && c % G == g && lane >= c && lane < nb) {
                            const int64_t o = (int64_t)(k + lane) + (int64_t)(k + c) * N;
                            const double w = V[lane * VP + c];
                            if (lane == c) {
                                a.L[o] = 1.0;
                                a.Dd[k + c] = w;
                            } else {
                                a.L[o] = w * s_rc[c];
                                const unsigned long long bw = absbits64(w);
                                bm = bw > bm ? bw : bm;
                            }
                        }
                        q_colmax(bm, &s_cmax[c], lane);
                    }
                }
                bar_comp();
                // ---- own rows: residues (a warp per row, lane = panel column)
                for (int r = wid; r < nr; r += 8) {
                    const double w = lane < nb ? V[(QN + r) * VP + lane] : 0.0;
                    const unsigned long long sm = s_sm[lane];
                    const int se = s_se[lane];
                    const int ef = (int)((__double_as_longlong(w) >> 52) & 0x7ff);
                    const int E = __reduce_max_sync(0xffffffffu, ef != 0 ? ef - 1023 + se : -100000) + 2;
                    const rns::Limbs x = rns::limbs(rns::scaled_int(w, sm, se, E, QB));
                    const uint32_t sa = w < 0.0 ? 0x8000u : 0u, sb = sa ^ (s_d[lane] < 0.0 ? 0x8000u : 0u);
                    const int64_t row = cb + r;
                    if (lane == 0) q.rowE[row] = E;
                    const int64_t at = q_at(row - (kfirst & 31), lane);
                    uint16_t *ra = reinterpret_cast<uint16_t *>(q.RA) + at;
                    uint16_t *rb = reinterpret_cast<uint16_t *>(q.RB) + at;
                    const int64_t ls = (int64_t)q.npad * QN;
#pragma unroll
                    for (int l = 0; l < RL; ++l) {
                        const float v = rns::residue(c_tab13, l, x);
                        const float vi = rns::mod(v * c_tab13.inv[l], c_tab13.p[l], c_tab13.pinv[l]);
                        // the BF16 of an integer of magnitude <= 256: the upper half of its FP32
                        ra[l * ls] = (uint16_t)((__float_as_uint(v) >> 16) ^ sa);
                        rb[l * ls] = (uint16_t)((__float_as_uint(vi) >> 16) ^ sb);
                    }
                }
                bar_comp();
            }
            if (tid < nb && s_cmax[tid]) atomicMax(&a.cmax[buf * 64 + tid], s_cmax[tid]);
            asm volatile("fence.proxy.async;" ::: "memory");   // the residues are read by bulk copies
        }
        if (!panel_barrier(a.bar, epoch, a.wait_ns)) break;
        // ---------------- the rule's column test, the same in every CTA
        {
            int keep = 1;
            if (tid < nb)
                keep = q_keeps(s_d[tid], __longlong_as_double((long long)__ldcg(&a.cmax[buf * 64 + tid])), zbits);
            if (!__syncthreads_and(keep)) {
                if (g == 0 && tid == 0) q_hand_over(a.st);   // st->k is this panel's first column
                break;
            }
            if (g == 0) {
                int pos = 0;
                if (tid < nb) {
                    a.kind[k + tid] = 1;
                    a.Doff[k + tid] = 0.0;
                    pos = s_d[tid] > 0.0 ? 1 : 0;
                }
                if (tid < QN) a.cmax[(buf ^ 1) * 64 + tid] = 0ULL;   // the next panel's maxima start at zero
                const int np = __syncthreads_count(pos);
                if (tid == 0) {
                    a.st->npos += np;
                    a.st->nneg += nb - np;
                    a.st->k = k + nb;
                    a.st->kb = nb;
                    // counted in panels of 64 columns, as the panel loop's
                    if (k + nb >= N || (k + nb - kfirst) % 64 == 0) a.st->nacc += 1;
                }
            }
        }
        if (k + nb >= N) break;
        // ---------------- trailing update
        const int base = k + nb;
        const QUpdate up{a.A, q.RA, q.RB, q.rowE, q.rowE, N, q.npad, base, base, kfirst & 31};
        const bool ok = q_update(up, G, g, ring, tmem, full, &tfull, &tempty, s_km, tl);
        if (!ok) atomicExch(&a.bar->err, 1);
        __threadfence();
        if (!panel_barrier(a.bar, epoch, a.wait_ns)) break;
    }
    release();
}

// ---------------------------------------------------------------------------
// The same update after a pivoting panel of at most 32 columns with 1x1 and 2x2
// pivots: X = L with column t scaled by 2^h_t, Y = W by 2^-h_t, 2 h_t the
// exponent of the pivot (block), which balances the two as |d|^1/2 does above.
// (N = 2003: 64-column panels with DFMA tiles 3.9 ms of updates, 31-column ones
// so 1.65, and the panels' own FP64 products halved.)
// ---------------------------------------------------------------------------
struct RnsTrailing {
    int N, npad;
    double *A;
    const double *L, *Dd, *Doff, *Wg, *maxabs;
    const PanelState *st;
    bf16 *RA, *RB;
    int *EA, *EB, *flag, *err;
    int tag;   // of this panel: *flag == tag when its update has to be done term by term
};

constexpr int RT_THREADS = 256;

// residues of the rows below the panel, a warp per row, lane = panel column
__global__ void __launch_bounds__(RT_THREADS) k_bk_rns_rows(RnsTrailing a) {
    pdl_wait();
    pdl_release();
    __shared__ int s_h[QN];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, N = a.N, kb = a.st->kb, first = a.st->k, k = first - kb;
    if (first >= N || kb <= 0) return;
    if (threadIdx.x < QN) {
        int h = 0;
        if (lane < kb) {
            double d = fabs(a.Dd[k + lane]);
            const double o = a.Doff[k + lane], p = lane > 0 ? a.Doff[k + lane - 1] : 0.0;
            if (o != 0.0) d = fmax(fmax(d, fabs(o)), fabs(a.Dd[k + lane + 1]));
            else if (p != 0.0) d = fmax(fmax(d, fabs(p)), fabs(a.Dd[k + lane - 1]));
            const int ef = (int)((__double_as_longlong(d) >> 52) & 0x7ff);
            if (ef != 0 && ef != 0x7ff) h = (ef - 1023) >> 1;
        }
        s_h[lane] = h;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && !(__ldg(a.maxabs) > 0x1p-900)) atomicExch(a.flag, a.tag);
    __syncthreads();
    const int h = s_h[lane];
    const int64_t ls = (int64_t)a.npad * QN;
    for (int i = first + (int)blockIdx.x * (RT_THREADS / 32) + wid; i < N; i += (int)gridDim.x * (RT_THREADS / 32)) {
        const int64_t at = q_at(i, lane);
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const double v = lane < kb ? (side ? a.Wg[i + (int64_t)lane * N] : a.L[i + (int64_t)(k + lane) * N]) : 0.0;
            const int se = side ? -h : h;
            const int ef = (int)((__double_as_longlong(v) >> 52) & 0x7ff);
            if (ef == 0x7ff) atomicExch(a.flag, a.tag);
            const int E = __reduce_max_sync(0xffffffffu, ef != 0 ? ef - 1023 + se : -100000) + 2;
            const rns::Limbs x = rns::limbs(rns::scaled_int(v, 1ULL << 63, se, E, QB));
            const uint32_t sg = v < 0.0 ? 0x8000u : 0u;
            if (lane == 0) (side ? a.EB : a.EA)[i] = E;
            uint16_t *out = reinterpret_cast<uint16_t *>(side ? a.RB : a.RA) + at;
#pragma unroll
            for (int l = 0; l < RL; ++l) {
                float r = rns::residue(c_tab13, l, x);
                if (side) r = rns::mod(r * c_tab13.inv[l], c_tab13.p[l], c_tab13.pinv[l]);
                out[l * ls] = (uint16_t)((__float_as_uint(r) >> 16) ^ sg);
            }
        }
    }
}

__global__ void __launch_bounds__(Q_THREADS, 1) k_bk_rns_trailing(RnsTrailing a) {
    pdl_wait();
    pdl_release();
    extern __shared__ uint8_t psm_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(psm_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint4 s_km[16];
    __shared__ __align__(8) uint64_t full[RL], tfull, tempty;
    __shared__ uint32_t s_tmem;
    const int N = a.N, kb = a.st->kb, first = a.st->k, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (first >= N || kb <= 0) return;
    if (*a.flag == a.tag) {   // entries that the integer form does not hold: term by term
        for (int64_t e = (int64_t)blockIdx.x * Q_THREADS + tid; e < (int64_t)(N - first) * (N - first);
             e += (int64_t)gridDim.x * Q_THREADS) {
            const int i = first + (int)(e % (N - first)), c = first + (int)(e / (N - first));
            if (c > i) continue;
            double s = 0.0;
            for (int t = 0; t < kb; ++t) s = fma(a.L[i + (int64_t)(first - kb + t) * N], a.Wg[c + (int64_t)t * N], s);
            a.A[i + (int64_t)c * N] -= s;
        }
        return;
    }
    q_update_init(full, &tfull, &tempty, s_km);
    if (tid == 0) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (wid == 0) tc::tmem_alloc(&s_tmem, 512);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    int tl = 0;
    const QUpdate up{a.A, a.RA, a.RB, a.EA, a.EB, N, a.npad, first & ~7, first, 0};
    if (!q_update(up, (int)gridDim.x, (int)blockIdx.x, ring, s_tmem, full, &tfull, &tempty, s_km, tl)) atomicExch(a.err, 1);
    if (wid == Q_EPI && tl > 0 && lane < RL) tc::mbar_wait(&full[lane], (tl - 1) & 1);   // no copy in flight on the way out
    tc::fence_before();
    __syncthreads();
    if (wid == 0) tc::tmem_dealloc(s_tmem, 512);
}

int64_t q_npad(int64_t N) { return (N + 127) / 128 * 128 + 128; }
size_t al256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

size_t persist64_scratch_bytes(int64_t N) {
    const size_t np = (size_t)q_npad(std::max<int64_t>(N, 1));
    return 2 * al256(RL * np * QN * sizeof(bf16)) + 2 * al256(np * sizeof(int)) + 256;
}

void launch_persist64(cudaStream_t s, int num_sms, int64_t N, const PersistArgs &pa, void *scratch) {
    P64Args q{};
    q.p = pa;
    q.npad = (int)q_npad(N);
    const size_t rb = al256((size_t)RL * q.npad * QN * sizeof(bf16));
    char *w = static_cast<char *>(scratch);
    q.RA = reinterpret_cast<bf16 *>(w);
    q.RB = reinterpret_cast<bf16 *>(w + rb);
    q.rowE = reinterpret_cast<int *>(w + 2 * rb);
    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_bk_persist64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQSmem);
    }));
    int per_sm = 0;
    MDSIP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bk_persist64, Q_THREADS, kQSmem));
    MDSIP_REQUIRE(per_sm >= 1, MDSIP_ERR_CUDA, "ldlt: persistent factorization does not fit an SM");
    // one CTA per 16 rows below the first block or per 128 x 16 part of the first
    // trailing update, whichever is more, at most one per SM
    const int64_t rest = std::max<int64_t>(0, N - QN), nbr = (rest + 127) / 128;
    const int64_t want = std::max<int64_t>({1, (rest + 15) / 16, 4 * nbr * (nbr + 1)});
    const int G = (int)std::min<int64_t>(want, (int64_t)num_sms);
    void *kargs[] = {&q};
    MDSIP_CUDA(cudaLaunchCooperativeKernel((const void *)k_bk_persist64, dim3(G), dim3(Q_THREADS), kargs, kQSmem, s));
    count_launch();
}

// Trailing update after the pivoting panel numbered `panel` (from 0) of at most
// 32 columns; rest: at most this many columns are left (the panel state says how
// many).  scratch: the persistent kernel's.
void launch_rns_trailing(cudaStream_t s, int num_sms, int64_t N, int64_t rest, int panel, double *A, const double *L,
                         const double *Dd, const double *Doff, const double *Wg, const double *maxabs,
                         const PanelState *st, int *err, void *scratch) {
    RnsTrailing a{};
    a.N = (int)N;
    a.npad = (int)q_npad(N);
    a.A = A;
    a.L = L;
    a.Dd = Dd;
    a.Doff = Doff;
    a.Wg = Wg;
    a.maxabs = maxabs;
    a.st = st;
    const size_t rb = al256((size_t)RL * a.npad * QN * sizeof(bf16)), eb = al256((size_t)a.npad * sizeof(int));
    char *w = static_cast<char *>(scratch);
    a.RA = reinterpret_cast<bf16 *>(w);
    a.RB = reinterpret_cast<bf16 *>(w + rb);
    a.EA = reinterpret_cast<int *>(w + 2 * rb);
    a.EB = reinterpret_cast<int *>(w + 2 * rb + eb);
    a.flag = reinterpret_cast<int *>(w + 2 * rb + 2 * eb);
    a.err = err;
    a.tag = panel + 1;
    static PerDeviceOnce once;
    MDSIP_CUDA(once.run([] {
        return cudaFuncSetAttribute(k_bk_rns_trailing, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQSmem);
    }));
    if (panel == 0) MDSIP_CUDA(cudaMemsetAsync(a.flag, 0, sizeof(int), s));
    const int64_t nbr = (rest + 7 + 127) / 128;
    launch_pdl(k_bk_rns_rows, (unsigned)std::min<int64_t>(4 * num_sms, ceil_div(rest, RT_THREADS / 32)), RT_THREADS, 0, s, 1, a);
    launch_pdl(k_bk_rns_trailing, (unsigned)std::min<int64_t>(num_sms, 4 * nbr * (nbr + 1)), Q_THREADS,
               (size_t)1024 + RL * Q_STAGE, s, 1, a);
}

}  // namespace mdsip
