// Residue number system for exact integer contractions on the BF16 tensor
// cores: tables of pairwise coprime moduli (<= 512, residues of magnitude <=
// 256, exact in BF16), Chinese remainder constants, and the scalar pieces the
// users share (syrk_rns.cu, ldlt_persist64.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace mdsip {
namespace rns {

constexpr int kModuli[14] = {512, 511, 509, 507, 505, 503, 499, 493, 491, 487, 479, 473, 467, 463};
constexpr int LIMB = 14;               // bits per limb of |X| when residues are formed
constexpr float kMagic = 12582912.0f;  // 1.5 2^23: adding and subtracting it rounds to an integer

template <int RN>
struct Tab {
    float p[RN], pinv[RN];
    float c1[RN], c2[RN], c3[RN];      // 2^14, 2^28, 2^42 mod p, symmetric
    float inv[RN];                     // (M / p)^-1 mod p, symmetric
    // moduli taken in pairs (a last one alone): sum_l y_l M/p_l is the sum over
    // pairs of z M/(p q), z = y_p q + y_q p, |z| < 2^19
    uint32_t mpair32[(RN + 1) / 2][4], mod32[4], bias32[4];   // M/(p q), M, 2^19 sum of M/(p q) modulo 2^128, 32-bit limbs
    float top, btop;                   // 2^96 / M; bias / M
};

constexpr int sym(int v, int p) {
    v %= p;
    if (v < 0) v += p;
    return v > p / 2 ? v - p : v;
}

template <int RN>
constexpr Tab<RN> make_tab() {
    Tab<RN> t{};
    unsigned __int128 M = 1, bias = 0;
    double bias_M = 0.0;
    for (int l = 0; l < RN; ++l) M *= (unsigned)kModuli[l];
    for (int l = 0; l < RN; ++l) {
        const int p = kModuli[l];
        t.p[l] = (float)p;
        t.pinv[l] = 1.0f / (float)p;
        t.c1[l] = (float)sym((int)((1LL << LIMB) % p), p);
        t.c2[l] = (float)sym((int)((1LL << (2 * LIMB)) % p), p);
        t.c3[l] = (float)sym((int)((1LL << (3 * LIMB)) % p), p);
        const unsigned __int128 h = M / (unsigned)p;
        const int hm = (int)(h % (unsigned)p);
        for (int v = 1; v < p; ++v)
            if ((v * hm) % p == 1) t.inv[l] = (float)sym(v, p);
    }
    for (int l = 0; l < RN; l += 2) {
        const unsigned __int128 h = M / (unsigned)kModuli[l] / (unsigned)(l + 1 < RN ? kModuli[l + 1] : 1);
        bias += h << 19;
        bias_M += (double)(1 << 19) / ((double)kModuli[l] * (l + 1 < RN ? kModuli[l + 1] : 1));
        for (int j = 0; j < 4; ++j) t.mpair32[l / 2][j] = (uint32_t)(h >> (32 * j));
    }
    for (int j = 0; j < 4; ++j) {
        t.mod32[j] = (uint32_t)(M >> (32 * j));
        t.bias32[j] = (uint32_t)(bias >> (32 * j));
    }
    t.top = (float)(79228162514264337593543950336.0 / (double)M);
    t.btop = (float)bias_M;   // (the bias itself passes 2^128 with 14 moduli)
    return t;
}

#ifdef __CUDACC__
// w^-1/2 = sm 2^(se - 63), sm accurate to about 63 bits (one Newton correction
// of the FP64 value with exact residuals), for w positive and well inside the
// FP64 range
__device__ __forceinline__ void rsqrt64(double v, unsigned long long &sm, int &se) {
    const double s = 1.0 / sqrt(v);
    const double h = v * s, hl = fma(v, s, -h);
    const double r = fma(-h, s, 1.0) - hl * s;             // 1 - v s^2
    se = (int)((__double_as_longlong(s) >> 52) & 0x7ff) - 1023;
    const unsigned long long mant =
        (((unsigned long long)__double_as_longlong(s) & 0xfffffffffffffULL) | 0x10000000000000ULL) << 11;
    const double cd = ldexp(0.5 * s * r, 63 - se);
    // (s is a rounded root's rounded reciprocal: up to 1.5 units, 3072 of cd, off)
    const long long c = __double2ll_rn(cd);
    sm = mant + (unsigned long long)c;
    if (c > 0 && sm < mant) {              // past 2^64
        sm = (sm >> 1) | (1ULL << 63);
        ++se;
    }
}

// |X| for X = rint(a s 2^(b - E)), s = sm 2^(se - 63), given that |a s| < 2^E; 0
// for a zero or subnormal
__device__ __forceinline__ unsigned long long scaled_int(double a, unsigned long long sm, int se, int E, int b) {
    const long long bits = __double_as_longlong(a);
    const int ef = (int)((bits >> 52) & 0x7ff);
    if (ef == 0) return 0ULL;
    const unsigned long long mant = (((unsigned long long)bits & 0xfffffffffffffULL) | 0x10000000000000ULL) << 11;
    // a s = hi 2^(ea + es - 62); X = hi >> sh with rounding, sh >= 64 - b
    const unsigned long long hi = __umul64hi(mant, sm);
    const int sh = 62 - b + E - (ef - 1023 + se) - 1;
    return sh < 64 ? ((hi >> sh) + 1ULL) >> 1 : 0ULL;
}

// limbs of |X| as FP32
struct Limbs {
    float x0, x1, x2, x3;
};
__device__ __forceinline__ Limbs limbs(unsigned long long X) {
    auto lf = [](unsigned u) { return __uint_as_float(0x4B000000u | u) - 8388608.0f; };
    return Limbs{lf((unsigned)X & 0x3fffu), lf((unsigned)(X >> LIMB) & 0x3fffu), lf((unsigned)(X >> (2 * LIMB)) & 0x3fffu),
                 lf((unsigned)(X >> (3 * LIMB)))};
}

// t mod p, |t| < 2^24 (the quotient rounded by the 1.5 2^23 trick)
__device__ __forceinline__ float mod(float t, float p, float pinv) {
    return fmaf(-p, __fadd_rn(fmaf(t, pinv, kMagic), -kMagic), t);
}

template <int RN>
__device__ __forceinline__ float residue(const Tab<RN> &tab, int l, const Limbs &x) {
    return mod(fmaf(tab.c3[l], x.x3, fmaf(tab.c2[l], x.x2, fmaf(tab.c1[l], x.x1, x.x0))), tab.p[l], tab.pinv[l]);
}

// the two's complement 128-bit integer u times 2^e, rounded to nearest, ties to
// even, in integers (an FP64 instruction costs as much as 64 integer ones)
__device__ __forceinline__ double to_double(unsigned __int128 u, int e) {
    if (u == 0) return 0.0;
    const bool neg = (long long)(u >> 64) < 0;
    if (neg) u = (unsigned __int128)0 - u;
    unsigned long long hi = (unsigned long long)(u >> 64);
    const int z = hi ? __clzll((long long)hi) : 64 + __clzll((long long)(unsigned long long)u);
    u <<= z;
    hi = (unsigned long long)(u >> 64);   // top bit set
    const int ex = 127 - z + e;           // exponent of the value
    double val;
    if (ex > -1022 && ex < 1023) {
        unsigned long long mant = hi >> 11;
        const unsigned rest = (unsigned)hi & 0x7ffu;
        mant += rest > 0x400u || (rest == 0x400u && ((unsigned long long)u != 0ULL || (mant & 1ULL)));
        val = __longlong_as_double((long long)(((unsigned long long)(ex + 1022) << 52) + mant));
    } else {
        val = scalbn((double)(hi | ((unsigned long long)u != 0ULL)), ex - 63);
    }
    return neg ? -val : val;
}

// packed FP32 pairs
__device__ __forceinline__ uint64_t pk(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 upk(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
#endif

}  // namespace rns
}  // namespace mdsip
