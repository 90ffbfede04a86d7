// rlb_fixed.cuh -- 64-bit fixed-point arithmetic of the FP64 step.
//
// One binary64 instruction occupies its scheduler's FP64 pipe for 65 clocks
// on GB300 (1.98 per SM per clock), against 1-2 clocks for a 32-bit integer
// add, shift or logic operation and 4 for a 32x32 -> 64 bit multiply-add.  So
// the sums, products and equilibria of a cell are formed in 64-bit integers
// and the FP64 pipe keeps the square root, one reciprocal and the final
// relaxation h + omega (eq - h) of every population.
//
// Block fixed point: the 19 populations of a set share the exponent of the
// largest one (binary64 exponent field emax), x = |v| 2^60 / 2^(emax - 1023),
// so a value keeps all its 53 bits while it lies within 2^-8 of the largest
// and is held to 2^-60 of it below that (binary64 sums round to 2^-53 of
// their result).  Sums of pairs are exact; the sum E (or S) of all 19 and the
// momentum sums carry 2^-56 of the largest population, rounded to nearest.
// E is then normalised to [2^61, 2^62) and every term of the relaxed
// equilibria is an integer in units of 2^-62 of the normalised scale, so the
// terms add without rounding and each sum is rounded once to binary64.
//
// Equilibria in terms of the moments (eps = 3P): with d = M / c_l,
// D = 3 E + eps = 2 E + sqrt(4 E^2 - 3 M^2), u = d / D, and
// (4/3) eps gamma^2 = D / 3, beta = 3 c_l u, Eqs. (equil1s), (equil2as),
// (equil2bs) become
//   f_i = w_i S (1 + 9 e_i.u)
//   g_i = w_i [E / c_l^2 + 13.5 (e_i.d)(e_i.u) - 7.5 d.u + 3 e_i.d],  i > 0
//   g_0 = w_0 [E (3 - 2 / c_l^2) + 1.5 d.u],
// which needs neither gamma^2 nor a subtraction of nearly equal terms.
//
// Weights: the lattice weights are the binary64 numbers nearest 1/3, 1/18 and
// 1/36, as in the binary64 kernels.  All three are (1 - 2^-54) of the
// fraction, so the equilibria carry that factor: over thousands of steps a
// scheme with the exact fractions would drift away from them by 2^-54 a step.
//
// Everything here is integer or explicitly rounded, so the kernels that use
// it (one cell per thread, eight lanes per cell) give the same values.  The
// functions compile for the host as well (checks of the arithmetic).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifndef __CUDACC__
#define RLB_FX inline
#else
#define RLB_FX __host__ __device__ __forceinline__
#endif

namespace rlb {

// A constant in [-2^63, 2^63) as the two 32-bit halves that the products use,
// value = h 2^32 + 2 l, and the rounding term of fx_mul: one half plus the
// mean of the low product it drops.
struct FxConst {
    int32_t h, l;
    uint32_t r;
};

// Per-run constants (made on the host, make_fx_run).
struct FxRun {
    FxConst kE;   // omega / (36 c_l^2)            x 2^65
    FxConst kU;   // omega / 12                    x 2^65
    FxConst kS;   // omega / 36                    x 2^65
    FxConst k0;   // omega (1 - 2 / (3 c_l^2))     x 2^62
    FxConst kQ;   // 5 / 9                         x 2^63
    FxConst kG;   // 1 / 6                         x 2^63
    FxConst kE1;  // 1 / (36 c_l^2)                x 2^65 (adjoint)
    FxConst kE0;  // (3 - 2 / c_l^2) / 3           x 2^62 (adjoint)
    double om4;   // omega / 4
    double omw;   // 1 - omega
    double m3cl2; // -3 c_l^2
    double three_cl;
    float m_max;  // largest |M|^2 / (c_l^2 E^2) of the fast path
    float q_scale;  // beta = q_scale x (high word of w); NaN where that is too coarse
    float c_l;
};

// Per-run constants of the equilibrium initialisation (make_fx_init).
struct FxInit {
    FxConst k6;    // 1 / (6 c_l^2)               x 2^65
    FxConst kEp;   // 1 / (108 c_l^2)             x 2^65
    FxConst k29;   // 2 / 9                       x 2^62
    FxConst kU;    // 2 c_l / 3                   x 2^(62 - sU)
    FxConst kQ, kG;  // as in FxRun
    FxConst k0;    // (1 - 2 / (3 c_l^2)) / 3     x 2^64
    FxConst kS;    // 1 / 36                      x 2^65
    FxConst kS12;  // 1 / (12 c_l)                x 2^65
    double rf, rg, rg0;  // reference populations: diagonal f and g, rest g
    int sU, on;
    int lo, hi;      // high words between which n and eps have to lie
    int re_f, re_g;  // least exponents of S and eps gamma^2 against the reference
};

#include "rlb_fixed_host.h"

RLB_FX int32_t fx_hi(double v) {
#ifdef __CUDA_ARCH__
    return __double2hiint(v);
#else
    uint64_t b;
    memcpy(&b, &v, 8);
    return (int32_t)(b >> 32);
#endif
}
RLB_FX uint32_t fx_lo(double v) {
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2loint(v);
#else
    uint64_t b;
    memcpy(&b, &v, 8);
    return (uint32_t)b;
#endif
}
RLB_FX double fx_double(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    uint64_t b = ((uint64_t)hi << 32) | lo;
    double v;
    memcpy(&v, &b, 8);
    return v;
#endif
}
RLB_FX int fx_clz(uint32_t v) {
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}
// v >> s for any s >= 0 (0 from 64 on)
RLB_FX uint64_t fx_shr(uint64_t v, uint32_t s) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
#else
    return s > 63 ? 0 : v >> s;
#endif
}

// Largest high word of N values without the sign, times 2; the binary64
// exponent field of the largest (0x7FF when one is not finite).
template <int N>
RLB_FX uint32_t fx_max_word(const double* v) {
    uint32_t m = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int i = 0; i < N; ++i) {
        const uint32_t t = (uint32_t)fx_hi(v[i]) << 1;
        m = t > m ? t : m;
    }
    return m;
}
template <int N>
RLB_FX int fx_max_exponent(const double* v) {
    return (int)(fx_max_word<N>(v) >> 21);
}
// The block exponent of values with the largest word m: 1023 for zeros (values
// below 2^-1042 count as zero), and 0x7FF, as for non-finite ones, when all lie
// below 2^-923, where fx_from would keep too few of their bits.
RLB_FX int fx_block_exponent(uint32_t m) { return m >= 100u << 21 ? (int)(m >> 21) : (m ? 0x7FF : 1023); }

// v 2^60 / 2^(emax - 1023), truncated towards zero; |result| < 2^61.
RLB_FX int64_t fx_from(double v, int emax) {
    const uint32_t hi = (uint32_t)fx_hi(v), lo = fx_lo(v);
    const int e = (int)((hi << 1) >> 21);
    // the mantissa with its leading bit at bit 63 (a zero or subnormal v is
    // shifted out entirely: emax is at least 100)
    const uint64_t m = ((uint64_t)((hi << 11) | (lo >> 21) | 0x80000000u) << 32) | (uint64_t)(lo << 11);
    const uint64_t x = fx_shr(m, (uint32_t)(emax + 3 - e));
    const int64_t s = (int64_t)((int32_t)hi >> 31);
    return (int64_t)((x ^ (uint64_t)s) - (uint64_t)s);
}

// the factor (1 - 2^-54) of the binary64 weights; for signed values, whose
// rounding must not have a mean, to nearest
RLB_FX int64_t fx_weight(int64_t v) { return v - (v >> 54); }
RLB_FX int64_t fx_weight_signed(int64_t v) { return v - ((v + (1ll << 53)) >> 54); }

// v 2^s for v >= 0 with v 2^s < 2^63 (truncated)
RLB_FX int64_t fx_fixed(double v, int s) {
    const uint32_t hi = (uint32_t)fx_hi(v), lo = fx_lo(v);
    const uint64_t m = ((uint64_t)((hi << 11) | (lo >> 21) | 0x80000000u) << 32) | (uint64_t)(lo << 11);
    return (int64_t)fx_shr(m, (uint32_t)(1086 - s - (int)(hi >> 20)));
}

// (x + 8) >> 4: from units of 2^-60 to 2^-56 of the block, rounded to nearest
RLB_FX int64_t fx_round4(int64_t x) { return (x + 8) >> 4; }
// Ties always rounded up are an error common to all cells: in signed sums that
// enter a sum over the lattice they go to even (also (x + 4) >> 3), or down in
// one half of the terms.
RLB_FX int64_t fx_round4_even(int64_t x) { return (x + 7 + ((x >> 4) & 1)) >> 4; }
RLB_FX int64_t fx_round3_even(int64_t x) { return (x + 3 + ((x >> 3) & 1)) >> 3; }

// t 2^eb rounded to nearest binary64, |t| < 2^63; the result is a normal
// number (eb from the block exponent, at least 100).
RLB_FX double fx_to(int64_t t, int eb) {
    const int32_t s = (int32_t)(t >> 63);
    uint64_t a = (uint64_t)((t ^ (int64_t)s) - (int64_t)s);
    int n;
    const uint32_t ah = (uint32_t)(a >> 32);
    if (ah != 0u) {
        n = fx_clz(ah) - 1;
    } else {  // far below the scale: rare
        if (a == 0) return 0.0;
        n = 31 + fx_clz((uint32_t)a);
    }
    a = (a << n) + 512u;  // leading bit at 62; round half up in the 53rd bit
    const uint64_t m = a >> 10;
    const uint32_t hi = (uint32_t)(m >> 32) + ((uint32_t)(1084 + eb - n) << 20);
    return fx_double(hi | ((uint32_t)s & 0x80000000u), (uint32_t)m);
}

// fx_to with ties to even: for sums of binary64 values, whose few excess bits
// make ties common (near rest, rounding them up is a bias of 2^-55 a cell).
RLB_FX double fx_to_even(int64_t t, int eb) {
    const int32_t s = (int32_t)(t >> 63);
    uint64_t a = (uint64_t)((t ^ (int64_t)s) - (int64_t)s);
    const uint32_t ah = (uint32_t)(a >> 32);
    if (a == 0) return 0.0;
    const int n = ah != 0u ? fx_clz(ah) - 1 : 31 + fx_clz((uint32_t)a);
    a <<= n;
    const uint64_t m = (a + 511u + ((uint32_t)(a >> 10) & 1u)) >> 10;
    const uint32_t hi = (uint32_t)(m >> 32) + ((uint32_t)(1084 + eb - n) << 20);
    return fx_double(hi | ((uint32_t)s & 0x80000000u), (uint32_t)m);
}

// x 2^-61 for x in [2^61, 2^62), ties to even
RLB_FX double fx_unit(int64_t x) {
    const int64_t r = (x + 255 + ((x >> 9) & 1)) >> 9;
    return fx_double((uint32_t)(r >> 32) + (1022u << 20), (uint32_t)r);
}

// a split for products: value = h 2^32 + 2 l (the lowest bit dropped)
struct FxSplit {
    int32_t h, l;
};
RLB_FX FxSplit fx_split(int64_t a) {
    return {(int32_t)(a >> 32), (int32_t)((uint32_t)a >> 1)};
}
// (a b) 2^-64 within one unit, without bias: the product of the low halves is
// replaced by its mean (2^29 in the units of mid for two arbitrary factors).
RLB_FX int64_t fx_mul(const FxSplit& a, const FxConst& b) {
    const int64_t mid = (int64_t)a.h * b.l + ((int64_t)a.l * b.h + (int64_t)(uint64_t)b.r);
    return (int64_t)a.h * b.h + (mid >> 31);
}
RLB_FX int64_t fx_mul(const FxSplit& a, const FxSplit& b) {
    const int64_t mid = (int64_t)a.h * b.l + ((int64_t)a.l * b.h + 0x60000000ll);
    return (int64_t)a.h * b.h + (mid >> 31);
}
// c + the high word of a b
RLB_FX uint32_t fx_madhi(uint32_t a, uint32_t b, uint32_t c) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b) + c;
#else
    return (uint32_t)(((uint64_t)a * b) >> 32) + c;
#endif
}
// The same with the product of the low halves itself (the mean is wrong where
// they are short: sums of binary32 values), and a's lowest bit rounded to even.
RLB_FX int64_t fx_mul_exact(int64_t a, const FxConst& b) {
    const FxSplit s = fx_split(a + ((a >> 1) & a & 1));
    const uint32_t low = fx_madhi((uint32_t)s.l << 1, (uint32_t)b.l, 1u << 30);
    const int64_t mid = (int64_t)s.h * b.l + ((int64_t)s.l * b.h + (int64_t)(uint64_t)low);
    return (int64_t)s.h * b.h + (mid >> 31);
}
// sum of up to 19 products (a b) 2^-64 of values below 2^61, rounded once.  The
// products of the low halves are added too: their mean in their place would
// be an error common to all cells whose values are short (binary32 lambda,
// zeros), 25 times the other errors' mean.
struct FxDot {
    int64_t hh, mid;
    uint32_t low;
    RLB_FX void add(int64_t x, int64_t y) {
        const FxSplit a = fx_split(x), b = fx_split(y);
        hh += (int64_t)a.h * b.h;
        mid += ((int64_t)a.h * b.l + (int64_t)a.l * b.h) >> 6;
        low = fx_madhi((uint32_t)x, (uint32_t)b.l >> 6, low);
    }
    RLB_FX int64_t result() const { return hh + ((mid + (int64_t)low + (1 << 24)) >> 25); }
};

// What a cell's equilibria are made of, in units of 2^-62 of the normalised
// scale (g0: 2^-59), the antisymmetric f terms for S.
struct FxG {
    int64_t A;                       // omega/36 (E/c_l^2 - 7.5 d.u)
    int64_t Pxx, Pyy, Pzz, Pxy, Pxz, Pyz;  // omega/36 13.5 d_a u_b
    int64_t ux, uy, uz;              // omega/36 3 d_a
    int64_t g0;                      // omega g_0^eq (units of 2^-59)
    FxSplit wx, wy, wz;              // omega u_a / 4, x 2^65
    int eb;                          // exponent of the units: value = t 2^eb
};

// Recovery in binary64 on scaled moments E in [1, 2), d = M / c_l: returns
// (omega / 4) / D.  In the fast path 4 E^2 - 3 M^2 lies in (E^2, 4 E^2].
RLB_FX float fx_seed_f32(double v) {  // binary32 of a positive normal v near 1, truncated
    const uint32_t b = ((uint32_t)(fx_hi(v) - (896 << 20)) << 3) | (fx_lo(v) >> 29);
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float f;
    memcpy(&f, &b, 4);
    return f;
#endif
}
RLB_FX double fx_widen(float f) {  // exact for positive normal f
#ifdef __CUDA_ARCH__
    const uint32_t u = __float_as_uint(f);
#else
    uint32_t u;
    memcpy(&u, &f, 4);
#endif
    return fx_double((u >> 3) + (896u << 20), u << 29);
}
RLB_FX double fx_reciprocal_D(double E, double dx, double dy, double dz, const FxRun& k, double& D) {
    const double E2 = fx_double((uint32_t)fx_hi(E) + (1u << 20), fx_lo(E));  // 2 E
    const double dd = fma(dx, dx, fma(dy, dy, dz * dz));
    const double disc = fma(k.m3cl2, dd, E2 * E2);
    const float df = fx_seed_f32(disc);
#ifdef __CUDA_ARCH__
    const float y = rsqrtf(df);
#else
    const float y = 1.0f / sqrtf(df);
#endif
    const double ys = fx_widen(y), hs = fx_widen(0.5f * y);
    double sq = disc * ys;
    sq = fma(fma(-sq, sq, disc), hs, sq);
    sq = fma(fma(-sq, sq, disc), hs, sq);
    D = E2 + sq;
#ifdef __CUDA_ARCH__
    const float yd = __fdividef(1.0f, fx_seed_f32(D));
#else
    const float yd = 1.0f / fx_seed_f32(D);
#endif
    const double x = fx_widen(yd);
    const double e = fma(-D, x, 1.0);     // third order: x (1 + e + e^2)
    return fma(x, fma(e, e, e), x);
}

// From the sums of the 19 g populations (units of 2^-56 of the block) to the
// terms of their equilibria; false when the cell has to take the general
// path (E <= 0, |M| close to or above E, extreme exponents).  u_d, r_d: the
// scaled momenta and (1/D) in binary64, for the exact positivity test.
RLB_FX bool fx_g_terms(int64_t E, int64_t dx, int64_t dy, int64_t dz, int emax, const FxRun& k, FxG& t, double* u_d,
                       double& r_d) {
    if (emax < 100 || emax > 1900) return false;
    const int32_t Eh = (int32_t)(E >> 32);
    if (Eh <= 0) return false;
    const int n = fx_clz((uint32_t)Eh) - 2;
    if (n > 12) return false;  // E much smaller than its largest population
    const float Ef = (float)Eh, xf = (float)(int32_t)(dx >> 32), yf = (float)(int32_t)(dy >> 32),
                zf = (float)(int32_t)(dz >> 32);
    if (!(xf * xf + yf * yf + zf * zf < k.m_max * (Ef * Ef))) return false;
    E <<= n;  // [2^61, 2^62)
    dx <<= n;
    dy <<= n;
    dz <<= n;
    t.eb = emax - 1080 - n;  // 2^-62 of the scaled value: 2^(emax-1023) 2^(61-56-n) 2^-62
    const double Ed = fx_unit(E);
    u_d[0] = fx_to(dx, -61);
    u_d[1] = fx_to(dy, -61);
    u_d[2] = fx_to(dz, -61);
    double D;
    r_d = fx_reciprocal_D(Ed, u_d[0], u_d[1], u_d[2], k, D);
    const double rW = r_d * k.om4;  // (omega / 4) / D
    const FxSplit r = fx_split(fx_weight(fx_fixed(rW, 65)));
    const FxSplit sx = fx_split(dx), sy = fx_split(dy), sz = fx_split(dz);
    // w = d r: (d 2^61)(rW 2^65) 2^-64 = w 2^62, then x 8
    t.wx = fx_split(fx_mul(sx, r) << 3);
    t.wy = fx_split(fx_mul(sy, r) << 3);
    t.wz = fx_split(fx_mul(sz, r) << 3);
    const FxSplit hx = fx_split(dx + (dx >> 1)), hy = fx_split(dy + (dy >> 1)), hz = fx_split(dz + (dz >> 1));
    t.Pxx = fx_mul(hx, t.wx);
    t.Pyy = fx_mul(hy, t.wy);
    t.Pzz = fx_mul(hz, t.wz);
    t.Pxy = fx_mul(hx, t.wy);
    t.Pxz = fx_mul(hx, t.wz);
    t.Pyz = fx_mul(hy, t.wz);
    t.ux = fx_mul(sx, k.kU);
    t.uy = fx_mul(sy, k.kU);
    t.uz = fx_mul(sz, k.kU);
    const FxSplit X = fx_split((t.Pxx + t.Pyy + t.Pzz) << 1);
    const FxSplit sE = fx_split(E);
    t.A = fx_mul(sE, k.kE) - fx_mul(X, k.kQ);
    t.g0 = fx_mul(sE, k.k0) + fx_mul(X, k.kG);
    return true;
}

// omega g^eq of pair p (units of FxG::eb): symmetric and antisymmetric part
RLB_FX void fx_g_pair(const FxG& t, int p, int64_t& sym, int64_t& asy) {
    switch (p) {
        case 0: sym = (t.A + t.Pxx) << 1; asy = t.ux << 1; break;
        case 1: sym = (t.A + t.Pyy) << 1; asy = t.uy << 1; break;
        case 2: sym = (t.A + t.Pzz) << 1; asy = t.uz << 1; break;
        case 3: sym = (t.A + t.Pxx + t.Pyy) + (t.Pxy << 1); asy = t.ux + t.uy; break;
        case 4: sym = (t.A + t.Pxx + t.Pyy) - (t.Pxy << 1); asy = t.ux - t.uy; break;
        case 5: sym = (t.A + t.Pxx + t.Pzz) + (t.Pxz << 1); asy = t.ux + t.uz; break;
        case 6: sym = (t.A + t.Pxx + t.Pzz) - (t.Pxz << 1); asy = t.ux - t.uz; break;
        case 7: sym = (t.A + t.Pyy + t.Pzz) + (t.Pyz << 1); asy = t.uy + t.uz; break;
        default: sym = (t.A + t.Pyy + t.Pzz) - (t.Pyz << 1); asy = t.uy - t.uz; break;
    }
}

// The f terms: S normalised, B = omega/36 S, F_a = omega/36 9 S u_a.
struct FxF {
    int64_t B, Fx, Fy, Fz;
    int eb;
};
RLB_FX bool fx_f_terms(int64_t S, int emax, const FxG& g, const FxRun& k, FxF& t) {
    if (emax < 100 || emax > 1900) return false;
    const int32_t Sh = (int32_t)(S >> 32);
    if (Sh <= 0) return false;
    const int n = fx_clz((uint32_t)Sh) - 2;
    if (n > 12) return false;
    t.eb = emax - 1080 - n;
    const FxSplit s = fx_split(S << n);
    t.B = fx_mul(s, k.kS);
    t.Fx = fx_mul(s, g.wx);
    t.Fy = fx_mul(s, g.wy);
    t.Fz = fx_mul(s, g.wz);
    return true;
}
RLB_FX void fx_f_pair(const FxF& t, int p, int64_t& sym, int64_t& asy) {
    sym = p < 3 ? t.B << 1 : t.B;
    switch (p) {
        case 0: asy = t.Fx << 1; break;
        case 1: asy = t.Fy << 1; break;
        case 2: asy = t.Fz << 1; break;
        case 3: asy = t.Fx + t.Fy; break;
        case 4: asy = t.Fx - t.Fy; break;
        case 5: asy = t.Fx + t.Fz; break;
        case 6: asy = t.Fx - t.Fz; break;
        case 7: asy = t.Fy + t.Fz; break;
        default: asy = t.Fy - t.Fz; break;
    }
}

#ifdef __CUDACC__
// 1/sqrt(a) for 0 < a <= 1, a normal: binary32 seed y, then the third-order
// step y (1 + e/2 + 3 e^2/8), e = 1 - a y^2.
__device__ __forceinline__ double rsqrt_unit(double a) {
    const double y = fx_widen(rsqrtf(fx_seed_f32(a)));
    const double e = fma(-a * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// The mantissa of a positive normal v in [2^61, 2^62) and its exponent:
// v = x 2^(e - 1023 - 61).
__device__ __forceinline__ int64_t fx_mantissa(double v, int& e) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    e = (int)(hi >> 20);
    return (int64_t)((((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo) << 9);
}
// v 2^s / 2^(e - 1023) for |v| below that range (truncated; s <= 62)
__device__ __forceinline__ int64_t fx_scaled(double v, int e, int s) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const int ev = (int)((hi << 1) >> 21);
    const uint64_t m = ((uint64_t)((hi << 11) | (lo >> 21) | 0x80000000u) << 32) | (uint64_t)(lo << 11);
    const uint64_t x = ev == 0 ? 0 : fx_shr(m, (uint32_t)(63 - s + e - ev));
    const int64_t sg = (int64_t)((int32_t)hi >> 31);
    return (int64_t)((x ^ (uint64_t)sg) - (uint64_t)sg);
}

// t 2^eb rounded to binary32 (c1 c2 = 2^(eb + 32)), and whether a value within
// 128 (d7 - 1) of t could round to another one: t is normalised to 31 leading
// bits and the bits below the 24th compared with one half.  d7 <= 2^nd.
struct F32Out {
    float c1, c2;
    uint32_t d7;
    int nd;
};
__device__ __forceinline__ float fx_to_f32(int64_t t, const F32Out& o, bool& ambiguous) {
    const int32_t hi = (int32_t)(t >> 32);
    const int n = __clz(hi ^ (hi >> 31)) - 1;
    const uint32_t nh = __funnelshift_l((uint32_t)t, (uint32_t)hi, n), nl = (uint32_t)t << n;
    const uint32_t w = __funnelshift_r(nl, nh, 7);  // the 32 bits below the 24 kept
    const uint32_t d = o.d7 << n;
    ambiguous |= (w + 0x80000000u + d) < 2u * d;
    ambiguous |= n + o.nd > 29;  // (also t = 0 and t below 2^32)
    // bit 0 set: the bits dropped from nh then never turn into a tie (an exact
    // tie is ambiguous)
    return (float)(int32_t)(nh | 1u) * __uint_as_float((uint32_t)(127 - n) << 23) * o.c1 * o.c2;
}
__device__ __forceinline__ float pow2f(int k) { return __uint_as_float((uint32_t)(127 + k) << 23); }
// Binary32 values to fixed point: as fx_from, v 2^60 / 2^(emax - 127).
__device__ __forceinline__ int64_t fx_from(float v, int emax) {
    const uint32_t u = __float_as_uint(v);
    const int e = (int)((u << 1) >> 24);
    const uint64_t m = (uint64_t)((u << 8) | 0x80000000u) << 32;
    const uint64_t x = fx_shr(m, (uint32_t)(emax + 3 - e));
    const int64_t s = (int64_t)((int32_t)u >> 31);
    return (int64_t)((x ^ (uint64_t)s) - (uint64_t)s);
}
template <int N>
__device__ __forceinline__ uint32_t fx_max_word(const float* v) {
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t t = __float_as_uint(v[i]) << 1;
        m = t > m ? t : m;
    }
    return m;
}
template <int N>
__device__ __forceinline__ int fx_max_exponent(const float* v) {
    return (int)(fx_max_word<N>(v) >> 24);
}
// The block exponent of N binary32 values for fx_from, which reads subnormals
// as normal numbers and shifts zeros out from an exponent of 61 on only: values
// all below 2^-63 are brought up by 2^96 (exactly) and `lift` says so.
template <int N>
__device__ __forceinline__ int fx_block_exponent(float* v, int& lift) {
    int e = fx_max_exponent<N>(v);
    lift = 0;
    if (e < 64) {
        lift = 96;
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] *= 0x1p96f;
        e = max(fx_max_exponent<N>(v), 64);
    }
    return e;
}
template <int N>
__device__ __forceinline__ int fx_block_exponent(double* v, int& lift) {
    lift = 0;
    return fx_block_exponent(fx_max_word<N>(v));
}

// The moments of a stored state's cell: E, S and d = M / c_l in binary64 (d
// also as integers x 2^(kb - 2)), t = -3 |M|^2 and 4 E^2 - 3 |M|^2.  T = float:
// deviations from (n_ref, eps_ref).  False unless the cell is clearly
// physical (E, S > 0, |M|^2 < 0.98 E^2) and its exponents are in range.
struct FxMoments {
    double E, S, x, y, z, t, disc;
    int64_t ix, iy, iz;
    int kb;
};
template <typename T>
__device__ __forceinline__ bool fx_moments(const T* h, const T* f, double m3cl2, double n_ref, double eps_ref, FxMoments& m) {
    constexpr bool DEV = sizeof(T) == 4;
    // LO: with E below 2^477 the quotients M / E stay above 2^-900 (fx_to)
    constexpr int BIAS = DEV ? 127 : 1023, LO = DEV ? 64 : 624, HI = DEV ? 250 : 1900;
    // the moving populations share an exponent; FP64: the rest population,
    // 9 c_l^2 times larger, is added in binary64; FP32: it shares it too (its
    // deviation carries 24 bits)
    const uint32_t wm = DEV ? fx_max_word<19>(h) : fx_max_word<18>(h + 1), wf = fx_max_word<19>(f);
    const int em = (int)(wm >> (DEV ? 24 : 21)), ef = (int)(wf >> (DEV ? 24 : 21));
    // deviations that are all zero, but not subnormal ones
    bool ok = ((DEV && wm == 0) || em > LO) && em < HI && ((DEV && wf == 0) || ef > LO) && ef < HI;
    double E = 0, sf = 0, dx = 0, dy = 0, dz = 0;
    if (!ok) return false;
    {
        int64_t ix = 0, iy = 0, iz = 0;
        int64_t e = DEV ? fx_round4(fx_from(h[0], em)) : 0, d[9];
        int64_t s = fx_round4(fx_from(f[0], ef));
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const int64_t a = fx_from(h[2 * p + 1], em), b = fx_from(h[2 * p + 2], em);
            e += fx_round4(a + b);
            d[p] = (a - b + 2) >> 2;  // units of 2^-58
            s += fx_round4(fx_from(f[2 * p + 1], ef) + fx_from(f[2 * p + 2], ef));
        }
        const int kb = em - BIAS - 56;
        if (DEV && em == 0) {  // every deviation zero
        } else {
            E = fx_to(e, kb);
            ix = ((d[0] + d[3]) + (d[4] + d[5])) + d[6];
            iy = ((d[1] + d[3]) - d[4]) + (d[7] + d[8]);
            iz = ((d[2] + d[5]) - d[6]) + (d[7] - d[8]);
            dx = fx_to(ix, kb - 2);
            dy = fx_to(iy, kb - 2);
            dz = fx_to(iz, kb - 2);
        }
        if (!(DEV && ef == 0)) sf = fx_to(s, ef - BIAS - 56);
        E += DEV ? eps_ref : (double)h[0];
        if (DEV) sf += n_ref;
        const double E2 = E + E;
        const double t = m3cl2 * fma(dx, dx, fma(dy, dy, dz * dz));  // -3 |M|^2
        const double disc = fma(E2, E2, t);
        // E and S positive, exponents in range, |M|^2 < 0.98 E^2
        const int Eh = __double2hiint(E), Sh = __double2hiint(sf), Dh = __double2hiint(disc);
        const int k = (Eh >> 20) - 1023;
        ok = Eh > (600 << 20) && Eh < (1500 << 20) && Sh > (600 << 20) && Sh < (1500 << 20) && Dh > 0;
        if (ok) {
            const float Em = fx_seed_f32(fx_double((uint32_t)Eh - ((uint32_t)k << 20), (uint32_t)__double2loint(E)));
            const float Dm = fx_seed_f32(fx_double((uint32_t)Dh - ((uint32_t)k << 21), (uint32_t)__double2loint(disc)));
            ok = Dm > 1.06f * Em * Em && Dm < 4.001f * Em * Em;
        }
        m.E = E, m.S = sf, m.x = dx, m.y = dy, m.z = dz, m.t = t, m.disc = disc;
        m.ix = ix, m.iy = iy, m.iz = iz, m.kb = kb;
    }
    return ok;
}

#endif

}  // namespace rlb
