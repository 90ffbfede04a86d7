// rlb_fields.cu -- between macroscopic fields and populations: the equilibrium
// initialisation and the macroscopic output.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "rlb_device.cuh"
#include "rlb_fixed.cuh"

namespace rlb {

// ---------------------------------------------------------------------------
// Equilibria of given fields in binary64 throughout (any lattice speed, any
// fields): Eqs. (equil1s), (equil2as), (equil2bs).
// ---------------------------------------------------------------------------
__device__ void equilibrium_f64(double n, double eps, double bx, double by, double bz, const Phys& ph, double* f,
                                double* g) {
    const double b2 = bx * bx + by * by + bz * bz;
    const double gam2 = 1.0 / (1.0 - b2);
    const double ng = n * sqrt(gam2);
    const double eg = eps * gam2;
    const double q[9] = {bx, by, bz, bx + by, bx - by, bx + bz, bx - bz, by + bz, by - bz};
    f[0] = kW0 * ng;
    g[0] = kW0 * (4.0 * eg - eps * (2.0 * ph.inv_cl2 + 1.0) - 2.0 * eg * b2 * ph.inv_cl2);
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const double w = pair_w(p);
        const double fa = 3.0 * q[p] * ph.inv_cl;
        f[2 * p + 1] = w * ng * (1.0 + fa);
        f[2 * p + 2] = w * ng * (1.0 - fa);
        const double gs = eps * ph.inv_cl2 + eg * (6.0 * q[p] * q[p] - 2.0 * b2) * ph.inv_cl2;
        const double ga = eg * 4.0 * q[p] * ph.inv_cl;
        g[2 * p + 1] = w * (gs + ga);
        g[2 * p + 2] = w * (gs - ga);
    }
}

// Rest equilibrium of the FP32 deviation reference.
__device__ __forceinline__ void reference_eq(const Phys& ph, double* fr, double* gr) {
    fr[0] = kW0 * ph.n_ref;
    gr[0] = kW0 * ph.eps_ref * (3.0 - 2.0 * ph.inv_cl2);
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const double w = pair_w(p);
        fr[2 * p + 1] = fr[2 * p + 2] = w * ph.n_ref;
        gr[2 * p + 1] = gr[2 * p + 2] = w * ph.eps_ref * ph.inv_cl2;
    }
}

// Initial populations of one cell in binary64 (deviations for T = float).
template <typename T>
__device__ __noinline__ void init_cell_general(T* A, const Geom& g, const Phys& ph, double n, double eps, double bx,
                                               double by, double bz, int idx) {
    const long long S = g.S;
    double f[19], gg[19];
    equilibrium_f64(n, eps, bx, by, bz, ph, f, gg);
    if constexpr (sizeof(T) == 4) {
        double fr[19], gr[19];
        reference_eq(ph, fr, gr);
        for (int i = 0; i < 19; ++i) {
            f[i] -= fr[i];
            gg[i] -= gr[i];
        }
    }
    for (int i = 0; i < 19; ++i) {
        A[RLB_CHK(i * S + idx, 38ll * S)] = (T)f[i];
        A[RLB_CHK((19 + i) * S + idx, 38ll * S)] = (T)gg[i];
    }
}

// binary64 to binary32, rounded to nearest (the integer-pipe conversion in
// the normal range)
__device__ __forceinline__ float round_f32(double v) {
    const int e = (__double2hiint(v) >> 20) & 0x7FF;
    return e > 900 && e < 1140 ? d2f(v) : (float)v;
}

// ---------------------------------------------------------------------------
// Equilibrium initialisation in 64-bit fixed point (rlb_fixed.cuh).
//
// With v = eps gamma^2 beta, Eqs. (equil1s), (equil2as), (equil2bs) are
//   36 f_i / w = S (1 + 3 e_i.beta / c_l),  36 w = 2 (axis) or 1 (diagonal),
//   g_i = 36 w_i [(4 eps gamma^2 - eps) / (108 c_l^2) - Q + P_ab sums + v.e_i / (9 c_l)],
//   P_ab = v_a beta_b / (6 c_l^2), Q = 5/9 (P_xx + P_yy + P_zz),
//   g_0 = (1 - 2 / (3 c_l^2)) (4 eps gamma^2 - eps) / 3 + 4/3 (P_xx + P_yy + P_zz).
// FP64 instructions: 12 (gamma, S = n gamma, eps gamma^2) instead of some 190,
// which bound the kernel at 65 clocks of a scheduler each.  A cell at rest
// takes six distinct values, formed in binary64.
//
// Binary32 states keep the bits of the binary64 form: its values lie within
// a known distance of the fixed-point ones (the sum of its roundings), and a
// cell with a deviation that close to the midpoint of two binary32 numbers is
// left to it (a few cells in 10^4 in the random box).
//
// Measured (4 to 8 blocks per SM alike): 512^3 FP32 72.6 -> 9.8 ms (2,085
// instructions per 32 cells, ALU pipe 64 % busy), 256^3 FP64 6.52 -> 1.19 ms,
// the sphere lattice FP32 1.25 -> 0.20 ms.
//
// The second state buffer is not written: a step writes every cell of it
// (the halo planes of a z slab excepted, which are initialised in both).
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(128, 6) k_init(const double* __restrict__ n, const double* __restrict__ eps,
                                              const double* __restrict__ beta, const uint8_t* __restrict__ solid,
                                              T* __restrict__ A, T* __restrict__ B, const __grid_constant__ Geom g,
                                              const __grid_constant__ Phys ph) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= g.N) return;
    const long long S = g.S;
    bool both = false;
    if (g.zhalo) {
        const int z = idx / g.nxy;
        both = z == 0 || z == g.nz - 1;
    }
    T* Ac = A + idx;
    T* Bc = B + idx;
    auto put = [&](int q, T v) {
        Ac[RLB_CHK_OFF(q * S, idx, 38ll * S)] = v;
        if (both) Bc[RLB_CHK_OFF(q * S, idx, 38ll * S)] = v;
    };
    if (solid && solid[idx]) {
        T m;
        if constexpr (sizeof(T) == 8) m = solid_marker_d(); else m = solid_marker_f();
#pragma unroll
        for (int q = 0; q < 38; ++q) put(q, m);
        return;
    }
    double nn, ee, bx, by, bz;
    if (g.xbc == XBC_INFLOW_OUTFLOW && idx % g.nx == 0) {
        nn = ph.n_in, ee = ph.eps_in, bx = ph.beta_in[0], by = ph.beta_in[1], bz = ph.beta_in[2];
    } else {
        nn = __ldg(n + idx), ee = __ldg(eps + idx);
        bx = __ldg(beta + idx), by = __ldg(beta + g.N + idx), bz = __ldg(beta + 2 * (long long)g.N + idx);
    }
    if (bx == 0.0 && by == 0.0 && bz == 0.0) {
        // at rest: the operations of equilibrium_f64 that are left
        const double gs = ee * ph.inv_cl2;
        double v[6] = {kW0 * nn, pair_w(0) * nn, pair_w(3) * nn,
                       kW0 * (4.0 * ee - ee * (2.0 * ph.inv_cl2 + 1.0)), pair_w(0) * gs, pair_w(3) * gs};
        T o[6];
        if constexpr (sizeof(T) == 4) {
            double fr[19], gr[19];
            reference_eq(ph, fr, gr);
            const double r[6] = {fr[0], fr[1], fr[7], gr[0], gr[1], gr[7]};
#pragma unroll
            for (int j = 0; j < 6; ++j) o[j] = round_f32(v[j] - r[j]);
        } else {
#pragma unroll
            for (int j = 0; j < 6; ++j) o[j] = v[j];
        }
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            put(i, o[i == 0 ? 0 : (i < 7 ? 1 : 2)]);
            put(19 + i, o[i == 0 ? 3 : (i < 7 ? 4 : 5)]);
        }
        return;
    }
    const FxInit& k = ph.fi;
    const double omb2 = 1.0 - fma(bx, bx, fma(by, by, bz * bz));
    const int oh = __double2hiint(omb2), nh = __double2hiint(nn), eh = __double2hiint(ee);
    // 1/64 < 1 - |beta|^2 <= 1; n and eps positive and well inside the range
    // of the output's exponents
    bool ok = k.on && oh > 0x3F900000 && oh < 0x3FF00001 && nh > k.lo && nh < k.hi && eh > k.lo && eh < k.hi;
    if (ok) {
        const double gam = rsqrt_unit(omb2);
        const double gam2 = gam * gam;
        const double eg = ee * gam2, sn = nn * gam;
        int ge, se;
        const int64_t xg = fx_mantissa(eg, ge);
        const FxSplit xs = fx_split(fx_mantissa(sn, se));
        F32Out og{}, of{}, o0{};
        int64_t rf = 0, rg = 0, rg0 = 0;  // the reference populations in the cell's units
        if constexpr (sizeof(T) == 4) {
            // exponents of the units: g 2^(ge - 1085), f 2^(se - 1085)
            const int kg = ge - 1085 + 32, kf = se - 1085 + 32;
            // distances of the binary64 form, in units: the roundings of each
            // of its operations at the size of their values (u = 2^-53 = 512
            // units; eg, S in [1, 2), b2 = |beta|^2):
            //   f_i: w S (1 + 3 beta) (1.5 b2 gamma^2 + 11) u, axis w = 1/18
            //   g_i: w eg [6 + 8 b2 (3 b2 gamma^2 + 16) + 4 beta (3 b2 gamma^2 + 11)] u / c_l
            //   g_0: 1/3 eg [46 + 40 b2 + 12 b2 gamma^2] u (units 8 times larger)
            // and three roundings of the reference populations
            const float b2 = 1.0f - fx_seed_f32(omb2) + 1e-6f, g2 = fx_seed_f32(gam2), b1 = sqrtf(b2), bg = b2 * g2;
            const float Sm = (float)xs.h * 0x1p-29f, em = (float)(int32_t)(xg >> 32) * 0x1p-29f;
            const float nr = 85.0f * (float)ph.n_ref * pow2f(1023 - se), er = 100.0f * (float)ph.eps_ref * pow2f(1023 - ge);
            auto set = [](F32Out& o, float units) {  // over 128, rounded up
                o.d7 = (uint32_t)(units * (1.03f / 128.0f)) + 2u;
                o.nd = 32 - __clz((int)o.d7);
            };
            set(of, 28.5f * Sm * (1.0f + 3.0f * b1) * (1.5f * bg + 11.0f) + nr);
            set(og, (28.5f * em * (6.0f + 8.0f * b2 * (3.0f * bg + 16.0f) + 4.0f * b1 * (3.0f * bg + 11.0f)) + er) * (float)ph.inv_cl);
            set(o0, 21.4f * em * (46.0f + 40.0f * b2 + 12.0f * bg) + er);
            og.c1 = pow2f(kg >> 1), og.c2 = pow2f(kg - (kg >> 1));
            o0.c1 = 8.0f * og.c1, o0.c2 = og.c2;
            of.c1 = pow2f(kf >> 1), of.c2 = pow2f(kf - (kf >> 1));
            // a cell far below the reference is left to the general path
            ok = se >= k.re_f && ge >= k.re_g;
            rf = fx_scaled(k.rf, se, 62);
            rg = fx_scaled(k.rg, ge, 62);
            rg0 = fx_scaled(k.rg0, ge, 59);
        }
        if (ok) {
            const FxSplit gx = fx_split(xg);
            const int64_t e6 = fx_mul(gx, k.k6);  // eg / (6 c_l^2)
            const FxSplit s6 = fx_split(e6 << 2);
            const FxSplit tx = fx_split(fx_scaled(bx, 1023, 62)), ty = fx_split(fx_scaled(by, 1023, 62)),
                          tz = fx_split(fx_scaled(bz, 1023, 62));
            const FxSplit vx = fx_split(fx_mul(s6, tx) << 2), vy = fx_split(fx_mul(s6, ty) << 2),
                          vz = fx_split(fx_mul(s6, tz) << 2);
            FxG t;
            t.Pxx = fx_mul(vx, tx);
            t.Pyy = fx_mul(vy, ty);
            t.Pzz = fx_mul(vz, tz);
            t.Pxy = fx_mul(vx, ty);
            t.Pxz = fx_mul(vx, tz);
            t.Pyz = fx_mul(vy, tz);
            t.ux = fx_mul(vx, k.kU) << k.sU;
            t.uy = fx_mul(vy, k.kU) << k.sU;
            t.uz = fx_mul(vz, k.kU) << k.sU;
            const int64_t xe = fx_scaled(ee, ge, 61);
            const FxSplit X = fx_split((t.Pxx + t.Pyy + t.Pzz) << 1);
            t.A = fx_mul(s6, k.k29) - fx_mul(fx_split(xe), k.kEp) - fx_mul(X, k.kQ) - rg;
            t.g0 = fx_mul(fx_split(xg - (xe >> 2)), k.k0) + fx_mul(X, k.kG) - rg0;
            const FxSplit s12 = fx_split(fx_mul(xs, k.kS12) << 2);
            FxF q;
            q.B = fx_mul(xs, k.kS) - rf;
            q.Fx = fx_mul(s12, tx);
            q.Fy = fx_mul(s12, ty);
            q.Fz = fx_mul(s12, tz);
            bool ambiguous = false;
            auto gput = [&](int i, int64_t v) {
                if constexpr (sizeof(T) == 8)
                    put(i, fx_to(v, ge - 1085));
                else
                    put(i, fx_to_f32(v, og, ambiguous));
            };
            auto fput = [&](int i, int64_t v) {
                if constexpr (sizeof(T) == 8)
                    put(i, fx_to(v, se - 1085));
                else
                    put(i, fx_to_f32(v, of, ambiguous));
            };
            if constexpr (sizeof(T) == 8) {
                put(19, fx_to(t.g0, ge - 1082));
                put(0, fx_to((q.B << 3) + (q.B << 2), se - 1085));
            } else {
                put(19, fx_to_f32(t.g0, o0, ambiguous));
                put(0, 8.0f * fx_to_f32(q.B + (q.B >> 1), of, ambiguous));
            }
#pragma unroll
            for (int p = 0; p < 9; ++p) {
                int64_t s, a;
                fx_g_pair(t, p, s, a);
                gput(20 + 2 * p, s + a);
                gput(21 + 2 * p, s - a);
                fx_f_pair(q, p, s, a);
                fput(1 + 2 * p, s + a);
                fput(2 + 2 * p, s - a);
            }
            if (!ambiguous) return;
        }
    }
    init_cell_general<T>(A, g, ph, nn, ee, bx, by, bz, idx);
    if (both) init_cell_general<T>(B, g, ph, nn, ee, bx, by, bz, idx);
}

// ---------------------------------------------------------------------------
// Macroscopic output of a stored state (no gather: the moments of the
// post-collision populations equal those of the gathered ones, the
// collision conserves them).
// ---------------------------------------------------------------------------

// One cell with IEEE square roots and divisions, any state: writes its fields
// and returns whether it is unphysical.
template <typename T>
__device__ __noinline__ bool macro_cell_general(const T* A, double* n, double* eps, double* beta, const Geom& g,
                                                const Phys& ph, int idx) {
    const long long S = g.S;
    double f[19], gg[19];
    for (int i = 0; i < 19; ++i) {
        f[i] = (double)A[RLB_CHK(i * S + idx, 38ll * S)];
        gg[i] = (double)A[RLB_CHK((19 + i) * S + idx, 38ll * S)];
    }
    double sf, E, mx, my, mz;
    moments_pairs(f, gg, sf, E, mx, my, mz);
    if constexpr (sizeof(T) == 4) {
        sf += ph.n_ref;
        E += ph.eps_ref;
    }
    mx *= ph.c_l;
    my *= ph.c_l;
    mz *= ph.c_l;
    const double m2 = mx * mx + my * my + mz * mz;
    const double disc = 4.0 * E * E - 3.0 * m2;
    const double e = sqrt(disc) - E;
    const double D = 3.0 * E + e;
    const double bx = 3.0 * mx / D, by = 3.0 * my / D, bz = 3.0 * mz / D;
    const double b2 = bx * bx + by * by + bz * bz;
    const double nn = sf * sqrt(1.0 - b2);
    n[idx] = nn;
    eps[idx] = e;
    beta[idx] = bx;
    beta[g.N + idx] = by;
    beta[2 * (long long)g.N + idx] = bz;
    return !(pos_finite(sf) && pos_finite(E) && nonneg_finite(disc) && pos_finite(e) && below_one(b2) &&
                       pos_finite(nn));
}

// The moment sums are 64-bit integers (exact below 2^-56 of the largest
// population), the recovery binary64 with the square roots and 1/D from
// binary32 seeds: eps = E - 3 M^2 / D, beta = 3 M / D, n = S sqrt(4 eps / D)
// (4 eps / D = 1 - beta^2), 26 FP64 instructions instead of some 120
// with the IEEE sequences, the conversions and the sums.  512^3 FP32 40.3 ->
// 6.5 ms (ALU pipe 84 % busy), 256^3 FP64 3.84 -> 0.94 ms; 4, 5 and 8 blocks
// per SM 8.1, 7.0 and 6.6 ms.
template <typename T>
__global__ void __launch_bounds__(128, 6) k_macro(const T* __restrict__ A, double* __restrict__ n,
                                               double* __restrict__ eps, double* __restrict__ beta,
                                               const __grid_constant__ Geom g, const __grid_constant__ Phys ph,
                                               unsigned long long* bad_count) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= g.N) return;
    const long long S = g.S;
    T h[19], f[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) h[i] = __ldg(RLB_CHK_PTR(A, (19 + i) * S + idx, 38ll * S));
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = __ldg(RLB_CHK_PTR(A, i * S + idx, 38ll * S));
    if (is_solid(f[0])) {
        const double nan = __longlong_as_double(0x7FF8000000000000ll);
        n[idx] = eps[idx] = beta[idx] = beta[g.N + idx] = beta[2 * (long long)g.N + idx] = nan;
        return;
    }
    FxMoments m;
    bool ok = fx_moments(h, f, ph.fx.m3cl2, ph.n_ref, ph.eps_ref, m);
    if (ok) {
        const double E = m.E, E2 = m.E + m.E, t = m.t, disc = m.disc, sf = m.S;
        double ys, hs;
        rsqrt_seed(disc, ys, hs);
        double sq = disc * ys;
        sq = fma(fma(-sq, sq, disc), hs, sq);
        sq = fma(fma(-sq, sq, disc), hs, sq);
        const double D = E2 + sq;
        const double x = rcp_seed(D);
        const double h = fma(-D, x, 1.0);
        const double rD = fma(x, fma(h, h, h), x);
        const double ee = fma(t, rD, E);
        const double r3 = rD * ph.three_cl;
        // sqrt(4 eps / D) = w y with w = eps / D in (0, 1/4]
        const double w = ee * rD;
        const double y = fx_widen(rsqrtf(fx_seed_f32(w)));
        const double s0 = w * y, q = fma(-s0, y, 1.0);
        const double rt = fma(s0 * q, fma(0.375, q, 0.5), s0);
        const double n2 = sf * rt;
        n[idx] = fx_double((uint32_t)__double2hiint(n2) + (1u << 20), (uint32_t)__double2loint(n2));  // 2 S sqrt(eps/D)
        eps[idx] = ee;
        // beta = d r3 in integers: (x 2^(kb - 2)) (r 2^(er - 1023 - 61))
        int er;
        const FxSplit r = fx_split(fx_mantissa(r3, er));
        const int eb = m.kb - 2 + er - 1084 + 64;
        beta[idx] = fx_to(fx_mul(fx_split(m.ix), r), eb);
        beta[g.N + idx] = fx_to(fx_mul(fx_split(m.iy), r), eb);
        beta[2 * (long long)g.N + idx] = fx_to(fx_mul(fx_split(m.iz), r), eb);
    }
    if (!ok && macro_cell_general<T>(A, n, eps, beta, g, ph, idx)) atomicAdd(bad_count, 1ull);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
FxInit make_fx_init(const Phys& ph, int prec) {
    FxInit k{};
    const double c = ph.c_l, c2 = c * c, c2l = fma(c, c, -c2);
    // num / (den c_l^2) and num / (den c_l) as constants times 2^s
    auto over_c2 = [&](double num, double den, int s) {
        double qh, ql;
        fx_div2(num, den, qh, ql);
        const double th = qh / c2, tl = (fma(-th, c2, qh) + (ql - th * c2l)) / c2;
        return fx_const_w(th, tl, s);
    };
    // FP64 populations lose low bits with c_l (see k_step_f64_fx); binary32
    // ones are rounded far above them
    k.on = c >= 1.0 && c <= (prec == 0 ? 2.0 : 16.0) ? 1 : 0;
    if (!k.on) return k;
    k.k6 = over_c2(1.0, 6.0, 65);
    k.kEp = over_c2(1.0, 108.0, 65);
    double qh, ql;
    fx_div2(2.0, 9.0, qh, ql);
    k.k29 = fx_const(qh, ql, 62);
    k.sU = 0;
    while (ldexp(1.0, k.sU) < 2.0 * c / 3.0) ++k.sU;
    fx_div2(2.0 * c, 3.0, qh, ql);
    k.kU = fx_const(qh, ql, 62 - k.sU);
    fx_div2(5.0, 9.0, qh, ql);
    k.kQ = fx_const(qh, ql, 63);
    fx_div2(1.0, 6.0, qh, ql);
    k.kG = fx_const(qh, ql, 63);
    // (1 - 2/(3 c_l^2)) / 3 = 1/3 - (2/9)/c_l^2
    fx_div2(2.0, 9.0, qh, ql);
    const double th = qh / c2, tl = (fma(-th, c2, qh) + (ql - th * c2l)) / c2;
    double oh, ol;
    fx_div2(1.0, 3.0, oh, ol);
    const double dh = oh - th, de = ((oh - dh) - th) + (ol - tl);
    k.k0 = fx_const_w(dh, de, 64);
    fx_div2(1.0, 36.0, qh, ql);
    k.kS = fx_const_w(qh, ql, 65);
    fx_div2(1.0, 12.0 * c, qh, ql);
    k.kS12 = fx_const_w(qh, ql, 65);
    // exponents (high words) that leave every product and the output in range:
    // a deviation that fx_to_f32 decides is at least 2^-29 of its cell's
    // scale, and below 2^-126 it would be rounded a second time
    k.lo = (prec == 0 ? 200 : 1023 - 96) << 20;
    k.hi = (prec == 0 ? 1800 : 1023 + 110) << 20;
    k.rf = ph.n_ref / 36.0;
    k.rg = ph.eps_ref / 36.0 * ph.inv_cl2;
    k.rg0 = kW0 * ph.eps_ref * (3.0 - 2.0 * ph.inv_cl2);
    // twice the sums, reference subtracted, stay below 2^63: the reference
    // below half the cell's scale (units of 2^-62), the rest one below 8
    // times it (units of 2^-59)
    k.re_f = ilogb(k.rf) + 1025;
    k.re_g = ilogb(k.rg) + 1025;
    if (ilogb(k.rg0) + 1021 > k.re_g) k.re_g = ilogb(k.rg0) + 1021;
    return k;
}

cudaError_t launch_init(int prec, const Geom& g, const Phys& ph, const double* n, const double* eps,
                        const double* beta, const uint8_t* solid, void* A, void* B, cudaStream_t st) {
    set_last_launch_count(1);
    if (prec == 0)
        k_init<double><<<(unsigned)((g.N + 127ll) / 128), 128, 0, st>>>(n, eps, beta, solid, (double*)A, (double*)B, g, ph);
    else
        k_init<float><<<(unsigned)((g.N + 127ll) / 128), 128, 0, st>>>(n, eps, beta, solid, (float*)A, (float*)B, g, ph);
    return cudaGetLastError();
}

cudaError_t launch_macro(int prec, const Geom& g, const Phys& ph, const void* A, double* n, double* eps,
                         double* beta, Counters cnt, cudaStream_t st) {
    set_last_launch_count(1);
    if (prec == 0)
        k_macro<double><<<(unsigned)((g.N + 127ll) / 128), 128, 0, st>>>((const double*)A, n, eps, beta, g, ph, cnt.macro_bad);
    else
        k_macro<float><<<(unsigned)((g.N + 127ll) / 128), 128, 0, st>>>((const float*)A, n, eps, beta, g, ph, cnt.macro_bad);
    return cudaGetLastError();
}

// Bounds-check count of this translation unit (0 in the release build).
RLB_OOB_TAKE_FN(oob_take_fields)

}  // namespace rlb
