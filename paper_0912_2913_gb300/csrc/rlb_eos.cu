// rlb_eos.cu -- the relativistic lattice Boltzmann step with a general
// equation of state (an ideal gas with rest mass m,
//     P = (Gamma - 1)(eps - n m)):
// the equilibria of Eqs. (equil1), (equil2a), (equil2b), the macroscopic
// constraints n gamma = sum f, (eps + P) gamma^2 - P = sum g,
// (eps + P) gamma^2 u = sum g c, and their inversion by a Newton iteration on
// P.  Gamma = 4/3, m = 0 is the eps = 3P scheme.  FP64 states only.
//
// Recovery: with D = sum f, E = sum g, M = sum g c and a trial P,
//     beta = M / (E + P),   eps = E - |M|^2 / (E + P),   n = D sqrt(1 - beta^2);
// P solves r(P) = (Gamma - 1)(eps(P) - m n(P)) - P = 0, with
//     r'(P) = (Gamma - 1)(beta^2 - m n beta^2 / ((E + P)(1 - beta^2))) - 1,
// started from the massless solution (the positive root of
// X^2 - Gamma E X + (Gamma - 1)|M|^2 = 0 for X = E + P, then
// P = (Gamma - 1)(eps - m n) at its eps and n) and iterated until
// |dP| <= 1e-14 (P + E), at most 100 iterations.  Reciprocals and inverse
// square roots are binary32 seeds refined by two FP64 Newton-Raphson steps
// (x -> x (2 - a x) and y -> y (3 - a y^2)/2), which are far cheaper than the
// IEEE FP64 sequences on this GPU's FP64 pipe.
#include <cuda_runtime.h>
#include <stdint.h>

#include "rlb_device.cuh"
#include "rlb_fixed.cuh"

namespace rlb {

namespace {

__device__ __forceinline__ double rcp64(double a) {
    double x = rcp_seed(a);
    x = fma(x, fma(-a, x, 1.0), x);
    x = fma(x, fma(-a, x, 1.0), x);
    return x;
}

__device__ __forceinline__ double rsqrt64(double a) {
    double y, half_y;
    rsqrt_seed(a, y, half_y);
    (void)half_y;
    y = y * fma(-0.5 * a * y, y, 1.5);
    y = y * fma(-0.5 * a * y, y, 1.5);
    return y;
}

__device__ __forceinline__ double eos_pressure(const Phys& ph, double n, double eps) {
    return (ph.eos_gamma - 1.0) * (eps - n * ph.eos_mass);
}

// Eqs. (equil1), (equil2a), (equil2b) in pair form: q_p = e_p . beta, so
// (c_i . u)/c_l^2 = +-q_p/c_l and (c_i . u)^2/c_l^4 = q_p^2/c_l^2.
__device__ __forceinline__ void equilibrium_general(double n, double eps, double P, double bx, double by, double bz,
                                                    const Phys& ph, double* f, double* g) {
    const double b2 = bx * bx + by * by + bz * bz;
    const double gam = rsqrt64(1.0 - b2);
    const double gam2 = gam * gam;
    const double h = (eps + P) * gam2;
    const double pr = P * rcp64(h);  // P / ((P + eps) gamma^2)
    const double rest = 3.0 * pr * ph.inv_cl2;
    const double ng = n * gam;
    f[0] = kW0 * ng;
    g[0] = kW0 * h * (3.0 - 3.0 * pr * (2.0 + ph.c_l * ph.c_l) * ph.inv_cl2 - 1.5 * b2 * ph.inv_cl2);
    const double q[9] = {bx, by, bz, bx + by, bx - by, bx + bz, bx - bz, by + bz, by - bz};
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const double w = pair_w(p);
        const double fa = 3.0 * q[p] * ph.inv_cl;
        f[2 * p + 1] = w * ng * (1.0 + fa);
        f[2 * p + 2] = w * ng * (1.0 - fa);
        const double gs = w * h * (rest + 4.5 * q[p] * q[p] * ph.inv_cl2 - 1.5 * b2 * ph.inv_cl2);
        const double ga = w * h * 3.0 * q[p] * ph.inv_cl;
        g[2 * p + 1] = gs + ga;
        g[2 * p + 2] = gs - ga;
    }
}

// Returns true when the state is unphysical (see the file header).
__device__ __forceinline__ bool recover_general(double D, double E, double mx, double my, double mz, const Phys& ph,
                                                double& n, double& eps, double& P, double& bx, double& by,
                                                double& bz) {
    const double M2 = mx * mx + my * my + mz * mz;
    const double g1 = ph.eos_gamma - 1.0;
    const double mass = ph.eos_mass;
    double p;
    {
        // massless solution: X = E + P, X^2 - Gamma E X + (Gamma - 1) M^2 = 0
        const double ge = ph.eos_gamma * E;
        const double disc = fma(ge, ge, -4.0 * g1 * M2);
        const double X = 0.5 * (ge + disc * rsqrt64(disc));
        const double rX = rcp64(X);
        const double b2 = M2 * rX * rX;
        const double omb = 1.0 - b2;
        p = g1 * ((E - M2 * rX) - mass * D * (omb * rsqrt64(omb)));
        const double lo = sqrt(M2) - E;
        if (!(p > lo)) p = lo + 1e-3 * (E > 0.0 ? E : 1.0);
    }
    bool conv = false;
    for (int it = 0; it < 100; ++it) {
        const double rW = rcp64(E + p);
        const double b2 = M2 * rW * rW;
        const double rs = rsqrt64(1.0 - b2);
        const double nn = D * ((1.0 - b2) * rs);
        const double ep = E - M2 * rW;
        const double r = g1 * (ep - mass * nn) - p;
        const double dr = g1 * (b2 - mass * D * rs * b2 * rW) - 1.0;  // n / (1 - b2) = D rs
        const double dp = -r * rcp64(dr);
        p = p + dp;
        if (fabs(dp) <= 1e-14 * (fabs(p) + fabs(E))) {
            conv = true;
            break;
        }
    }
    const double rW = rcp64(E + p);
    bx = mx * rW;
    by = my * rW;
    bz = mz * rW;
    const double b2 = bx * bx + by * by + bz * bz;
    n = D * ((1.0 - b2) * rsqrt64(1.0 - b2));
    eps = E - M2 * rW;
    P = p;
    return !(conv && pos_finite(D) && pos_finite(E) && pos_finite(p) && below_one(b2) && isfinite(n) &&
             isfinite(eps) && isfinite(bx) && isfinite(by) && isfinite(bz));
}

// One collided cell in binary64 throughout (any lattice speed, any state);
// false for a solid cell.
template <int XBC>
__device__ __forceinline__ bool step_cell_eos(const double* __restrict__ A, double* __restrict__ B, const Geom& g,
                                              const Phys& ph, int idx, int x, const PullOffsets& o, bool& unphys,
                                              bool& nonpos) {
    const long long S = g.S;
    double f[19], gg[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const int s = idx + o.src(i);
        f[i] = A[RLB_CHK(i * S + s, 38ll * S)];
        gg[i] = A[RLB_CHK((19 + i) * S + s, 38ll * S)];
    }
    if (is_solid(f[0])) {  // the cell itself is solid: keep the marker
        const double m = solid_marker_d();
        for (int q = 0; q < 38; ++q) B[RLB_CHK(q * S + idx, 38ll * S)] = m;
        return false;
    }
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        if (is_solid(f[i])) {  // link bounce-back
            f[i] = A[RLB_CHK(opp(i) * S + idx, 38ll * S)];
            gg[i] = A[RLB_CHK((19 + opp(i)) * S + idx, 38ll * S)];
        }
    }
    double sf, E, mx, my, mz;
    moments_pairs(f, gg, sf, E, mx, my, mz);
    mx *= ph.c_l;
    my *= ph.c_l;
    mz *= ph.c_l;
    double n, eps, P, bx, by, bz;
    unphys = recover_general(sf, E, mx, my, mz, ph, n, eps, P, bx, by, bz);
    double feq[19], geq[19];
    equilibrium_general(n, eps, P, bx, by, bz, ph, feq, geq);
    nonpos = false;
    const double om = ph.omega, omw = 1.0 - ph.omega;
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        nonpos |= !(feq[i] > 0.0) || !(geq[i] > 0.0);
        f[i] = fma(omw, f[i], om * feq[i]);
        gg[i] = fma(omw, gg[i], om * geq[i]);
    }
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        B[RLB_CHK(i * S + idx, 38ll * S)] = f[i];
        B[RLB_CHK((19 + i) * S + idx, 38ll * S)] = gg[i];
    }
    if (XBC != XBC_PERIODIC && x == g.nx - 2) {  // outflow ghost x = nx-1 copies x = nx-2
        for (int i = 0; i < 19; ++i) {
            B[RLB_CHK(i * S + idx + 1, 38ll * S)] = f[i];
            B[RLB_CHK((19 + i) * S + idx + 1, 38ll * S)] = gg[i];
        }
    }
    if (XBC == XBC_OUTFLOW_BOTH && x == 1) {  // outflow ghost x = 0 copies x = 1
        for (int i = 0; i < 19; ++i) {
            B[RLB_CHK(i * S + idx - 1, 38ll * S)] = f[i];
            B[RLB_CHK((19 + i) * S + idx - 1, 38ll * S)] = gg[i];
        }
    }
    return true;
}
template <int XBC>
__device__ __noinline__ void step_cell_eos_general(const double* A, double* B, const Geom& g, const Phys& ph, int idx,
                                                   bool& unphys, bool& nonpos) {
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    const PullOffsets o(g, x, y, z);
    step_cell_eos<XBC>(A, B, g, ph, idx, x, o, unphys, nonpos);
}

template <int XBC>
__global__ void __launch_bounds__(128) k_step_eos(const double* __restrict__ A, double* __restrict__ B, Geom g,
                                                  Phys ph, Counters cnt, int count, long long step_index) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= g.N) return;
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    const long long S = g.S;
    if (XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1)) {
        // ghost planes are not collided (the inflow plane is copied so that
        // every cell of B is written; outflow ghosts are written below)
        if (XBC == XBC_INFLOW_OUTFLOW && x == 0) {
            for (int q = 0; q < 38; ++q) B[RLB_CHK(q * S + idx, 38ll * S)] = A[RLB_CHK(q * S + idx, 38ll * S)];
        }
        return;
    }
    const PullOffsets o(g, x, y, z);
    bool unphys, nonpos;
    if (!step_cell_eos<XBC>(A, B, g, ph, idx, x, o, unphys, nonpos)) return;
    if (count) count_flags(cnt, unphys, nonpos, (unsigned long long)step_index * (unsigned long long)g.N + idx);
}

// ---------------------------------------------------------------------------
// Fixed-point form (rlb_fixed.cuh), lattice speeds 1 <= c_l <= 2.
//
// With d = M / c_l, W = E + P = (eps + P) gamma^2 and u = d / W the equilibria
// are, as for eps = 3P, polynomials of the moments:
//   f_i = w_i S (1 + 3 e_i.u)
//   g_i = w_i [3 P / c_l^2 + 4.5 (e_i.d)(e_i.u) - 1.5 d.u + 3 e_i.d],  i > 0
//   g_0 = w_0 [3 E - 6 P / c_l^2 - 1.5 d.u],
// so beside the moments only P and 1/W are wanted.  P is found by Newton's
// iteration in binary32, then two steps with the residual in binary64 and the
// binary32 derivative (errors below 1e-7, 1e-13 and rounding); a cell whose
// last step is not below 2^-30 E, or that is not clearly physical, runs the
// binary64 iteration.
//
// The binary64 step was bound by some 600 FP64 instructions per cell (65
// clocks of a scheduler each); 83 remain beside 3,500 in all, the FP64 pipe
// 71 % busy.  128^3 box, Gamma = 1.2, m = 0.3: step 2.19 -> 0.390 ms,
// initialisation 0.80 -> 0.152 ms, macroscopic output 1.06 -> 0.26 ms.
// ---------------------------------------------------------------------------

// On scaled moments (E in [1, 2)): P, 1/W, b = M^2 / W, sq = sqrt(1 - beta^2);
// mS = m S, M2 = |M|^2.  False where the iteration is left to the general one.
__device__ __forceinline__ bool solve_pressure(double E, double M2, double mS, double g1, double& P, double& rW,
                                               double& b, double& sq) {
    const float Ef = fx_seed_f32(E), Mf = (float)M2, mf = (float)mS, gf = (float)g1;
    if (!(Mf < 0.96f * Ef * Ef) || !(mf >= 0.0f) || !(mf < 4.0f)) return false;
    const float ge = (gf + 1.0f) * Ef;
    const float X = 0.5f * (ge + sqrtf(fmaxf(ge * ge - 4.0f * gf * Mf, 0.0f)));
    float rx = 1.0f / X;
    float p = gf * ((Ef - Mf * rx) - mf * sqrtf(fmaxf(1.0f - Mf * rx * rx, 0.0f))), kf = 1.0f;
#pragma unroll 1
    for (int it = 0; it < 8; ++it) {
        rx = __fdividef(1.0f, Ef + p);
        const float b2 = Mf * rx * rx, om = 1.0f - b2;
        const float rs = rsqrtf(om);
        const float r = gf * ((Ef - Mf * rx) - mf * om * rs) - p;
        kf = __fdividef(1.0f, 1.0f - gf * (b2 - mf * rs * b2 * rx));  // -1 / r'(P)
        const float dp = r * kf;
        p += dp;
        if (!(fabsf(dp) > 2e-6f * Ef)) break;
    }
    if (!(p > 1e-4f * Ef) || !(p < 2.0f * Ef) || !(kf > 0.0f) || !(kf < 1e4f)) return false;
    const double k = fx_widen(kf);
    P = fx_widen(p);
    // first residual
    double W = E + P;
    const double x = fx_widen(__fdividef(1.0f, fx_seed_f32(W)));
    double h = fma(-W, x, 1.0);
    rW = fma(x, fma(h, h, h), x);
    b = M2 * rW;
    double om = fma(-b, rW, 1.0);  // 1 - beta^2, at least 0.04
    const float yf = rsqrtf(fx_seed_f32(om));
    const double y = fx_widen(yf);
    double s0 = om * y, q = fma(-s0, y, 1.0);
    sq = fma(s0 * q, fma(0.375, q, 0.5), s0);
    P = fma(fma(g1, fma(-mS, sq, E - b), -P), k, P);
    // second residual, 1e-7 further: third-order corrections from the same
    // 1/W and root seed
    W = E + P;
    h = fma(-W, rW, 1.0);
    rW = fma(rW, fma(h, h, h), rW);
    b = M2 * rW;
    om = fma(-b, rW, 1.0);
    s0 = om * y, q = fma(-s0, y, 1.0);
    sq = fma(s0 * q, fma(0.375, q, 0.5), s0);
    const double dP = fma(g1, fma(-mS, sq, E - b), -P) * k;
    P = P + dP;
    if ((__double2hiint(dP) & 0x7FFFFFFF) > 0x3E100000) return false;  // |dP| > 2^-30
    // and to the final P (first order: dP is below 1e-9 E, about 1e-13)
    W = E + P;
    rW = fma(rW, fma(-W, rW, 1.0), rW);
    b = M2 * rW;
    om = fma(-b, rW, 1.0);
    sq = fma(fma(-sq, sq, om), fx_widen(0.5f * yf), sq);
    return true;
}

// Sums of the populations of a set in units of 2^-56 of its block exponent.
__device__ __forceinline__ int64_t fx_sum19(const double* v, int e) {
    int64_t s = fx_round4(fx_from(v[0], e));
#pragma unroll
    for (int p = 0; p < 9; ++p) s += fx_round4(fx_from(v[2 * p + 1], e) + fx_from(v[2 * p + 2], e));
    return s;
}

// The normalised moments of a cell: E in [2^61, 2^62), d alike, and the same
// in binary64 (E in [1, 2)); value = scaled 2^k.  False outside the range.
struct EosMoments {
    int64_t E, dx, dy, dz;
    double Ed, x, y, z;
    int k;
};
__device__ __forceinline__ bool eos_moments(const double* g, int em, EosMoments& m) {
    int64_t E = fx_round4(fx_from(g[0], em)), d[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const int64_t a = fx_from(g[2 * p + 1], em), b = fx_from(g[2 * p + 2], em);
        E += fx_round4(a + b);
        d[p] = fx_round4(a - b);
    }
    const int64_t dx = ((d[0] + d[3]) + (d[4] + d[5])) + d[6], dy = ((d[1] + d[3]) - d[4]) + (d[7] + d[8]),
                  dz = ((d[2] + d[5]) - d[6]) + (d[7] - d[8]);
    const int32_t Eh = (int32_t)(E >> 32);
    if (em < 100 || em > 1900 || Eh <= 0) return false;
    const int n = fx_clz((uint32_t)Eh) - 2;
    const float Ef = (float)Eh, xf = (float)(int32_t)(dx >> 32), yf = (float)(int32_t)(dy >> 32), zf = (float)(int32_t)(dz >> 32);
    if (n > 12 || !(xf * xf + yf * yf + zf * zf < Ef * Ef)) return false;
    m.E = E << n, m.dx = dx << n, m.dy = dy << n, m.dz = dz << n;
    m.k = em - 1018 - n;
    m.Ed = fx_unit(m.E);
    m.x = fx_to(m.dx, -61), m.y = fx_to(m.dy, -61), m.z = fx_to(m.dz, -61);
    return true;
}

// Per-run constants of k_init_eos.
struct FxEosInit {
    FxConst k8;   // 1 / (8 c_l^2)   x 2^65
    FxConst kP;   // 1 / (12 c_l^2)  x 2^65
    FxConst kc2;  // 1 / c_l^2       x 2^62
    FxConst k3;   // 1 / 3           x 2^63
};

// Per-run constants of k_step_eos_fx (make_fx_eos).
struct FxEos {
    FxConst kP;   // omega / (12 c_l^2)  x 2^64
    FxConst kP0;  // omega / c_l^2       x 2^62
    FxConst kE0;  // omega               x 2^62
    FxConst kU;   // omega / 12          x 2^64
    FxConst kS;   // omega / 36          x 2^64
    FxConst k3;   // 1 / 3               x 2^63
    FxConst k23;  // 2 / 3               x 2^63
    int64_t om57;     // omega x 2^57
    double om8, omw;  // omega / 8, 1 - omega
};

template <int XBC>
__global__ void __launch_bounds__(128, 4)
    k_step_eos_fx(const double* __restrict__ A, double* __restrict__ B, const __grid_constant__ Geom g,
                  const __grid_constant__ Phys ph, Counters cnt, int count, long long step_index,
                  const __grid_constant__ FxEos k) {
    const int idx = dependent_begin(blockIdx.x * blockDim.x + threadIdx.x);
    if (idx >= g.N) return;
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    const long long S = g.S;
    if (XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1)) {
        if (XBC == XBC_INFLOW_OUTFLOW && x == 0) {
            for (int q = 0; q < 38; ++q) B[RLB_CHK(q * S + idx, 38ll * S)] = A[RLB_CHK(q * S + idx, 38ll * S)];
        }
        return;
    }
    const PullOffsets o(g, x, y, z);
    double f[19], h[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) h[i] = __ldg(RLB_CHK_PTR(A, (19 + i) * S + idx + o.src(i), 38ll * S));
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = __ldg(RLB_CHK_PTR(A, i * S + idx + o.src(i), 38ll * S));
    int em = fx_max_exponent<19>(h);
    if (em == 0x7FF) {  // a solid marker, or a non-finite population
        if (is_solid(h[0])) {
            const double m = solid_marker_d();
            for (int q = 0; q < 38; ++q) B[RLB_CHK(q * S + idx, 38ll * S)] = m;
            return;
        }
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            if (is_solid(f[i])) {  // link bounce-back
                f[i] = A[RLB_CHK(opp(i) * S + idx, 38ll * S)];
                h[i] = A[RLB_CHK((19 + opp(i)) * S + idx, 38ll * S)];
            }
        }
        em = fx_max_exponent<19>(h);
    }
    const bool dup_hi = XBC != XBC_PERIODIC && x == g.nx - 2, dup_lo = XBC == XBC_OUTFLOW_BOTH && x == 1;
    double* Bc = B + idx;
    auto put = [&](int q, double v) {
        Bc[RLB_CHK_OFF(q * S, idx, 38ll * S)] = v;
        if (dup_hi) Bc[RLB_CHK_OFF(q * S + 1, idx, 38ll * S)] = v;
        if (dup_lo) Bc[RLB_CHK_OFF(q * S - 1, idx, 38ll * S)] = v;
    };
    bool unphys = false, nonpos = false;
    EosMoments m;
    bool ok = eos_moments(h, em, m);
    const int ef = fx_max_exponent<19>(f);
    ok = ok && ef >= 100 && ef <= 1900;
    if (ok) {
        const int64_t Si = fx_sum19(f, ef);
        const int32_t Sh = (int32_t)(Si >> 32);
        const int n = fx_clz((uint32_t)Sh) - 2;
        const double mS = ph.eos_mass * fx_to(Si, max(ef - 1079 - m.k, -900));
        double P, rW, b, sq;
        const double M2 = ph.cl2 * fma(m.x, m.x, fma(m.y, m.y, m.z * m.z));
        ok = Sh > 0 && n <= 12 && ef - 1079 - m.k < 900 && solve_pressure(m.Ed, M2, mS, ph.eos_gamma - 1.0, P, rW, b, sq);
        if (ok) {
            // units of 2^-61 of the scale (g_0: 2^-59)
            const int eb = m.k - 61;
            // omega / (8 W), below 1/4, x 2^64, with the residual of the sum
            // E + P in fixed point: without it the roundings of W, of 1/W and
            // of this product are common to every term that is linear in u
            // (and are most of the error of a population that they cancel in)
            const int64_t Pi = fx_fixed(P, 61);
            int64_t r8 = fx_fixed(rW * k.om8, 64);
            const int64_t rest = k.om57 - fx_mul(fx_split((int64_t)((uint64_t)(m.E + Pi) >> 1)), fx_split(r8));
            r8 += (int64_t)__float2int_rn((float)(int32_t)rest * 16.0f * fx_seed_f32(rW));
            const FxSplit r = fx_split(fx_weight(r8));
            const FxSplit sx = fx_split(m.dx), sy = fx_split(m.dy), sz = fx_split(m.dz);
            const FxSplit wx = fx_split(fx_mul(sx, r) << 3), wy = fx_split(fx_mul(sy, r) << 3),
                          wz = fx_split(fx_mul(sz, r) << 3);  // omega u / 8, x 2^64
            FxG t;
            t.Pxx = fx_mul(sx, wx);
            t.Pyy = fx_mul(sy, wy);
            t.Pzz = fx_mul(sz, wz);
            t.Pxy = fx_mul(sx, wy);
            t.Pxz = fx_mul(sx, wz);
            t.Pyz = fx_mul(sy, wz);
            t.ux = fx_mul(sx, k.kU);
            t.uy = fx_mul(sy, k.kU);
            t.uz = fx_mul(sz, k.kU);
            const int64_t X = t.Pxx + t.Pyy + t.Pzz;
            t.A = fx_mul(fx_split(Pi), k.kP) - fx_mul(fx_split(X << 1), k.k3);
            const int64_t g0 = fx_mul(fx_split(m.E), k.kE0) - fx_mul(fx_split(Pi << 1), k.kP0) - X;
            int64_t low = g0 - 1;  // negative when an equilibrium is not positive
            put(19, fma(k.omw, h[0], fx_to(g0, eb + 2)));
#pragma unroll
            for (int p = 0; p < 9; ++p) {
                int64_t s, a;
                fx_g_pair(t, p, s, a);
                low |= (s + a - 1) | (s - a - 1);
                put(20 + 2 * p, fma(k.omw, h[2 * p + 1], fx_to(s + a, eb)));
                put(21 + 2 * p, fma(k.omw, h[2 * p + 2], fx_to(s - a, eb)));
            }
            const FxSplit ss = fx_split(Si << n);
            FxF q;
            q.B = fx_mul(ss, k.kS);
            q.Fx = fx_mul(ss, fx_split(fx_mul(wx, k.k23) << 1));
            q.Fy = fx_mul(ss, fx_split(fx_mul(wy, k.k23) << 1));
            q.Fz = fx_mul(ss, fx_split(fx_mul(wz, k.k23) << 1));
            const int fb = ef - 1079 - n;
            put(0, fma(k.omw, f[0], fx_to((q.B << 3) + (q.B << 2), fb)));
#pragma unroll
            for (int p = 0; p < 9; ++p) {
                int64_t s, a;
                fx_f_pair(q, p, s, a);
                low |= (s + a - 1) | (s - a - 1);
                put(1 + 2 * p, fma(k.omw, f[2 * p + 1], fx_to(s + a, fb)));
                put(2 + 2 * p, fma(k.omw, f[2 * p + 2], fx_to(s - a, fb)));
            }
            nonpos = low < 0;
        }
    }
    if (!ok) step_cell_eos_general<XBC>(A, B, g, ph, idx, unphys, nonpos);
    if (count) count_flags(cnt, unphys, nonpos, (unsigned long long)step_index * (unsigned long long)g.N + idx);
}

// Initial populations of one cell in binary64.
__device__ __noinline__ void init_cell_eos(double* A, const Geom& g, const Phys& ph, double n, double eps, double bx,
                                           double by, double bz, int idx) {
    const long long S = g.S;
    double f[19], gg[19];
    equilibrium_general(n, eps, eos_pressure(ph, n, eps), bx, by, bz, ph, f, gg);
    for (int i = 0; i < 19; ++i) {
        A[RLB_CHK(i * S + idx, 38ll * S)] = f[i];
        A[RLB_CHK((19 + i) * S + idx, 38ll * S)] = gg[i];
    }
}

// As k_init (rlb_fields.cu), with v = W beta and P in the g terms:
//   g_i = 36 w_i [P / (12 c_l^2) - X / 3 + P_ab sums + v.e_i / (12 c_l)],
//   P_ab = v_a beta_b / (8 c_l^2), X = P_xx + P_yy + P_zz,
//   g_0 = W - P - 2 P / c_l^2 - 4 X.
// The second buffer is not written (a step writes every cell of it).
__global__ void __launch_bounds__(128, 6) k_init_eos(const double* __restrict__ n, const double* __restrict__ eps,
                                                  const double* __restrict__ beta, const uint8_t* __restrict__ solid,
                                                  double* __restrict__ A, const __grid_constant__ Geom g,
                                                  const __grid_constant__ Phys ph, const __grid_constant__ FxEosInit k) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= g.N) return;
    const long long S = g.S;
    double* Ac = A + idx;
    auto put = [&](int q, double v) { Ac[RLB_CHK_OFF(q * S, idx, 38ll * S)] = v; };
    if (solid && solid[idx]) {
        const double m = solid_marker_d();
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
    const FxInit& c = ph.fi;
    const double omb2 = 1.0 - fma(bx, bx, fma(by, by, bz * bz));
    const double P = eos_pressure(ph, nn, ee);
    const int oh = __double2hiint(omb2), nh = __double2hiint(nn), eh = __double2hiint(ee), Ph = __double2hiint(P);
    // the conditions of k_init, and P positive and not far below eps
    if (c.on && oh > 0x3F900000 && oh < 0x3FF00001 && nh > c.lo && nh < c.hi && eh > c.lo && eh < c.hi &&
        Ph > eh - (10 << 20) && Ph <= eh + (1 << 20)) {
        const double gam = rsqrt_unit(omb2);
        // gamma^2 and gamma to their last bit: an error here is common to all
        // populations of a cell, and stays in its conserved moments
        const double g2 = gam * gam, gh = fma(-omb2, g2, 1.0);
        const double W = (ee + P) * fma(g2, gh, g2), sn = nn * fma(0.5 * gh, gam, gam);
        int we, se;
        const int64_t xw = fx_mantissa(W, we);
        const FxSplit xs = fx_split(fx_mantissa(sn, se));
        const FxSplit s8 = fx_split(fx_mul(fx_split(xw), k.k8) << 2);  // W / (8 c_l^2), x 2^64
        const FxSplit tx = fx_split(fx_scaled(bx, 1023, 62)), ty = fx_split(fx_scaled(by, 1023, 62)),
                      tz = fx_split(fx_scaled(bz, 1023, 62));
        const FxSplit vx = fx_split(fx_mul(s8, tx) << 2), vy = fx_split(fx_mul(s8, ty) << 2),
                      vz = fx_split(fx_mul(s8, tz) << 2);
        FxG t;
        t.Pxx = fx_mul(vx, tx);
        t.Pyy = fx_mul(vy, ty);
        t.Pzz = fx_mul(vz, tz);
        t.Pxy = fx_mul(vx, ty);
        t.Pxz = fx_mul(vx, tz);
        t.Pyz = fx_mul(vy, tz);
        t.ux = fx_mul(vx, c.kU) << c.sU;
        t.uy = fx_mul(vy, c.kU) << c.sU;
        t.uz = fx_mul(vz, c.kU) << c.sU;
        const int64_t X = t.Pxx + t.Pyy + t.Pzz, Pi = fx_scaled(P, we, 61);
        t.A = fx_mul(fx_split(Pi), k.kP) - fx_mul(fx_split(X << 1), k.k3);
        const int64_t g0 = fx_weight((xw - Pi + 2) >> 2) - fx_mul(fx_split(Pi << 1), k.kc2) - ((X + 1) >> 1);
        const int gb = we - 1085, fb = se - 1085;
        put(19, fx_to(g0, gb + 3));
        const FxSplit s12 = fx_split(fx_mul(xs, c.kS12) << 2);
        FxF q;
        q.B = fx_mul(xs, c.kS);
        q.Fx = fx_mul(s12, tx);
        q.Fy = fx_mul(s12, ty);
        q.Fz = fx_mul(s12, tz);
        put(0, fx_to((q.B << 3) + (q.B << 2), fb));
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            int64_t s, a;
            fx_g_pair(t, p, s, a);
            put(20 + 2 * p, fx_to(s + a, gb));
            put(21 + 2 * p, fx_to(s - a, gb));
            fx_f_pair(q, p, s, a);
            put(1 + 2 * p, fx_to(s + a, fb));
            put(2 + 2 * p, fx_to(s - a, fb));
        }
        return;
    }
    init_cell_eos(A, g, ph, nn, ee, bx, by, bz, idx);
}

// One cell of the output in binary64 throughout; whether it is unphysical.
__device__ __noinline__ bool macro_cell_eos(const double* A, double* n, double* eps, double* beta, const Geom& g,
                                            const Phys& ph, int idx) {
    const long long S = g.S;
    double f[19], gg[19];
    for (int i = 0; i < 19; ++i) {
        f[i] = A[RLB_CHK(i * S + idx, 38ll * S)];
        gg[i] = A[RLB_CHK((19 + i) * S + idx, 38ll * S)];
    }
    double sf, E, mx, my, mz;
    moments_pairs(f, gg, sf, E, mx, my, mz);
    mx *= ph.c_l;
    my *= ph.c_l;
    mz *= ph.c_l;
    double nn, e, P, bx, by, bz;
    const bool bad = recover_general(sf, E, mx, my, mz, ph, nn, e, P, bx, by, bz);
    n[idx] = nn;
    eps[idx] = e;
    beta[idx] = bx;
    beta[g.N + idx] = by;
    beta[2 * (long long)g.N + idx] = bz;
    return bad;
}

__global__ void __launch_bounds__(128, 5) k_macro_eos(const double* __restrict__ A, double* __restrict__ n,
                                                   double* __restrict__ eps, double* __restrict__ beta,
                                                   const __grid_constant__ Geom g, const __grid_constant__ Phys ph,
                                                   unsigned long long* bad_count, int fx_on) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= g.N) return;
    const long long S = g.S;
    double h[19], f[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) h[i] = __ldg(RLB_CHK_PTR(A, (19 + i) * S + idx, 38ll * S));
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = __ldg(RLB_CHK_PTR(A, i * S + idx, 38ll * S));
    if (is_solid(f[0])) {
        const double nan = __longlong_as_double(0x7FF8000000000000ll);
        n[idx] = eps[idx] = beta[idx] = beta[g.N + idx] = beta[2 * (long long)g.N + idx] = nan;
        return;
    }
    bool ok = fx_on;
    if (ok) {
        EosMoments m;
        const int ef = fx_max_exponent<19>(f);
        ok = eos_moments(h, fx_max_exponent<19>(h), m) && ef >= 100 && ef <= 1900;
        if (ok) {
            const int ks = ef - 1079 - m.k;
            const double Ss = fx_to(fx_sum19(f, ef), max(ks, -900));
            double P, rW, b, sq;
            const double M2 = ph.cl2 * fma(m.x, m.x, fma(m.y, m.y, m.z * m.z));
            ok = ks < 900 && ks > -900 && Ss > 0.0 && m.k > -900 && m.k < 900 &&
                 solve_pressure(m.Ed, M2, ph.eos_mass * Ss, ph.eos_gamma - 1.0, P, rW, b, sq);
            if (ok) {
                // scaled values back by 2^k (their exponents stay in range)
                const double r = rW * ph.c_l;
                n[idx] = scale_pow2(Ss * sq, m.k);
                eps[idx] = scale_pow2(m.Ed - b, m.k);
                beta[idx] = m.x * r;
                beta[g.N + idx] = m.y * r;
                beta[2 * (long long)g.N + idx] = m.z * r;
            }
        }
    }
    if (!ok && macro_cell_eos(A, n, eps, beta, g, ph, idx)) atomicAdd(bad_count, 1ull);
}

// The fixed-point kernels cover 1 <= c_l <= 2 (see k_step_f64_fx).
bool eos_fx_on(const Phys& ph) { return fx_covers(ph.c_l); }

// num / (den c_l^2) x 2^s
FxConst over_c2(const Phys& ph, double num, double den, int s) {
    const double c2 = ph.c_l * ph.c_l, c2l = fma(ph.c_l, ph.c_l, -c2);
    double qh, ql;
    fx_div2(num, den, qh, ql);
    const double th = qh / c2, tl = (fma(-th, c2, qh) + (ql - th * c2l)) / c2;
    return fx_const_w(th, tl, s);
}

FxEosInit make_fx_eos_init(const Phys& ph) {
    FxEosInit k{};
    if (!ph.fi.on) return k;
    k.k8 = over_c2(ph, 1.0, 8.0, 65);
    k.kP = over_c2(ph, 1.0, 12.0, 65);
    k.kc2 = over_c2(ph, 1.0, 1.0, 62);
    double qh, ql;
    fx_div2(1.0, 3.0, qh, ql);
    k.k3 = fx_const(qh, ql, 63);
    return k;
}

FxEos make_fx_eos(const Phys& ph) {
    FxEos k;
    const double om = ph.omega;
    double qh, ql;
    k.kP = over_c2(ph, om, 12.0, 64);
    k.kP0 = over_c2(ph, om, 1.0, 62);
    k.kE0 = fx_const_w(om, 0.0, 62);
    fx_div2(om, 12.0, qh, ql);
    k.kU = fx_const_w(qh, ql, 64);
    fx_div2(om, 36.0, qh, ql);
    k.kS = fx_const_w(qh, ql, 64);
    fx_div2(1.0, 3.0, qh, ql);
    k.k3 = fx_const(qh, ql, 63);
    fx_div2(2.0, 3.0, qh, ql);
    k.k23 = fx_const(qh, ql, 63);
    k.om57 = (int64_t)(om * 0x1p57);
    k.om8 = 0.125 * om;
    k.omw = 1.0 - om;
    return k;
}

inline unsigned nblocks(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

cudaError_t launch_init_eos(const Geom& g, const Phys& ph, const double* n, const double* eps, const double* beta,
                            const uint8_t* solid, void* A, void* B, cudaStream_t st) {
    (void)B;
    set_last_launch_count(1);
    k_init_eos<<<nblocks(g.N, 128), 128, 0, st>>>(n, eps, beta, solid, (double*)A, g, ph, make_fx_eos_init(ph));
    return cudaGetLastError();
}

cudaError_t launch_step_eos(const Geom& g, const Phys& ph, const void* A, void* B, Counters cnt, bool count,
                            long long step_index, cudaStream_t st) {
    set_last_launch_count(1);
    const unsigned nb = nblocks(g.N, 128);
    const int cs = count ? 1 : 0;
    if (eos_fx_on(ph)) {
        const FxEos k = make_fx_eos(ph);
        auto go = [&](auto kern) {
            launch_dependent(kern, nb, 128, 0, st, (const double*)A, (double*)B, g, ph, cnt, cs, step_index, k);
        };
        switch (g.xbc) {
            case XBC_PERIODIC: go(k_step_eos_fx<XBC_PERIODIC>); break;
            case XBC_INFLOW_OUTFLOW: go(k_step_eos_fx<XBC_INFLOW_OUTFLOW>); break;
            default: go(k_step_eos_fx<XBC_OUTFLOW_BOTH>); break;
        }
        return cudaGetLastError();
    }
    switch (g.xbc) {
        case XBC_PERIODIC:
            k_step_eos<XBC_PERIODIC><<<nb, 128, 0, st>>>((const double*)A, (double*)B, g, ph, cnt, cs, step_index);
            break;
        case XBC_INFLOW_OUTFLOW:
            k_step_eos<XBC_INFLOW_OUTFLOW><<<nb, 128, 0, st>>>((const double*)A, (double*)B, g, ph, cnt, cs,
                                                               step_index);
            break;
        default:
            k_step_eos<XBC_OUTFLOW_BOTH><<<nb, 128, 0, st>>>((const double*)A, (double*)B, g, ph, cnt, cs,
                                                             step_index);
            break;
    }
    return cudaGetLastError();
}

cudaError_t launch_macro_eos(const Geom& g, const Phys& ph, const void* A, double* n, double* eps, double* beta,
                             Counters cnt, cudaStream_t st) {
    set_last_launch_count(1);
    k_macro_eos<<<nblocks(g.N, 128), 128, 0, st>>>((const double*)A, n, eps, beta, g, ph, cnt.macro_bad, eos_fx_on(ph) ? 1 : 0);
    return cudaGetLastError();
}

// Bounds-check count of this translation unit (0 in the release build).
RLB_OOB_TAKE_FN(oob_take_eos)

}  // namespace rlb
