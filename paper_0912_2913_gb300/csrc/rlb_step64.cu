// rlb_step64.cu -- the FP64 fused stream-and-collide step (Eqs. lbe1, lbe2
// with the eps = 3P equilibria Eqs. equil1s, equil2as, equil2bs).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "rlb_device.cuh"
#include "rlb_fixed.cuh"

namespace rlb {

// ---------------------------------------------------------------------------
// FP64 step.
// ---------------------------------------------------------------------------

// Moments S_f, E and d = M / c_l of the FP64 step, summed as a fixed tree
// over eight partials: partial j holds pair j, and for j < 2 also unit
// j + 8 (pair 8 for j = 0, the rest population for j = 1).  They are combined
// as ((P0 + P4) + (P2 + P6)) + ((P1 + P5) + (P3 + P7)), the order in which an
// xor butterfly over eight lanes (offsets 4, 2, 1) adds them on every lane,
// so k_step_f64_split, which spreads the units of a cell over eight lanes,
// forms the same sums; the partials of d that are identically zero are left
// out here (adding an exact zero leaves any value but -0 unchanged).
__device__ __forceinline__ void moments_tree8(const double* f, const double* g, double& sf, double& e, double& dx,
                                              double& dy, double& dz) {
    double sp[9], ep[9], d[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        sp[p] = f[2 * p + 1] + f[2 * p + 2];
        ep[p] = g[2 * p + 1] + g[2 * p + 2];
        d[p] = g[2 * p + 1] - g[2 * p + 2];
    }
    const double s0 = sp[0] + sp[8], s1 = sp[1] + f[0];
    const double e0 = ep[0] + ep[8], e1 = ep[1] + g[0];
    sf = ((s0 + sp[4]) + (sp[2] + sp[6])) + ((s1 + sp[5]) + (sp[3] + sp[7]));
    e = ((e0 + ep[4]) + (ep[2] + ep[6])) + ((e1 + ep[5]) + (ep[3] + ep[7]));
    // x: pairs 0, 3, 4, 5, 6; y: 1, 3, -4, 7, 8; z: 2, 5, -6, 7, -8
    dx = ((d[0] + d[4]) + d[6]) + (d[5] + d[3]);
    dy = (d[8] - d[4]) + (d[1] + (d[3] + d[7]));
    dz = (-d[8] + (d[2] - d[6])) + (d[5] + d[7]);
}

// One collided cell in binary64 throughout: any lattice speed, any state.
// Runs every cell of k_step_f64 and, in the fixed-point kernels, the cells
// whose state they do not cover (unphysical or near |M| = E, non-finite).
// Returns false for a solid cell (marker kept, nothing counted).
template <int XBC, bool SOLID>
__device__ __forceinline__ bool step_cell_f64(const double* __restrict__ A, double* __restrict__ B, const Geom& g,
                                              const Phys& ph, int idx, int x, const PullOffsets& o, bool& unphys,
                                              bool& nonpos) {
    const long long S = g.S;
    double f[19], gg[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const int s = idx + o.src(i);
        f[i] = __ldg(RLB_CHK_PTR(A, i * S + s, 38ll * S));
        gg[i] = __ldg(RLB_CHK_PTR(A, (19 + i) * S + s, 38ll * S));
    }
    if (SOLID) {
        if (is_solid(f[0])) {  // the cell itself is solid: keep the marker
            const double m = solid_marker_d();
#pragma unroll
            for (int q = 0; q < 38; ++q) B[RLB_CHK(q * S + idx, 38ll * S)] = m;
            return false;
        }
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            if (is_solid(f[i])) {  // link bounce-back
                f[i] = __ldg(RLB_CHK_PTR(A, opp(i) * S + idx, 38ll * S));
                gg[i] = __ldg(RLB_CHK_PTR(A, (19 + opp(i)) * S + idx, 38ll * S));
            }
        }
    }
    // d = M / c_l (the pair differences summed along each axis)
    double sf, E, dx, dy, dz;
    moments_tree8(f, gg, sf, E, dx, dy, dz);
    // Recovery with eps = 3P: eps = -E + sqrt(4E^2 - 3M^2), beta = 3M/(3E + eps).
    // Square root and reciprocals from binary32 seeds (converted on the integer
    // pipe, valid for any exponent of the argument) with two FP64 Newton
    // corrections each: full double accuracy at a fraction of the IEEE
    // sequences' cost on this GPU's FP64 pipe.
    const double m2 = fma(dx, dx, fma(dy, dy, dz * dz));  // |M|^2 / c_l^2
    const double disc = fma(4.0 * E, E, ph.m3cl2 * m2);   // 4E^2 - 3|M|^2
    double ys, hs;
    rsqrt_seed(disc, ys, hs);
    double sq = disc * ys;
    sq = fma(fma(-sq, sq, disc), hs, sq);
    sq = fma(fma(-sq, sq, disc), hs, sq);
    const double eps = sq - E;
    const double D = fma(3.0, E, eps);
    double rD = rcp_seed(D);
    rD = fma(rD, fma(-D, rD, 1.0), rD);
    rD = fma(rD, fma(-D, rD, 1.0), rD);
    const double r3 = ph.three_cl * rD;  // beta = 3 M / D = 3 c_l d / D
    const double bx = dx * r3, by = dy * r3, bz = dz * r3;
    const double b2 = fma(bx, bx, fma(by, by, bz * bz));
    const double omb2 = 1.0 - b2;
    double gam2 = rcp_seed(omb2);
    gam2 = fma(gam2, fma(-omb2, gam2, 1.0), gam2);
    gam2 = fma(gam2, fma(-omb2, gam2, 1.0), gam2);
    unphys = !(pos_finite(sf) && pos_finite(E) && nonneg_finite(disc) && pos_finite(eps) && below_one(b2));
    // beta rounded to binary32 on the integer pipe (the same rounding as a conversion)
    nonpos = nonpositive_eq(d2f(bx), d2f(by), d2f(bz), (float)ph.c_l);

    // The relaxed values omega eq + (1 - omega) h, with omega and the weights
    // folded into per-run constants (Phys::c_*):
    //   f^eq_i = w_i S_f (1 + 3 q_i / c_l)     (Eq. equil1s with n gamma = S_f)
    //   g^eq_i = w_i [eps/c_l^2 + eps gamma^2 (6 q^2/c_l^2 - 2 b2/c_l^2)] +- w_i eps gamma^2 4 q / c_l
    //   g_0^eq = w_0 [4 eps gamma^2 - eps (2 + c_l^2)/c_l^2 - 2 eps gamma^2 b2/c_l^2]   (Eq. equil2bs)
    const double omw = 1.0 - ph.omega;
    const double q[9] = {bx, by, bz, bx + by, bx - by, bx + bz, bx - bz, by + bz, by - bz};
    const double eg = eps * gam2;
    const double egb2 = eg * b2;
    const double t = fma(-2.0, egb2, eps);  // eps - 2 eg b2
    const double k1w[2] = {t * ph.c_k1[0], t * ph.c_k1[1]};
    const double k2w[2] = {eg * ph.c_k2[0], eg * ph.c_k2[1]};
    const double k3w[2] = {eg * ph.c_k3[0], eg * ph.c_k3[1]};
    const double fsw[2] = {sf * ph.c_fs[0], sf * ph.c_fs[1]};
    const double faw[2] = {sf * ph.c_fa[0], sf * ph.c_fa[1]};
    double outf[19], outg[19];
    outf[0] = fma(omw, f[0], sf * ph.c_f0);
    outg[0] = fma(omw, gg[0], fma(eg, ph.c_g0[0], fma(eps, ph.c_g0[1], egb2 * ph.c_g0[2])));
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const int cl = p < 3 ? 0 : 1;
        outf[2 * p + 1] = fma(omw, f[2 * p + 1], fma(faw[cl], q[p], fsw[cl]));
        outf[2 * p + 2] = fma(omw, f[2 * p + 2], fma(-faw[cl], q[p], fsw[cl]));
        const double gsym = fma(k2w[cl], q[p] * q[p], k1w[cl]);
        outg[2 * p + 1] = fma(omw, gg[2 * p + 1], fma(k3w[cl], q[p], gsym));
        outg[2 * p + 2] = fma(omw, gg[2 * p + 2], fma(-k3w[cl], q[p], gsym));
    }
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        B[RLB_CHK(i * S + idx, 38ll * S)] = outf[i];
        B[RLB_CHK((19 + i) * S + idx, 38ll * S)] = outg[i];
    }
    if (XBC != XBC_PERIODIC && x == g.nx - 2) {  // outflow ghost x = nx-1 copies x = nx-2
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            B[RLB_CHK(i * S + idx + 1, 38ll * S)] = outf[i];
            B[RLB_CHK((19 + i) * S + idx + 1, 38ll * S)] = outg[i];
        }
    }
    if (XBC == XBC_OUTFLOW_BOTH && x == 1) {  // outflow ghost x = 0 copies x = 1
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            B[RLB_CHK(i * S + idx - 1, 38ll * S)] = outf[i];
            B[RLB_CHK((19 + i) * S + idx - 1, 38ll * S)] = outg[i];
        }
    }
    return true;
}

template <int XBC, bool SOLID>
__global__ void __launch_bounds__(128) k_step_f64(const double* __restrict__ A, double* __restrict__ B, Geom g,
                                                  Phys ph, Counters cnt, int count, long long step_index) {
    const int idx = dependent_begin(blockIdx.x * blockDim.x + threadIdx.x);
    if (idx >= g.N) return;
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    if (g.zhalo && (z == 0 || z == g.nz - 1)) return;  // z halo planes: filled by the exchange
    const long long S = g.S;
    if (XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1)) {
        // Ghost planes are not collided.  The inflow plane keeps its fixed
        // equilibrium (copied so that every cell of B is written); outflow
        // ghosts are written by the cell they copy.
        if (XBC == XBC_INFLOW_OUTFLOW && x == 0) {
#pragma unroll
            for (int q = 0; q < 38; ++q) B[RLB_CHK(q * S + idx, 38ll * S)] = __ldg(RLB_CHK_PTR(A, q * S + idx, 38ll * S));
        }
        return;
    }
    const PullOffsets o(g, x, y, z);
    bool unphys, nonpos;
    if (!step_cell_f64<XBC, SOLID>(A, B, g, ph, idx, x, o, unphys, nonpos)) return;
    if (count) count_flags(cnt, unphys, nonpos, (unsigned long long)step_index * (unsigned long long)g.N + idx);
}

// ---------------------------------------------------------------------------
// FP64 step for small lattices (the 1600-cell shock tube): eight lanes per
// cell.  The FP64 pipe issues one warp instruction about every 76 cycles per
// scheduler on this GPU (1.68 FMA per SM per clock), whatever the number of
// active lanes, so a cell's ~200 FP64 instructions on one thread take some
// 15,000 cycles however few cells share a scheduler.  Here lane j of a cell's
// group pulls and relaxes pair j (and pair 8 for j = 0, the rest population
// for j = 1); the moments are the lanes' partials summed by an xor butterfly
// (the tree of moments_tree8), the recovery is repeated on every lane, and a
// warp issues about half the FP64 instructions.  The arithmetic is that of
// k_step_f64 term for term, so the two give the same values.
// ---------------------------------------------------------------------------
template <int XBC, bool SOLID>
__global__ void __launch_bounds__(128) k_step_f64_split(const double* __restrict__ A, double* __restrict__ B, Geom g,
                                                        Phys ph, Counters cnt, int count, long long step_index) {
    const unsigned full = 0xffffffffu;
    const int t = dependent_begin(blockIdx.x * blockDim.x + threadIdx.x);  // 8 N < 2^31 (small lattices; tests)
    const int j = threadIdx.x & 7;  // lane of the cell's group
    const int cell = (int)((unsigned)t >> 3);
    const bool live = cell < g.N;
    const int idx = live ? cell : 0;
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    const bool halo = g.zhalo && (z == 0 || z == g.nz - 1);  // filled by the exchange
    const bool ghost = XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1);
    const bool work = live && !halo && !ghost;  // a collided cell
    const long long S = g.S;
    const PullOffsets o(g, x, y, z);
    // this lane's populations: pair j (a: +, b: -); lane 0 also pair 8
    // (c: +, d: -), lane 1 the rest population (c)
    const int ia = 2 * j + 1, ib = 2 * j + 2;
    auto pull = [&](int i, double& fv, double& gv) {
        const int src = idx + o.src(i);
        fv = __ldg(RLB_CHK_PTR(A, i * S + src, 38ll * S));
        gv = __ldg(RLB_CHK_PTR(A, (19 + i) * S + src, 38ll * S));
        if (SOLID && is_solid(fv)) {  // link bounce-back
            fv = __ldg(RLB_CHK_PTR(A, opp(i) * S + idx, 38ll * S));
            gv = __ldg(RLB_CHK_PTR(A, (19 + opp(i)) * S + idx, 38ll * S));
        }
    };
    double fa = 0.0, fb = 0.0, ga = 0.0, gb = 0.0, fc = 0.0, fd = 0.0, gc = 0.0, gd = 0.0;
    bool own_solid = false;
    if (work) {
        pull(ia, fa, ga);
        pull(ib, fb, gb);
        if (j == 0) {
            pull(17, fc, gc);
            pull(18, fd, gd);
        } else if (j == 1) {
            fc = __ldg(RLB_CHK_PTR(A, idx, 38ll * S));
            gc = __ldg(RLB_CHK_PTR(A, 19 * S + idx, 38ll * S));
            own_solid = SOLID && is_solid(fc);
        }
    }
    const bool solid = __shfl_sync(full, own_solid, (threadIdx.x & 24) + 1);  // lane 1 holds f_0
    // partials of the moments (the tree of moments_tree8)
    double ps = fa + fb, pe = ga + gb;
    const double dj = ga - gb;
    if (j == 0) {
        ps = ps + (fc + fd);
        pe = pe + (gc + gd);
    } else if (j == 1) {
        ps = ps + fc;
        pe = pe + gc;
    }
    const double d8 = gc - gd;  // pair 8 on lane 0
    const int ex = pair_ex(j), ey = pair_ey(j), ez = pair_ez(j);
    double px = ex ? dj : 0.0;
    double py = j == 0 ? d8 : (ey > 0 ? dj : (ey < 0 ? -dj : 0.0));
    double pz = j == 0 ? -d8 : (ez > 0 ? dj : (ez < 0 ? -dj : 0.0));
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        ps += __shfl_xor_sync(full, ps, off);
        pe += __shfl_xor_sync(full, pe, off);
        px += __shfl_xor_sync(full, px, off);
        py += __shfl_xor_sync(full, py, off);
        pz += __shfl_xor_sync(full, pz, off);
    }
    const double sf = ps, E = pe, dx = px, dy = py, dz = pz;
    // recovery: as in k_step_f64
    const double m2 = fma(dx, dx, fma(dy, dy, dz * dz));
    const double disc = fma(4.0 * E, E, ph.m3cl2 * m2);
    double ys, hs;
    rsqrt_seed(disc, ys, hs);
    double sq = disc * ys;
    sq = fma(fma(-sq, sq, disc), hs, sq);
    sq = fma(fma(-sq, sq, disc), hs, sq);
    const double eps = sq - E;
    const double D = fma(3.0, E, eps);
    double rD = rcp_seed(D);
    rD = fma(rD, fma(-D, rD, 1.0), rD);
    rD = fma(rD, fma(-D, rD, 1.0), rD);
    const double r3 = ph.three_cl * rD;
    const double bx = dx * r3, by = dy * r3, bz = dz * r3;
    const double b2 = fma(bx, bx, fma(by, by, bz * bz));
    const double omb2 = 1.0 - b2;
    double gam2 = rcp_seed(omb2);
    gam2 = fma(gam2, fma(-omb2, gam2, 1.0), gam2);
    gam2 = fma(gam2, fma(-omb2, gam2, 1.0), gam2);
    const bool unphys = !(pos_finite(sf) && pos_finite(E) && nonneg_finite(disc) && pos_finite(eps) && below_one(b2));
    const bool nonpos = nonpositive_eq(d2f(bx), d2f(by), d2f(bz), (float)ph.c_l);
    // equilibria and relaxation of this lane's populations: as in k_step_f64
    const double omw = 1.0 - ph.omega;
    const double q[9] = {bx, by, bz, bx + by, bx - by, bx + bz, bx - bz, by + bz, by - bz};
    const double eg = eps * gam2;
    const double egb2 = eg * b2;
    const double tt = fma(-2.0, egb2, eps);
    const double k1w[2] = {tt * ph.c_k1[0], tt * ph.c_k1[1]};
    const double k2w[2] = {eg * ph.c_k2[0], eg * ph.c_k2[1]};
    const double k3w[2] = {eg * ph.c_k3[0], eg * ph.c_k3[1]};
    const double fsw[2] = {sf * ph.c_fs[0], sf * ph.c_fs[1]};
    const double faw[2] = {sf * ph.c_fa[0], sf * ph.c_fa[1]};
    double qj = q[0];
#pragma unroll
    for (int p = 1; p < 8; ++p) qj = j == p ? q[p] : qj;
    const int cl = j < 3 ? 0 : 1;
    const double fsc = cl ? fsw[1] : fsw[0], fac = cl ? faw[1] : faw[0];
    const double k1c = cl ? k1w[1] : k1w[0], k2c = cl ? k2w[1] : k2w[0], k3c = cl ? k3w[1] : k3w[0];
    const double ofa = fma(omw, fa, fma(fac, qj, fsc));
    const double ofb = fma(omw, fb, fma(-fac, qj, fsc));
    const double gsym = fma(k2c, qj * qj, k1c);
    const double oga = fma(omw, ga, fma(k3c, qj, gsym));
    const double ogb = fma(omw, gb, fma(-k3c, qj, gsym));
    double ofc, ofd = 0.0, ogc, ogd = 0.0;
    if (j == 0) {  // pair 8 (diagonal weight)
        ofc = fma(omw, fc, fma(faw[1], q[8], fsw[1]));
        ofd = fma(omw, fd, fma(-faw[1], q[8], fsw[1]));
        const double gs8 = fma(k2w[1], q[8] * q[8], k1w[1]);
        ogc = fma(omw, gc, fma(k3w[1], q[8], gs8));
        ogd = fma(omw, gd, fma(-k3w[1], q[8], gs8));
    } else {  // the rest population (lane 1)
        ofc = fma(omw, fc, sf * ph.c_f0);
        ogc = fma(omw, gc, fma(eg, ph.c_g0[0], fma(eps, ph.c_g0[1], egb2 * ph.c_g0[2])));
    }
    auto put = [&](int i, long long at, double fv, double gv) {
        B[RLB_CHK(i * S + at, 38ll * S)] = fv;
        B[RLB_CHK((19 + i) * S + at, 38ll * S)] = gv;
    };
    if (work) {
        if (solid) {  // the cell itself is solid: keep the marker
            const double m = solid_marker_d();
            put(ia, idx, m, m);
            put(ib, idx, m, m);
            if (j == 0) {
                put(17, idx, m, m);
                put(18, idx, m, m);
            } else if (j == 1) {
                put(0, idx, m, m);
            }
        } else {
            auto put_all = [&](long long at) {
                put(ia, at, ofa, oga);
                put(ib, at, ofb, ogb);
                if (j == 0) {
                    put(17, at, ofc, ogc);
                    put(18, at, ofd, ogd);
                } else if (j == 1) {
                    put(0, at, ofc, ogc);
                }
            };
            put_all(idx);
            if (XBC != XBC_PERIODIC && x == g.nx - 2) put_all(idx + 1);  // outflow ghost x = nx-1 copies x = nx-2
            if (XBC == XBC_OUTFLOW_BOTH && x == 1) put_all(idx - 1);      // outflow ghost x = 0 copies x = 1
        }
    } else if (XBC == XBC_INFLOW_OUTFLOW && live && !halo && x == 0) {
        // the inflow plane keeps its fixed equilibrium (copied)
        auto copy = [&](int i) {
            B[RLB_CHK(i * S + idx, 38ll * S)] = __ldg(RLB_CHK_PTR(A, i * S + idx, 38ll * S));
            B[RLB_CHK((19 + i) * S + idx, 38ll * S)] = __ldg(RLB_CHK_PTR(A, (19 + i) * S + idx, 38ll * S));
        };
        copy(ia);
        copy(ib);
        if (j == 0) {
            copy(17);
            copy(18);
        } else if (j == 1) {
            copy(0);
        }
    }
    if (count) {
        const bool mine = j == 0 && work && !solid;
        count_flags(cnt, mine && unphys, mine && nonpos, (unsigned long long)step_index * (unsigned long long)g.N + idx);
    }
}

// ---------------------------------------------------------------------------
// FP64 step in block fixed point (rlb_fixed.cuh), lattice speeds 1 <= c_l <= 2.
//
// k_step_f64 issues 203 FP64 instructions per cell, 13,200 clocks of the
// scheduler's FP64 pipe per 32 cells against 3,600 for the cell's 608 bytes
// at the HBM rate.  Here 53 remain (15 for the recovery, 38 relaxations
// h + omega (eq - h)) beside 2,989 instructions in all, 1,418 of them on the
// ALU pipe at two clocks each: the two pipes are loaded alike, and a warp's
// integer and FP64 phases overlap with those of the others.  256^3 box 6.07 ->
// 2.09 ms, 200x100x100 sphere 0.740 -> 0.285 ms per step.  Resident blocks of
// 128 threads: 4, 5 and 6 measure 2.20, 2.09 and 2.33 ms (0.291, 0.285 and
// 0.316 for the sphere).
//
// Lattice speed: all 19 populations of g share one exponent and the rest
// population is 9 c_l^2 times the moving ones, so with c_l they lose low bits;
// against 113-bit references the relaxed g are 3.3 times closer than those
// of the binary64 kernel at c_l = 1, 2.6 times at 2, 1.7 times at 3 and 12
// times further off at 10: the limit is 2, the range where the
// lattice speeds in use below that lie.
// ---------------------------------------------------------------------------

// Plane bases of both states as a kernel parameter: an address is a uniform
// base plus the cell's 32-bit offset.
struct PlaneTab64 {
    const double* a[38];
    double* b[38];
};

// The positivity decision of nonpositive_eq.  The flag depends on the largest
// |q_p| alone (the g bracket falls with |q| up to c_l / 3, beyond which the f
// bracket is negative), so beta in binary32 decides unless a bracket lies
// within 1e-4 of zero; then beta is formed in binary64 and rounded, as the
// general path does.  The step of this beta is q_scale = 12 c_l tau 2^-33, and a
// bracket can move by 68 of them (q by two steps times |12 q - 4 c_l| <= 25, b2
// by at most 3 times six): for tau c_l beyond 950 q_scale is NaN, which sends
// every cell to binary64.  (A margin that grows with tau, read from the
// constants instead of an immediate: 256^3 2.09 -> 2.17 ms.)
__device__ __forceinline__ bool fx_nonpositive(const FxG& t, const double* u, double rD, const FxRun& k) {
    const float bx = k.q_scale * (float)t.wx.h, by = k.q_scale * (float)t.wy.h, bz = k.q_scale * (float)t.wz.h;
    const float ax = fabsf(bx), ay = fabsf(by), az = fabsf(bz);
    const float q = fmaxf(ax + ay, fmaxf(ax + az, ay + az));
    const float b2 = fmaf(bx, bx, fmaf(by, by, bz * bz));
    const float m = fminf(fmaf(-3.0f, q, k.c_l), fmaf(q, fmaf(6.0f, q, -4.0f * k.c_l), fmaf(-3.0f, b2, 1.0f)));
    if (fabsf(m) > 1e-4f) return m < 0.0f;
    const double r3 = rD * k.three_cl;
    return nonpositive_eq(d2f(u[0] * r3), d2f(u[1] * r3), d2f(u[2] * r3), k.c_l);
}

template <int XBC>
__device__ __noinline__ bool step_cell_f64_general(const double* A, double* B, const Geom& g, const Phys& ph, int idx,
                                                   bool& unphys, bool& nonpos) {
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    const PullOffsets o(g, x, y, z);
    return step_cell_f64<XBC, true>(A, B, g, ph, idx, x, o, unphys, nonpos);
}

template <int XBC, int MINB>
__global__ void __launch_bounds__(128, MINB)
    k_step_f64_fx(const double* __restrict__ A, double* __restrict__ B, const __grid_constant__ Geom g,
                  const __grid_constant__ Phys ph, Counters cnt, int count, long long step_index,
                  const __grid_constant__ PlaneTab64 tab) {
    const int idx = dependent_begin(blockIdx.x * blockDim.x + threadIdx.x);
    if (idx >= g.N) return;
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    if (g.zhalo && (z == 0 || z == g.nz - 1)) return;  // z halo planes: filled by the exchange
    const long long S = g.S;
    auto pa = [&](int q, int off) { return __ldg(RLB_CHK_PTR(tab.a[q], (unsigned)off, S)); };
    // the inflow column keeps its populations: loaded with the warp's others,
    // through offsets of zero, and stored as loaded
    const bool keep = XBC == XBC_INFLOW_OUTFLOW && x == 0;
    if (XBC != XBC_PERIODIC && (x == g.nx - 1 || (x == 0 && !keep))) return;
    PullOffsets o(g, x, y, z);
    if (keep) o.xm = o.xp = o.ym = o.yp = o.zm = o.zp = 0;
    const FxRun& k = ph.fx;
    double h[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) h[i] = pa(19 + i, idx + o.src(i));
    // the f populations on their way to shared memory during the g phase, each
    // thread's into its own slots: loads after that phase were a third of the
    // stall cycles, and registers for them would cost two of the five blocks
    // (256^3: 2.34 -> 2.09 ms; 200x100x100 sphere: 300 -> 285 us)
    __shared__ double staged[19][128];
    const uint32_t slot = (uint32_t)__cvta_generic_to_shared(&staged[0][threadIdx.x]);
#pragma unroll
    for (int i = 0; i < 19; ++i)
        cp_async8(slot + (uint32_t)(i * 128 * 8), RLB_CHK_PTR(tab.a[i], (unsigned)(idx + o.src(i)), S));
    cp_async_commit();
    int em = fx_max_exponent<19>(h);
    unsigned bounced = 0u;
    if (em == 0x7FF) {  // a solid marker among them, or a non-finite population
        if (is_solid(h[0])) {  // the cell itself is solid: keep the marker
            const double m = solid_marker_d();
#pragma unroll
            for (int q = 0; q < 38; ++q) tab.b[q][RLB_CHK((unsigned)idx, S)] = m;
            cp_async_wait<0>();
            return;
        }
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            if (is_solid(h[i])) {  // link bounce-back
                bounced |= 1u << i;
                h[i] = pa(19 + (XBC == XBC_INFLOW_OUTFLOW && keep ? i : opp(i)), idx);
            }
        }
        em = fx_max_exponent<19>(h);
    }
    // the outflow ghosts that copy x (both when nx = 3)
    const bool dup_hi = XBC != XBC_PERIODIC && x == g.nx - 2, dup_lo = XBC == XBC_OUTFLOW_BOTH && x == 1;
    auto put = [&](int q, double v) {
        tab.b[q][RLB_CHK((unsigned)idx, S)] = v;
        if (dup_hi) tab.b[q][RLB_CHK((unsigned)idx + 1u, S)] = v;
        if (dup_lo) tab.b[q][RLB_CHK((unsigned)idx - 1u, S)] = v;
    };
    bool unphys = false, nonpos = false;
    FxG t;
    bool ok;
    {
        int64_t E = fx_round4(fx_from(h[0], em)), d[9];
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const int64_t a = fx_from(h[2 * p + 1], em), b = fx_from(h[2 * p + 2], em);
            E += fx_round4(a + b);
            d[p] = fx_round4(a - b);
        }
        double u[3], rD;
        ok = fx_g_terms(E, ((d[0] + d[3]) + (d[4] + d[5])) + d[6], ((d[1] + d[3]) - d[4]) + (d[7] + d[8]),
                        ((d[2] + d[5]) - d[6]) + (d[7] - d[8]), em, k, t, u, rD);
        if (ok) nonpos = fx_nonpositive(t, u, rD, k);
    }
    if (XBC == XBC_INFLOW_OUTFLOW && keep) {
        ok = true, nonpos = false;
#pragma unroll
        for (int i = 0; i < 19; ++i) tab.b[19 + i][RLB_CHK((unsigned)idx, S)] = h[i];
    } else if (ok) {
        put(19, fma(k.omw, h[0], fx_to(t.g0, t.eb + 3)));
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            int64_t s, a;
            fx_g_pair(t, p, s, a);
            put(20 + 2 * p, fma(k.omw, h[2 * p + 1], fx_to(s + a, t.eb)));
            put(21 + 2 * p, fma(k.omw, h[2 * p + 2], fx_to(s - a, t.eb)));
        }
    }
    cp_async_wait<0>();
    if (ok) {
        // ---- number populations f_i
#pragma unroll
        for (int i = 0; i < 19; ++i) h[i] = staged[i][threadIdx.x];
        if (bounced) {
#pragma unroll
            for (int i = 1; i < 19; ++i)
                if ((bounced >> i) & 1u) h[i] = pa(XBC == XBC_INFLOW_OUTFLOW && keep ? i : opp(i), idx);
        }
        const int ef = fx_max_exponent<19>(h);
        int64_t sum = fx_round4(fx_from(h[0], ef));
#pragma unroll
        for (int p = 0; p < 9; ++p) sum += fx_round4(fx_from(h[2 * p + 1], ef) + fx_from(h[2 * p + 2], ef));
        FxF q;
        ok = fx_f_terms(sum, ef, t, k, q);
        if (XBC == XBC_INFLOW_OUTFLOW && keep) {
            ok = true;
#pragma unroll
            for (int i = 0; i < 19; ++i) tab.b[i][RLB_CHK((unsigned)idx, S)] = h[i];
        } else if (ok) {
            put(0, fma(k.omw, h[0], fx_to((q.B << 3) + (q.B << 2), q.eb)));
#pragma unroll
            for (int p = 0; p < 9; ++p) {
                int64_t s, a;
                fx_f_pair(q, p, s, a);
                put(1 + 2 * p, fma(k.omw, h[2 * p + 1], fx_to(s + a, q.eb)));
                put(2 + 2 * p, fma(k.omw, h[2 * p + 2], fx_to(s - a, q.eb)));
            }
        }
    }
    if (!ok) step_cell_f64_general<XBC>(A, B, g, ph, idx, unphys, nonpos);
    if (count) count_flags(cnt, unphys, nonpos, (unsigned long long)step_index * (unsigned long long)g.N + idx);
}

// Eight lanes per cell (small lattices): lane j holds pair j (a: +, b: -),
// lane 0 also pair 8 (c: +, d: -), lane 1 the rest population (c).  The sums
// are integers, so the xor butterfly gives k_step_f64_fx's sums whatever the
// order, and the terms are formed by the same functions: the same values.
template <int XBC>
__global__ void __launch_bounds__(128)
    k_step_f64_fx_split(const double* __restrict__ A, double* __restrict__ B, const __grid_constant__ Geom g,
                        const __grid_constant__ Phys ph, Counters cnt, int count, long long step_index) {
    const unsigned full = 0xffffffffu;
    const int tid = dependent_begin(blockIdx.x * blockDim.x + threadIdx.x);  // 8 N < 2^31 (small lattices; tests)
    const int j = threadIdx.x & 7;  // lane of the cell's group
    const int cell = (int)((unsigned)tid >> 3);
    const bool live = cell < g.N;
    const int idx = live ? cell : 0;
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    const bool halo = g.zhalo && (z == 0 || z == g.nz - 1);  // filled by the exchange
    const bool ghost = XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1);
    const bool work = live && !halo && !ghost;  // a collided cell
    const long long S = g.S;
    const PullOffsets o(g, x, y, z);
    const FxRun& k = ph.fx;
    const int ia = 2 * j + 1, ib = 2 * j + 2;
    auto pull = [&](int i, double& fv, double& gv) {
        const int src = idx + o.src(i);
        fv = __ldg(RLB_CHK_PTR(A, i * S + src, 38ll * S));
        gv = __ldg(RLB_CHK_PTR(A, (19 + i) * S + src, 38ll * S));
        if (is_solid(fv)) {  // link bounce-back
            fv = __ldg(RLB_CHK_PTR(A, opp(i) * S + idx, 38ll * S));
            gv = __ldg(RLB_CHK_PTR(A, (19 + opp(i)) * S + idx, 38ll * S));
        }
    };
    double fa = 0.0, fb = 0.0, ga = 0.0, gb = 0.0, fc = 0.0, fd = 0.0, gc = 0.0, gd = 0.0;
    bool own_solid = false;
    if (work) {
        pull(ia, fa, ga);
        pull(ib, fb, gb);
        if (j == 0) {
            pull(17, fc, gc);
            pull(18, fd, gd);
        } else if (j == 1) {
            fc = __ldg(RLB_CHK_PTR(A, idx, 38ll * S));
            gc = __ldg(RLB_CHK_PTR(A, 19 * S + idx, 38ll * S));
            own_solid = is_solid(fc);
        }
    }
    const bool solid = __shfl_sync(full, own_solid, (threadIdx.x & 24) + 1);  // lane 1 holds f_0
    // block exponents of the cell's g and f populations
    const double gv[4] = {ga, gb, gc, gd}, fv[4] = {fa, fb, fc, fd};
    int em = fx_max_exponent<4>(gv), ef = fx_max_exponent<4>(fv);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        em = max(em, __shfl_xor_sync(full, em, off));
        ef = max(ef, __shfl_xor_sync(full, ef, off));
    }
    const int64_t xa = fx_from(ga, em), xb = fx_from(gb, em), xc = fx_from(gc, em), xd = fx_from(gd, em);
    long long E = fx_round4(xa + xb) + fx_round4(xc + xd);  // c, d: pair 8, the rest population, or zero
    long long s = fx_round4(fx_from(fa, ef) + fx_from(fb, ef)) + fx_round4(fx_from(fc, ef) + fx_from(fd, ef));
    const int64_t dj = fx_round4(xa - xb), d8 = fx_round4(xc - xd);  // d8: pair 8 on lane 0
    const int ex = pair_ex(j), ey = pair_ey(j), ez = pair_ez(j);
    long long dx = ex ? dj : 0;
    long long dy = j == 0 ? d8 : (ey > 0 ? dj : (ey < 0 ? -dj : 0));
    long long dz = j == 0 ? -d8 : (ez > 0 ? dj : (ez < 0 ? -dj : 0));
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        E += __shfl_xor_sync(full, E, off);
        s += __shfl_xor_sync(full, s, off);
        dx += __shfl_xor_sync(full, dx, off);
        dy += __shfl_xor_sync(full, dy, off);
        dz += __shfl_xor_sync(full, dz, off);
    }
    FxG t;
    FxF q;
    double u[3], rD;
    const bool ok = fx_g_terms(E, dx, dy, dz, em, k, t, u, rD) && fx_f_terms(s, ef, t, k, q);
    bool unphys = false, nonpos = false;
    if (work && solid) {  // keep the marker
        const double m = solid_marker_d();
        auto put = [&](int i) {
            B[RLB_CHK(i * S + idx, 38ll * S)] = m;
            B[RLB_CHK((19 + i) * S + idx, 38ll * S)] = m;
        };
        put(ia);
        put(ib);
        if (j == 0) {
            put(17);
            put(18);
        } else if (j == 1) {
            put(0);
        }
    } else if (work && ok) {
        // pair j: its axes (a, and b for a diagonal pair) selected by lane
        const bool axis = j < 3;
        const bool hx = ex != 0, hy = ey != 0;
        const int64_t Pa = hx ? t.Pxx : (hy ? t.Pyy : t.Pzz), Pb = axis ? 0 : (hx && hy ? t.Pyy : t.Pzz);
        int64_t Pc = axis ? 0 : (hx ? (hy ? t.Pxy : t.Pxz) : t.Pyz);
        const int64_t ua = hx ? t.ux : (hy ? t.uy : t.uz), Fa = hx ? q.Fx : (hy ? q.Fy : q.Fz);
        int64_t ub = axis ? 0 : (hx && hy ? t.uy : t.uz), Fb = axis ? 0 : (hx && hy ? q.Fy : q.Fz);
        if (j == 4 || j == 6) {  // the second axis negative
            Pc = -Pc;
            ub = -ub;
            Fb = -Fb;
        }
        const int sh = axis ? 1 : 0;
        const int64_t gs = (((t.A + Pa) + Pb) + (Pc << 1)) << sh, gy = (ua + ub) << sh;
        const int64_t fs = q.B << sh, fy = (Fa + Fb) << sh;
        const double ofa = fma(k.omw, fa, fx_to(fs + fy, q.eb)), ofb = fma(k.omw, fb, fx_to(fs - fy, q.eb));
        const double oga = fma(k.omw, ga, fx_to(gs + gy, t.eb)), ogb = fma(k.omw, gb, fx_to(gs - gy, t.eb));
        // pair 8 on lane 0, the rest population on lane 1
        const bool l0 = j == 0;
        int64_t s8, a8, f8, y8;
        fx_g_pair(t, 8, s8, a8);
        fx_f_pair(q, 8, f8, y8);
        double ofc = 0.0, ofd = 0.0, ogc = 0.0, ogd = 0.0;
        if (j < 2) {
            ofc = fma(k.omw, fc, fx_to(l0 ? f8 + y8 : (q.B << 3) + (q.B << 2), q.eb));
            ogc = fma(k.omw, gc, fx_to(l0 ? s8 + a8 : t.g0, l0 ? t.eb : t.eb + 3));
            ofd = fma(k.omw, fd, fx_to(f8 - y8, q.eb));
            ogd = fma(k.omw, gd, fx_to(s8 - a8, t.eb));
        }
        auto put = [&](int i, long long at, double fo, double go) {
            B[RLB_CHK(i * S + at, 38ll * S)] = fo;
            B[RLB_CHK((19 + i) * S + at, 38ll * S)] = go;
        };
        auto put_all = [&](long long at) {
            put(ia, at, ofa, oga);
            put(ib, at, ofb, ogb);
            if (j == 0) {
                put(17, at, ofc, ogc);
                put(18, at, ofd, ogd);
            } else if (j == 1) {
                put(0, at, ofc, ogc);
            }
        };
        put_all(idx);
        if (XBC != XBC_PERIODIC && x == g.nx - 2) put_all(idx + 1);  // outflow ghost x = nx-1 copies x = nx-2
        if (XBC == XBC_OUTFLOW_BOTH && x == 1) put_all(idx - 1);      // outflow ghost x = 0 copies x = 1
        if (j == 0) nonpos = fx_nonpositive(t, u, rD, k);
    } else if (work) {
        if (j == 0) step_cell_f64_general<XBC>(A, B, g, ph, idx, unphys, nonpos);
    } else if (XBC == XBC_INFLOW_OUTFLOW && live && !halo && x == 0) {
        // the inflow plane keeps its fixed equilibrium (copied)
        auto copy = [&](int i) {
            B[RLB_CHK(i * S + idx, 38ll * S)] = __ldg(RLB_CHK_PTR(A, i * S + idx, 38ll * S));
            B[RLB_CHK((19 + i) * S + idx, 38ll * S)] = __ldg(RLB_CHK_PTR(A, (19 + i) * S + idx, 38ll * S));
        };
        copy(ia);
        copy(ib);
        if (j == 0) {
            copy(17);
            copy(18);
        } else if (j == 1) {
            copy(0);
        }
    }
    if (count) count_flags(cnt, unphys, nonpos, (unsigned long long)step_index * (unsigned long long)g.N + idx);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
namespace {

template <int XBC>
void launch_step_f64_t(const Geom& g, const Phys& ph, const double* A, double* B, Counters cnt, bool count,
                       long long step_index, cudaStream_t st) {
    static int nsm = 0;
    if (nsm == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    }
    const int c = count ? 1 : 0;
    auto blocks = [](long long n, int bs) { return (unsigned)((n + bs - 1) / bs); };
    // eight lanes per cell while the lanes fit one warp per scheduler
    // (N <= 16 x SMs), unless RLB_F64_SPLIT says otherwise; same values.  The
    // 1600-cell tube, issued on the stream: 10.24 us per step in binary64, 8.20
    // in fixed point (20 instead of 103 FP64 instructions per warp), 6.25
    // launched back to back.
    const bool split = (g.f64split == 1 && g.N < (1 << 27)) || (g.f64split < 0 && g.N <= 16ll * nsm);
    if (ph.fx_on) {
        if (split) {
            launch_dependent(k_step_f64_fx_split<XBC>, blocks(8ll * g.N, 128), 128, 0, st, A, B, g, ph, cnt, c, step_index);
            return;
        }
        PlaneTab64 tab;
        for (int q = 0; q < 38; ++q) {
            tab.a[q] = A + (long long)q * g.S;
            tab.b[q] = B + (long long)q * g.S;
        }
        // small lattices spread over more SMs in 32-thread blocks
        const int tb = blocks(g.N, 128) < (unsigned)nsm ? 32 : 128;
        launch_dependent(k_step_f64_fx<XBC, 5>, blocks(g.N, tb), tb, 0, st, A, B, g, ph, cnt, c, step_index, tab);
        return;
    }
    if (split) {
        launch_dependent(k_step_f64_split<XBC, true>, blocks(8ll * g.N, 128), 128, 0, st, A, B, g, ph, cnt, c, step_index);
        return;
    }
    const int tb = blocks(g.N, 128) < (unsigned)nsm ? 32 : 128;
    launch_dependent(k_step_f64<XBC, true>, blocks(g.N, tb), tb, 0, st, A, B, g, ph, cnt, c, step_index);
}
}  // namespace

cudaError_t launch_step_f64(const Geom& g, const Phys& ph, const void* A, void* B, Counters cnt, bool count,
                            long long step_index, cudaStream_t st) {
    const double* a = (const double*)A;
    double* b = (double*)B;
    set_last_launch_count(1);
    switch (g.xbc) {
        case XBC_PERIODIC: launch_step_f64_t<XBC_PERIODIC>(g, ph, a, b, cnt, count, step_index, st); break;
        case XBC_INFLOW_OUTFLOW: launch_step_f64_t<XBC_INFLOW_OUTFLOW>(g, ph, a, b, cnt, count, step_index, st); break;
        default: launch_step_f64_t<XBC_OUTFLOW_BOTH>(g, ph, a, b, cnt, count, step_index, st); break;
    }
    return cudaGetLastError();
}

// Bounds-check count of this translation unit (0 in the release build).
RLB_OOB_TAKE_FN(oob_take_step64)

}  // namespace rlb
