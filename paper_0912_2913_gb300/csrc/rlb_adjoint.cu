// rlb_adjoint.cu -- discrete adjoint of the relativistic lattice Boltzmann
// step (the transpose of the exact Jacobian of Eqs. lbe1/lbe2 with the
// eps = 3P equilibria Eqs. equil1s, equil2as, equil2bs and the closed-form
// recovery), the adjoint of the macroscopic output and of the equilibrium
// initialisation.
//
// Step adjoint, push form.  With lambda_{t+1} = dL/dA_{t+1}, one thread per
// interior fluid cell x
//   1. gathers h(x) from A_t exactly as the forward step does,
//   2. takes mu(x) = lambda_{t+1}(x) (+ lambda_{t+1} of the outflow ghost that
//      copies x),
//   3. forms nu = J_C(h)^T mu, where C(h) = h + (eq(m(h)) - h)/tau:
//        nu = (1 - 1/tau) mu + (1/tau) P^T (d eq / d m)^T mu,
//      m = P h the five moments, by the chain rule through the equilibria and
//      the recovery (the partial derivatives are written out below),
//   4. scatters nu_i to lambda_t(x - e_i, i), or to lambda_t(x, opp(i)) when
//      x - e_i is solid (transpose of the pull with bounce-back).
// Every element of lambda_t has exactly one writer: the scatter above, or
// the owner cell writing 0 where nobody reads the population (a neighbour
// that is a ghost plane), or the identity at solid cells (never updated).
// dL/dtau = sum mu_i (h_i - eq_i)/tau^2 and, at the inflow plane (held at
// eq(n_in, eps_in, beta_in)), dL/dbeta_in = sum lambda_{t+1} d eq/d beta_in
// are summed per warp (binary32 for the FP32 path, binary64 otherwise), per
// block, and over the blocks in a fixed order: by the block that ends last
// (block_sums, FP64) or by a second kernel (k_finalize).
#include <cuda.h>  // CUcontext type only; cuCtxGetCurrent is taken through the runtime
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "rlb_device.cuh"
#include "rlb_fixed.cuh"

namespace rlb {

// ---------------------------------------------------------------------------
// Adjoint of the g equilibria (Eqs. equil2as, equil2bs) with respect to
// (eps, beta) at fixed mu:   a_eps = sum mu_i d g_i / d eps,
//                            a_beta = sum mu_i d g_i / d beta.
// g_{+-p} = w_p [eps/c_l^2 + eps gamma^2 (6 q_p^2 - 2 b2)/c_l^2] +- w_p eps gamma^2 4 q_p / c_l
// g_0     = w_0 [4 eps gamma^2 - eps (2 + c_l^2)/c_l^2 - 2 eps gamma^2 b2 / c_l^2]
// with q_p = e_p . beta, b2 = |beta|^2, d gamma^2 / d beta = 2 gamma^4 beta.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void g_eq_adjoint(const T* mug, T eps, T bx, T by, T bz, T b2, T gam2, T inv_cl,
                                             T inv_cl2, T& a_eps, T& abx, T& aby, T& abz) {
    const T q[9] = {bx, by, bz, bx + by, bx - by, bx + bz, bx - bz, by + bz, by - bz};
    T ae = 0, gg2 = 0, gb2 = 0;  // d/d eps, d/d gamma^2, d/d b2 (explicit)
    T Qp[9];
    T sw = 0;  // sum_p w_p sigma_p
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const T w = (T)pair_w(p);
        const T sig = mug[2 * p + 1] + mug[2 * p + 2];
        const T del = mug[2 * p + 1] - mug[2 * p + 2];
        const T sym = (6 * q[p] * q[p] - 2 * b2) * inv_cl2;
        const T asy = 4 * q[p] * inv_cl;
        ae += w * (sig * (inv_cl2 + gam2 * sym) + del * gam2 * asy);
        gg2 += w * (sig * sym + del * asy);
        sw += w * sig;
        // d/dq_p: w eps gamma^2 (sigma 12 q / c_l^2 + delta 4 / c_l)
        Qp[p] = w * (sig * 12 * q[p] * inv_cl2 + del * 4 * inv_cl);
    }
    const T w0 = (T)kW0;
    const T m0 = mug[0];
    ae += w0 * m0 * (4 * gam2 - (2 * inv_cl2 + 1) - 2 * gam2 * b2 * inv_cl2);
    gg2 += w0 * m0 * (4 - 2 * b2 * inv_cl2);
    gb2 = -2 * gam2 * inv_cl2 * (sw + w0 * m0);
    // chain: gamma^2 (factor eps), b2 (factor eps), q_p (factor eps gamma^2)
    const T eg = eps * gam2;
    const T rad = 2 * eps * (gb2 + gam2 * gam2 * gg2);  // coefficient of beta_a
    a_eps = ae;
    abx = eg * (Qp[0] + Qp[3] + Qp[4] + Qp[5] + Qp[6]) + rad * bx;
    aby = eg * (Qp[1] + Qp[3] - Qp[4] + Qp[7] + Qp[8]) + rad * by;
    abz = eg * (Qp[2] + Qp[5] - Qp[6] + Qp[7] - Qp[8]) + rad * bz;
}

// Adjoint of the f equilibria written as f_i = w_i S (1 + 3 q_i / c_l) with
// S = n gamma held fixed: a_S = sum mu_i w_i (1 + 3 q_i/c_l),
// a_beta = (3 S / c_l) sum_i mu_i w_i e_i.
template <typename T>
__device__ __forceinline__ void f_eq_adjoint_S(const T* muf, T S, T bx, T by, T bz, T inv_cl, T& aS, T& abx, T& aby,
                                               T& abz) {
    const T q[9] = {bx, by, bz, bx + by, bx - by, bx + bz, bx - bz, by + bz, by - bz};
    T s0 = (T)kW0 * muf[0], s1 = 0;
    T d[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const T w = (T)pair_w(p);
        s0 += w * (muf[2 * p + 1] + muf[2 * p + 2]);
        d[p] = w * (muf[2 * p + 1] - muf[2 * p + 2]);
        s1 += d[p] * q[p];
    }
    aS = s0 + 3 * inv_cl * s1;
    const T c = 3 * S * inv_cl;
    abx = c * (d[0] + d[3] + d[4] + d[5] + d[6]);
    aby = c * (d[1] + d[3] - d[4] + d[7] + d[8]);
    abz = c * (d[2] + d[5] - d[6] + d[7] - d[8]);
}

// Adjoint of the closed-form recovery: given adjoints (a_eps, a_beta) of
// eps = s - E and beta = 3M/D (s = sqrt(4E^2 - 3M^2), D = 3E + eps), the
// adjoints of E and M:
//   d eps/dE = 4E/s - 1,          d eps/dM_b = -3 M_b / s,
//   d beta_a/dE = -(beta_a/D)(3 + d eps/dE),
//   d beta_a/dM_b = 3 delta_ab / D + 3 beta_a M_b / (D s).
template <typename T>
__device__ __forceinline__ void recovery_adjoint(T a_eps, T abx, T aby, T abz, T E, T s, T D, T bx, T by, T bz, T Mx,
                                                 T My, T Mz, T& vE, T& vx, T& vy, T& vz) {
    const T ab_b = abx * bx + aby * by + abz * bz;
    const T rD = 1 / D;
    const T rs = 1 / s;
    const T depsdE = 4 * E * rs - 1;
    vE = a_eps * depsdE - ab_b * rD * (3 + depsdE);
    const T c = 3 * rs * (ab_b * rD - a_eps);
    vx = 3 * abx * rD + c * Mx;
    vy = 3 * aby * rD + c * My;
    vz = 3 * abz * rD + c * Mz;
}

// Warp partial sums written to red[(global warp)*4 + k], no block barrier:
// tau in binary32 across the warp for the FP32 path (the per-cell terms are
// binary32 already), the beta_in terms only when a lane has one.
template <typename T>
__device__ __forceinline__ void warp_partials(double tau, double b0, double b1, double b2, bool has_b, double* red) {
    const unsigned full = 0xffffffffu;
    double v0;
    if constexpr (sizeof(T) == 4) {
        float t = (float)tau;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(full, t, off);
        v0 = (double)t;
    } else {
        v0 = tau;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v0 += __shfl_xor_sync(full, v0, off);
    }
    double v1 = b0, v2 = b1, v3 = b2;
    if (__any_sync(full, has_b)) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            v1 += __shfl_xor_sync(full, v1, off);
            v2 += __shfl_xor_sync(full, v2, off);
            v3 += __shfl_xor_sync(full, v3, off);
        }
    }
    if ((threadIdx.x & 31) == 0) {
        const long long wg = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
        red[wg * 4 + 0] = v0;
        red[wg * 4 + 1] = v1;
        red[wg * 4 + 2] = v2;
        red[wg * 4 + 3] = v3;
    }
}

// Block reduction of four doubles into red[blockIdx.x*4 + k].
__device__ __forceinline__ void block_reduce4(double v0, double v1, double v2, double v3, double* red) {
    __shared__ double sm[4][32];
    double v[4] = {v0, v1, v2, v3};
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) sm[k][warp] = v[k];
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            double t = lane < nw ? sm[k][lane] : 0.0;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) t += __shfl_down_sync(0xffffffffu, t, off);
            if (lane == 0) red[blockIdx.x * 4 + k] = t;
        }
    }
}

// Where a persistent adjoint kernel leaves its sums: red[block*4 + k], then,
// by the last block to arrive at the ticket (which it resets to 0), the sum
// over the blocks added to the accumulators.  The ticket is the context's, also
// where red is shared by all contexts of a device: launches of two contexts
// that overlap spoil their own sums, not those of later ones.
struct AdjSums {
    double* red;
    unsigned* ticket;
    double* dtau;
    double* dbeta_in;
};

// The tail of a persistent adjoint kernel, reached by every thread of its
// (at most 128-thread) blocks.  The last block sums the block partials in an
// order that depends on the grid alone, so the result does not depend on
// scheduling; nothing waits.  Saves a launch per step (1600 cells 21 -> 18 us;
// in the staged FP32 kernels it cost the main loop 1.5 % on the 256^3 box, so
// they keep k_finalize).  BIN: the dL/dbeta_in terms exist (an inflow plane).
template <typename T, bool BIN>
__device__ __forceinline__ void block_sums(double tau, double b0, double b1, double b2, bool has_b, const AdjSums& out) {
    constexpr unsigned full = 0xffffffffu;
    constexpr int NC = BIN ? 4 : 1;
    __shared__ double part[4][NC];
    __shared__ double sm[128];
    __shared__ bool last;
    double v[4] = {tau, b0, b1, b2};
    if constexpr (sizeof(T) == 4) {
        float t = (float)tau;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(full, t, off);
        v[0] = (double)t;
    } else {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v[0] += __shfl_xor_sync(full, v[0], off);
    }
    if (BIN && __any_sync(full, has_b)) {
#pragma unroll
        for (int k = 1; k < 4; ++k)
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(full, v[k], off);
    }
    const int tid = threadIdx.x, nw = blockDim.x >> 5;
    if ((tid & 31) == 0)
#pragma unroll
        for (int k = 0; k < NC; ++k) part[tid >> 5][k] = v[k];
    __syncthreads();
    if (tid < NC) {
        double s = part[0][tid];
        for (int w = 1; w < nw; ++w) s += part[w][tid];
        out.red[blockIdx.x * 4 + tid] = s;
        __threadfence();
    }
    __syncthreads();
    if (tid == 0) {
        last = atomicAdd(out.ticket, 1u) == gridDim.x - 1;
        if (last) *out.ticket = 0u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int k = tid % NC, step = (int)blockDim.x / NC, nb = (int)gridDim.x;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    int b = tid / NC;
    for (; b + 3 * step < nb; b += 4 * step)
#pragma unroll
        for (int j = 0; j < 4; ++j) a[j] += __ldcg(out.red + (b + j * step) * 4 + k);
    for (int j = 0; j < 3; ++j)
        if (b + j * step < nb) a[j] += __ldcg(out.red + (b + j * step) * 4 + k);
    sm[tid] = (a[0] + a[1]) + (a[2] + a[3]);
    __syncthreads();
    for (int h = (int)blockDim.x / 2; h >= NC; h >>= 1) {
        if (tid < h) sm[tid] += sm[tid + h];
        __syncthreads();
    }
    if (tid == 0) {
        *out.dtau += sm[0];
        if (BIN) {
            out.dbeta_in[0] += sm[NC > 1 ? 1 : 0];
            out.dbeta_in[1] += sm[NC > 1 ? 2 : 0];
            out.dbeta_in[2] += sm[NC > 1 ? 3 : 0];
        }
    }
}

// Sum the partial-sum slots (one per warp or per block, 4 doubles each) and
// add them to the accumulators: block k sums component k (each on its own SM:
// the additions of the four together were bound by one SM's FP64 pipe, 10 us
// for 1824 slots), block 0 alone without an inflow plane, whose terms are all
// zero.  Thread t sums slots t, t+256, ... in a fixed grouping, then a fixed
// tree combines the 256 sums: the result does not depend on scheduling.
__global__ void __launch_bounds__(256) k_finalize(const double* __restrict__ red, int nslots, double* dtau,
                                                  double* dbeta_in) {
    __shared__ double sm[256];
    const int k = blockIdx.x, t = dependent_begin(threadIdx.x);
    if (k == 0 && !dtau) return;
    // four independent partial sums so that four loads are in flight; the
    // grouping depends only on nslots (deterministic)
    double a[4] = {0, 0, 0, 0};
    int b = t;
    for (; b + 3 * 256 < nslots; b += 4 * 256) {
#pragma unroll
        for (int j = 0; j < 4; ++j) a[j] += red[(b + j * 256) * 4 + k];
    }
#pragma unroll
    for (int j = 0; j < 3; ++j)
        if (b + j * 256 < nslots) a[j] += red[(b + j * 256) * 4 + k];
    sm[t] = (a[0] + a[1]) + (a[2] + a[3]);
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (t < h) sm[t] += sm[t + h];
        __syncthreads();
    }
    if (t == 0) {
        if (k == 0)
            *dtau += sm[0];
        else
            dbeta_in[k - 1] += sm[0];
    }
}

// Adjoint of eq(n, eps, beta) with respect to the fields (f with n gamma,
// gamma = (1 - b2)^-1/2, d gamma / d beta = gamma^3 beta).
__device__ __noinline__ void eq_fields_adjoint(const double* muf, const double* mug, double n, double eps, double bx, double by,
                                  double bz, const Phys& ph, double& an, double& ae, double& abx, double& aby,
                                  double& abz) {
    const double b2 = bx * bx + by * by + bz * bz;
    const double gam2 = 1.0 / (1.0 - b2);
    const double gam = sqrt(gam2);
    double aS, fbx, fby, fbz;
    f_eq_adjoint_S(muf, n * gam, bx, by, bz, ph.inv_cl, aS, fbx, fby, fbz);
    // S = n gamma: dS/dn = gamma, dS/dbeta = n gamma^3 beta
    an = aS * gam;
    const double cS = aS * n * gam * gam2;
    double gbx, gby, gbz;
    g_eq_adjoint(mug, eps, bx, by, bz, b2, gam2, ph.inv_cl, ph.inv_cl2, ae, gbx, gby, gbz);
    abx = fbx + gbx + cS * bx;
    aby = fby + gby + cS * by;
    abz = fbz + gbz + cS * bz;
}

// ---------------------------------------------------------------------------
// Step adjoint.  T = double: FP64 states and arithmetic.  T = float: FP32
// deviation states, binary32 arithmetic throughout (the recovery in the
// cancellation-free deviation form of cell_g).  Per cell two phases, g then
// f.  The per-cell mathematics (cell_g, cell_f, scatter_cell) is shared by
// the register kernel and the shared-memory staged kernel.
// ---------------------------------------------------------------------------
template <typename T>
struct AdjConst {
    T om, omw, c_l, inv_cl, inv_cl2, n_ref, g0a, g0b, eps_ref_t, inv_tau2_t;
    double inv_tau2;
    // per-run products for the binary64 cell functions (cell_g64 and after);
    // the _36 ones divided by 36, for the pair sums carried times 36
    double c2, c2p1;                  // 2/c_l^2, 2/c_l^2 + 1
    double i2_36, c2_36, c3_36, c4_36, c6_36, c12_36;  // 1/c_l^2, 2/c_l^2, 3/c_l, 4/c_l, 6/c_l^2, 12/c_l^2
    double three_cl, m3cl2, om_cl;    // 3 c_l, -3 c_l^2, omega c_l
    double g0_eg, g0_e, g0_egb2;      // g_0^eq = eg g0_eg + eps g0_e + eg b2 g0_egb2
};

template <typename T>
static AdjConst<T> make_adj_const(const Phys& ph) {
    AdjConst<T> c;
    c.om = (T)ph.omega;
    c.omw = (T)(1.0 - ph.omega);
    c.c_l = (T)ph.c_l;
    c.inv_cl = (T)ph.inv_cl;
    c.inv_cl2 = (T)ph.inv_cl2;
    c.n_ref = (T)ph.n_ref;
    c.g0a = (T)(3.0 - 2.0 * ph.inv_cl2);
    c.g0b = (T)(4.0 - 2.0 * ph.inv_cl2);
    c.eps_ref_t = (T)ph.eps_ref;
    c.inv_tau2 = ph.omega * ph.omega;
    c.inv_tau2_t = (T)c.inv_tau2;
    c.c2 = 2.0 * ph.inv_cl2;
    c.i2_36 = ph.inv_cl2 / 36.0;
    c.c2_36 = 2.0 * ph.inv_cl2 / 36.0;
    c.c3_36 = 3.0 * ph.inv_cl / 36.0;
    c.c4_36 = 4.0 * ph.inv_cl / 36.0;
    c.c6_36 = 6.0 * ph.inv_cl2 / 36.0;
    c.c12_36 = 12.0 * ph.inv_cl2 / 36.0;
    c.three_cl = 3.0 * ph.c_l;
    c.m3cl2 = -3.0 * ph.c_l * ph.c_l;
    c.om_cl = ph.omega * ph.c_l;
    c.g0_eg = 4.0 * kW0;
    c.g0_e = -kW0 * (2.0 * ph.inv_cl2 + 1.0);
    c.g0_egb2 = -2.0 * kW0 * ph.inv_cl2;
    c.c2p1 = 2.0 * ph.inv_cl2 + 1.0;
    return c;
}

// Sums over the 19 populations as shallow trees (independent partial sums
// instead of one 18-deep dependency chain).
template <typename T>
__device__ __forceinline__ T sum19(const T* h) {
    const T a0 = h[0] + h[1], a1 = h[2] + h[3], a2 = h[4] + h[5], a3 = h[6] + h[7], a4 = h[8] + h[9];
    const T a5 = h[10] + h[11], a6 = h[12] + h[13], a7 = h[14] + h[15], a8 = h[16] + h[17];
    return ((a0 + a1) + (a2 + a3)) + (((a4 + a5) + (a6 + a7)) + (a8 + h[18]));
}
template <typename T>
__device__ __forceinline__ T dot19(const T* a, const T* b) {
    T s0 = a[0] * b[0], s1 = a[1] * b[1], s2 = a[2] * b[2], s3 = a[3] * b[3];
#pragma unroll
    for (int i = 4; i < 16; i += 4) {
        s0 += a[i] * b[i];
        s1 += a[i + 1] * b[i + 1];
        s2 += a[i + 2] * b[i + 2];
        s3 += a[i + 3] * b[i + 3];
    }
    s0 += a[16] * b[16];
    s1 += a[17] * b[17];
    s2 += a[18] * b[18];
    return (s0 + s1) + (s2 + s3);
}

// What the g phase leaves for the f phase and the recovery adjoint.
template <typename T>
struct CellG {
    T mx, my, mz, Et, sqt, Dt, bx, by, bz;  // moments (cell_g64: M / c_l), recovery
    T tacc, ae, gbx, gby, gbz;              // sum mu_g (h - eq), d/d eps, d/d beta
    T rD, rs;                               // 1/D, 1/s (cell_g64)
};

// Moments and recovery from the 19 g populations h, then the g part of the
// collision adjoint at mu = mug.
template <typename T>
__device__ __forceinline__ void cell_g(const T* h, const T* mug, const AdjConst<T>& c, CellG<T>& r) {
    const T dE = sum19(h);
    T dd[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) dd[p] = h[2 * p + 1] - h[2 * p + 2];
    const T mx = c.c_l * (dd[0] + dd[3] + dd[4] + dd[5] + dd[6]);
    const T my = c.c_l * (dd[1] + dd[3] - dd[4] + dd[7] + dd[8]);
    const T mz = c.c_l * (dd[2] + dd[5] - dd[6] + dd[7] - dd[8]);
    T Et, sqt, Dt, epst, e0, bx, by, bz, b2, gam2;
    if constexpr (sizeof(T) == 8) {
        const double E = dE;
        const double sq = sqrt(4.0 * E * E - 3.0 * (mx * mx + my * my + mz * mz));
        const double eps = sq - E;
        const double D = 3.0 * E + eps;
        const double r3 = 3.0 / D;
        bx = mx * r3;
        by = my * r3;
        bz = mz * r3;
        b2 = bx * bx + by * by + bz * bz;
        gam2 = 1.0 / (1.0 - b2);
        Et = E;
        sqt = sq;
        Dt = D;
        epst = eps;
        e0 = eps;
    } else {
        // binary32 in deviation form (the coefficients of the adjoint need
        // no FP64): E = eps_ref + dE, s = sqrt(E^2 - 3/4 M^2), eps = 2 s - E,
        // and the deviation eps - eps_ref = 2 (s - eps_ref) - dE with
        // s - eps_ref = (dE (2 eps_ref + dE) - 3/4 M^2) / (s + eps_ref),
        // free of the cancellation of eps - eps_ref.
        const float er = c.eps_ref_t;
        const float m34 = 0.75f * fmaf(mx, mx, fmaf(my, my, mz * mz));
        const float num = fmaf(dE, fmaf(2.0f, er, dE), -m34);
        const float sr = sqrtf(fmaf(er, er, num));
        e0 = fmaf(2.0f, __fdividef(num, sr + er), -dE);
        epst = er + e0;
        Et = er + dE;
        sqt = 2.0f * sr;
        Dt = fmaf(3.0f, Et, epst);
        const float r3 = __fdividef(3.0f, Dt);
        bx = mx * r3;
        by = my * r3;
        bz = mz * r3;
        b2 = fmaf(bx, bx, fmaf(by, by, bz * bz));
        gam2 = __fdividef(1.0f, 1.0f - b2);
    }
    const T q[9] = {bx, by, bz, bx + by, bx - by, bx + bz, bx - bz, by + bz, by - bz};
    const T eg = epst * gam2;
    // Everything the collision adjoint needs from mu reduces to a few
    // weighted pair sums (sigma_p = mu_{+p} + mu_{-p}, delta_p = mu_{+p} -
    // mu_{-p}, weight w_p, q_p = e_p . beta):
    //   S1 = sum w sigma,  Sq2 = sum w sigma q^2,  Sdq = sum w delta q,
    //   Vq = sum w sigma q e_p,  Vd = sum w delta e_p.
    // With them (Eqs. equil2as/equil2bs and their derivatives):
    //   sum mu_i geq_i = mu_0 geq_0 + k1 S1 + k2 Sq2 + k3 Sdq,
    //   d/d eps = S1/c_l^2 + gamma^2 (SYM + ASY) + rest-particle term,
    //   d/d gamma^2 = eps (SYM + ASY + rest term), d/d b2 = -2 eps gamma^2 (S1 + w0 mu_0)/c_l^2,
    //   d/d beta = eps gamma^2 (12 Vq / c_l^2 + 4 Vd / c_l) + (chain through gamma^2 and b2) beta,
    // SYM = (6 Sq2 - 2 b2 S1)/c_l^2, ASY = 4 Sdq / c_l; and likewise for f.
    const T muh = dot19(mug, h);
    T S1 = 0, Sq2 = 0, Sdq = 0, Vq[3] = {0, 0, 0}, Vd[3] = {0, 0, 0};
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const T w = (T)pair_w(p);
        const T ws = w * (mug[2 * p + 1] + mug[2 * p + 2]);
        const T wd = w * (mug[2 * p + 1] - mug[2 * p + 2]);
        S1 += ws;
        const T wsq = ws * q[p];
        Sq2 += wsq * q[p];
        Sdq += wd * q[p];
        const int ex = pair_ex(p), ey = pair_ey(p), ez = pair_ez(p);
        if (ex) { Vq[0] += wsq; Vd[0] += wd; }
        if (ey > 0) { Vq[1] += wsq; Vd[1] += wd; }
        if (ey < 0) { Vq[1] -= wsq; Vd[1] -= wd; }
        if (ez > 0) { Vq[2] += wsq; Vd[2] += wd; }
        if (ez < 0) { Vq[2] -= wsq; Vd[2] -= wd; }
    }
    const T m0 = mug[0], w0 = (T)kW0;
    const T k1 = (e0 - 2 * eg * b2) * c.inv_cl2, k2 = 6 * eg * c.inv_cl2, k3 = 4 * eg * c.inv_cl;
    const T geq0 = (sizeof(T) == 8) ? w0 * (4 * eg - epst * (2 * c.inv_cl2 + 1) - 2 * eg * b2 * c.inv_cl2)
                                    : w0 * (e0 * c.g0a + eg * b2 * c.g0b);
    r.tacc = muh - (m0 * geq0 + k1 * S1 + k2 * Sq2 + k3 * Sdq);
    const T SYM = (6 * Sq2 - 2 * b2 * S1) * c.inv_cl2;
    const T ASY = 4 * c.inv_cl * Sdq;
    r.ae = c.inv_cl2 * S1 + gam2 * (SYM + ASY) + w0 * m0 * (4 * gam2 - (2 * c.inv_cl2 + 1) - 2 * gam2 * b2 * c.inv_cl2);
    const T gg2 = SYM + ASY + w0 * m0 * (4 - 2 * b2 * c.inv_cl2);
    const T gb2 = -2 * gam2 * c.inv_cl2 * (S1 + w0 * m0);
    const T rad = 2 * epst * (gb2 + gam2 * gam2 * gg2);
    const T cq = eg * 12 * c.inv_cl2, cd = eg * 4 * c.inv_cl;
    r.gbx = cq * Vq[0] + cd * Vd[0] + rad * bx;
    r.gby = cq * Vq[1] + cd * Vd[1] + rad * by;
    r.gbz = cq * Vq[2] + cd * Vd[2] + rad * bz;
    r.mx = mx;
    r.my = my;
    r.mz = mz;
    r.Et = Et;
    r.sqt = sqt;
    r.Dt = Dt;
    r.bx = bx;
    r.by = by;
    r.bz = bz;
}

// The f part: sum mu_f (h - eq) and the adjoints of S = n gamma and beta.
template <typename T>
__device__ __forceinline__ void cell_f(const T* h, const T* muf, const CellG<T>& r, const AdjConst<T>& c, T& tacc,
                                       T& aS, T& fbx, T& fby, T& fbz) {
    const T q[9] = {r.bx, r.by, r.bz, r.bx + r.by, r.bx - r.by, r.bx + r.bz, r.bx - r.bz, r.by + r.bz, r.by - r.bz};
    const T dS = sum19(h);
    const T Sfull = (sizeof(T) == 8) ? dS : dS + c.n_ref;
    const T muh = dot19(muf, h);
    T F1 = 0, Fdq = 0, Vf[3] = {0, 0, 0};
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const T w = (T)pair_w(p);
        const T ws = w * (muf[2 * p + 1] + muf[2 * p + 2]);
        const T wd = w * (muf[2 * p + 1] - muf[2 * p + 2]);
        F1 += ws;
        Fdq += wd * q[p];
        const int ex = pair_ex(p), ey = pair_ey(p), ez = pair_ez(p);
        if (ex) Vf[0] += wd;
        if (ey > 0) Vf[1] += wd;
        if (ey < 0) Vf[1] -= wd;
        if (ez > 0) Vf[2] += wd;
        if (ez < 0) Vf[2] -= wd;
    }
    const T w0 = (T)kW0;
    const T fa = 3 * Sfull * c.inv_cl;
    // f^eq_{+-p} = w_p (fb +- fa q_p), fb = S (values) or dS (deviations)
    tacc = muh - (muf[0] * w0 * dS + dS * F1 + fa * Fdq);
    aS = w0 * muf[0] + F1 + 3 * c.inv_cl * Fdq;
    fbx = fa * Vf[0];
    fby = fa * Vf[1];
    fbz = fa * Vf[2];
}

// nu = (1 - 1/tau) mu + (1/tau) P^T v for the 38 populations of the cell,
// handed to put(plane, velocity, value) (the transpose of the pull).
template <typename T, typename PUT>
__device__ __forceinline__ void scatter_cell(const T* muf, const T* mug, T aS, T vE, T vx, T vy, T vz,
                                             const AdjConst<T>& c, PUT put) {
    const T nuS = c.om * aS, nuE = c.om * vE;
#pragma unroll
    for (int i = 0; i < 19; ++i) put(i, i, c.omw * muf[i] + nuS);
    put(19, 0, c.omw * mug[0] + nuE);
    const T pm[9] = {vx, vy, vz, vx + vy, vx - vy, vx + vz, vx - vz, vy + vz, vy - vz};
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const T t = c.om * c.c_l * pm[p];
        put(20 + 2 * p, 2 * p + 1, c.omw * mug[2 * p + 1] + nuE + t);
        put(21 + 2 * p, 2 * p + 2, c.omw * mug[2 * p + 2] + nuE - t);
    }
}

// ---------------------------------------------------------------------------
// The same per-cell mathematics in binary64 with fewer FP64 instructions
// (the FP64 pipe bounds the FP64 adjoint):
//  * the square root and the reciprocals 1/D, 1/(1 - b2), 1/s from binary32
//    seeds and two Newton steps each (the forward step's recovery), 1/D and
//    1/s computed once for the recovery and its adjoint;
//  * the per-run products of 1/c_l, the weights and omega folded (AdjConst);
//    the weighted pair sums are carried times 36 (weights 2 and 1), the
//    1/36 folded into their coefficients;
//  * the pair sums that depend on beta formed from beta-free moments of mu:
//    with q_p = e_p . beta,
//      Sdq = sum w delta_p q_p = beta . Vd,     Vd = sum w delta_p e_p,
//      Vq  = sum w sigma_p q_p e_p = T beta,    T  = sum w sigma_p e_p e_p^T,
//      Sq2 = sum w sigma_p q_p^2 = beta . Vq.
// ---------------------------------------------------------------------------

// x = 1/a from a binary32 seed and two Newton steps
__device__ __forceinline__ double rcp_newton(double a) {
    double x = rcp_seed(a);
    x = fma(x, fma(-a, x, 1.0), x);
    return fma(x, fma(-a, x, 1.0), x);
}

// 36 sum w s_p (36 w = 2 for the axis pairs, 1 for the diagonal ones)
__device__ __forceinline__ double wsum9(const double* s) {
    return fma(2.0, (s[0] + s[1]) + s[2], ((s[3] + s[4]) + (s[5] + s[6])) + (s[7] + s[8]));
}
// 36 sum w d_p e_p (three components)
__device__ __forceinline__ void wvec9(const double* d, double& vx, double& vy, double& vz) {
    vx = fma(2.0, d[0], (d[3] + d[4]) + (d[5] + d[6]));
    vy = fma(2.0, d[1], (d[3] - d[4]) + (d[7] + d[8]));
    vz = fma(2.0, d[2], (d[5] - d[6]) + (d[7] - d[8]));
}

__device__ __forceinline__ void cell_g64(const double* h, const double* mug, const AdjConst<double>& c,
                                         CellG<double>& r) {
    const double E = sum19(h);
    double dd[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) dd[p] = h[2 * p + 1] - h[2 * p + 2];
    double dx, dy, dz;  // M / c_l
    dx = dd[0] + dd[3] + dd[4] + dd[5] + dd[6];
    dy = dd[1] + dd[3] - dd[4] + dd[7] + dd[8];
    dz = dd[2] + dd[5] - dd[6] + dd[7] - dd[8];
    const double m2 = fma(dx, dx, fma(dy, dy, dz * dz));
    const double disc = fma(4.0 * E, E, c.m3cl2 * m2);  // 4 E^2 - 3 M^2
    double ys, hs;
    rsqrt_seed(disc, ys, hs);
    double sq = disc * ys;
    sq = fma(fma(-sq, sq, disc), hs, sq);
    sq = fma(fma(-sq, sq, disc), hs, sq);
    const double eps = sq - E;
    const double D = fma(3.0, E, eps);
    const double rD = rcp_newton(D);
    const double r3 = c.three_cl * rD;  // beta = 3 M / D
    const double bx = dx * r3, by = dy * r3, bz = dz * r3;
    const double b2 = (r3 * r3) * m2;
    const double gam2 = rcp_newton(1.0 - b2);
    // beta-free moments of mu_g (all times 36)
    double sg[9], dg[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        sg[p] = mug[2 * p + 1] + mug[2 * p + 2];
        dg[p] = mug[2 * p + 1] - mug[2 * p + 2];
    }
    const double s34 = sg[3] + sg[4], s56 = sg[5] + sg[6], s78 = sg[7] + sg[8];
    const double S1 = fma(2.0, (sg[0] + sg[1]) + sg[2], (s34 + s56) + s78);
    const double Txx = fma(2.0, sg[0], s34 + s56);
    const double Tyy = fma(2.0, sg[1], s34 + s78);
    const double Tzz = fma(2.0, sg[2], s56 + s78);
    const double Txy = sg[3] - sg[4], Txz = sg[5] - sg[6], Tyz = sg[7] - sg[8];
    double Vdx, Vdy, Vdz;
    wvec9(dg, Vdx, Vdy, Vdz);
    const double Vqx = fma(Txx, bx, fma(Txy, by, Txz * bz));
    const double Vqy = fma(Txy, bx, fma(Tyy, by, Tyz * bz));
    const double Vqz = fma(Txz, bx, fma(Tyz, by, Tzz * bz));
    const double Sq2 = fma(Vqx, bx, fma(Vqy, by, Vqz * bz));
    const double Sdq = fma(Vdx, bx, fma(Vdy, by, Vdz * bz));
    // the coefficients (Eqs. equil2as/equil2bs and their derivatives), the
    // 1/36 of the sums folded into them
    const double eg = eps * gam2, egb2 = eg * b2;
    const double m0 = mug[0], w0m0 = kW0 * m0;
    const double k1 = fma(-2.0, egb2, eps) * c.i2_36, k2 = eg * c.c6_36, k3 = eg * c.c4_36;
    const double geq0 = fma(eg, c.g0_eg, fma(eps, c.g0_e, egb2 * c.g0_egb2));
    r.tacc = dot19(mug, h) - fma(m0, geq0, fma(k1, S1, fma(k2, Sq2, k3 * Sdq)));
    const double SA = fma(c.c6_36, Sq2, fma(-c.c2_36 * b2, S1, c.c4_36 * Sdq));  // SYM + ASY
    const double t4 = fma(-c.c2, b2, 4.0);                                          // 4 - 2 b2 / c_l^2
    r.ae = fma(c.i2_36, S1, fma(gam2, SA, w0m0 * fma(gam2, t4, -c.c2p1)));
    const double gg2 = fma(w0m0, t4, SA);
    const double gb2 = -(c.c2 * gam2) * fma(S1, 1.0 / 36.0, w0m0);
    const double rad = (2.0 * eps) * fma(gam2 * gam2, gg2, gb2);
    const double cq = eg * c.c12_36;  // the Vd coefficient is k3
    r.gbx = fma(cq, Vqx, fma(k3, Vdx, rad * bx));
    r.gby = fma(cq, Vqy, fma(k3, Vdy, rad * by));
    r.gbz = fma(cq, Vqz, fma(k3, Vdz, rad * bz));
    r.mx = dx;
    r.my = dy;
    r.mz = dz;
    r.Et = E;
    r.sqt = sq;
    r.Dt = D;
    r.rD = rD;
    r.rs = rcp_newton(sq);
    r.bx = bx;
    r.by = by;
    r.bz = bz;
}

__device__ __forceinline__ void cell_f64(const double* h, const double* muf, const CellG<double>& r,
                                         const AdjConst<double>& c, double& tacc, double& aS, double& fbx,
                                         double& fby, double& fbz) {
    const double dS = sum19(h);
    double sf[9], df[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        sf[p] = muf[2 * p + 1] + muf[2 * p + 2];
        df[p] = muf[2 * p + 1] - muf[2 * p + 2];
    }
    const double F1 = wsum9(sf);  // sums times 36
    double Vx, Vy, Vz;
    wvec9(df, Vx, Vy, Vz);
    const double Fdq = fma(Vx, r.bx, fma(Vy, r.by, Vz * r.bz));
    const double fa = c.c3_36 * dS;  // (3 S / c_l) / 36
    // f^eq_{+-p} = w_p (S +- 3 S q_p / c_l)
    tacc = dot19(muf, h) - fma(kW0 * muf[0], dS, fma(dS * (1.0 / 36.0), F1, fa * Fdq));
    aS = fma(F1, 1.0 / 36.0, fma(c.c3_36, Fdq, kW0 * muf[0]));
    fbx = fa * Vx;
    fby = fa * Vy;
    fbz = fa * Vz;
}

// recovery_adjoint with 1/D and 1/s given and d = M / c_l
__device__ __forceinline__ void recovery_adjoint64(double a_eps, double abx, double aby, double abz,
                                                   const CellG<double>& r, const AdjConst<double>& c, double& vE,
                                                   double& vx, double& vy, double& vz) {
    const double abD = fma(abx, r.bx, fma(aby, r.by, abz * r.bz)) * r.rD;
    const double depsdE = fma(4.0 * r.Et, r.rs, -1.0);
    vE = fma(a_eps, depsdE, -abD * (3.0 + depsdE));
    const double cc = (c.three_cl * r.rs) * (abD - a_eps);  // 3 (ab.beta / D - a_eps) / s, times c_l
    const double rD3 = 3.0 * r.rD;
    vx = fma(cc, r.mx, abx * rD3);
    vy = fma(cc, r.my, aby * rD3);
    vz = fma(cc, r.mz, abz * rD3);
}

template <typename PUT>
__device__ __forceinline__ void scatter_cell64(const double* muf, const double* mug, double aS, double vE, double vx,
                                               double vy, double vz, const AdjConst<double>& c, PUT put) {
    const double nuS = c.om * aS, nuE = c.om * vE;
#pragma unroll
    for (int i = 0; i < 19; ++i) put(i, i, fma(c.omw, muf[i], nuS));
    put(19, 0, fma(c.omw, mug[0], nuE));
    const double ux = c.om_cl * vx, uy = c.om_cl * vy, uz = c.om_cl * vz;
    const double t[9] = {ux, uy, uz, ux + uy, ux - uy, ux + uz, ux - uz, uy + uz, uy - uz};
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        put(20 + 2 * p, 2 * p + 1, fma(c.omw, mug[2 * p + 1], nuE) + t[p]);
        put(21 + 2 * p, 2 * p + 2, fma(c.omw, mug[2 * p + 2], nuE) - t[p]);
    }
}

// A ghost plane cell (non-periodic x): nobody reads its populations that do
// not point into the lattice; the others are written by the scatter of x +- 1.
// At the inflow plane (held at eq(n_in, eps_in, beta_in)) its adjoint adds
// lambda_{t+1} . d eq_in / d beta_in (a per-context table).
// TERMS = false: only the zeros (the dL/dbeta_in terms taken elsewhere).
template <typename T, int XBC, bool TERMS = true>
__device__ __forceinline__ void ghost_cell(int x, int idx, long long S, const T* __restrict__ A,
                                           const T* __restrict__ Lin, T* __restrict__ Lout,
                                           const T* __restrict__ inflow_t, double& bin0, double& bin1,
                                           double& bin2, bool& has_b) {
    const int inward = (x == 0) ? 1 : -1;
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        if (vel_x(i) != inward) {
            Lout[RLB_CHK(i * S + idx, 38ll * S)] = (T)0;
            Lout[RLB_CHK((19 + i) * S + idx, 38ll * S)] = (T)0;
        }
    }
    if (TERMS && XBC == XBC_INFLOW_OUTFLOW && x == 0 && !is_solid(A[RLB_CHK(idx, 38ll * S)])) {
        T a0 = 0, a1 = 0, a2 = 0;
#pragma unroll 2
        for (int q = 0; q < 38; ++q) {
            const T l = Lin[RLB_CHK(q * S + idx, 38ll * S)];
            a0 += l * inflow_t[3 * q + 0];
            a1 += l * inflow_t[3 * q + 1];
            a2 += l * inflow_t[3 * q + 2];
        }
        bin0 += (double)a0;
        bin1 += (double)a1;
        bin2 += (double)a2;
        has_b = true;
    }
}

// Populations of x that a ghost plane would pull: nobody reads them.
template <typename T, int XBC>
__device__ __forceinline__ void zero_to_ghost(int x, int nx, int idx, long long S, T* __restrict__ Lout) {
    if (XBC != XBC_PERIODIC && (x == 1 || x == nx - 2)) {
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const bool to_ghost = (x == 1 && vel_x(i) == -1) || (x == nx - 2 && vel_x(i) == 1);
            if (to_ghost) {
                Lout[RLB_CHK(i * S + idx, 38ll * S)] = (T)0;
                Lout[RLB_CHK((19 + i) * S + idx, 38ll * S)] = (T)0;
            }
        }
    }
}

// Register kernel.  PIPE: persistent grid-stride loop over the cells;
// otherwise one cell per thread.
template <typename T, int XBC, int MINB, bool PIPE>
__global__ void __launch_bounds__(128, MINB)
    k_adjoint_step(const T* __restrict__ A, const T* __restrict__ Lin, T* __restrict__ Lout, Geom g, Phys ph,
                   AdjConst<T> c, const AdjSums sums, const T* __restrict__ inflow_t) {
    const long long S = g.S;
    T tau_acc = 0;
    double bin0 = 0.0, bin1 = 0.0, bin2 = 0.0;
    bool has_b = false;
    const long long stride = PIPE ? (long long)gridDim.x * blockDim.x : (long long)g.N;
    // the loop ends for every thread before the warp reduction ('continue'
    // skips to the next cell); the counter is 64-bit so that the last
    // stride cannot wrap
    for (long long li = (long long)blockIdx.x * blockDim.x + threadIdx.x; li < g.N; li += stride) {
        const int idx = (int)li;
        int x, y, z;
        cell_coords(g, idx, x, y, z);
        if constexpr (sizeof(T) == 8 && XBC == XBC_INFLOW_OUTFLOW) {
            // dL/dbeta_in at the fluid inflow ghosts of this warp, their 38
            // products with the table spread over the active lanes (one lane
            // issuing all 114 would take a full FP64 warp slot for each)
            const unsigned act = __activemask();
            unsigned m = __ballot_sync(act, x == 0 && !is_solid(A[RLB_CHK(idx, 38ll * S)]));
            if (m) {
                const int lane = threadIdx.x & 31;
                const int rank = __popc(act & ((1u << lane) - 1u)), cnt = __popc(act);
                while (m) {
                    const int src = __ffs(m) - 1;
                    m &= m - 1;
                    const int gidx = __shfl_sync(act, idx, src);
                    for (int q = rank; q < 38; q += cnt) {
                        const T l = Lin[RLB_CHK((long long)q * S + gidx, 38ll * S)];
                        bin0 = fma(l, inflow_t[3 * q + 0], bin0);
                        bin1 = fma(l, inflow_t[3 * q + 1], bin1);
                        bin2 = fma(l, inflow_t[3 * q + 2], bin2);
                    }
                    has_b = true;
                }
            }
        }
        if ((XBC != XBC_PERIODIC) && (x == 0 || x == g.nx - 1)) {
            if constexpr (sizeof(T) == 8 && XBC == XBC_INFLOW_OUTFLOW)
                ghost_cell<T, XBC, false>(x, idx, S, A, Lin, Lout, inflow_t, bin0, bin1, bin2, has_b);
            else
                ghost_cell<T, XBC>(x, idx, S, A, Lin, Lout, inflow_t, bin0, bin1, bin2, has_b);
            continue;
        }
        if (is_solid(A[RLB_CHK(19 * S + idx, 38ll * S)])) {  // never updated: identity
#pragma unroll
            for (int q = 0; q < 38; ++q) Lout[RLB_CHK(q * S + idx, 38ll * S)] = Lin[RLB_CHK(q * S + idx, 38ll * S)];
            continue;
        }
        const PullOffsets o(g, x, y, z);
        // mu = lambda_{t+1}(x), plus the outflow ghost that copies x
        const int dup = dup_of<XBC>(x, g.nx);
        // rare cases (a cell copied by an outflow ghost, links to solid cells)
        // take branches, so the common cell runs straight-line loads/stores
        auto load_mu = [&](T* mu, int base) {
#pragma unroll
            for (int i = 0; i < 19; ++i) mu[i] = Lin[RLB_CHK((base + i) * S + idx, 38ll * S)];
            if (dup) {
#pragma unroll
                for (int i = 0; i < 19; ++i) mu[i] += Lin[RLB_CHK((base + i) * S + idx + dup, 38ll * S)];
                if (dup_both<XBC>(g.nx)) {
#pragma unroll
                    for (int i = 0; i < 19; ++i) mu[i] += Lin[RLB_CHK((base + i) * S + idx - 1, 38ll * S)];
                }
            }
        };
        if (!PIPE) {
            // f-phase populations and adjoints: start their trip from HBM into L2 now
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                asm volatile("prefetch.global.L2 [%0];" ::"l"(RLB_CHK_PTR(A, i * S + idx + o.src(i), 38ll * S)));
                asm volatile("prefetch.global.L2 [%0];" ::"l"(RLB_CHK_PTR(Lin, i * S + idx, 38ll * S)));
            }
        }
        // ---- g phase: gather, moments, recovery, g part of the adjoint
        unsigned bounced = 0u;
        T h[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) h[i] = A[RLB_CHK((19 + i) * S + idx + o.src(i), 38ll * S)];
        {
            // a pulled solid marker is a NaN: test the per-value markers only
            // when the sum of the gathered values is NaN
            if (isnan(sum19(h))) {
#pragma unroll
                for (int i = 1; i < 19; ++i) {
                    if (is_solid(h[i])) {
                        bounced |= 1u << i;
                        h[i] = A[RLB_CHK((19 + opp(i)) * S + idx, 38ll * S)];
                    }
                }
            }
        }
        T mug[19];
        load_mu(mug, 19);
        CellG<T> r;
        if constexpr (sizeof(T) == 8)
            cell_g64(h, mug, c, r);
        else
            cell_g(h, mug, c, r);
        // ---- f phase
#pragma unroll
        for (int i = 0; i < 19; ++i) h[i] = A[RLB_CHK(i * S + idx + o.src(i), 38ll * S)];
        if (bounced) {
#pragma unroll
            for (int i = 1; i < 19; ++i)
                if ((bounced >> i) & 1u) h[i] = A[RLB_CHK(opp(i) * S + idx, 38ll * S)];
        }
        T muf[19];
        load_mu(muf, 0);
        T tf, aS, fbx, fby, fbz;
        if constexpr (sizeof(T) == 8)
            cell_f64(h, muf, r, c, tf, aS, fbx, fby, fbz);
        else
            cell_f(h, muf, r, c, tf, aS, fbx, fby, fbz);
        tau_acc += (r.tacc + tf) * c.inv_tau2_t;
        T vE, vx, vy, vz;
        if constexpr (sizeof(T) == 8)
            recovery_adjoint64(r.ae, fbx + r.gbx, fby + r.gby, fbz + r.gbz, r, c, vE, vx, vy, vz);
        else
            recovery_adjoint<T>(r.ae, fbx + r.gbx, fby + r.gby, fbz + r.gbz, r.Et, r.sqt, r.Dt, r.bx, r.by, r.bz,
                                r.mx, r.my, r.mz, vE, vx, vy, vz);
        auto put = [&](int q, int i, T v) {
            if ((bounced >> i) & 1u)
                Lout[RLB_CHK((q - i + opp(i)) * S + idx, 38ll * S)] = v;
            else
                Lout[RLB_CHK(q * S + idx + o.src(i), 38ll * S)] = v;
        };
        if constexpr (sizeof(T) == 8)
            scatter_cell64(muf, mug, aS, vE, vx, vy, vz, c, put);
        else
            scatter_cell(muf, mug, aS, vE, vx, vy, vz, c, put);
        zero_to_ghost<T, XBC>(x, g.nx, idx, S, Lout);
    }
    if constexpr (PIPE)
        block_sums<T, XBC == XBC_INFLOW_OUTFLOW>((double)tau_acc, bin0, bin1, bin2, has_b, sums);
    else
        warp_partials<T>((double)tau_acc, bin0, bin1, bin2, has_b, sums.red);
}

// ---------------------------------------------------------------------------
// FP64 step adjoint with its sums in 64-bit fixed point (rlb_fixed.cuh),
// lattice speeds 1 <= c_l <= 2.
//
// With d = M / c_l, D = 2 E + s, s = sqrt(4 E^2 - 3 M^2), u = d / D and the
// equilibria written as in rlb_fixed.cuh, mu enters through integer moments
// (weights times 36): S1 = sum w sigma_p, T = sum w sigma_p e_p e_p^T,
// V = sum w delta_p e_p over the g pairs, F1 and F likewise over the f pairs:
//   G     = 13.5 T + (1.5 w0 mu_0 - 7.5 S1) I,     y = G u,
//   a_E   = S1 / c_l^2 + w0 mu_0 (3 - 2 / c_l^2),
//   a_S   = w0 mu_f0 + F1 + 9 F.u,
//   a_D   = -(u.y + 9 (S / D) F.u),
//   v_E   = a_E + a_D (2 + 4 E / s),
//   v_d   = 2 y + 3 V + 9 (S / D) F - 3 c_l^2 (a_D / s) d,
//   nu_f  = (1 - omega) mu_f + omega a_S,
//   nu_g  = (1 - omega) mu_g + omega (v_E + e_i.v_d),
//   sum mu eq = S a_S + E a_E + D u.y + 3 V.d,
// no gamma^2, 1 / (1 - b2) or weights per population.  sum mu h is an integer
// dot product.
//
// k_adjoint_step<double> (the other lattice speeds) issues 408 FP64
// instructions per collided cell, 26,500 clocks of a scheduler's FP64 pipe per
// 32 cells, against 5,400 for the cell's 912 bytes at the HBM rate; here 118
// remain (80 for recovery and algebra, 38 relaxations) beside 6,624
// instructions in all.  What bounds it now is the speed of a warp: with 12
// warps per SM 41 % of the issue slots and 45 % of the FP64 pipe are used, the
// rest being instruction latency and fetch.  mu and the gathered populations
// are staged in a shared-memory column per thread by asynchronous copies, so
// that they hold no registers, and the velocity pairs are walked in three
// rounds by one loop body (a third of the code to fetch).  200x100x100 sphere
// 1.51 -> 0.86 ms.  (Before the rounding below, 0.83 ms there and 2.35 on the
// 192^3 box, 5.1 in binary64; blocks of 64 threads: 5, 6 and 7 per SM 2.65, 2.35
// and 2.49 ms; all values in registers and unrolled, 3 blocks of 128: 2.35 ms on
// the box, 0.854 on the sphere.)
//
// Error against 113-bit references (1.5e6 cells, |beta_a| up to 0.5, lambda
// normal): nu 0.9e-16 rms, the terms of dL/dtau 1.1e-16 (binary64 5.5e-16 and
// 3.0e-16).  What the sum over the lattice, or over many steps, sees is their
// mean: of a term -5e-20 +- 9e-20 for lambda of zero mean (binary64 -3e-20 +-
// 2e-19), -3e-19 for binary32 lambda, -9e-19 for lambda of one sign (5.2e-17);
// of a value of nu next to an outflow plane 1e-18 of the largest.  That takes
// ties to even or balanced, weights rounded, and the products of the low halves
// themselves: with ties up, floors and a mean product they were -2.6e-18,
// +6.7e-17, -1.5e-17 and 2.4e-17 (0.83 ms on the sphere).
// ---------------------------------------------------------------------------

struct AdjFx {
    FxConst kS1;  // 5 / 3                        x 2^62
    FxConst kE1;  // 1 / (36 c_l^2)               x 2^65
    FxConst kE0;  // (3 - 2 / c_l^2) / 3          x 2^62
    FxConst kS36;  // 1 / 36                      x 2^65
};

// 2^k, |k| <= 1022
__device__ __forceinline__ double pow2d(int k) { return fx_double((uint32_t)(1023 + k) << 20, 0u); }
// k such that the largest of N values times 2^k is of order one (non-finite
// values: 0)
template <int N>
__device__ __forceinline__ int unit_shift(const double* v) {
    const int e = fx_max_exponent<N>(v);
    return e == 0x7FF ? 0 : max(-1022, min(1022, 1023 - e));
}

// A cell in binary64 throughout (any state); the terms of dL/dtau returned.
// lambda_t is linear in lambda and does not depend on the unit of the state,
// so both are brought to order one first (exactly, by powers of two): products
// of states of 1e-80 with lambda of 1e-240 lose no bits on the way.
template <int XBC>
__device__ __noinline__ double adjoint_cell_general(const double* A, const double* Lin, double* Lout, const Geom& g,
                                                    const AdjConst<double>& c, int idx) {
    const long long S = g.S;
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    const PullOffsets o(g, x, y, z);
    const int dup = dup_of<XBC>(x, g.nx);
    double h[19], mu[38];
    double *const muf = mu, *const mug = mu + 19;
    for (int q = 0; q < 38; ++q) mu[q] = Lin[RLB_CHK(q * S + idx, 38ll * S)];
    if (dup) {
        for (int q = 0; q < 38; ++q) mu[q] += Lin[RLB_CHK(q * S + idx + dup, 38ll * S)];
        if (dup_both<XBC>(g.nx))
            for (int q = 0; q < 38; ++q) mu[q] += Lin[RLB_CHK(q * S + idx - 1, 38ll * S)];
    }
    const int kl = unit_shift<38>(mu);
    for (int q = 0; q < 38; ++q) mu[q] *= pow2d(kl);
    unsigned bounced = 0u;
#pragma unroll
    for (int i = 0; i < 19; ++i) h[i] = A[RLB_CHK((19 + i) * S + idx + o.src(i), 38ll * S)];
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        if (is_solid(h[i])) {
            bounced |= 1u << i;
            h[i] = A[RLB_CHK((19 + opp(i)) * S + idx, 38ll * S)];
        }
    }
    const int kh = unit_shift<19>(h);
    for (int i = 0; i < 19; ++i) h[i] *= pow2d(kh);
    CellG<double> r;
    cell_g64(h, mug, c, r);
#pragma unroll
    for (int i = 0; i < 19; ++i)
        h[i] = ((bounced >> i) & 1u ? A[RLB_CHK(opp(i) * S + idx, 38ll * S)] : A[RLB_CHK(i * S + idx + o.src(i), 38ll * S)]) * pow2d(kh);
    double tf, aS, fbx, fby, fbz, vE, vx, vy, vz;
    cell_f64(h, muf, r, c, tf, aS, fbx, fby, fbz);
    recovery_adjoint64(r.ae, fbx + r.gbx, fby + r.gby, fbz + r.gbz, r, c, vE, vx, vy, vz);
    scatter_cell64(muf, mug, aS, vE, vx, vy, vz, c, [&](int q, int i, double v) {
        v *= pow2d(-kl);
        if ((bounced >> i) & 1u)
            Lout[RLB_CHK((q - i + opp(i)) * S + idx, 38ll * S)] = v;
        else
            Lout[RLB_CHK(q * S + idx + o.src(i), 38ll * S)] = v;
    });
    return (r.tacc + tf) * c.inv_tau2 * pow2d(-kh) * pow2d(-kl);
}

// Whether products of values with block exponents ea and eb can be formed by
// fx_to (sum mu h, units 2^(ea + eb - 2102)), whose result has to be a normal
// number: otherwise (states of 1e-80 with lambda of 1e-230) the exponent would
// wrap into the sign, and the cell is left to the binary64 form.
__device__ __forceinline__ bool dot_in_range(int ea, int eb) { return (unsigned)(ea + eb - 1080) <= 1982u; }

// What the f phase and the output need of a cell (see the formulas above).
struct AdjFxCell {
    double x, y, z, E4, rs, rD, ux, uy, uz, yx, yy, yz, uy_, vx, vy, vz, aE;  // d, 4 E, 1/s, 1/D, u, G u, u.y, 36 V, a_E
    double tsum;                      // sum mu (h - eq)
    double nuE, nuS, tx, ty, tz;      // omega v_E, omega a_S, omega v_d
};

// Recovery and the g moments of mu in binary64 (ties to even throughout: sums
// of equal values, as of lambda next to a boundary, meet them often, and an
// error that every step repeats adds up in lambda).  S*, P*, T*: the sums of
// sigma_p over the axis pairs (doubled), and over each plane's two diagonal
// pairs and their difference; units 2^-56 of the block exponents eh, em.
__device__ __forceinline__ void adj_fx_g(int64_t E, int64_t dx, int64_t dy, int64_t dz, int64_t dot, int64_t m0, int64_t Sx,
                                         int64_t Sy, int64_t Sz, int64_t Pxy, int64_t Pyz, int64_t Pzx, int64_t Txy,
                                         int64_t Tyz, int64_t Tzx, int64_t Vx, int64_t Vy, int64_t Vz, int eh, int em,
                                         const Phys& ph, const AdjFx& k, AdjFxCell& t) {
    const int kh = eh - 1079, km = em - 1079;
    const double Ed = fx_to_even(E, kh);
    t.x = fx_to_even(dx, kh), t.y = fx_to_even(dy, kh), t.z = fx_to_even(dz, kh);
    const double E2 = Ed + Ed;
    t.E4 = E2 + E2;
    const double dd = fma(t.x, t.x, fma(t.y, t.y, t.z * t.z));
    const double disc = fma(ph.fx.m3cl2, dd, E2 * E2);
    double ys, hs;
    rsqrt_seed(disc, ys, hs);
    double sq = disc * ys;
    sq = fma(fma(-sq, sq, disc), hs, sq);
    sq = fma(fma(-sq, sq, disc), hs, sq);
    const double e1 = fma(-sq, ys, 1.0);
    t.rs = fma(ys, fma(e1, e1, e1), ys);
    const double D = E2 + sq;
    const double r0 = rcp_seed(D);
    const double e2 = fma(-D, r0, 1.0);
    t.rD = fma(r0, fma(e2, e2, e2), r0);
    t.ux = t.x * t.rD, t.uy = t.y * t.rD, t.uz = t.z * t.rD;
    const int64_t sp = (Sx + Sy + Sz) + (Pxy + Pyz + Pzx);
    // 8 G: 13.5 / 36 = 3/8; the partial sums may wrap, the result does not
    const int64_t kap = (m0 << 2) - (fx_mul_exact(sp, k.kS1) << 2);
    auto g38 = [](int64_t v, int64_t k8) { return fx_weight_signed(fx_round3_even(v + (v << 1) + k8)); };
    auto g38_off = [](int64_t v) { return fx_weight_signed((v + (v << 1) + 4) >> 3); };  // u_a u_b has either sign
    const double Gxx = fx_to_even(g38(Sx + Pxy + Pzx, kap), km), Gyy = fx_to_even(g38(Sy + Pxy + Pyz, kap), km),
                 Gzz = fx_to_even(g38(Sz + Pyz + Pzx, kap), km);
    const double Gxy = fx_to_even(g38_off(Txy), km), Gxz = fx_to_even(g38_off(Tzx), km), Gyz = fx_to_even(g38_off(Tyz), km);
    t.yx = fma(Gxx, t.ux, fma(Gxy, t.uy, Gxz * t.uz));
    t.yy = fma(Gxy, t.ux, fma(Gyy, t.uy, Gyz * t.uz));
    t.yz = fma(Gxz, t.ux, fma(Gyz, t.uy, Gzz * t.uz));
    t.aE = fx_to_even(fx_mul_exact(sp, k.kE1) + fx_mul_exact(m0 << 3, k.kE0), km - 1);
    t.uy_ = fma(t.ux, t.yx, fma(t.uy, t.yy, t.uz * t.yz));
    t.vx = fx_to_even(Vx, km), t.vy = fx_to_even(Vy, km), t.vz = fx_to_even(Vz, km);
    const double Vd = fma(t.vx, t.x, fma(t.vy, t.y, t.vz * t.z));
    t.tsum = fx_to_even(dot, em + eh - 2102) - fma(Ed, t.aE, fma(D, t.uy_, Vd * (1.0 / 12.0)));
}

// The f moments (36 w0 mu_f0 + F1 and F times 36, S, the dot product) and the
// coefficients of the output.
__device__ __forceinline__ void adj_fx_f(int64_t Sf, int64_t fd, int64_t Fs, int64_t Fx, int64_t Fy, int64_t Fz, int fh,
                                         int ef, const Phys& ph, const AdjFx& k, AdjFxCell& t) {
    const double Sd = fx_to_even(Sf, fh - 1079);
    const int kf = ef - 1079;
    const double fx = fx_to_even(fx_weight_signed(Fx), kf), fy = fx_to_even(fx_weight_signed(Fy), kf), fz = fx_to_even(fx_weight_signed(Fz), kf);
    const double Fu = fma(fx, t.ux, fma(fy, t.uy, fz * t.uz));
    const double aS = fma(0.25, Fu, fx_to_even(fx_mul_exact(Fs, k.kS36), kf - 1));
    t.tsum += fx_to_even(fd, ef + fh - 2102) - Sd * aS;
    const double sD = (0.25 * Sd) * t.rD;
    const double aD = -fma(sD, Fu, t.uy_);
    t.nuE = ph.omega * fma(aD, fma(t.E4, t.rs, 2.0), t.aE);
    t.nuS = ph.omega * aS;
    const double c2 = (ph.fx.m3cl2 * t.rs) * aD;
    t.tx = ph.omega * fma(2.0, t.yx, fma(t.vx, 1.0 / 12.0, fma(sD, fx, c2 * t.x)));
    t.ty = ph.omega * fma(2.0, t.yy, fma(t.vy, 1.0 / 12.0, fma(sD, fy, c2 * t.y)));
    t.tz = ph.omega * fma(2.0, t.yz, fma(t.vz, 1.0 / 12.0, fma(sD, fz, c2 * t.z)));
}

// The 18 moving velocities as three rounds r = 0, 1, 2 over the axes
// (a, b) = (x, y), (y, z), (z, x): the axis pair of a and the two diagonal
// pairs of the plane (a, b).  Velocity numbers of a round: +-a at ax, ax + 1;
// (+,+) and (-,-) at pp, pp + 1; (+,-) at pm and (-,+) at mp.
struct Round {
    int ax, pp, pm, mp;
    __device__ __forceinline__ explicit Round(int r)
        : ax(1 + 2 * r), pp((0x0B0F07 >> (8 * r)) & 0xFF), pm((0x0E1109 >> (8 * r)) & 0xFF),
          mp((0x0D120A >> (8 * r)) & 0xFF) {}
};
__device__ __forceinline__ int opp_rt(int i) { return ((i - 1) ^ 1) + 1; }  // i > 0
template <typename V>
__device__ __forceinline__ void rotate3(V& a, V& b, V& c) {
    const V t = a;
    a = b;
    b = c;
    c = t;
}

constexpr int kAdjFxThreads = 64;  // threads per block (columns of the staging area)
constexpr int kAdjFxBlocks = 6;    // resident blocks per SM

template <int XBC>
__global__ void __launch_bounds__(kAdjFxThreads, kAdjFxBlocks)
    k_adjoint_step_fx(const double* __restrict__ A, const double* __restrict__ Lin, double* __restrict__ Lout,
                      const __grid_constant__ Geom g, const __grid_constant__ Phys ph,
                      const __grid_constant__ AdjConst<double> c, const __grid_constant__ AdjFx k, const AdjSums sums,
                      const double* __restrict__ inflow_t) {
    const long long S = g.S;
    // This thread's column: mu_f (0..18), mu_g (19..37), then h_g and later
    // h_f (38..56).  No other thread reads it.
    __shared__ double col[57][kAdjFxThreads];
    const int tid = threadIdx.x;
    const uint32_t scol = (uint32_t)__cvta_generic_to_shared(&col[0][tid]);
    auto stage = [&](int slot, const double* p) { cp_async8(scol + (uint32_t)(slot * kAdjFxThreads * 8), p); };
    double tau_acc = 0;
    double bin0 = 0.0, bin1 = 0.0, bin2 = 0.0;
    bool has_b = false;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long li = dependent_begin(blockIdx.x * blockDim.x + tid); li < g.N; li += stride) {
        const int idx = (int)li;
        int x, y, z;
        cell_coords(g, idx, x, y, z);
        if constexpr (XBC == XBC_INFLOW_OUTFLOW) {
            // dL/dbeta_in at the fluid inflow ghosts of this warp, their 38
            // products with the table spread over the active lanes
            const unsigned act = __activemask();
            unsigned m = __ballot_sync(act, x == 0 && !is_solid(A[RLB_CHK(idx, 38ll * S)]));
            if (m) {
                const int lane = tid & 31;
                const int rank = __popc(act & ((1u << lane) - 1u)), cnt = __popc(act);
                while (m) {
                    const int src = __ffs(m) - 1;
                    m &= m - 1;
                    const int gidx = __shfl_sync(act, idx, src);
                    for (int q = rank; q < 38; q += cnt) {
                        const double l = Lin[RLB_CHK((long long)q * S + gidx, 38ll * S)];
                        bin0 = fma(l, inflow_t[3 * q + 0], bin0);
                        bin1 = fma(l, inflow_t[3 * q + 1], bin1);
                        bin2 = fma(l, inflow_t[3 * q + 2], bin2);
                    }
                    has_b = true;
                }
            }
        }
        if ((XBC != XBC_PERIODIC) && (x == 0 || x == g.nx - 1)) {
            const int inward = x == 0 ? 1 : -1;
#pragma unroll 1
            for (int i = 0; i < 19; ++i) {
                if (vel_x(i) != inward) {
                    Lout[RLB_CHK(i * S + idx, 38ll * S)] = 0.0;
                    Lout[RLB_CHK((19 + i) * S + idx, 38ll * S)] = 0.0;
                }
            }
            continue;
        }
        const PullOffsets o(g, x, y, z);
        const int dup = dup_of<XBC>(x, g.nx);
        const double* Ac = A + idx;
        const double* Lc = Lin + idx;
        // offsets of the sources x - e along the axes: minus and plus
        int am = o.xm, ap = o.xp, bm = o.ym, bp = o.yp, cm = o.zm, cp = o.zp;
        auto gather = [&](int base) {  // the 19 pulled populations of a set
            stage(38, Ac + RLB_CHK_OFF(base * S, idx, 38ll * S));
#pragma unroll 1
            for (int r = 0; r < 3; ++r) {
                const Round v(r);
                auto one = [&](int i, int off) { stage(38 + i, Ac + RLB_CHK_OFF((base + i) * S + off, idx, 38ll * S)); };
                one(v.ax, am);
                one(v.ax + 1, ap);
                one(v.pp, am + bm);
                one(v.pp + 1, ap + bp);
                one(v.pm, am + bp);
                one(v.mp, ap + bm);
                rotate3(am, bm, cm);
                rotate3(ap, bp, cp);
            }
        };
        gather(19);
#pragma unroll 1
        for (int q = 19; q < 38; ++q) stage(q, Lc + RLB_CHK_OFF(q * S, idx, 38ll * S));
        cp_async_commit();
#pragma unroll 1
        for (int q = 0; q < 19; ++q) stage(q, Lc + RLB_CHK_OFF(q * S, idx, 38ll * S));
        cp_async_commit();
        cp_async_wait<1>();
        if (is_solid(col[38][tid])) {  // never updated: identity
            cp_async_wait<0>();
#pragma unroll 1
            for (int q = 0; q < 38; ++q) Lout[RLB_CHK(q * S + idx, 38ll * S)] = col[q][tid];
            continue;
        }
        auto max_word = [&](int base) {
            uint32_t m = 0;
#pragma unroll 4
            for (int i = 0; i < 19; ++i) m = max(m, (uint32_t)__double2hiint(col[base + i][tid]) << 1);
            return m;
        };
        // mu also takes lambda of the outflow ghosts that copy x
        auto add_dup = [&](int base) {
            for (int off = dup;; off = -1) {
#pragma unroll 4
                for (int i = 0; i < 19; ++i) col[base + i][tid] += Lc[RLB_CHK_OFF((base + i) * S + off, idx, 38ll * S)];
                if (!dup_both<XBC>(g.nx) || off < 0) break;
            }
        };
        int eh = (int)(max_word(38) >> 21);
        unsigned bounced = 0u;
        if (eh == 0x7FF) {  // links to solid cells, or a non-finite population
#pragma unroll 1
            for (int i = 1; i < 19; ++i) {
                if (is_solid(col[38 + i][tid])) {
                    bounced |= 1u << i;
                    col[38 + i][tid] = Ac[RLB_CHK_OFF((19 + opp_rt(i)) * S, idx, 38ll * S)];
                }
            }
            eh = (int)(max_word(38) >> 21);
        }
        if (dup) add_dup(19);
        // ---- g: moments of h and mu, their dot product
        const int em = fx_block_exponent(max_word(19));
        bool ok = eh >= 600 && eh <= 1400 && em <= 1900 && dot_in_range(em, eh);  // E^2 in range
        int64_t E, dx = 0, dy = 0, dz = 0, m0;
        FxDot dot{};
        // moments of mu: axis sums, plane sums and differences (xy, yz, zx), V
        int64_t Sx = 0, Sy = 0, Sz = 0, Pxy = 0, Pyz = 0, Pzx = 0, Txy = 0, Tyz = 0, Tzx = 0, Vx = 0, Vy = 0, Vz = 0;
        {
            const int64_t h0 = fx_from(col[38][tid], eh), u0 = fx_from(col[19][tid], em);
            E = fx_round4(h0);
            m0 = fx_round4_even(u0);
            dot.add(h0, u0);
#pragma unroll 1
            for (int r = 0; r < 3; ++r) {
                const Round v(r);
                int64_t d, sg, dl;
                auto pair = [&](int i, int j, int half) {
                    const int64_t a = fx_from(col[38 + i][tid], eh), b = fx_from(col[38 + j][tid], eh);
                    const int64_t ua = fx_from(col[19 + i][tid], em), ub = fx_from(col[19 + j][tid], em);
                    E += fx_round4(a + b);
                    dot.add(a, ua);
                    dot.add(b, ub);
                    d = fx_round4(a - b);
                    sg = (ua + ub + half) >> 4;
                    dl = fx_round4(ua - ub);
                };
                pair(v.ax, v.ax + 1, 7);  // sigma's ties: down for the axis pairs, up for the others (weights 6 and 6)
                dx += d;
                Sx = sg << 1;
                Vx += dl << 1;
                pair(v.pp, v.pp + 1, 8);
                dx += d, dy += d;
                Vx += dl, Vy += dl;
                Pxy = sg, Txy = sg;
                pair(v.pm, v.mp, 8);
                dx += d, dy -= d;
                Vx += dl, Vy -= dl;
                Pxy += sg, Txy -= sg;
                rotate3(dx, dy, dz);
                rotate3(Sx, Sy, Sz);
                rotate3(Vx, Vy, Vz);
                rotate3(Pxy, Pyz, Pzx);
                rotate3(Txy, Tyz, Tzx);
            }
        }
        gather(0);  // the h_f slots: every h_g of this column has been read
        cp_async_commit();
        {
            const int32_t Eh = (int32_t)(E >> 32);
            const float Ef = (float)Eh, xf = (float)(int32_t)(dx >> 32), yf = (float)(int32_t)(dy >> 32),
                        zf = (float)(int32_t)(dz >> 32);
            ok = ok && Eh > 0 && fx_clz((uint32_t)Eh) <= 14 && xf * xf + yf * yf + zf * zf < ph.fx.m_max * (Ef * Ef);
        }
        if (!ok) {
            cp_async_wait<0>();
            tau_acc += adjoint_cell_general<XBC>(A, Lin, Lout, g, c, idx);
            zero_to_ghost<double, XBC>(x, g.nx, idx, S, Lout);
            continue;
        }
        AdjFxCell t;
        adj_fx_g(E, dx, dy, dz, dot.result(), m0, Sx, Sy, Sz, Pxy, Pyz, Pzx, Txy, Tyz, Tzx, Vx, Vy, Vz, eh, em, ph, k, t);
        // ---- f
        cp_async_wait<0>();
        if (bounced) {
#pragma unroll 1
            for (int i = 1; i < 19; ++i)
                if ((bounced >> i) & 1u) col[38 + i][tid] = Ac[RLB_CHK_OFF(opp_rt(i) * S, idx, 38ll * S)];
        }
        if (dup) add_dup(0);
        {
            const int fh = fx_block_exponent(max_word(38)), ef = fx_block_exponent(max_word(0));
            ok = fh <= 1900 && ef <= 1900 && dot_in_range(ef, fh);
            const int64_t h0 = fx_from(col[38][tid], fh), u0 = fx_from(col[0][tid], ef);
            int64_t Sf = fx_round4(h0);
            FxDot fd{};
            fd.add(h0, u0);
            const int64_t u4 = fx_round4_even(u0);
            int64_t Fs = (u4 << 3) + (u4 << 2);  // 36 w0 mu_f0
            int64_t Fx = 0, Fy = 0, Fz = 0;
#pragma unroll 1
            for (int r = 0; r < 3; ++r) {
                const Round v(r);
                int64_t sg, dl;
                auto pair = [&](int i, int j, int half) {
                    const int64_t a = fx_from(col[38 + i][tid], fh), b = fx_from(col[38 + j][tid], fh);
                    const int64_t ua = fx_from(col[i][tid], ef), ub = fx_from(col[j][tid], ef);
                    Sf += fx_round4(a + b);
                    fd.add(a, ua);
                    fd.add(b, ub);
                    sg = (ua + ub + half) >> 4;
                    dl = fx_round4(ua - ub);
                };
                pair(v.ax, v.ax + 1, 7);
                Fs += sg << 1;
                Fx += dl << 1;
                pair(v.pp, v.pp + 1, 8);
                Fs += sg;
                Fx += dl, Fy += dl;
                pair(v.pm, v.mp, 8);
                Fs += sg;
                Fx += dl, Fy -= dl;
                rotate3(Fx, Fy, Fz);
            }
            adj_fx_f(Sf, fd.result(), Fs, Fx, Fy, Fz, fh, ef, ph, k, t);
        }
        if (!ok) {
            tau_acc += adjoint_cell_general<XBC>(A, Lin, Lout, g, c, idx);
            zero_to_ghost<double, XBC>(x, g.nx, idx, S, Lout);
            continue;
        }
        tau_acc = fma(t.tsum, c.inv_tau2, tau_acc);
        // ---- nu = (1 - omega) mu + omega (...), scattered.  omega (v_E +
        // e_i.v_d) as integers of one exponent; values beyond its range are
        // non-finite, about to overflow (ek >= 1900) or about to underflow
        const double nuE = t.nuE, nuS = t.nuS, kv[4] = {t.nuE, t.tx, t.ty, t.tz};
        const int ek = fx_block_exponent(fx_max_word<4>(kv));
        if (ek >= 1900) {
            adjoint_cell_general<XBC>(A, Lin, Lout, g, c, idx);
            zero_to_ghost<double, XBC>(x, g.nx, idx, S, Lout);
            continue;
        }
        const int64_t kE = fx_from(nuE, ek);
        int64_t ka = fx_from(t.tx, ek), kb = fx_from(t.ty, ek), kc = fx_from(t.tz, ek);
        double* Lo = Lout + idx;
        Lo[RLB_CHK_OFF(0, idx, 38ll * S)] = fma(ph.fx.omw, col[0][tid], nuS);
        Lo[RLB_CHK_OFF(19 * S, idx, 38ll * S)] = fma(ph.fx.omw, col[19][tid], nuE);
#pragma unroll 1
        for (int r = 0; r < 3; ++r) {
            const Round v(r);
            auto put = [&](int i, int off, int64_t kt) {
                const bool back = (bounced >> i) & 1u;
                const long long at = (long long)(back ? opp_rt(i) : i) * S + (back ? 0 : off);
                Lo[RLB_CHK_OFF(at, idx, 38ll * S)] = fma(ph.fx.omw, col[i][tid], nuS);
                Lo[RLB_CHK_OFF(19 * S + at, idx, 38ll * S)] = fma(ph.fx.omw, col[19 + i][tid], fx_to_even(kt, ek - 1083));
            };
            put(v.ax, am, kE + ka);
            put(v.ax + 1, ap, kE - ka);
            put(v.pp, am + bm, kE + ka + kb);
            put(v.pp + 1, ap + bp, kE - ka - kb);
            put(v.pm, am + bp, kE + ka - kb);
            put(v.mp, ap + bm, kE - ka + kb);
            rotate3(ka, kb, kc);
            rotate3(am, bm, cm);
            rotate3(ap, bp, cp);
        }
        zero_to_ghost<double, XBC>(x, g.nx, idx, S, Lout);
    }
    block_sums<double, XBC == XBC_INFLOW_OUTFLOW>(tau_acc, bin0, bin1, bin2, has_b, sums);
}

// Eight lanes per cell (lattices of at most 32 cells per SM, two warps per
// scheduler, where a step takes the time of one warp's instructions: 1600
// cells 29 -> 21 us, 4800 cells 29 -> 23 us): lane j holds pair j, lane 0 also pair 8,
// lane 1 the rest populations; the sums are gathered by shuffles and the
// binary64 part is repeated on every lane.
template <int XBC>
__global__ void __launch_bounds__(128)
    k_adjoint_step_fx_split(const double* __restrict__ A, const double* __restrict__ Lin, double* __restrict__ Lout,
                            const __grid_constant__ Geom g, const __grid_constant__ Phys ph,
                            const __grid_constant__ AdjConst<double> c, const __grid_constant__ AdjFx k, const AdjSums sums,
                            const double* __restrict__ inflow_t) {
    const unsigned full = 0xffffffffu;
    const long long S = g.S;
    const int t8 = dependent_begin(blockIdx.x * blockDim.x + threadIdx.x);
    const int j = threadIdx.x & 7, base = threadIdx.x & 24;  // lane of the group, its first lane in the warp
    const bool live = (t8 >> 3) < g.N;
    const int idx = live ? (int)(t8 >> 3) : 0;
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    const bool ghost = XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1);
    const PullOffsets o(g, x, y, z);
    const int dup = dup_of<XBC>(x, g.nx);
    // this lane's velocities: 2j + 1, 2j + 2 and (lane 0) 17, 18 or (lane 1) 0
    const int iv[4] = {2 * j + 1, 2 * j + 2, j == 0 ? 17 : 0, 18};
    const int nv = j == 0 ? 4 : (j == 1 ? 3 : 2);
    double hf[4], hg[4], uf[4], ug[4];
    unsigned back = 0u;
    double tau_acc = 0.0, bin0 = 0.0, bin1 = 0.0, bin2 = 0.0;
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        hf[n] = hg[n] = uf[n] = ug[n] = 0.0;
        if (live && n < nv) {
            uf[n] = __ldg(Lin + RLB_CHK(iv[n] * S + idx, 38ll * S));
            ug[n] = __ldg(Lin + RLB_CHK((19 + iv[n]) * S + idx, 38ll * S));
            if (!ghost) {
                const int src = idx + o.src(iv[n]);
                hf[n] = __ldg(A + RLB_CHK(iv[n] * S + src, 38ll * S));
                hg[n] = __ldg(A + RLB_CHK((19 + iv[n]) * S + src, 38ll * S));
                if (dup) {
                    uf[n] += __ldg(Lin + RLB_CHK(iv[n] * S + idx + dup, 38ll * S));
                    ug[n] += __ldg(Lin + RLB_CHK((19 + iv[n]) * S + idx + dup, 38ll * S));
                    if (dup_both<XBC>(g.nx)) {
                        uf[n] += __ldg(Lin + RLB_CHK(iv[n] * S + idx - 1, 38ll * S));
                        ug[n] += __ldg(Lin + RLB_CHK((19 + iv[n]) * S + idx - 1, 38ll * S));
                    }
                }
            }
        }
    }
    const bool own_solid = j == 1 && is_solid(ghost ? __ldg(A + RLB_CHK(idx, 38ll * S)) : hf[2]);
    const bool solid = __shfl_sync(full, own_solid, base + 1);
    const bool work = live && !ghost && !solid;
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        if (work && n < nv && iv[n] > 0 && is_solid(hf[n])) {  // link bounce-back
            back |= 1u << n;
            hf[n] = __ldg(A + RLB_CHK(opp_rt(iv[n]) * S + idx, 38ll * S));
            hg[n] = __ldg(A + RLB_CHK((19 + opp_rt(iv[n])) * S + idx, 38ll * S));
        }
    }
    uint32_t wh = fx_max_word<4>(hg), wm = fx_max_word<4>(ug), vh = fx_max_word<4>(hf), vm = fx_max_word<4>(uf);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        wh = max(wh, __shfl_xor_sync(full, wh, off));
        wm = max(wm, __shfl_xor_sync(full, wm, off));
        vh = max(vh, __shfl_xor_sync(full, vh, off));
        vm = max(vm, __shfl_xor_sync(full, vm, off));
    }
    const int eh = (int)(wh >> 21), em = fx_block_exponent(wm), fh = fx_block_exponent(vh), ef = fx_block_exponent(vm);
    bool ok = eh >= 600 && eh <= 1400 && em <= 1900 && fh <= 1900 && ef <= 1900 && dot_in_range(em, eh) && dot_in_range(ef, fh);
    long long hx[4], ux[4];
    // g
#pragma unroll
    for (int n = 0; n < 4; ++n) hx[n] = fx_from(hg[n], eh), ux[n] = fx_from(ug[n], em);
    auto dot4 = [&]() {
        FxDot d{};
#pragma unroll
        for (int n = 0; n < 4; ++n) d.add(hx[n], ux[n]);
        return d.result();
    };
    long long E = fx_round4(hx[0] + hx[1]) + fx_round4(hx[2] + hx[3]), dot = dot4();
    const long long d_j = fx_round4(hx[0] - hx[1]), d_8 = fx_round4(hx[2] - hx[3]);
    const int half = j < 3 ? 7 : 8;  // ties of the axis pairs down, of the others up
    const long long s_j = (ux[0] + ux[1] + half) >> 4, s_8 = j == 1 ? fx_round4_even(ux[2]) : fx_round4(ux[2] + ux[3]);  // lane 1's s_8: the rest population
    const long long l_j = fx_round4(ux[0] - ux[1]), l_8 = fx_round4(ux[2] - ux[3]);
    // f
#pragma unroll
    for (int n = 0; n < 4; ++n) hx[n] = fx_from(hf[n], fh), ux[n] = fx_from(uf[n], ef);
    long long Sf = fx_round4(hx[0] + hx[1]) + fx_round4(hx[2] + hx[3]), fd = dot4();
    const long long sf_j = (ux[0] + ux[1] + half) >> 4, sf_8 = j == 1 ? fx_round4_even(ux[2]) : fx_round4(ux[2] + ux[3]);
    const long long lf_j = fx_round4(ux[0] - ux[1]), lf_8 = fx_round4(ux[2] - ux[3]);
    long long Fs = (j < 3 ? sf_j << 1 : sf_j) + (j == 0 ? sf_8 : (j == 1 ? (sf_8 << 3) + (sf_8 << 2) : 0));
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        E += __shfl_xor_sync(full, E, off);
        dot += __shfl_xor_sync(full, dot, off);
        Sf += __shfl_xor_sync(full, Sf, off);
        fd += __shfl_xor_sync(full, fd, off);
        Fs += __shfl_xor_sync(full, Fs, off);
    }
    auto all9 = [&](long long vj, long long v8, long long* v) {  // the nine pairs' values
#pragma unroll
        for (int p = 0; p < 8; ++p) v[p] = __shfl_sync(full, vj, base + p);
        v[8] = __shfl_sync(full, v8, base);
    };
    auto vec9 = [](const long long* v, int sh, int64_t& a, int64_t& b, int64_t& d) {  // sum v_p e_p, axis pairs << sh
        a = (v[0] << sh) + ((v[3] + v[4]) + (v[5] + v[6]));
        b = (v[1] << sh) + ((v[3] - v[4]) + (v[7] + v[8]));
        d = (v[2] << sh) + ((v[5] - v[6]) + (v[7] - v[8]));
    };
    long long v[9];
    int64_t dx, dy, dz, Vx, Vy, Vz, Fx, Fy, Fz;
    all9(d_j, d_8, v);
    vec9(v, 0, dx, dy, dz);
    all9(l_j, l_8, v);
    vec9(v, 1, Vx, Vy, Vz);
    all9(lf_j, lf_8, v);
    vec9(v, 1, Fx, Fy, Fz);
    all9(s_j, s_8, v);
    const long long m0 = __shfl_sync(full, s_8, base + 1);
    const int32_t Eh = (int32_t)(E >> 32);
    const float Ef = (float)Eh, xf = (float)(int32_t)(dx >> 32), yf = (float)(int32_t)(dy >> 32), zf = (float)(int32_t)(dz >> 32);
    ok = ok && Eh > 0 && fx_clz((uint32_t)Eh) <= 14 && xf * xf + yf * yf + zf * zf < ph.fx.m_max * (Ef * Ef);
    AdjFxCell t;
    int ek = 0;
    if (ok) {
        adj_fx_g(E, dx, dy, dz, dot, m0, v[0] << 1, v[1] << 1, v[2] << 1, v[3] + v[4], v[7] + v[8], v[5] + v[6], v[3] - v[4],
                 v[7] - v[8], v[5] - v[6], Vx, Vy, Vz, eh, em, ph, k, t);
        adj_fx_f(Sf, fd, Fs, Fx, Fy, Fz, fh, ef, ph, k, t);
        const double kv[4] = {t.nuE, t.tx, t.ty, t.tz};
        ek = fx_block_exponent(fx_max_word<4>(kv));
        ok = ek < 1900;
    }
    if (work && ok) {
        const int64_t kE = fx_from(t.nuE, ek), kx = fx_from(t.tx, ek), ky = fx_from(t.ty, ek), kz = fx_from(t.tz, ek);
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            if (n < nv) {
                const int i = iv[n];
                const int ex = vel_x(i), ey = vel_y(i), ez = vel_z(i);
                const int64_t kt = kE + (ex > 0 ? kx : (ex < 0 ? -kx : 0)) + (ey > 0 ? ky : (ey < 0 ? -ky : 0)) +
                                   (ez > 0 ? kz : (ez < 0 ? -kz : 0));
                const bool bk = (back >> n) & 1u;
                const long long at = (long long)(bk ? opp_rt(i) : i) * S + idx + (bk ? 0 : o.src(i));
                Lout[RLB_CHK(at, 38ll * S)] = fma(ph.fx.omw, uf[n], t.nuS);
                Lout[RLB_CHK(19 * S + at, 38ll * S)] = fma(ph.fx.omw, ug[n], i == 0 ? t.nuE : fx_to_even(kt, ek - 1083));
            }
        }
        if (j == 0) tau_acc = t.tsum * c.inv_tau2;
    } else if (work) {
        if (j == 0) tau_acc = adjoint_cell_general<XBC>(A, Lin, Lout, g, c, idx);
    }
    if (live && !work) {
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            if (n < nv) {
                const int i = iv[n];
                if (ghost) {  // zero where nobody reads the population; the inflow's dL/dbeta_in
                    if (vel_x(i) != (x == 0 ? 1 : -1)) {
                        Lout[RLB_CHK(i * S + idx, 38ll * S)] = 0.0;
                        Lout[RLB_CHK((19 + i) * S + idx, 38ll * S)] = 0.0;
                    }
                    if (XBC == XBC_INFLOW_OUTFLOW && x == 0 && !solid) {
                        const double* tf = inflow_t + 3 * i;
                        const double* tg = tf + 57;
                        bin0 = fma(uf[n], tf[0], fma(ug[n], tg[0], bin0));
                        bin1 = fma(uf[n], tf[1], fma(ug[n], tg[1], bin1));
                        bin2 = fma(uf[n], tf[2], fma(ug[n], tg[2], bin2));
                    }
                } else {  // solid: identity
                    Lout[RLB_CHK(i * S + idx, 38ll * S)] = uf[n];
                    Lout[RLB_CHK((19 + i) * S + idx, 38ll * S)] = ug[n];
                }
            }
        }
    }
    if (XBC != XBC_PERIODIC && work && (x == 1 || x == g.nx - 2)) {  // populations that a ghost would pull
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const int ex = vel_x(iv[n]);
            if (n < nv && ((x == 1 && ex == -1) || (x == g.nx - 2 && ex == 1))) {
                Lout[RLB_CHK(iv[n] * S + idx, 38ll * S)] = 0.0;
                Lout[RLB_CHK((19 + iv[n]) * S + idx, 38ll * S)] = 0.0;
            }
        }
    }
    block_sums<double, XBC == XBC_INFLOW_OUTFLOW>(tau_acc, bin0, bin1, bin2, true, sums);
}

// ---------------------------------------------------------------------------
// Shared-memory staged FP32 kernel.  Persistent grid-stride loop; every
// thread stages the 38 values of each phase of its cells (19 pulled
// populations + 19 lambda_{t+1}) in its own column of a three-slot ring with
// 4-byte cp.async copies, one phase ahead of the arithmetic:
//
//     issue F_k | wait G_k, compute G_k | issue G_k+1 | wait F_k, compute F_k, scatter
//
// so the loads of the next phase are in flight during the arithmetic of the
// current one without holding registers.  Slots: G_k, F_k, G_k+1 (the G slot
// stays valid through F_k, whose scatter reads mu_g).  Each thread reads only
// the slots it wrote, so cp.async.wait_group alone orders the accesses.
// ---------------------------------------------------------------------------
constexpr int kStageThreads = 128;
constexpr int kStageSlots = 3;
constexpr size_t kStageSmemBytes = sizeof(float) * kStageSlots * 38 * kStageThreads;

// Base address of each of the 38 planes of the three buffers, a kernel
// parameter: with every plane number a compile-time constant after
// unrolling, an address is a 32-bit cell offset added to a uniform base.
struct PlaneTab {
    const float* a[38];
    const float* l[38];
    float* o[38];
};

// Every address of a cell's populations is its plane's base from the table
// plus a 32-bit cell offset (N < 2^31): the fewest address instructions at any
// accepted lattice size.
template <int XBC>
__global__ void __launch_bounds__(kStageThreads, 3)
    k_adjoint_step_staged(const float* __restrict__ A, const float* __restrict__ Lin, float* __restrict__ Lout,
                          Geom g, Phys ph, AdjConst<float> c, double* red, const float* __restrict__ inflow_t,
                          const __grid_constant__ PlaneTab tab) {
    extern __shared__ float stage[];  // [slot][value 0..37][thread]
    const long long S = g.S;
    // element q S + off of A, Lin, Lout (off a cell index, q a constant)
    auto pa = [&](int q, int off) -> const float* { return RLB_CHK_PTR(tab.a[q], off, S); };
    auto pl = [&](int q, int off) -> const float* { return RLB_CHK_PTR(tab.l[q], off, S); };
    auto po = [&](int q, int off) -> float* { return RLB_CHK_PTR(tab.o[q], off, S); };
    const int tid = threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const uint32_t scol = (uint32_t)__cvta_generic_to_shared(stage) + 4u * tid;
    auto sval = [&](int slot, int q) -> float { return stage[(slot * 38 + q) * kStageThreads + tid]; };
    auto is_ghost = [&](int x) { return XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1); };
    // one phase (base 19: g, base 0: f) of a cell (pull offsets o) into a slot
    auto issue = [&](int cidx, const PullOffsets& o, int base, int slot) {
        const uint32_t s0 = scol + 4u * (uint32_t)(slot * 38 * kStageThreads);
#pragma unroll
        for (int i = 0; i < 19; ++i) cp_async4(s0 + 4u * (uint32_t)(i * kStageThreads), pa(base + i, cidx + o.src(i)));
#pragma unroll
        for (int i = 0; i < 19; ++i) cp_async4(s0 + 4u * (uint32_t)((19 + i) * kStageThreads), pl(base + i, cidx));
    };

    float tau_acc = 0.0f;
    double bin0 = 0.0, bin1 = 0.0, bin2 = 0.0;
    bool has_b = false;
    // 64-bit loop counter: li + stride cannot wrap for any accepted N
    long long li = dependent_begin(blockIdx.x * blockDim.x + tid);
    int idx = li < g.N ? (int)li : 0;
    int x = 0, y = 0, z = 0;
    PullOffsets o{};
    if (li < g.N) {
        cell_coords(g, idx, x, y, z);
        o = PullOffsets(g, x, y, z);
        if (!is_ghost(x)) issue(idx, o, 19, 0);
    }
    cp_async_commit();
    int sg = 0;
    for (; li < g.N; li += stride) {
        idx = (int)li;
        const int sf = sg == kStageSlots - 1 ? 0 : sg + 1;
        const int sn = sf == kStageSlots - 1 ? 0 : sf + 1;
        const bool ghost = is_ghost(x);
        if (!ghost) issue(idx, o, 0, sf);
        cp_async_commit();
        const long long nl = (long long)idx + stride;  // 64-bit: cannot wrap
        const int nidx = nl < g.N ? (int)nl : 0;
        int xn = 0, yn = 0, zn = 0;
        PullOffsets on{};
        if (nl < g.N) {
            cell_coords(g, nidx, xn, yn, zn);
            on = PullOffsets(g, xn, yn, zn);
        }
        cp_async_wait<1>();  // G_k has landed
        // ---- g phase
        unsigned bounced = 0u;
        bool solid = false;
        const int dup = dup_of<XBC>(x, g.nx);
        float mug[19];
        CellG<float> r;
        if (!ghost) {
            float h[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) h[i] = sval(sg, i);
            solid = is_solid(h[0]);  // the cell's own g_0 (pull offset 0)
            if (!solid) {
                if (isnan(sum19(h))) {
#pragma unroll
                    for (int i = 1; i < 19; ++i) {
                        if (is_solid(h[i])) {
                            bounced |= 1u << i;
                            h[i] = *pa(19 + opp(i), idx);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < 19; ++i) mug[i] = sval(sg, 19 + i);
                if (dup) {
#pragma unroll
                    for (int i = 0; i < 19; ++i) mug[i] += *pl(19 + i, idx + dup);
                    if (dup_both<XBC>(g.nx)) {
#pragma unroll
                        for (int i = 0; i < 19; ++i) mug[i] += *pl(19 + i, idx - 1);
                    }
                }
                cell_g(h, mug, c, r);
            }
        }
        if (nl < g.N && !is_ghost(xn)) issue(nidx, on, 19, sn);
        cp_async_commit();
        cp_async_wait<1>();  // F_k has landed
        // ---- f phase, scatter
        if (ghost) {
            ghost_cell<float, XBC>(x, idx, S, A, Lin, Lout, inflow_t, bin0, bin1, bin2, has_b);
        } else if (solid) {  // never updated: identity
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                *po(i, idx) = sval(sf, 19 + i);
                *po(19 + i, idx) = sval(sg, 19 + i);
            }
        } else {
            float h[19], muf[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) h[i] = sval(sf, i);
            if (bounced) {
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    if ((bounced >> i) & 1u) h[i] = *pa(opp(i), idx);
            }
#pragma unroll
            for (int i = 0; i < 19; ++i) muf[i] = sval(sf, 19 + i);
            if (dup) {
#pragma unroll
                for (int i = 0; i < 19; ++i) muf[i] += *pl(i, idx + dup);
                if (dup_both<XBC>(g.nx)) {
#pragma unroll
                    for (int i = 0; i < 19; ++i) muf[i] += *pl(i, idx - 1);
                }
            }
            float tf, aS, fbx, fby, fbz;
            cell_f(h, muf, r, c, tf, aS, fbx, fby, fbz);
            tau_acc += (r.tacc + tf) * c.inv_tau2_t;
            float vE, vx, vy, vz;
            recovery_adjoint<float>(r.ae, fbx + r.gbx, fby + r.gby, fbz + r.gbz, r.Et, r.sqt, r.Dt, r.bx, r.by,
                                    r.bz, r.mx, r.my, r.mz, vE, vx, vy, vz);
            scatter_cell(muf, mug, aS, vE, vx, vy, vz, c, [&](int q, int i, float v) {
                if ((bounced >> i) & 1u)
                    *po(q - i + opp(i), idx) = v;
                else
                    *po(q, idx + o.src(i)) = v;
            });
            zero_to_ghost<float, XBC>(x, g.nx, idx, S, Lout);
        }
        sg = sn;
        x = xn;
        o = on;
    }
    cp_async_wait<0>();
    warp_partials<float>((double)tau_acc, bin0, bin1, bin2, has_b, red);
}

// Cooperative form of the staged kernel (the default FP32 adjoint kernel).
// The pulled populations are staged per thread as above; lambda_t+1, read at
// the cell's own index, is copied by the whole block in 16-byte chunks (a
// quarter of the copy instructions), so the block meets at two barriers per
// cell: after the G phase has landed (then every thread is past the f phase
// of the previous cell, and its slots can be refilled) and after the F phase
// has landed.  Because every cell's lambda_t+1 is in the ring, the ghost
// planes and the outflow-copy cells read theirs from it instead of from HBM
// (a lane that waits on HBM would hold the whole block at the next barrier).
template <int XBC>
__global__ void __launch_bounds__(kStageThreads, 3)
    k_adjoint_step_coop(const float* __restrict__ A, const float* __restrict__ Lin, float* __restrict__ Lout,
                          Geom g, Phys ph, AdjConst<float> c, double* red, const float* __restrict__ inflow_t,
                          const __grid_constant__ PlaneTab tab) {
    extern __shared__ float stage[];  // [slot][value 0..37][thread]
    const long long S = g.S;
    // element q S + off of A, Lin, Lout (off a cell index, q a constant)
    auto pa = [&](int q, int off) -> const float* { return RLB_CHK_PTR(tab.a[q], off, S); };
    auto pl = [&](int q, int off) -> const float* { return RLB_CHK_PTR(tab.l[q], off, S); };
    auto po = [&](int q, int off) -> float* { return RLB_CHK_PTR(tab.o[q], off, S); };
    const int tid = threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const uint32_t scol = (uint32_t)__cvta_generic_to_shared(stage) + 4u * tid;
    auto sval = [&](int slot, int q) -> float { return stage[(slot * 38 + q) * kStageThreads + tid]; };
    // another thread's column (lambda_t+1 of every cell of the block is staged)
    auto sval_c = [&](int slot, int q, int col) -> float { return stage[(slot * 38 + q) * kStageThreads + col]; };
    auto is_ghost = [&](int x) { return XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1); };
    // the pulled values of one phase (base 19: g, base 0: f) of this thread's
    // cell (pull offsets o) into its column of a slot
    auto issue = [&](int cidx, const PullOffsets& o, int base, int slot) {
        const uint32_t s0 = scol + 4u * (uint32_t)(slot * 38 * kStageThreads);
#pragma unroll
        for (int i = 0; i < 19; ++i) cp_async4(s0 + 4u * (uint32_t)(i * kStageThreads), pa(base + i, cidx + o.src(i)));
    };
    // lambda_t+1 of one phase for the block's cells [cb, cb + 128): warp w
    // copies planes w, w + 4, ..., lane l the 16 bytes of cells cb + 4l .. + 3
    // (S is a multiple of 4: a chunk lies wholly inside or outside a plane)
    const int wq = tid >> 5, lane4 = 4 * (tid & 31);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(stage);
    auto issue_lam = [&](long long cb, int base, int slot) {
        const long long cell = cb + lane4;
        if (cell >= S) return;
        const uint32_t s0 = sbase + 4u * (uint32_t)((slot * 38 + 19) * kStageThreads + lane4);
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const int q = wq + 4 * m;
            if (q < 19) cp_async16(s0 + 4u * (uint32_t)(q * kStageThreads), RLB_CHK_PTR(Lin, (long long)(base + q) * S + cell, 38ll * S));
        }
    };

    float tau_acc = 0.0f;
    float ga0 = 0.0f, ga1 = 0.0f, ga2 = 0.0f;  // this lane's share of the inflow plane's terms
    double bin0 = 0.0, bin1 = 0.0, bin2 = 0.0;
    bool has_b = false;
    // block-uniform loop over the block's cells [cb, cb + 128) (every thread
    // reaches every barrier); 64-bit: cb + stride cannot wrap
    long long cb = dependent_begin(blockIdx.x * blockDim.x);
    long long li = cb + tid;
    int idx = li < g.N ? (int)li : 0;
    int x = 0, y = 0, z = 0;
    PullOffsets o{};
    if (li < g.N) {
        cell_coords(g, idx, x, y, z);
        o = PullOffsets(g, x, y, z);
        if (!is_ghost(x)) issue(idx, o, 19, 0);
    }
    if (cb < g.N) issue_lam(cb, 19, 0);
    cp_async_commit();
    int sg = 0;
    for (; cb < g.N; cb += stride) {
        li = cb + tid;
        const bool act = li < g.N;
        idx = act ? (int)li : 0;
        const int sf = sg == kStageSlots - 1 ? 0 : sg + 1;
        const int sn = sf == kStageSlots - 1 ? 0 : sf + 1;
        const bool ghost = !act || is_ghost(x);
        // the inflow ghost's own f_0 (solid marker), loaded early
        const float own0 = (XBC == XBC_INFLOW_OUTFLOW && act && x == 0) ? *pa(0, idx) : 0.0f;
        const long long nl = li + stride;
        const int nidx = nl < g.N ? (int)nl : 0;
        int xn = 0, yn = 0, zn = 0;
        PullOffsets on{};
        if (nl < g.N) {
            cell_coords(g, nidx, xn, yn, zn);
            on = PullOffsets(g, xn, yn, zn);
        }
        cp_async_wait<0>();  // G_k has landed (this thread's copies)
        __syncthreads();     // ... and every thread's; all are past f phase k-1
        if (!ghost) issue(idx, o, 0, sf);
        issue_lam(cb, 0, sf);
        cp_async_commit();
        // ---- g phase
        unsigned bounced = 0u;
        bool solid = false;
        const int dup = dup_of<XBC>(x, g.nx);
        const int dcol = tid + dup;  // the copying ghost's column, when in this block
        const bool dup_in = dcol >= 0 && dcol < kStageThreads;
        float mug[19];
        CellG<float> r;
        if (!ghost) {
            float h[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) h[i] = sval(sg, i);
            solid = is_solid(h[0]);  // the cell's own g_0 (pull offset 0)
            if (!solid) {
                if (isnan(sum19(h))) {
#pragma unroll
                    for (int i = 1; i < 19; ++i) {
                        if (is_solid(h[i])) {
                            bounced |= 1u << i;
                            h[i] = *pa(19 + opp(i), idx);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < 19; ++i) mug[i] = sval(sg, 19 + i);
                if (dup) {
                    if (dup_in) {
#pragma unroll
                        for (int i = 0; i < 19; ++i) mug[i] += sval_c(sg, 19 + i, dcol);
                    } else {
#pragma unroll
                        for (int i = 0; i < 19; ++i) mug[i] += *pl(19 + i, idx + dup);
                    }
                    if (dup_both<XBC>(g.nx)) {
#pragma unroll
                        for (int i = 0; i < 19; ++i) mug[i] += *pl(19 + i, idx - 1);
                    }
                }
                cell_g(h, mug, c, r);
            }
        }
        if (nl < g.N && !is_ghost(xn)) issue(nidx, on, 19, sn);
        if (cb + stride < g.N) issue_lam(cb + stride, 19, sn);
        cp_async_commit();
        cp_async_wait<1>();  // F_k has landed (this thread's copies)
        __syncthreads();     // ... and every thread's
        // ---- f phase, scatter
        if (!act) {
        } else if (ghost) {
            // ghost_cell: its zeros and the inflow plane's dL/dbeta_in terms
            // are written below by the whole warp
        } else if (solid) {  // never updated: identity
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                *po(i, idx) = sval(sf, 19 + i);
                *po(19 + i, idx) = sval(sg, 19 + i);
            }
        } else {
            float h[19], muf[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) h[i] = sval(sf, i);
            if (bounced) {
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    if ((bounced >> i) & 1u) h[i] = *pa(opp(i), idx);
            }
#pragma unroll
            for (int i = 0; i < 19; ++i) muf[i] = sval(sf, 19 + i);
            if (dup) {
                if (dup_in) {
#pragma unroll
                    for (int i = 0; i < 19; ++i) muf[i] += sval_c(sf, 19 + i, dcol);
                } else {
#pragma unroll
                    for (int i = 0; i < 19; ++i) muf[i] += *pl(i, idx + dup);
                }
                if (dup_both<XBC>(g.nx)) {
#pragma unroll
                    for (int i = 0; i < 19; ++i) muf[i] += *pl(i, idx - 1);
                }
            }
            float tf, aS, fbx, fby, fbz;
            cell_f(h, muf, r, c, tf, aS, fbx, fby, fbz);
            tau_acc += (r.tacc + tf) * c.inv_tau2_t;
            float vE, vx, vy, vz;
            recovery_adjoint<float>(r.ae, fbx + r.gbx, fby + r.gby, fbz + r.gbz, r.Et, r.sqt, r.Dt, r.bx, r.by,
                                    r.bz, r.mx, r.my, r.mz, vE, vx, vy, vz);
            scatter_cell(muf, mug, aS, vE, vx, vy, vz, c, [&](int q, int i, float v) {
                if ((bounced >> i) & 1u)
                    *po(q - i + opp(i), idx) = v;
                else
                    *po(q, idx + o.src(i)) = v;
            });
        }
        if constexpr (XBC != XBC_PERIODIC) {
            // The zeros next to the ghost planes, spread over the warp (one
            // lane storing 28 or 10 of them would hold its block at the next
            // barrier): for each lane that is a ghost cell, lane q zeroes
            // population q of it where nobody reads it (velocity not pointing
            // inward); for each fluid cell at x = 1 or nx - 2, lane q zeroes
            // population q of it where the ghost would have pulled it.
            const int lane = tid & 31;
            const int vq = lane < 19 ? vel_x(lane) : 0;
            unsigned m = __ballot_sync(0xffffffffu, act && (ghost || (!solid && (x == 1 || x == g.nx - 2))));
            while (m) {
                const int src = __ffs(m) - 1;
                m &= m - 1;
                const int cx = __shfl_sync(0xffffffffu, x, src);
                const int cidx = __shfl_sync(0xffffffffu, idx, src);
                bool z;
                if (cx == 0 || cx == g.nx - 1)
                    z = vq != (cx == 0 ? 1 : -1);  // a ghost cell
                else  // next to a ghost (both, when nx = 3)
                    z = (cx == 1 && vq == -1) || (cx == g.nx - 2 && vq == 1);
                if (lane < 19 && z) {
                    Lout[RLB_CHK((long long)lane * S + cidx, 38ll * S)] = 0.0f;
                    Lout[RLB_CHK((long long)(19 + lane) * S + cidx, 38ll * S)] = 0.0f;
                }
            }
        }
        if constexpr (XBC == XBC_INFLOW_OUTFLOW) {
            // dL/dbeta_in = lambda_t+1 . d eq_in / d beta_in at each fluid
            // inflow ghost: its 38 terms spread over the warp (lane l takes
            // q = l and l + 32) from the ghost's column of the ring, each lane
            // adding into its own partial sums (summed over the warp at the end)
            unsigned m = __ballot_sync(0xffffffffu, act && x == 0 && !is_solid(own0));
            const int lane = tid & 31;
            while (m) {
                const int col = (tid & ~31) + __ffs(m) - 1;
                m &= m - 1;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int q = lane + 32 * r;
                    if (q < 38) {
                        const float l = q < 19 ? sval_c(sf, 19 + q, col) : sval_c(sg, q, col);
                        ga0 = fmaf(l, inflow_t[3 * q + 0], ga0);
                        ga1 = fmaf(l, inflow_t[3 * q + 1], ga1);
                        ga2 = fmaf(l, inflow_t[3 * q + 2], ga2);
                    }
                }
                has_b = true;
            }
        }
        sg = sn;
        x = xn;
        o = on;
    }
    cp_async_wait<0>();
    bin0 += (double)ga0;
    bin1 += (double)ga1;
    bin2 += (double)ga2;
    warp_partials<float>((double)tau_acc, bin0, bin1, bin2, has_b, red);
}

// d eq_j(n_in, eps_in, beta_in) / d beta_in,a for the 38 populations (one
// thread per population, FP64): the adjoint of the inflow plane.  The table
// is written twice: binary64, then rounded to binary32 after it.
__global__ void k_inflow_derivs(Phys ph, double* out) {
    const int j = threadIdx.x;
    if (j >= 38) return;
    double lf[19], lg[19];
    for (int i = 0; i < 19; ++i) lf[i] = lg[i] = 0.0;
    if (j < 19) lf[j] = 1.0; else lg[j - 19] = 1.0;
    double an, ae, ax, ay, az;
    eq_fields_adjoint(lf, lg, ph.n_in, ph.eps_in, ph.beta_in[0], ph.beta_in[1], ph.beta_in[2], ph, an, ae, ax, ay, az);
    out[3 * j + 0] = ax;
    out[3 * j + 1] = ay;
    out[3 * j + 2] = az;
    float* outf = reinterpret_cast<float*>(out + kInflowTable);
    outf[3 * j + 0] = (float)ax;
    outf[3 * j + 1] = (float)ay;
    outf[3 * j + 2] = (float)az;
}

// The inflow table in the kernels' precision.
template <typename T>
const T* inflow_table(const double* inflow_d) {
    if constexpr (sizeof(T) == 8)
        return inflow_d;
    else
        return reinterpret_cast<const float*>(inflow_d + kInflowTable);
}

cudaError_t launch_inflow_derivs(const Phys& ph, double* out, cudaStream_t st) {
    set_last_launch_count(1);
    k_inflow_derivs<<<1, 64, 0, st>>>(ph, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Adjoint of the macroscopic output: n = S sqrt(1 - b2), eps, beta.
// ---------------------------------------------------------------------------
// One cell in binary64 with IEEE roots and divisions, any state.
template <typename T>
__device__ __noinline__ void adjoint_macro_general(const T* A, const double* dn, const double* deps, const double* dbeta,
                                                   T* lam, const Geom& g, const Phys& ph, int idx) {
    const long long S = g.S;
    double h[38];
    for (int q = 0; q < 38; ++q) h[q] = (double)A[RLB_CHK(q * S + idx, 38ll * S)];
    double sf = 0, E = 0, Mx = 0, My = 0, Mz = 0;
    for (int i = 0; i < 19; ++i) {
        sf += h[i];
        E += h[19 + i];
        Mx += h[19 + i] * vel_x(i);
        My += h[19 + i] * vel_y(i);
        Mz += h[19 + i] * vel_z(i);
    }
    if (sizeof(T) == 4) {
        sf += ph.n_ref;
        E += ph.eps_ref;
    }
    Mx *= ph.c_l;
    My *= ph.c_l;
    Mz *= ph.c_l;
    const double sq = sqrt(4.0 * E * E - 3.0 * (Mx * Mx + My * My + Mz * Mz));
    const double eps = sq - E;
    const double D = 3.0 * E + eps;
    const double bx = 3.0 * Mx / D, by = 3.0 * My / D, bz = 3.0 * Mz / D;
    const double b2 = bx * bx + by * by + bz * bz;
    const double rt = sqrt(1.0 - b2);
    const double gdn = dn[idx];
    const double aS = gdn * rt;
    const double c = -gdn * sf / rt;
    const double abx = dbeta[idx] + c * bx;
    const double aby = dbeta[g.N + idx] + c * by;
    const double abz = dbeta[2 * (long long)g.N + idx] + c * bz;
    double vE, vx, vy, vz;
    recovery_adjoint<double>(deps[idx], abx, aby, abz, E, sq, D, bx, by, bz, Mx, My, Mz, vE, vx, vy, vz);
    for (int i = 0; i < 19; ++i) {
        lam[RLB_CHK(i * S + idx, 38ll * S)] = (T)aS;
        lam[RLB_CHK((19 + i) * S + idx, 38ll * S)] = (T)(vE + ph.c_l * (vel_x(i) * vx + vel_y(i) * vy + vel_z(i) * vz));
    }
}

// FP64 instructions: 60 instead of some 190, which bound the kernel (sphere
// lattice, FP32: 1.14 -> 0.29 ms).  The
// moments are integers (fx_moments); s = sqrt(4 E^2 - 3 M^2), 1/s, 1/D and
// sqrt(1 - beta^2) = 2 sqrt(eps / D) come from binary32 seeds; the 18 moving g
// values are integer sums of c_l v and v_E.  Binary32 lambdas keep the bits of
// the binary64 form: a cell with a value within its rounding error (64 u
// gamma^2 of the terms' sizes) of a binary32 midpoint is left to it.
template <typename T>
__global__ void __launch_bounds__(128, 6) k_adjoint_macro(const T* __restrict__ A, const double* __restrict__ dn,
                                                       const double* __restrict__ deps, const double* __restrict__ dbeta,
                                                       T* __restrict__ lam, const __grid_constant__ Geom g,
                                                       const __grid_constant__ Phys ph) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= g.N) return;
    const long long S = g.S;
    T* Lc = lam + idx;
    auto put = [&](int q, T v) { Lc[RLB_CHK_OFF(q * S, idx, 38ll * S)] = v; };
    const double gn = __ldg(dn + idx), ge = __ldg(deps + idx), gx = __ldg(dbeta + idx), gy = __ldg(dbeta + g.N + idx),
                 gz = __ldg(dbeta + 2 * (long long)g.N + idx);
    T h[19], f[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = __ldg(RLB_CHK_PTR(A, i * S + idx, 38ll * S));
    if (is_solid(f[0])) {
#pragma unroll
        for (int q = 0; q < 38; ++q) put(q, (T)0);
        return;
    }
#pragma unroll
    for (int i = 0; i < 19; ++i) h[i] = __ldg(RLB_CHK_PTR(A, (19 + i) * S + idx, 38ll * S));
    FxMoments m;
    if (fx_moments(h, f, ph.fx.m3cl2, ph.n_ref, ph.eps_ref, m)) {
        if (gn == 0.0 && ge == 0.0 && gx == 0.0 && gy == 0.0 && gz == 0.0) {  // zero only where the fields exist
#pragma unroll
            for (int q = 0; q < 38; ++q) put(q, (T)0);
            return;
        }
        const double E2 = m.E + m.E;
        double ys, hs;
        rsqrt_seed(m.disc, ys, hs);
        double sq = m.disc * ys;
        sq = fma(fma(-sq, sq, m.disc), hs, sq);
        sq = fma(fma(-sq, sq, m.disc), hs, sq);
        const double e1 = fma(-sq, ys, 1.0);
        const double rs = fma(ys, fma(e1, e1, e1), ys);
        const double D = E2 + sq;
        const double x0 = rcp_seed(D);
        const double e2 = fma(-D, x0, 1.0);
        const double rD = fma(x0, fma(e2, e2, e2), x0);
        const double r3 = rD * ph.three_cl;
        const double bx = m.x * r3, by = m.y * r3, bz = m.z * r3;
        // 1/sqrt(1 - beta^2) and its inverse from 4 eps / D
        const double w = 4.0 * (fma(m.t, rD, m.E) * rD);
        const double gam = rsqrt_unit(w);
        const double aS = gn * (w * gam), cc = -(gn * m.S) * gam;
        const double ax = fma(cc, bx, gx), ay = fma(cc, by, gy), az = fma(cc, bz, gz);
        const double ab = fma(ax, bx, fma(ay, by, az * bz)) * rD;
        const double dE = fma(E2 + E2, rs, -1.0);
        const double vE = fma(ge, dE, -ab * (3.0 + dE));
        const double c3 = (ph.three_cl * rs) * (ab - ge), rD3 = 3.0 * rD;
        // c_l v: v_a = 3 ab_a / D + 3 M_a (...) / s, M = c_l d
        const double vx = ph.c_l * fma(c3, m.x, ax * rD3), vy = ph.c_l * fma(c3, m.y, ay * rD3),
                     vz = ph.c_l * fma(c3, m.z, az * rD3);
        const double kv[4] = {vE, vx, vy, vz};
        const int ek = fx_max_exponent<4>(kv);
        bool ok = ek >= 200 && ek < 1800;
        if constexpr (sizeof(T) == 4) ok = ok && ek > 1023 - 80 && ek < 1023 + 80;
        if (ok) {
            const int64_t kE = fx_from(vE, ek), kx = fx_from(vx, ek), ky = fx_from(vy, ek), kz = fx_from(vz, ek);
            if constexpr (sizeof(T) == 8) {
#pragma unroll
                for (int i = 0; i < 19; ++i) put(i, aS);
                auto gput = [&](int p, int64_t t) {
                    put(20 + 2 * p, fx_to_even(kE + t, ek - 1083));
                    put(21 + 2 * p, fx_to_even(kE - t, ek - 1083));
                };
                put(19, vE);
                gput(0, kx), gput(1, ky), gput(2, kz), gput(3, kx + ky), gput(4, kx - ky), gput(5, kx + kz), gput(6, kx - kz);
                gput(7, ky + kz), gput(8, ky - kz);
                return;
            } else {
                // the rounding error of the binary64 form in units of 2^(ek - 1083):
                // 64 u gamma^2 at the size of the terms
                auto mag = [](double v) { return fabsf(d2f_seed(v)); };
                const float B = 3.0f * mag(ge) + 6.0f * mag(ab) + 3.0f * (float)ph.c_l * mag(rD) * (mag(ax) + mag(ay) + mag(az)) +
                                3.0f * mag(ph.cl2 * rs) * (mag(m.x) + mag(m.y) + mag(m.z)) * (mag(ab) + mag(ge));
                const float g1 = d2f_seed(gam), g2 = g1 * g1;
                const float units = 8192.0f * g2 * B * pow2f(1023 - ek);
                F32Out o;
                const int kb = ek - 1083 + 32;
                o.c1 = pow2f(kb >> 1), o.c2 = pow2f(kb - (kb >> 1));
                ok = units < 0x1p28f;
                o.d7 = (uint32_t)(units * (1.03f / 128.0f)) + 2u;
                o.nd = 32 - __clz((int)o.d7);
                bool ambiguous = !ok;
                float fs = 0.0f;
                if (gn != 0.0) {
                    int es;
                    const double as = fabs(aS);
                    const int64_t xs = fx_mantissa(as, es);
                    F32Out of;
                    const int kf = es - 1084 + 32;
                    ambiguous |= es < 1023 - 80 || es > 1023 + 80;
                    of.c1 = pow2f(kf >> 1), of.c2 = pow2f(kf - (kf >> 1));
                    of.d7 = (uint32_t)(256.0f * g2 * 1.03f) + 2u;
                    of.nd = 32 - __clz((int)of.d7);
                    fs = copysignf(fx_to_f32(xs, of, ambiguous), gn > 0.0 ? 1.0f : -1.0f);
                }
                if (!ambiguous) {
#pragma unroll
                    for (int i = 0; i < 19; ++i) put(i, fs);
                    auto gput = [&](int p, int64_t t) {
                        put(20 + 2 * p, fx_to_f32(kE + t, o, ambiguous));
                        put(21 + 2 * p, fx_to_f32(kE - t, o, ambiguous));
                    };
                    put(19, fx_to_f32(kE, o, ambiguous));
                    gput(0, kx), gput(1, ky), gput(2, kz), gput(3, kx + ky), gput(4, kx - ky), gput(5, kx + kz),
                        gput(6, kx - kz);
                    gput(7, ky + kz), gput(8, ky - kz);
                    if (!ambiguous) return;
                }
            }
        }
    }
    adjoint_macro_general<T>(A, dn, deps, dbeta, lam, g, ph, idx);
}

// ---------------------------------------------------------------------------
// Adjoint of the initialisation A_0 = eq(n0, eps0, beta0).
// ---------------------------------------------------------------------------
// The lambda moments are integers (weights times 36): S1, T, V over the g
// pairs, F1, F over the f pairs; with y = T beta, eg = eps gamma^2 and
//   Q = [6 beta.y - 2 |beta|^2 S1] / c_l^2 + 4 V.beta / c_l + w0 l_0 (4 - 2 |beta|^2 / c_l^2):
//   a_eps  = S1 / c_l^2 - w0 l_0 (2 / c_l^2 + 1) + gamma^2 Q
//   a_beta = eg [(12 y - 4 (S1 + w0 l_0) beta) / c_l^2 + 4 V / c_l + 2 gamma^2 Q beta]
//   a_S    = w0 l_f0 + F1 + 3 F.beta / c_l,   a_n = gamma a_S,
//   a_beta += 3 n gamma F / c_l + n gamma^3 a_S beta.
// 80 FP64 instructions instead of some 250 with the conversions, which bound
// the kernel (sphere lattice, FP32 lambdas: 1.72 -> 0.41 ms).
template <typename T>
__global__ void __launch_bounds__(128, 4) k_adjoint_fields(const double* __restrict__ n0, const double* __restrict__ e0,
                                                        const double* __restrict__ b0, const T* __restrict__ A0,
                                                        const T* __restrict__ lam, double* __restrict__ dn,
                                                        double* __restrict__ de, double* __restrict__ db,
                                                        const __grid_constant__ Geom g, const __grid_constant__ Phys ph,
                                                        double* red) {
    const long long S = g.S;
    double bin0 = 0.0, bin1 = 0.0, bin2 = 0.0;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < g.N) {
        double an = 0, ae = 0, ax = 0, ay = 0, az = 0;
        if (!is_solid(A0[RLB_CHK(idx, 38ll * S)])) {
            const bool inflow = g.xbc == XBC_INFLOW_OUTFLOW && idx % g.nx == 0;
            double n, e, bx, by, bz;
            if (inflow) {
                n = ph.n_in, e = ph.eps_in, bx = ph.beta_in[0], by = ph.beta_in[1], bz = ph.beta_in[2];
            } else {
                n = __ldg(n0 + idx), e = __ldg(e0 + idx);
                bx = __ldg(b0 + idx), by = __ldg(b0 + g.N + idx), bz = __ldg(b0 + 2 * (long long)g.N + idx);
            }
            T lf[19], lg[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) lg[i] = __ldg(RLB_CHK_PTR(lam, (19 + i) * S + idx, 38ll * S));
#pragma unroll
            for (int i = 0; i < 19; ++i) lf[i] = __ldg(RLB_CHK_PTR(lam, i * S + idx, 38ll * S));
            constexpr int BIAS = sizeof(T) == 4 ? 127 : 1023, HI = sizeof(T) == 4 ? 250 : 1900;
            int um, uf;
            const int em = fx_block_exponent<19>(lg, um), ef = fx_block_exponent<19>(lf, uf);
            const double b2 = fma(bx, bx, fma(by, by, bz * bz));
            const double omb2 = 1.0 - b2;
            const int oh = __double2hiint(omb2);
            if (em <= HI && ef <= HI && oh > 0x3F900000 && oh < 0x3FF00001) {
                const int km = em - BIAS - 56 - um, kf = ef - BIAS - 56 - uf;
                int64_t Sx = 0, Sy = 0, Sz = 0, Pxy = 0, Pxz = 0, Pyz = 0, Txy = 0, Txz = 0, Tyz = 0, Vx = 0, Vy = 0, Vz = 0;
                int64_t Fx = 0, Fy = 0, Fz = 0;
                const int64_t m0 = fx_round4(fx_from(lg[0], em)), u0 = fx_round4(fx_from(lf[0], ef));
                int64_t Fs = (u0 << 3) + (u0 << 2);
#pragma unroll
                for (int p = 0; p < 9; ++p) {
                    const int64_t a = fx_from(lg[2 * p + 1], em), b = fx_from(lg[2 * p + 2], em);
                    const int64_t c = fx_from(lf[2 * p + 1], ef), d = fx_from(lf[2 * p + 2], ef);
                    const int sh = p < 3 ? 1 : 0;
                    const int64_t sg = fx_round4(a + b) << sh, dl = fx_round4(a - b) << sh, df = fx_round4(c - d) << sh;
                    Fs += fx_round4(c + d) << sh;
                    if (p == 0) Sx = sg;
                    if (p == 1) Sy = sg;
                    if (p == 2) Sz = sg;
                    if (p == 3 || p == 4) Pxy += sg, Txy += p == 3 ? sg : -sg;
                    if (p == 5 || p == 6) Pxz += sg, Txz += p == 5 ? sg : -sg;
                    if (p == 7 || p == 8) Pyz += sg, Tyz += p == 7 ? sg : -sg;
                    if (pair_ex(p)) Vx += dl, Fx += df;
                    if (pair_ey(p) > 0) Vy += dl, Fy += df;
                    if (pair_ey(p) < 0) Vy -= dl, Fy -= df;
                    if (pair_ez(p) > 0) Vz += dl, Fz += df;
                    if (pair_ez(p) < 0) Vz -= dl, Fz -= df;
                }
                const double i2 = ph.inv_cl2, i1 = ph.inv_cl;
                const double gam = rsqrt_unit(omb2);
                const double gam2 = gam * gam, eg = e * gam2 * (1.0 / 36.0);
                const double S1 = fx_to((Sx + Sy + Sz) + (Pxy + Pxz + Pyz), km), l0 = 12.0 * fx_to(m0, km);
                const double Txx = fx_to(Sx + Pxy + Pxz, km), Tyy = fx_to(Sy + Pxy + Pyz, km), Tzz = fx_to(Sz + Pxz + Pyz, km);
                const double txy = fx_to(Txy, km), txz = fx_to(Txz, km), tyz = fx_to(Tyz, km);
                const double yx = fma(Txx, bx, fma(txy, by, txz * bz)), yy = fma(txy, bx, fma(Tyy, by, tyz * bz)),
                             yz = fma(txz, bx, fma(tyz, by, Tzz * bz));
                const double vx = fx_to(Vx, km), vy = fx_to(Vy, km), vz = fx_to(Vz, km);
                const double by_ = fma(bx, yx, fma(by, yy, bz * yz)), vb = fma(bx, vx, fma(by, vy, bz * vz));
                const double b2i = b2 * i2;
                const double Q = fma(6.0 * i2, by_, fma(4.0 * i1, vb, fma(-2.0 * b2i, S1 + l0, 4.0 * l0)));
                ae = fma(gam2, Q, fma(i2, S1, -l0 * fma(2.0, i2, 1.0))) * (1.0 / 36.0);
                const double cb = fma(-4.0 * i2, S1 + l0, 2.0 * gam2 * Q) * eg, cy = 12.0 * i2 * eg, cv = 4.0 * i1 * eg;
                const double fx = fx_to(Fx, kf), fy = fx_to(Fy, kf), fz = fx_to(Fz, kf);
                const double fb = fma(bx, fx, fma(by, fy, bz * fz));
                an = fma(3.0 * i1, fb, fx_to(Fs, kf)) * (gam * (1.0 / 36.0));
                const double ng = n * gam * (1.0 / 12.0) * i1, cs = fma(an * n, gam2, cb);
                ax = fma(cy, yx, fma(cv, vx, fma(ng, fx, cs * bx)));
                ay = fma(cy, yy, fma(cv, vy, fma(ng, fy, cs * by)));
                az = fma(cy, yz, fma(cv, vz, fma(ng, fz, cs * bz)));
            } else {
                double df[19], dg[19];
                for (int i = 0; i < 19; ++i) {
                    df[i] = (double)lf[i] * (uf ? 0x1p-96 : 1.0);
                    dg[i] = (double)lg[i] * (um ? 0x1p-96 : 1.0);
                }
                eq_fields_adjoint(df, dg, n, e, bx, by, bz, ph, an, ae, ax, ay, az);
            }
            if (inflow) {
                bin0 = ax, bin1 = ay, bin2 = az;
                an = ae = ax = ay = az = 0;
            }
        }
        dn[idx] = an;
        de[idx] = ae;
        db[idx] = ax;
        db[g.N + idx] = ay;
        db[2 * (long long)g.N + idx] = az;
    }
    block_reduce4(0.0, bin0, bin1, bin2, red);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
static inline int adj_blocks(int N) { return (N + 127) / 128; }

cudaError_t launch_adjoint_macro(int prec, const Geom& g, const Phys& ph, const void* A, const double* dn,
                                 const double* deps, const double* dbeta, void* lam, cudaStream_t st) {
    const unsigned nb = (unsigned)((g.N + 127) / 128);
    set_last_launch_count(1);
    if (prec == 0)
        k_adjoint_macro<double><<<nb, 128, 0, st>>>((const double*)A, dn, deps, dbeta, (double*)lam, g, ph);
    else
        k_adjoint_macro<float><<<nb, 128, 0, st>>>((const float*)A, dn, deps, dbeta, (float*)lam, g, ph);
    return cudaGetLastError();
}

namespace {
// The calling thread's current context (the device's primary context under
// the runtime API), through the driver entry point the runtime hands out, so
// that the library needs no link against the driver library.
CUcontext current_context() {
    using Fn = CUresult (*)(CUcontext*);
    static Fn fn = nullptr;
    static bool looked = false;
    if (!looked) {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 4000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<Fn>(f);
        looked = true;
    }
    CUcontext c = nullptr;
    if (fn) fn(&c);
    return c;
}

// The dynamic shared memory opt-in of a staged kernel, once per context and
// kernel (the attribute belongs to the kernel in a context: a new context
// after a reset needs it again; setting it on every launch costs a host-side
// call that held back the launch queue of short steps).
std::mutex g_optin_mu;
struct OptIn {
    CUcontext ctx;
    const void* kern;
};
OptIn g_optin[64];
int g_optin_n = 0;

cudaError_t smem_opt_in(const void* kern, int bytes) {
    const CUcontext ctx = current_context();
    std::lock_guard<std::mutex> lock(g_optin_mu);
    for (int i = 0; i < g_optin_n; ++i)
        if (g_optin[i].ctx == ctx && g_optin[i].kern == kern) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && g_optin_n < 64) g_optin[g_optin_n++] = {ctx, kern};
    return e;
}
}  // namespace

// Launch of the fixed-point FP64 adjoint: eight lanes per cell while the
// lanes fit two warps per scheduler, else persistent blocks of 64 threads.
struct AdjFxShape {
    bool split;
    int grid, threads;
};
static AdjFxShape adj_fx_shape(long long N, int nsm) {
    if (N <= kAdjSplitCells && N <= 32ll * nsm) return {true, (int)((8 * N + 127) / 128), 128};
    const long long nb = (N + kAdjFxThreads - 1) / kAdjFxThreads, most = (long long)nsm * kAdjFxBlocks;
    return {false, (int)(nb < most ? nb : most), kAdjFxThreads};
}

static void launch_adjoint_fx(const Geom& g, const Phys& ph, const AdjConst<double>& c, const double* A,
                              const double* Li, double* Lo, const AdjSums& sums, const AdjFxShape& sh, const double* inflow_t,
                              cudaStream_t st) {
    AdjFx k;
    double qh, ql;
    fx_div2(5.0, 3.0, qh, ql);
    k.kS1 = fx_const(qh, ql, 62);
    fx_div2(1.0, 36.0, qh, ql);
    k.kS36 = fx_const_w(qh, ql, 65);
    k.kE1 = ph.fx.kE1;
    k.kE0 = ph.fx.kE0;
    auto go = [&](auto kern) { launch_dependent(kern, sh.grid, sh.threads, 0, st, A, Li, Lo, g, ph, c, k, sums, inflow_t); };
    switch (g.xbc) {
        case XBC_PERIODIC:
            sh.split ? go(k_adjoint_step_fx_split<XBC_PERIODIC>) : go(k_adjoint_step_fx<XBC_PERIODIC>);
            break;
        case XBC_INFLOW_OUTFLOW:
            sh.split ? go(k_adjoint_step_fx_split<XBC_INFLOW_OUTFLOW>) : go(k_adjoint_step_fx<XBC_INFLOW_OUTFLOW>);
            break;
        default:
            sh.split ? go(k_adjoint_step_fx_split<XBC_OUTFLOW_BOTH>) : go(k_adjoint_step_fx<XBC_OUTFLOW_BOTH>);
            break;
    }
}

template <typename T>
static int adjoint_step_t(const Geom& g, const Phys& ph, const T* A, const T* Li, T* Lo, const AdjSums& sums, int nb,
                          const double* inflow_d, cudaStream_t st) {
    const AdjConst<T> c = make_adj_const<T>(ph);
    const T* inflow_t = inflow_table<T>(inflow_d);
    static int nsm = 0;
    auto persistent_grid = [&](int minb) {
        if (nsm == 0) {
            int dev = 0;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        }
        const int pg = nsm * minb;
        return pg < nb ? pg : nb;
    };
    // returns the number of warps whose partial sums are left for k_finalize
    // (0: a kernel that adds up its own)
    auto go = [&](auto kern, bool pipe, int minb) {
        const int grid = pipe ? persistent_grid(minb) : nb;
        kern<<<grid, 128, 0, st>>>(A, Li, Lo, g, ph, c, sums, inflow_t);
        return pipe ? 0 : grid * 4;
    };
    int warps = 0;
    if constexpr (sizeof(T) == 4) {
        if (g.adj_pipe == 2) {
            const int coop = g.adj_coop;
            PlaneTab tab;
            for (int q = 0; q < 38; ++q) {
                tab.a[q] = (const float*)A + (long long)q * g.S;
                tab.l[q] = (const float*)Li + (long long)q * g.S;
                tab.o[q] = (float*)Lo + (long long)q * g.S;
            }
            auto staged = [&](auto kern) {
                smem_opt_in((const void*)kern, (int)kStageSmemBytes);  // a failure shows at the launch
                const int grid = persistent_grid(3);
                launch_dependent(kern, grid, kStageThreads, kStageSmemBytes, st, A, Li, Lo, g, ph, c, sums.red, inflow_t, tab);
                return grid * (kStageThreads / 32);
            };
            // 16-byte copies of lambda_t+1: the buffer must be 16-byte aligned
            if (coop && ((uintptr_t)Li & 15u) == 0) {
                switch (g.xbc) {
                    case XBC_PERIODIC: return staged(k_adjoint_step_coop<XBC_PERIODIC>);
                    case XBC_INFLOW_OUTFLOW: return staged(k_adjoint_step_coop<XBC_INFLOW_OUTFLOW>);
                    default: return staged(k_adjoint_step_coop<XBC_OUTFLOW_BOTH>);
                }
            }
            switch (g.xbc) {
                case XBC_PERIODIC: return staged(k_adjoint_step_staged<XBC_PERIODIC>);
                case XBC_INFLOW_OUTFLOW: return staged(k_adjoint_step_staged<XBC_INFLOW_OUTFLOW>);
                default: return staged(k_adjoint_step_staged<XBC_OUTFLOW_BOTH>);
            }
        }
    }
    if constexpr (sizeof(T) == 8) {
        // persistent (the instantiation the allocation-free step runs too)
        if (ph.fx_on) {
            persistent_grid(1);  // the SM count
            const AdjFxShape sh = adj_fx_shape(g.N, nsm);
            launch_adjoint_fx(g, ph, c, A, Li, Lo, sums, sh, inflow_t, st);
            return 0;
        }
        switch (g.xbc) {
            case XBC_PERIODIC: warps = go(k_adjoint_step<T, XBC_PERIODIC, 2, true>, true, 2); break;
            case XBC_INFLOW_OUTFLOW: warps = go(k_adjoint_step<T, XBC_INFLOW_OUTFLOW, 2, true>, true, 2); break;
            default: warps = go(k_adjoint_step<T, XBC_OUTFLOW_BOTH, 2, true>, true, 2); break;
        }
    } else if (g.adj_pipe) {
        switch (g.xbc) {
            case XBC_PERIODIC: warps = go(k_adjoint_step<T, XBC_PERIODIC, 4, true>, true, 4); break;
            case XBC_INFLOW_OUTFLOW: warps = go(k_adjoint_step<T, XBC_INFLOW_OUTFLOW, 4, true>, true, 4); break;
            default: warps = go(k_adjoint_step<T, XBC_OUTFLOW_BOTH, 4, true>, true, 4); break;
        }
    } else {
        switch (g.xbc) {
            case XBC_PERIODIC: warps = go(k_adjoint_step<T, XBC_PERIODIC, 4, false>, false, 4); break;
            case XBC_INFLOW_OUTFLOW: warps = go(k_adjoint_step<T, XBC_INFLOW_OUTFLOW, 4, false>, false, 4); break;
            default: warps = go(k_adjoint_step<T, XBC_OUTFLOW_BOTH, 4, false>, false, 4); break;
        }
    }
    return warps;
}

cudaError_t launch_adjoint_step(int prec, const Geom& g, const Phys& ph, const void* A, const void* lam_in,
                                void* lam_out, double* red, unsigned* ticket, const double* inflow_d, double* dtau,
                                double* dbeta_in, cudaStream_t st) {
    const int nb = adj_blocks(g.N);
    const AdjSums sums{red, ticket, dtau, dbeta_in};
    int warps;
    if (prec == 0)
        warps = adjoint_step_t<double>(g, ph, (const double*)A, (const double*)lam_in, (double*)lam_out, sums, nb,
                                       inflow_d, st);
    else
        warps = adjoint_step_t<float>(g, ph, (const float*)A, (const float*)lam_in, (float*)lam_out, sums, nb,
                                      inflow_d, st);
    if (warps) launch_dependent(k_finalize, g.xbc == XBC_INFLOW_OUTFLOW ? 4 : 1, 256, 0, st, red, warps, dtau, dbeta_in);
    set_last_launch_count(warps ? 2 : 1);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_fields(int prec, const Geom& g, const Phys& ph, const double* n0, const double* eps0,
                                  const double* beta0, const void* A0, const void* lam0, double* dn0, double* deps0,
                                  double* dbeta0, double* red, double* dbeta_in, cudaStream_t st) {
    const int nb = adj_blocks(g.N);
    set_last_launch_count(2);
    if (prec == 0)
        k_adjoint_fields<double><<<nb, 128, 0, st>>>(n0, eps0, beta0, (const double*)A0, (const double*)lam0, dn0,
                                                     deps0, dbeta0, g, ph, red);
    else
        k_adjoint_fields<float><<<nb, 128, 0, st>>>(n0, eps0, beta0, (const float*)A0, (const float*)lam0, dn0, deps0,
                                                    dbeta0, g, ph, red);
    // without an inflow plane every dL/dbeta_in term is zero
    if (g.xbc == XBC_INFLOW_OUTFLOW)
        launch_dependent(k_finalize, 4, 256, 0, st, red, nb, (double*)nullptr, dbeta_in);
    else
        set_last_launch_count(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Allocation-free adjoint step.  Same kernels as launch_adjoint_step, always
// as the persistent grid-stride launch (grid = SMs x resident blocks, capped
// at the block count), with the partial sums in a fixed static device array
// instead of the context workspace.  Every launch writes all the slots it
// reads (4 per block, in the staged kernel per warp), so the array needs no
// zeroing; two launches that overlap in time on one device (other contexts)
// share it and race, for their own sums only (AdjSums).
// ---------------------------------------------------------------------------
static __device__ __align__(256) double g_adj_scratch[kAdjScratchDoubles];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
struct ScratchSetup {
    double* ptr;    // device address of g_adj_scratch in the context below
    int nsm;        // SM count of the device
    CUcontext ctx;  // the context the set-up was made in
};
ScratchSetup g_scratch[kMaxDevices];

// Set-up, with the device current: the device address of g_adj_scratch, the
// SM count, and every kernel this entry point launches loaded onto the
// device (cudaFuncGetAttributes loads a kernel that lazy module loading has
// not loaded yet), so that no later call loads code, which can allocate.
// Redone when the device's context is not the one it was made in (after
// cudaDeviceReset the old address is stale).
cudaError_t scratch_for_device(int dev, double** ptr, int* nsm) {
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    const CUcontext ctx = current_context();
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    ScratchSetup& s = g_scratch[dev];
    if (!s.ptr || s.ctx != ctx) {
        s.ptr = nullptr;
        double* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress((void**)&p, g_adj_scratch);
        if (e != cudaSuccess) return e;
        int n = 0;
        e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        const void* kernels[] = {
            (const void*)k_adjoint_step<double, XBC_PERIODIC, 2, true>,
            (const void*)k_adjoint_step<double, XBC_INFLOW_OUTFLOW, 2, true>,
            (const void*)k_adjoint_step<double, XBC_OUTFLOW_BOTH, 2, true>,
            (const void*)k_adjoint_step<float, XBC_PERIODIC, 4, true>,
            (const void*)k_adjoint_step<float, XBC_INFLOW_OUTFLOW, 4, true>,
            (const void*)k_adjoint_step<float, XBC_OUTFLOW_BOTH, 4, true>,
            (const void*)k_adjoint_step_fx<XBC_PERIODIC>,
            (const void*)k_adjoint_step_fx<XBC_INFLOW_OUTFLOW>,
            (const void*)k_adjoint_step_fx<XBC_OUTFLOW_BOTH>,
            (const void*)k_adjoint_step_fx_split<XBC_PERIODIC>,
            (const void*)k_adjoint_step_fx_split<XBC_INFLOW_OUTFLOW>,
            (const void*)k_adjoint_step_fx_split<XBC_OUTFLOW_BOTH>,
            (const void*)k_finalize,
        };
        for (const void* k : kernels) {
            cudaFuncAttributes attr;
            e = cudaFuncGetAttributes(&attr, k);
            if (e != cudaSuccess) return e;
        }
        // the FP32 staged kernels (block-copy and per-thread forms): loaded,
        // and their shared memory opted in
        const void* staged[] = {
            (const void*)k_adjoint_step_coop<XBC_PERIODIC>,   (const void*)k_adjoint_step_coop<XBC_INFLOW_OUTFLOW>,
            (const void*)k_adjoint_step_coop<XBC_OUTFLOW_BOTH>, (const void*)k_adjoint_step_staged<XBC_PERIODIC>,
            (const void*)k_adjoint_step_staged<XBC_INFLOW_OUTFLOW>, (const void*)k_adjoint_step_staged<XBC_OUTFLOW_BOTH>,
        };
        for (const void* k : staged) {
            cudaFuncAttributes attr;
            e = cudaFuncGetAttributes(&attr, k);
            if (e == cudaSuccess) e = smem_opt_in(k, (int)kStageSmemBytes);
            if (e != cudaSuccess) return e;
        }
        s.nsm = n;
        s.ctx = ctx;
        s.ptr = p;
    }
    *ptr = s.ptr;
    *nsm = s.nsm;
    return cudaSuccess;
}

template <typename T, int MINB>
int adjoint_step_noalloc_t(const Geom& g, const Phys& ph, const T* A, const T* Li, T* Lo, const AdjSums& sums, int grid,
                           const double* inflow_d, cudaStream_t st) {
    const AdjConst<T> c = make_adj_const<T>(ph);
    const T* inflow_t = inflow_table<T>(inflow_d);
    switch (g.xbc) {
        case XBC_PERIODIC:
            k_adjoint_step<T, XBC_PERIODIC, MINB, true><<<grid, 128, 0, st>>>(A, Li, Lo, g, ph, c, sums, inflow_t);
            break;
        case XBC_INFLOW_OUTFLOW:
            k_adjoint_step<T, XBC_INFLOW_OUTFLOW, MINB, true><<<grid, 128, 0, st>>>(A, Li, Lo, g, ph, c, sums, inflow_t);
            break;
        default:
            k_adjoint_step<T, XBC_OUTFLOW_BOTH, MINB, true><<<grid, 128, 0, st>>>(A, Li, Lo, g, ph, c, sums, inflow_t);
            break;
    }
    return grid;
}
}  // namespace

cudaError_t launch_adjoint_step_noalloc(int prec, const Geom& g, const Phys& ph, const void* A, const void* lam_in,
                                        void* lam_out, unsigned* ticket, const double* inflow_d, double* dtau,
                                        double* dbeta_in, cudaStream_t st, long long* need_doubles) {
    set_last_launch_count(0);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    double* red = nullptr;
    int nsm = 0;
    e = scratch_for_device(dev, &red, &nsm);
    const AdjSums sums{red, ticket, dtau, dbeta_in};
    if (e != cudaSuccess) return e;
    const int nb = adj_blocks(g.N);
    if (prec == 0 && ph.fx_on) {
        const AdjFxShape sh = adj_fx_shape(g.N, nsm);
        const long long need = 4ll * sh.grid;  // 4 partial sums per block (block_sums)
        if (need_doubles) *need_doubles = need;
        if (need > kAdjScratchDoubles) return cudaErrorInvalidValue;
        set_last_launch_count(1);
        launch_adjoint_fx(g, ph, make_adj_const<double>(ph), (const double*)A, (const double*)lam_in, (double*)lam_out,
                          sums, sh, inflow_table<double>(inflow_d), st);
        return cudaGetLastError();
    }
    if (prec != 0 && g.adj_pipe == 2) {
        // FP32 with the default kernel choice: the staged kernel that
        // rlb_adjoint_step runs (persistent, SMs x 3 blocks of 128)
        const int grid3 = nsm * 3 < nb ? nsm * 3 : nb;
        const long long need = 16ll * grid3;  // 4 partial sums per warp (k_finalize adds them up)
        if (need_doubles) *need_doubles = need;
        if (need > kAdjScratchDoubles) return cudaErrorInvalidValue;
        const int warps = adjoint_step_t<float>(g, ph, (const float*)A, (const float*)lam_in, (float*)lam_out, sums, nb,
                                                inflow_d, st);
        launch_dependent(k_finalize, g.xbc == XBC_INFLOW_OUTFLOW ? 4 : 1, 256, 0, st, red, warps, dtau, dbeta_in);
        set_last_launch_count(2);
        return cudaGetLastError();
    }
    const int minb = prec == 0 ? 2 : 4;
    const int grid = nsm * minb < nb ? nsm * minb : nb;
    const long long need = 4ll * grid;  // 4 partial sums per block (block_sums)
    if (need_doubles) *need_doubles = need;
    if (need > kAdjScratchDoubles) return cudaErrorInvalidValue;
    set_last_launch_count(1);
    if (prec == 0)
        adjoint_step_noalloc_t<double, 2>(g, ph, (const double*)A, (const double*)lam_in, (double*)lam_out, sums, grid,
                                          inflow_d, st);
    else
        adjoint_step_noalloc_t<float, 4>(g, ph, (const float*)A, (const float*)lam_in, (float*)lam_out, sums, grid,
                                         inflow_d, st);
    return cudaGetLastError();
}

// Bounds-check count of this translation unit (0 in the release build).
RLB_OOB_TAKE_FN(oob_take_adjoint)

}  // namespace rlb
