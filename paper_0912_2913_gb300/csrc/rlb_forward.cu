// rlb_forward.cu -- the FP32 fused stream-and-collide step of the relativistic
// lattice Boltzmann scheme (Eqs. lbe1, lbe2 with the eps = 3P equilibria Eqs.
// equil1s, equil2as, equil2bs); the FP64 one is in rlb_step64.cu, the
// equilibrium initialisation and the macroscopic output in rlb_fields.cu.
//
// One thread owns one cell.  A step pulls the 38 populations that arrive at
// the cell (h_i(x) = A_i(x - e_i), link bounce-back h_i(x) = A_opp(i)(x) when
// x - e_i is solid), forms the five moments, recovers (n gamma, eps, beta) in
// closed form, builds the equilibria pair by pair (velocities i and opp(i)
// share every term but the odd one) and writes the BGK-relaxed populations
// B_i = h_i + (eq_i - h_i)/tau.  State planes are structure-of-arrays, so a
// warp's loads and stores of one plane are 32 consecutive elements (the x
// neighbours are off by one element and share cache sectors).
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "rlb_collide.cuh"
#include "rlb_device.cuh"

namespace rlb {

namespace {
int g_last_launches = 0;
}
int last_launch_count() { return g_last_launches; }
void set_last_launch_count(int n) { g_last_launches = n; }


// ---------------------------------------------------------------------------
// FP32 deviation step.  Populations are stored as d_i = p_i - p_i^ref with
// p^ref the rest equilibrium of (n_ref, eps_ref): f_i^ref = w_i n_ref,
// g_i^ref = w_i eps_ref / c_l^2 (i > 0), g_0^ref = w_0 eps_ref (3 - 2/c_l^2).
// Streaming and BGK are linear and the reference is uniform and symmetric, so
// the step maps deviations to deviations.  The moments are the reference
// moments (n_ref, eps_ref, 0) plus the float sums of the deviations; the
// recovery, where the strong-shock cancellation sits, runs in FP64:
//   E = eps_ref + sum dg,  sqrt(E^2 - 3M^2/4) and 1/(3E + eps) each from a
//   binary32 seed and one FP64 Newton correction (relative error ~1e-14),
//   eps = 2 sqrt(...) - E, beta = 3 M / (3E + eps), 1 - |beta|^2 in FP64.
// The equilibrium deviations are formed without cancellation:
//   df_i = w_i [dS + 3 S q_i / c_l]
//   dg_i = w_i [d_eps / c_l^2 + eps gamma^2 (6 q_i^2 - 2 b2) / c_l^2] +- w_i eps gamma^2 4 q_i / c_l
//   dg_0 = w_0 [d_eps (3 - 2/c_l^2) + eps gamma^2 b2 (4 - 2/c_l^2)]
// with dS = sum df, d_eps = eps - eps_ref (FP64, then rounded).
// ---------------------------------------------------------------------------

// MINB: resident 256-thread blocks per SM the register budget is cut for;
// PREF: prefetch the populations of the f phase into L2 before the g phase
// runs (the default launch: the f loads then hit L2 instead of waiting on
// HBM, measured +16% on the 200x100x100 sphere).
// I: type of the element offsets, int when 38 S < 2^31 (fewer address
// instructions: measured +2 % / +6 % for two of the shapes on the
// 200x100x100 sphere), else long long.
// COMP: the compensated collision (collide_cell_f32c), run for c_l > 1.
// EARLY: the f populations are loaded before the g phase's arithmetic.
// TB: threads per block the register budget is cut for.
// BOTH: the one fluid plane of three is copied by both outflow ghosts (a test
// of nx beside the stores cost a lattice that is not so narrow 10 to 50 % of
// its step: 1600 cells 2.9 -> 4.3 us).
template <int XBC, bool SOLID, int MINB, bool PREF, typename I = long long, bool COMP = false, bool EARLY = false,
          int TB = 256, bool BOTH = false>
__global__ void __launch_bounds__(TB, MINB) k_step_f32(const float* __restrict__ A, float* __restrict__ B, Geom g,
                                                       Dev32 c, Counters cnt, int count, long long step_index) {
    const int idx = dependent_begin(blockIdx.x * blockDim.x + threadIdx.x);
    if (idx >= g.N) return;
    int x, y, z;
    cell_coords(g, idx, x, y, z);
    if (g.zhalo && (z == 0 || z == g.nz - 1)) return;  // z halo planes: filled by the exchange
    const I S = (I)g.S;
    // I = unsigned: the f planes (0..18) and the g planes (19..37) are
    // addressed from their own base pointers with unsigned 32-bit element
    // offsets (for lattices with 38 S >= 2^31 and 19 S < 2^32), which costs
    // no more address arithmetic than the int offsets.
    constexpr bool SPLIT = std::is_same<I, unsigned>::value;
    const float* __restrict__ Ag = SPLIT ? A + 19ll * g.S : A;
    float* Bg = SPLIT ? B + 19ll * g.S : B;
    const long long lim = (SPLIT ? 19ll : 38ll) * g.S;  // extent the checked builds test against
    auto pq = [](int q) { return (SPLIT && q >= 19) ? q - 19 : q; };  // plane number within its base
    auto abase = [&](int q) { return (SPLIT && q >= 19) ? Ag : A; };
    // The inflow column keeps its populations: its lanes load them through
    // offsets of zero and store them as loaded, along with their warp (a copy
    // loop of its own was a second pass over memory for every warp that holds
    // such a cell: all warps of a lattice 63 cells wide).
    const bool keep = XBC == XBC_INFLOW_OUTFLOW && x == 0;
    if (XBC != XBC_PERIODIC && (x == g.nx - 1 || (x == 0 && !keep))) return;
    PullOffsets o(g, x, y, z);
    if (keep) o.xm = o.xp = o.ym = o.yp = o.zm = o.zp = 0;
    const int dup = dup_of<XBC>(x, g.nx);
    float* Bc = B + idx;
    float* Bgc = Bg + idx;
    auto put = [&](int q, float v, float old) {
        if (XBC == XBC_INFLOW_OUTFLOW && keep) v = old;
        if constexpr (SPLIT) {
            float* b = q >= 19 ? Bgc : Bc;
            b[RLB_CHK_OFF(pq(q) * S, idx, lim)] = v;
            // the outflow copy: dup (+-1) moves the pointer, so that the
            // unsigned offset never has to hold a negative value
            if (dup) (b + dup)[RLB_CHK_OFF(pq(q) * S, idx + dup, lim)] = v;
        } else {
            Bc[RLB_CHK_OFF(q * S, idx, 38ll * S)] = v;
            if (dup) Bc[RLB_CHK_OFF(q * S + dup, idx, 38ll * S)] = v;
            if (BOTH) Bc[RLB_CHK_OFF(q * S - 1, idx, 38ll * S)] = v;
        }
    };
    if (PREF) {
#pragma unroll
        for (int i = 0; i < 19; ++i) asm volatile("prefetch.global.L2 [%0];" ::"l"(RLB_CHK_PTR(A, i * S + idx + o.src(i), lim)));
    }
    auto fetch = [&](int q, int i) {
        if constexpr (SPLIT)
            return __ldg(RLB_CHK_PTR(abase(q), pq(q) * S + idx + o.src(i), lim));
        else
            return __ldg(RLB_CHK_PTR(A, q * S + idx + o.src(i), 38ll * S));
    };
    auto bounce = [&](int q, int i) {  // link bounce-back
        const int r = XBC == XBC_INFLOW_OUTFLOW && keep ? q : q - i + opp(i);
        if constexpr (SPLIT)
            return __ldg(RLB_CHK_PTR(abase(q), pq(r) * S + idx, lim));
        else
            return __ldg(RLB_CHK_PTR(A, r * S + idx, 38ll * S));
    };
    bool unphys, nonpos, fluid;
    if (COMP)
        fluid = collide_cell_f32c<SOLID>(fetch, bounce, put, c, unphys, nonpos);
    else
        fluid = collide_cell_f32<SOLID, decltype(fetch), decltype(bounce), decltype(put), EARLY>(fetch, bounce, put, c,
                                                                                                unphys, nonpos);
    if (!fluid) {  // keep the marker (found among the gathered values: a load of it before them is a round trip more)
        const float m = solid_marker_f();
#pragma unroll
        for (int q = 0; q < 38; ++q) ((SPLIT && q >= 19) ? Bgc : Bc)[RLB_CHK_OFF(pq(q) * S, idx, lim)] = m;
        return;
    }
    if (count && !keep) count_flags(cnt, unphys, nonpos, (unsigned long long)step_index * (unsigned long long)g.N + idx);
}

// Persistent variant: a grid of (SMs x resident blocks) threads walks the
// lattice with a grid stride; before colliding its current cell a thread
// issues L2 prefetches for all 38 populations of its next cell, so every
// gather hits L2 while HBM streams the next cells in (software pipelining
// without registers).  Same per-cell arithmetic as k_step_f32.
template <int XBC, bool SOLID, bool CS>
__global__ void __launch_bounds__(256, 3) k_step_f32_pipe(const float* __restrict__ A, float* __restrict__ B, Geom g,
                                                          Dev32 c, Counters cnt, int count, long long step_index) {
    const long long S = g.S;
    const long long stride = (long long)gridDim.x * blockDim.x;
    auto prefetch_cell = [&](int idx) {
        int x, y, z;
        cell_coords(g, idx, x, y, z);
        if (XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1)) return;
        if (g.zhalo && (z == 0 || z == g.nz - 1)) return;
        const PullOffsets o(g, x, y, z);
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(RLB_CHK_PTR(A, (19 + i) * S + idx + o.src(i), 38ll * S)));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(RLB_CHK_PTR(A, i * S + idx + o.src(i), 38ll * S)));
        }
    };
    // 64-bit loop counter: li + stride cannot wrap for any accepted N
    long long li = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (li < g.N) prefetch_cell((int)li);
    for (; li < g.N; li += stride) {
        const int idx = (int)li;
        if (li + stride < g.N) prefetch_cell((int)(li + stride));
        int x, y, z;
        cell_coords(g, idx, x, y, z);
        if (g.zhalo && (z == 0 || z == g.nz - 1)) continue;
        if (XBC != XBC_PERIODIC && (x == 0 || x == g.nx - 1)) {
            if (XBC == XBC_INFLOW_OUTFLOW && x == 0) {
#pragma unroll
                for (int q = 0; q < 38; ++q) B[RLB_CHK(q * S + idx, 38ll * S)] = __ldg(RLB_CHK_PTR(A, q * S + idx, 38ll * S));
            }
            continue;
        }
        const PullOffsets o(g, x, y, z);
        const int dup = dup_of<XBC>(x, g.nx);
        float* Bc = B + idx;
        auto put = [&](int q, float v, float) {
            if (CS) {
                __stcs(Bc + q * S, v);
                if (dup) __stcs(Bc + q * S + dup, v);
            } else {
                Bc[RLB_CHK_OFF(q * S, idx, 38ll * S)] = v;
                if (dup) Bc[RLB_CHK_OFF(q * S + dup, idx, 38ll * S)] = v;
            }
        };
        if (SOLID && is_solid(__ldg(RLB_CHK_PTR(A, 19 * S + idx, 38ll * S)))) {
            const float m = solid_marker_f();
#pragma unroll
            for (int q = 0; q < 38; ++q) Bc[RLB_CHK_OFF(q * S, idx, 38ll * S)] = m;
            continue;
        }
        auto fetch = [&](int q, int i) { return __ldg(RLB_CHK_PTR(A, q * S + idx + o.src(i), 38ll * S)); };
        auto bounce = [&](int q, int i) { return __ldg(RLB_CHK_PTR(A, (q - i + opp(i)) * S + idx, 38ll * S)); };
        bool unphys, nonpos;
        collide_cell_f32<SOLID>(fetch, bounce, put, c, unphys, nonpos);
        if (count) count_flags(cnt, unphys, nonpos, (unsigned long long)step_index * (unsigned long long)g.N + idx);
    }
}

__global__ void k_conversions(const float* __restrict__ fi, const double* __restrict__ di, long long n,
                              double* __restrict__ fo, float* __restrict__ dout) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        fo[k] = f2d(fi[k]);
        dout[k] = d2f(di[k]);
    }
}

cudaError_t launch_conversions(const float* fi, const double* di, long long n, double* fo, float* dout) {
    if (n > 0) k_conversions<<<1024, 256>>>(fi, di, n, fo, dout);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    return e;
}

__global__ void k_check_solid_planes(Geom g, const uint8_t* __restrict__ solid, unsigned long long* flag) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int plane = g.ny * g.nz;
    if (t >= 4 * plane) return;
    const int which = t / plane, yz = t - which * plane;
    const int xs[4] = {0, 1, g.nx - 2, g.nx - 1};
    if (solid[(long long)yz * g.nx + xs[which]]) atomicAdd(flag, 1ull);
}

// ---------------------------------------------------------------------------
// Halo exchange of a z decomposition.  Plane q of a state is [z][y][x], so
// the values of one population on one z plane are nxy consecutive elements.
// blockIdx.y = 0..19: segments 0..9 carry the ten populations with e_z = +1
// (f then g) from lower's plane nz_l - 2 to upper's plane 0; segments 10..19
// the ten with e_z = -1 from upper's plane 1 to lower's plane nz_l - 1.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int zface_velocity(int j, int sign) {  // j-th velocity (0..4) with e_z = sign
    int k = 0;
    for (int i = 1; i < 19; ++i)
        if (vel_z(i) == sign) {
            if (k == j) return i;
            ++k;
        }
    return -1;
}

template <typename T>
__global__ void k_halo_exchange(long long nxy, T* __restrict__ lower, long long S_l, int nz_l, T* __restrict__ upper,
                                long long S_u) {
    const int seg = blockIdx.y;
    const bool up = seg < 10;
    const int j = up ? seg : seg - 10;
    const int i = zface_velocity(j % 5, up ? 1 : -1);
    const int q = (j < 5 ? 0 : 19) + i;
    const T* src = up ? lower + q * S_l + (long long)(nz_l - 2) * nxy : upper + q * S_u + nxy;
    T* dst = up ? upper + q * S_u : lower + q * S_l + (long long)(nz_l - 1) * nxy;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nxy; k += (long long)gridDim.x * blockDim.x)
        dst[k] = src[k];
}

cudaError_t launch_halo_exchange(int elem, long long nxy, void* lower, long long S_lower, int nz_lower, void* upper,
                                 long long S_upper, cudaStream_t st) {
    g_last_launches = 1;
    long long nb = (nxy + 255) / 256;
    if (nb > 4096) nb = 4096;
    const dim3 grid((unsigned)nb, 20);
    if (elem == 8)
        k_halo_exchange<double><<<grid, 256, 0, st>>>(nxy, (double*)lower, S_lower, nz_lower, (double*)upper, S_upper);
    else
        k_halo_exchange<float><<<grid, 256, 0, st>>>(nxy, (float*)lower, S_lower, nz_lower, (float*)upper, S_upper);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
static inline unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

Dev32 make_dev32(const Phys& ph) {
    Dev32 c;
    c.omega = (float)ph.omega;
    c.omw = (float)(1.0 - ph.omega);
    c.c_l = (float)ph.c_l;
    c.inv_cl = (float)ph.inv_cl;
    c.inv_cl2 = (float)ph.inv_cl2;
    c.n_ref = (float)ph.n_ref;
    c.g0a = (float)(3.0 - 2.0 * ph.inv_cl2);
    c.g0b = (float)(4.0 - 2.0 * ph.inv_cl2);
    c.eps_ref = ph.eps_ref;
    c.n_ref_d = ph.n_ref;
    c.c_l_d = ph.c_l;
    c.inv_cl_d = ph.inv_cl;
    c.inv_cl2_d = ph.inv_cl2;
    c.g0a_d = 3.0 - 2.0 * ph.inv_cl2;
    c.g0b_d = 4.0 - 2.0 * ph.inv_cl2;
    return c;
}

static int sm_count() {
    static int nsm = 0;
    if (nsm == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    }
    return nsm;
}

// Threads per block of the one-cell-per-thread step kernels: a lattice with
// fewer blocks than SMs (the 1600-cell shock tube) runs 32-thread blocks, so
// that its cells spread over up to 32x more SMs (the per-cell arithmetic,
// FP64 above all, is then the step's latency).  Results do not depend on it.
static int step_block(long long N, int full) { return blocks_for(N, full) < (unsigned)sm_count() ? 32 : full; }

// Launch shape of the FP32 step (all give the same bits), by how the lattice
// fills the chip: r = cells per SM / 128, one warp on each scheduler per unit.
// Shape 8, f loaded before the g arithmetic in 64-thread blocks x 12 per SM, is
// the fastest where blocks are many (us a step, shapes 2 / 7 / 8: 200x100x100
// sphere 102.5 / 93.6 / 91.5; 256^3 844 / 750 / 739; 512^3 6740 / 5982 / 5880)
// or fit easily (r = 0.5: 3.8 / 3.2 / 3.0; 2.5: 5.7 / 4.3 / 4.1).  In between a
// shape takes a step up where another block goes on the busiest SM (2 of 256
// threads at r = 4, 7 of 128 at 3.5, 8 of 64 at 3) and where its resident
// blocks are used up (7 at r = 7 and 14, 8 at 6 and 12), the same for
// 1D, 3D, periodic and inflow lattices:
//   r = 3.0    5.9 / 4.2 / 4.2     r = 3.01   5.8 / 4.7 / 6.1     r = 3.5    5.8 / 5.1 / 6.3
//   r = 3.51   5.8 / 6.8 / 6.3     r = 4.0    5.8 / 6.8 / 6.4     r = 4.01   8.7 / 6.8 / 6.4
//   r = 5.98   9.3 / 7.1 / 6.3     r = 6.1    9.4 / 7.1 / 7.2     r = 7.0    9.4 / 6.9 / 7.8
//   r = 8.0    9.3 / 8.4 / 8.5     r = 8.9   10.9 / 9.0 / 9.0     r = 11.9  12.9 / 10.7 / 10.8
//   r = 12.5  14.0 / 11.2 / 11.7   r = 14.0  15.0 / 12.6 / 13.2   r = 14.9  16.6 / 13.8 / 14.2
//   r = 16.0  17.5 / 15.4 / 15.2   r = 18.8  21.8 / 18.7 / 18.2   r = 32    35.8 / 33.3 / 31.0
static int f32_shape(long long N) {
    const long long r2 = (N + 64ll * sm_count() - 1) / (64ll * sm_count());  // 2 r, rounded up
    if (r2 == 7) return 7;
    if (r2 == 8) return 2;
    return (r2 > 12 && r2 <= 17) || (r2 > 24 && r2 <= 30) ? 7 : 8;
}

template <int XBC, bool SOLID>
static void launch_step_t(int prec, const Geom& g, const Phys& ph, const void* A, void* B, Counters cnt, bool count,
                          long long step_index, cudaStream_t st) {
    if (prec == 0) {
        if (g.f64df)
            launch_step_f64_df(g, ph, A, B, cnt, count, step_index, st, step_block(g.N, 128));
        else
            launch_step_f64(g, ph, A, B, cnt, count, step_index, st);
    } else {
        const Dev32 c = make_dev32(ph);
        const int tb = step_block(g.N, 256);
        const unsigned nb = blocks_for(g.N, tb);
        const int cs = count ? 1 : 0;
        const bool idx32 = 38 * g.S < (1ll << 31);
        const bool split32 = !idx32 && 19 * g.S < (1ll << 32);  // unsigned offsets per population set
        if constexpr (XBC == XBC_OUTFLOW_BOTH) {
            if (dup_both<XBC>(g.nx)) {  // every variant of the tuning knobs has the same bits
                const int t = tb < 128 ? tb : 128;
                auto go = [&](auto kern) {
                    launch_dependent(kern, blocks_for(g.N, t), t, 0, st, (const float*)A, (float*)B, g, c, cnt, cs, step_index);
                };
                if (ph.c_l > 1.0)
                    go(k_step_f32<XBC, SOLID, 5, false, long long, true, false, 128, true>);
                else
                    go(k_step_f32<XBC, SOLID, 7, false, long long, false, true, 128, true>);
                return;
            }
        }
        if (ph.c_l > 1.0) {
            // lattice speeds above 1: the compensated collision (one launch
            // shape; the TMA-staged and tuning variants use the binary32 one).
            // 128 threads x 5 per SM; 193x127x161, us a step: 256 x 2 614,
            // 128 x 5 561, 128 x 6 566, 64 x 12 568, 128 x 7 585
            const int t = tb < 128 ? tb : 128;
            const unsigned n = blocks_for(g.N, t);
            const float* a = (const float*)A;
            float* b = (float*)B;
            if (idx32)
                launch_dependent(k_step_f32<XBC, SOLID, 5, false, int, true, false, 128>, n, t, 0, st, a, b, g, c, cnt, cs, step_index);
            else if (split32)
                launch_dependent(k_step_f32<XBC, SOLID, 5, false, unsigned, true, false, 128>, n, t, 0, st, a, b, g, c, cnt, cs, step_index);
            else
                launch_dependent(k_step_f32<XBC, SOLID, 5, false, long long, true, false, 128>, n, t, 0, st, a, b, g, c, cnt, cs, step_index);
            return;
        }
        if (g.tma && launch_step_f32_tma(g, c, (const float*)A, (float*)B, cnt, count, step_index, st) == cudaSuccess)
            return;
        cudaGetLastError();
        const int variant = g.variant < 0 ? f32_shape(g.N) : g.variant;
        switch (variant) {
            case 0: launch_dependent(k_step_f32<XBC, SOLID, 3, false>, nb, tb, 0, st, (const float*)A, (float*)B, g, c, cnt, cs, step_index); break;
            case 1:
                if (idx32)
                    launch_dependent(k_step_f32<XBC, SOLID, 3, true, int>, nb, tb, 0, st, (const float*)A, (float*)B, g, c, cnt, cs, step_index);
                else if (split32)
                    launch_dependent(k_step_f32<XBC, SOLID, 3, true, unsigned>, nb, tb, 0, st, (const float*)A, (float*)B, g, c, cnt, cs,
                                                                               step_index);
                else
                    launch_dependent(k_step_f32<XBC, SOLID, 3, true>, nb, tb, 0, st, (const float*)A, (float*)B, g, c, cnt, cs, step_index);
                break;
            case 2:
                if (idx32)
                    launch_dependent(k_step_f32<XBC, SOLID, 4, false, int>, nb, tb, 0, st, (const float*)A, (float*)B, g, c, cnt, cs, step_index);
                else if (split32)
                    launch_dependent(k_step_f32<XBC, SOLID, 4, false, unsigned>, nb, tb, 0, st, (const float*)A, (float*)B, g, c, cnt, cs,
                                                                                step_index);
                else
                    launch_dependent(k_step_f32<XBC, SOLID, 4, false>, nb, tb, 0, st, (const float*)A, (float*)B, g, c, cnt, cs, step_index);
                break;
            case 3: launch_dependent(k_step_f32<XBC, SOLID, 4, true>, nb, tb, 0, st, (const float*)A, (float*)B, g, c, cnt, cs, step_index); break;
            case 6:
            case 7:
            case 8: {
                // the f populations loaded before the g arithmetic (EARLY), in
                // blocks of 128 threads x 6 or 7 per SM or 64 x 12 (80, 72 and
                // 80 registers)
                const float* a = (const float*)A;
                float* b = (float*)B;
                const int v = variant;
                const int t = v == 8 ? (tb < 64 ? tb : 64) : (tb < 128 ? tb : 128);
                const unsigned n = blocks_for(g.N, t);
#define RLB_EARLY_LAUNCH(MB, TBK)                                                                                        \
    do {                                                                                                                 \
        if (idx32) launch_dependent(k_step_f32<XBC, SOLID, MB, false, int, false, true, TBK>, n, t, 0, st, a, b, g, c, cnt, cs, step_index); \
        else if (split32) launch_dependent(k_step_f32<XBC, SOLID, MB, false, unsigned, false, true, TBK>, n, t, 0, st, a, b, g, c, cnt, cs, step_index); \
        else launch_dependent(k_step_f32<XBC, SOLID, MB, false, long long, false, true, TBK>, n, t, 0, st, a, b, g, c, cnt, cs, step_index); \
    } while (0)
                if (v == 6) RLB_EARLY_LAUNCH(6, 128);
                else if (v == 7) RLB_EARLY_LAUNCH(7, 128);
                else RLB_EARLY_LAUNCH(12, 64);
#undef RLB_EARLY_LAUNCH
                break;
            }
            case 4:
            case 5: {
                unsigned grid = (unsigned)sm_count() * (unsigned)(g.pipe_blocks > 0 ? g.pipe_blocks : 3);
                if (grid > nb) grid = nb;
                if (variant == 4)
                    k_step_f32_pipe<XBC, SOLID, false><<<grid, 256, 0, st>>>((const float*)A, (float*)B, g, c, cnt, cs, step_index);
                else
                    k_step_f32_pipe<XBC, SOLID, true><<<grid, 256, 0, st>>>((const float*)A, (float*)B, g, c, cnt, cs, step_index);
                break;
            }
            default: launch_dependent(k_step_f32<XBC, SOLID, 3, true>, nb, tb, 0, st, (const float*)A, (float*)B, g, c, cnt, cs, step_index); break;
        }
    }
}

cudaError_t launch_step(int prec, const Geom& g, const Phys& ph, const void* A, void* B, Counters cnt, bool count,
                        long long step_index, cudaStream_t st) {
    // The solid-marker checks are always compiled in: a lattice without
    // solid cells never matches the marker, and the check costs no memory
    // traffic.
    g_last_launches = 1;
    switch (g.xbc) {
        case XBC_PERIODIC: launch_step_t<XBC_PERIODIC, true>(prec, g, ph, A, B, cnt, count, step_index, st); break;
        case XBC_INFLOW_OUTFLOW:
            launch_step_t<XBC_INFLOW_OUTFLOW, true>(prec, g, ph, A, B, cnt, count, step_index, st);
            break;
        default: launch_step_t<XBC_OUTFLOW_BOTH, true>(prec, g, ph, A, B, cnt, count, step_index, st); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_check_solid_planes(const Geom& g, const uint8_t* solid, unsigned long long* flag,
                                      cudaStream_t st) {
    g_last_launches = 1;
    const long long n = 4ll * g.ny * g.nz;
    k_check_solid_planes<<<blocks_for(n, 256), 256, 0, st>>>(g, solid, flag);
    return cudaGetLastError();
}

// Bounds-check count of this translation unit (0 in the release build).
RLB_OOB_TAKE_FN(oob_take_forward)

#ifdef RLB_CHECK_BOUNDS
// The checker itself on one index (no memory is accessed with it): counts a
// violation and returns 0 when the index lies outside [0, n).
static __device__ long long g_rlb_chk_result;
__global__ void k_bounds_selftest(long long i, long long n) { g_rlb_chk_result = RLB_CHK(i, n); }

long long bounds_selftest(long long i, long long n, cudaStream_t s) {
    k_bounds_selftest<<<1, 1, 0, s>>>(i, n);
    long long r = -1;
    if (cudaMemcpyFromSymbolAsync(&r, g_rlb_chk_result, sizeof r, 0, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return -1;
    return r;
}
#endif

}  // namespace rlb
