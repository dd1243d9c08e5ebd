// Readout kernels (init, moments, population exchange, reductions) and the launcher
// table of the step kernels (plb_step.cuh), templated over lattice and storage.
// Instantiated once per storage precision (plb_kern_*.cu).
#pragma once
#include <cuda_runtime.h>

#include <map>
#include <utility>

#include "plb_device.cuh"
#include "plb_launch.h"
#include "plb_batch.cuh"
#include "plb_fused.cuh"
#include "plb_pair.cuh"
#include "plb_staged.cuh"
#include "plb_step.cuh"
#include "plb_tile.cuh"

// L2 prefetch one wave ahead in the FP32 fused pass (1) or not (0).
#ifndef PLB_L2_PREFETCH
#define PLB_L2_PREFETCH 1
#endif
// The same for FP16-shifted storage.
#ifndef PLB_L2_PREFETCH_HALF
#define PLB_L2_PREFETCH_HALF 0
#endif
// L2 prefetch distance of the fused pass in waves of resident blocks.
#ifndef PLB_PF_WAVES
#define PLB_PF_WAVES 1
#endif
// D3Q19 fused pass with the next plane staged in shared memory (plb_staged.cuh): FP16S storage
// (PLB_STAGED_HALF) and FP32 storage (PLB_STAGED_FLOAT).
#ifndef PLB_STAGED_HALF
#define PLB_STAGED_HALF 1
#endif
#ifndef PLB_STAGED_FLOAT
#define PLB_STAGED_FLOAT 0
#endif
// psi pass of FP16S storage over four cells per thread where nx is a multiple of 4.
#ifndef PLB_PSI_QUAD
#define PLB_PSI_QUAD 1
#endif
// Two cells per thread for FP16 storage (1) or one (0).
#ifndef PLB_HALF_PAIR
#define PLB_HALF_PAIR 1
#endif

namespace plb {

// Linear thread -> cell mapping (x fastest) for the readout kernels; 32-bit divisions where they do (the
// 64-bit ones are about 100 instructions each).
__device__ __forceinline__ bool cell_coords(const KParams &p, long long s, int &x, int &y, int &z) {
    if (s >= p.n) return false;
    if (p.n < (1LL << 31)) {
        const unsigned row = (unsigned)s / (unsigned)p.nx;
        x = (int)((unsigned)s - row * (unsigned)p.nx);
        z = (int)(row / (unsigned)p.ny);
        y = (int)(row - (unsigned)z * (unsigned)p.ny);
        return true;
    }
    const long long plane = (long long)p.nx * p.ny;
    z = (int)(s / plane);
    const long long r = s - (long long)z * plane;
    y = (int)(r / p.nx);
    x = (int)(r - (long long)y * p.nx);
    return true;
}

// ------------------------------------------------------------ init (a1)
// Records an invalid initial value: FLAG_BAD_INPUT and the smallest such index in `slot`.
__device__ __forceinline__ void bad_input(const KParams &p, int slot, long long idx) {
    atomicOr(p.flags, FLAG_BAD_INPUT);
    atomicMin(reinterpret_cast<unsigned long long *>(p.flags + slot), (unsigned long long)idx);
}

// f_i = f_i^eq(rho0, u0) in natural layout, for cells [c0, c0 + cn).  A rho0 that is not a
// positive finite number, or a non-finite u0 component, is recorded (bad_input).
template <class L, class S>
__global__ void k_init(KParams p, S *__restrict__ A, const double *__restrict__ rho0, const double *__restrict__ u0,
                       long long c0, long long cn, int has_u) {
    using T = typename Store<S>::T;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= cn) return;
    const long long s = c0 + k;
    const double r0 = rho0[k];
    if (!(r0 > 0.0) || !(r0 < INFINITY)) bad_input(p, FLAG_SLOT_RHO, s);
    const T rho = (T)r0;
    T u[3] = {0, 0, 0};
    if (has_u)
        for (int a = 0; a < L::D; ++a) {
            const double ua = u0[a * cn + k];
            if (!(fabs(ua) < INFINITY)) bad_input(p, FLAG_SLOT_U, a * p.n + s);
            u[a] = (T)ua;
        }
    if constexpr (std::is_same<S, double>::value) {
        // FP64: Eq. Single_Phase_EDF evaluated as the plain collision does
        double f[L::Q];
        plain::equilibrium<L>(r0, u, f);
#pragma unroll
        for (int i = 0; i < L::Q; ++i) Store<S>::st(A + (long long)i * p.pstride + s, f[i]);
        return;
    }
    const T usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const T rref = phys<T>(p).rho_ref;
    Unroll<0, L::Q>::run([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        const T cu = (T)L::cx(i) * u[0] + (T)L::cy(i) * u[1] + (T)L::cz(i) * u[2];
        const T feq = (T)L::w(i) * rho * ((T)1 - (T)1.5 * usq + (T)3 * cu + (T)4.5 * cu * cu);
        Store<S>::st(A + (long long)i * p.pstride + s, Store<S>::SHIFT ? feq - (T)L::w(i) * rref : feq);
    });
}

// -------------------------------------------------------------- moments (a6)
template <class L, class S>
__global__ void k_moments(KParams p, const S *__restrict__ A, const typename Store<S>::PsiT *__restrict__ psi, int odd,
                          double *__restrict__ rho_out, double *__restrict__ u_out, double *__restrict__ p_out,
                          long long c0, long long cn) {
    using T = typename Store<S>::T;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= cn) return;
    const long long s = c0 + k;
    int x, y, z;
    cell_coords(p, s, x, y, z);
    const Nbr nb = neighbours(p, x, y, z);
    T f[L::Q];
    load_pops<L, S>(p, A, x, y, z, nb, s, odd != 0, f);
    T rho = 0, j[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        rho += f[i];
        j[0] += (T)L::cx(i) * f[i];
        j[1] += (T)L::cy(i) * f[i];
        j[2] += (T)L::cz(i) * f[i];
    }
    T F[3];
    cell_force<L, T>(p, psi, psi_index(p, x, y, z), F);
    if (rho_out) rho_out[k] = (double)rho;
    if (u_out)
        for (int a = 0; a < L::D; ++a) u_out[a * cn + k] = (double)((j[a] + (T)0.5 * F[a]) / rho);
    if (p_out) p_out[k] = (double)eos_pressure<T>(p, rho);
}

// ------------------------------------------------- balanced start (plb_init_physical)
// At t = 0 (even parity, natural layout) the populations are f^eq(rho, u0), so sum f c = rho u0.
// Rewrites them as f^eq(rho, u0 - F / (2 rho)), F the force of the initial density (psi pass
// already run), so that the velocity of Eq. Momentum, (sum f c + F/2) / rho, is u0.  Each
// thread reads and writes its own cell only.
template <class L, class S>
__global__ void k_rebalance(KParams p, S *__restrict__ A, const typename Store<S>::PsiT *__restrict__ psi) {
    using T = typename Store<S>::T;
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int x, y, z;
    if (!cell_coords(p, s, x, y, z)) return;
    const Nbr nb = neighbours(p, x, y, z);
    T f[L::Q];
    load_pops<L, S>(p, A, x, y, z, nb, s, false, f);
    T rho = 0, j[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        rho += f[i];
        j[0] += (T)L::cx(i) * f[i];
        j[1] += (T)L::cy(i) * f[i];
        j[2] += (T)L::cz(i) * f[i];
    }
    T F[3];
    cell_force<L, T>(p, psi, psi_index(p, x, y, z), F);
    T u[3];
    for (int a = 0; a < 3; ++a) u[a] = (j[a] - (T)0.5 * F[a]) / rho;
    const T usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const T rref = phys<T>(p).rho_ref;
    Unroll<0, L::Q>::run([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        const T cu = (T)L::cx(i) * u[0] + (T)L::cy(i) * u[1] + (T)L::cz(i) * u[2];
        const T feq = (T)L::w(i) * rho * ((T)1 - (T)1.5 * usq + (T)3 * cu + (T)4.5 * cu * cu);
        Store<S>::st(A + (long long)i * p.pstride + s, Store<S>::SHIFT ? feq - (T)L::w(i) * rref : feq);
    });
}

// ------------------------------------------------------------- wetting walls
// psi_wall into the ghost rows y = -1 and y = ny of the padded psi field, over the ghost columns
// and planes too (every node beyond a wall).  Nothing else writes these rows when the walls
// are wetting (psi_ghosts skips them), so this runs once, when the lattice is created.
template <class L, class S>
__global__ void k_wall_fill(KParams p, typename Store<S>::PsiT *__restrict__ psi) {
    using T = typename Store<S>::T;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long cols = (long long)p.nx + 2, planes = L::D == 3 ? p.nz + 2 : 1;
    if (k >= cols * planes) return;
    const int x = (int)(k % cols) - 1;
    const int z = L::D == 3 ? (int)(k / cols) - 1 : 0;
    const typename Store<S>::PsiT v = (typename Store<S>::PsiT)phys<T>(p).psi_wall;
    psi[psi_index(p, x, -1, z)] = v;
    psi[psi_index(p, x, p.ny, z)] = v;
}

// ------------------------------------------------------ population exchange
template <class L, class S>
__global__ void k_get_pops(KParams p, const S *__restrict__ A, int odd, double *__restrict__ out, long long c0,
                           long long cn) {
    using T = typename Store<S>::T;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= cn) return;
    const long long s = c0 + k;
    int x, y, z;
    cell_coords(p, s, x, y, z);
    const Nbr nb = neighbours(p, x, y, z);
    T f[L::Q];
    load_pops<L, S>(p, A, x, y, z, nb, s, odd != 0, f);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) out[i * cn + k] = (double)f[i];
}

template <class L, class S>
__global__ void k_set_pops(KParams p, S *__restrict__ A, const double *__restrict__ in, long long c0, long long cn) {
    using T = typename Store<S>::T;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= cn) return;
    const long long s = c0 + k;
    const T rref = phys<T>(p).rho_ref;
    Unroll<0, L::Q>::run([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        const T v = (T)in[i * cn + k];
        Store<S>::st(A + (long long)i * p.pstride + s, Store<S>::SHIFT ? v - (T)L::w(i) * rref : v);
    });
}

// ----------------------------------------------------------- reductions (a4)
// A grid-stride loop per thread, warp-shuffle tree, one partial per block (4 doubles);
// k_reduce_final sums the partials in block order.
//
// What bounds the sums is the FP64 pipe: two operations per clock and SM on GB300.  Adding every
// population in FP64 took about 100 of them per cell, ten times the HBM time.  FP32 storage adds with
// error-free transformations on the FP32 pipe instead and converts once per thread; the speed
// maximum is searched in pairs of FP32 values, and FP64 evaluates the candidates only.  Mass, momentum,
// maximum speed and moments of 256 x 128 x 128 cells, D3Q19 FP32: 2140 -> 713 us.

// A sum of FP32 values in three FP32 parts, each the rounding error of the one before (TwoSum, Knuth
// 1969; the cascade of Ogita, Rump and Oishi 2005): about 70 bits, where FP64 keeps 53.
struct Sum3 {
    float h = 0.0f, m = 0.0f, l = 0.0f;
    __device__ __forceinline__ static float two_sum(float a, float b, float &err) {
        const float s = __fadd_rn(a, b), bb = __fadd_rn(s, -a);
        err = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb));
        return s;
    }
    __device__ __forceinline__ void add(float x) {
        float e1, e2;
        h = two_sum(h, x, e1);
        m = two_sum(m, e1, e2);
        l = __fadd_rn(l, e2);
    }
    // false where the sum has left FP32's range (or a term was not finite): its error terms are then NaN
    __device__ __forceinline__ bool finite() const { return fabsf(h) < INFINITY; }
    __device__ __forceinline__ double value() const { return (double)h + ((double)m + (double)l); }
    // the sum as a pair: hi the FP32 value nearest to it
    __device__ __forceinline__ void pair(float &hi, float &lo) const {
        hi = two_sum(h, __fadd_rn(m, l), lo);
    }
};

// speed^2 = |momentum|^2 / rho^2 of a cell as a pair of FP32 values, relative error below 2^-40: true where the
// pair says so.  Density and momentum are scaled by the power of two that brings the density to 1 .. 2
// (exact), so that no square leaves FP32's range for any density as long as the speed lies in 2^-45 .. 2^50.
// False for every other cell (its rounding errors could be subnormal, its squares overflow, or its density
// is 0, infinite or NaN).  A cell without momentum has speed 0.
__device__ __forceinline__ bool speed2_pair(const Sum3 &rho, const Sum3 m[3], int dims, float &qh, float &ql) {
    float rh, rl;
    rho.pair(rh, rl);
    int e = (int)(__float_as_uint(rh) >> 23 & 0xffu);
    e = e < 1 ? 1 : (e > 253 ? 253 : e);
    const float scale = __uint_as_float((unsigned)(254 - e) << 23);        // 2^(127 - e)
    rh = __fmul_rn(rh, scale);
    rl = __fmul_rn(rl, scale);
    float nh = 0.0f, nl = 0.0f, err;
    bool still = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (a >= dims) continue;
        float h, l;
        m[a].pair(h, l);
        still = still && h == 0.0f;
        h = __fmul_rn(h, scale);
        l = __fmul_rn(l, scale);
        const float s = __fmul_rn(h, h);
        const float r = fmaf(h, h, -s) + 2.0f * h * l;
        nh = Sum3::two_sum(nh, s, err);
        nl += err + r;
    }
    nh = Sum3::two_sum(nh, nl, nl);
    const float dh = __fmul_rn(rh, rh), dl = fmaf(rh, rh, -dh) + 2.0f * rh * rl;
    qh = __fdiv_rn(nh, dh);
    ql = __fdiv_rn(fmaf(-qh, dl, fmaf(-qh, dh, nh) + nl), dh);
    qh = Sum3::two_sum(qh, ql, ql);
    return (qh >= 0x1p-90f && qh <= 0x1p100f) || (still && rh >= 0x1p-10f && rh < 4.0f);
}

// Density and total momentum (half the force included) of a cell in FP64.
template <class L, class S>
__device__ __forceinline__ void cell_sums(const KParams &p, const S *__restrict__ A,
                                          const typename Store<S>::PsiT *__restrict__ psi, int odd, int what,
                                          long long s, int x, int y, int z, double &rho, double m[3]) {
    using T = typename Store<S>::T;
    const Nbr nb = neighbours(p, x, y, z);
    T f[L::Q];
    load_pops<L, S>(p, A, x, y, z, nb, s, odd != 0, f);
    rho = 0.0;
    double j[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < L::Q; ++i) rho += (double)f[i];
    if (what < 1 || what > 4) return;
    // terms with a zero velocity component add exactly 0 and are skipped
    Unroll<0, L::Q>::run([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if (L::cx(i) != 0) j[0] += (double)(L::cx(i) * f[i]);
        if (L::cy(i) != 0) j[1] += (double)(L::cy(i) * f[i]);
        if (L::cz(i) != 0) j[2] += (double)(L::cz(i) * f[i]);
    });
    T F[3];
    cell_force<L, T>(p, psi, psi_index(p, x, y, z), F);
    for (int a = 0; a < 3; ++a) m[a] = j[a] + 0.5 * (double)F[a];
}

// |u| of cell s in FP64.
template <class L, class S>
__device__ __forceinline__ double cell_speed(const KParams &p, const S *__restrict__ A,
                                             const typename Store<S>::PsiT *__restrict__ psi, int odd, long long s) {
    int x, y, z;
    double rho, m[3];
    cell_coords(p, s, x, y, z);
    cell_sums<L, S>(p, A, psi, odd, 2, s, x, y, z, rho, m);
    return sqrt((m[0] * m[0] + m[1] * m[1] + m[2] * m[2]) / (rho * rho));
}

// The block's partial from its threads' sums (or maxima).
__device__ __forceinline__ void block_partial(double acc[4], bool is_max, double *__restrict__ partials) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        double v = acc[c];
        for (int o = 16; o > 0; o >>= 1) {
            const double w = __shfl_down_sync(0xffffffffu, v, o);
            v = is_max ? fmax(v, w) : v + w;
        }
        acc[c] = v;
    }
    __shared__ double red[8][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
        for (int c = 0; c < 4; ++c) red[warp][c] = acc[c];
    __syncthreads();
    if (threadIdx.x < 4) {
        double v = 0.0;
        const int nw = blockDim.x >> 5;
        for (int w = 0; w < nw; ++w) v = is_max ? fmax(v, red[w][threadIdx.x]) : v + red[w][threadIdx.x];
        partials[blockIdx.x * 4 + threadIdx.x] = v;
    }
}

struct Box {
    int lo[3], hi[3];
    __device__ __forceinline__ bool holds(int x, int y, int z) const {
        return x >= lo[0] && x < hi[0] && y >= lo[1] && y < hi[1] && z >= lo[2] && z < hi[2];
    }
};

// Every reduction, in FP64: FP64 storage, and the means of |u|, u^2 and the pressure.
template <class L, class S>
__global__ void __launch_bounds__(256) k_reduce(KParams p, const S *__restrict__ A,
                                                const typename Store<S>::PsiT *__restrict__ psi, int odd, int what,
                                                Box box, double *__restrict__ partials) {
    using T = typename Store<S>::T;
    double acc[4] = {0, 0, 0, 0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < p.n; s += stride) {
        int x, y, z;
        cell_coords(p, s, x, y, z);
        if (!box.holds(x, y, z)) continue;
        double rho, m[3];
        cell_sums<L, S>(p, A, psi, odd, what, s, x, y, z, rho, m);
        if (what == 0 || what == 5) {
            acc[0] += rho;
        } else if (what == 6) {
            acc[0] += (double)eos_pressure<T>(p, (T)rho);
        } else if (what == 1) {
            acc[0] += m[0];
            acc[1] += m[1];
            acc[2] += m[2];
        } else {
            const double u2 = (m[0] * m[0] + m[1] * m[1] + m[2] * m[2]) / (rho * rho);
            if (what == 2) acc[0] = fmax(acc[0], sqrt(u2));
            else if (what == 3) acc[0] += sqrt(u2);
            else acc[0] += u2;
        }
    }
    block_partial(acc, what == 2, partials);
}

// FP32 arithmetic: density (WHAT 0), momentum (1) and the largest speed (2).  Four blocks per SM: at the
// 128 registers that it takes uncapped, two, a long chain of additions per cell has too little beside it
// (the four readouts of 256 x 128 x 128 cells, two / three / four / five blocks: 805 / 719 / 706 / 731 us).
//
// Largest speed: pairs of FP32 values rank a thread's cells, and FP64 evaluates the first in rank.  It also
// evaluates every cell that the pairs cannot rank: one that comes within 2^-36 of the thread's first (the
// pairs are good to 2^-40), unless its sums are those of the first in every bit (uniform and symmetric
// flows), and one outside the pairs' range.  So the cell of the largest speed is always among those
// evaluated, and the result is as accurate as a search in FP64.
template <class L, class S, int WHAT>
__global__ void __launch_bounds__(256, 4) k_reduce_f32(KParams p, const S *__restrict__ A, const float *__restrict__ psi,
                                                    int odd, Box box, double *__restrict__ partials) {
    double acc[4] = {0, 0, 0, 0};
    Sum3 sum[3];
    float bh = -1.0f, bl = 0.0f;               // WHAT 2: speed^2 of the thread's first cell in rank, the cell
    long long best = -1;
    __shared__ float first[WHAT == 2 ? 12 : 1][256];                       // its sums
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < p.n; s += stride) {
        int x, y, z;
        cell_coords(p, s, x, y, z);
        if (!box.holds(x, y, z)) continue;
        const Nbr nb = neighbours(p, x, y, z);
        float f[L::Q];
        load_pops<L, S>(p, A, x, y, z, nb, s, odd != 0, f);
        if constexpr (WHAT == 0) {
#pragma unroll
            for (int i = 0; i < L::Q; ++i) sum[0].add(f[i]);
        } else {
            if (WHAT == 2) sum[0] = sum[1] = sum[2] = Sum3();
            Unroll<0, L::Q>::run([&](auto ic) {
                constexpr int i = decltype(ic)::value;
                if (L::cx(i) != 0) sum[0].add(L::cx(i) * f[i]);
                if (L::cy(i) != 0) sum[1].add(L::cy(i) * f[i]);
                if (L::cz(i) != 0) sum[2].add(L::cz(i) * f[i]);
            });
            float F[3];
            cell_force<L, float>(p, psi, psi_index(p, x, y, z), F);
#pragma unroll
            for (int a = 0; a < L::D; ++a) sum[a].add(0.5f * F[a]);
            if constexpr (WHAT == 2) {
                Sum3 rho;
#pragma unroll
                for (int i = 0; i < L::Q; ++i) rho.add(f[i]);
                float qh, ql;
                const bool ranked = speed2_pair(rho, sum, L::D, qh, ql);
                const float d = (qh - bh) + (ql - bl), near = 0x1p-36f * bh;
                const float parts[12] = {rho.h, rho.m, rho.l, sum[0].h, sum[0].m, sum[0].l,
                                         sum[1].h, sum[1].m, sum[1].l, sum[2].h, sum[2].m, sum[2].l};
                if (ranked && (best < 0 || d > near)) {
                    bh = qh;
                    bl = ql;
                    best = s;
#pragma unroll
                    for (int k = 0; k < 12; ++k) first[k][threadIdx.x] = parts[k];
                } else if (!(ranked && (d < -near || qh == 0.0f))) {
                    bool same = ranked;
#pragma unroll
                    for (int k = 0; k < 12; ++k) same = same && first[k][threadIdx.x] == parts[k];
                    if (!same) acc[0] = fmax(acc[0], cell_speed<L, S>(p, A, psi, odd, s));
                }
            }
        }
    }
    if constexpr (WHAT < 2) {
        bool finite = true;
#pragma unroll
        for (int a = 0; a < (WHAT ? 3 : 1); ++a) {
            acc[a] = sum[a].value();
            finite = finite && sum[a].finite();
        }
        if (!finite) {
            // beyond FP32's range: this thread's cells again, in FP64
            acc[0] = acc[1] = acc[2] = 0.0;
#pragma unroll 1
            for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < p.n; s += stride) {
                int x, y, z;
                cell_coords(p, s, x, y, z);
                if (!box.holds(x, y, z)) continue;
                double rho, m[3];
                cell_sums<L, S>(p, A, psi, odd, WHAT, s, x, y, z, rho, m);
                if (WHAT == 0) acc[0] += rho;
                else
                    for (int a = 0; a < 3; ++a) acc[a] += m[a];
            }
        }
    } else {
        // the threads whose cell comes within 2^-20 of the block's largest evaluate it in FP64
        float top = bh;
        for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
        __shared__ float tops[8];
        if ((threadIdx.x & 31) == 0) tops[threadIdx.x >> 5] = top;
        __syncthreads();
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) top = fmaxf(top, tops[w]);
        if (best >= 0 && bh >= top * (1.0f - 0x1p-20f)) acc[0] = fmax(acc[0], cell_speed<L, S>(p, A, psi, odd, best));
    }
    block_partial(acc, WHAT == 2, partials);
}

// Total mass of the whole lattice.  In either AA layout every population of every cell sits in
// exactly one slot of the store, so the mass is the sum of the Q planes over the N cells (plus
// N rho_ref with the FP16 shift): no coordinates, no neighbour addressing, coalesced loads.
// FP32 arithmetic: each cell's Q values are summed with an error-free compensated sum (TwoSum),
// the cell's sum and correction then added in FP64 per thread; FP64 storage sums in FP64.
// One partial per block in partials[4 * block] (the final pass sums them in block order).
template <class L, class S>
__global__ void __launch_bounds__(256) k_mass_flat(KParams p, const S *__restrict__ A, double *__restrict__ partials) {
    using T = typename Store<S>::T;
    double acc = 0.0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < p.n; s += stride) {
        if constexpr (std::is_same<T, double>::value) {
            double r = 0.0;
#pragma unroll
            for (int i = 0; i < L::Q; ++i) r += Store<S>::ld(A + i * p.pstride + s);
            acc += r;
        } else {
            float sum = 0.0f, cor = 0.0f;
#pragma unroll
            for (int i = 0; i < L::Q; ++i) {
                const float x = Store<S>::ld(A + i * p.pstride + s);
                const float t = sum + x, bb = t - sum;
                cor += (sum - (t - bb)) + (x - bb);
                sum = t;
            }
            acc += (double)sum + (double)cor;
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    __shared__ double red[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w];
        if (Store<S>::SHIFT && blockIdx.x == 0) v += (double)p.n * p.d.rho_ref;
        partials[blockIdx.x * 4] = v;
        partials[blockIdx.x * 4 + 1] = partials[blockIdx.x * 4 + 2] = partials[blockIdx.x * 4 + 3] = 0.0;
    }
}

// ----------------------------------------------------------------- launchers
template <class L, class S> struct Launch {
    using PsiT = typename Store<S>::PsiT;
    static unsigned blocks(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }
    // SMs of the current device (queried once per device, up to 64 devices)
    static int sm_count() {
        static int cache[64] = {0};
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev < 0 || dev >= 64) return 152;
        if (cache[dev] == 0) {
            int n = 0;
            if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 152;
            cache[dev] = n;
        }
        return cache[dev];
    }

    static void init(const KParams &p, void *A, const double *rho0, const double *u0, long long c0, long long cn,
                     cudaStream_t st) {
        k_init<L, S><<<blocks(cn, 256), 256, 0, st>>>(p, (S *)A, rho0, u0, c0, cn, u0 != nullptr);
    }
    // Launches a step kernel so that it may start while the kernel before it in the stream runs out
    // (step_kernel_begin waits for that one).
    template <class... P, class... Args>
    static void go(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, const Args &...args) {
        go_if(true, kernel, grid, block, st, args...);
    }
    template <class... P, class... Args>
    static void go_if(bool early, void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, const Args &...args) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = block;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    }
    // The same for the collision kernels whose blocks run long (FP64, and FP16 D3Q19): early only if the grid
    // fills every SM or leaves half of them free.  Blocks that come early pile up on the SMs that come free
    // first, and the fullest SM then ends the step.  Microseconds a step, one step a call, early and not: FP64
    // 24^3 (144 blocks) 99 and 45, 32^3 104 and 74, 200^2 84 and 51, 16^2 (4 blocks) 21 and 23; FP16 64^3 26 and
    // 17, with a wait after each step 41 and 27, 10 x 16 x 9 (32 blocks) 13 and 15, 160^3 108 and 111.
    template <class... P, class... Args>
    static void go_long(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, const Args &...args) {
        static thread_local std::map<std::pair<const void *, unsigned>, int> cache;
        const unsigned threads = block.x * block.y;
        int &resident = cache[{(const void *)kernel, threads}];
        if (resident == 0 &&
            (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, kernel, (int)threads, 0) != cudaSuccess ||
             resident < 1))
            resident = 1;
        const long long n = (long long)grid.x * grid.y * grid.z;
        go_if(n >= (long long)resident * sm_count() || n <= sm_count() / 2, kernel, grid, block, st, args...);
    }
    static Planes<S> planes(const KParams &p, const void *A) {
        Planes<S> pl;
        for (int i = 0; i < 19; ++i) pl.p[i] = (S *)A + (i < L::Q ? (long long)i * p.pstride : 0);
        return pl;
    }
    static void dims3(const KParams &p, dim3 &grid, dim3 &block, int threads = 256) {
        int bx = p.nx >= threads ? threads : (p.nx + 31) / 32 * 32;
        int by = threads / bx;
        if (by > p.ny) by = p.ny;
        block = dim3(bx, by, 1);
        grid = dim3((p.nx + bx - 1) / bx, (p.ny + by - 1) / by, p.nzl);
    }
    // Two cells per thread with packed FP32 arithmetic where it applies (FP32 arithmetic,
    // even nx, fewer than 2^31 cells); one cell per thread otherwise.
    static bool use_pair(const KParams &p) {
        if (std::is_same<S, __half>::value && !PLB_HALF_PAIR) return false;
        // one population plane addressable with 32-bit cell indices and byte offsets
        return !std::is_same<S, double>::value && (p.nx % 2 == 0) && p.n * (long long)sizeof(S) < (1LL << 32);
    }
    static void dims_pair(const KParams &p, dim3 &grid, dim3 &block, int threads = 256) {
        const int npx = p.nx / 2;
        int bx = npx >= threads ? threads : (npx + 31) / 32 * 32;
        if (threads & (threads - 1)) bx = npx >= 64 ? 64 : (npx + 31) / 32 * 32;   // 64 wide
        int by = threads / bx;
        if (by > p.ny) by = p.ny;
        block = dim3(bx, by, 1);
        grid = dim3((npx + bx - 1) / bx, (p.ny + by - 1) / by, p.nzl);
    }
    template <bool ODD> static void psi_t(const KParams &p, const void *A, void *psi, cudaStream_t st) {
        dim3 grid, block;
        if constexpr (std::is_same<S, __half>::value) {
            if (PLB_PSI_QUAD && p.nx % 4 == 0 && p.n < (1LL << 31)) {
                const long long quads = (long long)(p.nx / 4) * p.ny;
                go(k_psi_quad<L, ODD>, dim3(blocks(quads, 256), 1, p.nzl), 256, st, p, planes(p, A), (float *)psi);
                return;
            }
        }
        if constexpr (!std::is_same<S, double>::value) {
            if (use_pair(p)) {
                dims_pair(p, grid, block);
                go(k_psi_pair<L, S, ODD>, grid, block, st, p, planes(p, A), (float *)psi);
                return;
            }
        }
        dims3(p, grid, block);
        if (p.n < (1LL << 31))
            go(k_psi_fast<L, S, ODD, int>, grid, block, st, p, planes(p, A), (PsiT *)psi);
        else
            go(k_psi_fast<L, S, ODD, long long>, grid, block, st, p, planes(p, A), (PsiT *)psi);
    }
    static void psi(const KParams &p, const void *A, void *psi, int odd, cudaStream_t st) {
        if (odd) psi_t<true>(p, A, psi, st);
        else psi_t<false>(p, A, psi, st);
    }
    // resident blocks per SM of the pair collide kernel (one wave = this x SM count)
    template <int MRT, bool ODD> static int pair_blocks_per_sm() {
        static int nb = 0;
        if (nb == 0) {
            int v = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_collide_pair<L, S, MRT, ODD, false>,
                                                              PLB_PAIR_THREADS, 0) != cudaSuccess || v < 1)
                v = 1;
            nb = v;
        }
        return nb;
    }
    template <int MRT, bool ODD, bool WIDE>
    static void staged_run(const KParams &p, void *A, const void *psi, const StagedSplit &sp, cudaStream_t st) {
        const dim3 grid(sp.segments, (p.ny + sp.rows - 1) / sp.rows, (p.nzl + PLB_STAGED_ZC - 1) / PLB_STAGED_ZC);
        if constexpr (Store<S>::SHIFT) {
            if (p.stochastic) {
                go_long(k_collide_staged<L, S, MRT, ODD, true, WIDE>, grid, sp.threads, st, p, planes(p, A),
                        (const float *)psi, sp);
                return;
            }
        }
        go_long(k_collide_staged<L, S, MRT, ODD, false, WIDE>, grid, sp.threads, st, p, planes(p, A),
                (const float *)psi, sp);
    }
    template <int MRT, bool ODD> static void collide_t(const KParams &p, void *A, const void *psi, cudaStream_t st) {
        dim3 grid, block;
        if constexpr (!std::is_same<S, double>::value) {
            if constexpr (std::is_same<L, D3Q19>::value) {
                if (use_pair(p) && (std::is_same<S, __half>::value ? PLB_STAGED_HALF : PLB_STAGED_FLOAT) != 0) {
                    bool wide = false;
                    const StagedSplit sp = staged_split(p.nx / 2, p.ny, (p.nzl + PLB_STAGED_ZC - 1) / PLB_STAGED_ZC,
                                                        sm_count(), wide);
                    if (wide) staged_run<MRT, ODD, true>(p, A, psi, sp, st);
                    else staged_run<MRT, ODD, false>(p, A, psi, sp, st);
                    return;
                }
            }
            if (use_pair(p)) {
                dims_pair(p, grid, block, PLB_PAIR_THREADS);
                // FP32 storage: prefetch into L2 for the block one wave (the resident blocks of
                // every SM) later; FP16S is bound by arithmetic and loses more to the extra
                // instructions than it gains
                KParams q = p;
                if ((std::is_same<S, float>::value ? PLB_L2_PREFETCH : PLB_L2_PREFETCH_HALF) != 0) {
                    const int ahead = PLB_PF_WAVES * pair_blocks_per_sm<MRT, ODD>() * sm_count();
                    q.prefetch_ahead = ahead;
                    q.pf_step[0] = ahead % (int)grid.x;
                    q.pf_step[1] = (ahead / (int)grid.x) % (int)grid.y;
                    q.pf_step[2] = ahead / ((int)grid.x * (int)grid.y);
                }
                if constexpr (Store<S>::SHIFT) {
                    if (p.stochastic) {
                        go(k_collide_pair<L, S, MRT, ODD, true>, grid, block, st, q, planes(p, A), (const float *)psi);
                        return;
                    }
                }
                go(k_collide_pair<L, S, MRT, ODD, false>, grid, block, st, q, planes(p, A), (const float *)psi);
                return;
            }
        }
        if constexpr (std::is_same<S, double>::value) {
            dims3(p, grid, block, 128);
            if (p.n < (1LL << 31))
                go_long(k_collide_plain<L, MRT, ODD, int>, grid, block, st, p, planes(p, A), (const double *)psi);
            else
                go_long(k_collide_plain<L, MRT, ODD, long long>, grid, block, st, p, planes(p, A), (const double *)psi);
            return;
        }
        dims3(p, grid, block);
        if (p.n < (1LL << 31))
            go(k_collide_fast<L, S, MRT, ODD, int>, grid, block, st, p, planes(p, A), (const PsiT *)psi);
        else
            go(k_collide_fast<L, S, MRT, ODD, long long>, grid, block, st, p, planes(p, A), (const PsiT *)psi);
    }
    static void collide_bgk(const KParams &p, void *A, const void *psi, int odd, cudaStream_t st) {
        if (odd) collide_t<0, true>(p, A, psi, st);
        else collide_t<0, false>(p, A, psi, st);
    }
    static void collide_mrt(const KParams &p, void *A, const void *psi, int odd, cudaStream_t st) {
        if (odd) collide_t<1, true>(p, A, psi, st);
        else collide_t<1, false>(p, A, psi, st);
    }
    static void moments(const KParams &p, const void *A, const void *psi, int odd, double *r, double *u, double *pr,
                        long long c0, long long cn, cudaStream_t st) {
        k_moments<L, S><<<blocks(cn, 256), 256, 0, st>>>(p, (const S *)A, (const PsiT *)psi, odd, r, u, pr, c0, cn);
    }
    static void get_pops(const KParams &p, const void *A, int odd, double *out, long long c0, long long cn,
                         cudaStream_t st) {
        k_get_pops<L, S><<<blocks(cn, 256), 256, 0, st>>>(p, (const S *)A, odd, out, c0, cn);
    }
    static void set_pops(const KParams &p, void *A, const double *in, long long c0, long long cn, cudaStream_t st) {
        k_set_pops<L, S><<<blocks(cn, 256), 256, 0, st>>>(p, (S *)A, in, c0, cn);
    }
    static void reduce(const KParams &p, const void *A, const void *psi, int odd, int what, const int lo[3],
                       const int hi[3], double *partials, int nblocks, cudaStream_t st) {
        const Box box = {{lo[0], lo[1], lo[2]}, {hi[0], hi[1], hi[2]}};
        if constexpr (!std::is_same<S, double>::value) {
            const S *a = (const S *)A;
            const float *ps = (const float *)psi;
            if (what == 0 || what == 5) {
                k_reduce_f32<L, S, 0><<<nblocks, 256, 0, st>>>(p, a, ps, odd, box, partials);
                return;
            }
            if (what == 1) {
                k_reduce_f32<L, S, 1><<<nblocks, 256, 0, st>>>(p, a, ps, odd, box, partials);
                return;
            }
            if (what == 2) {
                k_reduce_f32<L, S, 2><<<nblocks, 256, 0, st>>>(p, a, ps, odd, box, partials);
                return;
            }
        }
        k_reduce<L, S><<<nblocks, 256, 0, st>>>(p, (const S *)A, (const PsiT *)psi, odd, what, box, partials);
    }
    static void mass(const KParams &p, const void *A, double *partials, int nblocks, cudaStream_t st) {
        k_mass_flat<L, S><<<nblocks, 256, 0, st>>>(p, (const S *)A, partials);
    }
    static void wall_fill(const KParams &p, void *psi, cudaStream_t st) {
        const long long n = ((long long)p.nx + 2) * (L::D == 3 ? p.nz + 2 : 1);
        k_wall_fill<L, S><<<blocks(n, 256), 256, 0, st>>>(p, (PsiT *)psi);
    }
    static void rebalance(const KParams &p, void *A, const void *psi, cudaStream_t st) {
        k_rebalance<L, S><<<blocks(p.n, 256), 256, 0, st>>>(p, (S *)A, (const PsiT *)psi);
    }
    // resident blocks per SM of the single-pass kernel
    template <int MRT> static int fused_blocks_per_sm() {
        static int nb = 0;
        if (nb == 0) {
            int v = 0;
            if constexpr (!std::is_same<S, double>::value) {
                if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_fused_pair<L, S, MRT, false>,
                                                                  FusedTile<L, S>::THREADS, 0) != cudaSuccess || v < 1)
                    v = 1;
            }
            nb = v < 1 ? 1 : v;
        }
        return nb;
    }
    // single pass: tiles of FusedTile's size, each block walking a chunk of zc planes.  The chunk count
    // minimises (waves of resident blocks) x (planes per chunk + 0.5): a block also forms psi of the two
    // planes before its chunk, at about a third of a collided plane's cost each (measured with tiles of
    // 64 x 16 and kept for 64 x 8), and the last wave of a grid that is not a multiple of the resident
    // blocks runs partly idle.
    template <int MRT> static void fused_t(const KParams &p, const void *A, void *B, cudaStream_t st) {
        if constexpr (!std::is_same<S, double>::value) {
            using Tl = FusedTile<L, S>;
            const int gx = (p.nx + Tl::TX - 1) / Tl::TX, gy = (p.ny + Tl::TY - 1) / Tl::TY;
            int zc = 1, gz = 1;
            if (L::D == 3) {
                const long long tiles = (long long)gx * gy;
                const long long resident = (long long)fused_blocks_per_sm<MRT>() * sm_count();
                // the last search's result (one lattice stepped many times asks the same again)
                static thread_local long long key[3] = {-1, -1, -1};
                static thread_local int last[2] = {1, 1};
                if (key[0] != tiles || key[1] != resident || key[2] != p.nz) {
                    double best = 0.0;
                    const int gmax = p.nz < 4096 ? p.nz : 4096;
                    for (int g = 1; g <= gmax; ++g) {
                        const int zcg = (p.nz + g - 1) / g;
                        const int gzg = (p.nz + zcg - 1) / zcg;
                        if (gzg != g) continue;                       // the same chunking as a smaller g
                        const long long waves = (tiles * gzg + resident - 1) / resident;
                        const double cost = (double)waves * (zcg + 0.5);
                        if (g == 1 || cost < best) {
                            best = cost;
                            last[0] = zcg;
                            last[1] = gzg;
                        }
                    }
                    key[0] = tiles;
                    key[1] = resident;
                    key[2] = p.nz;
                }
                zc = last[0];
                gz = last[1];
            }
            const dim3 grid(gx, gy, gz), block(Tl::THREADS);
            if constexpr (Store<S>::SHIFT) {
                if (p.stochastic) {
                    k_fused_pair<L, S, MRT, true><<<grid, block, 0, st>>>(p, planes(p, A), planes(p, B), zc);
                    return;
                }
            }
            k_fused_pair<L, S, MRT, false><<<grid, block, 0, st>>>(p, planes(p, A), planes(p, B), zc);
        }
    }
    static void fused_bgk(const KParams &p, const void *A, void *B, cudaStream_t st) { fused_t<0>(p, A, B, st); }
    static void fused_mrt(const KParams &p, const void *A, void *B, cudaStream_t st) { fused_t<1>(p, A, B, st); }
    // kernel of the many-step launch for this lattice and collision form (FORM 1: the single pass's)
    template <int FORM> static const void *tile_kernel(const KParams &p, int mrt) {
        constexpr int M = FORM && !Store<S>::SHIFT && std::is_same<L, D3Q19>::value ? PLB_FUSED_MOMENT : -1;
        if constexpr (std::is_same<S, double>::value) {
            return mrt ? (const void *)&k_tile<L, S, 1, false, -1, 1> : (const void *)&k_tile<L, S, 0, false, -1, 1>;
        } else {
            if constexpr (Store<S>::SHIFT) {
                if (p.stochastic) {
                    if (p.nx % 2 == 0)
                        return mrt ? (const void *)&k_tile<L, S, 1, true, M, 2> : (const void *)&k_tile<L, S, 0, true, M, 2>;
                    return mrt ? (const void *)&k_tile<L, S, 1, true, -1, 1> : (const void *)&k_tile<L, S, 0, true, -1, 1>;
                }
            }
            if (p.nx % 2 == 0)
                return mrt ? (const void *)&k_tile<L, S, 1, false, M, 2> : (const void *)&k_tile<L, S, 0, false, M, 2>;
            return mrt ? (const void *)&k_tile<L, S, 1, false, -1, 1> : (const void *)&k_tile<L, S, 0, false, -1, 1>;
        }
    }
    static size_t tile_smem(const KParams &p, const TileArgs &t) {
        const int w = !std::is_same<S, double>::value && p.nx % 2 == 0 ? 2 : 1;
        const size_t v = w * sizeof(typename Store<S>::T);
        return ((size_t)L::Q * v + 4) * t.max_own + (size_t)(w * sizeof(PsiT) + 8) * t.max_region;
    }
    // Splits the lattice into tiles: the split with the least cost, which is the work of the fullest SM
    // (throughput) plus 256 threads' worth for every pass of a block over its cells (latency).
    // Which lattices and calls: those whose steps are then faster than by the kernels of a single step, of up to
    // 2^18 cells (the staging area holds the second copy).  A launch of tiles costs about 5 us more than its
    // steps, so larger lattices want more steps a call.  Microseconds a step, tiles and single steps:
    //   FP32 D3Q19, two cells a thread, 10 steps a call: 44^3 6.9 and 8.3, 48^3 7.3 and 8.4, 50^3 8.5 and 8.6, 60^3
    //     10.6 and 10.3, 100 steps: 50^3 8.0 and 8.6, 60^3 10.1 and 10.3, 64^3 11.0 and 10.7; one cell, 10 steps:
    //     33 x 32^2 5.2 and 6.8, 41 x 40^2 6.8 and 7.4, 49 x 48^2 8.6 and 8.5 (100 steps 8.1 and 8.4), 61 x 60^2
    //     12.8 and 10.7
    //   FP16 D3Q19: 64^3 10.7 and 17.5; one cell: 49 x 48^2 8.3 and 8.9, 63^3 13.6 and 11.5
    //   FP64 D2Q9: 256^2 61 and 70, 362^2 124 and 129, 400^2 152 and 156, 512^2 223 and 213; FP64 D3Q19 is bound
    //     by the FP64 pipe, where the ring's psi is extra work
    //   FP32 D2Q9 with 2 / 4 / 6 / 10 steps a call: 256^2 5.2 / 4.7 / 4.2 / 3.9 and 5.2, 362^2 6.3 / 5.2 / 4.9 / 4.6
    //     and 5.8, 512^2 8.3 / 7.3 / 6.9 / 6.6 and 7.1, one cell, 511^2 9.3 / 8.1 / 7.6 / 7.2 and 7.2
    template <int FORM> static bool tile_plan(const KParams &p, int mrt, TileArgs &t) {
        const void *k = tile_kernel<FORM>(p, mrt);
        const int w = !std::is_same<S, double>::value && p.nx % 2 == 0 ? 2 : 1;
        const int nw = p.nx / w, sms = sm_count();
        constexpr bool d3 = L::D == 3, fp64 = std::is_same<S, double>::value, fp32 = std::is_same<S, float>::value;
        const long long most_cells = fp64 ? (d3 ? 1 << 14 : 10 << 14)
                                   : FORM || !d3 ? 1 << 18
                                   : fp32        ? (w == 2 ? 14 << 14 : 7 << 14)
                                                 : (w == 2 ? 1 << 18 : 1 << 17);
        if (p.n > most_cells) return false;
        const long long work = p.n * (2 / w);
        t.least = FORM || fp64 || (d3 && !fp32 && w == 2) || work <= 1 << 16 ? 2
                : d3 && fp32 && w == 2 && p.n > 7 << 14 ? 16 : work <= 13 << 14 ? 4 : work <= 1 << 18 ? 6 : 10;
        const size_t most = 200 * 1024;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        long long best = -1;
        constexpr int ring = L::D == 3 ? 2 : 0;
        TileArgs c = t;
        const int unit = w == 2 ? tile_unit<S, 2> : tile_unit<S, 1>, units = tile_units(nw, unit);
        for (c.gx = 1; c.gx <= 16 && c.gx <= units; ++c.gx) {
            for (c.gz = 1; c.gz <= 32 && (c.gz == 1 || p.nz / c.gz >= 2); ++c.gz) {
                for (int per_sm = 1; per_sm <= 3; ++per_sm) {
                    c.gy = sms * per_sm / (c.gx * c.gz);
                    if (c.gy > p.ny / 2) c.gy = p.ny / 2;
                    if (c.gy < 1) c.gy = 1;
                    const long long tiles = (long long)c.gx * c.gy * c.gz;
                    if (tiles > kMaxTiles || tiles > (long long)sms * per_sm) continue;
                    int tw = (units + c.gx - 1) / c.gx * unit + (nw % unit == 1 ? 1 : 0);
                    tw = units == 1 || tw > nw ? nw : tw;
                    const int th = (p.ny + c.gy - 1) / c.gy, td = (p.nz + c.gz - 1) / c.gz;
                    if (tw > 1023 || th > 1023 || td > 1023) continue;
                    c.max_own = (tw * th * td + 1) & ~1;          // even: 8-byte alignment of what follows
                    c.max_region = ((tw + 2) * (th + 2) * (td + ring) + 1) & ~1;
                    const int here = (int)((tiles + sms - 1) / sms);       // blocks on the fullest SM
                    c.threads = TileThreads<L, S>::per_sm / here / 32 * 32;
                    if (c.threads > TileThreads<L, S>::most) c.threads = TileThreads<L, S>::most;
                    const int even = ((c.max_region + 31) / 32) * 32;
                    if (c.threads > even) c.threads = even < 64 ? 64 : even;
                    const long long fit = (long long)(227 * 1024) / (long long)(tile_smem(p, c) + 1024);
                    if (fit < here || tile_smem(p, c) > most) continue;
                    // a collision in units of psi of a region cell: 2 in FP32 (64^3: 1900 cycles a pass
                    // for psi, 4400 for the collision), 8 in FP64 (60 and 424 pipe operations)
                    const int cost = std::is_same<S, double>::value ? 8 : 2;
                    const long long rounds = (c.max_region + c.threads - 1) / c.threads +
                                             cost * ((c.max_own + c.threads - 1) / c.threads);
                    const long long work = here * ((long long)cost * c.max_own + c.max_region) + 256 * rounds;
                    if (best < 0 || work < best) {
                        best = work;
                        t = c;
                    }
                }
            }
        }
        if (best < 0) return false;
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, t.threads, tile_smem(p, t)) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        return (long long)nb * sms >= (long long)t.gx * t.gy * t.gz;
    }
    template <int FORM> static cudaError_t tile_run(const KParams &p, int mrt, const TileArgs &t, cudaStream_t st) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(t.gx * t.gy * t.gz, 1, 1);
        cfg.blockDim = dim3(t.threads, 1, 1);
        cfg.dynamicSmemBytes = tile_smem(p, t);
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        void *args[] = {const_cast<KParams *>(&p), const_cast<TileArgs *>(&t)};
        return cudaLaunchKernelExC(&cfg, tile_kernel<FORM>(p, mrt), args);
    }
    static const void *batch_bgk() { return reinterpret_cast<const void *>(&k_batch<L, S, 0>); }
    static const void *batch_mrt() { return reinterpret_cast<const void *>(&k_batch<L, S, 1>); }
    static constexpr Launchers table() {
        return Launchers{&init,     &psi,    {&collide_bgk, &collide_mrt}, &moments, &get_pops, &set_pops, &reduce,
                         {&batch_bgk, &batch_mrt}, &rebalance, &wall_fill,
                         {std::is_same<S, double>::value ? nullptr : &fused_bgk,
                          std::is_same<S, double>::value ? nullptr : &fused_mrt},
                         {&tile_plan<0>, &tile_plan<1>}, {&tile_run<0>, &tile_run<1>},
                         &mass};
    }
};

}  // namespace plb
