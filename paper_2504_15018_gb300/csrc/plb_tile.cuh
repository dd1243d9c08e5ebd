// Many time steps of a small lattice in one launch: every block keeps one tile of the lattice for
// all steps and waits for its neighbour tiles only.
//
// A small lattice's step is bound by launches, not by work: at 256 x 256 cells (D2Q9) a step needs
// about 1 us of the GPU but two launches of 4 us of host time each.  Here the blocks stay: for each
// step a block forms psi of its tile and of the ring around it in shared memory from the populations
// of copy A, collides its own cells and pushes them into copy B (the single-pass step's scheme, so
// one exchange between blocks per step instead of two); the copies change roles every step.  The
// populations that psi was formed from wait in shared memory for the collision.
//
// Neighbours: a tile's step reads populations of the tile and its ring, which the tiles around it
// (across the periodic wrap, diagonals included) wrote in the step before, and writes into the same
// set.  With tiles at least two rows, planes and (two-cell path) pairs thick, it is enough that these
// tiles have finished the step before: their step count is published with a release after the
// block's stores and read before a fence; populations bypass L1.  The counts only grow, and every
// launch starts from the block's own count, so nothing has to be cleared between launches.  The
// launch is cooperative (all tiles resident), and every wait is bounded: one that runs out records
// FLAG_TIMEOUT and the blocks leave, as do those of later launches until the counts are cleared (the
// tiles stand at different steps, and counts say nothing about neighbours any more).
//
// What bounds it: the chain poll -> L2 loads -> psi -> collision -> stores -> release, about 2.7 us a
// step when every thread has one cell or pair (clock64 of an 8 x 256 lattice: 1300 cycles psi, 930
// collision, 950 release, 2000 until the neighbours' counts arrive); the redundant psi of the ring is
// cheap beside it.  Microseconds a step, kernels of a single step (which start under the tail of the one
// before) and tiles, 100 steps a call: D2Q9 FP32 8 x 256 4.3 and 2.6, 256 x 256 5.2 and 3.5, 512 x 512 7.0 and
// 6.1; D3Q19 FP32 32^3 7.1 and 3.8, 48^3 8.4 and 6.8; D2Q9 FP64 256 x 256 70 and 61, 301 x 203 82 and 58.
#pragma once
#include "plb_pair.cuh"

namespace plb {

// Threads resident per SM that the register allocation leaves room for, and the largest block.
template <class L, class S> struct TileThreads { static constexpr int most = 512, per_sm = L::Q == 9 ? 768 : 512, regs = L::Q == 9 ? 80 : 128; };
template <class L> struct TileThreads<L, double> { static constexpr int most = 256, per_sm = L::Q == 9 ? 512 : 256, regs = L::Q == 9 ? 128 : 255; };

struct LdShared {
    template <class U> __device__ __forceinline__ static U ro(const U *a) { return *a; }
};

__device__ __forceinline__ unsigned ld_relaxed(const unsigned *a) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
    return v;
}

__device__ __forceinline__ void fence_acq_rel() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// First row (plane) of tile k of g over n; tile k ends where tile k + 1 begins.
__host__ __device__ inline int tile_lo(int n, int g, int k) { return (int)((long long)n * k / g); }
// The same along x, for n threads' worth of cells: tiles begin at multiples of `unit` (whole 128-byte
// lines of the populations); a last unit of one is left to the tile before it.
__host__ __device__ inline int tile_units(int n, int unit) {
    const int u = n / unit + (n % unit >= 2 ? 1 : 0);
    return u > 1 ? u : 1;
}
__host__ __device__ inline int tile_lo_x(int n, int unit, int g, int k) {
    const int x = unit * (int)((long long)tile_units(n, unit) * k / g);
    return k >= g || x > n ? n : x;
}
template <class S, int W> constexpr int tile_unit = 128 / (int)sizeof(S) / W;

// W = 2: two cells per thread (FP32 arithmetic, even nx); W = 1: one cell.
template <class L, class S, int MRT, bool SR, int MOM, int W>
__global__ void __maxnreg__((TileThreads<L, S>::regs)) k_tile(KParams p, TileArgs t) {
    using T = typename Store<S>::T;
    using PsiT = typename Store<S>::PsiT;
    using V = typename std::conditional<W == 2, f2, T>::type;       // a thread's cells
    extern __shared__ __align__(16) char tile_smem[];
    const int tid = threadIdx.x, tile = blockIdx.x;
    const int kx = tile % t.gx, ky = (tile / t.gx) % t.gy, kz = tile / (t.gx * t.gy);
    const int nw = p.nx / W;
    const int x0 = tile_lo_x(nw, tile_unit<S, W>, t.gx, kx), y0 = tile_lo(p.ny, t.gy, ky), z0 = tile_lo(p.nz, t.gz, kz);
    const int tw = tile_lo_x(nw, tile_unit<S, W>, t.gx, kx + 1) - x0, th = tile_lo(p.ny, t.gy, ky + 1) - y0;
    const int td = tile_lo(p.nz, t.gz, kz + 1) - z0;
    constexpr int zr = L::D == 3 ? 1 : 0;                          // ring in z
    const int own = tw * th * td, region = (tw + 2) * (th + 2) * (td + 2 * zr);
    // shared memory: populations of the own cells [Q][own], psi of the region, the region's cells, own cells
    V *pops = reinterpret_cast<V *>(tile_smem);
    PsiT *psi = reinterpret_cast<PsiT *>(pops + (size_t)L::Q * t.max_own);
    int2 *cells = reinterpret_cast<int2 *>(psi + (size_t)W * t.max_region);
    int *mine = reinterpret_cast<int *>(cells + t.max_region);
    const int sy = W * (tw + 2), sz = sy * (th + 2);
    const unsigned gave_up = ld_relaxed(t.counts);                 // (here, under the set-up)
    for (int r = tid; r < region; r += blockDim.x) {
        const int lx = r % (tw + 2), ly = (r / (tw + 2)) % (th + 2), lz = r / ((tw + 2) * (th + 2));
        const bool in = lx >= 1 && lx <= tw && ly >= 1 && ly <= th && lz >= zr && lz < td + zr;
        int x = x0 - 1 + lx, y = y0 - 1 + ly, z = z0 - zr + lz;
        x = x < 0 ? x + nw : (x >= nw ? x - nw : x);
        z = z < 0 ? z + p.nz : (z >= p.nz ? z - p.nz : z);
        bool fixed = false;
        if (p.wall_y) {
            fixed = p.wall_fixed && (y < 0 || y >= p.ny);          // wetting walls carry psi_wall
            y = y < 0 ? 0 : (y >= p.ny ? p.ny - 1 : y);            // neutral ones mirror the fluid row
        } else {
            y = y < 0 ? y + p.ny : (y >= p.ny ? y - p.ny : y);
        }
        int o = -1;
        if (in) {
            o = ((lz - zr) * th + (ly - 1)) * tw + lx - 1;
            mine[o] = (lx - 1) | (ly - 1) << 10 | (lz - zr) << 20;
        }
        cells[r] = make_int2(fixed ? -1 : W * x + p.nx * (y + p.ny * z), o);
    }
    // the neighbour tile whose count this thread watches (second warp)
    const unsigned *watch = nullptr;
    if (tid >= 32 && tid < 32 + (L::D == 3 ? 27 : 9)) {
        const int d = tid - 32;
        int ax = kx + d % 3 - 1, ay = ky + (d / 3) % 3 - 1, az = L::D == 3 ? kz + d / 9 - 1 : 0;
        const bool beyond = p.wall_y && (ay < 0 || ay >= t.gy);
        ax = (ax + t.gx) % t.gx;
        ay = (ay + t.gy) % t.gy;
        az = (az + t.gz) % t.gz;
        const int other = ax + t.gx * (ay + t.gy * az);
        if (!beyond && other != tile) watch = t.counts + kTilePitch * (1 + other);
    }
    unsigned *count = t.counts + kTilePitch * (1 + tile);
    const unsigned start = *reinterpret_cast<volatile unsigned *>(count);
    S *src = static_cast<S *>(t.a), *dst = static_cast<S *>(t.b);
    for (int s = 0; s < t.nsteps; ++s) {
        int ok = s > 0 || gave_up == 0;
        if (s > 0 && watch) {
            unsigned spins = 0;
            while ((int)(ld_relaxed(watch) - (start + (unsigned)s)) < 0) {
                if (++spins > t.spin_limit || ((spins & 63) == 0 && ld_relaxed(t.counts) != 0)) {
                    atomicExch(t.counts, 1u);
                    atomicOr(p.flags, FLAG_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
            fence_acq_rel();
        }
        if (!__syncthreads_and(ok)) return;
        // ---- psi of the tile and its ring
        Planes<S> A, B;
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            A.p[i] = src + (long long)i * p.pstride;
            B.p[i] = dst + (long long)i * p.pstride;
        }
        for (int r = tid; r < region; r += blockDim.x) {
            const int2 c = cells[r];
            if (c.x < 0) {
                const PsiT v = (PsiT)phys<T>(p).psi_wall;
                psi[W * r] = v;
                if (W == 2) psi[W * r + 1] = v;
                continue;
            }
            V f[L::Q];
            if constexpr (W == 2) {
#pragma unroll
                for (int i = 0; i < L::Q; ++i) f[i] = PairIO<S>::template ld2<LdCoherent>(elem(A.p[i], c.x));
                f2 rho = f[0];
#pragma unroll
                for (int i = 1; i < L::Q; ++i) rho += f[i];
                if (Store<S>::SHIFT) rho += f2(p.f.rho_ref);       // sum_i w_i rho_ref = rho_ref
                *reinterpret_cast<float2 *>(psi + 2 * r) = psi_pair_of(p, rho).v;
            } else {
#pragma unroll
                for (int i = 0; i < L::Q; ++i) f[i] = Store<S>::template ld<LdCoherent>(A.p[i] + c.x);
                psi[r] = psi_cell<L, S>(p, f);
            }
            if (c.y >= 0) {
#pragma unroll
                for (int i = 0; i < L::Q; ++i) pops[i * t.max_own + c.y] = f[i];
            }
        }
        __syncthreads();
        // ---- collision of the own cells, pushed into the other copy
        const unsigned salt = p.salt + (unsigned)s;
        for (int o = tid; o < own; o += blockDim.x) {
            const int m = mine[o], lx = m & 1023, ly = (m >> 10) & 1023, lz = m >> 20;
            const int y = y0 + ly, z = z0 + lz;
            V f[L::Q];
#pragma unroll
            for (int i = 0; i < L::Q; ++i) f[i] = pops[i * t.max_own + o];
            const PsiT *pc = psi + (W * (lx + 1) + sy * (ly + 1) + sz * (lz + zr));
            const bool wall = p.wall_y && (y == 0 || y == p.ny - 1);
            V F[3];
            if constexpr (W == 2) {
                auto at = [&](int cx, int cy, int cz) -> f2 {
                    const float *r = pc + cy * sy + cz * sz;
                    const float2 c = *reinterpret_cast<const float2 *>(r);
                    if (cx == 0) return f2(c);
                    if (cx < 0) return f2(r[-1], c.x);
                    return f2(c.y, r[2]);
                };
                force_pair_from<L>(p, at, F);
                GeoPair g;
                geo_pair_at(p, 2 * (x0 + lx), y, z, g);
                if (wall) collide_store_pair<L, S, MRT, true, true, SR, MOM>(p, B, g, f, F, salt);
                else collide_store_pair<L, S, MRT, true, false, SR, MOM>(p, B, g, f, F, salt);
            } else {
                Geo<int> g;
                geo_at<int>(p, x0 + lx, y, z, g);
                if constexpr (std::is_same<S, double>::value) {
                    plain::force<L, LdShared>(p, pc, sy, sz, F);
                    plain::collide<L, MRT>(p, f, F);
                } else {
                    force_fast<L, T, LdShared>(p, pc, sy, sz, F);
                    collide_fast<L, MRT, Store<S>::SHIFT, T>(p, f, F);
                }
                if (wall) store_fast<L, S, true, true, SR>(p, B, g, f, salt);
                else store_fast<L, S, true, false, SR>(p, B, g, f, salt);
            }
        }
        __syncthreads();
        if (tid == 0 && !(t.withhold && tile == 0))
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(count), "r"(start + (unsigned)s + 1) : "memory");
        S *const u = src;
        src = dst;
        dst = u;
    }
}

}  // namespace plb
