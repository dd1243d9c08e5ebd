// Persistent kernel of a batch of independent lattices: every step runs the psi pass over
// all tiles of its instances, a grid barrier, the fused force/collide/stream pass, and a
// second barrier, for nsteps steps in one launch (a batch larger than L2: one group of instances after
// the other, each for all steps).  Loads follow LdBatch (populations through
// L2 only, the psi stencil through L1 after the barrier's acquire):
// blocks read, across barriers, what other SMs wrote in the same launch.
#pragma once
#include "plb_pair.cuh"

namespace plb {

// Minimum resident 256-thread blocks per SM requested from the register allocator (D2Q9: 80 registers, 3
// blocks; D3Q19: 128, 2 blocks).  Most kernels spill a little there (24 to 72 bytes; D3Q19 FP64 BGK 256), which
// costs less than a block fewer: 24 D3Q19 lattices of 24 to 64 a side, FP32 BGK / MRT 81 / 84 us a step (107 / 114
// before the even tiles, with 0 / 12 bytes), eight in FP64 1235 / 2012 (2533 / 4013).
template <class L> struct BatchMinBlocks { static constexpr int value = L::Q == 9 ? 3 : 2; };

// Grid-wide barrier with a bounded wait.  Returns false (in every thread of the block) when
// any block gave up waiting, after which the kernel returns.
__device__ __forceinline__ bool grid_sync(GridBar *bar, unsigned expected, unsigned spin_limit) {
    __syncthreads();
    __shared__ int s_ok;
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        volatile unsigned *vgen = &bar->gen;
        volatile unsigned *verr = &bar->err;
        const unsigned gen = *vgen;
        __threadfence();
        const unsigned arrived = atomicAdd(&bar->count, 1u);
        if (arrived == expected - 1) {
            atomicExch(&bar->count, 0u);
            __threadfence();
            atomicAdd(&bar->gen, 1u);
        } else {
            unsigned spins = 0;
            while (*vgen == gen) {
                if (*verr) break;
                if (++spins > spin_limit) {
                    atomicOr(&bar->err, 1u);
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
        s_ok = *verr == 0;
    }
    __syncthreads();
    return s_ok != 0;
}

template <class L, class S, int MRT, bool PSI, bool SR>
__device__ __forceinline__ void batch_tile(const BatchInst &in, const BatchTile &tl, int odd, unsigned salt) {
    const KParams &p = in.kp;
    const Planes<S> &A = *reinterpret_cast<const Planes<S> *>(in.pl);
    using PsiT = typename Store<S>::PsiT;
    for (int u = tl.u0 + threadIdx.x; u < tl.u1; u += blockDim.x) {
        const int y = u / in.upr, xu = u - y * in.upr;
        const bool wall = odd && p.wall_y && (y == 0 || y == p.ny - 1);
        bool done = false;
        if constexpr (!std::is_same<S, double>::value) {
            if (in.pair) {
                GeoPair g;
                geo_pair_at(p, 2 * xu, y, tl.z, g);
                float *psi = static_cast<float *>(in.psi);
                if (PSI) {
                    if (!odd) psi_pair_body<L, S, false, false, LdBatch>(p, A, psi, g);
                    else if (wall) psi_pair_body<L, S, true, true, LdBatch>(p, A, psi, g);
                    else psi_pair_body<L, S, true, false, LdBatch>(p, A, psi, g);
                } else {
                    if (!odd) collide_pair_body<L, S, MRT, false, false, LdBatch, SR>(p, A, psi, g, salt);
                    else if (wall) collide_pair_body<L, S, MRT, true, true, LdBatch, SR>(p, A, psi, g, salt);
                    else collide_pair_body<L, S, MRT, true, false, LdBatch, SR>(p, A, psi, g, salt);
                }
                done = true;
            }
        }
        if (!done) {
            Geo<int> g;
            geo_at<int>(p, xu, y, tl.z, g);
            PsiT *psi = static_cast<PsiT *>(in.psi);
            if (PSI) {
                if (!odd) psi_body<L, S, false, false, LdBatch>(p, A, psi, g);
                else if (wall) psi_body<L, S, true, true, LdBatch>(p, A, psi, g);
                else psi_body<L, S, true, false, LdBatch>(p, A, psi, g);
            } else {
                if (!odd) collide_body<L, S, MRT, false, false, LdBatch, SR>(p, A, psi, g, salt);
                else if (wall) collide_body<L, S, MRT, true, true, LdBatch, SR>(p, A, psi, g, salt);
                else collide_body<L, S, MRT, true, false, LdBatch, SR>(p, A, psi, g, salt);
            }
        }
    }
}

// Instance descriptors that a block keeps in shared memory: its tiles are consecutive, so they belong to
// few instances, and parameters read from shared memory replace about 60 loads per cell from global
// memory, which the barriers' acquires drop from L1.
constexpr int kBatchWindow = 4;

template <class L, class S, int MRT>
__global__ void __launch_bounds__(256, BatchMinBlocks<L>::value) k_batch(BatchLaunch b) {
    __shared__ BatchInst window[kBatchWindow];
    const unsigned salt0 = *reinterpret_cast<volatile unsigned *>(&b.bar->salt);
    int held = -1;                                // first instance in the window (the same in all threads)
    auto instance = [&](int k) -> const BatchInst & {
        if (held < 0 || k < held || k >= held + kBatchWindow) {
            static_assert(sizeof(BatchInst) % 8 == 0, "copied in 8-byte words");
            __syncthreads();
            held = k;
            const int n = b.ninst - k < kBatchWindow ? b.ninst - k : kBatchWindow;
            const unsigned long long *src = reinterpret_cast<const unsigned long long *>(b.insts + k);
            unsigned long long *dst = reinterpret_cast<unsigned long long *>(window);
            for (int w = threadIdx.x; w < n * (int)(sizeof(BatchInst) / 8); w += blockDim.x) dst[w] = src[w];
            __syncthreads();
        }
        // (through a pointer of unknown origin: knowing that no store changes the window, the compiler
        // loads all parameters up front and spills 90 bytes)
        const BatchInst *in = window + (k - held);
        asm("" : "+l"(in));
        return *in;
    };
    // group by group, each for all steps; in a group, consecutive tiles, the same number (give or take one)
    // for every block
    for (int group = 0; group < b.ngroups; ++group) {
        const int g0 = b.groups[group], gn = b.groups[group + 1] - g0;
        const int t0 = g0 + (int)((long long)gn * blockIdx.x / gridDim.x);
        const int t1 = g0 + (int)((long long)gn * (blockIdx.x + 1) / gridDim.x);
        for (int step = 0; step < b.nsteps; ++step) {
            for (int t = t0; t < t1; ++t) {
                const BatchTile tl = b.tiles[t];
                const BatchInst &in = instance(tl.inst);
                batch_tile<L, S, MRT, true, false>(in, tl, (in.odd + step) & 1, 0);
            }
            if (!grid_sync(b.bar, b.expected, b.spin_limit)) return;
            for (int t = t0; t < t1; ++t) {
                const BatchTile tl = b.tiles[t];
                const BatchInst &in = instance(tl.inst);
                const int odd = (in.odd + step) & 1;
                if constexpr (Store<S>::SHIFT) {
                    if (in.kp.stochastic) {
                        batch_tile<L, S, MRT, false, true>(in, tl, odd, salt0 + step);
                        continue;
                    }
                }
                batch_tile<L, S, MRT, false, false>(in, tl, odd, 0);
            }
            if (!grid_sync(b.bar, b.expected, b.spin_limit)) return;
        }
    }
    // every block has passed the last barrier: advance the stored parities and the step salt
    if (blockIdx.x == 0) {
        if (b.nsteps & 1)
            for (int k = threadIdx.x; k < b.ninst; k += blockDim.x) b.insts[k].odd ^= 1;
        if (threadIdx.x == 0) b.bar->salt = salt0 + b.nsteps;
    }
}

}  // namespace plb
