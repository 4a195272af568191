// lbcm_fused.cuh -- the fused step kernel (params.step_kernel = 1): both passes of a step in one
// cooperative launch, for any storage (arXiv:1804.08923, Section II).
#pragma once
#include "lbcm_internal.h"
#include "lbcm_node.cuh"

namespace lbcm {

// ------------------------------------------------------- fused step (one launch)
// Both passes of a step in one cooperative launch (params.step_kernel = 1).  The work is a fixed
// sequence of items, each a 32 x kFusedRows tile of one plane: the gathers of a plane are issued
// lag planes before the collisions that read them (FusedCtl::ops), and block b takes items b,
// b + G, b + 2G, ... (G blocks, all resident).  A gather item counts itself into done[z] once its
// writes are visible device-wide; a collision item of plane z waits until planes z - 1, z, z + 1
// are counted complete.  Every item waits only for items earlier in the sequence, held by
// resident blocks that do not wait on it, so the waits end; each is also bounded, and on running
// out it sets f.err (reported by the next synchronising call) and goes on.  With the lag (about
// one round of G items) a collision item seldom waits, and a plane's 48-byte moments are read a
// few planes after they were written: they stay in L2 (stored with the evict-last policy) and,
// read once, their lines are dropped without being written back.  The step then moves close to
// the method's 448 bytes a node from DRAM (450-500 measured, against 522 for the two launches),
// but its blocks wait and synchronise at every item and it streams at a lower fraction of the
// bandwidth: on GB300 it is 3% slower than the two launches on the 256x256x1024 jet and about
// level with them on smaller ones, and the two launches, or the advance where a call takes several
// steps, stay the default.
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}


// Waits until the gathers of planes p0, p1, p2 are all counted complete (the three counters
// are read together).  Bounded by time, kFusedWaitNs, and as a backstop by the number of
// polls; on giving up it sets f.err and returns.
__device__ __forceinline__ void wait_planes(const FusedCtl &f, int p0, int p1, int p2) {
    const unsigned long long t0 = global_ns();
    for (long long k = 0;; ++k) {
        const unsigned long long d0 = ld_acquire_u64(f.done + p0), d1 = ld_acquire_u64(f.done + p1),
                                 d2 = ld_acquire_u64(f.done + p2);
        if (d0 >= f.target && d1 >= f.target && d2 >= f.target) return;
        if (global_ns() - t0 > kFusedWaitNs || k > kFusedSpinLimit) {
            atomicExch(f.err, 1);
            return;
        }
        __nanosleep(64);
    }
}

// K: a storage's gather and collision of one node (moments<W>, collide<kForce>), and its blocks per SM.
template <class K, bool kForce, bool W>
__global__ void __launch_bounds__(128, K::kBlocks) step_kernel(StepArgs a, FusedCtl f) {
    // items are 32 x kFusedRows tiles of a plane, taken by the blocks round-robin; each warp
    // walks kFusedRows / 4 rows of the tile
    const bool lead = threadIdx.x == 0 && threadIdx.y == 0;
    const int T = f.items_x * f.items_y;
    const long long total = (long long)f.nops * T;
    const unsigned long long pol = l2_evict_last_policy();
    for (long long it = blockIdx.x; it < total; it += gridDim.x) {
        const int op = (int)(it / T), t = (int)(it - (long long)op * T);
        const int2 o = f.ops[op];
        const int z = o.y;
        const int x = (t % f.items_x) * 32 + threadIdx.x;
        const int y0 = (t / f.items_x) * kFusedRows;
        if (o.x == 0) {  // gather: phase entries and moments of the tile
#pragma unroll 1
            for (int r = threadIdx.y; r < kFusedRows; r += 4) {
                const int y = y0 + r;
                if (x < a.nx && y < a.ny) K::template moments<W>(a, x, y, z, pol);
            }
            __syncthreads();
            if (lead) {
                __threadfence();
                atomicAdd(f.done + z, 1ull);
            }
        } else {  // collision of the tile, once the three planes of its stencil are gathered
            if (lead) {
                const bool pz = a.bc_zlo == BC_PERIODIC;
                wait_planes(f, z, (z > 0 || pz) ? (z > 0 ? z - 1 : a.nz - 1) : z,
                            (z < a.nz - 1 || pz) ? (z < a.nz - 1 ? z + 1 : 0) : z);
            }
            __syncthreads();
#pragma unroll 1
            for (int r = threadIdx.y; r < kFusedRows; r += 4) {
                const int y = y0 + r;
                const bool in = x < a.nx && y < a.ny;
                if (in) K::template collide<kForce>(a, x, y, z);
                if (f.discard) {  // every lane has read its moments: drop the lines
                    __syncwarp();
                    if (in && (threadIdx.x & 7) == 0) {
                        const size_t n = ((size_t)z * a.ny + y) * a.nx + x, NN = (size_t)a.NN;
                        l2_discard(a.mom + n);
                        l2_discard(a.mom + NN + n);
                        l2_discard(a.mom + 2 * NN + n);
                    }
                }
            }
        }
        __syncthreads();
    }
}

// Launches the fused kernel of K, or, occ not NULL, asks for its blocks per SM.
template <class K>
static cudaError_t fused_run(const StepArgs &a, const FusedCtl &f, int grid, cudaStream_t s, int *occ) {
    const bool force = a.gx != 0.0f || a.gy != 0.0f || a.gz != 0.0f;
    const bool walls = a.wall_x || a.wall_y;
    const void *fn = force ? (walls ? (const void *)step_kernel<K, true, true> : (const void *)step_kernel<K, true, false>)
                           : (walls ? (const void *)step_kernel<K, false, true> : (const void *)step_kernel<K, false, false>);
    if (occ) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, fn, 128, 0);
    void *args[] = {(void *)&a, (void *)&f};
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(32, 4, 1), args, 0, s);
}

}  // namespace lbcm
