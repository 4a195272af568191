// lbcm_fragments.cu -- fragment analysis of a state (arXiv:1804.08923, Section IV.B: binarise
// the order parameter, connected components, volume, equivalent spherical diameter).
//
// Labelling is union-find over the lattice with lock-free links: every jet node starts under the
// first of its run of jet nodes in a row (per warp), each node unites with its jet neighbours in
// the backward half of the neighbourhood (3 face neighbours, or 13 of the 26) where no run connects
// them anyway, and a union links the larger root under the smaller with atomicMin.  Parents only decrease and always stay inside the component, so
// after the unions every component is one tree whose root is its smallest linear node index:
// the labels are canonical (independent of the schedule) and comparable with a sequential
// flood fill.  Volumes come from integer atomics on the root; the roots are compacted in index
// order (per-block counts, one scan, per-block ballots), so the output is deterministic.
#include "lbcm_device.cuh"
#include "lbcm_internal.h"

#include <algorithm>

namespace lbcm {

// Smallest-index root of x (parents only decrease: at most x steps).  Volatile reads: other
// SMs relink parents during the union kernel, and a stale cached parent would only cost retries.
__device__ __forceinline__ int frag_find(const volatile int *p, int x, int limit, int *err) {
    for (int it = 0; it < limit; ++it) {
        const int q = p[x];
        if (q == x) return x;
        x = q;
    }
    *err = 1;
    return x;
}

__device__ __forceinline__ void frag_unite(int *p, int a, int b, int limit, int *err) {
    for (int it = 0; it < limit; ++it) {
        a = frag_find(p, a, limit, err);
        b = frag_find(p, b, limit, err);
        if (a == b) return;
        const int hi = max(a, b), lo = min(a, b);
        const int old = atomicMin(&p[hi], lo);
        if (old == hi) return;  // hi was a root and now hangs under lo
        a = old;                // hi was linked meanwhile: unite its new parent with lo
        b = lo;
    }
    *err = 1;
}

// Labels of jet nodes (phi > 0 of the state's colour densities), -1 elsewhere.  A warp holds 32
// consecutive nodes: each jet node starts under the first node of its run of jet nodes in the warp's
// part of its row, so that runs need no unions and chains start short.
template <int S>
__global__ void __launch_bounds__(256) frag_init_kernel(StepArgs a, int *label) {
    const int lane = threadIdx.x & 31;
    for (long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x - lane; b < a.NN; b += (long long)gridDim.x * blockDim.x) {
        const long long n = b + lane;
        bool jet = false, first = true;
        if (n < a.NN) {
            const int x = (int)(n % a.nx);
            float rr = 0.0f, rb = 0.0f;
            auto add = [&](float2 v) {
                rr += v.x;
                rb += v.y;
            };
            if constexpr (S == STORE_FP32) {
#pragma unroll
                for (int i = 0; i < 27; ++i) add(load_pop<S>(a, i, (int)n, no_shift()));
            } else {
                const Nbr nb(a, x, (int)((n / a.nx) % a.ny), (int)(n / a.plane));
#pragma unroll
                for (int i = 0; i < 27; ++i) add(stored_pop<S>(a, nb, i));
            }
            jet = rr * a.inv_rho_r0 > rb * a.inv_rho_b0;  // phi > 0  <=>  rho_r / rho_r0 > rho_b / rho_b0 (Eq. (23))
            first = x == 0;
        }
        // a run starts at a jet node that opens a row or follows a node outside the jet
        const unsigned in = __ballot_sync(0xffffffffu, jet);
        const unsigned starts = in & (__ballot_sync(0xffffffffu, first) | ~(in << 1));
        if (n < a.NN) label[n] = jet ? (int)(b + (31 - __clz(starts & (0xffffffffu >> (31 - lane))))) : -1;
    }
}

struct FragGeom {
    int nx, ny, nz, periodic_z, conn, wall_x, wall_y;
    long long NN, plane;
};

// Unites every jet node with its jet neighbours in the backward half of the neighbourhood: the node
// before it in its row, and the rows (dy, dz) with dz < 0, or dz = 0 and dy < 0.  Of a row's three
// neighbours (dx = -1, 0, 1; one, dx = 0, with face connectivity) only those are united that no run
// connects anyway: a jet neighbour at dx = 0 stands for those beside it, and where the node before
// is in the jet too it has united that one (dx = 0 here is dx = 1 there), or with face connectivity
// the pair before has been united if both of it are in the jet.
__global__ void __launch_bounds__(256) frag_union_kernel(FragGeom g, int *label, int *err) {
    const int limit = (int)min(g.NN, (long long)INT32_MAX);
    const volatile int *lab = label;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < g.NN; n += (long long)gridDim.x * blockDim.x) {
        if (lab[n] < 0) continue;
        const int x = (int)(n % g.nx), y = (int)((n / g.nx) % g.ny), z = (int)(n / g.plane);
        const bool left = x > 0 && lab[n - 1] >= 0;  // the run goes on from the node before
        if (left) {
            if ((n & 31) == 0) frag_unite(label, (int)n, (int)n - 1, limit, err);  // from another warp's part
        } else if (x == 0 && !g.wall_x && g.nx > 1 && lab[n + g.nx - 1] >= 0) {
            frag_unite(label, (int)n, (int)n + g.nx - 1, limit, err);  // across the periodic side
        }
        for (int dz = -1; dz <= 0; ++dz)
            for (int dy = -1; dy <= (dz ? 1 : -1); ++dy) {
                if (g.conn == 6 && dz && dy) continue;
                int zz = z + dz, yy = y + dy;
                if (zz < 0) {
                    if (!g.periodic_z) continue;
                    zz += g.nz;
                }
                if (yy < 0 || yy >= g.ny) {
                    if (g.wall_y) continue;  // no neighbour across a side wall
                    yy = yy < 0 ? yy + g.ny : yy - g.ny;
                }
                const long long row = (long long)zz * g.plane + (long long)yy * g.nx;
                const bool mid = lab[row + x] >= 0;
                auto unite = [&](int xx) {
                    const long long m = row + xx;
                    if (m != n && lab[m] >= 0) frag_unite(label, (int)n, (int)m, limit, err);
                };
                if (g.conn == 6) {
                    if (mid && !(left && lab[row + x - 1] >= 0)) unite(x);
                } else if (mid) {
                    if (!left) unite(x);
                } else {
                    if (!left) {
                        if (x > 0) unite(x - 1);
                        else if (!g.wall_x) unite(g.nx - 1);
                    }
                    if (x < g.nx - 1) unite(x + 1);
                    else if (!g.wall_x) unite(0);
                }
            }
    }
}

constexpr int kFragBlock = 1024;

// count[root] = nodes of the component, touch[root] = 1 if it has a node on z = 0, and the roots per
// block of kFragBlock nodes.  The lanes of a warp that share a root add to it once (a long column is
// one component: its nodes would queue at one address).
__global__ void __launch_bounds__(kFragBlock) frag_count_kernel(FragGeom g, const int *label, int *count, uint8_t *touch,
                                                               int *bc, int *err) {
    __shared__ int sh[32];
    const int limit = (int)min(g.NN, (long long)INT32_MAX);
    const long long n = (long long)blockIdx.x * kFragBlock + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int l = n < g.NN ? label[n] : -1;
    const int r = l >= 0 ? frag_find(label, l, limit, err) : -1;
    const unsigned same = __match_any_sync(0xffffffffu, r);
    if (r >= 0) {
        if (lane == __ffs(same) - 1) atomicAdd(&count[r], __popc(same));
        if (n < g.plane) touch[r] = 1;
    }
    const unsigned m = __ballot_sync(0xffffffffu, l >= 0 && l == (int)n);
    if (lane == 0) sh[threadIdx.x >> 5] = __popc(m);
    __syncthreads();
    if (threadIdx.x < 32) {
        int s = sh[threadIdx.x];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) bc[blockIdx.x] = s;
    }
}

// Exclusive scan of the block counts (one block; chunks of 1024 in order); total in bc[nblk].
__global__ void __launch_bounds__(1024) frag_scan_kernel(const int *bc, long long nblk, long long *boff) {
    __shared__ long long sh[1024];
    long long carry = 0;
    for (long long base = 0; base < nblk; base += 1024) {
        const long long i = base + threadIdx.x;
        const long long v = i < nblk ? bc[i] : 0;
        sh[threadIdx.x] = v;
        __syncthreads();
        for (int o = 1; o < 1024; o <<= 1) {  // inclusive Hillis-Steele scan
            const long long t = (int)threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
            __syncthreads();
            sh[threadIdx.x] += t;
            __syncthreads();
        }
        if (i < nblk) boff[i] = carry + sh[threadIdx.x] - v;
        const long long tot = sh[1023];
        __syncthreads();
        carry += tot;
    }
    if (threadIdx.x == 0) boff[nblk] = carry;
}

// Roots in index order with their volumes and z = 0 flags.
__global__ void __launch_bounds__(kFragBlock) frag_write_kernel(FragGeom g, const int *label, const int *count,
                                                               const uint8_t *touch, const long long *boff,
                                                               long long *out_root, long long *out_vol,
                                                               uint8_t *out_touch) {
    __shared__ int sh[32];
    const long long n = (long long)blockIdx.x * kFragBlock + threadIdx.x;
    const bool root = n < g.NN && label[n] == (int)n;
    const unsigned m = __ballot_sync(0xffffffffu, root);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) sh[warp] = __popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int w = 0; w < kFragBlock / 32; ++w) {
            const int c = sh[w];
            sh[w] = s;
            s += c;
        }
    }
    __syncthreads();
    if (root) {
        const long long k = boff[blockIdx.x] + sh[warp] + __popc(m & ((1u << lane) - 1u));
        out_root[k] = n;
        out_vol[k] = count[n];
        out_touch[k] = touch[n];
    }
}

static int frag_grid(long long n) {
    long long b = (n + 255) / 256;
    return (int)std::min<long long>(std::max<long long>(b, 1), 152ll * 32);
}

cudaError_t launch_fragments_label(const StepArgs &a, int storage, int connectivity, int *label, int *count,
                                   uint8_t *touch, int *bc, long long *boff, int *err, cudaStream_t s,
                                   long long *launches) {
    FragGeom g{a.nx, a.ny, a.nz, a.bc_zlo == BC_PERIODIC, connectivity, a.wall_x, a.wall_y, a.NN, a.plane};
    if (storage == STORE_FP16)
        frag_init_kernel<STORE_FP16><<<frag_grid(a.NN), 256, 0, s>>>(a, label);
    else if (storage == STORE_FP16_FIT)
        frag_init_kernel<STORE_FP16_FIT><<<frag_grid(a.NN), 256, 0, s>>>(a, label);
    else
        frag_init_kernel<STORE_FP32><<<frag_grid(a.NN), 256, 0, s>>>(a, label);
    frag_union_kernel<<<frag_grid(a.NN), 256, 0, s>>>(g, label, err);
    const long long nblk = (a.NN + kFragBlock - 1) / kFragBlock;
    frag_count_kernel<<<(unsigned)nblk, kFragBlock, 0, s>>>(g, label, count, touch, bc, err);
    frag_scan_kernel<<<1, 1024, 0, s>>>(bc, nblk, boff);
    *launches += 4;
    return cudaGetLastError();
}

cudaError_t launch_fragments_write(const StepArgs &a, int connectivity, const int *label, const int *count,
                                   const uint8_t *touch, const long long *boff, long long *out_root,
                                   long long *out_vol, uint8_t *out_touch, cudaStream_t s, long long *launches) {
    FragGeom g{a.nx, a.ny, a.nz, a.bc_zlo == BC_PERIODIC, connectivity, a.wall_x, a.wall_y, a.NN, a.plane};
    const long long nblk = (a.NN + kFragBlock - 1) / kFragBlock;
    frag_write_kernel<<<(unsigned)nblk, kFragBlock, 0, s>>>(g, label, count, touch, boff, out_root, out_vol, out_touch);
    *launches += 1;
    return cudaGetLastError();
}

}  // namespace lbcm
