// lbcm_step.cu -- the per-time-step kernels of the colour-gradient central-moment LB
// method (arXiv:1804.08923), FP32 populations and arithmetic, sm_103a.
//
// One step (state S(t) -> S(t+1)) is three launches on the context's stream:
//   1. boundary_plane_kernel  incoming z = 0 populations (inlet disc / free-slip mirror),
//                             free-slip top, and the convective outflow plane
//                             f(N, t+1) = [f(N, t) + lambda f(N-1, t+1)] / (1 + lambda)
//                             (Section IV.A).  One warp per (x, y) column.
//   2. moment_kernel          pull-gathers the 54 post-stream populations of a node (the
//                             step's only gather) and writes its order parameter phi
//                             (Eq. (23)) and total density rho (Section II, densities) for
//                             the gradient stencil, and the 12 moments the collision needs
//                             (colour densities, mass, momentum, raw second moment).  One
//                             thread per node.
//   3. collide_kernel         reads a node's moments, takes the isotropic gradients of phi
//                             and rho from the fields of step 2 (end of Section II), and
//                             applies the central-moment collision with the enhanced
//                             equilibrium and GMRT forcing (Eqs. (11), (18), (21), (28),
//                             (29)), the perturbation (Eq. (30)) and the recolouring
//                             (Eqs. (33), (34)); writes the 54 post-collision populations
//                             of the node (pull scheme: streaming happens in the next
//                             step's gathers).
// With relaxation rates other than the paper's the passes are those of lbcm_general.cu.  Several steps
// of one call take advance_kernel (lbcm_advance.cu) in place of a collision and the next gather.
//
// With the paper's rates s3 = s4 = s5 = s6 = 1 (Section II, below Eq. (17)), (I - K) removes every
// central moment of order three and above, so f* depends on f only through its moments of order
// <= 2: mass, momentum and the raw second moment Pi(f).  Those of f^e and F' have closed forms
// (Pi(f^e) = rho c_s^2 I + rho u u + nu (u g + g u + (u.g) I) with c_s^2 = 9(1 - alpha)/19 and
// g = grad rho; Pi(F') = u F + F u), so the collision (collide_node, lbcm_collide.cuh) needs no
// per-direction Delta and no forward transform.
#include "lbcm_collide.cuh"
#include "lbcm_device.cuh"
#include "lbcm_internal.h"
#include "lbcm_node.cuh"

namespace lbcm {

// ------------------------------------------------------------------ boundary planes
//   z = 0 (inlet or free-slip bottom): the 9 incoming c_z = +1 populations -> zin
//   z = N free-slip top: the 9 incoming c_z = -1 populations -> zout
//   z = N convective: hist(t+1) from hist(t) and the post-stream f(N-1, t+1) (Section IV.A)
// Two kernels with the same results, bit for bit.
// boundary_plane_kernel: one warp per (x, y) column, lane i < 27 handles direction i.  Many
// warps with few instructions each: the faster of the two on planes of fewer than
// kColumnKernelPlane columns.
template <int S>
__global__ void __launch_bounds__(128) boundary_plane_kernel(StepArgs a) {
    chain_begin();
    const int lane = threadIdx.x & 31;
    const long long col = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (col >= a.plane) return;  // whole warps leave together
    const int x = (int)(col % a.nx), y = (int)(col / a.nx);
    const long long P = a.plane, pxy = col;
    const int N = a.nz - 1;
    const int i = lane < 27 ? lane : 0;
    const int cxi = cx(i), cyi = cy(i), czi = cz(i);
    const bool mine = lane < 27;
    // source column of the pull of direction i, reflected at free-slip side walls, and the
    // direction that leaves it
    int xs = x - cxi, ys = y - cyi, cxs = cxi, cys = cyi;
    if (xs < 0 || xs >= a.nx) {
        if (a.wall_x) { xs = x; cxs = -cxi; } else xs = wrapi(xs, a.nx);
    }
    if (ys < 0 || ys >= a.ny) {
        if (a.wall_y) { ys = y; cys = -cyi; } else ys = wrapi(ys, a.ny);
    }
    const int ii = dir_of(cxs, cys, czi);

    if ((a.bc_zlo == BC_INLET || a.bc_zlo == BC_FREESLIP) && mine && czi == 1) {
        float vr, vb;
        if (a.bc_zlo == BC_INLET && a.disc[(long long)ys * a.nx + xs]) {
            vr = inlet_population_at(a, i, cxs, cys, xs, ys);
            vb = 0.0f;
        } else {  // half-way specular reflection at z = -1/2
            const float2 v = load_pop<S>(a, mirror_z(ii), ys * a.nx + xs, reader_shift<S>(a, (int)pxy));
            vr = v.x;
            vb = v.y;
        }
        a.zin[(long long)zrank(i) * P + pxy] = vr;
        a.zin[(long long)(9 + zrank(i)) * P + pxy] = vb;
    }
    if (a.bc_zhi == BC_FREESLIP && mine && czi == -1) {
        const float2 v = load_pop<S>(a, mirror_z(ii), (N * a.ny + ys) * a.nx + xs,
                                     reader_shift<S>(a, N * (int)P + (int)pxy));
        a.zout[(long long)zrank(i) * P + pxy] = v.x;
        a.zout[(long long)(9 + zrank(i)) * P + pxy] = v.y;
    }
    if (a.bc_zhi == BC_CONVECTIVE) {
        // post-stream populations of node (x, y, N-1) at t+1 (N-1 >= 1: plain pulls)
        const int z = N - 1;
        float fr = 0.0f, fb = 0.0f;
        if (mine) {
            const int zs = z - czi;
            const float2 v = load_pop<S>(a, ii, (zs * a.ny + ys) * a.nx + xs, reader_shift<S>(a, z * (int)P + (int)pxy));
            fr = v.x;
            fb = v.y;
        }
        // the node's moments from the lanes' populations, in every lane
        float2 all[27];
#pragma unroll
        for (int k = 0; k < 27; ++k)
            all[k] = make_float2(__shfl_sync(0xffffffffu, fr, k), __shfl_sync(0xffffffffu, fb, k));
        const float lam = outflow_lambda(a, moments_of(a, [&](int k) { return all[k]; }));
        const float inv = 1.0f / (1.0f + lam);
        if (mine) {
            const long long hr = (long long)i * P + pxy, hb = (long long)(27 + i) * P + pxy;
            a.hist_out[hr] = outflow_blend(__ldg(a.hist_in + hr), fr, lam, inv);
            a.hist_out[hb] = outflow_blend(__ldg(a.hist_in + hb), fb, lam, inv);
            if (a.fm_out) {
                a.fm_out[hr] = fr;
                a.fm_out[hb] = fb;
            }
        }
    }
}

// boundary_column_kernel: one thread per (x, y) column, looping over the directions, so that
// the loads and stores of a warp are consecutive columns of one direction's plane; on large
// planes it takes half the time of the warp-per-column kernel (measured on the 256 x 256
// plane: 0.023 against 0.050 ms), on small ones it has too few threads.
constexpr long long kColumnKernelPlane = 24576;
template <int S>
__global__ void __launch_bounds__(128) boundary_column_kernel(StepArgs a) {
    chain_begin();
    const long long col = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= a.plane) return;
    const int x = (int)(col % a.nx), y = (int)(col / a.nx);
    const long long P = a.plane, pxy = col;
    const int N = a.nz - 1;
    // source column x - c_x, y - c_y of a pull for c = -1, 0, +1, reflected onto the node's own
    // column at a free-slip side wall (where the direction leaving the source has that
    // component reversed: rx / ry)
    int xs3[3], ys3[3];
    bool rx3[3], ry3[3];
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
        int xs = x - d, ys = y - d;
        bool rx = false, ry = false;
        if (xs < 0 || xs >= a.nx) {
            if (a.wall_x) { xs = x; rx = true; } else xs = wrapi(xs, a.nx);
        }
        if (ys < 0 || ys >= a.ny) {
            if (a.wall_y) { ys = y; ry = true; } else ys = wrapi(ys, a.ny);
        }
        xs3[d + 1] = xs; ys3[d + 1] = ys; rx3[d + 1] = rx; ry3[d + 1] = ry;
    }

    if (a.bc_zlo == BC_INLET || a.bc_zlo == BC_FREESLIP) {
        const Own own = reader_shift<S>(a, (int)pxy);
#pragma unroll
        for (int i = 1; i < 27; ++i) {
            if (cz(i) != 1) continue;
            const int xs = xs3[cx(i) + 1], ys = ys3[cy(i) + 1];
            const int cxs = rx3[cx(i) + 1] ? -cx(i) : cx(i), cys = ry3[cy(i) + 1] ? -cy(i) : cy(i);
            float vr, vb;
            if (a.bc_zlo == BC_INLET && a.disc[(long long)ys * a.nx + xs]) {
                vr = inlet_population_at(a, i, cxs, cys, xs, ys);
                vb = 0.0f;
            } else {  // half-way specular reflection at z = -1/2
                const float2 v = load_pop<S>(a, mirror_z(i), ys * a.nx + xs, own, mirror_z(dir_of(cxs, cys, 1)));
                vr = v.x;
                vb = v.y;
            }
            a.zin[(long long)zrank(i) * P + pxy] = vr;
            a.zin[(long long)(9 + zrank(i)) * P + pxy] = vb;
        }
    }
    if (a.bc_zhi == BC_FREESLIP) {
        const Own own = reader_shift<S>(a, N * (int)P + (int)pxy);
#pragma unroll
        for (int i = 1; i < 27; ++i) {
            if (cz(i) != -1) continue;
            const int xs = xs3[cx(i) + 1], ys = ys3[cy(i) + 1];
            const int cxs = rx3[cx(i) + 1] ? -cx(i) : cx(i), cys = ry3[cy(i) + 1] ? -cy(i) : cy(i);
            const float2 v = load_pop<S>(a, mirror_z(i), (N * a.ny + ys) * a.nx + xs, own, mirror_z(dir_of(cxs, cys, -1)));
            a.zout[(long long)zrank(i) * P + pxy] = v.x;
            a.zout[(long long)(9 + zrank(i)) * P + pxy] = v.y;
        }
    }
    if (a.bc_zhi == BC_CONVECTIVE) {
        // post-stream populations of node (x, y, N-1) at t+1 (N-1 >= 1: plain pulls)
        const int z = N - 1;
        const Own own = reader_shift<S>(a, z * (int)P + (int)pxy);
        float2 f[27];
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            const int xs = xs3[cx(i) + 1], ys = ys3[cy(i) + 1];
            const int cxs = rx3[cx(i) + 1] ? -cx(i) : cx(i), cys = ry3[cy(i) + 1] ? -cy(i) : cy(i);
            f[i] = load_pop<S>(a, i, ((z - cz(i)) * a.ny + ys) * a.nx + xs, own, dir_of(cxs, cys, cz(i)));
        }
        const float lam = outflow_lambda(a, moments_of(a, [&](int i) { return f[i]; }));
        const float inv = 1.0f / (1.0f + lam);
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            const long long hr = (long long)i * P + pxy, hb = (long long)(27 + i) * P + pxy;
            a.hist_out[hr] = outflow_blend(__ldg(a.hist_in + hr), f[i].x, lam, inv);
            a.hist_out[hb] = outflow_blend(__ldg(a.hist_in + hb), f[i].y, lam, inv);
            if (a.fm_out) {
                a.fm_out[hr] = f[i].x;
                a.fm_out[hb] = f[i].y;
            }
        }
    }
}

// The boundary planes of a step, with the kernel that suits the plane size.
template <int S>
static void launch_boundary(const StepArgs &a, cudaStream_t s) {
    if (a.plane >= kColumnKernelPlane)
        launch_chained(boundary_column_kernel<S>, dim3((unsigned)((a.plane + 127) / 128)), dim3(128), 0, s, a);
    else
        launch_chained(boundary_plane_kernel<S>, dim3((unsigned)((a.plane + 3) / 4)), dim3(128), 0, s, a);
}

// ------------------------------------------- moment pass (K_A with the paper's rates)
// With s3 = s4 = s5 = s6 = 1 the collision needs only a node's colour densities, mass,
// momentum and raw second moment (see the header), so the one pull gather of a step happens
// here: the node's phase entry (as phase_field_kernel writes it) plus its 12 collision
// moments go to a.mom, and collide_kernel reads those instead of gathering again.
template <int S, bool W, bool kKeep>
__device__ __forceinline__ void moment_at(const StepArgs &a, int x, int y, int z, unsigned long long pol) {
    const Nbr nb(a, x, y, z);
    float fr[27], fb[27];
    if (z == 0 || z == a.nz - 1)
        gather<S, W, true>(a, nb, z, fr, fb);
    else
        gather<S, W, false>(a, nb, z, fr, fb);
    const Moments mo = moments_of(a, [&](int i) { return make_float2(fr[i], fb[i]); });
    if constexpr (S == STORE_FP32)
        a.phase[nb.n] = phase_entry(mo);
    else if constexpr (S == STORE_FP16)
        a.ph_cur[nb.n] = phase_entry_fp16(mo);
    else
        a.ph_cur[nb.n] = pack_fit_entry(mo.phi, mo.rho_r + mo.rho_b, fit_even(a, mo.rho_r, mo.rho_b, mo.phi),
                                        fit_odd_fp8(a, fr, fb));
    if constexpr (kKeep)
        store_moments_keep(a.mom, (size_t)a.NN, nb.n, mo, pol);
    else
        store_moments(a.mom, (size_t)a.NN, nb.n, mo);
}

template <int S, bool W>
__device__ __forceinline__ void moment_node(const StepArgs &a) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z + a.z_base;
    if (x >= a.nx || y >= a.ny) return;
    moment_at<S, W, false>(a, x, y, z, 0ull);
}

template <int S, bool W>
__global__ void __launch_bounds__(128) moment_kernel(StepArgs a) {
    chain_begin();
    moment_node<S, W>(a);
}
template <int S>
__global__ void __launch_bounds__(128, S == STORE_FP16_FIT ? 5 : 1) moment_wall_kernel(StepArgs a) {
    chain_begin();
    moment_node<S, true>(a);
}

// -------- collide, perturb, recolour (K_B) with the paper's rates s3 = s4 = s5 = s6 = 1
// Reads the node's moments from the moment pass (no population gather), takes the
// gradients from the 26 neighbours' phase entries and writes the 54 populations.
// kRec (FP32, adjoint recompute): also writes the node's gradients to a.grad4 / a.grad2 (its
// moments are already in a.mom).
// Blocks per SM (register bound): FP32 6, FP16 5, FP16_FIT 4 (its encoding needs the most
// registers).

// (phi, rho) of the neighbour x + c_j.  Ghosts: z = -1 is phi = 1, rho = rho_r0 inside the inlet
// disc and the mirror of z = 0 elsewhere; z = N + 1 mirrors z = N (the neighbour offsets are clamped
// onto the wall planes).  kEdge = false: the caller knows that z > 0.
template <int S, bool kEdge>
__device__ __forceinline__ float2 neighbour_phase(const StepArgs &a, const Nbr &nb, int z, int j) {
    float2 v;
    if constexpr (S == STORE_FP32) {
        v = __ldg(a.phase + nb.nbr(j));
    } else {
        const float4 e = __ldg(a.ph_cur + nb.nbr(j));
        v = make_float2(e.x, S == STORE_FP16 ? e.y : fit_entry_rho(e));
    }
    if (kEdge && cz(j) == -1 && z == 0 && a.bc_zlo == BC_INLET) {
        if (a.disc[nb.yo[1 - cy(j)] + nb.xo[1 - cx(j)]]) v = make_float2(1.0f, a.rho_r0);
    }
    return v;
}

template <bool kForce, int S, bool kRec, bool kOnce>
__device__ __forceinline__ void collide_at(const StepArgs &a, int x, int y, int z) {
    const Nbr nb(a, x, y, z);
    const Moments mo = kOnce ? load_moments_once(a.mom, (size_t)a.NN, nb.n) : load_moments(a.mom, (size_t)a.NN, nb.n);
    float2 gx, gy, gz;  // (grad phi, grad rho)
    if (z == 0)
        gradients([&](int j) { return neighbour_phase<S, true>(a, nb, z, j); }, gx, gy, gz);
    else
        gradients([&](int j) { return neighbour_phase<S, false>(a, nb, z, j); }, gx, gy, gz);
    if constexpr (kRec) {
        a.grad4[nb.n] = make_float4(gx.x, gy.x, gz.x, gx.y);
        a.grad2[nb.n] = make_float2(gy.y, gz.y);
    }
    collide_node<kForce>(a, mo, gx, gy, gz, [&](int i, float2 f) {
        return store_pop<S>(a, i, nb.n, f, S == STORE_FP32 || i == 0 ? no_shift() : dest_shift<S>(a, nb, i));
    }, [] {});
}

template <bool kForce, int S, bool kRec>
__global__ void __launch_bounds__(128, (S == STORE_FP32 ? 6 : (S == STORE_FP16 ? 5 : 4))) collide_kernel(StepArgs a) {
    chain_begin();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z + a.z_base;
    if (x >= a.nx || y >= a.ny) return;
    collide_at<kForce, S, kRec, false>(a, x, y, z);
}

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
// level with them on smaller ones, and the two launches stay the default.
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
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

// The fused kernel's wait on a plane that no gather completes (f.target beyond reach): one
// thread gives up after the wait's limit, sets f.err and records the time it waited in *ns.
__global__ void fused_wait_probe_kernel(FusedCtl f, unsigned long long *ns) {
    if (threadIdx.x != 0) return;
    const unsigned long long t0 = global_ns();
    wait_planes(f, 0, 0, 0);
    *ns = global_ns() - t0;
}

cudaError_t launch_fused_wait_probe(const FusedCtl &f, unsigned long long *ns, cudaStream_t s) {
    fused_wait_probe_kernel<<<1, 32, 0, s>>>(f, ns);
    return cudaGetLastError();
}

template <bool kForce, int S, bool W>
__global__ void __launch_bounds__(128, (S == STORE_FP32 ? 6 : (S == STORE_FP16 ? 5 : 4))) step_kernel(StepArgs a, FusedCtl f) {
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
                if (x < a.nx && y < a.ny) moment_at<S, W, true>(a, x, y, z, pol);
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
                if (in) collide_at<kForce, S, false, true>(a, x, y, z);
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

// ------------------------------------------------------------------------ launchers
template <int S, bool W>
static void launch_step_sw(const StepArgs &a, cudaStream_t s, cudaEvent_t *ev, long long *launches, int passes) {
    const bool paper_rates = a.s3 == 1.0f && a.s4 == 1.0f && a.s5 == 1.0f && a.s6 == 1.0f;
    const bool force = a.gx != 0.0f || a.gy != 0.0f || a.gz != 0.0f;
    dim3 blk(32, 4, 1), grd((a.nx + 31) / 32, (a.ny + 3) / 4, a.nz);
    if (passes & PASS_GATHER) {
        if (ev) cudaEventRecord(ev[0], s);
        if (a.bc_zlo != BC_PERIODIC || a.bc_zhi != BC_PERIODIC) {
            launch_boundary<S>(a, s);
            *launches += 1;
        }
        if (ev) cudaEventRecord(ev[1], s);
        // pass 1: the step's pull gather (phase field, and the collision moments when the
        // paper's rates let the collision work from them)
        if (paper_rates) {
            if constexpr (W && S != STORE_FP32)
                launch_chained(moment_wall_kernel<S>, grd, blk, 0, s, a);
            else
                launch_chained(moment_kernel<S, W>, grd, blk, 0, s, a);
        } else {
            launch_general_gather(a, S, s);
        }
        if (ev) cudaEventRecord(ev[2], s);
        *launches += 1;
    }
    if (!(passes & PASS_COLLIDE)) return;
    // pass 2: the collision, writing S(t+1)
    if (ev && !(passes & PASS_GATHER)) cudaEventRecord(ev[2], s);
    const bool rec = S == STORE_FP32 && a.grad4 != nullptr;  // paper rates only (adjoint)
    if (!paper_rates)
        launch_general_collide(a, S, s);
    else if (rec && force)
        launch_chained(collide_kernel<true, S, S == STORE_FP32>, grd, blk, 0, s, a);
    else if (rec)
        launch_chained(collide_kernel<false, S, S == STORE_FP32>, grd, blk, 0, s, a);
    else if (force)
        launch_chained(collide_kernel<true, S, false>, grd, blk, 0, s, a);
    else
        launch_chained(collide_kernel<false, S, false>, grd, blk, 0, s, a);
    if (ev) cudaEventRecord(ev[3], s);
    *launches += 1;
}

template <bool kForce, int S, bool W>
static cudaError_t launch_fused_sw(const StepArgs &a, const FusedCtl &f, int grid, cudaStream_t s) {
    void *args[] = {(void *)&a, (void *)&f};
    return cudaLaunchCooperativeKernel((const void *)step_kernel<kForce, S, W>, dim3(grid), dim3(32, 4, 1), args, 0, s);
}

template <int S>
static cudaError_t fused_sw(const StepArgs &a, const FusedCtl &f, int grid, cudaStream_t s, int *occ) {
    const bool force = a.gx != 0.0f || a.gy != 0.0f || a.gz != 0.0f;
    const bool walls = a.wall_x || a.wall_y;
    const void *fn = force ? (walls ? (const void *)step_kernel<true, S, true> : (const void *)step_kernel<true, S, false>)
                           : (walls ? (const void *)step_kernel<false, S, true> : (const void *)step_kernel<false, S, false>);
    if (occ) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, fn, 128, 0);
    if (force)
        return walls ? launch_fused_sw<true, S, true>(a, f, grid, s) : launch_fused_sw<true, S, false>(a, f, grid, s);
    return walls ? launch_fused_sw<false, S, true>(a, f, grid, s) : launch_fused_sw<false, S, false>(a, f, grid, s);
}

cudaError_t fused_occupancy(const StepArgs &a, int storage, int *blocks_per_sm) {
    if (storage == STORE_FP16) return fused_sw<STORE_FP16>(a, FusedCtl{}, 0, nullptr, blocks_per_sm);
    if (storage == STORE_FP16_FIT) return fused_sw<STORE_FP16_FIT>(a, FusedCtl{}, 0, nullptr, blocks_per_sm);
    return fused_sw<STORE_FP32>(a, FusedCtl{}, 0, nullptr, blocks_per_sm);
}

cudaError_t launch_fused_step(const StepArgs &a, int storage, const FusedCtl &f, int grid, cudaStream_t s,
                              cudaEvent_t *ev, long long *launches) {
    if (ev) cudaEventRecord(ev[0], s);
    if (a.bc_zlo != BC_PERIODIC || a.bc_zhi != BC_PERIODIC) {
        if (storage == STORE_FP16)
            launch_boundary<STORE_FP16>(a, s);
        else if (storage == STORE_FP16_FIT)
            launch_boundary<STORE_FP16_FIT>(a, s);
        else
            launch_boundary<STORE_FP32>(a, s);
        *launches += 1;
    }
    if (ev) cudaEventRecord(ev[1], s);
    cudaError_t e;
    if (storage == STORE_FP16)
        e = fused_sw<STORE_FP16>(a, f, grid, s, nullptr);
    else if (storage == STORE_FP16_FIT)
        e = fused_sw<STORE_FP16_FIT>(a, f, grid, s, nullptr);
    else
        e = fused_sw<STORE_FP32>(a, f, grid, s, nullptr);
    if (e != cudaSuccess) return e;
    *launches += 1;
    if (ev) {
        cudaEventRecord(ev[2], s);
        cudaEventRecord(ev[3], s);
    }
    return cudaGetLastError();
}

template <int S>
static void launch_step_s(const StepArgs &a, cudaStream_t s, cudaEvent_t *ev, long long *launches, int passes) {
    if (a.wall_x || a.wall_y)
        launch_step_sw<S, true>(a, s, ev, launches, passes);
    else
        launch_step_sw<S, false>(a, s, ev, launches, passes);
}

cudaError_t launch_step(const StepArgs &a, int storage, cudaStream_t s, cudaEvent_t *ev, long long *launches,
                        int passes) {
    if (storage == STORE_FP16)
        launch_step_s<STORE_FP16>(a, s, ev, launches, passes);
    else if (storage == STORE_FP16_FIT)
        launch_step_s<STORE_FP16_FIT>(a, s, ev, launches, passes);
    else
        launch_step_s<STORE_FP32>(a, s, ev, launches, passes);
    return cudaGetLastError();
}

}  // namespace lbcm
