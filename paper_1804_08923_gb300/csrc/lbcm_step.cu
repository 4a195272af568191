// lbcm_step.cu -- the per-time-step kernels of the colour-gradient central-moment LB
// method (arXiv:1804.08923), FP32 populations and arithmetic, sm_103a.
//
// One step (state S(t) -> S(t+1)) is three launches on the context's stream:
//   1. boundary_plane_kernel  incoming z = 0 populations (inlet disc / free-slip mirror),
//                             free-slip top, and the convective outflow plane
//                             f(N, t+1) = [f(N, t) + lambda f(N-1, t+1)] / (1 + lambda)
//                             (Section IV.A).
//   2. moment_kernel          pull-gathers the 54 post-stream populations of a node (the
//                             step's only gather) and writes its order parameter phi
//                             (Eq. (23)) and total density rho (Section II, densities) for
//                             the gradient stencil, and the moments the collision needs
//                             (colour densities, phi, momentum, raw second moment).  One
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
#include "lbcm_fused.cuh"
#include "lbcm_internal.h"
#include "lbcm_node.cuh"

namespace lbcm {

// ------------------------------------------------------------------ boundary planes
//   z = 0 (inlet or free-slip bottom): the 9 incoming c_z = +1 populations -> zin
//   z = N free-slip top: the 9 incoming c_z = -1 populations -> zout
//   z = N convective: hist(t+1) from hist(t) and the post-stream f(N-1, t+1) (Section IV.A)
// Two kernels with the same results, bit for bit.
// boundary_plane_kernel: one warp per (x, y) column and plane (blockIdx.y = 0: z = 0, 1: z = N), lane
// i < 27 handles direction i.  Many warps with few instructions each: the faster of the two on planes of
// fewer than kColumnKernelPlane columns.
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

    if (blockIdx.y == 0 && (a.bc_zlo == BC_INLET || a.bc_zlo == BC_FREESLIP) && mine && czi == 1) {
        float vr, vb;
        if (a.bc_zlo == BC_INLET && a.disc[(long long)ys * a.nx + xs]) {
            vr = inlet_population_at(a, i, cxs, cys, xs, ys);
            vb = 0.0f;
        } else {  // half-way specular reflection at z = -1/2
            const float2 v = load_pop<STORE_FP32>(a, mirror_z(ii), ys * a.nx + xs, no_shift());
            vr = v.x;
            vb = v.y;
        }
        a.zin[(long long)zrank(i) * P + pxy] = vr;
        a.zin[(long long)(9 + zrank(i)) * P + pxy] = vb;
    }
    if (blockIdx.y == 1 && a.bc_zhi == BC_FREESLIP && mine && czi == -1) {
        const float2 v = load_pop<STORE_FP32>(a, mirror_z(ii), (N * a.ny + ys) * a.nx + xs,
                                     no_shift());
        a.zout[(long long)zrank(i) * P + pxy] = v.x;
        a.zout[(long long)(9 + zrank(i)) * P + pxy] = v.y;
    }
    if (blockIdx.y == 1 && a.bc_zhi == BC_CONVECTIVE) {
        // post-stream populations of node (x, y, N-1) at t+1 (N-1 >= 1: plain pulls)
        const int z = N - 1;
        float fr = 0.0f, fb = 0.0f, hist_r = 0.0f, hist_b = 0.0f;
        const long long hr = (long long)i * P + pxy, hb = (long long)(27 + i) * P + pxy;
        if (mine) {
            hist_r = __ldg(a.hist_in + hr);
            hist_b = __ldg(a.hist_in + hb);
            const int zs = z - czi;
            const float2 v = load_pop<STORE_FP32>(a, ii, (zs * a.ny + ys) * a.nx + xs, no_shift());
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
            a.hist_out[hr] = outflow_blend(hist_r, fr, lam, inv);
            a.hist_out[hb] = outflow_blend(hist_b, fb, lam, inv);
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
        const Own own = no_shift();
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
                const float2 v = load_pop<STORE_FP32>(a, mirror_z(i), ys * a.nx + xs, own, mirror_z(dir_of(cxs, cys, 1)));
                vr = v.x;
                vb = v.y;
            }
            a.zin[(long long)zrank(i) * P + pxy] = vr;
            a.zin[(long long)(9 + zrank(i)) * P + pxy] = vb;
        }
    }
    if (a.bc_zhi == BC_FREESLIP) {
        const Own own = no_shift();
#pragma unroll
        for (int i = 1; i < 27; ++i) {
            if (cz(i) != -1) continue;
            const int xs = xs3[cx(i) + 1], ys = ys3[cy(i) + 1];
            const int cxs = rx3[cx(i) + 1] ? -cx(i) : cx(i), cys = ry3[cy(i) + 1] ? -cy(i) : cy(i);
            const float2 v = load_pop<STORE_FP32>(a, mirror_z(i), (N * a.ny + ys) * a.nx + xs, own, mirror_z(dir_of(cxs, cys, -1)));
            a.zout[(long long)zrank(i) * P + pxy] = v.x;
            a.zout[(long long)(9 + zrank(i)) * P + pxy] = v.y;
        }
    }
    if (a.bc_zhi == BC_CONVECTIVE) {
        // post-stream populations of node (x, y, N-1) at t+1 (N-1 >= 1: plain pulls)
        const int z = N - 1;
        const Own own = no_shift();
        float2 f[27];
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            const int xs = xs3[cx(i) + 1], ys = ys3[cy(i) + 1];
            const int cxs = rx3[cx(i) + 1] ? -cx(i) : cx(i), cys = ry3[cy(i) + 1] ? -cy(i) : cy(i);
            f[i] = load_pop<STORE_FP32>(a, i, ((z - cz(i)) * a.ny + ys) * a.nx + xs, own, dir_of(cxs, cys, cz(i)));
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
static void launch_boundary(const StepArgs &a, cudaStream_t s) {
    if (a.plane >= kColumnKernelPlane)
        launch_chained(boundary_column_kernel, dim3((unsigned)((a.plane + 127) / 128)), dim3(128), 0, s, a);
    else
        launch_chained(boundary_plane_kernel, dim3((unsigned)((a.plane + 3) / 4), 2), dim3(128), 0, s, a);
}

// ------------------------------------------- moment pass (K_A with the paper's rates)
// With s3 = s4 = s5 = s6 = 1 the collision needs only a node's colour densities, mass,
// momentum and raw second moment (see the header), so the one pull gather of a step happens
// here: the node's phase entry (as phase_field_kernel writes it) plus its 12 collision
// moments go to a.mom, and collide_kernel reads those instead of gathering again.
template <bool W, bool kKeep>
__device__ __forceinline__ void moment_at(const StepArgs &a, int x, int y, int z, unsigned long long pol) {
    const Nbr nb(a, x, y, z);
    float fr[27], fb[27];
    if (z == 0 || z == a.nz - 1)
        gather<STORE_FP32, W, true>(a, nb, z, fr, fb);
    else
        gather<STORE_FP32, W, false>(a, nb, z, fr, fb);
    const Moments mo = moments_of(a, [&](int i) { return make_float2(fr[i], fb[i]); });
    a.phase[nb.n] = phase_entry(mo);
    if constexpr (kKeep)
        store_moments_keep(a.mom, (size_t)a.NN, nb.n, mo, pol);
    else
        store_moments(a.mom, (size_t)a.NN, nb.n, mo);
}

template <bool W>
__device__ __forceinline__ void moment_node(const StepArgs &a) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z + a.z_base;
    if (x >= a.nx || y >= a.ny) return;
    moment_at<W, false>(a, x, y, z, 0ull);
}

template <bool W>
__global__ void __launch_bounds__(128) moment_kernel(StepArgs a) {
    chain_begin();
    moment_node<W>(a);
}

// -------- collide, perturb, recolour (K_B) with the paper's rates s3 = s4 = s5 = s6 = 1
// Reads the node's moments from the moment pass (no population gather), takes the
// gradients from the 26 neighbours' phase entries and writes the 54 populations.
// kRec (FP32, adjoint recompute): also writes the node's gradients to a.grad4 / a.grad2 (its
// moments are already in a.mom).
// Blocks per SM (register bound): 6.

// (phi, rho) of the neighbour x + c_j.  Ghosts: z = -1 is phi = 1, rho = rho_r0 inside the inlet
// disc and the mirror of z = 0 elsewhere; z = N + 1 mirrors z = N (the neighbour offsets are clamped
// onto the wall planes).  kEdge = false: the caller knows that z > 0.
template <bool kEdge>
__device__ __forceinline__ float2 neighbour_phase(const StepArgs &a, const Nbr &nb, int z, int j) {
    float2 v = __ldg(a.phase + nb.nbr(j));
    if (kEdge && cz(j) == -1 && z == 0 && a.bc_zlo == BC_INLET) {
        if (a.disc[nb.yo[1 - cy(j)] + nb.xo[1 - cx(j)]]) v = make_float2(1.0f, a.rho_r0);
    }
    return v;
}

template <bool kForce, bool kRec, bool kOnce>
__device__ __forceinline__ void collide_at(const StepArgs &a, int x, int y, int z) {
    const Nbr nb(a, x, y, z);
    const Moments mo = kOnce ? load_moments_once(a.mom, (size_t)a.NN, nb.n) : load_moments(a.mom, (size_t)a.NN, nb.n);
    float2 gx, gy, gz;  // (grad phi, grad rho)
    if (z == 0)
        gradients([&](int j) { return neighbour_phase<true>(a, nb, z, j); }, gx, gy, gz);
    else
        gradients([&](int j) { return neighbour_phase<false>(a, nb, z, j); }, gx, gy, gz);
    if constexpr (kRec) {
        a.grad4[nb.n] = make_float4(gx.x, gy.x, gz.x, gx.y);
        a.grad2[nb.n] = make_float2(gy.y, gz.y);
    }
    collide_node<kForce>(a, mo, gx, gy, gz, [&](int i, float2 f) {
        return store_pop<STORE_FP32>(a, i, nb.n, f, no_shift());
    }, [] {});
}

template <bool kForce, bool kRec>
__global__ void __launch_bounds__(128, 6) collide_kernel(StepArgs a) {
    chain_begin();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z + a.z_base;
    if (x >= a.nx || y >= a.ny) return;
    collide_at<kForce, kRec, false>(a, x, y, z);
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

// ------------------------------------------------------------------------ launchers
struct FusedFp32 {
    static constexpr int kBlocks = 6;
    template <bool W>
    static __device__ __forceinline__ void moments(const StepArgs &a, int x, int y, int z, unsigned long long pol) {
        moment_at<W, true>(a, x, y, z, pol);
    }
    template <bool kForce>
    static __device__ __forceinline__ void collide(const StepArgs &a, int x, int y, int z) {
        collide_at<kForce, false, true>(a, x, y, z);
    }
};

cudaError_t fused_occupancy(const StepArgs &a, int storage, int *blocks_per_sm) {
    return storage == STORE_FP32 ? fused_run<FusedFp32>(a, FusedCtl{}, 0, nullptr, blocks_per_sm)
                                 : half_fused(a, storage, FusedCtl{}, 0, nullptr, blocks_per_sm);
}

cudaError_t launch_fused_step(const StepArgs &a, int storage, const FusedCtl &f, int grid, cudaStream_t s,
                              cudaEvent_t *ev, long long *launches) {
    if (ev) cudaEventRecord(ev[0], s);
    if (a.bc_zlo != BC_PERIODIC || a.bc_zhi != BC_PERIODIC) {
        if (storage == STORE_FP32)
            launch_boundary(a, s);
        else
            launch_half_boundary(a, storage, s);
        *launches += 1;
    }
    if (ev) cudaEventRecord(ev[1], s);
    const cudaError_t e = storage == STORE_FP32 ? fused_run<FusedFp32>(a, f, grid, s, nullptr)
                                                : half_fused(a, storage, f, grid, s, nullptr);
    if (e != cudaSuccess) return e;
    *launches += 1;
    if (ev) {
        cudaEventRecord(ev[2], s);
        cudaEventRecord(ev[3], s);
    }
    return cudaGetLastError();
}

static void launch_fp32_step(const StepArgs &a, cudaStream_t s, cudaEvent_t *ev, long long *launches, int passes) {
    const bool paper_rates = a.s3 == 1.0f && a.s4 == 1.0f && a.s5 == 1.0f && a.s6 == 1.0f;
    const bool force = a.gx != 0.0f || a.gy != 0.0f || a.gz != 0.0f;
    const dim3 blk(32, 4, 1), grd((a.nx + 31) / 32, (a.ny + 3) / 4, a.nz);
    if (passes & PASS_GATHER) {
        if (ev) cudaEventRecord(ev[0], s);
        if (a.bc_zlo != BC_PERIODIC || a.bc_zhi != BC_PERIODIC) {
            launch_boundary(a, s);
            *launches += 1;
        }
        if (ev) cudaEventRecord(ev[1], s);
        // pass 1: the step's pull gather (phase field, and the collision moments when the
        // paper's rates let the collision work from them)
        if (!paper_rates)
            launch_general_gather(a, STORE_FP32, s);
        else if (a.wall_x || a.wall_y)
            launch_chained(moment_kernel<true>, grd, blk, 0, s, a);
        else
            launch_chained(moment_kernel<false>, grd, blk, 0, s, a);
        if (ev) cudaEventRecord(ev[2], s);
        *launches += 1;
    }
    if (!(passes & PASS_COLLIDE)) return;
    // pass 2: the collision, writing S(t+1)
    if (ev && !(passes & PASS_GATHER)) cudaEventRecord(ev[2], s);
    const bool rec = a.grad4 != nullptr;  // paper rates only (adjoint)
    if (!paper_rates)
        launch_general_collide(a, STORE_FP32, s);
    else if (rec && force)
        launch_chained(collide_kernel<true, true>, grd, blk, 0, s, a);
    else if (rec)
        launch_chained(collide_kernel<false, true>, grd, blk, 0, s, a);
    else if (force)
        launch_chained(collide_kernel<true, false>, grd, blk, 0, s, a);
    else
        launch_chained(collide_kernel<false, false>, grd, blk, 0, s, a);
    if (ev) cudaEventRecord(ev[3], s);
    *launches += 1;
}

cudaError_t launch_step(const StepArgs &a, int storage, cudaStream_t s, cudaEvent_t *ev, long long *launches,
                        int passes) {
    if (storage == STORE_FP32)
        launch_fp32_step(a, s, ev, launches, passes);
    else
        launch_half_step(a, storage, s, ev, launches, passes);
    return cudaGetLastError();
}

}  // namespace lbcm
