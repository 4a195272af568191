// lbcm_half.cu -- the step with half-precision population storage and the paper's rates
// (arXiv:1804.08923): the same three launches as with FP32 storage (lbcm_step.cu).
//
// The arithmetic is its own: sums over opposite pairs, the inverse transform evaluated direction by
// direction, contraction left to the compiler.  A population rounded to half precision falls on one
// side or the other by the last bit of its FP32 value, so another order of the same sums gives
// another run: populations of a 40 x 40 x 120 melt jet differ by 1e-4 (FP16) and 2e-5 (FP16_FIT) in
// the 2-norm after 50 steps, where FP32 ones differ by 3e-7.  So these storages take neither the
// collision of lbcm_collide.cuh nor the advance (which, built for FP16, gave 241 us a step on the
// 96 x 96 x 384 jet against 258 for the two passes).
#include "lbcm_device.cuh"
#include "lbcm_fused.cuh"
#include "lbcm_internal.h"
#include "lbcm_node.cuh"
#include "lbcm_pairs.cuh"

namespace lbcm {
namespace half_storage {

// ------------------------------------------------------------------ boundary planes
//   z = 0 (inlet or free-slip bottom): the 9 incoming c_z = +1 populations -> zin
//   z = N free-slip top: the 9 incoming c_z = -1 populations -> zout
//   z = N convective: hist(t+1) from hist(t) and the post-stream f(N-1, t+1) (Section IV.A)
// Two kernels with the same results up to the order of the outflow velocity's sums.
// boundary_plane_kernel: one warp per (x, y) column, lane i < 27 handles direction i.  Many
// warps with few instructions each: the faster of the two on planes of fewer than
// kColumnKernelPlane columns.
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

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
            // red equilibrium f^e(rho_r0, u_in) with alpha_r and Phi = 0, no blue
            InletVel iv;
            inlet_velocity(a.u_in, a.noise_amp, a.fourier, a.xc, a.yc, a.seed, a.step, xs, ys, a.nx, a.ny, iv);
            const float cu = (float)cxs * iv.ux + (float)cys * iv.uy + (float)czi * iv.uz;
            const float usq = iv.ux * iv.ux + iv.uy * iv.uy + iv.uz * iv.uz;
            vr = a.rho_r0 * (varphi(i, a.alpha_r, a.oma_r) + wgt(i) * eq_poly(cu, usq));
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
        const float s_ = fr + fb;
        const float rho = warp_sum_f(s_), jz = warp_sum_f((float)czi * s_);
        const float Fz = (rho - a.rho_b0) * a.gz;
        float lam = (jz + 0.5f * Fz) / rho;  // u_z(x, y, N-1, t+1), Eq. (13)
        lam = fminf(fmaxf(lam, 0.0f), 1.0f);
        const float inv = 1.0f / (1.0f + lam);
        if (mine) {
            const long long hr = (long long)i * P + pxy, hb = (long long)(27 + i) * P + pxy;
            a.hist_out[hr] = (__ldg(a.hist_in + hr) + lam * fr) * inv;
            a.hist_out[hb] = (__ldg(a.hist_in + hb) + lam * fb) * inv;
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
                // red equilibrium f^e(rho_r0, u_in) with alpha_r and Phi = 0, no blue
                InletVel iv;
                inlet_velocity(a.u_in, a.noise_amp, a.fourier, a.xc, a.yc, a.seed, a.step, xs, ys, a.nx, a.ny, iv);
                const float cu = (float)cxs * iv.ux + (float)cys * iv.uy + iv.uz;
                const float usq = iv.ux * iv.ux + iv.uy * iv.uy + iv.uz * iv.uz;
                vr = a.rho_r0 * (varphi(i, a.alpha_r, a.oma_r) + wgt(i) * eq_poly(cu, usq));
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
        float fr[27], fb[27];
        float rho = 0.0f, jz = 0.0f;
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            const int xs = xs3[cx(i) + 1], ys = ys3[cy(i) + 1];
            const int cxs = rx3[cx(i) + 1] ? -cx(i) : cx(i), cys = ry3[cy(i) + 1] ? -cy(i) : cy(i);
            const float2 v = load_pop<S>(a, i, ((z - cz(i)) * a.ny + ys) * a.nx + xs, own, dir_of(cxs, cys, cz(i)));
            fr[i] = v.x;
            fb[i] = v.y;
        }
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            const float s_ = fr[i] + fb[i];
            rho += s_;
            if (cz(i) > 0) jz += s_; else if (cz(i) < 0) jz -= s_;
        }
        const float Fz = (rho - a.rho_b0) * a.gz;
        float lam = (jz + 0.5f * Fz) / rho;  // u_z(x, y, N-1, t+1), Eq. (13)
        lam = fminf(fmaxf(lam, 0.0f), 1.0f);
        const float inv = 1.0f / (1.0f + lam);
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            const long long hr = (long long)i * P + pxy, hb = (long long)(27 + i) * P + pxy;
            a.hist_out[hr] = (__ldg(a.hist_in + hr) + lam * fr[i]) * inv;
            a.hist_out[hb] = (__ldg(a.hist_in + hb) + lam * fb[i]) * inv;
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
    PairMoments mo;
    pair_moments_of(fr, fb, mo);
    const float rr = mo.rho_r, rb = mo.rho_b;
    const float ph = order_parameter(rr, rb, a.inv_rho_r0, a.inv_rho_b0);
    if constexpr (S == STORE_FP16) {
        a.ph_cur[nb.n] = make_float4(ph, rr + rb, rr, rb);
    } else {
        a.ph_cur[nb.n] = pack_fit_entry(ph, rr + rb, fit_even(a, rr, rb, ph), fit_odd_fp8(a, fr, fb));
    }
    if constexpr (kKeep)
        store_pair_moments_keep(a.mom, (size_t)a.NN, nb.n, mo, pol);
    else
        store_pair_moments(a.mom, (size_t)a.NN, nb.n, mo);
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

// Collision, perturbation and recolouring of one node from its moments and gradients;
// writes the 54 post-collision populations of node n.
template <bool kForce, int S>
__device__ __forceinline__ void collide_from_moments(const StepArgs &a, const Nbr &nb, const PairMoments &mo, float gpx,
                                                     float gpy, float gpz, float grx, float gry, float grz) {
    const int n = nb.n;
    const float rho_r = mo.rho_r, rho_b = mo.rho_b, sf = mo.sf, jx = mo.jx, jy = mo.jy, jz = mo.jz;
    const float pxx = mo.pxx, pyy = mo.pyy, pzz = mo.pzz, pxy = mo.pxy, pxz = mo.pxz, pyz = mo.pyz;
    // macroscopic quantities (Eqs. (13), (48), (23)) and mixture parameters
    const float rho = rho_r + rho_b;
    const float inv_rho = 1.0f / rho;
    float Fx = 0.0f, Fy = 0.0f, Fz = 0.0f;
    if (kForce) {
        const float fo = rho - a.rho_b0;
        Fx = fo * a.gx; Fy = fo * a.gy; Fz = fo * a.gz;
    }
    const float jFx = fmaf(0.5f, Fx, jx), jFy = fmaf(0.5f, Fy, jy), jFz = fmaf(0.5f, Fz, jz);
    const float ux = jFx * inv_rho, uy = jFy * inv_rho, uz = jFz * inv_rho;
    const float phi = order_parameter(rho_r, rho_b, a.inv_rho_r0, a.inv_rho_b0);
    const float hp = 0.5f * (1.0f + phi), hm = 0.5f * (1.0f - phi);
    const float oma = one_minus_alpha_bar(a.alpha_mix, rho_r, rho_b, inv_rho, hp, hm, a.oma_r, a.oma_b);
    const float alpha = 1.0f - oma;
    const float nu = 1.0f / (hp * a.inv_nu_r + hm * a.inv_nu_b);
    const float tau = 3.0f * nu + 0.5f;
    const float s2nu = 1.0f / tau;
    const float Acoef = 2.25f * a.sigma / tau;  // A = 9 sigma / (4 tau)
    const float usq = ux * ux + uy * uy + uz * uz;
    const float ugr = ux * grx + uy * gry + uz * grz;
    const float uF = ux * Fx + uy * Fy + uz * Fz;

    // moments of Delta = f - f^e + F'/2: mass, momentum, raw second moment
    const float M = sf - rho;
    const float dx = fmaf(-rho, ux, jFx), dy = fmaf(-rho, uy, jFy), dz = fmaf(-rho, uz, jFz);
    const float cs2r = rho * oma * (9.0f / 19.0f);
    float Dxx = pxx - (cs2r + rho * ux * ux + nu * (2.0f * ux * grx + ugr));
    float Dyy = pyy - (cs2r + rho * uy * uy + nu * (2.0f * uy * gry + ugr));
    float Dzz = pzz - (cs2r + rho * uz * uz + nu * (2.0f * uz * grz + ugr));
    float Dxy = pxy - (rho * ux * uy + nu * (ux * gry + uy * grx));
    float Dxz = pxz - (rho * ux * uz + nu * (ux * grz + uz * grx));
    float Dyz = pyz - (rho * uy * uz + nu * (uy * grz + uz * gry));
    if (kForce) {
        Dxx += ux * Fx; Dyy += uy * Fy; Dzz += uz * Fz;
        Dxy += 0.5f * (ux * Fy + uy * Fx); Dxz += 0.5f * (ux * Fz + uz * Fx); Dyz += 0.5f * (uy * Fz + uz * Fy);
    }
    // central moments of Delta, then (I - K') applied
    const float k000 = (1.0f - a.s0) * M;
    const float o1 = 1.0f - a.s1;
    const float k100 = o1 * fmaf(-ux, M, dx), k010 = o1 * fmaf(-uy, M, dy), k001 = o1 * fmaf(-uz, M, dz);
    const float o2 = 1.0f - s2nu;
    const float cxx = Dxx - 2.0f * ux * dx + ux * ux * M;
    const float cyy = Dyy - 2.0f * uy * dy + uy * uy * M;
    const float czz = Dzz - 2.0f * uz * dz + uz * uz * M;
    const float k110 = o2 * (Dxy - ux * dy - uy * dx + ux * uy * M);
    const float k101 = o2 * (Dxz - ux * dz - uz * dx + ux * uz * M);
    const float k011 = o2 * (Dyz - uy * dz - uz * dy + uy * uz * M);
    float k200, k020, k002;
    {
        const float t = (1.0f - a.s2b) * (cxx + cyy + czz);
        const float e1 = o2 * (cxx - cyy), e2 = o2 * (cxx - czz);
        const float third = 1.0f / 3.0f;
        k200 = (t + e1 + e2) * third;
        k020 = (t - 2.0f * e1 + e2) * third;
        k002 = (t + e1 - 2.0f * e2) * third;
    }

    // inverse transform of the ten surviving moments: z sweep, y sweep (x sweep per direction)
    const InvAxis Ax(ux), Ay(uy), Az(uz);
    // z sweep of the columns (p, q): values V_pq[cz]
    float V00[3], V10[3], V01[3], V20[3], V02[3], V11[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        V00[c] = fmaf(Az.g0[c], k000, fmaf(Az.g1[c], k001, g2c(c - 1) * k002));
        V10[c] = fmaf(Az.g0[c], k100, Az.g1[c] * k101);
        V01[c] = fmaf(Az.g0[c], k010, Az.g1[c] * k011);
        V20[c] = Az.g0[c] * k200;
        V02[c] = Az.g0[c] * k020;
        V11[c] = Az.g0[c] * k110;
    }
    // y sweep: W_p[cy][cz]
    float W0[3][3], W1[3][3], W2[3][3];
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            W0[b][c] = fmaf(Ay.g0[b], V00[c], fmaf(Ay.g1[b], V01[c], g2c(b - 1) * V02[c]));
            W1[b][c] = fmaf(Ay.g0[b], V10[c], Ay.g1[b] * V11[c]);
            W2[b][c] = Ay.g0[b] * V20[c];
        }

    // perturbation (Eq. (30), squared numerator, both colours) and recolouring
    const float g2 = gpx * gpx + gpy * gpy + gpz * gpz;
    const float inv_gm = 1.0f / sqrtf(g2 + a.eps2);  // 1/|grad phi|_eps
    const float pert = Acoef * inv_gm;
    const float frac_r = rho_r * inv_rho, frac_b = rho_b * inv_rho;
    const float seg0 = a.beta * rho_r * rho_b * inv_rho * inv_gm;
    // moving populations written (as read back), per colour, summed as MassAcc sums them
    float2 sum = make_float2(0.0f, 0.0f);
    // opposite pairs (i, i+1), c_{i+1} = -c_i: c.u, c.grad rho and c.grad phi change sign;
    // f^e splits into an even part (rest weight, quadratic terms, Phi) and an odd part
    // (linear and cubic terms), the perturbation is even and the recolouring flux odd.
#pragma unroll
    for (int i = 1; i < 27; i += 2) {
        const float cu = (float)cx(i) * ux + (float)cy(i) * uy + (float)cz(i) * uz;
        const float cgr = (float)cx(i) * grx + (float)cy(i) * gry + (float)cz(i) * grz;
        const float cgp = (float)cx(i) * gpx + (float)cy(i) * gpy + (float)cz(i) * gpz;
        const float h = 4.5f * cu;
        const float ev = fmaf(h, cu, -1.5f * usq);                  // 9/2 cu^2 - 3/2 u^2
        const float od = cu * fmaf(h, cu, fmaf(-4.5f, usq, 3.0f));  // 3 cu + 9/2 cu^3 - 9/2 cu u^2
        const float rw = rho * wgt(i);
        float even = fmaf(rw, ev, rho * varphi(i, alpha, oma));
        even = fmaf(phi_corr(i) * nu * cu, cgr, even);                // Phi_i
        even = fmaf(pert, wgt(i) * cgp * cgp - bcoef(i) * g2, even);  // perturbation
        float odd = rw * od;
        if (kForce) {
            const float cF = (float)cx(i) * Fx + (float)cy(i) * Fy + (float)cz(i) * Fz;
            even = fmaf(0.5f * wgt(i), fmaf(9.0f * cu, cF, -3.0f * uF), even);  // F'/2, even part
            odd = fmaf(1.5f * wgt(i), cF, odd);                                   // F'/2, odd part
        }
        const int X = cx(i) + 1, Y = cy(i) + 1, Z = cz(i) + 1;
        const float rp = fmaf(Ax.g0[X], W0[Y][Z], fmaf(Ax.g1[X], W1[Y][Z], g2c(cx(i)) * W2[Y][Z]));
        const float rm = fmaf(Ax.g0[2 - X], W0[2 - Y][2 - Z], fmaf(Ax.g1[2 - X], W1[2 - Y][2 - Z], g2c(cx(i)) * W2[2 - Y][2 - Z]));
        const float fsp = (even + odd) + rp, fsm = (even - odd) + rm;
        const float seg = seg0 * varphi(i, alpha, oma) * inv_cnorm(i) * cgp;
        const float2 dp_ = store_pop<S>(a, i, n, make_float2(fmaf(frac_r, fsp, seg), fmaf(frac_b, fsp, -seg)),
                                        dest_shift<S>(a, nb, i));
        const float2 dm_ = store_pop<S>(a, i + 1, n, make_float2(fmaf(frac_r, fsm, -seg), fmaf(frac_b, fsm, seg)),
                                        dest_shift<S>(a, nb, i + 1));
        sum.x += dp_.x + dm_.x;
        sum.y += dp_.y + dm_.y;
    }
    const float sum_r = sum.x, sum_b = sum.y;
    // Rest direction.  In exact arithmetic the step keeps each colour's mass at this node
    // (sum_i f_i^k* = rho_k), so the rest population is that mass minus the moving ones as
    // they will be read back; this equals Eqs. (33), (34) for i = 0 and keeps the FP32
    // rounding of the lattice constants and any storage rounding from drifting the colour
    // masses step after step (the pairwise sum above is MassAcc's association).
    store_pop<S>(a, 0, n, make_float2(rho_r - sum_r, rho_b - sum_b), no_shift());
}

// -------- collide, perturb, recolour (K_B) with the paper's rates s3 = s4 = s5 = s6 = 1
// Reads the node's moments from the moment pass (no population gather), takes the
// gradients from the 26 neighbours' phase entries and writes the 54 populations.
// Blocks per SM (register bound): FP16 5, FP16_FIT 4 (its encoding needs the most registers).
template <bool kForce, int S, bool kOnce>
__device__ __forceinline__ void collide_at(const StepArgs &a, int x, int y, int z) {
    const Nbr nb(a, x, y, z);
    const PairMoments mo = kOnce ? load_pair_moments_once(a.mom, (size_t)a.NN, nb.n) : load_pair_moments(a.mom, (size_t)a.NN, nb.n);
    float gpx, gpy, gpz, grx, gry, grz;
    if (z == 0)
        stencil_gradients<S, true>(a, nb, z, gpx, gpy, gpz, grx, gry, grz);
    else
        stencil_gradients<S, false>(a, nb, z, gpx, gpy, gpz, grx, gry, grz);
    collide_from_moments<kForce, S>(a, nb, mo, gpx, gpy, gpz, grx, gry, grz);
}

template <bool kForce, int S>
__global__ void __launch_bounds__(128, S == STORE_FP16 ? 5 : 4) collide_kernel(StepArgs a) {
    chain_begin();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z + a.z_base;
    if (x >= a.nx || y >= a.ny) return;
    collide_at<kForce, S, false>(a, x, y, z);
}

// ------------------------------------------------------------------------ launchers
template <int S>
struct FusedHalf {
    static constexpr int kBlocks = S == STORE_FP16 ? 5 : 4;
    template <bool W>
    static __device__ __forceinline__ void moments(const StepArgs &a, int x, int y, int z, unsigned long long pol) {
        moment_at<S, W, true>(a, x, y, z, pol);
    }
    template <bool kForce>
    static __device__ __forceinline__ void collide(const StepArgs &a, int x, int y, int z) {
        collide_at<kForce, S, true>(a, x, y, z);
    }
};

template <int S>
static void launch_step_s(const StepArgs &a, cudaStream_t s, cudaEvent_t *ev, long long *launches, int passes) {
    const bool paper_rates = a.s3 == 1.0f && a.s4 == 1.0f && a.s5 == 1.0f && a.s6 == 1.0f;
    const bool force = a.gx != 0.0f || a.gy != 0.0f || a.gz != 0.0f;
    const dim3 blk(32, 4, 1), grd((a.nx + 31) / 32, (a.ny + 3) / 4, a.nz);
    if (passes & PASS_GATHER) {
        if (ev) cudaEventRecord(ev[0], s);
        if (a.bc_zlo != BC_PERIODIC || a.bc_zhi != BC_PERIODIC) {
            launch_boundary<S>(a, s);
            *launches += 1;
        }
        if (ev) cudaEventRecord(ev[1], s);
        if (!paper_rates)
            launch_general_gather(a, S, s);
        else if (a.wall_x || a.wall_y)
            launch_chained(moment_wall_kernel<S>, grd, blk, 0, s, a);
        else
            launch_chained(moment_kernel<S, false>, grd, blk, 0, s, a);
        if (ev) cudaEventRecord(ev[2], s);
        *launches += 1;
    }
    if (!(passes & PASS_COLLIDE)) return;
    if (ev && !(passes & PASS_GATHER)) cudaEventRecord(ev[2], s);
    if (!paper_rates)
        launch_general_collide(a, S, s);
    else if (force)
        launch_chained(collide_kernel<true, S>, grd, blk, 0, s, a);
    else
        launch_chained(collide_kernel<false, S>, grd, blk, 0, s, a);
    if (ev) cudaEventRecord(ev[3], s);
    *launches += 1;
}

}  // namespace half_storage

void launch_half_step(const StepArgs &a, int storage, cudaStream_t s, cudaEvent_t *ev, long long *launches, int passes) {
    if (storage == STORE_FP16)
        half_storage::launch_step_s<STORE_FP16>(a, s, ev, launches, passes);
    else
        half_storage::launch_step_s<STORE_FP16_FIT>(a, s, ev, launches, passes);
}

void launch_half_boundary(const StepArgs &a, int storage, cudaStream_t s) {
    if (storage == STORE_FP16)
        half_storage::launch_boundary<STORE_FP16>(a, s);
    else
        half_storage::launch_boundary<STORE_FP16_FIT>(a, s);
}

cudaError_t half_fused(const StepArgs &a, int storage, const FusedCtl &f, int grid, cudaStream_t s, int *occ) {
    return storage == STORE_FP16 ? fused_run<half_storage::FusedHalf<STORE_FP16>>(a, f, grid, s, occ)
                                 : fused_run<half_storage::FusedHalf<STORE_FP16_FIT>>(a, f, grid, s, occ);
}

}  // namespace lbcm
