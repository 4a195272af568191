// lbcm_general.cu -- the step with relaxation rates other than the paper's s3 = s4 = s5 = s6 = 1
// (arXiv:1804.08923, Section II): phase_field_kernel gathers the populations for the phase
// entries alone, and collide_general_kernel gathers them again and relaxes all 27 central moments.
//
// The collision applies T^-1 K T through the tensor-product central moments
//   kappa_abc = sum_i f_i (c_ix - u_x)^a (c_iy - u_y)^b (c_iz - u_z)^c,  a, b, c in {0,1,2},
// computed by three 1-D shifted sweeps and undone by three reverse sweeps.  The 27 rows
// of the paper's moment set (Eq. (14)) are, order by order, invertible combinations
// of these; K holds one rate per order except order 2, where the trace relaxes with s_2b
// and the deviatoric part with s_2nu.  Relaxing kappa with those rates is therefore the
// same linear map as T^-1 K T (exact up to rounding).  The forcing is folded in:
//   f* = f^e + F'/2 + T^-1 (I - K) T (f - f^e + F'/2)
// which equals f - T^-1 K T (f - f^e) + T^-1 (I - K/2) T F' (Eqs. (11) and (28)).
#include "lbcm_device.cuh"
#include "lbcm_internal.h"
#include "lbcm_node.cuh"
#include "lbcm_pairs.cuh"

namespace lbcm {

// --------------------------------------------------------------- phase field (K_A)
template <int S, bool W>
__device__ __forceinline__ void phase_field_node(const StepArgs &a) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= a.nx || y >= a.ny) return;
    const Nbr nb(a, x, y, z);
    float fr[27], fb[27];
    gather<S, W>(a, nb, z, fr, fb);
    MassAcc mr, mb;
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        mr.add(i, fr[i]);
        mb.add(i, fb[i]);
    }
    const float rr = mr.total(), rb = mb.total();
    const float ph = order_parameter(rr, rb, a.inv_rho_r0, a.inv_rho_b0);
    if constexpr (S == STORE_FP32) {
        a.phase[nb.n] = make_float2(ph, rr + rb);
    } else if constexpr (S == STORE_FP16) {
        a.ph_cur[nb.n] = make_float4(ph, rr + rb, rr, rb);  // also the FP16 shift densities of S(t+1)
    } else {  // the prediction S(t+1) is encoded against
        a.ph_cur[nb.n] = pack_fit_entry(ph, rr + rb, fit_even(a, rr, rb, ph), fit_odd_fp8(a, fr, fb));
    }
}

// Lattices without side walls (and FP32 with them); and, with separate register bounds, the
// FP16 encodings on lattices with side walls.  Measured on the 240x240x1200 UT lattice: FP16
// 1.97 -> 1.80 ms with a one-block bound, FP16_FIT 3.12 -> 2.52 ms with five; FP32 went the
// other way (2.17 -> 2.69 ms) and keeps the plain bound.
template <int S, bool W>
__global__ void __launch_bounds__(128) phase_field_kernel(StepArgs a) {
    phase_field_node<S, W>(a);
}
template <int S>
__global__ void __launch_bounds__(128, S == STORE_FP16_FIT ? 5 : 1) phase_field_wall_kernel(StepArgs a) {
    phase_field_node<S, true>(a);
}

// 1-D shifted moment sweep: values at c = -1, 0, +1 -> central moments of order 0, 1, 2
// about u:  m0 = sum v, m1 = sum v (c - u), m2 = sum v (c - u)^2.
__device__ __forceinline__ void sweep_fwd(float &a0, float &a1, float &a2, float u) {
    const float r0 = a0 + a1 + a2, r1 = a2 - a0, r2 = a2 + a0;
    a0 = r0;
    a1 = fmaf(-u, r0, r1);
    a2 = fmaf(u, fmaf(u, r0, -2.0f * r1), r2);
}
// Inverse of sweep_fwd: raw moments r1 = m1 + u m0, r2 = m2 + 2u m1 + u^2 m0, then
// v0 = r0 - r2, v+ = (r2 + r1)/2, v- = (r2 - r1)/2.
__device__ __forceinline__ void sweep_inv(float &a0, float &a1, float &a2, float u) {
    const float r0 = a0;
    const float r1 = fmaf(u, a0, a1);
    const float r2 = fmaf(u, fmaf(u, a0, 2.0f * a1), a2);
    a1 = r0 - r2;
    a0 = 0.5f * (r2 - r1);
    a2 = 0.5f * (r2 + r1);
}

// ------------------------- collide, perturb, recolour (K_B), any relaxation rates
template <int S, bool W>
__global__ void __launch_bounds__(128) collide_general_kernel(StepArgs a) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= a.nx || y >= a.ny) return;
    const Nbr nb(a, x, y, z);

    // post-stream populations, colour-blind sum and densities (same order as K_A)
    float f[27];
    float rho_r, rho_b;
    {
        float fr[27], fb[27];
        gather<S, W>(a, nb, z, fr, fb);
        MassAcc mr, mb;
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            mr.add(i, fr[i]);
            mb.add(i, fb[i]);
            f[i] = fr[i] + fb[i];
        }
        rho_r = mr.total();
        rho_b = mb.total();
    }

    float gpx, gpy, gpz, grx, gry, grz;
    stencil_gradients<S>(a, nb, z, gpx, gpy, gpz, grx, gry, grz);

    // macroscopic velocity with the Guo half-force (Eq. (13)), body force Eq. (48)
    const float rho = rho_r + rho_b;
    const float inv_rho = 1.0f / rho;
    const float Fx = (rho - a.rho_b0) * a.gx, Fy = (rho - a.rho_b0) * a.gy, Fz = (rho - a.rho_b0) * a.gz;
    float jx = 0.0f, jy = 0.0f, jz = 0.0f;
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        if (cx(i) != 0) jx += (float)cx(i) * f[i];
        if (cy(i) != 0) jy += (float)cy(i) * f[i];
        if (cz(i) != 0) jz += (float)cz(i) * f[i];
    }
    const float ux = (jx + 0.5f * Fx) * inv_rho, uy = (jy + 0.5f * Fy) * inv_rho, uz = (jz + 0.5f * Fz) * inv_rho;

    // order parameter (Eq. (23)) and mixture parameters
    const float phi = order_parameter(rho_r, rho_b, a.inv_rho_r0, a.inv_rho_b0);
    const float hp = 0.5f * (1.0f + phi), hm = 0.5f * (1.0f - phi);
    const float one_m_alpha = one_minus_alpha_bar(a.alpha_mix, rho_r, rho_b, inv_rho, hp, hm, a.oma_r, a.oma_b);
    const float alpha = 1.0f - one_m_alpha;
    const float nu = 1.0f / (hp * a.inv_nu_r + hm * a.inv_nu_b);  // harmonic mean
    const float tau = 3.0f * nu + 0.5f;                           // Eq. (16): 1/s_2nu
    const float s2nu = 1.0f / tau;
    const float Acoef = 2.25f * a.sigma / tau;                     // Eq. (32): A = 9 sigma / (4 tau)

    const float usq = ux * ux + uy * uy + uz * uz;
    const float ugr = ux * grx + uy * gry + uz * grz;
    const float uF = ux * Fx + uy * Fy + uz * Fz;

    // Delta = f - f^e + F'/2, scattered into the tensor-product layout
    float m[27];
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        const float cu = (float)cx(i) * ux + (float)cy(i) * uy + (float)cz(i) * uz;
        const float cg = (float)cx(i) * grx + (float)cy(i) * gry + (float)cz(i) * grz;
        const float cF = (float)cx(i) * Fx + (float)cy(i) * Fy + (float)cz(i) * Fz;
        const float Phi = csq(i) == 0 ? -3.0f * nu * ugr : phi_corr(i) * nu * cu * cg;
        const float fe = rho * fmaf(wgt(i), eq_poly(cu, usq), varphi(i, alpha, one_m_alpha)) + Phi;
        const float Fp = wgt(i) * (3.0f * (cF - uF) + 9.0f * cu * cF);
        m[cell(i)] = f[i] - fe + 0.5f * Fp;
    }

    // forward central-moment transform: z, then y, then x sweeps
#pragma unroll
    for (int p = 0; p < 9; ++p) sweep_fwd(m[p * 3 + 0], m[p * 3 + 1], m[p * 3 + 2], uz);
#pragma unroll
    for (int a0 = 0; a0 < 3; ++a0)
#pragma unroll
        for (int c = 0; c < 3; ++c) sweep_fwd(m[a0 * 9 + 0 + c], m[a0 * 9 + 3 + c], m[a0 * 9 + 6 + c], uy);
#pragma unroll
    for (int q = 0; q < 9; ++q) sweep_fwd(m[q], m[9 + q], m[18 + q], ux);

    // relaxation: kappa <- (I - K') kappa, K' = K in the tensor-product basis
    {
#define KAP(p, q, r) m[(p) * 9 + (q) * 3 + (r)]
        const float o0 = 1.0f - a.s0, o1 = 1.0f - a.s1, o2 = 1.0f - s2nu, o2b = 1.0f - a.s2b;
        const float o3 = 1.0f - a.s3, o4 = 1.0f - a.s4, o5 = 1.0f - a.s5, o6 = 1.0f - a.s6;
        KAP(0, 0, 0) *= o0;
        KAP(1, 0, 0) *= o1; KAP(0, 1, 0) *= o1; KAP(0, 0, 1) *= o1;
        KAP(1, 1, 0) *= o2; KAP(1, 0, 1) *= o2; KAP(0, 1, 1) *= o2;
        {
            const float tr = KAP(2, 0, 0) + KAP(0, 2, 0) + KAP(0, 0, 2);
            const float d1 = KAP(2, 0, 0) - KAP(0, 2, 0), d2 = KAP(2, 0, 0) - KAP(0, 0, 2);
            const float t = o2b * tr, e1 = o2 * d1, e2 = o2 * d2;
            const float third = 1.0f / 3.0f;
            KAP(2, 0, 0) = (t + e1 + e2) * third;
            KAP(0, 2, 0) = (t - 2.0f * e1 + e2) * third;
            KAP(0, 0, 2) = (t + e1 - 2.0f * e2) * third;
        }
        KAP(2, 1, 0) *= o3; KAP(2, 0, 1) *= o3; KAP(1, 2, 0) *= o3; KAP(0, 2, 1) *= o3;
        KAP(1, 0, 2) *= o3; KAP(0, 1, 2) *= o3; KAP(1, 1, 1) *= o3;
        KAP(2, 2, 0) *= o4; KAP(2, 0, 2) *= o4; KAP(0, 2, 2) *= o4;
        KAP(2, 1, 1) *= o4; KAP(1, 2, 1) *= o4; KAP(1, 1, 2) *= o4;
        KAP(2, 2, 1) *= o5; KAP(2, 1, 2) *= o5; KAP(1, 2, 2) *= o5;
        KAP(2, 2, 2) *= o6;
#undef KAP
    }

    // inverse transform: x, then y, then z sweeps
#pragma unroll
    for (int q = 0; q < 9; ++q) sweep_inv(m[q], m[9 + q], m[18 + q], ux);
#pragma unroll
    for (int a0 = 0; a0 < 3; ++a0)
#pragma unroll
        for (int c = 0; c < 3; ++c) sweep_inv(m[a0 * 9 + 0 + c], m[a0 * 9 + 3 + c], m[a0 * 9 + 6 + c], uy);
#pragma unroll
    for (int p = 0; p < 9; ++p) sweep_inv(m[p * 3 + 0], m[p * 3 + 1], m[p * 3 + 2], uz);

    // perturbation (Eq. (30), squared numerator, both colours) and recolouring
    const float g2 = gpx * gpx + gpy * gpy + gpz * gpz;
    const float inv_gm = 1.0f / sqrtf(g2 + a.eps2);  // 1/|grad phi|_eps
    const float frac_r = rho_r * inv_rho, frac_b = rho_b * inv_rho;
    const float seg0 = a.beta * rho_r * rho_b * inv_rho * inv_gm;  // beta rho_r rho_b / (rho |g|)
    const float pert = Acoef * inv_gm;
    const int n = nb.n;
    MassAcc sum_r, sum_b;  // moving populations written (as read back), per colour
#pragma unroll
    for (int i = 1; i < 27; ++i) {  // the rest direction is the per-colour remainder below
        const float cu = (float)cx(i) * ux + (float)cy(i) * uy + (float)cz(i) * uz;
        const float cg = (float)cx(i) * grx + (float)cy(i) * gry + (float)cz(i) * grz;
        const float cF = (float)cx(i) * Fx + (float)cy(i) * Fy + (float)cz(i) * Fz;
        const float Phi = phi_corr(i) * nu * cu * cg;
        const float fe = rho * fmaf(wgt(i), eq_poly(cu, usq), varphi(i, alpha, one_m_alpha)) + Phi;
        const float Fp = wgt(i) * (3.0f * (cF - uF) + 9.0f * cu * cF);
        const float cgp = (float)cx(i) * gpx + (float)cy(i) * gpy + (float)cz(i) * gpz;
        float fs = fe + 0.5f * Fp + m[cell(i)];
        fs += pert * (wgt(i) * cgp * cgp - bcoef(i) * g2);
        const float seg = seg0 * varphi(i, alpha, one_m_alpha) * cgp * inv_cnorm(i);
        const float2 d = store_pop<S>(a, i, n, make_float2(fmaf(frac_r, fs, seg), fmaf(frac_b, fs, -seg)),
                                      dest_shift<S>(a, nb, i));
        sum_r.add(i, d.x);
        sum_b.add(i, d.y);
    }
    // rest direction as the per-colour remainder (see collide_from_moments)
    store_pop<S>(a, 0, n, make_float2(rho_r - sum_r.s, rho_b - sum_b.s), no_shift());
}

// ------------------------------------------------------------------------ launchers
static dim3 node_block() { return dim3(32, 4, 1); }
static dim3 node_grid(const StepArgs &a) { return dim3((a.nx + 31) / 32, (a.ny + 3) / 4, a.nz); }

template <int S>
static void launch_phase_field(const StepArgs &a, cudaStream_t s) {
    const bool walls = a.wall_x || a.wall_y;
    if (walls && S != STORE_FP32)
        phase_field_wall_kernel<S><<<node_grid(a), node_block(), 0, s>>>(a);
    else if (walls)
        phase_field_kernel<S, true><<<node_grid(a), node_block(), 0, s>>>(a);
    else
        phase_field_kernel<S, false><<<node_grid(a), node_block(), 0, s>>>(a);
}
template <int S>
static void launch_collide(const StepArgs &a, cudaStream_t s) {
    if (a.wall_x || a.wall_y)
        collide_general_kernel<S, true><<<node_grid(a), node_block(), 0, s>>>(a);
    else
        collide_general_kernel<S, false><<<node_grid(a), node_block(), 0, s>>>(a);
}

void launch_general_gather(const StepArgs &a, int storage, cudaStream_t s) {
    if (storage == STORE_FP16)
        launch_phase_field<STORE_FP16>(a, s);
    else if (storage == STORE_FP16_FIT)
        launch_phase_field<STORE_FP16_FIT>(a, s);
    else
        launch_phase_field<STORE_FP32>(a, s);
}
void launch_general_collide(const StepArgs &a, int storage, cudaStream_t s) {
    if (storage == STORE_FP16)
        launch_collide<STORE_FP16>(a, s);
    else if (storage == STORE_FP16_FIT)
        launch_collide<STORE_FP16_FIT>(a, s);
    else
        launch_collide<STORE_FP32>(a, s);
}

}  // namespace lbcm
