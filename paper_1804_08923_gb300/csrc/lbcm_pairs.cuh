// lbcm_pairs.cuh -- per-node pieces in the association over the 13 pairs of opposite directions: the
// gradient stencil of the general-rates step and of the half-precision storages, the moments and the
// moment record of the latter, and their inverse 1-D sweep coefficients.
#pragma once
#include "lbcm_node.cuh"

namespace lbcm {

// Isotropic gradients of phi and rho (end of Section II): grad chi = 3 sum_j w_j chi(x + c_j)
// c_j, summed over the 13 pairs of opposite directions (j, j+1) as 3 w_j c_j (chi(x + c_j) -
// chi(x - c_j)), so that a uniform field gives exactly zero and nearby values subtract
// exactly.  Ghosts: z = -1 is phi = 1, rho = rho_r0 inside the inlet disc and the mirror of
// z = 0 elsewhere; z = N + 1 mirrors z = N.  kEdge = false: the caller knows that z > 0.
template <int S, bool kEdge = true>
__device__ __forceinline__ void stencil_gradients(const StepArgs &a, const Nbr &nb, int z, float &gpx, float &gpy,
                                                  float &gpz, float &grx, float &gry, float &grz) {
    const bool inlet_lo = kEdge && z == 0 && a.bc_zlo == BC_INLET;
    float ph[27], rh[27];
#pragma unroll
    for (int j = 1; j < 27; ++j) {
        // ghost planes were clamped onto z = 0 / z = N (mirror)
        if constexpr (S == STORE_FP32) {
            const float2 v = __ldg(a.phase + nb.nbr(j));
            ph[j] = v.x;
            rh[j] = v.y;
        } else if constexpr (S == STORE_FP16) {
            const float4 v = __ldg(a.ph_cur + nb.nbr(j));
            ph[j] = v.x;
            rh[j] = v.y;
        } else {
            const float4 v = __ldg(a.ph_cur + nb.nbr(j));
            ph[j] = v.x;
            rh[j] = fit_entry_rho(v);
        }
        if (cz(j) == -1 && inlet_lo) {
            if (a.disc[nb.yo[1 - cy(j)] + nb.xo[1 - cx(j)]]) {  // z = -1 inside the inlet disc
                ph[j] = 1.0f;
                rh[j] = a.rho_r0;
            }
        }
    }
    gpx = gpy = gpz = grx = gry = grz = 0.0f;
#pragma unroll
    for (int j = 1; j < 27; j += 2) {  // c_{j+1} = -c_j
        const float w3 = 3.0f * wgt(j);
        const float dp = ph[j] - ph[j + 1], dr = rh[j] - rh[j + 1];
        if (cx(j) != 0) { gpx = fmaf(w3 * cx(j), dp, gpx); grx = fmaf(w3 * cx(j), dr, grx); }
        if (cy(j) != 0) { gpy = fmaf(w3 * cy(j), dp, gpy); gry = fmaf(w3 * cy(j), dr, gry); }
        if (cz(j) != 0) { gpz = fmaf(w3 * cz(j), dp, gpz); grz = fmaf(w3 * cz(j), dr, grz); }
    }
}

// Coefficients of the inverse 1-D sweep: a value at c in {-1, 0, +1} from central moments
// (m0, m1, m2) about u is G0[c] m0 + G1[c] m1 + G2[c] m2 with
//   G0 = ((u^2 - u)/2, 1 - u^2, (u^2 + u)/2), G1 = (u - 1/2, -2u, u + 1/2), G2 = (1/2, -1, 1/2).
struct InvAxis {
    float g0[3], g1[3];
    __device__ __forceinline__ explicit InvAxis(float u) {
        const float u2 = u * u;
        g0[0] = 0.5f * (u2 - u);
        g0[1] = 1.0f - u2;
        g0[2] = 0.5f * (u2 + u);
        g1[0] = u - 0.5f;
        g1[1] = -2.0f * u;
        g1[2] = u + 0.5f;
    }
};
__device__ __forceinline__ constexpr float g2c(int c) { return c == 0 ? -1.0f : 0.5f; }

// Moments of the post-stream populations of one node that the paper-rate collision needs:
// colour densities, colour-blind mass, momentum and raw second moment, summed over opposite pairs.
struct PairMoments {
    float rho_r, rho_b, sf, jx, jy, jz, pxx, pyy, pzz, pxy, pxz, pyz;
};

// The moments above of gathered populations (fr, fb).
__device__ __forceinline__ void pair_moments_of(const float (&fr)[27], const float (&fb)[27], PairMoments &m) {
    float sf, jx = 0.0f, jy = 0.0f, jz = 0.0f;
    float pxx = 0.0f, pyy = 0.0f, pzz = 0.0f, pxy = 0.0f, pxz = 0.0f, pyz = 0.0f;
    MassAcc mr, mb;  // the phase-field kernel's association
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        mr.add(i, fr[i]);
        mb.add(i, fb[i]);
    }
    // opposite pairs (i, i+1): odd moments take the difference, even ones the sum
    sf = fr[0] + fb[0];
#pragma unroll
    for (int i = 1; i < 27; i += 2) {
        const float fp = fr[i] + fb[i], fm = fr[i + 1] + fb[i + 1];
        const float s2 = fp + fm, d2 = fp - fm;
        sf += s2;
        if (cx(i) > 0) jx += d2; else if (cx(i) < 0) jx -= d2;
        if (cy(i) > 0) jy += d2; else if (cy(i) < 0) jy -= d2;
        if (cz(i) > 0) jz += d2; else if (cz(i) < 0) jz -= d2;
        if (cx(i) != 0) pxx += s2;
        if (cy(i) != 0) pyy += s2;
        if (cz(i) != 0) pzz += s2;
        if (cx(i) * cy(i) > 0) pxy += s2; else if (cx(i) * cy(i) < 0) pxy -= s2;
        if (cx(i) * cz(i) > 0) pxz += s2; else if (cx(i) * cz(i) < 0) pxz -= s2;
        if (cy(i) * cz(i) > 0) pyz += s2; else if (cy(i) * cz(i) < 0) pyz -= s2;
    }
    m = PairMoments{mr.total(), mb.total(), sf, jx, jy, jz, pxx, pyy, pzz, pxy, pxz, pyz};
}

// The collision moments of a node as the moment pass stores them: three float4 planes of NN
// entries, (rho_r, rho_b, sf, jx), (jy, jz, pxx, pyy), (pzz, pxy, pxz, pyz).
__device__ __forceinline__ void store_pair_moments(float4 *__restrict__ mom, size_t NN, int n, const PairMoments &m) {
    mom[n] = make_float4(m.rho_r, m.rho_b, m.sf, m.jx);
    mom[NN + n] = make_float4(m.jy, m.jz, m.pxx, m.pyy);
    mom[2 * NN + n] = make_float4(m.pzz, m.pxy, m.pxz, m.pyz);
}
__device__ __forceinline__ PairMoments load_pair_moments(const float4 *__restrict__ mom, size_t NN, int n) {
    const float4 a = __ldg(mom + n), b = __ldg(mom + NN + n), c = __ldg(mom + 2 * NN + n);
    return PairMoments{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
}

// The same for the fused step kernel, where the moments were written earlier in the same launch
// and are read once: L1 is bypassed (ld.global.cg), and the L2 lines can be dropped afterwards.
__device__ __forceinline__ PairMoments load_pair_moments_once(const float4 *__restrict__ mom, size_t NN, int n) {
    const float4 a = __ldcg(mom + n), b = __ldcg(mom + NN + n), c = __ldcg(mom + 2 * NN + n);
    return PairMoments{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
}

// Moments stored with the evict-last policy (the fused step kernel reads them a few planes later).
__device__ __forceinline__ void store_pair_moments_keep(float4 *__restrict__ mom, size_t NN, int n, const PairMoments &m,
                                                   unsigned long long pol) {
    st_keep(mom + n, make_float4(m.rho_r, m.rho_b, m.sf, m.jx), pol);
    st_keep(mom + NN + n, make_float4(m.jy, m.jz, m.pxx, m.pyy), pol);
    st_keep(mom + 2 * NN + n, make_float4(m.pzz, m.pxy, m.pxz, m.pyz), pol);
}

}  // namespace lbcm
