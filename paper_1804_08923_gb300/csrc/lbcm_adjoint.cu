// lbcm_adjoint.cu -- discrete adjoint (reverse mode) of the FP32 step with the paper's rates
// s3 = s4 = s5 = s6 = 1 (arXiv:1804.08923, Section II; boundaries of Section IV.A).
//
// The step S(n) -> S(n+1) is
//   stream (pull, inlet / mirror / convective outflow)  f = P(S(n), hist(n))
//   densities and isotropic gradients                   rho_k = sum_i f_i^k, grad phi, grad rho
//   per-node collision, perturbation, recolouring        S(n+1) = C(f, grad phi, grad rho)
// and its transpose, given lambda = dJ/dS(n+1), runs in three launches:
//   adj_collide_kernel   per node: applies (dC/df)^T, (dC/dgrad)^T to lambda of S(n+1) from the
//                        forward step's recorded moments and gradients, and accumulates dJ/d(sigma,
//                        nu_r, nu_b); writes lambda of the two gradients and the node's record (below).
//   adj_stencil_kernel   per node: transposes the gradient stencil (with the ghost rules) into
//                        lambda_rho_k, the adjoint of the node's colour densities, and adds it to
//                        the record.
//   adj_boundary_kernel  per (x, y) column: inlet-disc gradients w.r.t. u_in and the 16 profile
//                        coefficients, and the transpose of the convective outflow
//                        f(N) = [hist + lambda f(N-1)] / (1 + lambda), lambda = clamp(u_z(N-1)).
// A node's collision depends on its 54 pulled populations through its colour densities, momentum and
// second moment, so their adjoint has the form
//   lambda_f_i^k(y) = l_j . c_i + c_i Lambda c_i + l_k,
// and the adjoint state between two reverse steps is those 11 numbers a node (AdjRec, 48 bytes) where
// the populations' adjoint would be 54: lambda of slot (x, i) of S(n) is lambda_f of the node y that
// pulls it, evaluated when it is needed.  On a convective lattice the outflow adds lx, 54 numbers
// a column, to the pulls of plane N - 1, and Lh = dJ/dhist(n).  Parameter gradients are summed per
// block in FP64 into one accumulator slot per block (deterministic, no atomics).
#include "lbcm_collide.cuh"
#include "lbcm_device.cuh"
#include "lbcm_internal.h"
#include "lbcm_node.cuh"

#include <algorithm>

namespace lbcm {

// Adds the block sums of v[0..NV) to acc[blk * NV + k] (FP64).  The sum over the block's
// threads is FP32 (shuffles, then one warp over the warp sums); only the block total is
// converted and accumulated in FP64, since FP64 throughput is a small fraction of FP32 here.
// Every thread of the block must call it (no early return before).
template <int NV>
__device__ __forceinline__ void block_accumulate(const float (&v)[NV], double *acc, long long blk) {
    __shared__ float sh[NV][32];
    const int nthr = blockDim.x * blockDim.y * blockDim.z;
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int lane = tid & 31, warp = tid >> 5, nwarp = (nthr + 31) >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        float d = v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
        if (lane == 0) sh[k][warp] = d;
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            float d = lane < nwarp ? sh[k][lane] : 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
            if (lane == 0) acc[blk * NV + k] += (double)d;
        }
    }
}

__device__ __forceinline__ long long block_id() {
    return blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z);
}

// The record of the node x + c_i: through L1 (RecNbr) or from the block's ring of planes in shared
// memory (RecRing; p[cz + 1] points at the node's own cell in the plane z + cz).
struct RecNbr {
    const AdjRec &r;
    const Nbr &nb;
    __device__ __forceinline__ float4 ld(int q, int i) const { return __ldg(r.p[q] + nb.nbr(i)); }
};
// Tile of the marching collide adjoint: TX x 128 / TX nodes and one more on each side.
template <int TX>
struct AdjTile {
    static constexpr int kTY = 128 / TX, kX = TX + 2, kN = kX * (kTY + 2);
};
template <int TX>
struct RecRing {
    using T = AdjTile<TX>;
    const float4 *p[3];
    __device__ __forceinline__ float4 ld(int q, int i) const { return p[cz(i) + 1][q * T::kN + cy(i) * T::kX + cx(i)]; }
};

// lambda_f of the pull of direction i by the node x + c_i, with the signs of c as given: the record's
// polynomial.  i selects which components are there at compile time; sx, sy, sz are their signs.
template <class R>
__device__ __forceinline__ float2 adj_pull(const R &r, int i, float sx, float sy, float sz) {
    const float4 v0 = r.ld(0, i);  // (l_r, l_b, l_jx, l_jy)
    if (i == 0) return make_float2(v0.x, v0.y);
    const float4 v1 = r.ld(1, i);  // (l_jz, L_xx, L_yy, L_zz)
    float t = 0.0f, q = 0.0f;
    if (cx(i) != 0) { t = sx * v0.z; q = v1.y; }
    if (cy(i) != 0) { t = fmaf(sy, v0.w, t); q += v1.z; }
    if (cz(i) != 0) { t = fmaf(sz, v1.x, t); q += v1.w; }
    if (csq(i) > 1) {
        const float4 v2 = r.ld(2, i);  // (L_xy, L_xz, L_yz, -), off-diagonal entries doubled
        if (cx(i) != 0 && cy(i) != 0) q = fmaf(sx * sy, v2.x, q);
        if (cx(i) != 0 && cz(i) != 0) q = fmaf(sx * sz, v2.y, q);
        if (cy(i) != 0 && cz(i) != 0) q = fmaf(sy * sz, v2.z, q);
    }
    t += q;
    return make_float2(v0.x + t, v0.y + t);
}

// lambda of slot (node nb.n at height z, direction i) of S(n+1): lambda_f of the node that pulls it, in
// the direction of its pull (beyond a wall that is the node of the wall layer, with the component
// reversed).  The inlet disc and the convective plane pull nothing; the pulls of plane N - 1 have the
// outflow's part too.  kEdge = false: the caller knows that 0 < z < N - 2.  On the first reverse step
// (g.lr_obj) S(T)'s own lambda, the objective's density adjoint, is the same for every direction.
template <bool W, bool kEdge, class R>
__device__ __forceinline__ float2 adj_slot(const StepArgs &a, const AdjArgs &g, const R &r, const Nbr &nb, int i, int z,
                                           bool own_in_disc) {
    const float sx = W && nb.gx(i) ? -(float)cx(i) : (float)cx(i), sy = W && nb.gy(i) ? -(float)cy(i) : (float)cy(i);
    if (!kEdge || a.bc_zlo == BC_PERIODIC) return adj_pull(r, i, sx, sy, (float)cz(i));
    const int zr = z + cz(i), N = a.nz - 1;
    if ((zr < 0 && own_in_disc) || (a.bc_zhi == BC_CONVECTIVE && zr >= N)) return make_float2(0.0f, 0.0f);
    const float sz = zr < 0 || zr > N ? -(float)cz(i) : (float)cz(i);
    float2 v = adj_pull(r, i, sx, sy, sz);
    if (a.bc_zhi == BC_CONVECTIVE && zr == N - 1) {
        const size_t P = (size_t)a.plane;
        const float *x = g.lx + dir_of((int)sx, (int)sy, cz(i)) * P + (nb.nbr(i) - (N - 1) * (int)P);
        v.x += x[0];
        v.y += x[27 * P];
    }
    return v;
}

__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

// 1-D transpose of the inverse transform of central moments about u (values v(+-1) = (t +- o)/2,
// v(0) = m0 - t with t = u^2 m0 + 2 u m1 + m2, o = u m0 + m1), two fields at once: (v0, v1, v2) become
// lambda of m0, twice that of m1 and twice that of m2.
__device__ __forceinline__ void sweep_inv_T(float2 &v0, float2 &v1, float2 &v2, float u) {
    const float2 s = __fadd2_rn(v2, v0), d = sub2(v2, v0), e = __ffma2_rn(both(-2.0f), v1, s);
    v0 = __ffma2_rn(both(0.5f * u * u), e, __ffma2_rn(both(0.5f * u), d, v1));
    v1 = __ffma2_rn(both(2.0f * u), e, d);
    v2 = e;
}

// Weighted raw moments m_pqr = sum_i v_i w_i cx^p cy^q cz^r (p, q, r <= 2) of 27 values in the
// tensor layout [cx+1][cy+1][cz+1], by 1-D sweeps: D3Q27's w_i is the product of the 1-D weights
// (1/6, 2/3, 1/6), here times 6 an axis.  Only the moments of total order <= 3 are kept (c^3 = c on the
// lattice).
struct RawMom {
    float m000, m100, m010, m001, m200, m020, m002, m110, m101, m011, m210, m201, m120, m021, m102, m012, m111;
};
__device__ __forceinline__ void wsweep(float2 &v0, float2 &v1, float2 &v2) {
    const float2 s = __fadd2_rn(v2, v0), d = sub2(v2, v0);
    v0 = __ffma2_rn(both(4.0f), v1, s);
    v1 = d;
    v2 = s;
}
// of two fields at once: A of the .x, B of the .y
__device__ __forceinline__ void raw_moments(float2 (&t)[27], RawMom &A, RawMom &B) {
#pragma unroll
    for (int q = 0; q < 9; ++q) wsweep(t[q], t[9 + q], t[18 + q]);
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int c = 0; c < 3; ++c) wsweep(t[p * 9 + c], t[p * 9 + 3 + c], t[p * 9 + 6 + c]);
#pragma unroll
    for (int p = 0; p < 9; ++p) wsweep(t[p * 3], t[p * 3 + 1], t[p * 3 + 2]);
    auto get = [&](int p, int q, int r, float &x, float &y) {
        const float2 v = __fmul2_rn(both(1.0f / 216.0f), t[p * 9 + q * 3 + r]);
        x = v.x;
        y = v.y;
    };
    get(0, 0, 0, A.m000, B.m000);
    get(1, 0, 0, A.m100, B.m100); get(0, 1, 0, A.m010, B.m010); get(0, 0, 1, A.m001, B.m001);
    get(2, 0, 0, A.m200, B.m200); get(0, 2, 0, A.m020, B.m020); get(0, 0, 2, A.m002, B.m002);
    get(1, 1, 0, A.m110, B.m110); get(1, 0, 1, A.m101, B.m101); get(0, 1, 1, A.m011, B.m011);
    get(2, 1, 0, A.m210, B.m210); get(2, 0, 1, A.m201, B.m201); get(1, 2, 0, A.m120, B.m120);
    get(0, 2, 1, A.m021, B.m021); get(1, 0, 2, A.m102, B.m102); get(0, 1, 2, A.m012, B.m012);
    get(1, 1, 1, A.m111, B.m111);
}
// M2 v (the second-moment tensor applied to a vector) and v.M2.w
__device__ __forceinline__ void m2v(const RawMom &M, float vx, float vy, float vz, float &ox, float &oy, float &oz) {
    ox = M.m200 * vx + M.m110 * vy + M.m101 * vz;
    oy = M.m110 * vx + M.m020 * vy + M.m011 * vz;
    oz = M.m101 * vx + M.m011 * vy + M.m002 * vz;
}
// A3(., u, u)_a = sum_i v_i w_i c_a (c.u)^2
__device__ __forceinline__ void m3uu(const RawMom &M, float ux, float uy, float uz, float &ox, float &oy, float &oz) {
    const float xx = ux * ux, yy = uy * uy, zz = uz * uz, xy = 2.0f * ux * uy, xz = 2.0f * ux * uz, yz = 2.0f * uy * uz;
    ox = M.m100 * xx + M.m120 * yy + M.m102 * zz + M.m210 * xy + M.m201 * xz + M.m111 * yz;
    oy = M.m210 * xx + M.m010 * yy + M.m012 * zz + M.m120 * xy + M.m111 * xz + M.m021 * yz;
    oz = M.m201 * xx + M.m021 * yy + M.m001 * zz + M.m111 * xy + M.m102 * xz + M.m012 * yz;
}

// ---------------------------------------------------------------- reverse collision
// Every per-direction sum of the reverse pass is linear in a_i = (rho_r lS^r_i + rho_b lS^b_i)/rho
// or b_i = lS^r_i - lS^b_i with coefficients that are polynomials in c_i times shell constants
// proportional to w_i (varphi_i(alpha) = 27/19 (1 - alpha) w_i, the Phi coefficient 9 w_i and
// B_i = w_i for i >= 1), so it is a combination of the weighted raw moments of a and b up to
// third order.  Only the recolouring's 1/|c_i| is not separable and is summed directly.
template <bool kForce, bool W, class Ring, class Next>
__device__ __forceinline__ void adj_collide_node(const StepArgs &a, const AdjArgs &g, const Nbr &nb, int z, const Ring &ring,
                                                 const float4 (*own)[128], const float2 *own2, float (&part)[3],
                                                 float2 *L_s, Next &&fetch_next) {
    const int N = a.nz - 1;

    // ---- the forward step's collision inputs of this node
    const Moments mo = unpack_moments(own[0][0], own[1][0], own[2][0]);
    const float rr = mo.rho_r, rb = mo.rho_b;
    const float rho = rr + rb, inv_rho = rcp_newton(rho);
    float Fx = 0.0f, Fy = 0.0f, Fz = 0.0f;
    if (kForce) {
        const float fo = rho - a.rho_b0;
        Fx = fo * a.gx; Fy = fo * a.gy; Fz = fo * a.gz;
    }
    const float ux = fmaf(0.5f, Fx, mo.jx) * inv_rho, uy = fmaf(0.5f, Fy, mo.jy) * inv_rho,
                uz = fmaf(0.5f, Fz, mo.jz) * inv_rho;
    const float phi = order_parameter(rr, rb, a.inv_rho_r0, a.inv_rho_b0);
    const float hp = 0.5f * (1.0f + phi), hm = 0.5f * (1.0f - phi);
    const float oma = one_minus_alpha_bar(a.alpha_mix, rr, rb, inv_rho, hp, hm, a.oma_r, a.oma_b), alpha = 1.0f - oma;
    const float nu = rcp_newton(hp * a.inv_nu_r + hm * a.inv_nu_b);
    const float tau = 3.0f * nu + 0.5f, s2nu = rcp_newton(tau);
    const float Acoef = 2.25f * a.sigma * s2nu;
    const float usq = ux * ux + uy * uy + uz * uz;
    const float uF = ux * Fx + uy * Fy + uz * Fz;
    const float cs2 = oma * (9.0f / 19.0f);
    float gpx, gpy, gpz, grx, gry, grz, ugr, Qxx, Qyy, Qzz, Qxy, Qxz, Qyz;
    // gradients and Q, the second central moment of f - f^e + F'/2 (Pi(f^e), Pi(F') in closed form)
    auto load_q = [&] {
        const float4 r1 = own[1][0], r2 = own[2][0], r3 = own[3][0];
        const float2 r4 = own2[0];
        const float dxz = r1.z, dyz = r1.w, pzz = r2.x;
        gpx = r3.x; gpy = r3.y; gpz = r3.z; grx = r3.w; gry = r4.x; grz = r4.y;
        ugr = ux * grx + uy * gry + uz * grz;
        Qxx = (pzz + dxz) - (rho * cs2 + rho * ux * ux + nu * (2.0f * ux * grx + ugr));
        Qyy = (pzz + dyz) - (rho * cs2 + rho * uy * uy + nu * (2.0f * uy * gry + ugr));
        Qzz = pzz - (rho * cs2 + rho * uz * uz + nu * (2.0f * uz * grz + ugr));
        Qxy = r2.y - (rho * ux * uy + nu * (ux * gry + uy * grx));
        Qxz = r2.z - (rho * ux * uz + nu * (ux * grz + uz * grx));
        Qyz = r2.w - (rho * uy * uz + nu * (uy * grz + uz * gry));
        if (kForce) {
            Qxx += ux * Fx; Qyy += uy * Fy; Qzz += uz * Fz;
            Qxy += 0.5f * (ux * Fy + uy * Fx); Qxz += 0.5f * (ux * Fz + uz * Fx); Qyz += 0.5f * (uy * Fz + uz * Fy);
        }
    };
    load_q();
    const float o2 = 1.0f - s2nu, o2b = 1.0f - a.s2b, third = 1.0f / 3.0f;
    float trQ = Qxx + Qyy + Qzz;
    const float k200 = o2 * (Qxx - trQ * third) + o2b * trQ * third;
    const float k020 = o2 * (Qyy - trQ * third) + o2b * trQ * third;
    const float k002 = o2 * (Qzz - trQ * third) + o2b * trQ * third;
    const float k110 = o2 * Qxy, k101 = o2 * Qxz, k011 = o2 * Qyz;
    // ---- a_i and b_i into this thread's column of shared memory (tensor layout): 54 registers less
    auto put = [&](int i, float2 l) { L_s[cell(i) * 128] = make_float2((rr * l.x + rb * l.y) * inv_rho, l.x - l.y); };
    if (g.lr_obj) {
        const float2 l = __ldg(g.lr_obj + nb.n);
#pragma unroll
        for (int i = 0; i < 27; ++i) put(i, l);
    } else if (z == 0 || z >= N - 2) {
        const bool own_in_disc = a.bc_zlo == BC_INLET && z == 0 && a.disc[nb.pxy];
#pragma unroll
        for (int i = 0; i < 27; ++i) put(i, adj_slot<W, true>(a, g, ring, nb, i, z, own_in_disc));
    } else {
#pragma unroll
        for (int i = 0; i < 27; ++i) put(i, adj_slot<W, false>(a, g, ring, nb, i, z, false));
    }
    const float a0 = L_s[13 * 128].x, b0 = L_s[13 * 128].y;  // rest direction: cell 13
    const float w0 = 8.0f / 27.0f, k27 = 27.0f / 19.0f;

    // ---- h_i = sum_t C_t psi_t,i(u): lambda_C_t, d/du and sum_i b_i h_i by the transposed 1-D sweeps
    float l200, l020, l002, l110, l101, l011, lux, luy, luz, bh;
    {
        float2 t[27];
#pragma unroll
        for (int c = 0; c < 27; ++c) t[c] = L_s[c * 128];
#pragma unroll
        for (int q = 0; q < 9; ++q) sweep_inv_T(t[q], t[9 + q], t[18 + q], ux);
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int c = 0; c < 3; ++c) sweep_inv_T(t[p * 9 + c], t[p * 9 + 3 + c], t[p * 9 + 6 + c], uy);
#pragma unroll
        for (int p = 0; p < 9; ++p) sweep_inv_T(t[p * 3], t[p * 3 + 1], t[p * 3 + 2], uz);
        // an entry holds 2^(number of its nonzero orders) times its moment
        const float h200 = 0.5f * k200, h020 = 0.5f * k020, h002 = 0.5f * k002, h110 = 0.25f * k110, h101 = 0.25f * k101,
                    h011 = 0.25f * k011;
        bh = h200 * t[18].y + h020 * t[6].y + h002 * t[2].y + h110 * t[12].y + h101 * t[10].y + h011 * t[4].y;
#define MM(p, q, r) t[(p) * 9 + (q) * 3 + (r)].x
        l200 = 0.5f * MM(2, 0, 0); l020 = 0.5f * MM(0, 2, 0); l002 = 0.5f * MM(0, 0, 2);
        l110 = 0.25f * MM(1, 1, 0); l101 = 0.25f * MM(1, 0, 1); l011 = 0.25f * MM(0, 1, 1);
        // with the values G_a[c](u) of the transform: dG0/du = G1, dG1/du = 2 G2, dG2/du = 0
        lux = 0.5f * (h020 * MM(1, 2, 0) + h002 * MM(1, 0, 2) + h011 * MM(1, 1, 1)) + 2.0f * (h110 * MM(2, 1, 0) + h101 * MM(2, 0, 1));
        luy = 0.5f * (h200 * MM(2, 1, 0) + h002 * MM(0, 1, 2) + h101 * MM(1, 1, 1)) + 2.0f * (h110 * MM(1, 2, 0) + h011 * MM(0, 2, 1));
        luz = 0.5f * (h200 * MM(2, 0, 1) + h020 * MM(0, 2, 1) + h110 * MM(1, 1, 1)) + 2.0f * (h101 * MM(1, 0, 2) + h011 * MM(0, 1, 2));
#undef MM
    }

    // ---- the gradients and Q once more: read again, they take no registers while the sweeps need them all
    asm volatile("" ::: "memory");
    load_q();
    trQ = Qxx + Qyy + Qzz;
    fetch_next();  // everything of this node is in registers or in L_s now
    const float g2 = gpx * gpx + gpy * gpy + gpz * gpz;
    const float inv_gm = rsqrt_newton(fmaxf(g2 + a.eps2, 1.1754944e-38f));  // of a normal number
    const float pert = Acoef * inv_gm;
    const float R = a.beta * rr * rb * inv_rho;

    // ---- moments of a and b
    RawMom A, B;
    float Dsum, Q1x, Q1y, Q1z;
    {
        float2 t[27];
#pragma unroll
        for (int c = 0; c < 27; ++c) t[c] = L_s[c * 128];
        // Q1 = 27/19 sum_{i>=1} b_i w_i c_i / |c_i|, opposite directions and the speed classes first
        auto d = [&](int i) { return t[cell(i)].y - t[cell(i + 1)].y; };  // c_{i+1} = -c_i
        const float d7 = d(7), d9 = d(9), d11 = d(11), d13 = d(13), d15 = d(15), d17 = d(17);
        const float d19 = d(19), d21 = d(21), d23 = d(23), d25 = d(25);  // (1,1,1) (1,1,-1) (1,-1,1) (-1,1,1)
        const float p = d19 + d21, q = d23 - d25, q1 = k27 * wgt(1) * inv_cnorm(1), q2 = k27 * wgt(7) * inv_cnorm(7),
                    q3 = k27 * wgt(19) * inv_cnorm(19);
        Q1x = fmaf(q1, d(1), fmaf(q2, (d7 + d9) + (d15 + d17), q3 * (p + q)));    // (1,1,0) (1,-1,0) (1,0,1) (1,0,-1)
        Q1y = fmaf(q1, d(3), fmaf(q2, (d7 - d9) + (d11 + d13), q3 * (p - q)));    // (0,1,1) (0,1,-1)
        Q1z = fmaf(q1, d(5), fmaf(q2, (d11 - d13) + (d15 - d17), q3 * ((d19 - d21) + (d23 + d25))));
        raw_moments(t, A, B);
    }
    // ---- of b: the recolouring weight D = sum_i f**_i b_i
    {
        const float B1u = B.m100 * ux + B.m010 * uy + B.m001 * uz;
        float Bux, Buy, Buz;
        m2v(B, ux, uy, uz, Bux, Buy, Buz);
        float B3x, B3y, B3z;
        m3uu(B, ux, uy, uz, B3x, B3y, B3z);
        const float uBu = ux * Bux + uy * Buy + uz * Buz;
        const float B3uuu = ux * B3x + uy * B3y + uz * B3z;
        float Bgx, Bgy, Bgz;
        m2v(B, gpx, gpy, gpz, Bgx, Bgy, Bgz);
        Dsum = rho * fmaf(alpha, b0, k27 * oma * (B.m000 - w0 * b0));
        Dsum = fmaf(rho, 3.0f * B1u + 4.5f * uBu - 1.5f * usq * B.m000 + 4.5f * B3uuu - 4.5f * usq * B1u, Dsum);
        Dsum += -3.0f * nu * ugr * b0 + 9.0f * nu * (grx * Bux + gry * Buy + grz * Buz);
        if (kForce)
            Dsum += 0.5f * (3.0f * (B.m100 * Fx + B.m010 * Fy + B.m001 * Fz) - 3.0f * uF * B.m000 +
                            9.0f * (Fx * Bux + Fy * Buy + Fz * Buz));
        Dsum += bh;
        Dsum = fmaf(pert, gpx * Bgx + gpy * Bgy + gpz * Bgz - g2 * (B.m000 - (2.0f / 3.0f) * b0), Dsum);
    }

    // ---- recolouring: S^r = (rho_r/rho) f** + seg, S^b = (rho_b/rho) f** - seg
    float lrr = Dsum * rb * inv_rho * inv_rho, lrb = -Dsum * rr * inv_rho * inv_rho;
    float lrho = 0.0f;
    const float gQ1 = gpx * Q1x + gpy * Q1y + gpz * Q1z;
    const float lR = oma * gQ1 * inv_gm;
    float lalpha = -R * inv_gm * gQ1;
    lrr = fmaf(lR * a.beta, rb * inv_rho, lrr);
    lrb = fmaf(lR * a.beta, rr * inv_rho, lrb);
    lrho = fmaf(-lR, R * inv_rho, lrho);
    const float sq = R * inv_gm * oma;
    float lgpx = sq * Q1x, lgpy = sq * Q1y, lgpz = sq * Q1z;
    float lgm = -R * lR * inv_gm;

    // ---- moments of a: perturbation, equilibrium, forcing
    float lnu, lgrx, lgry, lgrz, lFx = 0.0f, lFy = 0.0f, lFz = 0.0f, lA;
    {
        const float sB = A.m000 - (2.0f / 3.0f) * a0;  // sum_i a_i B_i
        float Agx, Agy, Agz, Aux, Auy, Auz, Arx, Ary, Arz;
        m2v(A, gpx, gpy, gpz, Agx, Agy, Agz);
        m2v(A, ux, uy, uz, Aux, Auy, Auz);
        m2v(A, grx, gry, grz, Arx, Ary, Arz);
        // perturbation Omega2_i = A (w_i cgp^2 - B_i |g|^2) / |g|_eps
        lA = (gpx * Agx + gpy * Agy + gpz * Agz - g2 * sB) * inv_gm;
        lgpx = fmaf(2.0f * pert, Agx, lgpx);
        lgpy = fmaf(2.0f * pert, Agy, lgpy);
        lgpz = fmaf(2.0f * pert, Agz, lgpz);
        float lg2 = -pert * sB;
        lgm = fmaf(-lA, pert, lgm);
        lg2 = fmaf(lgm, 0.5f * inv_gm, lg2);
        lgpx = fmaf(2.0f * gpx, lg2, lgpx);
        lgpy = fmaf(2.0f * gpy, lg2, lgpy);
        lgpz = fmaf(2.0f * gpz, lg2, lgpz);
        part[0] += lA * 2.25f * s2nu;
        // equilibrium f^e_i = rho (varphi_i(alpha) + w_i poly_i(u)) + Phi_i(nu, u, grad rho)
        const float A1u = A.m100 * ux + A.m010 * uy + A.m001 * uz;
        float A3x, A3y, A3z;
        m3uu(A, ux, uy, uz, A3x, A3y, A3z);
        const float uAu = ux * Aux + uy * Auy + uz * Auz;
        const float A3uuu = ux * A3x + uy * A3y + uz * A3z;
        lrho += fmaf(alpha, a0, k27 * oma * (A.m000 - w0 * a0)) + 3.0f * A1u + 4.5f * uAu - 1.5f * usq * A.m000 +
                4.5f * A3uuu - 4.5f * usq * A1u;
        lalpha = fmaf(rho, a0 - k27 * (A.m000 - w0 * a0), lalpha);
        const float c3 = 3.0f - 4.5f * usq, s_u = -3.0f * A.m000 - 9.0f * A1u;
        lux += rho * (c3 * A.m100 + 9.0f * Aux + 13.5f * A3x + ux * s_u);
        luy += rho * (c3 * A.m010 + 9.0f * Auy + 13.5f * A3y + uy * s_u);
        luz += rho * (c3 * A.m001 + 9.0f * Auz + 13.5f * A3z + uz * s_u);
        lnu = -3.0f * a0 * ugr + 9.0f * (ux * Arx + uy * Ary + uz * Arz);
        lux = fmaf(nu, fmaf(-3.0f * a0, grx, 9.0f * Arx), lux);
        luy = fmaf(nu, fmaf(-3.0f * a0, gry, 9.0f * Ary), luy);
        luz = fmaf(nu, fmaf(-3.0f * a0, grz, 9.0f * Arz), luz);
        lgrx = nu * fmaf(-3.0f * a0, ux, 9.0f * Aux);
        lgry = nu * fmaf(-3.0f * a0, uy, 9.0f * Auy);
        lgrz = nu * fmaf(-3.0f * a0, uz, 9.0f * Auz);
        // forcing F'_i = w_i (3 (c_i - u).F + 9 (c_i.u)(c_i.F)), weight 1/2 in f*
        if (kForce) {
            float AFx, AFy, AFz;
            m2v(A, Fx, Fy, Fz, AFx, AFy, AFz);
            lux += 0.5f * (-3.0f * Fx * A.m000 + 9.0f * AFx);
            luy += 0.5f * (-3.0f * Fy * A.m000 + 9.0f * AFy);
            luz += 0.5f * (-3.0f * Fz * A.m000 + 9.0f * AFz);
            lFx = 0.5f * (3.0f * A.m100 - 3.0f * ux * A.m000 + 9.0f * Aux);
            lFy = 0.5f * (3.0f * A.m010 - 3.0f * uy * A.m000 + 9.0f * Auy);
            lFz = 0.5f * (3.0f * A.m001 - 3.0f * uz * A.m000 + 9.0f * Auz);
        }
    }
    // ---- relaxation C = (1 - s2nu) dev Q + (1 - s2b) (tr Q / 3) I
    const float trl = l200 + l020 + l002;
    const float lQxx = o2 * (l200 - trl * third) + o2b * trl * third;
    const float lQyy = o2 * (l020 - trl * third) + o2b * trl * third;
    const float lQzz = o2 * (l002 - trl * third) + o2b * trl * third;
    const float lQxy = o2 * l110, lQxz = o2 * l101, lQyz = o2 * l011;
    const float ls2nu = -(l200 * (Qxx - trQ * third) + l020 * (Qyy - trQ * third) + l002 * (Qzz - trQ * third) +
                          l110 * Qxy + l101 * Qxz + l011 * Qyz);
    // ---- Q: symmetric Lambda (diagonal lQ_aa, off-diagonal lQ_ab / 2)
    const float Lxy = 0.5f * lQxy, Lxz = 0.5f * lQxz, Lyz = 0.5f * lQyz;
    const float Lux = lQxx * ux + Lxy * uy + Lxz * uz;
    const float Luy = Lxy * ux + lQyy * uy + Lyz * uz;
    const float Luz = Lxz * ux + Lyz * uy + lQzz * uz;
    const float Lgx = lQxx * grx + Lxy * gry + Lxz * grz;
    const float Lgy = Lxy * grx + lQyy * gry + Lyz * grz;
    const float Lgz = Lxz * grx + Lyz * gry + lQzz * grz;
    const float Ltr = lQxx + lQyy + lQzz;
    lrho += -(ux * Lux + uy * Luy + uz * Luz) - cs2 * Ltr;
    lux += -2.0f * rho * Lux - nu * (2.0f * Lgx + Ltr * grx);
    luy += -2.0f * rho * Luy - nu * (2.0f * Lgy + Ltr * gry);
    luz += -2.0f * rho * Luz - nu * (2.0f * Lgz + Ltr * grz);
    if (kForce) {
        lux += lQxx * Fx + Lxy * Fy + Lxz * Fz;
        luy += Lxy * Fx + lQyy * Fy + Lyz * Fz;
        luz += Lxz * Fx + Lyz * Fy + lQzz * Fz;
        lFx += Lux; lFy += Luy; lFz += Luz;
    }
    lalpha = fmaf(9.0f / 19.0f * rho, Ltr, lalpha);
    lnu += -(2.0f * (ux * Lgx + uy * Lgy + uz * Lgz) + Ltr * ugr);
    lgrx -= nu * fmaf(2.0f, Lux, Ltr * ux);
    lgry -= nu * fmaf(2.0f, Luy, Ltr * uy);
    lgrz -= nu * fmaf(2.0f, Luz, Ltr * uz);
    // ---- sigma, tau, nu (harmonic mean), alpha-bar
    const float ltau = -lA * Acoef * s2nu - ls2nu * s2nu * s2nu;
    lnu = fmaf(3.0f, ltau, lnu);
    const float lH = -lnu * nu * nu;
    float lphi = lH * 0.5f * (a.inv_nu_r - a.inv_nu_b);
    part[1] += -lH * hp * a.inv_nu_r * a.inv_nu_r;
    part[2] += -lH * hm * a.inv_nu_b * a.inv_nu_b;
    if (a.alpha_mix) {  // alpha-bar = (rho_r alpha_r + rho_b alpha_b) / rho
        lrr = fmaf(lalpha, (oma - a.oma_r) * inv_rho, lrr);  // (alpha_r - alpha-bar) / rho
        lrb = fmaf(lalpha, (oma - a.oma_b) * inv_rho, lrb);
    } else {
        lphi = fmaf(lalpha, 0.5f * (a.oma_b - a.oma_r), lphi);  // (alpha_r - alpha_b) / 2
    }
    // ---- u = (j + F/2) / rho, F = (rho - rho_b0) g
    const float ljx = lux * inv_rho, ljy = luy * inv_rho, ljz = luz * inv_rho;
    if (kForce) {
        lFx = fmaf(0.5f, ljx, lFx);
        lFy = fmaf(0.5f, ljy, lFy);
        lFz = fmaf(0.5f, ljz, lFz);
        lrho += lFx * a.gx + lFy * a.gy + lFz * a.gz;
    }
    lrho -= (lux * ux + luy * uy + luz * uz) * inv_rho;
    // ---- phi = (A - B)/(A + B), A = rho_r / rho_r0, B = rho_b / rho_b0
    {
        const float S_ = rr * a.inv_rho_r0 + rb * a.inv_rho_b0;
        const float t = lphi * rcp_newton(S_);
        lrr = fmaf(t * (1.0f - phi), a.inv_rho_r0, lrr);
        lrb = fmaf(-t * (1.0f + phi), a.inv_rho_b0, lrb);
    }
    lrr += lrho;
    lrb += lrho;

    // ---- outputs: the record of lambda_f_i^k = lambda_j . c_i + c_i Lambda_P c_i + lambda_rho_k
    g.lga[nb.n] = make_float4(lgpx, lgpy, lgpz, lgrx);
    g.lgb[nb.n] = make_float2(lgry, lgrz);
    g.rec_out.p[0][nb.n] = make_float4(lrr, lrb, ljx, ljy);
    g.rec_out.p[1][nb.n] = make_float4(ljz, lQxx, lQyy, lQzz);
    g.rec_out.p[2][nb.n] = make_float4(lQxy, lQxz, lQyz, 0.0f);
}

// Shared memory of a block of adj_collide_kernel: a ring of four planes of the tile's records, a_i and
// b_i of every node of the plane in hand, and the forward step's record of that node.
template <int TX>
struct AdjSmem {
    float4 ring[4][3 * AdjTile<TX>::kN];
    float4 own[4][128];
    float2 own2[128];
    float2 ab[27 * 128];
};

// A block marches chunk planes of a tile of TX x 128 / TX columns upwards.  While a plane is worked on, the
// tile's records of the plane after next and the own record of the next one arrive by cp.async.  What
// bounds it is the latency of the node's arithmetic (1700 instructions in 158 registers, three warps a
// scheduler; a fourth block an SM does not fit the registers), so memory is kept out of it: gathered
// straight from memory, the 73 16-byte loads of a node were 40% of the stall cycles and moved 650 bytes a
// node through L2.  64x64x256: 144 us gathered; 110 in the ring with a and b as pairs; 104 with the own
// record fetched before the arithmetic; 98 without spills (load_q reads twice); 83 with the reciprocals
// of lbcm_collide.cuh.
template <bool kForce, bool W, int TX>
__global__ void __launch_bounds__(128, 3) adj_collide_kernel(StepArgs a, AdjArgs g, int chunk) {
    chain_begin();
    extern __shared__ float4 adj_dsm[];
    using T = AdjTile<TX>;
    AdjSmem<TX> &S = *reinterpret_cast<AdjSmem<TX> *>(adj_dsm);
    const int t = threadIdx.x, tx = t % TX, ty = t / TX, P = (int)a.plane;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * T::kTY, z0 = blockIdx.z * chunk, z1 = min(z0 + chunk, a.nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool live = x < a.nx && y < a.ny;
    // this thread's two cells of the tile, wrapped or reflected at the sides as Nbr does; cells beyond
    // the node after the last are never read
    int cell0[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int c = t + 128 * k, xs = x0 - 1 + c % T::kX, ys = y0 - 1 + c / T::kX;
        const int xw = a.wall_x ? min(max(xs, 0), a.nx - 1) : (xs < 0 ? a.nx - 1 : (xs < a.nx ? xs : 0));
        const int yw = a.wall_y ? min(max(ys, 0), a.ny - 1) : (ys < 0 ? a.ny - 1 : (ys < a.ny ? ys : 0));
        cell0[k] = yw * a.nx + xw;
    }
    auto fetch_plane = [&](int z) {  // z in [-1, nz]
        int zs = z;
        if (a.bc_zlo == BC_PERIODIC) zs = wrapi(z, a.nz);
        zs = min(max(zs, 0), a.nz - 1);
        float4 *dst = S.ring[(z + 1) & 3];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int c = t + 128 * k;
            if (c < T::kN) {
#pragma unroll
                for (int q = 0; q < 3; ++q) cp_async<16>(dst + q * T::kN + c, g.rec_in.p[q] + (size_t)zs * P + cell0[k]);
            }
        }
    };
    const size_t NN = (size_t)a.NN;
    auto fetch_own = [&](int z) {
        if (!live) return;
        const size_t n = (size_t)z * P + (size_t)y * a.nx + x;
#pragma unroll
        for (int q = 0; q < 3; ++q) cp_async<16>(&S.own[q][t], g.mom + q * NN + n);
        cp_async<16>(&S.own[3][t], g.grad4 + n);
        cp_async<8>(&S.own2[t], g.grad2 + n);
    };
    const bool gather = g.lr_obj == nullptr;
    if (gather) {
        fetch_plane(z0 - 1);
        fetch_plane(z0);
        fetch_plane(z0 + 1);
    }
    fetch_own(z0);
    // parameter sums of this thread's column, compensated: the sum over a block keeps the rounding of a
    // sum of one term a thread
    float sum[3] = {0.0f, 0.0f, 0.0f}, low[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll 1
    for (int z = z0; z < z1; ++z) {
        cp_async_wait_all();
        __syncthreads();  // plane z + 1 is there for every thread, and nobody reads plane z - 2 any more
        if (gather && z + 1 < z1) fetch_plane(z + 2);
        if (live) {
            const Nbr nb(a, x, y, z);
            const int c = (ty + 1) * T::kX + tx + 1;
            const RecRing<TX> ring{{S.ring[z & 3] + c, S.ring[(z + 1) & 3] + c, S.ring[(z + 2) & 3] + c}};
            float part[3] = {0.0f, 0.0f, 0.0f};
            adj_collide_node<kForce, W>(a, g, nb, z, ring, reinterpret_cast<const float4 (*)[128]>(&S.own[0][t]), S.own2 + t, part, S.ab + t, [&] { if (z + 1 < z1) fetch_own(z + 1); });
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float s = sum[k] + part[k], bb = s - sum[k];
                low[k] += (sum[k] - (s - bb)) + (part[k] - bb);
                sum[k] = s;
            }
        }
    }
    float part[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) part[k] = sum[k] + low[k];
    block_accumulate<3>(part, g.acc_coll, block_id());
}

// --------------------------------------------------- transposed gradient stencil (K3)
// lambda_rho_k of node n from lambda_phi and lambda_rho; what it needs of the node is loaded ahead.
struct StencilNode {
    float4 r0;  // a reverse step: (rho_r, rho_b, phi, jx); the objective: (phi, rho, -, -)
    float2 l;   // the record's (l_r, l_b)
    __device__ __forceinline__ void load(const StepArgs &a, const AdjArgs &g, int n) {
        if (g.mom) {
            r0 = __ldg(g.mom + n);
            l = *reinterpret_cast<const float2 *>(g.rec_out.p[0] + n);
        } else {
            const float2 ph = __ldg(a.phase + n);
            r0 = make_float4(ph.x, ph.y, 0.0f, 0.0f);
        }
    }
};
__device__ __forceinline__ void adj_stencil_out(const StepArgs &a, const AdjArgs &g, int n, const StencilNode &s, float lphi,
                                                float lrho) {
    float phv, S_;  // phi and rho_r/rho_r0 + rho_b/rho_b0 of this node
    if (g.mom) {
        phv = order_parameter(s.r0.x, s.r0.y, a.inv_rho_r0, a.inv_rho_b0);
        S_ = s.r0.x * a.inv_rho_r0 + s.r0.y * a.inv_rho_b0;
    } else {
        phv = s.r0.x;
        S_ = s.r0.y / (a.rho_r0 * 0.5f * (1.0f + phv) + a.rho_b0 * 0.5f * (1.0f - phv));
    }
    const float t = lphi * rcp_newton(S_);
    const float2 l = make_float2(fmaf(t * (1.0f - phv), a.inv_rho_r0, lrho), fmaf(-t * (1.0f + phv), a.inv_rho_b0, lrho));
    if (g.mom)  // into the record
        *reinterpret_cast<float2 *>(g.rec_out.p[0] + n) = make_float2(s.l.x + l.x, s.l.y + l.y);
    else
        g.lr_out[n] = l;
}

// lambda_phi(y) = sum over the nodes x whose stencil reads y of 3 w_j c_j . lambda_gphi(x); a
// node x on z = 0 (z = N) reads y through the mirror ghost with c_j's z component flipped,
// except inside the inlet disc, where the ghost is a constant.  Same for rho.  Then
// lambda_rho_k(y) = lambda_phi dphi/drho_k + lambda_rho.
// A thread marches chunk planes of its column.  The nine readers in a plane z enter the sums of z - 1,
// z and z + 1 only as three numbers a field, so a plane's 18 loads are made once and not three times.
struct StencilPart {
    float2 in, xy, z;  // (phi, rho): sum for the plane itself; x, y and z terms for the planes next to it
};
template <bool W>
__global__ void __launch_bounds__(128) adj_stencil_kernel(StepArgs a, AdjArgs g, int chunk) {
    chain_begin();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= a.nx || y >= a.ny) return;
    const int z0 = blockIdx.z * chunk, z1 = min(z0 + chunk, a.nz), N = a.nz - 1;
    const bool pz = a.bc_zlo == BC_PERIODIC;
    const Nbr nb(a, x, y, z0);
    const bool lo_const = a.bc_zlo == BC_INLET && z0 == 0 && a.disc[nb.pxy];  // the disc ghost is a constant
    struct Readers {
        float4 A[9];
        float2 B[9];
    };
    auto load = [&](int z) {
        const size_t base = (size_t)z * (size_t)a.plane;
        Readers r;
#pragma unroll
        for (int q = 0; q < 9; ++q) {  // the node x - c, clamped onto a side wall: the mirrored reader
            const size_t n = base + nb.yo[q / 3] + nb.xo[q % 3];
            r.A[q] = __ldg(g.lga + n);
            r.B[q] = __ldg(g.lgb + n);
        }
        return r;
    };
    auto sums = [&](const Readers &r) {
        const float4(&A)[9] = r.A;
        const float2(&B)[9] = r.B;
        StencilPart o{{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int dx = q % 3 - 1, dy = q / 3 - 1, m = dx * dx + dy * dy;
            // beyond a side wall the reader reached y through its mirror ghost with that component of c
            // reversed
            const float sx = W && (dx > 0 ? nb.wxl : dx < 0 && nb.wxh) ? -(float)dx : (float)dx;
            const float sy = W && (dy > 0 ? nb.wyl : dy < 0 && nb.wyh) ? -(float)dy : (float)dy;
            const float w0 = m == 1 ? 6.0f / 27.0f : 3.0f / 54.0f, w1 = m == 0 ? 6.0f / 27.0f : m == 1 ? 3.0f / 54.0f : 3.0f / 216.0f;
            if (m > 0) {
                const float tp = dx == 0 ? sy * A[q].y : dy == 0 ? sx * A[q].x : fmaf(sx, A[q].x, sy * A[q].y);
                const float tr = dx == 0 ? sy * B[q].x : dy == 0 ? sx * A[q].w : fmaf(sx, A[q].w, sy * B[q].x);
                o.in.x = fmaf(w0, tp, o.in.x);
                o.in.y = fmaf(w0, tr, o.in.y);
                o.xy.x = fmaf(w1, tp, o.xy.x);
                o.xy.y = fmaf(w1, tr, o.xy.y);
            }
            o.z.x = fmaf(w1, A[q].z, o.z.x);
            o.z.y = fmaf(w1, B[q].y, o.z.y);
        }
        return o;
    };
    StencilPart lo{}, cur = sums(load(z0)), hi{};
    if (z0 > 0 || pz) lo = sums(load(z0 > 0 ? z0 - 1 : N));
#pragma unroll 1
    for (int z = z0; z < z1; ++z) {
        const int n = z * (int)a.plane + nb.pxy;
        StencilNode node;
        node.load(a, g, n);
        float lphi = cur.in.x, lrho = cur.in.y;
        if (z < N || pz) {
            hi = sums(load(z < N ? z + 1 : 0));
            lphi += hi.xy.x - hi.z.x;
            lrho += hi.xy.y - hi.z.y;
        } else {  // beyond a wall the reader is on this layer, with the z component of c reversed
            lphi += cur.xy.x + cur.z.x;
            lrho += cur.xy.y + cur.z.y;
        }
        if (z > 0 || pz) {
            lphi += lo.xy.x + lo.z.x;
            lrho += lo.xy.y + lo.z.y;
        } else if (!lo_const) {
            lphi += cur.xy.x - cur.z.x;
            lrho += cur.xy.y - cur.z.y;
        }
        adj_stencil_out(a, g, n, node, lphi, lrho);
        lo = cur;
        cur = hi;
    }
}

// ----------------------------------------------- inlet gradients and outflow transpose
// One warp per (x, y) column and plane (blockIdx.y = 0: z = 0, 1: z = N), lane i < 27 handling direction i
// (both colours).  Bound by the chain of its loads.
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// lambda_f of node n's own pull of direction c (components known at run time).
__device__ __forceinline__ float2 adj_pull_any(const AdjRec &r, size_t n, int c0, int c1, int c2) {
    const float4 v0 = r.p[0][n], v1 = r.p[1][n], v2 = r.p[2][n];
    const float x = (float)c0, y = (float)c1, z = (float)c2;
    const float t = x * v0.z + y * v0.w + z * v1.x + x * x * v1.y + y * y * v1.z + z * z * v1.w + x * y * v2.x + x * z * v2.y + y * z * v2.z;
    return make_float2(v0.x + t, v0.y + t);
}

__global__ void __launch_bounds__(128) adj_boundary_kernel(StepArgs a, AdjArgs g) {
    chain_begin();
    const int lane = threadIdx.x & 31;
    const long long col = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    float part[17];
#pragma unroll
    for (int k = 0; k < 17; ++k) part[k] = 0.0f;
    if (col < a.plane) {  // warp-uniform
        const int x = (int)(col % a.nx), y = (int)(col / a.nx);
        const size_t P = (size_t)a.plane, pxy = (size_t)col;
        const int i = lane < 27 ? lane : 0;
        const int cxi = (int)((kPackX >> (2 * i)) & 3ull) - 1, cyi = (int)((kPackY >> (2 * i)) & 3ull) - 1,
                  czi = (int)((kPackZ >> (2 * i)) & 3ull) - 1;
        // source column of the pull of direction i, reflected at free-slip side walls, and the
        // direction that leaves it
        int xs = x - cxi, ys = y - cyi, cxs = cxi, cys = cyi;
        if (xs < 0 || xs >= a.nx) {
            if (a.wall_x) { xs = x; cxs = -cxi; } else xs = wrapi(xs, a.nx);
        }
        if (ys < 0 || ys >= a.ny) {
            if (a.wall_y) { ys = y; cys = -cyi; } else ys = wrapi(ys, a.ny);
        }
        const int q = cxi * cxi + cyi * cyi + czi * czi;
        const float w_i = q == 0 ? 8.0f / 27.0f : q == 1 ? 2.0f / 27.0f : q == 2 ? 1.0f / 54.0f : 1.0f / 216.0f;
        if (blockIdx.y == 0 && a.bc_zlo == BC_INLET && lane < 27 && czi == 1) {
            const float lam = adj_pull_any(g.rec_out, pxy, cxi, cyi, czi).x;
            if (a.disc[(size_t)ys * a.nx + xs]) {
                InletVel iv;
                inlet_velocity(a.u_in, a.noise_amp, a.fourier, a.xc, a.yc, a.seed, a.step, xs, ys, a.nx, a.ny, iv);
                const float c0 = (float)cxs, c1 = (float)cys, c2 = (float)czi;  // direction leaving the ghost
                const float cu = c0 * iv.ux + c1 * iv.uy + c2 * iv.uz;
                const float usq = iv.ux * iv.ux + iv.uy * iv.uy + iv.uz * iv.uz;
                // d f^e_i / d u = rho_r0 w_i [(3 + 9 cu + 27/2 cu^2 - 9/2 u^2) c_i - (3 + 9 cu) u]
                const float sc = lam * a.rho_r0 * w_i;
                const float dp = fmaf(13.5f * cu, cu, fmaf(9.0f, cu, 3.0f)) - 4.5f * usq;
                const float du = fmaf(-9.0f, cu, -3.0f);
                const float gx_ = sc * fmaf(c0, dp, du * iv.ux);
                const float gy_ = sc * fmaf(c1, dp, du * iv.uy);
                const float gz_ = sc * fmaf(c2, dp, du * iv.uz);
                part[0] = gx_ * iv.dux + gy_ * iv.duy + gz_ * iv.prof;
#pragma unroll
                for (int m = 1; m <= 8; ++m) {
                    part[2 * m - 1] = gz_ * a.u_in * iv.cm[m];
                    part[2 * m] = gz_ * a.u_in * iv.sm[m];
                }
            }
        }
        if (blockIdx.y == 1 && a.bc_zhi == BC_CONVECTIVE) {
            const int N = a.nz - 1;
            const size_t hr = (size_t)i * P + pxy, hb = (size_t)(27 + i) * P + pxy;
            float fr = 0.0f, fb = 0.0f, lvr = 0.0f, lvb = 0.0f, hist_r = 0.0f, hist_b = 0.0f;
            if (lane < 27) {  // f(N-1) as the forward step pulled it; every load before the sums
                const float2 lN = adj_pull_any(g.rec_out, (size_t)N * P + pxy, cxi, cyi, czi);
                lvr = lN.x + g.lh_in[hr];
                lvb = lN.y + g.lh_in[hb];
                hist_r = a.hist_out[hr];
                hist_b = a.hist_out[hb];
                fr = __ldg(g.fm + (size_t)i * P + pxy);
                fb = __ldg(g.fm + (size_t)(27 + i) * P + pxy);
            }
            const float s_ = fr + fb;
            const float rho = warp_sum(s_), jz = warp_sum((float)czi * s_);
            const float Fz = (rho - a.rho_b0) * a.gz;
            const float lam_raw = (jz + 0.5f * Fz) / rho;
            const float lam = fminf(fmaxf(lam_raw, 0.0f), 1.0f);
            const float inv = 1.0f / (1.0f + lam);
            float part_l = 0.0f;
            if (lane < 27) {
                g.lh_out[hr] = lvr * inv;
                g.lh_out[hb] = lvb * inv;
                part_l = fmaf(lvr, fr - hist_r, lvb * (fb - hist_b));
            }
            const float llam = warp_sum(part_l) * inv;
            if (lane < 27) {
                const bool active = lam_raw > 0.0f && lam_raw < 1.0f;
                const float dl = active ? llam * ((float)czi + 0.5f * a.gz - lam_raw) / rho : 0.0f;
                g.lx[hr] = fmaf(lvr, lam * inv, dl);
                g.lx[hb] = fmaf(lvb, lam * inv, dl);
            }
        }
    }
    // only blocks holding inlet-disc columns have inlet gradients; the others skip the reduction
    // (the decision is block-uniform, so every thread of a block takes the same branch)
    bool any = false;
#pragma unroll
    for (int k = 0; k < 17; ++k) any |= part[k] != 0.0f;
    if (__syncthreads_or(any)) block_accumulate<17>(part, g.acc_inlet, block_id());
}

// ------------------------------------------------------------------- objectives
// (phi, rho) of a post-collision state: rho_k = sum_i S_i^k, as the collision summed.
__global__ void __launch_bounds__(256) obj_fields_kernel(StepArgs a, float2 *ph) {
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.NN; n += (long long)gridDim.x * blockDim.x) {
        float2 f[27];
#pragma unroll
        for (int i = 0; i < 27; ++i) f[i] = load_pop<STORE_FP32>(a, i, (int)n, no_shift());
        const float2 s = moving_mass([&](int i) { return f[i]; });
        const float rr = f[0].x + s.x, rb = f[0].y + s.y;
        ph[n] = make_float2(order_parameter(rr, rb, a.inv_rho_r0, a.inv_rho_b0), rr + rb);
    }
}

// Interface area sum over 1 <= z <= nz-2 of sqrt(|grad phi|^2 + eps^2) (isotropic stencil,
// periodic in x and y); writes lambda_grad phi = grad phi / sqrt(...) (zero elsewhere).
__global__ void __launch_bounds__(128) obj_area_kernel(StepArgs a, const float2 *ph, float4 *lga, float2 *lgb,
                                                      double *acc, float eps2) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    float part[1] = {0.0f};
    if (x < a.nx && y < a.ny) {
        const Nbr nb(a, x, y, z);
        float gx = 0.0f, gy = 0.0f, gz = 0.0f;
        const bool inside = z >= 1 && z <= a.nz - 2;
        if (inside) {
#pragma unroll
            for (int j = 1; j < 27; j += 2) {
                const float w3 = 3.0f * wgt(j);
                const float d = __ldg(ph + nb.nbr(j)).x - __ldg(ph + nb.nbr(j + 1)).x;
                gx = fmaf(w3 * cx(j), d, gx);
                gy = fmaf(w3 * cy(j), d, gy);
                gz = fmaf(w3 * cz(j), d, gz);
            }
            const float m = sqrtf(gx * gx + gy * gy + gz * gz + eps2);
            part[0] = m;
            const float im = 1.0f / m;
            gx *= im; gy *= im; gz *= im;
        }
        lga[nb.n] = make_float4(gx, gy, gz, 0.0f);
        lgb[nb.n] = make_float2(0.0f, 0.0f);
    }
    block_accumulate<1>(part, acc, block_id());
}

// Penetration length (smooth maximum): L = delta log sum_n H(phi_n) exp(z_n / delta) with the
// redness weight H = ((1 + phi)/2)^2, accumulated as sum H exp((z - N) / delta).
__global__ void __launch_bounds__(128) obj_pen_sum_kernel(StepArgs a, const float2 *ph, double *acc, float inv_delta) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    float part[1] = {0.0f};
    if (x < a.nx && y < a.ny) {
        const float h = 0.5f * (1.0f + __ldg(ph + ((size_t)z * a.plane + (size_t)y * a.nx + x)).x);
        part[0] = h * h * expf((float)(z - (a.nz - 1)) * inv_delta);
    }
    block_accumulate<1>(part, acc, block_id());
}

// lambda_S(T)(n, k, i) = dL/dphi_n dphi/drho_k for every i.
__global__ void __launch_bounds__(256) obj_pen_adjoint_kernel(StepArgs a, const float2 *ph, const double *Z,
                                                             float2 *lr, float inv_delta, float delta) {
    const float inv_Z = (float)(1.0 / *Z);
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.NN; n += (long long)gridDim.x * blockDim.x) {
        const float2 v = ph[n];
        const int z = (int)(n / a.plane);
        const float lphi = delta * 0.5f * (1.0f + v.x) * expf((float)(z - (a.nz - 1)) * inv_delta) * inv_Z;
        const float S_ = v.y / (a.rho_r0 * 0.5f * (1.0f + v.x) + a.rho_b0 * 0.5f * (1.0f - v.x));
        const float q = lphi / S_;
        lr[n] = make_float2(q * (1.0f - v.x) * a.inv_rho_r0, -q * (1.0f + v.x) * a.inv_rho_b0);
    }
}

// out[k] = sum_b acc[b * nv + k0 + k] (FP64, fixed order: deterministic).
__global__ void __launch_bounds__(1024) adj_reduce_kernel(const double *acc, long long nblk, int nv, int k0,
                                                         double *out) {
    __shared__ double sh[1024];
    const int k = blockIdx.x;
    double s = 0.0;
    for (long long b = threadIdx.x; b < nblk; b += blockDim.x) s += acc[b * nv + k0 + k];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[k] = sh[0];
}

// J of the penetration objective from Z: L = N + delta log Z.
__global__ void obj_pen_value_kernel(const double *Z, double *out, double N, double delta) {
    if (threadIdx.x == 0 && blockIdx.x == 0) out[0] = N + delta * log(*Z);
}

// dJ/dS(n) in the canonical layout [k][i][z][y][x] from the records.
__global__ void __launch_bounds__(256) adj_state_kernel(StepArgs a, AdjArgs g, float *out) {
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.NN; n += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(n % a.nx), y = (int)((n / a.nx) % a.ny), z = (int)(n / a.plane);
        const Nbr nb(a, x, y, z);
        const bool own_in_disc = a.bc_zlo == BC_INLET && z == 0 && a.disc[nb.pxy];
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            const float2 v = adj_slot<true, true>(a, g, RecNbr{g.rec_in, nb}, nb, i, z, own_in_disc);
            out[(size_t)i * a.NN + n] = v.x;
            out[(size_t)(27 + i) * a.NN + n] = v.y;
        }
    }
}

// ------------------------------------------------------------------------ launchers
static dim3 node_block() { return dim3(32, 4, 1); }
static dim3 node_grid(const StepArgs &a) { return dim3((a.nx + 31) / 32, (a.ny + 3) / 4, a.nz); }
static dim3 col_block() { return dim3(128, 1, 1); }  // four columns, one warp each
static dim3 col_grid(const StepArgs &a) { return dim3((unsigned)((a.plane + 3) / 4), 1, 1); }

long long adj_collide_blocks(const StepArgs &a) {
    const dim3 gr = node_grid(a);
    return (long long)gr.x * gr.y * gr.z;
}
long long adj_boundary_blocks(const StepArgs &a) {
    const dim3 gr = col_grid(a);
    return (long long)gr.x * gr.y * gr.z;
}

static long long tile_columns(const StepArgs &a, int tx) {
    return (long long)((a.nx + tx - 1) / tx) * ((a.ny + 128 / tx - 1) / (128 / tx));
}
// Tile width of the collide adjoint and the stencil: 32, or 16 where that takes fewer tiles (an 80 x 80
// plane: 50 against 60; a step of 80x80x300, forward and reverse, 473 -> 402 us).
static int tile_width(const StepArgs &a) { return tile_columns(a, 16) < tile_columns(a, 32) ? 16 : 32; }

// Planes a block of the collide adjoint marches: the length with the least estimated time.  A plane
// takes 3.8 us where a block has an SM to itself and 6.0 us where three share it; starting a block
// costs a tenth of a plane (the others on the SM hide it).  Step of 64x64x256 by length: 1 248 us, 5
// 259, 10 251, 19 (chosen) 249, 32 327; of 25x23x60: 1 (chosen) 50, 2 56, 5 65.
static int adj_chunk(const StepArgs &a, int tx) {
    const long long cols = tile_columns(a, tx), slots = 3 * 152;
    auto us = [&](long long blocks, int len) {
        const long long r = blocks % slots;
        return ((float)(blocks / slots) * 6.0f + (r ? 3.8f + 2.2f * (float)r / (float)slots : 0.0f)) * ((float)len + 0.1f);
    };
    int best = 1;
    float cost = 1e30f;
    for (int len = 1; len <= a.nz && len <= 64; ++len) {
        const long long full = cols * (a.nz / len);
        const int rest = a.nz % len;  // the last chunk; alongside the others where slots are left
        const float t = us(full, len) + (rest && full % slots + cols > slots ? us(cols, rest) : 0.0f);
        if (t < 0.985f * cost) { cost = t; best = len; }  // the shorter where it makes no difference
    }
    return best;
}

template <bool kForce, bool W, int TX>
static cudaError_t launch_adj_collide(const StepArgs &a, const AdjArgs &g, cudaStream_t s) {
    auto *fn = adj_collide_kernel<kForce, W, TX>;
    const int smem = (int)sizeof(AdjSmem<TX>), chunk = adj_chunk(a, TX);
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const dim3 gr((a.nx + TX - 1) / TX, (a.ny + 128 / TX - 1) / (128 / TX), (a.nz + chunk - 1) / chunk);
    launch_chained(fn, gr, dim3(128, 1, 1), smem, s, a, g, chunk);
    return cudaSuccess;
}
template <int TX>
static cudaError_t launch_adj_collide(const StepArgs &a, const AdjArgs &g, bool force, bool walls, cudaStream_t s) {
    return force ? (walls ? launch_adj_collide<true, true, TX>(a, g, s) : launch_adj_collide<true, false, TX>(a, g, s))
                 : (walls ? launch_adj_collide<false, true, TX>(a, g, s) : launch_adj_collide<false, false, TX>(a, g, s));
}

// Grid of the stencil: a thread marches the longest chunk of 16, 8, 4, 2, 1 planes that leaves five
// blocks an SM (a chunk reads two planes more than it writes).  Whole step of 64x64x256 by length: 1 245
// us, 4 232, 8 (chosen) 231, 16 247; of 41x38x90: 1 (chosen) 77.5, 2 76.4, 4 79.5, 16 99.8.
struct StencilGrid {
    dim3 grid, block;
    int chunk;
    explicit StencilGrid(const StepArgs &a) : chunk(16) {
        const int tx = tile_width(a), ty = 128 / tx;
        while (chunk > 1 && tile_columns(a, tx) * ((a.nz + chunk - 1) / chunk) < 5 * 152) chunk /= 2;
        block = dim3(tx, ty, 1);
        grid = dim3((a.nx + tx - 1) / tx, (a.ny + ty - 1) / ty, (a.nz + chunk - 1) / chunk);
    }
};

cudaError_t launch_adjoint_step(const StepArgs &a, const AdjArgs &g, cudaStream_t s, long long *launches) {
    const bool force = a.gx != 0.0f || a.gy != 0.0f || a.gz != 0.0f;
    const bool walls = a.wall_x || a.wall_y;
    const cudaError_t e = tile_width(a) == 16 ? launch_adj_collide<16>(a, g, force, walls, s) : launch_adj_collide<32>(a, g, force, walls, s);
    if (e != cudaSuccess) return e;
    const StencilGrid sg(a);
    launch_chained(walls ? adj_stencil_kernel<true> : adj_stencil_kernel<false>, sg.grid, sg.block, 0, s, a, g, sg.chunk);
    *launches += 2;
    if (a.bc_zlo == BC_INLET || a.bc_zhi == BC_CONVECTIVE) {
        launch_chained(adj_boundary_kernel, dim3(col_grid(a).x, 2), col_block(), 0, s, a, g);
        *launches += 1;
    }
    return cudaGetLastError();
}

static int stride_grid(long long n) {
    long long b = (n + 255) / 256;
    return (int)std::min<long long>(std::max<long long>(b, 1), 152ll * 32);
}

cudaError_t launch_objective(const StepArgs &a, const AdjArgs &g, int objective, const double *args, float2 *ph,
                             float2 *lr_obj, double *acc_obj, double *scalar, cudaStream_t s, long long *launches) {
    const long long nblk = adj_collide_blocks(a);
    obj_fields_kernel<<<stride_grid(a.NN), 256, 0, s>>>(a, ph);
    *launches += 1;
    if (objective == 0) {  // interface area
        AdjArgs o = g;
        o.lr_out = lr_obj;
        StepArgs ao = a;
        ao.phase = ph;
        const float eps = (float)args[0];
        obj_area_kernel<<<node_grid(a), node_block(), 0, s>>>(a, ph, g.lga, g.lgb, acc_obj, eps * eps);
        const StencilGrid sg(a);
        (a.wall_x || a.wall_y ? adj_stencil_kernel<true> : adj_stencil_kernel<false>)<<<sg.grid, sg.block, 0, s>>>(ao, o, sg.chunk);
        adj_reduce_kernel<<<1, 1024, 0, s>>>(acc_obj, nblk, 1, 0, scalar);
        *launches += 3;
    } else {  // penetration length
        const double delta = args[0];
        obj_pen_sum_kernel<<<node_grid(a), node_block(), 0, s>>>(a, ph, acc_obj, (float)(1.0 / delta));
        adj_reduce_kernel<<<1, 1024, 0, s>>>(acc_obj, nblk, 1, 0, scalar + 1);
        obj_pen_value_kernel<<<1, 32, 0, s>>>(scalar + 1, scalar, (double)(a.nz - 1), delta);
        obj_pen_adjoint_kernel<<<stride_grid(a.NN), 256, 0, s>>>(a, ph, scalar + 1, lr_obj, (float)(1.0 / delta), (float)delta);
        *launches += 4;
    }
    return cudaGetLastError();
}

cudaError_t launch_adjoint_reduce(const AdjArgs &g, long long nblk_coll, long long nblk_inlet, double *out,
                                  cudaStream_t s, long long *launches) {
    // out[1] = u_in, out[2..4] = sigma, nu_r, nu_b, out[5..20] = a_1, b_1, ..., a_8, b_8
    adj_reduce_kernel<<<1, 1024, 0, s>>>(g.acc_inlet, nblk_inlet, 17, 0, out + 1);
    adj_reduce_kernel<<<3, 1024, 0, s>>>(g.acc_coll, nblk_coll, 3, 0, out + 2);
    adj_reduce_kernel<<<16, 1024, 0, s>>>(g.acc_inlet, nblk_inlet, 17, 1, out + 5);
    *launches += 3;
    return cudaGetLastError();
}

cudaError_t launch_adjoint_state(const StepArgs &a, const AdjArgs &g, float *out, cudaStream_t s, long long *launches) {
    adj_state_kernel<<<stride_grid(a.NN), 256, 0, s>>>(a, g, out);
    *launches += 1;
    return cudaGetLastError();
}

}  // namespace lbcm
