// lbcm_collide.cuh -- collision, perturbation and recolouring of one node with the paper's rates
// s3 = s4 = s5 = s6 = 1 (arXiv:1804.08923, Section II), from the node's moments and the
// gradients of phi and rho.
//
// The kernels that use it (collide_kernel and step_kernel of lbcm_step.cu, advance_kernel of
// lbcm_advance.cu) have to give the same bits: a population that one block rebuilds for its halo
// is the one its owner accounts for.  Their translation units are therefore compiled without
// contraction (-fmad=false), and every fused multiply-add is written out.
#pragma once
#include "lbcm_node.cuh"

namespace lbcm {

// 1/x and 1/sqrt(x) of normal positive x: the hardware approximation and one Newton step in FMA
// arithmetic, three and five instructions where the IEEE forms take about ten, with a branch for the
// special cases.  Over every mantissa 1/x is the IEEE division's result; 1/sqrt(x) is off by at most 1
// ulp, 0.33 rms (a division by the square root: 1.49 and 0.43).
__device__ __forceinline__ float rcp_newton(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ float rsqrt_newton(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(0.5f * r, fmaf(-(x * r), r, 1.0f), r);
}

// a - b in one packed instruction (the product by -1 is exact)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }

// Isotropic gradients of phi (.x) and rho (.y) (end of Section II): 3 sum_j w_j chi(x + c_j) c_j.
// at(j) is (phi, rho) of the neighbour x + c_j.  Opposite neighbours are subtracted first, so that
// a uniform field gives exactly zero and nearby values subtract exactly; the differences are
// summed by speed class, both fields at once in packed arithmetic (each lane rounds as a scalar).
template <class L>
__device__ __forceinline__ void gradients(L &&at, float2 &gx, float2 &gy, float2 &gz) {
    auto d = [&](int j) { return sub2(at(j), at(j + 1)); };  // c_{j+1} = -c_j
    const float2 ax = d(1), ay = d(3), az = d(5);
    const float2 d7 = d(7), d9 = d(9), d11 = d(11), d13 = d(13), d15 = d(15), d17 = d(17);
    const float2 fx = __fadd2_rn(__fadd2_rn(d7, d9), __fadd2_rn(d15, d17));    // (1,1,0) (1,-1,0) (1,0,1) (1,0,-1)
    const float2 fy = __fadd2_rn(sub2(d7, d9), __fadd2_rn(d11, d13));          // (0,1,1) (0,1,-1)
    const float2 fz = __fadd2_rn(sub2(d11, d13), sub2(d15, d17));
    const float2 d19 = d(19), d21 = d(21), d23 = d(23), d25 = d(25);  // (1,1,1) (1,1,-1) (1,-1,1) (-1,1,1)
    const float2 p = __fadd2_rn(d19, d21), q = sub2(d23, d25);
    const float2 kx = __fadd2_rn(p, q), ky = sub2(p, q);
    const float2 kz = __fadd2_rn(sub2(d19, d21), __fadd2_rn(d23, d25));
    constexpr float w1 = 6.0f / 27.0f, w2 = 3.0f / 54.0f, w3 = 3.0f / 216.0f;
    const float2 W1 = make_float2(w1, w1), W2 = make_float2(w2, w2), W3 = make_float2(w3, w3);
    gx = __ffma2_rn(W1, ax, __ffma2_rn(W2, fx, __fmul2_rn(W3, kx)));
    gy = __ffma2_rn(W1, ay, __ffma2_rn(W2, fy, __fmul2_rn(W3, ky)));
    gz = __ffma2_rn(W1, az, __ffma2_rn(W2, fz, __fmul2_rn(W3, kz)));
}

// One axis of the inverse transform of second-order central moments about u, on half values:
// from half the moments (m0, m1, m2) of a line, half of t = u^2 m0 + 2 u m1 + m2 and of
// o = u m0 + m1 give the values v(+1) = (t + o)/2, v(-1) = (t - o)/2, v(0) = m0 - t.
struct Axis {
    float u, u2, uu;
    __device__ __forceinline__ explicit Axis(float v) : u(v), u2(2.0f * v), uu(v * v) {}
};

// The collision of one node, up to the evaluation of single directions.
//
// Every term but the recolouring's 1/|c_i| and the relaxed second moment is w_i times a polynomial
// in c_i for i >= 1: varphi_i(alpha) = (27/19) w_i (1 - alpha), Phi_i = 9 w_i nu (c_i.u)(c_i.grad
// rho), B_i = w_i.  So the even part of a pair of opposite directions is w_i (C0 + c_i^T Q c_i)
// with one symmetric Q per node, and the odd part w_i (c_i.u)(lb + ld (c_i.u)^2) (+ the force).  The
// relaxed second moment K goes through the inverse central-moment transform about u by 1-D
// sweeps (K has no moments of order 0 and 1: those of f - f^e + F'/2 vanish).
//
// Reversing the sign of one component of every vector and tensor reverses that component of c_i in the
// result and nothing else, bit for bit: products and sums only change sign.  The halo versions below
// rest on it.
template <bool kForce>
struct Collision {
    float rho_r, rho_b, rho, ux, uy, uz, Fx, Fy, Fz, gpx, gpy, gpz;
    float C0, qxx, qyy, qzz, qxy, qxz, qyz, lb, ld, frac_r, frac_b, sg1, sg2, sg3;
    float V00[3], V10[3], V01[3], V20[3], V02[3], V11[3];  // [c_z + 1], moments (p, q) in (x, y), half values

    // ax, ay, az: gravity
    __device__ __forceinline__ Collision(const StepArgs &a, const Moments &mo, float2 gx, float2 gy, float2 gz, float ax,
                                         float ay, float az) {
        gpx = gx.x; gpy = gy.x; gpz = gz.x;
        const float grx = gx.y, gry = gy.y, grz = gz.y;
        rho_r = mo.rho_r;
        rho_b = mo.rho_b;
        // macroscopic quantities (Eqs. (13), (48), (23)) and mixture parameters
        rho = mo.rho_r + mo.rho_b;
        const float inv_rho = rcp_newton(rho);
        Fx = Fy = Fz = 0.0f;
        if (kForce) {
            const float fo = rho - a.rho_b0;
            Fx = fo * ax; Fy = fo * ay; Fz = fo * az;
        }
        ux = (kForce ? fmaf(0.5f, Fx, mo.jx) : mo.jx) * inv_rho;
        uy = (kForce ? fmaf(0.5f, Fy, mo.jy) : mo.jy) * inv_rho;
        uz = (kForce ? fmaf(0.5f, Fz, mo.jz) : mo.jz) * inv_rho;
        const float hp = fmaf(0.5f, mo.phi, 0.5f), hm = fmaf(-0.5f, mo.phi, 0.5f);
        const float oma = a.alpha_mix ? fmaf(mo.rho_r, a.oma_r, mo.rho_b * a.oma_b) * inv_rho : fmaf(hp, a.oma_r, hm * a.oma_b);
        const float nu = rcp_newton(fmaf(hp, a.inv_nu_r, hm * a.inv_nu_b));
        const float s2nu = rcp_newton(fmaf(3.0f, nu, 0.5f));  // 1/tau
        const float usq = fmaf(ux, ux, fmaf(uy, uy, uz * uz));
        const float g2 = fmaf(gpx, gpx, fmaf(gpy, gpy, gpz * gpz));
        const float inv_gm = rsqrt_newton(fmaxf(g2 + a.eps2, 1.1754944e-38f));  // 1/|grad phi|_eps, a normal number
        const float pert = (2.25f * a.sigma) * s2nu * inv_gm;  // A / |grad phi|, A = 9 sigma / (4 tau)

        // S = rho u u + nu (u g + g u), the anisotropic second moment of f^e; Fh = (u F + F u) / 2
        const float rux = rho * ux, ruy = rho * uy, ruz = rho * uz;
        float Sxx = fmaf(rux, ux, nu * (2.0f * ux * grx)), Syy = fmaf(ruy, uy, nu * (2.0f * uy * gry)),
              Szz = fmaf(ruz, uz, nu * (2.0f * uz * grz));
        float Sxy = fmaf(rux, uy, nu * fmaf(ux, gry, uy * grx)), Sxz = fmaf(rux, uz, nu * fmaf(ux, grz, uz * grx)),
              Syz = fmaf(ruy, uz, nu * fmaf(uy, grz, uz * gry));
        // second central moments of Delta = f - f^e + F'/2, without the isotropic part of f^e
        float uF = 0.0f;
        float Txx = Sxx, Tyy = Syy, Tzz = Szz, Txy = Sxy, Txz = Sxz, Tyz = Syz;  // what Delta takes off Pi(f)
        if (kForce) {
            uF = fmaf(ux, Fx, fmaf(uy, Fy, uz * Fz));
            const float hxx = ux * Fx, hyy = uy * Fy, hzz = uz * Fz;
            const float hxy = 0.5f * fmaf(ux, Fy, uy * Fx), hxz = 0.5f * fmaf(ux, Fz, uz * Fx), hyz = 0.5f * fmaf(uy, Fz, uz * Fy);
            Txx -= hxx; Tyy -= hyy; Tzz -= hzz; Txy -= hxy; Txz -= hxz; Tyz -= hyz;
            Sxx += hxx; Syy += hyy; Szz += hzz; Sxy += hxy; Sxz += hxz; Syz += hyz;
        }
        // K: shear part with 1 - 1/tau, trace with 1 - s2b (0 with the paper's s2b = 1); halved
        const float o2 = 1.0f - s2nu, h2 = 0.5f * o2, t3 = (0.5f / 3.0f) * o2;
        const float k110 = h2 * (mo.pxy - Txy), k101 = h2 * (mo.pxz - Txz), k011 = h2 * (mo.pyz - Tyz);
        const float e1 = t3 * (mo.dxz - (Txx - Tzz)), e2 = t3 * (mo.dyz - (Tyy - Tzz));
        float k200 = fmaf(2.0f, e1, -e2), k020 = fmaf(2.0f, e2, -e1), k002 = -(e1 + e2);
        if (a.s2b != 1.0f) {
            const float ugr = fmaf(ux, grx, fmaf(uy, gry, uz * grz));
            const float iso = fmaf(rho * oma, 9.0f / 19.0f, nu * ugr);
            const float tr = (fmaf(3.0f, mo.pzz, mo.dxz + mo.dyz) - ((Txx + Tyy) + Tzz)) - 3.0f * iso;
            const float t = (0.5f / 3.0f) * (1.0f - a.s2b) * tr;
            k200 += t; k020 += t; k002 += t;
        }

        // even part of the pairs: C0 + c^T Q c (off-diagonal entries doubled)
        C0 = fmaf(rho * oma, 27.0f / 19.0f, fmaf(-1.5f * rho, usq, fmaf(-pert, g2, -1.5f * uF)));
        const float px = pert * gpx, py = pert * gpy;
        qxx = fmaf(4.5f, Sxx, px * gpx); qyy = fmaf(4.5f, Syy, py * gpy); qzz = fmaf(4.5f, Szz, pert * gpz * gpz);
        qxy = fmaf(9.0f, Sxy, 2.0f * px * gpy); qxz = fmaf(9.0f, Sxz, 2.0f * px * gpz); qyz = fmaf(9.0f, Syz, 2.0f * py * gpz);
        // odd part: (c.u) (lb + ld (c.u)^2) + 3/2 c.F
        lb = rho * fmaf(-4.5f, usq, 3.0f);
        ld = 4.5f * rho;
        // recolouring: +- seg_i, seg_i = w_i/|c_i| seg0 (c_i.grad phi), seg0 = beta rho_r rho_b (27/19)
        // (1 - alpha) / (rho |grad phi|)
        frac_r = mo.rho_r * inv_rho;
        frac_b = mo.rho_b * inv_rho;
        const float seg0 = a.beta * mo.rho_r * frac_b * inv_gm * (oma * (27.0f / 19.0f));
        sg1 = (2.0f / 27.0f) * seg0;
        sg2 = (float)(0.70710678118654752 / 54.0) * seg0;
        sg3 = (float)(0.57735026918962576 / 216.0) * seg0;
        // inverse transform, z sweep; a line that has one moment only, of order 0, 1 or 2
        const Axis Z(uz);
        auto line0 = [&](float m0, float (&v)[3]) {
            const float t = Z.uu * m0, o = Z.u * m0;
            v[0] = 0.5f * (t - o); v[1] = m0 - t; v[2] = 0.5f * (t + o);
        };
        auto line1 = [&](float m1, float (&v)[3]) {
            const float t = Z.u2 * m1;
            v[0] = 0.5f * (t - m1); v[1] = -t; v[2] = 0.5f * (t + m1);
        };
        V00[0] = 0.5f * k002; V00[1] = -k002; V00[2] = 0.5f * k002;
        line1(k101, V10);
        line1(k011, V01);
        line0(k200, V20);
        line0(k020, V02);
        line0(k110, V11);
    }

    // y sweep of the plane c = c_z + 1: half the moments of order 0, 1, 2 in x of the line c_y = b - 1
    __device__ __forceinline__ void yline(const Axis &Y, int c, float (&W0)[3], float (&W1)[3], float (&W2)[3]) const {
        {
            const float t = fmaf(Y.uu, V00[c], fmaf(Y.u2, V01[c], V02[c])), o = fmaf(Y.u, V00[c], V01[c]);
            W0[0] = 0.5f * (t - o); W0[1] = V00[c] - t; W0[2] = 0.5f * (t + o);
        }
        {
            const float t = fmaf(Y.uu, V10[c], Y.u2 * V11[c]), o = fmaf(Y.u, V10[c], V11[c]);
            W1[0] = 0.5f * (t - o); W1[1] = V10[c] - t; W1[2] = 0.5f * (t + o);
        }
        {
            const float t = Y.uu * V20[c], o = Y.u * V20[c];
            W2[0] = 0.5f * (t - o); W2[1] = V20[c] - t; W2[2] = 0.5f * (t + o);
        }
    }
    // x sweep of a line: the values of K at c_x = -1, 0, +1
    static __device__ __forceinline__ void xline(const Axis &X, float w0, float w1, float w2, float &vm, float &v0, float &vp) {
        const float t = fmaf(X.uu, w0, fmaf(X.u2, w1, w2)), o = fmaf(X.u, w0, w1);
        vm = t - o;
        vp = t + o;
        v0 = 2.0f * (w0 - t);
    }
    __device__ __forceinline__ float odd(float cu, float cF) const {
        const float p = fmaf(ld, cu * cu, lb);
        return kForce ? fmaf(p, cu, 1.5f * cF) : p * cu;
    }
    // the first (kSecond = false) or second direction of an opposite pair, of the class of i
    template <bool kSecond>
    __device__ __forceinline__ float2 one(int i, float ev, float cu, float cF, float cgp, float sg, float r) const {
        const float od = odd(cu, cF), seg = sg * cgp;
        // One rounding at the population's size, where ev + od would be rounded at that of rho.  Distance
        // of u after one step from double precision, against a collision that adds even and odd part by
        // direction, mean of seven scenes: 0.88 (0.97 with ev + od; 1.2 to 1.3 on a static droplet, whose
        // velocities are below FP32 resolution either way).
        const float s = fmaf(wgt(i), ev, fmaf(wgt(i), kSecond ? -od : od, r));
        return kSecond ? make_float2(fmaf(frac_r, s, -seg), fmaf(frac_b, s, seg))
                       : make_float2(fmaf(frac_r, s, seg), fmaf(frac_b, s, -seg));
    }
};

// emit(i, f) stores the populations (red, blue) f of direction i and returns them as they will be
// read back (with a half-precision storage, rounded); the mass of the moving ones is summed from
// those, in the association of z_class / finish_moments (lbcm_node.cuh), so that the reader of an
// unchanged set gets the node's colour densities back exactly.
// ready() is called once, when the moments have been used and nothing has been emitted yet.
template <bool kForce, class E, class R>
__device__ __forceinline__ void collide_node(const StepArgs &a, const Moments &mo, float2 gx, float2 gy, float2 gz,
                                             E &&emit, R &&ready) {
    const Collision<kForce> q(a, mo, gx, gy, gz, a.gx, a.gy, a.gz);
    ready();
    const Axis X(q.ux), Y(q.uy);
    float W0[3][3], W1[3][3], W2[3][3];  // [c_z + 1][c_y + 1]
#pragma unroll
    for (int c = 0; c < 3; ++c) q.yline(Y, c, W0[c], W1[c], W2[c]);
    auto xline = [&](int b, int c, float &vm, float &v0, float &vp) { q.xline(X, W0[c][b], W1[c][b], W2[c][b], vm, v0, vp); };
    auto pair = [&](int i, int j, float ev, float cu, float cF, float cgp, float sg, float ri, float rj, float2 &fi,
                    float2 &fj) {
        fi = emit(i, q.template one<false>(i, ev, cu, cF, cgp, sg, ri));
        fj = emit(j, q.template one<true>(i, ev, cu, cF, cgp, sg, rj));
    };
    const float cx0 = q.C0 + q.qxx, cy0 = q.C0 + q.qyy, cz0 = q.C0 + q.qzz;
    const float exy = cx0 + q.qyy, exz = cx0 + q.qzz, eyz = cy0 + q.qzz, exyz = exy + q.qzz;
    const float ux = q.ux, uy = q.uy, uz = q.uz, Fx = q.Fx, Fy = q.Fy, Fz = q.Fz, gpx = q.gpx, gpy = q.gpy, gpz = q.gpz;
    const float qxy = q.qxy, qxz = q.qxz, qyz = q.qyz, sg1 = q.sg1, sg2 = q.sg2, sg3 = q.sg3;

    auto add = [](float2 &acc, float2 v) { acc = __fadd2_rn(acc, v); };
    float2 s0, sp, sm;  // masses of the moving populations by c_z = 0, +1, -1, each a running sum (z_class)
    float m_, z_, p_, n_, y_, q_;
    // line (0, 0): +-x; lines (+-1, 0): +-y and the xy diagonals
    const float uxy = ux + uy, vxy = ux - uy, gxy = gpx + gpy, hxy = gpx - gpy;
    const float Fxy = Fx + Fy, Hxy = Fx - Fy;
    {
        float2 f1, f2, f4, f7, f8, f9, f10;
        xline(1, 1, m_, z_, p_);
        pair(1, 2, cx0, ux, Fx, gpx, sg1, p_, m_, f1, f2);
        xline(2, 1, m_, z_, p_);
        xline(0, 1, n_, y_, q_);
        pair(3, 4, cy0, uy, Fy, gpy, sg1, z_, y_, s0, f4);
        add(s0, f1); add(s0, f4); add(s0, f2);
        pair(7, 8, exy + qxy, uxy, Fxy, gxy, sg2, p_, n_, f7, f8);
        pair(9, 10, exy - qxy, vxy, Hxy, hxy, sg2, q_, m_, f9, f10);
        add(s0, f7); add(s0, f9); add(s0, f8); add(s0, f10);
    }
    // lines (0, +-1): +-z and the xz diagonals
    float2 f15, f16, f17, f18;
    xline(1, 2, m_, z_, p_);
    xline(1, 0, n_, y_, q_);
    pair(5, 6, cz0, uz, Fz, gpz, sg1, z_, y_, sp, sm);
    pair(15, 16, exz + qxz, ux + uz, Fx + Fz, gpx + gpz, sg2, p_, n_, f15, f16);
    pair(17, 18, exz - qxz, ux - uz, Fx - Fz, gpx - gpz, sg2, q_, m_, f17, f18);
    // lines (1, 1) / (-1, -1) and (1, -1) / (-1, 1): the yz diagonals and the corners
    const float qp = qxy + qxz, qm = qxy - qxz;
    float2 f11, f12, f13, f14, f19, f20, f21, f22, f23, f24, f25, f26;
    xline(2, 2, m_, z_, p_);
    xline(0, 0, n_, y_, q_);
    pair(11, 12, eyz + qyz, uy + uz, Fy + Fz, gpy + gpz, sg2, z_, y_, f11, f12);
    add(sp, f11); add(sp, f15);
    pair(19, 20, exyz + (qp + qyz), uxy + uz, Fxy + Fz, gxy + gpz, sg3, p_, n_, f19, f20);
    pair(25, 26, exyz + (qyz - qp), uz - vxy, Fz - Hxy, gpz - hxy, sg3, m_, q_, f25, f26);
    xline(2, 0, m_, z_, p_);
    xline(0, 2, n_, y_, q_);
    pair(13, 14, eyz - qyz, uy - uz, Fy - Fz, gpy - gpz, sg2, z_, y_, f13, f14);
    add(sm, f13); add(sm, f17); add(sm, f12); add(sm, f16);
    add(sp, f14); add(sp, f18); add(sp, f19);
    pair(21, 22, exyz + (qm - qyz), uxy - uz, Fxy - Fz, gxy - gpz, sg3, p_, n_, f21, f22);
    pair(23, 24, exyz - (qm + qyz), vxy + uz, Hxy + Fz, hxy + gpz, sg3, q_, m_, f23, f24);
    add(sm, f21); add(sm, f26); add(sm, f20); add(sm, f24);
    add(sp, f23); add(sp, f22); add(sp, f25);
    const float2 s = __fadd2_rn(__fadd2_rn(s0, sp), sm);
    // Rest direction.  In exact arithmetic the step keeps each colour's mass at this node
    // (sum_i f_i^k* = rho_k), so the rest population is that mass minus the moving ones as
    // they will be read back; this equals Eqs. (33), (34) for i = 0 and keeps the FP32 rounding
    // of the lattice constants and any storage rounding from drifting the colour masses.
    emit(0, make_float2(q.rho_r - s.x, q.rho_b - s.y));
}

// The populations of a halo node that enter the tile beside it, put(i, f) for each of the nine: those
// with c_y = +1 (halo_y) or c_x = +1 (halo_x) of the node mirrored in that axis when s = -1, that is,
// the node's own ones with c_y (c_x) = s, direction i mirrored.
template <bool kForce, class E, class R>
__device__ __forceinline__ void collide_halo_y(const StepArgs &a, Moments mo, float2 gx, float2 gy, float2 gz, float s,
                                               E &&put, R &&ready) {
    mo.jy *= s; mo.pxy *= s; mo.pyz *= s;
    const Collision<kForce> q(a, mo, gx, make_float2(s * gy.x, s * gy.y), gz, a.gx, s * a.gy, a.gz);
    ready();
    const Axis X(q.ux), Y(q.uy);
    float W0[3], W1[3], W2[3];
    float m_, z_, p_;
    const float cy0 = q.C0 + q.qyy, exy = (q.C0 + q.qxx) + q.qyy, eyz = cy0 + q.qzz, exyz = exy + q.qzz;
    const float uxy = q.ux + q.uy, vxy = q.ux - q.uy, gxy = q.gpx + q.gpy, hxy = q.gpx - q.gpy, Fxy = q.Fx + q.Fy, Hxy = q.Fx - q.Fy;
    const float qp = q.qxy + q.qxz, qm = q.qxy - q.qxz;
    q.yline(Y, 1, W0, W1, W2);
    q.xline(X, W0[2], W1[2], W2[2], m_, z_, p_);
    put(3, q.template one<false>(3, cy0, q.uy, q.Fy, q.gpy, q.sg1, z_));
    put(7, q.template one<false>(7, exy + q.qxy, uxy, Fxy, gxy, q.sg2, p_));
    put(10, q.template one<true>(9, exy - q.qxy, vxy, Hxy, hxy, q.sg2, m_));
    q.yline(Y, 2, W0, W1, W2);
    q.xline(X, W0[2], W1[2], W2[2], m_, z_, p_);
    put(11, q.template one<false>(11, eyz + q.qyz, q.uy + q.uz, q.Fy + q.Fz, q.gpy + q.gpz, q.sg2, z_));
    put(19, q.template one<false>(19, exyz + (qp + q.qyz), uxy + q.uz, Fxy + q.Fz, gxy + q.gpz, q.sg3, p_));
    put(25, q.template one<false>(25, exyz + (q.qyz - qp), q.uz - vxy, q.Fz - Hxy, q.gpz - hxy, q.sg3, m_));
    q.yline(Y, 0, W0, W1, W2);
    q.xline(X, W0[2], W1[2], W2[2], m_, z_, p_);
    put(13, q.template one<false>(13, eyz - q.qyz, q.uy - q.uz, q.Fy - q.Fz, q.gpy - q.gpz, q.sg2, z_));
    put(21, q.template one<false>(21, exyz + (qm - q.qyz), uxy - q.uz, Fxy - q.Fz, gxy - q.gpz, q.sg3, p_));
    put(24, q.template one<true>(23, exyz - (qm + q.qyz), vxy + q.uz, Hxy + q.Fz, hxy + q.gpz, q.sg3, m_));
}
template <bool kForce, class E, class R>
__device__ __forceinline__ void collide_halo_x(const StepArgs &a, Moments mo, float2 gx, float2 gy, float2 gz, float s,
                                               E &&put, R &&ready) {
    mo.jx *= s; mo.pxy *= s; mo.pxz *= s;
    const Collision<kForce> q(a, mo, make_float2(s * gx.x, s * gx.y), gy, gz, s * a.gx, a.gy, a.gz);
    ready();
    const Axis X(q.ux), Y(q.uy);
    float W0[3], W1[3], W2[3];
    const float cx0 = q.C0 + q.qxx, exy = cx0 + q.qyy, exz = cx0 + q.qzz, exyz = exy + q.qzz;
    const float uxy = q.ux + q.uy, vxy = q.ux - q.uy, gxy = q.gpx + q.gpy, hxy = q.gpx - q.gpy, Fxy = q.Fx + q.Fy, Hxy = q.Fx - q.Fy;
    const float qp = q.qxy + q.qxz, qm = q.qxy - q.qxz;
    q.yline(Y, 1, W0, W1, W2);
    auto xplus = [&](int b) {
        float m_, z_, p_;
        q.xline(X, W0[b], W1[b], W2[b], m_, z_, p_);
        return p_;
    };
    put(1, q.template one<false>(1, cx0, q.ux, q.Fx, q.gpx, q.sg1, xplus(1)));
    put(7, q.template one<false>(7, exy + q.qxy, uxy, Fxy, gxy, q.sg2, xplus(2)));
    put(9, q.template one<false>(9, exy - q.qxy, vxy, Hxy, hxy, q.sg2, xplus(0)));
    q.yline(Y, 2, W0, W1, W2);
    put(15, q.template one<false>(15, exz + q.qxz, q.ux + q.uz, q.Fx + q.Fz, q.gpx + q.gpz, q.sg2, xplus(1)));
    put(19, q.template one<false>(19, exyz + (qp + q.qyz), uxy + q.uz, Fxy + q.Fz, gxy + q.gpz, q.sg3, xplus(2)));
    put(23, q.template one<false>(23, exyz - (qm + q.qyz), vxy + q.uz, Hxy + q.Fz, hxy + q.gpz, q.sg3, xplus(0)));
    q.yline(Y, 0, W0, W1, W2);
    put(17, q.template one<false>(17, exz - q.qxz, q.ux - q.uz, q.Fx - q.Fz, q.gpx - q.gpz, q.sg2, xplus(1)));
    put(21, q.template one<false>(21, exyz + (qm - q.qyz), uxy - q.uz, Fxy - q.Fz, gxy - q.gpz, q.sg3, xplus(2)));
    put(26, q.template one<true>(25, exyz + (q.qyz - qp), q.uz - vxy, q.Fz - Hxy, q.gpz - hxy, q.sg3, xplus(0)));
}

}  // namespace lbcm
