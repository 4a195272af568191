// lbcm_node.cuh -- per-node pieces shared by the forward step and its adjoint: the
// pull gather of the post-stream populations, the isotropic gradient stencil, the moments
// the paper-rate collision needs and the inverse 1-D central-moment sweep coefficients
// (arXiv:1804.08923, Section II).
#pragma once
#include "lbcm_device.cuh"

namespace lbcm {

// Direction i of the gather: the boundary planes at z = 0 / z = N, else the pull from the
// source node, reading the populations of direction j there.  With the fitted FP16 encoding
// the pull is loaded and decoded unconditionally (the source offsets are clamped onto the
// lattice, so the address is valid on the boundary planes too) and the boundary value replaces
// it afterwards: with the load inside the branch, the long decoding kept real branches around
// each load, which then could not be issued together (the phase-field pass ran 3x slower).
// The other storages keep the load inside the branch, which measured faster for them.
template <int S>
__device__ __forceinline__ void gather_one(const StepArgs &a, const Nbr &nb, int i, bool lo, bool slip_hi, size_t P,
                                           const Own &own, int j, float (&fr)[27], float (&fb)[27]) {
    if constexpr (S == STORE_FP16_FIT) {
        const float2 v = load_pop<S>(a, i, nb.src(i), own, j);
        fr[i] = v.x;
        fb[i] = v.y;
    }
    if (cz(i) == 1 && lo) {
        fr[i] = a.zin[zrank(i) * P + nb.pxy];
        fb[i] = a.zin[(9 + zrank(i)) * P + nb.pxy];
    } else if (cz(i) == -1 && slip_hi) {
        fr[i] = a.zout[zrank(i) * P + nb.pxy];
        fb[i] = a.zout[(9 + zrank(i)) * P + nb.pxy];
    } else if constexpr (S != STORE_FP16_FIT) {
        const float2 v = load_pop<S>(a, i, nb.src(i), own, j);
        fr[i] = v.x;
        fb[i] = v.y;
    }
}

// Post-stream populations of node (x, y, z) (Eq. (9), pull form) with the boundary
// planes of this step substituted.  Branches are uniform across a warp (one z per warp).
// kEdge = false: the caller knows that 0 < z < nz - 1, and the boundary-plane tests of every
// direction drop out of the code.
template <int S, bool W, bool kEdge = true>
__device__ __forceinline__ void gather(const StepArgs &a, const Nbr &nb, int z, float (&fr)[27], float (&fb)[27]) {
    const size_t P = (size_t)a.plane;
    const int N = a.nz - 1;
    const bool periodic_z = a.bc_zlo == BC_PERIODIC;
    const bool lo = kEdge && (z == 0) && !periodic_z;
    const bool conv = kEdge && (z == N) && a.bc_zhi == BC_CONVECTIVE;
    const bool slip_hi = kEdge && (z == N) && a.bc_zhi == BC_FREESLIP;
    if (conv) {
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            fr[i] = a.hist_out[i * P + nb.pxy];
            fb[i] = a.hist_out[(27 + i) * P + nb.pxy];
        }
        return;
    }
    const Own own = reader_shift<S>(a, nb.n);
    // W: the lattice has side walls, where a pull reflects (the direction leaving the source is
    // nb.pulled(i), selected at run time).  Only warps holding a wall node take that path; the
    // others, and lattices without side walls, index every plane at compile time.
    bool reflect = false;
    if constexpr (W) reflect = __any_sync(__activemask(), nb.wxl || nb.wxh || nb.wyl || nb.wyh);
    if (reflect) {
        if constexpr (S == STORE_FP16_FIT) {
            const OwnFlip of = flip_own(own, nb.wxl, nb.wxh, nb.wyl, nb.wyh);
#pragma unroll
            for (int i = 0; i < 27; ++i) {
                const float2 v = load_pop_flip(a, i, nb.src(i), of, nb.pulled(i));
                fr[i] = v.x;
                fb[i] = v.y;
                if (cz(i) == 1 && lo) {
                    fr[i] = a.zin[zrank(i) * P + nb.pxy];
                    fb[i] = a.zin[(9 + zrank(i)) * P + nb.pxy];
                } else if (cz(i) == -1 && slip_hi) {
                    fr[i] = a.zout[zrank(i) * P + nb.pxy];
                    fb[i] = a.zout[(9 + zrank(i)) * P + nb.pxy];
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 27; ++i) gather_one<S>(a, nb, i, lo, slip_hi, P, own, nb.pulled(i), fr, fb);
        }
    } else if constexpr (S == STORE_FP16_FIT) {
        // opposite pulls (i, i+1) were both encoded for this node, with odd terms of opposite
        // sign: one odd sum and one odd product decode the pair
        const float2 *rest = reinterpret_cast<const float2 *>(a.pin);
        const __half2 *mov = reinterpret_cast<const __half2 *>(rest + a.NN);
        const float2 f0 = __ldg(rest + nb.src(0));
        fr[0] = f0.x;
        fb[0] = f0.y;
#pragma unroll
        for (int i = 1; i < 27; i += 2) {
            const float2 hp = __half22float2(__ldg(mov + (size_t)(i - 1) * a.NN + nb.src(i)));
            const float2 hm = __half22float2(__ldg(mov + (size_t)i * a.NN + nb.src(i + 1)));
            const __half2 e = fit_odd_h(a, i, odd_sum(i, own));
            const float2 pp = fit_pred_h(a, i, own.Ah, e), pm = fit_pred_h(a, i, own.Ah, __hneg2(e));
            fr[i] = fmaf(hp.x, a.inv_dev_scale, pp.x);
            fb[i] = fmaf(hp.y, a.inv_dev_scale, pp.y);
            fr[i + 1] = fmaf(hm.x, a.inv_dev_scale, pm.x);
            fb[i + 1] = fmaf(hm.y, a.inv_dev_scale, pm.y);
        }
#pragma unroll
        for (int i = 1; i < 27; ++i) {
            if (cz(i) == 1 && lo) {
                fr[i] = a.zin[zrank(i) * P + nb.pxy];
                fb[i] = a.zin[(9 + zrank(i)) * P + nb.pxy];
            } else if (cz(i) == -1 && slip_hi) {
                fr[i] = a.zout[zrank(i) * P + nb.pxy];
                fb[i] = a.zout[(9 + zrank(i)) * P + nb.pxy];
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < 27; ++i) gather_one<S>(a, nb, i, lo, slip_hi, P, own, i, fr, fb);
    }
}

// Moments of the post-stream populations of one node that the paper-rate collision needs:
// colour densities, order parameter, colour-blind momentum and raw second moment Pi, its diagonal as
// dxz = Pi_xx - Pi_zz, dyz = Pi_yy - Pi_zz and Pi_zz (the collision relaxes the differences, and the
// trace only with a bulk rate other than 1).
struct Moments {
    float rho_r, rho_b, phi, jx, jy, jz, dxz, dyz, pzz, pxy, pxz, pyz;
};

// The sums are taken by the three classes of c_z, each in one fixed order, so that a kernel that
// marches along z and meets the classes of a node one plane after another (advance_kernel) gives
// the same bits as one that holds all 27.  Within a class mirrored directions are subtracted
// before they are added up, and the differences dxz and dyz are taken class by class, so that a
// resting uniform node has exactly zero momentum and no second moment but its trace.  The axis
// population (a), the two pairs of faces (fx, fy) and the corners (k, with what the sums fx and fy
// rounded off) are kept apart until the classes c_z = +-1 are subtracted: their differences are nearly
// exact, where a class's sum is rounded at the size of the class.  Error of j_z of populations about
// equilibrium, against that of differences taken pair by pair: 0.96 so, 1.14 without the
// remainders in k, 1.64 with faces and corners added up in one sum, which made u_z after one step of a
// jet 1.27 times as far from double precision.  The colour masses of a class are one running sum: at
// a density ratio of 1000 a node's rest population holds all but 0.05% of its mass, FP32 resolves what
// moves only down to 6% of the Laplace jump, and how a droplet settles depends on the association
// (100^3, R = 25, 1e5 steps, jump off by 1.2% when all 13 pairs were added up in one sum, red and blue
// mass by -6e-5 and 1.3e-4; by 1.2%, -5e-5 and 3e-5 with this order, by 3.5% with balanced trees).
struct ZClass {
    float2 m;  // colour masses of the class's moving populations
    float a, fx, fy, k, X, Y, XY;
    __device__ __forceinline__ float b() const { return (fx + fy) + k; }
    // c_z = 0: the class's part of dxz, dyz; c_z = +-1: minus that part
    template <int cz>
    __device__ __forceinline__ float ex() const { return cz == 0 ? fx + k : a + fy; }
    template <int cz>
    __device__ __forceinline__ float ey() const { return cz == 0 ? fy + k : a + fx; }
};
// at(i) is (red, blue) of direction i; cz = 0 leaves the rest direction out (a = 0).
template <int cz, class L>
__device__ __forceinline__ ZClass z_class(L &&at) {
    ZClass o;
    const float2 v_y = at(dir_of(0, 1, cz)), vmy = at(dir_of(0, -1, cz)), v_x = at(dir_of(1, 0, cz)),
                 vmx = at(dir_of(-1, 0, cz)), v_k = at(dir_of(1, 1, cz)), vmk = at(dir_of(-1, -1, cz)),
                 v_q = at(dir_of(1, -1, cz)), vmq = at(dir_of(-1, 1, cz));
    o.a = 0.0f;
    o.m = v_y;
    if constexpr (cz != 0) {
        const float2 v0 = at(dir_of(0, 0, cz));
        o.a = v0.x + v0.y;
        o.m = __fadd2_rn(v0, v_y);
    }
    o.m = __fadd2_rn(__fadd2_rn(__fadd2_rn(o.m, v_x), vmy), vmx);
    o.m = __fadd2_rn(__fadd2_rn(__fadd2_rn(__fadd2_rn(o.m, v_k), v_q), vmk), vmq);
    const float y0 = v_y.x + v_y.y;
    const float y1 = vmy.x + vmy.y;
    const float x0 = v_x.x + v_x.y;
    const float x1 = vmx.x + vmx.y;
    const float k0 = v_k.x + v_k.y, k1 = vmk.x + vmk.y, q0 = v_q.x + v_q.y, q1 = vmq.x + vmq.y;
    const float ks = k0 + k1, qs = q0 + q1, kd = k0 - k1, qd = q0 - q1;
    o.fx = x0 + x1;
    o.fy = y0 + y1;
    o.k = ks + qs;
    // what x0 + x1 and y0 + y1 rounded off (x0 and x1 lie within a factor of two, so it is exact)
    if constexpr (cz != 0) o.k += (x1 - (o.fx - x0)) + (y1 - (o.fy - y0));
    o.X = (x0 - x1) + (kd + qd);
    o.Y = (y0 - y1) + (kd - qd);
    o.XY = ks - qs;
    return o;
}
// The classes c_z = +1 and 0 of a node, and its rest population.
struct HalfNode {
    float2 f0, m;
    float a, fx, fy, k, X, Y, jx, jy, dx, dy, XY;
};
__device__ __forceinline__ HalfNode join_classes(const ZClass &p, const ZClass &o, float2 f0) {
    return HalfNode{f0,        __fadd2_rn(o.m, p.m), p.a, p.fx, p.fy, p.k, p.X, p.Y,
                    o.X + p.X, o.Y + p.Y, o.ex<0>() - p.ex<1>(), o.ey<0>() - p.ey<1>(), o.XY + p.XY};
}
// All 27: the colour masses are f_0 + ((class 0 + class +1) + class -1), the association in which
// the collision sums the moving populations it writes before it takes the rest population as the
// remainder; fl(fl(rho - s) + s) = rho then keeps a uniform state an exact fixed point.
__device__ __forceinline__ Moments finish_moments(const StepArgs &a, const HalfNode &h, const ZClass &n) {
    const float2 rho = __fadd2_rn(h.f0, __fadd2_rn(h.m, n.m));
    Moments m;
    m.rho_r = rho.x;
    m.rho_b = rho.y;
    m.phi = order_parameter(rho.x, rho.y, a.inv_rho_r0, a.inv_rho_b0);
    m.jx = h.jx + n.X;
    m.jy = h.jy + n.Y;
    m.jz = (h.a - n.a) + (((h.fx - n.fx) + (h.fy - n.fy)) + (h.k - n.k));
    m.dxz = h.dx - n.ex<-1>();
    m.dyz = h.dy - n.ey<-1>();
    m.pzz = (h.a + n.a) + (((h.fx + h.fy) + h.k) + n.b());
    m.pxy = h.XY + n.XY;
    m.pxz = h.X - n.X;
    m.pyz = h.Y - n.Y;
    return m;
}
// Colour masses of the 26 moving populations in that association.
template <class L>
__device__ __forceinline__ float2 moving_mass(L &&at) {
    return __fadd2_rn(__fadd2_rn(z_class<0>(at).m, z_class<1>(at).m), z_class<-1>(at).m);
}
template <class L>
__device__ __forceinline__ Moments moments_of(const StepArgs &a, L &&at) {
    return finish_moments(a, join_classes(z_class<1>(at), z_class<0>(at), at(0)), z_class<-1>(at));
}

// Convective outflow (Section IV.A): the convective speed lambda = u_z(N - 1, t + 1) (Eq. (13))
// from the node's moments, clamped to [0, 1], and the blend f(N, t + 1) = [f(N, t) + lambda
// f(N - 1, t + 1)] / (1 + lambda) with inv = 1 / (1 + lambda).
__device__ __forceinline__ float outflow_lambda(const StepArgs &a, const Moments &m) {
    const float rho = m.rho_r + m.rho_b;
    const float lam = fmaf(0.5f * (rho - a.rho_b0), a.gz, m.jz) / rho;
    return fminf(fmaxf(lam, 0.0f), 1.0f);
}
__device__ __forceinline__ float outflow_blend(float hist, float f, float lam, float inv) { return fmaf(lam, f, hist) * inv; }

// Red population of the inlet disc that leaves a ghost column of velocity u in direction (cxs, cys,
// 1), of the speed class of i (reflected at a side wall, c differs from c_i in signs): f^e(rho_r0, u)
// with alpha_r and Phi = 0.
__device__ __forceinline__ float inlet_population(const StepArgs &a, int i, int cxs, int cys, float ux, float uy, float uz) {
    const float cu = ((float)cxs * ux + (float)cys * uy) + uz;
    const float usq = (ux * ux + uy * uy) + uz * uz;
    return a.rho_r0 * (varphi(i, a.alpha_r, a.oma_r) + wgt(i) * eq_poly(cu, usq));
}
__device__ __forceinline__ float inlet_population_at(const StepArgs &a, int i, int cxs, int cys, int xs, int ys) {
    InletVel iv;
    inlet_velocity(a.u_in, a.noise_amp, a.fourier, a.xc, a.yc, a.seed, a.step, xs, ys, a.nx, a.ny, iv);
    return inlet_population(a, i, cxs, cys, iv.ux, iv.uy, iv.uz);
}

// The phase entry of a node (FP32 storage).
__device__ __forceinline__ float2 phase_entry(const Moments &m) { return make_float2(m.phi, m.rho_r + m.rho_b); }

// The collision moments of a node as the moment pass stores them: three float4 planes of NN
// entries, (rho_r, rho_b, phi, jx), (jy, jz, dxz, dyz), (pzz, pxy, pxz, pyz).
__device__ __forceinline__ Moments unpack_moments(float4 a, float4 b, float4 c) {
    return Moments{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
}
__device__ __forceinline__ void store_moments(float4 *__restrict__ mom, size_t NN, int n, const Moments &m) {
    mom[n] = make_float4(m.rho_r, m.rho_b, m.phi, m.jx);
    mom[NN + n] = make_float4(m.jy, m.jz, m.dxz, m.dyz);
    mom[2 * NN + n] = make_float4(m.pzz, m.pxy, m.pxz, m.pyz);
}
__device__ __forceinline__ Moments load_moments(const float4 *__restrict__ mom, size_t NN, int n) {
    return unpack_moments(__ldg(mom + n), __ldg(mom + NN + n), __ldg(mom + 2 * NN + n));
}

// The same for the fused step kernel, where the moments were written earlier in the same launch
// and are read once: L1 is bypassed (ld.global.cg), and the L2 lines can be dropped afterwards.
__device__ __forceinline__ Moments load_moments_once(const float4 *__restrict__ mom, size_t NN, int n) {
    return unpack_moments(__ldcg(mom + n), __ldcg(mom + NN + n), __ldcg(mom + 2 * NN + n));
}

// L2 cache policy that keeps lines over evict-first and evict-normal ones.
__device__ __forceinline__ unsigned long long l2_evict_last_policy() {
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void st_keep(float4 *p, float4 v, unsigned long long pol) {
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "f"(v.x), "f"(v.y),
                 "f"(v.z), "f"(v.w), "l"(pol)
                 : "memory");
}
// Moments stored with the evict-last policy (the fused step kernel reads them a few planes later).
__device__ __forceinline__ void store_moments_keep(float4 *__restrict__ mom, size_t NN, int n, const Moments &m,
                                                   unsigned long long pol) {
    st_keep(mom + n, make_float4(m.rho_r, m.rho_b, m.phi, m.jx), pol);
    st_keep(mom + NN + n, make_float4(m.jy, m.jz, m.dxz, m.dyz), pol);
    st_keep(mom + 2 * NN + n, make_float4(m.pzz, m.pxy, m.pxz, m.pyz), pol);
}
// Drops the 128-byte L2 line at p (128-byte aligned) without writing it back: its contents
// become undefined.  For data that is dead (read for the last time by every thread that
// shares the line).
__device__ __forceinline__ void l2_discard(const void *p) {
    asm volatile("discard.global.L2 [%0], 128;" ::"l"(p) : "memory");
}

}  // namespace lbcm
