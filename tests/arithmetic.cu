// Error sums of the device functions that the step kernels share, for test_gpu_arithmetic.py.
#include "lbcm_collide.cuh"
#include "lbcm_node.cuh"
#include "lbcm_pairs.cuh"

using namespace lbcm;

// Over n consecutive floats from the bit pattern lo: out[0] = how often rcp_newton differs from 1/x;
// out[1], out[2] = squared errors of rsqrt_newton and of 1/sqrtf in units of the result's last place.
__global__ void reciprocals_kernel(unsigned lo, unsigned n, double *out) {
    double v[3] = {0.0, 0.0, 0.0};
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float x = __uint_as_float(lo + i);
        v[0] += rcp_newton(x) != 1.0f / x;
        const double e = 1.0 / sqrt((double)x), u = (double)__uint_as_float(__float_as_uint((float)e) & 0x7f800000u);
        const double a = ((double)rsqrt_newton(x) - e) / u, b = ((double)(1.0f / sqrtf(x)) - e) / u;
        v[1] += a * a;
        v[2] += b * b;
    }
    for (int k = 0; k < 3; ++k) atomicAdd(out + k, v[k]);
}

// Squared errors of (jx, jy, jz) of n nodes near equilibrium (rho = 1, |u| up to 0.05, both colours, 1%
// disturbed): out[0..2] summed by classes of c_z, out[3..5] over the 13 pairs of opposite directions.
__global__ void momentum_kernel(int n, double *out) {
    StepArgs a{};
    a.inv_rho_r0 = a.inv_rho_b0 = 1.0f;
    double v[6] = {};
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        unsigned s = 0x9E3779B9u * (unsigned)(t + 1);
        auto rnd = [&] {  // in [-1, 1)
            s = s * 1664525u + 1013904223u;
            return (float)(s >> 8) / 8388608.0f - 1.0f;
        };
        const float ux = 0.05f * rnd(), uy = 0.05f * rnd(), uz = 0.05f * rnd(), c = 0.5f + 0.5f * rnd();
        float fr[27], fb[27];
        double j[3] = {0.0, 0.0, 0.0};
        for (int i = 0; i < 27; ++i) {
            const float cu = cx(i) * ux + cy(i) * uy + cz(i) * uz;
            const float f = wgt(i) * (1.0f + 3.0f * cu + 4.5f * cu * cu - 1.5f * (ux * ux + uy * uy + uz * uz)) * (1.0f + 0.01f * rnd());
            fr[i] = f * c;
            fb[i] = f - fr[i];
            const double d = (double)fr[i] + (double)fb[i];
            j[0] += cx(i) * d;
            j[1] += cy(i) * d;
            j[2] += cz(i) * d;
        }
        const Moments m = moments_of(a, [&](int i) { return make_float2(fr[i], fb[i]); });
        PairMoments p;
        pair_moments_of(fr, fb, p);
        const float got[6] = {m.jx, m.jy, m.jz, p.jx, p.jy, p.jz};
        for (int k = 0; k < 6; ++k) v[k] += ((double)got[k] - j[k % 3]) * ((double)got[k] - j[k % 3]);
    }
    for (int k = 0; k < 6; ++k) atomicAdd(out + k, v[k]);
}

extern "C" __attribute__((visibility("default"))) int reciprocals(unsigned lo, unsigned n, double *out) {
    reciprocals_kernel<<<1024, 256>>>(lo, n, out);
    return (int)cudaDeviceSynchronize();
}
extern "C" __attribute__((visibility("default"))) int momentum(int n, double *out) {
    momentum_kernel<<<256, 128>>>(n, out);
    return (int)cudaDeviceSynchronize();
}
