// lbcm_advance.cu -- the steps between the first gather and the last collision of one lb_step call
// with the paper's rates (arXiv:1804.08923, Section II, boundaries of Section IV.A).
//
// With s3 = s4 = s5 = s6 = 1 the collision depends on a node's 54 populations only through its 12
// collision moments (lbcm_collide.cuh).  So inside one call the state between two steps is kept as
// the moment record and the phase entry of the post-stream node (56 bytes with FP32 storage) and
// advance_kernel takes one such state to the next: it rebuilds the populations that the collision
// would have written (rounded as the storage rounds them), streams them through shared memory and
// sums the next moments.  lb_step(n) is one gather pass, n - 1 advances and one collision pass,
// with the same bits as n gather and n collision passes.
//
// A block owns a TX x TY tile of columns and a run of planes and marches along z.  Per plane k:
//   collide  a warp takes a row of the tile, its halo rows or its halo columns (of which only the nine
//            populations that enter the tile are built), from prefetched moments and the gradients,
//            and writes the populations to shared memory;
//   gradient of plane k + 1, from a ring of four phase planes in shared memory, while other warps are
//            still colliding;
//   gather   each thread of the tile reads the 27 pulls that come from plane k: c_z = -1 completes
//            the node of plane k - 1, c_z = 0 is joined to plane k, c_z = +1 starts plane k + 1
//            (z_class, join_classes, finish_moments; 24 registers hold the two open planes).
// What bounds it: instruction issue and the shared-memory pipe, in turn rather than together (96 x 96 x
// 384 jet: issue slots 74%, FMA pipe 58%, 1238 instructions a node with its share of the halo; DRAM 104
// bytes a node, a third of its bandwidth), because the warps of a block go through the same phase at
// the same time.  96 registers a thread; the outflow epilogue, which one run of a column takes after its
// march, spills 27 pairs (about 450 bytes).  256 x 256 x 512: 23.4 G nodes/s.  Tried there, before the
// present order of the sums (22.4): 32 x 16 tile, 20 warps, a barrier after each phase 19.2; halo warps of
// their own 20.2; gradient moved between arriving at and waiting on the first barrier, the scalar
// part of the collision before the second 22.4; both barriers split in two halves 21.5.  Two
// population buffers and one barrier (32 x 11, 14 warps) 16.3 when the first form had 17.2.
#include <algorithm>
#include <iterator>
#include <type_traits>

#include "lbcm_collide.cuh"
#include "lbcm_device.cuh"
#include "lbcm_internal.h"
#include "lbcm_node.cuh"

namespace lbcm {

template <int TX, int TY>
struct AdvanceTile {
    static constexpr int BX = TX + 2, RX = TX + 4, RY = TY + 4;  // row of collided nodes, ring of phase nodes
    static constexpr int NB = BX * (TY + 2), NR = RX * RY;
    // threads: the nodes of the tile, the two halo rows, the halo columns with the corners, in whole warps
    static constexpr int kRows = TX * TY, kHaloY = 2 * TX, NT = kRows + kHaloY + (2 * (TY + 2) + 31) / 32 * 32;
    // bytes: populations [27][NB] float2, moments [3][NT] float4, ring [4][NR] float2, inlet velocities [NB] float4
    static constexpr int kMom = (27 * NB * (int)sizeof(float2) + 15) / 16 * 16;
    static constexpr int kRing = kMom + 3 * NT * (int)sizeof(float4);
    static constexpr int kInflow = kRing + 4 * NR * (int)sizeof(float2);
    static constexpr int kBar = kInflow + NB * (int)sizeof(float4);
    static constexpr int kBytes = kBar + 16;
    static_assert(kBytes <= 227 * 1024 && NR <= 2 * NT && kRows % 32 == 0 && kHaloY % 32 == 0, "layout");
};

// Barrier of the block's warps in two halves: a warp arrives when it has written what it shares, goes
// on with work of its own and waits when it needs the others'.  The wait is bounded by the number of
// tries (1.4 us each when they fail); a wait that runs out (none does while every warp arrives once a
// phase) sets *err and the word after the barrier and goes on, and later waits of the block that find
// that word set try once.
constexpr int kWaitTries = 1 << 20;  // 1.5 s
__device__ __forceinline__ void warps_init(unsigned bar, int warps) {
    asm volatile("mbarrier.init.shared.b64 [%0], %1;\n" ::"r"(bar), "r"(warps) : "memory");
    asm volatile("st.shared.u32 [%0 + 8], 0;\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void warps_arrive(unsigned bar) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void warps_wait(unsigned bar, int phase, int *err, int tries = kWaitTries) {
    for (int n = 0; n < tries; ++n) {
        unsigned done, given_up;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done)
                     : "r"(bar), "r"(phase & 1)
                     : "memory");
        if (done) return;
        asm volatile("ld.volatile.shared.u32 %0, [%1 + 8];\n" : "=r"(given_up) : "r"(bar) : "memory");
        if (given_up) return;
    }
    *err = 1;
    asm volatile("st.volatile.shared.u32 [%0 + 8], 1;\n" ::"r"(bar) : "memory");
}

// That wait on a barrier at which only one of two warps arrives, twice; *ns receives the time both took.
__global__ void __launch_bounds__(64) advance_wait_probe_kernel(int *err, int tries, unsigned long long *ns) {
    __shared__ __align__(16) unsigned char smem[16];
    const unsigned bar = (unsigned)__cvta_generic_to_shared(smem);
    if (threadIdx.x == 0) warps_init(bar, 2);
    __syncthreads();
    const unsigned long long t0 = global_ns();
    if (threadIdx.x < 32) warps_arrive(bar);
    warps_wait(bar, 0, err, tries);
    warps_wait(bar, 0, err, tries);
    if (threadIdx.x == 0) *ns = global_ns() - t0;
}

// Barrier of the whole block that the warps may reach at different places of the code.
template <int NT>
__device__ __forceinline__ void block_sync() {
    asm volatile("barrier.sync 1, %0;\n" ::"n"(NT) : "memory");
}

__device__ __forceinline__ int pmod(int a, int n) {
    const int r = a % n;
    return r < 0 ? r + n : r;
}

// The run that ends at a convective top computes the outflow after its march, as long as six planes take;
// it gets that many fewer.  By that number of planes (us a step): 64x64x256 jet 0 72.5, 2 66.3, 4 60.8, 6
// 56.5, 8 57.2; 96x96x384 jet 180, 177, 171, 167.0, 167.4 (52.7 and 159.3 now); runs shorter than 8 planes
// stay equal.
constexpr int kTail = 6;

template <bool kForce, bool W, int TX, int TY, int MB>
__global__ void __launch_bounds__(AdvanceTile<TX, TY>::NT, MB) advance_kernel(StepArgs a, AdvanceArgs v) {
    chain_begin();
    using T = AdvanceTile<TX, TY>;
    constexpr int BX = T::BX, RX = T::RX, NB = T::NB, NT = T::NT;
    extern __shared__ __align__(16) unsigned char smem[];
    float4 *mb = reinterpret_cast<float4 *>(smem + T::kMom);
    float2 *ring = reinterpret_cast<float2 *>(smem + T::kRing);
    float4 *inflow = reinterpret_cast<float4 *>(smem + T::kInflow);

    const int t = threadIdx.x;
    const int tile = blockIdx.x % v.tiles, chunk = blockIdx.x / v.tiles;
    const int x0 = (tile % v.tiles_x) * TX, y0 = (tile / v.tiles_x) * TY;
    const int nx = a.nx, ny = a.ny, N = a.nz - 1, P = (int)a.plane;
    const bool pz = a.bc_zlo == BC_PERIODIC, conv = a.bc_zhi == BC_CONVECTIVE;
    const int tail = conv && v.planes >= 8 * v.chunks ? kTail : 0;
    auto cut = [&](int c) { return min((int)((long long)(v.planes + tail) * c / v.chunks), v.planes); };
    const int z0 = cut(chunk), z1 = cut(chunk + 1);
    const bool top = !pz && z1 == v.planes;  // the run that ends at z = N (conv: planes = N)
    const int kb = pz ? z0 - 1 : max(z0 - 1, 0), ke = pz ? z1 : min(z1, N);

    // the node this thread collides, at position (bx, by) of the tile with its halo, wrapped where
    // periodic; nothing lies beyond a side wall
    const int line = t / TX, lane = t % TX, e = t - T::kRows - T::kHaloY;
    const bool row = line < TY, halo_y = !row && line < TY + 2;  // warp-uniform
    const int bx = e < 0 ? lane + 1 : (e & 1 ? BX - 1 : 0),
              by = row ? line + 1 : (halo_y ? (line == TY ? 0 : TY + 1) : e >> 1);
    const float side = e < 0 ? (by == 0 ? 1.0f : -1.0f) : (bx == 0 ? 1.0f : -1.0f);  // halo: the component that enters
    int xs = x0 + bx - 1, ys = y0 + by - 1;
    const bool wx = W && a.wall_x, wy = W && a.wall_y;
    const bool collider = by < TY + 2 && xs <= nx && ys <= ny && !(wx && (xs < 0 || xs >= nx)) && !(wy && (ys < 0 || ys >= ny));
    const bool inside = row && xs < nx && ys < ny;  // a node of the tile: this thread gathers it too
    const int pos = by * BX + bx, rpos = (by + 1) * RX + bx + 1;
    const int x = xs, y = ys;
    xs = wrapi(xs, nx);
    ys = wrapi(ys, ny);
    const int cxy = collider ? ys * nx + xs : 0;
    // the one or two ring positions this thread fills, clamped at side walls (mirror ghosts)
    int fill[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = t + q * NT;
        int X = x0 + e % RX - 2, Y = y0 + e / RX - 2;
        X = wx ? min(max(X, 0), nx - 1) : pmod(X, nx);
        Y = wy ? min(max(Y, 0), ny - 1) : pmod(Y, ny);
        fill[q] = Y * nx + X;
    }
    const unsigned s_ring = (unsigned)__cvta_generic_to_shared(ring), s_mb = (unsigned)__cvta_generic_to_shared(mb);
    // planes beyond z walls mirror the wall plane
    auto plane_of = [&](int k) { return pz ? pmod(k, a.nz) : min(max(k, 0), N); };
    auto plane_after = [&](int z) { return z < N ? z + 1 : (pz ? 0 : N); };
    auto fill_ring = [&](int k, int z) {  // slot of plane k from plane z
        const float2 *src = v.phase + z * P;
        const unsigned dst = s_ring + ((k & 3) * T::NR + t) * (int)sizeof(float2);
        cp_async<sizeof(float2)>(dst, src + fill[0]);
        if (t + NT < T::NR) cp_async<sizeof(float2)>(dst + NT * (int)sizeof(float2), src + fill[1]);
    };
    auto fetch_moments = [&](int z) {
        const int n = z * P + cxy;
        cp_async<16>(s_mb + t * 16, v.mom[0] + n);
        cp_async<16>(s_mb + (NT + t) * 16, v.mom[1] + n);
        cp_async<16>(s_mb + (2 * NT + t) * 16, v.mom[2] + n);
    };
    auto write_out = [&](int z, const Moments &m) {
        const int n = z * P + cxy;
        v.mom_out[0][n] = make_float4(m.rho_r, m.rho_b, m.phi, m.jx);
        v.mom_out[1][n] = make_float4(m.jy, m.jz, m.dxz, m.dyz);
        v.mom_out[2][n] = make_float4(m.pzz, m.pxy, m.pxz, m.pyz);
        v.phase_out[n] = phase_entry(m);
    };

    fill_ring(kb - 1, plane_of(kb - 1));
    fill_ring(kb, plane_of(kb));
    fill_ring(kb + 1, plane_of(kb + 1));
    int zr = plane_after(plane_of(kb + 1));  // the last plane in the ring
    fill_ring(kb + 2, zr);
    int zm = plane_of(kb);      // the plane whose moments are here or on their way
    fetch_moments(zm);
    cp_async_commit();
    const unsigned bar_full = (unsigned)__cvta_generic_to_shared(smem + T::kBar);
    if (t == 0) warps_init(bar_full, NT / 32);
    cp_async_wait();
    if (!pz && kb == 0 && a.bc_zlo == BC_INLET) {  // ghost plane z = -1 inside the inlet disc (own entries)
        float2 *g = ring + 3 * T::NR;
        for (int q = 0; q < 2; ++q)
            if (t + q * NT < T::NR && a.disc[fill[q]]) g[t + q * NT] = make_float2(1.0f, a.rho_r0);
    }
    if (!pz && kb == 0 && a.bc_zlo == BC_INLET && collider) {  // velocity of the ghost columns inside the disc
        float4 u = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (a.disc[cxy]) {
            InletVel iv;
            inlet_velocity(a.u_in, a.noise_amp, a.fourier, a.xc, a.yc, a.seed, a.step, xs, ys, nx, ny, iv);
            u = make_float4(iv.ux, iv.uy, iv.uz, 1.0f);
        }
        inflow[pos] = u;
    }
    __syncthreads();

    // gradients of plane k's node from ring planes k - 1, k, k + 1
    float2 gx, gy, gz;
    auto gradient = [&](int k) {
        const float2 *r[3] = {ring + ((k - 1) & 3) * T::NR + rpos, ring + (k & 3) * T::NR + rpos,
                             ring + ((k + 1) & 3) * T::NR + rpos};
        gradients([&](int j) { return r[cz(j) + 1][cy(j) * RX + cx(j)]; }, gx, gy, gz);
        if (a.grad4 && inside && k >= z0 && (k < z1 || top)) {
            a.grad4[k * P + cxy] = make_float4(gx.x, gy.x, gz.x, gx.y);
            a.grad2[k * P + cxy] = make_float2(gy.y, gz.y);
        }
    };
    // collides plane k; the rest population of a node of the tile stays with its thread
    auto collide = [&](int k, float2 &rest) {
        float2 *out = reinterpret_cast<float2 *>(smem) + pos;
        const float4 *m = mb + t;
        const Moments mo = unpack_moments(m[0], m[NT], m[2 * NT]);
        // the record is in registers: its place takes the next plane's; the populations' place is free
        // once every warp has gathered plane k - 1
        auto ready = [&] {
            if (k < ke) fetch_moments(plane_after(zm));
            if (k > kb) block_sync<NT>();
        };
        if (row)
            collide_node<kForce>(a, mo, gx, gy, gz, [&](int i, float2 f) {
                if (i == 0)
                    rest = f;
                else
                    out[i * NB] = f;
                return f;
            }, ready);
        else if (halo_y)
            collide_halo_y<kForce>(a, mo, gx, gy, gz, side,
                                   [&](int i, float2 f) { out[(side > 0.0f ? i : flip_y(i)) * NB] = f; }, ready);
        else
            collide_halo_x<kForce>(a, mo, gx, gy, gz, side,
                                   [&](int i, float2 f) { out[(side > 0.0f ? i : flip_x(i)) * NB] = f; }, ready);
    };

    ZClass up{};      // class c_z = +1 of plane k + 1
    HalfNode open{};  // classes +1 and 0 of plane k
    const float2 *pop = reinterpret_cast<const float2 *>(smem);
    // The pull of direction i comes from tile position pos - c_i; wall: beyond a free-slip side wall it
    // comes from the wall node itself, with that velocity component reversed (half-way specular
    // reflection).  Blocks without wall nodes take the plain form.
    const bool wxl = wx && x == 0, wxh = wx && x == nx - 1, wyl = wy && y == 0, wyh = wy && y == ny - 1;
    const bool walled = (wx && (x0 == 0 || x0 + TX >= nx)) || (wy && (y0 == 0 || y0 + TY >= ny));
    auto gather = [&](int k, float2 rest, auto wall) {
        constexpr bool kWall = decltype(wall)::value;
        auto fx = [&](int i) { return kWall && (cx(i) > 0 ? wxl : (cx(i) < 0 ? wxh : false)); };
        auto fy = [&](int i) { return kWall && (cy(i) > 0 ? wyl : (cy(i) < 0 ? wyh : false)); };
        auto from = [&](int i) { return pos - (fy(i) ? 0 : cy(i) * BX) - (fx(i) ? 0 : cx(i)); };
        auto slot = [&](int i) { return fx(i) ? (fy(i) ? flip_xy(i) : flip_x(i)) : (fy(i) ? flip_y(i) : i); };
        auto at = [&](int i) { return pop[slot(i) * NB + from(i)]; };
        // reflected at a z wall: the slot whose direction has c_z reversed too
        auto mirrored = [&](int i) {
            const int m = mirror_z(i);
            return pop[(fx(i) ? (fy(i) ? flip_xy(m) : flip_x(m)) : (fy(i) ? flip_y(m) : m)) * NB + from(i)];
        };
        if (!pz && k == 0)  // what enters plane 0 from z = -1: the inlet, or plane 0's own reflected
            up = z_class<1>([&](int i) {
                if (a.bc_zlo == BC_INLET) {
                    const float4 u = inflow[from(i)];
                    if (u.w != 0.0f)
                        return make_float2(inlet_population(a, i, fx(i) ? -cx(i) : cx(i), fy(i) ? -cy(i) : cy(i), u.x, u.y, u.z), 0.0f);
                }
                return mirrored(i);
            });
        if (k > z0) write_out(k - 1, finish_moments(a, open, z_class<-1>(at)));
        if (top && conv && k >= N - 2) {
            // the outflow plane N needs the populations of plane N - 1 one by one: they are kept
            // in this column's slots of the next history until the march is over
            const size_t p = (size_t)P;
#pragma unroll
            for (int i = 0; i < 27; ++i)
                if (cz(i) == N - 1 - k) {
                    const float2 f = i == 0 ? rest : at(i);
                    a.hist_out[i * p + cxy] = f.x;
                    a.hist_out[(27 + i) * p + cxy] = f.y;
                }
        }
        open = join_classes(up, z_class<0>(at), rest);
        up = z_class<1>(at);
        if (top && !conv && k == N) write_out(N, finish_moments(a, open, z_class<-1>(mirrored)));
    };
    if (collider) gradient(kb);
    __syncthreads();  // the first refill of the ring takes the place of plane kb - 1
    for (int k = kb; k <= ke; ++k) {
        float2 rest;
        if (collider)
            collide(k, rest);
        else if (k > kb)  // no warp runs ahead of the ring's readers
            block_sync<NT>();
        warps_arrive(bar_full);
        zm = plane_after(zm);
        zr = plane_after(zr);
        if (k + 2 <= ke) fill_ring(k + 3, zr);  // over plane k - 1, whose last reader was gradient(k)
        cp_async_commit();
        if (collider && k < ke) gradient(k + 1);
        warps_wait(bar_full, k - kb, v.err);
        if (inside) {
            if (W && walled)
                gather(k, rest, std::true_type{});
            else
                gather(k, rest, std::false_type{});
        }
        cp_async_wait();
    }
    if (top && conv && inside) {  // f(N, t + 1) from f(N - 1, t + 1) and f(N, t)
        const size_t p = (size_t)P;
        float2 f[27];
#pragma unroll
        for (int i = 0; i < 27; ++i) f[i] = make_float2(a.hist_out[i * p + cxy], a.hist_out[(27 + i) * p + cxy]);
        const float lam = outflow_lambda(a, moments_of(a, [&](int i) { return f[i]; }));
        const float inv = 1.0f / (1.0f + lam);
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            if (i % 6 == 0) asm volatile("" ::: "memory");  // six directions' loads in flight, not all 27 in registers
            if (a.fm_out) {
                a.fm_out[i * p + cxy] = f[i].x;
                a.fm_out[(27 + i) * p + cxy] = f[i].y;
            }
            f[i] = make_float2(outflow_blend(__ldg(a.hist_in + i * p + cxy), f[i].x, lam, inv),
                               outflow_blend(__ldg(a.hist_in + (27 + i) * p + cxy), f[i].y, lam, inv));
            a.hist_out[i * p + cxy] = f[i].x;
            a.hist_out[(27 + i) * p + cxy] = f[i].y;
        }
        write_out(N, moments_of(a, [&](int i) { return f[i]; }));
    }
}

// ------------------------------------------------------------------------ launchers
cudaError_t launch_advance_wait_probe(int *err, int tries, unsigned long long *ns, cudaStream_t s) {
    advance_wait_probe_kernel<<<1, 64, 0, s>>>(err, tries, ns);
    return cudaGetLastError();
}

template <bool kForce, bool W, int TX, int TY, int MB>
static cudaError_t launch_tile(const StepArgs &a, AdvanceArgs v, int chunks, cudaStream_t s) {
    using T = AdvanceTile<TX, TY>;
    auto *fn = advance_kernel<kForce, W, TX, TY, MB>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, T::kBytes);
    if (e != cudaSuccess) return e;
    v.tiles_x = (a.nx + TX - 1) / TX;
    v.tiles = v.tiles_x * ((a.ny + TY - 1) / TY);
    v.planes = a.bc_zhi == BC_CONVECTIVE ? a.nz - 1 : a.nz;
    v.chunks = std::min(chunks, v.planes);
    for (int q = 1; q < 3; ++q) {
        v.mom[q] = v.mom[0] + q * a.NN;
        v.mom_out[q] = v.mom_out[0] + q * a.NN;
    }
    return launch_chained(fn, dim3((unsigned)v.tiles * v.chunks), dim3(T::NT), T::kBytes, s, a, v);
}

template <int TX, int TY, int MB>
static cudaError_t launch_shape(const StepArgs &a, const AdvanceArgs &v, int chunks, cudaStream_t s) {
    const bool force = a.gx != 0.0f || a.gy != 0.0f || a.gz != 0.0f;
    if (a.wall_x || a.wall_y)
        return force ? launch_tile<true, true, TX, TY, MB>(a, v, chunks, s) : launch_tile<false, true, TX, TY, MB>(a, v, chunks, s);
    return force ? launch_tile<true, false, TX, TY, MB>(a, v, chunks, s) : launch_tile<false, false, TX, TY, MB>(a, v, chunks, s);
}

constexpr int kSMs = 152;

// The tiles.  Per plane and resident block (us, from 256 x 256 x 512 periodic and the jets): 3.15 for
// 32 x 16 (one block of 20 warps on an SM), 2.9 for 16 x 30 (18 warps), 2.85 for 16 x 14 (two blocks of
// 9 warps; 1.9 when a block has the SM to itself).  They reach 21.7, 21.5 and 20.9 G nodes/s on that
// lattice; the 16-wide ones waste less on extents that are no multiple of 32, and the smallest fills the
// chip with fewer columns (it replaced 32 x 7, 10 warps for the same 224 nodes, 18.4).  Over lattices of
// 48 to 192 nodes a side the estimate is 7% (up to 23%) below that of 32 x 16 and 32 x 7 alone; the
// walled 120 x 120 x 600 jet took 507 us a step in 16 x 30 and 530 in 32 x 16 (487 now; estimated 404:
// the estimate knows no side walls, whose blocks take the longer gather).
struct TileShape {
    int tx, ty, resident;
    float plane_us, alone_us;
};
constexpr TileShape kShapes[] = {{32, 16, 1, 3.15f, 3.15f}, {16, 30, 1, 2.9f, 2.9f}, {16, 14, 2, 2.85f, 1.9f}};

// Which tile and how many runs of planes: the least estimated time of the last wave's end.  A run
// collides one plane more at each end, and about 12 us go into filling and draining it.
AdvancePlan plan_advance(const StepArgs &a) {
    const int planes = a.bc_zhi == BC_CONVECTIVE ? a.nz - 1 : a.nz;
    AdvancePlan best{0, 1, 1e30f};
    for (int k = 0; k < (int)std::size(kShapes); ++k) {
        const TileShape &h = kShapes[k];
        const long long tiles = (long long)((a.nx + h.tx - 1) / h.tx) * ((a.ny + h.ty - 1) / h.ty), slots = h.resident * kSMs;
        for (int chunks = 1; chunks <= planes && chunks <= 4 * kSMs; ++chunks) {
            const long long blocks = tiles * chunks;
            const float us = (float)((blocks + slots - 1) / slots) * (float)((planes + chunks - 1) / chunks + 2) *
                                 (blocks <= kSMs ? h.alone_us : h.plane_us) + 12.0f;
            if (us < best.us) best = AdvancePlan{k, chunks, us};
        }
    }
    return best;
}

cudaError_t launch_advance(const StepArgs &a, const AdvancePlan &p, const AdvanceArgs &v, cudaStream_t s,
                           long long *launches) {
    *launches += 1;
    switch (p.shape) {
        case 0: return launch_shape<kShapes[0].tx, kShapes[0].ty, kShapes[0].resident>(a, v, p.chunks, s);
        case 1: return launch_shape<kShapes[1].tx, kShapes[1].ty, kShapes[1].resident>(a, v, p.chunks, s);
        default: return launch_shape<kShapes[2].tx, kShapes[2].ty, kShapes[2].resident>(a, v, p.chunks, s);
    }
}

}  // namespace lbcm
