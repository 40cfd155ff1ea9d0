// pf_march2d.cu -- the explicit step of large 2D FP32 grids: warps that march
// along y with their rows in registers.
//
// Method and discretisation are those of pf_step2d.cu, through the same
// cell_rate and face_flux.  A warp owns a strip of 60 columns and `rows` rows.
// Lane l holds the cells 2l and 2l+1 of the strip's 64 (two of them stale on
// either side) as one two-lane vector, so x neighbours are one shuffle and y
// neighbours are the registers of the rows before.  The warp reads rows y0-2 ...
// y1+1; on reading row r it evaluates the rate of row r-1, that row's x faces, the
// y faces between r-2 and r-1, and updates row r-2.  There is no shared memory and
// no barrier.
//
// What bounds it: issue and the dependent chain of a row (logarithms, rate,
// fluxes), 500 instructions per 64 cells against 890 in the tile kernel, whose
// phases also wait for one another at four barriers.  Three warps per scheduler
// at 168 registers: four at 128 spill (1024^2: 26.7 us per step instead of 22.6),
// two hide less (2048^2: 107 instead of 70), unrolling by two or three to rename
// the rows spills as well (2048^2: 106 and 93).  Per step, tile kernel and this
// one: 1024^2 24.1 and 20.4 us, 2048^2 93.7 and 65.7 us.
#include <algorithm>
#include "pf_internal.cuh"
#include "pf_kernels.h"
#include "pf_lanes.cuh"

namespace pf {

namespace {

constexpr int MARCH_WARPS = 4;                 // per block

__device__ __forceinline__ float2 from_right(float2 v) {   // v at x + 1
    return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1));
}
__device__ __forceinline__ float2 from_left(float2 v) {    // v at x - 1
    return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x);
}

}  // namespace

__device__ __forceinline__ float word(const float* p, unsigned off) {
    float v;   // issued here, a row ahead of its use
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(reinterpret_cast<const char*>(p) + off));
    return v;
}
__device__ __forceinline__ void put(float* p, unsigned off, bool a, bool b, bool even, float2 v) {
    float* q = reinterpret_cast<float*>(reinterpret_cast<char*>(p) + off);
    if (even) {
        if (b) *reinterpret_cast<float2*>(q) = v;
    } else {
        if (a) q[0] = v.x;
        if (b) q[1] = v.y;
    }
}

template <bool L9, bool AI, bool STD>
__global__ void __launch_bounds__(32 * MARCH_WARPS, MARCH_PER_SM / MARCH_WARPS)
march2d_kernel(const float* phi_in, const float* c_in, const float* d_in, const float* clo_in,
               float* __restrict__ phi_out, float* __restrict__ c_out, float* __restrict__ d_out,
               float* __restrict__ clo_out, const PairConsts<float2> K, const GridConsts<float> G, const int strips,
               const int rows, const bool even) {
    using V = float2;
    const int w = blockIdx.x * MARCH_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int nx = G.n[0], ny = G.n[1];
    const int xw = (w % strips) * MARCH_X - 2, x = xw + 2 * lane;   // the warp's and the lane's first column
    const int y0 = (w / strips) * rows, y1 = min(y0 + rows, ny);
    if (y0 >= ny) return;   // a whole warp
    const int ma = map_coord(x, nx, G.bc_lo[0], G.bc_hi[0]), mb = map_coord(x + 1, nx, G.bc_lo[0], G.bc_hi[0]);
    const bool ghost_a = ma < 0, ghost_b = mb < 0;
    const bool inside = xw >= 0 && xw + 64 <= nx;   // no column of the warp lies outside the grid
    const bool own = lane >= 1 && lane <= 30;
    const unsigned oa = 4u * (ghost_a ? 0 : ma), ob = 4u * (ghost_b ? 0 : mb);   // of the columns in a row
    const bool st_a = own && x < nx, st_b = own && x + 1 < nx;
    const unsigned pitch = 4u * nx;
    // theta at the mirror / wrap image
    const V ke_theta = vpair(G.ke_theta0 - G.ke_G * ((float(ghost_a ? x : ma) + 0.5f) * G.dx),
                             G.ke_theta0 - G.ke_G * ((float(ghost_b ? x + 1 : mb) + 0.5f) * G.dx));
    const bool ghosts = (!inside && (G.bc_lo[0] == BC_DIRICHLET || G.bc_hi[0] == BC_DIRICHLET)) ||
                        ((y0 < 2 || y1 + 2 > ny) && (G.bc_lo[1] == BC_DIRICHLET || G.bc_hi[1] == BC_DIRICHLET));
    const bool twos = even && inside;   // 8-byte stores

    V nf, nc, nd;   // the next row
    auto fetch = [&](int y) {
        const unsigned row = (unsigned)max(map_coord(y, ny, G.bc_lo[1], G.bc_hi[1]), 0) * pitch;
        nf = vpair(word(phi_in, row + oa), word(phi_in, row + ob));
        nc = vpair(word(c_in, row + oa), word(c_in, row + ob));
        nd = vpair(word(d_in, row + oa), word(d_in, row + ob));
    };
    // rows r-1 ("1") and r-2 ("2"); components 0..3 = phi, Y, mu_s, mu_l; n = R - v,
    // D = R - L, LR = L + R of phi; cs12, cl12: rows r-1 and r-2 summed
    const V zero = vpair(0.f, 0.f);
    V v1[4], v2[4], n1[4], D1[4], D2[4], LR1 = zero, LR2 = zero, cs1 = zero, cl1 = zero, cs12 = zero, cl12 = zero, rate2 = zero;
    V yFc = zero, yFd = zero, xFc2 = zero, xFd2 = zero, c1 = zero, d1 = zero, c2 = zero, d2 = zero;
#pragma unroll
    for (int k = 0; k < 4; ++k) v1[k] = v2[k] = n1[k] = D1[k] = D2[k] = zero;

    grid_wait(phi_in, c_in, d_in, clo_in);
    fetch(y0 - 2);
    unsigned out = (unsigned)(y0 - 4) * pitch;   // of row r-2; wraps before the first use
#pragma unroll 1
    for (int r = y0 - 2; r <= y1 + 1; ++r, out += pitch) {
        // ---- row r
        V v0[4];
        v0[0] = nf;
        V c = nc, d = nd;
        if (ghosts) {   // beyond a Dirichlet boundary
            const bool gy = map_coord(r, ny, G.bc_lo[1], G.bc_hi[1]) < 0;
            if (gy || ghost_a) v0[0].x = G.dir_phi, c.x = G.dir_c, d.x = G.dir_d;
            if (gy || ghost_b) v0[0].y = G.dir_phi, c.y = G.dir_c, d.y = G.dir_d;
        }
        if (r <= y1) fetch(r + 1);
        const V p = vp_of<AI, STD>(K, v0[0]);
        const V cs0 = vfma(vsub(vlit<V>(1.0), p), d, c);
        const V cl0 = vsub(c, vmul(p, d));
        v0[2] = vsub(vlog(cs0), K.log_ke);
        v0[3] = vlog(cl0);
        v0[1] = vfma(p, vsub(v0[2], v0[3]), v0[3]);

        V n0[4], D0[4], g[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            n0[k] = vsub(from_right(v0[k]), v0[k]);
            D0[k] = vadd(n0[k], from_left(n0[k]));
            g[k] = vsub(v0[k], v2[k]);   // y differences at row r-1
        }
        const V LR0 = vadd(from_left(v0[0]), from_right(v0[0]));

        // ---- rate of row r-1
        V lap;
        {
            const V faces = vadd(LR1, vadd(v0[0], v2[0]));
            if (L9)
                lap = vmul(vlit<V>(1.0 / 6), vfma(vlit<V>(4.0), vsub(faces, vfma(vlit<V>(4.0), v1[0], v1[0])),
                                                  vadd(LR0, LR2)));
            else
                lap = vsub(faces, vmul(vlit<V>(4.0), v1[0]));
        }
        const V g2 = vfma(D1[0], D1[0], vmul(g[0], g[0]));
        const V ds = vfma(D1[2], D1[0], vmul(g[2], g[0])), dl = vfma(D1[3], D1[0], vmul(g[3], g[0]));
        V rate1 = cell_rate<AI, STD>(K, v1[0], lap, g2, ds, dl, cs1, cl1, v1[2], v1[3], ke_theta);
        if (ghosts) {
            const bool gy = map_coord(r - 1, ny, G.bc_lo[1], G.bc_hi[1]) < 0;
            rate1 = vmask(rate1, ghost_a || gy, ghost_b || gy);
        }

        // ---- x faces of row r-1, and their difference
        V xFc1, xFd1;
        {
            V t1[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) t1[k] = vadd(g[k], from_right(g[k]));
            face_flux<V, false, AI, STD>(K, vfma(vlit<V>(0.5), n1[0], v1[0]), vadd(cs1, from_right(cs1)),
                                         vadd(cl1, from_right(cl1)), vadd(rate1, from_right(rate1)), n1, t1, t1, xFc1,
                                         xFd1);
            if (!inside) {
                const bool shut_a = x == nx - 1 && G.bc_hi[0] == BC_NOFLUX;
                const bool shut_b = (x + 1 == nx - 1 && G.bc_hi[0] == BC_NOFLUX) ||
                                    (x + 1 == -1 && G.bc_lo[0] == BC_NOFLUX);
                xFc1 = vmask(xFc1, shut_a, shut_b);
                xFd1 = vmask(xFd1, shut_a, shut_b);
            }
            xFc1 = vsub(xFc1, from_left(xFc1));
            xFd1 = vsub(xFd1, from_left(xFd1));
        }

        // ---- y faces between rows r-2 and r-1
        V Fc, Fd;
        {
            V t1[4], n[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) t1[k] = vadd(D2[k], D1[k]), n[k] = vsub(v1[k], v2[k]);
            face_flux<V, false, AI, STD>(K, vmul(vlit<V>(0.5), vadd(v2[0], v1[0])), cs12, cl12, vadd(rate2, rate1), n, t1, t1,
                                         Fc, Fd);
            if ((r == 1 && G.bc_lo[1] == BC_NOFLUX) || (r - 1 == ny && G.bc_hi[1] == BC_NOFLUX)) Fc = Fd = zero;
        }

        // ---- conservative update of row r-2
        if (r >= y0 + 2) {
            const V phi_new = vfma(K.dt_dx2, rate2, v2[0]);
            const V d_new = vfma(K.dt_dx2, vadd(xFd2, vsub(Fd, yFd)), d2);
            const V dcv = vmul(K.dt_dx2, vadd(xFc2, vsub(Fc, yFc)));
            V c_new;
            if (clo_in != nullptr) {
                // compensated (TwoSum) update of c = hi + lo
                const V lo_k = vpair(word(clo_in, out + oa), word(clo_in, out + ob));
                const V s_ = vadd(c2, dcv);
                const V bv = vsub(s_, c2);
                const V err = vadd(vsub(c2, vsub(s_, bv)), vsub(dcv, bv));
                const V lo = vadd(lo_k, err);
                c_new = vadd(s_, lo);
                put(clo_out, out + 4u * x, st_a, st_b, twos, vsub(lo, vsub(c_new, s_)));
            } else {
                c_new = vadd(c2, dcv);
                if (clo_out != nullptr) put(clo_out, out + 4u * x, st_a, st_b, twos, c_new);
            }
            put(phi_out, out + 4u * x, st_a, st_b, twos, phi_new);
            put(c_out, out + 4u * x, st_a, st_b, twos, c_new);
            put(d_out, out + 4u * x, st_a, st_b, twos, d_new);
        }
        yFc = Fc, yFd = Fd, xFc2 = xFc1, xFd2 = xFd1, rate2 = rate1, LR2 = LR1, LR1 = LR0;
        cs12 = vadd(cs0, cs1), cl12 = vadd(cl0, cl1), cs1 = cs0, cl1 = cl0;
        c2 = c1, d2 = d1, c1 = c, d1 = d;
#pragma unroll
        for (int k = 0; k < 4; ++k) v2[k] = v1[k], v1[k] = v0[k], n1[k] = n0[k], D2[k] = D1[k], D1[k] = D0[k];
    }
}

cudaError_t launch_march2d(const StepLaunch& a, const Consts<float>& C, const Clock<float>& Kc, bool* taken) {
    *taken = false;
    const HostProblem& P = *a.prob;
    if ((long long)C.n[0] * C.n[1] >= 1ll << 30) return cudaSuccess;   // byte offsets are 32-bit
    static DeviceSetup setup;
    int dev = 0, sms = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= DeviceSetup::MAX_DEVICES) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(setup.mu);
        if (!setup.done[dev]) {
            e = cudaDeviceGetAttribute(&setup.sms[dev], cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
            setup.done[dev] = true;
        }
        sms = setup.sms[dev];
    }
    const long long strips = (C.n[0] + MARCH_X - 1) / MARCH_X;
    const long long rows = march2d_rows(C.n[0], C.n[1], sms);
    if (rows == 0) return cudaSuccess;
    const long long warps = strips * ((C.n[1] + rows - 1) / rows);
    *taken = true;
    const PairConsts<float2> K = make_pair_consts<float>(P, C);
    const GridConsts<float> G = make_grid_consts<float>(P, Kc);
    // default physics or not x 9- or 5-point Laplacian x shape parameter a != 0 or a = 0
    decltype(&march2d_kernel<true, true, true>) kerns[2][2][2] = {
        {{march2d_kernel<false, false, false>, march2d_kernel<false, true, false>},
         {march2d_kernel<true, false, false>, march2d_kernel<true, true, false>}},
        {{march2d_kernel<false, false, true>, march2d_kernel<false, true, true>},
         {march2d_kernel<true, false, true>, march2d_kernel<true, true, true>}}};
    auto kern = kerns[std_physics(P, false) ? 1 : 0][C.lap == 9 ? 1 : 0][P.a != 0.0 ? 1 : 0];
    bool even = C.n[0] % 2 == 0;   // rows start on 8-byte boundaries in every array
    for (const void* q : {a.phi_in, a.c_in, a.d_in, a.clo_in, (const void*)a.phi_out, (const void*)a.c_out,
                          (const void*)a.d_out, (const void*)a.clo_out})
        even = even && reinterpret_cast<uintptr_t>(q) % 8 == 0;
    return launch_after(
        kern, dim3((unsigned)((warps + MARCH_WARPS - 1) / MARCH_WARPS)), dim3(32 * MARCH_WARPS), 0, a.stream,
        static_cast<const float*>(a.phi_in), static_cast<const float*>(a.c_in), static_cast<const float*>(a.d_in),
        static_cast<const float*>(a.clo_in), static_cast<float*>(a.phi_out), static_cast<float*>(a.c_out),
        static_cast<float*>(a.d_out), static_cast<float*>(a.clo_out), K, G, (int)strips, (int)rows, even);
}

}  // namespace pf
