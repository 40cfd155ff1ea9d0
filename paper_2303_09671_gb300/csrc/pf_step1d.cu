// pf_step1d.cu -- several steps of one 1D line per launch.
//
// A single line is bound by latency: one step per launch cost a launch, a kernel
// of three barriers and, with a moving window, a second kernel per shift (1000
// cells, FP32: 8.5 us per step; 1024 cells, FP64, with F_h after every step:
// 43 us).  Here a warp takes a strip of the line (pf_line.cuh) with a halo of two
// cells per step through registers for up to KS steps, so that strips exchange
// nothing within a launch; the window's shifts are changes of index, applied when
// the strip is written.  The halo is computed twice: 32 of 64 cells hold results
// where the line leaves SMs idle, 112 of 128 where it does not.  FP64 is bound by
// the FP64 pipe of an SM, which issues one warp instruction in about 18 cycles:
// a short line is spread with one cell per lane, 16 of 32 cells holding results.
// Measured: 1.45 us per FP32 step (1000 cells), 6.4 us per FP64 step with its energy.
//
// The energy of the state before each step is summed from the values the step
// evaluates anyway (c_s, c_l, their potentials), per strip in a fixed order.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include "pf_internal.cuh"
#include "pf_kernels.h"
#include "pf_line.cuh"

namespace pf {

constexpr int LINE_KMAX = 8;   // steps per launch at most

template <typename E>
struct LineArgs {
    using M = typename LineNum<E>::M;
    const M *phi, *c, *d, *clo, *plo;
    M *phi_out, *c_out, *d_out, *clo_out, *plo_out;   // phi_out null: nothing is stored
    LineConsts<E> K;
    typename LineNum<E>::V dtq;
    int n, steps, strips;
    int periodic;
    int m[LINE_KMAX + 1];          // window shifts before each step, and after the last
    double ke_theta0[LINE_KMAX];
    // energies: partial of strip s and step k at epart[(erec + k) strips + s]; those of negative records are left out
    double* epart;
    long long erec;
    double H, grad;                // well height; sigma / (2 dx^2)
};

// a strip's sum of the energy density over the cells lo .. hi - 1
struct LineEnergy {
    static constexpr bool on = true;
    int i0, lo, hi, last;          // last: the cell whose right neighbour is a ghost, or -1
    double H, grad;
    double* sum;
    __device__ __forceinline__ void operator()(int q, double f, double fR, double p, double cs, double cl, double mus,
                                               double mul, double, double ke_theta) const {
        const int i = i0 + q;
        if (i < lo || i >= hi) return;
        const double g = vmul(f, vsub(1.0, f)), d = vsub(fR, f);
        const double fs = vsub(vmul(cs, vsub(mus, 1.0)), ke_theta), fl = vmul(cl, vsub(mul, 1.0));
        const double w = i == last ? 0.5 * grad : grad;
        *sum = vadd(*sum, vfma(w, vmul(d, d), vfma(H, vmul(g, g), vfma(p, vsub(fs, fl), fl))));
    }
};

// KS: steps per launch at most; a strip is 32 J cells, 2 KS of them halo on either side
template <typename E, int J, int KS, bool STD, int COMP, bool ENERGY>
__global__ void __launch_bounds__(128) line_kernel(const __grid_constant__ LineArgs<E> a) {
    using M = typename LineNum<E>::M;
    using X = typename LineNum<E>::X;
    constexpr int LN = LineNum<E>::LANES, H = J / LN, USE = 32 * J - 4 * KS;
    const int strip = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x & 31;
    if (strip >= a.strips) return;
    const int n = a.n, mt = a.m[a.steps];
    // first cell of the strip and of the lane, in the frame before the launch
    const int s0 = mt + strip * USE - 2 * KS, i0 = s0 + lane * J;
    Strip<E, J, COMP> s;
    auto get = [&](const M* p, M ghost, X (&x)[H]) {
        M w[J];
#pragma unroll
        for (int k = 0; k < J; ++k) {
            int i = i0 + k;
            if (a.periodic) {
                i %= n;
                i += i < 0 ? n : 0;
            }
            w[k] = i >= 0 && i < n ? p[i] : ghost;
        }
#pragma unroll
        for (int k = 0; k < H; ++k) x[k] = x_join<X>(w[k], w[(k + H) % J]);
    };
    grid_wait();
    get(a.phi, a.K.gphi, s.phi);
    get(a.c, a.K.fc, s.c);
    get(a.d, a.K.fd, s.d);
    if constexpr (COMP == 1) {
        get(a.plo, a.K.gphi_lo, s.plo);
        get(a.clo, a.K.fc_lo, s.clo);
    }
    const bool edge = !a.periodic && (s0 <= mt + 1 || s0 + 32 * J + 1 >= n);   // an end of the line in the strip
    auto run = [&](auto e) {
        constexpr bool EDGE = decltype(e)::value;
        for (int k = 0; k < a.steps; ++k) {
            if constexpr (ENERGY) {
                double sum = 0.0;
                LineEnergy en;
                en.i0 = i0;
                en.lo = strip * USE;
                en.hi = min(en.lo + USE, n);
                en.last = a.periodic || a.K.hot_noflux ? -1 : n - 1;
                en.H = a.H;
                en.grad = a.grad;
                en.sum = &sum;
                line_step<STD, EDGE, E, J, COMP>(a.K, s, i0, n, a.m[k], a.dtq, a.ke_theta0[k], en);
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (lane == 0 && a.erec + k >= 0) a.epart[(a.erec + k) * a.strips + strip] = sum;
            } else {
                line_step<STD, EDGE, E, J, COMP>(a.K, s, i0, n, a.m[k], a.dtq, a.ke_theta0[k], NoRecord());
            }
        }
    };
    if (edge) run(std::true_type());
    else run(std::false_type());
    if (a.phi_out == nullptr) return;
#pragma unroll
    for (int k = 0; k < J; ++k) {
        const int j = i0 + k - mt, u = lane * J + k;      // the window has dropped mt cells
        if (u < 2 * KS || u >= 32 * J - 2 * KS || j >= n) continue;
        a.phi_out[j] = k < H ? x_lo(s.phi[k % H]) : x_hi(s.phi[k % H]);
        a.c_out[j] = k < H ? x_lo(s.c[k % H]) : x_hi(s.c[k % H]);
        a.d_out[j] = k < H ? x_lo(s.d[k % H]) : x_hi(s.d[k % H]);
        if constexpr (COMP == 1) {
            a.plo_out[j] = k < H ? x_lo(s.plo[k % H]) : x_hi(s.plo[k % H]);
            a.clo_out[j] = k < H ? x_lo(s.clo[k % H]) : x_hi(s.clo[k % H]);
        }
    }
}

// out[2 r] = dV times the sum of record r's strips, in a fixed order
__global__ void __launch_bounds__(32) line_energy_sum(const double* __restrict__ epart, int strips, double dV,
                                                      double* __restrict__ out) {
    const double* p = epart + (long long)blockIdx.x * strips;
    double s = 0.0;
    for (int i = threadIdx.x; i < strips; i += 32) s += p[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) out[2 * blockIdx.x] = s * dV;
}

namespace {

// FP32: two cells per lane and 8 steps while every SM has at most four strips
// (one per scheduler), else four cells and 4 steps.  FP64: one cell and 4 steps
// while there are SMs for all strips, else two cells and 2 steps.
struct LinePlan {
    int J, ks, strips, warps;
};
LinePlan plan_for(const HostProblem& P, int sms) {
    const int n = (int)P.n[0];
    auto strips = [&](int J, int ks) { return (n + 32 * J - 4 * ks - 1) / (32 * J - 4 * ks); };
    if (P.precision == 1) {
        if (strips(1, 4) <= sms) return {1, 4, strips(1, 4), 1};
        return {2, 2, strips(2, 2), 1};
    }
    if (strips(2, 8) <= 4 * sms) return {2, 8, strips(2, 8), 1};
    return {4, 4, strips(4, 4), 4};
}

int line_sms() {
    static DeviceSetup setup;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= DeviceSetup::MAX_DEVICES) {
        cudaGetLastError();
        return 1;
    }
    std::lock_guard<std::mutex> lock(setup.mu);
    if (!setup.done[dev]) {
        int n = 1;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            n = 1;
        }
        setup.sms[dev] = n;
        setup.done[dev] = true;
    }
    return setup.sms[dev];
}

template <typename E>
LineArgs<E> line_args(const HostProblem& P, const LinePlan& pl) {
    LineArgs<E> a = {};
    a.K = make_line_consts<E>(P, -1);
    a.dtq = line_splat<typename LineNum<E>::V>((typename LineNum<E>::S)(P.dt / (P.dx * P.dx)));
    a.n = (int)P.n[0];
    a.strips = pl.strips;
    a.periodic = P.bc_lo[0] == BC_PERIODIC;
    a.H = P.H;
    a.grad = 0.5 * P.sigma / (P.dx * P.dx);
    return a;
}

template <typename E>
void line_state(LineArgs<E>& a, const Fields& in, const Fields* out) {
    using M = typename LineNum<E>::M;
    a.phi = (const M*)in.phi; a.c = (const M*)in.c; a.d = (const M*)in.d;
    a.clo = (const M*)in.clo; a.plo = (const M*)in.plo;
    a.phi_out = out ? (M*)out->phi : nullptr;
    if (!out) return;
    a.c_out = (M*)out->c; a.d_out = (M*)out->d; a.clo_out = (M*)out->clo; a.plo_out = (M*)out->plo;
}

// steps until nothing is left, state buffers and clock advanced
template <typename E, int J, int KS, int COMP, bool ENERGY>
cudaError_t line_run(const HostProblem& P, const LinePlan& pl, LineRun& r, int64_t count) {
    static_assert(KS <= LINE_KMAX, "steps per launch");
    LineArgs<E> a = line_args<E>(P, pl);
    a.epart = r.epart;
    const bool std_phys = line_std(P);
    const int blocks = (pl.strips + pl.warps - 1) / pl.warps;
    for (int64_t done = 0; done < count; done += a.steps) {
        a.steps = (int)std::min<int64_t>(KS, count - done);
        int64_t shifts = r.shifts;
        for (int k = 0; k < a.steps; ++k) {
            const double t = (double)(r.step + k) * P.dt;
            a.m[k] = (int)(shifts - r.shifts);
            a.ke_theta0[k] = (1.0 - P.k_e) *
                             (P.theta_ref + P.G_theta * (P.x0 + P.v_pull * t - (double)shifts * P.dx));
            if (P.shift && r.store) {
                const double tn = (double)(r.step + k + 1) * P.dt;
                while (P.v_pull * tn >= (double)(shifts + 1) * P.dx) shifts += 1;
            }
        }
        a.m[a.steps] = (int)(shifts - r.shifts);
        a.erec = r.erec;
        line_state(a, r.buf[r.cur], r.store ? &r.buf[r.cur ^ 1] : nullptr);
        const cudaError_t e = launch_after(std_phys ? line_kernel<E, J, KS, true, COMP, ENERGY>
                                                    : line_kernel<E, J, KS, false, COMP, ENERGY>,
                                           dim3(blocks), dim3(32 * pl.warps), 0, r.stream, a);
        if (e != cudaSuccess) return e;
        r.erec += a.steps;
        if (r.store) {
            r.cur ^= 1;
            r.step += a.steps;
            r.shifts = shifts;
        }
    }
    return cudaSuccess;
}

}  // namespace

bool line_eligible(const HostProblem& P) {
    if (P.dim != 1) return false;
    const bool periodic = P.bc_lo[0] == BC_PERIODIC;
    return periodic ? (P.G_theta == 0.0 && !P.shift)
                    : P.bc_lo[0] == BC_NOFLUX && (P.bc_hi[0] == BC_NOFLUX || P.bc_hi[0] == BC_DIRICHLET);
}

int line_energy_strips(const HostProblem& P) {
    if (!line_eligible(P) || P.precision != 1) return 0;
    const LinePlan pl = plan_for(P, line_sms());
    return pl.J == 1 ? pl.strips : 0;
}

cudaError_t line_steps(const HostProblem& P, LineRun& r, int64_t count) {
    const LinePlan pl = plan_for(P, line_sms());
    if (P.precision == 1) {
        if (pl.J == 1)
            return r.epart ? line_run<Mono, 1, 4, 0, true>(P, pl, r, count) : line_run<Mono, 1, 4, 0, false>(P, pl, r, count);
        return line_run<double, 2, 2, 0, false>(P, pl, r, count);
    }
    if (pl.J == 2) return line_run<float, 2, 8, 1, false>(P, pl, r, count);
    return line_run<float, 4, 4, 1, false>(P, pl, r, count);
}

cudaError_t line_energy_records(const HostProblem& P, const double* epart, int strips, int64_t count, double* out,
                                cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    line_energy_sum<<<(unsigned)count, 32, 0, s>>>(epart, strips, P.dx, out);
    return cudaGetLastError();
}

}  // namespace pf
