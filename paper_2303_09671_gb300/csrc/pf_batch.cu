// pf_batch.cu -- batched 1D pulled fronts in one persistent launch.
//
// Each 1D directional-solidification instance (frozen temperature of Eq. ds1,
// moving window of Sec. "Numerical technique", no-flux cold end, fixed hot end)
// belongs to one CTA, or to a cluster of CTAs where there are fewer instances
// than SMs, which keeps its state phi, c = p c_s + (1-p) c_l, d = c_s - c_l in
// shared memory for `nsteps` steps; global memory is touched only at the start
// and the end of a launch.  Warps step strips of the line in registers
// (pf_line.cuh): the discrete step is the one of the other kernels (Eq.
// phasefield_nonvar with the re-derived driving force at cells; the brackets of
// Eqs. cs_nonvar / cl_nonvar at faces; forward Euler on phi, c, d).  Every
// `check_every` steps the instance's k_v = c_inf / c_max (Sec. "Effect of
// parameter A on velocity-dependent partition coefficient") is evaluated and the
// instance marked converged once |dk_v/dt| stays below a tolerance over a window
// of at least `window` time units; converged instances return at once in later
// launches.  Instances are grouped by block size; the groups run concurrently
// on forked streams and the whole chunk of launches is captured in a CUDA graph
// and replayed.
//
// Bound (256 fronts of 512..8192 cells, FP32): the FP32 pipe, on which a packed
// instruction takes two cycles, at 60 % of its cycles; the rest is warps waiting
// at the block barrier for uneven numbers of strips.  500 steps: 17 ms with one
// cell per thread through shared memory, every face evaluated twice with IEEE
// divisions (634 instructions per cell and step), 4.5 ms with strips (115).  16
// fronts of 2048 cells (a few SMs' work, bound by a step's latency): 8.9 us per
// step, now 1.5 us on clusters of 8.  Their tangents: 32 us, now 3.9 us.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>
#include "pf.h"
#include "pf_dual.cuh"
#include "pf_internal.cuh"
#include "pf_kernels.h"
#include "pf_line.cuh"
#include <cooperative_groups.h>

namespace pf {

namespace cg = cooperative_groups;

// per-instance persistent state (device)
struct BatchState {
    long long off;      // offset of the instance's cells in the packed field arrays
    int n;              // cells
    int converged;      // 0 running, 1 converged, 2 stopped: the state became non-finite
    long long step, shifts;
    double k_prev, t_prev, k_last, dkdt_last;
};

template <typename T>
struct BatchArgs {
    const T* phi;       // packed fields before the launch
    const T* c;
    const T* d;
    const BatchState* st;
    T* phi_out;         // and after it (the same arrays, or others)
    T* c_out;
    T* d_out;
    // COMP: the low words of the values of phi, c, d, one array after the other
    const typename LineNum<T>::S* low;
    typename LineNum<T>::S* low_out;
    long long low_stride;
    BatchState* st_out;
    const int* ids;     // instances of this launch group
    const double* v;    // per-instance pulling velocity
    const double* dt;   // per-instance time step
    int count;
    int nsteps;
    int check_every;
    int cluster;        // CTAs per instance
    int room;           // cells of one buffer of a CTA
    double tol, window, min_travel;
    LineConsts<T> K;    // shared model parameters
    Consts<double> C;   // the same in FP64, rounded to T (energy records, clock)
    double theta_ref, G_theta, x0, c_inf;
    long long energy_every;         // record F_h every this many steps (0: never)
    int energy_slots;               // records per instance in `energy`
    double* energy;                 // [instance][slot] F_h records (device)
    double dir_phi;                 // hot-end ghost phi, for the gradient energy
    T* rec;                         // if set: every step's state and intermediates,
                                    // [instance block of 6 rec_steps n][step][phi|c_s|c_l|mu_s|mu_l|dx^2 phidot][n]
    long long rec_steps;
    double inv_dx2;
};

constexpr int BATCH_TAB = 32;       // steps whose clock is tabulated at once
// cells per lane at most.  FP32: four (8192-cell fronts 4.6 ms per 512 steps;
// with eight, whose 168 registers leave 12 warps per CTA, 4.9 ms).  FP64, bound
// by the FP64 pipe, and runs with derivatives: two (with four, 12 FP64 fronts
// took 5.4 ms instead of 2.9, and the tangents of 16 fronts spilled).
template <typename T>
constexpr int batch_jmax() {
    return sizeof(T) == 4 ? 4 : 2;
}
// warps per CTA at most: FP32 fits 128 registers a thread, the others 168
template <typename T>
constexpr int batch_warps() {
    return sizeof(T) == 4 ? 16 : 12;
}
constexpr int BATCH_WARPS = 16;     // the largest of them
constexpr int BATCH_CLUSTER = 8;    // CTAs per instance at most

// a pair's phi, c_s and c_l before the step and its potentials and rate, into the record
// of the step (cells i of the line go to i - m)
template <typename T, int J>
struct LineRecord {
    using X = typename LineNum<T>::X;
    T* base;          // nullptr: nothing is recorded
    int n, i0, m;
    static constexpr bool on = true;
    __device__ __forceinline__ void one(int i, T f, T c, T d, T s, T l, T r) const {
        if (i < 0 || i >= n) return;
        base[i] = f;
        base[n + i] = c;
        base[2 * n + i] = d;
        base[3 * n + i] = s;
        base[4 * n + i] = l;
        base[5 * n + i] = r;
    }
    template <typename V>
    __device__ __forceinline__ void operator()(int q, const X& f, const X&, const X&, const X& c, const X& d,
                                               const X& s, const X& l, const X& r, const V&) const {
        if (base == nullptr) return;
        const int i = i0 - m + q;
        one(i, x_lo(f), x_lo(c), x_lo(d), x_lo(s), x_lo(l), x_lo(r));
        one(i + J / 2, x_hi(f), x_hi(c), x_hi(d), x_hi(s), x_hi(l), x_hi(r));
    }
};

// J consecutive elements between shared memory and registers, in the widest
// accesses their alignment (J elements, at most 16 bytes) allows
template <typename T, int J>
struct CellBlock {
    using W = typename std::conditional<(J * sizeof(T)) % 16 == 0, uint4, uint2>::type;
    static constexpr int N = (int)(J * sizeof(T) / sizeof(W));
};
template <int J, typename T>
__device__ __forceinline__ void load_cells(const T* p, T (&w)[J]) {
    using B = CellBlock<T, J>;
    typename B::W u[B::N];
#pragma unroll
    for (int k = 0; k < B::N; ++k) u[k] = reinterpret_cast<const typename B::W*>(p)[k];
    memcpy(w, u, sizeof(u));
}
template <int J, typename T>
__device__ __forceinline__ void store_cells(T* p, const T (&w)[J]) {
    using B = CellBlock<T, J>;
    typename B::W u[B::N];
    memcpy(u, w, sizeof(u));
#pragma unroll
    for (int k = 0; k < B::N; ++k) reinterpret_cast<typename B::W*>(p)[k] = u[k];
}

// One instance per cluster of a.cluster CTAs (one CTA: no cluster launch).  Each
// CTA keeps a segment of the line's (phi, c, d) in shared memory, twice; in a
// block of up to J/2 steps every warp takes strips of the line from one copy
// through registers (pf_line.cuh) into the other, so that there is one barrier
// per block and none inside it.  Cells at a segment's ends are also written to
// the neighbouring CTA's copy of them (distributed shared memory).
//
// MODE: a plain run, or one for derivatives without and with records.  COMP: the
// values of phi, c and d are kept as unevaluated FP32 pairs in the runs for
// derivatives, whose error is mostly that of the values' accumulated rounding.
enum { BATCH_PLAIN = 0, BATCH_DERIV = 1, BATCH_RECORD = 2 };
template <typename T, int J, bool STD, int MODE>
__global__ void __launch_bounds__(32 * batch_warps<T>())
batch_kernel(const __grid_constant__ BatchArgs<T> a) {
    using X = typename LineNum<T>::X;
    using V = typename LineNum<T>::V;
    using S = typename LineNum<T>::S;
    constexpr int H = J / 2;
    constexpr int USE = 30 * J;      // cells of a strip that hold results
    constexpr bool REC = MODE == BATCH_RECORD;
    constexpr int COMP = MODE != BATCH_PLAIN && sizeof(S) == 4 ? 2 : 0;
    const int csize = a.cluster;
    const int inst = a.ids[blockIdx.x / csize];
    const BatchState St = a.st[inst];
    if (St.converged) return;        // the same for every CTA of the cluster
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = csize > 1 ? (int)cluster.block_rank() : 0;
    const int n = St.n;
    // The line is stored up to a whole number of strips, its cells from n on
    // holding the Dirichlet state (J of them at least: a block of J/2 steps moves
    // the window by fewer).  Each CTA keeps `mine` cells from lo on, with J copies
    // of its neighbours' cells on either side.
    const int strips = (n + J + USE - 1) / USE;
    const int seg = (strips + csize - 1) / csize * USE;
    const int lo = rank * seg;
    const int mine = max(0, min(seg, strips * USE - lo));
    const LineConsts<T>& K = a.K;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[BATCH_WARPS], cred[BATCH_CLUSTER];
    __shared__ double th0[BATCH_TAB];           // (1 - k_e) theta0 of the tabulated steps
    __shared__ int sh[BATCH_TAB + 1];           // window shifts before each of them since the first, and after the last
    __shared__ int s_done;

    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, warps = NT >> 5;
    const long long off = St.off;
    const int room = a.room;                    // cells of one field: J + segment + J
    T* const sm = reinterpret_cast<T*>(smem) + J;   // own cell 0 of the first field
    S* const sl = reinterpret_cast<S*>(reinterpret_cast<T*>(smem) + 6 * room) + J;   // and of its low word
    for (int i = tid - J; i < room - J; i += NT) {
        const int g = lo + i;
        const bool in = g >= 0 && g < n;
        const T f = in ? a.phi[off + g] : T(K.gphi), c = in ? a.c[off + g] : T(K.fc), d = in ? a.d[off + g] : T(K.fd);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            sm[3 * b * room + i] = f;
            sm[(3 * b + 1) * room + i] = c;
            sm[(3 * b + 2) * room + i] = d;
        }
        if constexpr (COMP) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const S l = in ? a.low[k * a.low_stride + off + g] : k == 0 ? K.gphi_lo : k == 1 ? K.fc_lo : K.fd_lo;
                sl[k * room + i] = l;
                sl[(3 + k) * room + i] = l;
            }
        }
    }
    long long step = St.step, shifts = St.shifts;
    double k_prev = St.k_prev, t_prev = St.t_prev, k_last = St.k_last, dkdt_last = St.dkdt_last;
    int converged = 0;
    const double v = a.v[inst], dtd = a.dt[inst], dxd = a.C.dx;
    const S dtq1 = S(dtd * a.inv_dx2);
    V dtq;
    dtq.x = dtq1;
    dtq.y = dtq1;
    if (tid == 0) s_done = 0;
    auto sync = [&]() {
        if (csize > 1) cluster.sync();
        else __syncthreads();
    };
    // steps to the next look at the state
    int to_check = a.check_every > 0 ? a.check_every - (int)(step % a.check_every) : 0x7fffffff;
    long long to_energy = a.energy_every > 0 ? a.energy_every - step % a.energy_every : 0x7fffffffffffffffll;
    sync();

    int cur = 0;                       // offset of the current copy
    int tab = BATCH_TAB;               // next entry of the clock table (full: refill)
    long long tab_shifts = shifts;     // shifts at the table's first step
    for (int it = 0; it < a.nsteps;) {
        if (tab == BATCH_TAB) {
            // the clock of the next steps: shifts after step j is the smallest
            // count whose successor's distance the window has not yet covered
            if (warp == 0) {
                const double t = (double)(step + lane) * dtd;
                long long k = shifts;
                if (lane > 0)
                    while (v * t >= (double)(k + 1) * dxd) k += 1;
                sh[lane] = (int)(k - shifts);
                th0[lane] = K.one_m_ke * (a.theta_ref + a.G_theta * (a.x0 + v * t - (double)k * dxd));
                if (lane == 31) {
                    const double t2 = (double)(step + BATCH_TAB) * dtd;
                    while (v * t2 >= (double)(k + 1) * dxd) k += 1;
                    sh[BATCH_TAB] = (int)(k - shifts);
                }
            }
            tab = 0;
            tab_shifts = shifts;
            __syncthreads();
        }
        // a block: up to J/2 steps, ending where the state is looked at
        int kb = min(min(H, a.nsteps - it), min(BATCH_TAB - tab, to_check));
        if (to_energy < kb) kb = (int)to_energy;
        const int s0 = sh[tab];
        const int mt = sh[tab + kb] - s0;                 // shifts in the block
        const int nxt = 3 * room - cur;
        for (int u = warp * USE; u < mine; u += warps * USE) {
            const int w0 = u + (lane - 1) * J;            // own index; lane 0 and lane 31: the strip's stale ends
            const int i0 = lo + w0;
            Strip<T, J, COMP> s;
            {
                const T* p = sm + cur + w0;
                T w[J];
                auto get = [&](const T* q, X (&x)[H]) {
                    load_cells<J>(q, w);
#pragma unroll
                    for (int k = 0; k < H; ++k) x[k] = x_pair(w[k], w[k + H]);
                };
                get(p, s.phi);
                get(p + room, s.c);
                get(p + 2 * room, s.d);
                if constexpr (COMP) {
                    const S* l = sl + cur + w0;
                    S z[J];
                    auto getl = [&](const S* q, V (&x)[H]) {
                        load_cells<J>(q, z);
#pragma unroll
                        for (int k = 0; k < H; ++k) x[k] = x_pair(z[k], z[k + H]);
                    };
                    getl(l, s.plo);
                    getl(l + room, s.clo);
                    getl(l + 2 * room, s.dlo);
                }
            }
            // an end of the line in the strip
            const bool edge = lo + u < mt + J + 1 || lo + u + USE + J >= n;
            auto steps = [&](auto e) {
                constexpr bool EDGE = decltype(e)::value;
                for (int k = 0; k < kb; ++k) {
                    const int m = sh[tab + k] - s0;
                    if constexpr (REC) {
                        LineRecord<T, J> rec;
                        rec.base = (lane == 0 || lane == 31)
                                       ? nullptr
                                       : a.rec + 6 * a.rec_steps * off + (long long)(it + k) * 6 * n;
                        rec.n = n;
                        rec.i0 = i0;
                        rec.m = m;
                        line_step<STD, EDGE, T, J, COMP>(K, s, i0, n, m, dtq, th0[tab + k], rec);
                    } else {
                        line_step<STD, EDGE, T, J, COMP>(K, s, i0, n, m, dtq, th0[tab + k], NoRecord());
                    }
                }
            };
            if (edge) steps(std::true_type());
            else steps(std::false_type());
            if (lane != 0 && lane != 31) {
                if (mt == 0) {
                    auto put = [&](T* q, const X (&x)[H]) {
                        T w[J];
#pragma unroll
                        for (int k = 0; k < H; ++k) {
                            w[k] = x_lo(x[k]);
                            w[k + H] = x_hi(x[k]);
                        }
                        store_cells<J>(q, w);
                    };
                    auto putl = [&](S* q, const V (&x)[H]) {
                        S w[J];
#pragma unroll
                        for (int k = 0; k < H; ++k) {
                            w[k] = x[k].x;
                            w[k + H] = x[k].y;
                        }
                        store_cells<J>(q, w);
                    };
                    auto put3 = [&](T* p, S* l) {
                        put(p, s.phi);
                        put(p + room, s.c);
                        put(p + 2 * room, s.d);
                        if constexpr (COMP) {
                            putl(l, s.plo);
                            putl(l + room, s.clo);
                            putl(l + 2 * room, s.dlo);
                        }
                    };
                    T* const p = sm + nxt + w0;
                    S* const l = sl + nxt + w0;
                    put3(p, l);
                    // the neighbours' copies of this CTA's first and last cells
                    if (csize > 1) {
                        auto put_at = [&](int by, int r) {
                            put3(cluster.map_shared_rank(p + by, r), cluster.map_shared_rank(l + by, r));
                        };
                        if (w0 == 0 && rank > 0) put_at(seg, rank - 1);
                        if (w0 + J == seg && rank < csize - 1) put_at(-seg, rank + 1);
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < J; ++k) {
                        const int i = i0 + k - mt;      // the window has dropped mt cells
                        if (i < 0) continue;
                        // cell l of CTA r
                        auto put1 = [&](int l, int r) {
                            T* q = sm + nxt + l;
                            S* z = sl + nxt + l;
                            if (r != rank) {
                                q = cluster.map_shared_rank(q, r);
                                z = cluster.map_shared_rank(z, r);
                            }
                            q[0] = k < H ? x_lo(s.phi[k % H]) : x_hi(s.phi[k % H]);
                            q[room] = k < H ? x_lo(s.c[k % H]) : x_hi(s.c[k % H]);
                            q[2 * room] = k < H ? x_lo(s.d[k % H]) : x_hi(s.d[k % H]);
                            if constexpr (COMP) {
                                z[0] = k < H ? s.plo[k % H].x : s.plo[k % H].y;
                                z[room] = k < H ? s.clo[k % H].x : s.clo[k % H].y;
                                z[2 * room] = k < H ? s.dlo[k % H].x : s.dlo[k % H].y;
                            }
                        };
                        const int r = i >= lo ? rank : rank - 1;     // mt < seg
                        const int l = i - r * seg;
                        put1(l, r);
                        if (csize > 1) {
                            if (l < J && r > 0) put1(l + seg, r - 1);
                            if (l >= seg - J && r < csize - 1) put1(l - seg, r + 1);
                        }
                    }
                }
            }
        }
        it += kb;
        step += kb;
        tab += kb;
        to_check -= kb;
        to_energy -= kb;
        shifts = tab_shifts + sh[tab];
        cur = nxt;
        sync();
        const int own = min(mine, n - lo);     // own cells of the line (may be negative)
        T* const sPhi = sm + cur;
        T* const sC = sPhi + room;
        T* const sD = sC + room;
        // F_h of the new state (the discrete free energy of pf_energy), FP64
        if (to_energy == 0) {
            to_energy = a.energy_every;
            const double tn = (double)step * dtd;
            const Consts<double>& C = a.C;
            const double th = a.theta_ref + a.G_theta * (a.x0 + v * tn - (double)shifts * dxd);
            double e = 0.0;
            for (int i = tid; i < own; i += NT) {
                const double f = (double)value_of(sPhi[i]), cc = (double)value_of(sC[i]), dd = (double)value_of(sD[i]);
                const double g = f * (1.0 - f);
                const double p = p_of(C, f);
                const double cs = cc + (1.0 - p) * dd, cl = cc - p * dd;
                const double tx = th - C.G_theta * (((double)(lo + i) + 0.5) * dxd);
                const double fs = -C.one_m_ke * tx + cs * (log(cs) - C.log_ke - 1.0);
                const double fl = cl * (log(cl) - 1.0);
                // gradient energy: each pair of cells once, from its left cell;
                // mirror ghosts add nothing and the pair with a Dirichlet ghost
                // counts half, as in pf_energy
                double gs = 0.0;
                if (lo + i < n - 1) {
                    const double dphi = (double)value_of(sPhi[i + 1]) - f;
                    gs = dphi * dphi;
                } else if (!K.hot_noflux) {
                    const double dphi = a.dir_phi - f;
                    gs = 0.5 * dphi * dphi;
                }
                e += C.H * g * g + p * fs + (1.0 - p) * fl + 0.5 * C.sigma * gs / (dxd * dxd);
            }
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (lane == 0) red[warp] = e;
            __syncthreads();
            if (tid == 0) {
                double tot = 0.0;
                for (int w = 0; w < warps; ++w) tot += red[w];
                if (csize > 1) *cluster.map_shared_rank(&cred[rank], 0) = tot;
                else cred[0] = tot;
            }
            sync();
            if (tid == 0 && rank == 0) {
                double tot = 0.0;
                for (int r = 0; r < csize; ++r) tot += cred[r];
                const long long slot = step / a.energy_every - 1;
                if (slot < a.energy_slots) a.energy[(long long)inst * a.energy_slots + slot] = tot * dxd;
            }
            sync();
        }
        // steady-state check on k_v = c_inf / c_max
        if (to_check == 0) {
            to_check = a.check_every;
            const double tn = (double)step * dtd;
            // a maximum that keeps a NaN (fmax would drop it): a state that has
            // stopped being finite must not look steady
            auto nanmax = [](double x, double y) { return (y > x || y != y) ? y : x; };
            double cm = -1e300;
            for (int i = tid; i < own; i += NT) cm = nanmax(cm, (double)value_of(sC[i]));
            for (int o = 16; o > 0; o >>= 1) cm = nanmax(cm, __shfl_xor_sync(0xffffffffu, cm, o));
            if (lane == 0) red[warp] = cm;
            __syncthreads();
            if (tid == 0) {
                double m = red[0];
                for (int w = 1; w < warps; ++w) m = nanmax(m, red[w]);
                for (int r = 0; r < csize; ++r) {      // every CTA keeps its own copy of the maxima
                    if (csize > 1) *cluster.map_shared_rank(&cred[rank], r) = m;
                    else cred[0] = m;
                }
            }
            sync();
            if (tid == 0) {
                double m = cred[0];
                for (int r = 1; r < csize; ++r) m = nanmax(m, cred[r]);
                const double k = a.c_inf / m;
                k_last = k;
                if (!isfinite(m)) {
                    s_done = 2;   // non-finite state: the instance stops, not converged
                } else if (tn - t_prev >= a.window) {
                    dkdt_last = fabs(k - k_prev) / (tn - t_prev);
                    s_done = (t_prev > 0.0 && dkdt_last < a.tol && v * tn >= a.min_travel) ? 1 : 0;
                    k_prev = k;
                    t_prev = tn;
                }
            }
            sync();
            if (s_done) {
                converged = s_done;
                break;
            }
        }
    }
    for (int i = tid; i < min(mine, n - lo); i += NT) {
        a.phi_out[off + lo + i] = sm[cur + i];
        a.c_out[off + lo + i] = sm[cur + room + i];
        a.d_out[off + lo + i] = sm[cur + 2 * room + i];
        if constexpr (COMP)
            for (int k = 0; k < 3; ++k) a.low_out[k * a.low_stride + off + lo + i] = sl[cur + k * room + i];
    }
    if (tid == 0 && rank == 0)
        a.st_out[inst] = BatchState{off, n, converged, step, shifts, k_prev, t_prev, k_last, dkdt_last};
}


// (phi, c_s, c_l) -> (phi, c, d) for packed instances, with their low words
// [phi, c, d][n] if low is set
template <typename T>
__global__ void batch_to_state(const T* __restrict__ cs, const T* __restrict__ cl, T* __restrict__ phi,
                               T* __restrict__ c, T* __restrict__ d, long long n, int interp, double a,
                               T* __restrict__ low = nullptr) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double f = (double)phi[i], s = (double)cs[i], l = (double)cl[i];
        const double g = f * (1.0 - f);
        const double h = (interp == 1) ? f * f * (3.0 - 2.0 * f) : f * f * f * (6.0 * f * f - 15.0 * f + 10.0);
        const double p = h + a * (f - 0.5) * g * g;
        const double cc = p * s + (1.0 - p) * l, dd = s - l;
        c[i] = (T)cc;
        d[i] = (T)dd;
        if (low != nullptr) {
            low[i] = T(0);
            low[n + i] = (T)(cc - (double)(T)cc);
            low[2 * n + i] = (T)(dd - (double)(T)dd);
        }
    }
}

template <typename T>
__global__ void batch_from_state(const T* __restrict__ phi, const T* __restrict__ c, const T* __restrict__ d,
                                 T* __restrict__ cs, T* __restrict__ cl, long long n, int interp, double a) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double f = (double)phi[i], cc = (double)c[i], dd = (double)d[i];
        const double g = f * (1.0 - f);
        const double h = (interp == 1) ? f * f * (3.0 - 2.0 * f) : f * f * f * (6.0 * f * f - 15.0 * f + 10.0);
        const double p = h + a * (f - 0.5) * g * g;
        cs[i] = (T)(cc + (1.0 - p) * dd);
        cl[i] = (T)(cc - p * dd);
    }
}

namespace {

// cells per lane: the request rounded to what the type's kernels have (two at
// least, as cells are computed in pairs)
template <typename T>
int cells_per_lane(int cpt) {
    return std::max(2, std::min(cpt, batch_jmax<T>()));
}

// warps of a CTA that has `strips` strips to take: as few as finish them in the
// smallest number of rounds
int warps_for(int64_t strips, int most) {
    const int64_t rounds = (strips + most - 1) / most;
    return (int)((strips + rounds - 1) / rounds);
}

template <typename T>
using BatchFn = void (*)(const BatchArgs<T>);
template <typename T, bool STD, int MODE>
BatchFn<T> batch_fn_J(int J) {
    if constexpr (batch_jmax<T>() >= 4 && MODE == BATCH_PLAIN)
        if (J == 4) return batch_kernel<T, 4, STD, MODE>;
    return batch_kernel<T, 2, STD, MODE>;
}
// the instance for J cells per lane, the default physics or not, and a mode (in
// FP64, which has no low words, BATCH_DERIV is the plain run of the values; dual
// numbers are only run for derivatives and never recorded)
template <typename T>
BatchFn<T> batch_fn(int J, bool std_phys, int mode) {
    if constexpr (IsDual<T>::value) {
        return std_phys ? batch_fn_J<T, true, BATCH_DERIV>(J) : batch_fn_J<T, false, BATCH_DERIV>(J);
    } else {
        if (mode == BATCH_RECORD)
            return std_phys ? batch_fn_J<T, true, BATCH_RECORD>(J) : batch_fn_J<T, false, BATCH_RECORD>(J);
        if constexpr (sizeof(T) == 4)
            if (mode == BATCH_DERIV)
                return std_phys ? batch_fn_J<T, true, BATCH_DERIV>(J) : batch_fn_J<T, false, BATCH_DERIV>(J);
        return std_phys ? batch_fn_J<T, true, BATCH_PLAIN>(J) : batch_fn_J<T, false, BATCH_PLAIN>(J);
    }
}
// bytes of shared memory per cell of a CTA: two copies of the state
template <typename T>
size_t batch_cell_bytes(int mode) {
    using S = typename LineNum<T>::S;
    return 2 * 3 * (sizeof(T) + (mode != BATCH_PLAIN && sizeof(S) == 4 ? sizeof(S) : 0));
}

// `count` clusters of `cluster` CTAs (1: a plain launch)
template <typename Args>
cudaError_t launch_clusters(void (*kern)(const Args), int count, int cluster, int warps, size_t smem, cudaStream_t s,
                            const Args& a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(count * cluster);
    cfg.blockDim = dim3(32 * warps);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cluster;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// CTAs per instance: an instance is spread over a cluster where that fills SMs
// that would otherwise have no instance (16 fronts of 2048 cells, FP32: 2.9 us
// per step on one CTA each, 1.5 us on clusters of 8; sizes in between that are
// no power of two were no faster)
int cluster_for(int64_t strips, int instances, int sms) {
    int c = 1;
    while (2 * c <= BATCH_CLUSTER && 2 * c <= strips && (int64_t)2 * c * instances <= sms) c *= 2;
    return c;
}

// raise each instantiation's dynamic shared-memory limit to what the device
// allows next to the kernel's static shared memory
template <typename K>
cudaError_t raise_smem(K kern, int optin) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                optin - (int)fa.sharedSizeBytes);
}

template <typename T>
cudaError_t set_smem_limits(size_t* max_dynamic, int* sms) {
    static DeviceSetup setup;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= DeviceSetup::MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(setup.mu);
    if (!setup.done[dev]) {
        int optin = 0;
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        for (int J = 2; J <= batch_jmax<T>(); J *= 2) {
            for (int i = 0; i < 6 && e == cudaSuccess; ++i) e = raise_smem(batch_fn<T>(J, i & 1, i / 2), optin);
        }
        int n = 1;
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        setup.sms[dev] = n;
        setup.value[dev] = (size_t)optin - 1024;   // static part: clock table, reduction scratch, flag
        setup.err[dev] = e;
        setup.done[dev] = true;
    }
    *max_dynamic = setup.value[dev];
    *sms = setup.sms[dev];
    return setup.err[dev];
}

// device arrays of one call: listed, then allocated together and freed together
// (ten allocations and frees took 0.3 ms of a call)
struct Arena {
    std::vector<std::pair<void**, size_t>> want;
    void* base = nullptr;
    template <typename P>
    void add(P** p, size_t bytes) {
        want.push_back({reinterpret_cast<void**>(p), (bytes + 255) / 256 * 256});
    }
    cudaError_t allocate() {
        size_t total = 0;
        for (auto& w : want) total += w.second;
        cudaError_t e = cudaMalloc(&base, total > 0 ? total : 256);
        if (e != cudaSuccess) {
            base = nullptr;
            return e;
        }
        char* p = static_cast<char*>(base);
        for (auto& w : want) {
            *w.first = p;
            p += w.second;
        }
        return e;
    }
    ~Arena() {
        if (base) cudaFree(base);
    }
};

struct Group {
    int warps;         // of a CTA
    int dir = -1;      // seeded parameter of a tangent run (0 M_phi, 1 A, 2 b), -1 none
    int room = 0;      // cells of one shared-memory copy
    std::vector<int> ids;
    int* d_ids = nullptr;
    cudaStream_t stream = nullptr;
    cudaEvent_t done = nullptr;
};

template <typename T>
struct BatchRun {
    const pf_batch_desc& D;
    cudaStream_t main;
    std::string& err;
    int64_t total = 0;
    std::vector<int64_t> off;
    std::vector<double> dt;
    T *phi = nullptr, *c = nullptr, *d = nullptr;
    BatchState* st = nullptr;
    typename LineNum<T>::S* low = nullptr;   // runs for derivatives, FP32: [copy][phi, c, d][total] low words
    bool deriv = false;                      // a run for derivatives
    int64_t slot_in = 0, slot_out = 0;   // the copies of the state a launch reads and writes
    double *dv = nullptr, *ddt = nullptr;
    Arena mem;
    int* ids = nullptr;         // instance numbers, group after group
    std::vector<int> ids_host;
    std::vector<Group> groups;
    int J = 2, cluster = 1;     // cells per lane and CTAs per instance of the groups
    bool std_phys = false;
    int sms = 1;
    size_t max_dyn = 0;         // dynamic shared memory of a CTA
    std::vector<int> rep_dir;   // tangent runs: seeded parameter of each instance
    double* energy = nullptr;   // F_h records [instance][slot] (device), or null
    int energy_slots = 0;
    T* rec = nullptr;           // reverse sweeps: per-step state record (not owned)
    long long rec_steps = 0;
    cudaEvent_t fork = nullptr, t0 = nullptr, t1 = nullptr;
    int64_t launches = 0;

    BatchRun(const pf_batch_desc& d_, cudaStream_t s, std::string& e) : D(d_), main(s), err(e) {}
    ~BatchRun() {
        drop_groups();
        if (fork) cudaEventDestroy(fork);
        if (t0) cudaEventDestroy(t0);
        if (t1) cudaEventDestroy(t1);
    }

    int mode() const { return rec ? BATCH_RECORD : low ? BATCH_DERIV : BATCH_PLAIN; }

    // the line of the batch as a problem description (lengths and clocks are the instances')
    HostProblem problem() const {
        pf_grid g1{1, {8, 1, 1}, D.dx};
        HostProblem P;
        fill_problem(P, &g1, &D.bc, &D.params);
        return P;
    }

    BatchArgs<T> args(const Group& g, int nsteps) const {
        BatchArgs<T> a;
        const int64_t i = slot_in * total, o = slot_out * total;
        a.phi = phi + i; a.c = c + i; a.d = d + i; a.st = st + slot_in * D.n_instances;
        a.phi_out = phi + o; a.c_out = c + o; a.d_out = d + o; a.st_out = st + slot_out * D.n_instances;
        a.low = low + (low ? 3 * i : 0);
        a.low_out = low + (low ? 3 * o : 0);
        a.low_stride = total;
        a.ids = g.d_ids; a.v = dv; a.dt = ddt;
        a.count = (int)g.ids.size();
        a.nsteps = nsteps;
        a.check_every = (int)D.check_every;
        a.tol = D.tol;
        a.window = D.window;
        a.min_travel = D.min_travel;
        a.cluster = cluster;
        a.room = g.room;
        const HostProblem P = problem();
        a.K = make_line_consts<T>(P, g.dir);
        using S = typename LineNum<T>::S;
        auto r = [](double x) { return (double)S(x); };
        Consts<double>& C = a.C;
        C = Consts<double>{};
        C.interp = P.interp; C.mobility = P.mobility;
        C.dx = r(P.dx); C.H = r(P.H); C.sigma = r(P.sigma); C.D_s = r(P.D_s); C.D_l = r(P.D_l);
        C.log_ke = r(std::log(P.k_e)); C.one_m_ke = r(1.0 - P.k_e); C.a = r(P.a); C.G_theta = r(P.G_theta);
        set_coefficients(C);
        a.inv_dx2 = 1.0 / (P.dx * P.dx);
        a.theta_ref = P.theta_ref; a.G_theta = P.G_theta; a.x0 = P.x0; a.c_inf = P.c_inf;
        a.energy_every = D.energy_every;
        a.energy_slots = energy_slots;
        a.energy = energy;
        a.dir_phi = D.bc.dir_phi;
        a.rec = rec;
        a.rec_steps = rec_steps;
        return a;
    }

    // `count` launches of nsteps steps each, every group's on its own stream: a
    // group does not wait for the others' launches until the last is done
    cudaError_t issue(int nsteps, int count = 1) {
        cudaError_t e = groups.size() > 1 ? cudaEventRecord(fork, main) : cudaSuccess;
        for (Group& g : groups) {
            const cudaStream_t on = g.stream ? g.stream : main;
            if (e == cudaSuccess && g.stream) e = cudaStreamWaitEvent(on, fork, 0);
            const BatchArgs<T> a = args(g, nsteps);
            for (int l = 0; l < count && e == cudaSuccess; ++l)
                e = launch_clusters(batch_fn<T>(J, std_phys, mode()), a.count, cluster, g.warps,
                                    g.room * batch_cell_bytes<T>(mode()), on, a);
            if (e == cudaSuccess && g.stream) e = cudaEventRecord(g.done, on);
            launches += count;
        }
        for (Group& g : groups)
            if (e == cudaSuccess && g.stream) e = cudaStreamWaitEvent(main, g.done, 0);
        return e;
    }

    void drop_groups() {
        for (Group& g : groups) {
            if (g.stream) cudaStreamDestroy(g.stream);
            if (g.done) cudaEventDestroy(g.done);
        }
        groups.clear();
    }

    cudaError_t make_groups(int cpt) {
        if (!groups.empty()) {   // an earlier choice: its copies of ids may still be read
            const cudaError_t e = cudaStreamSynchronize(main);
            if (e != cudaSuccess) return e;
            drop_groups();
        }
        J = deriv ? 2 : cells_per_lane<T>(cpt);
        std_phys = line_std(problem());
        const int64_t use = 30 * J;
        int64_t most = 0;
        for (int i = 0; i < D.n_instances; ++i) most = std::max(most, (D.n[i] + J + use - 1) / use);
        cluster = cluster_for(most, D.n_instances, sms);
        // a segment has to fit a CTA's shared memory
        const size_t cell = batch_cell_bytes<T>(deriv ? BATCH_DERIV : BATCH_PLAIN);
        while (2 * cluster <= BATCH_CLUSTER && ((most + cluster - 1) / cluster * use + 2 * J) * cell > max_dyn)
            cluster *= 2;
        std::map<std::pair<int, int>, Group> by;
        for (int i = 0; i < D.n_instances; ++i) {
            const int64_t strips = ((D.n[i] + J + use - 1) / use + cluster - 1) / cluster;
            // few block sizes, so that few launches make up a chunk
            const int top = batch_warps<T>();
            int w = warps_for(strips, top);
            for (int step : {1, 2, 4, 6, 9, 12, 16})
                if (w <= step) {
                    w = std::min(step, top);
                    break;
                }
            const int dir = rep_dir.empty() ? -1 : rep_dir[i];
            Group& g = by[{w, dir}];
            g.warps = w;
            g.dir = dir;
            g.room = std::max(g.room, (int)(strips * use + 2 * J));
            g.ids.push_back(i);
        }
        // largest instances first inside a group: the long CTAs start early.  The
        // last group runs on the main stream, the others on their own.
        ids_host.clear();
        for (auto& kv : by) {
            Group g = kv.second;
            std::sort(g.ids.begin(), g.ids.end(), [&](int x, int y) { return D.n[x] > D.n[y]; });
            g.d_ids = ids + ids_host.size();
            ids_host.insert(ids_host.end(), g.ids.begin(), g.ids.end());
            cudaError_t e = cudaSuccess;
            if (groups.size() + 1 < by.size()) {
                e = cudaStreamCreateWithFlags(&g.stream, cudaStreamNonBlocking);
                if (e == cudaSuccess) e = cudaEventCreateWithFlags(&g.done, cudaEventDisableTiming);
            }
            groups.push_back(g);
            if (e != cudaSuccess) return e;
        }
        return cudaMemcpyAsync(ids, ids_host.data(), ids_host.size() * sizeof(int), cudaMemcpyHostToDevice, main);
    }
};

}  // namespace

// per-instance time step: the given one, or 0.9 of the stable step capped so
// that the window moves at most half a cell per step
static bool batch_time_steps(const pf_batch_desc& D, std::vector<double>& out, std::string& err) {
    pf_grid g1{1, {8, 1, 1}, D.dx};
    double dts = 0;
    pf_stable_dt(&g1, &D.params, &dts);
    out.resize(D.n_instances);
    for (int i = 0; i < D.n_instances; ++i) {
        double dt = (D.dt && D.dt[i] > 0) ? D.dt[i] : 0.9 * dts;
        if (!(D.dt && D.dt[i] > 0) && D.v_pull[i] > 0) dt = std::min(dt, 0.5 * D.dx / D.v_pull[i]);
        if (!(dt > 0) || dt > dts * (1 + 1e-12) || D.v_pull[i] * dt >= D.dx) {
            err = "invalid or unstable time step for instance " + std::to_string(i);
            return false;
        }
        out[i] = dt;
    }
    return true;
}

template <typename T>
static int run_batch_T(const pf_batch_desc& D, pf_batch_result* R, cudaStream_t main, std::string& err) {
    BatchRun<T> B(D, main, err);
    const int N = D.n_instances;
    B.off.resize(N);
    B.dt.resize(N);
    for (int i = 0; i < N; ++i) {
        B.off[i] = B.total;
        B.total += D.n[i];
    }
    if (!batch_time_steps(D, B.dt, err)) return PF_EINVAL;
    const size_t fb = (size_t)B.total * sizeof(T);
    T *scs = nullptr, *scl = nullptr;   // c_s and c_l, on the way in and out
    B.mem.add(&B.phi, fb);
    B.mem.add(&B.c, fb);
    B.mem.add(&B.d, fb);
    B.mem.add(&B.st, N * sizeof(BatchState));
    B.mem.add(&B.dv, N * sizeof(double));
    B.mem.add(&B.ddt, N * sizeof(double));
    B.mem.add(&B.ids, N * sizeof(int));
    B.mem.add(&scs, fb);
    B.mem.add(&scl, fb);
    if (D.energy_every > 0) {
        // one record per energy_every steps up to max_steps, NaN where never written
        B.energy_slots = (int)(D.max_steps / D.energy_every);
        B.mem.add(&B.energy, (size_t)N * B.energy_slots * sizeof(double));
    }
    cudaError_t e = B.mem.allocate();
    if (e != cudaSuccess) {
        cudaGetLastError();
        err = std::string("device allocation failed: ") + cudaGetErrorString(e);
        return PF_ENOMEM;
    }
    if (D.energy_every > 0)
        e = cudaMemsetAsync(B.energy, 0xff, (size_t)N * B.energy_slots * sizeof(double), main);
    std::vector<BatchState> hs(N);
    for (int i = 0; i < N; ++i) {
        hs[i] = BatchState{B.off[i], (int)D.n[i], 0, 0, 0, 0.0, 0.0, 0.0, 0.0};
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.phi, D.phi0, fb, cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(scs, D.cs0, fb, cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(scl, D.cl0, fb, cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.st, hs.data(), N * sizeof(BatchState), cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.dv, D.v_pull, N * sizeof(double), cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.ddt, B.dt.data(), N * sizeof(double), cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) {
        batch_to_state<T><<<1216, 256, 0, main>>>(scs, scl, B.phi, B.c, B.d, B.total, D.params.interp, D.params.a);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = set_smem_limits<T>(&B.max_dyn, &B.sms);
    if (e == cudaSuccess) {
        int64_t nbig = 0;
        for (int i = 0; i < N; ++i) nbig = std::max(nbig, (int64_t)D.n[i]);
        if ((size_t)6 * (nbig + 34 * batch_jmax<T>()) * sizeof(T) > B.max_dyn) {   // a copy's padding included
            err = "longest instance does not fit in shared memory";
            return PF_EINVAL;
        }
    }
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&B.fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreate(&B.t0);
    if (e == cudaSuccess) e = cudaEventCreate(&B.t1);
    if (e != cudaSuccess) {
        err = std::string("batch set-up: ") + cudaGetErrorString(e);
        return PF_ECUDA;
    }

    // The cells per lane: the one kernel there is (FP64); for a short run two
    // where the instances leave SMs over for clusters (the run is then bound by
    // the latency of a step) and four otherwise; for a run of at least 1024 steps,
    // in which it is 6 % at most, a timed probe of both on a scratch copy of the
    // initial state.
    int cpt = D.cells_per_thread;
    if (cpt == 0 && batch_jmax<T>() == 2) cpt = 2;
    if (cpt == 0 && D.max_steps < 1024) cpt = 2 * N <= B.sms ? 2 : 4;
    if (cpt == 0) {
        T *bp = nullptr, *bc = nullptr, *bd = nullptr;
        e = cudaMalloc(&bp, fb);
        if (e == cudaSuccess) e = cudaMalloc(&bc, fb);
        if (e == cudaSuccess) e = cudaMalloc(&bd, fb);
        if (e == cudaSuccess) e = cudaMemcpyAsync(bp, B.phi, fb, cudaMemcpyDeviceToDevice, main);
        if (e == cudaSuccess) e = cudaMemcpyAsync(bc, B.c, fb, cudaMemcpyDeviceToDevice, main);
        if (e == cudaSuccess) e = cudaMemcpyAsync(bd, B.d, fb, cudaMemcpyDeviceToDevice, main);
        float best = 1e30f;
        const int probe = 32;
        for (int cand : {2, 4}) {
            if (e != cudaSuccess) break;
            e = B.make_groups(cand);
            if (e == cudaSuccess) e = cudaEventRecord(B.t0, main);
            if (e == cudaSuccess) e = B.issue(probe);
            if (e == cudaSuccess) e = cudaEventRecord(B.t1, main);
            if (e == cudaSuccess) e = cudaEventSynchronize(B.t1);
            float ms = 0;
            if (e == cudaSuccess) cudaEventElapsedTime(&ms, B.t0, B.t1);
            if (e == cudaSuccess && ms < best) {
                best = ms;
                cpt = cand;
            }
            // restore the state the probe advanced
            if (e == cudaSuccess) e = cudaMemcpyAsync(B.phi, bp, fb, cudaMemcpyDeviceToDevice, main);
            if (e == cudaSuccess) e = cudaMemcpyAsync(B.c, bc, fb, cudaMemcpyDeviceToDevice, main);
            if (e == cudaSuccess) e = cudaMemcpyAsync(B.d, bd, fb, cudaMemcpyDeviceToDevice, main);
            if (e == cudaSuccess) e = cudaMemcpyAsync(B.st, hs.data(), N * sizeof(BatchState), cudaMemcpyHostToDevice, main);
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(main);
        if (bp) cudaFree(bp);
        if (bc) cudaFree(bc);
        if (bd) cudaFree(bd);
        if (e != cudaSuccess) {
            err = std::string("batch autotune: ") + cudaGetErrorString(e);
            return PF_ECUDA;
        }
        B.launches = 0;
    }
    e = B.make_groups(cpt);
    if (e != cudaSuccess) {
        err = std::string("batch groups: ") + cudaGetErrorString(e);
        return PF_ECUDA;
    }

    // capture a chunk of launches as a CUDA graph and replay it; a run of fewer than
    // two chunks launches them directly (the capture costs more than it saves)
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    if (D.max_steps / D.launches_per_graph >= 2 * D.steps_per_launch) {
        e = cudaStreamBeginCapture(main, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) e = B.issue((int)D.steps_per_launch, D.launches_per_graph);
        cudaError_t e2 = cudaStreamEndCapture(main, &graph);
        if (e == cudaSuccess) e = e2;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
        if (e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            err = std::string("batch graph: ") + cudaGetErrorString(e);
            return PF_ECUDA;
        }
    }
    const int64_t per_replay = D.steps_per_launch * D.launches_per_graph;
    B.launches = 0;
    float total_ms = 0;
    int64_t done_steps = 0;
    for (;;) {
        // whole graph replays, then the remainder of max_steps launched directly,
        // so that no instance takes more than max_steps steps
        const int64_t left = D.max_steps - done_steps;
        const bool whole = left >= per_replay;
        e = cudaEventRecord(B.t0, main);
        if (whole) {
            if (e == cudaSuccess)
                e = exec ? cudaGraphLaunch(exec, main) : B.issue((int)D.steps_per_launch, D.launches_per_graph);
        } else {
            for (int64_t r = left; r > 0 && e == cudaSuccess; r -= D.steps_per_launch)
                e = B.issue((int)std::min<int64_t>(r, D.steps_per_launch));
        }
        if (e == cudaSuccess) e = cudaEventRecord(B.t1, main);
        if (e == cudaSuccess) e = cudaMemcpyAsync(hs.data(), B.st, N * sizeof(BatchState), cudaMemcpyDeviceToHost, main);
        if (e == cudaSuccess) e = cudaStreamSynchronize(main);
        if (e != cudaSuccess) break;
        float ms = 0;
        cudaEventElapsedTime(&ms, B.t0, B.t1);
        total_ms += ms;
        if (whole && exec) B.launches += (int64_t)D.launches_per_graph * (int64_t)B.groups.size();
        done_steps += whole ? per_replay : left;
        bool all = true;
        for (int i = 0; i < N; ++i)
            if (!hs[i].converged) all = false;
        if (all || done_steps >= D.max_steps) break;
    }
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
        err = std::string("batch run: ") + cudaGetErrorString(e);
        return PF_ECUDA;
    }
    for (int i = 0; i < N; ++i) {
        if (R->k_v) R->k_v[i] = hs[i].k_last;
        if (R->dkdt) R->dkdt[i] = hs[i].dkdt_last;
        if (R->t) R->t[i] = (double)hs[i].step * B.dt[i];
        if (R->steps) R->steps[i] = hs[i].step;
        if (R->converged) R->converged[i] = hs[i].converged == 1 ? 1 : 0;
    }
    R->cells_per_thread = B.J;
    R->launches = B.launches;
    R->gpu_ms = total_ms;
    if (R->energy && B.energy) {
        e = cudaMemcpyAsync(R->energy, B.energy, (size_t)N * B.energy_slots * sizeof(double),
                            cudaMemcpyDeviceToHost, main);
        if (e == cudaSuccess) e = cudaStreamSynchronize(main);
        if (e != cudaSuccess) {
            err = std::string("batch energy records: ") + cudaGetErrorString(e);
            return PF_ECUDA;
        }
    }
    if (R->phi && R->cs && R->cl) {
        batch_from_state<T><<<1216, 256, 0, main>>>(B.phi, B.c, B.d, scs, scl, B.total, D.params.interp, D.params.a);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(R->phi, B.phi, fb, cudaMemcpyDeviceToHost, main);
        if (e == cudaSuccess) e = cudaMemcpyAsync(R->cs, scs, fb, cudaMemcpyDeviceToHost, main);
        if (e == cudaSuccess) e = cudaMemcpyAsync(R->cl, scl, fb, cudaMemcpyDeviceToHost, main);
        if (e == cudaSuccess) e = cudaStreamSynchronize(main);
        if (e != cudaSuccess) {
            err = std::string("batch fields: ") + cudaGetErrorString(e);
            return PF_ECUDA;
        }
    }
    return PF_OK;
}

// Runs on a private non-blocking stream forked from the caller's (which may be
// the legacy default stream, not capturable) and joined back at the end.
template <typename T>
static int run_batch_forked(const pf_batch_desc& D, pf_batch_result* R, cudaStream_t caller, std::string& err) {
    cudaStream_t work = nullptr;
    cudaEvent_t ev = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&work, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(ev, caller);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(work, ev, 0);
    int rc = PF_ECUDA;
    if (e == cudaSuccess) {
        rc = run_batch_T<T>(D, R, work, err);
        cudaError_t e2 = cudaEventRecord(ev, work);
        if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(caller, ev, 0);
        if (e2 == cudaSuccess) e2 = cudaStreamSynchronize(work);
        if (rc == PF_OK && e2 != cudaSuccess) {
            err = std::string("batch join: ") + cudaGetErrorString(e2);
            rc = PF_ECUDA;
        }
    } else {
        err = std::string("batch stream: ") + cudaGetErrorString(e);
    }
    if (ev) cudaEventDestroy(ev);
    if (work) cudaStreamDestroy(work);
    return rc;
}

int run_batch(const pf_batch_desc* D, pf_batch_result* R, void* stream, std::string& err) {
    if (!D || !R) { err = "null argument"; return PF_EINVAL; }
    const pf_params& P = D->params;
    const int64_t nmax = (P.precision == PF_FP64) ? 4096 : 8192;
    if (D->n_instances <= 0 || !D->n || !D->v_pull || !D->phi0 || !D->cs0 || !D->cl0) {
        err = "empty batch or null array";
        return PF_EINVAL;
    }
    for (int i = 0; i < D->n_instances; ++i) {
        if (D->n[i] < 8 || D->n[i] > nmax) { err = "instance length outside 8.." + std::to_string(nmax); return PF_EINVAL; }
        if (!(D->v_pull[i] >= 0) || !std::isfinite(D->v_pull[i])) { err = "negative or non-finite velocity"; return PF_EINVAL; }
    }
    if (!(D->dx > 0) || !(P.k_e > 0 && P.k_e < 1) || !(P.b > 0) || !(P.M_phi > 0) || !(P.H > 0) ||
        !(P.sigma > 0) || !(P.D_s > 0) || !(P.D_l > 0) || !(P.c_inf > 0)) {
        err = "invalid model parameters";
        return PF_EINVAL;
    }
    if (P.precision != PF_FP32 && P.precision != PF_FP64) { err = "precision must be PF_FP32 or PF_FP64"; return PF_EINVAL; }
    if (D->bc.lo[0] != PF_BC_NOFLUX || (D->bc.hi[0] != PF_BC_DIRICHLET && D->bc.hi[0] != PF_BC_NOFLUX)) {
        err = "batch instances need a no-flux cold end and a Dirichlet or no-flux hot end";
        return PF_EINVAL;
    }
    if (D->energy_every < 0 || (D->energy_every > 0 && D->max_steps / D->energy_every > (int64_t)1 << 26)) {
        err = "energy_every must be 0 or leave at most 2^26 records per instance";
        return PF_EINVAL;
    }
    if (D->bc.hi[0] == PF_BC_NOFLUX) {
        for (int i = 0; i < D->n_instances; ++i)
            if (D->v_pull[i] != 0.0) { err = "a moving window needs the Dirichlet hot end"; return PF_EINVAL; }
    }
    if (!(D->bc.dir_cs > 0) || !(D->bc.dir_cl > 0)) { err = "Dirichlet concentrations must be positive"; return PF_EINVAL; }
    if (D->steps_per_launch <= 0 || D->launches_per_graph <= 0 || D->check_every <= 0 || D->max_steps <= 0 ||
        D->steps_per_launch > (1 << 30)) {
        err = "steps_per_launch, launches_per_graph, check_every and max_steps must be positive";
        return PF_EINVAL;
    }
    const int cpt = D->cells_per_thread;
    if (cpt != 0 && cpt != 1 && cpt != 2 && cpt != 4 && cpt != 8) { err = "cells_per_thread must be 0, 1, 2, 4 or 8"; return PF_EINVAL; }
    if (cpt != 0)
        for (int i = 0; i < D->n_instances; ++i)
            if (D->n[i] > (int64_t)1024 * cpt) { err = "cells_per_thread too small for the longest instance"; return PF_EINVAL; }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (P.precision == PF_FP64) return run_batch_forked<double>(*D, R, s, err);
    return run_batch_forked<float>(*D, R, s, err);
}


// ------------------------------------------------------------------ tangents
// packed value state (phi, c, d) of the instances -> the Dual state of every
// (direction, instance) replica, derivative 0 (the initial fields do not
// depend on the parameters)
template <typename V>
__global__ void adjoint_replicate(const V* __restrict__ phi, const V* __restrict__ c, const V* __restrict__ d,
                                  const V* __restrict__ low, long long total, int reps, Dual<V>* P, Dual<V>* Cc,
                                  Dual<V>* Dd, V* __restrict__ L) {
    const long long n = total * reps;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const long long s = k % total;
        P[k] = make_dual<V>(phi[s], V(0));
        Cc[k] = make_dual<V>(c[s], V(0));
        Dd[k] = make_dual<V>(d[s], V(0));
        if (low != nullptr)
            for (int q = 0; q < 3; ++q) L[q * n + k] = low[q * total + s];
    }
}

// per replica: max_x c and the derivative of c at the maximising cell (lowest
// index among ties)
template <typename V>
__global__ void __launch_bounds__(256) adjoint_cmax(const Dual<V>* __restrict__ c, const V* __restrict__ clo,
                                                    const BatchState* __restrict__ st, double* __restrict__ out) {
    const BatchState S = st[blockIdx.x];
    double best = -INFINITY, tan = 0.0;
    int bi = 0x7fffffff;
    for (int i = threadIdx.x; i < S.n; i += blockDim.x) {
        const Dual<V> x = c[S.off + i];
        const double v = (double)x.v + (clo != nullptr ? (double)clo[S.off + i] : 0.0);
        if (v > best || (v == best && i < bi)) {
            best = v;
            tan = (double)x.t;
            bi = i;
        }
    }
    __shared__ double sb[256], st_[256];
    __shared__ int si[256];
    sb[threadIdx.x] = best;
    st_[threadIdx.x] = tan;
    si[threadIdx.x] = bi;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            const double vb = sb[threadIdx.x + o];
            const int ib = si[threadIdx.x + o];
            if (vb > sb[threadIdx.x] || (vb == sb[threadIdx.x] && ib < si[threadIdx.x])) {
                sb[threadIdx.x] = vb;
                st_[threadIdx.x] = st_[threadIdx.x + o];
                si[threadIdx.x] = ib;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[2 * blockIdx.x] = sb[0];
        out[2 * blockIdx.x + 1] = st_[0];
    }
}

template <typename V>
static int run_adjoint_T(const pf_adjoint_desc& A, pf_adjoint_result* R, cudaStream_t main, std::string& err) {
    using T = Dual<V>;
    const pf_batch_desc& D = A.batch;
    const int N = D.n_instances;
    std::vector<int> dirs;
    for (int j = 0; j < 3; ++j)
        if ((A.wrt >> j) & 1) dirs.push_back(j);
    const int ND = (int)dirs.size();
    const int M = N * ND;
    // replicas r = q N + i: instance i, parameter dirs[q]
    std::vector<int64_t> rn(M);
    std::vector<double> rv(M), rdt(M);
    std::vector<int> rdir(M);
    std::vector<double> dt1;
    if (!batch_time_steps(D, dt1, err)) return PF_EINVAL;
    for (int q = 0; q < ND; ++q)
        for (int i = 0; i < N; ++i) {
            rn[q * N + i] = D.n[i];
            rv[q * N + i] = D.v_pull[i];
            rdt[q * N + i] = dt1[i];
            rdir[q * N + i] = dirs[q];
        }
    pf_batch_desc RD = D;
    RD.n_instances = M;
    RD.n = rn.data();
    RD.v_pull = rv.data();
    RD.dt = rdt.data();
    RD.check_every = 0;   // fixed number of steps, no convergence test
    RD.energy_every = 0;
    BatchRun<T> B(RD, main, err);
    B.rep_dir = rdir;
    B.off.resize(M);
    B.dt = rdt;
    int64_t total1 = 0;
    for (int i = 0; i < N; ++i) total1 += D.n[i];
    for (int r = 0; r < M; ++r) {
        B.off[r] = B.total;
        B.total += rn[r];
    }
    const size_t fb = (size_t)B.total * sizeof(T), vb = (size_t)total1 * sizeof(V);
    B.deriv = true;
    V *vphi = nullptr, *vcs = nullptr, *vcl = nullptr, *vc = nullptr, *vd = nullptr, *vlow = nullptr;
    double* dout = nullptr;
    for (T** p : {&B.phi, &B.c, &B.d}) B.mem.add(p, fb);
    B.mem.add(&B.st, M * sizeof(BatchState));
    B.mem.add(&B.dv, M * sizeof(double));
    B.mem.add(&B.ddt, M * sizeof(double));
    B.mem.add(&B.ids, M * sizeof(int));
    for (V** p : {&vphi, &vcs, &vcl, &vc, &vd}) B.mem.add(p, vb);
    if (sizeof(V) == 4) {
        B.mem.add(&vlow, 3 * vb);
        B.mem.add(&B.low, 3 * (size_t)B.total * sizeof(V));
    }
    B.mem.add(&dout, 2 * M * sizeof(double));
    cudaError_t e = B.mem.allocate();
    if (e != cudaSuccess) {
        cudaGetLastError();
        err = std::string("device allocation failed: ") + cudaGetErrorString(e);
        return PF_ENOMEM;
    }
    std::vector<BatchState> hs(M);
    for (int r = 0; r < M; ++r) hs[r] = BatchState{B.off[r], (int)rn[r], 0, 0, 0, 0.0, 0.0, 0.0, 0.0};
    e = cudaMemcpyAsync(vphi, D.phi0, vb, cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(vcs, D.cs0, vb, cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(vcl, D.cl0, vb, cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.st, hs.data(), M * sizeof(BatchState), cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.dv, rv.data(), M * sizeof(double), cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.ddt, rdt.data(), M * sizeof(double), cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) {
        batch_to_state<V><<<1216, 256, 0, main>>>(vcs, vcl, vphi, vc, vd, total1, D.params.interp, D.params.a, vlow);
        adjoint_replicate<V><<<1216, 256, 0, main>>>(vphi, vc, vd, vlow, total1, ND, B.phi, B.c, B.d, B.low);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = set_smem_limits<T>(&B.max_dyn, &B.sms);
    if (e == cudaSuccess) {
        int64_t nbig = 0;
        for (int i = 0; i < N; ++i) nbig = std::max(nbig, (int64_t)D.n[i]);
        if ((size_t)6 * (nbig + 34 * batch_jmax<T>()) * sizeof(T) > B.max_dyn) {   // a copy's padding included
            err = "longest instance does not fit in shared memory";
            return PF_EINVAL;
        }
    }
    const int cpt = D.cells_per_thread > 0 ? D.cells_per_thread : 8;
    if (e == cudaSuccess) e = B.make_groups(cpt);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&B.fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreate(&B.t0);
    if (e == cudaSuccess) e = cudaEventCreate(&B.t1);
    const int64_t chunk = D.steps_per_launch > 0 ? D.steps_per_launch : A.nsteps;
    if (e == cudaSuccess) e = cudaEventRecord(B.t0, main);
    for (int64_t done = 0; done < A.nsteps && e == cudaSuccess; done += chunk)
        e = B.issue((int)std::min(chunk, A.nsteps - done));
    if (e == cudaSuccess) e = cudaEventRecord(B.t1, main);
    if (e == cudaSuccess) {
        adjoint_cmax<V><<<M, 256, 0, main>>>(B.c, B.low ? B.low + B.total : nullptr, B.st, dout);
        e = cudaGetLastError();
    }
    std::vector<double> hout(2 * M);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hout.data(), dout, 2 * M * sizeof(double), cudaMemcpyDeviceToHost, main);
    if (e == cudaSuccess) e = cudaStreamSynchronize(main);
    float ms = 0;
    if (e == cudaSuccess) cudaEventElapsedTime(&ms, B.t0, B.t1);
    if (e != cudaSuccess) {
        err = std::string("adjoint run: ") + cudaGetErrorString(e);
        return PF_ECUDA;
    }
    // k_i = c_inf / c_max,i and dk_i = -c_inf dc_max,i / c_max,i^2; the loss
    const double cinf = D.params.c_inf;
    R->loss = 0.0;
    R->grad[0] = R->grad[1] = R->grad[2] = 0.0;
    for (int i = 0; i < N; ++i) {
        const double cm = hout[2 * i];
        const double k = cinf / cm;
        if (R->k) R->k[i] = k;
        double dk[3] = {0.0, 0.0, 0.0};
        for (int q = 0; q < ND; ++q) dk[dirs[q]] = -cinf * hout[2 * (q * N + i) + 1] / (cm * cm);
        if (R->dk)
            for (int j = 0; j < 3; ++j) R->dk[3 * i + j] = dk[j];
        if (A.k_target) {
            const double res = k - A.k_target[i];
            R->loss += res * res;
            for (int j = 0; j < 3; ++j) R->grad[j] += 2.0 * res * dk[j];
        }
    }
    R->gpu_ms = ms;
    return PF_OK;
}

// ---------------------------------------------------------------------------
// Reverse sweep (pf_adjoint, PF_ADJ_REVERSE): the adjoint of one step of
// batch_kernel, applied backwards over recorded states.  lambda = dk/du for
// the state u = (phi, c, d) of one instance; the parameter derivatives collect
// dk/d(1/M_phi), dk/dA, dk/db from every use inside the step.

// constants of the reverse sweep beside the step's
template <typename T>
struct RevConsts {
    using V = typename LineNum<T>::V;
    V A, oA, b, bm1, c4, dx2, H, inv_Mphi;   // oA = 1 - A, bm1 = b - 1, c4 = 4 dx^2
    T gphi, gcs, gcl, gmus, gmul;            // Dirichlet (hot end) ghost
};

// adjoints of a face's inputs (and of A, b) from those of its fluxes (gc, gd)
template <typename V>
struct FaceAdj {
    V f, cs, cl, pd;          // of each of the two cells' phi, c_s, c_l, rate (half the face's)
    V nphi, nY, nS, nL;       // of the normal differences
    V A, b;                   // of the parameters
};

template <bool STD, typename T, typename V>
__device__ __forceinline__ void line_face_rev(const LineConsts<T>& K, const RevConsts<T>& R, V fL, V fR, V csL, V csR,
                                              V clL, V clR, V pdL, V pdR, V n1, V n2, V n3, V gc, V gd,
                                              FaceAdj<V>& o) {
    const V half = vlit<V>(0.5), two = vlit<V>(2.0), zero = vlit<V>(0.0);
    // forward values (line_face)
    const V f = vmul(vadd(fL, fR), half), cs = vmul(vadd(csL, csR), half), cl = vmul(vadd(clL, clR), half);
    const V d = vsub(cs, cl), P = vmul(vadd(pdL, pdR), half);
    const V p = line_p<STD>(K, f);
    const V omp = vsub(vlit<V>(1.0), p);
    const V Ms = line_M<STD>(K.Ms_c, K.Ms_0, cs), Ml = line_M<STD>(K.Ml_c, K.Ml_0, cl);
    const V bMl = vmul(R.b, Ml);
    const V n0 = vsub(fR, fL), nn = vmul(n0, n0);
    const V M = vfma(bMl, p, vmul(Ms, omp)), G = vadd(nn, K.delta2_dx2);
    V iM, r;
    if constexpr (STD) {
        const V t = vrcp_n(vmul(M, G));
        iM = vmul(t, G);
        r = vmul(t, M);
    } else {
        iM = vrcp_n(M);
        r = vrcp_n(G);
    }
    // F_c = q n_Y w + rd Z + a e afn, F_d = rd (T_s - T_l) + a e (as line_face with
    // a derivative, whose comment gives the reason)
    const V rd = vmul(K.delta2_dx2, r), w = vmul(nn, r), e = vmul(n0, r);
    const V Ts = vmul(Ms, n2), Tl = vmul(Ml, n3), TD = vsub(Ts, Tl);
    const V oAd = vmul(R.oA, d), av = vmul(oAd, P);
    const V u = vfma(R.b, p, omp), ui = vmul(u, iM), MsMl = vmul(Ms, Ml), q = vmul(MsMl, ui);
    const V ppo = vmul(p, omp), D = vsub(Ms, bMl), pi = vmul(ppo, iM);
    const V afn = vmul(D, pi);
    // reverse
    const V gcq = vmul(gc, q), gcn = vmul(gc, n1);
    o.nY = vmul(gcq, w);
    const V lrd = vfma(gc, vfma(p, TD, Tl), vmul(gd, TD));
    const V gae = vfma(gc, afn, gd);                      // adjoint of a e
    const V lnphi = vfma(vmul(vmul(e, rd), two), vsub(vmul(gcq, n1), lrd),
                         vmul(vmul(av, gae), vmul(r, vsub(rd, w))));
    const V gr = vmul(gc, rd), gdr = vmul(gd, rd);
    const V lTs = vfma(gr, p, gdr), lTl = vsub(vmul(gr, omp), gdr);
    V lp = vmul(gr, TD);
    const V lafn = vmul(gc, vmul(av, e)), lD = vmul(lafn, D);
    const V lq = vmul(gcn, w);
    const V w1 = vmul(lafn, pi);
    V lMs = vfma(lq, vmul(Ml, ui), w1), lbMl = vsub(zero, w1), lMl = vmul(vmul(lq, Ms), ui);
    lp = vfma(lD, vmul(iM, vsub(omp, p)), lp);
    const V lqM = vmul(lq, MsMl), lu = vmul(lqM, iM);
    const V liM = vfma(lD, ppo, vmul(lqM, u));
    lp = vfma(lu, R.bm1, lp);
    V lb = vmul(lu, p);
    const V la = vmul(e, gae);
    const V loAd = vmul(la, P);                           // adjoint of (1 - A) d
    const V ld = vmul(loAd, R.oA);
    o.A = vsub(zero, vmul(loAd, d));
    o.pd = vmul(vmul(la, oAd), half);
    lMs = vfma(lTs, n2, lMs);
    o.nS = vmul(lTs, Ms);
    lMl = vfma(lTl, n3, lMl);
    o.nL = vmul(lTl, Ml);
    const V lMb = vsub(zero, vmul(liM, vmul(iM, iM)));
    lMs = vfma(lMb, omp, lMs);
    lp = vsub(lp, vmul(lMb, D));
    lbMl = vfma(lMb, p, lbMl);
    lMl = vfma(lbMl, R.b, lMl);
    o.b = vfma(lbMl, Ml, lb);
    o.nphi = lnphi;
    o.cs = vmul(vfma(lMs, K.Ms_c, ld), half);
    o.cl = vmul(vsub(vmul(lMl, K.Ml_c), ld), half);
    o.f = vmul(vmul(lp, line_dp<STD>(K, f)), half);
}

// adjoints of a rate's inputs from that of the rate, lpd
template <typename V>
struct RateAdj {
    V f, cs, cl, mus, mul, p;   // of the cell's own values (phi without the stencil terms)
    V lap, gp, gs, gl;          // of the stencil sums f_W - 2 f + f_E, f_E - f_W, mu_E - mu_W
    V iMphi, A, b;              // of the parameters
};

template <bool STD, typename T, typename V>
__device__ __forceinline__ void line_rate_rev(const LineConsts<T>& K, const RevConsts<T>& R, V f, V fL, V fR, V sL,
                                              V sR, V lL, V lR, V cs, V cl, V mus, V mul, V p, V pd, V ke_theta, V lpd,
                                              RateAdj<V>& o) {
    const V zero = vlit<V>(0.0), one = vlit<V>(1.0), two = vlit<V>(2.0);
    // forward values (line_rate)
    const V gp = vsub(fR, fL), gs = vsub(sR, sL), gl = vsub(lR, lL);
    const V dp = line_dp<STD>(K, f);
    const V omp = vsub(one, p);
    const V Ms = line_M<STD>(K.Ms_c, K.Ms_0, cs), Ml = line_M<STD>(K.Ml_c, K.Ml_0, cl);
    const V bMl = vmul(R.b, Ml), Msq = vmul(Ms, omp);
    const V M = vfma(bMl, p, Msq), G = vfma(gp, gp, K.delta2_4dx2);
    const V u = vfma(R.b, p, omp);
    V iM, rr, iu;
    if constexpr (STD) {
        const V t = vrcp_n(vmul(M, G));
        iM = vmul(t, G);
        rr = vmul(t, M);
    } else {
        iM = vrcp_n(M);
        rr = vrcp_n(G);
    }
    iu = vrcp_n(u);
    const V d = vsub(cs, cl), pq = vmul(p, omp);
    const V oAb = vmul(R.oA, R.b), dd = vmul(d, d);
    const V com = vmul(vmul(R.c4, vmul(rr, iM)), iu);              // 4 dx^2 rr / (Mbar u)
    const V K2 = vmul(vmul(R.oA, oAb), vmul(com, vmul(dd, pq)));
    const V iKc = vrcp_n(vadd(R.inv_Mphi, K2));
    const V dmu = vsub(mus, mul);
    const V AbMl = vmul(R.A, bMl), pp = vmul(p, p), oAo = vsub(one, vmul(R.A, omp));
    const V Nv = vfma(Msq, oAo, vmul(AbMl, pp));
    const V Dd = vmul(Nv, iM);
    const V Ddd = vmul(Dd, d);
    const V dG = vsub(vsub(vmul(vsub(cs, Ddd), dmu), d), ke_theta);
    const V W = vsub(vmul(Ms, gs), vmul(bMl, gl));
    const V X = vmul(vmul(W, gp), rr);
    // reverse: rate = R / Kc
    const V lRt = vmul(lpd, iKc);
    const V lKc = vsub(zero, vmul(lRt, pd));
    o.iMphi = lKc;
    o.lap = vmul(lRt, K.sigma);
    const V lZ = vmul(lRt, R.dx2);
    const V ldG = vsub(zero, vmul(lZ, dp));
    const V ldp = vsub(zero, vmul(lZ, dG));
    // Z = (1-A) d pq iM X
    const V zi = vmul(lZ, iM), zX = vmul(lZ, X), dpq = vmul(d, pq), oAzX = vmul(R.oA, zX);
    V loA = vmul(vmul(zX, iM), dpq);
    const V e1 = vmul(oAzX, iM);
    V ld = vmul(e1, pq), lpq = vmul(e1, d), liM = vmul(oAzX, dpq);
    const V lX = vmul(vmul(R.oA, zi), dpq);
    const V lW = vmul(lX, vmul(gp, rr));
    // d(gp rr)/dgp = rr (1 - 2 gp^2 rr), without the terms that cancel
    const V lgp0 = vmul(vmul(vmul(lX, W), rr), vfma(vmul(vmul(gp, gp), rr), vlit<V>(-2.0), one));
    V lMs = vmul(lW, gs), lbMl = vsub(zero, vmul(lW, gl));
    o.gs = vmul(lW, Ms);
    o.gl = vsub(zero, vmul(lW, bMl));
    // Kc = 1/M_phi + (1-A)^2 b c4 d^2 pq rr iM / u
    const V ko = vmul(lKc, R.oA), kob = vmul(lKc, oAb);
    const V kd = vmul(dd, pq);
    loA = vfma(vmul(two, kob), vmul(com, kd), loA);
    const V kk = vmul(ko, oAb);                                    // lKc (1-A)^2 b
    ld = vfma(vmul(two, kk), vmul(com, dpq), ld);
    V lb = vmul(vmul(ko, R.oA), vmul(com, kd));
    lpq = vfma(kk, vmul(com, dd), lpq);
    const V kcd = vmul(vmul(kk, vmul(R.c4, iu)), kd);
    const V lrr = vmul(kcd, iM);                                   // of Kc's rr alone
    liM = vfma(kcd, rr, liM);
    const V lu = vsub(zero, vmul(lKc, vmul(K2, iu)));
    V lp = vmul(lu, R.bm1);
    lb = vfma(lu, p, lb);
    // dG = cs dmu - d - (1-k_e) theta - Dd d dmu
    V lcs = vmul(ldG, dmu);
    const V ldmu = vmul(ldG, vsub(cs, Ddd));
    ld = vsub(ld, vmul(ldG, vfma(Dd, dmu, one)));
    const V lDd = vsub(zero, vmul(ldG, vmul(d, dmu)));
    // Dd = Nv iM
    const V lN = vmul(lDd, iM);
    liM = vfma(lDd, Nv, liM);
    V lMsq = vmul(lN, oAo);
    o.A = vsub(vmul(lN, vsub(vmul(bMl, pp), vmul(Msq, omp))), loA);   // (1-A) = 1 - A
    lp = vfma(lN, vmul(R.A, vfma(vmul(two, bMl), p, Msq)), lp);
    lbMl = vfma(lN, vmul(R.A, pp), lbMl);
    // pq, rr, iM, Msq, bMl, Ms, Ml, d
    lp = vfma(lpq, vsub(omp, p), lp);
    o.gp = vsub(lgp0, vmul(vmul(two, lrr), vmul(vmul(rr, rr), gp)));
    const V lden = vsub(zero, vmul(liM, vmul(iM, iM)));
    lMsq = vadd(lMsq, lden);
    lbMl = vfma(lden, p, lbMl);
    lp = vfma(lden, bMl, lp);
    lMs = vfma(lMsq, omp, lMs);
    lp = vsub(lp, vmul(lMsq, Ms));
    const V lMl = vmul(lbMl, R.b);
    o.b = vfma(lbMl, Ml, lb);
    o.cs = vadd(lcs, vfma(lMs, K.Ms_c, ld));
    o.cl = vsub(vmul(lMl, K.Ml_c), ld);
    o.mus = ldmu;
    o.mul = vsub(zero, ldmu);
    o.p = lp;
    // phi of the cell itself: f_dw' and p' (f_dw'' = 2 (1 - 6 phi + 6 phi^2))
    const V ddw = vmul(vfma(f, vfma(f, vlit<V>(6.0), vlit<V>(-6.0)), one), two);
    o.f = vsub(vmul(ldp, line_d2p<STD>(K, f)), vmul(vmul(lZ, R.H), ddw));
}

// a running sum kept as an unevaluated pair in FP32 (TwoSum)
template <typename V>
struct RunningSum {
    V hi, lo;
    __device__ __forceinline__ void add(V x) {
        if constexpr (sizeof(V) == sizeof(float2)) {
            const V s = vadd(hi, x), bb = vsub(s, hi);
            lo = vadd(lo, vadd(vsub(hi, vsub(s, bb)), vsub(x, bb)));
            hi = s;
        } else {
            hi = vadd(hi, x);
        }
    }
    __device__ __forceinline__ double total() const {
        return ((double)hi.x + (double)hi.y) + ((double)lo.x + (double)lo.y);
    }
};

template <typename T>
struct RevArgs {
    const T* rec;            // recorded states and intermediates of the segment (batch_kernel layout)
    long long rec_steps;
    T* lphi;                 // adjoint state, packed like the value state
    T* lc;
    T* ld;
    double* grad;            // [instance][3]: d k_i / d(1/M_phi, A, b), accumulated
    const BatchState* st0;   // per instance at the segment start (off, n, step, shifts)
    const double* v;
    const double* dt;
    int nsteps;              // steps of this segment (<= RMAX_SEG)
    int cluster, room;       // as BatchArgs
    LineConsts<T> K;
    RevConsts<T> R;
    double theta_ref, G_theta, x0, dx, inv_dx2;
};

constexpr int RMAX_SEG = 1024;
template <typename T>
constexpr int rev_warps() {
    return sizeof(T) == 4 ? 12 : 8;   // 168 or 255 registers a thread
}

// Bound by the latency of a step's chain of dependent operations and by the
// shuffles.  It replaces one CTA of 512 threads per instance with 13 arrays of the
// line in shared memory and FP64 sums in every thread: 16 fronts of 2048 cells
// take 4.1 us per step instead of 9.5.
//
// One instance per cluster, as batch_kernel, with two cells per lane: one step
// backwards moves information by two cells, so the first and the last lane of a
// strip are stale after it, and a block is one step.  lambda is kept in the
// frame of the state before the step that is swept next.
template <typename T, bool STD>
__global__ void __launch_bounds__(32 * rev_warps<T>()) reverse_kernel(const __grid_constant__ RevArgs<T> a) {
    using V = typename LineNum<T>::V;
    constexpr int J = 2, USE = 30 * J;
    const int csize = a.cluster;
    const int inst = blockIdx.x / csize;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = csize > 1 ? (int)cluster.block_rank() : 0;
    const BatchState S0 = a.st0[inst];
    const int n = S0.n;
    const long long off = S0.off;
    const int strips = (n + J + USE - 1) / USE;
    const int seg = (strips + csize - 1) / csize * USE;
    const int lo = rank * seg;
    const int mine = max(0, min(seg, strips * USE - lo));
    const LineConsts<T>& K = a.K;
    const RevConsts<T>& R = a.R;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int nsh[RMAX_SEG];         // window shifts that followed each step
    __shared__ double th0[RMAX_SEG];      // (1 - k_e) theta0 of each step
    __shared__ double red[rev_warps<T>()][3], cred[BATCH_CLUSTER][3];
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, warps = NT >> 5;
    const int room = a.room;
    T* const sm = reinterpret_cast<T*>(smem) + J;
    const double v = a.v[inst], dtd = a.dt[inst];
    V dtq;
    dtq.x = dtq.y = T(dtd * a.inv_dx2);
    // batch_kernel's clock over the segment: the shifts after j steps are the
    // smallest count, from the segment's start on, that the distance covers
    auto shifts_at = [&](int j) {
        if (j == 0) return S0.shifts;
        const double t = (double)(S0.step + j) * dtd;
        long long k = max(S0.shifts, (long long)floor(v * t / a.dx) - 1);
        while (v * t >= (double)(k + 1) * a.dx) k += 1;
        return k;
    };
    for (int j = tid; j < a.nsteps; j += NT) {
        const long long k0 = shifts_at(j);
        nsh[j] = (int)(shifts_at(j + 1) - k0);
        th0[j] = K.one_m_ke *
                 (a.theta_ref + a.G_theta * (a.x0 + v * ((double)(S0.step + j) * dtd) - (double)k0 * a.dx));
    }
    __syncthreads();
    {
        // lambda after the last step, moved back by the shifts that followed it
        const int s = nsh[a.nsteps - 1];
        for (int i = tid - J; i < room - J; i += NT) {
            const int g = lo + i, j = g - s;
            const bool in = j >= 0 && g < n;
            const T f = in ? a.lphi[off + j] : T(0), c = in ? a.lc[off + j] : T(0), d = in ? a.ld[off + j] : T(0);
            sm[i] = f;
            sm[room + i] = c;
            sm[2 * room + i] = d;
            sm[3 * room + i] = sm[4 * room + i] = sm[5 * room + i] = T(0);
        }
    }
    auto sync = [&]() {
        if (csize > 1) cluster.sync();
        else __syncthreads();
    };
    sync();
    RunningSum<V> gM, gA, gB;
    gM.hi = gM.lo = gA.hi = gA.lo = gB.hi = gB.lo = vlit<V>(0.0);
    // the recorded values of a lane's two cells: phi, c_s, c_l, mu_s, mu_l, rate
    struct Cells {
        T a[12];
    };
    auto fetch = [&](int it, int u) {
        Cells w;
        const int i0 = lo + u + (lane - 1) * J;
        const T* r = a.rec + 6 * a.rec_steps * off + (long long)it * 6 * n;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int i = i0 + k;
            const bool in = i >= 0 && i < n;
            w.a[k] = in ? r[i] : R.gphi;
            w.a[2 + k] = in ? r[n + i] : R.gcs;
            w.a[4 + k] = in ? r[2 * n + i] : R.gcl;
            w.a[6 + k] = in ? r[3 * n + i] : R.gmus;
            w.a[8 + k] = in ? r[4 * n + i] : R.gmul;
            w.a[10 + k] = in ? r[5 * n + i] : T(0);
        }
        return w;
    };
    Cells next = {};
    if (warp * USE < mine) next = fetch(a.nsteps - 1, warp * USE);
    int cur = 0;
    for (int it = a.nsteps - 1; it >= 0; --it) {
        const int nxt = 3 * room - cur;
        const int s = it > 0 ? nsh[it - 1] : 0;     // shifts before this step: into the earlier frame
        for (int u = warp * USE; u < mine; u += warps * USE) {
            const int w0 = u + (lane - 1) * J, i0 = lo + w0;
            const Cells w = u == warp * USE ? next : fetch(it, u);
            auto pair = [](T x, T y) { return x_pair(x, y); };
            const V f = pair(w.a[0], w.a[1]), cs = pair(w.a[2], w.a[3]), cl = pair(w.a[4], w.a[5]);
            const V mus = pair(w.a[6], w.a[7]), mul = pair(w.a[8], w.a[9]), pd = pair(w.a[10], w.a[11]);
            const T* q = sm + cur + w0;
            const V lf = pair(q[0], q[1]), lc = pair(q[room], q[room + 1]), ld = pair(q[2 * room], q[2 * room + 1]);
            if (u == warp * USE && it > 0) next = fetch(it - 1, u);
            auto left_of = [&](V x) { return x_pair(from_below(x.y), x.x); };
            auto right_of = [&](V x) { return x_pair(x.y, from_above(x.x)); };
            const V p = line_p<STD>(K, f), omp = vsub(vlit<V>(1.0), p);
            const V dmu = vsub(mus, mul), Y = vfma(p, dmu, mul);
            const V fR = right_of(f), sR = right_of(mus), lR = right_of(mul);
            // R1: the face to the right, by its left cell
            const bool real0 = i0 >= 0 && i0 < n, real1 = i0 + 1 >= 0 && i0 + 1 < n;
            FaceAdj<V> o;
            line_face_rev<STD>(K, R, f, fR, cs, right_of(cs), cl, right_of(cl), pd, right_of(pd),
                               vsub(right_of(Y), Y), vsub(sR, mus), vsub(lR, mul), vmul(dtq, vsub(lc, right_of(lc))),
                               vmul(dtq, vsub(ld, right_of(ld))), o);
            auto keep = [&](V x) { return vmask(x, !real0, !real1); };   // no face left of the line or beyond its ghost
            o.f = keep(o.f); o.cs = keep(o.cs); o.cl = keep(o.cl); o.pd = keep(o.pd);
            o.nphi = keep(o.nphi); o.nY = keep(o.nY); o.nS = keep(o.nS); o.nL = keep(o.nL);
            const bool useful = lane != 0 && lane != 31;
            // this cell as the face's left side, and as the right side of its left face
            V af = vadd(vsub(o.f, o.nphi), left_of(vadd(o.f, o.nphi)));
            V acs = vadd(o.cs, left_of(o.cs)), acl = vadd(o.cl, left_of(o.cl));
            const V lpd = vfma(dtq, lf, vadd(o.pd, left_of(o.pd)));
            const V lY = vsub(left_of(o.nY), o.nY);
            // Y = mu_l + p (mu_s - mu_l)
            V ams = vfma(lY, p, vsub(left_of(o.nS), o.nS)), aml = vfma(lY, omp, vsub(left_of(o.nL), o.nL));
            V ap = vmul(lY, dmu);
            // R2: the rate, backwards (cold end: mirror ghost; hot end: Dirichlet)
            V fL = left_of(f), sL = left_of(mus), lL = left_of(mul);
            if (i0 == 0) { fL.x = f.x; sL.x = mus.x; lL.x = mul.x; }
            if (i0 == -1) { fL.y = f.y; sL.y = mus.y; lL.y = mul.y; }
            V xc;
            xc.x = T(i0) + T(0.5);
            xc.y = T(i0 + 1) + T(0.5);
            V th;
            th.x = th.y = T(th0[it]);
            RateAdj<V> z;
            line_rate_rev<STD>(K, R, f, fL, fR, sL, sR, lL, lR, cs, cl, mus, mul, p, pd, vfma(K.ke_G, xc, th), lpd, z);
            auto only = [&](V x) { return vmask(x, !real0, !real1); };
            z.lap = only(z.lap); z.gp = only(z.gp); z.gs = only(z.gs); z.gl = only(z.gl);
            if (useful) {
                gM.add(only(z.iMphi));
                gA.add(vadd(only(z.A), keep(o.A)));
                gB.add(vadd(only(z.b), keep(o.b)));
            }
            // R3: the own rate's stencil centre and its neighbours' stencils
            af = vadd(af, vfma(z.lap, vlit<V>(-2.0), z.f));
            ams = vadd(ams, z.mus);
            aml = vadd(aml, z.mul);
            ap = vadd(ap, z.p);
            acs = vadd(acs, z.cs);
            acl = vadd(acl, z.cl);
            const V up = vadd(z.lap, z.gp), dn = vsub(z.lap, z.gp);   // to the east and to the west neighbour
            V fromL = left_of(up), sfromL = left_of(z.gs), lfromL = left_of(z.gl);
            V fromR = right_of(dn), sfromR = right_of(z.gs), lfromR = right_of(z.gl);
            // the mirrored cold end: the first cell is its own west neighbour
            if (i0 == 0) { fromL.x = dn.x; sfromL.x = -z.gs.x; lfromL.x = -z.gl.x; }
            if (i0 == -1) { fromL.y = dn.y; sfromL.y = -z.gs.y; lfromL.y = -z.gl.y; }
            af = vadd(af, vadd(fromL, fromR));
            ams = vadd(ams, vsub(sfromL, sfromR));
            aml = vadd(aml, vsub(lfromL, lfromR));
            // the pointwise values
            acs = vfma(ams, vrcp_n(cs), acs);
            acl = vfma(aml, vrcp_n(cl), acl);
            const V asum = vadd(acs, acl);
            ap = vsub(ap, vmul(vsub(cs, cl), asum));
            const V nf = only(vadd(lf, vfma(ap, line_dp<STD>(K, f), af)));
            const V nc = only(vadd(lc, asum));
            const V nd = only(vadd(ld, vsub(vmul(acs, omp), vmul(acl, p))));
            const T out[6] = {nf.x, nf.y, nc.x, nc.y, nd.x, nd.y};
            auto put = [&](T* t, int k) {
                t[0] = out[k];
                t[room] = out[2 + k];
                t[2 * room] = out[4 + k];
            };
            if (useful || (s > 0 && i0 < 0)) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int i = i0 + k + s;       // its place in the earlier frame
                    if (i < 0 || i >= n) continue;
                    const int r = i < lo + seg ? rank : rank + 1;
                    const int l = i - r * seg;
                    T* const t = sm + nxt + l;
                    put(r == rank ? t : cluster.map_shared_rank(t, r), k);
                    if (csize > 1) {
                        if (l < J && r > 0)
                            put(r - 1 == rank ? t + seg : cluster.map_shared_rank(t + seg, r - 1), k);
                        if (l >= seg - J && r < csize - 1)
                            put(r + 1 == rank ? t - seg : cluster.map_shared_rank(t - seg, r + 1), k);
                    }
                }
            }
        }
        cur = nxt;
        sync();
    }
    for (int i = tid; i < min(mine, n - lo); i += NT) {
        a.lphi[off + lo + i] = sm[cur + i];
        a.lc[off + lo + i] = sm[cur + room + i];
        a.ld[off + lo + i] = sm[cur + 2 * room + i];
    }
    // parameter derivatives: sums over the lanes, the warps and the CTAs in fixed order
    double vals[3] = {gM.total(), gA.total(), gB.total()};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        for (int o = 16; o > 0; o >>= 1) vals[q] += __shfl_xor_sync(0xffffffffu, vals[q], o);
        if (lane == 0) red[warp][q] = vals[q];
    }
    __syncthreads();
    if (tid < 3) {
        double tot = 0.0;
        for (int w = 0; w < warps; ++w) tot += red[w][tid];
        if (csize > 1) *cluster.map_shared_rank(&cred[rank][tid], 0) = tot;
        else cred[0][tid] = tot;
    }
    sync();
    if (rank == 0 && tid < 3) {
        double tot = 0.0;
        for (int r = 0; r < csize; ++r) tot += cred[r][tid];
        a.grad[3 * inst + tid] += tot;
    }
}

// per instance: max_x c and the lowest maximising index
template <typename V>
__global__ void __launch_bounds__(256) value_cmax(const V* __restrict__ c, const V* __restrict__ clo,
                                                  const BatchState* __restrict__ st, double* __restrict__ cmax,
                                                  int* __restrict__ imax) {
    const BatchState S = st[blockIdx.x];
    double best = -INFINITY;
    int bi = 0x7fffffff;
    for (int i = threadIdx.x; i < S.n; i += blockDim.x) {
        const double x = (double)c[S.off + i] + (clo != nullptr ? (double)clo[S.off + i] : 0.0);
        if (x > best || (x == best && i < bi)) {
            best = x;
            bi = i;
        }
    }
    __shared__ double sb[256];
    __shared__ int si[256];
    sb[threadIdx.x] = best;
    si[threadIdx.x] = bi;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            const double vb = sb[threadIdx.x + o];
            const int ib = si[threadIdx.x + o];
            if (vb > sb[threadIdx.x] || (vb == sb[threadIdx.x] && ib < si[threadIdx.x])) {
                sb[threadIdx.x] = vb;
                si[threadIdx.x] = ib;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        cmax[blockIdx.x] = sb[0];
        imax[blockIdx.x] = si[0];
    }
}

// lambda at the end of the run: d k_i / d c at the maximising cell, -c_inf / c_max^2
template <typename V>
__global__ void seed_lambda(V* __restrict__ lc, const BatchState* __restrict__ st, const double* __restrict__ cmax,
                            const int* __restrict__ imax, double cinf, int N) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    // a run that went non-finite has no maximising cell: nothing is seeded (k is NaN)
    if (i < N && imax[i] >= 0 && imax[i] < st[i].n) lc[st[i].off + imax[i]] = V(-cinf / (cmax[i] * cmax[i]));
}

// the reverse sweep's kernel limits, per device
template <typename V>
static cudaError_t reverse_setup(size_t* max_dynamic) {
    static DeviceSetup setup;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= DeviceSetup::MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(setup.mu);
    if (!setup.done[dev]) {
        int optin = 0;
        cudaFuncAttributes fa = {};
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (e == cudaSuccess) e = raise_smem(reverse_kernel<V, true>, optin);
        if (e == cudaSuccess) e = raise_smem(reverse_kernel<V, false>, optin);
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, reverse_kernel<V, true>);
        setup.err[dev] = e;
        setup.value[dev] = (size_t)optin - fa.sharedSizeBytes;
        setup.done[dev] = true;
    }
    *max_dynamic = setup.value[dev];
    return setup.err[dev];
}

template <typename V>
static int run_adjoint_reverse_T(const pf_adjoint_desc& A, pf_adjoint_result* R, cudaStream_t main, std::string& err) {
    pf_batch_desc D = A.batch;
    D.check_every = 0;   // a fixed number of steps
    D.energy_every = 0;
    const int N = D.n_instances;
    BatchRun<V> B(D, main, err);
    B.off.resize(N);
    for (int i = 0; i < N; ++i) {
        B.off[i] = B.total;
        B.total += D.n[i];
    }
    if (!batch_time_steps(D, B.dt, err)) return PF_EINVAL;
    int64_t nmax = 0;
    for (int i = 0; i < N; ++i) nmax = std::max(nmax, (int64_t)D.n[i]);
    const int64_t most = std::min<int64_t>(RMAX_SEG, A.nsteps);
    int64_t seg = std::min<int64_t>(
        A.checkpoint_every > 0 ? (int64_t)A.checkpoint_every : (int64_t)std::ceil(std::sqrt((double)A.nsteps)), most);
    int64_t nseg = 0;
    const size_t fb = (size_t)B.total * sizeof(V);
    B.deriv = true;
    V *scs = nullptr, *scl = nullptr, *rec = nullptr, *lphi = nullptr, *lc = nullptr, *ld = nullptr;
    double *grad = nullptr, *cmax = nullptr;
    int* imax = nullptr;
    cudaError_t e = cudaSuccess;
    for (;; seg = std::min(2 * seg, most)) {
        nseg = (A.nsteps + seg - 1) / seg;
        // States before every segment (each segment's run reads its own and writes
        // the next), the final state, and one for the re-runs' results, which nothing
        // reads: slots 0 .. nseg + 1 of every array.
        const size_t slots = (size_t)nseg + 2;
        B.mem.want.clear();
        for (V** p : {&B.phi, &B.c, &B.d}) B.mem.add(p, fb * slots);
        if (sizeof(V) == 4) B.mem.add(&B.low, 3 * fb * slots);
        B.mem.add(&B.st, N * slots * sizeof(BatchState));
        B.mem.add(&B.dv, N * sizeof(double));
        B.mem.add(&B.ddt, N * sizeof(double));
        B.mem.add(&B.ids, N * sizeof(int));
        for (V** p : {&scs, &scl, &lphi, &lc, &ld}) B.mem.add(p, fb);
        B.mem.add(&rec, fb * 6 * seg * 2);
        B.mem.add(&grad, 3 * N * sizeof(double));
        B.mem.add(&cmax, N * sizeof(double));
        B.mem.add(&imax, N * sizeof(int));
        e = B.mem.allocate();
        // Checkpoints that do not fit are taken twice as far apart (the results' sums
        // then group otherwise, no more), while that saves more than the records (12
        // words a cell and step of a segment) grow: with their low words FP32 checkpoints take 6 words, and dense
        // ones that fitted with 3 still have to run.
        if (e == cudaSuccess || seg == most || 4 * seg >= nseg) break;
        cudaGetLastError();
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        err = std::string("device allocation failed: ") + cudaGetErrorString(e);
        return PF_ENOMEM;
    }
    std::vector<BatchState> hs(N);
    for (int i = 0; i < N; ++i) hs[i] = BatchState{B.off[i], (int)D.n[i], 0, 0, 0, 0.0, 0.0, 0.0, 0.0};
    e = cudaMemcpyAsync(B.phi, D.phi0, fb, cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(scs, D.cs0, fb, cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(scl, D.cl0, fb, cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.st, hs.data(), N * sizeof(BatchState), cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.dv, D.v_pull, N * sizeof(double), cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(B.ddt, B.dt.data(), N * sizeof(double), cudaMemcpyHostToDevice, main);
    if (e == cudaSuccess) e = cudaMemsetAsync(lphi, 0, fb, main);
    if (e == cudaSuccess) e = cudaMemsetAsync(lc, 0, fb, main);
    if (e == cudaSuccess) e = cudaMemsetAsync(ld, 0, fb, main);
    if (e == cudaSuccess) e = cudaMemsetAsync(grad, 0, 3 * N * sizeof(double), main);
    if (e == cudaSuccess) {
        batch_to_state<V><<<1216, 256, 0, main>>>(scs, scl, B.phi, B.c, B.d, B.total, D.params.interp, D.params.a,
                                                  B.low);
        e = cudaGetLastError();
    }
    size_t max_rev = 0;
    if (e == cudaSuccess) e = set_smem_limits<V>(&B.max_dyn, &B.sms);
    if (e == cudaSuccess) e = reverse_setup<V>(&max_rev);
    constexpr int RUSE = 60;                       // reverse_kernel's cells per strip that hold results
    const int64_t rstrips = (nmax + 2 + RUSE - 1) / RUSE;
    const int rcluster = cluster_for(rstrips, N, B.sms);
    const int64_t rper = (rstrips + rcluster - 1) / rcluster;
    const int rroom = (int)(rper * RUSE + 4);
    const size_t rsmem = (size_t)6 * rroom * sizeof(V);
    if (e == cudaSuccess && rsmem > max_rev) {
        err = "longest instance does not fit in shared memory for the reverse sweep";
        return PF_EINVAL;
    }
    if (e == cudaSuccess && (size_t)6 * (nmax + 34 * batch_jmax<V>()) * sizeof(V) > B.max_dyn) {
        err = "longest instance does not fit in shared memory";
        return PF_EINVAL;
    }
    const int cpt = D.cells_per_thread > 0 ? D.cells_per_thread : 2;
    if (e == cudaSuccess) e = B.make_groups(cpt);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&B.fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreate(&B.t0);
    if (e == cudaSuccess) e = cudaEventCreate(&B.t1);
    if (e == cudaSuccess) e = cudaEventRecord(B.t0, main);
    // forward: segment s from slot s into slot s + 1
    for (int64_t s = 0; s < nseg && e == cudaSuccess; ++s) {
        const int64_t len = std::min(seg, A.nsteps - s * seg);
        B.slot_in = s;
        B.slot_out = s + 1;
        e = B.issue((int)len);
    }
    if (e == cudaSuccess) {
        const V* cf = B.c + nseg * B.total;
        const BatchState* sf = B.st + nseg * N;
        value_cmax<V><<<N, 256, 0, main>>>(cf, B.low ? B.low + (3 * nseg + 1) * B.total : nullptr, sf, cmax, imax);
        seed_lambda<V><<<(N + 255) / 256, 256, 0, main>>>(lc, sf, cmax, imax, D.params.c_inf, N);
        e = cudaGetLastError();
    }
    // backwards: re-run each segment recording every step (main stream, the
    // batch kernel) and sweep it (a second stream, the reverse kernel).  The
    // records are double-buffered, so the re-run of segment s-1 overlaps the
    // sweep of segment s; the sweeps run in order on their stream.
    cudaStream_t rs = nullptr;
    cudaEvent_t erec[2] = {nullptr, nullptr}, erev[2] = {nullptr, nullptr};
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&rs, cudaStreamNonBlocking);
    for (int b = 0; b < 2 && e == cudaSuccess; ++b) {
        e = cudaEventCreateWithFlags(&erec[b], cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&erev[b], cudaEventDisableTiming);
    }
    B.rec_steps = seg;
    const size_t rec_elems = (size_t)6 * seg * B.total;
    auto rerun = [&](int64_t s) {
        const int b = (int)(s & 1);
        const int64_t len = std::min(seg, A.nsteps - s * seg);
        cudaError_t x = cudaSuccess;
        if (s + 2 < nseg) x = cudaStreamWaitEvent(main, erev[b], 0);   // the sweep of s+2 read this buffer
        B.slot_in = s;
        B.slot_out = nseg + 1;
        B.rec = rec + b * rec_elems;
        if (x == cudaSuccess) x = B.issue((int)len);
        if (x == cudaSuccess) x = cudaEventRecord(erec[b], main);
        return x;
    };
    RevArgs<V> ra = {};
    {
        const HostProblem P = B.problem();
        auto v2 = [](double x) {
            typename LineNum<V>::V r;
            r.x = r.y = V(x);
            return r;
        };
        const double dx2 = P.dx * P.dx;
        ra.K = make_line_consts<V>(P, -1);
        ra.R.A = v2(P.A); ra.R.oA = v2(1.0 - P.A); ra.R.b = v2(P.b); ra.R.bm1 = v2(P.b - 1.0);
        ra.R.c4 = v2(4.0 * dx2); ra.R.dx2 = v2(dx2); ra.R.H = v2(P.H); ra.R.inv_Mphi = v2(1.0 / P.M_phi);
        ra.R.gphi = ra.K.gphi; ra.R.gcs = V(P.dir_cs); ra.R.gcl = V(P.dir_cl);
        ra.R.gmus = V(std::log(P.dir_cs) - std::log(P.k_e));
        ra.R.gmul = V(std::log(P.dir_cl));
        ra.rec_steps = seg;
        ra.lphi = lphi; ra.lc = lc; ra.ld = ld; ra.grad = grad; ra.v = B.dv; ra.dt = B.ddt;
        ra.cluster = rcluster; ra.room = rroom;
        ra.theta_ref = P.theta_ref; ra.G_theta = P.G_theta; ra.x0 = P.x0;
        ra.dx = (double)V(P.dx);
        ra.inv_dx2 = 1.0 / dx2;
    }
    if (e == cudaSuccess) e = rerun(nseg - 1);
    for (int64_t s = nseg - 1; s >= 0 && e == cudaSuccess; --s) {
        const int b = (int)(s & 1);
        e = cudaStreamWaitEvent(rs, erec[b], 0);
        if (e == cudaSuccess) {
            ra.rec = rec + b * rec_elems;
            ra.st0 = B.st + s * N;
            ra.nsteps = (int)std::min(seg, A.nsteps - s * seg);
            e = launch_clusters(B.std_phys ? reverse_kernel<V, true> : reverse_kernel<V, false>, N, rcluster,
                                warps_for(rper, rev_warps<V>()), rsmem, rs, ra);
        }
        if (e == cudaSuccess) e = cudaEventRecord(erev[b], rs);
        if (e == cudaSuccess && s > 0) e = rerun(s - 1);
    }
    if (e == cudaSuccess) e = cudaStreamWaitEvent(main, erev[0], 0);   // the sweep of segment 0
    if (rs) {
        cudaStreamSynchronize(rs);
        cudaStreamDestroy(rs);
    }
    for (int b = 0; b < 2; ++b) {
        if (erec[b]) cudaEventDestroy(erec[b]);
        if (erev[b]) cudaEventDestroy(erev[b]);
    }
    if (e == cudaSuccess) e = cudaEventRecord(B.t1, main);
    std::vector<double> hg(3 * N), hc(N);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hg.data(), grad, 3 * N * sizeof(double), cudaMemcpyDeviceToHost, main);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hc.data(), cmax, N * sizeof(double), cudaMemcpyDeviceToHost, main);
    if (e == cudaSuccess) e = cudaStreamSynchronize(main);
    float ms = 0;
    if (e == cudaSuccess) cudaEventElapsedTime(&ms, B.t0, B.t1);
    if (e != cudaSuccess) {
        err = std::string("reverse adjoint run: ") + cudaGetErrorString(e);
        return PF_ECUDA;
    }
    const double cinf = D.params.c_inf, Mphi = D.params.M_phi;
    R->loss = 0.0;
    R->grad[0] = R->grad[1] = R->grad[2] = 0.0;
    for (int i = 0; i < N; ++i) {
        const double k = cinf / hc[i];
        if (R->k) R->k[i] = k;
        // d k / d(1/M_phi) -> d k / d M_phi
        const double all[3] = {hg[3 * i] * (-1.0 / (Mphi * Mphi)), hg[3 * i + 1], hg[3 * i + 2]};
        double dk[3];
        for (int j = 0; j < 3; ++j) dk[j] = ((A.wrt >> j) & 1) ? all[j] : 0.0;
        if (R->dk)
            for (int j = 0; j < 3; ++j) R->dk[3 * i + j] = dk[j];
        if (A.k_target) {
            const double res = k - A.k_target[i];
            R->loss += res * res;
            for (int j = 0; j < 3; ++j) R->grad[j] += 2.0 * res * dk[j];
        }
    }
    R->gpu_ms = ms;
    return PF_OK;
}

int run_adjoint(const pf_adjoint_desc* A, pf_adjoint_result* R, void* stream, std::string& err) {
    if (!A || !R) { err = "null argument"; return PF_EINVAL; }
    const pf_batch_desc& D = A->batch;
    const pf_params& P = D.params;
    if (A->nsteps <= 0 || A->nsteps > (int64_t(1) << 40)) { err = "nsteps must be positive"; return PF_EINVAL; }
    if (A->wrt <= 0 || A->wrt > 7) { err = "wrt must be a non-empty set of PF_ADJ_* bits"; return PF_EINVAL; }
    if (A->mode != PF_ADJ_TANGENT && A->mode != PF_ADJ_REVERSE) { err = "mode must be PF_ADJ_TANGENT or PF_ADJ_REVERSE"; return PF_EINVAL; }
    if (A->checkpoint_every < 0) { err = "checkpoint_every must be >= 0"; return PF_EINVAL; }
    const int64_t nmax = (P.precision == PF_FP64) ? 2048 : 4096;
    if (D.n_instances <= 0 || !D.n || !D.v_pull || !D.phi0 || !D.cs0 || !D.cl0) { err = "empty batch or null array"; return PF_EINVAL; }
    for (int i = 0; i < D.n_instances; ++i) {
        if (D.n[i] < 8 || D.n[i] > nmax) { err = "instance length outside 8.." + std::to_string(nmax); return PF_EINVAL; }
        if (!(D.v_pull[i] >= 0) || !std::isfinite(D.v_pull[i])) { err = "negative or non-finite velocity"; return PF_EINVAL; }
    }
    if (!(D.dx > 0) || !(P.k_e > 0 && P.k_e < 1) || !(P.b > 0) || !(P.M_phi > 0) || !(P.H > 0) ||
        !(P.sigma > 0) || !(P.D_s > 0) || !(P.D_l > 0) || !(P.c_inf > 0)) {
        err = "invalid model parameters";
        return PF_EINVAL;
    }
    if (P.precision != PF_FP32 && P.precision != PF_FP64) { err = "precision must be PF_FP32 or PF_FP64"; return PF_EINVAL; }
    if (D.bc.lo[0] != PF_BC_NOFLUX || D.bc.hi[0] != PF_BC_DIRICHLET) {
        err = "instances need a no-flux cold end and a Dirichlet hot end";
        return PF_EINVAL;
    }
    if (!(D.bc.dir_cs > 0) || !(D.bc.dir_cl > 0)) { err = "Dirichlet concentrations must be positive"; return PF_EINVAL; }
    const int cpt = D.cells_per_thread;
    if (cpt != 0 && cpt != 1 && cpt != 2 && cpt != 4 && cpt != 8) { err = "cells_per_thread must be 0, 1, 2, 4 or 8"; return PF_EINVAL; }
    for (int i = 0; i < D.n_instances; ++i)
        if (D.n[i] > (int64_t)1024 * (cpt > 0 ? cpt : 8)) { err = "cells_per_thread too small for the longest instance"; return PF_EINVAL; }
    if (D.steps_per_launch < 0 || D.steps_per_launch > (1 << 30)) { err = "steps_per_launch must be in 0..2^30"; return PF_EINVAL; }
    if (D.steps_per_launch == 0 && A->nsteps > (1 << 30)) { err = "nsteps above 2^30 needs steps_per_launch"; return PF_EINVAL; }
    cudaStream_t caller = static_cast<cudaStream_t>(stream);
    cudaStream_t work = nullptr;
    cudaEvent_t ev = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&work, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(ev, caller);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(work, ev, 0);
    int rc = PF_ECUDA;
    if (e == cudaSuccess) {
        if (A->mode == PF_ADJ_REVERSE)
            rc = (P.precision == PF_FP64) ? run_adjoint_reverse_T<double>(*A, R, work, err)
                                          : run_adjoint_reverse_T<float>(*A, R, work, err);
        else
            rc = (P.precision == PF_FP64) ? run_adjoint_T<double>(*A, R, work, err) : run_adjoint_T<float>(*A, R, work, err);
        cudaError_t e2 = cudaEventRecord(ev, work);
        if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(caller, ev, 0);
        if (e2 == cudaSuccess) e2 = cudaStreamSynchronize(work);
        if (rc == PF_OK && e2 != cudaSuccess) {
            err = std::string("adjoint join: ") + cudaGetErrorString(e2);
            rc = PF_ECUDA;
        }
    } else {
        err = std::string("adjoint stream: ") + cudaGetErrorString(e);
    }
    if (ev) cudaEventDestroy(ev);
    if (work) cudaStreamDestroy(work);
    return rc;
}

}  // namespace pf

namespace {
thread_local std::string g_batch_error;
}

extern "C" int pf_run_batch(const pf_batch_desc* desc, pf_batch_result* res, void* stream) {
    g_batch_error.clear();
    const int rc = pf::run_batch(desc, res, stream, g_batch_error);
    if (rc != PF_OK) pf::set_create_error(g_batch_error);
    return rc;
}

extern "C" int pf_adjoint(const pf_adjoint_desc* desc, pf_adjoint_result* res, void* stream) {
    g_batch_error.clear();
    const int rc = pf::run_adjoint(desc, res, stream, g_batch_error);
    if (rc != PF_OK) pf::set_create_error(g_batch_error);
    return rc;
}
