// pf_diag.cu -- FP64 diagnostics (discrete free energy, total solute, front,
// c_max), the 1D moving-window shift and the conversions between the
// caller's (phi, c_s, c_l) and the device state (phi, c, d[, c_lo]).
//
// Reductions are deterministic: a grid fixed by the problem size and the
// device (at most 8 blocks per SM, fewer for small grids, so that a 1D run does
// not launch a thousand idle blocks every step) writes one partial per block
// (warp-shuffle tree inside the block), and a single block sums the partials in
// a fixed order.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include "pf_internal.cuh"
#include "pf_kernels.h"
#include "pf_words.cuh"

namespace pf {

static constexpr int DIAG_THREADS = 256;

size_t diag_scratch_doubles(const HostProblem&) { return 2 * (size_t)DIAG_MAX_BLOCKS; }

// largest grid of the reductions and conversions on the current device: 8
// blocks of 256 threads per SM (the SM count queried once per device), at most
// DIAG_MAX_BLOCKS
static int diag_grid() {
    static DeviceSetup setup;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= DeviceSetup::MAX_DEVICES) {
        cudaGetLastError();
        return DIAG_MAX_BLOCKS;
    }
    std::lock_guard<std::mutex> lock(setup.mu);
    if (!setup.done[dev]) {
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
            cudaGetLastError();
            sms = DIAG_MAX_BLOCKS / 8;
        }
        setup.value[dev] = (size_t)std::min(8 * sms, DIAG_MAX_BLOCKS);
        setup.done[dev] = true;
    }
    return (int)setup.value[dev];
}

// blocks for a grid-stride pass over `items`: one per 64 items up to
// diag_grid(), so that small FP64 problems spread their (slow) FP64 work over
// many SMs
static int diag_blocks(long long items) {
    const long long b = (items + 63) / 64;
    const long long cap = diag_grid();
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

// The FP64 pipe of a GB300 runs at about 1/70 of the FP32 rate, so the sums over FP32
// states are formed in three FP32 words (pf_words.cuh) for a few cells at a time
// and added in FP64.

struct DiagConsts {
    int n[3], bc_lo[3], bc_hi[3], dim, lap, interp;
    double dir_phi, dx, H, sigma, k_e, a, theta0, G_theta, dV;
    // in FP32 words, for FP32 states: 1 + ln k_e, H, -(1 - k_e) theta = th + Gx (i + 1/2), a, dir_phi
    Triple lk3, H3, th3, Gx3, a3, dir3;
};

__device__ __forceinline__ double p_d(const DiagConsts& C, double f) {
    double g = f * (1.0 - f);
    double h = (C.interp == 1) ? f * f * (3.0 - 2.0 * f) : f * f * f * (6.0 * f * f - 15.0 * f + 10.0);
    return h + C.a * (f - 0.5) * g * g;
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// block reduction of two values (sum or max), result valid in thread 0
template <bool MAX>
__device__ void block_reduce2(double& a, double& b) {
    __shared__ double sa[DIAG_THREADS / 32], sb[DIAG_THREADS / 32];
    a = MAX ? warp_max(a) : warp_sum(a);
    b = MAX ? warp_max(b) : warp_sum(b);
    const int w = threadIdx.x / 32, l = threadIdx.x % 32;
    if (l == 0) { sa[w] = a; sb[w] = b; }
    __syncthreads();
    if (w == 0) {
        a = (l < DIAG_THREADS / 32) ? sa[l] : (MAX ? -INFINITY : 0.0);
        b = (l < DIAG_THREADS / 32) ? sb[l] : (MAX ? -INFINITY : 0.0);
        a = MAX ? warp_max(a) : warp_sum(a);
        b = MAX ? warp_max(b) : warp_sum(b);
    }
}

// state accessors: c (with its FP32 low word), d -> c_s, c_l in FP64
template <typename T>
struct StateView {
    const T* phi;
    const T* c;
    const T* d;
    const T* clo;   // nullptr in FP64
    __device__ __forceinline__ double cval(long long i) const {
        return (double)c[i] + (clo ? (double)clo[i] : 0.0);
    }
    // total c, and (ENERGY) phi, p(phi), c_s, c_l of cell i
    template <bool ENERGY>
    __device__ __forceinline__ void cell(const DiagConsts& C, long long i, double& cc, double& f, double& p,
                                         double& s, double& l) const {
        cc = cval(i);
        if (!ENERGY) return;
        f = (double)phi[i];
        const double dd = (double)d[i];
        p = p_d(C, f);
        s = cc + (1.0 - p) * dd;
        l = cc - p * dd;
    }
    // total c, c_s and c_l of cell i in FP32 words, from its p
    __device__ __forceinline__ void cell32(long long i, Triple p, Triple& cc, Triple& s, Triple& l) const {
        cc = {(float)c[i], clo ? (float)clo[i] : 0.0f, 0.0f};
        const float dd = (float)d[i];
        l = cc - p * dd;
        s = l + dd;
    }
};

// the caller's fields (phi, c_s, c_l) read directly (pf_energy_solute_noalloc)
template <typename T>
struct FieldView {
    const T* phi;
    const T* cs;
    const T* cl;
    template <bool ENERGY>
    __device__ __forceinline__ void cell(const DiagConsts& C, long long i, double& cc, double& f, double& p,
                                         double& s, double& l) const {
        f = (double)phi[i];
        s = (double)cs[i];
        l = (double)cl[i];
        p = p_d(C, f);
        cc = p * s + (1.0 - p) * l;   // Eq. model1 with g = p
    }
    __device__ __forceinline__ void cell32(long long i, Triple p, Triple& cc, Triple& s, Triple& l) const {
        s = {(float)cs[i], 0.0f, 0.0f};
        l = {(float)cl[i], 0.0f, 0.0f};
        cc = p * widen(sum2(s.h, -l.h)) + l.h;
    }
};

// A sum of weighted squared differences.
template <typename T>
struct SquareSum;
template <>
struct SquareSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double v, double f, double weight) { s += weight * ((v - f) * (v - f)); }
    __device__ __forceinline__ double total() const { return s; }
};
template <>
struct SquareSum<float> {
    float h = 0.0f, l = 0.0f;
    __device__ __forceinline__ void add(Pair d, float weight) {   // weight: a power of two
        const Pair p = prod2(d.h, d.h);
        const Pair s = sum2(h, weight * p.h);
        h = s.h;
        l += s.l + weight * __fmaf_rn(2.0f * d.h, d.l, p.l);
    }
    __device__ __forceinline__ void add(float v, float f, float weight) { add(sum2(v, -f), weight); }
    __device__ __forceinline__ void settle() {   // after a cell: a small l is added to with small errors
        const Pair s = sum2(h, l);
        h = s.h;
        l = s.l;
    }
    __device__ __forceinline__ double total() const { return (double)h + (double)l; }
};

// position of a cell and the step of a grid-stride loop, advanced without divisions
struct Cursor {
    int i, j, k, si, sj, sk;
    __device__ Cursor(const DiagConsts& C, long long c, long long stride) {
        const long long row = c / C.n[0];
        i = (int)(c - row * C.n[0]);
        k = (int)(row / C.n[1]);
        j = (int)(row - (long long)k * C.n[1]);
        const long long srow = stride / C.n[0];
        si = (int)(stride - srow * C.n[0]);
        sk = (int)(srow / C.n[1]);
        sj = (int)(srow - (long long)sk * C.n[1]);
    }
    __device__ __forceinline__ void next(const DiagConsts& C) {
        i += si;
        if (i >= C.n[0]) { i -= C.n[0]; j += 1; }
        j += sj;
        if (j >= C.n[1]) { j -= C.n[1]; k += 1; }
        k += sk;
    }
};

// Gradient energy: every pair of a cell c and a neighbour of its stencil with the
// Laplacian's weight, s1 the face neighbours', s2 the edge neighbours' (corners of
// a square in 2D).  A pair of cells of the grid is added once, by its lower cell;
// a pair with a ghost beyond a mirror, Dirichlet or halo side belongs to one cell
// only and counts half.
template <int LAP, typename T, typename S>
__device__ __forceinline__ void gradient_pairs(const DiagConsts& C, const T* __restrict__ phi, long long c, int i,
                                               int j, int k, T f, SquareSum<S>& s1, SquareSum<S>& s2) {
    constexpr int DIM = LAP == 3 ? 1 : LAP <= 9 && LAP != 7 ? 2 : 3;
    constexpr bool DIAG = LAP == 9 || LAP == 19;
    const int nx = C.n[0], ny = C.n[1], nz = C.n[2];
    const long long oy = nx, oz = (long long)nx * ny;
    const bool perx = C.bc_hi[0] == BC_PERIODIC, pery = DIM >= 2 && C.bc_hi[1] == BC_PERIODIC,
               perz = DIM == 3 && C.bc_hi[2] == BC_PERIODIC;
    // the neighbour above (p) and below (m) along each axis: in the grid, or wrapped
    const bool px = i < nx - 1 || perx, mx = i > 0 || perx;
    const bool py = DIM >= 2 && (j < ny - 1 || pery), my = DIM >= 2 && (j > 0 || pery);
    const bool pz = DIM == 3 && (k < nz - 1 || perz), mz = DIM == 3 && (k > 0 || perz);
    const long long xp = i < nx - 1 ? 1 : -(long long)(nx - 1), xm = i > 0 ? -1 : nx - 1;
    const long long yp = j < ny - 1 ? oy : -(ny - 1) * oy, ym = j > 0 ? -oy : (ny - 1) * oy;
    const long long zp = k < nz - 1 ? oz : -(nz - 1) * oz;
    const T* q = phi + c;
    const S one = S(1);
    s1.add(px ? q[xp] : f, f, one);
    if constexpr (DIM >= 2) s1.add(py ? q[yp] : f, f, one);
    if constexpr (DIM == 3) s1.add(pz ? q[zp] : f, f, one);
    if constexpr (DIAG) {
        s2.add(px && py ? q[xp + yp] : f, f, one);
        s2.add(mx && py ? q[xm + yp] : f, f, one);
        if constexpr (DIM == 3) {
            s2.add(px && pz ? q[xp + zp] : f, f, one);
            s2.add(mx && pz ? q[xm + zp] : f, f, one);
            s2.add(py && pz ? q[yp + zp] : f, f, one);
            s2.add(my && pz ? q[ym + zp] : f, f, one);
        }
    }
    const bool yz = (DIM < 2 || (py && my)) && (DIM < 3 || (pz && mz));
    if (px && mx && yz) return;
    // A mirror side along x, away from the other sides (the same lanes of a warp
    // throughout the loop when rows are whole warps): the ghosts are the cell's own
    // column, so only its edge neighbours differ.
    if (yz && (px || C.bc_hi[0] == BC_NOFLUX) && (mx || C.bc_lo[0] == BC_NOFLUX)) {
        if constexpr (DIAG) {
            s2.add(q[yp], f, S(0.5));
            s2.add(q[ym], f, S(0.5));
            if constexpr (DIM == 3) {
                s2.add(q[zp], f, S(0.5));
                s2.add(q[k > 0 ? -oz : (nz - 1) * oz], f, S(0.5));
            }
        }
        return;
    }
    for (int dz = (DIM == 3 ? -1 : 0); dz <= (DIM == 3 ? 1 : 0); ++dz)
        for (int dy = (DIM >= 2 ? -1 : 0); dy <= (DIM >= 2 ? 1 : 0); ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                const int away = (dx != 0) + (dy != 0) + (dz != 0);
                if (away == 0 || away > (DIAG ? 2 : 1)) continue;
                const bool in = (dx == 0 || (dx > 0 ? px : mx)) && (dy == 0 || (dy > 0 ? py : my)) &&
                                (dz == 0 || (dz > 0 ? pz : mz));
                if (in) continue;
                SquareSum<S>& s = away == 1 ? s1 : s2;
                const int mi = map_coord(i + dx, nx, C.bc_lo[0], C.bc_hi[0]);
                const int mj = DIM >= 2 ? map_coord(j + dy, ny, C.bc_lo[1], C.bc_hi[1]) : 0;
                const int mk = DIM == 3 ? map_coord(k + dz, nz, C.bc_lo[2], C.bc_hi[2]) : 0;
                if (mi < 0 || mj < 0 || mk == DIR_GHOST) {
                    if constexpr (sizeof(S) == 4) {
                        const Triple d = C.dir3 + -f;
                        s.add(Pair{d.h, d.l}, 0.5f);
                    }
                    else s.add(C.dir_phi, f, 0.5);
                } else {
                    s.add(phi[((long long)mk * ny + mj) * nx + mi], f, S(0.5));
                }
            }
}

// FP64 energy density of a cell without its gradient part
__device__ __forceinline__ double bulk_energy(const DiagConsts& C, double f, double p, double s, double l, int i,
                                              double log_ke) {
    const double theta = C.theta0 - C.G_theta * (((double)i + 0.5) * C.dx);
    const double fs = -(1.0 - C.k_e) * theta + s * (log(s) - log_ke - 1.0);
    const double fl = l * (log(l) - 1.0);
    const double fdw = f * f * (1.0 - f) * (1.0 - f);
    return C.H * fdw + p * fs + (1.0 - p) * fl;
}

// cells whose terms a thread sums in FP32 words before it adds them to its FP64 sums
// (12 operations of the FP64 pipe; 2 % of the time of 32 cells)
constexpr int ENERGY_RUN = 32;

// F_h and S_h.  The FP64 form is bound by the FP64 pipe (two logarithms and the
// pairs).  The terms of an FP32 state's cells are formed in three FP32 words, which
// leaves F_h as exact as FP64 arithmetic does (against extended precision, 48 states
// of 3000 to 130,000 cells: 1e-16 rms either way, the last bit; with two words, whose
// cells of equal value all repeat one rounding, 1.3e-15).  256^3: 0.74 ms, bound
// by instruction issue; two words took 0.53, FP64 arithmetic with each pair of
// neighbours taken twice 5.9.  Threads whose sums are not finite (a concentration
// below ln_triple's range, an overflow) repeat their cells in FP64.
template <int LAP, typename View, typename T>
__global__ void __launch_bounds__(DIAG_THREADS, sizeof(T) == 4 ? 3 : 1)
energy_kernel(View S, const T* __restrict__ phi, const DiagConsts C, const __grid_constant__ LogTable logs,
              double* __restrict__ part) {
    const long long N = (long long)C.n[0] * C.n[1] * C.n[2];
    const long long stride = (long long)gridDim.x * blockDim.x, first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double eF = 0.0, eS = 0.0;
    const double w1 = (LAP == 9 ? 2.0 / 3.0 : LAP == 19 ? 1.0 / 3.0 : 1.0), w2 = 1.0 / 6.0;
    const double grad = 0.5 * C.sigma / (C.dx * C.dx);   // a pair counts twice in the sum over cells, each 1/4
    bool exact = sizeof(T) == 8;
    if constexpr (sizeof(T) == 4) {
        __shared__ LogTable table;   // a copy that lanes read at different entries
        for (int t = threadIdx.x; t < 128; t += DIAG_THREADS) {
            table.r[t] = logs.r[t];
            table.a[t] = logs.a[t];
            table.b[t] = logs.b[t];
            table.c[t] = logs.c[t];
            table.d[t] = logs.d[t];
        }
        __syncthreads();
        const Triple lk = C.lk3, H = C.H3, th = C.th3, Gx = C.Gx3, ai = C.a3;
        Cursor at(C, first, stride);
        for (long long c = first; c < N && !exact;) {
            SquareSum<float> s1, s2;
            Triple E = {0.0f, 0.0f, 0.0f}, Sc = E;
            for (int k = 0; k < ENERGY_RUN && c < N; ++k, c += stride) {
                const float f = phi[c];
                gradient_pairs<LAP>(C, phi, c, at.i, at.j, at.k, f, s1, s2);
                s1.settle();
                s2.settle();
                // p = h + a (f - 1/2) g^2, g = f (1 - f)
                const Triple ff = widen(prod2(f, f));
                Triple p;
                if (C.interp == 1) p = ff * widen(sum2(3.0f, -(f + f)));
                else p = (ff * f) * ((widen(prod2(-15.0f, f)) + 10.0f) + ff * 6.0f);
                const Triple g = widen(sum2(1.0f, -f)) * f, gg = g * g;
                if (C.a != 0.0) p = p + (ai * widen(sum2(f, -0.5f))) * gg;
                Triple cc, s, l;
                S.cell32(c, p, cc, s, l);
                const Triple fl = l * (ln_triple(table, l) + -1.0f);
                Triple fs = s * (ln_triple(table, s) - lk) + th;
                if (C.G_theta != 0.0) fs = fs + Gx * widen(sum2((float)(at.i & ~4095), (float)(at.i & 4095) + 0.5f));
                E = E + ((fl + p * (fs - fl)) + H * gg);
                Sc = Sc + cc;
                at.next(C);
            }
            eS += value(Sc);
            eF += value(E) + grad * (w1 * s1.total() + w2 * s2.total());
            exact = !(isfinite(eF) && isfinite(eS));
        }
    }
    if (exact) {
        SquareSum<double> s1, s2;
        eF = eS = 0.0;
        const double log_ke = log(C.k_e);
        Cursor at(C, first, stride);
        for (long long c = first; c < N; c += stride) {
            double cc, f = 0.0, p = 0.0, s = 0.0, l = 0.0;
            S.template cell<true>(C, c, cc, f, p, s, l);
            eS += cc;
            gradient_pairs<LAP>(C, phi, c, at.i, at.j, at.k, phi[c], s1, s2);
            eF += bulk_energy(C, f, p, s, l, at.i, log_ke);
            at.next(C);
        }
        eF += grad * (w1 * s1.s + w2 * s2.s);
    }
    block_reduce2<false>(eF, eS);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = eF;
        part[gridDim.x + blockIdx.x] = eS;
    }
}

// total c of an FP64 state
__global__ void __launch_bounds__(DIAG_THREADS)
solute_f64_kernel(const double* __restrict__ c, long long n, double* __restrict__ part) {
    double s = 0.0, unused = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        s += c[i];
    block_reduce2<false>(s, unused);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = 0.0;
        part[gridDim.x + blockIdx.x] = s;
    }
}

// out[0..1] = the two sums; with `slot`, out[2 k..2 k+1] for k = *slot, then
// *slot = k + 1 (a record written from a replayed graph)
__global__ void __launch_bounds__(DIAG_THREADS)
finish_sum2(const double* __restrict__ part, int nb, double scale, double* __restrict__ out,
            long long* __restrict__ slot) {
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        a += part[i];
        b += part[nb + i];
    }
    block_reduce2<false>(a, b);
    if (threadIdx.x == 0) {
        long long k = 0;
        if (slot != nullptr) {
            k = *slot;
            *slot = k + 1;
        }
        out[2 * k] = a * scale;
        out[2 * k + 1] = b * scale;
    }
}

// The largest phi = 0.5 crossing along x and the largest c.  Every cell is one
// step of a grid-stride loop (a thread per x row read 32 rows' cells per warp
// access: 0.56 ms at 256^3); a row's largest crossing is the one the scan from
// the hot end would meet first.  An FP32 c is compared word by word: hi + lo is
// normalised, so the pairs order as their sums do; NaN in either word is passed
// over, as fmax passes it over.
template <typename T>
__global__ void __launch_bounds__(DIAG_THREADS)
front_kernel(StateView<T> S, DiagConsts C, double* __restrict__ part) {
    const long long N = (long long)C.n[0] * C.n[1] * C.n[2];
    const long long stride = (long long)gridDim.x * blockDim.x, first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double xf = -INFINITY;
    T bh = -INFINITY, bl = T(0);
    Cursor at(C, first, stride);
    for (long long c = first; c < N; c += stride) {
        const T f = S.phi[c], h = S.c[c], l = S.clo != nullptr ? S.clo[c] : T(0);
        if (at.i < C.n[0] - 1) {
            const T g = S.phi[c + 1];
            if (f >= T(0.5) && g < T(0.5)) {
                const double a = (double)f, b = (double)g;
                xf = fmax(xf, ((double)at.i + 0.5 + (a - 0.5) / (a - b)) * C.dx);
            }
        }
        if ((h > bh || (h == bh && l > bl)) && l == l) {
            bh = h;
            bl = l;
        }
        at.next(C);
    }
    double cm = (double)bh + (double)bl;
    block_reduce2<true>(xf, cm);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = xf;
        part[gridDim.x + blockIdx.x] = cm;
    }
}

__global__ void __launch_bounds__(DIAG_THREADS)
finish_max2(const double* __restrict__ part, int nb, double* __restrict__ out) {
    double a = -INFINITY, b = -INFINITY;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        a = fmax(a, part[i]);
        b = fmax(b, part[nb + i]);
    }
    block_reduce2<true>(a, b);
    if (threadIdx.x == 0) {
        out[0] = (a == -INFINITY) ? NAN : a;
        out[1] = b;
    }
}

// store an FP64 value of c as the state's c (and low word in FP32)
template <typename T>
__device__ __forceinline__ void put_c(T* c, T* clo, long long i, double v) {
    const T hi = (T)v;
    c[i] = hi;
    if (clo) clo[i] = (T)(v - (double)hi);
}

template <typename T>
__global__ void shift_kernel(StateView<T> in, const T* plo_in, T* po, T* co, T* dout, T* clo_out,
                             T* plo_out, int n, double fphi, double fc, double fd) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (i < n - 1) {
            po[i] = in.phi[i + 1];
            co[i] = in.c[i + 1];
            dout[i] = in.d[i + 1];
            if (clo_out) clo_out[i] = in.clo[i + 1];
            if (plo_out) plo_out[i] = plo_in[i + 1];
        } else {
            po[i] = (T)fphi;
            dout[i] = (T)fd;
            put_c(co, clo_out, i, fc);
            if (plo_out) plo_out[i] = (T)(fphi - (double)(T)fphi);
        }
    }
}

template <typename T>
__global__ void to_state_kernel(const T* __restrict__ phi, const T* __restrict__ cs,
                                const T* __restrict__ cl, long long n, DiagConsts C, T* po,
                                T* co, T* dout, T* clo) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double f = (double)phi[i], s = (double)cs[i], l = (double)cl[i];
        const double p = p_d(C, f);
        po[i] = phi[i];
        put_c(co, clo, i, p * s + (1.0 - p) * l);
        dout[i] = (T)(s - l);
    }
}

// FP32 input: the conversion in FP32 arithmetic (the FP64 units of a GB300
// are a small fraction of its FP32 rate).  p(phi) is evaluated in FP32 and
// c = c_l + p (c_s - c_l) is kept exactly as an unevaluated sum hi + lo of
// two floats: c_s - c_l and c_l + p d by TwoSum, p d by an FMA-based exact
// product (Knuth; Dekker), so the stored (c, c_lo) carries ~2^-48 relative
// error with respect to that p.
// one cell: (phi, c_s, c_l) -> (c, c_lo, d)
__device__ __forceinline__ void convert_f32(float f, float s, float l, float a, bool cubic, float& c,
                                            float& clo, float& d) {
    const float g = f * (1.0f - f);
    const float h = cubic ? f * f * (3.0f - 2.0f * f) : f * f * f * (f * (6.0f * f - 15.0f) + 10.0f);
    const float p = h + a * (f - 0.5f) * g * g;
    float dh, dl;
    two_sum(s, -l, dh, dl);
    const float prod = p * dh;
    const float small = fmaf(p, dl, fmaf(p, dh, -prod));
    float hi, e;
    two_sum(l, prod, hi, e);
    const float lo = e + small;
    c = hi + lo;
    clo = lo - (c - hi);
    d = dh;
}

__global__ void __launch_bounds__(DIAG_THREADS)
to_state_f32_kernel(const float* __restrict__ phi, const float* __restrict__ cs,
                    const float* __restrict__ cl, long long n, DiagConsts C, float* __restrict__ po,
                    float* __restrict__ co, float* __restrict__ dout, float* __restrict__ clo,
                    float* __restrict__ plo) {
    const float a = (float)C.a;
    const bool cubic = C.interp == 1;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const float f = phi[i];
        float c, lo, d;
        convert_f32(f, cs[i], cl[i], a, cubic, c, lo, d);
        po[i] = f;
        if (plo) plo[i] = 0.0f;
        co[i] = c;
        clo[i] = lo;
        dout[i] = d;
    }
}

// The same with 16-byte loads and stores, 4 cells per thread and iteration,
// for 16-byte aligned arrays (the conversion from host memory is bound by the
// link, and wide requests keep more bytes in flight per thread); cells
// [4 (n / 4), n) are left to the scalar kernel.
__global__ void __launch_bounds__(DIAG_THREADS)
to_state_f32x4_kernel(const float4* __restrict__ phi, const float4* __restrict__ cs,
                      const float4* __restrict__ cl, long long n4, DiagConsts C, float4* __restrict__ po,
                      float4* __restrict__ co, float4* __restrict__ dout, float4* __restrict__ clo,
                      float4* __restrict__ plo) {
    const float a = (float)C.a;
    const bool cubic = C.interp == 1;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
         i += (long long)gridDim.x * blockDim.x) {
        const float4 f = phi[i], s = cs[i], l = cl[i];
        float4 c, lo, d;
        convert_f32(f.x, s.x, l.x, a, cubic, c.x, lo.x, d.x);
        convert_f32(f.y, s.y, l.y, a, cubic, c.y, lo.y, d.y);
        convert_f32(f.z, s.z, l.z, a, cubic, c.z, lo.z, d.z);
        convert_f32(f.w, s.w, l.w, a, cubic, c.w, lo.w, d.w);
        po[i] = f;
        if (plo) plo[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        co[i] = c;
        clo[i] = lo;
        dout[i] = d;
    }
}

// FP32 conversion of cells [0, n): the wide kernel where every array is 16-byte
// aligned, the scalar kernel for the rest
static void to_state_f32(const float* phi, const float* cs, const float* cl, long long n, const DiagConsts& C,
                         float* po, float* co, float* dout, float* clo, float* plo, int blocks,
                         cudaStream_t s) {
    auto al = [](const void* p) { return p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    long long n4 = 0;
    if (al(phi) && al(cs) && al(cl) && al(po) && al(co) && al(dout) && al(clo) && al(plo)) {
        n4 = n / 4;
        if (n4 > 0)
            to_state_f32x4_kernel<<<blocks, DIAG_THREADS, 0, s>>>(
                (const float4*)phi, (const float4*)cs, (const float4*)cl, n4, C, (float4*)po, (float4*)co,
                (float4*)dout, (float4*)clo, (float4*)plo);
    }
    const long long d = 4 * n4;
    if (d < n)
        to_state_f32_kernel<<<blocks, DIAG_THREADS, 0, s>>>(phi + d, cs + d, cl + d, n - d, C, po + d, co + d,
                                                            dout + d, clo + d, plo ? plo + d : nullptr);
}

// FP32 state: total of c = c_hi + c_lo.  Each thread accumulates its cells as
// a renormalised float pair (TwoSum), so the FP32 pipes do the work; the
// per-thread totals then enter the FP64 block reduction.  Deterministic: the
// cells of a thread and the reduction order are fixed.
__global__ void __launch_bounds__(DIAG_THREADS)
solute_f32_kernel(const float* __restrict__ c, const float* __restrict__ clo, long long n,
                  double* __restrict__ part) {
    float ah = 0.0f, al = 0.0f;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n4 = n / 4;
    const float4* c4 = reinterpret_cast<const float4*>(c);
    const float4* l4 = reinterpret_cast<const float4*>(clo);
    auto add = [&](float x, float y) {
        float s, e;
        two_sum(ah, x, s, e);
        const float t = al + (e + y);
        ah = s + t;
        al = t - (ah - s);
    };
    for (long long i = t0; i < n4; i += stride) {
        const float4 x = c4[i], y = l4[i];
        add(x.x, y.x);
        add(x.y, y.y);
        add(x.z, y.z);
        add(x.w, y.w);
    }
    for (long long i = 4 * n4 + t0; i < n; i += stride) add(c[i], clo[i]);
    double v = (double)ah + (double)al, unused = 0.0;
    block_reduce2<false>(v, unused);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = 0.0;
        part[gridDim.x + blockIdx.x] = v;
    }
}

template <typename T>
__global__ void from_state_kernel(StateView<T> S, long long n, DiagConsts C, T* phi, T* cs, T* cl) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double f = (double)S.phi[i], c = S.cval(i), d = (double)S.d[i];
        const double p = p_d(C, f);
        phi[i] = S.phi[i];
        cs[i] = (T)(c + (1.0 - p) * d);
        cl[i] = (T)(c - p * d);
    }
}

// FP32 state -> (phi, c_s, c_l) in FP32 arithmetic: p(phi) in FP32, then
// c_s = c_hi + fma(1 - p, d, c_lo), c_l = c_hi + fma(-p, d, c_lo), so that the
// low word of c enters before the one rounding of each result
__device__ __forceinline__ void from_f32(float f, float hi, float lo, float d, float a, bool cubic, float& s,
                                         float& l) {
    const float g = f * (1.0f - f);
    const float h = cubic ? f * f * (3.0f - 2.0f * f) : f * f * f * (f * (6.0f * f - 15.0f) + 10.0f);
    const float p = h + a * (f - 0.5f) * g * g;
    s = hi + fmaf(1.0f - p, d, lo);
    l = hi + fmaf(-p, d, lo);
}

__global__ void __launch_bounds__(DIAG_THREADS)
from_state_f32_kernel(const float* __restrict__ phi, const float* __restrict__ c, const float* __restrict__ clo,
                      const float* __restrict__ d, long long n, DiagConsts C, float* __restrict__ po,
                      float* __restrict__ cs, float* __restrict__ cl) {
    const float a = (float)C.a;
    const bool cubic = C.interp == 1;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        float s, l;
        from_f32(phi[i], c[i], clo[i], d[i], a, cubic, s, l);
        po[i] = phi[i];
        cs[i] = s;
        cl[i] = l;
    }
}

// the same, 4 cells per thread and iteration with 16-byte accesses (every
// array 16-byte aligned): the read-back to page-locked host memory is bound by
// the host link, and wide requests keep more bytes in flight per thread
__global__ void __launch_bounds__(DIAG_THREADS)
from_state_f32x4_kernel(const float4* __restrict__ phi, const float4* __restrict__ c,
                        const float4* __restrict__ clo, const float4* __restrict__ d, long long n4, DiagConsts C,
                        float4* __restrict__ po, float4* __restrict__ cs, float4* __restrict__ cl) {
    const float a = (float)C.a;
    const bool cubic = C.interp == 1;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
         i += (long long)gridDim.x * blockDim.x) {
        const float4 f = phi[i], h = c[i], lo = clo[i], dd = d[i];
        float4 s, l;
        from_f32(f.x, h.x, lo.x, dd.x, a, cubic, s.x, l.x);
        from_f32(f.y, h.y, lo.y, dd.y, a, cubic, s.y, l.y);
        from_f32(f.z, h.z, lo.z, dd.z, a, cubic, s.z, l.z);
        from_f32(f.w, h.w, lo.w, dd.w, a, cubic, s.w, l.w);
        po[i] = f;
        cs[i] = s;
        cl[i] = l;
    }
}

static DiagConsts make_diag(const HostProblem& P, int64_t step, int64_t shifts) {
    DiagConsts C;
    for (int a = 0; a < 3; ++a) {
        C.n[a] = (int)P.n[a];
        C.bc_lo[a] = P.bc_lo[a];
        C.bc_hi[a] = P.bc_hi[a];
    }
    C.dim = P.dim;
    C.lap = P.lap;
    C.interp = P.interp;
    C.dir_phi = P.dir_phi;
    C.dx = P.dx;
    C.H = P.H;
    C.sigma = P.sigma;
    C.k_e = P.k_e;
    C.a = P.a;
    const double t = (double)step * P.dt;
    C.theta0 = P.theta_ref + P.G_theta * (P.x0 + P.v_pull * t - (double)shifts * P.dx);
    C.G_theta = P.G_theta;
    C.dV = std::pow(P.dx, P.dim);
    const double log_ke = std::log(P.k_e), lk = 1.0 + log_ke;   // what its rounding leaves goes into the last word
    C.lk3 = triple_of(lk);
    C.lk3.t += (float)((1.0 - (lk - (lk - 1.0))) + (log_ke - (lk - 1.0)));
    C.H3 = triple_of(P.H);
    C.th3 = triple_of((P.k_e - 1.0) * C.theta0);
    C.Gx3 = triple_of((1.0 - P.k_e) * P.G_theta * P.dx);
    C.a3 = triple_of(P.a);
    C.dir3 = triple_of(P.dir_phi);
    return C;
}

template <typename T>
static StateView<T> view(const Fields& f) {
    return StateView<T>{(const T*)f.phi, (const T*)f.c, (const T*)f.d, (const T*)f.clo};
}

template <typename T, typename View>
static void launch_energy(const View& v, const T* phi, const DiagConsts& C, int nb, double* scratch, cudaStream_t s) {
    auto k = C.lap == 3 ? energy_kernel<3, View, T> : C.lap == 5 ? energy_kernel<5, View, T>
           : C.lap == 9 ? energy_kernel<9, View, T> : C.lap == 7 ? energy_kernel<7, View, T>
                                                                  : energy_kernel<19, View, T>;
    static const LogTable logs(0);
    k<<<nb, DIAG_THREADS, 0, s>>>(v, phi, C, logs, scratch);
}

cudaError_t launch_energy_solute(const HostProblem& P, const Fields& f, int64_t step,
                                 int64_t shifts, bool with_energy, double* scratch, double* out,
                                 cudaStream_t s, long long* slot) {
    const DiagConsts C = make_diag(P, step, shifts);
    const int nb = diag_blocks(P.cells());
    if (with_energy) {
        if (P.precision == 1) launch_energy<double>(view<double>(f), (const double*)f.phi, C, nb, scratch, s);
        else launch_energy<float>(view<float>(f), (const float*)f.phi, C, nb, scratch, s);
    } else if (P.precision == 1) {
        solute_f64_kernel<<<nb, DIAG_THREADS, 0, s>>>((const double*)f.c, P.cells(), scratch);
    } else {
        solute_f32_kernel<<<nb, DIAG_THREADS, 0, s>>>((const float*)f.c, (const float*)f.clo, P.cells(), scratch);
    }
    finish_sum2<<<1, DIAG_THREADS, 0, s>>>(scratch, nb, C.dV, out, slot);
    return cudaGetLastError();
}

cudaError_t launch_energy_solute_fields(const HostProblem& P, const void* phi, const void* cs, const void* cl,
                                        int64_t step, int64_t shifts, double* scratch, double* out,
                                        cudaStream_t s) {
    const DiagConsts C = make_diag(P, step, shifts);
    const int nb = diag_blocks(P.cells());
    if (P.precision == 1)
        launch_energy<double>(FieldView<double>{(const double*)phi, (const double*)cs, (const double*)cl},
                              (const double*)phi, C, nb, scratch, s);
    else
        launch_energy<float>(FieldView<float>{(const float*)phi, (const float*)cs, (const float*)cl},
                             (const float*)phi, C, nb, scratch, s);
    finish_sum2<<<1, DIAG_THREADS, 0, s>>>(scratch, nb, C.dV, out, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_front(const HostProblem& P, const Fields& f, double* scratch, double* out,
                         cudaStream_t s) {
    const DiagConsts C = make_diag(P, 0, 0);
    const int nb = diag_blocks(P.cells());
    if (P.precision == 1)
        front_kernel<double><<<nb, DIAG_THREADS, 0, s>>>(view<double>(f), C, scratch);
    else
        front_kernel<float><<<nb, DIAG_THREADS, 0, s>>>(view<float>(f), C, scratch);
    finish_max2<<<1, DIAG_THREADS, 0, s>>>(scratch, nb, out);
    return cudaGetLastError();
}

static double p_host(const HostProblem& P, double f) {
    const double g = f * (1.0 - f);
    const double h = (P.interp == 1) ? f * f * (3.0 - 2.0 * f) : f * f * f * (6.0 * f * f - 15.0 * f + 10.0);
    return h + P.a * (f - 0.5) * g * g;
}

cudaError_t launch_shift(const HostProblem& P, const Fields& in, const Fields& out, cudaStream_t s) {
    const int n = (int)P.n[0];
    const int blocks = (n + 255) / 256;
    const double p = p_host(P, P.dir_phi);
    const double fc = p * P.dir_cs + (1.0 - p) * P.dir_cl, fd = P.dir_cs - P.dir_cl;
    if (P.precision == 1)
        shift_kernel<double><<<blocks, 256, 0, s>>>(view<double>(in), nullptr, (double*)out.phi,
                                                    (double*)out.c, (double*)out.d, nullptr, nullptr, n,
                                                    P.dir_phi, fc, fd);
    else
        shift_kernel<float><<<blocks, 256, 0, s>>>(view<float>(in), (const float*)in.plo, (float*)out.phi,
                                                   (float*)out.c, (float*)out.d, (float*)out.clo,
                                                   (float*)out.plo, n, P.dir_phi, fc, fd);
    return cudaGetLastError();
}

cudaError_t launch_to_state(const HostProblem& P, const void* phi, const void* cs, const void* cl,
                            const Fields& out, cudaStream_t s) {
    const DiagConsts C = make_diag(P, 0, 0);
    const long long n = P.cells();
    if (P.precision == 1)
        to_state_kernel<double><<<diag_grid(), DIAG_THREADS, 0, s>>>(
            (const double*)phi, (const double*)cs, (const double*)cl, n, C, (double*)out.phi,
            (double*)out.c, (double*)out.d, nullptr);
    else
        to_state_f32((const float*)phi, (const float*)cs, (const float*)cl, n, C, (float*)out.phi,
                     (float*)out.c, (float*)out.d, (float*)out.clo, (float*)out.plo, diag_grid(), s);
    return cudaGetLastError();
}

cudaError_t launch_to_state_range(const HostProblem& P, const void* phi, const void* cs, const void* cl,
                                  const Fields& out, long long first, long long count, int blocks,
                                  cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    const DiagConsts C = make_diag(P, 0, 0);
    const int nb = blocks > 0 ? blocks : diag_grid();
    if (P.precision == 1) {
        auto at = [&](const void* p) { return static_cast<const double*>(p) + first; };
        auto to = [&](void* p) { return static_cast<double*>(p) + first; };
        to_state_kernel<double><<<nb, DIAG_THREADS, 0, s>>>(at(phi), at(cs), at(cl), count, C, to(out.phi),
                                                            to(out.c), to(out.d), nullptr);
    } else {
        auto at = [&](const void* p) { return static_cast<const float*>(p) + first; };
        auto to = [&](void* p) { return p ? static_cast<float*>(p) + first : nullptr; };
        to_state_f32(at(phi), at(cs), at(cl), count, C, to(out.phi), to(out.c), to(out.d), to(out.clo),
                     to(out.plo), nb, s);
    }
    return cudaGetLastError();
}

cudaError_t launch_from_state(const HostProblem& P, const Fields& in, void* phi, void* cs, void* cl,
                              cudaStream_t s, int blocks) {
    const DiagConsts C = make_diag(P, 0, 0);
    const long long n = P.cells();
    const int nb = blocks > 0 ? blocks : diag_grid();
    if (P.precision == 1) {
        from_state_kernel<double><<<nb, DIAG_THREADS, 0, s>>>(
            view<double>(in), n, C, (double*)phi, (double*)cs, (double*)cl);
        return cudaGetLastError();
    }
    if (in.clo == nullptr) {   // no low word of c (not a state of this library's FP32 handles)
        from_state_kernel<float><<<nb, DIAG_THREADS, 0, s>>>(
            view<float>(in), n, C, (float*)phi, (float*)cs, (float*)cl);
        return cudaGetLastError();
    }
    auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    const float *f = (const float*)in.phi, *c = (const float*)in.c, *lo = (const float*)in.clo,
                *d = (const float*)in.d;
    long long n4 = 0;
    if (al(f) && al(c) && al(lo) && al(d) && al(phi) && al(cs) && al(cl)) {
        n4 = n / 4;
        if (n4 > 0)
            from_state_f32x4_kernel<<<nb, DIAG_THREADS, 0, s>>>(
                (const float4*)f, (const float4*)c, (const float4*)lo, (const float4*)d, n4, C, (float4*)phi,
                (float4*)cs, (float4*)cl);
    }
    const long long o = 4 * n4;
    if (o < n)
        from_state_f32_kernel<<<nb, DIAG_THREADS, 0, s>>>(f + o, c + o, lo + o, d + o, n - o, C,
                                                                   (float*)phi + o, (float*)cs + o,
                                                                   (float*)cl + o);
    return cudaGetLastError();
}

}  // namespace pf
