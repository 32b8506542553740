// pic_particles.cu -- marker kernels of libpic (sm_103a).
//
// Markers are stored as structure-of-arrays (cell int32, offset t from the cell's centre, momentum p,
// iterates delta and p_new, caller index id) and kept sorted by the key
// (cell, velocity bin), so the 32 lanes of a warp hold markers of one or two
// cells with similar displacements.  Each warp of a sweep owns one contiguous range
// of markers, reads it coalesced one step ahead, evaluates the fields from the
// polynomial of each cell (pic_poly.cuh) through the L1 cache, and sums its
// deposits as moments of the cells in a register window, written to global memory
// when the window moves on.  No shared memory, so nothing is staged per block and
// the field tables may be of any size.
//
// Precision discipline of the FP32 form: per-marker arithmetic is float; the
// marker weight w, the cell width dx and every spline normalisation enter in double,
// when the tables are formed and when the solves read the moments; the momentum and
// position updates share one float factor tau = dt/dx (fields are staged as
// e dx and a), so the discrete work identity (p^(k+1) - p^n) vbar =
// (Ebar - F)(x^(k+1) - x^n) of Sec. 4.2 holds with the same rounded factor on both
// sides.
#include <algorithm>
#include <climits>
#include <mutex>
#include <type_traits>

#include "pic_internal.h"
#include "pic_poly.cuh"
#include "pic_solve.cuh"
#include "pic_sweep.cuh"

namespace pic {

template <int K, typename R, int ACC>
__global__ void __launch_bounds__(SweepShape<R, K>::threads1, SweepShape<R, K>::blocks1) k_sweep1(Sweep1Args A)
{
    long long wb, we;
    grid_warp_chunk(A.np, wb, we);
    double dmax = 0.0;
    bool bad = false;
    sweep1_range<K, R, ACC, false>(A, wb, we, dmax, bad);
    if (bad) atomicOr(&A.ctrl->status, STATUS_NUMERIC);
    sweep_max_to(&A.ctrl->dmax_bits, dmax);
}

// ---------------------------------------------------------------------------
// Start of subsystem I with a predicted field: the proposal x^(0) = x^n + delta^(0)
// (the explicit predictor dt p^n / gamma(p^n, A(x^n)), written here, or the learned
// one already in delta) and its path-integrated current j^(0), deposited as in the
// sweeps, so that the fixed-point loop can start from e^(0) = e^n - M1^{-1} j^(0),
// the field consistent with x^(0).  The fixed point does not depend on the start;
// the starting field sets how far the first sweep's kick is off.
// ---------------------------------------------------------------------------
template <int K, typename R, int ACC>
__global__ void __launch_bounds__(SweepShape<R, K>::threads1, SweepShape<R, K>::blocks1) k_predeposit(Sweep1Args A)
{
    long long wb, we;
    grid_warp_chunk(A.np, wb, we);
    double dmax = 0.0;
    bool bad = false;
    sweep1_range<K, R, ACC, true>(A, wb, we, dmax, bad);
    if (bad) atomicOr(&A.ctrl->status, STATUS_NUMERIC);
}

// Instantiations: double form with double lanes; float form with compensated
// lanes for every degree, and with plain float or double lanes (kept to
// compare the deposit accumulations) for k = 3 and 5.
#define PIC_FOR_SWEEP_VARIANTS(X)                                                                   \
    X(2, double, ACC_NATIVE) X(3, double, ACC_NATIVE) X(4, double, ACC_NATIVE) X(5, double, ACC_NATIVE) \
    X(2, float, ACC_COMP) X(3, float, ACC_COMP) X(4, float, ACC_COMP) X(5, float, ACC_COMP)             \
    X(3, float, ACC_NATIVE) X(5, float, ACC_NATIVE) X(3, float, ACC_DOUBLE) X(5, float, ACC_DOUBLE)

bool sweep_variant_ok(int K, int fp32, int acc)
{
#define OKV(KK, RR, AA) if (K == KK && (fp32 != 0) == std::is_same<RR, float>::value && acc == AA) return true;
    PIC_FOR_SWEEP_VARIANTS(OKV)
#undef OKV
    return false;
}

int launch_sweep1(const Sweep1Args &a, int grid, cudaStream_t s)
{
#define L1(KK, RR, AA)                                                                              \
    if (a.K == KK && (a.fp32 != 0) == std::is_same<RR, float>::value && a.acc == AA) {              \
        k_sweep1<KK, RR, AA><<<grid, SweepShape<RR, KK>::threads1, 0, s>>>(a);                      \
        return 0;                                                                                   \
    }
    PIC_FOR_SWEEP_VARIANTS(L1)
#undef L1
    return 1;
}

// four consecutive markers' numbers (none beyond end)
template <typename T>
__device__ __forceinline__ void load4_to(const T *q, long long a, long long end, T (&v)[4])
{
    if (a + 4 <= end) {
        load4(q + a, v);
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = a + u < end ? q[a + u] : T(0);
    }
}

// ---------------------------------------------------------------------------
// Path-integrated current of given displacements (pic_deposit CURRENT): the
// deposit half of the sweep above, in the form's precision.  A path inside one cell
// has length d exactly, a path across knots ends at the offset of t0 + d.  Adding every
// basis value to a shared-memory row by a double atomic (a compare-and-swap loop) took
// 4.2 ms for 1e7 markers; the register window takes 0.32 ms, bound by the displacements'
// scattered loads and the FP64 pipe.
// ---------------------------------------------------------------------------
// The deposit is the path's pieces cell by cell, h S_m in each (displacements may be tiny
// here, which the difference of the end points' moments would not resolve).
template <int K, typename R>
__global__ void __launch_bounds__(kSweepThreads) k_current(CurrentArgs A)
{
    const int32_t *__restrict__ cp = A.P.cell;
    const int32_t *__restrict__ id = A.P.id;
    const R *__restrict__ vp = static_cast<const R *>(A.P.t);
    const int lane = threadIdx.x & 31, M = A.M;
    const double inv = 1.0 / A.dx;
    const R half = R(0.5);
    long long wb, we;
    grid_warp_chunk(A.np, wb, we);
    if (wb >= we) return;
    MomentWindow<kWin1, K, AccNative<double>> win;
    win.clear();
    int base = cp[wb];
    unsigned used = 0u;
    bool bad = false;
    for (long long s = wb; s < we; s += 32) {
        const long long a = s + lane;
        const bool act = a < we;
        const unsigned amask = __ballot_sync(0xffffffffu, act);
        const int c = act ? cp[a] : 0;
        const R v0 = act ? vp[a] : R(0);
        R d = act ? (R)(A.disp[id[a]] * inv) : R(0);
        if (!(fabs(d) <= (R)A.Dlim)) { bad = true; d = R(0); }
        int n;
        R v1;
        path_end(v0, d, n, v1);
        int r0 = rel_cell(c, base, M), r1 = r0 + n;
        bool in = act && (unsigned)r0 < (unsigned)kWin1 && (unsigned)r1 < (unsigned)kWin1;
        if (__popc(__ballot_sync(0xffffffffu, act && !in)) > kWindowMisses) {
            int off = window_move<kWin1>(min(r0, r1), min(r0, r1), act, amask);
            if (off > 0 && off < kWin1) {
                for (; off > 0; --off) {
                    win.shift(A.mom, base, used);
                    used >>= 1;
                    base = base + 1 == M ? 0 : base + 1;
                }
            } else if (off != 0) {
                win.flush(A.mom, base, used, M);
                used = 0u;
                base = wrap_cell(base + off, M);
            }
            r0 = rel_cell(c, base, M);
            r1 = r0 + n;
            in = act && (unsigned)r0 < (unsigned)kWin1 && (unsigned)r1 < (unsigned)kWin1;
        }
        const int lo = min(r0, r1), hi = max(r0, r1);
        const unsigned mine = in ? (2u << hi) - (1u << lo) : 0u;
        const unsigned mask = __reduce_or_sync(0xffffffffu, mine);
        used |= mask;
#pragma unroll
        for (int w = 0; w < kWin1; ++w) {
            if (mask & (1u << w)) {
                if (mine & (1u << w)) {
                    const R va = r0 == w ? v0 : (r0 < w ? -half : half), vb = r1 == w ? v1 : (r1 < w ? -half : half);
                    R x[K];
                    piece_moments<K, R>(va, vb, n == 0 ? d : vb - va, x);
#pragma unroll
                    for (int m = 0; m < K; ++m) win.acc[w][m].add((double)x[m]);
                }
            }
        }
        if (act && !in) {
            int g = c;
            for (int q = 0; q <= abs(n); ++q) {
                const R va = q == 0 ? v0 : (n > 0 ? -half : half);
                const R vb = q == abs(n) ? v1 : (n > 0 ? half : -half);
                R x[K];
                piece_moments<K, R>(va, vb, n == 0 ? d : vb - va, x);
#pragma unroll
                for (int m = 0; m < K; ++m) atomicAdd(&A.mom[(size_t)g * K + m], (double)x[m]);
                g = wrap_once(g + (n > 0 ? 1 : -1), M);
            }
        }
    }
    win.flush(A.mom, base, used, M);
    if (bad) atomicOr(&A.ctrl->status, STATUS_NUMERIC);
}

template <typename R>
static int launch_current_t(const CurrentArgs &a, int grid, cudaStream_t s)
{
    switch (a.K) {
    case 2: k_current<2, R><<<grid, kSweepThreads, 0, s>>>(a); break;
    case 3: k_current<3, R><<<grid, kSweepThreads, 0, s>>>(a); break;
    case 4: k_current<4, R><<<grid, kSweepThreads, 0, s>>>(a); break;
    case 5: k_current<5, R><<<grid, kSweepThreads, 0, s>>>(a); break;
    default: return 1;
    }
    return 0;
}

int launch_current(const CurrentArgs &a, int grid, cudaStream_t s)
{
    return a.fp32 ? launch_current_t<float>(a, grid, s) : launch_current_t<double>(a, grid, s);
}

template <int K, typename R, int ACC>
__global__ void __launch_bounds__(SweepShape<R, K>::threads2, SweepShape<R, K>::blocks2) k_sweep2(Sweep2Args A)
{
    long long wb, we;
    grid_warp_chunk(A.np, wb, we);
    sweep2_range<K, R, ACC>(A, wb, we);
}

// The predicted start's current only sets where the fixed-point iteration starts
// (the fixed point and its stopping test do not depend on it), so its lanes sum in
// the form's own precision: plain float lanes in the FP32 form, whatever
// accumulation the sweeps use.
#define PIC_FOR_PREDEPOSIT_VARIANTS(X)                                                              \
    X(2, double, ACC_NATIVE) X(3, double, ACC_NATIVE) X(4, double, ACC_NATIVE) X(5, double, ACC_NATIVE) \
    X(2, float, ACC_NATIVE) X(3, float, ACC_NATIVE) X(4, float, ACC_NATIVE) X(5, float, ACC_NATIVE)

int launch_predeposit(const Sweep1Args &a, int grid, cudaStream_t s)
{
#define LP(KK, RR, AA)                                                                              \
    if (a.K == KK && (a.fp32 != 0) == std::is_same<RR, float>::value) {                             \
        k_predeposit<KK, RR, AA><<<grid, SweepShape<RR, KK>::threads1, 0, s>>>(a);                  \
        return 0;                                                                                   \
    }
    PIC_FOR_PREDEPOSIT_VARIANTS(LP)
#undef LP
    return 1;
}

int launch_sweep2(const Sweep2Args &a, int grid, cudaStream_t s)
{
#define L2(KK, RR, AA)                                                                              \
    if (a.K == KK && (a.fp32 != 0) == std::is_same<RR, float>::value && a.acc == AA) {              \
        k_sweep2<KK, RR, AA><<<grid, SweepShape<RR, KK>::threads2, 0, s>>>(a);                      \
        return 0;                                                                                   \
    }
    PIC_FOR_SWEEP_VARIANTS(L2)
#undef L2
    return 1;
}

// ---------------------------------------------------------------------------
// Diagnostics, evaluated in double from the stored state.
// ---------------------------------------------------------------------------
// charge moments sum_a v^m per cell, halved, as 64-bit integers (AccFixed): with double sums
// the FP64 pipe bounds it (1e7 float markers: 274 us, 88 now, the pipe 30 % busy).  Four blocks
// an SM: left alone the compiler takes 70 registers in degrees 2 and 3, which leaves three
// (112 us).
template <int K, typename R>
__global__ void __launch_bounds__(kSweepThreads, K <= 3 ? 4 : 1) k_charge(DiagArgs A)
{
    const int32_t *__restrict__ cp = A.P.cell;
    const R *__restrict__ vp = static_cast<const R *>(A.P.t);
    const int lane = threadIdx.x & 31, M = A.M;
    long long wb, we;
    grid_warp_chunk(A.np, wb, we);
    if (wb >= we) return;
    MomentWindow<kWin2, K + 1, AccFixed> win;
    win.clear();
    int base = cp[wb];
    unsigned used = 0u;
    int adds = 0;
    for (long long s = wb; s < we; s += 32) {
        const long long a = s + lane;
        const bool act = a < we;
        const unsigned amask = __ballot_sync(0xffffffffu, act);
        const int c = act ? cp[a] : 0;
        const double v = act ? as_double(vp[a]) : 0.0;
        const bool num = is_offset(v);          // what is none goes to global memory as it is
        int rel = rel_cell(c, base, M);
        bool in = act && num && (unsigned)rel < (unsigned)kWin2;
        if (__popc(__ballot_sync(0xffffffffu, act && !in)) > kWindowMisses) {
            int off = window_move<kWin2>(rel, rel, act, amask);
            if (off > 0 && off < kWin2) {
                for (; off > 0; --off) {
                    win.shift(A.mom, base, used, 2.0);
                    used >>= 1;
                    base = base + 1 == M ? 0 : base + 1;
                }
            } else if (off != 0) {
                win.flush(A.mom, base, used, M, 2.0);
                used = 0u;
                base = wrap_cell(base + off, M);
            }
            rel = rel_cell(c, base, M);
            in = act && num && (unsigned)rel < (unsigned)kWin2;
        }
        const unsigned mask = __reduce_or_sync(0xffffffffu, in ? 1u << rel : 0u);
        used |= mask;
        long long x[K + 1], y[K];
        point_moments_fixed<K>(v, y);
        x[0] = 1LL << 55;
#pragma unroll
        for (int m = 1; m <= K; ++m) x[m] = y[m - 1];
        win.add(mask, in ? rel : -1, x);
        if (act && !in) {
            double pw = 1.0;
#pragma unroll
            for (int m = 0; m <= K; ++m) {
                atomicAdd(&A.mom[(size_t)c * (K + 1) + m], pw);
                pw *= v;
            }
        }
        if (++adds == kFixedAdds) { win.flush(A.mom, base, used, M, 2.0); used = 0u; adds = 0; }
    }
    win.flush(A.mom, base, used, M, 2.0);
}

// A.tab: the field's polynomial of each cell in double (launch_cell_coefs)
template <int D, typename R>
__global__ void __launch_bounds__(256) k_gather(DiagArgs A)
{
    const R *tp = static_cast<const R *>(A.P.t);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < A.np; a += stride) {
        double c[D + 1];
        load_coef<D + 1>(A.tab + (size_t)A.P.cell[a] * CoefPad<double, D + 1>::v, c);
        A.out[A.P.id[a]] = horner<D + 1>(c, as_double(tp[a]));
    }
}

template <int K, typename R>
__global__ void __launch_bounds__(256) k_kinetic(DiagArgs A)
{
    __shared__ double s_red[32];
    const R *tp = static_cast<const R *>(A.P.t);
    const R *pp = static_cast<const R *>(A.P.p);
    double acc = 0.0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < A.np; a += stride) {
        const int c = A.P.cell[a];
        double v[K + 1];
        bspline_vals<K, double>(as_double(tp[a]) + 0.5, v);
        double Ay = 0.0, Az = 0.0;
#pragma unroll
        for (int r = 0; r <= K; ++r) {
            const int i = wrap_cell(c - r, A.M);
            Ay += A.c0[i] * v[r];
            Az += A.c1[i] * v[r];
        }
        const double p = as_double(pp[a]);
        const double q = p * p + Ay * Ay + Az * Az;
        acc += quotient(A.w * q, 1.0 + root(1.0 + q));      // w (gamma - 1) without cancellation
    }
    block_sum_to(A.acc, acc, s_red);
}

template <typename R>
static int launch_charge_t(const DiagArgs &a, int grid, cudaStream_t s)
{
    switch (a.K) {
    case 2: k_charge<2, R><<<grid, kSweepThreads, 0, s>>>(a); break;
    case 3: k_charge<3, R><<<grid, kSweepThreads, 0, s>>>(a); break;
    case 4: k_charge<4, R><<<grid, kSweepThreads, 0, s>>>(a); break;
    case 5: k_charge<5, R><<<grid, kSweepThreads, 0, s>>>(a); break;
    default: return 1;
    }
    return 0;
}

int launch_charge(const DiagArgs &a, int grid, cudaStream_t s)
{
    return a.fp32 ? launch_charge_t<float>(a, grid, s) : launch_charge_t<double>(a, grid, s);
}

template <typename R>
static int launch_gather_t(const DiagArgs &a, int d, int grid, int block, cudaStream_t s)
{
    switch (d) {
    case 1: k_gather<1, R><<<grid, block, 0, s>>>(a); break;
    case 2: k_gather<2, R><<<grid, block, 0, s>>>(a); break;
    case 3: k_gather<3, R><<<grid, block, 0, s>>>(a); break;
    case 4: k_gather<4, R><<<grid, block, 0, s>>>(a); break;
    case 5: k_gather<5, R><<<grid, block, 0, s>>>(a); break;
    default: return 1;
    }
    return 0;
}

int launch_gather(const DiagArgs &a, int d, int grid, int block, cudaStream_t s)
{
    return a.fp32 ? launch_gather_t<float>(a, d, grid, block, s)
                  : launch_gather_t<double>(a, d, grid, block, s);
}

// Path mean of E_x,h = sum_i e_i Lambda^1_i along x_a -> x_a + d_a (Sec. 4.2, the
// (1/dt) int Lambda_1(X(tau)) dtau . e of subsystem I), in double: the path is
// split at the knots and each piece contributes (h/d) sum_m E_m S_m (A.tab holds
// E_m / (m + 1)); a zero displacement gives E_x,h(x_a).  On entry
// out[id] holds d (length units); it is overwritten with the mean.  Bound by the FP64 pipe:
// 32 operations a marker took 604 us for 1e7 float markers, cubic; 450 us now.
template <int K, typename R>
__global__ void __launch_bounds__(256) k_gather_path(DiagArgs A)
{
    const R *tp = static_cast<const R *>(A.P.t);
    bool bad = false;
    constexpr int PE = CoefPad<double, K>::v;
    const double inv = 1.0 / A.dx;
    const long long lim = __double_as_longlong((double)A.Dlim);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < A.np; a += stride) {
        int g = A.P.cell[a];
        const int id = A.P.id[a];
        const double d = A.out[id] * inv;
        // |d| <= Dlim, as integers (a NaN is larger)
        if ((__double_as_longlong(d) & LLONG_MAX) > lim) { bad = true; A.out[id] = 0.0; continue; }
        const double v0 = as_double(tp[a]);
        int n;
        double v1;
        path_end(v0, d, n, v1);
        const int an = abs(n);
        const bool right = n > 0;
        const double edge = right ? 0.5 : -0.5;
        double S[K], c[K];
        const double vb = an == 0 ? v1 : edge;
        path_sums<K, double>(v0, vb, S);
        load_coef<K>(A.tab + (size_t)g * PE, c);
        double e = c[0];
#pragma unroll
        for (int m = 1; m < K; ++m) e = fma(c[m], S[m], e);
        if (an > 0) {
            double W = vb - v0, sum = W * e;
            for (int q = 1; q <= an; ++q) {
                g = wrap_once(g + (right ? 1 : -1), A.M);
                const double ve = q == an ? v1 : edge;
                edge_sums<K, double>(right, -edge, ve, S);
                load_coef<K>(A.tab + (size_t)g * PE, c);
                e = c[0];
#pragma unroll
                for (int m = 1; m < K; ++m) e = fma(c[m], S[m], e);
                const double h = ve + edge;
                sum = fma(h, e, sum);
                W += h;
            }
            e = quotient(sum, W);
        }
        A.out[id] = e;
    }
    if (bad) atomicOr(A.status, STATUS_NUMERIC);
}

// ---------------------------------------------------------------------------
// Spin (double form): deposit, rotation (subsystem III) and Zeeman energy.  Spin
// components live in caller order; markers are visited in stored order and
// their spins addressed through id.
// ---------------------------------------------------------------------------
// dA/dx at a marker: sum_i (G a)_i Lambda^1_i(x), (G a)_i = (a_i - a_{i-1}) / dx
template <int K>
__device__ __forceinline__ void spin_field_grad(const SpinArgs &A, int c, double off, double &Y, double &Z)
{
    double v[K];
    bspline_vals<K - 1, double>(off + 0.5, v);
    Y = 0.0;
    Z = 0.0;
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int i = wrap_cell(c - r, A.M), im = wrap_cell(c - r - 1, A.M);
        Y += v[r] * (A.ay[i] - A.ay[im]);
        Z += v[r] * (A.az[i] - A.az[im]);
    }
    Y /= A.dx;
    Z /= A.dx;
}

// Moments s_y v^m, s_z v^m (m < K) per cell: windows of cells in registers as in k_charge
// (adding each marker's 2 K basis values to nodes in shared memory, where a double addition
// is a compare-and-swap loop, took 36 us for 1e4 markers).
template <int K>
__global__ void __launch_bounds__(kSweepThreads) k_spin_deposit(SpinArgs A)
{
    const int32_t *__restrict__ cp = A.P.cell;
    const double *__restrict__ vp = static_cast<const double *>(A.P.t);
    const int lane = threadIdx.x & 31, M = A.M;
    long long wb, we;
    grid_warp_chunk(A.np, wb, we);
    if (wb >= we) return;
    MomentWindow<kWin2, K, AccNative<double>> wy, wz;
    wy.clear();
    wz.clear();
    int base = cp[wb];
    unsigned used = 0u;
    for (long long s = wb; s < we; s += 32) {
        const long long a = s + lane;
        const bool act = a < we;
        const unsigned amask = __ballot_sync(0xffffffffu, act);
        const int c = act ? cp[a] : 0;
        const double v = act ? vp[a] : 0.0;
        const int id = act ? A.P.id[a] : 0;
        double y[K], z[K];
        y[0] = act ? A.sy[id] : 0.0;
        z[0] = act ? A.sz[id] : 0.0;
#pragma unroll
        for (int m = 1; m < K; ++m) {
            y[m] = y[m - 1] * v;
            z[m] = z[m - 1] * v;
        }
        int rel = rel_cell(c, base, M);
        bool in = act && (unsigned)rel < (unsigned)kWin2;
        if (__popc(__ballot_sync(0xffffffffu, act && !in)) > kWindowMisses) {
            int off = window_move<kWin2>(rel, rel, act, amask);
            if (off > 0 && off < kWin2) {
                for (; off > 0; --off) {
                    wy.shift(A.dy, base, used);
                    wz.shift(A.dz, base, used);
                    used >>= 1;
                    base = base + 1 == M ? 0 : base + 1;
                }
            } else if (off != 0) {
                wy.flush(A.dy, base, used, M);
                wz.flush(A.dz, base, used, M);
                used = 0u;
                base = wrap_cell(base + off, M);
            }
            rel = rel_cell(c, base, M);
            in = act && (unsigned)rel < (unsigned)kWin2;
        }
        const unsigned mask = __reduce_or_sync(0xffffffffu, in ? 1u << rel : 0u);
        used |= mask;
        wy.add(mask, in ? rel : -1, y);
        wz.add(mask, in ? rel : -1, z);
        if (act && !in) {
#pragma unroll
            for (int m = 0; m < K; ++m) {
                atomicAdd(&A.dy[(size_t)c * K + m], y[m]);
                atomicAdd(&A.dz[(size_t)c * K + m], z[m]);
            }
        }
    }
    wy.flush(A.dy, base, used, M);
    wz.flush(A.dz, base, used, M);
}

// Subsystem III
template <int K>
__global__ void __launch_bounds__(256) k_spin_rotate(SpinArgs A)
{
    const double *tp = static_cast<const double *>(A.P.t);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < A.np; a += stride) {
        const int id = A.P.id[a];
        double Y, Z;
        spin_field_grad<K>(A, A.P.cell[a], tp[a], Y, Z);
        spin_turn(A.dt, Y, Z, A.sx[id], A.sy[id], A.sz[id]);
    }
}

template <int K>
__global__ void __launch_bounds__(256) k_spin_energy(SpinArgs A)
{
    __shared__ double s_red[32];
    const double *tp = static_cast<const double *>(A.P.t);
    double acc = 0.0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < A.np; a += stride) {
        const int id = A.P.id[a];
        double Y, Z;
        spin_field_grad<K>(A, A.P.cell[a], tp[a], Y, Z);
        acc += A.w * (A.sy[id] * Z - A.sz[id] * Y);
    }
    block_sum_to(A.acc, acc, s_red);
}

#define PIC_SPIN_LAUNCH(NAME)                                                            \
    switch (a.K) {                                                                       \
    case 2: NAME<2><<<grid, 256, 0, s>>>(a); break;                                      \
    case 3: NAME<3><<<grid, 256, 0, s>>>(a); break;                                      \
    case 4: NAME<4><<<grid, 256, 0, s>>>(a); break;                                      \
    case 5: NAME<5><<<grid, 256, 0, s>>>(a); break;                                      \
    default: return 1;                                                                   \
    }                                                                                    \
    return 0;

int launch_spin_deposit(const SpinArgs &a, int grid, cudaStream_t s)
{
    // at least 128 markers a warp: a warp's windows cost it a reduction of their cells
    const int most = (int)std::max<long long>(1, a.np / (128 * kSweepWarps));
    if (grid > most) grid = most;
    PIC_SPIN_LAUNCH(k_spin_deposit)
}

int launch_spin_rotate(const SpinArgs &a, int grid, cudaStream_t s) { PIC_SPIN_LAUNCH(k_spin_rotate) }

int launch_spin_energy(const SpinArgs &a, int grid, cudaStream_t s) { PIC_SPIN_LAUNCH(k_spin_energy) }

#undef PIC_SPIN_LAUNCH

int launch_gather_path(const DiagArgs &a, int grid, int block, cudaStream_t s)
{
#define GP(KK)                                                                                  \
    case KK:                                                                                    \
        if (a.fp32) k_gather_path<KK, float><<<grid, block, 0, s>>>(a);                         \
        else k_gather_path<KK, double><<<grid, block, 0, s>>>(a);                               \
        break;
    switch (a.K) {
    GP(2) GP(3) GP(4) GP(5)
    default: return 1;
    }
#undef GP
    return 0;
}

template <typename R>
static int launch_kinetic_t(const DiagArgs &a, int grid, int block, cudaStream_t s)
{
    switch (a.K) {
    case 2: k_kinetic<2, R><<<grid, block, 0, s>>>(a); break;
    case 3: k_kinetic<3, R><<<grid, block, 0, s>>>(a); break;
    case 4: k_kinetic<4, R><<<grid, block, 0, s>>>(a); break;
    case 5: k_kinetic<5, R><<<grid, block, 0, s>>>(a); break;
    default: return 1;
    }
    return 0;
}

int launch_kinetic(const DiagArgs &a, int grid, int block, cudaStream_t s)
{
    return a.fp32 ? launch_kinetic_t<float>(a, grid, block, s)
                  : launch_kinetic_t<double>(a, grid, block, s);
}

template <typename R>
__global__ void __launch_bounds__(256) k_finalize1(long long np, int M, PartPtrs P, bool zero_delta)
{
    finalize1_range<R>(np, M, P, (long long)blockIdx.x * blockDim.x + threadIdx.x,
                       (long long)gridDim.x * blockDim.x, zero_delta);
}

int launch_finalize1(int fp32, long long np, int M, PartPtrs P, bool zero_delta, int grid, int block,
                     cudaStream_t s)
{
    if (fp32) k_finalize1<float><<<grid, block, 0, s>>>(np, M, P, zero_delta);
    else k_finalize1<double><<<grid, block, 0, s>>>(np, M, P, zero_delta);
    return 0;
}

// ---------------------------------------------------------------------------
// Load / store between the caller's FP64 (x, p) arrays and the stored form.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(256) k_load(long long np, int M, double dx, const double *x,
                                              const double *p, PartPtrs P)
{
    R *tp = static_cast<R *>(P.t);
    R *pp = static_cast<R *>(P.p);
    R *dp = static_cast<R *>(P.delta);
    R *pnp = static_cast<R *>(P.pnew);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < np; a += stride) {
        const double u = x[a] / dx;
        const double f = ::floor(u);
        P.cell[a] = wrap_cell((int)f, M);
        tp[a] = (R)((u - f) - 0.5);
        pp[a] = (R)p[a];
        pnp[a] = (R)p[a];
        dp[a] = R(0);
        P.id[a] = (int32_t)a;
    }
}

int launch_load(int fp32, long long np, int M, double dx, const double *x, const double *p,
                PartPtrs P, int grid, int block, cudaStream_t s)
{
    if (fp32) k_load<float><<<grid, block, 0, s>>>(np, M, dx, x, p, P);
    else k_load<double><<<grid, block, 0, s>>>(np, M, dx, x, p, P);
    return 0;
}

// position of a marker in [0, L): the centre of its cell plus its offset (an offset of a
// whole half cell may reach L).  Two FP64 operations a marker: with conversions and the
// comparison on the FP64 pipe (ten) the stores were bound by it (2e7 dealt float markers:
// 374 us, the pipe 86 % busy; now 224).
template <typename R>
__device__ __forceinline__ double position(int c, R v, double dx, double L)
{
    const double x = (cell_centre(c) + as_double(v)) * dx;
    // x >= L, as integers (L > 0)
    return __double_as_longlong(x) >= __double_as_longlong(L) ? x - L : x;
}

template <typename R>
__global__ void __launch_bounds__(256) k_store(long long np, int M, double dx, PartPtrs P, double *x, double *p)
{
    const R *tp = static_cast<const R *>(P.t);
    const R *pp = static_cast<const R *>(P.p);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < np; a += stride) {
        const long long i = P.id[a];
        if (x) x[i] = position(P.cell[a], tp[a], dx, M * dx);
        if (p) p[i] = as_double(pp[a]);
    }
}

int launch_store(int fp32, long long np, int M, double dx, PartPtrs P, double *x, double *p,
                 int grid, int block, cudaStream_t s)
{
    if (fp32) k_store<float><<<grid, block, 0, s>>>(np, M, dx, P, x, p);
    else k_store<double><<<grid, block, 0, s>>>(np, M, dx, P, x, p);
    return 0;
}

// The same for a whole state in device memory: x and p in caller order, the fields and the
// spins, in one launch.
template <typename R>
__global__ void __launch_bounds__(256) k_store_state(long long np, int M, double dx, PartPtrs P, StateOut o)
{
    const R *vp = static_cast<const R *>(P.t);
    const R *pp = static_cast<const R *>(P.p);
    const double L = M * dx;
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
    if (o.x || o.p)
        for (long long a = first; a < np; a += stride) {
            const long long i = P.id[a];
            if (o.x) o.x[i] = position(P.cell[a], vp[a], dx, L);
            if (o.p) o.p[i] = as_double(pp[a]);
        }
    for (int f = 0; f < o.n; ++f)
        for (long long a = first; a < o.len[f]; a += stride) o.dst[f][a] = o.src[f][a];
}

int launch_store_state(int fp32, long long np, int M, double dx, PartPtrs P, const StateOut &o, int grid, int block,
                       cudaStream_t s)
{
    if (fp32) k_store_state<float><<<grid, block, 0, s>>>(np, M, dx, P, o);
    else k_store_state<double><<<grid, block, 0, s>>>(np, M, dx, P, o);
    return 0;
}

// Stored order to caller order for more markers than L2 holds outputs for.  Scattered
// directly, every 8-byte write is a sector of its own by the time it leaves L2 (1e8
// markers: 6.8 ms).  Instead the markers are first dealt into at most 256 buckets of
// 2^shift consecutive caller indices (a tile of 2048 markers is ordered by bucket in shared
// memory, so a bucket's part of it is one run of some 128 bytes), then each bucket
// is written out while its range of x and p stays in L2.  Every bucket is full (the
// indices are a permutation), so bucket b starts at b 2^shift and needs no histogram.
// 2e7 float markers: deal 175 us (512 threads 202, 1024 271; loading cell, v and p only after
// the ranks 257), store 224 us; 1e8: 6.8 -> 2.0 ms.
template <typename R> struct StoreRec;
template <> struct StoreRec<float> { int id, cell; float v, p; };
template <> struct StoreRec<double> { double v, p; int id, cell; };
constexpr int kDealThreads = 256, kDealPer = 8, kDealTile = kDealThreads * kDealPer, kDealBuckets = 256;

__global__ void k_deal_start(int *cursor, int shift) { cursor[threadIdx.x] = (int)((long long)threadIdx.x << shift); }

template <typename R>
__global__ void __launch_bounds__(kDealThreads) k_deal(long long np, int shift, PartPtrs P, StoreRec<R> *rec, int *cursor)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    StoreRec<R> *s_rec = reinterpret_cast<StoreRec<R> *>(s_raw);
    __shared__ int s_cnt[kDealBuckets], s_off[kDealBuckets], s_dst[kDealBuckets], s_warp[kDealBuckets / 32];
    const R *vp = static_cast<const R *>(P.t);
    const R *pp = static_cast<const R *>(P.p);
    const long long base = (long long)blockIdx.x * kDealTile;
    const int n = (int)min((long long)kDealTile, np - base);
    if (threadIdx.x < kDealBuckets) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    int id[kDealPer], c[kDealPer], rank[kDealPer];
    R v[kDealPer], p[kDealPer];
#pragma unroll
    for (int j = 0; j < kDealPer; j += 4) {
        const long long a = base + j * kDealThreads + 4 * threadIdx.x;
        load4_to(P.id, a, np, *reinterpret_cast<int (*)[4]>(id + j));
        load4_to(P.cell, a, np, *reinterpret_cast<int (*)[4]>(c + j));
        load4_to(vp, a, np, *reinterpret_cast<R (*)[4]>(v + j));
        load4_to(pp, a, np, *reinterpret_cast<R (*)[4]>(p + j));
    }
#pragma unroll
    for (int j = 0; j < kDealPer; ++j)
        if ((j & ~3) * kDealThreads + 4 * threadIdx.x + (j & 3) < n) rank[j] = atomicAdd(&s_cnt[id[j] >> shift], 1);
    __syncthreads();
    if (threadIdx.x < kDealBuckets) {          // exclusive scan of the counts, and the runs' places
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, m = s_cnt[threadIdx.x];
        int sum = m;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += u;
        }
        if (lane == 31) s_warp[w] = sum;
        s_off[threadIdx.x] = sum - m;
        s_dst[threadIdx.x] = m ? atomicAdd(&cursor[threadIdx.x], m) : 0;
    }
    __syncthreads();
    if (threadIdx.x < kDealBuckets) {
        int add = 0;
        for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) add += s_warp[w];
        s_off[threadIdx.x] += add;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kDealPer; ++j) {
        if ((j & ~3) * kDealThreads + 4 * threadIdx.x + (j & 3) < n) {
            StoreRec<R> r;
            r.id = id[j];
            r.cell = c[j];
            r.v = v[j];
            r.p = p[j];
            s_rec[s_off[id[j] >> shift] + rank[j]] = r;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kDealThreads) {
        const StoreRec<R> r = s_rec[i];
        const int b = r.id >> shift;
        rec[(size_t)s_dst[b] + (i - s_off[b])] = r;
    }
}

template <typename R>
__global__ void __launch_bounds__(256) k_store_dealt(long long np, double dx, double L, const StoreRec<R> *rec,
                                                     double *x, double *p)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    const StoreRec<R> r = rec[i];
    if (x) x[r.id] = position(r.cell, r.v, dx, L);
    if (p) p[r.id] = as_double(r.p);
}

template <typename R>
static int launch_store_dealt_t(long long np, int M, double dx, PartPtrs P, void *rec, int *cursor, double *x, double *p,
                                cudaStream_t s)
{
    int shift = 0;
    while ((np - 1) >> shift >= kDealBuckets) ++shift;
    const size_t smem = kDealTile * sizeof(StoreRec<R>);
    if (cudaFuncSetAttribute(k_deal<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 1;
    k_deal_start<<<1, kDealBuckets, 0, s>>>(cursor, shift);
    k_deal<R><<<(unsigned)((np + kDealTile - 1) / kDealTile), kDealThreads, smem, s>>>(
        np, shift, P, static_cast<StoreRec<R> *>(rec), cursor);
    k_store_dealt<R><<<(unsigned)((np + 255) / 256), 256, 0, s>>>(np, dx, M * dx, static_cast<StoreRec<R> *>(rec), x, p);
    return 0;
}

int launch_store_dealt(int fp32, long long np, int M, double dx, PartPtrs P, void *rec, int *cursor, double *x, double *p,
                       cudaStream_t s)
{
    return fp32 ? launch_store_dealt_t<float>(np, M, dx, P, rec, cursor, x, p, s)
                : launch_store_dealt_t<double>(np, M, dx, P, rec, cursor, x, p, s);
}

// inv[id[a]] = a: where the marker of each caller index is stored
__global__ void __launch_bounds__(256) k_inverse_id(long long np, const int32_t *__restrict__ id,
                                                    int32_t *__restrict__ inv)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < np; a += stride)
        inv[id[a]] = (int32_t)a;
}

// x[i], p[i] in caller order, each read from where marker i is stored: the writes are
// consecutive, so the destination may be page-locked host memory written over the host
// link (the same values as k_store)
template <typename R>
__global__ void __launch_bounds__(256) k_store_ordered(long long np, int M, double dx, PartPtrs P,
                                                       const int32_t *__restrict__ inv, double *x, double *p)
{
    const R *tp = static_cast<const R *>(P.t);
    const R *pp = static_cast<const R *>(P.p);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < np; i += stride) {
        const long long a = inv[i];
        if (x) x[i] = position(P.cell[a], tp[a], dx, M * dx);
        if (p) p[i] = as_double(pp[a]);
    }
}

int launch_store_ordered(int fp32, long long np, int M, double dx, PartPtrs P, int32_t *inv, double *x, double *p,
                         int grid, int block, cudaStream_t s)
{
    k_inverse_id<<<grid, block, 0, s>>>(np, P.id, inv);
    if (fp32) k_store_ordered<float><<<grid, block, 0, s>>>(np, M, dx, P, inv, x, p);
    else k_store_ordered<double><<<grid, block, 0, s>>>(np, M, dx, P, inv, x, p);
    return 0;
}

// ---------------------------------------------------------------------------
// Counting sort of the markers by key = cell * nbins + velocity bin, the bin being
// the expected displacement tau p in units of 1/per cell (nbins = 16 per, clamped),
// so that a warp's markers share cells and piece counts.  Runs between steps; delta and
// p_new are not carried (each step's first sweep or warm start writes them
// before they are read, and delta is all zero where the iteration starts from
// it).  Atomics are aggregated per warp over equal keys.
// counts: sort_counts(nkeys) int32 (histogram, cursors, the scan's tile totals).
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ int sort_key(int c, R p, float taup, int nbins)
{
    int b = (int)floorf((float)p * taup) + nbins / 2;
    b = b < 0 ? 0 : (b >= nbins ? nbins - 1 : b);
    return c * nbins + b;
}

// Both passes give each block a contiguous chunk of the markers.  The markers are
// nearly sorted (they were sorted a few steps ago), so the blocks running at the
// same time then touch different keys' counters; in a grid-stride order every
// block would work on the same few cells at once and serialise on their counters.
// chunk [beg, end) of block b among nb blocks (a multiple of 128 markers)
__device__ __forceinline__ void chunk_of(long long np, int b, int nb, long long &beg, long long &end)
{
    long long chunk = (np + nb - 1) / nb;
    chunk = (chunk + 127) & ~127LL;
    beg = (long long)b * chunk;
    end = beg + chunk < np ? beg + chunk : np;
}

template <typename R>
__device__ __forceinline__ void hist_range(long long beg, long long end, float tau, int nbins, const PartPtrs &S,
                                           int32_t *counts)
{
    const R *ps = static_cast<const R *>(S.p);
    const int lane = threadIdx.x & 31;
    for (long long base = beg; base < end; base += 4 * blockDim.x) {
        const long long a = base + 4 * threadIdx.x;
        int c[4];
        R p[4];
        load4_to(S.cell, a, end, c);
        load4_to(ps, a, end, p);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int key = a + u < end ? sort_key(c[u], p[u], tau, nbins) : -1;
            const unsigned grp = __match_any_sync(0xffffffffu, key);
            if (key >= 0 && lane == __ffs(grp) - 1) atomicAdd(&counts[key], __popc(grp));
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(256) k_hist(long long np, float tau, int nbins, PartPtrs S, int32_t *counts)
{
    long long beg, end;
    chunk_of(np, blockIdx.x, gridDim.x, beg, end);
    hist_range<R>(beg, end, tau, nbins, S, counts);
}

// Exclusive scan of nkeys counts into the cursors behind them: a block a tile of
// kScanTile keys sums it into the totals behind the cursors, then a block a tile adds the
// totals before its own and scans it.  (One block with a range of keys a thread, whose
// loads are strided, took 227 us for 131072 keys.)
__device__ __forceinline__ int block_sum(int v)
{
    __shared__ int s_part[32];
    v = __reduce_add_sync(0xffffffffu, v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
    __syncthreads();
    int t = 0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) t += s_part[w];
    return t;
}

__device__ __forceinline__ void scan_totals(int nkeys, int tile, int32_t *counts)
{
    int s = 0;
    const int end = min(nkeys, (tile + 1) * kScanTile);
    for (int i = tile * kScanTile + threadIdx.x; i < end; i += blockDim.x) s += counts[i];
    s = block_sum(s);
    if (threadIdx.x == 0) counts[2 * (size_t)nkeys + tile] = s;
}

__device__ __forceinline__ void scan_tile(int nkeys, int tile, int32_t *counts)
{
    __shared__ int s_warp[32];
    int before = 0;
    for (int i = threadIdx.x; i < tile; i += blockDim.x) before += counts[2 * (size_t)nkeys + i];
    before = block_sum(before);
    constexpr int kPer = kScanTile / 256;      // consecutive keys a thread
    const int lane = threadIdx.x & 31, lo = tile * kScanTile + threadIdx.x * kPer;
    int v[kPer], s = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        v[i] = lo + i < nkeys ? counts[lo + i] : 0;
        s += v[i];
    }
    int incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_warp[threadIdx.x >> 5] = incl;
    __syncthreads();
    int run = before + incl - s;
    for (int w = 0; w < (int)threadIdx.x / 32; ++w) run += s_warp[w];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        if (lo + i < nkeys) counts[nkeys + lo + i] = run;
        run += v[i];
    }
}

__global__ void __launch_bounds__(256) k_scan_totals(int nkeys, int32_t *counts) { scan_totals(nkeys, blockIdx.x, counts); }
__global__ void __launch_bounds__(256) k_scan(int nkeys, int32_t *counts) { scan_tile(nkeys, blockIdx.x, counts); }

template <typename R>
__device__ __forceinline__ void scatter_range(long long beg, long long end, float tau, int nbins, const PartPtrs &S,
                                              const PartPtrs &D, int32_t *cursor)
{
    const R *ts = static_cast<const R *>(S.t);
    const R *ps = static_cast<const R *>(S.p);
    R *td = static_cast<R *>(D.t);
    R *pd = static_cast<R *>(D.p);
    const int lane = threadIdx.x & 31;
    // four markers a thread per pass: their loads and cursor atomics are independent, so
    // the warp waits for the returned slots once per pass instead of once a marker
    for (long long base = beg; base < end; base += 4 * blockDim.x) {
        const long long a = base + 4 * threadIdx.x;
        int c[4], id[4], key[4], first[4];
        R p[4], t[4];
        unsigned grp[4];
        load4_to(S.cell, a, end, c);
        load4_to(ps, a, end, p);
        load4_to(ts, a, end, t);
        load4_to(S.id, a, end, id);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            key[u] = a + u < end ? sort_key(c[u], p[u], tau, nbins) : -1;
            grp[u] = __match_any_sync(0xffffffffu, key[u]);
            first[u] = 0;
            if (key[u] >= 0 && lane == __ffs(grp[u]) - 1) first[u] = atomicAdd(&cursor[key[u]], __popc(grp[u]));
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int f = __shfl_sync(0xffffffffu, first[u], __ffs(grp[u]) - 1);
            if (key[u] < 0) continue;
            const long long j = (long long)f + __popc(grp[u] & ((1u << lane) - 1u));
            D.cell[j] = c[u];
            td[j] = t[u];
            pd[j] = p[u];
            D.id[j] = id[u];
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(256) k_scatter(long long np, float tau, int nbins, PartPtrs S, PartPtrs D,
                                                 int32_t *cursor)
{
    long long beg, end;
    chunk_of(np, blockIdx.x, gridDim.x, beg, end);
    scatter_range<R>(beg, end, tau, nbins, S, D, cursor);
}

// Batched sorts (ensembles): block row y = run, its counts zeroed, histogrammed,
// scanned and scattered in five launches for all runs due.
__global__ void __launch_bounds__(256) k_sort_zero_ens(const SortRun *runs)
{
    const SortRun &r = runs[blockIdx.y];
    const int n = r.M * r.nbins;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) r.counts[i] = 0;
}

template <typename R>
__global__ void __launch_bounds__(256) k_hist_ens(const SortRun *runs)
{
    const SortRun &r = runs[blockIdx.y];
    long long beg, end;
    chunk_of(r.np, blockIdx.x, gridDim.x, beg, end);
    hist_range<R>(beg, end, r.taup, r.nbins, r.src, r.counts);
}

__global__ void __launch_bounds__(256) k_scan_totals_ens(const SortRun *runs)
{
    const SortRun &r = runs[blockIdx.y];
    for (int t = blockIdx.x; t * kScanTile < r.M * r.nbins; t += gridDim.x) scan_totals(r.M * r.nbins, t, r.counts);
}
__global__ void __launch_bounds__(256) k_scan_ens(const SortRun *runs)
{
    const SortRun &r = runs[blockIdx.y];
    for (int t = blockIdx.x; t * kScanTile < r.M * r.nbins; t += gridDim.x) {
        scan_tile(r.M * r.nbins, t, r.counts);
        __syncthreads();
    }
}

template <typename R>
__global__ void __launch_bounds__(256) k_scatter_ens(const SortRun *runs)
{
    const SortRun &r = runs[blockIdx.y];
    long long beg, end;
    chunk_of(r.np, blockIdx.x, gridDim.x, beg, end);
    scatter_range<R>(beg, end, r.taup, r.nbins, r.src, r.dst, r.counts + (size_t)r.M * r.nbins);
}

int launch_sort_ens(int fp32, const SortRun *runs, int nruns, int grid_x, cudaStream_t s)
{
    if (nruns < 1) return 0;
    const dim3 g(grid_x, nruns);
    k_sort_zero_ens<<<g, 256, 0, s>>>(runs);
    if (fp32) k_hist_ens<float><<<g, 256, 0, s>>>(runs);
    else k_hist_ens<double><<<g, 256, 0, s>>>(runs);
    k_scan_totals_ens<<<dim3(8, nruns), 256, 0, s>>>(runs);
    k_scan_ens<<<dim3(8, nruns), 256, 0, s>>>(runs);
    if (fp32) k_scatter_ens<float><<<g, 256, 0, s>>>(runs);
    else k_scatter_ens<double><<<g, 256, 0, s>>>(runs);
    return 0;
}

int launch_sort(int fp32, long long np, int M, double tau, int per, PartPtrs src, PartPtrs dst,
                int32_t *counts, int num_sms, cudaStream_t s)
{
    // more blocks than fit: their chunks are short, so the blocks running together write a
    // narrow range of the sorted order (2e7 float markers: scatter 180 us at 4 blocks a SM,
    // 176 at 8, 150 at 16; histogram 41, 32, 32)
    const int grid = 16 * num_sms;
    const int nbins = kVelBinsBase * per;
    const int nkeys = M * nbins;
    const float taup = (float)(tau * per);
    if (cudaMemsetAsync(counts, 0, sizeof(int32_t) * (size_t)nkeys, s) != cudaSuccess) return 1;
    if (fp32) k_hist<float><<<grid, 256, 0, s>>>(np, taup, nbins, src, counts);
    else k_hist<double><<<grid, 256, 0, s>>>(np, taup, nbins, src, counts);
    const int tiles = (nkeys + kScanTile - 1) / kScanTile;
    k_scan_totals<<<tiles, 256, 0, s>>>(nkeys, counts);
    k_scan<<<tiles, 256, 0, s>>>(nkeys, counts);
    if (fp32) k_scatter<float><<<grid, 256, 0, s>>>(np, taup, nbins, src, dst, counts + nkeys);
    else k_scatter<double><<<grid, 256, 0, s>>>(np, taup, nbins, src, dst, counts + nkeys);
    return 0;
}

// ---------------------------------------------------------------------------
// Batched ensemble sweeps: persistent blocks claim work items (run, marker range)
// until the queue built by the plan kernel is empty; an item is shared out among the
// block's warps.
// ---------------------------------------------------------------------------
template <typename Args>
__device__ __forceinline__ bool ens_claim(EnsQueue *Q, const Args *runs, int nruns, int &run,
                                          long long &beg, long long &end)
{
    __shared__ int s_item;
    __syncthreads();                       // s_item of the previous claim is consumed
    if (threadIdx.x == 0) s_item = atomicAdd(&Q->next, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= Q->nitems) return false;
    // the run r with item_start[r] <= item < item_start[r + 1]
    int lo = 0, hi = nruns;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (Q->item_start[mid] <= item) lo = mid; else hi = mid;
    }
    run = lo;
    const long long im = Q->item_markers;
    const long long ib = (long long)(item - Q->item_start[run]) * im;
    const long long ie = ib + im < runs[run].np ? ib + im : runs[run].np;
    warp_chunk(ib, ie, threadIdx.x >> 5, blockDim.x >> 5, beg, end);
    return true;
}

template <int K, typename R>
__global__ void __launch_bounds__(SweepShape<R, K>::threads1, SweepShape<R, K>::blocks1)
    k_sweep1_ens(const Sweep1Args *runs, int nruns, EnsQueue *Q)
{
    if (blockIdx.x * Q->shares >= gridDim.x * Q->share) return;
    int run;
    long long beg, end;
    while (ens_claim(Q, runs, nruns, run, beg, end)) {
        double dmax = 0.0;
        bool bad = false;
        sweep1_range<K, R, DefaultAcc<R>::v, false>(runs[run], beg, end, dmax, bad);
        if (bad) atomicOr(&runs[run].ctrl->status, STATUS_NUMERIC);
        sweep_max_to(&runs[run].ctrl->dmax_bits, dmax);
    }
}

// the predicted start of every run (sweep1_range's PRE mode over the work queue)
template <int K, typename R>
__global__ void __launch_bounds__(SweepShape<R, K>::threads1, SweepShape<R, K>::blocks1)
    k_predeposit_ens(const Sweep1Args *runs, int nruns, EnsQueue *Q)
{
    if (blockIdx.x * Q->shares >= gridDim.x * Q->share) return;
    int run;
    long long beg, end;
    while (ens_claim(Q, runs, nruns, run, beg, end)) {
        double dmax = 0.0;
        bool bad = false;
        sweep1_range<K, R, ACC_NATIVE, true>(runs[run], beg, end, dmax, bad);
        if (bad) atomicOr(&runs[run].ctrl->status, STATUS_NUMERIC);
    }
}

template <int K, typename R>
__global__ void __launch_bounds__(SweepShape<R, K>::threads2, SweepShape<R, K>::blocks2)
    k_sweep2_ens(const Sweep2Args *runs, int nruns, EnsQueue *Q)
{
    if (blockIdx.x * Q->shares >= gridDim.x * Q->share) return;
    int run;
    long long beg, end;
    while (ens_claim(Q, runs, nruns, run, beg, end)) sweep2_range<K, R, DefaultAcc<R>::v>(runs[run], beg, end);
}

template <typename R>
static int launch_sweep_ens_t(int which, int K, const void *runs, int nruns, EnsQueue *Q, int grid, cudaStream_t s)
{
#define ENS(KK)                                                                                          \
    case KK: {                                                                                           \
        constexpr int b1 = SweepShape<R, KK>::threads1, b2 = SweepShape<R, KK>::threads2;                \
        if (which == 1) k_sweep1_ens<KK, R><<<grid, b1, 0, s>>>((const Sweep1Args *)runs, nruns, Q);     \
        else if (which == 2) k_sweep2_ens<KK, R><<<grid, b2, 0, s>>>((const Sweep2Args *)runs, nruns, Q); \
        else k_predeposit_ens<KK, R><<<grid, b1, 0, s>>>((const Sweep1Args *)runs, nruns, Q);            \
        break;                                                                                           \
    }
    switch (K) {
    ENS(2) ENS(3) ENS(4) ENS(5)
    default: return 1;
    }
#undef ENS
    return 0;
}

int launch_sweep1_ens(int K, int fp32, const Sweep1Args *runs, int nruns, EnsQueue *Q, int grid, cudaStream_t s)
{
    return fp32 ? launch_sweep_ens_t<float>(1, K, runs, nruns, Q, grid, s)
                : launch_sweep_ens_t<double>(1, K, runs, nruns, Q, grid, s);
}

int launch_sweep2_ens(int K, int fp32, const Sweep2Args *runs, int nruns, EnsQueue *Q, int grid, cudaStream_t s)
{
    return fp32 ? launch_sweep_ens_t<float>(2, K, runs, nruns, Q, grid, s)
                : launch_sweep_ens_t<double>(2, K, runs, nruns, Q, grid, s);
}

int launch_predeposit_ens(int K, int fp32, const Sweep1Args *runs, int nruns, EnsQueue *Q, int grid, cudaStream_t s)
{
    return fp32 ? launch_sweep_ens_t<float>(0, K, runs, nruns, Q, grid, s)
                : launch_sweep_ens_t<double>(0, K, runs, nruns, Q, grid, s);
}

// End of subsystem I for every run (block row = run); runs stopped by an error
// keep their markers.
template <typename R>
__global__ void __launch_bounds__(256) k_finalize1_ens(const RunDesc *runs)
{
    const RunDesc &D = runs[blockIdx.y];
    if (D.ctrl->status & (STATUS_NUMERIC | STATUS_TIMEOUT)) return;
    finalize1_range<R>(D.np, D.M, D.P, (long long)blockIdx.x * blockDim.x + threadIdx.x,
                       (long long)gridDim.x * blockDim.x, true);
}

int launch_finalize1_ens(int fp32, const RunDesc *R, int nruns, int grid_x, cudaStream_t s)
{
    if (fp32) k_finalize1_ens<float><<<dim3(grid_x, nruns), 256, 0, s>>>(R);
    else k_finalize1_ens<double><<<dim3(grid_x, nruns), 256, 0, s>>>(R);
    return 0;
}

int sweep_blocks_per_sm(int K, int fp32, int acc, int which)
{
    int n = 0;
    cudaError_t e = cudaErrorInvalidValue;
#define OCC(KK, RR, AA)                                                                                   \
    if (K == KK && (fp32 != 0) == std::is_same<RR, float>::value && acc == AA)                           \
        e = which == 1 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_sweep1<KK, RR, AA>, SweepShape<RR, KK>::threads1, 0) \
                       : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_sweep2<KK, RR, AA>, SweepShape<RR, KK>::threads2, 0);
    PIC_FOR_SWEEP_VARIANTS(OCC)
#undef OCC
    return e == cudaSuccess ? n : 0;
}

}  // namespace pic
