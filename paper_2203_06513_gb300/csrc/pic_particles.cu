// pic_particles.cu -- marker kernels of libpic (sm_103a).
//
// Markers are stored as structure-of-arrays (cell int32, offset t, momentum p,
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

namespace pic {

template <typename R>
struct Real;
template <>
struct Real<float> { static constexpr bool fp32 = true; };
template <>
struct Real<double> { static constexpr bool fp32 = false; };

// Correctly rounded division: an approximate reciprocal carries a systematic
// bias that the discrete-gradient identity turns into a steady energy drift.
template <typename R> __device__ __forceinline__ R fdiv_(R a, R b) { return a / b; }

// Contiguous chunk of markers owned by one block (a multiple of 32, so every
// warp's lanes see consecutive, sorted markers).
__device__ __forceinline__ void block_chunk(long long np, long long &beg, long long &end)
{
    long long chunk = (np + gridDim.x - 1) / gridDim.x;
    chunk = (chunk + 31) & ~31LL;
    beg = (long long)blockIdx.x * chunk;
    end = beg + chunk < np ? beg + chunk : np;
}

// Range of one warp among `nw` that share [beg, end): contiguous, a multiple of 32.
__device__ __forceinline__ void warp_chunk(long long beg, long long end, long long w, long long nw, long long &wb,
                                           long long &we)
{
    long long chunk = (end - beg + nw - 1) / nw;
    chunk = (chunk + 31) & ~31LL;
    wb = beg + w * chunk;
    we = wb + chunk < end ? wb + chunk : end;
}

// The grid's warps take consecutive ranges block by block in turn (warp q of block b is
// number q * grid + b), so that a launch with fewer ranges than warps uses every SM.
__device__ __forceinline__ void grid_warp_chunk(long long np, long long &wb, long long &we)
{
    const long long nw = (long long)gridDim.x * kSweepWarps;
    warp_chunk(0, np, (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x, nw, wb, we);
}

// Largest value of the block, one atomic per block.
__device__ __forceinline__ void sweep_max_to(unsigned long long *dst, double v)
{
    __shared__ double s_max[kSweepWarps];
    v = warp_max(v);
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double u = s_max[0];
        for (int i = 1; i < kSweepWarps; ++i) {
            const double x = s_max[i];
            u = (x > u || x != x) ? x : u;
        }
        if (u != 0.0) atomic_max_nonneg(dst, u);
    }
    __syncthreads();
}

// Start-point cache of the double form: (A_y, A_z, gamma, unused) per marker, as two
// 16-byte accesses.  A(x^n) and gamma(p^n, A(x^n)) do not change during a fixed-point
// loop: its first sweep stores them and the later ones read them back (32 bytes a
// marker against about 20 operations on the narrow FP64 pipe; in the float form the
// bytes would cost more than the operations).
__device__ __forceinline__ void start_cache_store(void *base, long long a, double y, double z, double g)
{
    double2 *q = reinterpret_cast<double2 *>(base) + 2 * a;
    q[0] = make_double2(y, z);
    q[1] = make_double2(g, 0.0);
}

__device__ __forceinline__ void start_cache_load(const void *base, long long a, double &y, double &z, double &g)
{
    const double2 *q = reinterpret_cast<const double2 *>(base) + 2 * a;
    const double2 u = q[0], w = q[1];
    y = u.x;
    z = u.y;
    g = w.x;
}

// ---------------------------------------------------------------------------
// Subsystem I: one Picard sweep (Sec. 4.2).  Per marker, with x^n = (c0, t0),
// the iterate x^(k) = x^n + delta^(k) and ebar = (e^n + e^(k))/2:
//   A0 = A_h(x^n), A1 = A_h(x^(k)), Ebar and D = (A1-A0)/(x^(k)-x^n) the path means
//   of ebar and G a on x^n -> x^(k),
//   p^(k+1) = p^n + dt Ebar - dt (A1+A0).D / (g(p^n,A1) + g(p^n,A0)),
//   delta^(k+1) = dt (p^n + p^(k+1)) / (g(p^n,A1) + g(p^(k+1),A1)) / dx,
//   j_i += w int_{x^n}^{x^n+delta^(k+1)} Lambda^1_i.
// In cell units with tau = dt/dx: p^(k+1) = p^n + tau (Ebar dx - (A1+A0).D dx/(...)).
// The path is split at the knots; a piece of length h in one cell contributes
//   h sum_m E_m S_m to the integral of ebar and h sum_m A_{m+1} S_m to A1 - A0
// (path_sums), and the deposit adds h S_m to the moments of that cell.
//
// What bounds it: the FP32 form instruction issue, the FP64 form the FP64 pipe (1/64 of
// the FP32 rate).  A sweep that evaluates the triangle of basis values at both ends and
// the piece means of every path piece from nodes staged in shared memory, and deposits
// two cumulative bases through a switch over window offsets, took 453 us in float
// (2e7 markers, 2048 cells, cubic: 652 warp instructions per 32 markers) and 854 us in
// double (2e6 markers); the cell polynomials take 336 us (458) and 537 us.
// PRE: the predicted start instead of a sweep -- the proposal delta^(0) (the
// explicit predictor when A.warm, else the one already in delta) is written back
// and its path current deposited into A.mom; no gather walk, no momentum update.
// ---------------------------------------------------------------------------
template <int K, typename R, int ACC, bool PRE>
__device__ __forceinline__ void sweep1_range(const Sweep1Args &A, long long beg, long long end, double &dmax_out,
                                             bool &bad_out)
{
    constexpr int NC = K + 1;                           // coefficients of A in a cell
    constexpr int PA = CoefPad<R, NC>::v, PE = CoefPad<R, K>::v;
    const R one = R(1), half = R(0.5);
    double *mom = A.mom;
    bool warm = A.warm != 0;
    bool first = A.first != 0;
    if (!PRE && A.graph) {                  // replayed by a graph: buffers by sweep parity
        const int it = *reinterpret_cast<volatile const int *>(&A.ctrl->iter);
        mom = A.mpair[it & 1];
        warm = warm && it == 0;
        first = it == 0;
    }
    const int M = A.M;
    const bool hasz = A.zforce || *reinterpret_cast<volatile const int *>(&A.ctrl->zany) != 0;
    const int32_t *__restrict__ cp = A.P.cell;
    const R *__restrict__ tp = static_cast<const R *>(A.P.t);
    const R *__restrict__ pp = static_cast<const R *>(A.P.p);
    R *dp = static_cast<R *>(A.P.delta);
    R *pnp = static_cast<R *>(A.P.pnew);
    const R *TA = static_cast<const R *>(A.T.A), *TE = static_cast<const R *>(A.T.E);
    const R tau = (R)(A.dt / A.dx);
    const R dlim = (R)A.Dlim;
    const int lane = threadIdx.x & 31;
    R dmax = R(0);
    bool bad = false;
    MomentWindow<kWin1, K, typename AccOf<R, ACC>::T> win;
    win.start();
    int adds = 0;

    // the next step's markers are loaded while this one's are computed
    int nc = 0;
    R nt = half, npn = R(0), nd = R(0);
    auto fetch = [&](long long s) {
        const long long a = s + lane;
        if (a < end) {
            nc = cp[a];
            nt = tp[a];
            npn = pp[a];
            if (!warm) nd = dp[a];
        } else {
            nt = half;
            npn = R(0);
            nd = R(0);
        }
    };
    if (beg < end) fetch(beg);
    for (long long s = beg; s < end; s += 32) {
        const long long a = s + lane;
        const bool act = a < end;
        const unsigned amask = __ballot_sync(0xffffffffu, act);
        const int cw = nc;                               // in [0, M)
        const R t0 = nt, pn = npn, dread = nd;
        if (s + 32 < end) fetch(s + 32);
        const R v0 = t0 - half;
        // A(x^n), gamma(p^n, A(x^n))
        R ay[NC], az[NC];
        R A0y, A0z = R(0), g0;
        load_coef<NC>(TA + (size_t)cw * (2 * PA), ay);
#pragma unroll
        for (int m = 0; m < NC; ++m) az[m] = R(0);
        if (hasz) load_coef<NC>(TA + (size_t)cw * (2 * PA) + PA, az);
        bool cached = false;
        if constexpr (!Real<R>::fp32 && !PRE) cached = !first && A.a0 != nullptr;
        if (cached) {
            if constexpr (!Real<R>::fp32) {
                if (act) start_cache_load(A.a0, a, A0y, A0z, g0);
                else { A0y = R(0); g0 = one; }
            }
        } else {
            A0y = horner<NC>(ay, v0);
            R q0 = fma(A0y, A0y, fma(pn, pn, one));
            if (hasz) {
                A0z = horner<NC>(az, v0);
                q0 = fma(A0z, A0z, q0);
            }
            g0 = sqrt_(q0);
            if constexpr (!Real<R>::fp32 && !PRE)
                if (A.a0 && act) start_cache_store(A.a0, a, A0y, A0z, g0);
        }
        R dold = warm ? fdiv_(tau * pn, g0) : dread;
        if (!(fabs(dold) <= dlim)) { bad = bad || act; dold = R(0); }
        R dnew = R(0), pnew = R(0);
        if constexpr (PRE) {
            dnew = dold;
        } else {
            int n;
            R t1;
            path_end(t0, dold, n, t1);
            const int an = abs(n);
            const bool right = n > 0;
            // first piece (the whole path when no knot is crossed)
            R h0, EI, Qy, Qz = R(0), W;
            {
                const R tb = an == 0 ? t1 : (right ? one : R(0));
                h0 = tb - t0;
                R S[K], ec[K];
                path_sums<K, R>(v0, tb - half, S);
                load_coef<K>(TE + (size_t)cw * PE, ec);
                R e = ec[0], y = ay[1], z = az[1];
#pragma unroll
                for (int m = 1; m < K; ++m) {
                    e = fma(ec[m], S[m], e);
                    y = fma(ay[m + 1], S[m], y);
                }
                if (hasz) {
#pragma unroll
                    for (int m = 1; m < K; ++m) z = fma(az[m + 1], S[m], z);
                }
                // one piece: the means are e, y, z themselves (weight 1, no division by h)
                const R hw = an == 0 ? one : h0;
                EI = hw * e;
                Qy = hw * y;
                Qz = hw * z;
                W = hw;
            }
            R D2y = R(0), D2z = R(0);
            if constexpr (!Real<R>::fp32) {
                if (A.hbar != 0.0) {
                    // path integral of d^2A/dx^2 (cell units) for the Zeeman term:
                    // the difference quotient of A' = sum_m m A_m v^(m-1)
                    R S[K];
                    path_sums<K, R>(v0, (an == 0 ? t1 : (right ? one : R(0))) - half, S);
#pragma unroll
                    for (int m = 2; m <= K; ++m) {
                        D2y = fma(R(m) * ay[m], S[m - 2], D2y);
                        D2z = fma(R(m) * az[m], S[m - 2], D2z);
                    }
                    const R hw = an == 0 ? one : h0;
                    D2y *= hw;
                    D2z *= hw;
                }
            }
            const int nmax = __reduce_max_sync(0xffffffffu, act ? an : 0);
            int g = cw;
            for (int q = 1; q <= nmax; ++q) {
                g += right ? 1 : -1;
                g = g >= M ? g - M : (g < 0 ? g + M : g);
                const bool on = q <= an;
                const R ta = right ? R(0) : one;
                const R tb = q == an ? t1 : (right ? one : R(0));
                const R h = on ? tb - ta : R(0);
                R S[K], ec[K], by[NC];
                path_sums<K, R>(ta - half, tb - half, S);
                load_coef<K>(TE + (size_t)g * PE, ec);
                load_coef<NC>(TA + (size_t)g * (2 * PA), by);
                R e = ec[0], y = by[1];
#pragma unroll
                for (int m = 1; m < K; ++m) {
                    e = fma(ec[m], S[m], e);
                    y = fma(by[m + 1], S[m], y);
                }
                EI = fma(h, e, EI);
                Qy = fma(h, y, Qy);
                W += h;
                if constexpr (!Real<R>::fp32) {
                    if (A.hbar != 0.0) {
                        R d2 = R(0);
#pragma unroll
                        for (int m = 2; m <= K; ++m) d2 = fma(R(m) * by[m], S[m - 2], d2);
                        D2y = fma(h, d2, D2y);
                    }
                }
                if (hasz) {
                    R bz[NC];
                    load_coef<NC>(TA + (size_t)g * (2 * PA) + PA, bz);
                    R z = bz[1];
#pragma unroll
                    for (int m = 1; m < K; ++m) z = fma(bz[m + 1], S[m], z);
                    Qz = fma(h, z, Qz);
                    if constexpr (!Real<R>::fp32) {
                        if (A.hbar != 0.0) {
                            R d2 = R(0);
#pragma unroll
                            for (int m = 2; m <= K; ++m) d2 = fma(R(m) * bz[m], S[m - 2], d2);
                            D2z = fma(h, d2, D2z);
                        }
                    }
                }
            }
            // A(x^(k)) = A(x^n) + the path integral of dA/dx, of the staged field
            const R hs = an == 0 ? h0 : one;
            const R A1y = fma(hs, Qy, A0y), A1z = fma(hs, Qz, A0z);

            // p^(k+1) = p^n + tau (Ebar - (A1 + A0).D / (g1 + g0)) with Ebar = EI/W,
            // D = Q/W (W the summed pieces, 1 for a single one), as one division
            R q1 = fma(A1y, A1y, one), nm = (A1y + A0y) * Qy;
            if (hasz) {
                q1 = fma(A1z, A1z, q1);
                nm = fma(A1z + A0z, Qz, nm);
            }
            const R g1 = sqrt_(fma(pn, pn, q1));
            const R G = g1 + g0;
            const R num = fma(EI, G, -nm);
            R kick = fdiv_(num, W * G);
            if constexpr (!Real<R>::fp32) {
                if (A.hbar != 0.0 && act) {
                    const int id = A.P.id[a];
                    kick -= A.hbar / A.dx * ((A.sy[id] * D2z - A.sz[id] * D2y) / W);
                }
            }
            pnew = fma(tau, kick, pn);
            const R g2 = sqrt_(fma(pnew, pnew, q1));
            dnew = fdiv_(tau * (pn + pnew), g1 + g2);
            if (!(fabs(dnew) <= dlim)) { bad = bad || act; dnew = R(0); }
        }

        // deposit of the path x^n -> x^(k+1); its end is the position finalize stores
        {
            int n;
            R t1;
            path_end(t0, dnew, n, t1);
            deposit_paths<kWin1, K>(win, mom, M, act, amask, warp_unwrap_cell(cw, act, M), t0, n, t1);
            if (++adds == kMaxLaneAdds) { win.flush(mom, M); adds = 0; }
        }
        if (act) {
            dp[a] = dnew;
            if constexpr (!PRE) {
                pnp[a] = pnew;
                R inc = fabs(dnew - dold);
                if (Real<R>::fp32) inc = __fdividef(inc, fmax(one, fabs(dnew)));   // convergence metric only
                dmax = (inc > dmax || inc != inc) ? inc : dmax;
            }
        }
    }
    win.flush(mom, M);
    dmax_out = (double)dmax > dmax_out || dmax != dmax ? (double)dmax : dmax_out;
    bad_out = bad_out || bad;
}

template <int K, typename R, int ACC>
__global__ void __launch_bounds__(kSweepThreads, SweepOcc<R, K>::v1) k_sweep1(Sweep1Args A)
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
__global__ void __launch_bounds__(kSweepThreads, SweepOcc<R, K>::v1) k_predeposit(Sweep1Args A)
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
        k_sweep1<KK, RR, AA><<<grid, kSweepThreads, 0, s>>>(a);                                     \
        return 0;                                                                                   \
    }
    PIC_FOR_SWEEP_VARIANTS(L1)
#undef L1
    return 1;
}

// ---------------------------------------------------------------------------
// Path-integrated current of given displacements (pic_deposit CURRENT): the
// deposit half of the sweep above, in the form's precision.  A path inside one cell
// has length d exactly, a path across knots ends at the offset of t0 + d.  Adding every
// basis value to a shared-memory row by a double atomic (a compare-and-swap loop) took
// 4.2 ms for 1e7 markers; the register window takes 0.32 ms.
// ---------------------------------------------------------------------------
template <int K, typename R>
__global__ void __launch_bounds__(kSweepThreads) k_current(CurrentArgs A)
{
    const int32_t *__restrict__ cp = A.P.cell;
    const int32_t *__restrict__ id = A.P.id;
    const R *__restrict__ tp = static_cast<const R *>(A.P.t);
    const int lane = threadIdx.x & 31, M = A.M;
    const double inv = 1.0 / A.dx;
    long long wb, we;
    grid_warp_chunk(A.np, wb, we);
    MomentWindow<kWin1, K, AccNative<double>> win;
    win.start();
    bool bad = false;
    for (long long s = wb; s < we; s += 32) {
        const long long a = s + lane;
        const bool act = a < we;
        const unsigned amask = __ballot_sync(0xffffffffu, act);
        const int cw = act ? cp[a] : 0;
        const R t0 = act ? tp[a] : R(0.5);
        R d = act ? (R)(A.disp[id[a]] * inv) : R(0);
        if (!(fabs(d) <= (R)A.Dlim)) { bad = true; d = R(0); }
        int n;
        R t1;
        path_end(t0, d, n, t1);
        const int c0 = warp_unwrap_cell(cw, act, M), c1 = c0 + n;
        const int lo = min(c0, c1), hi = max(c0, c1);
        const int nb = window_base<kWin1>(win.base, lo, hi, act, amask);
        if (nb != win.base) win.move(nb, A.mom, M);
        const bool in = act && lo >= win.base && hi < win.base + kWin1;
        const int rlo = __reduce_min_sync(0xffffffffu, in ? lo - win.base : kWin1);
        const int rhi = __reduce_max_sync(0xffffffffu, in ? hi - win.base : -1);
        const int b0 = in ? c0 - win.base : 4 * kWin1, b1 = in ? c1 - win.base : 4 * kWin1;
#pragma unroll
        for (int w = 0; w < kWin1; ++w) {
            if (w >= rlo && w <= rhi) {
                win.used |= 1u << w;
                const R ta = clip_end(b0 - w, t0), tb = clip_end(b1 - w, t1);
                R S[K];
                path_sums<K, R>(ta - R(0.5), tb - R(0.5), S);
                const R h = (n == 0 && in && b0 == w) ? d : tb - ta;
#pragma unroll
                for (int m = 0; m < K; ++m) win.acc[w][m].add((double)(m == 0 ? h : h * S[m]));
            }
        }
        if (act && !in) {
            if (n == 0) {
                R S[K];
                path_sums<K, R>(t0 - R(0.5), t1 - R(0.5), S);
#pragma unroll
                for (int m = 0; m < K; ++m)
                    atomicAdd(&A.mom[(size_t)cw * K + m], (double)(m == 0 ? d : d * S[m]));
            } else {
                deposit_path_global<K, R>(A.mom, M, c0, t0, c1, t1);
            }
        }
    }
    win.flush(A.mom, M);
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

// ---------------------------------------------------------------------------
// Subsystem II: one fixed-point sweep (Sec. 4.2).  Markers frozen at x; with
// A0 = A^n_h(x), A1 = A^(k)_h(x):
//   s_i += w (A0 + A1) Lambda^0_i(x) / (g(p,A0) + g(p,A1))   (y and z),
// deposited as the moments f v^m of each cell.  Same warp ranges as subsystem I.  From
// basis values and node windows: 287 us in float (2e7 markers, 2048 cells, cubic), 413 us
// in double (2e6 markers); from cell polynomials and moments 153 us and 166 us.
// Z: the z component is not identically zero (a linearly polarised wave keeps
// A_z = 0 exactly, and then neither its gathers nor its moments are needed).
// ---------------------------------------------------------------------------
template <int K, typename R, int ACC, bool Z>
__device__ __forceinline__ void sweep2_range_z(const Sweep2Args &A, long long beg, long long end, double *my, double *mz,
                                               bool first)
{
    constexpr int NC = K + 1;
    constexpr int PA = CoefPad<R, NC>::v;
    constexpr int NW = Z ? kWin2z : kWin2;
    const R one = R(1), half = R(0.5);
    const int M = A.M;
    const int32_t *__restrict__ cp = A.P.cell;
    const R *__restrict__ tp = static_cast<const R *>(A.P.t);
    const R *__restrict__ pp = static_cast<const R *>(A.P.p);
    const R *TA = static_cast<const R *>(A.T.A), *TK = static_cast<const R *>(A.T.Kt);
    const float *TL = A.T.L;
    const int lane = threadIdx.x & 31;
    using Acc = typename AccOf<R, ACC>::T;
    MomentWindow<NW, NC, Acc> wy, wz;
    wy.start();
    if (Z) wz.start();
    int adds = 0;
    int nc = 0;
    R nt = half, npn = R(0);
    auto fetch = [&](long long s) {
        const long long a = s + lane;
        if (a < end) {
            nc = cp[a];
            nt = tp[a];
            npn = pp[a];
        }
    };
    if (beg < end) fetch(beg);
    for (long long s = beg; s < end; s += 32) {
        const long long a = s + lane;
        const bool act = a < end;
        const unsigned amask = __ballot_sync(0xffffffffu, act);
        const int cw = nc;
        const R v = nt - half, p = npn;
        if (s + 32 < end) fetch(s + 32);
        const R pp1 = fma(p, p, one);
        const size_t row = (size_t)cw * (2 * PA);
        R A0y, A1y, A0z = R(0), A1z = R(0), Ly = R(0), Lz = R(0), g0;
        bool cached = false;
        if constexpr (!Real<R>::fp32) cached = !first && A.a0 != nullptr;
        if (cached) {
            if constexpr (!Real<R>::fp32) {
                if (act) start_cache_load(A.a0, a, A0y, A0z, g0);
                else { A0y = R(0); g0 = one; }
            }
        } else {
            R c[NC];
            load_coef<NC>(TA + row, c);
            A0y = horner<NC>(c, v);
            R q = fma(A0y, A0y, pp1);
            if (Z) {
                load_coef<NC>(TA + row + PA, c);
                A0z = horner<NC>(c, v);
                q = fma(A0z, A0z, q);
            }
            g0 = sqrt_(q);
            if constexpr (!Real<R>::fp32)
                if (A.a0 && act) start_cache_store(A.a0, a, A0y, A0z, g0);
        }
        R c[NC];
        load_coef<NC>(TK + row, c);
        A1y = horner<NC>(c, v);
        R q1 = fma(A1y, A1y, pp1);
        if (Z) {
            load_coef<NC>(TK + row + PA, c);
            A1z = horner<NC>(c, v);
            q1 = fma(A1z, A1z, q1);
        }
        const R g1 = sqrt_(q1);
        if constexpr (Real<R>::fp32) {
            // The float rounding of a coefficient is the same for every marker of its
            // cell, so it does not average out over markers: in the exchange term
            // (A1 - A0)(A1 + A0)/(g0 + g1) it shows as an energy error of about 1e-11
            // per step.  The residues of the sum a^n + a^(k) enter the numerator before
            // its one rounding, which leaves only per-marker rounding.
            load_coef<NC>(TL + row, c);
            Ly = horner<NC>(c, v);
            if (Z) {
                load_coef<NC>(TL + row + PA, c);
                Lz = horner<NC>(c, v);
            }
        }
        const R cf = fdiv_(one, g0 + g1);
        const R sy = A0y + A1y, sz = A0z + A1z;
        R fy, fz = R(0);
        if constexpr (Real<R>::fp32) {
            // f = cf (s + L) rounded once: the residue L is far below half an ulp of s,
            // so s + L in float would drop it.  The product's own rounding error (exact
            // by an fma) and cf L are added before the one rounding.
            const float py = cf * sy;
            fy = py + (fmaf(cf, sy, -py) + cf * Ly);
            if (Z) {
                const float pz = cf * sz;
                fz = pz + (fmaf(cf, sz, -pz) + cf * Lz);
            }
        } else {
            fy = cf * sy;
            fz = cf * sz;
        }
        const int cu = warp_unwrap_cell(cw, act, M);
        const int nb = window_base<NW>(wy.base, cu, cu, act, amask);
        if (nb != wy.base) {
            wy.move(nb, my, M);
            if (Z) wz.move(nb, mz, M);
        }
        R x[NC], pw[NC];
        pw[0] = one;
#pragma unroll
        for (int m = 1; m < NC; ++m) pw[m] = pw[m - 1] * v;
#pragma unroll
        for (int m = 0; m < NC; ++m) x[m] = m == 0 ? fy : fy * pw[m];
        deposit_points<NW, NC>(wy, my, M, act, cu, x);
        if (Z) {
#pragma unroll
            for (int m = 0; m < NC; ++m) x[m] = m == 0 ? fz : fz * pw[m];
            deposit_points<NW, NC>(wz, mz, M, act, cu, x);
        }
        if (++adds == kMaxLaneAdds) {
            wy.flush(my, M);
            if (Z) wz.flush(mz, M);
            adds = 0;
        }
    }
    wy.flush(my, M);
    if (Z) wz.flush(mz, M);
}

template <int K, typename R, int ACC>
__device__ __forceinline__ void sweep2_range(const Sweep2Args &A, long long beg, long long end)
{
    double *my = A.mom_y, *mz = A.mom_z;
    bool first = A.first != 0;
    if (A.graph) {                          // replayed by a graph: buffers by sweep parity
        const int it = *reinterpret_cast<volatile const int *>(&A.ctrl->iter);
        my = A.mypair[it & 1];
        mz = A.mzpair[it & 1];
        first = it == 0;
    }
    if (A.zforce || *reinterpret_cast<volatile const int *>(&A.ctrl->zany) != 0)
        sweep2_range_z<K, R, ACC, true>(A, beg, end, my, mz, first);
    else
        sweep2_range_z<K, R, ACC, false>(A, beg, end, my, mz, first);
}

template <int K, typename R, int ACC>
__global__ void __launch_bounds__(kSweepThreads, SweepOcc<R, K>::v2) k_sweep2(Sweep2Args A)
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
        k_predeposit<KK, RR, AA><<<grid, kSweepThreads, 0, s>>>(a);                                 \
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
        k_sweep2<KK, RR, AA><<<grid, kSweepThreads, 0, s>>>(a);                                     \
        return 0;                                                                                   \
    }
    PIC_FOR_SWEEP_VARIANTS(L2)
#undef L2
    return 1;
}

// ---------------------------------------------------------------------------
// Diagnostics, evaluated in double from the stored state.
// ---------------------------------------------------------------------------
// charge moments sum_a v^m per cell
template <int K, typename R>
__global__ void __launch_bounds__(kSweepThreads) k_charge(DiagArgs A)
{
    const int32_t *__restrict__ cp = A.P.cell;
    const R *__restrict__ tp = static_cast<const R *>(A.P.t);
    const int lane = threadIdx.x & 31, M = A.M;
    long long wb, we;
    grid_warp_chunk(A.np, wb, we);
    MomentWindow<kWin2, K + 1, AccNative<double>> win;
    win.start();
    for (long long s = wb; s < we; s += 32) {
        const long long a = s + lane;
        const bool act = a < we;
        const unsigned amask = __ballot_sync(0xffffffffu, act);
        const int c = warp_unwrap_cell(act ? cp[a] : 0, act, M);
        const double v = act ? (double)tp[a] - 0.5 : 0.0;
        const int nb = window_base<kWin2>(win.base, c, c, act, amask);
        if (nb != win.base) win.move(nb, A.mom, M);
        double x[K + 1];
        x[0] = 1.0;
#pragma unroll
        for (int m = 1; m <= K; ++m) x[m] = x[m - 1] * v;
        deposit_points<kWin2, K + 1>(win, A.mom, M, act, c, x);
    }
    win.flush(A.mom, M);
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
        A.out[A.P.id[a]] = horner<D + 1>(c, (double)tp[a] - 0.5);
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
        bspline_vals<K, double>((double)tp[a], v);
        double Ay = 0.0, Az = 0.0;
#pragma unroll
        for (int r = 0; r <= K; ++r) {
            const int i = wrap_cell(c - r, A.M);
            Ay += A.c0[i] * v[r];
            Az += A.c1[i] * v[r];
        }
        const double p = (double)pp[a];
        const double q = p * p + Ay * Ay + Az * Az;
        acc += A.w * q / (1.0 + sqrt(1.0 + q));      // w (gamma - 1) without cancellation
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
// out[id] holds d (length units); it is overwritten with the mean.
template <int K, typename R>
__global__ void __launch_bounds__(256) k_gather_path(DiagArgs A)
{
    const R *tp = static_cast<const R *>(A.P.t);
    bool bad = false;
    constexpr int PE = CoefPad<double, K>::v;
    const double inv = 1.0 / A.dx;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < A.np; a += stride) {
        int g = A.P.cell[a];
        const int id = A.P.id[a];
        const double d = A.out[id] * inv;
        if (!(fabs(d) <= (double)A.Dlim)) { bad = true; A.out[id] = 0.0; continue; }
        const double t0 = (double)tp[a];
        int n;
        double t1;
        path_end(t0, d, n, t1);
        const int an = abs(n);
        const bool right = n > 0;
        double sum = 0.0, W = 0.0;
        for (int q = 0; q <= an; ++q) {
            const double ta = q == 0 ? t0 : (right ? 0.0 : 1.0);
            const double tb = q == an ? t1 : (right ? 1.0 : 0.0);
            double S[K], c[K];
            path_sums<K, double>(ta - 0.5, tb - 0.5, S);
            load_coef<K>(A.tab + (size_t)g * PE, c);
            double e = c[0];
#pragma unroll
            for (int m = 1; m < K; ++m) e = fma(c[m], S[m], e);
            const double h = an == 0 ? 1.0 : tb - ta;
            sum = fma(h, e, sum);
            W += h;
            g += right ? 1 : -1;
            g = g >= A.M ? g - A.M : (g < 0 ? g + A.M : g);
        }
        A.out[id] = an == 0 ? sum : sum / W;
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
__device__ __forceinline__ void spin_field_grad(const SpinArgs &A, int c, double t, double &Y, double &Z)
{
    double v[K];
    bspline_vals<K - 1, double>(t, v);
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

template <int K>
__global__ void __launch_bounds__(256) k_spin_deposit(SpinArgs A)
{
    extern __shared__ __align__(16) double s_dep[];
    double *sy = s_dep, *sz = s_dep + A.M;
    for (int i = threadIdx.x; i < 2 * A.M; i += blockDim.x) s_dep[i] = 0.0;
    __syncthreads();
    const double *tp = static_cast<const double *>(A.P.t);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < A.np; a += stride) {
        const int c = A.P.cell[a];
        const int id = A.P.id[a];
        double v[K];
        bspline_vals<K - 1, double>(tp[a], v);
        const double wy = A.w * A.sy[id], wz = A.w * A.sz[id];
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const int i = wrap_cell(c - r, A.M);
            atomicAdd(&sy[i], wy * v[r]);
            atomicAdd(&sz[i], wz * v[r]);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < A.M; i += blockDim.x) {
        if (sy[i] != 0.0) atomicAdd(&A.dy[i], sy[i]);
        if (sz[i] != 0.0) atomicAdd(&A.dz[i], sz[i]);
    }
}

// Subsystem III (Eq. spin_rodrigue): s <- s + sin(dt|r|)/|r| (r x s)
//                                         + (1/2) (sin(dt|r|/2)/(|r|/2))^2 r x (r x s),
// r = (0, Z, -Y), Y = dA_y/dx, Z = dA_z/dx at the marker.
template <int K>
__global__ void __launch_bounds__(256) k_spin_rotate(SpinArgs A)
{
    const double *tp = static_cast<const double *>(A.P.t);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < A.np; a += stride) {
        const int id = A.P.id[a];
        double Y, Z;
        spin_field_grad<K>(A, A.P.cell[a], tp[a], Y, Z);
        const double r1 = Z, r2 = -Y;
        const double nr = sqrt(r1 * r1 + r2 * r2);
        const double s0 = A.sx[id], s1 = A.sy[id], s2 = A.sz[id];
        // c1 = r x s, c2 = r x c1, with r0 = 0
        const double c1x = r1 * s2 - r2 * s1, c1y = r2 * s0, c1z = -r1 * s0;
        const double c2x = r1 * c1z - r2 * c1y, c2y = r2 * c1x, c2z = -r1 * c1x;
        double f1, f2;
        if (nr > 0.0) {
            f1 = sin(A.dt * nr) / nr;
            const double hh = sin(0.5 * A.dt * nr) / (0.5 * nr);
            f2 = 0.5 * hh * hh;
        } else {
            f1 = A.dt;
            f2 = 0.5 * A.dt * A.dt;
        }
        A.sx[id] = s0 + f1 * c1x + f2 * c2x;
        A.sy[id] = s1 + f1 * c1y + f2 * c2y;
        A.sz[id] = s2 + f1 * c1z + f2 * c2z;
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

#define PIC_SPIN_LAUNCH(NAME, SMEM)                                                      \
    switch (a.K) {                                                                       \
    case 2: NAME<2><<<grid, 256, SMEM, s>>>(a); break;                                   \
    case 3: NAME<3><<<grid, 256, SMEM, s>>>(a); break;                                   \
    case 4: NAME<4><<<grid, 256, SMEM, s>>>(a); break;                                   \
    case 5: NAME<5><<<grid, 256, SMEM, s>>>(a); break;                                   \
    default: return 1;                                                                   \
    }                                                                                    \
    return 0;

int launch_spin_deposit(const SpinArgs &a, int grid, cudaStream_t s)
{
    const size_t smem = 2 * (size_t)a.M * sizeof(double);
    PIC_SPIN_LAUNCH(k_spin_deposit, smem)
}

int launch_spin_rotate(const SpinArgs &a, int grid, cudaStream_t s) { PIC_SPIN_LAUNCH(k_spin_rotate, 0) }

int launch_spin_energy(const SpinArgs &a, int grid, cudaStream_t s) { PIC_SPIN_LAUNCH(k_spin_energy, 0) }

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

// ---------------------------------------------------------------------------
// End of subsystem I: x^{n+1} = x^n + delta (re-split into cell and offset,
// wrapped periodically), p^{n+1} = p^(k+1).  delta is cleared only where the
// next iteration starts from it (no warm start): the warm starts overwrite it
// before any sweep reads it.
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ void finalize1_range(long long np, int M, const PartPtrs &P, long long a0,
                                                long long stride, bool zero_delta)
{
    R *tp = static_cast<R *>(P.t);
    R *pp = static_cast<R *>(P.p);
    R *dp = static_cast<R *>(P.delta);
    const R *pnp = static_cast<const R *>(P.pnew);
    for (long long a = a0; a < np; a += stride) {
        const R s = tp[a] + dp[a];
        const R f = floor_(s);
        int c = P.cell[a] + (int)f;
        R t = s - f;
        if (t >= R(1)) { t -= R(1); c += 1; }
        P.cell[a] = wrap_cell(c, M);
        tp[a] = t;
        pp[a] = pnp[a];
        if (zero_delta) dp[a] = R(0);
    }
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
        int c = (int)f;
        R t = (R)(u - f);
        if (t >= R(1)) { t = R(0); c += 1; }
        P.cell[a] = wrap_cell(c, M);
        tp[a] = t;
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

template <typename R>
__global__ void __launch_bounds__(256) k_store(long long np, double dx, PartPtrs P, double *x, double *p)
{
    const R *tp = static_cast<const R *>(P.t);
    const R *pp = static_cast<const R *>(P.p);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < np; a += stride) {
        const long long i = P.id[a];
        if (x) x[i] = ((double)P.cell[a] + (double)tp[a]) * dx;
        if (p) p[i] = (double)pp[a];
    }
}

int launch_store(int fp32, long long np, double dx, PartPtrs P, double *x, double *p,
                 int grid, int block, cudaStream_t s)
{
    if (fp32) k_store<float><<<grid, block, 0, s>>>(np, dx, P, x, p);
    else k_store<double><<<grid, block, 0, s>>>(np, dx, P, x, p);
    return 0;
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
__global__ void __launch_bounds__(256) k_store_ordered(long long np, double dx, PartPtrs P,
                                                       const int32_t *__restrict__ inv, double *x, double *p)
{
    const R *tp = static_cast<const R *>(P.t);
    const R *pp = static_cast<const R *>(P.p);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < np; i += stride) {
        const long long a = inv[i];
        if (x) x[i] = ((double)P.cell[a] + (double)tp[a]) * dx;
        if (p) p[i] = (double)pp[a];
    }
}

int launch_store_ordered(int fp32, long long np, double dx, PartPtrs P, int32_t *inv, double *x, double *p,
                         int grid, int block, cudaStream_t s)
{
    k_inverse_id<<<grid, block, 0, s>>>(np, P.id, inv);
    if (fp32) k_store_ordered<float><<<grid, block, 0, s>>>(np, dx, P, inv, x, p);
    else k_store_ordered<double><<<grid, block, 0, s>>>(np, dx, P, inv, x, p);
    return 0;
}

// ---------------------------------------------------------------------------
// Counting sort of the markers by key = cell * nbins + velocity bin, the bin being
// the expected displacement tau p in units of 1/per cell (nbins = 16 per, clamped),
// so that a warp's markers share cells and piece counts.  Runs between steps; delta and
// p_new are not carried (each step's first sweep or warm start writes them
// before they are read, and delta is all zero where the iteration starts from
// it).  Atomics are aggregated per warp over equal keys.
// counts: 2 * nkeys int32 (histogram, then cursors).
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
// chunk [beg, end) of block b among nb blocks (a multiple of 32 markers)
__device__ __forceinline__ void chunk_of(long long np, int b, int nb, long long &beg, long long &end)
{
    long long chunk = (np + nb - 1) / nb;
    chunk = (chunk + 31) & ~31LL;
    beg = (long long)b * chunk;
    end = beg + chunk < np ? beg + chunk : np;
}

template <typename R>
__device__ __forceinline__ void hist_range(long long beg, long long end, float tau, int nbins, const PartPtrs &S,
                                           int32_t *counts)
{
    const R *ps = static_cast<const R *>(S.p);
    const int lane = threadIdx.x & 31;
    for (long long base = beg; base < end; base += blockDim.x) {
        const long long a = base + threadIdx.x;
        const bool act = a < end;
        const int key = act ? sort_key(S.cell[a], ps[a], tau, nbins) : -1;
        const unsigned grp = __match_any_sync(0xffffffffu, key);
        if (act && lane == __ffs(grp) - 1) atomicAdd(&counts[key], __popc(grp));
    }
}

template <typename R>
__global__ void __launch_bounds__(256) k_hist(long long np, float tau, int nbins, PartPtrs S, int32_t *counts)
{
    long long beg, end;
    block_chunk(np, beg, end);
    hist_range<R>(beg, end, tau, nbins, S, counts);
}

__device__ __forceinline__ void scan_block(int nkeys, int32_t *counts)
{
    // exclusive scan of nkeys counts into cursors (single block)
    __shared__ int s_part[1024];
    const int per = (nkeys + blockDim.x - 1) / blockDim.x;
    const int lo = threadIdx.x * per, hi = min(nkeys, lo + per);
    int s = 0;
    for (int i = lo; i < hi; ++i) s += counts[i];
    s_part[threadIdx.x] = s;
    __syncthreads();
    for (int off = 1; off < (int)blockDim.x; off <<= 1) {
        const int v = threadIdx.x >= (unsigned)off ? s_part[threadIdx.x - off] : 0;
        __syncthreads();
        s_part[threadIdx.x] += v;
        __syncthreads();
    }
    int run = s_part[threadIdx.x] - s;     // exclusive prefix of this thread's range
    for (int i = lo; i < hi; ++i) { const int v = counts[i]; counts[nkeys + i] = run; run += v; }
}

__global__ void __launch_bounds__(1024) k_scan(int nkeys, int32_t *counts) { scan_block(nkeys, counts); }

template <typename R>
__device__ __forceinline__ void scatter_range(long long beg, long long end, float tau, int nbins, const PartPtrs &S,
                                              const PartPtrs &D, int32_t *cursor)
{
    const R *ts = static_cast<const R *>(S.t);
    const R *ps = static_cast<const R *>(S.p);
    R *td = static_cast<R *>(D.t);
    R *pd = static_cast<R *>(D.p);
    const int lane = threadIdx.x & 31;
    // kSortU markers a thread per pass: their cursor atomics are independent, so
    // the warp waits for the returned slots once per pass instead of once a marker
    constexpr int kSortU = 4;
    for (long long base = beg; base < end; base += kSortU * (long long)blockDim.x) {
        int c[kSortU], key[kSortU], first[kSortU];
        R p[kSortU];
        unsigned grp[kSortU];
#pragma unroll
        for (int u = 0; u < kSortU; ++u) {
            const long long a = base + u * (long long)blockDim.x + threadIdx.x;
            const bool act = a < end;
            c[u] = act ? S.cell[a] : 0;
            p[u] = act ? ps[a] : R(0);
            key[u] = act ? sort_key(c[u], p[u], tau, nbins) : -1;
        }
#pragma unroll
        for (int u = 0; u < kSortU; ++u) {
            grp[u] = __match_any_sync(0xffffffffu, key[u]);
            first[u] = 0;
            if (key[u] >= 0 && lane == __ffs(grp[u]) - 1) first[u] = atomicAdd(&cursor[key[u]], __popc(grp[u]));
        }
#pragma unroll
        for (int u = 0; u < kSortU; ++u) {
            const long long a = base + u * (long long)blockDim.x + threadIdx.x;
            const int f = __shfl_sync(0xffffffffu, first[u], __ffs(grp[u]) - 1);
            if (key[u] < 0) continue;
            const long long j = (long long)f + __popc(grp[u] & ((1u << lane) - 1u));
            D.cell[j] = c[u];
            td[j] = ts[a];
            pd[j] = p[u];
            D.id[j] = S.id[a];
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(256) k_scatter(long long np, float tau, int nbins, PartPtrs S, PartPtrs D,
                                                 int32_t *cursor)
{
    long long beg, end;
    block_chunk(np, beg, end);
    scatter_range<R>(beg, end, tau, nbins, S, D, cursor);
}

// Batched sorts (ensembles): block row y = run, its counts zeroed, histogrammed,
// scanned (one block a run) and scattered in four launches for all runs due.
__global__ void __launch_bounds__(256) k_sort_zero_ens(const SortRun *runs)
{
    const SortRun &r = runs[blockIdx.y];
    const int n = 2 * r.M * r.nbins;
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

__global__ void __launch_bounds__(1024) k_scan_ens(const SortRun *runs)
{
    const SortRun &r = runs[blockIdx.x];
    scan_block(r.M * r.nbins, r.counts);
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
    k_scan_ens<<<nruns, 1024, 0, s>>>(runs);
    if (fp32) k_scatter_ens<float><<<g, 256, 0, s>>>(runs);
    else k_scatter_ens<double><<<g, 256, 0, s>>>(runs);
    return 0;
}

int launch_sort(int fp32, long long np, int M, double tau, int per, PartPtrs src, PartPtrs dst,
                int32_t *counts, int grid, int block, cudaStream_t s)
{
    const int nbins = kVelBinsBase * per;
    const int nkeys = M * nbins;
    const float taup = (float)(tau * per);
    if (cudaMemsetAsync(counts, 0, sizeof(int32_t) * 2 * (size_t)nkeys, s) != cudaSuccess) return 1;
    if (fp32) k_hist<float><<<grid, block, 0, s>>>(np, taup, nbins, src, counts);
    else k_hist<double><<<grid, block, 0, s>>>(np, taup, nbins, src, counts);
    k_scan<<<1, 1024, 0, s>>>(nkeys, counts);
    if (fp32) k_scatter<float><<<grid, block, 0, s>>>(np, taup, nbins, src, dst, counts + nkeys);
    else k_scatter<double><<<grid, block, 0, s>>>(np, taup, nbins, src, dst, counts + nkeys);
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
    warp_chunk(ib, ie, threadIdx.x >> 5, kSweepWarps, beg, end);
    return true;
}

template <int K, typename R>
__global__ void __launch_bounds__(kSweepThreads, SweepOcc<R, K>::v1)
    k_sweep1_ens(const Sweep1Args *runs, int nruns, EnsQueue *Q)
{
    if ((int)blockIdx.x >= Q->nblocks) return;
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
__global__ void __launch_bounds__(kSweepThreads, SweepOcc<R, K>::v1)
    k_predeposit_ens(const Sweep1Args *runs, int nruns, EnsQueue *Q)
{
    if ((int)blockIdx.x >= Q->nblocks) return;
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
__global__ void __launch_bounds__(kSweepThreads, SweepOcc<R, K>::v2)
    k_sweep2_ens(const Sweep2Args *runs, int nruns, EnsQueue *Q)
{
    if ((int)blockIdx.x >= Q->nblocks) return;
    int run;
    long long beg, end;
    while (ens_claim(Q, runs, nruns, run, beg, end)) sweep2_range<K, R, DefaultAcc<R>::v>(runs[run], beg, end);
}

template <typename R>
static int launch_sweep_ens_t(int which, int K, const void *runs, int nruns, EnsQueue *Q, int grid, cudaStream_t s)
{
    const int b = kSweepThreads;
#define ENS(KK)                                                                                          \
    case KK:                                                                                             \
        if (which == 1) k_sweep1_ens<KK, R><<<grid, b, 0, s>>>((const Sweep1Args *)runs, nruns, Q);      \
        else if (which == 2) k_sweep2_ens<KK, R><<<grid, b, 0, s>>>((const Sweep2Args *)runs, nruns, Q); \
        else k_predeposit_ens<KK, R><<<grid, b, 0, s>>>((const Sweep1Args *)runs, nruns, Q);             \
        break;
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

static int set_attrs_spin(size_t smem)
{
    int rc = 0;
    rc |= cudaFuncSetAttribute(k_spin_deposit<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess;
    rc |= cudaFuncSetAttribute(k_spin_deposit<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess;
    rc |= cudaFuncSetAttribute(k_spin_deposit<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess;
    rc |= cudaFuncSetAttribute(k_spin_deposit<5>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess;
    return rc;
}

int spin_optin(int M)
{
    static std::mutex mu;
    static size_t have = 0;
    std::lock_guard<std::mutex> lock(mu);
    const size_t need = 2 * (size_t)M * sizeof(double);
    if (need <= have) return 0;
    if (set_attrs_spin(need)) return 1;
    have = need;
    return 0;
}

int sweep_blocks_per_sm(int K, int fp32, int acc, int which)
{
    int n = 0;
    cudaError_t e = cudaErrorInvalidValue;
#define OCC(KK, RR, AA)                                                                                   \
    if (K == KK && (fp32 != 0) == std::is_same<RR, float>::value && acc == AA)                           \
        e = which == 1 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_sweep1<KK, RR, AA>, kSweepThreads, 0) \
                       : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_sweep2<KK, RR, AA>, kSweepThreads, 0);
    PIC_FOR_SWEEP_VARIANTS(OCC)
#undef OCC
    return e == cudaSuccess ? n : 0;
}

}  // namespace pic
