// pic_sweep.cuh -- the marker sweeps of subsystems I and II and the end of subsystem I, as
// device functions over a warp's range of markers (launched by pic_particles.cu, and all
// in one kernel by pic_small.cuh).
#pragma once

#include <climits>
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
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
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
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
            const double x = s_max[i];
            u = (x > u || x != x) ? x : u;
        }
        if (u != 0.0) atomic_max_nonneg(dst, u);      // (a NaN is not equal to 0)
    }
    __syncthreads();
}

// Start-point cache of the double form: (A_y, gamma) and, with the z component, (A_z, 0)
// per marker, 16-byte accesses.  A(x^n) and gamma(p^n, A(x^n)) do not change during a
// fixed-point loop: its first sweep stores them and the later ones read them back (the
// bytes against a dozen operations on the narrow FP64 pipe; in the float form the bytes
// would cost more than the operations).
template <bool Z>
__device__ __forceinline__ void start_cache_store(void *base, long long a, double y, double z, double g)
{
    double2 *q = reinterpret_cast<double2 *>(base) + 2 * a;
    q[0] = make_double2(y, g);
    if (Z) q[1] = make_double2(z, 0.0);
}

template <bool Z>
__device__ __forceinline__ void start_cache_load(const void *base, long long a, double &y, double &z, double &g)
{
    const double2 *q = reinterpret_cast<const double2 *>(base) + 2 * a;
    const double2 u = q[0];
    y = u.x;
    g = u.y;
    if (Z) z = q[1].x;
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
// (path_sums); the deposit adds the end point's moments and the knots crossed.
//
// What bounds it: the FP32 form instruction issue, the FP64 form the FP64 pipe (1/64 of
// the FP32 rate).  us a launch, float (1e8 markers, 2048 cells, cubic) and double (1e7):
//   basis triangles at both ends, piece means, node windows     2160   4200
//   cell polynomials, path moments h S_m in every cell visited  1680   2680
//   end-point moments and knot counts, centred offsets, roots
//   and quotients without exception paths, two markers a lane    992   1513
//   double: path ends, moments and seeds off the FP64 pipe         -   1042
// PRE: the predicted start instead of a sweep -- the proposal delta^(0) (the
// explicit predictor when A.warm, else the one already in delta) is written back
// and its path current deposited into A.mom; no gather walk, no momentum update.
// ---------------------------------------------------------------------------
// The update of one marker from the iterate v0 -> v0 + d: path integrals over the first
// piece, over the q-th piece (in the cells beyond), and the new momentum and displacement.
// ay, az: coefficients of A in the marker's cell.  S: with spin terms.
template <int K, typename R, bool Z, bool S>
struct Kick {
    static constexpr int NC = K + 1, PA = CoefPad<R, NC>::v, PE = CoefPad<R, K>::v;
    R v1, h0, EI, Qy, Qz, W, D2y, D2z;
    int an, g;
    bool right;
    __device__ __forceinline__ void start(const R *TE, int cell, R v0, R d, const R (&ay)[NC], const R (&az)[NC], bool spin)
    {
        const R one = R(1), half = R(0.5);
        int n;
        path_end_open(v0, d, n, v1);
        // callers loop up to an: bounded for a position that is not a number.  By a mask: a
        // minimum here or in the loops takes 977 .. 987 us a launch (1e8 markers, cubic), this
        // 971, as without a bound
        an = abs(n) & kMaxPathCells;
        right = n > 0;
        g = cell;
        const R vb = an == 0 ? v1 : (right ? half : -half);
        h0 = vb - v0;
        R P[K], ec[K];
        path_sums<K, R>(v0, vb, P);
        load_coef<K>(TE + (size_t)cell * PE, ec);
        R e = ec[0], y = ay[1], z = Z ? az[1] : R(0);
#pragma unroll
        for (int m = 1; m < K; ++m) {
            e = fma(ec[m], P[m], e);
            y = fma(ay[m + 1], P[m], y);
            if (Z) z = fma(az[m + 1], P[m], z);
        }
        // one piece: the means are e, y, z themselves (weight 1, no division by h)
        const R hw = an == 0 ? one : h0;
        EI = hw * e;
        Qy = hw * y;
        Qz = Z ? hw * z : R(0);
        W = hw;
        D2y = D2z = R(0);
        if constexpr (S) {
            if (spin) {
                // path integral of d^2A/dx^2 (cell units) for the Zeeman term: the
                // difference quotient of A' = sum_m m A_m v^(m-1)
#pragma unroll
                for (int m = 2; m <= K; ++m) {
                    D2y = fma(R(m) * ay[m], P[m - 2], D2y);
                    D2z = fma(R(m) * az[m], P[m - 2], D2z);
                }
                D2y *= hw;
                D2z *= hw;
            }
        }
    }
    __device__ __forceinline__ void piece(const R *TA, const R *TE, int M, int q, bool spin)
    {
        const R half = R(0.5);
        g = wrap_once(g + (right ? 1 : -1), M);
        const R va = right ? -half : half;
        const R vb = q == an ? v1 : -va;
        const R h = q <= an ? vb - va : R(0);
        R P[K], ec[K], by[NC];
        edge_sums<K, R>(right, va, vb, P);
        load_coef<K>(TE + (size_t)g * PE, ec);
        load_coef<NC>(TA + (size_t)g * (2 * PA), by);
        R e = ec[0], y = by[1];
#pragma unroll
        for (int m = 1; m < K; ++m) {
            e = fma(ec[m], P[m], e);
            y = fma(by[m + 1], P[m], y);
        }
        EI = fma(h, e, EI);
        Qy = fma(h, y, Qy);
        if (an != 0) W += h;
        R bz[NC];
        if (Z) {
            load_coef<NC>(TA + (size_t)g * (2 * PA) + PA, bz);
            R z = bz[1];
#pragma unroll
            for (int m = 1; m < K; ++m) z = fma(bz[m + 1], P[m], z);
            Qz = fma(h, z, Qz);
        }
        if constexpr (S) {
            if (spin) {
                R y2 = R(0), z2 = R(0);
#pragma unroll
                for (int m = 2; m <= K; ++m) {
                    y2 = fma(R(m) * by[m], P[m - 2], y2);
                    z2 = fma(R(m) * bz[m], P[m - 2], z2);
                }
                D2y = fma(h, y2, D2y);
                D2z = fma(h, z2, D2z);
            }
        }
    }
    // zeeman(W, D2y, D2z): the kick of the spin term
    template <class F>
    __device__ __forceinline__ void finish(R pn, R A0y, R A0z, R g0, R tau, F &&zeeman, R &pnew, R &dnew) const
    {
        // A(x^(k)) = A(x^n) + the path integral of dA/dx, of the staged field
        const R one = R(1), hs = an == 0 ? h0 : one;
        const R A1y = fma(hs, Qy, A0y);
        // p^(k+1) = p^n + tau (Ebar - (A1 + A0).D / (g1 + g0)) with Ebar = EI/W,
        // D = Q/W (W the summed pieces, 1 for a single one), as one division
        R q1 = fma(A1y, A1y, one), nm = (A1y + A0y) * Qy;
        if (Z) {
            const R A1z = fma(hs, Qz, A0z);
            q1 = fma(A1z, A1z, q1);
            nm = fma(A1z + A0z, Qz, nm);
        }
        const R g1 = root(fma(pn, pn, q1));
        const R G = g1 + g0;
        R kick = quotient(fma(EI, G, -nm), W * G);
        if constexpr (S) kick -= zeeman(W, D2y, D2z);
        pnew = fma(tau, kick, pn);
        dnew = quotient(tau * (pn + pnew), g1 + root(fma(pnew, pnew, q1)));
    }
};

// Z: the z component is not identically zero (a linearly polarised wave keeps A_z = 0
// exactly, and then none of its terms are needed).
template <int K, typename R, int ACC, bool PRE, bool Z>
__device__ __forceinline__ void sweep1_range_z(const Sweep1Args &A, long long beg, long long end, double &dmax_out,
                                               bool &bad_out)
{
    constexpr int NC = K + 1;                           // coefficients of A in a cell
    constexpr int PA = CoefPad<R, NC>::v;
    constexpr int U = SweepU<R>::v;                     // markers a lane and step
    constexpr bool kSpin = !Real<R>::fp32 && !PRE && Z;
    const R one = R(1);
    double *mom = A.mom;
    int *flux = A.flux;
    bool warm = A.warm != 0;
    bool first = A.first != 0;
    if (!PRE && A.graph) {                  // replayed by a graph: buffers by sweep parity
        const int it = *reinterpret_cast<volatile const int *>(&A.ctrl->iter);
        mom = A.mpair[it & 1];
        flux = A.fpair[it & 1];
        warm = warm && it == 0;
        first = it == 0;
    }
    const int M = A.M;
    const int32_t *cp = A.P.cell;
    const R *vp = static_cast<const R *>(A.P.t);
    const R *pp = static_cast<const R *>(A.P.p);
    R *dp = static_cast<R *>(A.P.delta);
    R *pnp = static_cast<R *>(A.P.pnew);
    const R *TA = static_cast<const R *>(A.T.A), *TE = static_cast<const R *>(A.T.E);
    const R tau = (R)(A.dt / A.dx);
    const R dlim = (R)A.Dlim;
    const bool spin = kSpin && A.hbar != 0.0;
    const bool cached = !Real<R>::fp32 && !PRE && !first && A.a0 != nullptr;
    const bool keep = !Real<R>::fp32 && !PRE && first && A.a0 != nullptr;
    const int lane = threadIdx.x & 31;
    R dmax = R(0);
    bool bad = false;
    if (beg >= end) return;
    constexpr bool kFixed = !Real<R>::fp32 && ACC == ACC_NATIVE;
    PathDeposit<K, U, typename std::conditional<kFixed, AccFixed, typename AccOf<R, ACC>::T>::type> dep;
    dep.start(mom, flux, M, cp[beg]);

    // the next step's markers are loaded while this one's are computed
    int nc[U];
    R nv[U], npn[U], nd[U];
    auto fetch = [&](long long s) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long a = s + 32 * u + lane;
            if (a < end) {
                nc[u] = cp[a];
                nv[u] = vp[a];
                npn[u] = pp[a];
                if (!warm) nd[u] = dp[a];
            } else {
                nv[u] = R(0);
                npn[u] = R(0);
                nd[u] = R(0);
            }
        }
    };
#pragma unroll
    for (int u = 0; u < U; ++u) { nc[u] = 0; nd[u] = R(0); }
    fetch(beg);
    for (long long s = beg; s < end; s += 32 * U) {
        bool act[U];
        int cw[U];
        R v0[U], pn[U], dold[U], dnew[U], pnew[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            act[u] = s + 32 * u + lane < end;
            cw[u] = nc[u];
            v0[u] = nv[u];
            pn[u] = npn[u];
            dold[u] = nd[u];
        }
        if (s + 32 * U < end) fetch(s + 32 * U);
        // A(x^n), gamma(p^n, A(x^n))
        R A0y[U], A0z[U], g0[U], ay[U][NC], az[U][NC];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t row = (size_t)cw[u] * (2 * PA);
            load_coef<NC>(TA + row, ay[u]);
            if (Z) load_coef<NC>(TA + row + PA, az[u]);
            A0z[u] = R(0);
            if (cached) {
                if constexpr (!Real<R>::fp32) {
                    A0y[u] = R(0);
                    g0[u] = one;
                    if (act[u]) start_cache_load<Z>(A.a0, s + 32 * u + lane, A0y[u], A0z[u], g0[u]);
                }
            } else {
                A0y[u] = horner<NC>(ay[u], v0[u]);
                R q0 = fma(A0y[u], A0y[u], fma(pn[u], pn[u], one));
                if (Z) {
                    A0z[u] = horner<NC>(az[u], v0[u]);
                    q0 = fma(A0z[u], A0z[u], q0);
                }
                g0[u] = root(q0);
                if constexpr (!Real<R>::fp32)
                    if (keep && act[u]) start_cache_store<Z>(A.a0, s + 32 * u + lane, A0y[u], A0z[u], g0[u]);
            }
            if (warm) dold[u] = quotient(tau * pn[u], g0[u]);
            if (!within(dold[u], dlim)) { bad = bad || act[u]; dold[u] = R(0); }
        }
        if constexpr (PRE) {
#pragma unroll
            for (int u = 0; u < U; ++u) dnew[u] = dold[u];
        } else {
            Kick<K, R, Z, kSpin> k[U];
            int nmax = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                k[u].start(TE, cw[u], v0[u], dold[u], ay[u], az[u], spin);
                nmax = max(nmax, k[u].an);
            }
            nmax = __reduce_max_sync(0xffffffffu, nmax);
            for (int q = 1; q <= nmax; ++q) {
#pragma unroll
                for (int u = 0; u < U; ++u) k[u].piece(TA, TE, M, q, spin);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                k[u].finish(pn[u], A0y[u], A0z[u], g0[u], tau, [&](R W, R D2y, R D2z) -> R {
                    if (!spin || !act[u]) return R(0);
                    const int id = A.P.id[s + 32 * u + lane];
                    return (R)(A.hbar / A.dx * ((A.sy[id] * D2z - A.sz[id] * D2y) / W));
                }, pnew[u], dnew[u]);
                if (!within(dnew[u], dlim)) { bad = bad || act[u]; dnew[u] = R(0); }
                if (act[u]) {
                    R inc = fabs(dnew[u] - dold[u]);
                    if constexpr (Real<R>::fp32) inc *= approx_rcp(fmaxf(one, fabsf(dnew[u])));   // convergence metric only
                    dmax = max_nonneg(dmax, inc);
                }
            }
        }
        // deposit of the path x^n -> x^(k+1); its end is the position finalize stores
        int n1[U];
        R ve[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            path_end_open(v0[u], dnew[u], n1[u], ve[u]);
            if (act[u]) {
                const long long a = s + 32 * u + lane;
                dp[a] = dnew[u];
                if constexpr (!PRE) pnp[a] = pnew[u];
            }
        }
        dep.step(act, cw, n1, ve);
    }
    dep.flush();
    dmax_out = max_nonneg(dmax_out, (double)dmax);
    bad_out = bad_out || bad;
}

template <int K, typename R, int ACC, bool PRE>
__device__ __forceinline__ void sweep1_range(const Sweep1Args &A, long long beg, long long end, double &dmax, bool &bad)
{
    if (A.zforce || *reinterpret_cast<volatile const int *>(&A.ctrl->zany) != 0)
        sweep1_range_z<K, R, ACC, PRE, true>(A, beg, end, dmax, bad);
    else
        sweep1_range_z<K, R, ACC, PRE, false>(A, beg, end, dmax, bad);
}

// ---------------------------------------------------------------------------
// Subsystem II: one fixed-point sweep (Sec. 4.2).  Markers frozen at x; with
// A0 = A^n_h(x), A1 = A^(k)_h(x):
//   s_i += w (A0 + A1) Lambda^0_i(x) / (g(p,A0) + g(p,A1))   (y and z),
// deposited as the moments f v^m of each cell.  Same warp ranges as subsystem I.
// us a launch, float (1e8 markers, cubic) and double (1e7): basis values and node windows
// 1260 and 2060, cell polynomials and moments 767 and 830, as here (centred offsets, the
// short root and quotient, two markers a lane) 570 and 672, with their seeds refined off the
// FP64 pipe 610 in double, with the moments as 64-bit integers 303 (301 with one scale a
// warp instead of one a cell, which took the digits of weak fields in its range).
// Z: the z component is not identically zero, as in subsystem I.
// f = (s + L) / G, s = A^n + A^(k) of a component, G = g0 + g1, L the float form's residue.
// The float rounding of a coefficient is the same for every marker of its cell, so it
// does not average out over markers: in the exchange term (A1 - A0)(A1 + A0)/(g0 + g1) it
// shows as an energy error of about 1e-11 per step.  The residues L of the sum a^n + a^(k)
// enter before its one rounding, which leaves only per-marker rounding: the quotient's
// reciprocal times s, rounded once, with the product's own rounding error (exact by an
// fma) and the reciprocal times L added to it (L is far below half an ulp of s).
template <typename R, bool Z>
__device__ __forceinline__ void exchange(R sy, R sz, R G, R Ly, R Lz, R &fy, R &fz)
{
    const R cf = quotient(R(1), G);
    if constexpr (Real<R>::fp32) {
        const float py = cf * sy;
        fy = py + fmaf(cf, Ly, fmaf(cf, sy, -py));
        if (Z) {
            const float pz = cf * sz;
            fz = pz + fmaf(cf, Lz, fmaf(cf, sz, -pz));
        }
    } else {
        fy = cf * sy;
        if (Z) fz = cf * sz;
    }
}

template <int K, typename R, int ACC, bool Z>
__device__ __forceinline__ void sweep2_range_z(const Sweep2Args &A, long long beg, long long end, double *my, double *mz,
                                               bool first)
{
    constexpr int NC = K + 1;
    constexpr int PA = CoefPad<R, NC>::v;
    constexpr int NW = Z ? kWin2z : kWin2;
    constexpr int U = SweepU<R>::v;
    const R one = R(1);
    const int M = A.M;
    const int32_t *cp = A.P.cell;
    const R *vp = static_cast<const R *>(A.P.t);
    const R *pp = static_cast<const R *>(A.P.p);
    const R *TA = static_cast<const R *>(A.T.A), *TK = static_cast<const R *>(A.T.Kt);
    const float *TL = A.T.L;
    const bool cached = !Real<R>::fp32 && !first && A.a0 != nullptr;
    const bool keep = !Real<R>::fp32 && first && A.a0 != nullptr;
    const int lane = threadIdx.x & 31;
    if (beg >= end) return;
    constexpr bool kFixed = !Real<R>::fp32 && ACC == ACC_NATIVE;
    using Window = typename std::conditional<kFixed, ScaledWindow<NW, NC>, MomentWindow<NW, NC, typename AccOf<R, ACC>::T>>::type;
    Window wy, wz;
    wy.clear();
    if (Z) wz.clear();
    int base = cp[beg], adds = 0;
    unsigned used = 0u;
    auto flush = [&]() {
        wy.flush(my, base, used, M);
        if (Z) wz.flush(mz, base, used, M);
        used = 0u;
        adds = 0;
    };
    int nc[U];
    R nv[U], npn[U];
    auto fetch = [&](long long s) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long a = s + 32 * u + lane;
            if (a < end) {
                nc[u] = cp[a];
                nv[u] = vp[a];
                npn[u] = pp[a];
            }
        }
    };
#pragma unroll
    for (int u = 0; u < U; ++u) { nc[u] = 0; nv[u] = R(0); npn[u] = R(0); }
    fetch(beg);
    for (long long s = beg; s < end; s += 32 * U) {
        bool act[U], in[U];
        int cw[U], rel[U], miss = 0;
        R v[U], p[U], fy[U], fz[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            act[u] = s + 32 * u + lane < end;
            cw[u] = nc[u];
            v[u] = nv[u];
            p[u] = npn[u];
        }
        if (s + 32 * U < end) fetch(s + 32 * U);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const R pp1 = fma(p[u], p[u], one);
            const size_t row = (size_t)cw[u] * (2 * PA);
            R A0y, A1y, A0z = R(0), A1z = R(0), g0;
            R c[NC];
            if (cached) {
                if constexpr (!Real<R>::fp32) {
                    A0y = R(0);
                    g0 = one;
                    if (act[u]) start_cache_load<Z>(A.a0, s + 32 * u + lane, A0y, A0z, g0);
                }
            } else {
                load_coef<NC>(TA + row, c);
                A0y = horner<NC>(c, v[u]);
                R q = fma(A0y, A0y, pp1);
                if (Z) {
                    load_coef<NC>(TA + row + PA, c);
                    A0z = horner<NC>(c, v[u]);
                    q = fma(A0z, A0z, q);
                }
                g0 = root(q);
                if constexpr (!Real<R>::fp32)
                    if (keep && act[u]) start_cache_store<Z>(A.a0, s + 32 * u + lane, A0y, A0z, g0);
            }
            load_coef<NC>(TK + row, c);
            A1y = horner<NC>(c, v[u]);
            R q1 = fma(A1y, A1y, pp1);
            if (Z) {
                load_coef<NC>(TK + row + PA, c);
                A1z = horner<NC>(c, v[u]);
                q1 = fma(A1z, A1z, q1);
            }
            R Ly = R(0), Lz = R(0);
            if constexpr (Real<R>::fp32) {
                load_coef<NC>(TL + row, c);
                Ly = horner<NC>(c, v[u]);
                if (Z) {
                    load_coef<NC>(TL + row + PA, c);
                    Lz = horner<NC>(c, v[u]);
                }
            }
            exchange<R, Z>(A0y + A1y, A0z + A1z, g0 + root(q1), Ly, Lz, fy[u], fz[u]);
            rel[u] = rel_cell(cw[u], base, M);
            in[u] = act[u] && (unsigned)rel[u] < (unsigned)NW;
            // infinities, NaN: to global memory as they are
            if constexpr (kFixed) in[u] = in[u] && exponent_of(fy[u]) < 2000 && (!Z || exponent_of(fz[u]) < 2000);
            miss += __popc(__ballot_sync(0xffffffffu, act[u] && !in[u]));
        }
        if (miss > kWindowMisses) {
            int lo = INT_MAX;
#pragma unroll
            for (int u = 0; u < U; ++u) lo = act[u] ? min(lo, rel[u]) : lo;
            const unsigned amask = __ballot_sync(0xffffffffu, act[0]);
            int off = window_move<NW>(lo, rel[0], act[0], amask);
            if (off > 0 && off < NW) {
                for (; off > 0; --off) {
                    wy.shift(my, base, used);
                    if (Z) wz.shift(mz, base, used);
                    used >>= 1;
                    base = base + 1 == M ? 0 : base + 1;
                }
            } else if (off != 0) {
                flush();
                base = wrap_cell(base + off, M);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                rel[u] = rel_cell(cw[u], base, M);
                in[u] = act[u] && (unsigned)rel[u] < (unsigned)NW;
                if constexpr (kFixed) in[u] = in[u] && exponent_of(fy[u]) < 2000 && (!Z || exponent_of(fz[u]) < 2000);
            }
        }
        unsigned bits = 0u;
#pragma unroll
        for (int u = 0; u < U; ++u) bits |= in[u] ? 1u << rel[u] : 0u;
        const unsigned mask = __reduce_or_sync(0xffffffffu, bits);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int r = in[u] ? rel[u] : -1;
            if constexpr (kFixed) {
                const long long q = to_fixed<63>(v[u]);
                wy.add(my, base, used, M, mask, r, fy[u], q);
                if (Z) wz.add(mz, base, used, M, mask, r, fz[u], q);
            } else {
                R x[NC], pw = one;
                x[0] = fy[u];
                R pws[NC];
                pws[0] = one;
#pragma unroll
                for (int m = 1; m < NC; ++m) { pw = m == 1 ? v[u] : pw * v[u]; pws[m] = pw; x[m] = fy[u] * pw; }
                wy.add(mask, r, x);
                if (act[u] && !in[u]) {
                    double *dst = my + (size_t)cw[u] * NC;
#pragma unroll
                    for (int m = 0; m < NC; ++m)
                        if (x[m] != R(0)) atomicAdd(&dst[m], (double)x[m]);
                }
                if (Z) {
                    x[0] = fz[u];
#pragma unroll
                    for (int m = 1; m < NC; ++m) x[m] = fz[u] * pws[m];
                    wz.add(mask, r, x);
                    if (act[u] && !in[u]) {
                        double *dst = mz + (size_t)cw[u] * NC;
#pragma unroll
                        for (int m = 0; m < NC; ++m)
                            if (x[m] != R(0)) atomicAdd(&dst[m], (double)x[m]);
                    }
                }
            }
            if constexpr (kFixed) {
                if (act[u] && !in[u]) {
                    double *dy = my + (size_t)cw[u] * NC, *dz = mz + (size_t)cw[u] * NC;
                    R xy = fy[u], xz = Z ? fz[u] : R(0);
#pragma unroll
                    for (int m = 0; m < NC; ++m) {
                        if (xy != R(0)) atomicAdd(&dy[m], (double)xy);
                        if (Z && xz != R(0)) atomicAdd(&dz[m], (double)xz);
                        xy *= v[u];
                        if (Z) xz *= v[u];
                    }
                }
            }
        }
        used |= mask;
        if (++adds == (kFixed ? kFixedAdds : kMaxLaneAdds) / U) flush();
    }
    flush();
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
    // four markers a thread and pass: the kernel only moves memory (28 bytes a marker in the
    // float form), and one marker's loads did not keep enough of it in flight (2e7 float
    // markers: 162 us one at a time, 80 us so, 7.0 TB/s)
    for (long long i = a0; i < np / 4; i += stride) {
        const int4 c = reinterpret_cast<const int4 *>(P.cell)[i];
        R t[4], d[4], p[4];
        load4(tp + 4 * i, t);
        load4(dp + 4 * i, d);
        load4(pnp + 4 * i, p);
        int g[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int n;
            path_end(t[j], d[j], n, t[j]);
            g[j] = wrap_cell(g[j] + n, M);
            d[j] = R(0);
        }
        reinterpret_cast<int4 *>(P.cell)[i] = make_int4(g[0], g[1], g[2], g[3]);
        store4(tp + 4 * i, t);
        store4(pp + 4 * i, p);
        if (zero_delta) store4(dp + 4 * i, d);
    }
    for (long long a = (np & ~3LL) + a0; a < np; a += stride) {
        int n;
        R v;
        path_end(tp[a], dp[a], n, v);
        P.cell[a] = wrap_cell(P.cell[a] + n, M);
        tp[a] = v;
        pp[a] = pnp[a];
        if (zero_delta) dp[a] = R(0);
    }
}

}  // namespace pic
