// pic_solve.cuh -- grid-side device functions: circulant solves with the convergence
// decision, preparation and end of the substeps (launched by pic_grid.cu, and all in
// one kernel by pic_small.cuh).
#pragma once

#include "pic_internal.h"
#include "pic_poly.cuh"

namespace pic {

// ---------------------------------------------------------------------------
// Convergence decision, made by the last block of a solve kernel.
// FP64 form (Sec. 5, tolerance tol): max |x^(k+1) - x^(k)| <= tol (length) and
// max |e^(k+1) - e^(k)| <= tol.  FP32 form: position increments at the float
// resolution of the offset (dtol, relative to max(1, |delta|)) and field
// increments below tol or no longer shrinking (stagnation at float noise).
// ---------------------------------------------------------------------------
// The test itself: sweep `iter` (counted from 1) moved the markers by at most d (cells; in
// the float form relative to max(1, |delta|)) and the field by e, the sweep before by dp
// and ep; emag: the field's max-norm.
static __device__ bool fixed_point_reached(const ConvArgs &A, int iter, double d, double dp, double e, double ep,
                                           double emag)
{
    if (A.subsystem != 1) d = 0.0;
    if (!A.fp32) return (d * A.dx <= A.tol) && (e <= A.tol);
    // Float iterates stop improving at rounding noise, so increments alone never
    // reach a tight tolerance.  Estimate the remaining error of the new iterate
    // from the increment v_k and the observed contraction r = v_k / v_{k-1}
    // (geometric tail v_k r / (1 - r), r capped at 0.9), and stop when both the
    // position and field estimates are below tolerance, or when both increments
    // have stopped shrinking at noise level.
    auto est = [](double v, double vprev) {
        if (v == 0.0) return 0.0;
        // no previous increment (first sweep): no contraction estimate yet
        double r = (vprev < 1e300) ? v / vprev : 0.9;
        if (!(r < 0.9)) r = 0.9;
        return v * r / (1.0 - r);
    };
    // field tolerance.  Subsystem I: the absolute tol, or erel of the field's
    // max-norm when that is larger, on the last increment itself: the markers'
    // momenta were updated with the field of the sweep before, and that
    // mismatch is proportional to the last increment (not to the estimated
    // remaining error), with a sign that does not average out over steps: a
    // rule on the estimate accepted increments near 1e-7 of the field and let
    // the energy drift by 1e-12 of the total a step on C2.
    // Subsystem II: the estimated remaining error below the absolute tol.  Its
    // markers do not move, the sweep is deterministic, and the remaining field
    // error enters the transverse energy directly.
    const bool dok = (A.subsystem == 1) ? (est(d, dp) <= A.dtol) : true;
    const bool eok = (A.subsystem == 1) ? (e <= fmax(A.tol, A.erel * emag)) : (est(e, ep) <= A.tol);
    const bool dstag = (A.subsystem == 1) ? (d >= 0.5 * dp && d <= 1e-4) : true;
    const bool estag = e >= 0.5 * ep && e <= 1e-8;
    return (dok && eok) || (iter >= 3 && dstag && estag);
}

// The decision taken by the last block of a solve kernel, on the control block.
static __device__ void decide(const ConvArgs &A)
{
    DevCtrl *c = A.ctrl;
    __threadfence();
    if (A.count) *A.count += 1;
    const int iter = c->iter + 1;
    c->iter = iter;
    const bool ok = fixed_point_reached(A, iter, bits_to_double(c->dmax_bits), bits_to_double(c->dprev_bits),
                                        bits_to_double(c->emax_bits), bits_to_double(c->eprev_bits),
                                        bits_to_double(c->emag_bits));
    bool stop = ok;
    if (!ok && iter >= A.max_iter) {
        c->status |= STATUS_NOCONV;
        stop = true;
    }
    if (c->status & (STATUS_NUMERIC | STATUS_TIMEOUT)) stop = true;
    c->converged = stop ? 1 : 0;
    c->dprev_bits = c->dmax_bits;
    c->eprev_bits = c->emax_bits;
    c->dmax_bits = 0ull;
    c->emax_bits = 0ull;
    c->emag_bits = 0ull;
    c->ticket = 0u;
    __threadfence();
    if (A.graph && A.cond_handle)
        cudaGraphSetConditional((cudaGraphConditionalHandle)A.cond_handle, stop ? 0u : 1u);
}

// Spline pieces of every degree (pic_poly.cuh).  Grid kernels take the degree at run time.
static __constant__ SplineTab c_spline = make_spline_tab();

// Pieces of C_i = sum_{j >= i} Lambda^0_j in the cells i + r, r = 0 .. d - 1: the running
// sums over r of the pieces of N^d.
constexpr SplineTab make_cumulative_tab()
{
    SplineTab T = make_spline_tab();
    for (int d = 0; d <= kMaxDegree; ++d)
        for (int r = 1; r <= d; ++r)
            for (int m = 0; m <= d; ++m) T.b[d][r][m] += T.b[d][r - 1][m];
    return T;
}
static __constant__ SplineTab c_cumulative = make_cumulative_tab();

// Stores coefficient m of row `row` (pad numbers a row) in the form's type.
__device__ __forceinline__ void put_coef(void *tab, int fp32, size_t row, int pad, int m, double v)
{
    if (fp32) static_cast<float *>(tab)[row * pad + m] = (float)v;
    else static_cast<double *>(tab)[row * pad + m] = v;
}

// Coefficient m of the degree-D polynomial in the cell whose node r steps down has value at(r).
template <int D, class At>
__device__ __forceinline__ double cell_coef(int m, At &&at)
{
    double s = 0.0;
#pragma unroll
    for (int r = 0; r <= D; ++r) s = fma(c_spline.b[D][r][m], at(r), s);
    return s;
}

// Coefficient m of ebar dx in a cell, divided by m + 1 (the table E).
template <int K, class At>
__device__ __forceinline__ double e_coef(int m, double dx, At &&at)
{
    const double s = cell_coef<K - 1>(m, at) * dx;
    return m == 0 ? s : (m == 1 ? 0.5 * s : s / (double)(m + 1));
}

// Value of a deposit at node j from the moments of degree D (path: coefficient m over m + 1).
__device__ __forceinline__ double node_value(int M, int D, bool path, const double *mom, int j)
{
    const int NV = D + 1;
    double s[kMaxDegree + 1] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    int c = j;
    for (int r = 0; r < NV; ++r) {
        const double *row = mom + (size_t)c * NV;
#pragma unroll
        for (int m = 0; m <= kMaxDegree; ++m)
            if (m < NV) s[m] = fma(c_spline.b[D][r][m], row[m], s[m]);
        c = c + 1 == M ? 0 : c + 1;
    }
    double v = 0.0;
#pragma unroll
    for (int m = 0; m <= kMaxDegree; ++m)
        if (m < NV) v += path ? s[m] * (1.0 / (m + 1)) : s[m];
    return v;
}

// Path current at a node over w dx (pic_poly.cuh): the polynomials of C on the change of the
// moments dm(r, m) in the cells r = 0 .. K - 1 from the node up, and the crossings f(r) of
// their left edges, f(K) of the knot after them.
template <int K, class Dm, class F>
__device__ __forceinline__ double path_node_value(Dm &&dm, F &&f)
{
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int r = 0; r < K; ++r) {
        s0 = fma(c_cumulative.b[K][r][0], (double)(f(r) - f(r + 1)), s0);
#pragma unroll
        for (int m = 1; m <= K; ++m) {
            double &s = (m & 1) ? s1 : s0;
            s = fma(c_cumulative.b[K][r][m], dm(r, m - 1), s);
        }
    }
    return (s0 + s1) + (double)f(K);
}

// The residue of a^n + a^(k) after both coefficients were rounded to float.
__device__ __forceinline__ float sum_residue(double n, double k)
{
    return (float)((n - (double)(float)n) + (k - (double)(float)k));
}

// y_i = sum_n taps[n] in[(i - (d_start + n)) mod M] for the kConvOut nodes
// i0 - K .. i0 - K + kConvOut - 1 of block bx, i0 = bx (kConvOut - K): the block owns the
// last kConvOut - K of them and recomputes the K below, which the polynomials of its cells
// need.  Each half warp sums a share of the taps for all nodes.  What bounds it is latency
// -- a few dependent round trips to L2 and chains on the FP64 pipe -- so a block has few
// nodes (the pipe of one SM takes 16 cycles a warp operation), every loop is unrolled for
// the degree, and loads the epilogue needs are issued at the start.  M = 2048, cubic, event
// to event: 20.8 us with 32 nodes a block and the degree at run time, 12 us so.
// Returns true in the one block that finished the run's solve last (after the
// convergence decision, in the solve modes).  With max_e != NULL the maxima go to
// max_e[0 .. 1] (increment, field) and no decision is taken.  given: the nodes of the component
// when a pass has formed them (ConvArgs::node), else null.
constexpr int kConvOut = 16, kConvThreads = 160, kConvMaxWarps = 8;

// nodes: they are given (conv_block), no moments are staged
inline size_t conv_smem(int K, int ntap, bool nodes)
{
    const int nq = kConvOut + ntap - 1;
    return ((size_t)nq + ntap + (nodes ? 0 : (size_t)(nq + K) * (K + 1)) + kConvMaxWarps * kConvOut + 2 * kConvOut) *
               sizeof(double) +
           (size_t)(nq + K + 1) * sizeof(int);
}
inline int conv_blocks(int M, int K) { return (M + kConvOut - K - 1) / (kConvOut - K); }

// max over the warp of non-negative doubles (NaN counts as the largest), by integer compares
__device__ __forceinline__ double warp_max_nonneg(double v)
{
    long long x = __double_as_longlong(v);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long y = __shfl_xor_sync(0xffffffffu, x, o);
        x = y > x ? y : x;
    }
    return __longlong_as_double(x);
}

// Node j of subsystem II's deposit: r-th cell's moments at(r, m).
template <int K, class At>
__device__ __forceinline__ double solve2_node(const ConvArgs &A, At &&at)
{
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int r = 0; r <= K; ++r)
#pragma unroll
        for (int m = 0; m <= K; ++m) {
            double &s = (m & 1) ? s1 : s0;
            s = fma(c_spline.b[K][r][m], at(r, m), s);
        }
    return A.scale * (s0 + s1);
}

// Node j of component comp into A.node (sweep `it` of the loop).
template <int K>
__device__ __forceinline__ void node_pass(const ConvArgs &A, int it, int j, int comp)
{
    if (j >= A.M) return;
    const double *mom = A.graph ? A.pair[comp][it & 1] : A.mom[comp];
    A.node[comp][j] = solve2_node<K>(A, [&](int r, int m) { return mom[(size_t)wrap_once(j + r, A.M) * (K + 1) + m]; });
}

template <int K>
static __device__ __forceinline__ bool conv_block(const ConvArgs &A, const double *given, CoefTables T, int it, int bx,
                                                  int comp, double *sm, unsigned long long *max_e)
{
    const int M = A.M, i0 = bx * (kConvOut - K), ntap = A.ntap;
    const int nq = kConvOut + ntap - 1;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
    double *s_in = sm, *s_tap = s_in + nq, *s_part = s_tap + ntap;
    double *s_val = s_part + kConvMaxWarps * kConvOut, *s_an = s_val + kConvOut, *s_mom = s_an + kConvOut;
    int *s_flux = reinterpret_cast<int *>(s_mom + (size_t)(nq + K) * K);       // (subsystem I)
    const double *mom = A.mom[comp];
    double *zero = A.zero[comp];
    const int *flux = A.flux;
    int *zflux = A.zflux;
    if (A.graph && A.mode != CONV_PLAIN) {   // buffers by sweep parity
        mom = A.pair[comp][it & 1];
        zero = A.pair[comp][(it + 1) & 1];
        flux = A.fpair[it & 1];
        zflux = A.fpair[(it + 1) & 1];
    }
    if (given) mom = nullptr;
    // the epilogue's loads (lanes 0 .. 15 of warp 0: one node each)
    const int o = lane & (kConvOut - 1), i = i0 - K + o;
    const int iw = wrap_cell(i, M);
    const bool own = wid == 0 && lane < kConvOut && o >= K && i < M;
    double en = 0.0, an = 0.0, eold = 0.0;
    if (wid == 0 && A.mode != CONV_PLAIN) {
        en = A.en[comp][iw];
        if (A.mode == CONV_SOLVE2) an = A.an[comp][iw];
        eold = A.ek[comp][iw];
    }
    // s_in[q]: node (g0 + q) mod M
    const int g0 = wrap_cell(i0 - K - (A.d_start + ntap - 1), M);
    auto node = [&](int q) { int g = g0 + q; while (g >= M) g -= M; return g; };
    for (int n = tid; n < ntap; n += nt) s_tap[n] = A.taps[n];
    if (mom && A.subsystem == 1) {
        for (int q = tid; q < (nq + K) * K; q += nt) {
            const int cell = node(q / K), m = q % K;
            s_mom[q] = mom[(size_t)cell * K + m] - A.mom0[(size_t)cell * K + m];
        }
        for (int q = tid; q < nq + K + 1; q += nt) s_flux[q] = flux[node(q)];
        __syncthreads();
        for (int q = tid; q < nq; q += nt)
            s_in[q] = A.scale * path_node_value<K>([&](int r, int m) { return s_mom[(q + r) * K + m]; },
                                                   [&](int r) { return s_flux[q + r]; });
    } else if (mom) {
        for (int q = tid; q < (nq + K) * (K + 1); q += nt)
            s_mom[q] = mom[(size_t)node(q / (K + 1)) * (K + 1) + q % (K + 1)];
        __syncthreads();
        for (int q = tid; q < nq; q += nt)
            s_in[q] = fma(A.dt, solve2_node<K>(A, [&](int r, int m) { return s_mom[(q + r) * (K + 1) + m]; }),
                          A.b[comp][node(q)]);
    } else {
        const double *in = given ? given : A.in[comp];
        for (int q = tid; q < nq; q += nt) {
            const int g = node(q);
            const double s = in[g];
            s_in[q] = A.mode == CONV_SOLVE2 ? fma(A.dt, s, A.b[comp][g]) : s;
        }
    }
    __syncthreads();
    {
        const int groups = 2 * nw, per = (ntap + groups - 1) / groups;
        const int n0 = (2 * wid + (lane >> 4)) * per, n1 = min(ntap, n0 + per);
        const double *base = s_in + o + ntap - 1;
        double a0 = 0.0, a1 = 0.0;
        int n = n0;
        for (; n + 1 < n1; n += 2) {
            a0 = fma(s_tap[n], base[-n], a0);
            a1 = fma(s_tap[n + 1], base[-n - 1], a1);
        }
        if (n < n1) a0 = fma(s_tap[n], base[-n], a0);
        a0 += a1;
        a0 += __shfl_xor_sync(0xffffffffu, a0, 16);
        if (lane < kConvOut) s_part[wid * kConvOut + o] = a0;
    }
    __syncthreads();
    double diff = 0.0, mag = 0.0;
    if (wid == 0) {
        double y = 0.0;
        for (int w = lane >> 4; w < nw; w += 2) y += s_part[w * kConvOut + o];
        y += __shfl_xor_sync(0xffffffffu, y, 16);
        if (A.mode == CONV_PLAIN) {
            if (own) A.out[comp][i] = y;
        } else {
            const bool two = A.mode == CONV_SOLVE2;
            const double enew = two ? y : en - y;        // P e^(k+1) = b + dt s;  e^(k+1) = e^n - M1^{-1} j
            const double sum = en + enew;
            const double aux = two ? fma(-0.5 * A.dt, sum, an) : 0.5 * sum;   // a^(k+1); ebar for the next sweep
            if (lane < kConvOut) {
                s_val[o] = aux;
                s_an[o] = an;
            }
            if (own) {
                if (A.mode != CONV_START1) {
                    diff = fabs(enew - eold);
                    mag = fabs(enew);
                }
                A.ek[comp][i] = enew;
                A.aux[comp][i] = aux;
            }
        }
    }
    if (A.mode == CONV_PLAIN) return false;
    __syncthreads();
    // the cells' polynomials of the new field, and the next sweep's moments cleared
    const int ncell = min(kConvOut - K, M - i0);
    if (A.mode != CONV_SOLVE2) {
        const int pad = coef_pad(A.fp32, K);
        for (int q = tid; q < ncell * K; q += nt) {
            const int j = q / K, m = q % K;
            put_coef(T.E, A.fp32, (size_t)(i0 + j), pad, m, e_coef<K>(m, A.dx, [&](int r) { return s_val[K + j - r]; }));
        }
    } else {
        const int pad = coef_pad(A.fp32, K + 1);
        for (int q = tid; q < ncell * (K + 1); q += nt) {
            const int j = q / (K + 1), m = q % (K + 1);
            const size_t row = 2 * (size_t)(i0 + j) + comp;
            const double k = cell_coef<K>(m, [&](int r) { return s_val[K + j - r]; });
            put_coef(T.Kt, A.fp32, row, pad, m, k);
            if (A.fp32) T.L[row * pad + m] = sum_residue(cell_coef<K>(m, [&](int r) { return s_an[K + j - r]; }), k);
        }
    }
    if (A.mode == CONV_START1) return false;
    const int NV = A.subsystem == 1 ? K : K + 1;
    if (zero)
        for (int q = tid; q < ncell * NV; q += nt) zero[(size_t)i0 * NV + q] = 0.0;
    if (zflux && A.subsystem == 1)
        for (int q = tid; q < ncell; q += nt) zflux[i0 + q] = 0;
    if (max_e) {
        if (wid == 0) {
            diff = warp_max_nonneg(diff);
            mag = warp_max_nonneg(mag);
            if (lane == 0) {
                atomic_max_nonneg(max_e, diff);
                atomic_max_nonneg(max_e + 1, mag);
            }
        }
        return false;
    }
    __shared__ int s_last;
    if (wid == 0) {
        diff = warp_max_nonneg(diff);
        mag = warp_max_nonneg(mag);
        if (lane == 0) {
            atomic_max_nonneg(&A.ctrl->emax_bits, diff);
            atomic_max_nonneg(&A.ctrl->emag_bits, mag);
            __threadfence();
            const unsigned int nblk = (unsigned)(((M + kConvOut - K - 1) / (kConvOut - K)) * A.ncomp);
            const unsigned int t = atomicAdd(&A.ctrl->ticket, 1u);
            s_last = (t == nblk - 1) ? 1 : 0;
            if (s_last) decide(A);
        }
    }
    __syncthreads();
    return s_last != 0;
}

// the sweep count of the running loop, for the buffers by parity (replayed by a graph)
__device__ __forceinline__ int conv_iter(const ConvArgs &A)
{
    return A.graph && A.mode != CONV_PLAIN ? *reinterpret_cast<volatile const int *>(&A.ctrl->iter) : 0;
}

// Control block at the start of a fixed-point loop (the error bits and the field
// history counts stay).
__device__ __forceinline__ void ctrl_loop_reset(DevCtrl *ctrl)
{
    ctrl->dmax_bits = 0ull;
    ctrl->emax_bits = 0ull;
    ctrl->emag_bits = 0ull;
    ctrl->dprev_bits = 0x7ff0000000000000ull;
    ctrl->eprev_bits = 0x7ff0000000000000ull;
    ctrl->iter = 0;
    ctrl->converged = 0;
    ctrl->ticket = 0u;
}

// Starting field of a fixed-point iteration.  The fixed point does not depend on
// it, only the number of sweeps to reach it does: e^n extrapolated in time by the
// polynomial through the last q + 1 states, q = min(stored changes, order):
// e^n, e^n + d0, e^n + 2 d0 - d1, e^n + 3 d0 - 3 d1 + d2.
__device__ __forceinline__ double start_field(double e, double *const d[kMaxStartOrder], int i, int q)
{
    switch (q) {
    case 0: return e;
    case 1: return e + d[0][i];
    case 2: return e + (2.0 * d[0][i] - d[1][i]);
    default: return e + (3.0 * (d[0][i] - d[1][i]) + d[2][i]);
    }
}

// ---------------------------------------------------------------------------
// Preparations, cut into independent tasks of a few operations (they are latency): task
// (cell, q) with prep1_tasks<K> or prep2_tasks<K> values of q.
// ---------------------------------------------------------------------------
// Subsystem I: e^(0), ebar^(0) = (e^n + e^(0)) / 2, the cells' polynomials of a^n and
// ebar^(0), cleared moments.
template <int K> constexpr int prep1_tasks = 3 * K + 3;      // A: 2 (K + 1), E: K, the rest: 1

// ebar^(0) at a node (q: stored field changes to use)
__device__ __forceinline__ double ebar0(const RunDesc &R, int g, int q)
{
    const double e = R.ex[g];
    return 0.5 * (e + start_field(e, R.fh.x, g, q));
}

template <int K>
__device__ __forceinline__ void prep1_e(int i, int m, const RunDesc &R, int q)
{
    put_coef(R.T.E, R.fp32, (size_t)i, coef_pad(R.fp32, K), m,
             e_coef<K>(m, R.dx, [&](int r) { return ebar0(R, wrap_once(i - r, R.M), q); }));
}

template <int K>
__device__ __forceinline__ void prep1_task(int i, int t, const RunDesc &R)
{
    const int M = R.M;
    const int q = min(R.ctrl->hist1, R.fh.order1);    // hist1: written only by the commit kernel
    if (t < 2 * (K + 1)) {
        const int c = t / (K + 1), m = t % (K + 1);
        const double *a = c ? R.az : R.ay;
        put_coef(R.T.A, R.fp32, 2 * (size_t)i + c, coef_pad(R.fp32, K + 1), m,
                 cell_coef<K>(m, [&](int r) { return a[wrap_once(i - r, M)]; }));
    } else if (t < 3 * K + 2) {
        prep1_e<K>(i, t - 2 * (K + 1), R, q);
    } else {
        R.ek[i] = start_field(R.ex[i], R.fh.x, i, q);
        R.ebar[i] = ebar0(R, i, q);
        for (int m = 0; m < K; ++m) R.m1[0][(size_t)i * K + m] = R.m1[1][(size_t)i * K + m] = 0.0;
        R.flux[0][i] = R.flux[1][i] = 0;
        if (R.az[i] != 0.0) R.ctrl->zany = 1;
        if (i == 0) ctrl_loop_reset(R.ctrl);
    }
}

// Zeeman source of subsystem II at a node: b_y -= dt hbar (G^T d_z)_j, b_z += dt hbar
// (G^T d_y)_j, d = Lambda_1(X)^T W S from the moments s v^m of the markers (degree K - 1);
// c = dt hbar w / dx.
__device__ __forceinline__ void spin_source_at(int M, int K, double c, const double *mom_y, const double *mom_z,
                                               double *by, double *bz, int j, int comp)
{
    const int jp = j + 1 == M ? 0 : j + 1;
    const double *m = comp ? mom_y : mom_z;
    const double v = c * (node_value(M, K - 1, false, m, j) - node_value(M, K - 1, false, m, jp));
    if (comp) bz[j] += v;
    else by[j] -= v;
}

// Subsystem III (Eq. spin_rodrigue): s <- s + sin(dt|r|)/|r| (r x s)
// + 2 (sin(dt|r|/2)/|r|)^2 r x (r x s), r = (0, Z, -Y), Y = dA_y/dx, Z = dA_z/dx at the marker.
__device__ __forceinline__ void spin_turn(double dt, double Y, double Z, double &sx, double &sy, double &sz)
{
    const double r1 = Z, r2 = -Y, nr = sqrt(r1 * r1 + r2 * r2);
    const double s0 = sx, s1 = sy, s2 = sz;
    const double c1x = r1 * s2 - r2 * s1, c1y = r2 * s0, c1z = -r1 * s0;
    const double c2x = r1 * c1z - r2 * c1y, c2y = r2 * c1x, c2z = -r1 * c1x;
    double f1 = dt, f2 = 0.5 * dt * dt;
    if (nr > 0.0) {
        double sn, cs;
        sincos(0.5 * dt * nr, &sn, &cs);
        const double q = sn / nr;
        f1 = 2.0 * q * cs;
        f2 = 2.0 * q * q;
    }
    sx = s0 + f1 * c1x + f2 * c2x;
    sy = s1 + f1 * c1y + f2 * c2y;
    sz = s2 + f1 * c1z + f2 * c2z;
}

// Subsystem II: b = (M0 - dt^2/4 K) e^n + dt K a^n (banded circulant products), e^(0),
// a^(0) = a^n - dt/2 (e^n + e^(0)), cleared moments, the cells' polynomials.
template <int K> constexpr int prep2_tasks = 2 * (K + 1) + 2;

__device__ __forceinline__ double a0_node(const double *a, const double *e, double *const d[kMaxStartOrder], double dt,
                                          int g, int q)
{
    return fma(-0.5 * dt, e[g] + start_field(e[g], d, g, q), a[g]);
}

// table row entry (cell, component, coefficient); with_a: also the polynomial of a^n
template <int K>
__device__ __forceinline__ void prep2_coef(int i, int c, int m, const RunDesc &R, CoefTables T, int q, bool with_a)
{
    const int M = R.M, pad = coef_pad(R.fp32, K + 1);
    const double *a = c ? R.az : R.ay, *e = c ? R.ez : R.ey;
    double *const *d = c ? R.fh.z : R.fh.y;
    const size_t row = 2 * (size_t)i + c;
    const double k = cell_coef<K>(m, [&](int r) { return a0_node(a, e, d, R.dt, wrap_once(i - r, M), q); });
    put_coef(T.Kt, R.fp32, row, pad, m, k);
    if (with_a || R.fp32) {
        const double n = cell_coef<K>(m, [&](int r) { return a[wrap_once(i - r, M)]; });
        if (with_a) put_coef(T.A, R.fp32, row, pad, m, n);
        if (R.fp32) T.L[row * pad + m] = sum_residue(n, k);
    }
}

// (K c)_i for the stiffness K = G^T M1 G, as M1 on the second differences of c over dx^2:
// neighbouring coefficients of a resolved wave are close, so the differences are exact or
// nearly so, where the rows of K (entries of both signs near 1/dx) lose as many digits as
// K c is smaller than its terms.
template <int K>
__device__ __forceinline__ double stiffness(const double *c, int i, int M, const double *m1, double dx)
{
    double w[2 * K + 1], d[2 * K];
#pragma unroll
    for (int s = 0; s <= 2 * K; ++s) w[s] = c[wrap_once(i + s - K, M)];
#pragma unroll
    for (int s = 0; s < 2 * K; ++s) d[s] = w[s + 1] - w[s];
    double u = m1[0] * (d[K - 1] - d[K]);
#pragma unroll
    for (int s = 1; s < K; ++s) u = fma(m1[s], (d[K - 1 + s] - d[K + s]) + (d[K - 1 - s] - d[K - s]), u);
    return u / (dx * dx);
}

// one component at a node: b = (M0 - dt^2/4 K) e^n + dt K a^n, e^(0), a^(0)
template <int K>
__device__ __forceinline__ void prep2_node(int i, int c, const RunDesc &R, int q)
{
    const int M = R.M;
    const double dt = R.dt;
    const double *a = c ? R.az : R.ay, *e = c ? R.ez : R.ey;
    double *const *d = c ? R.fh.z : R.fh.y;
    double v = R.rowM0[0] * e[i];
#pragma unroll
    for (int s = 1; s <= K; ++s) v = fma(R.rowM0[s], e[wrap_once(i + s, M)] + e[wrap_once(i - s, M)], v);
    const double ke = stiffness<K>(e, i, M, R.rowM1, R.dx), ka = stiffness<K>(a, i, M, R.rowM1, R.dx);
    (c ? R.bz : R.by)[i] = fma(dt, fma(-0.25 * dt, ke, ka), v);
    (c ? R.ekz : R.eky)[i] = start_field(e[i], d, i, q);
    (c ? R.akz : R.aky)[i] = a0_node(a, e, d, dt, i, q);
}

template <int K>
__device__ __forceinline__ void prep2_task(int i, int t, const RunDesc &R)
{
    const int q = min(R.ctrl->hist2, R.fh.order2);    // hist2: written only by the commit kernel
    if (t < 2 * (K + 1)) {
        prep2_coef<K>(i, t / (K + 1), t % (K + 1), R, R.T, q, true);
    } else {
        const int c = t - 2 * (K + 1);
        prep2_node<K>(i, c, R, q);
        for (int m = 0; m <= K; ++m)
            for (int b = 0; b < 2; ++b) (c ? R.mz : R.my)[b][(size_t)i * (K + 1) + m] = 0.0;
        if (c && (R.az[i] != 0.0 || R.ez[i] != 0.0)) R.ctrl->zany = 1;
        if (i == 0 && c == 0) ctrl_loop_reset(R.ctrl);
    }
}

// e^{n+1} = e^(k) replaces e^n; its change enters the history (d[2] = d[1],
// d[1] = d[0], d[0] = e^{n+1} - e^n), as deep as the extrapolation order needs.
__device__ __forceinline__ void commit_field(int i, const double *ek, double *e, double *const d[kMaxStartOrder],
                                             int order)
{
    const double v = ek[i];
    for (int m = order - 1; m > 0; --m) d[m][i] = d[m - 1][i];
    if (order > 0) d[0][i] = v - e[i];
    e[i] = v;
}

// End of a substep: I: e_x = e^(k); II: e_perp = e^(k), a_perp = a^(k).  Thread
// 0 counts the stored changes (up to kMaxStartOrder) for the next preparation.
// last: index of the last sweep of subsystem I's loop.
__device__ __forceinline__ void commit_at(int i, const RunDesc &R, int which, int last)
{
    if (i < R.M) {
        if (which == 1) {
            commit_field(i, R.ek, R.ex, R.fh.x, R.fh.order1);
            // the end points of the last sweep are the next step's start points
            const double *ends = R.m1[last & 1];
            for (int m = 0; m < R.K; ++m) R.m0[(size_t)i * R.K + m] = ends[(size_t)i * R.K + m];
        } else {
            commit_field(i, R.eky, R.ey, R.fh.y, R.fh.order2);
            commit_field(i, R.ekz, R.ez, R.fh.z, R.fh.order2);
            R.ay[i] = R.aky[i];
            R.az[i] = R.akz[i];
        }
    }
    if (i == 0) {
        int *h = which == 1 ? &R.ctrl->hist1 : &R.ctrl->hist2;
        if (*h < kMaxStartOrder) *h += 1;
    }
}

}  // namespace pic
