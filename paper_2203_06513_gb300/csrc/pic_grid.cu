// pic_grid.cu -- grid-side kernels of libpic (double precision) and the host
// algebra of the periodic spline matrices.
//
// Every matrix of the method is a symmetric circulant on M nodes (Sec. 3.1):
//   M0 (degree k), M1 (degree k-1), K = G^T M1 G, P = M0 + dt^2/4 K.
// Solves apply the exact inverse as a circulant convolution: the inverse of a
// banded SPD circulant has a first row that decays geometrically, so it is
// truncated where its entries fall below 1e-17 of the largest (or kept whole).
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "pic_internal.h"
#include "pic_poly.cuh"

namespace pic {

// ---------------------------------------------------------------------------
// Host: exact mass-matrix bands.  (M_d)_{0,r} = int N^d(s) N^d(s - r) ds * dx,
// the autocorrelation of the cardinal B-spline, equals dx N^{2d+1}(d + 1 + r).
// N^n is evaluated from the truncated-power form
//   N^n(s) = 1/n! sum_{i=0}^{n+1} (-1)^i C(n+1, i) (s - i)_+^n,
// exact in rational arithmetic; at the integer arguments used here every term
// is an integer divided by n!, so double evaluation is exact for n <= 11.
// ---------------------------------------------------------------------------
static double cardinal_tp(int n, double s)
{
    double acc = 0.0, binom = 1.0, fact = 1.0;
    for (int i = 1; i <= n; ++i) fact *= i;
    for (int i = 0; i <= n + 1; ++i) {
        const double u = s - i;
        if (u > 0.0) acc += ((i & 1) ? -1.0 : 1.0) * binom * std::pow(u, n);
        binom = binom * (n + 1 - i) / (i + 1);
    }
    return acc / fact;
}

void mass_band(int d, double dx, double *band)
{
    for (int r = 0; r <= d; ++r) band[r] = dx * cardinal_tp(2 * d + 1, (double)(d + 1 + r));
}

// First row g of the inverse of the symmetric circulant with band c_0..c_bw:
// eigenvalues lambda_m = c_0 + 2 sum_d c_d cos(2 pi m d / M), g_d = 1/M sum_m
// cos(2 pi m d / M) / lambda_m, with one step of iterative refinement.  The
// cosine table is made exactly symmetric (cs[M - j] = cs[j]), so both transforms
// are symmetric in their output index bit for bit and only the first half is
// summed; indices m q mod M advance by addition.
static void inverse_taps_compute(const double *band, int bw, int M, double cut, double *g, int *d_start,
                                 int *ntap, double *taps)
{
    const double twopi = 6.283185307179586476925286766559;
    std::vector<double> cs(M), lam(M), r(M), corr(M);
    for (int m = 0; m <= M / 2; ++m) cs[m] = std::cos(twopi * (double)m / (double)M);
    for (int m = M / 2 + 1; m < M; ++m) cs[m] = cs[M - m];
    for (int m = 0; m < M; ++m) {
        double l = band[0];
        for (int d = 1; d <= bw; ++d) l += 2.0 * band[d] * cs[(long long)m * d % M];
        lam[m] = 1.0 / l;
    }
    // y_k = sum_j v_j cs[k j mod M] for k = 0 .. M/2, mirrored; four interleaved
    // compensated partial sums (independent chains), added at the end
    auto cos_transform = [&](const std::vector<double> &v, std::vector<double> &y) {
        for (int k = 0; k <= M / 2; ++k) {
            double s[4] = {0.0, 0.0, 0.0, 0.0}, comp[4] = {0.0, 0.0, 0.0, 0.0};
            int idx = 0;
            for (int j = 0; j < M; ++j) {
                const int l = j & 3;
                const double t = v[j] * cs[idx] - comp[l];
                const double tt = s[l] + t;
                comp[l] = (tt - s[l]) - t;
                s[l] = tt;
                idx += k;
                if (idx >= M) idx -= M;
            }
            y[k] = ((s[0] + s[1]) + (s[2] + s[3])) - ((comp[0] + comp[1]) + (comp[2] + comp[3]));
        }
        for (int k = M / 2 + 1; k < M; ++k) y[k] = y[M - k];
    };
    auto apply_inv = [&](const std::vector<double> &rhs_even, std::vector<double> &out) {
        // rhs is symmetric (even) so its DFT is real: R_m = sum_q rhs_q cos(2 pi m q / M)
        std::vector<double> R(M);
        cos_transform(rhs_even, R);
        for (int m = 0; m < M; ++m) R[m] *= lam[m];
        cos_transform(R, out);
        for (int d = 0; d < M; ++d) out[d] /= (double)M;
    };
    std::vector<double> e0(M, 0.0), gv(M);
    e0[0] = 1.0;
    apply_inv(e0, gv);
    // refinement: r = e0 - A g, g += A^{-1} r
    for (int i = 0; i < M; ++i) {
        double s = band[0] * gv[i];
        for (int d = 1; d <= bw; ++d) s += band[d] * (gv[(i + d) % M] + gv[(i - d + M) % M]);
        r[i] = e0[i] - s;
    }
    apply_inv(r, corr);
    for (int i = 0; i < M; ++i) gv[i] += corr[i];
    for (int i = 0; i < M; ++i) g[i] = gv[i];
    double gmax = 0.0;
    for (int i = 0; i < M; ++i) gmax = std::fmax(gmax, std::fabs(gv[i]));
    int T = 0;
    for (int d = 1; d <= M / 2; ++d)
        if (std::fabs(gv[d]) > cut * gmax) T = d;
    if (2 * T + 1 <= M && !(M % 2 == 0 && T == M / 2)) {
        *d_start = -T;
        *ntap = 2 * T + 1;
        for (int n = 0; n < 2 * T + 1; ++n) taps[n] = gv[(n - T + M) % M];
    } else {  // whole circulant: offsets -(M/2 - 1) .. M/2 (M entries)
        const int lo = -(M / 2 - 1 + (M % 2));
        *d_start = lo;
        *ntap = M;
        for (int n = 0; n < M; ++n) taps[n] = gv[((lo + n) % M + M) % M];
    }
}

// The taps of one (band, M, cut) are the same for every handle that asks: a
// process-wide table of the recent ones spares repeated set-ups the O(M^2) work.
void inverse_taps(const double *band, int bw, int M, double cut, double *g, int *d_start, int *ntap,
                  double *taps)
{
    struct Entry {
        std::vector<double> key, g, taps;
        int d_start, ntap;
    };
    static std::mutex mu;
    static std::vector<Entry> table;
    std::vector<double> key(band, band + bw + 1);
    key.push_back((double)M);
    key.push_back(cut);
    {
        std::lock_guard<std::mutex> lock(mu);
        for (const Entry &e : table)
            if (e.key == key) {
                std::copy(e.g.begin(), e.g.end(), g);
                std::copy(e.taps.begin(), e.taps.end(), taps);
                *d_start = e.d_start;
                *ntap = e.ntap;
                return;
            }
    }
    inverse_taps_compute(band, bw, M, cut, g, d_start, ntap, taps);
    std::lock_guard<std::mutex> lock(mu);
    if (table.size() >= 64) table.clear();
    table.push_back(Entry{key, std::vector<double>(g, g + M), std::vector<double>(taps, taps + *ntap), *d_start,
                          *ntap});
}

// ---------------------------------------------------------------------------
// Convergence decision, made by the last block of a solve kernel.
// FP64 form (Sec. 5, tolerance tol): max |x^(k+1) - x^(k)| <= tol (length) and
// max |e^(k+1) - e^(k)| <= tol.  FP32 form: position increments at the float
// resolution of the offset (dtol, relative to max(1, |delta|)) and field
// increments below tol or no longer shrinking (stagnation at float noise).
// ---------------------------------------------------------------------------
__device__ void decide(const ConvArgs &A)
{
    DevCtrl *c = A.ctrl;
    __threadfence();
    if (A.count) *A.count += 1;
    const double d = (A.subsystem == 1) ? bits_to_double(c->dmax_bits) : 0.0;
    const double e = bits_to_double(c->emax_bits);
    const double ep = bits_to_double(c->eprev_bits);
    c->iter += 1;
    bool ok;
    if (!A.fp32) {
        ok = (d * A.dx <= A.tol) && (e <= A.tol);
    } else {
        // Float iterates stop improving at rounding noise, so increments alone never
        // reach a tight tolerance.  Estimate the remaining error of the new iterate
        // from the increment v_k and the observed contraction r = v_k / v_{k-1}
        // (geometric tail v_k r / (1 - r), r capped at 0.9), and stop when both the
        // position and field estimates are below tolerance, or when both increments
        // have stopped shrinking at noise level.
        const double dp = bits_to_double(c->dprev_bits);
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
        const double emag = bits_to_double(c->emag_bits);
        const bool dok = (A.subsystem == 1) ? (est(d, dp) <= A.dtol) : true;
        const bool eok = (A.subsystem == 1) ? (e <= fmax(A.tol, A.erel * emag)) : (est(e, ep) <= A.tol);
        const bool dstag = (A.subsystem == 1) ? (d >= 0.5 * dp && d <= 1e-4) : true;
        const bool estag = e >= 0.5 * ep && e <= 1e-8;
        ok = (dok && eok) || (c->iter >= 3 && dstag && estag);
    }
    bool stop = ok;
    if (!ok && c->iter >= A.max_iter) {
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
__constant__ SplineTab c_spline = make_spline_tab();

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
__constant__ SplineTab c_cumulative = make_cumulative_tab();

// Stores coefficient m of row `row` (pad numbers a row) in the form's type.
__device__ __forceinline__ void put_coef(void *tab, int fp32, size_t row, int pad, int m, double v)
{
    if (fp32) static_cast<float *>(tab)[row * pad + m] = (float)v;
    else static_cast<double *>(tab)[row * pad + m] = v;
}

// Coefficient m of the degree-D polynomial in the cell whose node r steps down has value at(r).
template <class At>
__device__ __forceinline__ double cell_coef(int D, int m, At &&at)
{
    double s = 0.0;
    for (int r = 0; r <= D; ++r) s = fma(c_spline.b[D][r][m], at(r), s);
    return s;
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

// Path current at node j over w dx (pic_poly.cuh): the polynomials of C_j on the change of
// the moments in the cells j .. j + K - 1, and the crossings of the knot j + K.
__device__ __forceinline__ double path_node_value(int M, int K, const double *mom, const double *mom0,
                                                  const int *flux, int j)
{
    double s0 = 0.0, s1 = 0.0;
    int c = j, f = flux[j];
    for (int r = 0; r < K; ++r) {
        const int cn = c + 1 == M ? 0 : c + 1;
        const int fn = flux[cn];
        s0 = fma(c_cumulative.b[K][r][0], (double)(f - fn), s0);
        for (int m = 1; m <= K; ++m) {
            const size_t q = (size_t)c * K + m - 1;
            s1 = fma(c_cumulative.b[K][r][m], mom[q] - mom0[q], s1);
        }
        c = cn;
        f = fn;
    }
    return (s0 + s1) + (double)f;
}

// The residue of a^n + a^(k) after both coefficients were rounded to float.
__device__ __forceinline__ float sum_residue(double n, double k)
{
    return (float)((n - (double)(float)n) + (k - (double)(float)k));
}

// y_i = sum_n taps[n] in[(i - (d_start + n)) mod M] for the kConvOut nodes
// i0 - K .. i0 - K + kConvOut - 1 of block bx, i0 = bx (kConvOut - K): the block owns the
// last kConvOut - K of them and recomputes the K below, which the polynomials of
// its cells need.  One warp computes a quarter of the taps for all nodes (lane =
// node): with a few dozen nodes a block the solve spreads over the SMs instead of
// waiting on one SM's FP64 pipe, and only the block's part of the deposit is staged
// (M = 2048, cubic: 35 us with one thread a node and the whole row staged twice by every
// block, 18 us so; both with cold caches).
// Returns true in the one block that finished the run's solve last (after the
// convergence decision, in the solve modes).
constexpr int kConvOut = 32, kConvThreads = 128;

inline size_t conv_smem(int ntap)
{
    const int nq = kConvOut + ntap - 1;
    return ((size_t)nq + ntap + 4 * kConvOut + 2 * kConvOut) * sizeof(double);
}
inline int conv_blocks(int M, int K) { return (M + kConvOut - K - 1) / (kConvOut - K); }

__device__ bool conv_block(const ConvArgs &A, int bx, int comp, double *sm)
{
    const int M = A.M, K = A.K, TB = kConvOut - K, i0 = bx * TB;
    const int NV = A.subsystem == 1 ? K : K + 1;       // moments a cell
    const int nq = kConvOut + A.ntap - 1;
    double *s_in = sm, *s_tap = s_in + nq, *s_part = s_tap + A.ntap;
    double *s_val = s_part + 4 * kConvOut, *s_an = s_val + kConvOut;
    const double *mom = A.mom[comp];
    double *zero = A.zero[comp];
    const int *flux = A.flux;
    int *zflux = A.zflux;
    if (A.graph && A.mode != CONV_PLAIN) {   // replayed by a graph: buffers by sweep parity
        const int it = *reinterpret_cast<volatile const int *>(&A.ctrl->iter);
        mom = A.pair[comp][it & 1];
        zero = A.pair[comp][(it + 1) & 1];
        flux = A.fpair[it & 1];
        zflux = A.fpair[(it + 1) & 1];
    }
    // s_in[q]: node (g0 + q) mod M
    const int g0 = wrap_cell(i0 - K - (A.d_start + A.ntap - 1), M);
    for (int n = threadIdx.x; n < A.ntap; n += kConvThreads) s_tap[n] = A.taps[n];
    if (mom) {
        for (int q = threadIdx.x; q < nq; q += kConvThreads) {
            const int g = (g0 + q) % M;
            double s = A.scale * (A.subsystem == 1 ? path_node_value(M, K, mom, A.mom0, flux, g)
                                                   : node_value(M, K, false, mom, g));
            if (A.mode == CONV_SOLVE2) s = fma(A.dt, s, A.b[comp][g]);
            s_in[q] = s;
        }
    } else {
        for (int q = threadIdx.x; q < nq; q += kConvThreads) {
            const int g = (g0 + q) % M;
            const double s = A.in[comp][g];
            s_in[q] = A.mode == CONV_SOLVE2 ? fma(A.dt, s, A.b[comp][g]) : s;
        }
    }
    __syncthreads();
    const int o = threadIdx.x & 31, wid = threadIdx.x >> 5;
    {
        const int per = (A.ntap + 3) >> 2, n0 = wid * per, n1 = min(A.ntap, n0 + per);
        const double *base = s_in + o + A.ntap - 1;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int n = n0;
        for (; n + 3 < n1; n += 4) {
            a0 = fma(s_tap[n], base[-n], a0);
            a1 = fma(s_tap[n + 1], base[-n - 1], a1);
            a2 = fma(s_tap[n + 2], base[-n - 2], a2);
            a3 = fma(s_tap[n + 3], base[-n - 3], a3);
        }
        for (; n < n1; ++n) a0 = fma(s_tap[n], base[-n], a0);
        s_part[wid * kConvOut + o] = (a0 + a1) + (a2 + a3);
    }
    __syncthreads();
    double diff = 0.0, mag = 0.0;
    if (wid == 0) {
        const double y = (s_part[o] + s_part[kConvOut + o]) + (s_part[2 * kConvOut + o] + s_part[3 * kConvOut + o]);
        const int i = i0 - K + o;
        const bool own = o >= K && i < M;
        const int iw = wrap_cell(i, M);
        if (A.mode == CONV_PLAIN) {
            if (own) A.out[comp][i] = y;
        } else if (A.mode != CONV_SOLVE2) {              // START1, SOLVE1
            const double en = A.en[0][iw];
            const double enew = en - y;                  // e^(k+1) = e^n - M1^{-1} j
            const double eb = 0.5 * (en + enew);         // ebar for the next sweep
            s_val[o] = eb;
            if (own) {
                if (A.mode == CONV_SOLVE1) {
                    diff = fabs(enew - A.ek[0][i]);
                    mag = fabs(enew);
                }
                A.ek[0][i] = enew;
                A.aux[0][i] = eb;
            }
        } else {                                         // P e^(k+1) = b + dt s
            const double en = A.en[comp][iw], an = A.an[comp][iw];
            const double enew = y;
            const double ak = an - 0.5 * A.dt * (en + enew);   // a^(k+1)
            s_val[o] = ak;
            s_an[o] = an;
            if (own) {
                diff = fabs(enew - A.ek[comp][i]);
                mag = fabs(enew);
                A.ek[comp][i] = enew;
                A.aux[comp][i] = ak;
            }
        }
    }
    if (A.mode == CONV_PLAIN) return false;
    __syncthreads();
    // the cells' polynomials of the new field, and the next sweep's moments cleared
    const int ncell = min(TB, M - i0);
    if (A.mode != CONV_SOLVE2) {
        const int pad = coef_pad(A.fp32, K);
        for (int q = threadIdx.x; q < ncell * K; q += kConvThreads) {
            const int j = q / K, m = q % K;
            const double v = cell_coef(K - 1, m, [&](int r) { return s_val[K + j - r]; });
            put_coef(A.T.E, A.fp32, (size_t)(i0 + j), pad, m, v * A.dx / (double)(m + 1));
        }
    } else {
        const int pad = coef_pad(A.fp32, K + 1);
        for (int q = threadIdx.x; q < ncell * (K + 1); q += kConvThreads) {
            const int j = q / (K + 1), m = q % (K + 1);
            const size_t row = 2 * (size_t)(i0 + j) + comp;
            const double k = cell_coef(K, m, [&](int r) { return s_val[K + j - r]; });
            put_coef(A.T.Kt, A.fp32, row, pad, m, k);
            if (A.fp32) {
                const double n = cell_coef(K, m, [&](int r) { return s_an[K + j - r]; });
                A.T.L[row * pad + m] = sum_residue(n, k);
            }
        }
    }
    if (A.mode == CONV_START1) return false;
    if (zero)
        for (int q = threadIdx.x; q < ncell * NV; q += kConvThreads) zero[(size_t)i0 * NV + q] = 0.0;
    if (zflux && A.subsystem == 1)
        for (int q = threadIdx.x; q < ncell; q += kConvThreads) zflux[i0 + q] = 0;
    __shared__ int s_last;
    if (wid == 0) {
        diff = warp_max(diff);
        mag = warp_max(mag);
        if (o == 0) {
            atomic_max_nonneg(&A.ctrl->emax_bits, diff);
            atomic_max_nonneg(&A.ctrl->emag_bits, mag);
            __threadfence();
            const unsigned int nblk = (unsigned)(((M + TB - 1) / TB) * A.ncomp);
            const unsigned int t = atomicAdd(&A.ctrl->ticket, 1u);
            s_last = (t == nblk - 1) ? 1 : 0;
            if (s_last) decide(A);
        }
    }
    __syncthreads();
    return s_last != 0;
}

__global__ void __launch_bounds__(kConvThreads) k_conv(ConvArgs A)
{
    extern __shared__ __align__(16) double s_conv[];
    conv_block(A, blockIdx.x, blockIdx.y, s_conv);
}

// Batched solves of an ensemble: block (bx, run, comp).  Runs that are not in
// the current sweep (converged, or stopped by an error) are skipped.  After a
// run's decision, the last run to decide in this sweep records whether any run
// goes on, and sets the loop's conditional handle (graph mode).
__global__ void __launch_bounds__(kConvThreads) k_conv_ens(const ConvArgs *runs, EnsQueue *Q, int *sweeps,
                                                           unsigned long long cond)
{
    extern __shared__ __align__(16) double s_conv[];
    const int r = blockIdx.y, comp = blockIdx.z;
    const ConvArgs &A = runs[r];
    if (A.mode != CONV_PLAIN && !Q->active[r]) return;
    if (comp >= A.ncomp || (int)blockIdx.x * (kConvOut - A.K) >= A.M) return;
    const bool last = conv_block(A, blockIdx.x, comp, s_conv);
    if (!last || threadIdx.x != 0) return;
    atomicAdd(&sweeps[2 * r + A.subsystem - 1], 1);
    if (!A.ctrl->converged) atomicAdd(&Q->n_continue, 1);
    __threadfence();
    const int t = atomicAdd(&Q->n_decided, 1);
    if (t == Q->nactive - 1) {
        __threadfence();
        const int go = atomicAdd(&Q->n_continue, 0) > 0 ? 1 : 0;
        Q->go = go;
        Q->loops[A.subsystem - 1] += 1;
        if (cond) cudaGraphSetConditional((cudaGraphConditionalHandle)cond, (unsigned)go);
    }
}

// Raises a solve kernel's dynamic shared-memory limit (never lowers it).  Inverse rows
// that decay slowly (large dt/dx in subsystem II) may keep as many taps as nodes.
static int conv_optin(const void *fn, size_t smem, size_t &opted)
{
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    if (smem > 48 * 1024 && smem > opted) {
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return 1;
        opted = smem;
    }
    return 0;
}

static size_t g_conv_ens_opted = 0;

// raise the shared-memory limit of k_conv_ens before any capture of it
int conv_ens_optin(int ntap_max)
{
    return conv_optin((const void *)k_conv_ens, conv_smem(ntap_max), g_conv_ens_opted);
}

int launch_conv_ens(const ConvArgs *runs, int nruns, int Mmax, int K, int ncomp, int ntap_max, EnsQueue *Q,
                    int *sweeps, unsigned long long cond, cudaStream_t s)
{
    const size_t smem = conv_smem(ntap_max);
    if (smem > 48 * 1024 && smem > g_conv_ens_opted) return 1;   // conv_ens_optin first
    dim3 grid(conv_blocks(Mmax, K), nruns, ncomp);
    k_conv_ens<<<grid, kConvThreads, smem, s>>>(runs, Q, sweeps, cond);
    return 0;
}

int launch_conv(const ConvArgs &a, cudaStream_t s)
{
    const size_t smem = conv_smem(a.ntap);
    static size_t opted = 0;   // largest dynamic shared memory opted in so far
    if (conv_optin((const void *)k_conv, smem, opted)) return 1;
    k_conv<<<dim3(conv_blocks(a.M, a.K), a.ncomp), kConvThreads, smem, s>>>(a);
    return 0;
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
// Subsystem I preparation: e^(0), ebar^(0) = (e^n + e^(0)) / 2, the cells' polynomials
// of a^n and ebar^(0), cleared moments, the control block reset for the loop.
// ---------------------------------------------------------------------------
// both rows of the polynomials of (cy, cz) in cell i, and whether cz has a non-zero
__device__ __forceinline__ void a_rows(int i, int M, int K, int fp32, const double *cy, const double *cz, void *tab)
{
    const int pad = coef_pad(fp32, K + 1);
    for (int m = 0; m <= K; ++m) {
        put_coef(tab, fp32, 2 * (size_t)i, pad, m, cell_coef(K, m, [&](int r) { return cy[wrap_cell(i - r, M)]; }));
        put_coef(tab, fp32, 2 * (size_t)i + 1, pad, m, cell_coef(K, m, [&](int r) { return cz[wrap_cell(i - r, M)]; }));
    }
}

__device__ __forceinline__ void prep1_at(int i, const RunDesc &R)
{
    const int M = R.M, K = R.K;
    const int q = min(R.ctrl->hist1, R.fh.order1);    // hist1: written only by the commit kernel
    if (i < M) {
        auto ebar = [&](int g) { return 0.5 * (R.ex[g] + start_field(R.ex[g], R.fh.x, g, q)); };
        R.ek[i] = start_field(R.ex[i], R.fh.x, i, q);
        R.ebar[i] = ebar(i);
        a_rows(i, M, K, R.fp32, R.ay, R.az, R.T.A);
        const int pad = coef_pad(R.fp32, K);
        for (int m = 0; m < K; ++m) {
            const double v = cell_coef(K - 1, m, [&](int r) { return ebar(wrap_cell(i - r, M)); });
            put_coef(R.T.E, R.fp32, (size_t)i, pad, m, v * R.dx / (double)(m + 1));
            R.m1[0][(size_t)i * K + m] = 0.0;
            R.m1[1][(size_t)i * K + m] = 0.0;
        }
        R.flux[0][i] = 0;
        R.flux[1][i] = 0;
        if (R.az[i] != 0.0) R.ctrl->zany = 1;
    }
    if (i == 0) ctrl_loop_reset(R.ctrl);
}

__global__ void k_prep1(RunDesc R) { prep1_at(blockIdx.x * blockDim.x + threadIdx.x, R); }

__global__ void k_prep1_ens(const RunDesc *runs)
{
    prep1_at(blockIdx.x * blockDim.x + threadIdx.x, runs[blockIdx.y]);
}

int launch_prep1_ens(const RunDesc *R, int nruns, int Mmax, cudaStream_t s)
{
    k_prep1_ens<<<dim3((Mmax + 63) / 64, nruns), 64, 0, s>>>(R);
    return 0;
}

int launch_prep1(const RunDesc &R, cudaStream_t s)
{
    k_prep1<<<(R.M + 63) / 64, 64, 0, s>>>(R);
    return 0;
}

// ---------------------------------------------------------------------------
// Subsystem II preparation: b = (M0 - dt^2/4 K) e^n + dt K a^n (banded
// circulant products), e^(0), a^(0) = a^n - dt/2 (e^n + e^(0)), cleared
// moments, the cells' polynomials, the control block reset for the loop.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void prep2_at(int i, const RunDesc &R)
{
    const int M = R.M, K = R.K;
    const double dt = R.dt;
    const int q = min(R.ctrl->hist2, R.fh.order2);    // hist2: written only by the commit kernel
    if (i < M) {
        const double *ey = R.ey, *ez = R.ez, *ay = R.ay, *az = R.az;
        auto a0 = [&](const double *a, const double *e, double *const d[kMaxStartOrder], int g) {
            return a[g] - 0.5 * dt * (e[g] + start_field(e[g], d, g, q));
        };
        const double ey0 = start_field(ey[i], R.fh.y, i, q);
        const double ez0 = start_field(ez[i], R.fh.z, i, q);
        const double ay0 = a0(ay, ey, R.fh.y, i), az0 = a0(az, ez, R.fh.z, i);
        {
            double kn[2][kMaxDegree + 1], kk[2][kMaxDegree + 1];     // nodes i, i - 1, .. i - K
            for (int r = 0; r <= K; ++r) {
                const int g = wrap_cell(i - r, M);
                kn[0][r] = ay[g];
                kn[1][r] = az[g];
                kk[0][r] = a0(ay, ey, R.fh.y, g);
                kk[1][r] = a0(az, ez, R.fh.z, g);
            }
            const int pad = coef_pad(R.fp32, K + 1);
            for (int c = 0; c < 2; ++c) {
                const size_t row = 2 * (size_t)i + c;
                for (int m = 0; m <= K; ++m) {
                    const double n = cell_coef(K, m, [&](int r) { return kn[c][r]; });
                    const double k = cell_coef(K, m, [&](int r) { return kk[c][r]; });
                    put_coef(R.T.A, R.fp32, row, pad, m, n);
                    put_coef(R.T.Kt, R.fp32, row, pad, m, k);
                    if (R.fp32) R.T.L[row * pad + m] = sum_residue(n, k);
                }
            }
        }
        double vy = R.rowPm[0] * ey[i] + dt * R.rowK[0] * ay[i];
        double vz = R.rowPm[0] * ez[i] + dt * R.rowK[0] * az[i];
        for (int d = 1; d <= K; ++d) {
            const int ip = (i + d) % M, im = (i - d + M) % M;
            vy += R.rowPm[d] * (ey[ip] + ey[im]) + dt * R.rowK[d] * (ay[ip] + ay[im]);
            vz += R.rowPm[d] * (ez[ip] + ez[im]) + dt * R.rowK[d] * (az[ip] + az[im]);
        }
        R.by[i] = vy;
        R.bz[i] = vz;
        R.eky[i] = ey0;
        R.ekz[i] = ez0;
        R.aky[i] = ay0;
        R.akz[i] = az0;
        for (int m = 0; m <= K; ++m)
            for (int b = 0; b < 2; ++b) {
                R.my[b][(size_t)i * (K + 1) + m] = 0.0;
                R.mz[b][(size_t)i * (K + 1) + m] = 0.0;
            }
        if (az[i] != 0.0 || ez[i] != 0.0) R.ctrl->zany = 1;
    }
    if (i == 0) ctrl_loop_reset(R.ctrl);
}

__global__ void k_prep2(RunDesc R) { prep2_at(blockIdx.x * blockDim.x + threadIdx.x, R); }

__global__ void k_prep2_ens(const RunDesc *runs)
{
    prep2_at(blockIdx.x * blockDim.x + threadIdx.x, runs[blockIdx.y]);
}

int launch_prep2_ens(const RunDesc *R, int nruns, int Mmax, cudaStream_t s)
{
    k_prep2_ens<<<dim3((Mmax + 63) / 64, nruns), 64, 0, s>>>(R);
    return 0;
}

int launch_prep2(const RunDesc &R, cudaStream_t s)
{
    k_prep2<<<(R.M + 63) / 64, 64, 0, s>>>(R);
    return 0;
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
__device__ __forceinline__ void commit_at(int i, const RunDesc &R, int which)
{
    if (i < R.M) {
        if (which == 1) {
            commit_field(i, R.ek, R.ex, R.fh.x, R.fh.order1);
            // the end points of the last sweep are the next step's start points
            const double *last = R.m1[(R.ctrl->iter - 1) & 1];
            for (int m = 0; m < R.K; ++m) R.m0[(size_t)i * R.K + m] = last[(size_t)i * R.K + m];
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

__global__ void k_commit(RunDesc R, int which) { commit_at(blockIdx.x * blockDim.x + threadIdx.x, R, which); }

int launch_commit(const RunDesc &R, int which, cudaStream_t s)
{
    k_commit<<<(R.M + 255) / 256, 256, 0, s>>>(R, which);
    return 0;
}

// The same for every run of an ensemble.  Runs stopped by an error keep their
// fields and history.
__global__ void k_commit_ens(const RunDesc *runs, int which)
{
    const RunDesc &R = runs[blockIdx.y];
    if (R.ctrl->status & (STATUS_NUMERIC | STATUS_TIMEOUT)) return;
    commit_at(blockIdx.x * blockDim.x + threadIdx.x, R, which);
}

int launch_commit_ens(const RunDesc *R, int nruns, int Mmax, int which, cudaStream_t s)
{
    k_commit_ens<<<dim3((Mmax + 255) / 256, nruns), 256, 0, s>>>(R, which);
    return 0;
}

// Work list of the next batched sweep: the runs still iterating (not converged,
// not stopped by an error), each cut into items of item_markers markers;
// item_start is the exclusive prefix sum of the items per run.
__global__ void __launch_bounds__(1024) k_ens_plan(EnsQueue *Q, const EnsRun *runs, int nruns,
                                                   unsigned long long cond)
{
    __shared__ int s_scan[1024];
    __shared__ int s_nact[32];
    const int r = threadIdx.x;
    int items = 0, act = 0;
    if (r < nruns) {
        const DevCtrl *c = runs[r].ctrl;
        act = (!c->converged && !(c->status & (STATUS_NUMERIC | STATUS_TIMEOUT))) ? 1 : 0;
        const long long im = Q->item_markers;
        items = act ? (int)((runs[r].np + im - 1) / im) : 0;
        Q->active[r] = act;
    }
    // inclusive scan (Hillis-Steele) over the block
    s_scan[r] = items;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const int v = r >= o ? s_scan[r - o] : 0;
        __syncthreads();
        s_scan[r] += v;
        __syncthreads();
    }
    if (r < nruns) Q->item_start[r + 1] = s_scan[r];
    const unsigned b = __ballot_sync(0xffffffffu, act != 0);
    if ((r & 31) == 0) s_nact[r >> 5] = __popc(b);
    __syncthreads();
    if (r == 0) {
        int n = 0;
        for (int w = 0; w < 32; ++w) n += s_nact[w];
        Q->item_start[0] = 0;
        Q->nitems = s_scan[nruns - 1];
        Q->nactive = n;
        Q->next = 0;
        Q->n_decided = 0;
        Q->n_continue = 0;
        Q->go = 0;
        // no run left (every run stopped by an error): no solve will decide, so the
        // loop is ended here
        if (n == 0 && cond) cudaGraphSetConditional((cudaGraphConditionalHandle)cond, 0u);
    }
}

__global__ void k_ens_status(const EnsRun *runs, int nruns, int *status)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < nruns) status[r] = runs[r].ctrl->status;
}

int launch_ens_status(const EnsRun *runs, int nruns, int *status, cudaStream_t s)
{
    k_ens_status<<<(nruns + 255) / 256, 256, 0, s>>>(runs, nruns, status);
    return 0;
}

int launch_ens_plan(EnsQueue *Q, const EnsRun *runs, int nruns, unsigned long long cond, cudaStream_t s)
{
    if (nruns < 1 || nruns > kEnsMaxRuns) return 1;
    k_ens_plan<<<1, 1024, 0, s>>>(Q, runs, nruns, cond);
    return 0;
}

__global__ void k_moments_to_nodes(int M, int D, bool path, double scale, const double *mom, double *out)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    out[j] = scale * node_value(M, D, path, mom, j);
}

int launch_moments_to_nodes(int M, int D, bool path, double scale, const double *mom, double *out, cudaStream_t s)
{
    k_moments_to_nodes<<<(M + 63) / 64, 64, 0, s>>>(M, D, path, scale, mom, out);
    return 0;
}

__global__ void k_path_nodes(int M, int K, double scale, const double *mom, const double *mom0, const int *flux,
                             double *out)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < M) out[j] = scale * path_node_value(M, K, mom, mom0, flux, j);
}

int launch_path_nodes(int M, int K, double scale, const double *mom, const double *mom0, const int *flux, double *out,
                      cudaStream_t s)
{
    k_path_nodes<<<(M + 63) / 64, 64, 0, s>>>(M, K, scale, mom, mom0, flux, out);
    return 0;
}

__global__ void k_start_moments(int M, int K, const double *charge, double *mom0)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M * K) return;
    mom0[i] = charge[(size_t)(i / K) * (K + 1) + i % K + 1];
}

int launch_start_moments(int M, int K, const double *charge, double *mom0, cudaStream_t s)
{
    k_start_moments<<<(M * K + 255) / 256, 256, 0, s>>>(M, K, charge, mom0);
    return 0;
}

__global__ void k_cell_coefs(int M, int D, bool path, const double *c, double *tab)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    const int pad = coef_pad(0, D + 1);
    for (int m = 0; m <= D; ++m) {
        const double v = cell_coef(D, m, [&](int r) { return c[wrap_cell(i - r, M)]; });
        tab[(size_t)i * pad + m] = path ? v / (double)(m + 1) : v;
    }
}

int launch_cell_coefs(int M, int D, bool path, const double *c, double *tab, cudaStream_t s)
{
    k_cell_coefs<<<(M + 63) / 64, 64, 0, s>>>(M, D, path, c, tab);
    return 0;
}

__global__ void k_tables2(int M, int K, int fp32, const double *an_y, const double *an_z, const double *ak_y,
                          const double *ak_z, CoefTables T)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    a_rows(i, M, K, fp32, an_y, an_z, T.A);
    a_rows(i, M, K, fp32, ak_y, ak_z, T.Kt);
    if (!fp32) return;
    const int pad = coef_pad(fp32, K + 1);
    for (int c = 0; c < 2; ++c) {
        const double *n = c ? an_z : an_y, *k = c ? ak_z : ak_y;
        for (int m = 0; m <= K; ++m)
            T.L[(2 * (size_t)i + c) * pad + m] =
                sum_residue(cell_coef(K, m, [&](int r) { return n[wrap_cell(i - r, M)]; }),
                            cell_coef(K, m, [&](int r) { return k[wrap_cell(i - r, M)]; }));
    }
}

int launch_tables2(int M, int K, int fp32, const double *an_y, const double *an_z, const double *ak_y,
                   const double *ak_z, CoefTables T, cudaStream_t s)
{
    k_tables2<<<(M + 63) / 64, 64, 0, s>>>(M, K, fp32, an_y, an_z, ak_y, ak_z, T);
    return 0;
}

// Discrete Poisson right side: with r = -rho + dx, d = M1 e_x solves
// (d_j - d_{j+1}) / dx = r_j (Remark 2, Sec. 4.2): a running sum made mean-free.
__global__ void k_poisson_rhs(int M, double dx, const double *rho, double *d)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double run = 0.0, sum = 0.0;
    for (int j = 0; j < M; ++j) {
        d[j] = run;
        sum += run;
        run -= dx * (dx - rho[j]);
    }
    const double mean = sum / M;
    for (int j = 0; j < M; ++j) d[j] -= mean;
}

int launch_poisson_rhs(int M, double dx, const double *rho, double *d, cudaStream_t s)
{
    k_poisson_rhs<<<1, 32, 0, s>>>(M, dx, rho, d);
    return 0;
}

// Field energies (Eq. discrete_H) and the Gauss-law residual (Remark 2, Sec. 4.2).
__global__ void k_energy_grid(int M, int K, double dx, const double *rowM0, const double *rowM1,
                              const double *rowK, const double *ex, const double *ey,
                              const double *ez, const double *ay, const double *az,
                              const double *rho, double *diag)
{
    __shared__ double s_red[32];
    double eex = 0.0, eperp = 0.0, aperp = 0.0, gres = 0.0;
    for (int i = threadIdx.x; i < M; i += blockDim.x) {
        double m1e = rowM1[0] * ex[i], m1e_next = 0.0;
        const int inx = (i + 1) % M;
        m1e_next = rowM1[0] * ex[inx];
        for (int d = 1; d <= K - 1; ++d) {
            m1e += rowM1[d] * (ex[(i + d) % M] + ex[(i - d + M) % M]);
            m1e_next += rowM1[d] * (ex[(inx + d) % M] + ex[(inx - d + M) % M]);
        }
        double m0y = rowM0[0] * ey[i], m0z = rowM0[0] * ez[i];
        double ky = rowK[0] * ay[i], kz = rowK[0] * az[i];
        for (int d = 1; d <= K; ++d) {
            const int ip = (i + d) % M, im = (i - d + M) % M;
            m0y += rowM0[d] * (ey[ip] + ey[im]);
            m0z += rowM0[d] * (ez[ip] + ez[im]);
            ky += rowK[d] * (ay[ip] + ay[im]);
            kz += rowK[d] * (az[ip] + az[im]);
        }
        eex += 0.5 * ex[i] * m1e;
        eperp += 0.5 * (ey[i] * m0y + ez[i] * m0z);
        aperp += 0.5 * (ay[i] * ky + az[i] * kz);
        const double r = (m1e - m1e_next) / dx + rho[i] - dx;
        gres = fmax(gres, fabs(r));
    }
    double v;
    v = warp_sum(eex);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) { double s = 0; for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += s_red[w]; diag[1] = s; }
    __syncthreads();
    v = warp_sum(eperp);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) { double s = 0; for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += s_red[w]; diag[2] = s; }
    __syncthreads();
    v = warp_sum(aperp);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) { double s = 0; for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += s_red[w]; diag[3] = s; }
    __syncthreads();
    v = warp_max(gres);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) { double s = 0; for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s = fmax(s, s_red[w]); diag[5] = s; }
}

int launch_energy_grid(int M, int K, double dx, const double *rowM0, const double *rowM1,
                       const double *rowK, const double *ex, const double *ey, const double *ez,
                       const double *ay, const double *az, const double *rho, double *diag,
                       cudaStream_t s)
{
    k_energy_grid<<<1, 256, 0, s>>>(M, K, dx, rowM0, rowM1, rowK, ex, ey, ez, ay, az, rho, diag);
    return 0;
}

__global__ void k_ctrl_reset(DevCtrl *c)
{
    c->dmax_bits = 0ull;
    c->emax_bits = 0ull;
    c->emag_bits = 0ull;
    c->dprev_bits = 0x7ff0000000000000ull;
    c->eprev_bits = 0x7ff0000000000000ull;
    c->iter = 0;
    c->converged = 0;
    c->status = 0;
    c->ticket = 0u;
    c->hist1 = 0;
    c->hist2 = 0;
    c->zany = 0;
    c->acc[0] = c->acc[1] = c->acc[2] = c->acc[3] = 0.0;
}

int launch_ctrl_reset(DevCtrl *ctrl, cudaStream_t s)
{
    k_ctrl_reset<<<1, 1, 0, s>>>(ctrl);
    return 0;
}

}  // namespace pic

// Zeeman source of subsystem II (Sec. 4.2): b_y -= dt hbar (G^T d_z)_j and
// b_z += dt hbar (G^T d_y)_j, (G^T v)_j = (v_j - v_{j+1}) / dx, d = Lambda_1(X)^T W S.
__global__ void k_spin_rhs(int M, double dx, double c, const double *dy, const double *dz, double *by,
                           double *bz)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    const int jp = j + 1 == M ? 0 : j + 1;
    by[j] -= c * (dz[j] - dz[jp]) / dx;
    bz[j] += c * (dy[j] - dy[jp]) / dx;
}

namespace pic {
int launch_spin_rhs(int M, double dx, double dt, double hbar, const double *dy, const double *dz, double *by,
                    double *bz, cudaStream_t s)
{
    k_spin_rhs<<<(M + 255) / 256, 256, 0, s>>>(M, dx, dt * hbar, dy, dz, by, bz);
    return 0;
}
}  // namespace pic

// Split runs (markers over several processes): the marker-side results of a sweep
// that every process must agree on, packed as doubles for a max-reduction over
// processes: the largest position increment, and one entry per error bit (the max
// of 0/1 entries is their logical or).
__global__ void k_split_pack(const pic::DevCtrl *c, double *buf)
{
    buf[0] = pic::bits_to_double(c->dmax_bits);
    buf[1] = (c->status & pic::STATUS_NUMERIC) ? 1.0 : 0.0;
    buf[2] = (c->status & pic::STATUS_TIMEOUT) ? 1.0 : 0.0;
}

__global__ void k_split_unpack(pic::DevCtrl *c, const double *buf)
{
    c->dmax_bits = (unsigned long long)__double_as_longlong(buf[0]);
    if (buf[1] != 0.0) c->status |= pic::STATUS_NUMERIC;
    if (buf[2] != 0.0) c->status |= pic::STATUS_TIMEOUT;
}

namespace pic {
int launch_split_pack(const DevCtrl *c, double *buf, cudaStream_t s)
{
    k_split_pack<<<1, 1, 0, s>>>(c, buf);
    return 0;
}
int launch_split_unpack(DevCtrl *c, const double *buf, cudaStream_t s)
{
    k_split_unpack<<<1, 1, 0, s>>>(c, buf);
    return 0;
}
}  // namespace pic
