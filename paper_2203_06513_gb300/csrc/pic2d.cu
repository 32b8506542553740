// pic2d.cu -- subsystem I of the two-dimensional scheme (Sec. 4.3) on the GPU, FP64.
//
// Spaces (Sec. 3.2): tensor-product B-splines on a uniform periodic M1 x M2 grid,
// node i = i1 * M2 + i2; A_z on N^k x N^k, the 1-form e_xy as e_x on N^{k-1} x N^k
// and e_y on N^k x N^{k-1}.  As in one dimension (pic_poly.cuh) every field is one
// polynomial per cell, here in both centred offsets (v1, v2) with coefficients
// sum_{r1, r2} c_{c1-r1, c2-r2} B[r1][a] B[r2][b], and deposits are moments v1^a v2^b of
// the cell: the marker kernel evaluates no basis function, and the grid kernels convert
// between nodes and cells once per sweep.  One thread per marker and sweep:
//   * the path means of both V1 components along x^n -> x^(k) (the straight path split at
//     every knot crossing of either coordinate, k-point Gauss--Legendre on each piece: the
//     integrand is a polynomial of degree 2k - 1 there), e_bar evaluated by Horner's rule
//     at the quadrature points;
//   * the coordinate-increment difference quotients D of A_z: along x1 at x2^(k) the
//     polynomial contracted over v2 (which gives A(x^(k)) as well) and its exact divided
//     difference, along x2 at x1^n the same with the contraction over v1, which does not
//     change during the fixed point and is kept from its first sweep;
//   * with spins (hbar != 0), the quotients of the Zeeman term hbar s . B,
//     B = (dA/dx2, -dA/dx1, b_z), the same way from the contracted derivatives;
//   * the momentum and position updates of the discrete-gradient scheme;
//   * the moments of the new path x^n -> x^(k+1), added to the cells in global memory.
// The grid side applies M1^{-1} = diag(M1_x^{-1} (x) M0_y^{-1}, M0_x^{-1} (x) M1_y^{-1})
// as two circulant passes with the exact inverse rows of the 1D mass matrices.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "pic2d.h"
#include "pic_hostcopy.h"
#include "pic_internal.h"
#include "pic_poly.cuh"

namespace pic {
namespace {

constexpr int kMax2DNodes = 4096;     // largest M1 * M2
constexpr int kMaxCross = 16;         // knot crossings per coordinate and path

__constant__ SplineTab c_spline2 = make_spline_tab();

// coefficients per cell, rows padded to 16 bytes: A (K+1)^2, e_x K (K+1) as [a][b], e_y
// (K+1) K, b_z K^2; moments of the two current components like e_x and e_y, unpadded
template <int K> struct Dim2 {
    static constexpr int nA = (K + 1) * (K + 1), nE = K * (K + 1), nB = K * K;
    static constexpr int pA = (nA + 1) & ~1, pE = (nE + 1) & ~1, pB = (nB + 1) & ~1;
    static constexpr int nCache = K + 2;    // contraction over v1 (b = 1 .. K), A(x^n), gamma
};
inline int pad2(int n) { return (n + 1) & ~1; }

struct Args2D {
    int M1, M2;
    long long np;
    double dx1, dx2, dt, w;
    double idx1, idx2;      // 1 / dx1, 1 / dx2
    int2 *cell;
    double2 *v;             // centred offsets
    double *cache;          // nCache x np, written by the first sweep of a step
    int first;              // this is the step's first sweep
    const double2 *pn;
    double2 *d;             // displacement iterate (cell units), in/out
    double2 *pk;            // momentum iterate, in/out
    const double *TA, *TEx, *TEy, *TB;
    double *mx, *my;        // moments of this sweep (zeroed before)
    double hbar;            // Zeeman terms on when non-zero (spins given)
    const double *s;        // np x 3 spins
    unsigned long long *dmax_bits, *pmax_bits;
    int *status;
    long long gls[5], glw[5];   // K-point Gauss--Legendre on [0, 1], times 2^62
};

__device__ __forceinline__ int wrapi(int i, int M)
{
    int r = i % M;
    return r < 0 ? r + M : r;
}

// Pieces of the path (v1, v2) -> + (d1, d2) between knot crossings, n1 and n2 cells over:
// f(sa, sb, k1, k2) for consecutive parameter values 0 = s_0 < ... = 1, in the cell k1, k2
// over.
template <class F>
__device__ __forceinline__ void walk2(double v1, double v2, double d1, double d2, int n1, int n2, F &&f)
{
    double sa = 0.0, sb = 1.0, r1 = 0.0, r2 = 0.0;
    int k1 = 0, k2 = 0;
    const bool multi = n1 != 0 || n2 != 0;
    const int g1 = n1 > 0 ? 1 : -1, g2 = n2 > 0 ? 1 : -1;
    if (multi) {
        r1 = n1 != 0 ? 1.0 / d1 : 0.0;
        r2 = n2 != 0 ? 1.0 / d2 : 0.0;
    }
    for (int guard = 0; guard < 2 * kMaxCross + 2; ++guard) {
        double b1 = 2.0, b2 = 2.0;
        bool go = true, last = true;        // a path in one cell compares nothing
        if (multi) {
            if (k1 != n1) b1 = ((double)k1 + 0.5 * g1 - v1) * r1;
            if (k2 != n2) b2 = ((double)k2 + 0.5 * g2 - v2) * r2;
            sb = fmin(fmin(b1, b2), 1.0);
            go = sb > sa;
            last = sb >= 1.0;
        }
        if (go) f(sa, sb, k1, k2);
        if (last) return;
        if (b1 <= sb) k1 += g1;
        if (b2 <= sb) k2 += g2;
        sa = fmax(sa, sb);
    }
}

// row[q] = sum_b c[q][b] y^b for the rows q = 0 .. NR - 1 of NC coefficients at `c`
template <int NR, int NC>
__device__ __forceinline__ void contract_rows(const double *c, double y, double (&row)[NR])
{
    double q[NR * NC];
    load_coef<NR * NC>(c, q);
#pragma unroll
    for (int a = 0; a < NR; ++a) {
        double s = q[a * NC + NC - 1];
#pragma unroll
        for (int b = NC - 2; b >= 0; --b) s = fma(s, y, q[a * NC + b]);
        row[a] = s;
    }
}

// col[q] = sum_a c[a][q] x^a
template <int NR, int NC>
__device__ __forceinline__ void contract_cols(const double *c, double x, double (&col)[NC])
{
    double q[NR * NC];
    load_coef<NR * NC>(c, q);
#pragma unroll
    for (int b = 0; b < NC; ++b) {
        double s = q[(NR - 1) * NC + b];
#pragma unroll
        for (int a = NR - 2; a >= 0; --a) s = fma(s, x, q[a * NC + b]);
        col[b] = s;
    }
}

// d/dy of the rows: row[q] = sum_{b >= 1} b c[q][b] y^(b-1)
template <int NR, int NC>
__device__ __forceinline__ void contract_rows_dy(const double *c, double y, double (&row)[NR])
{
#pragma unroll
    for (int a = 0; a < NR; ++a) {
        double s = (double)(NC - 1) * c[a * NC + NC - 1];
#pragma unroll
        for (int b = NC - 2; b >= 1; --b) s = fma(s, y, (double)b * c[a * NC + b]);
        row[a] = s;
    }
}

template <int NR, int NC>
__device__ __forceinline__ void contract_cols_dx(const double *c, double x, double (&col)[NC])
{
#pragma unroll
    for (int b = 0; b < NC; ++b) {
        double s = (double)(NR - 1) * c[(NR - 1) * NC + b];
#pragma unroll
        for (int a = NR - 2; a >= 1; --a) s = fma(s, x, (double)a * c[a * NC + b]);
        col[b] = s;
    }
}

// One piece of a coordinate-increment quotient: the sums of a path along one coordinate
// (n cells over, from v0 to the end offset ve), piece q of 0 .. |n|.  h: its length, or 1
// for a path in one cell (the mean itself).
template <int N>
__device__ __forceinline__ double quotient_piece(int q, int n, double v0, double ve, double (&S)[N])
{
    const int an = abs(n);
    const double edge = n > 0 ? 0.5 : -0.5;
    const double va = q == 0 ? v0 : -edge, vb = q == an ? ve : edge;
    path_sums<N, double>(va, vb, S);
    return an == 0 ? 1.0 : vb - va;
}

// sum_{q >= 1} c_q S_{q-1}: the divided difference of the polynomial c
template <int N>
__device__ __forceinline__ double divided(const double (&c)[N], const double (&S)[N - 1])
{
    double s = c[1];
#pragma unroll
    for (int q = 2; q < N; ++q) s = fma(c[q], S[q - 1], s);
    return s;
}

// The means of x^a y^b (a, b <= K, not both K) over a path piece in one cell, from (xa, ya)
// to (xb, yb) (offsets, 1/2 in size and rounding), by K Gauss points, which are exact.  In
// integers of 64 bits, beside the FP64 pipe: the offsets times 2^63, the means times
// 2^(60 + a + b), since x^a y^b is at most 2^-(a + b).  Relative to that the means are off by
// 1e-16 at most (rms, degrees 2 to 5), where the same sums in double are off by 2e-16; with
// 2^60 for all of them the highest means of degree 5 were off by 1e-15.
template <int K>
__device__ __forceinline__ void piece_means2(const Args2D &A, double xa, double ya, double xb, double yb,
                                             double (&md)[K + 1][K + 1])
{
    const long long x0 = to_fixed<63>(xa), y0 = to_fixed<63>(ya);
    const long long dx = (to_fixed<63>(xb) >> 1) - (x0 >> 1), dy = (to_fixed<63>(yb) >> 1) - (y0 >> 1);   // 2^62
    long long m[K + 1][K + 1];
#pragma unroll
    for (int g = 0; g < K; ++g) {
        const long long x = x0 + (__mul64hi(dx, A.gls[g]) << 3), y = y0 + (__mul64hi(dy, A.gls[g]) << 3);
        long long yp[K + 1];                            // y^b 2^(62 + b)
        yp[0] = 0;
        yp[1] = y;
#pragma unroll
        for (int b = 2; b <= K; ++b) yp[b] = __mul64hi(yp[b - 1], y) << 2;
        long long xw = A.glw[g];                        // w x^a 2^(62 + a)
#pragma unroll
        for (int a = 0; a <= K; ++a) {
            if (a > 0) xw = __mul64hi(xw, x) << 2;
#pragma unroll
            for (int b = 0; b <= K; ++b) {
                if (a == K && b == K) continue;
                const long long t = b == 0 ? xw >> 2 : __mul64hi(xw, yp[b]);
                m[a][b] = g == 0 ? t : m[a][b] + t;
            }
        }
    }
#pragma unroll
    for (int a = 0; a <= K; ++a)
#pragma unroll
        for (int b = 0; b <= K; ++b)
            if (a < K || b < K) md[a][b] = from_fixed60(m[a][b], a + b);
}

// f(cell, h, means) for the pieces of the path from v over d, which ends at (e1, e2) n1 and
// n2 cells over; h: the fraction of the path in the piece
template <int K, class F>
__device__ __forceinline__ void path_pieces(const Args2D &A, int2 c, double2 v, double2 d, int n1, int n2, double e1,
                                            double e2, F &&f)
{
    walk2(v.x, v.y, d.x, d.y, n1, n2, [&](double sa, double sb, int k1, int k2) {
        int cell = c.x * A.M2 + c.y;
        double xa = v.x, ya = v.y, xb = e1, yb = e2, h = 1.0;
        if (n1 != 0 || n2 != 0) {
            cell = wrapi(c.x + k1, A.M1) * A.M2 + wrapi(c.y + k2, A.M2);
            const double x0 = v.x - (double)k1, y0 = v.y - (double)k2;
            xa = fma(sa, d.x, x0);
            ya = fma(sa, d.y, y0);
            xb = fma(sb, d.x, x0);
            yb = fma(sb, d.y, y0);
            h = sb - sa;
        }
        double md[K + 1][K + 1];
        piece_means2<K>(A, xa, ya, xb, yb, md);
        f(cell, h, md);
    });
}

// (Ex, Ey) = the path means of e_bar's two components
template <int K>
__device__ __forceinline__ void gather_path(const Args2D &A, int2 c, double2 v, double2 d, int n1, int n2, double e1,
                                            double e2, double &Ex, double &Ey)
{
    Ex = Ey = 0.0;
    path_pieces<K>(A, c, v, d, n1, n2, e1, e2, [&](int cell, double h, const double (&md)[K + 1][K + 1]) {
        double ex[K * (K + 1)], ey[K * (K + 1)];
        load_coef<K * (K + 1)>(A.TEx + (size_t)cell * Dim2<K>::pE, ex);
        load_coef<K * (K + 1)>(A.TEy + (size_t)cell * Dim2<K>::pE, ey);
        double sx = ex[0] * md[0][0], sy = ey[0] * md[0][0];
#pragma unroll
        for (int a = 0; a <= K; ++a)
#pragma unroll
            for (int b = 0; b <= K; ++b) {
                if (a + b == 0) continue;
                if (a < K) sx = fma(ex[a < K ? a * (K + 1) + b : 0], md[a][b], sx);
                if (b < K) sy = fma(ey[b < K ? a * K + b : 0], md[a][b], sy);
            }
        Ex = fma(h, sx, Ex);
        Ey = fma(h, sy, Ey);
    });
}

// (wx, wy) x the path moments of the two components to the cells, one addition in global
// memory per moment and piece
template <int K>
__device__ __forceinline__ void deposit_path(const Args2D &A, int2 c, double2 v, double2 d, int n1, int n2, double e1,
                                             double e2, double wx, double wy)
{
    const bool bx = wx != 0.0, by = wy != 0.0;
    path_pieces<K>(A, c, v, d, n1, n2, e1, e2, [&](int cell, double h, const double (&md)[K + 1][K + 1]) {
        double *px = A.mx + (size_t)cell * Dim2<K>::nE, *py = A.my + (size_t)cell * Dim2<K>::nE;
        const double hx = h * wx, hy = h * wy;
#pragma unroll
        for (int a = 0; a <= K; ++a)
#pragma unroll
            for (int b = 0; b <= K; ++b) {
                if (a < K && bx) atomicAdd(px + a * (K + 1) + b, hx * md[a][b]);
                if (b < K && by) atomicAdd(py + a * K + b, hy * md[a][b]);
            }
    });
}

__device__ __forceinline__ void max_bits(unsigned long long *dst, double v)
{
    // non-negative doubles order like their bit patterns; NaN maps to the largest
    const unsigned long long b = (v == v) ? (unsigned long long)__double_as_longlong(v) : 0x7ff8000000000000ull;
    atomicMax(dst, b);
}

// PRE: the predicted start instead of a sweep -- A(x^n) stored, the explicit
// predictor delta^(0) = dt p^n / gamma(p^n, A(x^n)) written and the current of
// x^n -> x^n + delta^(0) deposited, so that the fixed point can start from the
// field consistent with it; no gather, no momentum update, no increments.
//
// Bound by the FP64 pipe.  With basis values at the quadrature points and 24 weights per
// piece, added to the block's shared rows by compare-and-swap, the sweep took 1068 FP64
// operations a marker (cubic, path in one cell) and 4.1 ms for 2e6 markers.
constexpr int kTile2 = 256;          // markers a warp groups at a time
template <int K> constexpr int sweep2d_blocks = K <= 3 ? 2 : 1;      // resident on an SM
template <int K, bool PRE = false>
__global__ void __launch_bounds__(256, sweep2d_blocks<K>) k2_sweep(Args2D A)
{
    using Dm = Dim2<K>;
    constexpr int NC = K + 1;
    __shared__ unsigned char s_perm[8][kTile2];
    double dm = 0.0, pm = 0.0;
    bool bad = false;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    // a run of markers per warp
    const long long warps = gridDim.x * 8LL, run = ((A.np + warps - 1) / warps + 31) & ~31LL;
    const long long beg = (blockIdx.x * 8LL + wid) * run, end = beg + run < A.np ? beg + run : A.np;
    for (long long base = beg; base < end; base += kTile2) {
        // The warp's next markers in two groups, paths within one cell first and paths
        // across a knot last (by the current iterate; the new path mostly follows it): the
        // extra pieces of a crossing then run only in the steps that hold crossing markers,
        // instead of nearly every step running them for one lane.  By warps, not blocks:
        // the warps of a block with the crossings kept the others waiting (388 us for 5e5
        // cubic markers, 293 so).
        const int n = (int)(end - base < kTile2 ? end - base : kTile2);
        int front = 0, back = n;
        for (int q = 0; q < n; q += 32) {
            const long long b = base + q + lane;
            const bool act = q + lane < n;
            bool multi = true;
            if (act) {
                const double2 v = A.v[b];
                double2 d = A.d[b];
                if (PRE) {                      // the predicted start's path is within dt p (gamma >= 1)
                    const double2 p = A.pn[b];
                    d = make_double2(A.dt * p.x * A.idx1, A.dt * p.y * A.idx2);
                }
                multi = !within(v.x + d.x, 0.5) || !within(v.y + d.y, 0.5);
            }
            const unsigned one = __ballot_sync(0xffffffffu, !multi), more = __ballot_sync(0xffffffffu, act && multi);
            if (act) s_perm[wid][multi ? back - 1 - __popc(more & lt) : front + __popc(one & lt)] = (unsigned char)(q + lane);
            front += __popc(one);
            back -= __popc(more);
        }
        __syncwarp();
        for (int q = lane; q < n; q += 32) {
            const long long a = base + s_perm[wid][q];
            const int2 c = A.cell[a];
            const double2 v = A.v[a], p = A.pn[a];
            double2 d = PRE ? make_double2(0.0, 0.0) : A.d[a];
            const double pp1 = fma(p.x, p.x, fma(p.y, p.y, 1.0));
            // beta_b: A contracted over v1 at x1^n; A(x^n) and gamma(p^n, A(x^n)); the same in
            // every sweep of the step
            double be[NC], A0, g0;
            if (PRE || A.first) {
                contract_cols<NC, NC>(A.TA + (size_t)(c.x * A.M2 + c.y) * Dm::pA, v.x, be);
                A0 = horner<NC>(be, v.y);
                g0 = root(fma(A0, A0, pp1));
    #pragma unroll
                for (int b = 1; b <= K; ++b) A.cache[(size_t)(b - 1) * A.np + a] = be[b];
                A.cache[(size_t)K * A.np + a] = A0;
                A.cache[(size_t)(K + 1) * A.np + a] = g0;
            } else {
                be[0] = 0.0;
    #pragma unroll
                for (int b = 1; b <= K; ++b) be[b] = A.cache[(size_t)(b - 1) * A.np + a];
                A0 = A.cache[(size_t)K * A.np + a];
                g0 = A.cache[(size_t)(K + 1) * A.np + a];
            }
            if constexpr (PRE) {
                const double r = quotient(A.dt, g0);
                const double x0 = r * p.x, x1 = r * p.y;
                d = make_double2(x0 * A.idx1, x1 * A.idx2);
                if (!within(d.x, 1024.0) || !within(d.y, 1024.0)) { bad = true; continue; }
                int n1, n2;
                double e1, e2;
                path_end(v.x, d.x, n1, e1);
                path_end(v.y, d.y, n2, e2);
                if (abs(n1) > kMaxCross || abs(n2) > kMaxCross) bad = true;
                else deposit_path<K>(A, c, v, d, n1, n2, e1, e2, A.w * x0, A.w * x1);
                A.d[a] = d;
                continue;
            }
            int n1, n2;
            double e1, e2;
            path_end(v.x, d.x, n1, e1);
            path_end(v.y, d.y, n2, e2);
            const bool spin = A.hbar != 0.0;
            double sx = 0.0, sy = 0.0, sz = 0.0, Z1 = 0.0, Z2 = 0.0;
            if (spin) {
                sx = A.s[3 * a] * A.idx2;           // s_x dA/dx2, s_y dA/dx1 in cell units
                sy = A.s[3 * a + 1] * A.idx1;
                sz = A.s[3 * a + 2];
            }
            // along x1 at x2^(k): alpha_a, A contracted over v2; A(x^(k)) in the last cell
            double D1 = 0.0, W1 = 0.0, A1 = 0.0;
            for (int q = 0; q <= abs(n1); ++q) {
                int cell = c.x * A.M2 + c.y;
                if (n1 != 0 || n2 != 0)
                    cell = wrapi(c.x + (n1 > 0 ? q : -q), A.M1) * A.M2 + wrapi(c.y + n2, A.M2);
                double al[NC], S[K];
                const double *row = A.TA + (size_t)cell * Dm::pA;
                contract_rows<NC, NC>(row, e2, al);
                const double h = quotient_piece<K>(q, n1, v.x, e1, S);
                D1 = fma(h, divided<NC>(al, S), D1);
                W1 += h;
                if (q == abs(n1)) A1 = horner<NC>(al, e1);
                if (spin) {
                    // f = s_x dA/dx2 - s_y dA/dx1 + s_z b_z contracted over v2, its quotient
                    double ady[NC], bz[K], f[NC];
                    contract_rows_dy<NC, NC>(row, e2, ady);
                    contract_rows<K, K>(A.TB + (size_t)cell * Dm::pB, e2, bz);
    #pragma unroll
                    for (int m = 0; m <= K; ++m) {
                        f[m] = sx * ady[m];
                        if (m < K) f[m] += sz * bz[m < K ? m : 0] - sy * (double)(m + 1) * al[m < K ? m + 1 : 0];
                    }
                    Z1 = fma(h, divided<NC>(f, S), Z1);
                }
            }
            // along x2 at x1^n
            double D2 = 0.0, W2 = 0.0;
            for (int q = 0; q <= abs(n2); ++q) {
                const int cell = q == 0 ? c.x * A.M2 + c.y : c.x * A.M2 + wrapi(c.y + (n2 > 0 ? q : -q), A.M2);
                const double *row = A.TA + (size_t)cell * Dm::pA;
                double bq[NC], S[K];
                if (q == 0) {
    #pragma unroll
                    for (int b = 0; b <= K; ++b) bq[b] = be[b];
                } else {
                    contract_cols<NC, NC>(row, v.x, bq);
                }
                const double h = quotient_piece<K>(q, n2, v.y, e2, S);
                D2 = fma(h, divided<NC>(bq, S), D2);
                W2 += h;
                if (spin) {
                    double adx[NC], bz[K], f[NC];
                    contract_cols_dx<NC, NC>(row, v.x, adx);
                    contract_cols<K, K>(A.TB + (size_t)cell * Dm::pB, v.x, bz);
    #pragma unroll
                    for (int m = 0; m <= K; ++m) {
                        f[m] = -sy * adx[m];
                        if (m < K) f[m] += sz * bz[m < K ? m : 0] + sx * (double)(m + 1) * bq[m < K ? m + 1 : 0];
                    }
                    Z2 = fma(h, divided<NC>(f, S), Z2);
                }
            }
            if (n1 != 0) { D1 = quotient(D1, W1); Z1 = Z1 / W1; }
            if (n2 != 0) { D2 = quotient(D2, W2); Z2 = Z2 / W2; }
            double Ex, Ey;
            gather_path<K>(A, c, v, d, n1, n2, e1, e2, Ex, Ey);
            const double g1 = root(fma(A1, A1, pp1));
            const double f = quotient(A.dt * (A1 + A0), g1 + g0);
            double q0 = fma(A.dt, Ex, p.x) - f * (D1 * A.idx1);
            double q1 = fma(A.dt, Ey, p.y) - f * (D2 * A.idx2);
            if (spin) {
                q0 -= A.dt * A.hbar * Z1 * A.idx1;
                q1 -= A.dt * A.hbar * Z2 * A.idx2;
            }
            const double g2 = root(fma(q0, q0, fma(q1, q1, fma(A1, A1, 1.0))));
            const double r = quotient(A.dt, g1 + g2);
            const double x0 = r * (p.x + q0), x1 = r * (p.y + q1);
            const double2 dn = make_double2(x0 * A.idx1, x1 * A.idx2);
            if (!within(dn.x, 1024.0) || !within(dn.y, 1024.0)) { bad = true; continue; }
            // the current of the new path
            path_end(v.x, dn.x, n1, e1);
            path_end(v.y, dn.y, n2, e2);
            if (abs(n1) > kMaxCross || abs(n2) > kMaxCross) bad = true;
            else deposit_path<K>(A, c, v, dn, n1, n2, e1, e2, A.w * x0, A.w * x1);
            const double2 po = A.pk[a];
            dm = max_nonneg(dm, max_nonneg(fabs(dn.x - d.x) * A.dx1, fabs(dn.y - d.y) * A.dx2));
            pm = max_nonneg(pm, max_nonneg(fabs(q0 - po.x), fabs(q1 - po.y)));
            A.d[a] = dn;
            A.pk[a] = make_double2(q0, q1);
        }
        __syncwarp();
    }
    if (bad) atomicOr(A.status, STATUS_NUMERIC);
    if (PRE) return;
    // block maxima of the increments
    __shared__ double s_m[2][8];
    for (int o = 16; o > 0; o >>= 1) {
        dm = max_nonneg(dm, __shfl_xor_sync(0xffffffffu, dm, o));
        pm = max_nonneg(pm, __shfl_xor_sync(0xffffffffu, pm, o));
    }
    if ((threadIdx.x & 31) == 0) {
        s_m[0][threadIdx.x >> 5] = dm;
        s_m[1][threadIdx.x >> 5] = pm;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            a = max_nonneg(a, s_m[0][w]);
            b = max_nonneg(b, s_m[1][w]);
        }
        max_bits(A.dmax_bits, a);
        max_bits(A.pmax_bits, b);
    }
}

// Coefficient (a, b) of the degree (D1, D2) field with nodes c in every cell: thread per
// (cell, a, b), coefficients fastest; rows of `pad` numbers.
template <int D1, int D2>
__device__ __forceinline__ void table2_at(long long t, int M1, int M2, const double *c, double *tab, int pad)
{
    constexpr int n = (D1 + 1) * (D2 + 1);
    const int cell = (int)(t / n), q = (int)(t % n), a = q / (D2 + 1), b = q % (D2 + 1);
    const int c1 = cell / M2, c2 = cell % M2;
    int o2[D2 + 1];
#pragma unroll
    for (int r = 0; r <= D2; ++r) o2[r] = wrapi(c2 - r, M2);
    double s = 0.0;
#pragma unroll
    for (int r1 = 0; r1 <= D1; ++r1) {
        const double *row = c + (size_t)wrapi(c1 - r1, M1) * M2;
        double u = 0.0;
#pragma unroll
        for (int r2 = 0; r2 <= D2; ++r2) u = fma(c_spline2.b[D2][r2][b], row[o2[r2]], u);
        s = fma(c_spline2.b[D1][r1][a], u, s);
    }
    tab[(size_t)cell * pad + q] = s;
}

template <int D1, int D2>
__global__ void __launch_bounds__(128) k2_table(int M1, int M2, const double *c, double *tab, int pad)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < (long long)M1 * M2 * (D1 + 1) * (D2 + 1)) table2_at<D1, D2>(t, M1, M2, c, tab, pad);
}

// both components of e_bar (blockIdx.y)
template <int K>
__global__ void __launch_bounds__(128) k2_table_e(int M1, int M2, const double *ebx, const double *eby, double *TEx,
                                                  double *TEy)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)M1 * M2 * K * (K + 1)) return;
    if (blockIdx.y == 0) table2_at<K - 1, K>(t, M1, M2, ebx, TEx, Dim2<K>::pE);
    else table2_at<K, K - 1>(t, M1, M2, eby, TEy, Dim2<K>::pE);
}

// node values of a current component from its moments: degree (D1, D2), moments [a][b]
template <int D1, int D2>
__device__ __forceinline__ double node2_at(int M1, int M2, const double *m, int i1, int i2)
{
    double s = 0.0;
#pragma unroll
    for (int r1 = 0; r1 <= D1; ++r1) {
        const int c1 = wrapi(i1 + r1, M1) * M2;
#pragma unroll
        for (int r2 = 0; r2 <= D2; ++r2) {
            const double *row = m + (size_t)(c1 + wrapi(i2 + r2, M2)) * ((D1 + 1) * (D2 + 1));
#pragma unroll
            for (int a = 0; a <= D1; ++a) {
                double u = 0.0;
#pragma unroll
                for (int b = 0; b <= D2; ++b) u = fma(c_spline2.b[D2][r2][b], row[a * (D2 + 1) + b], u);
                s = fma(c_spline2.b[D1][r1][a], u, s);
            }
        }
    }
    return s;
}

template <int K>
__global__ void __launch_bounds__(64) k2_nodes(int M1, int M2, const double *mx, const double *my, double *jx, double *jy)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M1 * M2) return;
    if (blockIdx.y == 0) jx[i] = node2_at<K - 1, K>(M1, M2, mx, i / M2, i % M2);
    else jy[i] = node2_at<K, K - 1>(M1, M2, my, i / M2, i % M2);
}

// sum_q g[(i - q) mod M] in[q stride]: a quarter of the terms a thread, kCirc outputs a block
// of 4 kCirc threads (a whole sum a thread is one chain of M dependent reads: 28 us along
// x1 of 64 x 64 nodes, 11 so).  The sum is returned to the block's first kCirc threads.
constexpr int kCirc = 16;
__device__ __forceinline__ double circ_at(int M, int i, const double *__restrict__ g, const double *__restrict__ in,
                                          int stride)
{
    __shared__ double s_part[3][kCirc];
    const int part = threadIdx.x / kCirc, o = threadIdx.x % kCirc;
    const int q1 = (part + 1) * M / 4;
    double s[2] = {0.0, 0.0};
    int q = part * M / 4, k = i - q < 0 ? i - q + M : i - q;
    for (; q < q1; ++q) {
        s[q & 1] = fma(g[k], in[(size_t)q * stride], s[q & 1]);
        k = k == 0 ? M - 1 : k - 1;
    }
    const double t = s[0] + s[1];
    if (part > 0) s_part[part - 1][o] = t;
    __syncthreads();
    return part > 0 ? 0.0 : (t + s_part[0][o]) + (s_part[1][o] + s_part[2][o]);
}

// pass along x2 of both components (blockIdx.y): out[i1, i2] = sum_q g[(i2 - q) mod M2] in[i1, q]
__global__ void __launch_bounds__(4 * kCirc) k2_circ2(int M1, int M2, const double *gx, const double *gy, const double *jx,
                                               const double *jy, double *ox, double *oy)
{
    const int i = blockIdx.x * kCirc + threadIdx.x % kCirc, n = min(i, M1 * M2 - 1);
    const int i1 = n / M2, i2 = n % M2;
    const bool y = blockIdx.y != 0;
    const double v = circ_at(M2, i2, y ? gy : gx, (y ? jy : jx) + (size_t)i1 * M2, 1);
    if (threadIdx.x < kCirc && i < M1 * M2) (y ? oy : ox)[i] = v;
}

// pass along x1, then e^(k+1) = e^n - M1^{-1} j, its increment's max-norm, e_bar for the
// next sweep
__global__ void __launch_bounds__(4 * kCirc) k2_circ1(int M1, int M2, const double *gx, const double *gy, const double *tx,
                                               const double *ty, const double *enx, const double *eny, double *ekx,
                                               double *eky, double *ebx, double *eby, unsigned long long *emax_bits)
{
    const int i = blockIdx.x * kCirc + threadIdx.x % kCirc, n = min(i, M1 * M2 - 1);
    const bool y = blockIdx.y != 0;
    const double sol = circ_at(M1, n / M2, y ? gy : gx, (y ? ty : tx) + n % M2, M2);
    double m = 0.0;
    if (threadIdx.x < kCirc && i < M1 * M2) {
        const double en = (y ? eny : enx)[i], v = en - sol;
        double *ek = y ? eky : ekx;
        m = fabs(v - ek[i]);
        ek[i] = v;
        (y ? eby : ebx)[i] = 0.5 * (en + v);
    }
    for (int o = 16; o > 0; o >>= 1) m = max_nonneg(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) max_bits(emax_bits, m);
}

// acc[0] += sum_a w (g(p_a, A(x_a)) - 1); with spins, acc[1] += sum_a w hbar
// (s_x dA/dx2 - s_y dA/dx1 + s_z b_z)(x_a)
template <int K>
__global__ void __launch_bounds__(256) k2_energy(Args2D A, const double2 *p, double *acc)
{
    constexpr int NC = K + 1;
    double s = 0.0, z = 0.0;
    for (long long a = blockIdx.x * (long long)blockDim.x + threadIdx.x; a < A.np;
         a += (long long)gridDim.x * blockDim.x) {
        const int cell = A.cell[a].x * A.M2 + A.cell[a].y;
        const double2 v = A.v[a], q = p[a];
        const double *row = A.TA + (size_t)cell * Dim2<K>::pA;
        double al[NC];
        contract_rows<NC, NC>(row, v.y, al);
        const double Az = horner<NC>(al, v.x);
        s += A.w * (sqrt(1.0 + q.x * q.x + q.y * q.y + Az * Az) - 1.0);
        if (A.hbar != 0.0) {
            double ady[NC], bz[K];
            contract_rows_dy<NC, NC>(row, v.y, ady);
            contract_rows<K, K>(A.TB + (size_t)cell * Dim2<K>::pB, v.y, bz);
            double d1 = (double)K * al[K];
#pragma unroll
            for (int m = K - 1; m >= 1; --m) d1 = fma(d1, v.x, (double)m * al[m]);
            z += A.w * A.hbar * (A.s[3 * a] * horner<NC>(ady, v.x) * A.idx2 - A.s[3 * a + 1] * d1 * A.idx1 +
                                 A.s[3 * a + 2] * horner<K>(bz, v.x));
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(acc, s);
        if (A.hbar != 0.0) atomicAdd(acc + 1, z);
    }
}

// x^{n+1} = x^n + delta (cells wrapped around the box), p^{n+1} = p^(k)
__global__ void k2_finalize(long long np, int M1, int M2, int2 *cell, double2 *v, double2 *p, const double2 *d,
                            const double2 *pk)
{
    for (long long a = blockIdx.x * (long long)blockDim.x + threadIdx.x; a < np;
         a += (long long)gridDim.x * blockDim.x) {
        int n1, n2;
        double2 u = v[a];
        const double2 dd = d[a];
        path_end(u.x, dd.x, n1, u.x);
        path_end(u.y, dd.y, n2, u.y);
        const int2 c = cell[a];
        if (n1 != 0 || n2 != 0) cell[a] = make_int2(wrapi(c.x + n1, M1), wrapi(c.y + n2, M2));
        v[a] = u;
        p[a] = pk[a];
    }
}

// positions in the box <-> cells and centred offsets
__global__ void k2_load(long long np, int M1, int M2, double dx1, double dx2, const double2 *x, int2 *cell, double2 *v)
{
    for (long long a = blockIdx.x * (long long)blockDim.x + threadIdx.x; a < np;
         a += (long long)gridDim.x * blockDim.x) {
        const double u1 = x[a].x / dx1, u2 = x[a].y / dx2;
        const double f1 = floor(u1), f2 = floor(u2);
        cell[a] = make_int2(wrapi((int)f1, M1), wrapi((int)f2, M2));
        v[a] = make_double2((u1 - f1) - 0.5, (u2 - f2) - 0.5);
    }
}

__global__ void k2_store(long long np, double L1, double L2, double dx1, double dx2, const int2 *cell, const double2 *v,
                         double2 *x)
{
    for (long long a = blockIdx.x * (long long)blockDim.x + threadIdx.x; a < np;
         a += (long long)gridDim.x * blockDim.x) {
        double x1 = (((double)cell[a].x + 0.5) + v[a].x) * dx1, x2 = (((double)cell[a].y + 0.5) + v[a].y) * dx2;
        x1 = x1 >= L1 ? x1 - L1 : (x1 < 0.0 ? 0.0 : x1);
        x2 = x2 >= L2 ? x2 - L2 : (x2 < 0.0 ? 0.0 : x2);
        x[a] = make_double2(x1, x2);
    }
}

// K-point Gauss--Legendre nodes and weights on [-1, 1] by Newton's method on the
// three-term recurrence of the Legendre polynomials
void gauss_legendre(int n, double *x, double *w)
{
    const double pi = 3.14159265358979323846;
    for (int i = 0; i < n; ++i) {
        double z = std::cos(pi * (i + 0.75) / (n + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int j = 1; j < n; ++j) {
                const double p2 = ((2.0 * j + 1.0) * z * p1 - j * p0) / (j + 1.0);
                p0 = p1;
                p1 = p2;
            }
            double pn = n == 0 ? 1.0 : p1, pm = n == 0 ? 0.0 : p0;
            if (n == 1) { pn = z; pm = 1.0; }
            dp = n * (z * pn - pm) / (z * z - 1.0);
            const double dz = pn / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

}  // namespace
}  // namespace pic

using namespace pic;

struct pic2d_handle {
    pic2d_config cfg{};
    int device = 0, num_sms = 1;
    cudaStream_t stream = nullptr;
    double dx1 = 0.0, dx2 = 0.0;
    int N = 0;
    int2 *cell = nullptr;
    double2 *v = nullptr, *p = nullptr, *d = nullptr, *pk = nullptr;
    double *cache = nullptr;
    double *ex = nullptr, *ey = nullptr, *exk = nullptr, *eyk = nullptr, *ebx = nullptr, *eby = nullptr;
    double *az = nullptr, *TA = nullptr, *TEx = nullptr, *TEy = nullptr;   // A_z; cell polynomials of A_z and e_bar
    double *spin = nullptr, *bz = nullptr, *TB = nullptr;       // pic2d_set_spin
    double *mom = nullptr;                   // moments of both current components, x then y
    double *jx = nullptr, *jy = nullptr, *tx = nullptr, *ty = nullptr;
    double *g1x = nullptr, *g0y = nullptr, *g0x = nullptr, *g1y = nullptr;   // inverse rows
    unsigned long long *bits = nullptr;      // dmax, pmax, emax; then the status word
    int *status = nullptr;                   // (inside bits' allocation)
    unsigned long long *h_bits = nullptr;    // page-locked copy of both
    double *acc = nullptr;
    std::vector<double> m0x, m1x, m0y, m1y;  // 1D mass rows (host) for the field energy
    double gls[5] = {0, 0, 0, 0, 0}, glw[5] = {0, 0, 0, 0, 0};
    pic::HostCopy copy;
    std::string err;
};

static thread_local std::string g_err2d;

static int fail2d(pic2d_handle *h, int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    if (h) h->err = buf;
    else g_err2d = buf;
    return code;
}

#define CK2(call)                                                                        \
    do {                                                                                 \
        cudaError_t e_ = (call);                                                         \
        if (e_ != cudaSuccess) return fail2d(h, PIC_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

static void free2d(pic2d_handle *h)
{
    void *arrs[] = {h->cell, h->v, h->p, h->d, h->pk, h->cache, h->ex, h->ey, h->exk, h->eyk, h->ebx, h->eby,
                    h->az, h->TA, h->TEx, h->TEy, h->mom, h->jx, h->jy, h->tx, h->ty, h->g1x, h->g0y,
                    h->g0x, h->g1y, h->acc, h->bits, h->spin, h->bz, h->TB};
    for (void *a : arrs)
        if (a) cudaFree(a);
    if (h->h_bits) cudaFreeHost(h->h_bits);
}

// full periodic circulant row of the degree-d mass matrix (band folded onto M nodes)
static std::vector<double> mass_row_full(int d, int M, double dx)
{
    std::vector<double> band(d + 1), row(M, 0.0);
    mass_band(d, dx, band.data());
    for (int r = -d; r <= d; ++r) row[((r % M) + M) % M] += band[r < 0 ? -r : r];
    return row;
}

static std::vector<double> inverse_row(int d, int M, double dx)
{
    std::vector<double> band(d + 1), g(M), taps(M);
    mass_band(d, dx, band.data());
    int start = 0, n = 0;
    inverse_taps(band.data(), d, M, 0.0, g.data(), &start, &n, taps.data());
    return g;
}

// the body for the degree K (a compile-time constant in it)
#define PIC2D_DEGREE(K_, ...)                                                             \
    switch (K_) {                                                                         \
    case 2: { constexpr int K = 2; __VA_ARGS__; break; }                                  \
    case 3: { constexpr int K = 3; __VA_ARGS__; break; }                                  \
    case 4: { constexpr int K = 4; __VA_ARGS__; break; }                                  \
    default: { constexpr int K = 5; __VA_ARGS__; break; }                                 \
    }

static Args2D make_args(pic2d_handle *h)
{
    const pic2d_config &c = h->cfg;
    Args2D a{};
    a.M1 = c.M1; a.M2 = c.M2; a.np = c.np; a.dx1 = h->dx1; a.dx2 = h->dx2; a.dt = c.dt; a.w = c.weight;
    a.idx1 = 1.0 / h->dx1; a.idx2 = 1.0 / h->dx2;
    a.cell = h->cell; a.v = h->v; a.cache = h->cache; a.pn = h->p; a.d = h->d; a.pk = h->pk;
    a.TA = h->TA; a.TEx = h->TEx; a.TEy = h->TEy; a.TB = h->TB;
    a.mx = h->mom; a.my = h->mom + (size_t)h->N * c.degree * (c.degree + 1);
    a.hbar = h->spin ? c.hbar : 0.0;
    a.s = h->spin;
    a.dmax_bits = h->bits; a.pmax_bits = h->bits + 1; a.status = h->status;
    for (int g = 0; g < 5; ++g) { a.gls[g] = std::llrint(std::ldexp(h->gls[g], 62)); a.glw[g] = std::llrint(std::ldexp(h->glw[g], 62)); }
    return a;
}

static int marker_grid2d(const pic2d_handle *h) { return (int)std::min<long long>((h->cfg.np + 255) / 256, 8LL * h->num_sms); }

// cell polynomials of e_bar
static int tables_e(pic2d_handle *h)
{
    const pic2d_config &c = h->cfg;
    const dim3 grid((unsigned)(((long long)h->N * c.degree * (c.degree + 1) + 127) / 128), 2);
    PIC2D_DEGREE(c.degree, (k2_table_e<K><<<grid, 128, 0, h->stream>>>(c.M1, c.M2, h->ebx, h->eby, h->TEx, h->TEy)))
    CK2(cudaGetLastError());
    return PIC_OK;
}

// e^(k+1) = e^n - M1^{-1} j from the sweep's moments, its increment, e_bar and its polynomials
static int solve2d(pic2d_handle *h)
{
    const pic2d_config &c = h->cfg;
    const Args2D a = make_args(h);
    const dim3 grid((h->N + 63) / 64, 2), circ((h->N + kCirc - 1) / kCirc, 2);
    cudaStream_t s = h->stream;
    PIC2D_DEGREE(c.degree, (k2_nodes<K><<<grid, 64, 0, s>>>(c.M1, c.M2, a.mx, a.my, h->jx, h->jy)))
    // along x2 with the rows of component x's N^k and y's N^{k-1}, then along x1
    k2_circ2<<<circ, 4 * kCirc, 0, s>>>(c.M1, c.M2, h->g0y, h->g1y, h->jx, h->jy, h->tx, h->ty);
    k2_circ1<<<circ, 4 * kCirc, 0, s>>>(c.M1, c.M2, h->g1x, h->g0x, h->tx, h->ty, h->ex, h->ey, h->exk, h->eyk, h->ebx, h->eby,
                                 h->bits + 2);
    CK2(cudaGetLastError());
    return tables_e(h);
}

extern "C" int pic2d_init(const pic2d_config *cfg, const double *x, const double *p, const double *ex,
                          const double *ey, const double *az, int32_t mem, void *stream, pic2d_handle **out)
{
    if (!cfg || !x || !p || !ex || !ey || !az || !out) return fail2d(nullptr, PIC_ERR_INVALID, "null argument");
    *out = nullptr;
    const pic2d_config &c = *cfg;
    if (!(c.L1 > 0.0) || !(c.L2 > 0.0) || c.M1 < 1 || c.M2 < 1 || (long long)c.M1 * c.M2 > kMax2DNodes ||
        c.degree < 2 || c.degree > 5 || c.np < 1 || !(c.dt > 0.0) || !(c.tol > 0.0) || c.max_iter < 1 ||
        (c.warm != 0 && c.warm != 1) ||
        !std::isfinite(c.weight) || !std::isfinite(c.hbar) || (mem != PIC_MEM_HOST && mem != PIC_MEM_DEVICE))
        return fail2d(nullptr, PIC_ERR_INVALID, "bad 2D configuration");
    pic2d_handle *h = new (std::nothrow) pic2d_handle();
    if (!h) return fail2d(nullptr, PIC_ERR_NOMEM, "handle");
    h->cfg = c;
    h->stream = (cudaStream_t)stream;
    cudaGetDevice(&h->device);
    h->dx1 = c.L1 / c.M1;
    h->dx2 = c.L2 / c.M2;
    h->N = c.M1 * c.M2;
    const size_t np = (size_t)c.np, N = (size_t)h->N;
    auto bail = [&](int rc) {
        g_err2d = h->err.empty() ? "pic2d_init failed" : h->err;
        free2d(h);
        delete h;
        return rc;
    };
    cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
    const int K = c.degree;
    struct { void **p; size_t bytes; } allocs[] = {
        {(void **)&h->cell, np * sizeof(int2)}, {(void **)&h->v, np * sizeof(double2)},
        {(void **)&h->p, np * sizeof(double2)}, {(void **)&h->d, np * sizeof(double2)},
        {(void **)&h->pk, np * sizeof(double2)}, {(void **)&h->cache, np * (K + 2) * sizeof(double)},
        {(void **)&h->TA, N * pad2((K + 1) * (K + 1)) * sizeof(double)},
        {(void **)&h->TEx, N * pad2(K * (K + 1)) * sizeof(double)},
        {(void **)&h->TEy, N * pad2(K * (K + 1)) * sizeof(double)},
        {(void **)&h->mom, 2 * N * K * (K + 1) * sizeof(double)},
        {(void **)&h->g1x, c.M1 * sizeof(double)}, {(void **)&h->g0x, c.M1 * sizeof(double)},
        {(void **)&h->g0y, c.M2 * sizeof(double)}, {(void **)&h->g1y, c.M2 * sizeof(double)},
        {(void **)&h->bits, 4 * sizeof(unsigned long long)}, {(void **)&h->acc, 2 * sizeof(double)}};
    for (auto &al : allocs)
        if (cudaMalloc(al.p, al.bytes) != cudaSuccess) return bail(PIC_ERR_NOMEM);
    double **grids[] = {&h->ex, &h->ey, &h->exk, &h->eyk, &h->ebx, &h->eby, &h->az, &h->jx, &h->jy, &h->tx, &h->ty};
    for (double **a : grids)
        if (cudaMalloc((void **)a, N * sizeof(double)) != cudaSuccess) return bail(PIC_ERR_NOMEM);
    h->status = reinterpret_cast<int *>(h->bits + 3);
    if (cudaMallocHost((void **)&h->h_bits, 4 * sizeof(unsigned long long)) != cudaSuccess) return bail(PIC_ERR_NOMEM);
    // positions must lie in the box
    const cudaMemcpyKind kind = mem == PIC_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    if (mem == PIC_MEM_HOST) {
        for (size_t a = 0; a < np; ++a)
            if (!(x[2 * a] >= 0.0 && x[2 * a] < c.L1 && x[2 * a + 1] >= 0.0 && x[2 * a + 1] < c.L2) ||
                !std::isfinite(p[2 * a]) || !std::isfinite(p[2 * a + 1])) {
                fail2d(h, PIC_ERR_INVALID, "marker %zu outside the box or not finite", a);
                return bail(PIC_ERR_INVALID);
            }
    }
    // the positions pass through the displacement array
    if (cudaMemcpyAsync(h->d, x, np * sizeof(double2), kind, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(h->p, p, np * sizeof(double2), kind, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(h->ex, ex, N * sizeof(double), kind, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(h->ey, ey, N * sizeof(double), kind, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(h->az, az, N * sizeof(double), kind, h->stream) != cudaSuccess)
        return bail(fail2d(h, PIC_ERR_CUDA, "input copies"));
    k2_load<<<marker_grid2d(h), 256, 0, h->stream>>>(c.np, c.M1, c.M2, h->dx1, h->dx2, h->d, h->cell, h->v);
    PIC2D_DEGREE(c.degree, (k2_table<K, K><<<(unsigned)((N * Dim2<K>::nA + 127) / 128), 128, 0, h->stream>>>(
                               c.M1, c.M2, h->az, h->TA, Dim2<K>::pA)))
    if (cudaGetLastError() != cudaSuccess) return bail(fail2d(h, PIC_ERR_CUDA, "input kernels"));
    {
        std::vector<double> g1x = inverse_row(c.degree - 1, c.M1, h->dx1), g0x = inverse_row(c.degree, c.M1, h->dx1);
        std::vector<double> g1y = inverse_row(c.degree - 1, c.M2, h->dx2), g0y = inverse_row(c.degree, c.M2, h->dx2);
        h->m0x = mass_row_full(c.degree, c.M1, h->dx1);
        h->m1x = mass_row_full(c.degree - 1, c.M1, h->dx1);
        h->m0y = mass_row_full(c.degree, c.M2, h->dx2);
        h->m1y = mass_row_full(c.degree - 1, c.M2, h->dx2);
        if (cudaMemcpyAsync(h->g1x, g1x.data(), c.M1 * sizeof(double), cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
            cudaMemcpyAsync(h->g0x, g0x.data(), c.M1 * sizeof(double), cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
            cudaMemcpyAsync(h->g1y, g1y.data(), c.M2 * sizeof(double), cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
            cudaMemcpyAsync(h->g0y, g0y.data(), c.M2 * sizeof(double), cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
            cudaStreamSynchronize(h->stream) != cudaSuccess)
            return bail(fail2d(h, PIC_ERR_CUDA, "grid uploads"));
    }
    gauss_legendre(c.degree, h->gls, h->glw);
    for (int g = 0; g < c.degree; ++g) {        // on [0, 1]
        h->gls[g] = 0.5 * (1.0 + h->gls[g]);
        h->glw[g] *= 0.5;
    }
    *out = h;
    return PIC_OK;
}

extern "C" int pic2d_substep1(pic2d_handle *h, int32_t *iters)
{
    if (!h) return PIC_ERR_INVALID;
    const pic2d_config &c = h->cfg;
    if (c.hbar != 0.0 && !h->spin)
        return fail2d(h, PIC_ERR_INVALID, "hbar != 0: pic2d_set_spin must give the spins and b_z first");
    const size_t np = (size_t)c.np, N = (size_t)h->N;
    const size_t mom_bytes = 2 * N * c.degree * (c.degree + 1) * sizeof(double);
    cudaStream_t s = h->stream;
    CK2(cudaMemsetAsync(h->d, 0, np * sizeof(double2), s));
    CK2(cudaMemcpyAsync(h->pk, h->p, np * sizeof(double2), cudaMemcpyDeviceToDevice, s));
    double *copies[][2] = {{h->exk, h->ex}, {h->eyk, h->ey}, {h->ebx, h->ex}, {h->eby, h->ey}};
    for (auto &q : copies) CK2(cudaMemcpyAsync(q[0], q[1], N * sizeof(double), cudaMemcpyDeviceToDevice, s));
    CK2(cudaMemsetAsync(h->bits, 0, 4 * sizeof(unsigned long long), s));
    Args2D a = make_args(h);
    const int grid = marker_grid2d(h);
    int rc, it = 0;
    const bool warm = c.warm != 0;
    if (warm) {
        // the predicted start: delta^(0) and its current, then e^(0) = e^n - M1^{-1} j^(0)
        // and e_bar = (e^n + e^(0)) / 2 for the first sweep
        CK2(cudaMemsetAsync(h->mom, 0, mom_bytes, s));
        PIC2D_DEGREE(c.degree, (k2_sweep<K, true><<<std::min(grid, sweep2d_blocks<K> * h->num_sms), 256, 0, s>>>(a)))
        CK2(cudaGetLastError());
        if ((rc = solve2d(h))) return rc;
    } else if ((rc = tables_e(h))) {
        return rc;
    }
    for (;;) {
        CK2(cudaMemsetAsync(h->mom, 0, mom_bytes, s));
        CK2(cudaMemsetAsync(h->bits, 0, 3 * sizeof(unsigned long long), s));
        a.first = !warm && it == 0;          // the predicted start filled the cache already
        PIC2D_DEGREE(c.degree, (k2_sweep<K><<<std::min(grid, sweep2d_blocks<K> * h->num_sms), 256, 0, s>>>(a)))
        CK2(cudaGetLastError());
        if ((rc = solve2d(h))) return rc;
        CK2(cudaMemcpyAsync(h->h_bits, h->bits, 4 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
        CK2(cudaStreamSynchronize(s));
        ++it;
        double dm, pm, em;
        int hs;
        std::memcpy(&dm, &h->h_bits[0], 8);
        std::memcpy(&pm, &h->h_bits[1], 8);
        std::memcpy(&em, &h->h_bits[2], 8);
        std::memcpy(&hs, &h->h_bits[3], sizeof(int));
        if (hs & STATUS_NUMERIC) return fail2d(h, PIC_ERR_NUMERIC, "2D subsystem I: non-finite value or a path beyond %d cells", kMaxCross);
        if (!(dm == dm && pm == pm && em == em)) return fail2d(h, PIC_ERR_NUMERIC, "2D subsystem I: NaN increment");
        if (dm <= c.tol && pm <= c.tol && em <= c.tol) break;
        if (it >= c.max_iter) {
            if (iters) *iters = it;
            return fail2d(h, PIC_ERR_NOCONVERGE, "2D subsystem I: no convergence in %d sweeps", c.max_iter);
        }
    }
    if (iters) *iters = it;
    k2_finalize<<<grid, 256, 0, s>>>(c.np, c.M1, c.M2, h->cell, h->v, h->p, h->d, h->pk);
    CK2(cudaMemcpyAsync(h->ex, h->exk, N * sizeof(double), cudaMemcpyDeviceToDevice, s));
    CK2(cudaMemcpyAsync(h->ey, h->eyk, N * sizeof(double), cudaMemcpyDeviceToDevice, s));
    CK2(cudaGetLastError());
    CK2(cudaStreamSynchronize(s));
    return PIC_OK;
}

// e^T (A (x) B) e / 2 with circulant rows a (M1) and b (M2), on the host
static double kron_quad(const std::vector<double> &e, const std::vector<double> &ra, const std::vector<double> &rb,
                        int M1, int M2)
{
    double s = 0.0;
    for (int i1 = 0; i1 < M1; ++i1)
        for (int i2 = 0; i2 < M2; ++i2) {
            double v = 0.0;
            for (int q1 = 0; q1 < M1; ++q1) {
                const double ca = ra[((q1 - i1) % M1 + M1) % M1];
                if (ca == 0.0) continue;
                for (int q2 = 0; q2 < M2; ++q2) v += ca * rb[((q2 - i2) % M2 + M2) % M2] * e[q1 * M2 + q2];
            }
            s += e[i1 * M2 + i2] * v;
        }
    return 0.5 * s;
}

extern "C" int pic2d_energy(pic2d_handle *h, double out[4])
{
    if (!h || !out) return PIC_ERR_INVALID;
    const pic2d_config &c = h->cfg;
    CK2(cudaMemsetAsync(h->acc, 0, 2 * sizeof(double), h->stream));
    const int grid = (int)std::min<long long>((c.np + 255) / 256, 1024);
    const Args2D args = make_args(h);
    PIC2D_DEGREE(c.degree, (k2_energy<K><<<grid, 256, 0, h->stream>>>(args, h->p, h->acc)))
    CK2(cudaGetLastError());
    std::vector<double> ex(h->N), ey(h->N);
    double acc[2] = {0.0, 0.0};
    CK2(cudaMemcpyAsync(acc, h->acc, sizeof(acc), cudaMemcpyDeviceToHost, h->stream));
    CK2(cudaMemcpyAsync(ex.data(), h->ex, h->N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    CK2(cudaMemcpyAsync(ey.data(), h->ey, h->N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    CK2(cudaStreamSynchronize(h->stream));
    const double fe = kron_quad(ex, h->m1x, h->m0y, c.M1, c.M2) + kron_quad(ey, h->m0x, h->m1y, c.M1, c.M2);
    out[0] = acc[0];
    out[1] = fe;
    out[2] = acc[1];
    out[3] = acc[0] + fe + acc[1];
    return PIC_OK;
}

extern "C" int pic2d_set_spin(pic2d_handle *h, const double *s, const double *bz, int32_t mem)
{
    if (!h || !s || !bz || (mem != PIC_MEM_HOST && mem != PIC_MEM_DEVICE)) return PIC_ERR_INVALID;
    const pic2d_config &c = h->cfg;
    const size_t N = (size_t)h->N, n3 = 3 * (size_t)c.np;
    if (!h->spin) {
        double *sp = nullptr, *b0 = nullptr, *tb = nullptr;
        if (cudaMalloc((void **)&sp, n3 * sizeof(double)) != cudaSuccess ||
            cudaMalloc((void **)&b0, N * sizeof(double)) != cudaSuccess ||
            cudaMalloc((void **)&tb, N * pad2(c.degree * c.degree) * sizeof(double)) != cudaSuccess) {
            for (double *q : {sp, b0, tb})
                if (q) cudaFree(q);
            return fail2d(h, PIC_ERR_NOMEM, "spin and b_z arrays");
        }
        h->spin = sp;
        h->bz = b0;
        h->TB = tb;
    }
    const cudaMemcpyKind kind = mem == PIC_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    std::vector<double> b(N);
    CK2(cudaMemcpyAsync(h->spin, s, n3 * sizeof(double), kind, h->stream));
    CK2(cudaMemcpyAsync(h->bz, bz, N * sizeof(double), kind, h->stream));
    CK2(cudaMemcpyAsync(b.data(), h->bz, N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    CK2(cudaStreamSynchronize(h->stream));
    for (size_t i = 0; i < N; ++i)
        if (!std::isfinite(b[i])) return fail2d(h, PIC_ERR_INVALID, "b_z not finite at node %zu", i);
    PIC2D_DEGREE(c.degree, (k2_table<K - 1, K - 1><<<(unsigned)((N * Dim2<K>::nB + 127) / 128), 128, 0, h->stream>>>(
                               c.M1, c.M2, h->bz, h->TB, Dim2<K>::pB)))
    CK2(cudaGetLastError());
    CK2(cudaStreamSynchronize(h->stream));
    return PIC_OK;
}

extern "C" int pic2d_get_state(pic2d_handle *h, double *x, double *p, double *ex, double *ey, int32_t mem)
{
    if (!h || (mem != PIC_MEM_HOST && mem != PIC_MEM_DEVICE)) return PIC_ERR_INVALID;
    const cudaMemcpyKind kind = mem == PIC_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    const size_t bytes = (size_t)h->cfg.np * sizeof(double2), N = (size_t)h->N;
    // markers to the host: by several threads where the memory is pageable
    auto markers = [&](double *dst, const double2 *src) -> int {
        if (mem == PIC_MEM_HOST) {
            cudaPointerAttributes at{};
            const bool pageable = cudaPointerGetAttributes(&at, dst) != cudaSuccess || at.type == cudaMemoryTypeUnregistered;
            cudaGetLastError();
            if (pageable) {
                CK2(cudaStreamSynchronize(h->stream));
                if (h->copy.run(dst, src, bytes, h->device)) return PIC_OK;
            }
        }
        CK2(cudaMemcpyAsync(dst, src, bytes, kind, h->stream));
        return PIC_OK;
    };
    int rc;
    if (x) {
        // host positions pass through the displacement array (free between substeps)
        double2 *dst = mem == PIC_MEM_HOST ? h->d : reinterpret_cast<double2 *>(x);
        k2_store<<<marker_grid2d(h), 256, 0, h->stream>>>(h->cfg.np, h->cfg.L1, h->cfg.L2, h->dx1, h->dx2, h->cell, h->v, dst);
        CK2(cudaGetLastError());
        if (mem == PIC_MEM_HOST && (rc = markers(x, dst))) return rc;
    }
    if (p && (rc = markers(p, h->p))) return rc;
    if (ex) CK2(cudaMemcpyAsync(ex, h->ex, N * sizeof(double), kind, h->stream));
    if (ey) CK2(cudaMemcpyAsync(ey, h->ey, N * sizeof(double), kind, h->stream));
    CK2(cudaStreamSynchronize(h->stream));
    return PIC_OK;
}

extern "C" int pic2d_destroy(pic2d_handle *h)
{
    if (!h) return PIC_OK;
    if (h->stream) cudaStreamSynchronize(h->stream);
    free2d(h);
    delete h;
    return PIC_OK;
}

extern "C" const char *pic2d_last_error(const pic2d_handle *h)
{
    return h ? h->err.c_str() : g_err2d.c_str();
}
