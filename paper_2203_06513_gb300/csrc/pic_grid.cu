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
#include "pic_solve.cuh"

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

// the body for the degree K (a compile-time constant in it)
#define PIC_FOR_DEGREE(K_, ...)                                                           \
    switch (K_) {                                                                         \
    case 2: { constexpr int K = 2; __VA_ARGS__; break; }                                  \
    case 3: { constexpr int K = 3; __VA_ARGS__; break; }                                  \
    case 4: { constexpr int K = 4; __VA_ARGS__; break; }                                  \
    case 5: { constexpr int K = 5; __VA_ARGS__; break; }                                  \
    default: break;                                                                       \
    }

template <int K>
__global__ void __launch_bounds__(kConvThreads) k_conv(ConvArgs A)
{
    extern __shared__ __align__(16) double s_conv[];
    conv_block<K>(A, A.node[blockIdx.y], A.T, conv_iter(A), blockIdx.x, blockIdx.y, s_conv, nullptr);
}

// Batched solves of an ensemble: block (bx, run, comp).  Runs that are not in
// the current sweep (converged, or stopped by an error) are skipped.  After a
// run's decision, the last run to decide in this sweep records whether any run
// goes on, and sets the loop's conditional handle (graph mode).
template <int K>
__global__ void __launch_bounds__(kConvThreads) k_conv_ens(const ConvArgs *runs, EnsQueue *Q, int *sweeps,
                                                           unsigned long long cond)
{
    extern __shared__ __align__(16) double s_conv[];
    const int r = blockIdx.y, comp = blockIdx.z;
    const ConvArgs &A = runs[r];
    if (A.mode != CONV_PLAIN && !Q->active[r]) return;
    if (comp >= A.ncomp || (int)blockIdx.x * (kConvOut - K) >= A.M) return;
    const bool last = conv_block<K>(A, A.node[comp], A.T, conv_iter(A), blockIdx.x, comp, s_conv, nullptr);
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

// The nodes of a solve of subsystem II, each formed once (ConvArgs::node).
constexpr int kNodeThreads = 64;

template <int K>
__global__ void __launch_bounds__(kNodeThreads) k_nodes(ConvArgs A)
{
    node_pass<K>(A, conv_iter(A), blockIdx.x * kNodeThreads + threadIdx.x, blockIdx.y);
}

template <int K>
__global__ void __launch_bounds__(kNodeThreads) k_nodes_ens(const ConvArgs *runs, const EnsQueue *Q)
{
    if (!Q->active[blockIdx.y]) return;
    const ConvArgs &A = runs[blockIdx.y];
    node_pass<K>(A, conv_iter(A), blockIdx.x * kNodeThreads + threadIdx.x, blockIdx.z);
}

long long conv_node_ops(int M, int K, int ntap)
{
    return 2LL * conv_blocks(M, K) * (kConvOut + ntap - 1) * (K + 1) * (K + 1);
}

// Inverse rows that decay slowly (large dt/dx in subsystem II) may keep as many taps as
// nodes, which takes more shared memory than the default.
static SmemOptin g_conv_optin[kMaxDegree + 1], g_conv_ens_optin[kMaxDegree + 1];

// raise the shared-memory limit of k_conv_ens before any capture of it
int conv_ens_optin(int K_, int ntap1, int ntap2, bool nodes)
{
    const size_t smem = std::max(conv_smem(K_, ntap1, false), conv_smem(K_, ntap2, nodes));
    PIC_FOR_DEGREE(K_, return g_conv_ens_optin[K].raise((const void *)k_conv_ens<K>, smem) ? 0 : 1)
    return 1;
}

int launch_conv_ens(const ConvArgs *runs, int nruns, int Mmax, int K_, int ncomp, int ntap_max, bool nodes, EnsQueue *Q,
                    int *sweeps, unsigned long long cond, cudaStream_t s)
{
    const size_t smem = conv_smem(K_, ntap_max, nodes);
    if (!g_conv_ens_optin[K_].allowed(smem)) return 1;   // conv_ens_optin first
    if (nodes) {
        const dim3 ngrid((Mmax + kNodeThreads - 1) / kNodeThreads, nruns, ncomp);
        PIC_FOR_DEGREE(K_, (k_nodes_ens<K><<<ngrid, kNodeThreads, 0, s>>>(runs, Q)))
    }
    dim3 grid(conv_blocks(Mmax, K_), nruns, ncomp);
    PIC_FOR_DEGREE(K_, (k_conv_ens<K><<<grid, kConvThreads, smem, s>>>(runs, Q, sweeps, cond)))
    return 0;
}

int launch_conv(const ConvArgs &a, cudaStream_t s)
{
    const size_t smem = conv_smem(a.K, a.ntap, a.node[0] != nullptr);
    const dim3 grid(conv_blocks(a.M, a.K), a.ncomp), ngrid((a.M + kNodeThreads - 1) / kNodeThreads, a.ncomp);
    PIC_FOR_DEGREE(a.K, {
        if (!g_conv_optin[K].raise((const void *)k_conv<K>, smem)) return 1;
        if (a.node[0]) k_nodes<K><<<ngrid, kNodeThreads, 0, s>>>(a);
        k_conv<K><<<grid, kConvThreads, smem, s>>>(a);
    })
    return 0;
}

// preparation WHICH, task t = blockIdx.x blockDim.x + threadIdx.x = (q, cell), cells fastest
template <int K, int WHICH>
__device__ __forceinline__ void prep_thread(int t, const RunDesc &R)
{
    constexpr int n = WHICH == 1 ? prep1_tasks<K> : prep2_tasks<K>;
    const int q = t / R.M, i = t - q * R.M;
    if (q >= n) return;
    if (WHICH == 1) prep1_task<K>(i, q, R);
    else prep2_task<K>(i, q, R);
}

template <int K, int WHICH>
__global__ void __launch_bounds__(128) k_prep(RunDesc R)
{
    prep_thread<K, WHICH>(blockIdx.x * blockDim.x + threadIdx.x, R);
}

template <int K, int WHICH>
__global__ void __launch_bounds__(128) k_prep_ens(const RunDesc *runs)
{
    prep_thread<K, WHICH>(blockIdx.x * blockDim.x + threadIdx.x, runs[blockIdx.y]);
}

template <int K, int WHICH>
static int prep_grid(int M)
{
    return (M * (WHICH == 1 ? prep1_tasks<K> : prep2_tasks<K>) + 127) / 128;
}

int launch_prep1_ens(const RunDesc *R, int nruns, int K_, int Mmax, cudaStream_t s)
{
    PIC_FOR_DEGREE(K_, (k_prep_ens<K, 1><<<dim3(prep_grid<K, 1>(Mmax), nruns), 128, 0, s>>>(R)))
    return 0;
}

int launch_prep1(const RunDesc &R, cudaStream_t s)
{
    PIC_FOR_DEGREE(R.K, (k_prep<K, 1><<<prep_grid<K, 1>(R.M), 128, 0, s>>>(R)))
    return 0;
}

int launch_prep2_ens(const RunDesc *R, int nruns, int K_, int Mmax, cudaStream_t s)
{
    PIC_FOR_DEGREE(K_, (k_prep_ens<K, 2><<<dim3(prep_grid<K, 2>(Mmax), nruns), 128, 0, s>>>(R)))
    return 0;
}

int launch_prep2(const RunDesc &R, cudaStream_t s)
{
    PIC_FOR_DEGREE(R.K, (k_prep<K, 2><<<prep_grid<K, 2>(R.M), 128, 0, s>>>(R)))
    return 0;
}

__global__ void k_commit(RunDesc R, int which) 
{
    commit_at(blockIdx.x * blockDim.x + threadIdx.x, R, which, R.ctrl->iter - 1);
}

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
    commit_at(blockIdx.x * blockDim.x + threadIdx.x, R, which, R.ctrl->iter - 1);
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

template <int K>
__global__ void k_path_nodes(int M, double scale, const double *mom, const double *mom0, const int *flux, double *out)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    out[j] = scale * path_node_value<K>(
                         [&](int r, int m) {
                             const size_t q = (size_t)wrap_cell(j + r, M) * K + m;
                             return mom[q] - mom0[q];
                         },
                         [&](int r) { return flux[wrap_cell(j + r, M)]; });
}

int launch_path_nodes(int M, int K_, double scale, const double *mom, const double *mom0, const int *flux, double *out,
                      cudaStream_t s)
{
    PIC_FOR_DEGREE(K_, (k_path_nodes<K><<<(M + 63) / 64, 64, 0, s>>>(M, scale, mom, mom0, flux, out)))
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

template <int D>
__global__ void k_cell_coefs(int M, bool path, const double *c, double *tab)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x, i = t / (D + 1), m = t % (D + 1);
    if (i >= M) return;
    const double v = cell_coef<D>(m, [&](int r) { return c[wrap_cell(i - r, M)]; });
    tab[(size_t)i * coef_pad(0, D + 1) + m] = path ? v / (double)(m + 1) : v;
}

int launch_cell_coefs(int M, int D, bool path, const double *c, double *tab, cudaStream_t s)
{
    const int grid = (M * (D + 1) + 127) / 128;
    switch (D) {
    case 1: k_cell_coefs<1><<<grid, 128, 0, s>>>(M, path, c, tab); break;
    case 2: k_cell_coefs<2><<<grid, 128, 0, s>>>(M, path, c, tab); break;
    case 3: k_cell_coefs<3><<<grid, 128, 0, s>>>(M, path, c, tab); break;
    case 4: k_cell_coefs<4><<<grid, 128, 0, s>>>(M, path, c, tab); break;
    case 5: k_cell_coefs<5><<<grid, 128, 0, s>>>(M, path, c, tab); break;
    default: return 1;
    }
    return 0;
}

template <int K>
__global__ void k_tables2(int M, int fp32, const double *an_y, const double *an_z, const double *ak_y,
                          const double *ak_z, CoefTables T)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x, i = t / (2 * (K + 1)), c = t / (K + 1) & 1, m = t % (K + 1);
    if (i >= M) return;
    const double *a = c ? an_z : an_y, *b = c ? ak_z : ak_y;
    const int pad = coef_pad(fp32, K + 1);
    const size_t row = 2 * (size_t)i + c;
    const double n = cell_coef<K>(m, [&](int r) { return a[wrap_cell(i - r, M)]; });
    const double k = cell_coef<K>(m, [&](int r) { return b[wrap_cell(i - r, M)]; });
    put_coef(T.A, fp32, row, pad, m, n);
    put_coef(T.Kt, fp32, row, pad, m, k);
    if (fp32) T.L[row * pad + m] = sum_residue(n, k);
}

int launch_tables2(int M, int K_, int fp32, const double *an_y, const double *an_z, const double *ak_y,
                   const double *ak_z, CoefTables T, cudaStream_t s)
{
    PIC_FOR_DEGREE(K_, (k_tables2<K><<<(M * 2 * (K + 1) + 127) / 128, 128, 0, s>>>(M, fp32, an_y, an_z, ak_y, ak_z, T)))
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

// Field energies (Eq. discrete_H) and the Gauss-law residual (Remark 2, Sec. 4.2).  The
// potential's energy applies the stiffness as the steps do (by differences): with its rows,
// whose rounding is an operator error of 1e-16 (dx k)^-2, the energy of a run that conserves
// it showed a change of 6e-12 (2048 cells, 1000 steps).
template <int K>
__global__ void k_energy_grid(int M, double dx, const double *rowM0, const double *rowM1, const double *ex,
                              const double *ey, const double *ez, const double *ay, const double *az,
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
        for (int d = 1; d <= K; ++d) {
            const int ip = (i + d) % M, im = (i - d + M) % M;
            m0y += rowM0[d] * (ey[ip] + ey[im]);
            m0z += rowM0[d] * (ez[ip] + ez[im]);
        }
        eex += 0.5 * ex[i] * m1e;
        eperp += 0.5 * (ey[i] * m0y + ez[i] * m0z);
        aperp += 0.5 * (ay[i] * pic::stiffness<K>(ay, i, M, rowM1, dx) + az[i] * pic::stiffness<K>(az, i, M, rowM1, dx));
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

int launch_energy_grid(int M, int K_, double dx, const double *rowM0, const double *rowM1, const double *ex,
                       const double *ey, const double *ez, const double *ay, const double *az, const double *rho,
                       double *diag, cudaStream_t s)
{
    PIC_FOR_DEGREE(K_, (k_energy_grid<K><<<1, 256, 0, s>>>(M, dx, rowM0, rowM1, ex, ey, ez, ay, az, rho, diag)))
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

__global__ void k_spin_source(int M, int K, double c, const double *mom_y, const double *mom_z, double *by, double *bz)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < 2 * M) pic::spin_source_at(M, K, c, mom_y, mom_z, by, bz, q % M, q / M);
}

namespace pic {
int launch_spin_source(int M, int K, double c, const double *mom_y, const double *mom_z, double *by, double *bz,
                       cudaStream_t s)
{
    k_spin_source<<<(2 * M + 63) / 64, 64, 0, s>>>(M, K, c, mom_y, mom_z, by, bz);
    return 0;
}

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
