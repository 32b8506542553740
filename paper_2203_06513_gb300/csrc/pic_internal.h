// pic_internal.h -- launchers shared by the translation units of libpic.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pic_device.cuh"
#include "pic_optin.h"

namespace pic {

// velocity bins of the marker sort key (cell, bin): bins_per_cell bins per cell of
// expected displacement, 16 per cell of it in all (displacements of +-8 cells a step;
// faster markers share the end bins).  Finer bins keep a warp's markers closer
// together after they move (fewer deposit-window misses): measured on C2 (48,828
// markers a cell) with sorting every second step, 64 quarter-cell bins 13.1 ms a step
// against 13.4 ms for 16 whole-cell bins.  With few markers a cell they buy nothing and
// the keys cost the scan time, so sparse runs keep whole cells.
constexpr int kVelBinsBase = 16;
constexpr int kScanTile = 2048;      // keys a block of the sort's scan takes
constexpr size_t sort_counts(size_t nkeys) { return 2 * nkeys + (nkeys + kScanTile - 1) / kScanTile; }
inline int bins_per_cell(long long np, int M) { return np >= 8192LL * M ? 4 : 1; }
// most threads per block of the marker kernels that split their range by warps
constexpr int kSweepThreads = 256;
constexpr int kSweepWarps = kSweepThreads / 32;
// cells a warp's deposit window holds: subsystem I (paths of sorted markers visit two
// or three cells, one more after a step without a sort), subsystem II without and with
// the z component (whose window doubles the registers)
constexpr int kWin1 = 4, kWin2 = 3, kWin2z = 2;
// markers a lane takes per step: two in float, whose steps are bound by issue and the
// latency of their chains; one in double, bound by the FP64 pipe
template <typename R> struct SweepU { static constexpr int v = 1; };
template <> struct SweepU<float> { static constexpr int v = 2; };
// Shape of the sweep kernels: threads a block and resident blocks an SM they are compiled
// for, which set the registers a thread may take (65536 / (threads x blocks)).  The float
// sweeps keep two markers and a window in registers; with fewer registers they spill, with
// more the SM holds too few warps.  Measured, us a launch (sweep I / II; cubic: 1e8
// markers, quintic: 5e7):
//   cubic    256 x 3 (85 registers)  1822 /  607     quintic  256 x 2 (128)  834 / 440
//            256 x 2 (128)            992 /  770              128 x 5 (102)    - / 378
//            128 x 7 (73)               - /  570              128 x 4 (128)  833 / 440
//            128 x 5 (102)           1606 /  662              128 x 3 (170)  624 /   -
// The double form is bound by the FP64 pipe and does not mind (1042 / 303 us for 1e7
// markers, cubic, at 16 warps an SM; with 24 warps sweep I 4 % slower).
template <typename R, int K> struct SweepShape {
    static constexpr int threads1 = 256, blocks1 = 2, threads2 = 256, blocks2 = 2;
};
template <int K> struct SweepShape<float, K> {
    static constexpr int threads1 = K <= 4 ? 256 : 128, blocks1 = K <= 4 ? 2 : 3;
    static constexpr int threads2 = 128, blocks2 = K <= 3 ? 7 : 5;
};

// ---------------------------------------------------------------- particles
struct PartPtrs {
    int32_t *cell;      // cell index in [0, M)
    void *t;            // offset from the cell's centre in [-1/2, 1/2]: float or double
    void *p;            // momentum
    void *delta;        // subsystem-I iterate: displacement x^(k) - x^n, cell units
    void *pnew;         // subsystem-I iterate p^(k+1)
    int32_t *id;        // caller index of each stored marker
};

// Coefficient tables of the sweeps (pic_poly.cuh): per cell one row of the field's
// polynomial in the cell, of the form's real type (float rows are rounded once from
// double coefficients).  Rows are padded for 16-byte loads (coef_pad).
struct CoefTables {
    void *A;            // a^n: y row, z row (K + 1 coefficients each)
    void *E;            // ebar dx, coefficient m divided by m + 1 (K coefficients)
    void *Kt;           // a^(k): y row, z row
    float *L;           // float form: residues of a^n + a^(k) after both roundings
};

struct Sweep1Args {
    int M, Dlim, K, fp32;
    int acc;            // deposit window accumulator (ACC_*)
    long long np;
    double dx, dt;
    PartPtrs P;
    CoefTables T;
    double *mom;        // deposit: M x K moments v, .. v^K of the paths' ends
    int *flux;          // deposit: net crossings (to the right) of the left edge of each cell
    DevCtrl *ctrl;
    int warm;           // 1: delta^(0) = explicit predictor, computed in-kernel (first sweep)
    int first;          // 1: the first sweep of the loop (writes the start-point cache)
    // graph mode (the launch is replayed by a CUDA graph): the deposit buffer is
    // mpair / fpair[iter & 1], and the explicit warm start and the first-sweep role apply
    // when iter == 0, with iter read from ctrl at kernel start
    int graph;
    double *mpair[2];
    int *fpair[2];
    // double form: start-point cache, 4 reals a marker (A_y(x^n), A_z(x^n),
    // gamma(p^n, A(x^n)), unused): written by the loop's first sweep, read by the later
    // ones; NULL: none
    void *a0;
    int zforce;         // 1: treat the z component as present whatever ctrl->zany says
    // spin (double form, hbar != 0): spin components in caller order (indexed by id)
    double hbar;
    const double *sy, *sz;
};

struct Sweep2Args {
    int M, K, fp32;
    int acc;            // deposit window accumulator (ACC_*)
    long long np;
    PartPtrs P;
    CoefTables T;
    double *mom_y, *mom_z;      // deposits: M x (K + 1) moments f v^m (without w)
    int first;
    // graph mode: deposits go to mypair/mzpair[iter & 1], iter read from ctrl
    int graph;
    const DevCtrl *ctrl;
    double *mypair[2], *mzpair[2];
    void *a0;           // double form: (A_y, A_z, gamma) at a^n, as in subsystem I
    int zforce;
};

struct CurrentArgs {
    int M, Dlim, K, fp32;
    long long np;
    double dx;
    PartPtrs P;
    const double *disp;     // caller order, length units
    double *mom;            // M x K moments
    DevCtrl *ctrl;
};

struct DiagArgs {
    int M, K, fp32;
    long long np;
    double dx, w;
    PartPtrs P;
    const double *c0, *c1;  // field coefficients (kinetic: a_y, a_z)
    const double *tab;      // gathers: cell polynomials (launch_cell_coefs)
    double *out;            // gather output (caller order)
    double *mom;            // charge: M x (K + 1) moments
    double *acc;            // kinetic sum
    int Dlim;               // path gathers: largest displacement (cells)
    int *status;            // path gathers: error bits (STATUS_NUMERIC)
};

int launch_sweep1(const Sweep1Args &a, int grid, cudaStream_t s);
// the predicted start of subsystem I: delta^(0) (explicit when a.warm) and its current
// into a.mom; the sweep's launch shape
int launch_predeposit(const Sweep1Args &a, int grid, cudaStream_t s);
int launch_sweep2(const Sweep2Args &a, int grid, cudaStream_t s);
int launch_current(const CurrentArgs &a, int grid, cudaStream_t s);
int launch_charge(const DiagArgs &a, int grid, cudaStream_t s);
int launch_gather(const DiagArgs &a, int field_degree, int grid, int block, cudaStream_t s);
int launch_gather_path(const DiagArgs &a, int grid, int block, cudaStream_t s);
int launch_kinetic(const DiagArgs &a, int grid, int block, cudaStream_t s);
int launch_finalize1(int fp32, long long np, int M, PartPtrs P, bool zero_delta, int grid, int block,
                     cudaStream_t s);
int launch_load(int fp32, long long np, int M, double dx, const double *x, const double *p,
                PartPtrs P, int grid, int block, cudaStream_t s);
int launch_store(int fp32, long long np, int M, double dx, PartPtrs P, double *x, double *p,
                 int grid, int block, cudaStream_t s);
// device destinations of a state: x and p in caller order (NULL: skipped) and n plain arrays
struct StateOut {
    double *x, *p;
    int n;
    double *dst[8];
    const double *src[8];
    long long len[8];
};
int launch_store_state(int fp32, long long np, int M, double dx, PartPtrs P, const StateOut &o, int grid, int block,
                       cudaStream_t s);
// x and p (device) through buckets of caller indices; rec: scratch of 16 (float) or 24
// (double) bytes a marker, cursor: 256 int32
int launch_store_dealt(int fp32, long long np, int M, double dx, PartPtrs P, void *rec, int *cursor, double *x, double *p,
                       cudaStream_t s);
// more markers than this are dealt: their x and p exceed half of L2
constexpr long long kDealMarkers = 1LL << 22;
// the same values in caller order through an inverse permutation (inv: np int32 of
// scratch); consecutive writes, so x and p may be device addresses of page-locked host memory
int launch_store_ordered(int fp32, long long np, int M, double dx, PartPtrs P, int32_t *inv, double *x, double *p,
                         int grid, int block, cudaStream_t s);
int sweep_blocks_per_sm(int K, int fp32, int acc, int which);
// whether the sweep kernels are built for (degree, form, accumulator)
bool sweep_variant_ok(int K, int fp32, int acc);
// one run's counting sort in a batched launch (key: cell * nbins + velocity bin)
struct SortRun {
    long long np;
    int M, nbins;
    float taup;             // dt / dx times the bins per cell
    PartPtrs src, dst;
    int32_t *counts;        // sort_counts(M nbins): histogram, cursors, tile totals
};
constexpr int kSortEnsLaunches = 5;
int launch_sort_ens(int fp32, const SortRun *runs, int nruns, int grid_x, cudaStream_t s);
int launch_sort(int fp32, long long np, int M, double tau, int per, PartPtrs src, PartPtrs dst,
                int32_t *counts, int num_sms, cudaStream_t s);

// ---------------------------------------------------------------- grid
// FP32 form, subsystem I: the last field increment must be below this fraction of
// the field's max-norm.  The momenta of the last sweep were updated with the field
// of the sweep before, so the energy error of a step is proportional to that
// increment.  Started from e^n the field converges from one side and the error has
// one sign, step after step (a drift, measured 1e-12 of the energy a step on C2 at
// 1e-9): 1e-10 is needed.  Started from the field of the proposal (warm_field) the
// last increment's sign varies and 3e-9 leaves no drift.
constexpr double kFieldIncrementRel = 1e-10;
constexpr double kFieldIncrementRelPredicted = 3e-9;

// CONV_START1: e^(0) = e^n - M1^{-1} j^(0) and ebar^(0), without a convergence decision
enum ConvMode { CONV_PLAIN = 0, CONV_SOLVE1 = 1, CONV_SOLVE2 = 2, CONV_START1 = 3 };

struct ConvArgs {
    int M, K, d_start, ntap, mode, ncomp;
    const double *taps;
    // input: the moments of the deposit times scale (subsystem I: mom, mom0 and flux of
    // the paths, II: mom), or nodes (in) where mom is null
    const double *mom[2];
    const double *mom0;     // subsystem I: moments of the start points
    const int *flux;
    const double *in[2];
    double *node[2];        // SOLVE2 with long rows: the nodes, formed once by a pass before the solve
    double scale;
    double *out[2];
    const double *en[2];    // e^n
    double *ek[2];          // e^(k) (in: previous, out: new)
    double *aux[2];         // SOLVE1: ebar out; SOLVE2: a^(k) out
    const double *an[2];    // SOLVE2: a^n
    const double *b[2];     // SOLVE2: right side b of P e = b + dt s
    double *zero[2];        // moments of the next sweep, cleared here
    int *zflux;
    double dt, dx, tol, dtol;
    double erel;        // FP32 subsystem I: field increment tolerance relative to the field's max-norm
    int max_iter, fp32, subsystem;
    DevCtrl *ctrl;
    // graph mode: mom[c] = pair[c][iter & 1], zero[c] = pair[c][(iter + 1) & 1] (flux and
    // zflux from fpair the same way)
    // (iter read from ctrl at kernel start), and the decision sets the loop's
    // conditional handle (1 = run another sweep)
    int graph;
    double *pair[2][2];
    int *fpair[2];
    unsigned long long cond_handle;
    CoefTables T;       // START1 / SOLVE1: E; SOLVE2: Kt, L
    int *count;         // graph mode of single runs: sweeps counted by the decision (or NULL)
};

// the solve, after a pass that forms its nodes when a.node is given (two launches)
int launch_conv(const ConvArgs &a, cudaStream_t s);
// FP64 operations a solve of subsystem II (all runs of an ensemble) spends on its nodes when
// every block forms those of its own tap window: long rows (large dt/dx) repeat a node some
// ntap / (16 - K) times.  From kNodePassOps on the nodes are formed once, in a pass before
// the solve, which costs a launch (or a barrier).  us a step, blocks and pass, double form:
//   M, k, dt/dx    operations   4e3 markers (one kernel)   6e4 (graph)
//   128, 3, 8        0.05e6          164   169               383   388
//   2048, 3, 1       0.60e6          252   249               338   343
//   512, 3, 16       0.68e6          200   189               387   367
//   2048, 3, 4       0.88e6          273   262               364   357
//   2048, 3, 8       1.67e6          301   265               374   348
//   4000, 5, 16      16.9e6          792   506               733   544
//   4000, 5, 64      66.1e6         1725   723              2206   942
long long conv_node_ops(int M, int K, int ntap);
constexpr long long kNodePassOps = 800000;

// ---------------------------------------------------------------- spin (double form)
// Spin components are kept in caller order (sx[id], sy[id], sz[id]).
struct SpinArgs {
    int M, K;
    long long np;
    double dx, w, dt, hbar;
    PartPtrs P;                 // markers in stored order (cell, t as double, id)
    const double *ay, *az;
    double *sx, *sy, *sz;
    double *dy, *dz;            // spin deposit outputs (M x K moments each)
    double *acc;                // Zeeman energy sum (without hbar)
};
// moments sum_a s_y,a v_a^m per cell, s_z likewise: d_y,i = sum_a w s_y,a Lambda^1_i(x_a) follows
// from them (Lambda_1(X)^T W S of subsystem II)
int launch_spin_deposit(const SpinArgs &a, int grid, cudaStream_t s);
// subsystem III: exact rotation of every spin
int launch_spin_rotate(const SpinArgs &a, int grid, cudaStream_t s);
// *acc += sum_a w (s_y dA_z/dx - s_z dA_y/dx)(x_a)
int launch_spin_energy(const SpinArgs &a, int grid, cudaStream_t s);
// b_y -= dt hbar (G^T d_z), b_z += dt hbar (G^T d_y), (G^T v)_j = (v_j - v_{j+1}) / dx
int launch_spin_rhs(int M, double dx, double dt, double hbar, const double *dy, const double *dz,
                    double *by, double *bz, cudaStream_t s);
// the same from the moments
int launch_spin_source(int M, int K, double c, const double *mom_y, const double *mom_z, double *by, double *bz,
                       cudaStream_t s);

// split runs: buf[0..2] = (max increment, numeric bit, timeout bit) of the control block
int launch_split_pack(const DevCtrl *c, double *buf, cudaStream_t s);
int launch_split_unpack(DevCtrl *c, const double *buf, cudaStream_t s);

// ---------------------------------------------------------------- batched ensemble
// Many independent runs advance together: one launch of each kernel covers every
// run.  The particle sweeps are persistent kernels that claim work items (a run
// and a range of item_markers of its markers) from a queue built before each
// sweep from the runs still iterating; grid-side kernels take one block row per run.
constexpr int kEnsMaxRuns = 1024;

struct EnsQueue {
    int next;                // claim counter of the current sweep
    int nitems;              // items of the current sweep
    int nactive;             // runs in the current sweep
    int n_decided;           // runs that took their convergence decision in this sweep
    int n_continue;          // ... and go on
    int go;                  // 1: some run goes on after this sweep
    int item_markers;        // markers per item (a multiple of 1024)
    int share, shares;       // share of shares of a sweep's blocks claim items (the rest leave at once)
    int loops[2];            // sweeps of the loops of subsystems I and II (all runs together)
    int item_start[kEnsMaxRuns + 1];
    int active[kEnsMaxRuns];
};

struct EnsRun {
    long long np;
    DevCtrl *ctrl;
};

// per-run pointers of the grid-side kernels
// Field changes of the last solves of each subsystem (x: subsystem I's e_x; y, z:
// subsystem II's e_y, e_z): d[0] = e^n - e^{n-1}, d[1] = e^{n-1} - e^{n-2}, ...
// order1 / order2: the degree of the time extrapolation that starts each
// subsystem's iteration (0: e^(0) = e^n), at most kMaxStartOrder.
constexpr int kMaxStartOrder = 3;
struct FieldHist {
    double *x[kMaxStartOrder], *y[kMaxStartOrder], *z[kMaxStartOrder];
    int order1, order2;
};

struct RunDesc {
    int M, K, fp32;
    long long np;
    double dx, dt;
    PartPtrs P;
    double *ex, *ek, *ebar, *ay, *az, *m1[2], *m0;   // M x K moments of subsystem I: ends (by sweep parity), starts
    int *flux[2];
    const double *rowM0, *rowM1;
    double *ey, *ez, *by, *bz, *eky, *ekz, *aky, *akz, *my[2], *mz[2];   // M x (K + 1) moments
    DevCtrl *ctrl;
    CoefTables T;
    FieldHist fh;
};

int launch_ens_plan(EnsQueue *Q, const EnsRun *runs, int nruns, unsigned long long cond, cudaStream_t s);
int launch_ens_status(const EnsRun *runs, int nruns, int *status, cudaStream_t s);
int conv_ens_optin(int K, int ntap1, int ntap2, bool nodes);
// nodes: a pass that forms the runs' nodes comes first (ConvArgs::node)
int launch_conv_ens(const ConvArgs *runs, int nruns, int Mmax, int K, int ncomp, int ntap_max, bool nodes, EnsQueue *Q,
                    int *sweeps, unsigned long long cond, cudaStream_t s);
int launch_prep1_ens(const RunDesc *R, int nruns, int K, int Mmax, cudaStream_t s);
int launch_prep2_ens(const RunDesc *R, int nruns, int K, int Mmax, cudaStream_t s);
int launch_commit_ens(const RunDesc *R, int nruns, int Mmax, int which, cudaStream_t s);
int launch_sweep1_ens(int K, int fp32, const Sweep1Args *runs, int nruns, EnsQueue *Q, int grid, cudaStream_t s);
int launch_sweep2_ens(int K, int fp32, const Sweep2Args *runs, int nruns, EnsQueue *Q, int grid, cudaStream_t s);
// the predicted start of every run in the queue (delta^(0) and its current into each run's a.mom)
int launch_predeposit_ens(int K, int fp32, const Sweep1Args *runs, int nruns, EnsQueue *Q, int grid, cudaStream_t s);
int launch_finalize1_ens(int fp32, const RunDesc *R, int nruns, int grid_x, cudaStream_t s);
// ---------------------------------------------------------------- small plasmas
// Whole steps in one cooperative kernel (pic_small.cuh), one marker a thread: up to
// num_sms * kSmallThreads markers.
constexpr int kSmallThreads = 256;
constexpr int kSmallSteps = 256;        // most steps a launch
struct SmallSync {
    // by subsystem and sweep mod 3: marker increment, field increment, field
    unsigned long long maxima[2][3][3];
    unsigned arrived;       // barrier arrivals since the launch (zeroed before it)
    int abort;
};
struct SmallArgs {
    RunDesc d;
    Sweep1Args a1;
    ConvArgs c1, c1p, c2;   // c1p: the predicted start (warm_field)
    int nsteps, strang, warm, warm_field, zero_delta;
    SmallSync *sync;
    double w, hbar;
    double *sx, *sy, *sz;   // spins, caller order (hbar != 0)
    double *sm_y, *sm_z;    // M x K moments of the spin deposit
};
// kSmallRefused: the device does not hold the grid at once (nothing was launched)
constexpr int kSmallRefused = 2;
int launch_small_f32(const SmallArgs &a, int num_sms, cudaStream_t s);
int launch_small_f64(const SmallArgs &a, int num_sms, cudaStream_t s);
int launch_prep1(const RunDesc &R, cudaStream_t s);
int launch_prep2(const RunDesc &R, cudaStream_t s);
// end of a substep (which = 1, 2): the converged iterate becomes the state, and
// its change is recorded for the next starting field
int launch_commit(const RunDesc &R, int which, cudaStream_t s);
// node values of a deposit from its moments of degree D (times scale; path: coefficient m
// divided by m + 1): out[j] = scale sum_r sum_m B_D[r][m] mom[j + r][m]
int launch_moments_to_nodes(int M, int D, bool path, double scale, const double *mom, double *out, cudaStream_t s);
// node values of the path current of subsystem I (ConvArgs: mom, mom0, flux, scale)
int launch_path_nodes(int M, int K, double scale, const double *mom, const double *mom0, const int *flux, double *out,
                      cudaStream_t s);
// start-point moments (m = 1 .. K) from charge moments (m = 0 .. K)
int launch_start_moments(int M, int K, const double *charge, double *mom0, cudaStream_t s);
// double cell polynomials of the degree-D spline with coefficients c (path: m-th divided by m + 1)
int launch_cell_coefs(int M, int D, bool path, const double *c, double *tab, cudaStream_t s);
// the tables of a subsystem-II sweep with given a^n and a^(k) (T.A, T.Kt, T.L)
int launch_tables2(int M, int K, int fp32, const double *an_y, const double *an_z, const double *ak_y,
                   const double *ak_z, CoefTables T, cudaStream_t s);
int launch_poisson_rhs(int M, double dx, const double *rho, double *d, cudaStream_t s);
int launch_energy_grid(int M, int K, double dx, const double *rowM0, const double *rowM1, const double *ex,
                       const double *ey, const double *ez, const double *ay, const double *az, const double *rho,
                       double *diag, cudaStream_t s);
int launch_ctrl_reset(DevCtrl *ctrl, cudaStream_t s);

// learned warm start (pic_mlp.cu)
struct WarmArgs {
    int M, K, fp32;
    long long np;
    double dx, dt;
    PartPtrs P;
    const double *ex;
    const void *coefA;  // a^n's table (CoefTables)
    const float *params, *norm;
    int *status;        // error bits (STATUS_TIMEOUT)
};
int launch_warm_mlp(const WarmArgs &a, int grid, cudaStream_t s);

// message returned by pic_last_error(NULL) on the calling thread
void set_thread_error(const char *msg);

// host-side spline algebra (exact rows and inverse taps of the circulant matrices)
void mass_band(int d, double dx, double *band /* d+1 */);
void inverse_taps(const double *band, int bw, int M, double cut, double *g_full /* M */,
                  int *d_start, int *ntap, double *taps /* M */);

}  // namespace pic
