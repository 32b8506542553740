// pic_handle.h -- the state behind a pic_handle (private to libpic).
#pragma once

#include <string>
#include <utility>
#include <vector>

#include "pic.h"
#include "pic_hostcopy.h"
#include "pic_internal.h"

using pic::PartPtrs;
using pic::DevCtrl;
using pic::kSweepThreads;
using pic::CoefTables;

struct pic_handle {
    pic_config cfg{};
    cudaStream_t stream = nullptr;
    int device = 0, num_sms = 0;
    int M = 0, K = 0, Dlim = 0, fp32 = 0;
    int acc = 0;                    // deposit window accumulator of the sweeps (pic::ACC_*)
    long long np = 0;
    double dx = 0.0;
    size_t rsize = 8;               // bytes of one particle real
    long long steps_done = 0;

    // marker state: two copies of (cell, t, p, id) for the counting sort
    PartPtrs P[2]{};
    // one device block per copy holds its four arrays; between sorts the copy not
    // in use (P[1 - cur]) is free, and the host transfers stage doubles in it
    char *Pblk[2] = {nullptr, nullptr};
    int cur = 0;
    void *delta = nullptr, *pnew = nullptr;
    void *a0 = nullptr;             // start-point cache of a fixed-point loop (4 reals a marker; FP64 form)
    // spin (hbar != 0, FP64 form): components in caller order, and the spin deposits
    double *spx = nullptr, *spy = nullptr, *spz = nullptr;
    double *sdy = nullptr, *sdz = nullptr;      // spin moments, M x K each

    // split run: the markers of one plasma spread over several processes; marker
    // sums and maxima go through this reduction (NULL: all markers are here)
    pic_reduce_fn reduce = nullptr;
    void *rctx = nullptr;
    double *red = nullptr;          // 4 doubles: packed control entries

    // one step as a CUDA graph with device-ended loops (one per marker copy cur)
    cudaGraphExec_t step_exec[2] = {nullptr, nullptr};
    int step_graph_nodes[2] = {0, 0};   // kernel nodes outside the loops
    cudaStream_t cap = nullptr;         // private capture stream
    int *d_count = nullptr;             // sweeps of subsystems I and II (graph mode)
    int *h_count = nullptr;             // pinned readback of d_count
    int host_steps = 0;                 // steps taken by host loops (the first one opts kernels in)
    pic::SmallSync *small = nullptr;    // barrier of the one-kernel steps of small plasmas
    bool small_refused = false;         // the device would not hold their grid at once
    bool lost = false;                  // a one-kernel step gave up at a barrier: no state to go on from

    // grid state (double)
    double *ex = nullptr, *ey = nullptr, *ez = nullptr, *ay = nullptr, *az = nullptr;
    double *ek = nullptr, *ebar = nullptr, *jb[2] = {nullptr, nullptr};
    double *eky = nullptr, *ekz = nullptr, *aky = nullptr, *akz = nullptr;
    double *by = nullptr, *bz = nullptr;
    double *sy[2] = {nullptr, nullptr}, *sz[2] = {nullptr, nullptr};    // node deposits (split runs)
    // moments of the sweeps' deposits (M x K and, per component, M x (K + 1)), by sweep
    // parity, with subsystem I's knot crossings and start-point moments; moments of the
    // deposit entry points; double cell polynomials of the gathers
    int *flux[2] = {nullptr, nullptr};
    double *m0 = nullptr;
    double *m1[2] = {nullptr, nullptr}, *my[2] = {nullptr, nullptr}, *mz[2] = {nullptr, nullptr};
    double *mdep = nullptr, *gtab = nullptr;
    double *rho = nullptr, *work = nullptr, *diag = nullptr;
    double *node = nullptr;         // 2 M: nodes of subsystem II's deposits, formed in a pass of
    bool node_pass = false;         // their own before its solves (long inverse rows)
    int32_t *counts = nullptr;

    // circulant bands and inverse taps
    double *d_rowM0 = nullptr, *d_rowM1 = nullptr;
    double *d_tapM1 = nullptr, *d_tapP = nullptr;
    int tapM1_start = 0, tapM1_n = 0, tapP_start = 0, tapP_n = 0;

    CoefTables T{};                 // cell polynomials of the sweeps' fields
    pic::FieldHist fh{};            // field changes of the last solves (starting fields)
    DevCtrl *ctrl = nullptr;
    DevCtrl *h_ctrl = nullptr;      // pinned: full control block readback

    int grid1 = 0, grid2 = 0;       // blocks of the sweeps of subsystems I and II

    // timing: event pairs recorded around the timed launches, read back (and the
    // pairs reused) by pic_timing_read or when kMaxTimedLaunches are pending
    int timing = 0;
    struct Timed {
        cudaEvent_t b, e;
        int kind;                   // 0 sweep I, 1 sweep II, 2 solve, 3 warm start
    };
    std::vector<Timed> timed;       // pairs in use, in launch order
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> spare;
    double t_sw1 = 0, t_sw2 = 0, t_solve = 0;
    long long n_sw1 = 0, n_sw2 = 0, n_solve = 0, launches = 0, marker_sweeps = 0;

    double t_warm = 0;
    long long n_warm = 0;
    pic_mlp *mlp = nullptr;         // borrowed warm-start network

    pic::HostCopy copy;             // pageable host transfers

    std::string err;
};

namespace pic {
// marker sort of one handle (swaps its current buffer); its current marker arrays
int handle_sort(pic_handle *h);
// room for the nodes of a pass before the solves (pic_handle::node)
int handle_nodes(pic_handle *h);
PartPtrs handle_parts(pic_handle *h);
// the grid-side pointers of one handle (preparation and commit kernels)
RunDesc handle_desc(pic_handle *h);
// kernel arguments of the sweeps and solves of one handle (time step dt of subsystem I)
Sweep1Args make_sweep1_args(pic_handle *h, double dt);
Sweep2Args make_sweep2_args(pic_handle *h);
ConvArgs make_conv1_args(pic_handle *h, double dt);
ConvArgs make_conv2_args(pic_handle *h);
}  // namespace pic
