// pic_small.cuh -- whole time steps of a small plasma in one cooperative kernel.
//
// A step is some twenty dependent launches (each fixed-point sweep, its solve, the
// preparations), and with fewer markers than the GPU has threads each of them takes less
// time than starting it and waiting for its chains of dependent loads.  Here a thread owns
// one marker, whose position, momentum and field coefficients stay in registers over the
// loops and from step to step; the solves are shared out over the blocks; and a barrier over
// the grid stands where the step graph has a kernel boundary.  Every block takes the
// convergence decision itself from the published maxima, so no block waits for one that
// decides.  Spin runs take the same kernel: their source is deposited while the markers are
// moved, the rotation follows subsystem II, and neither needs a barrier of its own.
//
// The barrier is bounded: a block that waits longer than its limit sets STATUS_TIMEOUT
// and an abort flag, and every block returns at its next barrier.  The launch is
// cooperative, so all blocks are resident; where the device does not hold them at once (fewer
// SMs for this process than it reports) the launch is refused and the steps go on as graphs.
#pragma once

#include <algorithm>

#include "pic_internal.h"
#include "pic_poly.cuh"
#include "pic_solve.cuh"
#include "pic_sweep.cuh"

namespace pic {

namespace {

constexpr unsigned kBarrierTries = 1u << 22;        // polls of about a microsecond

// Counts arrivals since the launch (the host zeroes it): generation g is complete at
// g * gridDim.x.  Returns false after a timeout here or elsewhere.
__device__ __forceinline__ bool grid_barrier(SmallSync *S, unsigned &gen, DevCtrl *ctrl)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ++gen;
        const unsigned target = gen * gridDim.x;
        __threadfence();
        atomicAdd(&S->arrived, 1u);
        bool ok = false;
        for (unsigned i = 0; i < kBarrierTries; ++i) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&S->arrived) : "memory");
            if ((int)(v - target) >= 0) { ok = true; break; }
            if ((i & 1023) == 1023 && *reinterpret_cast<volatile int *>(&S->abort)) break;
        }
        if (!ok) {
            atomicOr(&ctrl->status, STATUS_TIMEOUT);
            atomicExch(&S->abort, 1);
        }
        __threadfence();
        s_ok = ok ? 1 : 0;
    }
    __syncthreads();
    return s_ok != 0;
}

// What a loop's decision carries from sweep to sweep (thread 0 of every block, the same in
// all of them).
struct LoopState {
    double dprev, eprev;
    int it;                 // sweeps done
    bool failed;            // a marker went bad in this launch, or an error was there before it
    __device__ __forceinline__ void reset()
    {
        dprev = eprev = bits_to_double(0x7ff0000000000000ull);
        it = 0;
    }
};

// After the barrier behind the solve of sweep L.it: true when the loop ends.  Each
// subsystem has its maxima, slot s of them for the sweeps s, s + 3, ..: the slot of the next
// sweep is cleared two barriers before it is used, and a subsystem's slots after the
// barrier that ends it (a slower block may be reading them until then).  A marker that goes
// bad publishes a NaN increment in the sweep's slot: the control block's status is for the
// host alone, since a block that has gone on to the next sweep may set its bits before a slower
// one has taken this decision, and all have to take the same.
__device__ __forceinline__ bool loop_decision(const ConvArgs &C, unsigned long long (*maxima)[3], LoopState &L)
{
    __shared__ int s_stop;
    if (threadIdx.x == 0) {
        const int slot = L.it % 3;
        volatile unsigned long long *m = maxima[slot];
        const unsigned long long moved = m[0];
        const double d = bits_to_double(moved), e = bits_to_double(m[1]), mag = bits_to_double(m[2]);
        L.it += 1;
        bool stop = fixed_point_reached(C, L.it, d, L.dprev, e, L.eprev, mag);
        if (!stop && L.it >= C.max_iter) {
            stop = true;
            if (blockIdx.x == 0) atomicOr(&C.ctrl->status, STATUS_NOCONV);
        }
        L.failed = L.failed || moved > 0x7ff0000000000000ull;     // a NaN
        if (L.failed) stop = true;
        L.dprev = d;
        L.eprev = e;
        if (blockIdx.x == 0) {
            if (C.count) *C.count += 1;
            volatile unsigned long long *z = maxima[(slot + 2) % 3];
            z[0] = z[1] = z[2] = 0ull;
        }
        s_stop = stop ? 1 : 0;
    } else {
        L.it += 1;
    }
    __syncthreads();
    return s_stop != 0;
}

// Subsystem III from the coefficients of a^{n+1} in the marker's cell.
template <int K>
__device__ __forceinline__ void spin_rotate_one(const SmallArgs &A, const double (&cy)[K + 1], const double (&cz)[K + 1],
                                                double v, int id)
{
    double Y = K * cy[K], Z = K * cz[K];
#pragma unroll
    for (int m = K - 1; m >= 1; --m) {
        Y = fma(Y, v, m * cy[m]);
        Z = fma(Z, v, m * cz[m]);
    }
    spin_turn(A.d.dt, Y / A.d.dx, Z / A.d.dx, A.sx[id], A.sy[id], A.sz[id]);
}

template <int K, typename R>
__global__ void __launch_bounds__(kSmallThreads, 1) k_small(const __grid_constant__ SmallArgs A)
{
    extern __shared__ __align__(16) double s_conv[];
    constexpr int NC = K + 1, PA = CoefPad<R, NC>::v;
    constexpr bool kSpin = !Real<R>::fp32;
    const RunDesc &D = A.d;
    DevCtrl *ctrl = D.ctrl;
    SmallSync *S = A.sync;
    const int M = D.M, nconv = (M + kConvOut - K - 1) / (kConvOut - K);
    // task and marker numbering: consecutive warps on different SMs
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int me = (wid * gridDim.x + blockIdx.x) * 32 + lane, all = gridDim.x * kSmallThreads;
    unsigned gen = 0;
    const bool spin = kSpin && A.hbar != 0.0;
    const bool act = me < D.np;
    const unsigned any = __ballot_sync(0xffffffffu, act);
    R *vp = static_cast<R *>(D.P.t), *pp = static_cast<R *>(D.P.p), *dp = static_cast<R *>(D.P.delta);
    int c = 0, id = 0;
    R v = R(0), p = R(0), d = R(0);
    if (act) {
        c = D.P.cell[me];
        v = vp[me];
        p = pp[me];
        if (spin) id = D.P.id[me];
    }
    CoefTables T = D.T;             // A and Kt change places after every subsystem II
    LoopState L;
    L.failed = (*reinterpret_cast<volatile int *>(&ctrl->status) & (STATUS_NUMERIC | STATUS_TIMEOUT)) != 0;
    int hist2 = ctrl->hist2;
#define PIC_BARRIER() do { if (!grid_barrier(S, gen, ctrl)) return; } while (0)
    // ---- what a step finds prepared: the polynomials of a^n and of ebar^(0) = e^n, cleared
    // moments, crossings, spin moments and maxima
    for (int q = me; q < M * prep1_tasks<K>; q += all) prep1_task<K>(q % M, q / M, D);
    for (int q = me; q < M * (K + 1); q += all)
        for (int b = 0; b < 2; ++b) D.my[b][q] = D.mz[b][q] = 0.0;
    if (spin)
        for (int q = me; q < M * K; q += all) A.sm_y[q] = A.sm_z[q] = 0.0;
    if (me < 18) (&S->maxima[0][0][0])[me] = 0ull;
    PIC_BARRIER();
    for (int step = 0; step < A.nsteps; ++step) {
        for (int part = 0; part < (A.strang ? 3 : 2); ++part) {
            L.reset();
            if (part != 1) {
                // ---- subsystem I
                if (me < 9) S->maxima[1][me / 3][me % 3] = 0ull;
                const Sweep1Args &S1 = A.a1;
                const R tau = (R)(S1.dt / S1.dx), dlim = (R)S1.Dlim;
                const R *TA = static_cast<const R *>(T.A), *TE = static_cast<const R *>(T.E);
                R ay[NC], az[NC];
                load_coef<NC>(TA + (size_t)c * (2 * PA), ay);
                load_coef<NC>(TA + (size_t)c * (2 * PA) + PA, az);
                const R A0y = horner<NC>(ay, v), A0z = horner<NC>(az, v);
                const R g0 = root(fma(A0z, A0z, fma(A0y, A0y, fma(p, p, R(1)))));
                bool bad = false;
                d = R(0);
                if (A.warm) {
                    d = quotient(tau * p, g0);
                    if (!within(d, dlim)) { bad = act; d = R(0); }
                }
                if (A.warm_field) {
                    int n;
                    R ve;
                    path_end(v, d, n, ve);
                    if (act) deposit_path_global<K, R>(D.m1[1], D.flux[1], M, c, n, ve);
                    if (bad) atomicOr(&ctrl->status, STATUS_NUMERIC);
                    PIC_BARRIER();
                    for (int b = blockIdx.x; b < nconv; b += gridDim.x) {
                        conv_block<K>(A.c1p, nullptr, T, 0, b, 0, s_conv, nullptr);
                        __syncthreads();
                    }
                    PIC_BARRIER();
                }
                R pnew = p;
                for (;;) {
                    R inc = R(0);
                    if (any) {
                        Kick<K, R, true, kSpin> k;
                        k.start(TE, c, v, d, ay, az, spin);
                        const int nmax = __reduce_max_sync(0xffffffffu, k.an);
                        for (int q = 1; q <= nmax; ++q) k.piece(TA, TE, M, q, spin);
                        R dnew;
                        k.finish(p, A0y, A0z, g0, tau, [&](R W, R D2y, R D2z) -> R {
                            if (!spin || !act) return R(0);
                            return (R)(A.hbar / D.dx * ((A.sy[id] * D2z - A.sz[id] * D2y) / W));
                        }, pnew, dnew);
                        if (!within(dnew, dlim)) { bad = act; dnew = R(0); }
                        int n;
                        R ve;
                        path_end(v, dnew, n, ve);
                        if (act) {
                            deposit_path_global<K, R>(D.m1[L.it & 1], D.flux[L.it & 1], M, c, n, ve);
                            inc = fabs(dnew - d);
                            if constexpr (Real<R>::fp32) inc *= approx_rcp(fmaxf(1.f, fabsf(dnew)));
                        }
                        d = dnew;
                        const double big = warp_max_nonneg((double)inc);
                        if (lane == 0 && big != 0.0) atomic_max_nonneg(&S->maxima[0][L.it % 3][0], big);
                        if (bad) {
                            atomicOr(&ctrl->status, STATUS_NUMERIC);
                            atomicMax(&S->maxima[0][L.it % 3][0], 0x7ff8000000000000ull);
                        }
                    }
                    PIC_BARRIER();
                    for (int b = blockIdx.x; b < nconv; b += gridDim.x) {
                        conv_block<K>(A.c1, nullptr, T, L.it, b, 0, s_conv, S->maxima[0][L.it % 3] + 1);
                        __syncthreads();
                    }
                    PIC_BARRIER();
                    if (loop_decision(A.c1, S->maxima[0], L)) break;
                }
                // ---- end of subsystem I, preparation of II
                int n;
                path_end(v, d, n, v);
                c = wrap_cell(c + n, M);
                p = pnew;
                const int last = (L.it - 1) & 1;
                if (spin && part == 0 && act) {
                    const double sy = A.sy[id], sz = A.sz[id];
                    double pw = 1.0;
                    const size_t row = (size_t)c * K;
#pragma unroll
                    for (int m = 0; m < K; ++m) {
                        atomicAdd(&A.sm_y[row + m], sy * pw);
                        atomicAdd(&A.sm_z[row + m], sz * pw);
                        pw *= (double)v;
                    }
                }
                for (int i = me; i < M; i += all) {
                    commit_at(i, D, 1, last);
                    for (int m = 0; m < K; ++m) D.m1[last][(size_t)i * K + m] = 0.0;
                    D.flux[last][i] = 0;
                }
                if (part == 0) {
                    const int q2 = min(hist2, D.fh.order2);
                    for (int q = me; q < M * 2 * (K + 1); q += all)
                        prep2_coef<K>(q % M, q / M / (K + 1), q / M % (K + 1), D, T, q2, false);
                    for (int q = me; q < 2 * M; q += all) prep2_node<K>(q % M, q / M, D, q2);
                }
                PIC_BARRIER();
                if (part == 2) {
                    if (me < 9) S->maxima[0][me / 3][me % 3] = 0ull;
                    for (int q = me; q < M * K; q += all) prep1_e<K>(q % M, q / M, D, 0);
                    for (int i = me; i < M; i += all) D.ek[i] = D.ex[i];
                    PIC_BARRIER();
                }
            } else {
                // ---- subsystem II
                if (me < 9) S->maxima[0][me / 3][me % 3] = 0ull;
                if (spin)
                    for (int q = me; q < 2 * M; q += all) spin_source_at(M, K, A.d.dt * A.hbar * A.w / A.d.dx, A.sm_y, A.sm_z, D.by, D.bz, q % M, q / M);
                const R *TA = static_cast<const R *>(T.A), *TK = static_cast<const R *>(T.Kt);
                const size_t row = (size_t)c * (2 * PA);
                R cy[NC], cz[NC];
                load_coef<NC>(TA + row, cy);
                load_coef<NC>(TA + row + PA, cz);
                const R A0y = horner<NC>(cy, v), A0z = horner<NC>(cz, v), pp1 = fma(p, p, R(1));
                const R g0 = root(fma(A0z, A0z, fma(A0y, A0y, pp1)));
                for (;;) {
                    if (any) {
                        load_coef<NC>(TK + row, cy);
                        load_coef<NC>(TK + row + PA, cz);
                        const R A1y = horner<NC>(cy, v), A1z = horner<NC>(cz, v);
                        const R g1 = root(fma(A1z, A1z, fma(A1y, A1y, pp1)));
                        R Ly = R(0), Lz = R(0), fy, fz;
                        if constexpr (Real<R>::fp32) {
                            R l[NC];
                            load_coef<NC>(T.L + row, l);
                            Ly = horner<NC>(l, v);
                            load_coef<NC>(T.L + row + PA, l);
                            Lz = horner<NC>(l, v);
                        }
                        exchange<R, true>(A0y + A1y, A0z + A1z, g0 + g1, Ly, Lz, fy, fz);
                        if (act) {
                            double *my = D.my[L.it & 1] + (size_t)c * NC, *mz = D.mz[L.it & 1] + (size_t)c * NC;
                            R pw = R(1);
#pragma unroll
                            for (int m = 0; m < NC; ++m) {
                                if (m > 0) pw = m == 1 ? v : pw * v;
                                const R xy = m == 0 ? fy : fy * pw, xz = m == 0 ? fz : fz * pw;
                                if (xy != R(0)) atomicAdd(&my[m], (double)xy);
                                if (xz != R(0)) atomicAdd(&mz[m], (double)xz);
                            }
                        }
                    }
                    PIC_BARRIER();
                    if (A.c2.node[0]) {
                        for (int q = me; q < 2 * M; q += all) node_pass<K>(A.c2, L.it, q % M, q / M);
                        PIC_BARRIER();
                    }
                    for (int b = blockIdx.x; b < 2 * nconv; b += gridDim.x) {
                        conv_block<K>(A.c2, A.c2.node[b / nconv], T, L.it, b % nconv, b / nconv, s_conv, S->maxima[1][L.it % 3] + 1);
                        __syncthreads();
                    }
                    PIC_BARRIER();
                    if (loop_decision(A.c2, S->maxima[1], L)) break;
                }
                // ---- end of subsystem II: a^{n+1} has its polynomials in Kt
                const int last = (L.it - 1) & 1;
                if constexpr (kSpin) {
                    if (spin && act) {
                        load_coef<NC>(TK + row, cy);
                        load_coef<NC>(TK + row + PA, cz);
                        spin_rotate_one<K>(A, cy, cz, v, id);
                    }
                }
                for (int i = me; i < M; i += all) commit_at(i, D, 2, 0);
                hist2 = min(hist2 + 1, kMaxStartOrder);
                for (int q = me; q < M * (K + 1); q += all) D.my[last][q] = D.mz[last][q] = 0.0;
                if (spin)
                    for (int q = me; q < M * K; q += all) A.sm_y[q] = A.sm_z[q] = 0.0;
                for (int q = me; q < M * K; q += all) prep1_e<K>(q % M, q / M, D, 0);
                for (int i = me; i < M; i += all) D.ek[i] = D.ex[i];
                void *t = T.A;
                T.A = T.Kt;
                T.Kt = t;
                PIC_BARRIER();
            }
        }
    }
#undef PIC_BARRIER
    if (act) {
        D.P.cell[me] = c;
        vp[me] = v;
        pp[me] = p;
        if (A.zero_delta) dp[me] = R(0);
    }
}

template <int K, typename R>
int launch_small_kr(const SmallArgs &a, int grid, size_t smem, cudaStream_t s)
{
    static SmemOptin optin;
    if (!optin.raise((const void *)k_small<K, R>, smem)) return 1;
    void *args[] = {const_cast<SmallArgs *>(&a)};
    const cudaError_t e =
        cudaLaunchCooperativeKernel((const void *)k_small<K, R>, dim3(grid), dim3(kSmallThreads), args, smem, s);
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources || e == cudaErrorNotSupported) {
        cudaGetLastError();
        return kSmallRefused;
    }
    return e != cudaSuccess;
}

template <typename R>
int launch_small_r(const SmallArgs &a, int num_sms, cudaStream_t s)
{
    // a block a warp of markers where that suffices, and a block for every solve block
    const long long want = std::max<long long>((a.d.np + 31) / 32, 2 * conv_blocks(a.d.M, a.d.K));
    const int grid = (int)std::min<long long>(num_sms, want);
    if (a.d.np > (long long)grid * kSmallThreads) return 1;
    const size_t smem = std::max(conv_smem(a.d.K, a.c1.ntap, false), conv_smem(a.d.K, a.c2.ntap, a.c2.node[0] != nullptr));
    switch (a.d.K) {
    case 2: return launch_small_kr<2, R>(a, grid, smem, s);
    case 3: return launch_small_kr<3, R>(a, grid, smem, s);
    case 4: return launch_small_kr<4, R>(a, grid, smem, s);
    case 5: return launch_small_kr<5, R>(a, grid, smem, s);
    default: return 1;
    }
}

}  // namespace

}  // namespace pic
