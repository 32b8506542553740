// pic_device.cuh -- device-side building blocks of libpic (sm_103a).
//
// Positions are stored as (cell c, offset v in [-1/2, 1/2] from its centre) in cell units:
// x = (c + 1/2 + v) dx.  In cell c the degree-d periodic basis functions j = c - r
// (r = 0..d) are nonzero with values N^d(r + 1/2 + v), N^d the cardinal B-spline on the integer knots (Sec. 3.1:
// Lambda^0_j = N^k_j, Lambda^1_j = N^{k-1}_j, supp N^d_j = [x_j, x_{j+d+1})).
#pragma once

#include <climits>
#include <type_traits>

#include <cuda_runtime.h>
#include <stdint.h>

namespace pic {

// ---------------------------------------------------------------------------
// Device control block of one fixed-point loop.
// Non-negative doubles are kept as their bit patterns so that integer atomicMax
// orders them; NaN (0x7ff8...) compares above +Inf, so it reads "not converged".
// ---------------------------------------------------------------------------
struct DevCtrl {
    unsigned long long dmax_bits;      // max particle increment of this sweep
    unsigned long long emax_bits;      // max field increment of this sweep
    unsigned long long dprev_bits;     // previous sweep's values (stagnation test)
    unsigned long long eprev_bits;
    unsigned long long emag_bits;      // max |e^(k+1)| of this sweep (field scale)
    int iter;                          // sweeps done in the current loop
    int converged;                     // 1 once the test passed
    int status;                        // error bits, see STATUS_*
    unsigned int ticket;               // last-block election in multi-block grid kernels
    int hist1, hist2;                  // field changes stored for the starting fields
    int zany;                          // a_z or e_z was non-zero at some node
    double acc[4];                     // reductions for diagnostics (energy, residual)
};

enum : int {
    STATUS_NUMERIC = 1,    // NaN/Inf or displacement beyond the halo
    STATUS_NOCONV  = 2,
    STATUS_TIMEOUT = 4,    // a bounded wait (tensor cores, grid barrier) gave up
};

// accumulator kinds of the sweeps (pic_config.deposit)
enum : int { ACC_NATIVE = 0, ACC_COMP = 1, ACC_DOUBLE = 2 };

// numbers a row of n polynomial coefficients takes (pic_poly.cuh): rows are read by
// 16-byte loads
__host__ __device__ inline int coef_pad(int fp32, int n) { return fp32 ? (n <= 4 ? 4 : 8) : ((n + 1) & ~1); }

// ---------------------------------------------------------------------------
// mbarriers in shared memory (completion of the tensor cores' work).  Every wait is
// bounded: after kMaxWaitTries polls it returns false and the caller records
// STATUS_TIMEOUT and leaves.
// ---------------------------------------------------------------------------
constexpr unsigned long long kMaxWaitTries = 1ull << 26;

__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity)
{
    for (unsigned long long i = 0; i < kMaxWaitTries; ++i) {
        unsigned ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void atomic_max_nonneg(unsigned long long *addr, double v)
{
    // v >= 0 or NaN: the IEEE bit pattern is monotone in v for non-negative values
    atomicMax(addr, (unsigned long long)__double_as_longlong(v));
}

__device__ __forceinline__ double bits_to_double(unsigned long long b)
{
    return __longlong_as_double((long long)b);
}

__device__ __forceinline__ int wrap_cell(int c, int M)
{
    c %= M;
    return c < 0 ? c + M : c;
}

// ---------------------------------------------------------------------------
// Uniform B-spline values by the triangular (de Boor) scheme:
// level 0: b = [1]; level n: b'_r = ((t + r) b_r + (n + 1 - t - r) b_{r-1}) / n,
// with b_{-1} = b_n = 0.  After level d, v[r] = N^d(r + t), r = 0..d.
// ---------------------------------------------------------------------------
template <int D, typename R>
__device__ __forceinline__ void bspline_vals(R t, R *v)
{
    v[0] = R(1);
#pragma unroll
    for (int n = 1; n <= D; ++n) {
        const R inv = R(1) / R(n);
        v[n] = (R(1) - t) * v[n - 1] * inv;
#pragma unroll
        for (int r = n - 1; r >= 1; --r)
            v[r] = ((t + R(r)) * v[r] + (R(n + 1 - r) - t) * v[r - 1]) * inv;
        v[0] = t * v[0] * inv;
    }
}

template <typename T>
__device__ __forceinline__ T warp_max(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        T w = __shfl_xor_sync(0xffffffffu, v, o);
        v = (w > v || w != w) ? w : v;       // NaN wins
    }
    return v;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void block_sum_to(double *dst, double v, double *s_red)
{
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) s_red[wid] = v;
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        double u = lane < nw ? s_red[lane] : 0.0;
        u = warp_sum(u);
        if (lane == 0) atomicAdd(dst, u);
    }
    __syncthreads();
}

}  // namespace pic
