// pic_mlp.cu -- the learned warm start of the subsystem-I fixed point.
//
// A small network proposes each marker's displacement x^(0) - x^n for the
// implicit substep of subsystem I (Sec. 4.2); the Picard iteration then runs to
// the same tolerance, so the proposal changes only the number of sweeps, never
// the converged state or the conservation properties.
//
// Network: 6 inputs (cell-relative x, p, E_x(x^n), A_y(x^n), A_z(x^n), dt), each
// normalised by (v - shift) * scale; three hidden layers of width 64 with ReLU;
// 2 outputs, scaled by out_scale, read as
//   y0 = (x^{n+1} - x^n - dt p/gamma(p, A(x^n))) / dt^2   (residual of the explicit predictor)
//   y1 = (p^{n+1} - p^n - dt E_x(x^n)) / dt^2.
// Parameters: one float vector W1 (64x6, row-major [out][in]), b1, W2 (64x64),
// b2, W3, b3, W4 (2x64), b4 -- 8898 numbers.
//
// Inference runs on the 5th-generation tensor cores (tcgen05.mma, bf16 activations
// and fp32 accumulators in tensor memory, weights in shared memory), 128 markers per
// tile; the ReLU is part of each thread's conversion of its accumulator row to bf16.  Training
// (forward + backward + Adam) runs in fp32 on the CUDA cores.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <vector>

#include "pic.h"
#include "pic_internal.h"
#include "pic_poly.cuh"

namespace pic {

constexpr int kIn = 6, kHid = 64, kOut = 2;
constexpr int kNParams = kHid * kIn + kHid + 2 * (kHid * kHid + kHid) + kOut * kHid + kOut;   // 8898
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kHid * kIn, kOffW2 = kOffB1 + kHid,
              kOffB2 = kOffW2 + kHid * kHid, kOffW3 = kOffB2 + kHid, kOffB3 = kOffW3 + kHid * kHid,
              kOffW4 = kOffB3 + kHid, kOffB4 = kOffW4 + kOut * kHid;
static_assert(kOffB4 + kOut == kNParams, "parameter packing");
constexpr int kNorm = 2 * kIn + kOut;     // shift[6], scale[6], out_scale[2]

__device__ __forceinline__ float relu(float z) { return fmaxf(z, 0.f); }

// derivative of the ReLU, taken as 0 at z = 0
__device__ __forceinline__ float relu_grad(float z) { return z > 0.f ? 1.f : 0.f; }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    uint32_t u;
    memcpy(&u, &v, 4);
    return u;
}

// ReLU of two pre-activations, rounded to bf16 and packed.  NaN = true: a NaN becomes 0 (one
// packed max more); false: it stays a NaN, one conversion does both.
template <bool NaN>
__device__ __forceinline__ uint32_t relu_bf16x2(float z0, float z1)
{
    uint32_t o;
    if (NaN) {
        const __nv_bfloat162 out = __hmax2(__floats2bfloat162_rn(z0, z1), __float2bfloat162_rn(0.f));
        memcpy(&o, &out, 4);
    } else {
        asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(o) : "f"(z1), "f"(z0));
    }
    return o;
}

// ---------------------------------------------------------------------------
// Tensor-core inference with tcgen05 (5th-generation tensor cores, accumulators
// in tensor memory).  One block of 640 threads per SM runs 5 independent chains,
// one per warpgroup; a chain takes 128 markers at a time, one row per thread.  Per
// layer every thread stores its row's bf16 activations to the chain's operand columns
// of tensor memory, one thread issues the layer's tcgen05.mma instructions (M = 128,
// N = 64, K = 16 each) and commits them to the chain's mbarrier, every thread waits
// (bounded), loads its row of the fp32 accumulator and applies the ReLU.  While one
// chain waits for the tensor cores, the others run their epilogues.  Weights are staged
// once per block, in the canonical K-major layout (8-row x 16-byte core matrices) in
// shared memory, and shared by the chains.
//
// Activations stay out of shared memory: as the A operand there they cost 48 KB written
// and 48 KB read back a tile at 128 bytes a clock, more than the products themselves
// (32 clocks a step).  Warm start of 2e7 markers: 666 us with 8 chains on operands in
// shared memory, 582 us so, 562 us with the next tile's features formed beside the
// second layer (605 us with the ReLU as a packed maximum of its own).  What bounds it:
// the tensor pipe is busy half of the time, the rest is the chains' own latency.
// The tensor memory holds 5 chains: 64 accumulator and 32 operand columns each, and 8
// columns of the constant operand for the biases.
// ---------------------------------------------------------------------------
constexpr int kRows = 128;                       // markers per tile (UMMA M) = threads per chain
constexpr int kChains = 5;                       // warpgroups per block
constexpr int kMlpThreads = kRows * kChains;     // 640
constexpr int kTmemCols = 512;
constexpr int kChainCols = 96;                   // chain g: columns 96 g .. : 64 accumulators, 32 operands
constexpr int kOnesCol = kChains * kChainCols;   // 8 columns: 1 in operand column 0, else 0
static_assert(kOnesCol + 8 <= kTmemCols, "tensor memory");
constexpr int kOutN = 16;                        // output layer padded to the smallest N for M = 128

// byte offset of element (r, k) in a K-major no-swizzle operand with K columns:
// core matrix (r/8, k/8) at (r/8) * (K/8) * 128 + (k/8) * 128, row r%8 at 16 (r%8)
__host__ __device__ constexpr int kmaj_off(int r, int k, int K)
{
    return (r >> 3) * (K >> 3) * 128 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

struct MlpChain {
    unsigned long long bar;         // MMA completion
    int abort;                      // a wait gave up
    int pad;
};

// The biases of layers 1-3 ride on the tensor cores: layer 1 takes b1 as weight
// column 6 against a constant feature 1; layers 2 and 3 add one K = 16 step of the
// constant operand, whose column 0 is 1, against a bias block whose column 0 is b.
struct MlpUmma {
    __nv_bfloat16 W1[64 * 16];      // [n][k], K = 16: 6 weights, b1, zeros
    __nv_bfloat16 W2[64 * 64];
    __nv_bfloat16 W3[64 * 64];
    __nv_bfloat16 W4[kOutN * 64];   // rows 0, 1 used
    __nv_bfloat16 B2[64 * 16];      // column 0 = b2
    __nv_bfloat16 B3[64 * 16];      // column 0 = b3
    MlpChain C[kChains];
    float b4[2];
    float norm[kNorm];
    uint32_t tmem;                  // tensor-memory base address
    int last_ok;                    // the output layer's row 0 has no NaN
};

// shared-memory matrix descriptor (tcgen05): start, leading (K-direction core
// matrix) and stride (8-row group) byte offsets, version 1, no swizzle
__device__ __forceinline__ uint64_t umma_desc(const void *p, uint32_t lbo, uint32_t sbo)
{
    const uint32_t a = smem_u32(p);
    return (uint64_t)((a & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor, kind::f16: D f32, A and B bf16, both K-major, M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D (tensor memory) = A (tensor memory: lane = row, two bf16 a column) x B (shared memory)
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void umma_commit(unsigned long long *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// barrier of one chain (named barrier 1 + g, its 128 threads)
__device__ __forceinline__ void chain_sync(int g)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(kRows) : "memory");
}

// 64 consecutive fp32 columns of this thread's tensor-memory lane, and the wait
// for them, in one statement (the registers are valid only after the wait)
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, uint32_t (&r)[64])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,"
        "%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
          "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
          "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
          "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
          "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr)
        : "memory");
}

// 32 and 8 consecutive columns of this thread's lane; complete after tmem_st_wait
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31};\n" ::
          "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]),
        "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%5,%5,%5};\n" ::"r"(taddr), "r"(a), "r"(b),
                 "r"(c), "r"(d), "r"(0u)
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld2(uint32_t taddr, float (&v)[2])
{
    uint32_t r0, r1;
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r0), "=r"(r1)
        : "r"(taddr)
        : "memory");
    v[0] = __uint_as_float(r0);
    v[1] = __uint_as_float(r1);
}

__device__ __forceinline__ void put_bf16(void *base, int off, float v)
{
    *reinterpret_cast<__nv_bfloat16 *>(reinterpret_cast<char *>(base) + off) = __float2bfloat16(v);
}

// Four columns k .. k + 3 of row n, bf16, at a multiple of four columns (8 bytes of a core matrix row).
__device__ __forceinline__ void put_bf16x4(void *base, int n, int k, int K, float4 w)
{
    *reinterpret_cast<uint2 *>(reinterpret_cast<char *>(base) + kmaj_off(n, k, K)) =
        make_uint2(pack_bf16(w.x, w.y), pack_bf16(w.z, w.w));
}

// Stage the network (fp32 parameters in global memory) into the operand layouts: rows of W2
// and W3 four columns at a time, all of a thread's loads in flight together (one element at
// a time the staging was most of the 12.7 us of an inference of 4096 rows; now 9.0).
__device__ void stage_umma(MlpUmma &S, const float *params, const float *norm)
{
    constexpr int kQ = kHid * kHid / 4, kPer = (2 * kQ + kMlpThreads - 1) / kMlpThreads;
    float4 w[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int q = threadIdx.x + j * kMlpThreads;
        if (q < 2 * kQ)
            w[j] = reinterpret_cast<const float4 *>(params + (q < kQ ? kOffW2 : kOffW3))[q < kQ ? q : q - kQ];
    }
    static_assert(kOffW2 % 4 == 0 && kOffW3 % 4 == 0 && kOffW4 % 4 == 0, "float4 rows");
    for (int i = threadIdx.x; i < 64 * 16; i += blockDim.x) {
        const int n = i >> 4, k = i & 15;
        put_bf16(S.W1, kmaj_off(n, k, 16),
                 k < kIn ? params[kOffW1 + n * kIn + k] : (k == kIn ? params[kOffB1 + n] : 0.f));
        put_bf16(S.B2, kmaj_off(n, k, 16), k == 0 ? params[kOffB2 + n] : 0.f);
        put_bf16(S.B3, kmaj_off(n, k, 16), k == 0 ? params[kOffB3 + n] : 0.f);
    }
    if (threadIdx.x < kOutN * kHid / 4) {
        const int n = threadIdx.x / (kHid / 4), k = 4 * (threadIdx.x % (kHid / 4));
        put_bf16x4(S.W4, n, k, 64,
                   n < kOut ? *reinterpret_cast<const float4 *>(params + kOffW4 + n * kHid + k) : make_float4(0.f, 0.f, 0.f, 0.f));
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int q = threadIdx.x + j * kMlpThreads;
        if (q < 2 * kQ) put_bf16x4(q < kQ ? S.W2 : S.W3, (q % kQ) / 16, 4 * (q % 16), 64, w[j]);
    }
    if (threadIdx.x < kOut) S.b4[threadIdx.x] = params[kOffB4 + threadIdx.x];
    if (threadIdx.x < kNorm) S.norm[threadIdx.x] = norm[threadIdx.x];
    if (threadIdx.x < 32) {
        const float w = params[kOffW4 + threadIdx.x] + params[kOffW4 + 32 + threadIdx.x];
        const int ok = __all_sync(0xffffffffu, !isnan(w)) && !isnan(params[kOffB4]) && !isnan(norm[2 * kIn]);
        if (threadIdx.x == 0) S.last_ok = ok;
    }
}

// Block prologue: chain barriers, tensor memory (warp 0 allocates all 512
// columns: one block per SM), staged weights.
__device__ __forceinline__ void umma_begin(MlpUmma &S, const float *params, const float *norm)
{
    if (threadIdx.x < kChains) {
        mbar_init(&S.C[threadIdx.x].bar, 1);
        S.C[threadIdx.x].abort = 0;
    }
    if (threadIdx.x == 0) fence_mbar_init();
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    stage_umma(S, params, norm);
    fence_proxy_async();           // weights: visible to the tensor cores
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x < kRows) {     // the constant operand, a lane a thread
        tmem_st8(S.tmem + ((threadIdx.x & ~31u) << 16) + kOnesCol, pack_bf16(1.f, 0.f), 0u, 0u, 0u);
        tmem_st_wait();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}

// Block epilogue: report chains that gave up, and give their MMAs in flight one more
// bounded wait before the tensor memory is freed.
__device__ __forceinline__ void umma_end(MlpUmma &S, int g, unsigned phase, int *status)
{
    tc_fence_before();
    __syncthreads();
    if (*reinterpret_cast<volatile int *>(&S.C[g].abort)) {
        atomicOr(status, STATUS_TIMEOUT);
        mbar_wait(&S.C[g].bar, phase ^ 1u);
    }
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(S.tmem), "r"(kTmemCols)
                     : "memory");
}

// This thread's lane of its chain's columns.  Warp w reaches lanes 32 (w % 4) .. + 31.
__device__ __forceinline__ uint32_t umma_cols(const MlpUmma &S, int g, int r)
{
    return S.tmem + ((uint32_t)(r & ~31) << 16) + (uint32_t)(kChainCols * g);
}

// Write this thread's feature row (normalised, bf16) into its chain's operand.
__device__ __forceinline__ void umma_put_features(MlpUmma &S, int g, int r, const float f[kIn])
{
    tmem_st8(umma_cols(S, g, r) + 64,
             pack_bf16((f[0] - S.norm[0]) * S.norm[kIn + 0], (f[1] - S.norm[1]) * S.norm[kIn + 1]),
             pack_bf16((f[2] - S.norm[2]) * S.norm[kIn + 2], (f[3] - S.norm[3]) * S.norm[kIn + 3]),
             pack_bf16((f[4] - S.norm[4]) * S.norm[kIn + 4], (f[5] - S.norm[5]) * S.norm[kIn + 5]),
             pack_bf16(1.f, 0.f));     // feature 6 = 1 (carries b1)
}

// One layer of chain g: issue (the chain's first thread), wait (all of its threads).
// A wait that gives up marks the chain; its threads all leave at the next layer's
// barrier (false), before anything else is issued.  beside() runs while the layer does.
template <typename Beside>
__device__ __forceinline__ bool umma_layer(MlpUmma &S, int g, int r, int K, const __nv_bfloat16 *Bop,
                                           const __nv_bfloat16 *bias, uint32_t idesc, unsigned &phase, Beside &&beside)
{
    MlpChain &C = S.C[g];
    tmem_st_wait();                // this thread's activations
    tc_fence_before();
    chain_sync(g);
    tc_fence_after();
    if (*reinterpret_cast<volatile int *>(&C.abort)) return false;
    if (r == 0) {
        const uint32_t sbo = (uint32_t)K * 16;    // K/8 core matrices of 128 bytes per 8-row group
        const uint32_t d = S.tmem + (uint32_t)(kChainCols * g);
        for (int kt = 0; kt < K / 16; ++kt)       // 16 bf16 = 8 operand columns a step
            umma_bf16(d, d + 64 + 8 * kt, umma_desc(reinterpret_cast<const char *>(Bop) + kt * 256, 128, sbo), idesc,
                      kt > 0);
        if (bias)      // + ones x bias^T
            umma_bf16(d, S.tmem + kOnesCol, umma_desc(bias, 128, 256), idesc, 1u);
        umma_commit(&C.bar);
    }
    __syncwarp();
    beside();
    if (!mbar_wait(&C.bar, phase)) atomicExch(&C.abort, 1);
    __syncwarp();
    phase ^= 1u;
    tc_fence_after();
    return true;
}

// ReLU of this thread's accumulator row (the chain's 64 columns, bias included)
// into its row of the next layer's operand.
template <bool NaN>
__device__ __forceinline__ void umma_epilogue(MlpUmma &S, int g, int r)
{
    const uint32_t cols = umma_cols(S, g, r);
    uint32_t v[64], o[32];
    tmem_ld64(cols, v);
#pragma unroll
    for (int i = 0; i < 32; ++i) o[i] = relu_bf16x2<NaN>(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
    tmem_st32(cols + 64, o);
}

// The network on chain g's 128 feature rows.  Returns false after a bounded wait
// gave up; y = this row's scaled outputs.  beside() runs while the tensor cores work.
template <bool NaN, typename Beside>
__device__ __forceinline__ bool umma_network(MlpUmma &S, int g, int r, unsigned &phase, float (&y)[2], Beside &&beside)
{
    auto nothing = [] {};
    constexpr uint32_t kHidDesc = idesc_bf16(kRows, kHid), kOutDesc = idesc_bf16(kRows, kOutN);
    if (!umma_layer(S, g, r, 16, S.W1, nullptr, kHidDesc, phase, nothing)) return false;
    umma_epilogue<NaN>(S, g, r);
    if (!umma_layer(S, g, r, 64, S.W2, S.B2, kHidDesc, phase, beside)) return false;
    umma_epilogue<NaN>(S, g, r);
    if (!umma_layer(S, g, r, 64, S.W3, S.B3, kHidDesc, phase, nothing)) return false;
    umma_epilogue<NaN>(S, g, r);
    if (!umma_layer(S, g, r, 64, S.W4, nullptr, kOutDesc, phase, nothing)) return false;
    float o[2];
    tmem_ld2(umma_cols(S, g, r), o);
    y[0] = (o[0] + S.b4[0]) * S.norm[2 * kIn];
    y[1] = (o[1] + S.b4[1]) * S.norm[2 * kIn + 1];
    return true;
}

// ---------------------------------------------------------------------------
// Standalone inference: X (B x 6 raw features, fp32) -> Y (B x 2 scaled outputs).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kMlpThreads, 1) k_mlp_infer(const float *params, const float *norm,
                                                             const float *X, long long B, float *Y, int *status)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    MlpUmma &S = *reinterpret_cast<MlpUmma *>(smem);
    umma_begin(S, params, norm);
    const int g = threadIdx.x / kRows, r = threadIdx.x % kRows;
    unsigned phase = 0;
    const long long stride = (long long)gridDim.x * kChains * kRows;
    // the next tile's inputs are loaded while the network runs on this one
    float nx[kIn];
    const long long base0 = ((long long)blockIdx.x * kChains + g) * kRows;
#pragma unroll
    for (int i = 0; i < kIn; ++i) nx[i] = base0 + r < B ? X[(base0 + r) * kIn + i] : 0.f;
    for (long long base = base0; base < B; base += stride) {
        const long long a = base + r;
        float f[kIn];
#pragma unroll
        for (int i = 0; i < kIn; ++i) f[i] = a < B ? nx[i] : S.norm[i];
        const long long an = a + stride;
#pragma unroll
        for (int i = 0; i < kIn; ++i) nx[i] = an < B ? X[an * kIn + i] : 0.f;
        umma_put_features(S, g, r, f);
        float y[2];
        if (!umma_network<true>(S, g, r, phase, y, [] {})) break;
        if (a < B) {
            Y[2 * a] = y[0];
            Y[2 * a + 1] = y[1];
        }
    }
    umma_end(S, g, phase, status);
}

// ---------------------------------------------------------------------------
// Warm start of subsystem I: delta^(0) = tau p/g0 + y0 dt^2/dx for every marker, with the
// features at x^n: a^n from the cells' polynomials (the preparation of the substep writes
// them), e_x^n from the nodes staged in shared memory.  The features of a chain's next
// tile are formed while the tensor cores run the second layer of this one.
// ---------------------------------------------------------------------------
template <int K, typename R>
__global__ void __launch_bounds__(kMlpThreads, 1) k_warm_mlp(WarmArgs A)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    MlpUmma &S = *reinterpret_cast<MlpUmma *>(smem);
    constexpr int H = K + 1, kPad = CoefPad<R, K + 1>::v;
    const int W = A.M + 2 * H;
    float *s_e = reinterpret_cast<float *>(smem + ((sizeof(MlpUmma) + 127) & ~size_t(127)));
    for (int i = threadIdx.x; i < W; i += blockDim.x) s_e[i] = (float)A.ex[wrap_cell(i - H, A.M)];
    umma_begin(S, A.params, A.norm);
    const int g = threadIdx.x / kRows, r = threadIdx.x % kRows;
    const R *tp = static_cast<const R *>(A.P.t);
    const R *pp = static_cast<const R *>(A.P.p);
    R *dp = static_cast<R *>(A.P.delta);
    const float tau = (float)(A.dt / A.dx);
    const float c2 = (float)(A.dt * A.dt / A.dx);
    unsigned phase = 0;
    const long long stride = (long long)gridDim.x * kChains * kRows;
    int c = 0;
    R t = R(0), p = R(0);
    auto fetch = [&](long long a) {
        if (a >= A.np) return;
        c = A.P.cell[a];
        t = tp[a];
        p = pp[a];
    };
    float f[kIn], expl = 0.f;
    auto features = [&](long long a) {
        if (a >= A.np) {
#pragma unroll
            for (int i = 0; i < kIn; ++i) f[i] = S.norm[i];
            return;
        }
        const float v = (float)t, pn = (float)p, tc = v + 0.5f;      // tc: cell-relative position
        float u[K];
        bspline_vals<K - 1, float>(tc, u);
        float Ex = 0.f, Af[2];
#pragma unroll
        for (int q = 0; q < K; ++q) Ex += s_e[c - q + H] * u[q];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            R co[K + 1];
            load_coef<K + 1>(static_cast<const R *>(A.coefA) + ((size_t)2 * c + i) * kPad, co);
            Af[i] = (float)horner(co, t);
        }
        f[0] = tc; f[1] = pn; f[2] = Ex; f[3] = Af[0]; f[4] = Af[1]; f[5] = (float)A.dt;
        expl = quotient(tau * pn, root(fmaf(pn, pn, fmaf(Af[0], Af[0], fmaf(Af[1], Af[1], 1.f)))));
    };
    const long long base0 = ((long long)blockIdx.x * kChains + g) * kRows;
    fetch(base0 + r);
    features(base0 + r);
    fetch(base0 + r + stride);
    for (long long base = base0; base < A.np; base += stride) {
        const long long a = base + r;
        umma_put_features(S, g, r, f);
        const float now = expl;
        float y[2];
        auto next = [&] {
            features(a + stride);
            fetch(a + 2 * stride);
        };
        if (!umma_network<false>(S, g, r, phase, y, next)) break;
        // a hidden value that is no number proposes nothing (the inference takes it as 0)
        if (isnan(y[0]) && S.last_ok) y[0] = 0.f;
        if (a < A.np) dp[a] = (R)(now + y[0] * c2);
    }
    umma_end(S, g, phase, A.status);
}

// ---------------------------------------------------------------------------
// Training: loss = mean over the batch of sum_o (y_o - T_o / out_scale_o)^2 on
// the normalised outputs; gradients by the chain rule in fp32.
//
// A block takes tiles of 32 samples; its 256 threads hold 2 samples x 4 neurons of a
// layer's values (forward: products along the inputs, backward: along the neurons) and
// 4 x 4 of a weight gradient (products along the samples), all operands in shared memory
// read four numbers at a time: 32 multiply-adds per 6 loads, 16 per 2.  The row strides
// keep these reads free of bank conflicts (kWS: 8 rows of one column group; kHS: two
// rows of 16 columns).  The weights are loaded four numbers at a time, all of a thread's
// loads in flight together; the weight gradients stay in registers over a block's tiles; a
// cluster of blocks sums them through distributed shared memory and adds them to the global
// gradient once.  4096 samples, cold caches: 83 us with one product a thread at a time and
// gradients through shared memory, 29 us with these tiles, 19.7 us with the weights' loads
// together, 18.2 us with clusters of 4 (26.3 us with clusters of 8, whose blocks share SMs).
// ---------------------------------------------------------------------------
constexpr int kTB = 32, kTrainThreads = 256, kTrainCluster = 4;
constexpr int kWS = kHid + 4, kHS = kHid + 16;
struct TrainSmem {
    float W2[kHid * kWS], W3[kHid * kWS];
    float h1[kTB * kHS], h2[kTB * kHS], h3[kTB * kHS];
    float d1[kTB * kHS], d2[kTB * kHS];
    float W1[kHid * kIn], W4[kOut * kHid];
    float b1[kHid], b2[kHid], b3[kHid], b4[kOut];
    float h0[kTB * kIn];
    float y[kTB * kOut], tg[kTB * kOut];
    float norm[kNorm];
    double loss[kTrainThreads / 32];
};

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float dot4(float4 a, float4 b, float acc)
{
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}

// hout[s][n] = relu(b[n] + sum_k W[n][k] hin[s][k]): samples sg and sg + 16, neurons ng + 16 j
__device__ __forceinline__ void dense_fwd(const float *W, const float *b, const float *hin, float *hout)
{
    const int ng = threadIdx.x & 15, sg = threadIdx.x >> 4;
    float acc[2][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[0][j] = acc[1][j] = b[ng + 16 * j];
#pragma unroll 4
    for (int k = 0; k < kHid; k += 4) {
        const float4 x0 = ld4(hin + sg * kHS + k), x1 = ld4(hin + (sg + 16) * kHS + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 w = ld4(W + (ng + 16 * j) * kWS + k);
            acc[0][j] = dot4(w, x0, acc[0][j]);
            acc[1][j] = dot4(w, x1, acc[1][j]);
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        hout[sg * kHS + ng + 16 * j] = relu(acc[0][j]);
        hout[(sg + 16) * kHS + ng + 16 * j] = relu(acc[1][j]);
    }
}

// dout[s][k] = relu'(h[s][k]) sum_n din[s][n] W[n][k]: samples sg and sg + 16, inputs 4 kg .. 4 kg + 3
__device__ __forceinline__ void dense_bwd(const float *W, const float *din, const float *h, float *dout)
{
    const int k = 4 * (threadIdx.x & 15), sg = threadIdx.x >> 4;
    float acc[2][4] = {};
#pragma unroll 4
    for (int n = 0; n < kHid; n += 4) {
        float x[2][4];
        *reinterpret_cast<float4 *>(x[0]) = ld4(din + sg * kHS + n);
        *reinterpret_cast<float4 *>(x[1]) = ld4(din + (sg + 16) * kHS + n);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 w = ld4(W + (n + j) * kWS + k);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                acc[i][0] = fmaf(x[i][j], w.x, acc[i][0]);
                acc[i][1] = fmaf(x[i][j], w.y, acc[i][1]);
                acc[i][2] = fmaf(x[i][j], w.z, acc[i][2]);
                acc[i][3] = fmaf(x[i][j], w.w, acc[i][3]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int s = sg + 16 * i;
        const float4 z = ld4(h + s * kHS + k);
        *reinterpret_cast<float4 *>(dout + s * kHS + k) =
            make_float4(acc[i][0] * relu_grad(z.x), acc[i][1] * relu_grad(z.y), acc[i][2] * relu_grad(z.z),
                        acc[i][3] * relu_grad(z.w));
    }
}

// G[i][j] += sum_s d[s][4 ng + i] h[s][4 kg + j],  gb[i] += sum_s d[s][4 ng + i]
__device__ __forceinline__ void dense_grad(const float *d, const float *h, float (&G)[4][4], float (&gb)[4])
{
    const int k = 4 * (threadIdx.x & 15), n = 4 * (threadIdx.x >> 4);
#pragma unroll 4
    for (int s = 0; s < kTB; ++s) {
        const float4 a = ld4(d + s * kHS + n), b = ld4(h + s * kHS + k);
        const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            G[i][0] = fmaf(av[i], b.x, G[i][0]);
            G[i][1] = fmaf(av[i], b.y, G[i][1]);
            G[i][2] = fmaf(av[i], b.z, G[i][2]);
            G[i][3] = fmaf(av[i], b.w, G[i][3]);
            gb[i] += av[i];
        }
    }
}

// this thread's part of a layer's gradient to the block's
__device__ __forceinline__ void put_grad(float *gW, float *gB, const float (&G)[4][4], const float (&gb)[4])
{
    const int k = 4 * (threadIdx.x & 15), n = 4 * (threadIdx.x >> 4);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4 *>(gW + (n + i) * kHid + k) = make_float4(G[i][0], G[i][1], G[i][2], G[i][3]);
    if (k == 0) *reinterpret_cast<float4 *>(gB + n) = make_float4(gb[0], gb[1], gb[2], gb[3]);
}
static_assert(kOffB2 % 4 == 0 && kOffB3 % 4 == 0, "float4 stores");

__global__ void __launch_bounds__(kTrainThreads, 2) k_mlp_train(const float *params, const float *norm,
                                                                const float *X, const float *Tg, long long B,
                                                                float *grad, double *loss)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(smem);
    const int tid = threadIdx.x;
    {   // the weights, all loads in flight together
        constexpr int kPer = kHid * kHid / 4 / kTrainThreads;
        float4 w2[kPer], w3[kPer];
        float w1[2];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            w2[j] = reinterpret_cast<const float4 *>(params + kOffW2)[tid + j * kTrainThreads];
            w3[j] = reinterpret_cast<const float4 *>(params + kOffW3)[tid + j * kTrainThreads];
        }
        w1[0] = params[kOffW1 + tid];
        w1[1] = tid < kHid * kIn - kTrainThreads ? params[kOffW1 + kTrainThreads + tid] : 0.f;
        if (tid < kHid) {
            S.b1[tid] = params[kOffB1 + tid];
            S.b2[tid] = params[kOffB2 + tid];
            S.b3[tid] = params[kOffB3 + tid];
        }
        if (tid < kOut * kHid) S.W4[tid] = params[kOffW4 + tid];
        if (tid < kOut) S.b4[tid] = params[kOffB4 + tid];
        if (tid < kNorm) S.norm[tid] = norm[tid];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int q = tid + j * kTrainThreads, o = (q / 16) * kWS + 4 * (q % 16);
            *reinterpret_cast<float4 *>(S.W2 + o) = w2[j];
            *reinterpret_cast<float4 *>(S.W3 + o) = w3[j];
        }
        S.W1[tid] = w1[0];
        if (tid < kHid * kIn - kTrainThreads) S.W1[kTrainThreads + tid] = w1[1];
        static_assert(kHid * kIn >= kTrainThreads && kHid * kIn <= 2 * kTrainThreads, "W1");
    }
    float G2[4][4] = {}, G3[4][4] = {}, gb2[4] = {}, gb3[4] = {}, g1[2] = {}, gb1 = 0.f, g4 = 0.f;
    double sum = 0.0;
    for (long long s0 = (long long)blockIdx.x * kTB; s0 < B; s0 += (long long)gridDim.x * kTB) {
        const int ns = (int)min((long long)kTB, B - s0);
        const float x = tid < ns * kIn ? X[s0 * kIn + tid] : 0.f;
        const float tg = tid < ns * kOut ? Tg[s0 * kOut + tid] : 0.f;
        __syncthreads();                          // the weights; the last tile's reads
        if (tid < kTB * kIn) S.h0[tid] = tid < ns * kIn ? (x - S.norm[tid % kIn]) * S.norm[kIn + tid % kIn] : 0.f;
        if (tid < kTB * kOut) S.tg[tid] = tid < ns * kOut ? tg / S.norm[2 * kIn + tid % kOut] : 0.f;
        __syncthreads();
        {
            const int ng = tid & 15, sg = tid >> 4;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int n = ng + 16 * j;
                float a0 = S.b1[n], a1 = a0;
#pragma unroll
                for (int k = 0; k < kIn; ++k) {
                    const float w = S.W1[n * kIn + k];
                    a0 = fmaf(w, S.h0[sg * kIn + k], a0);
                    a1 = fmaf(w, S.h0[(sg + 16) * kIn + k], a1);
                }
                S.h1[sg * kHS + n] = relu(a0);
                S.h1[(sg + 16) * kHS + n] = relu(a1);
            }
        }
        __syncthreads();
        dense_fwd(S.W2, S.b2, S.h1, S.h2);
        __syncthreads();
        dense_fwd(S.W3, S.b3, S.h2, S.h3);
        __syncthreads();
        {   // outputs and dL/dy, four threads an output; a sample beyond the batch has none
            const int s = tid >> 3, o = (tid >> 2) & 1, q = tid & 3;
            float acc = 0.f;
#pragma unroll
            for (int k = 0; k < kHid; k += 16) acc = dot4(ld4(S.W4 + o * kHid + k + 4 * q), ld4(S.h3 + s * kHS + k + 4 * q), acc);
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            if (q == 0) {
                float dy = 0.f;
                if (s < ns) {
                    const float r = acc + S.b4[o] - S.tg[s * kOut + o];
                    dy = 2.f * r / (float)B;
                    sum += (double)r * (double)r;
                }
                S.y[s * kOut + o] = dy;
            }
        }
        __syncthreads();
        if (tid < kOut * kHid) {                  // W4
            const int o = tid / kHid, k = tid % kHid;
#pragma unroll 8
            for (int s = 0; s < kTB; ++s) g4 = fmaf(S.y[s * kOut + o], S.h3[s * kHS + k], g4);
        } else if (tid < kOut * kHid + kOut) {    // b4
            for (int s = 0; s < kTB; ++s) g4 += S.y[s * kOut + tid - kOut * kHid];
        }
        for (int i = tid; i < kTB * kHid; i += kTrainThreads) {
            const int s = i / kHid, k = i % kHid;
            const float acc = fmaf(S.y[s * kOut + 1], S.W4[kHid + k], S.y[s * kOut] * S.W4[k]);
            S.d1[s * kHS + k] = acc * relu_grad(S.h3[s * kHS + k]);
        }
        static_assert(kOut == 2, "output layer");
        __syncthreads();
        dense_bwd(S.W3, S.d1, S.h2, S.d2);
        dense_grad(S.d1, S.h2, G3, gb3);
        __syncthreads();
        dense_bwd(S.W2, S.d2, S.h1, S.d1);
        dense_grad(S.d2, S.h1, G2, gb2);
        __syncthreads();
        {   // W1, b1: neuron tid % 64, inputs tid / 64 and tid / 64 + 4
            const int n = tid % kHid, k0 = tid / kHid, k1 = k0 + 4 < kIn ? k0 + 4 : k0;
#pragma unroll 8
            for (int s = 0; s < kTB; ++s) {
                const float d = S.d1[s * kHS + n];
                g1[0] = fmaf(d, S.h0[s * kIn + k0], g1[0]);
                g1[1] = fmaf(d, S.h0[s * kIn + k1], g1[1]);
                gb1 += d;
            }
        }
    }
    // the block's gradient over its weights, then the cluster's: a block sums one part of it
    // over the blocks and adds that to the global gradient
    float *G = reinterpret_cast<float *>(smem);
    static_assert(kNParams * sizeof(float) <= offsetof(TrainSmem, d1), "gradient over weights and activations");
    __syncthreads();
    put_grad(G + kOffW2, G + kOffB2, G2, gb2);
    put_grad(G + kOffW3, G + kOffB3, G3, gb3);
    {
        const int n = tid % kHid, k0 = tid / kHid;
        G[kOffW1 + n * kIn + k0] = g1[0];
        if (k0 + 4 < kIn) G[kOffW1 + n * kIn + k0 + 4] = g1[1];
        if (k0 == 3) G[kOffB1 + n] = gb1;
        if (tid < kOut * kHid + kOut) G[kOffW4 + tid] = g4;
    }
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    cl.sync();
    const int nb = (int)cl.num_blocks(), part = (kNParams / 2 + nb - 1) / nb;
    for (int i = (int)cl.block_rank() * part + tid; i < min(kNParams / 2, ((int)cl.block_rank() + 1) * part);
         i += kTrainThreads) {
        float2 t = make_float2(0.f, 0.f);
        for (int b = 0; b < nb; ++b) {
            const float2 u = *reinterpret_cast<const float2 *>(cl.map_shared_rank(G, b) + 2 * i);
            t.x += u.x;
            t.y += u.y;
        }
        atomicAdd(reinterpret_cast<float2 *>(grad) + i, t);
    }
    static_assert(kNParams % 2 == 0, "pairs");
    cl.sync();                                    // the others' reads of G
    static_assert(kOffB4 == kOffW4 + kOut * kHid && kTrainThreads == 4 * kHid && kIn <= 8, "gradient layout");
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (tid % 32 == 0) S.loss[tid / 32] = sum;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int i = 0; i < kTrainThreads / 32; ++i) t += S.loss[i];
        atomicAdd(loss, t / (double)B);
    }
}

__global__ void k_adam(float *params, float *m, float *v, const float *g, int n, float lr, float b1, float b2,
                       float eps, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    params[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Every block allocates all 512 tensor-memory columns of its SM, so only one
// block may be resident per SM (a second would wait in tcgen05.alloc): the
// shared-memory request is padded above half of the SM's.
constexpr size_t kMinUmmaSmem = 120 * 1024;

size_t mlp_infer_smem() { return sizeof(MlpUmma) > kMinUmmaSmem ? sizeof(MlpUmma) : kMinUmmaSmem; }

// Grids up to this many staged nodes (M + 2 (K + 1)); larger ones are refused.
constexpr size_t kMaxWarmNodes = 3296;

size_t warm_mlp_smem(int M, int K)
{
    const size_t W = (size_t)M + 2 * (size_t)(K + 1);
    const size_t s = ((sizeof(MlpUmma) + 127) & ~size_t(127)) + W * sizeof(float);
    return s > kMinUmmaSmem ? s : kMinUmmaSmem;
}

int launch_warm_mlp(const WarmArgs &a, int grid, cudaStream_t s)
{
    if ((size_t)a.M + 2 * (size_t)(a.K + 1) > kMaxWarmNodes) return 1;
    const size_t smem = warm_mlp_smem(a.M, a.K);
    static SmemOptin optin;
#define FN(KK) (const void *)k_warm_mlp<KK, float>, (const void *)k_warm_mlp<KK, double>
    const void *const fn[] = {FN(2), FN(3), FN(4), FN(5)};
#undef FN
    if (!optin.raise(fn, smem)) return 1;
#define LAUNCH(KK)                                                                               \
    case KK:                                                                                     \
        if (a.fp32) k_warm_mlp<KK, float><<<grid, kMlpThreads, smem, s>>>(a);                          \
        else k_warm_mlp<KK, double><<<grid, kMlpThreads, smem, s>>>(a);                                \
        break;
    switch (a.K) {
        LAUNCH(2) LAUNCH(3) LAUNCH(4) LAUNCH(5)
    default: return 1;
    }
#undef LAUNCH
    return 0;
}

}  // namespace pic

using namespace pic;

struct pic_mlp {
    cudaStream_t stream = nullptr;
    int num_sms = 0;
    float *params = nullptr, *norm = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    double *loss = nullptr;
    int *status = nullptr;          // error bits of the inference kernel
    long long t = 0;
};

static int mlp_fail(int code, const char *msg)
{
    set_thread_error(msg);
    return code;
}

extern "C" int pic_mlp_create(const float *params, const float *norm, void *stream, pic_mlp **out)
{
    if (!out || !norm) return mlp_fail(PIC_ERR_INVALID, "pic_mlp_create: out and norm are required");
    *out = nullptr;
    pic_mlp *m = new (std::nothrow) pic_mlp();
    if (!m) return PIC_ERR_NOMEM;
    m->stream = (cudaStream_t)stream;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&m->num_sms, cudaDevAttrMultiProcessorCount, dev);
    bool ok = cudaMalloc((void **)&m->params, kNParams * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void **)&m->norm, kNorm * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void **)&m->grad, kNParams * sizeof(float) + sizeof(double)) == cudaSuccess &&
              cudaMalloc((void **)&m->m, kNParams * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void **)&m->v, kNParams * sizeof(float)) == cudaSuccess &&
              cudaMalloc((void **)&m->status, sizeof(int)) == cudaSuccess;
    if (!ok) {
        pic_mlp_destroy(m);
        return mlp_fail(PIC_ERR_NOMEM, "pic_mlp_create: cudaMalloc failed");
    }
    static_assert(kNParams % 2 == 0, "the loss behind the gradient is aligned");
    m->loss = reinterpret_cast<double *>(m->grad + kNParams);
    std::vector<float> zero(kNParams, 0.f);
    cudaMemcpyAsync(m->params, params ? params : zero.data(), kNParams * sizeof(float), cudaMemcpyHostToDevice, m->stream);
    cudaMemcpyAsync(m->norm, norm, kNorm * sizeof(float), cudaMemcpyHostToDevice, m->stream);
    cudaMemsetAsync(m->m, 0, kNParams * sizeof(float), m->stream);
    cudaMemsetAsync(m->v, 0, kNParams * sizeof(float), m->stream);
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) {
        pic_mlp_destroy(m);
        return mlp_fail(PIC_ERR_CUDA, "pic_mlp_create: upload failed");
    }
    *out = m;
    return PIC_OK;
}

extern "C" int pic_mlp_destroy(pic_mlp *m)
{
    if (!m) return PIC_OK;
    cudaStreamSynchronize(m->stream);
    cudaFree(m->params); cudaFree(m->norm); cudaFree(m->grad); cudaFree(m->m); cudaFree(m->v);
    cudaFree(m->status);
    delete m;
    return PIC_OK;
}

extern "C" int pic_mlp_get_params(pic_mlp *m, float *params_host)
{
    if (!m || !params_host) return mlp_fail(PIC_ERR_INVALID, "pic_mlp_get_params: null argument");
    if (cudaMemcpyAsync(params_host, m->params, kNParams * sizeof(float), cudaMemcpyDeviceToHost, m->stream) ||
        cudaStreamSynchronize(m->stream))
        return mlp_fail(PIC_ERR_CUDA, "pic_mlp_get_params: copy failed");
    return PIC_OK;
}

extern "C" int pic_mlp_grad(pic_mlp *m, const float *X, const float *T, int64_t B, float *grad_out, double *loss_out)
{
    if (!m || !X || !T || B < 1) return mlp_fail(PIC_ERR_INVALID, "pic_mlp_grad: invalid argument");
    static SmemOptin optin;
    if (!optin.raise((const void *)k_mlp_train, sizeof(TrainSmem)))
        return mlp_fail(PIC_ERR_CUDA, "pic_mlp_grad: shared-memory opt-in failed");
    cudaMemsetAsync(m->grad, 0, kNParams * sizeof(float) + sizeof(double), m->stream);    // and the loss behind it
    // two blocks are resident on an SM; beyond that the tiles of a block follow each other
    const long long tiles = std::min<long long>((B + kTB - 1) / kTB, 2LL * m->num_sms);
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = tiles >= kTrainCluster ? kTrainCluster : 1;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((tiles + at.val.clusterDim.x - 1) / at.val.clusterDim.x * at.val.clusterDim.x));
    cfg.blockDim = dim3(kTrainThreads);
    cfg.dynamicSmemBytes = sizeof(TrainSmem);
    cfg.stream = m->stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, k_mlp_train, (const float *)m->params, (const float *)m->norm, X, T, (long long)B, m->grad,
                           m->loss) != cudaSuccess)
        return mlp_fail(PIC_ERR_CUDA, "pic_mlp_grad: launch failed");
    if (cudaGetLastError() != cudaSuccess) return mlp_fail(PIC_ERR_CUDA, "pic_mlp_grad: launch failed");
    if (grad_out && cudaMemcpyAsync(grad_out, m->grad, kNParams * sizeof(float), cudaMemcpyDeviceToDevice, m->stream))
        return mlp_fail(PIC_ERR_CUDA, "pic_mlp_grad: copy failed");
    if (loss_out) {
        if (cudaMemcpyAsync(loss_out, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream) ||
            cudaStreamSynchronize(m->stream))
            return mlp_fail(PIC_ERR_CUDA, "pic_mlp_grad: loss copy failed");
    }
    return PIC_OK;
}

extern "C" int pic_mlp_train_step(pic_mlp *m, const float *X, const float *T, int64_t B, float lr, double *loss_out)
{
    int rc = pic_mlp_grad(m, X, T, B, nullptr, nullptr);
    if (rc) return rc;
    m->t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)m->t), c2 = 1.f - powf(b2, (float)m->t);
    k_adam<<<(kNParams + 255) / 256, 256, 0, m->stream>>>(m->params, m->m, m->v, m->grad, kNParams, lr, b1, b2,
                                                         1e-8f, c1, c2);
    if (cudaGetLastError() != cudaSuccess) return mlp_fail(PIC_ERR_CUDA, "pic_mlp_train_step: launch failed");
    if (loss_out) {
        if (cudaMemcpyAsync(loss_out, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream) ||
            cudaStreamSynchronize(m->stream))
            return mlp_fail(PIC_ERR_CUDA, "pic_mlp_train_step: loss copy failed");
    }
    return PIC_OK;
}

extern "C" int pic_mlp_infer(pic_mlp *m, const float *X, int64_t B, float *Y)
{
    if (!m || !X || !Y || B < 0) return mlp_fail(PIC_ERR_INVALID, "pic_mlp_infer: invalid argument");
    if (B == 0) return PIC_OK;
    const size_t smem = mlp_infer_smem();
    static SmemOptin optin;
    if (!optin.raise((const void *)k_mlp_infer, smem))
        return mlp_fail(PIC_ERR_CUDA, "pic_mlp_infer: shared-memory opt-in failed");
    long long blocks = (B + kMlpThreads - 1) / kMlpThreads;
    if (blocks > (long long)m->num_sms) blocks = (long long)m->num_sms;
    if (cudaMemsetAsync(m->status, 0, sizeof(int), m->stream) != cudaSuccess)
        return mlp_fail(PIC_ERR_CUDA, "pic_mlp_infer: status reset failed");
    k_mlp_infer<<<(unsigned)blocks, kMlpThreads, smem, m->stream>>>(m->params, m->norm, X, B, Y, m->status);
    int st = 0;
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(&st, m->status, sizeof(int), cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess)
        return mlp_fail(PIC_ERR_CUDA, "pic_mlp_infer: kernel failed");
    if (st) return mlp_fail(PIC_ERR_CUDA, "pic_mlp_infer: a bounded wait on the tensor cores gave up");
    return PIC_OK;
}

// accessors for the handle code (pic_api.cu)
const float *mlp_params(const pic_mlp *m) { return m->params; }
const float *mlp_norm(const pic_mlp *m) { return m->norm; }
