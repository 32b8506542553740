// pic_noalloc.cu -- the path-integrated current deposit without any allocation.
//
// Some callers cannot allocate device memory at the point where they need a
// deposit: code running inside a memory pool that must not grow, a host that
// has handed the whole device heap to another component, or a plugin that is
// not allowed to own CUDA allocations.  pic_deposit_current_noalloc() serves
// them: it needs no handle, and its only scratch is the file-scope device array
// below (2 MiB per GPU that loads the library, held until the process exits).
//
// Scratch layout (doubles): [0, 64) header (status word), then the path moments of the
// cells (pic_poly.cuh: K per cell), in several replicas that the blocks take in turn.
// Every call clears what it uses first, so the contents left by the previous call do not
// leak into the result.  All calls share the array: two calls whose kernels overlap on
// the GPU (different streams, or different host threads) race and corrupt each other's
// result; order them on one stream.
//
// The markers come in any order, so their moments go straight to the scratch by double
// additions in L2, K per path piece, which is what bounds the call: 91 us for 1e6 markers
// on 1000 cells, reach 1.5 cells, degree 3.  (Rows of nodes per block in shared memory,
// where a double addition is a compare-and-swap loop, and one thread per node to add the
// rows: 529 us.)
#include <algorithm>
#include <cmath>
#include <mutex>

#include "pic.h"
#include "pic_internal.h"
#include "pic_poly.cuh"

namespace {

constexpr size_t kScratchDoubles = size_t(1) << 18;   // 2 MiB
constexpr int kHeader = 64;                            // doubles reserved for the status word
constexpr int kMaxDisp = 64;                           // cells a displacement may span
constexpr int kMaxDevices = 64;

static __device__ __align__(256) double g_scratch[kScratchDoubles];

__constant__ pic::SplineTab c_spline_na = pic::make_spline_tab();

struct NoallocArgs {
    int M, reps;
    long long np;
    double dx, w;
    const double *x, *disp;
    double *mom;        // scratch: reps x M x K moments h S_m
    int *status;        // scratch header
};

template <int K>
__global__ void __launch_bounds__(256) k_noalloc_moments(NoallocArgs A)
{
    double *mom = A.mom + (size_t)(blockIdx.x % A.reps) * A.M * K;
    const double span = (double)A.M;
    bool bad = false;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < A.np; a += stride) {
        double u = pic::quotient(A.x[a], A.dx);
        const double d = pic::quotient(A.disp[a], A.dx);
        // positions and displacements must be finite and a displacement may span at most
        // kMaxDisp cells
        if (!isfinite(u) || !isfinite(d) || !(fabs(d) <= (double)kMaxDisp)) { bad = true; continue; }
        // periodic: wrap the cell coordinate into [0, M) before taking its integer part
        if (!(u >= 0.0 && u < span)) u -= span * ::floor(u / span);
        const double f = ::floor(u);
        int g = pic::wrap_cell((int)f, A.M);
        const double v0 = (u - f) - 0.5;
        int n;
        double v1;
        pic::path_end(v0, d, n, v1);
        const int an = abs(n);
        const double edge = n > 0 ? 0.5 : -0.5;
        for (int q = 0; q <= an; ++q) {
            const double va = q == 0 ? v0 : -edge, vb = q == an ? v1 : edge;
            double x[K];
            pic::piece_moments<K, double>(va, vb, an == 0 ? d : vb - va, x);
#pragma unroll
            for (int m = 0; m < K; ++m) atomicAdd(&mom[(size_t)g * K + m], x[m]);
            g = pic::wrap_once(g + (n > 0 ? 1 : -1), A.M);
        }
    }
    if (bad) atomicOr(A.status, 1);
}

// out[i] = w dx sum_r sum_m B_{K-1}[r][m] / (m + 1) (sum over the replicas, in order, of the
// moments of cell i + r).  A block takes kNodes nodes and the K - 1 cells above them.
constexpr int kNodes = 32;

template <int K>
__global__ void __launch_bounds__(128) k_noalloc_reduce(NoallocArgs A, double *out)
{
    __shared__ double s_mom[(kNodes + K) * K];
    const int i0 = blockIdx.x * kNodes;
    for (int q = threadIdx.x; q < (kNodes + K - 1) * K; q += blockDim.x) {
        const double *src = A.mom + (size_t)pic::wrap_cell(i0 + q / K, A.M) * K + q % K;
        double s = 0.0;
        for (int r = 0; r < A.reps; ++r) s += src[(size_t)r * A.M * K];
        s_mom[q] = s;
    }
    __syncthreads();
    const int i = i0 + threadIdx.x;
    if (threadIdx.x >= kNodes || i >= A.M) return;
    double v = 0.0;
#pragma unroll
    for (int m = 0; m < K; ++m) {
        double s = 0.0;
#pragma unroll
        for (int r = 0; r < K; ++r) s = fma(c_spline_na.b[K - 1][r][m], s_mom[(threadIdx.x + r) * K + m], s);
        v += s / (double)(m + 1);
    }
    out[i] = A.w * A.dx * v;
}

__global__ void k_noalloc_clear(int *status, double *mom, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *status = 0;
    for (long long q = i; q < n; q += (long long)gridDim.x * blockDim.x) mom[q] = 0.0;
}

struct DeviceSetup {
    double *scratch = nullptr;   // device address of g_scratch on this device
    int num_sms = 0;
};

std::mutex g_mu;
DeviceSetup g_dev[kMaxDevices];

// Once per device, with that device current: resolve the scratch address.
int setup_device(int dev, DeviceSetup **out, const char **why)
{
    std::lock_guard<std::mutex> lk(g_mu);
    DeviceSetup &d = g_dev[dev];
    if (!d.scratch) {
        double *p = nullptr;
        if (cudaGetSymbolAddress((void **)&p, g_scratch) != cudaSuccess || !p) {
            *why = "cudaGetSymbolAddress of the deposit scratch failed";
            return PIC_ERR_CUDA;
        }
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            *why = "cudaDeviceGetAttribute failed";
            return PIC_ERR_CUDA;
        }
        d.num_sms = sms;
        d.scratch = p;
    }
    *out = &d;
    return PIC_OK;
}

int fail_nohandle(int code, const char *msg)
{
    pic::set_thread_error(msg);
    return code;
}

}  // namespace

extern "C" int pic_deposit_current_noalloc(double L, int32_t nx, int32_t degree, int64_t np,
                                           double weight, const double *x, const double *disp,
                                           double *out, void *stream)
{
    if (!(L > 0) || nx < 8 || degree < 2 || degree > 5 || np < 0 || np > 2147483647LL || !out ||
        (np > 0 && (!x || !disp)) || !std::isfinite(weight))
        return fail_nohandle(PIC_ERR_INVALID, "pic_deposit_current_noalloc: invalid argument");
    if (nx > 8192)
        return fail_nohandle(PIC_ERR_INVALID,
                             "pic_deposit_current_noalloc: nx > 8192 exceeds the fixed 2 MiB scratch");
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return fail_nohandle(PIC_ERR_CUDA, "pic_deposit_current_noalloc: no usable current device");
    DeviceSetup *d = nullptr;
    const char *why = nullptr;
    int rc = setup_device(dev, &d, &why);
    if (rc) return fail_nohandle(rc, why);

    NoallocArgs a{};
    a.M = nx;
    a.np = np;
    a.dx = L / nx;
    a.w = weight;
    a.x = x;
    a.disp = disp;
    a.status = reinterpret_cast<int *>(d->scratch);
    a.mom = d->scratch + kHeader;
    // replicas spread the additions of a small grid; clearing and adding them up costs more
    // than it gives beyond some 2^16 doubles
    const long long row = (long long)nx * degree;
    const int grid = (int)std::max<long long>(1, std::min<long long>(8LL * d->num_sms, (np + 255) / 256));
    a.reps = (int)std::max<long long>(1, std::min<long long>(std::min<long long>(32, grid), (1LL << 16) / row));
    static_assert(kHeader + 8192 * 5 <= kScratchDoubles && kHeader + (1u << 16) <= kScratchDoubles, "scratch");
    k_noalloc_clear<<<(unsigned)((a.reps * row + 1023) / 1024), 256, 0, s>>>(a.status, a.mom, a.reps * row);
    const int nodes = (nx + kNodes - 1) / kNodes;
#define NOALLOC(K)                                           \
    k_noalloc_moments<K><<<grid, 256, 0, s>>>(a);            \
    k_noalloc_reduce<K><<<nodes, 128, 0, s>>>(a, out);       \
    break;
    switch (degree) {
    case 2: NOALLOC(2)
    case 3: NOALLOC(3)
    case 4: NOALLOC(4)
    default: NOALLOC(5)
    }
#undef NOALLOC
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail_nohandle(PIC_ERR_CUDA, cudaGetErrorString(e));
    int status = 0;
    e = cudaMemcpyAsync(&status, a.status, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return fail_nohandle(PIC_ERR_CUDA, cudaGetErrorString(e));
    if (status)
        return fail_nohandle(PIC_ERR_NUMERIC,
                             "pic_deposit_current_noalloc: a position or displacement is not finite, or a displacement spans more than 64 cells");
    return PIC_OK;
}
