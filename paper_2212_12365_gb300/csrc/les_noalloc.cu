// les_diag_sums_noalloc: the residual / conservation reduction of
// les_get_diagnostics for callers that must not allocate device memory.
//
// Who needs it: code that runs inside a framework whose caching allocator has
// reserved (nearly) all device memory, so a cudaMalloc would fail or fragment
// the pool; and monitoring hooks called every step, where cudaMalloc/cudaFree
// would add allocation latency and may synchronise the whole device, stalling
// other streams.  Such callers pass their own state and residual buffers and
// get the sums back in their own output buffer; this entry point allocates
// nothing (no cudaMalloc, cudaFree or allocating library call).
//
// Its only scratch is the file-scope array g_partials below: SUM_PART doubles
// per reduction block, at most SUM_MAX_BLOCKS blocks.  Every GPU that loads
// the library holds it (41 KB) until the process exits.
#include <cstdio>
#include <mutex>

#include "les_internal.cuh"
#include "les_sums.cuh"

namespace {

using namespace les;

// Partials of the reduction blocks; every call overwrites what it reads.
static __device__ __align__(256) double g_partials[SUM_MAX_BLOCKS * SUM_PART];

// Points are strided over the whole grid in a fixed order, so the result
// depends only on the inputs and npoints.
__global__ void __launch_bounds__(SUM_BLOCK, SUM_BLOCKS_PER_SM) k_na_partials(const double *__restrict__ qhat,
                                                              const double *__restrict__ rhs,
                                                              long long npoints, double *part)
{
    const long long stride = (long long)gridDim.x * SUM_BLOCK;
    const long long p0 = blockIdx.x * (long long)SUM_BLOCK + threadIdx.x;
    sum_block((npoints + stride - 1) / stride,
              [&](long long t, double q[5], double r[5]) {
                  const long long p = p0 + t * stride;
#pragma unroll
                  for (int f = 0; f < 5; ++f) {
                      q[f] = p < npoints ? __ldcs(qhat + f * npoints + p) : 0.0;
                      r[f] = p < npoints ? __ldcs(rhs + f * npoints + p) : 0.0;
                  }
              },
              part);
}

__global__ void __launch_bounds__(SUM_FINAL_THREADS) k_na_final(const double *__restrict__ part, int nblocks,
                                                                double *out)
{
    sum_final(part, nblocks, out);
}

// Device address of g_partials per device.  In host code the name
// g_partials denotes a host-side stand-in, not device memory, so the address
// is looked up once per device (with that device current) and cached.
constexpr int NA_MAX_DEVICES = 64;
double *g_partials_addr[NA_MAX_DEVICES] = {nullptr};
std::mutex g_setup_mutex;

} // namespace

extern "C" int les_diag_sums_noalloc(const double *qhat, const double *rhs, int64_t npoints,
                                     double *out, void *stream)
{
    if (!qhat || !rhs || !out || npoints < 1) return LES_ERR_ARG;
    if (npoints > (int64_t)LES_NOALLOC_MAX_POINTS) {
        std::fprintf(stderr,
                     "les_diag_sums_noalloc: %lld points exceed the fixed scratch limit of %lld "
                     "points; use les_get_diagnostics for larger grids\n",
                     (long long)npoints, (long long)LES_NOALLOC_MAX_POINTS);
        return LES_ERR_ARG;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) return LES_ERR_CUDA;
    double *part = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (!g_partials_addr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_partials) != cudaSuccess || !p) {
                cudaGetLastError();
                return LES_ERR_CUDA;
            }
            g_partials_addr[dev] = (double *)p;
        }
        part = g_partials_addr[dev];
    }
    const int nblocks = sum_blocks(npoints);
    cudaStream_t st = (cudaStream_t)stream;
    k_na_partials<<<nblocks, SUM_BLOCK, 0, st>>>(qhat, rhs, (long long)npoints, part);
    k_na_final<<<1, SUM_FINAL_THREADS, 0, st>>>(part, nblocks, out);
    if (cudaGetLastError() != cudaSuccess) return LES_ERR_CUDA;
    return LES_OK;
}
