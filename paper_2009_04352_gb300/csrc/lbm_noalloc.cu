// Plane profile of the current state without any device allocation.
//
// Some callers cannot allocate device memory at the point where they want a
// measurement: code that runs while another component owns the allocator (a
// fixed memory budget, a pool that must not grow), host loops that have to
// stay free of allocation calls because those synchronise the device, or
// real-time drivers that forbid allocation after start-up. lbm_plane_profile
// needs block partial sums (scratch), which the rest of the library takes from
// cudaMallocAsync. Here the scratch is a file-scope __device__ array of fixed
// size instead, so the call allocates nothing.
#include <mutex>

#include "lbm.h"
#include "lbm_handle.h"
#include "lbm_fields.cuh"
#include "lbm_kernels.cuh"

namespace {

constexpr int kMaxNy = 2048;        // largest ny the fixed scratch holds
constexpr int kBlocksPerPlane = 8;  // partial sums per wall-normal plane at ny = kMaxNy (more on fewer planes)
constexpr int kMaxDevices = 64;

// Block partials [ny][blocks][K_STATS], ny * blocks <= kMaxNy * kBlocksPerPlane: 1.44 MB, held by every GPU
// that loads the library until the process exits. Every call overwrites the
// entries it uses (nothing is accumulated in place), so no clearing is needed;
// two calls whose kernels overlap on the GPU (different streams or handles)
// race on this array.
static __device__ __align__(256) double g_profile_scratch[kMaxNy * kBlocksPerPlane * lbm::K_STATS];

std::mutex g_setup_mutex;
double *g_scratch_addr[kMaxDevices] = {};

// Device address of the scratch array on the current device. In host code
// g_profile_scratch names a host-side stand-in, not device memory, so the
// address is looked up once per device (with that device current).
int scratch_on_current_device(double **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return lbm_record_error(LBM_ERR_CUDA, cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return lbm_record_error(LBM_ERR_ARG, "device ordinal out of range");
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_profile_scratch);
        if (e != cudaSuccess || !p) return lbm_record_error(LBM_ERR_CUDA, "cudaGetSymbolAddress of the profile scratch failed");
        g_scratch_addr[dev] = static_cast<double *>(p);
    }
    *out = g_scratch_addr[dev];
    return LBM_OK;
}

// The partials of each plane (k_plane_sums of lbm_fields.cuh) in fixed order, one block
// of 256 a plane: sixteen groups of threads share the partials, a column a thread (few
// planes have hundreds of partials each; added by one thread they took 40 us of a
// call at 291x13x65).
__global__ void __launch_bounds__(256) k_profile_finish(const double *__restrict__ scratch, int blocks, double *__restrict__ out)
{
    __shared__ double red[16][16];
    const int y = blockIdx.x, k = threadIdx.x & 15, grp = threadIdx.x >> 4;
    double v = 0.0;
    if (k < lbm::K_STATS) {
        const double *q = scratch + (long long)y * blocks * lbm::K_STATS + k;
#pragma unroll 4
        for (int b = grp; b < blocks; b += 16) v += q[b * lbm::K_STATS];
    }
    red[grp][k] = v;
    __syncthreads();
    if (threadIdx.x >= lbm::K_STATS) return;
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i) s += red[i][k];
    out[y * lbm::K_STATS + k] = s;
}

}  // namespace

extern "C" int lbm_plane_profile_noalloc(lbm_handle *h, double *out_dev)
{
    if (!h || !out_dev) return lbm_record_error(LBM_ERR_ARG, "NULL argument");
    if (h->g.ny > kMaxNy)
        return lbm_record_error(LBM_ERR_ARG,
                                "lbm_plane_profile_noalloc: ny exceeds the fixed scratch limit of 2048 planes");
    double *scratch = nullptr;
    const int rc = scratch_on_current_device(&scratch);
    if (rc != LBM_OK) return rc;
    // the scratch array holds kMaxNy * kBlocksPerPlane partials in all
    const int blocks = lbm::plane_sum_blocks(h, kMaxNy * kBlocksPerPlane / h->g.ny);
    lbm::plane_sums<true>(h, blocks, scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return lbm_record_error(LBM_ERR_CUDA, cudaGetErrorString(e));
    k_profile_finish<<<h->g.ny, 256, 0, h->stream>>>(scratch, blocks, out_dev);
    e = cudaGetLastError();
    if (e != cudaSuccess) return lbm_record_error(LBM_ERR_CUDA, cudaGetErrorString(e));
    return LBM_OK;
}
