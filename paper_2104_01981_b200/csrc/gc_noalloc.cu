// gc_compress_noalloc: exact top-k compression of one tensor whose scratch memory is a fixed
// array inside the library image, for callers that must not allocate device memory.
#include "gc.h"

#include <mutex>

#include "gc_direct.cuh"

using namespace gc;

namespace {

constexpr uint32_t kMaxN = GC_NOALLOC_MAX_N;
static_assert(sizeof(DirectScratch) == 29184, "the documented size of the fixed scratch (about 29 KB)");

// The scratch itself.  Every GPU that loads this library carries these 29,184 bytes until the
// process exits; every launch clears what it needs of them.  In host code this name is only a handle
// for cudaGetSymbolAddress; it is not a device address and must never be handed to a kernel directly.
static __device__ __align__(256) DirectScratch g_noalloc_scratch;

struct PerDevice {
    DirectScratch* scratch = nullptr;     // device address of g_noalloc_scratch on this device
    int sms = 0;
};
constexpr int kMaxDevices = 64;
PerDevice g_dev[kMaxDevices];
std::mutex g_dev_mutex;

// k = 0: nothing is sent, but the gradient still has to reach the error-feedback residual
// (r' = g + r, one rounding), exactly as the top-k rule leaves every unsent entry.
__global__ void __launch_bounds__(256) k_noalloc_fold_only(const float* __restrict__ g, float* __restrict__ r,
                                                           uint32_t n, int32_t* status_out) {
    const uint32_t nth = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += nth) r[i] = __fadd_rn(g[i], r[i]);
    if (status_out != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *status_out = GC_OK;
}

}  // namespace

extern "C" int gc_compress_noalloc(const float* grad, float* residual, uint32_t n, uint32_t k,
                                   uint32_t* out_idx, float* out_val, int32_t* device_status,
                                   void* stream) {
    if (n > kMaxN) return GC_E_TOO_LARGE;        // beyond the fixed scratch: use gc_plan + gc_compress
    if (k > n) return GC_E_INVALID;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (n > 0 && (grad == nullptr || residual == nullptr)) return GC_E_INVALID;
    if (k > 0 && (out_idx == nullptr || out_val == nullptr)) return GC_E_INVALID;
    if ((reinterpret_cast<uintptr_t>(grad) & 15u) || (reinterpret_cast<uintptr_t>(residual) & 15u))
        return GC_E_INVALID;
    if (k == 0) {
        // nothing to select (and the scratch is not needed): fold only, or just report success
        if (n > 0 || device_status != nullptr) {
            const uint32_t blocks = n == 0 ? 1u : (n + 1023u) / 1024u;
            k_noalloc_fold_only<<<(int)(blocks < 1184u ? blocks : 1184u), 256, 0, s>>>(grad, residual, n, device_status);
            if (cudaGetLastError() != cudaSuccess) return GC_E_CUDA;
        }
        return GC_OK;
    }
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        (void)cudaGetLastError();
        return GC_E_CUDA;
    }
    PerDevice pd;
    {
        // one-time set-up per device, with that device current: resolve the device address of
        // the scratch and let the kernel use as much shared memory as a share may take.  Nothing here
        // allocates.
        std::lock_guard<std::mutex> lock(g_dev_mutex);
        if (g_dev[dev].scratch == nullptr) {
            void* ptr = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
            int sms = 0, coop = 0, nb = 0, nb2 = 0;
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_topk_direct<GradF32, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDirectResident);
            if (e == cudaSuccess)
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_topk_direct<GradF32, true, true>, kBlock, kDirectResident);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb2, k_topk_direct<GradF32, false, true>, kBlock, 0);
            if (e != cudaSuccess || ptr == nullptr || sms < 1 || coop == 0 || nb < 2 || nb2 < 3) {
                (void)cudaGetLastError();
                return GC_E_CUDA;
            }
            g_dev[dev].sms = sms;
            g_dev[dev].scratch = static_cast<DirectScratch*>(ptr);
        }
        pd = g_dev[dev];
    }
    DirectArgs da{};
    da.g = grad; da.r = residual; da.n = n; da.k = k; da.out_idx = out_idx; da.out_val = out_val;
    da.status_out = device_status; da.s = pd.scratch;
    const DirectGeom dg = direct_geometry(n, pd.sms);
    // No caller can replace this array, and what two calls that overlapped against the rules left in it must not
    // outlive them: the form that clears it.
    void* args[] = {&da};
    const void* fn = dg.resident ? (const void*)k_topk_direct<GradF32, true, true> : (const void*)k_topk_direct<GradF32, false, true>;
    if (cudaLaunchCooperativeKernel(fn, dim3(dg.G), dim3(kBlock), args, dg.smem, s) != cudaSuccess) {
        (void)cudaGetLastError();
        return GC_E_CUDA;
    }
    return GC_OK;
}
