// Spectral bounds without any device allocation (fo_spectral_bounds_noalloc).
//
// Some callers cannot allocate device memory at the point where they need the bounds: code
// running inside a memory pool they do not own, a host thread that must not touch the
// allocator while another component holds it, or an embedding that forbids cudaMalloc after
// start-up. This entry point needs neither a context nor a workspace: its per-block partial
// results live in a fixed file-scope device array, and the caller provides H and the output.
//
// The array is shared by every call on a device and keeps the contents of the last call.
// Each call writes every partial it later reads, so nothing has to be cleared; calls whose
// kernels overlap on the GPU (different streams, or several host threads) race on it and
// must be serialised by the caller.
#include <cuda_runtime.h>

#include "internal.cuh"

namespace fo {
namespace {

// The partials of launch_bounds_two: 3 doubles per kGershRows rows, at most 4096 of them in 128 KiB.
// The rows and their reduction are the context entry point's, hence the same bits; every size runs
// the same two kernels, so that one call loads all the device code a later, captured one needs.
constexpr int kMaxBlocks = FO_NOALLOC_MAX_N / kGershRows;
static __device__ __align__(256) double g_scratch[4 * kMaxBlocks];

// Device address of g_scratch on the current device. In host code the symbol itself is only
// a host-side stand-in and must never be passed to a kernel. The address is looked up on
// every call (cudaGetSymbolAddress is cheap and allocates nothing) rather than cached: after
// a device reset or a re-created primary context the module is loaded anew, possibly at
// another address, and a cached pointer would be stale.
cudaError_t scratch_address(double** out) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess) return e;
    *out = static_cast<double*>(p);
    return cudaSuccess;
}

}  // namespace
}  // namespace fo

extern "C" fo_status fo_spectral_bounds_noalloc(const double* dH, int64_t n, int64_t ld,
                                                double* d_bounds, void* stream) {
    using namespace fo;
    if (!dH || !d_bounds || n < 1 || ld < n) return FO_ERR_ARG;
    if (n > FO_NOALLOC_MAX_N) return FO_ERR_ARG;   // beyond the fixed scratch capacity
    double* part = nullptr;
    if (scratch_address(&part) != cudaSuccess) {
        cudaGetLastError();
        return FO_ERR_CUDA;
    }
    const cudaError_t e = launch_bounds_two(dH, n, ld, part, d_bounds, reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? FO_OK : FO_ERR_CUDA;
}
