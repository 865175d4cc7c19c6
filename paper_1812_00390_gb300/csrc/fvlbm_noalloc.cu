// Total mass without any allocation by the call.
//
// fvlbm_mass keeps its block partial sums in the solver's workspace.  This
// variant keeps them in a fixed array in the library's own device memory
// instead, so a call needs no device (or host) allocation at all.  It exists
// for callers that may not allocate while they run: processes whose device
// memory is reserved up front by another allocator (a framework's caching pool
// or a fixed serving budget), and real-time loops or plugins that are not
// allowed to touch the device heap.  The paper has no counterpart.
//
// The array belongs to this file's device module.  With CUDA's default lazy
// module loading the module, and so the array, is loaded into a device's
// memory the first time the process uses it there: the first call's
// cudaGetSymbolAddress.  That first call per device can therefore allocate;
// callers make it once before the region in which they may not allocate (and
// before any stream capture).  Later calls allocate nothing.
#include <mutex>

#include <cuda_runtime.h>

#include "fvlbm_device.cuh"
#include "fvlbm_internal.h"

namespace fvlbm {

namespace {

constexpr int64_t NA_MAX_CHUNKS = 8192;   // chunks of 4096 cells: up to 33.5 M cells
constexpr int64_t NA_MAX_INST = 4096;     // instances per solver
constexpr int NA_MAX_DEVICES = 64;

// Partial sums and per-instance sums as the reduction of fvlbm_mass has them in the
// solver's workspace (DevView::part, DevView::red), then the masses.  Every GPU on which the
// module is loaded (first call there) holds these 608 KB until the process exits.
constexpr int64_t NA_PART = 2 * RED_PARTS * NA_MAX_CHUNKS, NA_RED = 2 * NA_MAX_INST;
static __device__ __align__(256) double g_noalloc_scratch[NA_PART + NA_RED + NA_MAX_INST];

std::mutex g_setup_mutex;
double* g_scratch_ptr[NA_MAX_DEVICES] = {};

__global__ void masses_kernel(const double* red, double* mass, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) mass[k] = red[2 * k];
}

// Device address of the scratch array on the current device, looked up once
// per device (the host-side symbol is only a stand-in, not a device address),
// with which the kernels of every precision are loaded.
int scratch_address(int device, double** out) {
    if (device < 0 || device >= NA_MAX_DEVICES) return fail(FVLBM_ERR_ARG, "device %d out of range", device);
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_ptr[device]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess)
            return fail(FVLBM_ERR_CUDA, "cudaGetSymbolAddress(scratch): %s", cudaGetErrorString(e));
        cudaFuncAttributes a;
        int rc = load_reduce();
        if (!rc && cudaFuncGetAttributes(&a, (const void*)masses_kernel) != cudaSuccess)
            rc = fail(FVLBM_ERR_CUDA, "mass kernel: %s", cudaGetErrorString(cudaGetLastError()));
        if (rc) return rc;
        g_scratch_ptr[device] = (double*)p;
    }
    *out = g_scratch_ptr[device];
    return FVLBM_OK;
}

}  // namespace
}  // namespace fvlbm

using namespace fvlbm;

extern "C" int fvlbm_mass_noalloc(fvlbm_solver* s, double* mass) {
    clear_error();
    SolverRef r;
    if (!mass) return fail(FVLBM_ERR_ARG, "fvlbm_mass_noalloc: mass is null");
    int rc = solver_ref(s, &r);
    if (rc) return rc;
    DevView v = *r.view;
    if (v.n_chunk > NA_MAX_CHUNKS || v.n_inst > NA_MAX_INST)
        return fail(FVLBM_ERR_ARG,
                    "fvlbm_mass_noalloc: solver too large for the fixed scratch (%lld chunks of 4096 cells, "
                    "%d instances; limits %lld chunks = %lld cells, %lld instances)",
                    (long long)v.n_chunk, v.n_inst, (long long)NA_MAX_CHUNKS, (long long)(NA_MAX_CHUNKS * 4096),
                    (long long)NA_MAX_INST);
    DeviceGuard dg(r.device);
    if (!dg.ok) return fail(FVLBM_ERR_CUDA, "fvlbm_mass_noalloc: cannot select device %d", r.device);
    double* scratch = nullptr;
    rc = scratch_address(r.device, &scratch);
    if (rc) return rc;
    // the reduction of fvlbm_mass itself, on this scratch: the same bits
    v.part = scratch;
    v.red = scratch + NA_PART;
    rc = launch_reduce(v, r.prec, r.stream, RED_MASS);
    if (rc) return rc;
    double* res = v.red + NA_RED;
    masses_kernel<<<(unsigned)((v.n_inst + 127) / 128), 128, 0, (cudaStream_t)r.stream>>>(v.red, res, v.n_inst);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(mass, res, sizeof(double) * v.n_inst, cudaMemcpyDeviceToHost, (cudaStream_t)r.stream);
    if (e != cudaSuccess) return fail(FVLBM_ERR_CUDA, "fvlbm_mass_noalloc: %s", cudaGetErrorString(e));
    return solver_sync_check(s);
}
