// Halo exchange of a partitioned solve on one device: after each stage, the
// stored state of every ghost cell is copied from the part that owns it (see
// fvlbm_partition.cpp for which cells and why).  One launch covers every
// message; thread (entry, unit) copies one stored unit of a cell (16 bytes where the format has them).  Sources are
// owned cells and destinations ghost cells, so no thread reads what another
// writes.
#include <cuda_runtime.h>

#include "fvlbm_device.cuh"
#include "fvlbm_internal.h"

namespace fvlbm {

namespace {

struct PartPtrs {
    void* p[FVLBM_MAX_PARTS];
};

// Copies of one cell between two buffers of a stored format, unit u of UNITS
// (16-byte units, then the remaining values; see PlainIO and SplitIO).
template <typename S> struct CellCopy {
    static constexpr int UNITS = CellIO<S>::UNITS + 1;
    static __device__ __forceinline__ void copy(void* dst, uint32_t to, const void* src, uint32_t from, int u) {
        typedef typename CellIO<S>::V V;
        if (u < CellIO<S>::UNITS) ((V*)CellIO<S>::pairs(dst, to))[u * BLK] = CellIO<S>::pairs(src, from)[u * BLK];
        else *(S*)CellIO<S>::rest(dst, to) = *CellIO<S>::rest(src, from);
    }
};
template <> struct CellCopy<__half> {
    static constexpr int UNITS = 2;
    static __device__ __forceinline__ void copy(void* dst, uint32_t to, const void* src, uint32_t from, int u) {
        if (u == 0) *(uint4*)CellIO<__half>::head(dst, to) = *CellIO<__half>::head(src, from);
        else *(uint2*)CellIO<__half>::tail(dst, to) = *CellIO<__half>::tail(src, from);
    }
};

template <typename S>
__global__ void halo_copy_kernel(const int4* __restrict__ ent, int64_t n, PartPtrs ptr) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * CellCopy<S>::UNITS) return;
    const int64_t e = t / CellCopy<S>::UNITS;
    const int4 x = ent[e];   // src part, src cell, dst part, dst cell
    CellCopy<S>::copy(ptr.p[x.z], (uint32_t)x.w, ptr.p[x.x], (uint32_t)x.y, (int)(t - e * CellCopy<S>::UNITS));
}

template <typename S>
int launch(cudaStream_t st, const int4* ent, int64_t n, const PartPtrs& p) {
    if (n == 0) return FVLBM_OK;
    const int threads = 256;
    halo_copy_kernel<S><<<(unsigned)((n * CellCopy<S>::UNITS + threads - 1) / threads), threads, 0, st>>>(ent, n, p);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? FVLBM_OK : fail(FVLBM_ERR_CUDA, "halo exchange: %s", cudaGetErrorString(e));
}

}  // namespace

int launch_halo_copy(int prec, void* stream, const int4* entries, int64_t n, void* const* part_state, int n_parts) {
    if (n_parts < 1 || n_parts > FVLBM_MAX_PARTS) return fail(FVLBM_ERR_ARG, "halo exchange: %d parts", n_parts);
    PartPtrs p{};
    for (int k = 0; k < n_parts; k++) p.p[k] = part_state[k];
    cudaStream_t st = (cudaStream_t)stream;
    switch (prec) {
        case FVLBM_FP64: return launch<double>(st, entries, n, p);
        case FVLBM_FP32_DEV: return launch<float>(st, entries, n, p);
        case FVLBM_FP16_DEV:
        case FVLBM_BF16_DEV: return launch<__half>(st, entries, n, p);
    }
    return fail(FVLBM_ERR_ARG, "halo exchange: unknown precision %d", prec);
}

}  // namespace fvlbm
