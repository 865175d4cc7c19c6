// The resident stage loop instantiated for the bf16 state.
#include "fvlbm_resident.cuh"

namespace fvlbm {
FVLBM_RESIDENT_DECL(resident_bf16) {
    return resident_t<__nv_bfloat16>(v, r, (cudaStream_t)stream, scheme, stages, epoch, ab2_started, max_ctas);
}
}  // namespace fvlbm
