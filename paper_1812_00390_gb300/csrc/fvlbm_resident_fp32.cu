// The resident stage loop instantiated for the fp32 state.
#include "fvlbm_resident.cuh"

namespace fvlbm {
FVLBM_RESIDENT_DECL(resident_fp32) {
    return resident_t<float>(v, r, (cudaStream_t)stream, scheme, stages, epoch, ab2_started, max_ctas);
}
}  // namespace fvlbm
