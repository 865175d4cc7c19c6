// The resident stage loop instantiated for the fp64 state.
#include "fvlbm_resident.cuh"

namespace fvlbm {
FVLBM_RESIDENT_DECL(resident_fp64) {
    return resident_t<double>(v, r, (cudaStream_t)stream, scheme, stages, epoch, ab2_started, max_ctas);
}
}  // namespace fvlbm
