// fp32 search kernels for query tiles of up to 128 (TY = 16).
#include "search_f32.cuh"

namespace oprag {
namespace f32 {

template cudaError_t launch_ty<16, false>(const Config&, const CUtensorMap&, const CUtensorMap&,
                                         const Params&, cudaStream_t);
template cudaError_t launch_ty<16, true>(const Config&, const CUtensorMap&, const CUtensorMap&,
                                         const Params&, cudaStream_t);

}  // namespace f32
}  // namespace oprag
