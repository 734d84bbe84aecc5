// fp32 search kernels for query tiles of up to 32 (TY = 4).
#include "search_f32.cuh"

namespace oprag {
namespace f32 {

template cudaError_t launch_ty<4, false>(const Config&, const CUtensorMap&, const CUtensorMap&,
                                         const Params&, cudaStream_t);

}  // namespace f32
}  // namespace oprag
