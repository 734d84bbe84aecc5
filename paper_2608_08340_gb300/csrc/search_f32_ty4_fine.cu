// fp32 search kernels for query tiles of up to 32 (TY = 4), finer sums.
#include "search_f32.cuh"

namespace oprag {
namespace f32 {

template cudaError_t launch_ty<4, true>(const Config&, const CUtensorMap&, const CUtensorMap&,
                                         const Params&, cudaStream_t);

}  // namespace f32
}  // namespace oprag
