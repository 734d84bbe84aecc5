// fp32 search kernels for query tiles of up to 64 (TY = 8).
#include "search_f32.cuh"

namespace oprag {
namespace f32 {

cudaError_t launch_ty8(const Config& c, const CUtensorMap& mq, const CUtensorMap& me,
                       const Params& p, cudaStream_t st) {
  switch (c.TM) {
    case 5: return launch_tm<8, 5>(c, mq, me, p, st);
    case 6: return launch_tm<8, 6>(c, mq, me, p, st);
    case 7: return launch_tm<8, 7>(c, mq, me, p, st);
    default: return launch_tm<8, 8>(c, mq, me, p, st);
  }
}

}  // namespace f32
}  // namespace oprag
