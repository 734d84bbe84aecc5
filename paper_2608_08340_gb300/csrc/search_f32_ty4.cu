// fp32 search kernels for query tiles of up to 32 (TY = 4).
#include "search_f32.cuh"

namespace oprag {
namespace f32 {

cudaError_t launch_ty4(const Config& c, const CUtensorMap& mq, const CUtensorMap& me,
                       const Params& p, cudaStream_t st) {
  switch (c.TM) {
    case 1: return launch_tm<4, 1>(c, mq, me, p, st);
    case 2: return launch_tm<4, 2>(c, mq, me, p, st);
    case 3: return launch_tm<4, 3>(c, mq, me, p, st);
    case 4: return launch_tm<4, 4>(c, mq, me, p, st);
    case 5: return launch_tm<4, 5>(c, mq, me, p, st);
    case 6: return launch_tm<4, 6>(c, mq, me, p, st);
    case 7: return launch_tm<4, 7>(c, mq, me, p, st);
    default: return launch_tm<4, 8>(c, mq, me, p, st);
  }
}

}  // namespace f32
}  // namespace oprag
