// Instantiations of the tensor-core TTM of strided or unaligned BF16 data.
#include <algorithm>

#include "tk_ttm_lowp.cuh"

namespace tk {
namespace tc {

void ttm_lowp_run_bf16(const Ctx& c, int64_t npad, bool kmajor, const CUtensorMap& tx, const CUtensorMap& tb,
                     const LowpArgs& a) {
    ttm_lowp_dispatch<2>(c, npad, kmajor, tx, tb, a);
}

}  // namespace tc
}  // namespace tk
