// Instantiations of the plain FP32 tensor-core TTM for any size and alignment (cp.async loaders).
#include <algorithm>

#include "tk_ttm_tf32.cuh"

namespace tk {
namespace tc {

void ttm_tf32_run_flat(const Ctx& c, int64_t npad, bool kmajor, const CUtensorMap& tx, const CUtensorMap& tb,
                      const TtmArgs& a) {
    ttm_tf32_dispatch<true>(c, npad, kmajor, tx, tb, a);
}

}  // namespace tc
}  // namespace tk
