// Instantiations of the plain FP32 tensor-core TTM fused with a residual.
#include <algorithm>

#include "tk_ttm_tf32.cuh"

namespace tk {
namespace tc {

void ttm_tf32_run_residual(const Ctx& c, bool flat, const CUtensorMap& tx, const CUtensorMap& tb, const TtmResArgs& a) {
    if (flat) ttm_tf32_launch<64, false, true, true>(c, tx, tb, a);
    else ttm_tf32_launch<64, false, false, true>(c, tx, tb, a);
}

}  // namespace tc
}  // namespace tk
