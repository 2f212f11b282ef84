// Launch interface of the fused residual kernel (tk_tc_residual.cu).
#pragma once
#include "tk_ttm_tf32.cuh"

namespace tk {
namespace tc {

struct ResidArgs {
    int64_t L, nj, R, m;
    int64_t ntiles, tiles_per_r, nk, nblk;  // work item = (row tile, block of NPAD output columns)
    void* out;                              // EPI 2: alpha * (xref - product) (XR)
    const void* xref;                       // tensor compared with the product (same layout, XR)
    float alpha;
    float xr_scale;                         // xref element = stored value * xr_scale (FP8: 1 / scale)
    double* partials;                       // per CTA {sum (xref - product)^2, sum xref^2}
    unsigned* flags;
};

// dx: EPI 2 (also store alpha * (xref - product)); npad: 16, 32, 48 or 64.
void ttm_residual_run(const Ctx& c, int64_t npad, tk_dtype xrdt, bool dx, const CUtensorMap& tx, const CUtensorMap& th,
                      const CUtensorMap& tl, const CUtensorMap& txr, const ResidArgs& a);

}  // namespace tc
}  // namespace tk
