// Launch interface of the expansion kernel (tk_expand_tf32.cu).
#pragma once
#include "tk_ttm_tf32.cuh"

namespace tk {
namespace tc {

constexpr int64_t kExpandK = 64;        // contracted elements of a plain expansion, at most
constexpr int64_t kExpandKResid = 128;  // of a fused residual

struct ExpandArgs {
    int64_t L, nj, m;
    const float* W;           // L x nj x R
    uint32_t rows;            // L R
    uint32_t ntiles, nblk;    // row tiles, blocks of output columns
    uint32_t ncs, nitems;     // parts the blocks of a tile are split into; items = ntiles ncs
    uint32_t nk;              // K chunks of 32
    void* out;                // EPI 0: the product (FP32); EPI 2: alpha * (xref - product) (XR)
    const void* xref;         // EPI 1, 2: tensor compared with the product (its layout, R == 1)
    float alpha;
    float xr_scale;           // xref element = stored value * xr_scale (FP8: 1 / scale)
    double* partials;         // EPI 1, 2: per CTA {sum (xref - product)^2, sum xref^2}
    uint32_t bulk;            // EPI 1, 2: xref has no 16-byte column stride, its tiles come by bulk copies
    int64_t xclip;            // bulk: xref's bytes below this are covered by 16-byte copies inside it
    unsigned* flags;
    const FactorInfo* info;
};
static_assert(sizeof(ExpandArgs) <= 128, "see TtmResArgs");

// The row tile (256, or 128 for nj > kExpandK) and the output columns per block.
inline int64_t expand_tile(int64_t nj) { return nj <= kExpandK ? 256 : 128; }
inline int64_t expand_cols(int64_t nj) { return nj <= kExpandK ? 32 : 64; }

// epi 0: plain product; 1: norms; 2: norms and dx.  tb: map of (M_hi, M_lo) with boxes of 32 x
// expand_cols(nj) x 2; txr: map of xref with boxes of expand_tile x expand_cols (unused when bulk).
void expand_run(const Ctx& c, int epi, tk_dtype xrdt, const CUtensorMap& tb, const CUtensorMap& txr,
                const ExpandArgs& a);
// CTAs the launch will use (pairs of partial sums).
int expand_ctas(const Ctx& c, const ExpandArgs& a);

}  // namespace tc
}  // namespace tk
