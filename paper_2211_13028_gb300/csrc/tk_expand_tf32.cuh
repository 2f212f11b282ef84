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

// The parts a tile's column blocks are split into: one CTA runs an item (a tile's part) per wave, and an item converts its
// tile of W again, about as long as 1.2 blocks of output take from two buffers (K <= 32), 2.8 else; the parts whose waves
// end first.  152 SMs, loss: 262144 x 512, K = 39 (1024 tiles, 16 blocks): one part 197 us, two 215, eight 385; 40000 x 512:
// 85, 81, 107; 8800 x 391: two 60, four 57, one block each 69; 1600 x 4992 BF16, K = 39 (7 tiles, 156 blocks): one
// block each 45 us, the 21 parts of a wave 18.
inline int64_t expand_parts(int64_t ntiles, int64_t nblk, int64_t nj, int64_t sms) {
    int64_t best = 1;
    double least = 1e300;
    const double convert = nj <= kChunk ? 1.2 : 2.8;
    const int64_t most = nblk < 8 * sms ? nblk : 8 * sms;
    for (int64_t ncs = 1; ncs <= most; ++ncs) {
        const int64_t waves = (ntiles * ncs + sms - 1) / sms;
        if ((double)waves * (convert + 1.0) >= least) break;
        const int64_t full = waves * sms / ntiles;  // the most parts that take no more waves
        ncs = full < most ? full : most;
        const double t = (double)waves * (convert + (double)((nblk + ncs - 1) / ncs));
        if (t < least) {
            least = t;
            best = ncs;
        }
    }
    return best;
}

// epi 0: plain product; 1: norms; 2: norms and dx.  tb: map of (M_hi, M_lo) with boxes of 32 x
// expand_cols(nj) x 2; txr: map of xref with boxes of expand_tile x expand_cols (unused when bulk).
void expand_run(const Ctx& c, int epi, tk_dtype xrdt, const CUtensorMap& tb, const CUtensorMap& txr,
                const ExpandArgs& a);
// CTAs the launch will use (pairs of partial sums).
int expand_ctas(const Ctx& c, const ExpandArgs& a);

}  // namespace tc
}  // namespace tk
