// Expansions: TTMs of FP32 data with a short contraction and many output columns, the last products of a
// reconstruction (tens of elements in, hundreds of columns out), plain or fused with the comparison with X:
//
//   P[l + L*(a + m*r)] = sum_i M(i, a) W[l + L*(i + K*r)]     (W viewed as L x K x R), K <= 64 (128 fused)
//
// (3xTF32 as in tk_ttm_tf32.cuh).  They are bound by the output or by the tensor it is compared with, so
// the operand W is held: a CTA converts a tile of W rows once into TMEM (hi / lo, every K chunk) and
// runs over the tile's blocks of output columns, streaming the factor's columns and X's tiles.  The
// general kernel's order, a tile of W loaded and converted again for every block of 64 columns, bounds
// such passes (both measured with the same issue and split code): fused residual 1024^3 BF16, K = 64:
// 1327 -> 664 us; 160^4 FP32, K = 40: 983 -> 743; 512^3 FP32, K = 64: 123 (5.3 TB/s); plain 512^3,
// K = 32: 262 -> 103.  What is left at K = 64 are the MMAs (345 us of tensor time at N = 32) and the
// wait for a new tile of W, whose one buffer the last blocks still read.
//
// Persistent, one CTA per SM, 28 warps:
//   warp 0       TMA (one thread): the factor's 32 x NB chunks (hi, lo).
//   warp 1       allocates TMEM; one thread issues tcgen05.mma: per block and row subtile first the small
//                terms of every K step, A_hi * M_lo and A_lo * M_hi, then A_hi * M_hi, all into one
//                accumulator.  The tensor core rounds each addition toward zero: in this order only
//                the K / 8 last ones round at the size of the result.  Plain products, and the comparison of FP32
//                data at K <= 32, keep the even and the odd steps apart, half as many each: dX of 256^3, ranks 16,
//                1.72e-6 -> 1.62e-6 from 64 bits (FP32 FMAs 1.62e-6); 512^3, ranks 32, with dX 186 -> 201 us, the norms
//                alone 102 -> 117.  BF16 data, whose rounding is far larger, do not.
//   warps 2, 3   X's tiles: one thread by TMA, or, where X's columns have no 16-byte stride (`bulk`), two
//                by one bulk copy per column, widened to 16-byte bounds (half of the columns each).
//   warps 4-11   converters: W from global memory (any alignment; rows L*R numbered without regard to
//                slabs), split, into TMEM; the next tile's W is prefetched into L2.
//   warps 12-27  epilogue: tcgen05.ld, then stores (EPI 0), or the comparison with X's tile (EPI 1, and
//                EPI 2, which also stores alpha * (X - P)).  Two groups of 8 warps take alternate blocks.
// SUB = 2: 256-row tiles (two 128-row subtiles share every factor block, which halves its L2
// traffic: at K = 64 a block's factor is as many bytes as its BF16 tile of X), NB = 32, K <= 64.
// SUB = 1: 128-row tiles, NB = 64, K <= 128.  TMEM: four accumulators of 64 columns (or two pairs), A in the other
// 256 columns (two buffers where SUB * chunks <= 2).  FP32 data with K <= 12: residual_fma_kernel (tk_kernels.cu).
#include <algorithm>
#include <type_traits>

#include "tk_expand_tf32.cuh"

namespace tk {
namespace tc {

// NK: K chunks of 32 (compile time: the MMA thread shares its scheduler with six other warps, and a loop
// with run-time bounds and stage indexes issued an MMA in ~45 cycles, which bound K = 64: 1110 -> 664 us at 1024^3 BF16).
template <int NK, int EPI, typename XR>
struct ExpandCfg {
    static constexpr int SUB = NK <= 2 ? 2 : 1;
    static constexpr int kTile = 128 * SUB;
    static constexpr int kNB = 64 / SUB;
    static constexpr int kBStage = kNB * 256;                 // a 32 x NB chunk of M_hi and of M_lo
    static constexpr int kBS = SUB == 2 ? 6 : NK;             // factor stages (a multiple of NK)
    static constexpr int kXPitch = kTile * (int)sizeof(XR);   // bytes of a tile column (bulk: + 16)
    static constexpr int kXSlot = kNB * (kXPitch + 16);
    static constexpr int kXB = EPI ? (sizeof(XR) == 4 ? 4 : (sizeof(XR) == 2 ? 8 : 12)) : 0;  // X tiles (~130 KB in flight)
    static constexpr int kSmem = kBS * kBStage + kXB * kXSlot + 1024 + 512;
    // plain products, and the comparison of FP32 data at K <= 32: the even and the odd K steps have accumulators of
    // their own, added in the epilogue, rounding to nearest
    static constexpr bool kHalves = EPI == 0 || (NK == 1 && sizeof(XR) == 4);
    static constexpr uint32_t kAcc = kHalves ? 2 : 4;         // blocks in TMEM's accumulators (256 columns)
    static constexpr uint32_t kAccCols = 256 / kAcc;
    static constexpr int kThreads = 32 * 28;
    static constexpr int kEpi = 16;                           // epilogue warps, in two groups
    static constexpr int kEpiG = kEpi / 2;
    static constexpr int kFirstEpi = 12;
    static_assert(kXSlot % 128 == 0, "X tiles start on 128 bytes");
    static_assert(kSmem <= 227 * 1024, "SMEM budget");
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// The CTA's items once more, by exact_dot: the infinite and NaN elements of a plain product, or the whole comparison.
template <int TILE, int NB, int EPI, typename XR>
__device__ __forceinline__ void exact_expand(const ExpandArgs& args) {
    double sr = 0.0, sx = 0.0;
    for (uint32_t w = blockIdx.x; w < args.nitems; w += gridDim.x) {
        const uint32_t tile = w / args.ncs, cs = w - tile * args.ncs;
        const int64_t a0 = (int64_t)((uint64_t)args.nblk * cs / args.ncs) * NB;
        const int64_t ae = (int64_t)((uint64_t)args.nblk * (cs + 1) / args.ncs) * NB, a1 = ae < args.m ? ae : args.m;
        const int64_t l0 = (int64_t)tile * TILE, l1 = l0 + TILE < args.rows ? l0 + TILE : args.rows;
        if constexpr (EPI != 0) {
            exact_compare<XR>(args.W, args.L, args.nj, *args.info, l0, l1, a0, a1, args.xref, args.xr_scale,
                              EPI == 2 ? args.out : nullptr, args.alpha, sr, sx);
        } else {
            for (int64_t e = threadIdx.x; e < (l1 - l0) * (a1 - a0); e += blockDim.x) {
                const int64_t g = l0 + e % (l1 - l0), a = a0 + e / (l1 - l0), r = g / args.L, l = g - r * args.L;
                float* const o = static_cast<float*>(args.out) + l + args.L * (a + args.m * r);
                if (fabsf(*o) <= 3.402823466e38f) continue;
                *o = exact_dot(args.W + l + args.L * args.nj * r, args.L, 0, args.nj, *args.info, a, 1.f);
            }
        }
    }
    if (EPI != 0) residual_sums_cta(sr, sx, args.partials);
}

template <int NK, int EPI, typename XR>
__global__ void __launch_bounds__(ExpandCfg<NK, EPI, XR>::kThreads, 1)
    expand_tf32x3_kernel(const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmXr,
                         ExpandArgs args) {
    kernel_begin();
    using C = ExpandCfg<NK, EPI, XR>;
    constexpr int SUB = C::SUB;
    constexpr int NB = C::kNB;
    constexpr int XB = C::kXB ? C::kXB : 1;
    constexpr int es = (int)sizeof(XR);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* xbuf = smem + C::kBS * C::kBStage;
    uint64_t* bfull = reinterpret_cast<uint64_t*>(xbuf + C::kXB * C::kXSlot);  // [kBS] factor chunk landed
    uint64_t* bempty = bfull + C::kBS;   // [kBS] factor chunk consumed (MMA commit)
    uint64_t* xfull = bempty + C::kBS;   // [XB] X tile landed
    uint64_t* xempty = xfull + XB;       // [XB] X tile compared (epilogue warps)
    uint64_t* afull = xempty + XB;       // [2] W tile converted (converter warps)
    uint64_t* aempty = afull + 2;        // [2] W tile consumed (MMA commit)
    uint64_t* accfull = aempty + 2;      // [4] accumulator complete (MMA commit)
    uint64_t* accempty = accfull + 4;    // [4] accumulator read (the epilogue warps of a group)
    uint64_t* done = accempty + 4;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    __shared__ int again;  // infinities or NaN in the product's operands, or in the comparison (exact_dot); static: its address takes no register

    const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const bool bulk = EPI != 0 && args.bulk;
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kBS; ++s) {
            mbar_init(&bfull[s], 1);
            mbar_init(&bempty[s], 1);
        }
        for (int s = 0; s < XB; ++s) {
            mbar_init(&xfull[s], bulk ? 2 : 1);
            mbar_init(&xempty[s], C::kEpiG);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&afull[b], 8);
            mbar_init(&aempty[b], 1);
        }
        for (int b = 0; b < 4; ++b) {
            mbar_init(&accfull[b], 1);
            mbar_init(&accempty[b], C::kEpiG);
        }
        mbar_init(done, 1);
        *abort = 0;
        again = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = warp_uniform(*tmem_slot);
    unsigned* flags = args.flags;
    const uint32_t ncs = args.ncs;
    constexpr uint32_t nk = NK;
    constexpr uint32_t acols = SUB * NK * 64;             // TMEM columns of one converted tile
    constexpr uint32_t nab = 2 * acols <= 256 ? 2 : 1;    // buffers of them
    // every load a producer issued has landed before the CTA can exit
    auto drain = [&](uint64_t* bar, uint32_t n, uint32_t ring) {
        for (uint32_t q = n - (n < ring ? n : ring); q < n; ++q) {
            const uint64_t t0 = gtimer();
            while (!mbar_try_wait(&bar[q % ring], (q / ring) & 1) && gtimer() - t0 < kTimeoutNs) {
            }
        }
    };
    auto block0 = [&](uint32_t cs) { return (uint32_t)((uint64_t)args.nblk * cs / ncs); };

    if (warp == 0) {
        // ------------------------------------------------ TMA producer of the factor
        if (elect_one()) {
            uint32_t bs = 0, bph = 1, n = 0;
            bool ok = true;
            for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
                const uint32_t cs = w % ncs, b1 = block0(cs + 1);
                for (uint32_t b = block0(cs); b < b1 && ok; ++b) {
                    for (uint32_t kc = 0; kc < nk; ++kc) {
                        if (!mbar_wait(&bempty[bs], bph, abort, flags)) {
                            ok = false;
                            break;
                        }
                        mbar_expect_tx(&bfull[bs], C::kBStage);
                        tma_load_3d(smem + bs * C::kBStage, &tmB, (int)(kc * kChunk), (int)(b * NB), 0, &bfull[bs]);
                        ++n;
                        if (++bs == C::kBS) {
                            bs = 0;
                            bph ^= 1;
                        }
                    }
                }
            }
            drain(bfull, n, C::kBS);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (elect_one()) {
            const uint64_t bdesc0 = desc_sw128(smem_u32(smem));
            uint32_t bs = 0, bph = 0, a = 0, aph = 1, ab = 0, abph = 0;
            bool ok = true;
            for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
                const uint32_t tile = w / ncs, cs = w - tile * ncs, b1 = block0(cs + 1);
                if (!mbar_wait(&afull[ab], abph, abort, flags)) break;
                for (uint32_t b = block0(cs); b < b1 && ok; ++b) {
                    if (!mbar_wait(&accempty[a], aph, abort, flags)) {
                        ok = false;
                        break;
                    }
                    // the block's factor chunks, all of them before the first product
#pragma unroll
                    for (int kc = 0; kc < NK; ++kc) ok = ok && mbar_wait(&bfull[bs + kc], bph, abort, flags);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t bhi0 = bdesc0 + bs * (C::kBStage >> 4);
                    const uint32_t d0 = tbase + a * C::kAccCols, a0 = tbase + 256 + ab * acols;
#pragma unroll
                    for (int big = 0; big < 2; ++big) {
#pragma unroll
                        for (int kc = 0; kc < NK; ++kc) {
                            const uint64_t bhi = bhi0 + kc * (C::kBStage >> 4), blo = bhi + ((NB * 128) >> 4);
#pragma unroll
                            for (int sub = 0; sub < SUB; ++sub) {
                                const uint32_t a_hi = a0 + (sub * NK + kc) * 64;
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    const int step = kc * 4 + k;
                                    const bool second = C::kHalves && (step & 1);
                                    const uint32_t d = d0 + sub * NB + (second ? 64 : 0);
                                    const uint32_t more = step < (C::kHalves ? 2 : 1) ? 0u : 1u;
                                    if (big) {
                                        mma_tf32_ts(d, a_hi + 8 * k, bhi + 2 * k, idesc_tf32(NB), 1u);
                                    } else {
                                        mma_tf32_ts(d, a_hi + 8 * k, blo + 2 * k, idesc_tf32(NB), more);
                                        mma_tf32_ts(d, a_hi + 32 + 8 * k, bhi + 2 * k, idesc_tf32(NB), 1u);
                                    }
                                }
                            }
                        }
                    }
#pragma unroll
                    for (int kc = 0; kc < NK; ++kc) tc_commit(&bempty[bs + kc]);
                    bs += NK;
                    if (bs == C::kBS) {
                        bs = 0;
                        bph ^= 1;
                    }
                    tc_commit(&accfull[a]);
                    if (++a == C::kAcc) {
                        a = 0;
                        aph ^= 1;
                    }
                }
                if (!ok) break;
                tc_commit(&aempty[ab]);
                if (++ab == nab) {
                    ab = 0;
                    abph ^= 1;
                }
            }
            tc_commit(done);
            const uint64_t t0 = gtimer();
            while (!mbar_try_wait(done, 0) && gtimer() - t0 < kTimeoutNs) {
            }
        }
        __syncwarp();
    } else if (warp < 4) {
        // ------------------------------------------------ X tiles
        if (EPI && !bulk && warp == 2 && elect_one()) {
            uint32_t xs = 0, xph = 1, n = 0;
            bool ok = true;
            for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
                const uint32_t tile = w / ncs, cs = w - tile * ncs, b1 = block0(cs + 1);
                for (uint32_t b = block0(cs); b < b1; ++b) {
                    if (!mbar_wait(&xempty[xs], xph, abort, flags)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(&xfull[xs], NB * C::kXPitch);
                    tma_load_2d(xbuf + xs * C::kXSlot, &tmXr, (int)(tile * C::kTile), (int)(b * NB), &xfull[xs]);
                    ++n;
                    if (++xs == XB) {
                        xs = 0;
                        xph ^= 1;
                    }
                }
            }
            drain(xfull, n, XB);
        }
        if (bulk && elect_one()) {  // columns of any alignment
            const uint32_t j0 = (warp - 2) * (NB / 2);
            const uint8_t* X = static_cast<const uint8_t*>(args.xref);
            uint32_t xs = 0, xph = 1, nx = 0;
            bool ok = true;
            for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
                const uint32_t tile = w / ncs, cs = w - tile * ncs, b1 = block0(cs + 1);
                const int64_t l0 = (int64_t)tile * C::kTile;
                const int64_t nrow = args.L - l0 < C::kTile ? args.L - l0 : C::kTile;
                for (uint32_t b = block0(cs); b < b1; ++b) {
                    if (!mbar_wait(&xempty[xs], xph, abort, flags)) {
                        ok = false;
                        break;
                    }
                    const int64_t a0 = (int64_t)b * NB + j0;
                    // column a: bytes [beg, beg + nrow es) of X, copied from the 16-byte bound below to
                    // the one above (inside X)
                    auto span = [&](int64_t a, int64_t& src) -> uint32_t {
                        if (a >= args.m) return 0u;
                        const int64_t beg = (l0 + args.L * a) * es;
                        src = beg & ~(int64_t)15;
                        int64_t end = (beg + nrow * es + 15) & ~(int64_t)15;
                        if (end > args.xclip) end = args.xclip;
                        return end > src ? (uint32_t)(end - src) : 0u;
                    };
                    uint32_t total = 0;
                    int64_t src = 0;
                    for (int j = 0; j < NB / 2; ++j) total += span(a0 + j, src);
                    if (total) mbar_expect_tx(&xfull[xs], total);
                    else mbar_arrive(&xfull[xs]);
                    const uint32_t dst = smem_u32(xbuf + xs * C::kXSlot) + j0 * (C::kXPitch + 16);
                    for (int j = 0; j < NB / 2; ++j) {
                        const uint32_t n = span(a0 + j, src);
                        if (n) bulk_load(dst + j * (C::kXPitch + 16), X + src, n, &xfull[xs]);
                    }
                    ++nx;
                    if (++xs == XB) {
                        xs = 0;
                        xph ^= 1;
                    }
                }
            }
            drain(xfull, nx, XB);
        }
        __syncwarp();
        if (warp == 3) {  // whether the factor has such values
            int any = 0;
#pragma unroll 8
            for (uint32_t i = lane; i < args.info->nbad; i += 32) any |= args.info->bad[i];
            if (any) again = 1;
        }
    } else if (warp < C::kFirstEpi) {
        // ------------------------------------------------ converters: W tile -> TF32 hi / lo in TMEM
        const int q = warp & 3, hs = (warp - 4) >> 2;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        const uint32_t L = (uint32_t)args.L, nj = (uint32_t)args.nj;
        // the offset into W of this lane's row of a subtile, -1 beyond the last row
        auto row_of = [&](uint32_t tile, int sub) -> int64_t {
            const uint32_t g = tile * C::kTile + sub * 128 + 32 * q + lane;
            if (g >= args.rows) return -1;
            const uint32_t r = L == 1 ? g : g / L;
            return (int64_t)(g - r * L) + args.L * args.nj * r;
        };
        uint32_t ab = 0, abph = 1;
        float bad = 0.f;
        bool ok = true;
        for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
            const uint32_t tile = w / ncs, nst = SUB * nk;  // steps: (subtile, K chunk)
            // a step's loads are in flight while the one before is converted, and the first two before the
            // buffer is free
            float v[2][16];
            auto load = [&](uint32_t st, float (&x)[16]) {
                const int64_t base = row_of(tile, SUB == 2 && st >= nk ? 1 : 0);
                const uint32_t i0 = (st >= nk && SUB == 2 ? st - nk : st) * kChunk + 16 * hs;
#pragma unroll
                for (int ii = 0; ii < 16; ++ii)
                    x[ii] = base >= 0 && i0 + ii < nj ? args.W[base + args.L * (i0 + ii)] : 0.f;
            };
            auto store = [&](uint32_t st, const float (&x)[16]) {
                uint32_t hi[16], lo[16];
#pragma unroll
                for (int ii = 0; ii < 16; ++ii) {
                    split_tf32(x[ii], hi[ii], lo[ii]);
                    bad = fmaf(__uint_as_float(lo[ii]), 0.f, bad);  // a NaN once lo is infinite or one
                }
                const uint32_t ta = tbase + lane_base + 256 + ab * acols + st * 64 + 16 * hs;
                __syncwarp();
                tmem_st16(ta, hi);
                tmem_st16(ta + 32, lo);
            };
            load(0, v[0]);
            if (nst > 1) load(1, v[1]);
            if (!__all_sync(0xffffffffu, mbar_wait(&aempty[ab], abph, abort, flags))) {
                ok = false;
                break;
            }
            tc_fence_after();
            for (uint32_t st = 0; st < nst; st += 2) {
                store(st, v[0]);
                if (st + 2 < nst) load(st + 2, v[0]);
                if (st + 1 < nst) {
                    store(st + 1, v[1]);
                    if (st + 3 < nst) load(st + 3, v[1]);
                }
            }
            if (!ok) break;
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&afull[ab]);
            if (++ab == nab) {
                ab = 0;
                abph ^= 1;
            }
            // the next item's rows into L2 while this one's blocks run
            if (w + gridDim.x < args.nitems) {
                const uint32_t next = (w + gridDim.x) / ncs;
                for (int sub = 0; sub < SUB; ++sub) {
                    const int64_t base = row_of(next, sub);
                    if (base < 0) continue;
                    for (uint32_t i = 16 * hs; i < nj; i += (i & 15) == 15 ? 17 : 1)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(args.W + base + args.L * i));
                }
                __syncwarp();
            }
        }
        if (bad != bad) again = 1;
    } else if (warp < C::kFirstEpi + C::kEpi) {
        // ------------------------------------------------ epilogue
        // warp e: group e / 8; within it TMEM lane quarter warp % 4 and the subtile (SUB = 2) or the block's
        // column half; two 16-column slices each
        const int e = warp - C::kFirstEpi, q = warp & 3;
        const uint32_t grp = e >> 3;
        const int part = (e >> 2) & 1, sub = SUB == 2 ? part : 0;
        const int cbase = SUB == 2 ? 0 : 32 * part;
        const int rho = sub * 128 + 32 * q + lane;  // row of the tile
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        const uint32_t L = (uint32_t)args.L;
        const int ostep = bulk ? (int)((args.L * es) & 15) : 0;
        // running sums as double-float pairs (hi + lo, Knuth two-sum): FP32 instructions only, the FP64
        // pipe (1/64 of FP32 here) stays out of the per-item work
        float srh = 0.f, srl = 0.f, sxh = 0.f, sxl = 0.f;
        uint32_t it = 0, xs = grp, xph = 0;  // (kXB is even: a slot always falls to the same group)
        bool ok = true;
        for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
            const uint32_t tile = w / ncs, cs = w - tile * ncs, b1 = block0(cs + 1);
            const uint32_t g = tile * C::kTile + rho;
            const bool valid = g < args.rows;
            const uint32_t r = L == 1 ? g : g / L;
            const int64_t obase = (int64_t)(g - r * L) + args.L * args.m * r;
            for (uint32_t b = block0(cs); b < b1; ++b, ++it) {
                if ((it & 1) != grp) continue;
                const uint32_t a = it % C::kAcc;
                bool got = mbar_wait(&accfull[a], (it / C::kAcc) & 1, abort, flags);
                if (EPI) got = got && mbar_wait(&xfull[xs], xph, abort, flags);
                if (!__all_sync(0xffffffffu, got)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t ta = tbase + lane_base + a * C::kAccCols + sub * NB + cbase;
#pragma unroll
                for (int sl = 0; sl < 2; ++sl) {
                    const int c16 = cbase + 16 * sl;
                    float p[16], p2[16];
                    __syncwarp();
                    tmem_ld16(ta + 16 * sl, p);
                    if (C::kHalves) tmem_ld16(ta + 64 + 16 * sl, p2);
                    const int64_t col = (int64_t)b * NB + c16;
                    const int ncol = args.m - col < 16 ? (int)(args.m - col) : 16;  // valid columns of the slice
                    XR x[16];
                    if (EPI != 0 && valid) {
                        if (!bulk) {
                            const XR* xt = reinterpret_cast<const XR*>(xbuf + xs * C::kXSlot) + c16 * C::kTile + rho;
#pragma unroll
                            for (int i = 0; i < 16; ++i) x[i] = xt[i * C::kTile];
                        } else {
                            // column j of the tile starts at its first element's offset from a 16-byte bound
                            const uint8_t* xt = xbuf + xs * C::kXSlot + c16 * (C::kXPitch + 16) + rho * es;
                            const int o0 = (int)((((int64_t)tile * C::kTile + col * args.L) * es) & 15);
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                                x[i] = *reinterpret_cast<const XR*>(xt + i * (C::kXPitch + 16) +
                                                                    ((o0 + i * ostep) & 15));
                            if ((obase + (col + 15) * args.L + 1) * es > args.xclip) {
                                // the last elements of X, which 16-byte copies inside it cannot reach
                                const XR* xp = static_cast<const XR*>(args.xref) + obase + col * args.L;
#pragma unroll
                                for (int i = 0; i < 16; ++i)
                                    if (i < ncol && (obase + (col + i) * args.L + 1) * es > args.xclip)
                                        x[i] = xp[i * args.L];
                            }
                        }
                    }
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (C::kHalves) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) p[i] += p2[i];
                    }
                    if (sl == 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&accempty[a]);
                    }
                    if (!valid) continue;
                    if (EPI == 0) {
                        float* op = static_cast<float*>(args.out) + obase + col * args.L;
                        if (ncol == 16) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) op[i * args.L] = p[i];
                        } else {
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                                if (i < ncol) op[i * args.L] = p[i];
                        }
                    } else {
                        float fr = 0.f, fx = 0.f;
                        XR* op = EPI == 2 ? static_cast<XR*>(args.out) + obase + col * args.L : nullptr;
                        auto one = [&](int i) {
                            float xv = x_to_f32(x[i]);
                            if constexpr (std::is_same<XR, __nv_fp8_e4m3>::value) xv *= args.xr_scale;  // 1 / scale
                            const float dv = xv - p[i];
                            fr = fmaf(dv, dv, fr);
                            fx = fmaf(xv, xv, fx);
                            if constexpr (EPI == 2) xr_store(op + i * args.L, args.alpha * dv);
                        };
                        if (ncol == 16) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) one(i);
                        } else {
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                                if (i < ncol) one(i);
                        }
                        if (!(fr <= 3.402823466e38f)) again = 1;
                        ef_add(srh, srl, fr);
                        ef_add(sxh, sxl, fx);
                    }
                }
                if (EPI) {
                    __syncwarp();  // the warp's reads of the tile are done before lane 0 releases it
                    if (lane == 0) mbar_arrive(&xempty[xs]);
                    xs += 2;
                    if (xs >= (uint32_t)XB) {
                        xs = grp;
                        xph ^= 1;
                    }
                }
            }
        }
        if (EPI != 0) {
            residual_sums<C::kEpi>(e, lane, ef_value(srh, srl), ef_value(sxh, sxl), args.partials);
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tbase) : "memory");
    }
    if (again && !*abort) exact_expand<C::kTile, C::kNB, EPI, XR>(args);
}

int expand_ctas(const Ctx& c, const ExpandArgs& a) { return (int)std::min<int64_t>(a.nitems, grid_sms(c)); }

template <int NK, int EPI, typename XR>
static void launch_one(const Ctx& c, const CUtensorMap& tb, const CUtensorMap& txr, const ExpandArgs& a) {
    using Cf = ExpandCfg<NK, EPI, XR>;
    auto kern = expand_tf32x3_kernel<NK, EPI, XR>;
    static std::atomic<uint64_t> opted{0};
    smem_opt_in(opted, reinterpret_cast<const void*>(kern), Cf::kSmem);
    run_kernel(c, kern, expand_ctas(c, a), Cf::kThreads, Cf::kSmem, tb, txr, a);
}

void expand_run(const Ctx& c, int epi, tk_dtype xrdt, const CUtensorMap& tb, const CUtensorMap& txr,
                const ExpandArgs& a) {
    if (epi == 0) {
        if (a.nk == 1) launch_one<1, 0, float>(c, tb, txr, a);
        else launch_one<2, 0, float>(c, tb, txr, a);
        return;
    }
#define TK_EXPAND(NK)                                                                     \
    case NK:                                                                              \
        if (xrdt == TK_FP8_E4M3) launch_one<NK, 1, __nv_fp8_e4m3>(c, tb, txr, a);           \
        else if (xrdt == TK_BF16 && epi == 1) launch_one<NK, 1, __nv_bfloat16>(c, tb, txr, a); \
        else if (xrdt == TK_BF16) launch_one<NK, 2, __nv_bfloat16>(c, tb, txr, a);          \
        else if (epi == 1) launch_one<NK, 1, float>(c, tb, txr, a);                         \
        else launch_one<NK, 2, float>(c, tb, txr, a);                                       \
        break;
    switch (a.nk) {
        TK_EXPAND(1)
        TK_EXPAND(2)
        TK_EXPAND(3)
        TK_EXPAND(4)
        default: fail(TK_ERR_SHAPE, "expand: contraction too long");
    }
#undef TK_EXPAND
}

}  // namespace tc
}  // namespace tk
