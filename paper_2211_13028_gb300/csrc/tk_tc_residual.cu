// The fused residual on tensor cores: the last TTM of a reconstruction (a strided mode of FP32 data, the
// arithmetic of tk_ttm_tf32.cuh), whose product is compared with X in the epilogue instead of being stored.
//
// Persistent, one CTA per SM.  Warp roles: 0 TMA producer, 1 TMEM allocation + MMA issue, 2-3 idle, 8
// converter warps (only the small reconstruction operand is converted), 16 epilogue warps (every element
// of X is compared): four per TMEM lane quarter, splitting the columns.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <type_traits>

#include "tk_tc_residual.cuh"

namespace tk {
namespace tc {

struct Warps {
    static constexpr int kConv = 8;
    static constexpr int kEpi = 16;    // epilogue warps: 4 lane quarters x column groups
    static constexpr int kColGroups = kEpi / 4;
    static constexpr int kFirstConv = 4;
    static constexpr int kFirstEpi = 4 + kConv;
    static constexpr int kThreads = 32 * (4 + kConv + kEpi);
};

template <int NPAD, typename XR>
struct Cfg {
    static constexpr int kBBytes = NPAD * 128;  // one of M_hi / M_lo: NPAD rows of 128 B
    static constexpr int kStage = kXBytes + 2 * kBBytes;
    static constexpr int kXrBytes = kRows * NPAD * (int)sizeof(XR);  // X tile compared in the epilogue
    // X tiles in flight: about 128 KB, enough to cover HBM latency at one SM's share of
    // the bandwidth (2 to 8 tiles)
    static constexpr int kXrFit = (128 * 1024) / kXrBytes;
    static constexpr int kXrBufs = kXrFit > 8 ? 8 : (kXrFit < 2 ? 2 : kXrFit);
    static constexpr int kBudget = 210 * 1024 - kXrBufs * kXrBytes;
    static constexpr int kStages = kBudget / kStage > 12 ? 12 : kBudget / kStage;
    static constexpr int kAccCols = 2 * NPAD;      // accumulators: 2 x (2*NPAD) columns
    static constexpr int kAcc0 = 0;
    static constexpr int kABuf = 2 * kAccCols;     // A buffers: NA x 64 columns (hi 32 | lo 32)
    static constexpr int kNA = (512 - kABuf) / 64 > 6 ? 6 : (512 - kABuf) / 64;  // >= 2
    static constexpr int kSmem = kStages * kStage + kXrBufs * kXrBytes + 1024 + 512;
    static_assert(kNA >= 2, "TMEM budget");
    static_assert(kStages >= 2, "SMEM budget");
};

// (hi, lo) += b with Knuth's two-sum on the high part; the low part collects
// the rounding errors (a double-float running sum of FP32 terms).
__device__ __forceinline__ void ef_add(float& hi, float& lo, float b) {
    const float s = __fadd_rn(hi, b);
    const float v = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, v)), __fsub_rn(b, v));
    hi = s;
    lo = __fadd_rn(lo, e);
}

__device__ __forceinline__ float xr_to_f32(float v) { return v; }
__device__ __forceinline__ float xr_to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float xr_to_f32(__nv_fp8_e4m3 v) { return static_cast<float>(v); }
__device__ __forceinline__ void xr_store(float* p, float v) { *p = v; }
__device__ __forceinline__ void xr_store(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// EPI 1: accumulate the residual norms against xref; 2: as 1 and also store alpha * (xref - product).  XR: element type of xref
// and of the EPI 2 output (FP32, or BF16 for BF16 data).
template <int NPAD, int EPI, typename XR>
__global__ void __launch_bounds__(Warps::kThreads, 1)
    ttm_residual_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmBhi,
                      const __grid_constant__ CUtensorMap tmBlo, const __grid_constant__ CUtensorMap tmXr,
                      ResidArgs args) {
    using C = Cfg<NPAD, XR>;
    constexpr int S = C::kStages;
    constexpr int NA = C::kNA;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    float* xr_buf = reinterpret_cast<float*>(smem + S * C::kStage);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * C::kStage + C::kXrBufs * C::kXrBytes);
    uint64_t* full = bars;               // [S] TMA landed
    uint64_t* xfree = bars + S;          // [S] stage consumed (one arrival per converter warp + 1 MMA commit)
    uint64_t* afull = bars + 2 * S;      // [NA] A buffer written (one arrival per converter warp)
    uint64_t* aempty = afull + NA;       // [NA] A buffer consumed (MMA commit)
    uint64_t* accfull = aempty + NA;     // [2] accumulator complete (MMA commit)
    uint64_t* accempty = accfull + 2;    // [2] accumulator drained (one arrival per epilogue warp)
    constexpr int XB = C::kXrBufs;
    uint64_t* xrfull = accempty + 2;     // [XB] residual X tile landed
    uint64_t* xrempty = xrfull + XB;     // [XB] residual X tile consumed (one arrival per epilogue warp)
    uint64_t* done = xrempty + XB;       // [1] every issued MMA complete
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    using W = Warps;
    __shared__ double red[2 * W::kEpi];

    const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&xfree[s], 9);   // 8 converter warps + 1 MMA commit
        }
        for (int b = 0; b < NA; ++b) {
            mbar_init(&afull[b], 8);   // 8 converter warps
            mbar_init(&aempty[b], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accfull[b], 1);
            mbar_init(&accempty[b], W::kEpi);   // one arrival per epilogue warp
        }
        for (int b = 0; b < XB; ++b) {
            mbar_init(&xrfull[b], 1);
            mbar_init(&xrempty[b], W::kEpi);
        }
        mbar_init(done, 1);
        *abort = 0;
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
    const int64_t nk = args.nk;
    const int64_t nitems = args.ntiles * args.nblk;

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (elect_one()) {
            int64_t it = 0, item = 0;
            bool ok = true;
            for (int64_t w = blockIdx.x; w < nitems && ok; w += gridDim.x, ++item) {
                const int64_t t = w / args.nblk, nb = w % args.nblk;
                const int64_t rr = t / args.tiles_per_r, l0 = (t % args.tiles_per_r) * kRows;
                {  // the X tile the epilogue compares this item's product with
                    const int xb = (int)(item % XB);
                    if (!mbar_wait(&xrempty[xb], (uint32_t)(((item / XB) & 1) ^ 1), abort, flags)) break;
                    mbar_expect_tx(&xrfull[xb], C::kXrBytes);
                    tma_load_3d(reinterpret_cast<uint8_t*>(xr_buf) + xb * C::kXrBytes, &tmXr, (int)l0, (int)(nb * NPAD),
                                (int)rr, &xrfull[xb]);
                }
                for (int64_t kc = 0; kc < nk; ++kc, ++it) {
                    const int s = (int)(it % S);
                    const uint32_t ph = (uint32_t)((it / S) & 1);
                    if (!mbar_wait(&xfree[s], ph ^ 1, abort, flags)) {
                        ok = false;
                        break;
                    }
                    uint8_t* xs = smem + s * C::kStage;
                    uint8_t* bs = xs + kXBytes;
                    mbar_expect_tx(&full[s], C::kStage);
                    // one unswizzled 128 x 32 box: rows i of 128 floats (512 B)
                    tma_load_3d(xs, &tmX, (int)l0, (int)(kc * kChunk), (int)rr, &full[s]);
                    tma_load_2d(bs, &tmBhi, (int)(kc * kChunk), (int)(nb * NPAD), &full[s]);
                    tma_load_2d(bs + C::kBBytes, &tmBlo, (int)(kc * kChunk), (int)(nb * NPAD), &full[s]);
                }
            }
            // drain: every issued load has landed before the CTA can exit
            const int64_t n_out = it < S ? it : S;
            for (int64_t q = it - n_out; q < it; ++q) {
                const uint64_t t0 = gtimer();
                while (!mbar_try_wait(&full[q % S], (uint32_t)((q / S) & 1)) && gtimer() - t0 < kTimeoutNs) {
                }
            }
            const int64_t n_xr = item < XB ? item : XB;
            for (int64_t q = item - n_xr; q < item; ++q) {
                const uint64_t t0 = gtimer();
                while (!mbar_try_wait(&xrfull[q % XB], (uint32_t)((q / XB) & 1)) && gtimer() - t0 < kTimeoutNs) {
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (elect_one()) {
            int64_t it = 0, ab = 0, acc = 0;
            bool ok = true;
            for (int64_t w = blockIdx.x; w < nitems && ok; w += gridDim.x, ++acc) {
                const int a = (int)(acc & 1);
                if (!mbar_wait(&accempty[a], (uint32_t)(((acc >> 1) & 1) ^ 1), abort, flags)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d_tmem = tbase + C::kAcc0 + a * C::kAccCols;
                for (int64_t kc = 0; kc < nk; ++kc, ++it, ++ab) {
                    const int s = (int)(it % S);
                    const int b = (int)(ab % NA);
                    if (!mbar_wait(&full[s], (uint32_t)((it / S) & 1), abort, flags) ||
                        !mbar_wait(&afull[b], (uint32_t)((ab / NA) & 1), abort, flags)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t bs = smem_u32(smem + s * C::kStage + kXBytes);
                    const uint32_t a_hi = tbase + C::kABuf + 64 * b;
#pragma unroll
                    for (int k8 = 0; k8 < kChunk / 8; ++k8) {
                        const uint64_t bdesc = desc_sw128(bs + 32 * k8);
                        mma_tf32_ts(d_tmem, a_hi + 8 * k8, bdesc, idesc_tf32(2 * NPAD), (kc | k8) ? 1u : 0u);
                        mma_tf32_ts(d_tmem + NPAD, a_hi + 32 + 8 * k8, bdesc, idesc_tf32(NPAD), 1u);
                    }
                    tc_commit(&aempty[b]);
                    tc_commit(&xfree[s]);
                }
                if (!ok) break;
                tc_commit(&accfull[a]);
            }
            tc_commit(done);
            const uint64_t t0 = gtimer();
            while (!mbar_try_wait(done, 0) && gtimer() - t0 < kTimeoutNs) {
            }
        }
    } else if (warp >= W::kFirstConv && warp < W::kFirstEpi) {
        // ------------------------------------------------ converters: X chunk -> TF32 hi / lo in TMEM
        // two warps per TMEM lane quarter, half hs converting K columns [16 hs, 16 hs + 16)
        const int q = warp & 3, hs = ((warp - W::kFirstConv) >> 2) & 1;
        const int rho = 32 * q + lane;  // tile row == TMEM lane
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        int64_t it = 0, ab = 0;
        bool ok = true;
        for (int64_t w = blockIdx.x; w < nitems && ok; w += gridDim.x) {
            for (int64_t kc = 0; kc < nk; ++kc, ++it, ++ab) {
                const int s = (int)(it % S);
                const int b = (int)(ab % NA);
                bool got = mbar_wait(&full[s], (uint32_t)((it / S) & 1), abort, flags) &&
                           mbar_wait(&aempty[b], (uint32_t)(((ab / NA) & 1) ^ 1), abort, flags);
                if (!__all_sync(0xffffffffu, got)) {  // warp-uniform: tcgen05.st below is .aligned
                    ok = false;
                    break;
                }
                const uint8_t* xs = smem + s * C::kStage;
                float v[16];
                // rows i of 128 floats (512 B, no swizzle): lanes read consecutive words
                const float* xf = reinterpret_cast<const float*>(xs);
#pragma unroll
                for (int ii = 0; ii < 16; ++ii) v[ii] = xf[rho + (16 * hs + ii) * kRows];
                uint32_t hi[16], lo[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) split_tf32(v[i], hi[i], lo[i]);
                const uint32_t ta = tbase + lane_base + C::kABuf + 64 * b + 16 * hs;
                __syncwarp();
                tmem_st16(ta, hi);
                tmem_st16(ta + 32, lo);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();  // the warp's TMEM stores and SMEM reads are ordered before lane 0's arrivals
                if (lane == 0) {
                    mbar_arrive(&afull[b]);
                    mbar_arrive(&xfree[s]);
                }
            }
        }
    } else if (warp >= W::kFirstEpi) {
        // ------------------------------------------------ epilogue
        // warp e drains TMEM lane quarter warp % 4 (the quarter a warp may access) and the
        // 16-column slices cg, cg + kColGroups, ... of the accumulator
        const int q = warp & 3;
        const int cg = (warp - W::kFirstEpi) >> 2;
        const int rho = 32 * q + lane;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        // running sums as double-float pairs (hi + lo, Knuth two-sum): FP32 instructions only, the FP64
        // pipe (1/64 of FP32 here) stays out of the per-item work
        float srh = 0.f, srl = 0.f, sxh = 0.f, sxl = 0.f;
        int64_t acc = 0;
        for (int64_t w = blockIdx.x; w < nitems; w += gridDim.x, ++acc) {
            const int64_t t = w / args.nblk, nb = w % args.nblk;
            const int a = (int)(acc & 1);
            const int xb = (int)(acc % XB);
            bool got = mbar_wait(&accfull[a], (uint32_t)((acc >> 1) & 1), abort, flags);
            got = got && mbar_wait(&xrfull[xb], (uint32_t)((acc / XB) & 1), abort, flags);
            if (!__all_sync(0xffffffffu, got)) break;  // warp-uniform: tcgen05.ld below is .aligned
            tc_fence_after();
            const int64_t l = (t % args.tiles_per_r) * kRows + rho;
            const bool valid = l < args.L;
            int64_t base = l + args.L * args.m * (t / args.tiles_per_r);
            const int64_t stride = args.L;
            const int64_t col0 = nb * NPAD;
            base += col0 * stride;
            const int64_t ncol = args.m - col0;  // valid columns in this block (may exceed NPAD)
            const uint32_t ta = tbase + lane_base + C::kAcc0 + a * C::kAccCols;
            // [column][row] of the residual X tile
            const XR* xt = reinterpret_cast<const XR*>(reinterpret_cast<const uint8_t*>(xr_buf) + xb * C::kXrBytes);
#pragma unroll
            for (int c0 = 16 * cg; c0 < NPAD; c0 += 16 * W::kColGroups) {
                float h[16], g[16];
                __syncwarp();
                tmem_ld16(ta + c0, h);
                tmem_ld16(ta + NPAD + c0, g);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (valid) {
                    float fr = 0.f, fx = 0.f;
                    const XR* xcol = xt + c0 * kRows + rho;
                    XR* op = EPI == 2 ? static_cast<XR*>(args.out) + base + c0 * stride : nullptr;
                    auto one = [&](int i) {
                        float xv = xr_to_f32(xcol[i * kRows]);
                        if constexpr (std::is_same<XR, __nv_fp8_e4m3>::value) xv *= args.xr_scale;  // 1 / scale
                        const float dv = xv - (h[i] + g[i]);
                        fr = fmaf(dv, dv, fr);
                        fx = fmaf(xv, xv, fx);
                        if constexpr (EPI == 2) xr_store(op + i * stride, args.alpha * dv);
                    };
                    if (c0 + 16 <= ncol) {  // a full slice: no per-column test
#pragma unroll
                        for (int i = 0; i < 16; ++i) one(i);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (c0 + i < ncol) one(i);
                    }
                    ef_add(srh, srl, fr);
                    ef_add(sxh, sxl, fx);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&accempty[a]);
                mbar_arrive(&xrempty[xb]);
            }
        }
        // reduce over the epilogue threads: warp shuffles, then named barrier 1, then one
        // thread sums the warps in a fixed order
        double sr = (double)srh + (double)srl, sx = (double)sxh + (double)sxl;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sr += __shfl_xor_sync(0xffffffffu, sr, o);
            sx += __shfl_xor_sync(0xffffffffu, sx, o);
        }
        const int e = warp - W::kFirstEpi;
        if (lane == 0) {
            red[2 * e] = sr;
            red[2 * e + 1] = sx;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * W::kEpi) : "memory");
        if (e == 0 && lane == 0) {
            double a0 = 0.0, a1 = 0.0;
            for (int i = 0; i < W::kEpi; ++i) {
                a0 += red[2 * i];
                a1 += red[2 * i + 1];
            }
            args.partials[2 * blockIdx.x] = a0;
            args.partials[2 * blockIdx.x + 1] = a1;
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tbase) : "memory");
    }
}

template <int NPAD, int EPI, typename XR>
static void launch_one(const Ctx& c, const CUtensorMap& tx, const CUtensorMap& th, const CUtensorMap& tl,
                       const CUtensorMap& txr, const ResidArgs& a) {
    using Cf = Cfg<NPAD, XR>;
    auto kern = ttm_residual_kernel<NPAD, EPI, XR>;
    static bool attr_set = false;
    if (!attr_set) {
        TK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cf::kSmem));
        attr_set = true;
    }
    const int grid = (int)std::min<int64_t>(a.ntiles * a.nblk, grid_sms(c));
    kern<<<grid, Warps::kThreads, Cf::kSmem, c.stream>>>(tx, th, tl, txr, a);
}

void ttm_residual_run(const Ctx& c, int64_t npad, tk_dtype xrdt, bool dx, const CUtensorMap& tx, const CUtensorMap& th,
                      const CUtensorMap& tl, const CUtensorMap& txr, const ResidArgs& a) {
#define TK_TC_CASE(NP)                                                                     \
    case NP:                                                                               \
        if (xrdt == TK_FP8_E4M3) launch_one<NP, 1, __nv_fp8_e4m3>(c, tx, th, tl, txr, a);    \
        else if (xrdt == TK_BF16 && !dx) launch_one<NP, 1, __nv_bfloat16>(c, tx, th, tl, txr, a); \
        else if (xrdt == TK_BF16) launch_one<NP, 2, __nv_bfloat16>(c, tx, th, tl, txr, a);  \
        else if (!dx) launch_one<NP, 1, float>(c, tx, th, tl, txr, a);                       \
        else launch_one<NP, 2, float>(c, tx, th, tl, txr, a);                                \
        break;
    switch (npad) {
        TK_TC_CASE(16)
        TK_TC_CASE(32)
        TK_TC_CASE(48)
        TK_TC_CASE(64)
        default: fail(TK_ERR_SHAPE, "ttm_residual: unsupported width");
    }
#undef TK_TC_CASE
}

}  // namespace tc
}  // namespace tk
