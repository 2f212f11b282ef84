// The tcgen05 kernel of a plain mode-j contraction (TTM) of BF16 or FP8 (E4M3) data whose layout the kernels
// of tk_tc_bf16.cu and tk_tc_fp8.cu do not take: FP8 along any mode but the contiguous one, and either type
// with strides that are no multiple of 16 bytes.
//
//   out[l + L*(a + m*r)] = sum_i M(i, a) X[l + L*(i + n_j*r)]     (X viewed as L x n_j x R)
//
// BF16 and E4M3 values are TF32 values, so X needs no split: x*M = x*M_hi + x*M_lo with the TF32 parts of the
// factor that the FP32 kernel uses (22 bits of it), one MMA per 8-deep K step (N = 2*NPAD), FP32 accumulation.
//
// Kernel structure (persistent, one CTA per SM), as tk_ttm_tf32.cuh's with 64-deep K chunks:
//   warp 0      TMA producer (one thread): the factor's chunk, and with 16-byte strides X's (args.tma).
//   warp 1      allocates TMEM; one thread issues tcgen05.mma.
//   warps 2-3   loaders (!args.tma): X by 16-byte cp.async.  A chunk is a set of byte runs (a K row of the tile,
//               or a row's K range for L == 1) that start anywhere: each is fetched as the 16-byte pieces that
//               cover it, into a slot of its own, and the converters read at the run's offset in its slot.
//               That offset is the same for every chunk, as 64 steps of any stride are a multiple of 16 bytes.
//   converters  (two groups of 8 warps, alternate chunks) widen the chunk to FP32 and write it to TMEM, A's place.
//   epilogue    (8 warps, up to 16 columns 4): each chunk's accumulator is added in FP32 registers, rounding to
//               nearest (the tensor core's own additions round toward zero), rows written to global memory.
// 64 steps a chunk rather than 32 because a chunk of FP8 is little to load: 176 cycles of the SM's share of HBM
// at 32, less than a chunk takes.  Instruction issue still bounds it at 64 (ncu: 68% of the slots; a chunk takes
// 900 to 1400 cycles whether X is loaded or not, and its share of HBM is 350 for FP8, 700 for BF16).  SIMT and this
// kernel: FP8 768^3 along the last mode, 9 columns 1541 -> 176 us (2.7 TB/s); 689 x 690 x 700, 10 columns, along the
// last mode BF16 1064 -> 219, FP8 1147 -> 186; along the first BF16 3435 -> 178, FP8 3425 -> 168.  (Of these, the
// search for infinite and NaN results takes up to 14 us.)
//
// Every mbarrier wait is bounded by a wall-clock limit; on expiry the CTA raises FLAG_TIMEOUT, stops
// issuing work, drains what it issued and frees its TMEM.
#pragma once
#include <cuda_fp8.h>

#include "tk_ttm_tf32.cuh"

namespace tk {
namespace tc {

constexpr int kLowpChunk = 64;   // K elements per pipeline stage
constexpr int kLowpMaxStages = 12;

struct LowpArgs {
    int64_t L, nj, R, m;
    // work item = (row tile, block of NPAD output columns, part of the K chunks)
    uint32_t ntiles, tiles_per_r, nk, nblk, nitems;
    uint32_t pack;     // 32 <= L < 64: a tile holds `pack` consecutive r of L rows each; 1 otherwise
    uint32_t ksplit;   // parts of a tile's K chunks, each with its own partial product; 1 otherwise
    uint32_t stages;   // ring length (even: a stage always belongs to one converter group)
    uint32_t xstage;   // bytes of X's part of a stage (a multiple of 1 KB)
    uint32_t slot;     // bytes from one run of the chunk to the next (a multiple of 16)
    uint32_t tma;      // X by TMA (16-byte strides), the runs unshifted
    uint32_t xbytes;   // TMA bytes of X a chunk (0: loaders)
    float x_inv;       // factor of the result: 1 / scale of X
    const uint8_t* X;
    int64_t out_numel;
    float* out;        // the product, or the first of the ksplit partial ones
    unsigned* flags;
    const FactorInfo* info;
};
static_assert(sizeof(LowpArgs) <= 128, "see TtmResArgs");
static_assert(sizeof(LowpArgs) <= 128, "see TtmResArgs");

template <int NPAD>
struct LowpCfg {
    static constexpr int kBBytes = NPAD * 128;             // 32 K of M_hi or of M_lo
    static constexpr int kBStage = 4 * kBBytes;            // [K half][hi, lo]
    static constexpr int kNA = NPAD <= 32 ? 4 : 2;         // A buffers of 64 columns
    static constexpr int kABuf = 512 - 64 * kNA;
    static constexpr int kFit = kABuf / (2 * NPAD);
    static constexpr int kAcc = kFit > 8 ? 8 : kFit;       // accumulators of 2*NPAD columns
    static constexpr int kBudget = 222 * 1024;
    static constexpr int kLoad = 2, kFirstLoad = 2, kFirstConv = 4, kFirstEpi = 20;
    static constexpr int kEpi = NPAD <= 16 ? 4 : 8;        // at most one per 16 columns and lane quarter (idle ones
                                                           // poll: FP8 768^3, 9 columns 209 -> 172 us)
    static constexpr int kThreads = 32 * (kFirstEpi + kEpi);
    static_assert(kAcc >= 2, "TMEM budget");
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid) : "memory");
}

__device__ __forceinline__ uint32_t lds8(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t a) {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}

// Two E4M3 values (the low 16 bits) as FP32 bit patterns.
__device__ __forceinline__ void fp8_pair(uint32_t two, uint32_t& a, uint32_t& b) {
    const __half2_raw h = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)two, __NV_E4M3);
    const float2 f = __half22float2(__half2(h));
    a = __float_as_uint(f.x);
    b = __float_as_uint(f.y);
}

// The elements at shared addresses p0 and p1 as FP32 bit patterns.
template <int ES>
__device__ __forceinline__ void widen(uint32_t p0, uint32_t p1, uint32_t& a, uint32_t& b) {
    if (ES == 1) {
        fp8_pair(lds8(p0) | lds8(p1) << 8, a, b);
    } else {
        a = lds16(p0) << 16;
        b = lds16(p1) << 16;
    }
}

// A row's elements of 32 consecutive runs, SLOT bytes apart, the first `shift` mod 16 into its slot and each
// next one `step` mod 16 further.
template <int ES, int SLOT>
__device__ __forceinline__ void convert_runs(uint32_t xs, uint32_t shift, uint32_t step, uint32_t (&v)[2][16]) {
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        const uint32_t a0 = xs + ((shift + i * step) & 15), a1 = xs + ((shift + (i + 1) * step) & 15);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            widen<ES>(a0 + (16 * h + i) * SLOT, a1 + (16 * h + i + 1) * SLOT, v[h][i], v[h][i + 1]);
    }
}

template <int NPAD, bool KMAJOR, int ES>
__global__ void __launch_bounds__(LowpCfg<NPAD>::kThreads, 1)
    ttm_lowp_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmB, LowpArgs args) {
    kernel_begin();
    using C = LowpCfg<NPAD>;
    constexpr uint32_t NA = C::kNA;
    constexpr int K = kLowpChunk;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t S = args.stages, xstage = args.xstage, stage = xstage + C::kBStage;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * stage);
    uint64_t* full = bars;                          // [S] X and factor chunk landed
    uint64_t* xfree = full + kLowpMaxStages;        // [S] stage consumed (8 converter warps + 1 MMA commit)
    uint64_t* afull = xfree + kLowpMaxStages;       // [NA] A buffer written (8 converter warps)
    uint64_t* aempty = afull + NA;                  // [NA] A buffer consumed (MMA commit)
    uint64_t* accfull = aempty + NA;                // [kAcc] accumulator complete (MMA commit)
    uint64_t* accempty = accfull + C::kAcc;         // [kAcc] accumulator drained (the epilogue warps)
    uint64_t* done = accempty + C::kAcc;            // [1] every issued MMA complete
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    __shared__ int again;  // infinite or NaN results (exact_items); static: its address takes no register

    const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < S; ++s) {
            mbar_init(&full[s], args.tma ? 1 : 1 + 32 * C::kLoad);
            mbar_init(&xfree[s], 9);
        }
        for (uint32_t b = 0; b < NA; ++b) {
            mbar_init(&afull[b], 8);
            mbar_init(&aempty[b], 1);
        }
        for (int b = 0; b < C::kAcc; ++b) {
            mbar_init(&accfull[b], 1);
            mbar_init(&accempty[b], C::kEpi);
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
    const uint32_t nk = args.nk, ksplit = args.ksplit;
    // the K chunks [chunk0, chunk1) of item w, its row tile and column block
    auto chunk0 = [&](uint32_t w) { return ksplit == 1 ? 0u : (uint32_t)((uint64_t)nk * (w % ksplit) / ksplit); };
    auto chunk1 = [&](uint32_t w) { return ksplit == 1 ? nk : (uint32_t)((uint64_t)nk * (w % ksplit + 1) / ksplit); };
    auto tile_of = [&](uint32_t w) { return (ksplit == 1 ? w : w / ksplit) / args.nblk; };
    // strided: the tile's first slab r and first row l
    auto slab_of = [&](uint32_t t, uint32_t& r, uint32_t& l0) {
        const uint32_t q = args.tiles_per_r == 1 ? t : t / args.tiles_per_r;
        r = q * args.pack;
        l0 = (t - q * args.tiles_per_r) * kRows;
    };

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (elect_one()) {
            uint32_t s = 0, ph = 1, issued = 0;
            bool ok = true;
            for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
                const uint32_t t = tile_of(w), nb = args.nblk == 1 ? 0 : (ksplit == 1 ? w : w / ksplit) % args.nblk;
                const uint32_t kc1 = chunk1(w);
                uint32_t rr = 0, l0 = 0;
                if (!KMAJOR) slab_of(t, rr, l0);
                for (uint32_t kc = chunk0(w); kc < kc1; ++kc) {
                    if (!mbar_wait(&xfree[s], ph, abort, flags)) {
                        ok = false;
                        break;
                    }
                    uint8_t* xs = smem + s * stage;
                    uint8_t* bs = xs + xstage;
                    mbar_expect_tx(&full[s], args.xbytes + C::kBStage);
                    if (!KMAJOR && args.tma)
                        tma_load_3d(xs, &tmX, (int)l0, (int)(kc * K), (int)rr, &full[s]);
#pragma unroll
                    for (int h = 0; h < 2; ++h)  // 32 K of M_hi, then of M_lo
                        tma_load_3d(bs + h * 2 * C::kBBytes, &tmB, (int)(kc * K) + 32 * h, (int)(nb * NPAD), 0,
                                    &full[s]);
                    ++issued;
                    if (++s == S) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            // drain: every issued load has landed before the CTA can exit
            const uint32_t n_out = issued < S ? issued : S;
            for (uint32_t q = issued - n_out; q < issued; ++q) {
                const uint64_t t0 = gtimer();
                while (!mbar_try_wait(&full[q % S], (q / S) & 1) && gtimer() - t0 < kTimeoutNs) {
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (elect_one()) {
            uint32_t s = 0, ph = 0, b = 0, bph = 0, a = 0, aph = 1;
            bool ok = true;
            for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
                const uint32_t nc = chunk1(w) - chunk0(w);
                for (uint32_t kc = 0; kc < nc; ++kc) {
                    if (!mbar_wait(&accempty[a], aph, abort, flags) || !mbar_wait(&full[s], ph, abort, flags) ||
                        !mbar_wait(&afull[b], bph, abort, flags)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t bdesc = desc_sw128(smem_u32(smem + s * stage + xstage));
                    const uint32_t a_x = tbase + C::kABuf + 64 * b, d = tbase + a * (2 * NPAD);
#pragma unroll
                    for (int k8 = 0; k8 < K / 8; ++k8)  // 8 K = 32 B along the swizzled row
                        mma_tf32_ts(d, a_x + 8 * k8, bdesc + (k8 >> 2) * (2 * C::kBBytes / 16) + 2 * (k8 & 3),
                                    idesc_tf32(2 * NPAD), k8 ? 1u : 0u);
                    tc_commit(&aempty[b]);
                    tc_commit(&xfree[s]);
                    tc_commit(&accfull[a]);
                    if (++s == S) {
                        s = 0;
                        ph ^= 1;
                    }
                    if (++b == NA) {
                        b = 0;
                        bph ^= 1;
                    }
                    if (++a == C::kAcc) {
                        a = 0;
                        aph ^= 1;
                    }
                }
            }
            tc_commit(done);
            const uint64_t t0 = gtimer();
            while (!mbar_try_wait(done, 0) && gtimer() - t0 < kTimeoutNs) {
            }
        }
        __syncwarp();
    } else if (warp < C::kFirstConv) {
        // ------------------------------------------------ loaders
        if (!args.tma) {
            const uint32_t tid = threadIdx.x - 32 * C::kFirstLoad;
            constexpr uint32_t T = 32 * C::kLoad;
            const uint32_t npc = args.slot / 16;  // 16-byte pieces a run
            // lane -> (run, piece): groups of npc lanes take a run each, every G-th; a lane keeps its piece, so that
            // a whole chunk costs it an address step and a cp.async a run (with an index computed for each
            // piece the loaders bound the pass: 689 x 690 x 700 BF16, strided 498 us, contiguous 377)
            const uint32_t nrun = KMAJOR ? kRows : K, G = T / npc, g = tid / npc, pc = tid % npc;
            const uint64_t X = reinterpret_cast<uint64_t>(args.X);
            const uint64_t end = X + (uint64_t)ES * args.L * args.nj * args.R;
            const uint64_t run = (uint64_t)ES * (KMAJOR ? args.nj : args.L);  // from one run to the next
            const uint64_t slab = (uint64_t)ES * args.L * args.nj;
            uint32_t s = 0, ph = 1;
            bool ok = true;
            for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
                const uint32_t t = tile_of(w), kc1 = chunk1(w);
                uint32_t rr = 0, l0 = 0;
                if (!KMAJOR) slab_of(t, rr, l0);
                const uint64_t base = KMAJOR ? X + run * t * kRows : X + slab * rr + (uint64_t)ES * l0;
                for (uint32_t kc = chunk0(w); kc < kc1; ++kc) {
                    if (!__all_sync(0xffffffffu, mbar_wait(&xfree[s], ph, abort, flags))) {
                        ok = false;
                        break;
                    }
                    const uint32_t xs = smem_u32(smem + s * stage);
                    const uint64_t kb = base + (uint64_t)kc * K * (KMAJOR ? (uint64_t)ES : run);
                    const uint64_t last = kb + (args.pack - 1) * slab + (nrun - 1) * run;  // the chunk's last run
                    const bool whole = last + args.slot <= end &&
                                       (KMAJOR || (kc * K + K <= args.nj && rr + args.pack <= args.R));
                    if (g < G) {
                        for (uint32_t pk = 0; pk < args.pack; ++pk) {
                            uint64_t p = kb + pk * slab + g * run + 16 * pc;
                            uint32_t dst = xs + (pk * nrun + g) * args.slot + 16 * pc;
                            const uint64_t dp = G * run;
                            const uint32_t dd = G * args.slot;
                            if (whole) {
#pragma unroll 4
                                for (uint32_t i = g; i < nrun; i += G) {
                                    cp_async16(dst, reinterpret_cast<const void*>(p & ~uint64_t(15)), 16);
                                    p += dp;
                                    dst += dd;
                                }
                            } else {
                                for (uint32_t i = g; i < nrun; i += G) {
                                    const bool in = KMAJOR ? (int64_t)t * kRows + i < args.R
                                                           : kc * K + i < args.nj && rr + pk < args.R;
                                    const uint64_t a = p & ~uint64_t(15);
                                    const uint32_t n = in && a < end ? (end - a < 16 ? (uint32_t)(end - a) : 16u) : 0u;
                                    cp_async16(dst, reinterpret_cast<const void*>(n ? a : X), n);
                                    p += dp;
                                    dst += dd;
                                }
                            }
                        }
                    }
                    cp_async_arrive(&full[s]);
                    if (++s == S) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            asm volatile("cp.async.wait_all;" ::: "memory");  // nothing in flight when the CTA exits
        }
    } else if (warp < C::kFirstEpi) {
        // ------------------------------------------------ converters: X chunk -> TMEM
        // two groups of 8 warps; within a group two warps per TMEM lane quarter, half hs converting K
        // columns [32 hs, 32 hs + 32)
        const int cw = warp - C::kFirstConv;
        const int q = warp & 3, hs = (cw >> 2) & 1;
        const uint32_t grp = cw >> 3;
        const uint32_t rho = 32 * q + lane;  // tile row == TMEM lane
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        // strided: tile row rho is row l of slab p of the tile
        const uint32_t p = args.pack > 1 ? rho / (uint32_t)args.L : 0, l = rho - p * (uint32_t)args.L * (args.pack > 1);
        const bool real = p < args.pack;
        const uint32_t slot = args.slot;
        const uint32_t row = KMAJOR ? rho * slot : (real ? (p * K + 32 * hs) * slot + l * ES : 0);
        const uint32_t step = (uint32_t)args.L * ES;  // (mod 16: the shift from one run to the next)
        uint32_t s = 0, ph = 0, b = 0, bph = 1, it = 0;
        bool ok = true;
        for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
            const uint32_t c0 = chunk0(w), nc = chunk1(w) - c0, t = tile_of(w);
            uint32_t shift;  // byte offset (mod 16) of the row's, or of the half's first, run in its slot
            if (KMAJOR) {
                shift = (uint32_t)args.nj * ES * (t * kRows + rho) & 15;
            } else {
                uint32_t rr, l0;
                slab_of(t, rr, l0);
                shift = step * ((uint32_t)args.nj * (rr + p) + 32 * hs);
            }
            for (uint32_t kc = 0; kc < nc; ++kc, ++it) {
                if ((it & 1) == grp) {
                    if (!__all_sync(0xffffffffu, mbar_wait(&full[s], ph, abort, flags))) {
                        ok = false;
                        break;
                    }
                    const uint32_t xs = smem_u32(smem + s * stage) + row;
                    uint32_t v[2][16];
                    if (KMAJOR) {
                        // 32 elements from byte `shift` of the half's window: whole words, shifted down
                        constexpr int NW = 8 * ES;  // words wanted
                        uint32_t u[NW + 4];
#pragma unroll
                        for (int j = 0; j < NW / 4 + 1; ++j) {
                            const uint4 f = lds128(xs + 32 * ES * hs + 16 * j);
                            u[4 * j] = f.x;
                            u[4 * j + 1] = f.y;
                            u[4 * j + 2] = f.z;
                            u[4 * j + 3] = f.w;
                        }
#pragma unroll
                        for (int j = 0; j < NW + 2; ++j) u[j] = shift & 8 ? u[j + 2] : u[j];
#pragma unroll
                        for (int j = 0; j < NW + 1; ++j) u[j] = shift & 4 ? u[j + 1] : u[j];
#pragma unroll
                        for (int j = 0; j < NW; ++j) u[j] = __funnelshift_r(u[j], u[j + 1], (shift & 3) * 8);
#pragma unroll
                        for (int i = 0; i < 32; i += 2) {
                            uint32_t &x0 = v[i >> 4][i & 15], &x1 = v[i >> 4][(i & 15) + 1];
                            if (ES == 1) {
                                fp8_pair(u[i / 4] >> (8 * (i & 2)), x0, x1);
                            } else {
                                x0 = u[i / 2] << 16;
                                x1 = u[i / 2] & 0xFFFF0000u;
                            }
                        }
                        const int64_t left = args.nj - (int64_t)(c0 + kc) * K - 32 * hs;
                        if (left < 32) {  // past the row's end: the next row's elements
#pragma unroll
                            for (int i = 0; i < 32; ++i) v[i >> 4][i & 15] = i < left ? v[i >> 4][i & 15] : 0u;
                        }
                    } else if (args.pack == 1) {
                        // (constant slots; the shifts repeat every 16 runs)
                        if (args.tma) convert_runs<ES, kRows * ES>(xs, 0, 0, v);
                        else convert_runs<ES, kRows * ES + 16>(xs, shift, step, v);
                    } else if (real) {
#pragma unroll
                        for (int i = 0; i < 32; i += 2) {
                            uint32_t sh[2];
#pragma unroll
                            for (int e = 0; e < 2; ++e) sh[e] = args.tma ? 0 : (shift + (i + e) * step) & 15;
                            widen<ES>(xs + i * slot + sh[0], xs + (i + 1) * slot + sh[1], v[i >> 4][i & 15],
                                      v[i >> 4][(i & 15) + 1]);
                        }
                    }
                    if (!KMAJOR && !real) {  // packed tiles: the rows past L pack
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i >> 4][i & 15] = 0u;
                    }
                    if (!__all_sync(0xffffffffu, mbar_wait(&aempty[b], bph, abort, flags))) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t ta = tbase + lane_base + C::kABuf + 64 * b + 32 * hs;
                    tmem_st16(ta, v[0]);
                    tmem_st16(ta + 16, v[1]);
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    tc_fence_before();
                    __syncwarp();  // the warp's TMEM stores and SMEM reads are ordered before lane 0's arrivals
                    if (lane == 0) {
                        mbar_arrive(&afull[b]);
                        mbar_arrive(&xfree[s]);
                    }
                }
                if (++s == S) {
                    s = 0;
                    ph ^= 1;
                }
                if (++b == NA) {
                    b = 0;
                    bph ^= 1;
                }
            }
        }
    } else {
        // ------------------------------------------------ epilogue
        // warp e drains TMEM lane quarter warp % 4 (the quarter a warp may access), 16-column slices half, half + 2
        const int q = warp & 3, half = (warp - C::kFirstEpi) >> 2;
        const uint32_t rho = 32 * q + lane;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        const int64_t m = args.m;
        uint32_t a = 0, aph = 0;
        for (uint32_t w = blockIdx.x; w < args.nitems; w += gridDim.x) {
            const uint32_t w2 = ksplit == 1 ? w : w / ksplit, sk = w - w2 * ksplit;
            const uint32_t t = tile_of(w), nb = args.nblk == 1 ? 0 : w2 % args.nblk;
            const uint32_t nc = chunk1(w) - chunk0(w);
            float* const outp = args.out + sk * args.out_numel;
            int64_t base, stride;
            bool valid;
            if (KMAJOR) {
                const int64_t r = (int64_t)t * kRows + rho;
                valid = r < args.R;
                base = r * m;
                stride = 1;
            } else {
                uint32_t rr, l0, p = 0, l = rho;
                slab_of(t, rr, l0);
                if (args.pack > 1) {
                    p = rho / (uint32_t)args.L;
                    l = rho - p * (uint32_t)args.L;
                }
                valid = p < args.pack && rr + p < args.R && l0 + l < args.L;
                base = l0 + l + args.L * m * (int64_t)(rr + p);
                stride = args.L;
            }
            const int col0 = (int)nb * NPAD;
            base += col0 * stride;
            const int ncol = (int)(m - col0);  // valid columns in this block (may exceed NPAD)
            constexpr int kSl = (NPAD / 16 + 1) / 2;
            float v[kSl][16];
            bool ok = true;
            for (uint32_t f = 0; f < nc; ++f) {
                if (!__all_sync(0xffffffffu, mbar_wait(&accfull[a], aph, abort, flags))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t ta = tbase + lane_base + a * (2 * NPAD) + 16 * half;
#pragma unroll
                for (int j = 0; j < kSl; ++j) {
                    if (16 * half + 32 * j >= NPAD) break;  // warp-uniform
                    float h[16], g[16];
                    __syncwarp();
                    tmem_ld16(ta + 32 * j + NPAD, g);
                    tmem_ld16(ta + 32 * j, h);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[j][i] = f ? v[j][i] + (h[i] + g[i]) : h[i] + g[i];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&accempty[a]);
                if (++a == C::kAcc) {
                    a = 0;
                    aph ^= 1;
                }
            }
            if (!ok) break;
            if (valid) {
#pragma unroll
                for (int j = 0; j < kSl; ++j) {
                    const int c0 = 16 * half + 32 * j;
                    if (c0 >= NPAD) break;
                    if (any_nonfinite(v[j])) again = 1;
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[j][i] *= args.x_inv;
                    if (KMAJOR && (m & 3) == 0) {  // 16-byte stores along the row
#pragma unroll
                        for (int i = 0; i < 16; i += 4)
                            if (c0 + i < ncol)
                                *reinterpret_cast<float4*>(outp + base + c0 + i) =
                                    make_float4(v[j][i], v[j][i + 1], v[j][i + 2], v[j][i + 3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (c0 + i < ncol) outp[base + (c0 + i) * stride] = v[j][i];
                    }
                }
            }
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tbase) : "memory");
    }
    if (again && !*abort)
        exact_items<typename std::conditional<ES == 1, __nv_fp8_e4m3, __nv_bfloat16>::type, KMAJOR, false>(
            args, NPAD, K, args.x_inv);
}

template <int NPAD, bool KMAJOR, int ES>
static void ttm_lowp_launch(const Ctx& c, const CUtensorMap& tx, const CUtensorMap& tb, LowpArgs a) {
    using Cf = LowpCfg<NPAD>;
    const uint32_t stage = a.xstage + Cf::kBStage;
    a.stages = std::min<uint32_t>(kLowpMaxStages, Cf::kBudget / stage) & ~1u;
    TK_REQUIRE(a.stages >= 2, TK_ERR_SHAPE, "ttm_lowp: stage too large");
    auto kern = ttm_lowp_kernel<NPAD, KMAJOR, ES>;
    constexpr int kMaxSmem = Cf::kBudget + 2048;
    static std::atomic<uint64_t> opted{0};
    smem_opt_in(opted, reinterpret_cast<const void*>(kern), kMaxSmem);
    const int grid = (int)std::min<int64_t>(a.nitems, grid_sms(c));
    run_kernel(c, kern, grid, Cf::kThreads, a.stages * stage + 2048, tx, tb, a);
}

// The kernel for npad output columns per block (a multiple of 16 up to 64) and elements of ES bytes.
template <int ES>
static void ttm_lowp_dispatch(const Ctx& c, int64_t npad, bool kmajor, const CUtensorMap& tx, const CUtensorMap& tb,
                              const LowpArgs& a) {
#define TK_LOWP_CASE(NP)                                               \
    case NP:                                                           \
        if (kmajor) ttm_lowp_launch<NP, true, ES>(c, tx, tb, a);       \
        else ttm_lowp_launch<NP, false, ES>(c, tx, tb, a);             \
        break;
    switch (npad) {
        TK_LOWP_CASE(16)
        TK_LOWP_CASE(32)
        TK_LOWP_CASE(48)
        TK_LOWP_CASE(64)
        default: fail(TK_ERR_SHAPE, "ttm_lowp: unsupported width");
    }
#undef TK_LOWP_CASE
}

void ttm_lowp_run_bf16(const Ctx& c, int64_t npad, bool kmajor, const CUtensorMap& tx, const CUtensorMap& tb,
                       const LowpArgs& a);
void ttm_lowp_run_fp8(const Ctx& c, int64_t npad, bool kmajor, const CUtensorMap& tx, const CUtensorMap& tb,
                      const LowpArgs& a);

}  // namespace tc
}  // namespace tk
