// The tcgen05 kernel of a plain mode-j contraction (TTM) of FP32 data:
//
//   out[l + L*(a + m*r)] = sum_i M(i, a) X[l + L*(i + n_j*r)]     (X viewed as L x n_j x R)
//
// FP32 accuracy from TF32 tensor cores by the split-product ("3xTF32") method:
// x = x_hi + x_lo and M = M_hi + M_lo with TF32 parts, and x*M ~ x_hi*M_hi +
// x_hi*M_lo + x_lo*M_hi with FP32 accumulation.
//
// Kernel structure (persistent, one CTA per SM):
//   warp 0      TMA producer (one thread): 32-deep K chunks of a 128-row tile of X (16 KB) plus the
//               matching 32 x NPAD chunks of M_hi and M_lo, into an SMEM ring.
//   warp 1      allocates TMEM; one thread issues tcgen05.mma.
//   loaders     (FLAT only, 8 warps) bring the X chunk with cp.async instead of TMA, see below.
//   converters  (two groups of 8 warps taking alternate chunks; FLAT: one) read their row's values of the chunk
//               from SMEM, split them into TF32 hi / lo and write them to TMEM with tcgen05.st.  The
//               MMA reads A from TMEM, so X is read from SMEM exactly once, and a contraction over a
//               non-contiguous mode needs no transpose: only the element each lane reads differs.
//   epilogue    (8 warps, two per TMEM lane quarter; up to 16 columns 4): tcgen05.ld, sums, rows written to global
//               memory.
// The issuing threads are chosen by elect.sync (tk_tc_common.cuh), so that neither the MMAs (288 of
// the 700 cycles that HBM gives a chunk at NPAD = 48) nor their issue bounds the pass.
//
// One MMA per 8-deep K step computes A_hi * [M_hi ; M_lo] (N = 2*NPAD, the two halves land in separate
// TMEM columns); a second adds A_lo * M_hi into the second half, with the other small term.  The
// tensor core's FP32 accumulation rounds each addition toward zero, a bias that grows with the number
// of additions into one A_hi * M_hi sum.  So an accumulator takes the products of `fill` chunks only (1 up
// to 8 columns, 4 up to 64, 16 above; half a chunk for FLAT, whose shapes the SIMT kernels took before, with every addition
// rounded to nearest), and the epilogue adds the fills of an item in FP32 registers, rounding to nearest,
// while the next ones are computed: TMEM holds a ring of as many accumulators as fit beside the A
// buffers.  Errors against FP64: 512^3, 42 columns 2.4e-6 with one accumulator an item, 7.2e-7 so (100 ->
// 104 us); 413 x 350 x 275, 36 columns 4.1e-7 with one chunk an accumulator, 3.6e-7 with half (SIMT 4.3e-7).
//
// RES: the product is not stored but compared with a tensor of its shape: fused residuals whose contraction is longer
// than tk_expand_tf32.cu holds (128).
//
// FLAT = false: TMA.  Needs 16-byte strides (L % 4 == 0, or n_j % 4 == 0 for L == 1).  A strided mode
// with fewer than 64 rows before it packs several slabs into each 128-row tile (pack).
// FLAT = true: any L and n_j.  The L*R rows are numbered without regard to slabs (so no row of a tile
// is padding, whatever L is), every loader lane keeps the addresses of its rows, and 4-byte cp.async
// (8-byte when L, or n_j for L == 1, is even) fill the same stages in the same layout, with zeros
// beyond n_j and the last row; each loader's cp.async arrive on the stage's barrier when they land.
//
// Every mbarrier wait is bounded by a wall-clock limit; on expiry the CTA raises FLAG_TIMEOUT, stops
// issuing work, drains what it issued and frees its TMEM.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "tk_tc_common.cuh"

namespace tk {
namespace tc {

constexpr int kRows = 128;    // tile rows (TMEM lanes)
constexpr int kChunk = 32;    // K elements per pipeline stage
constexpr int kXBytes = kRows * kChunk * 4;

// D[tmem] (+)= A[tmem] * B[smem desc], kind::tf32, M = 128.
__device__ __forceinline__ void mma_tf32_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Instruction descriptor: D F32, A/B TF32, both K-major, M = 128, N = n.
__host__ __device__ constexpr uint32_t idesc_tf32(int n) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}

// x = hi + lo: hi is x rounded to TF32 (ties away, as cvt.rna) by integer addition; lo = x - hi (exact), whose
// bits below TF32 the tensor core ignores: an odd last bit is dropped where cvt.rna rounds it away, an
// error of the same size.  NaN survives in lo.  The conversion unit, two cvt.rna per element, bounded the
// pass (512^3, 42 columns: 135 -> 115 us).
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
    hi = (__float_as_uint(x) + 0x1000u) & 0xFFFFE000u;
    lo = __float_as_uint(x - __uint_as_float(hi));
}

// The sums (sr, sx) of the lanes of N epilogue warps, in a fixed order, into the CTA's pair of partials.
template <int N>
__device__ __forceinline__ void residual_sums(int e, int lane, double sr, double sx, double* partials) {
    __shared__ double red[2 * N];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
    }
    if (lane == 0) {
        red[2 * e] = sr;
        red[2 * e + 1] = sx;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * N) : "memory");
    if (e == 0 && lane == 0) {
        double a0 = 0.0, a1 = 0.0;
        for (int i = 0; i < N; ++i) {
            a0 += red[2 * i];
            a1 += red[2 * i + 1];
        }
        partials[2 * blockIdx.x] = a0;
        partials[2 * blockIdx.x + 1] = a1;
    }
}

// What a kernel has to know of the factor besides its parts, written beside them by the kernel that splits it (in
// memory: the kernels' arguments have no room for it, see TtmResArgs): the factor as the caller gave it, M(i, a) =
// M[i + ldm a], or M[a + ldm i] with mtrans (dt: F32 or F64), and a flag of each block that split it, set when a part
// is infinite or NaN.
struct FactorInfo {
    const void* M;
    int64_t ldm;
    int dt, mtrans;
    uint32_t nbad;
    int bad[1];
};

__device__ __forceinline__ void xr_store(float* p, float v) { *p = v; }
__device__ __forceinline__ void xr_store(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ float x_to_f32(float v) { return v; }
__device__ __forceinline__ float x_to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float x_to_f32(__nv_fp8_e4m3 v) { return static_cast<float>(v); }

// Elements of the product that come out infinite or NaN are formed again by FP32 FMAs, from the factor as the caller
// gave it: for an infinity, or a value that rounds to one, the split gives a NaN (x_hi M_lo with M_lo = 0 or of the
// other sign).  The epilogue only notes that there are some; the CTA goes over its items once more at its end, when
// nothing is kept in registers (a call in the epilogue itself: 135 -> 150 us for the core of 512^3, from the spills).
//
// The sum over i0 <= i < i1 of M(i, a) x[i step] inv.
template <typename TX>
__device__ __forceinline__ float exact_dot(const TX* x, int64_t step, int64_t i0, int64_t i1, const FactorInfo& f, int64_t a,
                                           float inv) {
    float s = 0.f;
    const int64_t fa = f.mtrans ? a : f.ldm * a, fi = f.mtrans ? f.ldm : 1;
#pragma unroll 4
    for (int64_t i = i0; i < i1; ++i) {
        const int64_t o = fa + fi * i;
        const float mv = f.dt == TK_F64 ? (float)static_cast<const double*>(f.M)[o] : static_cast<const float*>(f.M)[o];
        s = fmaf(mv, x_to_f32(x[i * step]) * inv, s);
    }
    return s;
}

// Forms the infinite and NaN elements among the results of this CTA's items again (every thread, after a barrier).
template <typename TX, bool KMAJOR, bool FLAT, typename Args>
__device__ __forceinline__ void exact_items(const Args& g, int npad, int chunk, float inv) {
    for (uint32_t w = blockIdx.x; w < g.nitems; w += gridDim.x) {
        const uint32_t w2 = w / g.ksplit, sk = w - w2 * g.ksplit, t = w2 / g.nblk, nb = w2 - t * g.nblk;
        const int64_t i0 = (int64_t)((uint64_t)g.nk * sk / g.ksplit) * chunk;
        const int64_t ie = (int64_t)((uint64_t)g.nk * (sk + 1) / g.ksplit) * chunk, i1 = ie < g.nj ? ie : g.nj;
        float* const out = g.out + sk * g.out_numel;
        for (int e = threadIdx.x; e < 128 * npad; e += blockDim.x) {
            const int rho = e & 127;
            const int64_t c = (int64_t)nb * npad + (e >> 7);
            if (c >= g.m) break;
            int64_t l, r;  // the row's place in its slab, its slab
            if (KMAJOR) {
                l = 0;
                r = (int64_t)t * 128 + rho;
            } else if (FLAT) {
                r = ((int64_t)t * 128 + rho) / g.L;
                l = (int64_t)t * 128 + rho - r * g.L;
            } else if (g.pack > 1) {
                const int p = rho / (int)g.L;
                l = p < (int)g.pack ? rho - p * g.L : g.L;
                r = (int64_t)t * g.pack + p;
            } else {
                r = t / g.tiles_per_r;
                l = (int64_t)(t - r * g.tiles_per_r) * 128 + rho;
            }
            if (l >= g.L || r >= g.R) continue;
            float* const o = out + l + g.L * (c + g.m * r);
            if (fabsf(*o) <= 3.402823466e38f) continue;
            *o = exact_dot(reinterpret_cast<const TX*>(g.X) + l + g.L * g.nj * r, g.L, i0, i1, *g.info, c, inv);
        }
    }
}

// A CTA whose part of a fused residual met such elements compares all of it again: element (l, a) of the rows [l0, l1)
// and columns [a0, a1), with the sums in FP64.
template <typename XR>
__device__ __forceinline__ void exact_compare(const float* W, int64_t L, int64_t nj, const FactorInfo& f, int64_t l0,
                                              int64_t l1, int64_t a0, int64_t a1, const void* xref, float xr_scale,
                                              void* dx, float alpha, double& sr, double& sx) {
    const int64_t rows = l1 - l0;
    for (int64_t e = threadIdx.x; e < rows * (a1 - a0); e += blockDim.x) {
        const int64_t l = l0 + e % rows, a = a0 + e / rows;
        const float xv = x_to_f32(static_cast<const XR*>(xref)[l + L * a]) * xr_scale;
        const float dv = xv - exact_dot(W + l, L, 0, nj, f, a, 1.f);
        sr += (double)dv * dv;
        sx += (double)xv * xv;
        if constexpr (!std::is_same<XR, __nv_fp8_e4m3>::value)
            if (dx) xr_store(static_cast<XR*>(dx) + l + L * a, alpha * dv);
    }
}

// Whether one of the values is infinite or NaN.
__device__ __forceinline__ bool any_nonfinite(const float (&v)[16]) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) t = fmaf(v[i], 0.f, t);
    return t != t;
}

// The same over every thread of the CTA (after a barrier).
__device__ __forceinline__ void residual_sums_cta(double sr, double sx, double* partials) {
    __shared__ double red[2 * 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = sr;
        red[32 + (threadIdx.x >> 5)] = sx;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double t = 0.0;
        for (uint32_t i = 0; i < blockDim.x / 32; ++i) t += red[32 * threadIdx.x + i];
        partials[2 * blockIdx.x + threadIdx.x] = t;
    }
}

struct TtmArgs {
    int64_t L, nj, R, m;
    // work item = (row tile, block of NPAD output columns, part of the K chunks)
    uint32_t ntiles, tiles_per_r, nk, nblk, nitems;
    // strided mode with L < 64 (TMA): a tile holds `pack` consecutive r of L rows each (pack L <= 128
    // rows) instead of one r, so that short rows fill the 128-row tile; 1 otherwise
    uint32_t pack;
    uint32_t xbytes;  // TMA bytes of one X chunk (128 x 32 x 4, or L x 32 x pack x 4; 0: FLAT)
    // few row tiles: the K chunks of a tile are split over ksplit work items, each writing its
    // partial product to out + s out_numel (summed in order by a second kernel); 1 otherwise
    uint32_t ksplit;
    uint32_t fill;         // chunks per accumulator (TMA)
    uint32_t vec;          // FLAT: floats per cp.async (1 or 2)
    const float* X;        // FLAT
    int64_t out_numel;
    float* out;            // the product, or the first of the ksplit partial ones
    unsigned* flags;
    const FactorInfo* info;
};
static_assert(sizeof(TtmArgs) <= 128, "see TtmResArgs");

// RES: the tensor compared with the product (its layout, R == 1; elements of type xrdt, times xr_scale),
// dx = alpha * (xref - product) in its type (may be NULL), per-CTA sums {(xref - product)^2, xref^2}.  (Arguments of their
// own: kernels get slower where theirs pass 128 bytes beside the two maps, ttm_lowp_kernel 170 -> 199 us.)
struct TtmResArgs : TtmArgs {
    const void* xref;
    void* dx;
    int xrdt;
    float alpha, xr_scale;
    double* partials;
};

template <typename XR>
__device__ __forceinline__ void residual_load(const void* xref, int64_t o, int64_t L, int n, float (&x)[8]) {
    const XR* xp = static_cast<const XR*>(xref) + o;
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = i < n ? x_to_f32(xp[i * L]) : 0.f;
}
template <typename XR>
__device__ __forceinline__ void residual_store(void* dx, int64_t o, int64_t L, int n, const float (&x)[8]) {
    XR* xp = static_cast<XR*>(dx) + o;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (i < n) xr_store(xp + i * L, x[i]);
}

// RES: 8 columns p of a row, of which n are the product's, against xref from its element o.
__device__ __forceinline__ void residual_columns(const TtmResArgs& a, int64_t o, int n, const float* p, float& fr,
                                                 float& fx) {
    float x[8];
    if (a.xrdt == TK_F32) residual_load<float>(a.xref, o, a.L, n, x);
    else if (a.xrdt == TK_BF16) residual_load<__nv_bfloat16>(a.xref, o, a.L, n, x);
    else residual_load<__nv_fp8_e4m3>(a.xref, o, a.L, n, x);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        x[i] *= a.xr_scale;
        fx = fmaf(x[i], x[i], fx);
        x[i] = i < n ? x[i] - p[i] : 0.f;
        fr = fmaf(x[i], x[i], fr);
        x[i] *= a.alpha;
    }
    if (!a.dx) return;
    if (a.xrdt == TK_F32) residual_store<float>(a.dx, o, a.L, n, x);
    else residual_store<__nv_bfloat16>(a.dx, o, a.L, n, x);
}

// RES: the whole of a CTA's part again.
__device__ __forceinline__ void exact_residual(const TtmResArgs& args, int npad) {
    double sr = 0.0, sx = 0.0;
    for (uint32_t w = blockIdx.x; w < args.nitems; w += gridDim.x) {
        const uint32_t t = w / args.nblk, nb = w - t * args.nblk;
        const int64_t l0 = (int64_t)t * kRows, a0 = (int64_t)nb * npad;
        const int64_t l1 = l0 + kRows < args.L ? l0 + kRows : args.L, a1 = a0 + npad < args.m ? a0 + npad : args.m;
        if (args.xrdt == TK_F32)
            exact_compare<float>(args.X, args.L, args.nj, *args.info, l0, l1, a0, a1, args.xref, args.xr_scale, args.dx,
                                 args.alpha, sr, sx);
        else if (args.xrdt == TK_BF16)
            exact_compare<__nv_bfloat16>(args.X, args.L, args.nj, *args.info, l0, l1, a0, a1, args.xref, args.xr_scale,
                                         args.dx, args.alpha, sr, sx);
        else
            exact_compare<__nv_fp8_e4m3>(args.X, args.L, args.nj, *args.info, l0, l1, a0, a1, args.xref, args.xr_scale,
                                         args.dx, args.alpha, sr, sx);
    }
    residual_sums_cta(sr, sx, args.partials);
}

template <int NPAD, bool KMAJOR, bool FLAT>
struct TtmCfg {
    static constexpr int kBBytes = NPAD * 128;  // one of M_hi / M_lo: NPAD rows of 128 B
    static constexpr int kStage = kXBytes + 2 * kBBytes;
    // a tile of the result, staged (L == 1, more than 16 columns: below, a copy a tile costs more than the
    // scattered stores do, 413 x 350 x 275 with 6 columns 47 -> 52 us)
    static constexpr int kOut = KMAJOR && NPAD > 16 ? kRows * NPAD * 4 : 0;
    static constexpr int kBudget = kOut ? 222 * 1024 - kOut : 210 * 1024;
    // FLAT: a shorter ring, which leaves the SM's L1, where each cp.async in flight holds its lines, some
    // room (413 x 350 x 275 along its first mode, 5 columns: 58 us with 10 stages, 47 with 6)
    static constexpr int kStages = FLAT ? (NPAD <= 32 ? 6 : 4) : (kBudget / kStage > 12 ? 12 : kBudget / kStage);
    static constexpr int kNA = NPAD <= 32 ? 4 : 2;      // A buffers of 64 columns (hi 32 | lo 32)
    static constexpr int kABuf = 512 - 64 * kNA;
    static constexpr int kFit = kABuf / (2 * NPAD);     // accumulators of 2*NPAD columns
    static constexpr int kAcc = kFit > 8 ? 8 : kFit;
    static constexpr int kSmem = kStages * kStage + kOut + 1024 + 512;
    static constexpr int kLoad = FLAT ? 8 : 0;          // loader warps, from warp 2
    static constexpr int kFirstConv = FLAT ? 12 : 4;    // (a multiple of 4: warp % 4 is the TMEM lane quarter)
    static constexpr int kGroups = FLAT ? 1 : 2;        // converter groups of 8 warps
    static constexpr int kFirstEpi = kFirstConv + 8 * kGroups;
    static constexpr int kEpi = NPAD <= 16 ? 4 : 8;     // epilogue warps: at most one per 16 columns and lane
                                                        // quarter (idle ones poll: 160^4, 5 columns 534 -> 502 us)
    static constexpr int kThreads = 32 * (kFirstEpi + kEpi);
    static_assert(kAcc >= 2, "TMEM budget");
    static_assert(kStages >= 4, "SMEM budget");
    // The converter groups take alternate chunks, so with an odd ring a stage alternates between them,
    // and a group must not test a stage's barrier a whole ring early (the parity of the phase before
    // would read as complete): chunk c + S comes after its own chunk c + S - 2, whose A buffer waited for
    // the MMAs of chunk c + S - 2 - kNA, hence for chunk c's load.
    static_assert(kGroups == 1 || kStages % 2 == 0 || kStages >= kNA + 2, "converter groups could overrun the ring");
};

template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, uint32_t valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(BYTES), "r"(valid) : "memory");
}
// One arrival on bar (counted in its expected arrivals) once this thread's earlier cp.async have landed.
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

template <int NPAD, bool KMAJOR, bool FLAT, bool RES = false>
__global__ void __launch_bounds__(TtmCfg<NPAD, KMAJOR, FLAT>::kThreads, 1)
    ttm_tf32x3_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmB,
                      typename std::conditional<RES, TtmResArgs, TtmArgs>::type args) {
    kernel_begin();
    using C = TtmCfg<NPAD, KMAJOR, FLAT>;
    constexpr uint32_t S = C::kStages;
    constexpr uint32_t NA = C::kNA;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    float* stg = reinterpret_cast<float*>(smem + S * C::kStage);  // kOut: a tile of the result
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * C::kStage + C::kOut);
    uint64_t* full = bars;                   // [S] X and factor chunk landed
    uint64_t* xfree = bars + S;              // [S] stage consumed (8 converter warps + 1 MMA commit)
    uint64_t* afull = bars + 2 * S;          // [NA] A buffer written (8 converter warps)
    uint64_t* aempty = afull + NA;           // [NA] A buffer consumed (MMA commit)
    uint64_t* accfull = aempty + NA;         // [kAcc] accumulator complete (MMA commit)
    uint64_t* accempty = accfull + C::kAcc; // [kAcc] accumulator drained (the epilogue warps)
    uint64_t* done = accempty + C::kAcc;    // [1] every issued MMA complete
    uint64_t* stgfree = done + 1;           // [1] staged tile copied out (kOut)
    uint64_t* stgfull = stgfree + 1;        // [1] tile staged (the epilogue warps)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(stgfull + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    __shared__ int again;  // infinite or NaN results (exact_items); static: its address takes no register

    const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        again = 0;
        for (uint32_t s = 0; s < S; ++s) {
            mbar_init(&full[s], 1 + 32 * C::kLoad);
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
        mbar_init(stgfree, 1);
        mbar_init(stgfull, C::kEpi);
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
    const uint32_t nk = args.nk, ksplit = args.ksplit;
    // the K chunks [kc0, kc1) of item w
    auto chunk0 = [&](uint32_t w) { return ksplit == 1 ? 0u : (uint32_t)((uint64_t)nk * (w % ksplit) / ksplit); };
    auto chunk1 = [&](uint32_t w) { return ksplit == 1 ? nk : (uint32_t)((uint64_t)nk * (w % ksplit + 1) / ksplit); };

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (elect_one()) {
            uint32_t s = 0, ph = 1, issued = 0;
            bool ok = true;
            for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
                const uint32_t w2 = ksplit == 1 ? w : w / ksplit;
                const uint32_t t = args.nblk == 1 ? w2 : w2 / args.nblk, nb = args.nblk == 1 ? 0 : w2 % args.nblk;
                const uint32_t kc1 = chunk1(w);
                int rr = 0, l0 = 0;
                if (!FLAT && !KMAJOR) {
                    const uint32_t q = args.tiles_per_r == 1 ? t : t / args.tiles_per_r;
                    rr = (int)(q * args.pack);
                    l0 = (int)((t - q * args.tiles_per_r) * kRows);
                }
                for (uint32_t kc = chunk0(w); kc < kc1; ++kc) {
                    if (!mbar_wait(&xfree[s], ph, abort, flags)) {
                        ok = false;
                        break;
                    }
                    uint8_t* xs = smem + s * C::kStage;
                    uint8_t* bs = xs + kXBytes;
                    mbar_expect_tx(&full[s], args.xbytes + 2 * C::kBBytes);
                    if (!FLAT) {
                        if (KMAJOR)
                            tma_load_2d(xs, &tmX, (int)(kc * kChunk), (int)(t * kRows), &full[s]);
                        else  // one unswizzled 128 x 32 box: rows i of 128 floats (512 B)
                            tma_load_3d(xs, &tmX, l0, (int)(kc * kChunk), rr, &full[s]);
                    }
                    tma_load_3d(bs, &tmB, (int)(kc * kChunk), (int)(nb * NPAD), 0, &full[s]);  // M_hi, then M_lo
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
                uint32_t in = 0;  // chunks in the current accumulator
                for (uint32_t kc = 0; kc < nc; ++kc) {
                    if ((!FLAT && in == 0 && !mbar_wait(&accempty[a], aph, abort, flags)) ||
                        !mbar_wait(&full[s], ph, abort, flags) || !mbar_wait(&afull[b], bph, abort, flags)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t bdesc = desc_sw128(smem_u32(smem + s * C::kStage + kXBytes));
                    const uint32_t a_hi = tbase + C::kABuf + 64 * b;
                    if (FLAT) {
                        // half a chunk per accumulator
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            ok = ok && mbar_wait(&accempty[a], aph, abort, flags);
                            if (!ok) break;
                            tc_fence_after();
                            const uint32_t d = tbase + a * (2 * NPAD);
#pragma unroll
                            for (int k8 = 2 * h; k8 < 2 * h + 2; ++k8) {
                                mma_tf32_ts(d, a_hi + 8 * k8, bdesc + 2 * k8, idesc_tf32(2 * NPAD), k8 & 1 ? 1u : 0u);
                                mma_tf32_ts(d + NPAD, a_hi + 32 + 8 * k8, bdesc + 2 * k8, idesc_tf32(NPAD), 1u);
                            }
                            tc_commit(&accfull[a]);
                            if (++a == C::kAcc) {
                                a = 0;
                                aph ^= 1;
                            }
                        }
                        if (!ok) break;
                    } else {
                        const uint32_t d = tbase + a * (2 * NPAD);
                        const uint32_t again = in ? 1u : 0u;
#pragma unroll
                        for (int k8 = 0; k8 < kChunk / 8; ++k8) {  // 8 K = 32 B along the swizzled row
                            mma_tf32_ts(d, a_hi + 8 * k8, bdesc + 2 * k8, idesc_tf32(2 * NPAD), k8 ? 1u : again);
                            mma_tf32_ts(d + NPAD, a_hi + 32 + 8 * k8, bdesc + 2 * k8, idesc_tf32(NPAD), 1u);
                        }
                    }
                    tc_commit(&aempty[b]);
                    tc_commit(&xfree[s]);
                    if (++s == S) {
                        s = 0;
                        ph ^= 1;
                    }
                    if (++b == NA) {
                        b = 0;
                        bph ^= 1;
                    }
                    if (!FLAT && (++in == args.fill || kc + 1 == nc)) {
                        tc_commit(&accfull[a]);
                        in = 0;
                        if (++a == C::kAcc) {
                            a = 0;
                            aph ^= 1;
                        }
                    }
                }
            }
            tc_commit(done);
            const uint64_t t0 = gtimer();
            while (!mbar_try_wait(done, 0) && gtimer() - t0 < kTimeoutNs) {
            }
        }
        __syncwarp();
    } else if (FLAT && warp >= 2 && warp < 2 + C::kLoad) {
        // ------------------------------------------------ loaders: X chunks by cp.async
        // Few instructions per cp.async: every lane keeps the pointers of its rows and steps them by a constant
        // (a loader warp issues, not waits, for most of its time).
        constexpr int kPart = kChunk / (C::kLoad ? C::kLoad : 1);    // K rows per warp and chunk (strided)
        constexpr int kPartR = kRows / (C::kLoad ? C::kLoad : 1);    // tile rows per warp (L == 1)
        const int lw = warp - 2;
        const uint32_t rows = (uint32_t)(args.L * args.R), L = (uint32_t)args.L, nj = (uint32_t)args.nj;
        const bool two = args.vec == 2;
        uint32_t s = 0, ph = 1;
        bool ok = true;
        for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
            const uint32_t w2 = ksplit == 1 ? w : w / ksplit;
            const uint32_t t = args.nblk == 1 ? w2 : w2 / args.nblk;
            const uint32_t kc0 = chunk0(w), kc1 = chunk1(w);
            // strided: the lane's 4 rows lane + 32 q of the tile (8-byte: 2 row pairs 2 lane + 64 q), at
            // K row kc0 * 32 + lw * kPart; L == 1: K element(s) k of row lw * kPartR (8-byte: + its half)
            const float* src[4];
            uint32_t vb[4];
            if (!KMAJOR) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t g = t * kRows + (two ? 2 * lane + 64 * q : lane + 32 * q);
                    const uint32_t r = g / L;
                    const bool in = g < rows && (!two || q < 2);
                    vb[q] = in ? (two ? 8 : 4) : 0;
                    src[q] = in ? args.X + (int64_t)(g - r * L) + args.L * (args.nj * r + kc0 * kChunk + lw * kPart)
                                : args.X;
                }
            }
            for (uint32_t kc = kc0; kc < kc1; ++kc) {
                if (!__all_sync(0xffffffffu, mbar_wait(&xfree[s], ph, abort, flags))) {
                    ok = false;
                    break;
                }
                const uint32_t xs = smem_u32(smem + s * C::kStage);
                if (!KMAJOR) {
                    // rows i of 128 floats
                    const uint32_t i0 = kc * kChunk + lw * kPart;
                    const uint32_t dst = xs + (lw * kPart * kRows + (two ? 2 * lane : lane)) * 4;
#pragma unroll
                    for (int u = 0; u < kPart; ++u) {
                        const bool in = i0 + u < nj;
                        if (two) {
#pragma unroll
                            for (int q = 0; q < 2; ++q)
                                cp_async<8>(dst + (u * kRows + 64 * q) * 4,
                                            in && vb[q] ? src[q] + (int64_t)u * args.L : args.X, in ? vb[q] : 0);
                        } else {
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                cp_async<4>(dst + (u * kRows + 32 * q) * 4,
                                            in && vb[q] ? src[q] + (int64_t)u * args.L : args.X, in ? vb[q] : 0);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) src[q] += vb[q] ? args.L * kChunk : 0;
                } else {
                    // rows g of 128 B, the 16-byte chunk j of row rr stored at chunk j ^ (rr & 7)
                    const uint32_t k = two ? (lane & 15) * 2 : lane, sub = two ? lane >> 4 : 0;
                    const uint32_t i = kc * kChunk + k, g0 = t * kRows + lw * kPartR + sub;
                    const float* p = args.X + (int64_t)nj * g0 + i;
                    const uint32_t row0 = xs + (lw * kPartR + sub) * 128 + (k & 3) * 4;
                    const bool kin = i < nj;
                    if (two) {
#pragma unroll
                        for (int u = 0; u < kPartR / 2; ++u, p += 2 * args.nj) {
                            const bool in = kin && g0 + 2 * u < rows;
                            cp_async<8>(row0 + u * 256 + (((k >> 2) ^ ((2 * u + sub) & 7)) << 4), in ? p : args.X,
                                        in ? 8 : 0);
                        }
                    } else {
#pragma unroll
                        for (int u = 0; u < kPartR; ++u, p += args.nj) {
                            const bool in = kin && g0 + u < rows;
                            cp_async<4>(row0 + u * 128 + (((k >> 2) ^ (u & 7)) << 4), in ? p : args.X, in ? 4 : 0);
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
    } else if (warp >= C::kFirstConv && warp < C::kFirstEpi) {
        // ------------------------------------------------ converters: X chunk -> TF32 hi / lo in TMEM
        // two groups of 8 warps, group g taking the even / odd chunks; within a group two warps per
        // TMEM lane quarter, half hs converting K columns [16 hs, 16 hs + 16).
        const int cw = warp - C::kFirstConv;
        const int q = warp & 3, hs = (cw >> 2) & 1;
        const uint32_t grp = cw >> 3;
        const int rho = 32 * q + lane;  // tile row == TMEM lane
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        const int Lp = (int)args.L;     // packed tiles only (L < 64)
        const int pack = (int)args.pack;
        const int xoff = pack > 1 ? (rho < Lp * pack ? (rho / Lp) * kChunk * Lp + rho % Lp : -1) : rho;
        const int istride = pack > 1 ? Lp : kRows;
        uint32_t s = 0, ph = 0, b = 0, bph = 1, it = 0;
        bool ok = true;
        for (uint32_t w = blockIdx.x; w < args.nitems && ok; w += gridDim.x) {
            const uint32_t nc = chunk1(w) - chunk0(w);
            for (uint32_t kc = 0; kc < nc; ++kc, ++it) {
                if (C::kGroups == 1 || (it & 1) == grp) {
                    if (!__all_sync(0xffffffffu, mbar_wait(&full[s], ph, abort, flags))) {
                        ok = false;
                        break;
                    }
                    const uint8_t* xs = smem + s * C::kStage;
                    float v[16];
                    if (KMAJOR) {
                        // row rho: 128 B, 16-byte chunk j stored at chunk j ^ (rho & 7)
                        const uint8_t* row = xs + rho * 128;
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj) {
                            const int j = 4 * hs + jj;
                            const float4 f = *reinterpret_cast<const float4*>(row + ((j ^ (rho & 7)) << 4));
                            v[4 * jj] = f.x;
                            v[4 * jj + 1] = f.y;
                            v[4 * jj + 2] = f.z;
                            v[4 * jj + 3] = f.w;
                        }
                    } else {
                        // rows i of 128 floats (512 B, no swizzle): lanes read consecutive words.  Packed
                        // tiles hold [p][i][l] (p < pack, rows of L floats): tile row rho = l + L p; the
                        // rows past L pack are padding (zero)
                        const float* xf = reinterpret_cast<const float*>(xs);
#pragma unroll
                        for (int ii = 0; ii < 16; ++ii) {
                            const int i = 16 * hs + ii;
                            v[ii] = xoff >= 0 ? xf[xoff + i * istride] : 0.f;
                        }
                    }
                    uint32_t hi[16], lo[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) split_tf32(v[i], hi[i], lo[i]);
                    if (!__all_sync(0xffffffffu, mbar_wait(&aempty[b], bph, abort, flags))) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t ta = tbase + lane_base + C::kABuf + 64 * b + 16 * hs;
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
    } else if (warp >= C::kFirstEpi) {
        // ------------------------------------------------ epilogue
        // warp e drains TMEM lane quarter warp % 4 (the quarter a warp may access)
        const int q = warp & 3, half = (warp - C::kFirstEpi) >> 2;
        const int rho = 32 * q + lane;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        const int64_t m = args.m;
        uint32_t a = 0, aph = 0, sph = 0;
        const bool copier = warp == C::kFirstEpi && lane == 0;
        float srh = 0.f, srl = 0.f, sxh = 0.f, sxl = 0.f;  // RES: running sums as double-float pairs
        for (uint32_t w = blockIdx.x; w < args.nitems; w += gridDim.x) {
            const uint32_t w2 = ksplit == 1 ? w : w / ksplit, sk = w - w2 * ksplit;
            const uint32_t t = args.nblk == 1 ? w2 : w2 / args.nblk, nb = args.nblk == 1 ? 0 : w2 % args.nblk;
            const uint32_t nc = chunk1(w) - chunk0(w);
            const uint32_t nfill = FLAT ? 2 * nc : (nc + args.fill - 1) / args.fill;
            float* const outp = args.out + sk * args.out_numel;
            int64_t base, stride;
            bool valid;
            if (KMAJOR) {
                const int64_t r = (int64_t)t * kRows + rho;
                valid = r < args.R;
                base = r * m;
                stride = 1;
            } else {
                int64_t l, rr;
                if (FLAT) {
                    const uint32_t g = t * kRows + rho, L = (uint32_t)args.L, r = g / L;
                    valid = g < (uint32_t)(args.L * args.R);
                    l = g - r * L;
                    rr = r;
                } else if (args.pack > 1) {  // packed tile: row rho = l + L p holds (l, r = pack t + p)
                    const int Lp = (int)args.L;
                    rr = (int64_t)t * args.pack + rho / Lp;
                    l = rho % Lp;
                    valid = rho < Lp * (int)args.pack && rr < args.R;
                } else {
                    const uint32_t r = args.tiles_per_r == 1 ? t : t / args.tiles_per_r;
                    rr = r;
                    l = (int64_t)(t - r * args.tiles_per_r) * kRows + rho;
                    valid = l < args.L;
                }
                base = l + args.L * m * rr;
                stride = args.L;
            }
            const int col0 = (int)nb * NPAD;
            base += col0 * stride;
            const int ncol = (int)(m - col0);  // valid columns in this block (may exceed NPAD)
            // the warp's 16-column slices half, half + 2, ...: each fill's small terms, then its large ones, in
            // the order of the fills; the loads of a slice are in flight together
            constexpr int kSl = (NPAD / 16 + 1) / 2;
            float v[kSl][16];
            bool ok = true;
            if constexpr (RES) {
                // the warp's columns of xref on their way into L2 while the product is formed, a column a lane
                const int c = 16 * half + (lane & 15) + 32 * (lane >> 4);
                const int64_t l = (int64_t)t * kRows + 32 * q, rows = args.L - l < 32 ? args.L - l : 32;
                if (c < ncol && rows > 0) {
                    const int es = args.xrdt == TK_F32 ? 4 : (args.xrdt == TK_BF16 ? 2 : 1);
                    const char* x = static_cast<const char*>(args.xref) + (l + (col0 + c) * args.L) * es;
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(x));
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(x + rows * es - 1));
                }
            }
            for (uint32_t f = 0; f < nfill; ++f) {
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
            bool bad = any_nonfinite(v[0]);
#pragma unroll
            for (int j = 1; j < kSl; ++j)
                if (16 * half + 32 * j < NPAD) bad = bad || any_nonfinite(v[j]);
            if (valid && bad) again = 1;  // (see exact_items)
            if constexpr (RES) {
                if (valid) {
#pragma unroll
                    for (int j = 0; j < 2 * kSl; ++j) {
                        const int c0 = 16 * half + 32 * (j >> 1) + 8 * (j & 1);
                        const float* p = &v[j >> 1][8 * (j & 1)];
                        const int64_t o = base + c0 * stride;
                        float fr = 0.f, fx = 0.f;
                        residual_columns(args, o, ncol - c0, p, fr, fx);
                        ef_add(srh, srl, fr);
                        ef_add(sxh, sxl, fx);
                    }
                }
                continue;
            }
            // L == 1: the tile's rows are one run of the result.  Unless its lanes can store them in 16 bytes, it
            // goes out as one bulk copy from a staged copy (4-byte stores of each lane's row reach L2 as pieces of
            // sectors: 512^3, 42 columns 127 -> 98 us; 413 x 350 x 275, 30 columns 59 -> 56)
            float* const tile = outp + (int64_t)t * kRows * m;
            if (C::kOut && (m & 3) != 0 && args.nblk == 1 && (int64_t)(t + 1) * kRows <= args.R &&
                (reinterpret_cast<uintptr_t>(tile) & 15) == 0) {
                if (copier) {
                    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // the tile before has been read
                    mbar_arrive(stgfree);
                }
                if (!__all_sync(0xffffffffu, mbar_wait(stgfree, sph, abort, flags))) break;
                float* const row = stg + rho * (int)m;
#pragma unroll
                for (int j = 0; j < kSl; ++j) {
                    const int c0 = 16 * half + 32 * j;
                    if (c0 >= NPAD) break;
                    if ((m & 1) == 0) {
#pragma unroll
                        for (int i = 0; i < 16; i += 2)
                            if (c0 + i < ncol) *reinterpret_cast<float2*>(row + c0 + i) = make_float2(v[j][i], v[j][i + 1]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (c0 + i < ncol) row[c0 + i] = v[j][i];
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the copy reads what was written here
                __syncwarp();
                if (lane == 0) mbar_arrive(stgfull);
                if (copier) {
                    if (mbar_wait(stgfull, sph, abort, flags)) {
                        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(tile),
                                     "r"(smem_u32(stg)), "r"((uint32_t)(kRows * 4 * m))
                                     : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
                __syncwarp();
                sph ^= 1;
                continue;
            }
            if (valid) {
#pragma unroll
                for (int j = 0; j < kSl; ++j) {
                    const int c0 = 16 * half + 32 * j;
                    if (c0 >= NPAD) break;
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
        if (C::kOut && copier) asm volatile("cp.async.bulk.wait_group 0;\n\tfence.proxy.async;" ::: "memory");
        if constexpr (RES)
            residual_sums<C::kEpi>(warp - C::kFirstEpi, lane, ef_value(srh, srl), ef_value(sxh, sxl), args.partials);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tbase) : "memory");
    }
    if (again && !*abort) {
        if constexpr (RES) {
            exact_residual(args, NPAD);
        } else {
            exact_items<float, KMAJOR, FLAT>(args, NPAD, kChunk, 1.f);
        }
    }
}

template <int NPAD, bool KMAJOR, bool FLAT, bool RES = false>
static void ttm_tf32_launch(const Ctx& c, const CUtensorMap& tx, const CUtensorMap& tb,
                            typename std::conditional<RES, TtmResArgs, TtmArgs>::type a) {
    using Cf = TtmCfg<NPAD, KMAJOR, FLAT>;
    // above 64 columns a drain every 4 chunks would bound the pass (512^3, 81 columns: 174 against 121 us);
    // up to 8, the sketch widths, every chunk is drained: the FP32 FMA kernel that streamed those before
    // rounds every addition to nearest (512^3 sketches: 2.4e-7, FMA 3.3e-7, 5.8e-7 with 4 chunks; 104 and
    // 98 us a pass, FMA 131 and 115, 94 and 90 with 4)
    a.fill = a.m <= 8 ? 1 : (NPAD <= 64 ? 4 : 16);
    auto kern = ttm_tf32x3_kernel<NPAD, KMAJOR, FLAT, RES>;
    static std::atomic<uint64_t> opted{0};
    smem_opt_in(opted, reinterpret_cast<const void*>(kern), Cf::kSmem);
    const int grid = (int)std::min<int64_t>(a.nitems, grid_sms(c));
    run_kernel(c, kern, grid, Cf::kThreads, Cf::kSmem, tx, tb, a);
}

// The kernel for npad output columns per block (a multiple of 16 up to 96).
template <bool FLAT>
static void ttm_tf32_dispatch(const Ctx& c, int64_t npad, bool kmajor, const CUtensorMap& tx, const CUtensorMap& tb,
                              const TtmArgs& a) {
#define TK_TC_CASE(NP)                                                           \
    case NP:                                                                     \
        if (kmajor) ttm_tf32_launch<NP, true, FLAT>(c, tx, tb, a);               \
        else ttm_tf32_launch<NP, false, FLAT>(c, tx, tb, a);                     \
        break;
    switch (npad) {
        TK_TC_CASE(16)
        TK_TC_CASE(32)
        TK_TC_CASE(48)
        TK_TC_CASE(64)
        TK_TC_CASE(80)
        TK_TC_CASE(96)
        default: fail(TK_ERR_SHAPE, "ttm_tc: unsupported width");
    }
#undef TK_TC_CASE
}

void ttm_tf32_run_tma(const Ctx& c, int64_t npad, bool kmajor, const CUtensorMap& tx, const CUtensorMap& tb,
                      const TtmArgs& a);
void ttm_tf32_run_flat(const Ctx& c, int64_t npad, bool kmajor, const CUtensorMap& tx, const CUtensorMap& tb,
                       const TtmArgs& a);
// Fused with the comparison with xref (RES): blocks of 64 columns.
void ttm_tf32_run_residual(const Ctx& c, bool flat, const CUtensorMap& tx, const CUtensorMap& tb, const TtmResArgs& a);

}  // namespace tc
}  // namespace tk
