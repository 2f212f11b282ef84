// Host side of the TF32 tensor-core TTMs on sm_103a (kernels: tk_ttm_tf32.cuh, tk_ttm_lowp.cuh,
// tk_expand_tf32.cu): the TF32 split of the factors, the choice of tiles, tensor maps and launches.
#include <algorithm>
#include <cmath>

#include "tk_expand_tf32.cuh"
#include "tk_ttm_lowp.cuh"
#include "tk_ttm_tf32.cuh"

namespace tk {
namespace tc {

__device__ __forceinline__ uint32_t tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// The blocks that split a factor of n values, each of which sets or clears a flag of its own: whether a part is
// infinite or NaN (an infinity or NaN in M, or a value that rounds to an infinity).
constexpr int kSplitThreads = 256;
inline int64_t split_blocks(int64_t n) { return std::min<int64_t>((n + kSplitThreads - 1) / kSplitThreads, 1024); }
inline size_t info_bytes(int64_t n) { return sizeof(FactorInfo) + sizeof(int) * (size_t)split_blocks(n); }

// hi = rn_tf32(M(i, a)), lo = rn_tf32(M(i, a) - hi), stored K-major: (i, a) at i + ldo*a,
// a in [0, rows_b) with zero padding beyond m.
struct SplitJob {
    const void* M;
    int dt, mtrans;
    int64_t ldm, nj, m, rows_b, ldo;
    float* hi;
    float* lo;
    FactorInfo* info;
    uint32_t blocks;
};
constexpr int kMaxSplitJobs = 8;
template <int NB>
struct SplitBatch {
    SplitJob job[NB];
};

// One factor, or several in one launch (blockIdx.y).
template <int NB>
__global__ void __launch_bounds__(kSplitThreads) split_tf32_kernel(const __grid_constant__ SplitBatch<NB> sb) {
    kernel_begin();
    const SplitJob& jb = sb.job[NB > 1 ? blockIdx.y : 0];
    if (blockIdx.x >= jb.blocks) return;
    float t = 0.f;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < jb.ldo * jb.rows_b;
         idx += (int64_t)jb.blocks * blockDim.x) {
        const int64_t i = idx % jb.ldo, a = idx / jb.ldo;
        double v = 0.0;
        if (i < jb.nj && a < jb.m) {
            const int64_t o = jb.mtrans ? a + jb.ldm * i : i + jb.ldm * a;
            v = jb.dt == TK_F64 ? static_cast<const double*>(jb.M)[o] : (double)static_cast<const float*>(jb.M)[o];
        }
        const float h = __uint_as_float(tf32_rna((float)v));
        const float l = __uint_as_float(tf32_rna((float)(v - (double)h)));
        jb.hi[idx] = h;
        jb.lo[idx] = l;
        t = fmaf(l, 0.f, t);
    }
    const int bad = __syncthreads_or(t != t);
    if (threadIdx.x != 0) return;
    jb.info->bad[blockIdx.x] = bad;
    if (blockIdx.x == 0) {
        jb.info->M = jb.M;
        jb.info->ldm = jb.ldm;
        jb.info->dt = jb.dt;
        jb.info->mtrans = jb.mtrans;
        jb.info->nbad = jb.blocks;
    }
}

// out = the sum of the ksplit partial products part[s n .. s n + n), in order of s.
__global__ void splitk_sum_kernel(const float* __restrict__ part, int ksplit, int64_t n, float* __restrict__ out) {
    kernel_begin();
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        float v = part[e];
        for (int sk = 1; sk < ksplit; ++sk) v += part[(int64_t)sk * n + e];
        out[e] = v;
    }
}

// Self-test of the bounded wait: one warp waits, through the same mbar_wait_warp
// the tcgen05 kernels use, on an mbarrier that nothing ever arrives at, so the
// wait must give up after limit_ns, raise FLAG_TIMEOUT and let the kernel
// return.  waited[0] receives the nanoseconds the wait lasted.
__global__ void __launch_bounds__(32) wait_selftest_kernel(uint64_t limit_ns, unsigned* flags, long long* waited) {
    kernel_begin();
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort;
    if (threadIdx.x == 0) {
        abort = 0;
        mbar_init(&bar, 1);
    }
    __syncthreads();
    const uint64_t t0 = gtimer();
    const bool ok = mbar_wait_warp(&bar, 0, &abort, flags, limit_ns);
    if (threadIdx.x == 0) waited[0] = ok ? -1 : (long long)(gtimer() - t0);
}

}  // namespace tc

void launch_wait_selftest(const Ctx& c, uint64_t limit_ns, long long* waited) {
    if (!c.exec) return;
    run_kernel(c, tc::wait_selftest_kernel, 1, 32, 0, limit_ns, c.dflags, waited);
    c.counted();
    c.check_launch();
}

// How a product of contraction length nj and m output columns is blocked, which also fixes the layout of the
// factor's split.  Expansions (a short contraction into many columns, every fused residual among them):
// blocks of 32 or 64 columns (tk_expand_tf32.cu).  Plain ones take that kernel from twice as many columns
// out as elements in (512^3, 32 -> 512: 103 us against 262), but not along the leading mode or with few
// rows before it, where its rows of W are scattered (64^3 -> 1024 x 64 x 64: 77 us against 16).  Other products: up to 96
// columns in one block padded to 16, else blocks of 64.  BF16 and FP8 data (tk_ttm_lowp.cuh, stages of 64 K):
// equal blocks of up to 64.
struct Blocks {
    int64_t npad, nblk;
    bool expand;
};

static Blocks tc_blocks(int64_t L, int64_t nj, int64_t m, bool residual, tk_dtype dt) {
    if (dt != TK_F32) {
        const int64_t nb = (m + 63) / 64;
        return {((m + nb - 1) / nb + 15) / 16 * 16, nb, false};
    }
    if (residual || (L >= 32 && nj <= tc::kExpandK && m >= 64 && m >= 2 * nj)) {
        const int64_t nb = tc::expand_cols(nj);
        return {nb, (m + nb - 1) / nb, true};
    }
    if (m <= 96) return {(m + 15) / 16 * 16, 1, false};
    return {64, (m + 63) / 64, false};
}

// The factor splits that tensor-core TTMs about to run will need, made in one
// launch and entered in the call's split cache (c.split_cache must be on while
// those TTMs run).  Factors already split are skipped.
void tc_presplit(Ctx& c, const std::vector<TcSplitReq>& reqs) {
    tc::SplitBatch<tc::kMaxSplitJobs> sb{};
    int nj_ = 0;
    int64_t most = 0, blocks = 1;
    for (const TcSplitReq& q : reqs) {
        const Blocks bl = tc_blocks(q.L, q.nj, q.m, q.residual, q.dt);
        const int64_t npad = bl.npad, ldo = (q.nj + 3) / 4 * 4, rows_b = npad * bl.nblk;
        bool have = false;
        for (const Ctx::Split& e : c.splits)
            have = have || (e.p == q.M.p && e.dt == (int)q.M.dt && e.ld == q.M.ld && e.mtrans == (q.mtrans ? 1 : 0) &&
                            e.nj == q.nj && e.m == q.m && e.npad == npad && e.rows == rows_b);
        if (have || nj_ == tc::kMaxSplitJobs) continue;
        float* hi = c.alloc<float>(ldo * rows_b);
        float* lo = c.alloc<float>(ldo * rows_b);
        const int64_t nb = tc::split_blocks(ldo * rows_b);
        auto* info = static_cast<tc::FactorInfo*>(c.alloc_bytes(tc::info_bytes(ldo * rows_b)));
        c.splits.push_back({q.M.p, q.M.ld, q.nj, q.m, npad, rows_b, (int)q.M.dt, q.mtrans ? 1 : 0, hi, lo, info});
        sb.job[nj_++] = {q.M.p, (int)q.M.dt, q.mtrans ? 1 : 0, q.M.ld, q.nj, q.m, rows_b, ldo, hi, lo, info, (uint32_t)nb};
        most = std::max(most, ldo * rows_b);
        blocks = std::max(blocks, nb);
    }
    if (!c.exec || nj_ == 0) return;
    ProfScope ps(c, "elementwise", 16.0 * most * nj_, 0.0);
    run_kernel(c, tc::split_tf32_kernel<tc::kMaxSplitJobs>, dim3((unsigned)blocks, (unsigned)nj_), tc::kSplitThreads, 0, sb);
    c.counted();
    c.check_launch();
}

// The strides and base address TMA needs for a TTM of FP32 data along mode j.
static bool tma_ok(const Tens& X, int j) {
    const int64_t L = X.left(j), nj = X.n[j], R = X.right(j);
    if (X.dt != TK_F32 || ((uintptr_t)X.p % 16) != 0) return false;
    if (L >= ((int64_t)1 << 31) || R >= ((int64_t)1 << 31) || nj >= ((int64_t)1 << 31)) return false;
    return L == 1 ? nj % 4 == 0 : L % 4 == 0;
}

enum class TcRoute { None, Tma, Flat, Lowp };

// The estimated times (us) of a product that both the SIMT kernels and the tensor cores could take, fitted to a sweep
// over 20 .. 300001 rows, n_j = 2 .. 9001 and m = 3 .. 120 in every data type.
//  * SIMT: 6.5 us, a CTA per slab: 0.06 to 0.2 us per step of a part, 0.65 products a ps, 1.5 us and 7 ns a step for each
//    further wave; else n_j steps of 0.1 us, 2.3 products a ps, 1.2 TB/s, and for the tiled kernel 4.4 products a ps
//    with n_j padded to 16 and m to 32.
//  * Tensor cores: 14 us on the device with the split of the factor, 7 on the host for its launch, which is what calls
//    on small tensors wait for; 3 TB/s (expansions 4.5), and for each further wave of tiles 0.035 us a column, or 0.75 us
//    for each chunk of 32 (0.65 of 64 for BF16 and FP8), and 1.2 us (2.2) where the tile has one chunk only.
// E.g. 413 x 350 x 275 along its last mode, 36 columns: 1337 us SIMT, 57; 9001 x 333, 20: 78 and 10; 900000 x 2,
// 26 columns: 104 and 150; 2512 x 48 along the first mode, 5 columns: 15 and 16 in two launches.
struct TtmTimes {
    double simt, tc;
};

static TtmTimes ttm_times(const Tens& X, int j, int64_t m) {
    const int64_t L = X.left(j), nj = X.n[j], R = X.right(j), rows = L * R;
    const bool f32 = X.dt == TK_F32;
    const double work = (double)rows * (double)nj * (double)m;
    const double bytes = (double)rows * (double)((int64_t)dtype_size(X.dt) * nj + 4 * m);
    TtmTimes t;
    if (ttm_simt_slab(L, nj, R, m, 4)) {
        const double waves = std::ceil((double)R / (8 * 152)) - 1.0, step = 0.06 + 0.0006 * (double)(L * m);
        t.simt = 6.5 + std::max({step * (double)nj / ttm_simt_slab_parts(L, m), work / 0.65e6, waves * (1.5 + 0.007 * nj)});
    } else {
        t.simt = std::max({0.1 * (double)nj, work / 2.3e6, bytes / 1.2e6});
        if (!ttm_simt_direct(rows, nj, m))
            t.simt = std::max(t.simt, (double)rows * (double)((nj + 15) / 16 * 16) * (double)((m + 31) / 32 * 32) / 4.4e6);
    }
    t.tc = 21.0;
    const Blocks bl = tc_blocks(L, nj, m, false, X.dt);
    if (bl.expand) {
        t.tc += bytes / 4.5e6;
    } else {
        const double tiles = (double)((rows + tc::kRows - 1) / tc::kRows) * (double)bl.nblk;
        const double chunks = (double)(f32 ? (nj + 31) / 32 : (nj + 63) / 64);
        const double tile = std::max((chunks > 1.0 ? 0.0 : (f32 ? 1.2 : 2.2)) + 0.035 * (double)std::min(m, bl.npad),
                                     (f32 ? 0.75 : 0.65) * chunks);
        t.tc += std::max(bytes / 3e6, (std::ceil(tiles / 152.0) - 1.0) * tile);
    }
    return t;
}

static bool tc_faster(const Tens& X, int j, int64_t m) {
    const TtmTimes t = ttm_times(X, j, m);
    return t.simt >= t.tc;
}

// Which form of the tensor-core kernel takes a TTM.
//  * TMA: 16-byte strides, n_j >= 32, and rows enough to fill tiles: L == 1 with R >= 128, or L >= 32 (below
//    64 by packing slabs).
//  * everything else the SIMT kernels could take as well: the tensor cores where they are the faster ones.
//  * BF16 and FP8 that their own kernels do not take: the same rule, for L == 1 or L >= 32 (shorter runs
//    cost more in their 16-byte pieces than they hold).  E.g. BF16 689 x 690 x 700 along its first mode, 10 columns:
//    3435 us SIMT, 178; FP8 768^3 along its last, 9: 1541 and 176.
static TcRoute lowp_route(const Tens& X, int j, int64_t m) {
    const int64_t L = X.left(j), nj = X.n[j], R = X.right(j);
    if (ttm_bf16_eligible(X, j, m, TK_F32) || ttm_fp8_eligible(X, j, m, TK_F32)) return TcRoute::None;
    if (nj < 1 || ((uintptr_t)X.p % 16) != 0 || nj >= ((int64_t)1 << 31) || (L != 1 && L < 32)) return TcRoute::None;
    const int64_t rows = L * R;
    if (rows < 1 || rows >= ((int64_t)1 << 31) - tc::kRows) return TcRoute::None;
    return tc_faster(X, j, m) ? TcRoute::Lowp : TcRoute::None;
}

static TcRoute tc_route(const Tens& X, int j, int64_t m, tk_dtype out_dt) {
    if (out_dt != TK_F32 || X.dt == TK_F64) return TcRoute::None;
    if (m < 1 || m > 65535) return TcRoute::None;
    if (X.dt != TK_F32) return lowp_route(X, j, m);
    const int64_t L = X.left(j), nj = X.n[j], R = X.right(j);
    const bool tma = tma_ok(X, j) && (L == 1 ? R >= tc::kRows : L >= 32);
    if (nj >= 32 && tma) return TcRoute::Tma;
    if (nj < 1 || ((uintptr_t)X.p % 16) != 0 || nj >= ((int64_t)1 << 31)) return TcRoute::None;
    const int64_t rows = L * R;
    if (rows < 1 || rows >= ((int64_t)1 << 31) - tc::kRows) return TcRoute::None;
    // streams of 4 million elements and more with 16-byte strides: HBM-bound at 2-3 times the SIMT rate
    if (rows * nj >= ((int64_t)1 << 22) && tma_ok(X, j)) return tma ? TcRoute::Tma : TcRoute::Flat;
    if (!tc_faster(X, j, m)) return TcRoute::None;
    return tma ? TcRoute::Tma : TcRoute::Flat;
}

bool ttm_tc_eligible(const Tens& X, int j, int64_t m, tk_dtype out_dt) {
    return tc_route(X, j, m, out_dt) != TcRoute::None;
}

double ttm_estimate(const Tens& X, int j, int64_t m, bool use_tc) {
    const TtmTimes t = ttm_times(X, j, m);
    if (!use_tc || !ttm_tc_eligible(X, j, m, TK_F32)) return t.simt + 5.0;
    // the device's part; a tile row's outputs are contiguous along the leading mode: 0.9 (192 columns from 9) to 1.7 TB/s
    const double tc = t.tc - 7.0;
    return X.left(j) == 1 ? std::max(tc, 14.0 + 4.0 * (double)X.right(j) * (double)m / 1e6) : tc;
}

// The TF32 parts of factor M in the layout the kernels load, from the call's split cache or made here.
struct Factor {
    float* hi = nullptr;
    float* lo = nullptr;
    tc::FactorInfo* info = nullptr;
    int64_t ldo = 0, rows_b = 0;
    bool have = false;
};

static Factor factor_alloc(Ctx& c, const Mat& M, bool mtrans, int64_t nj, int64_t m, int64_t npad, int64_t nblk) {
    Factor f;
    f.ldo = (nj + 3) / 4 * 4;
    f.rows_b = npad * nblk;
    if (c.split_cache) {
        for (const Ctx::Split& e : c.splits)
            if (e.p == M.p && e.dt == (int)M.dt && e.ld == M.ld && e.mtrans == (mtrans ? 1 : 0) && e.nj == nj &&
                e.m == m && e.npad == npad && e.rows == f.rows_b) {
                f.hi = e.hi;
                f.lo = e.lo;
                f.info = static_cast<tc::FactorInfo*>(e.info);
                f.have = true;
                return f;
            }
    }
    f.hi = c.alloc<float>(f.ldo * f.rows_b);
    f.lo = c.alloc<float>(f.ldo * f.rows_b);
    f.info = static_cast<tc::FactorInfo*>(c.alloc_bytes(tc::info_bytes(f.ldo * f.rows_b)));
    if (c.split_cache)
        c.splits.push_back({M.p, M.ld, nj, m, npad, f.rows_b, (int)M.dt, mtrans ? 1 : 0, f.hi, f.lo, f.info});
    return f;
}

// Splits the factor unless it already is, and makes the tensor map of its parts: hi and lo as the two layers of
// one tensor (lo lies above hi in the workspace), so that one load brings both.
static void factor_map(Ctx& c, const Factor& f, const Mat& M, bool mtrans, int64_t nj, int64_t m, int64_t npad,
                       CUtensorMap* tb) {
    if (!f.have) {
        const int64_t tot = f.ldo * f.rows_b;
        ProfScope ps(c, "elementwise", 8.0 * tot + 8.0 * nj * m, 0.0);
        const int64_t nb = tc::split_blocks(tot);
        const tc::SplitBatch<1> sb{{{M.p, (int)M.dt, mtrans ? 1 : 0, M.ld, nj, m, f.rows_b, f.ldo, f.hi, f.lo, f.info,
                                     (uint32_t)nb}}};
        run_kernel(c, tc::split_tf32_kernel<1>, (unsigned)nb, tc::kSplitThreads, 0, sb);
        c.counted();
        c.check_launch();
    }
    const uint64_t dims[3] = {(uint64_t)nj, (uint64_t)f.rows_b, 2};
    const uint64_t str[2] = {(uint64_t)f.ldo * 4, (uint64_t)((char*)f.lo - (char*)f.hi)};
    const uint32_t box[3] = {tc::kChunk, (uint32_t)npad, 2};
    tc::encode(tb, f.hi, 3, dims, str, box);
}

// The tensor map of X's chunks along mode j for a strided contraction: 128 rows x 32 K elements, or L rows of pack
// consecutive slabs (L x 4 bytes: a multiple of 16).
static void strided_map(const Tens& X, int j, int64_t pack, CUtensorMap* tx) {
    const int64_t L = X.left(j), nj = X.n[j];
    const uint64_t dims[3] = {(uint64_t)L, (uint64_t)nj, (uint64_t)X.right(j)};
    const uint64_t str[2] = {(uint64_t)L * 4, (uint64_t)L * nj * 4};
    const uint32_t box[3] = {pack > 1 ? (uint32_t)L : (uint32_t)tc::kRows, tc::kChunk, (uint32_t)pack};
    tc::encode(tx, X.p, 3, dims, str, box, false);
}

// The expansion kernel's work: row tiles x parts of their column blocks.
static tc::ExpandArgs expand_args(const Ctx& c, const Tens& W, int j, int64_t m, const Blocks& bl) {
    tc::ExpandArgs a{};
    a.L = W.left(j);
    a.nj = W.n[j];
    a.m = m;
    a.W = static_cast<const float*>(W.p);
    const int64_t rows = a.L * W.right(j), tile = tc::expand_tile(a.nj), sms = tc::grid_sms(c);
    a.rows = (uint32_t)rows;
    const int64_t ntiles = (rows + tile - 1) / tile;
    const int64_t ncs = tc::expand_parts(ntiles, bl.nblk, a.nj, sms);
    TK_REQUIRE(ntiles * ncs < ((int64_t)1 << 31), TK_ERR_SHAPE, "ttm_tc: too many tiles");
    a.ntiles = (uint32_t)ntiles;
    a.nblk = (uint32_t)bl.nblk;
    a.ncs = (uint32_t)ncs;
    a.nitems = (uint32_t)(ntiles * ncs);
    a.nk = (uint32_t)((a.nj + tc::kChunk - 1) / tc::kChunk);
    a.flags = c.dflags;
    return a;
}

// Few row tiles: the K chunks of each are split over several items, at least two chunks each.
static int64_t split_chunks(const Ctx& c, int64_t items, int64_t nk) {
    const int64_t sms = tc::grid_sms(c);
    return items * 2 <= sms && nk >= 4 ? std::max<int64_t>(1, std::min<int64_t>(nk / 2, sms / items)) : 1;
}

static void sum_parts(Ctx& c, const float* part, int64_t ksplit, int64_t n, float* out) {
    run_kernel(c, tc::splitk_sum_kernel, (unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, part,
               (int)ksplit, n, out);
    c.counted();
    c.check_launch();
}

// BF16 / FP8 data (tk_ttm_lowp.cuh).  TMA where the strides are multiples of 16 bytes and a mode is before the
// contracted one, else the loaders, whose runs (a K row of the tile; with L == 1 a row's 64 elements) begin anywhere.
static void launch_ttm_lowp(Ctx& c, const Tens& X, int j, const Mat& M, bool mtrans, int64_t m, float* out,
                            const char* name) {
    const int64_t L = X.left(j), nj = X.n[j], R = X.right(j), es = (int64_t)dtype_size(X.dt);
    const bool kmajor = L == 1;
    const Blocks bl = tc_blocks(L, nj, m, false, X.dt);
    const Factor f = factor_alloc(c, M, mtrans, nj, m, bl.npad, bl.nblk);
    const int64_t pack = !kmajor && L < tc::kRows / 2 ? tc::kRows / L : 1;
    const int64_t nk = (nj + tc::kLowpChunk - 1) / tc::kLowpChunk;
    const int64_t tiles_per_r = kmajor || pack > 1 ? 1 : (L + tc::kRows - 1) / tc::kRows;
    const int64_t ntiles = kmajor ? (R + tc::kRows - 1) / tc::kRows : (pack > 1 ? (R + pack - 1) / pack : R * tiles_per_r);
    const int64_t ksplit = split_chunks(c, ntiles * bl.nblk, nk);
    TK_REQUIRE(ntiles * bl.nblk * ksplit < ((int64_t)1 << 31), TK_ERR_SHAPE, "ttm_lowp: too many tiles");
    float* part = ksplit > 1 ? c.alloc<float>(ksplit * L * m * R) : nullptr;
    if (!c.exec) return;
    const bool tma = !kmajor && (L * es) % 16 == 0;
    const int64_t run = es * (pack > 1 ? L : tc::kRows);  // bytes of a tile's K row in one slab
    CUtensorMap tx, tb;
    factor_map(c, f, M, mtrans, nj, m, bl.npad, &tb);
    tx = tb;  // unused by the loaders
    if (tma) {
        const uint64_t dims[3] = {(uint64_t)L, (uint64_t)nj, (uint64_t)R};
        const uint64_t str[2] = {(uint64_t)(L * es), (uint64_t)(L * nj * es)};
        const uint32_t box[3] = {(uint32_t)(pack > 1 ? L : tc::kRows), tc::kLowpChunk, (uint32_t)pack};
        tc::encode(&tx, X.p, 3, dims, str, box, false,
                   es == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16);
    }
    tc::LowpArgs a{};
    a.L = L;
    a.nj = nj;
    a.R = R;
    a.m = m;
    a.ntiles = (uint32_t)ntiles;
    a.tiles_per_r = (uint32_t)tiles_per_r;
    a.nk = (uint32_t)nk;
    a.nblk = (uint32_t)bl.nblk;
    a.nitems = (uint32_t)(ntiles * bl.nblk * ksplit);
    a.pack = (uint32_t)pack;
    a.ksplit = (uint32_t)ksplit;
    // a run that starts anywhere spans up to 15 bytes more than it has
    a.slot = (uint32_t)(tma ? run : (kmajor ? tc::kLowpChunk * es + 16 : (run + 15 + 15) / 16 * 16));
    const uint32_t runs = (uint32_t)(kmajor ? tc::kRows : tc::kLowpChunk * pack);
    a.xstage = (runs * a.slot + 1023) / 1024 * 1024;
    a.tma = tma ? 1 : 0;
    a.xbytes = tma ? runs * a.slot : 0;
    a.x_inv = X.dt == TK_FP8_E4M3 ? 1.f / X.scale : 1.f;
    a.X = static_cast<const uint8_t*>(X.p);
    a.info = f.info;
    a.out_numel = L * m * R;
    a.out = ksplit > 1 ? part : out;
    a.flags = c.dflags;
    {
        ProfScope ps(c, name, (double)es * L * R * nj + 8.0 * nj * m + 4.0 * (double)L * R * m,
                     2.0 * (double)L * R * nj * m);
        if (es == 1) tc::ttm_lowp_run_fp8(c, bl.npad, kmajor, tx, tb, a);
        else tc::ttm_lowp_run_bf16(c, bl.npad, kmajor, tx, tb, a);
        c.counted();
        c.check_launch();
    }
    if (ksplit > 1) sum_parts(c, part, ksplit, L * m * R, out);
}

void launch_ttm_tc(Ctx& c, const Tens& X, int j, const Mat& M, bool mtrans, int64_t m, float* out) {
    const int64_t L = X.left(j), R = X.right(j);
    // kernel classes: "xpass_tc" streams all of X (a pass over the input),
    // "ttm_tc" contracts an intermediate
    const char* name = ((const void*)X.p == c.xdata || L * R * m == c.xnumel) ? (c.background ? "xpass_tc_bg" : "xpass_tc")
                                                                              : "ttm_tc";
    const int64_t nj = X.n[j];
    const TcRoute route = tc_route(X, j, m, TK_F32);
    TK_REQUIRE(route != TcRoute::None, TK_ERR_SHAPE, "ttm_tc: shape not supported");
    if (route == TcRoute::Lowp) {
        launch_ttm_lowp(c, X, j, M, mtrans, m, out, name);
        return;
    }
    const bool flat = route == TcRoute::Flat, kmajor = (L == 1);
    const Blocks bl = tc_blocks(L, nj, m, false, TK_F32);
    const int64_t npad = bl.npad, nblk = bl.nblk;
    const Factor f = factor_alloc(c, M, mtrans, nj, m, npad, nblk);
    if (bl.expand && L * R < ((int64_t)1 << 31) - 256) {  // (more rows: the general kernel, same blocks)
        if (!c.exec) return;
        CUtensorMap tb;
        factor_map(c, f, M, mtrans, nj, m, npad, &tb);
        tc::ExpandArgs a = expand_args(c, X, j, m, bl);
        a.out = out;
        a.info = f.info;
        ProfScope ps(c, name, 4.0 * (double)L * R * nj + 8.0 * nj * m + 4.0 * (double)L * R * m,
                     2.0 * (double)L * R * nj * m);
        tc::expand_run(c, 0, TK_F32, tb, tb, a);
        c.counted();
        c.check_launch();
        return;
    }
    // the work items: 128-row tiles (TMA: a strided mode with under 64 rows before it packs several slabs
    // per tile) x blocks of NPAD output columns; too few of them for half the SMs split each tile's
    // K chunks over several items (at least two chunks each), whose partial products are summed in
    // order afterwards
    const int64_t pack = (!flat && !kmajor && L < tc::kRows / 2) ? tc::kRows / L : 1;
    const int64_t nk = (nj + tc::kChunk - 1) / tc::kChunk;
    const int64_t tiles_per_r = (flat || kmajor || pack > 1) ? 1 : (L + tc::kRows - 1) / tc::kRows;
    const int64_t ntiles = flat ? (L * R + tc::kRows - 1) / tc::kRows
                                : (kmajor ? (R + tc::kRows - 1) / tc::kRows
                                          : (pack > 1 ? (R + pack - 1) / pack : R * tiles_per_r));
    const int64_t ksplit = split_chunks(c, ntiles * nblk, nk);
    TK_REQUIRE(ntiles * nblk * ksplit < ((int64_t)1 << 31), TK_ERR_SHAPE, "ttm_tc: too many tiles");
    float* part = ksplit > 1 ? c.alloc<float>(ksplit * L * m * R) : nullptr;
    if (!c.exec) return;
    CUtensorMap tx, tb;
    factor_map(c, f, M, mtrans, nj, m, npad, &tb);
    if (flat) {
        tx = tb;  // unused
    } else if (kmajor) {
        const uint64_t dims[2] = {(uint64_t)nj, (uint64_t)R};
        const uint64_t str[1] = {(uint64_t)nj * 4};
        const uint32_t box[2] = {tc::kChunk, tc::kRows};
        tc::encode(&tx, X.p, 2, dims, str, box);
    } else {
        strided_map(X, j, pack, &tx);
    }
    tc::TtmArgs a{};
    a.L = L;
    a.nj = nj;
    a.R = R;
    a.m = m;
    a.ntiles = (uint32_t)ntiles;
    a.tiles_per_r = (uint32_t)tiles_per_r;
    a.nk = (uint32_t)nk;
    a.nblk = (uint32_t)nblk;
    a.nitems = (uint32_t)(ntiles * nblk * ksplit);
    a.pack = (uint32_t)pack;
    a.xbytes = (uint32_t)(flat ? 0 : (pack > 1 ? L * tc::kChunk * pack * 4 : tc::kXBytes));
    a.ksplit = (uint32_t)ksplit;
    a.vec = (kmajor ? nj : L) % 2 == 0 ? 2 : 1;
    a.X = static_cast<const float*>(X.p);
    a.info = f.info;
    a.out_numel = L * m * R;
    a.out = ksplit > 1 ? part : out;
    a.flags = c.dflags;
    {
        ProfScope ps(c, name, 4.0 * (double)L * R * nj + 8.0 * nj * m + 4.0 * (double)L * R * m,
                     2.0 * (double)L * R * nj * m);
        if (flat) tc::ttm_tf32_run_flat(c, npad, kmajor, tx, tb, a);
        else tc::ttm_tf32_run_tma(c, npad, kmajor, tx, tb, a);
        c.counted();
        c.check_launch();
    }
    if (ksplit > 1) sum_parts(c, part, ksplit, L * m * R, out);
}

// Fused residuals of a contraction longer than the expansion kernel holds run on the plain kernel, whose epilogue then
// compares instead of storing (512^3 FP32, K = 160: norms 573 us, with dX 653; stored and compared by kernels of their
// own 672 and 1206 us, and Xhat's 512 MB of workspace.  BF16 1024 x 1024 x 512, K = 192, where the MMAs bound it: 2754
// and 2586, with 2 GB).
static bool residual_plain(int64_t nj) { return nj > tc::kExpandKResid; }

bool ttm_tc_residual_eligible(const Tens& W, int j, int64_t m) {
    const int64_t rows = W.left(j), nj = W.n[j];
    return W.dt == TK_F32 && W.right(j) == 1 && nj >= 1 && nj < ((int64_t)1 << 31) && m >= 1 && m <= 65535 &&
           rows >= 1 && rows < ((int64_t)1 << 31) - 256 && ((uintptr_t)W.p % 16) == 0;
}

int tc_residual_ctas(const Ctx& c, const Tens& W, int j, int64_t m) {
    const Blocks bl = tc_blocks(W.left(j), W.n[j], m, true, TK_F32);
    if (!residual_plain(W.n[j])) return tc::expand_ctas(c, expand_args(c, W, j, m, bl));
    const int64_t ntiles = (W.left(j) + tc::kRows - 1) / tc::kRows;
    return (int)std::min<int64_t>(ntiles * bl.nblk, tc::grid_sms(c));
}

void launch_ttm_tc_residual(Ctx& c, const Tens& W, int j, const Mat& M, bool mtrans, int64_t m, const void* xref,
                            tk_dtype xrdt, void* dx, float alpha, double* partials, float xr_scale) {
    const int64_t L = W.left(j), nj = W.n[j];
    TK_REQUIRE(xrdt == TK_F32 || xrdt == TK_BF16 || (xrdt == TK_FP8_E4M3 && !dx), TK_ERR_DTYPE,
               "ttm_tc: residual reference must be F32/BF16 (FP8: norms only)");
    const Blocks bl = tc_blocks(L, nj, m, true, TK_F32);
    const Factor f = factor_alloc(c, M, mtrans, nj, m, bl.npad, bl.nblk);
    if (!c.exec) return;
    CUtensorMap tb, txr;
    factor_map(c, f, M, mtrans, nj, m, bl.npad, &tb);
    const int64_t es = (int64_t)dtype_size(xrdt);
    ProfScope ps(c, c.background ? "xpass_tc_bg" : "xpass_tc",
                 4.0 * (double)L * nj + 8.0 * nj * m + (dx ? 2.0 : 1.0) * es * (double)L * m, 2.0 * (double)L * nj * m);
    if (residual_plain(nj)) {
        const bool flat = !tma_ok(W, j) || L < tc::kRows;
        CUtensorMap tw = tb;  // unused by the loaders
        if (!flat) strided_map(W, j, 1, &tw);
        tc::TtmResArgs a{};
        a.L = L;
        a.nj = nj;
        a.R = 1;
        a.m = m;
        a.tiles_per_r = a.ntiles = (uint32_t)((L + tc::kRows - 1) / tc::kRows);
        a.nk = (uint32_t)((nj + tc::kChunk - 1) / tc::kChunk);
        a.nblk = (uint32_t)bl.nblk;
        TK_REQUIRE((int64_t)a.ntiles * bl.nblk < ((int64_t)1 << 31), TK_ERR_SHAPE, "ttm_tc: too many tiles");
        a.nitems = a.ntiles * a.nblk;
        a.pack = a.ksplit = 1;
        a.xbytes = flat ? 0 : (uint32_t)tc::kXBytes;
        a.vec = L % 2 == 0 ? 2 : 1;
        a.X = static_cast<const float*>(W.p);
        a.info = f.info;
        a.flags = c.dflags;
        a.xref = xref;
        a.xrdt = (int)xrdt;
        a.dx = dx;
        a.alpha = alpha;
        a.xr_scale = xr_scale;
        a.partials = partials;
        tc::ttm_tf32_run_residual(c, flat, tw, tb, a);
        c.counted();
        c.check_launch();
        return;
    }
    tc::ExpandArgs a = expand_args(c, W, j, m, bl);
    a.info = f.info;
    a.bulk = (L * es) % 16 != 0;
    a.xclip = (L * m * es) & ~(int64_t)15;
    txr = tb;  // unused when bulk
    if (!a.bulk) {
        const uint64_t dims[2] = {(uint64_t)L, (uint64_t)m};
        const uint64_t str[1] = {(uint64_t)(L * es)};
        const uint32_t box[2] = {(uint32_t)tc::expand_tile(nj), (uint32_t)tc::expand_cols(nj)};
        tc::encode(&txr, xref, 2, dims, str, box, false,
                   es == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                           : (es == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32));
    }
    a.out = dx;
    a.xref = xref;
    a.alpha = alpha;
    a.xr_scale = xr_scale;
    a.partials = partials;
    tc::expand_run(c, dx ? 2 : 1, xrdt, tb, txr, a);
    c.counted();
    c.check_launch();
}

}  // namespace tk
