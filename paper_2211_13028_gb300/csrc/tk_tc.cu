// Host side of the FP32 tensor-core TTMs on sm_103a (kernels: tk_ttm_tf32.cuh, tk_tc_residual.cu): the
// TF32 split of the factors, the choice of tiles, tensor maps and launches.
#include <algorithm>

#include "tk_tc_residual.cuh"
#include "tk_ttm_tf32.cuh"

namespace tk {
namespace tc {

__device__ __forceinline__ uint32_t tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// hi = rn_tf32(M(i, a)), lo = rn_tf32(M(i, a) - hi), stored K-major: (i, a) at i + ldo*a,
// a in [0, npad) with zero padding beyond m.
__global__ void split_tf32_kernel(const void* M, tk_dtype dt, int64_t ldm, int mtrans, int64_t nj, int64_t m,
                                  int64_t npad, int64_t ldo, float* hi, float* lo) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= ldo * npad) return;
    int64_t i = idx % ldo, a = idx / ldo;
    double v = 0.0;
    if (i < nj && a < m) {
        int64_t o = mtrans ? a + ldm * i : i + ldm * a;
        v = dt == TK_F64 ? static_cast<const double*>(M)[o] : (double)static_cast<const float*>(M)[o];
    }
    float h = __uint_as_float(tf32_rna((float)v));
    float l = __uint_as_float(tf32_rna((float)(v - (double)h)));
    hi[idx] = h;
    lo[idx] = l;
}

// Several factors split in one launch (blockIdx.y = factor): the same split
// as split_tf32_kernel for each.
struct SplitJob {
    const void* M;
    int dt, mtrans;
    int64_t ldm, nj, m, rows_b, ldo;
    float* hi;
    float* lo;
};
constexpr int kMaxSplitJobs = 8;
struct SplitBatch {
    SplitJob job[kMaxSplitJobs];
};

__global__ void split_tf32_batch_kernel(SplitBatch sb) {
    const SplitJob& jb = sb.job[blockIdx.y];
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < jb.ldo * jb.rows_b;
         idx += (int64_t)gridDim.x * blockDim.x) {
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
    }
}

// out = the sum of the ksplit partial products part[s n .. s n + n), in order of s.
__global__ void splitk_sum_kernel(const float* __restrict__ part, int ksplit, int64_t n, float* __restrict__ out) {
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
    tc::wait_selftest_kernel<<<1, 32, 0, c.stream>>>(limit_ns, c.dflags, waited);
    c.counted();
    c.check_launch();
}

// Output columns: up to 96 (64 for the residual epilogue, whose X tiles share
// shared memory with the pipeline) in one block padded to 16, else blocks of 64.
static void tc_blocks(int64_t m, int64_t& npad, int64_t& nblk, bool residual = false) {
    if (m <= (residual ? 64 : 96)) {
        npad = (m + 15) / 16 * 16;
        nblk = 1;
    } else {
        npad = 64;
        nblk = (m + 63) / 64;
    }
}

// The factor splits that tensor-core TTMs about to run will need, made in one
// launch and entered in the call's split cache (c.split_cache must be on while
// those TTMs run).  Factors already split are skipped.
void tc_presplit(Ctx& c, const std::vector<TcSplitReq>& reqs) {
    tc::SplitBatch sb;
    int nj_ = 0;
    int64_t most = 0;
    for (const TcSplitReq& q : reqs) {
        int64_t npad, nblk;
        tc_blocks(q.m, npad, nblk, q.residual);
        const int64_t ldo = (q.nj + 3) / 4 * 4, rows_b = npad * nblk;
        bool have = false;
        for (const Ctx::Split& e : c.splits)
            have = have || (e.p == q.M.p && e.dt == (int)q.M.dt && e.ld == q.M.ld && e.mtrans == (q.mtrans ? 1 : 0) &&
                            e.nj == q.nj && e.m == q.m && e.npad == npad && e.rows == rows_b);
        if (have || nj_ == tc::kMaxSplitJobs) continue;
        float* hi = c.alloc<float>(ldo * rows_b);
        float* lo = c.alloc<float>(ldo * rows_b);
        c.splits.push_back({q.M.p, q.M.ld, q.nj, q.m, npad, rows_b, (int)q.M.dt, q.mtrans ? 1 : 0, hi, lo});
        sb.job[nj_++] = {q.M.p, (int)q.M.dt, q.mtrans ? 1 : 0, q.M.ld, q.nj, q.m, rows_b, ldo, hi, lo};
        most = std::max(most, ldo * rows_b);
    }
    if (!c.exec || nj_ == 0) return;
    ProfScope ps(c, "elementwise", 16.0 * most * nj_, 0.0);
    tc::split_tf32_batch_kernel<<<dim3((unsigned)std::min<int64_t>((most + 255) / 256, 1024), (unsigned)nj_), 256, 0,
                                  c.stream>>>(sb);
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

enum class TcRoute { None, Tma, Flat };

// Which form of the tensor-core kernel takes a TTM.
//  * TMA: 16-byte strides, n_j >= 32, and rows enough to fill tiles: L == 1 with R >= 128, or L >= 32 (below
//    64 by packing slabs).
//  * everything else the SIMT kernels could take as well: the tensor cores where they are the faster
//    ones by the times below (us), fitted to a sweep over 1000 .. 300001 rows, n_j = 7 .. 333 and
//    m = 5 .. 45.  The SIMT kernels walk n_j in one thread (0.1 us a step), reach 2300 products a ns and
//    1.2 TB/s; the tensor cores need two launches (14 us with the split of the factor, and as much again
//    on the host, which is what calls on small tensors wait for) and stream 3 TB/s.
//    E.g. 413 x 350 x 275 along its last mode, 36 columns: 1337 us SIMT; 9001 x 333, 20: 78.
static TcRoute tc_route(const Tens& X, int j, int64_t m, tk_dtype out_dt) {
    if (X.dt != TK_F32 || out_dt != TK_F32) return TcRoute::None;
    if (m < 1 || m > 65535) return TcRoute::None;
    const int64_t L = X.left(j), nj = X.n[j], R = X.right(j);
    const bool tma = tma_ok(X, j) && (L == 1 ? R >= tc::kRows : L >= 32);
    if (nj >= 32 && tma) return TcRoute::Tma;
    if (nj < 1 || ((uintptr_t)X.p % 16) != 0 || nj >= ((int64_t)1 << 31)) return TcRoute::None;
    const int64_t rows = L * R;
    if (rows < 1 || rows >= ((int64_t)1 << 31) - tc::kRows) return TcRoute::None;
    const double bytes = 4.0 * (double)rows * (double)(nj + m);
    const double simt = std::max({0.1 * (double)nj, (double)rows * (double)nj * (double)m / 2.3e6, bytes / 1.2e6});
    if (simt < 28.0 + bytes / 3e6) return TcRoute::None;
    return tma ? TcRoute::Tma : TcRoute::Flat;
}

bool ttm_tc_eligible(const Tens& X, int j, int64_t m, tk_dtype out_dt) {
    return tc_route(X, j, m, out_dt) != TcRoute::None;
}

// The TF32 parts of factor M in the layout the kernels load, from the call's split cache or made here.
struct Factor {
    float* hi = nullptr;
    float* lo = nullptr;
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
                f.have = true;
                return f;
            }
    }
    f.hi = c.alloc<float>(f.ldo * f.rows_b);
    f.lo = c.alloc<float>(f.ldo * f.rows_b);
    if (c.split_cache) c.splits.push_back({M.p, M.ld, nj, m, npad, f.rows_b, (int)M.dt, mtrans ? 1 : 0, f.hi, f.lo});
    return f;
}

// Splits the factor unless it already is, and makes the tensor maps of its parts.
static void factor_maps(Ctx& c, const Factor& f, const Mat& M, bool mtrans, int64_t nj, int64_t m, int64_t npad,
                        CUtensorMap* th, CUtensorMap* tl) {
    if (!f.have) {
        const int64_t tot = f.ldo * f.rows_b;
        ProfScope ps(c, "elementwise", 8.0 * tot + 8.0 * nj * m, 0.0);
        tc::split_tf32_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, c.stream>>>(M.p, M.dt, M.ld, mtrans ? 1 : 0,
                                                                                   nj, m, f.rows_b, f.ldo, f.hi, f.lo);
        c.counted();
        c.check_launch();
    }
    const uint64_t dims[2] = {(uint64_t)nj, (uint64_t)f.rows_b};
    const uint64_t str[1] = {(uint64_t)f.ldo * 4};
    const uint32_t box[2] = {tc::kChunk, (uint32_t)npad};
    tc::encode(th, f.hi, 2, dims, str, box);
    tc::encode(tl, f.lo, 2, dims, str, box);
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
    const bool flat = route == TcRoute::Flat, kmajor = (L == 1);
    int64_t npad, nblk;
    tc_blocks(m, npad, nblk);
    const Factor f = factor_alloc(c, M, mtrans, nj, m, npad, nblk);
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
    int64_t ksplit = 1;
    {
        const int64_t items = ntiles * nblk, sms = tc::grid_sms(c);
        if (items * 2 <= sms && nk >= 4) ksplit = std::max<int64_t>(1, std::min<int64_t>(nk / 2, sms / items));
    }
    TK_REQUIRE(ntiles * nblk * ksplit < ((int64_t)1 << 31), TK_ERR_SHAPE, "ttm_tc: too many tiles");
    float* part = ksplit > 1 ? c.alloc<float>(ksplit * L * m * R) : nullptr;
    if (!c.exec) return;
    CUtensorMap tx, th, tl;
    factor_maps(c, f, M, mtrans, nj, m, npad, &th, &tl);
    if (flat) {
        tx = th;  // unused
    } else if (kmajor) {
        const uint64_t dims[2] = {(uint64_t)nj, (uint64_t)R};
        const uint64_t str[1] = {(uint64_t)nj * 4};
        const uint32_t box[2] = {tc::kChunk, tc::kRows};
        tc::encode(&tx, X.p, 2, dims, str, box);
    } else {
        const uint64_t dims[3] = {(uint64_t)L, (uint64_t)nj, (uint64_t)R};
        const uint64_t str[2] = {(uint64_t)L * 4, (uint64_t)L * nj * 4};
        uint32_t box[3] = {tc::kRows, tc::kChunk, 1};
        if (pack > 1) {  // L rows of pack consecutive r per box (L x 4 bytes: a multiple of 16)
            box[0] = (uint32_t)L;
            box[2] = (uint32_t)pack;
        }
        tc::encode(&tx, X.p, 3, dims, str, box, false);
    }
    tc::TtmArgs a;
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
    a.part = part;
    a.out_numel = L * m * R;
    a.out = out;
    a.flags = c.dflags;
    {
        ProfScope ps(c, name, 4.0 * (double)L * R * nj + 8.0 * nj * m + 4.0 * (double)L * R * m,
                     2.0 * (double)L * R * nj * m);
        if (flat) tc::ttm_tf32_run_flat(c, npad, kmajor, tx, th, tl, a);
        else tc::ttm_tf32_run_tma(c, npad, kmajor, tx, th, tl, a);
        c.counted();
        c.check_launch();
    }
    if (ksplit > 1) {
        const int64_t n = L * m * R;
        tc::splitk_sum_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, c.stream>>>(
            part, (int)ksplit, n, out);
        c.counted();
        c.check_launch();
    }
}

int tc_num_ctas(const Ctx& c, const Tens& X, int j, int64_t m, bool residual) {
    int64_t npad, nblk;
    tc_blocks(m, npad, nblk, residual);
    const int64_t L = X.left(j), R = X.right(j);
    const int64_t tiles = (L == 1) ? (R + tc::kRows - 1) / tc::kRows : R * ((L + tc::kRows - 1) / tc::kRows);
    return (int)std::min<int64_t>(tiles * nblk, tc::grid_sms(c));
}

bool ttm_tc_residual_eligible(const Tens& W, int j, int64_t m) {
    int64_t npad, nblk;
    tc_blocks(m, npad, nblk, true);
    // the residual X tile is a (128 rows x npad columns) TMA box: keep it inside the tensor
    return W.n[j] >= 32 && W.left(j) >= tc::kRows && m >= npad && m <= 65535 && tma_ok(W, j);
}

void launch_ttm_tc_residual(Ctx& c, const Tens& W, int j, const Mat& M, bool mtrans, int64_t m, const void* xref,
                            tk_dtype xrdt, void* dx, float alpha, double* partials, float xr_scale) {
    const int64_t L = W.left(j), nj = W.n[j], R = W.right(j);
    TK_REQUIRE(L > 1, TK_ERR_SHAPE, "ttm_tc: the fused residual needs a non-leading mode");
    TK_REQUIRE(xrdt == TK_F32 || xrdt == TK_BF16 || (xrdt == TK_FP8_E4M3 && !dx), TK_ERR_DTYPE,
               "ttm_tc: residual reference must be F32/BF16 (FP8: norms only)");
    int64_t npad, nblk;
    tc_blocks(m, npad, nblk, true);
    const Factor f = factor_alloc(c, M, mtrans, nj, m, npad, nblk);
    if (!c.exec) return;
    CUtensorMap tx, th, tl, txr;
    factor_maps(c, f, M, mtrans, nj, m, npad, &th, &tl);
    {
        const uint64_t dims[3] = {(uint64_t)L, (uint64_t)nj, (uint64_t)R};
        const uint64_t str[2] = {(uint64_t)L * 4, (uint64_t)L * nj * 4};
        const uint32_t box[3] = {tc::kRows, tc::kChunk, 1};
        tc::encode(&tx, W.p, 3, dims, str, box, false);
    }
    const uint64_t es = xrdt == TK_FP8_E4M3 ? 1 : (xrdt == TK_BF16 ? 2 : 4);
    {
        const uint64_t dims[3] = {(uint64_t)L, (uint64_t)m, (uint64_t)R};
        const uint64_t str[2] = {(uint64_t)L * es, (uint64_t)L * m * es};
        const uint32_t box[3] = {tc::kRows, (uint32_t)npad, 1};
        tc::encode(&txr, xref, 3, dims, str, box, false,
                   es == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                           : (es == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32));
    }
    tc::ResidArgs a;
    a.L = L;
    a.nj = nj;
    a.R = R;
    a.m = m;
    a.tiles_per_r = (L + tc::kRows - 1) / tc::kRows;
    a.ntiles = R * a.tiles_per_r;
    a.nk = (nj + tc::kChunk - 1) / tc::kChunk;
    a.nblk = nblk;
    a.out = dx;
    a.xref = xref;
    a.alpha = alpha;
    a.xr_scale = xr_scale;
    a.partials = partials;
    a.flags = c.dflags;
    ProfScope ps(c, c.background ? "xpass_tc_bg" : "xpass_tc",
                 4.0 * (double)L * R * nj + 8.0 * nj * m + (dx ? 2.0 : 1.0) * es * (double)L * R * m,
                 2.0 * (double)L * R * nj * m);
    tc::ttm_residual_run(c, npad, xrdt, dx != nullptr, tx, th, tl, txr, a);
    c.counted();
    c.check_launch();
}

}  // namespace tk
