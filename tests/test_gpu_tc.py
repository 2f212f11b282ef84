"""GPU parity of the tensor-core (tcgen05, 3xTF32) TTM path against the FP64 oracle.

Shapes are chosen so that the tensor-core kernel is the one that runs (FP32
data, 16-byte strides, contracted mode >= 32): contraction over the contiguous
mode (K-major), over the last mode and over a middle mode (MN-major), every
supported output width (16..96 columns after padding), several 128-row tiles
with ragged row and K tails.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2211_13028_gb300 import synth
from paper_2211_13028_gb300 import tucker as T
from tests.gpu_helpers import make_X, mats, rel, require_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


@pytest.mark.parametrize("s", [(5, 3), (17, 16), (49, 42), (96, 81), (33, 64)])
def test_tc_two_way_both_majors(dev, s):
    # 100 x 1665: mode 1 -> K-major (K = 100, 13 tiles + 1 ragged row), mode 2 -> MN-major (L = 100 < 128).
    g = _rng(1)
    dims = (100, 1665)
    X, xv, _ = make_X(g.standard_normal(dims), "f32", dev)
    oms = synth.sketch_factors_reuse(dims, s, seed=2, dtype="f32")
    Y = T.tucker_sketch(X, mats(oms, "f32", dev))
    assert rel(to_np(Y[0]), O.ttm(xv, oms[1].T, 1)) <= 1e-5
    assert rel(to_np(Y[1]), O.ttm(xv, oms[0].T, 0)) <= 1e-5


@pytest.mark.parametrize("dims", [(64, 70, 9), (36, 20, 300), (128, 33, 40)])
def test_tc_three_way_middle_and_last(dev, dims):
    g = _rng(3)
    X, xv, _ = make_X(g.standard_normal(dims), "f32", dev)
    s = (7, 6, 5)
    oms = synth.sketch_factors_reuse(dims, s, seed=4, dtype="f32")
    Y = T.tucker_sketch(X, mats(oms, "f32", dev))
    for n in range(3):
        ref = O.multi_ttm(xv, [(j, oms[j].T) for j in range(3) if j != n])
        assert rel(to_np(Y[n]), ref) <= 1e-5


def test_tc_core_wide_factors(dev):
    # the core multi-TTM with k_j near the largest supported width
    g = _rng(5)
    dims, k = (160, 96, 200), (96, 81, 49)
    X, xv, _ = make_X(g.standard_normal(dims), "f32", dev)
    qs = [synth.round_to(O.thin_qr(g.standard_normal((n, kk))), "f32") for n, kk in zip(dims, k)]
    G = T.tucker_core(X, mats(qs, "f32", dev))
    assert rel(to_np(G), O.multi_ttm(xv, [(j, qs[j].T) for j in range(3)])) <= 1e-5


def test_tc_full_size_bench_tensor(dev):
    # the 512^3 FP32 field of the benchmark: mode-1 and mode-3 contractions as the bench runs them
    X = synth.gaussian_bumps(512, 3, 200, 0, 1e-4, dev, "f32")
    xv = synth.from_fortran(X)
    s = (6, 7, 7)
    oms = synth.sketch_factors_reuse(X.shape, s, seed=1, dtype="f32")
    Y = T.tucker_sketch(X, mats(oms, "f32", dev))
    for n in range(3):
        ref = O.multi_ttm(xv, [(j, oms[j].T) for j in range(3) if j != n])
        assert rel(to_np(Y[n]), ref) <= 1e-5
    st, _ = T.tk_sync_status(dev)
    assert st == 0


@pytest.mark.parametrize("need_dx", [False, True])
def test_tc_fused_residual_loss_and_gradient(dev, need_dx):
    # last reconstruction step fused with the residual on tensor cores (r_3 >= 32), gradients from
    # sketches of X plus FP64 core corrections
    g = _rng(7)
    dims, rk = (96, 80, 72), (12, 10, 36)
    x = synth.round_to(g.standard_normal(dims), "f32")
    G = synth.round_to(g.standard_normal(rk), "f32")
    U = [synth.round_to(g.standard_normal((nn, k)) / np.sqrt(nn), "f32") for nn, k in zip(dims, rk)]
    Xd, Gd, Ud = synth.fortran(x, "f32", dev), synth.fortran(G, "f32", dev), mats(U, "f32", dev)
    ref_loss = O.loss(x, G, U)
    assert abs(T.tucker_loss(Xd, Gd, Ud) - ref_loss) <= 1e-5 * ref_loss
    dG, dU, dX = T.tucker_reconstruct_backward(Xd, Gd, Ud, grad_scale=0.25, need_dX=need_dx)
    ref = O.loss_grads(x, G, U)
    assert rel(to_np(dG), 0.25 * ref["dG"]) <= 1e-4
    for j in range(3):
        assert rel(to_np(dU[j]), 0.25 * ref["dU"][j]) <= 1e-4
    if need_dx:
        assert rel(to_np(dX), 0.25 * ref["dX"]) <= 1e-5
    st, _ = T.tk_sync_status(dev)
    assert st == 0


def test_tc_rel_err_fused_matches_oracle(dev):
    # rHKron-re with r_3 = 32 so the relative error uses the fused tensor-core residual
    dims, r, p = (128, 96, 112), (20, 24, 32), 6
    core = synth.decaying_core((40, 40, 40), 0.8, seed=31)
    x = synth.tucker_tensor(dims, (40, 40, 40), seed=32, noise_rel=1e-3, core=core)
    X, xv, _ = make_X(x, "f32", dev)
    s = O.subranks_reuse(r, p)[0]
    oms = synth.sketch_factors_reuse(dims, s, seed=33, dtype="f32")
    G, U, err = T.tucker_rhkron(X, r, p, mats(oms, "f32", dev))
    ref = O.rhkron(xv, r, oms)
    assert abs(err - O.rel_err(xv, ref["G"], ref["U"])) <= 1e-5
    # the error the GPU reports is the error of the factors it returned
    assert abs(err - O.rel_err(xv, to_np(G), [to_np(u) for u in U])) <= 1e-6


@pytest.mark.parametrize("dims,k", [((40, 96, 77), (40, 20, 77)), ((32, 130, 65), (32, 48, 65)),
                                    ((60, 64, 50), (60, 16, 50)), ((44, 512, 9), (44, 64, 9))])
def test_tc_short_rows_packed_tiles(dev, dims, k):
    # the first product contracts mode 2 with only L = dims[0] (32..60) rows before it: the tensor-core
    # kernel packs floor(128 / L) consecutive slabs into each 128-row tile (the last one partial)
    g = _rng(11)
    X, xv, _ = make_X(g.standard_normal(dims), "f32", dev)
    qs = [synth.round_to(O.thin_qr(g.standard_normal((n, kk))), "f32") for n, kk in zip(dims, k)]
    T.tk_profile(True, dev)
    G = T.tucker_core(X, mats(qs, "f32", dev))
    prof = T.tk_profile_read(dev)
    T.tk_profile(False, dev)
    assert "xpass_tc" in prof  # X was streamed by the tensor-core kernel
    ref = O.multi_ttm(xv, [(j, qs[j].T) for j in range(3)])
    assert rel(to_np(G), ref) <= 1e-5


@pytest.mark.parametrize("dims,k", [((500, 40, 40), (48, 40, 40)), ((40, 40, 500), (40, 40, 44)),
                                    ((48, 44, 1000), (48, 44, 64))])
def test_tc_few_tiles_split_k(dev, dims, k):
    # the first product has a long contraction (500-1000) and only 13-17 row tiles: its K chunks are
    # split over several CTAs and the partial products summed in order afterwards
    g = _rng(12)
    X, xv, _ = make_X(g.standard_normal(dims), "f32", dev)
    qs = [synth.round_to(O.thin_qr(g.standard_normal((n, kk))), "f32") for n, kk in zip(dims, k)]
    T.tk_profile(True, dev)
    G = T.tucker_core(X, mats(qs, "f32", dev))
    prof = T.tk_profile_read(dev)
    T.tk_profile(False, dev)
    assert "xpass_tc" in prof
    ref = O.multi_ttm(xv, [(j, qs[j].T) for j in range(3)])
    assert rel(to_np(G), ref) <= 1e-5
    G2 = T.tucker_core(X, mats(qs, "f32", dev))
    assert torch.equal(G, G2)  # the partial sums are added in a fixed order


@pytest.mark.parametrize("dims,k", [
    ((251, 97, 203), (251, 97, 50)),    # strided, odd slab (4-byte loads), K tail 203 = 6 chunks + 11
    ((86, 161, 151), (86, 60, 151)),    # strided, L = 86: 8-byte loads, a tile holds rows of two slabs
    ((203, 151, 97), (40, 151, 97)),    # contiguous mode of odd length (4-byte loads), ragged last tile
    ((202, 151, 97), (49, 151, 97)),    # contiguous mode, 8-byte loads
    ((7, 333, 401), (7, 40, 401)),      # rows of 7: 18 slabs per tile
    ((501, 21, 700), (501, 20, 700)),   # fewer than 32 contracted (one partial chunk)
    ((500, 21, 700), (500, 20, 700)),   # the same with 16-byte strides (TMA)
    ((150, 141, 131), (150, 120, 131)),  # two blocks of output columns
    ((9, 9, 5001), (9, 9, 100)),        # one row tile, K split over many CTAs
    ((130, 129, 128), (90, 129, 128)),  # one element past 128: last tile of 2 x 64 rows, 90 columns
])
def test_tc_any_size_and_alignment(dev, dims, k):
    # the loaders that take any L and n_j, and the short contractions, against the FP64 oracle.  Bound: the
    # split drops x_lo M_lo and rounds each low part (2^-22 of a product in all), and each FP32 sum adds
    # at most 2^-23 per addition of one chunk's products, 4 x 2^-23, and per chunk: below 2e-6
    g = _rng(21)
    X, xv, _ = make_X(g.standard_normal(dims), "f32", dev)
    qs = [np.eye(n) if n == kk else synth.round_to(O.thin_qr(g.standard_normal((n, kk))), "f32")
          for n, kk in zip(dims, k)]
    mode = [j for j in range(3) if dims[j] != k[j]][0]
    om = [synth.fmat(q, "f32", dev) for q in qs]
    T.tk_profile(True, dev)
    G = T.tucker_core(X, om)
    prof = T.tk_profile_read(dev)
    T.tk_profile(False, dev)
    assert "xpass_tc" in prof
    assert rel(to_np(G), O.ttm(xv, qs[mode].T, mode)) <= 2e-6
    st, _ = T.tk_sync_status(dev)
    assert st == 0


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("dims,k", [
    ((251, 97, 203), (251, 97, 50)),        # strided, odd slab (runs off 16 bytes), K tail 203 = 3 chunks + 11
    ((16, 1760, 203), (16, 1760, 40)),      # strided, 16-byte strides (TMA), no padding in the last tile
    ((16, 1763, 203), (16, 1763, 40)),      # the same, 48 rows in the last tile of the slab
    ((203, 151, 97), (40, 151, 97)),        # contiguous mode of odd length, ragged last tile
    ((202, 151, 97), (49, 151, 97)),        # contiguous mode, runs off 16 but on 2 bytes
    ((33, 333, 401), (33, 40, 401)),        # 3 slabs of 33 rows a tile, 29 rows of it unused; 401 = 133 x 3 + 2
    ((4, 8, 333, 101), (4, 8, 40, 101)),    # 4 slabs of 32 rows a tile (TMA)
    ((90, 333, 401), (90, 40, 401)),        # slabs of less than a tile
    ((501, 21, 700), (501, 20, 700)),       # a third of one chunk contracted
    ((150, 141, 131), (150, 120, 131)),     # two blocks of output columns
    ((9, 9, 5001), (9, 9, 100)),            # one row tile, K split over many CTAs
    ((5001, 9, 9), (100, 9, 9)),            # the same along the contiguous mode
    ((700, 130, 129), (12, 130, 129)),      # 16-column accumulators
])
def test_tc_lowp_any_size_and_alignment(dev, dims, k, dtype):
    # BF16 and FP8 data against the FP64 oracle on the stored values, in the layouts that their own kernels do
    # not take.  Bound: the factor's two TF32 parts hold it to 2^-22, and each FP32 sum adds at most 2^-23 per
    # addition of the 8 MMAs of a chunk and per chunk: below 2e-6 (BF16 of 16-byte strides: the factor's two BF16
    # parts, 2^-17)
    g = _rng(29)
    X, xv, sc = make_X(g.standard_normal(dims), dtype, dev)
    qs = [np.eye(n) if n == kk else synth.round_to(O.thin_qr(g.standard_normal((n, kk))), "f32")
          for n, kk in zip(dims, k)]
    mode = [j for j in range(len(dims)) if dims[j] != k[j]][0]
    om = [synth.fmat(q, "f32", dev) for q in qs]
    T.tk_profile(True, dev)
    G = T.tucker_core(X, om, **({"scale": sc} if dtype == "fp8" else {}))
    prof = T.tk_profile_read(dev)
    T.tk_profile(False, dev)
    assert "xpass_tc" in prof and "xpass_simt" not in prof
    own = dtype == "bf16" and int(np.prod(dims[:mode])) % 8 == 0
    assert rel(to_np(G), O.ttm(xv, qs[mode].T, mode)) <= (1e-5 if own else 2e-6)
    st, _ = T.tk_sync_status(dev)
    assert st == 0


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("dims,rk", [
    ((130, 7, 66), (9, 5, 33)),     # 910 rows: FP32 columns off 16 bytes; K = 33, two chunks; 66 = 2 x 32 + 2 columns
    ((33, 31, 129), (8, 8, 20)),    # odd rows (every dtype off 16 bytes), one column in the last block
    ((64, 48, 257), (8, 8, 64)),    # 16-byte columns in every dtype; K = 64
    ((40, 37, 90), (6, 7, 90)),     # K = 90: three chunks, 128-row tiles
    ((41, 37, 130), (5, 6, 128)),   # K = 128: four chunks, odd rows
    ((130, 11, 200), (6, 5, 129)),  # K = 129: the plain kernel's chunks, rows by 8 bytes, last block of 8 columns
    ((43, 31, 161), (5, 6, 160)),   # K = 160, odd rows
    ((64, 48, 257), (8, 8, 256)),   # K = 256, rows by TMA, one column in the last block
    ((5, 9, 300), (3, 4, 290)),     # K above 256, less than a tile of rows
    ((3, 5, 40), (2, 3, 4)),        # fewer rows than 16 bytes hold
    ((16, 16, 257), (4, 4, 5)),     # exactly one 256-row tile
    ((257, 1, 32), (4, 1, 5)),      # one row in the second tile, one full block
])
def test_fused_residual_sizes_and_alignment(dev, dims, rk, dtype):
    # the fused residual (loss, and dX where the dtype has one) at the edges of its tiles, blocks, chunks and
    # of the copies of X's unaligned columns.  X - P is formed in FP32 from a product good to ~1e-6 of
    # ||P||, and ||X - P|| ~ ||X|| here: 1e-5 of the loss and of dX (BF16 dX: its rounding, 2^-8)
    g = _rng(23)
    X, xv, sc = make_X(g.standard_normal(dims), dtype, dev)
    G = synth.round_to(g.standard_normal(rk), "f32")
    U = [synth.round_to(g.standard_normal((n, k)) / np.sqrt(n), "f32") for n, k in zip(dims, rk)]
    Gd, Ud = synth.fortran(G, "f32", dev), mats(U, "f32", dev)
    ref = O.loss(xv, G, U)
    T.tk_profile(True, dev)
    assert abs(T.tucker_loss(X, Gd, Ud, scale=sc) - ref) <= 1e-5 * ref
    prof = T.tk_profile_read(dev)
    T.tk_profile(False, dev)
    fma = dtype == "f32" and rk[2] <= 12  # a short contraction of FP32 data: FP32 FMAs
    assert ("xpass_simt" if fma else "xpass_tc") in prof and "residual" not in prof  # Xhat is never formed
    if dtype == "fp8":
        return
    norms = torch.zeros(2, dtype=torch.float64, device=dev)
    _, _, dX = T.tucker_reconstruct_backward(X, Gd, Ud, 0.5, need_dG=False, need_dU=False, norms2=norms)
    res = xv - O.reconstruct(G, U)
    assert rel(to_np(dX.float() if dtype == "bf16" else dX), res) <= (1e-5 if dtype == "f32" else 2.0 ** -8)
    assert abs(norms[0].item() - ref) <= 1e-5 * ref and abs(norms[1].item() - np.sum(xv ** 2)) <= 1e-5 * np.sum(xv ** 2)
    st, _ = T.tk_sync_status(dev)
    assert st == 0


@pytest.mark.parametrize("dims,rk,order,tc", [
    # the order of the modes' products, and those on tensor cores; the last is an expansion
    ((201, 187, 211), (20, 24, 30), (0, 2, 1), (1,)),  # odd rows, slabs after it
    ((202, 188, 260), (20, 24, 60), (0, 2, 1), (2, 1)),  # two expansions
    ((160, 130, 70, 40), (5, 6, 7, 8), (0, 3, 2, 1), (1,)),  # 4-way
    ((300, 500, 256), (10, 20, 12), (0, 2, 1), (1,)),
    ((201, 187, 211), (40, 40, 30), (1, 0, 2), (1, 0, 2)),  # no slabs after it: K = 30, last block of 19 columns
    ((202, 188, 260), (60, 56, 60), (0, 1, 2), (0, 1, 2)),  # K = 60: two chunks
    ((300, 500, 256), (30, 60, 12), (0, 1, 2), (1, 2)),
    ((160, 60, 70, 130), (16, 12, 14, 6), (0, 1, 2, 3), (3,)),
])
def test_reconstruct_expansions(dev, dims, rk, order, tc):
    # a reconstruction whose last product takes the expansion kernel (a short contraction into more columns, rows enough
    # before it).  Bound as test_tc_any_size_and_alignment, once per product
    last = order[-1]
    assert np.prod(dims[:last]) >= 32 and rk[last] <= 64 <= dims[last] and 2 * rk[last] <= dims[last]
    g = _rng(24)
    G = synth.round_to(g.standard_normal(rk), "f32")
    U = [synth.round_to(g.standard_normal((n, k)) / np.sqrt(n), "f32") for n, k in zip(dims, rk)]
    T.tk_profile(True, dev)
    Xh = T.tucker_reconstruct(synth.fortran(G, "f32", dev), mats(U, "f32", dev))
    prof = T.tk_profile_read(dev)
    T.tk_profile(False, dev)
    sh, flops = list(rk), 0.0
    for j in order:
        sh[j] = dims[j]
        flops += 2.0 * np.prod(sh) * rk[j] if j in tc else 0.0
    assert prof["ttm_tc"]["flops"] == flops, prof
    assert rel(to_np(Xh), O.reconstruct(G, U)) <= len(dims) * 2e-6
    st, _ = T.tk_sync_status(dev)
    assert st == 0


@pytest.mark.parametrize("dims,rk,order", [
    ((81, 26, 31, 27, 19), (2, 2, 9, 7, 2), (2, 3, 4, 1, 0)),  # smallest growth first: 178 us, the leading mode first 251
    ((94, 7, 189, 34), (3, 4, 80, 5), (1, 2, 3, 0)),  # 45, 63
    ((384, 160, 160), (16, 16, 16), (0, 1, 2)),  # the leading mode's scattered outputs are the smaller then
    ((160, 40, 40, 40), (4, 10, 10, 10), (1, 2, 3, 0)),  # 61, 90
])
def test_reconstruct_expands_in_the_faster_order(dev, dims, rk, order):
    g = _rng(25)
    G = synth.round_to(g.standard_normal(rk), "f32")
    U = [synth.round_to(g.standard_normal((n, k)) / np.sqrt(n), "f32") for n, k in zip(dims, rk)]
    T.tk_profile(True, dev)
    Xh = T.tucker_reconstruct(synth.fortran(G, "f32", dev), mats(U, "f32", dev))
    prof = T.tk_profile_read(dev)
    T.tk_profile(False, dev)
    flops, sh = 0.0, list(rk)
    for j in order:
        sh[j] = dims[j]
        flops += 2.0 * np.prod(sh) * rk[j]
    assert sum(v["flops"] for v in prof.values()) == flops, prof
    assert rel(to_np(Xh), O.reconstruct(G, U)) <= len(dims) * 2e-6


@pytest.mark.parametrize("dims,r,dtype,want", [
    # X's pass to (r_1, all else): a product of few rows and steps takes one SIMT launch, not a split and a tensor-core one
    ((2512, 48), (5, 34), "f32", "xpass_simt"),  # 15 us against 16 in two launches, and their 7 on the host
    ((889, 16, 21), (3, 4, 4), "f32", "xpass_simt"),  # 12, 16
    ((9001, 333), (20, 9), "f32", "xpass_tc"),  # long contractions: 78, 10
    ((333, 9001), (20, 9), "f32", "xpass_tc"),
    ((413, 35, 275), (36, 4, 4), "f32", "xpass_tc"),
    ((1030, 97), (8, 4), "fp8", "xpass_simt"),
    ((203, 690, 70), (20, 4, 4), "fp8", "xpass_tc"),
])
def test_first_product_takes_the_faster_kernel(dev, dims, r, dtype, want):
    g = _rng(41)
    X, xv, xs = make_X(g.standard_normal(dims), dtype, dev)
    U = [synth.round_to(g.standard_normal((n, k)) / np.sqrt(n), "f32") for n, k in zip(dims, r)]
    T.tk_profile(True, dev)
    G = T.tucker_core(X, mats(U, "f32", dev), scale=xs)
    prof = T.tk_profile_read(dev)
    T.tk_profile(False, dev)
    assert [k for k in ("xpass_tc", "xpass_simt") if k in prof] == [want], prof
    ref = xv
    for j, u in enumerate(U):
        ref = O.ttm(ref, u.T, j)
    assert rel(to_np(G), ref) <= len(dims) * 2e-6

@pytest.mark.parametrize("rows", [4096, 4099])
@pytest.mark.parametrize("K", [1, 3, 4, 5, 8, 9, 12, 13, 16, 24, 32])
def test_residual_of_short_contractions_keeps_fp32_digits(dev, K, rows):
    # dX of X = 0 is -P, P = W U^T with W = u g^T rounded once per entry, so the product alone is seen.  Up to 12 terms
    # it is summed by FMAs that round to nearest: no bias (a truncating sum has about -2^-25 = 3e-8), and an error
    # of at most sqrt(K + 1) 2^-25.  Above, two accumulators take half of the 8-term steps each: at most
    # two truncations by 2^-23 of half the sum, 2^-23 = 1.2e-7
    g = torch.Generator(device=dev)
    g.manual_seed(K)
    m = 1000
    u, w, U = (torch.randn(b, a, generator=g, device=dev).t() for a, b in ((rows, 1), (1, K), (m, K)))
    ref = (u * w).double() @ U.double().t()
    X = torch.zeros(m, rows, device=dev).t()
    norms = torch.zeros(2, dtype=torch.float64, device=dev)
    _, _, dX = T.tucker_reconstruct_backward(X, w, [u, U], 0.5, need_dG=False, need_dU=False, norms2=norms)
    err = -dX.double() - ref
    if K <= 12:
        assert float((err * ref.sign()).sum() / ref.abs().sum()) >= -5e-9
        assert float(err.norm() / ref.norm()) <= (K + 1) ** 0.5 * 2.0 ** -25
    else:
        assert float(err.norm() / ref.norm()) <= 2.0 ** -23
    assert abs(float(norms[0]) - float((ref ** 2).sum())) <= 1e-6 * float((ref ** 2).sum()) and float(norms[1]) == 0.0
