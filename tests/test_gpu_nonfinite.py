"""Infinities, NaN and the largest finite values: a product contains what FP32 arithmetic gives, in the rows that meet
them only, on every kernel that takes the TTMs of FP32 data and of odd BF16 / FP8 layouts."""
import numpy as np
import pytest
import torch

from paper_2211_13028_gb300 import tucker as T
from tests.gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu

FLT_MAX = 3.4028234e38


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _colmajor(rows, cols, dev, seed, dtype=torch.float32):
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    return torch.randn(cols, rows, generator=g, device=dev).to(dtype).t()


def _same(got, ref, tol):
    """Infinities (with their signs) and NaN in the same places, the other entries close."""
    got = got.double()
    assert torch.equal(torch.isnan(got), torch.isnan(ref))
    assert torch.equal(torch.isinf(got), torch.isinf(ref))
    assert torch.equal(got[torch.isinf(ref)], ref[torch.isinf(ref)])
    ok = torch.isfinite(ref)
    # the rows with the largest values aside, whose sums are on another scale
    small = ok & (ref.abs() < 1e30)
    assert float((got - ref)[small].norm()) <= tol * float(ref[small].norm())
    large = ok & ~small
    if bool(large.any()):
        assert float(((got - ref)[large] / FLT_MAX).norm()) <= tol * float((ref[large] / FLT_MAX).norm())


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float8_e4m3fn])
@pytest.mark.parametrize("n1,n2,m", [
    (4096, 128, 6),    # the sketch widths, 16-byte strides
    (4096, 128, 20),   # 16-byte strides
    (4099, 203, 50),   # any stride
    (4098, 700, 90),   # two or more blocks or slices
    (40000, 21, 10),   # fewer than 32 contracted
    (130, 9000, 12),   # few rows, K split over CTAs
])
def test_products_keep_infinities_nan_and_large_values(dev, n1, n2, m, dtype):
    x = _colmajor(n1, n2, dev, 1, dtype)
    vals = [float("nan")] if dtype == torch.float8_e4m3fn else [float("inf"), -float("inf"), float("nan")]
    if dtype == torch.float32:
        vals += [FLT_MAX, -3.4026e38]
    for i, v in enumerate(vals):
        x[(17 + 31 * i) % n1, (5 + 7 * i) % n2] = v
    om = [_colmajor(n1, m, dev, 2) * 0.01, _colmajor(n2, m, dev, 3) * 0.01]
    xd = x.double()
    Y = T.tucker_sketch(x, om)
    own = dtype != torch.float32 and n1 % 16 == 0  # the kernels that multiply 16- and 8-bit data as they are
    if not own:
        _same(Y[0], xd @ om[1].double(), 2e-6)
    # along the contiguous mode every column of X that holds one of the values is a row of the product
    if not (dtype != torch.float32 and n1 % (8 if dtype == torch.bfloat16 else 16) == 0):
        _same(Y[1], om[0].double().t() @ xd, 2e-6)
    st, _ = T.tk_sync_status(dev)
    assert st == 0


@pytest.mark.parametrize("where", ["x", "factor"])
def test_infinite_factor_or_core(dev, where):
    # 200 x 300 from 30 x 20: the products of a reconstruction, with an infinity in the core or in a factor
    G, U = _colmajor(30, 20, dev, 1), [_colmajor(2000, 30, dev, 2), _colmajor(3000, 20, dev, 3)]
    if where == "x":
        G[3, 4] = float("inf")
    else:
        U[1][11, 7] = -float("inf")
    w = U[0].double() @ G.double()
    _same(T.tucker_reconstruct(G, U), w @ U[1].double().t(), 4e-6)


@pytest.mark.parametrize("K", [8, 24, 60, 100, 200])
@pytest.mark.parametrize("n1", [4096, 1001])
def test_residual_of_infinite_data(dev, n1, K):
    # the loss is infinite with an infinity in X, a NaN with a NaN; dX holds it in its own place only, and a
    # product that is infinite in one row of P leaves the others alone
    G, U = _colmajor(1, K, dev, 1), [_colmajor(n1, 1, dev, 2), _colmajor(500, K, dev, 3)]
    x = _colmajor(n1, 500, dev, 4)
    x[7, 9] = float("inf")
    assert T.tucker_loss(x, G, U) == float("inf")
    _, _, dX = T.tucker_reconstruct_backward(x, G, U, 0.5, need_dG=False, need_dU=False)
    ref = x.double() - (U[0] * G).double() @ U[1].double().t()
    _same(dX, ref, 2e-6)
    x[7, 9] = 1.0
    U[0][3, 0] = float("inf")
    _, _, dX = T.tucker_reconstruct_backward(x, G, U, 0.5, need_dG=False, need_dU=False)
    _same(dX, x.double() - (U[0] * G).double() @ U[1].double().t(), 2e-6)
    x[8, 1] = float("nan")
    assert np.isnan(T.tucker_loss(x, G, U))
