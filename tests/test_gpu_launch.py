"""Launches that overlap must not cost more than they save."""
import pytest
import torch

from paper_2211_13028_gb300 import synth
from paper_2211_13028_gb300 import tucker as T
from tests.gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


@pytest.mark.parametrize("dims,s", [((144, 16, 640), (20, 9, 4)), ((32, 96, 592), (12, 20, 6))])
def test_fp64_products_of_few_blocks_are_spread_over_the_sms(dev, dims, s):
    # products of 5 to 36 blocks, bound by the FP64 pipes of the SMs they run on, after one that fills every SM:
    # the call takes its kernels' own times (recorded one after another) and launch gaps, a fifth at most,
    # not the multiple that blocks sharing an SM take
    g = torch.Generator(device=dev)
    g.manual_seed(3)
    X = synth.fortran(torch.randn(dims, generator=g, device=dev, dtype=torch.float64).cpu().numpy(), "f64", dev)
    om = [torch.randn(k, n, generator=g, device=dev, dtype=torch.float64).t() for n, k in zip(dims, s)]
    T.tucker_sketch(X, om)
    T.tk_profile(True, dev)
    T.tucker_sketch(X, om)
    alone = sum(e["end_us"] - e["start_us"] for e in T.tk_profile_trace(dev))
    T.tk_profile(False, dev)
    best = float("inf")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        T.tucker_sketch(X, om)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    assert best <= 1.2 * alone, (best, alone)
