"""The workloads this library's speed is judged on, each one pass through its
public entry points.

A case names an entry point (``op``), the tensor's dims, the data type it is
stored in and the ranks.  Tensors are column-major on the GPU, as every entry
point takes them.  Two kinds of data are used:

* ``field``: a smooth field (200 anisotropic Gaussian bumps plus noise), the
  character of the simulation data that Tucker compression is used on; for the
  single contractions, whose results depend smoothly on it.
* ``tucker``: a core of decaying entries (three-way: mostly a decaying
  superdiagonal, as in the paper's accuracy experiment) times random orthonormal
  factors, plus noise; for whole decompositions and truncations, where the singular values
  must be apart for single columns of U to be determined by the data.

``listed`` holds the configurations the repository itself is run on (64^3 FP64,
512^3 FP32, 160^4 FP32, 1024^3 BF16, 256^3 for the gradient) and ragged sizes
between them; ``draw`` covers the same operations over the whole range of
sizes, aligned and not.
"""
from __future__ import annotations

import math
from typing import Dict, List, Sequence

import torch

from paper_2211_13028_gb300 import tucker as T

DEV = "cuda"
_TORCH = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.float8_e4m3fn}
_BYTES = {"f64": 8, "f32": 4, "bf16": 2, "fp8": 1}


def _ints(text: str) -> List[int]:
    return [int(v) for v in str(text).split("x")]


def _text(values: Sequence[int]) -> str:
    return "x".join(str(int(v)) for v in values)


def _case(op, dims, dtype, ranks, **more) -> dict:
    return dict(op=op, dims=_text(dims), dtype=dtype, ranks=_text(ranks), **more)


def listed() -> List[dict]:
    return [
        # the smallest whole call: one decomposition of a 64^3 double-precision tensor; latency and launches
        dict(_case("rhkron", (64, 64, 64), "f64", (8, 8, 8), p=4), name="rhkron_f64_64"),
        # the thin QR of the three sketches of a 512^3 field, as each rank of the sharded form calls it
        dict(_case("orth", (512, 512, 512), "f32", (32, 32, 32), p=8), name="orth_f32_512"),
        # the truncation of a 49 x 42 x 42 core, the step after the core of a 512^3 field (sharded form)
        dict(_case("sthosvd", (512, 512, 512), "f32", (32, 32, 32), p=8), name="sthosvd_f32_512"),
        # decompression of a mid-sized tensor of ragged dims
        dict(_case("reconstruct", (203, 187, 211), "f32", (20, 24, 18)), name="reconstruct_f32_ragged"),
        # one gradient step of the fit by descent
        dict(_case("backward", (256, 256, 256), "f32", (16, 16, 16)), name="backward_f32_256"),
        # the Kronecker sketches of a 512^3 field (first step of rHKron-re)
        dict(_case("sketch", (512, 512, 512), "f32", (32, 32, 32), p=8), name="sketch_f32_512"),
        # the core multi-TTM of a 512^3 field (third step)
        dict(_case("core", (512, 512, 512), "f32", (32, 32, 32), p=8), name="core_f32_512"),
        # the same step on a grid whose dims are no multiples of anything
        dict(_case("core", (413, 350, 275), "f32", (24, 20, 28), p=6), name="core_f32_ragged"),
        # one decomposition of a 512^3 tensor with its relative error
        dict(_case("rhkron", (512, 512, 512), "f32", (32, 32, 32), p=8), name="rhkron_f32_512"),
        # four-way data, uneven ranks, last mode first
        dict(_case("rsthkron", (160, 160, 160, 160), "f32", (10, 20, 30, 40), p=6, last_first=True),
             name="rsthkron_f32_160x4"),
        # a tensor stored in 16 bits, four times the size of the others
        dict(_case("rhkron", (1024, 1024, 1024), "bf16", (64, 64, 64), p=16), name="rhkron_bf16_1024"),
        # the sketches of a tensor stored in 8 bits with one scale
        dict(_case("sketch", (768, 768, 768), "fp8", (64, 64, 64), p=16), name="sketch_fp8_768"),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    op = rng.choice(["sketch", "sketch", "core", "core", "rhkron", "rhkron", "rsthkron", "reconstruct", "backward",
                     "orth", "sthosvd"])
    dtype = "f32"
    if op in ("sketch", "core", "rhkron"):
        dtype = rng.choice(["f32", "f32", "f32", "f64", "bf16", "fp8"])
    ways = 4 if rng.random() < 0.2 else 3
    lo, hi = {"f64": (48, 200), "f32": (64, 512), "bf16": (96, 800), "fp8": (96, 640)}[dtype]
    if ways == 4:
        lo, hi = 24, (48 if dtype == "f64" else 128)
    dims = [_log_int(rng, lo, hi) for _ in range(ways)]
    if rng.random() < 0.4:  # grids are often multiples of a power of two
        dims = [max(16, n // 16 * 16) for n in dims]
    # ranks of one magnitude, none above a third of its mode; 8-bit data holds only the leading directions
    top = min(48 if ways == 3 else 20, min(dims) // 3, 12 if dtype == "fp8" and op == "rhkron" else 48)
    base = _log_int(rng, 5, max(6, top))
    ranks = [max(3, int(base * rng.uniform(0.8, 1.0))) for n in dims]
    if op in ("reconstruct", "backward"):
        return _case(op, dims, dtype, ranks)
    more = dict(p=rng.choice([4, 5, 6, 8]))
    if op == "rsthkron":
        more["last_first"] = rng.random() < 0.5
    return _case(op, dims, dtype, ranks, **more)


# ------------------------------------------------------------------ inputs

def _colmajor(rev: torch.Tensor, dtype) -> torch.Tensor:
    """A tensor with reversed dims (last mode first, C order) as the column-major tensor it holds."""
    t = rev.to(dtype).contiguous()
    return t.permute(*reversed(range(t.dim())))


def _gen(seed: int) -> torch.Generator:
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62) + 17)
    return g


def _randn(g, *shape, dtype=torch.float32) -> torch.Tensor:
    return torch.randn(*shape, generator=g, device=DEV, dtype=dtype)


def _orthonormal(g, n: int, k: int, dtype=torch.float32) -> torch.Tensor:
    return torch.linalg.qr(_randn(g, n, k, dtype=torch.float64))[0].to(dtype)


def _colmajor_matrix(a: torch.Tensor) -> torch.Tensor:
    return a.t().contiguous().t()


def _expand(x: torch.Tensor, mats: Sequence[torch.Tensor]) -> torch.Tensor:
    """x (dims reversed) times mats[j] (rows x cols) along mode j, whose axis is d-1-j."""
    d = x.dim()
    for j, u in enumerate(mats):
        ax = d - 1 - j
        x = torch.movedim(torch.tensordot(x, u, dims=([ax], [1])), -1, ax)
    return x


def _field(g, dims: Sequence[int], noise: float) -> torch.Tensor:
    bumps = 200
    amp = torch.rand(bumps, generator=g, device=DEV) + 0.5
    facs = []
    for n in dims:
        c = torch.rand(bumps, generator=g, device=DEV) * n
        s = n / 64.0 + torch.rand(bumps, generator=g, device=DEV) * (n / 8.0 - n / 64.0)
        i = torch.arange(n, device=DEV, dtype=torch.float32)[:, None]
        facs.append(torch.exp(-((i - c) ** 2) / (2 * s * s)))
    kr = facs[-1] * amp
    for f in reversed(facs[1:-1]):
        kr = (kr[:, None, :] * f[None, :, :]).reshape(-1, bumps)
    x = (kr @ facs[0].t()).reshape(*reversed(list(dims)))
    e = _randn(g, *x.shape)
    return x.add_(e, alpha=float(noise * x.norm() / e.norm()))


def _decaying(g, ranks: Sequence[int], last: float = 0.05) -> torch.Tensor:
    """A dense core whose entries decay geometrically, to ``last`` along each mode."""
    core = _randn(g, *reversed(list(ranks)))
    for ax in range(core.dim()):
        r = core.shape[ax]
        w = last ** (torch.arange(r, device=DEV, dtype=torch.float32) / r)
        core = core * w.reshape([-1 if a == ax else 1 for a in range(core.dim())])
    return core


def _spread_core(g, ranks: Sequence[int]) -> torch.Tensor:
    """A core whose unfoldings have singular values apart from one another.  Three-way: a superdiagonal
    that decays geometrically to a twentieth, plus a dense part of a twentieth of its norm.  Four-way: dense
    with a mild decay; its unfoldings have so many columns that their rows are nearly orthogonal."""
    if len(ranks) > 3:
        return _decaying(g, ranks, 0.2)
    k = min(ranks)
    core = _decaying(g, ranks)
    diag = 0.05 ** (torch.arange(k, device=DEV, dtype=torch.float32) / k)
    core = core * (0.05 * diag.norm() / core.norm())
    i = torch.arange(k, device=DEV)
    core[(i,) * len(ranks)] += diag
    return core


def _tucker(g, dims: Sequence[int], ranks: Sequence[int], noise: float) -> torch.Tensor:
    x = _expand(_spread_core(g, ranks), [_orthonormal(g, n, k) for n, k in zip(dims, ranks)]).contiguous()
    e = _randn(g, *x.shape)
    return x.add_(e, alpha=float(noise * x.norm() / e.norm()))


def _store(x: torch.Tensor, dtype: str):
    """(column-major tensor in the storage type, scale): FP8 holds x * scale with the largest value at 448."""
    scale = 1.0
    if dtype == "fp8":
        scale = float(448.0 / x.abs().max())
        x = x * scale
    return _colmajor(x, _TORCH[dtype]), scale


def _widths(dims, ranks, p):
    s, w = T.tucker_subranks_reuse(ranks, p)
    return s, [min(n, k) for n, k in zip(dims, w)]


def _order(case: dict, d: int):
    return list(reversed(range(d))) if case.get("last_first") else list(range(d))


def prepare(case: dict, seed: int) -> Dict:
    g = _gen(seed)
    dims, ranks, op, dtype = _ints(case["dims"]), _ints(case["ranks"]), case["op"], case["dtype"]
    d = len(dims)
    fac = torch.float64 if dtype == "f64" else torch.float32
    st: Dict = dict(op=op, ranks=ranks, p=case.get("p", 0), scale=1.0)
    if op == "reconstruct":
        st["G"] = _colmajor(_decaying(g, ranks), fac)
        st["U"] = [_colmajor_matrix(_orthonormal(g, n, k, fac)) for n, k in zip(dims, ranks)]
        return st
    if op == "backward":
        # a fit under way: the parameters are a few percent from the tensor's own
        core = _decaying(g, ranks)
        us = [_orthonormal(g, n, k) for n, k in zip(dims, ranks)]
        x = _expand(core, us).contiguous()
        e = _randn(g, *x.shape)
        st["X"] = _colmajor(x.add_(e, alpha=float(1e-2 * x.norm() / e.norm())), torch.float32)
        st["G"] = _colmajor(core + _randn(g, *core.shape) * (0.05 * core.norm() / math.sqrt(core.numel())),
                            torch.float32)
        st["U"] = [_colmajor_matrix(u + _randn(g, *u.shape) * (0.05 / math.sqrt(u.shape[0]))) for u in us]
        return st
    s, k = _widths(dims, ranks, st["p"])
    if op == "orth":
        # sketches of decaying data: each column a mix of the leading directions, as X x Omega gives them
        st["Y"] = []
        for n in range(d):
            rows, cols = dims[n], math.prod(s) // s[n]
            a = _randn(g, rows, min(rows, cols + 16))
            w = 0.85 ** torch.arange(a.shape[1], device=DEV, dtype=torch.float32)
            y = (a * w) @ _randn(g, a.shape[1], cols) + 1e-2 * _randn(g, rows, cols)
            perm = [s[j] for j in reversed(range(d)) if j != n]
            y = torch.movedim(y.reshape(rows, *perm), 0, d - 1 - n)
            st["Y"].append(_colmajor(y, torch.float32))
        return st
    if op == "sthosvd":
        st["G"] = _colmajor(_spread_core(g, k), torch.float32)
        st["Q"] = [_colmajor_matrix(_orthonormal(g, n, kk)) for n, kk in zip(dims, k)]
        return st
    if op in ("sketch", "core"):
        x = _field(g, dims, 1e-4)
    else:
        x = _tucker(g, dims, [min(n, r + 8) for n, r in zip(dims, ranks)], 1e-3)
    st["X"], st["scale"] = _store(x, dtype)
    del x
    if op == "core":
        st["Q"] = [_colmajor_matrix(_orthonormal(g, n, kk, fac)) for n, kk in zip(dims, k)]
    elif op == "rsthkron":
        st["order"] = _order(case, d)
        S, w = T.tucker_subranks_matrix(ranks, st["p"], st["order"])
        kd = [min(n, ww) for n, ww in zip(dims, w)]
        keys, shapes, _ = T.rsthkron_factor_plan(dims, S, kd, st["order"])
        st["Omega"] = {key: _colmajor_matrix(_randn(g, *sh, dtype=fac)) for key, sh in zip(keys, shapes)}
    else:
        st["Omega"] = [_colmajor_matrix(_randn(g, n, sj, dtype=fac)) for n, sj in zip(dims, s)]
    return st


# ------------------------------------------------------------------ one pass

def run(st: Dict):
    op = st["op"]
    if op == "sketch":
        return T.tucker_sketch(st["X"], st["Omega"], scale=st["scale"])
    if op == "core":
        return T.tucker_core(st["X"], st["Q"], scale=st["scale"])
    if op == "orth":
        return T.tucker_orth_sketches(st["Y"])
    if op == "sthosvd":
        G, U = T.tucker_sthosvd(st["G"], st["Q"], st["ranks"])
        return {"G": G, "U": U}
    if op == "rhkron":
        G, U, err = T.tucker_rhkron(st["X"], st["ranks"], st["p"], st["Omega"], scale=st["scale"])
        return {"G": G, "U": U, "err": err}
    if op == "rsthkron":
        G, U, err = T.tucker_rsthkron(st["X"], st["ranks"], st["p"], st["Omega"], order=st["order"])
        return {"G": G, "U": U, "err": err}
    if op == "reconstruct":
        return T.tucker_reconstruct(st["G"], st["U"])
    dG, dU, dX = T.tucker_reconstruct_backward(st["X"], st["G"], st["U"], 0.5)
    return {"dG": dG, "dU": dU, "dX": dX}


# ------------------------------------------------------------------ the same in 64 bits, by plain torch

def _ttm64(x: torch.Tensor, m: torch.Tensor, j: int) -> torch.Tensor:
    """x (dims in order) times m^T along mode j, m: n_j x cols."""
    return torch.movedim(torch.tensordot(x, m.double(), dims=([j], [0])), -1, j)


def _unfold64(x: torch.Tensor, j: int) -> torch.Tensor:
    """The mode-j unfolding, columns in column-major order of the other modes."""
    y = torch.movedim(x, j, 0)
    return y.permute(0, *reversed(range(1, y.dim()))).reshape(x.shape[j], -1)


def _qr64(y: torch.Tensor) -> torch.Tensor:
    if y.shape[1] >= y.shape[0]:
        return torch.eye(y.shape[0], device=y.device, dtype=torch.float64)
    q, r = torch.linalg.qr(y)
    return q * torch.where(torch.diagonal(r) < 0, -1.0, 1.0)


def _sthosvd64(g: torch.Tensor, qs, ranks, order):
    d = g.dim()
    us: List = [None] * d
    for j in order:
        v = torch.linalg.svd(_unfold64(g, j), full_matrices=False)[0][:, :ranks[j]]
        us[j] = qs[j].double() @ v
        g = _ttm64(g, v, j)
    for j in range(d):  # sign gauge: each column's entry of largest magnitude is positive
        at = us[j].abs().argmax(dim=0)
        sg = torch.where(us[j].gather(0, at[None, :])[0] < 0, -1.0, 1.0).double()
        us[j] = us[j] * sg
        g = g * sg.reshape([-1 if a == j else 1 for a in range(d)])
    return g, us


def _error64(x: torch.Tensor, g: torch.Tensor, us) -> float:
    xh = g
    for j, u in enumerate(us):
        xh = _ttm64(xh, u.t(), j)
    return float((x - xh).norm() / x.norm())


def exact(case: dict, seed: int):
    st = prepare(case, seed)
    op, ranks = st["op"], st["ranks"]
    if op == "orth":
        return [_qr64(_unfold64(y.double(), n)) for n, y in enumerate(st["Y"])]
    if op == "sthosvd":
        g, us = _sthosvd64(st["G"].double(), st["Q"], ranks, list(range(len(ranks))))
        return {"G": g, "U": us}
    if op == "reconstruct":
        x = st["G"].double()
        for j, u in enumerate(st["U"]):
            x = _ttm64(x, u.t(), j)
        return x
    x = st["X"].double() / st["scale"]
    st["X"] = None
    d = x.dim()
    if op == "sketch":
        out = []
        for n in range(d):
            y = x
            for j in reversed(range(d)):
                if j != n:
                    y = _ttm64(y, st["Omega"][j], j)
            out.append(y)
        return out
    if op == "core":
        for j in reversed(range(d)):
            x = _ttm64(x, st["Q"][j], j)
        return x
    if op == "backward":
        g, us = st["G"].double(), [u.double() for u in st["U"]]
        xh = g
        for j, u in enumerate(us):
            xh = _ttm64(xh, u.t(), j)
        res = x - xh
        dg, du = res, []
        for n in range(d):
            y = res
            for j in reversed(range(d)):
                if j != n:
                    y = _ttm64(y, us[j], j)
            du.append(-(_unfold64(y, n) @ _unfold64(g, n).t()))
            if n == 0:
                dg = -_ttm64(y, us[0], 0)
        return {"dG": dg, "dU": du, "dX": res}
    if op == "rhkron":
        qs = []
        for n in range(d):
            y = x
            for j in reversed(range(d)):
                if j != n:
                    y = _ttm64(y, st["Omega"][j], j)
            qs.append(_qr64(_unfold64(y, n)))
        core, order = x, list(range(d))
        for j in reversed(range(d)):
            core = _ttm64(core, qs[j], j)
    else:
        core, order, qs = x, st["order"], [None] * d
        for j in order:
            y = core
            for i in reversed(range(d)):
                if i != j:
                    y = _ttm64(y, st["Omega"][(j, i)], i)
            qs[j] = _qr64(_unfold64(y, j))
            core = _ttm64(core, qs[j], j)
    g, us = _sthosvd64(core, qs, ranks, order)
    return {"G": g, "U": us, "err": _error64(x, g, us)}


# ------------------------------------------------------------------ what a pass cannot do without

def work(case: dict) -> Dict[str, float]:
    dims, ranks, op, dtype = _ints(case["dims"]), _ints(case["ranks"]), case["op"], case["dtype"]
    d, numel, e = len(dims), math.prod(dims), _BYTES[case["dtype"]]
    acc = 8 if dtype == "f64" else 4
    s, k = _widths(dims, ranks, case.get("p", 0))
    factors = sum(n * r for n, r in zip(dims, ranks)) * acc + math.prod(ranks) * acc

    def chain(ms):  # flops of a multi-TTM over all modes, cheapest order
        cur, total = numel, 0.0
        for n, m in sorted(zip(dims, ms), key=lambda t: t[1] / t[0]):
            total += 2.0 * cur * m
            cur = cur // n * m
        return total

    if op == "sketch":
        outs = sum(n * math.prod(s) // s[j] for j, n in enumerate(dims))
        return {"bytes": numel * e + outs * acc + sum(n * v for n, v in zip(dims, s)) * acc,
                "flops": 2.0 * numel * (s[0] + s[-1])}
    if op == "core":
        return {"bytes": numel * e + (sum(n * v for n, v in zip(dims, k)) + math.prod(k)) * acc, "flops": chain(k)}
    if op == "orth":
        cols = [math.prod(s) // v for v in s]
        return {"bytes": sum(n * c * 4 + n * min(n, c) * 8 for n, c in zip(dims, cols)),
                "flops": sum(4.0 * n * min(n, c) ** 2 for n, c in zip(dims, cols))}
    if op == "sthosvd":
        return {"bytes": (math.prod(k) + sum(n * v for n, v in zip(dims, k))) * 4 + factors,
                "flops": sum(2.0 * math.prod(k) * v + 2.0 * n * v * r for n, v, r in zip(dims, k, ranks))}
    if op == "reconstruct":
        return {"bytes": numel * acc + factors, "flops": chain(ranks)}
    if op == "backward":
        return {"bytes": 2.0 * numel * e + 2 * factors, "flops": 3.0 * chain(ranks)}
    return {"bytes": numel * e + factors + sum(n * v for n, v in zip(dims, s)) * acc,
            "flops": 2.0 * numel * (s[0] + s[-1]) + chain(k) + chain(ranks)}


def tolerance(case: dict):
    """About four times the largest error against ``exact`` seen over the declared ranges (three seeds of
    each listed case, some hundred drawn ones)."""
    op, dtype = case["op"], case["dtype"]
    if op == "orth":  # double-float arithmetic (about 48 bits) on FP32 sketches
        return {"rel": 5e-12, "max": 2e-10}
    if op == "sthosvd":
        return {"rel": 2e-6, "max": 5e-5}
    if op in ("rhkron", "rsthkron"):  # single columns of U follow the rounding over the singular values' gaps
        if dtype == "f64":
            return {"rel": 1e-12, "max": 1e-11}
        return {"rel": 1e-4, "max": 2e-3} if len(_ints(case["dims"])) == 3 else {"rel": 1e-3, "max": 2e-2}
    if dtype == "f64":
        return {"rel": 1e-14, "max": 1e-13}
    if op == "backward":  # differences of nearly equal FP32 products
        return {"rel": 2e-4, "max": 2e-3}
    return {"rel": 1e-5, "max": 1e-4}
