"""The solver's work as its users call it, and the ranges it comes in.

Matrices are symmetric positive definite with a chosen spectrum and dense,
incoherent eigenvectors: A = Q diag(lambda) Q^T, Q = D0 H D1 H, with random signs
D0, D1 and the orthogonal Hartley transform H (H_jk = cas(2 pi j k / n) / sqrt n).
H diag(lambda) H has a closed form, so A costs two passes of FFTs at any n, odd
and prime sizes included.  Spectra: "log", log-spaced in [1, kappa]; "gram", the
square Gram matrix M M^T / n (its limiting law, lambda = s^2 with s from the
semicircle on [-2, 2]) plus a 1e-2 ridge.
"""
import math

import torch

from paper_2601_14466_gb300 import autograd, jmg

DEV = "cuda"


def listed():
    return [
        # many small independent systems in one call (per-cell or per-site solves)
        {"name": "batched_n48", "kind": "batched", "n": 48, "nrhs": 1, "batch": 1000, "dtype": "f64"},
        # one latency-bound small system, solved and certified in one kernel
        {"name": "onekernel_n1024", "kind": "mixed", "n": 1024, "nrhs": 1, "prec": "fp32",
         "words": 1, "spectrum": "log", "kappa": 10.0},
        # the smallest plain FP64 solve: one system, one right-hand side
        {"name": "posv_fp64_n1024", "kind": "posv", "n": 1024, "nrhs": 1, "dtype": "f64",
         "kappa": 10.0},
        # a Gaussian-process style step on a ragged size: factor, solve, log det
        {"name": "factor_fp64_n5000", "kind": "factor", "n": 5000, "nrhs": 16, "dtype": "f64",
         "kappa": 1e4},
        # the plain FP64 solve with many right-hand sides
        {"name": "posv_fp64_n16384", "kind": "posv", "n": 16384, "nrhs": 64, "dtype": "f64",
         "kappa": 1e6},
        # new right-hand sides against a factor that the program keeps
        {"name": "potrs_fp64_n12288", "kind": "potrs", "n": 12288, "nrhs": 8, "dtype": "f64"},
        # float32 data: factor, solve, log det
        {"name": "factor_fp32_n8192", "kind": "factor", "n": 8192, "nrhs": 16, "dtype": "f32",
         "kappa": 100.0},
        # mixed precision at three sizes and factor types, to a certified FP64 residual
        {"name": "mixed_fp16x2_n16384", "kind": "mixed", "n": 16384, "nrhs": 64, "prec": "fp16",
         "words": 2, "spectrum": "log", "kappa": 1e3},
        {"name": "mixed_bf16_n32768", "kind": "mixed", "n": 32768, "nrhs": 16, "prec": "bf16",
         "words": 1, "spectrum": "log", "kappa": 100.0},
        {"name": "mixed_fp8_n65536", "kind": "mixed", "n": 65536, "nrhs": 32, "prec": "fp8",
         "words": 1, "spectrum": "gram", "kappa": 400.0},
        # a differentiable solve inside a training step: forward and backward
        {"name": "grad_fp64_n3000", "kind": "grad", "n": 3000, "nrhs": 4, "prec": "fp64",
         "words": 1, "kappa": 10.0},
        {"name": "grad_bf16x2_n8192", "kind": "grad", "n": 8192, "nrhs": 16, "prec": "bf16",
         "words": 2, "kappa": 10.0},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["batched", "onekernel", "posv", "factor", "factor32", "potrs", "mixed",
                       "mixed", "mixed8", "grad"])
    kappa = 10.0 ** rng.uniform(1.0, 4.0)
    if kind == "batched":
        return {"kind": "batched", "n": rng.randint(3, 128), "nrhs": _log_int(rng, 1, 32),
                "batch": _log_int(rng, 16, 2048), "dtype": rng.choice(["f64", "f32"])}
    if kind == "onekernel":
        return {"kind": "mixed", "n": _log_int(rng, 64, 2048), "nrhs": _log_int(rng, 1, 64),
                "prec": "fp32", "words": 1, "spectrum": "log", "kappa": min(kappa, 1e3)}
    if kind == "posv":
        return {"kind": "posv", "n": _log_int(rng, 200, 14000), "nrhs": _log_int(rng, 1, 100),
                "dtype": rng.choice(["f64", "f64", "f32"]), "kappa": min(kappa, 1e3)}
    if kind == "factor":
        return {"kind": "factor", "n": _log_int(rng, 300, 12000), "nrhs": _log_int(rng, 1, 64),
                "dtype": "f64", "kappa": kappa}
    if kind == "factor32":
        return {"kind": "factor", "n": _log_int(rng, 300, 16384), "nrhs": _log_int(rng, 1, 64),
                "dtype": "f32", "kappa": min(kappa, 100.0)}
    if kind == "potrs":
        return {"kind": "potrs", "n": _log_int(rng, 500, 16384), "nrhs": _log_int(rng, 1, 64),
                "dtype": rng.choice(["f64", "f64", "f32"])}
    if kind == "mixed":
        return {"kind": "mixed", "n": _log_int(rng, 2000, 32768), "nrhs": _log_int(rng, 1, 64),
                "prec": rng.choice(["bf16", "fp16"]), "words": rng.choice([1, 2, 2, 3]),
                "spectrum": "log", "kappa": min(kappa, 1e3)}
    if kind == "mixed8":
        return {"kind": "mixed", "n": _log_int(rng, 4000, 50000), "nrhs": _log_int(rng, 1, 48),
                "prec": "fp8", "words": 1, "spectrum": "gram", "kappa": 400.0}
    prec = rng.choice(["fp64", "bf16", "fp16"])
    return {"kind": "grad", "n": _log_int(rng, 500, 8192), "nrhs": _log_int(rng, 1, 16),
            "prec": prec, "words": 1 if prec == "fp64" else rng.choice([1, 2]),
            "kappa": min(kappa, 100.0)}


def _dtype(case):
    return torch.float32 if case.get("dtype") == "f32" else torch.float64


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _hartley_rows(x):
    n = x.shape[1]
    f = torch.fft.rfft(x, dim=1)
    h = torch.empty_like(x)
    m = n // 2 + 1
    h[:, :m] = f.real - f.imag
    if n > 2:
        h[:, m:] = (f.real + f.imag)[:, 1:n - m + 1].flip(1)
    return h.div_(math.sqrt(n))


def _spectrum(n, spectrum, kappa, g):
    t = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) / n
    if spectrum == "gram":
        grid = torch.linspace(0.0, math.pi / 2, 4097, dtype=torch.float64, device=DEV)
        cdf = (2.0 * grid - torch.sin(2.0 * grid)) / math.pi  # of |s| = 2 cos(theta), from the top
        i = torch.searchsorted(cdf, t).clamp_(1, 4096)
        w = (t - cdf[i - 1]) / (cdf[i] - cdf[i - 1])
        theta = grid[i - 1] + w * (grid[i] - grid[i - 1])
        lam = (2.0 * torch.cos(theta)).square() + 1e-2
    else:
        lam = torch.exp(t * math.log(kappa))
    return lam[torch.randperm(n, generator=g, device=DEV)]


def _spd(n, spectrum, kappa, g, dtype=torch.float64):
    """An n x n SPD matrix with the given spectrum, exactly symmetric."""
    lam = _spectrum(n, spectrum, kappa, g)
    f = torch.fft.fft(lam) / n
    wt = torch.float64 if n <= 40000 else torch.float32
    cos, sin = f.real.to(wt), (-f.imag).to(wt)
    d0, d1 = (torch.randint(0, 2, (n,), generator=g, device=DEV).to(wt) * 2 - 1 for _ in range(2))
    j = torch.arange(n, device=DEV)
    step = max(1, min(n, (1 << 27) // n))
    y = torch.empty((n, n), dtype=wt, device=DEV)
    for i0 in range(0, n, step):  # Y = (D1 H Lambda H D1) H
        i = torch.arange(i0, min(n, i0 + step), device=DEV)[:, None]
        c = cos[(i - j) % n] + sin[(i + j) % n]
        y[i0:i0 + step] = _hartley_rows(c.mul_(d1[i]).mul_(d1))
    a = torch.empty((n, n), dtype=dtype, device=DEV)
    for i0 in range(0, n, step):  # rows of A = D0 (H Y) D0, A symmetric
        z = _hartley_rows(y[:, i0:i0 + step].t().contiguous())
        a[i0:i0 + step] = z.mul_(d0[i0:i0 + step, None]).mul_(d0)
    del y
    for i0 in range(0, n, step):  # the upper triangle from the lower one
        i1 = min(n, i0 + step)
        a[:i0, i0:i1] = a[i0:i1, :i0].t()
        a[i0:i1, i0:i1] = a[i0:i1, i0:i1].tril() + a[i0:i1, i0:i1].tril(-1).t()
    return a


def _factor(n, g, dtype):
    """The Cholesky factor of a random Wishart matrix with 2n degrees of freedom over n (Bartlett)."""
    low = torch.randn((n, n), generator=g, device=DEV, dtype=dtype).div_(math.sqrt(n)).tril_(-1)
    i = torch.arange(n, device=DEV, dtype=torch.float64)
    low.diagonal().copy_(torch.sqrt((2 * n - i) / n))
    return low


def prepare(case, seed):
    g = _generator(seed)
    n, nrhs, kind = case["n"], case["nrhs"], case["kind"]
    dt = _dtype(case)
    state = {"case": dict(case)}
    if kind == "batched":
        m = torch.randn((case["batch"], n, 2 * n), generator=g, device=DEV, dtype=torch.float64)
        a = m @ m.mT / (2 * n)
        a = 0.5 * (a + a.mT) + 0.1 * torch.eye(n, device=DEV, dtype=torch.float64)
        state["A"] = a.to(dt)
        state["B"] = torch.randn((case["batch"], n, nrhs), generator=g, device=DEV, dtype=dt)
    elif kind == "potrs":
        state["L"] = jmg.colmajor_copy(_factor(n, g, dt))
        state["B"] = torch.randn((n, nrhs), generator=g, device=DEV, dtype=dt)
    else:
        a = _spd(n, case.get("spectrum", "log"), case["kappa"], g, dt)
        x = torch.rand((n, nrhs), generator=g, device=DEV, dtype=dt) * 2 - 1
        state["B"] = a @ x
        state["A"] = a
        if kind == "grad":
            a.requires_grad_(True)
            state["B"].requires_grad_(True)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batched":
        x, low, info = jmg.posv_batched(state["A"], state["B"])
        return {"X": x, "L": low, "info": info}
    if kind == "posv":
        return {"X": jmg.posv(state["A"].mT, state["B"], prec="fp64")[0]}
    if kind == "mixed":
        return {"X": jmg.posv(state["A"].mT, state["B"], prec=case["prec"],
                              words=case["words"])[0]}
    if kind == "factor":
        low = jmg.colmajor_copy(state["A"])
        info = jmg.potrf_(low)
        x = jmg.potrs_(low, jmg.colmajor_copy(state["B"]))
        return {"L": low, "X": x, "logdet": jmg.logdet(low), "info": info}
    if kind == "potrs":
        return {"X": jmg.potrs_(state["L"], jmg.colmajor_copy(state["B"]))}
    x = autograd.solve(state["A"], state["B"], prec=case["prec"], words=case["words"])
    loss = 0.5 * x.square().sum()
    ga, gb = torch.autograd.grad(loss, (state["A"], state["B"]))
    return {"X": x.detach(), "gA": ga, "gB": gb}


def work(case):
    n, r, kind = case["n"], case["nrhs"], case["kind"]
    es = 4 if case.get("dtype") == "f32" else 8
    tri, rhs = n * (n + 1) / 2, 2.0 * n * r
    if kind == "batched":
        b = case["batch"]
        return {"bytes": es * b * (2 * tri + rhs), "flops": b * (n ** 3 / 3 + 2.0 * n * n * r)}
    if kind == "potrs":
        return {"bytes": es * (tri + rhs), "flops": 2.0 * n * n * r}
    if kind == "factor":
        return {"bytes": es * (2 * tri + rhs), "flops": n ** 3 / 3 + 2.0 * n * n * r}
    if kind == "grad":
        return {"bytes": es * (tri + n * n + 2 * rhs), "flops": n ** 3 / 3 + 6.0 * n * n * r}
    return {"bytes": es * (tri + rhs), "flops": n ** 3 / 3 + 2.0 * n * n * r}


def _solve64(a, b):
    """A^-1 B in 64 bits: a Cholesky factor, in 32 bits where 64 would take too long, and refinement in 64."""
    n = a.shape[0]
    wt = torch.float64 if n <= 20000 else torch.float32
    low = torch.linalg.cholesky(a.to(wt))
    x = torch.zeros_like(b)
    for _ in range(2 if wt == torch.float64 else 8):
        r = b - a @ x
        x += torch.cholesky_solve(r.to(wt), low).to(torch.float64)
    return x


def exact(case, seed):
    kind = case["kind"]
    s = prepare(case, seed)
    b = s["B"].detach().double()
    if kind == "batched":
        a = s["A"].double()
        low = torch.linalg.cholesky(a)
        return {"X": torch.cholesky_solve(b, low), "L": low.mT.triu() + a.tril(-1), "info": None}
    if kind == "potrs":
        low = s["L"].double()
        y = torch.linalg.solve_triangular(low, b, upper=False)
        return {"X": torch.linalg.solve_triangular(low.mT, y, upper=True)}
    a = s["A"].detach().double()
    if kind in ("posv", "mixed"):
        return {"X": _solve64(a, b)}
    if kind == "factor":
        low = torch.linalg.cholesky(a)
        return {"L": low + a.triu(1), "X": torch.cholesky_solve(b, low),
                "logdet": 2.0 * low.diagonal().log().sum(), "info": None}
    low = torch.linalg.cholesky(a)
    x = torch.cholesky_solve(b, low)
    gb = torch.cholesky_solve(x, low)
    m = gb @ x.t()
    return {"X": x, "gA": -0.5 * (m + m.t()), "gB": gb}
