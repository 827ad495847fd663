"""The measured work of the library: what a program asks of it, through ``ls.Solver``.

Four kinds of call, over the grids of the workloads and of the serving mix (2D n = 32 .. 1024,
3D n = 16 .. 64, omega / 2 pi = n / 8, media of Gaussian bumps or smoothed noise):

* ``apply``  the operator (I + K omega^2 m) x on device vectors, in FP32 ("mixed"),
  float-float ("ff") or FP64 arithmetic: the product that a caller's own iteration needs;
* ``rhs``    the plane-wave right-hand sides of a medium;
* ``far``    the far-field pattern of solved fields in a set of directions;
* ``solve``  one scattering problem: factorization of the medium, its plane-wave right-hand
  sides and their solution, in mixed precision to 1e-6 or in FP64 to 1e-10.

The results of FP32 arithmetic are kept as a program at that accuracy keeps them, in complex64.
"""

from __future__ import annotations

import cmath
import functools
import math

import numpy as np
import torch

from paper_1408_4495_gb300 import ls, workloads as W

PREC = {"mixed": ls.LS_PREC_MIXED, "ff": ls.LS_PREC_FF, "fp64": ls.LS_PREC_FP64}


def _case(kind, d, n, nrhs, prec, medium="bumps", nobs=0, kernel="helmholtz"):
    return {"kind": kind, "d": d, "n": n, "nrhs": nrhs, "prec": prec, "medium": medium, "nobs": nobs, "kernel": kernel}


def listed():
    return [
        # the smallest call: one vector on the grid of the single-bump workload
        dict(_case("apply", 2, 32, 1, "mixed"), name="apply_mixed_2d_n32_1"),
        # a batch of vectors on the largest 2D grid of the serving mix
        dict(_case("apply", 2, 512, 16, "mixed"), name="apply_mixed_2d_n512_16"),
        # 3D, the radix-3 grid of the serving mix, an odd number of vectors
        dict(_case("apply", 3, 48, 7, "mixed"), name="apply_mixed_3d_n48_7"),
        # the operator at residual accuracy (what refinement checks are made with), an odd batch
        dict(_case("apply", 2, 512, 13, "ff"), name="apply_ff_2d_n512_13"),
        # the plain FP64 operator on the batched 2D workload's grid
        dict(_case("apply", 2, 256, 16, "fp64"), name="apply_fp64_2d_n256_16"),
        # the right-hand sides of the batched 3D workload
        dict(_case("rhs", 3, 64, 8, "mixed"), name="rhs_3d_n64_8"),
        # the pattern of a serving request's fields in 64 directions
        dict(_case("far", 2, 512, 32, "mixed", nobs=64), name="far_2d_n512_32x64"),
        # the plain FP64 workload: one wave on the smallest grid, where latency counts
        dict(_case("solve", 2, 32, 1, "fp64"), name="solve_fp64_2d_n32_1"),
        # a serving request on the small 2D grid, a ragged number of waves
        dict(_case("solve", 2, 128, 21, "mixed"), name="solve_mixed_2d_n128_21"),
        # the batched 2D workload
        dict(_case("solve", 2, 256, 16, "mixed"), name="solve_mixed_2d_n256_16"),
        # a serving request on the large 3D grid of the mix
        dict(_case("solve", 3, 48, 8, "mixed"), name="solve_mixed_3d_n48_8"),
        # the headline workload: 64 waves on the large 2D grid in a noise medium
        dict(_case("solve", 2, 1024, 64, "mixed", medium="noise"), name="solve_mixed_2d_n1024_64"),
    ]


def _count(rng, most):
    """1 .. most, spread over the logarithm."""
    return max(1, min(most, int(round(math.exp(rng.uniform(0.0, math.log(most + 0.49)))))))


def draw(rng):
    shapes = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _draw(rng)
        if case not in shapes:
            return case


def _draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "rhs", "far", "solve", "solve", "solve"])
    d = rng.choice([2, 2, 3])
    n2, n3 = [32, 48, 64, 128, 256, 512, 1024], [16, 24, 32, 48, 64]
    if kind == "solve":
        prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        if prec == "fp64":
            n = rng.choice([32, 48, 64, 128, 256] if d == 2 else [16, 24])
            return _case(kind, d, n, _count(rng, 16), prec)
        n = rng.choice([32, 48, 64, 128, 256, 512] if d == 2 else [16, 24, 32, 48])
        return _case(kind, d, n, _count(rng, 32), prec, medium=rng.choice(["bumps", "noise"]))
    n = rng.choice(n2 if d == 2 else n3)
    if kind == "far":
        n = min(n, 512 if d == 2 else 48)
        nrhs, nobs = _count(rng, 32), _count(rng, 128)
        while nrhs * nobs * n**d > 1 << 31:
            nobs = (nobs + 1) // 2
        return _case(kind, d, n, nrhs, "mixed", nobs=nobs)
    prec = rng.choice(["mixed", "ff", "fp64"]) if kind == "apply" else rng.choice(["mixed", "mixed", "fp64"])
    kernel = rng.choice(["helmholtz", "laplace"]) if kind == "apply" and d == 3 else "helmholtz"
    most = min(64, max(1, (1 << (22 if prec == "fp64" else 25)) // n**d))
    return _case(kind, d, n, _count(rng, most), prec, kernel=kernel)


# ------------------------------------------------------------------------------ inputs
def _omega(case):
    return 2.0 * math.pi * case["n"] / 8.0


def _medium(case, seed):
    """The medium m (the potential V of the Laplace kernel) on the grid, zero in the buffer layers."""
    n, d = case["n"], case["d"]
    if case["kernel"] == "laplace":
        return W.enforce_buffer(W.laplace_3d(n, 1).V * np.random.default_rng(seed).uniform(0.5, 1.0), 2)
    if case["medium"] == "noise":
        return W.enforce_buffer(W.smooth_noise(n, d, seed, 4.0, 0.2), 2)
    rng = np.random.default_rng(seed)
    k = int(rng.integers(4, 9))
    m = W.bumps(n, d, rng.uniform(-0.3, 0.3, k), rng.uniform(0.05, 0.12, k), rng.uniform(0.25, 0.75, (k, d)))
    return W.enforce_buffer(m * min(1.0, 0.3 / np.max(np.abs(m))), 2)


def _directions(d, count, seed):
    rng = np.random.default_rng(seed)
    if d == 2:
        a = rng.uniform(0.0, 2.0 * math.pi) + 2.0 * math.pi * np.arange(count) / count
        return np.stack([np.cos(a), np.sin(a)], axis=1)
    return W.directions_sphere(count, seed)


def _inputs(case, seed):
    """Medium, directions and vectors of a case, as arrays and device tensors."""
    n, d, nrhs = case["n"], case["d"], case["nrhs"]
    inp = {"m": _medium(case, seed), "dirs": torch.tensor(_directions(d, nrhs, seed), device="cuda")}
    if case["kind"] == "far":
        inp["obs"] = torch.tensor(_directions(d, case["nobs"], seed + 1), device="cuda")
    if case["kind"] in ("apply", "far"):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        inp["x"] = torch.randn((nrhs,) + (n,) * d, dtype=torch.complex128, device="cuda", generator=gen)
    return inp


def prepare(case, seed):
    """The solver of the medium (tables of the grid and frequency) and the call's inputs; the
    solver works on the program's own stream."""
    inp = _inputs(case, seed)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    solver = ls.Solver(inp["m"], _omega(case), mixed=case["prec"] != "fp64", stream=stream,
                       laplace=case["kernel"] == "laplace")
    return {"case": case, "solver": solver, "stream": stream, "in": inp}


def run(state):
    case, s, inp = state["case"], state["solver"], state["in"]
    kind, prec = case["kind"], case["prec"]
    with torch.cuda.stream(state["stream"]):
        if kind == "apply":
            y = s.apply(inp["x"], prec=PREC[prec])
            return y.to(torch.complex64) if prec == "mixed" else y
        if kind == "rhs":
            return s.rhs_plane_wave(inp["dirs"])
        if kind == "far":
            return s.far_field(inp["dirs"], inp["x"], inp["obs"])
        s.factor()
        u, _ = s.solve(s.rhs_plane_wave(inp["dirs"]), tol=1e-10 if prec == "fp64" else 1e-6)
        return u if prec == "fp64" else u.to(torch.complex64)


def work(case):
    """Inputs read and outputs written once (tables of the medium and the symbol included), the
    transforms at 5 P log2 P, a direct sum of one product per point and pair of directions, and
    for a solve the factors written and read twice per iteration, two iterations."""
    n, d, nrhs = case["n"], case["d"], case["nrhs"]
    N, P = n**d, (2 * n) ** d
    c = 8 if case["prec"] == "mixed" else 16
    fft = 2 * 5 * P * math.log2(P) * nrhs
    tables = (n + 1) ** d * c + N * c // 2
    if case["kind"] == "apply":
        return {"bytes": 32 * N * nrhs + tables, "flops": fft}
    if case["kind"] == "rhs":
        return {"bytes": 16 * N * nrhs + tables, "flops": fft}
    if case["kind"] == "far":
        return {"bytes": 16 * N * nrhs + 8 * N, "flops": 8.0 * N * nrhs * case["nobs"]}
    # fronts of nested dissection: entries and complex LU of separators of n^(d-1) points
    entries = 31 * N * math.log2(n) / 8 if d == 2 else 16 * n**4
    factor = 160.0 * n**3 if d == 2 else 12.0 * n**6
    return {"bytes": 32 * N * nrhs + tables + entries * c * 5,
            "flops": factor + 2 * (fft + 16.0 * entries * nrhs)}


# ------------------------------------------------------------------------------ 64-bit values
def _hankel1(order, z):
    """H_0 or H_1 of the first kind by the trapezoidal rule on Poisson's integral, s = v^2 in
    sqrt(2 / (pi z)) e^{i (z - order pi / 2 - pi / 4)} / Gamma(order + 1/2)
    int_0^inf e^{-s} (s (1 + i s / (2 z)))^{order - 1/2} ds  (z >= 0.4: error below 1e-15)."""
    step, acc = 0.1, torch.zeros_like(z, dtype=torch.complex128)
    for j in range(64):
        v = j * step
        f = torch.complex(torch.ones_like(z), 0.5 * v * v / z) ** (order - 0.5)
        acc += (1.0 if j else 0.5) * math.exp(-v * v) * v ** (2 * order) * f
    phase = torch.polar(torch.sqrt(2.0 / (math.pi * z)), z - order * 0.5 * math.pi - 0.25 * math.pi)
    return phase * acc * (2.0 * step / math.gamma(order + 0.5))


@functools.lru_cache(maxsize=1)
def _symbol(d, n, omega):
    """DFT of the circulant embedding of the Nystrom weights (omega = 0: the Laplace kernel)."""
    h, L = 1.0 / (n + 1), 2 * n
    k = torch.arange(L, device="cuda")
    t = torch.where(k <= n, k, L - k).double()
    r2 = sum((t * t).reshape([-1 if a == b else 1 for b in range(d)]) for a in range(d))
    r2[(0,) * d] = 1.0
    r = h * torch.sqrt(r2)
    if d == 2:
        q = 0.25j * h**2 * _hankel1(0, omega * r[: n + 1, : n + 1])
        K = torch.cat([q, q[1:n].flip(0)])
        K = torch.cat([K, K[:, 1:n].flip(1)], dim=1)
        a = h / math.sqrt(math.pi)
        h1 = complex(_hankel1(1, torch.tensor(omega * a, dtype=torch.float64)))
        k0 = 0.5j * math.pi * a / omega * h1 - 1.0 / omega**2
    else:
        K = torch.polar(h**3 / (4.0 * math.pi * r), omega * r)
        a = h * (3.0 / (4.0 * math.pi)) ** (1.0 / 3.0)
        k0 = cmath.exp(1j * omega * a) * (1.0 / omega**2 - 1j * a / omega) - 1.0 / omega**2 if omega else 0.5 * a * a
    K[(0,) * d] = k0
    for a in range(d):
        K.index_fill_(a, torch.tensor([n], device="cuda"), 0)
    return torch.fft.fftn(K)


def _convolve(sym, v, d, n):
    """K v for one field v."""
    return torch.fft.ifftn(torch.fft.fftn(v, s=(2 * n,) * d) * sym)[(slice(0, n),) * d]


def _plane_wave(case, direction):
    n, d = case["n"], case["d"]
    x = (torch.arange(n, device="cuda", dtype=torch.float64) + 1.0) / (n + 1)
    u = torch.ones((n,) * d, dtype=torch.complex128, device="cuda")
    for a in range(d):
        e = torch.polar(torch.ones_like(x), _omega(case) * float(direction[a]) * x)
        u = u * e.reshape([-1 if a == b else 1 for b in range(d)])
    return u


def _gmres(op, g, tol=1e-13, most=200):
    """The solution of op(u) = g to rounding, or None."""
    beta = float(torch.linalg.vector_norm(g))
    V = torch.empty((most + 1, g.numel()), dtype=g.dtype, device=g.device) if g.numel() * most < 1 << 31 else None
    if V is None:
        return None
    V[0] = g.reshape(-1) / beta
    H = np.zeros((most + 1, most), dtype=complex)
    for k in range(most):
        w = op(V[k].reshape(g.shape)).reshape(-1)
        for _ in range(2):
            c = V[: k + 1].conj() @ w
            w = w - c @ V[: k + 1]
            H[: k + 1, k] += c.cpu().numpy()
        H[k + 1, k] = float(torch.linalg.vector_norm(w))
        V[k + 1] = w / H[k + 1, k]
        if k % 4 == 3:
            e = np.zeros(k + 2, dtype=complex)
            e[0] = beta
            y = np.linalg.lstsq(H[: k + 2, : k + 1], e, rcond=None)[0]
            if np.linalg.norm(e - H[: k + 2, : k + 1] @ y) <= tol * beta:
                return (torch.tensor(y, device=g.device) @ V[: k + 1]).reshape(g.shape)
    return None


def exact(case, seed):
    n, d = case["n"], case["d"]
    inp = _inputs(case, seed)
    m, dirs = torch.tensor(inp["m"], device="cuda"), inp["dirs"].cpu().numpy()
    omega = _omega(case)
    if case["kind"] == "far":
        h, x = 1.0 / (n + 1), (torch.arange(n, device="cuda", dtype=torch.float64) + 1.0) / (n + 1)
        c = cmath.exp(0.25j * math.pi) / math.sqrt(8.0 * math.pi * omega) if d == 2 else 1.0 / (4.0 * math.pi)
        rows = []
        for r in range(case["nrhs"]):
            t = (omega**2 * m * (_plane_wave(case, dirs[r]) + inp["x"][r])).expand((case["nobs"],) + (n,) * d)
            for a in range(d - 1, -1, -1):
                e = torch.exp(-1j * omega * inp["obs"][:, a, None] * x[None])
                t = torch.einsum("k...j,kj->k...", t, e)
            rows.append(-c * h**d * t)
        return torch.stack(rows)
    laplace = case["kernel"] == "laplace"
    sym = _symbol(d, n, 0.0 if laplace else omega)
    w = m if laplace else omega**2 * m
    if case["kind"] == "apply":
        return torch.stack([x + _convolve(sym, w * x, d, n) for x in inp["x"]])
    rhs = [_convolve(sym, -w * _plane_wave(case, dr), d, n) for dr in dirs]
    if case["kind"] == "rhs":
        return torch.stack(rhs)
    us = []
    for g in rhs:
        u = _gmres(lambda v: v + _convolve(sym, w * v, d, n), g)
        if u is None:
            return None
        us.append(u)
    return torch.stack(us)
