"""What the library is measured on: emulated FP64 matrix products through its
public entry points, over the range its users call it with.

A case is a dict of plain values:

  entry   "dgemm" (oz2_dgemm), "noalloc" (oz2_dgemm_noalloc), "ex"
          (oz2_dgemm_ex with a workspace the caller keeps) or "host"
          (oz2_dgemm_host on pinned host buffers)
  m, n, k sizes of C = A·B (A m×k, B k×n, all column-major)
  r       moduli count (the accuracy asked for)
  phi     exponent spread of the entries, U(-1/2, 1/2)·exp(phi·N(0, 1))
  wide    share of A's rows scaled by 2^±300 (they take the native FP64 path)
  pad     rows beyond the matrix in each leading dimension (a submatrix of a
          larger array)
  quant, scale   the quantiser and scale rule of the "ex" entry
"""
from __future__ import annotations

import ctypes
import math

import torch

import paper_2606_06510_gb300 as oz


def _case(entry, m, n, k, r=12, phi=0.5, wide=0.0, pad=0, quant="tz", scale="r2", name=None):
    c = {"entry": entry, "m": m, "n": n, "k": k, "r": r, "phi": phi, "wide": wide, "pad": pad,
         "quant": quant, "scale": scale}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # One tile, a k that is no multiple of anything, for a caller that may
        # not allocate (blocks of a blocked solver, a plug-in): latency.
        _case("noalloc", 96, 80, 200, name="noalloc_96x80x200"),
        # A small square product, as panels and tests use: latency and launches.
        _case("dgemm", 256, 256, 256, name="dgemm_256"),
        # Odd sizes inside a larger array: a trailing update of a factorisation.
        _case("dgemm", 1000, 777, 1333, pad=3, name="ragged_1000x777x1333"),
        # A middle-sized product at reduced accuracy (few moduli), as iterative
        # refinement takes it.
        _case("dgemm", 2048, 2048, 2048, r=8, name="dgemm_2048_r8"),
        # The workhorse: the square product the benchmark quotes.
        _case("dgemm", 4096, 4096, 4096, name="dgemm_4096"),
        # Rounding to nearest, the crude scale bound and a high moduli count, in
        # a workspace of the caller's, odd sizes.
        _case("ex", 2500, 3001, 2047, r=15, phi=1.0, quant="rn", scale="r1", name="ex_rn_r1_2500x3001x2047"),
        # The large square product (accuracy at long k takes r = 13).
        _case("dgemm", 16384, 16384, 16384, r=13, phi=1.0, name="dgemm_16384"),
        # Tall k: an overlap or normal-equations product.
        _case("dgemm", 1024, 1024, 65536, name="dgemm_tallk"),
        # Low intensity: a rank-64 update of a large matrix with a wide dynamic
        # range and rows that leave the admissible one.
        _case("dgemm", 16384, 16384, 64, phi=4.0, wide=0.01, name="dgemm_k64_wide"),
        # A large matrix against 16 right-hand sides (batched GEMV).
        _case("dgemm", 16384, 16, 16384, name="gemv_batch16"),
        # A Gram-type block: a small C over a long k.
        _case("dgemm", 256, 256, 65536, name="gram_256"),
        # Operands and result in pinned host memory, copies included.
        _case("host", 4096, 4096, 4096, name="host_4096"),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(("small", "noalloc", "general", "general", "ex", "tallk", "shortk", "skinny", "gram", "host"))
    phi = rng.choice((0.5, 0.5, 1.0, 2.0))
    r = rng.choice((6, 8, 10, 11, 12, 12, 12, 13, 14, 16))
    pad = rng.choice((0, 0, 1, 2, 5))
    if kind == "small":
        return _case("dgemm", _log(rng, 16, 600), _log(rng, 16, 600), _log(rng, 16, 1500), r, phi, pad=pad)
    if kind == "noalloc":
        return _case("noalloc", _log(rng, 16, 400), _log(rng, 16, 400), _log(rng, 16, 400), r, phi, pad=pad)
    if kind == "general":
        return _case("dgemm", _log(rng, 300, 6000), _log(rng, 300, 6000), _log(rng, 300, 6000), r, phi, pad=pad)
    if kind == "ex":
        return _case("ex", _log(rng, 200, 4000), _log(rng, 200, 4000), _log(rng, 200, 4000), r, phi, pad=pad,
                     quant=rng.choice(("tz", "rn")), scale=rng.choice(("r2", "r1")))
    if kind == "tallk":
        return _case("dgemm", _log(rng, 512, 1600), _log(rng, 512, 1600), _log(rng, 16000, 80000), r, phi, pad=pad)
    if kind == "shortk":
        return _case("dgemm", _log(rng, 3000, 16384), _log(rng, 3000, 16384), _log(rng, 16, 256), r,
                     rng.choice((0.5, 2.0, 4.0)), rng.choice((0.0, 0.01)), pad)
    if kind == "skinny":
        a, b, k = _log(rng, 3000, 16384), rng.randint(1, 40), _log(rng, 3000, 16384)
        return _case("dgemm", *((a, b) if rng.random() < 0.7 else (b, a)), k, r, phi, pad=pad)
    if kind == "gram":
        return _case("dgemm", _log(rng, 48, 500), _log(rng, 48, 500), _log(rng, 8000, 100000), r, phi, pad=pad)
    return _case("host", _log(rng, 500, 4096), _log(rng, 500, 4096), _log(rng, 500, 4096), r, phi, pad=pad)


def _matrix(rows, cols, phi, pad, gen):
    """rows×cols column-major on the GPU, leading dimension rows + pad."""
    x = torch.empty((cols, rows + pad), dtype=torch.float64, device="cuda").normal_(generator=gen)
    x.mul_(phi).exp_()
    u = torch.empty_like(x).uniform_(-0.5, 0.5, generator=gen)
    return x.mul_(u).t()[:rows]


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    m, n, k, pad = case["m"], case["n"], case["k"], case["pad"]
    A = _matrix(m, k, case["phi"], pad, gen)
    B = _matrix(k, n, case["phi"], pad, gen)
    cnt = math.ceil(case["wide"] * m)
    if cnt:
        rows = torch.randperm(m, generator=gen, device="cuda")[:cnt]
        s = torch.ones(m, dtype=torch.float64, device="cuda")
        s[rows[:cnt // 2]] = 2.0 ** 300
        s[rows[cnt // 2:]] = 2.0 ** -300
        A *= s[:, None]
    return A, B


def _pinned(t):
    """A pinned host copy of a column-major matrix, with its leading dimension."""
    rows, cols = t.shape
    h = torch.empty((cols, t.stride(1)), dtype=torch.float64, pin_memory=True)
    h[:, :rows].copy_(t.t())
    return h.t()[:rows]


def prepare(case, seed):
    A, B = _inputs(case, seed)
    m, n, k = case["m"], case["n"], case["k"]
    C = torch.zeros((n, m + case["pad"]), dtype=torch.float64, device="cuda").t()[:m]
    state = {"case": case, "A": A, "B": B, "C": C}
    if case["entry"] == "host":
        state["A"], state["B"], state["C"] = _pinned(A), _pinned(B), _pinned(C)
    elif case["entry"] == "ex":
        state["ws"] = torch.empty(oz.oz2_workspace_size(m, n, k, case["r"]), dtype=torch.uint8, device="cuda")
    elif case["entry"] == "noalloc":  # no binding of its own: the C entry point
        state["call"] = (m, n, k, *(v for t in (A, B, C) for v in (ctypes.c_void_p(t.data_ptr()), t.stride(1))),
                         case["r"])
    return state


def run(state):
    case, A, B, C = state["case"], state["A"], state["B"], state["C"]
    entry, r = case["entry"], case["r"]
    if entry == "dgemm":
        return oz.oz2_dgemm(A, B, C, num_moduli=r)
    if entry == "host":
        return oz.oz2_dgemm_host(A, B, C, num_moduli=r)
    if entry == "ex":
        return oz.oz2_dgemm_ex(A, B, C, r, case["quant"], case["scale"], workspace=state["ws"])[0]
    code = oz.lib().oz2_dgemm_noalloc(*state["call"], ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if code != oz.OZ2_OK:
        raise oz.Oz2Error(code, "oz2_dgemm_noalloc")
    return C


def work(case):
    """A, B read and C written once; the 3r FP8 plane products of the method
    (2mnk each) are the operations (the library's FP8 rate is twice bf16's)."""
    m, n, k = case["m"], case["n"], case["k"]
    return {"bytes": 8 * (m * k + k * n + m * n), "flops": 3 * case["r"] * 2 * m * n * k}


def exact(case, seed):
    A, B = _inputs(case, seed)
    C = torch.matmul(A, B)
    return C.cpu() if case["entry"] == "host" else C
