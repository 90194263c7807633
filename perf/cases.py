"""Performance cases of the emulated FP64 / complex128 GEMM library.

Each case is one call (or one batch) that a program makes through the Python binding
``paper_2503_22875_gb300.ozg``: single real and complex products with a fixed slice count, the
3M complex product, products whose slice count the learned selector chooses, and grouped batches
on device and on host memory.  ``listed`` names the fixed cases, ``draw`` gives more of the same
ranges.  Matrices are column-major; a column-major m x n matrix is a torch tensor of shape (n, m).
"""
from __future__ import annotations

import functools
import math
import os
import random

import numpy as np
import torch

from paper_2503_22875_gb300 import ozg

SELECTOR = os.path.join(os.path.dirname(os.path.abspath(ozg.__file__)), "data", "selector_v3.ozgsel")
TARGET = 1e-12  # componentwise error relative to |A||B| that learned calls aim at
ALIGN = 32      # elements between the matrices of a flat batch buffer (256 bytes)


def _case(op, m, n, k, s, name=None, ta="N", tb="N", phi=0.0, alpha=1.0, beta=0.0):
    c = {"op": op, "m": m, "n": n, "k": k, "s": s, "ta": ta, "tb": tb, "phi": phi, "alpha": alpha, "beta": beta}
    return {"name": name, **c} if name else c


def _batch(op, count, lo, hi, s_lo, s_hi, shapes, name=None):
    """A batch of `count` uneven products, sizes log-uniform in [lo, hi]; slice counts uniform in
    s_lo .. s_hi, or chosen by the selector when s_lo is 0."""
    c = {"op": op, "count": count, "lo": lo, "hi": hi, "s_lo": s_lo, "s_hi": s_hi, "shapes": shapes}
    return {"name": name, **c} if name else c


def listed():
    return [
        # one small product, U(-1, 1): the latency of a call that does little work
        _case("dgemm", 256, 256, 256, 7, name="dgemm_256_s7"),
        # odd sizes, a transposed operand, alpha and beta: a general BLAS call of middling size
        _case("dgemm", 1537, 2001, 1111, 10, name="dgemm_ragged_tn_s10", ta="T", phi=4.0, alpha=1.5, beta=0.5),
        # an ordinary square product
        _case("dgemm", 2048, 2048, 2048, 8, name="dgemm_2048_s8", phi=2.0),
        # the largest: a whole-machine product, the smallest count that meets 1e-12 at this spread
        _case("dgemm", 8192, 8192, 8192, 7, name="dgemm_8192_s7", phi=0.5),
        # short k, large C: the trailing update of a blocked factorisation
        _case("dgemm", 6000, 6000, 192, 9, name="dgemm_rank192_s9", tb="T", phi=1.0, alpha=-1.0),
        # block-structured complex product of a multiple-scattering code (113 blocks of 32)
        _case("zgemm", 3616, 3616, 3616, 7, name="zgemm_kkr_3616_s7"),
        # the same structure on a small cluster, conjugate-transposed operand, fewer slices
        _case("zgemm", 768, 768, 768, 6, name="zgemm_kkr_768_cn_s6", ta="C"),
        # the 3M form of the complex product
        _case("zgemm3m", 1824, 1824, 1824, 7, name="zgemm3m_kkr_1824_s7"),
        # one product whose slice count is left to the selector, the check judging the result
        _case("dgemm", 2500, 3100, 1900, 0, name="dgemm_learned_2500", phi=1.5),
        # many uneven products in one launch sequence, learned counts: the library's batch workload
        _batch("grouped", 2048, 32, 2048, 0, 0, 4, name="grouped_learned_2048"),
        # a batch of small uneven products with counts fixed by the caller, mixed transposes
        _batch("grouped", 256, 24, 512, 5, 10, 6, name="grouped_fixed_256"),
        # a batch in page-locked host memory through the staged entry point
        _batch("host", 192, 32, 1024, 0, 0, 8, name="host_batch_192"),
    ]


def _log_int(rng: random.Random, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["dgemm", "dgemm", "dgemm", "zgemm", "zgemm3m", "learned", "grouped", "grouped", "host"])
    if kind in ("grouped", "host"):
        learned = kind == "host" or rng.random() < 0.5
        return _batch(kind, _log_int(rng, 12, 160 if kind == "host" else 640), rng.choice([17, 24, 32, 48]),
                      _log_int(rng, 256, 1024 if kind == "host" else 1536), 0 if learned else 5,
                      0 if learned else rng.choice([7, 9, 10]), rng.randrange(1 << 20))
    cplx = kind.startswith("z")
    m, n, k = (_log_int(rng, 48, 3200 if cplx else 6144) for _ in range(3))
    s = 0 if kind == "learned" else rng.randint(4, 10 if cplx else 12)
    ta, tb = (rng.choice("NTC" if cplx else "NT") for _ in range(2))
    alpha, beta = rng.choice([(1.0, 0.0), (1.0, 0.0), (-1.0, 0.0), (0.75, 0.5)])
    phi = 0.0 if cplx else round(rng.uniform(0.0, 4.0), 2)
    return _case("dgemm" if kind == "learned" else kind, m, n, k, s, ta=ta, tb=tb, phi=phi, alpha=alpha, beta=beta)


# ---------------------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _real(cols, rows, phi, g):
    """Entries (u - 0.5) exp(phi z), or U(-1, 1) for phi = 0; shape (cols, rows)."""
    u = torch.rand((cols, rows), generator=g, device="cuda", dtype=torch.float64)
    if phi == 0.0:
        return 2.0 * u - 1.0
    return (u - 0.5) * torch.exp(phi * torch.randn((cols, rows), generator=g, device="cuda", dtype=torch.float64))


def _kkr(cols, rows, g):
    """Block-structured complex entries: normal, scaled per 32 x 32 block by exp(-distance) of two
    atom sites, with a shifted diagonal."""
    nb = (max(cols, rows) + 31) // 32
    r = torch.rand((nb, 3), generator=g, device="cuda", dtype=torch.float64) * nb ** (1.0 / 3.0)
    scale = torch.exp(-torch.cdist(r, r)).repeat_interleave(32, 0).repeat_interleave(32, 1)[:cols, :rows]
    z = torch.randn((cols, rows), generator=g, device="cuda", dtype=torch.complex128) * scale
    z.diagonal().add_(1.0 + 0.1j)
    return z.contiguous()


def _shapes(case):
    """(m, n, k, transa, transb, phi, s) of every product of a batch, fixed by the case."""
    g = np.random.Generator(np.random.PCG64(case["shapes"]))
    lo, hi = case["lo"], case["hi"]
    dims = np.exp(g.uniform(np.log(lo), np.log(hi), size=(case["count"], 3))).round().astype(int)
    phi = g.uniform(0.0, 4.0, size=case["count"])
    tr = g.integers(0, 2, size=(case["count"], 2)) if case["s_lo"] else np.zeros((case["count"], 2), int)
    s = g.integers(case["s_lo"], case["s_hi"] + 1, size=case["count"])
    return [(int(d[0]), int(d[1]), int(d[2]), "NT"[t[0]], "NT"[t[1]], float(p), int(x))
            for d, t, p, x in zip(dims, tr, phi, s)]


def _batch_buffers(case, seed):
    """Flat buffers of a batch's A, B and C and each product's views into them."""
    g = _gen(seed)
    shapes = _shapes(case)

    def offsets(sizes):
        ends = np.cumsum([(z + ALIGN - 1) // ALIGN * ALIGN for z in sizes])
        return [0] + [int(e) for e in ends[:-1]], int(ends[-1])

    oa, na = offsets([m * k for m, n, k, *_ in shapes])
    ob, nb = offsets([k * n for m, n, k, *_ in shapes])
    oc, nc = offsets([m * n for m, n, k, *_ in shapes])
    A, B = (torch.zeros(z, device="cuda", dtype=torch.float64) for z in (na, nb))
    for (m, n, k, _, _, phi, _), a, b in zip(shapes, oa, ob):
        A[a:a + m * k] = _real(1, m * k, phi, g)[0]
        B[b:b + k * n] = _real(1, k * n, phi, g)[0]
    return shapes, A, B, nc, oa, ob, oc


@functools.lru_cache(maxsize=None)
def _handle(learned):
    """The context that a program keeps for its single calls."""
    ctx = ozg.Context()
    if learned:
        ctx.load_selector(SELECTOR)
        ctx.set_target_error(TARGET)
    return ctx


def prepare(case, seed):
    if case["op"] in ("grouped", "host"):
        shapes, A, B, nc, oa, ob, oc = _batch_buffers(case, seed)
        if case["op"] == "host":
            A, B = (x.cpu().pin_memory() for x in (A, B))
            C = torch.zeros(nc, dtype=torch.float64).pin_memory()
        else:
            C = torch.zeros(nc, dtype=torch.float64, device="cuda")
        # a batch that is submitted again and again keeps its context, and with it its plan
        stream = torch.cuda.Stream()
        ctx = ozg.Context(stream=stream)
        if case["s_lo"] == 0:
            ctx.load_selector(SELECTOR)
            ctx.set_target_error(TARGET)
        calls = [(ta, tb, m, n, k, 1.0, A[a:a + m * k], m if ta == "N" else k, B[b:b + k * n], k if tb == "N" else n,
                  0.0, C[c:c + m * n], m) for (m, n, k, ta, tb, _, _), a, b, c in zip(shapes, oa, ob, oc)]
        torch.cuda.synchronize()
        return {"op": case["op"], "ctx": ctx, "stream": stream, "calls": calls, "s": [x[6] for x in shapes], "A": A,
                "B": B, "C": C}
    m, n, k = case["m"], case["n"], case["k"]
    g = _gen(seed)
    a, b = ((k, m) if case["ta"] == "N" else (m, k)), ((n, k) if case["tb"] == "N" else (k, n))
    if case["op"] == "dgemm":
        A, B = _real(*a, case["phi"], g), _real(*b, case["phi"], g)
        C0 = _real(n, m, case["phi"], g) if case["beta"] else None
    else:
        A, B = _kkr(*a, g), _kkr(*b, g)
        C0 = _kkr(n, m, g) if case["beta"] else None
    C = torch.zeros((n, m), dtype=A.dtype, device="cuda")
    torch.cuda.synchronize()
    args = (case["ta"], case["tb"], m, n, k, case["alpha"], A, a[1], B, b[1], case["beta"], C, m, case["s"])
    return {"op": case["op"], "ctx": _handle(case["s"] == 0), "args": args, "C0": C0, "C": C}


def run(state):
    ctx = state["ctx"]
    if state["op"] == "grouped":
        ctx.dgemm_grouped(state["calls"], state["s"])
    elif state["op"] == "host":
        ctx.dgemm_grouped_host(state["calls"], state["s"])
    else:
        if state["C0"] is not None:  # beta != 0 updates C: each pass starts from the same C
            state["C"].copy_(state["C0"])
        getattr(ctx, state["op"])(*state["args"])
    return state["C"]


def _products(case):
    """(real multiply-adds, elements of A and B, elements of C, slice count) of every product."""
    if "count" in case:
        return [(m * n * k, m * k + k * n, m * n, s or 8) for m, n, k, _, _, _, s in _shapes(case)]
    m, n, k = case["m"], case["n"], case["k"]
    per = {"dgemm": 1, "zgemm": 4, "zgemm3m": 3}[case["op"]]
    return [(per * m * n * k, m * k + k * n, m * n * (2 if case["beta"] else 1), case["s"] or 8)]


def work(case):
    """Inputs read once and outputs written once; the slice products of the method, s (s + 1) / 2
    integer products per real multiply-add (about s = 8 where the selector chooses)."""
    size = 8 if case["op"] in ("dgemm", "grouped", "host") else 16
    p = _products(case)
    return {"bytes": sum(size * (ab + c) for _, ab, c, _ in p),
            "flops": sum(2 * mac * (s * (s + 1) // 2) for mac, _, _, s in p)}


def exact(case, seed):
    if case["op"] in ("grouped", "host"):
        shapes, A, B, nc, oa, ob, oc = _batch_buffers(case, seed)
        C = torch.zeros(nc, dtype=torch.float64, device="cuda")
        for (m, n, k, ta, tb, _, _), a, b, c in zip(shapes, oa, ob, oc):
            At, Bt = A[a:a + m * k], B[b:b + k * n]
            At = At.view(k, m) if ta == "N" else At.view(m, k).T
            Bt = Bt.view(n, k) if tb == "N" else Bt.view(k, n).T
            C[c:c + m * n] = (Bt @ At).reshape(-1)
        return C
    st = prepare(case, seed)
    A, B = st["args"][6], st["args"][8]
    At, Bt = (x if t == "N" else x.T if t == "T" else x.conj().T for x, t in ((A, case["ta"]), (B, case["tb"])))
    C = case["alpha"] * (Bt.resolve_conj() @ At.resolve_conj())
    return C if st["C0"] is None else C + case["beta"] * st["C0"]
