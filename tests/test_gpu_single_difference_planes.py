"""Single calls large enough for the difference-plane kernel (one product per unordered plane pair,
256 x 256 tiles on CTA pairs): the same integers as the plane-by-plane kernels, so C is bit for bit
that of the stacked kernel (tile variant 5, forced) over the whole matrix and the oracle's on sampled
rows and columns at tile edges (a row of op(A) and a column of op(B) are split by themselves)."""
import os

import numpy as np
import pytest

import oracle
from paper_2503_22875_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SELECTOR = os.path.join(os.path.dirname(os.path.abspath(workloads.__file__)), "data", "selector_v3.ozgsel")


@pytest.fixture(scope="module")
def ozg():
    from paper_2503_22875_gb300 import build, ozg
    build.build()
    ozg.load()
    return ozg


def draw(shape, phi, cplx, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kw = dict(generator=g, device="cuda", dtype=torch.float64)
    x = (torch.rand(shape, **kw) - 0.5) * torch.exp(phi * torch.randn(shape, **kw))
    if not cplx:
        return x
    return torch.complex(x, (torch.rand(shape, **kw) - 0.5) * torch.exp(phi * torch.randn(shape, **kw)))


def edges(n):
    return sorted({i for e in range(0, n + 256, 128) for i in (e - 1, e, e + 1) if 0 <= i < n} | {n - 1})[-14:]


def operands(cplx, m, n, k, ta, tb, phi, seed):
    """Column-major op storage: a tensor of shape (columns, rows)."""
    A = draw((k, m) if ta == "N" else (m, k), phi, cplx, seed)
    B = draw((n, k) if tb == "N" else (k, n), phi, cplx, seed + 1)
    return A, B, draw((n, m), phi, cplx, seed + 2)


def both(ozg, cplx, m, n, k, s, ta, tb, alpha, beta, A, B, C0, setup=lambda c: None, report=False):
    out = []
    for variant in (-1, 5):
        ctx = ozg.Context()
        setup(ctx)
        ctx.set_tile_variant(variant)
        C = C0.clone()
        torch.cuda.synchronize()
        rep = (ctx.zgemm if cplx else ctx.dgemm)(ta, tb, m, n, k, alpha, A, A.shape[1], B, B.shape[1], beta, C, m, s,
                                                 report=report)
        ctx.sync()
        ctx.close()
        out.append((torch.view_as_real(C) if cplx else C, rep))
    return out


# one and two windows, chains cut at 1024 products (k = 1025, 4097), k below one 64-wide sub-tile,
# rows and columns on, before and past 128 and 256 edges, every transpose, alpha and beta
REAL = [(1920, 1801, 2560, 5, "N", "N", 0.5, 1.0, 0.0), (1793, 2047, 2305, 7, "T", "N", 2.0, -0.5, 0.25),
        (2048, 1800, 4097, 9, "N", "T", 1.0, 1.0, 0.0), (1665, 1919, 4033, 10, "T", "T", 4.0, 1.5, 1.0),
        (1700, 1700, 8200, 3, "N", "N", 0.0, 1.0, 0.0)]
COMPLEX = [(900, 1025, 257, 7, "N", "C", 0.5, 1.0, 0.0), (1000, 833, 96, 6, "C", "N", 2.0, 0.5 - 1j, 0.25j),
           (769, 1153, 64, 5, "T", "C", 1.0, 1.0, 0.0), (961, 897, 1025, 9, "N", "N", 3.0, 1j, 1.0),
           (1000, 1000, 33, 4, "C", "T", 1.0, 1.0, 0.0), (1024, 1024, 1, 4, "N", "N", 0.5, 1.0, 0.0),
           (1100, 770, 65, 10, "T", "N", 1.0, -1.0, 0.5), (1200, 650, 4100, 8, "N", "T", 1.0, 1.0, 0.0),
           (900, 900, 700, 2, "N", "N", 1.0, 1.0, 0.0)]


@pytest.mark.parametrize("case", REAL + COMPLEX, ids=lambda c: "-".join(str(x) for x in c[:6]))
def test_difference_planes_bit_exact(ozg, case):
    m, n, k, s, ta, tb, phi, alpha, beta = case
    cplx = case in COMPLEX
    A, B, C0 = operands(cplx, m, n, k, ta, tb, phi, seed=m + n + k + s)
    (C, _), (E, _) = both(ozg, cplx, m, n, k, s, ta, tb, alpha, beta, A, B, C0)
    assert torch.equal(C, E)
    rows, cols = edges(m), edges(n)
    As, Bs = A.cpu().numpy().T, B.cpu().numpy().T  # m x k or k x m storage
    As = As[rows] if ta == "N" else As[:, rows]
    Bs = Bs[:, cols] if tb == "N" else Bs[cols]
    Cs = np.asfortranarray(C0.cpu().numpy().T[np.ix_(rows, cols)])
    emu = oracle.zgemm_emu if cplx else oracle.dgemm_emu
    want = emu(np.asfortranarray(As), np.asfortranarray(Bs), s, ta, tb, alpha, beta, Cs)
    got = (torch.view_as_complex(C) if cplx else C).cpu().numpy().T[np.ix_(rows, cols)]
    assert np.array_equal(got, want)


@pytest.mark.parametrize("target,beta", [(1e-12, 0.5), (1e-17, 0.0)])
def test_learned_counts_with_and_without_differences(ozg, target, beta):
    """The selected count runs on the difference planes; the fallback that an unreachable target
    forces (13, above them) on the digit planes of the same set."""
    m, n, k = 1801, 1920, 2305
    A, B, C0 = operands(False, m, n, k, "N", "N", 1.0, seed=5)

    def setup(c):
        c.load_selector(SELECTOR)
        c.set_target_error(target)

    (C, r), (E, q) = both(ozg, False, m, n, k, 0, "N", "N", 1.0, beta, A, B, C0, setup, report=True)
    assert torch.equal(C, E)
    assert (r.selected, r.slices_used, r.repaired) == (q.selected, q.slices_used, q.repaired)
    assert r.repaired == (1 if target < 1e-16 else 0)


def test_nonfinite_input_takes_the_native_kernel(ozg):
    m, n, k = 900, 1025, 257
    A, B, C0 = operands(True, m, n, k, "N", "N", 1.0, seed=9)
    A[3, 7] = complex(float("nan"), 0.0)
    (C, r), (E, q) = both(ozg, True, m, n, k, 7, "N", "N", 1.0, 0.0, A, B, C0, report=True)
    assert r.nonfinite == 1 and q.nonfinite == 1
    assert torch.equal(torch.isnan(C), torch.isnan(E))
    assert torch.equal(torch.nan_to_num(C), torch.nan_to_num(E))
