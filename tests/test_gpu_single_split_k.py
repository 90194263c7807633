"""Single calls with few output tiles: the stacked kernel with every tile's k range cut into parts,
whose window sums meet in memory and are rounded by a kernel of their own.  The sums are exact
integers, so C is bit for bit that of whole tiles (tile variant 5, forced), also where a third
window continues in FP64, and the oracle's where two windows hold the sum."""
import numpy as np
import pytest

import oracle
from paper_2503_22875_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ozg():
    from paper_2503_22875_gb300 import build, ozg
    build.build()
    ozg.load()
    return ozg


# (complex, m, n, k, s, transa, transb, alpha, beta): a last part shorter than the others, parts of
# one 64-wide sub-tile, one entry, tile edges, one to three windows, more parts than SMs can hold
CASES = [(False, 256, 256, 256, 7, "N", "N", 1.0, 0.0), (False, 1, 1, 700, 7, "T", "N", -0.5, 0.25),
         (False, 130, 257, 1100, 4, "N", "T", 1.0, 1.0), (False, 129, 128, 4287, 10, "T", "T", 1.5, 0.0),
         (False, 60, 70, 6000, 12, "N", "N", 1.0, 0.5), (False, 127, 383, 129, 9, "N", "N", 1.0, 0.0),
         (True, 65, 64, 2248, 7, "C", "C", 0.5 + 1j, 0.25j), (True, 142, 100, 1265, 10, "T", "N", 1.0, 0.0),
         (True, 33, 190, 450, 5, "N", "C", 1j, 1.0), (True, 20, 20, 3000, 12, "N", "N", 1.0, 0.0)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c[:7]))
def test_split_k_bit_exact(ozg, case):
    cplx, m, n, k, s, ta, tb, alpha, beta = case
    g = workloads.rng(m + n + k + s)

    def draw(r, c):
        x = workloads.wide_exponent((r, c), 1.0, g)
        return np.asfortranarray(x + 1j * workloads.wide_exponent((r, c), 1.0, g)) if cplx else x

    A, B = draw(*((m, k) if ta == "N" else (k, m))), draw(*((k, n) if tb == "N" else (n, k)))
    C0 = draw(m, n)
    dA, dB = ozg.to_device(A), ozg.to_device(B)
    out = []
    for variant in (-1, 5):
        ctx = ozg.Context()
        ctx.set_tile_variant(variant)
        for _ in range(2):  # twice on one context: the sums start from zero each time
            dC = ozg.to_device(C0)
            (ctx.zgemm if cplx else ctx.dgemm)(ta, tb, m, n, k, alpha, dA, A.shape[0], dB, B.shape[0], beta, dC, m, s)
            ctx.sync()
            out.append(ozg.from_device(dC, m, n))
        ctx.close()
    assert all(np.array_equal(C, out[0]) for C in out[1:])
    want = (oracle.zgemm_emu if cplx else oracle.dgemm_emu)(A, B, s, ta, tb, alpha, beta, C0)
    if s <= 10:  # two windows at any k
        assert np.array_equal(out[0], want)
