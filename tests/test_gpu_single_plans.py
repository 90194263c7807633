"""Single calls checked together with the way they run: the plan of each is asked first, so that a change of
the cost model cannot quietly leave a path untested.  Difference planes at the counts and depths that small
matrices no longer take them at, and learned calls whose selected count lies below or above the difference
planes of their plane set, with and without the re-run at the fallback count."""
import os

import numpy as np
import pytest

import oracle
from paper_2503_22875_gb300 import workloads
from test_gpu_single_difference_planes import both, edges, operands

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SELECTOR = os.path.join(os.path.dirname(os.path.abspath(workloads.__file__)), "data", "selector_v3.ozgsel")


@pytest.fixture(scope="module")
def ozg():
    from paper_2503_22875_gb300 import build, ozg
    build.build()
    ozg.load()
    return ozg


def plan(ozg, cplx, m, n, k, s, **kw):
    return ozg.single_plan(torch.cuda.get_device_properties(0).multi_processor_count, cplx, m, n, k, s, **kw)


# one slice, one and two windows, chains cut at 1024 products, tiles past 128 and 256 edges
FIXED = [(3073, 2815, 2560, 5, "N", "N", 0.5, 1.0, 0.0), (2500, 3100, 4033, 10, "T", "T", 4.0, 1.5, 1.0),
         (3071, 2561, 8200, 3, "N", "T", 0.0, 1.0, 0.0), (2048, 2047, 2048, 1, "T", "N", 1.0, -1.0, 0.5)]


@pytest.mark.parametrize("case", FIXED, ids=lambda c: "-".join(str(x) for x in c[:6]))
def test_fixed_counts_on_difference_planes(ozg, case):
    m, n, k, s, ta, tb, phi, alpha, beta = case
    assert plan(ozg, False, m, n, k, s)["kd"] == s
    A, B, C0 = operands(False, m, n, k, ta, tb, phi, seed=m + n + k + s)
    (C, _), (E, _) = both(ozg, False, m, n, k, s, ta, tb, alpha, beta, A, B, C0)
    assert torch.equal(C, E)
    rows, cols = edges(m), edges(n)
    As, Bs = A.cpu().numpy().T, B.cpu().numpy().T
    As = As[rows] if ta == "N" else As[:, rows]
    Bs = Bs[:, cols] if tb == "N" else Bs[cols]
    Cs = np.asfortranarray(C0.cpu().numpy().T[np.ix_(rows, cols)])
    want = oracle.dgemm_emu(np.asfortranarray(As), np.asfortranarray(Bs), s, ta, tb, alpha, beta, Cs)
    assert np.array_equal(C.cpu().numpy().T[np.ix_(rows, cols)], want)


# (complex, m, n, k, phi, target, beta): selected count above the set's difference planes, re-run
LEARNED = [((False, 2500, 3100, 1900, 1.0, 1e-12, 0.5), False, False), ((False, 2500, 3100, 1900, 1.0, 1e-17, 0.0), False, True),
           ((False, 2500, 3100, 1900, 0.0, 3e-16, 0.0), True, False), ((False, 2500, 3100, 1900, 4.0, 1e-18, 0.5), True, True),
           ((True, 1100, 1000, 700, 1.0, 1e-13, 0.5j), False, False), ((True, 1100, 1000, 700, 1.0, 1e-17, 0.5), False, True),
           ((True, 1100, 1000, 700, 0.0, 1e-15, 0.0), True, False), ((True, 1100, 1000, 700, 4.0, 1e-18, 0.0), True, True)]


@pytest.mark.parametrize("case,above,repaired", LEARNED, ids=lambda c: "-".join(map(str, c)) if type(c) is tuple else str(c))
def test_learned_counts_on_a_set_with_differences(ozg, case, above, repaired):
    cplx, m, n, k, phi, target, beta = case
    kd = plan(ozg, cplx, m, n, k, 0, sel_max=12, fallback=13)["kd"]
    assert kd == 10
    A, B, C0 = operands(cplx, m, n, k, "N", "N", phi, seed=5)

    def setup(c):
        c.load_selector(SELECTOR)
        c.set_target_error(target)

    (C, r), (E, q) = both(ozg, cplx, m, n, k, 0, "N", "N", 1.0, beta, A, B, C0, setup, report=True)
    assert (r.selected > kd, r.repaired) == (above, int(repaired))
    assert torch.equal(C, E)
    assert (r.selected, r.slices_used, r.repaired) == (q.selected, q.slices_used, q.repaired)
