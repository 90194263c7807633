"""The plan of single calls (host only, no GPU).  A call cut along k keeps as many window words per
output as the kernels index: their windows follow from k padded to whole 128-wide stages."""
import pytest

from paper_2503_22875_gb300 import build, ozg

SMS = 152


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


def kernel_windows(s, k, cplx):
    """Windows the stacked kernel walks: the first of len0 groups, then `win` groups at a time."""
    gmax = s * (-(-k // 128) * 128) * 127 * 127 * (2 if cplx else 1)
    win = max(1, (62 - gmax.bit_length()) // 7 + 1)
    len0 = min(s, win)
    if win < s <= 2 * win and (win - s) % 2 and s - (win - 1) <= win:
        len0 = win - 1
    n, start, length = 0, 2, len0
    while start <= s + 1:
        n, start = n + 1, start + length
        length = min(win, s + 2 - start)
    return n


@pytest.mark.parametrize("cplx", [False, True])
def test_window_words_of_cut_calls(cplx):
    """Every fixed count and 600 sub-tile counts of k, and the learned calls, which may run any count."""
    bad = []
    for kb in range(1, 601):
        most = 0
        for s in range(1, 17):
            k = 64 * kb - (s * 7) % 64
            p = ozg.single_plan(SMS, cplx, 64, 64, k, s)
            most = max(most, kernel_windows(s, k, cplx))
            if p["parts"] > 1 and p["part_windows"] < kernel_windows(s, k, cplx):
                bad.append((s, k))
        p = ozg.single_plan(SMS, cplx, 64, 64, 64 * kb, 0, sel_max=12, fallback=13)
        need = max(kernel_windows(s, 64 * kb, cplx) for s in range(1, 14))
        if p["parts"] > 1 and p["part_windows"] < need:
            bad.append((0, 64 * kb))
    assert not bad, f"{len(bad)} calls, e.g. {bad[:5]}"


@pytest.mark.parametrize("call", [(False, 256, 256, 1344, 6), (False, 200, 130, 700, 11), (False, 1300, 700, 1300, 6),
                                  (True, 64, 64, 320, 11), (True, 64, 64, 320, 12), (False, 130, 257, 1281, 6)])
def test_words_at_the_padding_edge(call):
    """Calls whose window is one group shorter for the padded k than for whole 64-wide sub-tiles."""
    cplx, m, n, k, s = call
    p = ozg.single_plan(SMS, cplx, m, n, k, s)
    assert p["parts"] > 1 and p["part_windows"] == kernel_windows(s, k, cplx)


@pytest.mark.parametrize("call", [(False, 2500, 3100, 1900), (False, 4096, 4096, 4096), (False, 300, 200, 3000),
                                  (True, 1800, 1700, 1900), (False, 1537, 2001, 1111)])
def test_learned_plan_does_not_depend_on_a_low_fallback(call):
    """A learned call is planned by the counts the selector can choose, whether the fallback count adds
    digit planes above the selector's largest class (13), ends at it (12) or below."""
    plans = [ozg.single_plan(SMS, *call, 0, sel_max=12, fallback=f) for f in (13, 12, 10, 7)]
    how = [(p["kd"], p["parts"], p["part_kb"]) for p in plans]
    assert how == how[:1] * len(how)
    if call == (False, 2500, 3100, 1900):
        assert plans[0]["kd"] == 10
