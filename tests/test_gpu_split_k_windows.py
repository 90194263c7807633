"""Single calls cut along k where the padded k holds one slice group less per window than k itself:
bit for bit whole tiles (tile variant 5, forced), and the same again on the same context."""
import numpy as np
import pytest

from paper_2503_22875_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (complex, m, n, k, s): the smallest and largest k of the ranges, one tile, tiles by the edge, many
CASES = [(False, 256, 256, 1344, 6), (False, 130, 257, 1281, 6), (False, 200, 130, 700, 11), (False, 1, 1, 641, 11),
         (True, 64, 64, 320, 11), (True, 64, 64, 257, 12), (True, 65, 130, 320, 12), (False, 1300, 700, 1300, 6)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c))
def test_windows_of_cut_calls(case):
    from paper_2503_22875_gb300 import build, ozg
    build.build()
    cplx, m, n, k, s = case
    p = ozg.single_plan(torch.cuda.get_device_properties(0).multi_processor_count, cplx, m, n, k, s)
    assert p["parts"] > 1
    g = workloads.rng(m + n + k + s)

    def draw(r, c):
        x = workloads.wide_exponent((r, c), 1.0, g)
        return np.asfortranarray(x + 1j * workloads.wide_exponent((r, c), 1.0, g)) if cplx else x

    A, B = ozg.to_device(draw(m, k)), ozg.to_device(draw(k, n))
    out = []
    for variant in (5, -1, -1):
        if variant == 5 or len(out) == 1:
            ctx = ozg.Context()
            ctx.set_tile_variant(variant)
        C = torch.zeros((n, m), dtype=torch.complex128 if cplx else torch.float64, device="cuda")
        torch.cuda.synchronize()
        (ctx.zgemm if cplx else ctx.dgemm)("N", "N", m, n, k, 1.0, A, m, B, k, 0.0, C, m, s)
        ctx.sync()
        out.append(torch.view_as_real(C) if cplx else C)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
    assert float(out[0].abs().max()) > 0
