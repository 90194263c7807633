"""Single calls of the kernels whose MMA warp issues as a whole (difference planes, stacked pairs,
stacked pairs on parts of k), repeated on two contexts and streams at once: every wait ends in its
phase (no time-out is raised) and every result has the bits of the first."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CALLS = [(2048, 2048, 2048, 8, "kd"), (1537, 1100, 1500, 16, "whole"), (300, 260, 1111, 9, "parts")]


def test_repeated_calls_on_two_streams():
    from paper_2503_22875_gb300 import build, ozg
    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator(device="cuda").manual_seed(3)
    work = []
    for m, n, k, s, way in CALLS:
        p = ozg.single_plan(sms, False, m, n, k, s)
        assert way == ("kd" if p["kd"] else "parts" if p["parts"] > 1 else "whole")
        A, B = (torch.rand(x, dtype=torch.float64, device="cuda", generator=g) - 0.5 for x in ((k, m), (n, k)))
        work.append((m, n, k, s, A, B))
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    ctx = [ozg.Context(stream=st) for st in streams]
    first, last = {}, {}
    for rep in range(40):
        for i, (m, n, k, s, A, B) in enumerate(work):
            for j in range(2):
                with torch.cuda.stream(streams[j]):
                    C = torch.zeros((n, m), dtype=torch.float64, device="cuda")
                    ctx[j].dgemm("N", "N", m, n, k, 1.0, A, m, B, k, 0.0, C, m, s)
                (last if (i, j) in first else first)[(i, j)] = C
    for c in ctx:
        c.sync()  # raises when a bounded wait gave up
    torch.cuda.synchronize()
    for key, C in last.items():
        assert torch.equal(C, first[key]) and torch.equal(C, first[(key[0], 0)])
