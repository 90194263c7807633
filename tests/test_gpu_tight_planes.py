"""Calls whose workspace has no room for digit planes on whole 128-byte lines (here: a reserved
workspace that cannot grow while the stream is captured) run on 16-byte rows with the same bits."""
import pytest

pytestmark = pytest.mark.gpu
N = 12000
RESERVED = 200 << 20  # between the two layouts' needs at N x N x 13, s = 8 (at most 180 and at least 270 MB)


@pytest.mark.parametrize("op,ta,tb,k", [("d", "N", "N", 8), ("d", "T", "N", 13), ("d", "N", "T", 1), ("z", "N", "C", 13)])
def test_tight_planes(op, ta, tb, k):
    import torch

    from paper_2503_22875_gb300 import ozg
    g = torch.Generator(device="cuda").manual_seed(5)
    w = 2 if op == "z" else 1
    A = torch.rand(N * k * w, dtype=torch.float64, device="cuda", generator=g) - 0.5
    B = torch.rand(N * k * w, dtype=torch.float64, device="cuda", generator=g) - 0.5
    lda, ldb = (N if ta == "N" else k), (k if tb == "N" else N)
    out = []
    for reserved in (0, RESERVED):
        C = torch.zeros(N * N * w, dtype=torch.float64, device="cuda")
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        ctx = ozg.Context(reserved, stream=st)
        ctx.set_check_samples(0)
        call = lambda: getattr(ctx, op + "gemm")(ta, tb, N, N, k, 1.0, A, lda, B, ldb, 0.0, C, N, 8)
        if reserved:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                call()
            graph.replay()
        else:
            call()
        torch.cuda.synchronize()
        out.append(C)
        ctx.close()
    assert torch.equal(out[0].view(torch.int64), out[1].view(torch.int64))
    assert float(out[0].abs().max()) > 0
