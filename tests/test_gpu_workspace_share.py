"""On a device whose memory a program has mostly taken, a single call keeps to the digit planes it needs
(the difference planes would leave less than three quarters of the rest free), with the same bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
N, S = 3000, 8
LEAVE = 1536 << 20


def test_call_on_a_nearly_full_device():
    from paper_2503_22875_gb300 import build, ozg
    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert ozg.single_plan(sms, False, N, N, N, S)["kd"] == S
    g = torch.Generator(device="cuda").manual_seed(1)
    A, B = (torch.rand((N, N), dtype=torch.float64, device="cuda", generator=g) - 0.5 for _ in range(2))
    out, used, held = [], [], None
    try:
        for full in (False, True):
            C = torch.zeros((N, N), dtype=torch.float64, device="cuda")
            if full:
                torch.cuda.empty_cache()
                held = torch.empty(torch.cuda.mem_get_info()[0] - LEAVE, dtype=torch.uint8, device="cuda")
            ctx = ozg.Context()
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            ctx.dgemm("N", "N", N, N, N, 1.0, A, N, B, N, 0.0, C, N, S)
            ctx.sync()
            used.append(free - torch.cuda.mem_get_info()[0])
            ctx.close()
            out.append(C)
    finally:
        del held
        torch.cuda.empty_cache()
    lean = 9 * (2 * S * N * 3008 * 2 + sms * 128 * 256 * 16) // 8  # digit planes and the epilogue's scratch
    assert used[0] > 2 * lean  # the difference planes, where there is room
    assert used[1] <= lean + (LEAVE - lean) // 4 + (8 << 20)
    assert torch.equal(out[0], out[1])
