"""The autotuner on single calls that the cost model runs on difference planes: they are timed once against
the tile variants, the choice is saved under a bucket of their own and later contexts run as it says.  What
ran shows in the workspace: difference planes take about twice the memory of a call on tiles."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
M, N, K, S = 2048, 2047, 2300, 8


@pytest.fixture(scope="module")
def run():
    from paper_2503_22875_gb300 import build, ozg
    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert ozg.single_plan(sms, False, M, N, K, S)["kd"] == S
    g = torch.Generator(device="cuda").manual_seed(2)
    A, B = (torch.rand(x, dtype=torch.float64, device="cuda", generator=g) - 0.5 for x in ((K, M), (N, K)))

    def call(path, tune, beta=0.0, variant=-1, calls=1):
        """C and the workspace that the calls' context took."""
        C = torch.zeros((N, M), dtype=torch.float64, device="cuda")
        ctx = ozg.Context()
        ctx.set_autotune(tune, str(path) if path else None)
        ctx.set_tile_variant(variant)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for _ in range(calls):
            ctx.dgemm("N", "N", M, N, K, 1.0, A, M, B, K, beta, C, M, S)
        ctx.sync()
        used = free - torch.cuda.mem_get_info()[0]
        ctx.close()
        return C, used

    call(None, False)  # the kernels are loaded
    return call


def lines(path):
    return [x.split() for x in path.read_text().splitlines()]


def test_choice_is_timed_once_saved_and_read_back(run, tmp_path):
    path = tmp_path / "tune.txt"
    want, _ = run(None, False, variant=5)
    C, _ = run(path, True, calls=2)
    assert torch.equal(C, want)
    (bucket, choice), = lines(path)
    assert int(bucket, 16) >> 63 == 1 and choice in ("0", "1", "2", "3", "5", "6")
    C, _ = run(path, True)
    assert torch.equal(C, want) and len(lines(path)) == 1


def test_saved_choices_are_what_runs(run, tmp_path):
    path = tmp_path / "tune.txt"
    want, _ = run(None, False, variant=5)
    _, differences = run(None, False)
    run(path, True)
    (bucket, _), = lines(path)
    for choice in ("1", "5", "6"):
        path.write_text(f"{bucket} {choice}\n")
        for tune in (False, True):
            C, got = run(path, tune)
            assert torch.equal(C, want) and (got > 0.9 * differences) == (choice == "6") and got < 1.1 * differences
            assert got > 0.9 * differences or got < 0.75 * differences
    path.write_text("%x 1\n" % (int(bucket, 16) & ~(1 << 63)))  # made without difference planes in the comparison
    C, got = run(path, False)
    assert torch.equal(C, want) and got > 0.9 * differences


def test_updates_of_c_are_not_timed(run, tmp_path):
    path = tmp_path / "tune.txt"
    run(path, True, beta=0.5)
    assert not path.exists() or path.read_text() == ""


def test_captured_calls_are_not_timed(tmp_path):
    """A call that is captured into a graph runs as planned: timing it would need the stream."""
    from paper_2503_22875_gb300 import build, ozg
    build.build()
    path = tmp_path / "tune.txt"
    g = torch.Generator(device="cuda").manual_seed(2)
    out = []
    for shape in ((M, N, K, S), (300, 200, 500, 6)):  # difference planes; cut along k
        m, n, k, s = shape
        A, B = (torch.rand(x, dtype=torch.float64, device="cuda", generator=g) - 0.5 for x in ((k, m), (n, k)))
        for capture in (False, True):
            C = torch.zeros((n, m), dtype=torch.float64, device="cuda")
            st = torch.cuda.Stream()
            st.wait_stream(torch.cuda.current_stream())
            ctx = ozg.Context(1 << 30, stream=st)
            ctx.set_autotune(capture, str(path))
            call = lambda: ctx.dgemm("N", "N", m, n, k, 1.0, A, m, B, k, 0.0, C, m, s)
            if capture:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=st):
                    call()
                graph.replay()
            else:
                call()
            torch.cuda.synchronize()
            ctx.close()
            out.append(C)
        assert torch.equal(out[-1], out[-2])
    assert not path.exists() or path.read_text() == ""
