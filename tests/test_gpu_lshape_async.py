"""On the L the mixed-precision cycle, the float32 step and the float32 restriction run no planar level: they return without
waiting for the stream, and the two float32 calls can be captured into a graph."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    from paper_1502_04070_gb300.solver import Solver
    n = 128
    gen = torch.Generator(device="cuda").manual_seed(9)
    u, f = (torch.rand(2, 2 * n + 1, 2 * n + 1, generator=gen, device="cuda") - 0.5 for _ in range(2))
    p, g = (torch.rand(n + 1, n + 1, generator=gen, device="cuda") - 0.5 for _ in range(2))
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    S = Solver(7, 1.0, precision="mixed", domain="lshape", coarse_level=1, stream=stream)
    yield S, stream, (u, p, f, g), [t.double() for t in (u, p, f, g)]
    torch.cuda.synchronize()
    S.close()


def test_calls_return_before_the_work_ahead_of_them(setup):
    S, stream, x32, x64 = setup
    calls = [lambda: S.cycle(*x64), lambda: S.smooth_f32(*x32, 1), lambda: S.residual_restrict_f32(*x32)]
    with torch.cuda.stream(stream):
        for call in calls:
            call()   # graphs are built by the first call
            torch.cuda.synchronize()
            ahead = torch.cuda.Event()
            torch.cuda._sleep(400_000_000)   # about 0.2 s
            ahead.record()
            call()
            assert not ahead.query()
            torch.cuda.synchronize()


def test_float32_calls_are_capturable(setup):
    S, stream, x32, _ = setup
    u, p, f, g = x32
    with torch.cuda.stream(stream):
        v, q = u.clone(), p.clone()
        want = [t.clone() for t in S.smooth_f32(v, q, f, g, 2)] + list(S.residual_restrict_f32(u, p, f, g))
        w, r = u.clone(), p.clone()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            S.smooth_f32(w, r, f, g, 2)
            fc, gc = S.residual_restrict_f32(u, p, f, g)
        graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, (w, r, fc, gc)))
