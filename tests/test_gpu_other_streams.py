"""GPU test of what a large single-map call leaves to other streams: its CTAs of
1024 threads take an SM each, and a small kernel on another stream has to fit beside
them.  Small kernels launched while a long row of calls runs are done well
before the row is; when the calls' registers fill the SMs, they are done only
after it."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["rsmss_filter", "rbsm_visibility"])
def test_small_kernels_run_beside_large_calls(what):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1711_07793_gb300 import api
    g = torch.Generator(device="cuda").manual_seed(1)
    w, h = 3840, 2160
    n = w * h
    depth = torch.where(torch.rand((1024, 1024), generator=g, device="cuda") < 0.003, 0.3, 1.0)
    tex = api.MapTexture(depth)
    xyz = [(torch.arange(w, device="cuda") / w * 0.8 + 0.1).repeat(h),
           (torch.arange(h, device="cuda") / h * 0.5 + 0.1).repeat_interleave(w), torch.full((n,), 0.75, device="cuda")]
    vis = torch.empty(n, device="cuda")
    small, out = torch.rand(1 << 20, device="cuda"), torch.empty(1 << 20, device="cuda")
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(two):
        torch.mul(small, 2.0, out=out)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=two):
            for _ in range(200):
                torch.mul(small, 2.0, out=out)
    begin, calls, others = (torch.cuda.Event(enable_timing=True) for _ in range(3))

    def run(rounds):
        torch.cuda.synchronize()
        with torch.cuda.stream(one):
            begin.record()
            for _ in range(rounds):
                getattr(api, what)(tex, *xyz, vis=vis)
            calls.record()
        with torch.cuda.stream(two):
            two.wait_event(begin)
            graph.replay()
            others.record()
        torch.cuda.synchronize()
        return begin.elapsed_time(calls), begin.elapsed_time(others)

    run(5)
    row, beside = sorted((run(100) for _ in range(5)), key=lambda t: t[1] / t[0])[2]
    assert beside < 0.75 * row, (row, beside)
