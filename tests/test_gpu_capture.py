"""Calls as programmatic dependents of whatever the caller queued before them:
captured in a CUDA graph, after a copy and after a wait for another stream's
event, each bitwise as an eager call on its own."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    hd = gbgemm.Handle(0)
    yield hd
    hd.close()


# path, then SIMT, direct (one launch and workspace slices), packed, packed with
# k slices, packed pair tiles
CALLS = [(0, 300, 200, 60), (0, 256, 256, 256), (0, 500, 500, 16400), (2, 300, 200, 200), (2, 300, 200, 4000),
         (2, 700, 900, 1000)]


def operands(m, n, k):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(m + k)
    uni = lambda *s: torch.empty(*s, device="cuda").uniform_(-1.0, 1.0, generator=g)
    return uni(k, m), uni(n, k), uni(n, m)


def call(h, stream, path, m, n, k, A, B, C):
    h.set_stream(stream)
    h.set_path(path)
    h.sgemm("N", "N", m, n, k, 1.5, A, m, B, k, -0.25, C, m)


@pytest.mark.parametrize("path,m,n,k", CALLS)
def test_graph_replay_after_a_kernel_and_a_copy(h, path, m, n, k):
    import torch
    A0, B, C0 = operands(m, n, k)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        want = C0.clone()
        call(h, s, path, m, n, k, A0, B, want)  # workspace and kernels are there before the capture
        A, C = torch.zeros_like(A0), torch.zeros_like(C0)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            A.copy_(A0)              # a copy,
            C.copy_(C0)
            A.mul_(2.0).mul_(0.5)    # kernels, and the call right behind them
            call(h, s, path, m, n, k, A, B, C)
        for _ in range(3):
            A.zero_()
            C.fill_(float("nan"))
            graph.replay()
            s.synchronize()
            assert torch.equal(C, want)
    assert h.get_device_status() == 0


@pytest.mark.parametrize("path,m,n,k", CALLS)
def test_after_an_event_of_another_stream(h, path, m, n, k):
    import torch
    A0, B, C0 = operands(m, n, k)
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    want = C0.clone()
    call(h, torch.cuda.current_stream(), path, m, n, k, A0, B, want)
    A, C = torch.zeros_like(A0), C0.clone()
    big = torch.zeros(64 << 20, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        for _ in range(8):
            big.add_(1.0)            # some time passes before A is written
        A.copy_(A0)
        e = torch.cuda.Event()
        e.record(other)
    with torch.cuda.stream(s):
        s.wait_event(e)
        call(h, s, path, m, n, k, A, B, C)
    torch.cuda.synchronize()
    assert torch.equal(C, want)
    assert h.get_device_status() == 0
