"""sgemv between the shapes its kernels were tuned on: results against FP64 at
the edges of the steps, and times that do not jump there."""

import numpy as np
import pytest

from paper_1608_05265_gb300 import synth

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    import torch
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    hd = gbgemm.Handle(0)
    hd.set_stream(torch.cuda.current_stream())
    yield hd
    hd.close()


def check(h, trans, m, n, pad, incx=1):
    import torch
    ld = (m + 3) // 4 * 4 + pad
    A = synth.uniform_pm1(synth.draws(97, 1, n * ld)).astype(np.float32)
    lx, ly = (n, m) if trans == "N" else (m, n)
    x = synth.uniform_pm1(synth.draws(97, 2, lx * abs(incx))).astype(np.float32)
    y = synth.uniform_pm1(synth.draws(97, 3, ly)).astype(np.float32)
    dy = dev(y)
    h.sgemv(trans, m, n, 1.25, dev(A), ld, dev(x), incx, -0.5, dy, 1)
    torch.cuda.synchronize()
    a = A.reshape(n, ld)[:, :m].T.astype(np.float64)
    xs = x[::abs(incx)][:lx].astype(np.float64)
    xs = xs if incx > 0 else xs[::-1]
    op = a if trans == "N" else a.T
    want = 1.25 * op @ xs - 0.5 * y.astype(np.float64)
    bound = 2 * lx * 2.0 ** -24 * (1.25 * np.abs(op) @ np.abs(xs) + 0.5 * np.abs(y))
    assert np.all(np.abs(dy.cpu().numpy() - want) <= bound)


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("m,n", [(1023, 40), (1024, 7), (1025, 700), (1100, 2500), (2049, 33), (2304, 12), (2305, 12),
                                 (4097, 610), (4100, 2500), (6001, 4)])
def test_transposed(h, m, n, pad):
    check(h, "T", m, n, pad)
    check(h, "T", m, n, pad, incx=-2)


def timed(h, trans, m, n, pad):
    import torch
    ld = (m + 3) // 4 * 4 + pad
    calls = []
    for _ in range(3):
        A = torch.rand(n, ld, device="cuda")
        x = torch.rand(n if trans == "N" else m, device="cuda")
        y = torch.rand(m if trans == "N" else n, device="cuda")
        calls.append(lambda A=A, x=x, y=y: h.sgemv(trans, m, n, 1.0, A, ld, x, 1, 0.5, y, 1))
    best = 1e30
    for _ in range(10):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for i in range(30):
            calls[i % 3]()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


def test_transposed_time_does_not_jump(h):
    """One row more than a step of four rows a thread cost 1.56 times the time."""
    assert timed(h, "T", 1100, 16384, 0) <= 1.3 * timed(h, "T", 1000, 16384, 0)
    assert timed(h, "T", 1025, 4096, 0) <= 1.2 * timed(h, "T", 1025, 4096, 1)


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("m,n", [(1025, 1), (1030, 20), (1536, 9), (2050, 64), (3000, 65), (5003, 3), (16384, 20)])
def test_not_transposed_few_columns(h, m, n, pad):
    check(h, "N", m, n, pad)
    check(h, "N", m, n, pad, incx=-3)


def test_few_columns_cost_no_more_aligned_than_not(h):
    """Blocks of 1024 rows took 1.3 times as long as those of unaligned columns."""
    assert timed(h, "N", 16384, 20, 0) <= 1.15 * timed(h, "N", 16384, 20, 1)
    assert timed(h, "N", 4097, 20, 0) <= 1.15 * timed(h, "N", 4097, 20, 1)
