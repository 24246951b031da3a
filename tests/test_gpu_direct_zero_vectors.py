"""The split path without a packing pass on operands whose K-vectors are zero
in the first steps: throughout (padded or masked operands), up to some k
(triangular, banded), well or badly scaled after, or infinite.  They cost what
dense operands cost, and the results are those of exponents from the true
maxima."""

import numpy as np
import pytest

from oracle import oracle as O
from paper_1608_05265_gb300 import synth

from gpu_util import SPLIT, check_full, dev

pytestmark = pytest.mark.gpu

AUTO = 0


@pytest.fixture(scope="module")
def h():
    import torch
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    hd = gbgemm.Handle(0)
    hd.set_stream(torch.cuda.current_stream())
    yield hd
    hd.close()


def vectors(seed, rows, k, span):
    """rows x k, by row: zero up to some k (any step's edge or middle), then at
    a scale of its own within 2^+-span, or well scaled, or one single entry;
    some zero throughout and some dense."""
    x = synth.uniform_pm1(synth.draws(seed, 1, rows * k)).reshape(rows, k).astype(np.float64)
    e = synth.int_range(synth.draws(seed, 2, rows), -span, span).astype(np.int64)
    first = np.array([31, 32, 33, 63, 64, 65, 95, 127, 128, 129, 200, k // 2, k - 1])
    for i in range(rows):
        kind = i % 5
        if kind == 0:
            x[i] = 0.0
        elif kind < 4:
            x[i, : min(first[(i // 5) % len(first)], k - 1)] = 0.0
            if kind == 1:
                x[i] = np.ldexp(x[i], int(e[i]))
            elif kind == 2:
                x[i, (7 * i) % k + 1:] = 0.0
    return x.astype(np.float32)


def operand(x, mode):
    """Stored form of the K-vectors x and its leading dimension and transposition."""
    rows, k = x.shape
    if mode == "rows":
        return np.ascontiguousarray(x.T).reshape(-1), rows, False
    ld = k + (1 if mode == "scalar" else 0)
    X = np.zeros((rows, ld), dtype=np.float32)
    X[:, :k] = x
    return X.reshape(-1), ld, True


@pytest.mark.parametrize("ma", ["rows", "vec", "scalar"])
@pytest.mark.parametrize("mb", ["rows", "vec", "scalar"])
@pytest.mark.parametrize("m,n,k,want", [(200, 150, 300, 1), (130, 70, 700, 1), (300, 260, 2048, 1), (500, 500, 16384, 2)])
def test_results(h, ma, mb, m, n, k, want):
    import torch
    A, lda, ta = operand(vectors(91, m, k, 60), ma)
    B, ldb, nb = operand(vectors(92, n, k, 40), mb)
    C = synth.uniform_matrix(93, 4, m, n, m)
    h.profile_begin()
    check_full(h, AUTO, "T" if ta else "N", "N" if nb else "T", m, n, k, 1.0, A, lda, B, ldb, 0.0, C, m, nthreads=4)
    torch.cuda.synchronize()
    assert h.profile_end()[2] == want and h.last_path() == SPLIT


@pytest.mark.parametrize("mode", ["rows", "vec", "scalar"])
def test_infinity_after_zeros(h, mode):
    import torch
    m, n, k = 150, 96, 640
    x = vectors(94, m, k, 60)
    x[7] = 0.0
    x[7, 300] = np.inf
    x[8] = 0.0
    x[8, 301], x[8, 400] = 2.0 ** -60, np.nan
    A, lda, ta = operand(x, mode)
    B = synth.uniform_pm1(synth.draws(95, 2, n * k)).astype(np.float32)
    C = np.zeros(m * n, dtype=np.float32)
    h.set_path(AUTO)
    dC = dev(C)
    h.sgemm("T" if ta else "N", "N", m, n, k, 1.0, dev(A), lda, dev(B), k, 0.0, dC, m)
    torch.cuda.synchronize()
    c64, bnd = O.gemm_f64("T" if ta else "N", "N", m, n, k, 1.0, A, lda, B, k, 0.0, C, m)
    got = synth.logical(dC.cpu().numpy(), m, n, m)
    assert np.array_equal(np.isfinite(got), np.isfinite(c64))
    keep = [i for i in range(m) if i not in (7, 8)]
    assert O.error_ratio(got[keep], c64[keep], bnd[keep]) <= 1.0


@pytest.mark.parametrize("ta,pad", [("N", 0), ("T", 0), ("T", 1)])
@pytest.mark.parametrize("step", [2, 64])
def test_zero_rows_cost_no_more_than_dense_ones(h, ta, pad, step):
    """Every second row, or one in 64, of op(A) zero: within a quarter of the
    time of a dense operand (a barrier a step and an atomic a value took up to
    twice its time)."""
    import torch
    m = n = 512
    k = 65536
    ar, ac = (m, k) if ta == "N" else (k, m)
    B, C = torch.rand(n, k, device="cuda") - 0.5, torch.zeros(n, m, device="cuda")
    times = {}
    h.set_path(AUTO)
    for zero in (False, True):
        A = torch.rand(ac, ar + pad, device="cuda") - 0.5
        if zero:
            (A[:, ::step] if ta == "N" else A[::step]).zero_()
        call = lambda: h.sgemm(ta, "N", m, n, k, 1.0, A, ar + pad, B, k, 0.0, C, m)
        best = 1e30
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(10):
                call()
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times[zero] = best
    assert times[True] <= 1.25 * times[False], times
