"""The parts of the triangular solves that a factorisation's own pivots and
factors do not reach: row exchanges in every order (run many at a time on the
GPU), and the back substitution's quotients, which have to be the correctly
rounded ones over the whole exponent range."""

import numpy as np
import pytest

from paper_1608_05265_gb300 import synth

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


def solve(h, lu, ipiv, b):
    """x of the packed factors lu (n x n, row major view) for columns b (n x nrhs)."""
    import torch
    n, nrhs = b.shape
    d = torch.from_numpy(np.asfortranarray(lu.astype(np.float32)).ravel(order="F").copy()).cuda()
    p = torch.from_numpy(ipiv.astype(np.int32)).cuda()
    x = torch.from_numpy(np.asfortranarray(b.astype(np.float32)).ravel(order="F").copy()).cuda()
    h.sgetrs(n, nrhs, d, n, p, x, n)
    torch.cuda.synchronize()
    assert h.get_device_status() == 0
    return x.cpu().numpy().reshape(nrhs, n).T


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("order", ["any", "near", "same", "chain", "back", "outside"])
@pytest.mark.parametrize("n", [1, 31, 33, 64, 200, 1100])
def test_row_exchanges_in_order(h, n, order, nrhs):
    j = np.arange(n)
    u = synth.int_range(synth.draws(71, n, n), 0, n - 1).astype(np.int64) if n > 1 else np.zeros(1, np.int64)
    p = {"any": u, "near": (j + u % 5).clip(max=n - 1), "same": np.full(n, n // 2), "chain": (j + 1).clip(max=n - 1),
         "back": n - 1 - j, "outside": np.where(u % 3 == 0, n + u, np.where(u % 3 == 1, -1 - u, u))}[order]
    b = np.arange(1, n * nrhs + 1, dtype=np.float64).reshape(n, nrhs)
    want = b.copy()
    for r, q in enumerate(p):
        if 0 <= q < n:
            want[[r, q]] = want[[q, r]]
    got = solve(h, np.eye(n), p + 1, b)  # unit factors: the solve only exchanges
    assert np.array_equal(got, want.astype(np.float32))


@pytest.mark.parametrize("span_d,span_b", [(0, 0), (20, 20), (59, 59), (61, 61), (100, 20), (20, 100), (62, 64)])
@pytest.mark.parametrize("nrhs", [1, 2])
@pytest.mark.parametrize("n", [5, 32, 300])
def test_quotients_are_correctly_rounded(h, n, nrhs, span_d, span_b):
    def vec(slot, count, span):
        m = synth.uniform_pm1(synth.draws(72, slot, count)).astype(np.float32)
        e = synth.int_range(synth.draws(73, slot, count), -span, span).astype(np.int64)
        m = np.where(np.abs(m) < 0.5, np.copysign(m + np.copysign(np.float32(0.5), m), m), m).astype(np.float32)
        return np.ldexp(m, e).astype(np.float32)
    d = vec(1, n, span_d)
    b = vec(2, n * nrhs, span_b).reshape(n, nrhs)
    b[n // 2] = 0.0
    got = solve(h, np.diag(d), np.arange(1, n + 1), b)
    assert np.array_equal(got, b / d[:, None])
