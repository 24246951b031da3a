"""The register-resident LU panel at the sizes where its layout changes: one
block up to 384 rows, then clusters with one to four rows a thread, panels
narrower than 32 columns, and the pivot rule on ties and NaNs (the first row
of largest magnitude; a column of NaNs keeps its row).  Every expected pivot
follows from how the matrix was built."""

import numpy as np
import pytest

from paper_1608_05265_gb300 import synth

from gpu_util import dev

pytestmark = pytest.mark.gpu

EPS32 = 2.0 ** -24


@pytest.fixture(scope="module")
def h():
    import torch
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    hd = gbgemm.Handle(0)
    hd.set_stream(torch.cuda.current_stream())
    yield hd
    hd.close()


def factor(h, A):
    import torch
    n, lda = A.shape[0], A.shape[0] + 1
    d = dev(synth.place_colmajor(np.ascontiguousarray(A.T).reshape(-1), n, n, lda))
    ipiv = torch.zeros(n, dtype=torch.int32, device="cuda")
    info = torch.full((1,), -7, dtype=torch.int32, device="cuda")
    h.sgetrf(n, d, lda, ipiv, info)
    torch.cuda.synchronize()
    assert h.get_device_status() == 0
    out = d.cpu().numpy()
    assert synth.padding_is_sentinel(out, n, n, lda)
    return synth.logical(out, n, n, lda), ipiv.cpu().numpy(), int(info.item())


def pivots_of(order):
    """LAPACK's exchanges that bring row order[i] to position i, in order."""
    n = len(order)
    at, row = np.arange(n), np.arange(n)  # position of each row, row at each position
    ipiv = np.empty(n, dtype=np.int64)
    for j in range(n):
        p = at[order[j]]
        ipiv[j] = p + 1
        row[j], row[p] = row[p], row[j]
        at[row[j]], at[row[p]] = j, p
    return ipiv


@pytest.mark.parametrize("n", [31, 33, 97, 384, 385, 1030, 2049, 2081, 4130])
def test_pivots_fixed_by_construction(h, n):
    rng = np.random.default_rng(n)
    s = 1.0 / np.sqrt(n)
    L = np.tril(rng.uniform(-0.5 * s, 0.5 * s, (n, n)), -1) + np.eye(n)
    U = np.triu(rng.uniform(-s, s, (n, n)), 1) + np.diag(rng.uniform(1, 2, n))
    order = rng.permutation(n)
    A = np.empty((n, n))
    A[order] = L @ U
    lu, ipiv, info = factor(h, A.astype(np.float32))
    assert info == 0
    assert np.array_equal(ipiv, pivots_of(order))
    # well conditioned, entries O(1): a few n eps between FP32 and exact factors
    assert np.max(np.abs(lu - (np.tril(L, -1) + U))) <= 16 * n * EPS32


@pytest.mark.parametrize("n", [40, 385, 700, 2500])
def test_ties_take_the_first_row(h, n):
    """L and U with a few entries of +-1 per column: every product and partial
    sum is a small integer, many multipliers are +-1, so the pivot ties with
    rows below and must stay; the factors are exact."""
    rng = np.random.default_rng(n)
    L, U = np.eye(n), np.eye(n)
    for j in range(n - 1):
        rows = rng.integers(j + 1, n, 3)
        L[rows, j] = rng.choice([-1.0, 1.0], 3)
        U[j, rng.integers(j + 1, n)] = rng.choice([-1.0, 1.0])
    lu, ipiv, info = factor(h, (L @ U).astype(np.float32))
    assert info == 0
    assert np.array_equal(ipiv, np.arange(1, n + 1))
    assert np.array_equal(lu, (np.tril(L, -1) + U).astype(np.float32))


@pytest.mark.parametrize("n", [50, 600])
def test_nan_columns_keep_their_rows(h, n):
    A = np.random.default_rng(n).uniform(-1, 1, (n, n)).astype(np.float32)
    A[:, 0] = np.nan
    lu, ipiv, info = factor(h, A)
    assert info == 0
    assert np.array_equal(ipiv, np.arange(1, n + 1))
    assert np.all(np.isnan(lu[1:, :])) and np.array_equal(lu[0, 1:], A[0, 1:])
