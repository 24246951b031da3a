"""The split path without a packing pass: K-vectors whose first nonzero step
holds a value so small that a later one, scaled by its exponent, is beyond
FP32.  The result has to be that of exponents from the true maxima, in every
way an operand is read, with two and three parts, with k slices in a cluster
and through the workspace, and for strided batches."""

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


def vectors(rows, k, small, large):
    """rows x k: every chunk of 32 k begins with `small` (so that whichever
    slice and step a vector is first seen in holds nothing else), one entry of
    every vector is `large`, anywhere, and all others are zero: no smaller
    neighbour of a `large` entry tells of it.  Every fifth vector is `small`
    throughout, every eleventh ordinary."""
    x = np.zeros((rows, k), dtype=np.float32)
    x[:, ::32] = small
    i = np.arange(rows)
    x[i, (37 * i + 100) % k] = large
    x[::5] = small
    u = synth.uniform_pm1(synth.draws(81, 1, rows * k)).reshape(rows, k).astype(np.float32)
    x[::11] = u[::11]
    return x


@pytest.mark.parametrize("small,large", [(1e-40, 1.0), (2.0 ** -100, 2.0 ** 40), (-(2.0 ** -149), -3.0)])
@pytest.mark.parametrize("mode", ["rows", "vec", "scalar"])
@pytest.mark.parametrize("which", ["A", "B"])
@pytest.mark.parametrize("m,n,k,want", [(200, 150, 300, 1), (200, 150, 700, 1), (300, 260, 2048, 1),
                                        (500, 500, 16384, 2)])
def test_scaled_value_beyond_fp32(h, which, mode, m, n, k, want, small, large):
    import torch
    rows = m if which == "A" else n
    x = vectors(rows, k, small, large)
    y = synth.uniform_pm1(synth.draws(82, 2, (m + n - rows) * k)).reshape(m + n - rows, k).astype(np.float32)
    ld = rows if mode == "rows" else k + (1 if mode == "scalar" else 0)
    if mode == "rows":
        X = np.ascontiguousarray(x.T).reshape(-1)   # rows contiguous
    else:
        X = np.zeros((rows, ld), dtype=np.float32)  # k contiguous
        X[:, :k] = x
        X = X.reshape(-1)
    Y = y.reshape(-1)
    trans = "N" if (mode == "rows") == (which == "A") else "T"
    args = ((trans, "N", m, n, k, 1.0, X, ld, Y, k) if which == "A"
            else ("T", trans, m, n, k, 1.0, Y, k, X, ld))
    C = synth.uniform_matrix(83, 4, m, n, m)
    h.profile_begin()
    check_full(h, AUTO, *args, 0.5, C, m, nthreads=4)
    torch.cuda.synchronize()
    assert h.profile_end()[2] == want and h.last_path() == SPLIT


@pytest.mark.parametrize("ta", ["N", "T"])
def test_strided_batch(h, ta):
    import torch
    m, n, k, batch = 130, 70, 600, 9
    x = np.stack([np.roll(vectors(m, k, 1e-40, 1.0), z, axis=0) for z in range(batch)])
    A = np.ascontiguousarray(x.transpose(0, 2, 1) if ta == "N" else x)
    lda = m if ta == "N" else k
    B = synth.uniform_pm1(synth.draws(84, 2, batch * n * k)).astype(np.float32)
    dA, dB, dC = dev(A.reshape(-1)), dev(B), torch.zeros(batch * m * n, device="cuda")
    h.set_path(AUTO)
    h.sgemm_strided_batched(ta, "N", m, n, k, 1.0, dA, lda, m * k, dB, k, k * n, 0.0, dC, m, m * n, batch)
    out = dC.cpu().numpy().reshape(batch, n, m)
    zero = np.zeros(m * n, dtype=np.float32)
    for z in range(batch):
        c64, bnd = O.gemm_f64(ta, "N", m, n, k, 1.0, A[z].reshape(-1), lda, B[z * n * k:], k, 0.0, zero, m)
        assert O.error_ratio(out[z].T, c64, bnd) <= 1.0
