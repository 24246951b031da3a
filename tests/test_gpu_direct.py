"""The split path without a packing pass (path AUTO, small outputs or long k):
one kernel launch, or two when k slices are reduced through the workspace.
Every way an operand is read (rows contiguous, k contiguous and aligned, k
contiguous at any alignment), tile edges, k remainders, cluster and workspace
slices, strided batches, and the scaling of badly scaled vectors: exponents
from the first nonzero step, kept, given late, or replaced by those of the
true maxima.  Each against the FP64 oracle under the componentwise bound; the
packed path (SPLIT forced, at least two launches) on the same inputs meets the
same bound, so both answer every form alike."""

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


def launches(h, fn):
    import torch
    h.profile_begin()
    r = fn()
    torch.cuda.synchronize()
    return r, h.profile_end()[2]


def check_both(h, *args, want=1):
    r, n = launches(h, lambda: check_full(h, AUTO, *args, nthreads=4))
    assert n == want and h.last_path() == SPLIT, f"{n} launches"
    _, n = launches(h, lambda: check_full(h, SPLIT, *args, nthreads=4))
    assert n >= 2
    return r


@pytest.mark.parametrize("ta,tb,pad", [("N", "N", 0), ("N", "N", 1), ("T", "N", 0), ("T", "N", 3), ("N", "T", 2),
                                       ("T", "T", 0), ("T", "T", 5)])
@pytest.mark.parametrize("m,n,k", [
    (1, 1, 128), (129, 65, 129), (256, 256, 256), (200, 130, 511),     # three parts
    (128, 64, 512), (127, 191, 545), (257, 260, 1001), (700, 310, 640)  # two parts
])
def test_every_operand_form(h, ta, tb, pad, m, n, k):
    A, lda, B, ldb, C, ldc = synth.gemm_problem("uniform", 61, ta, tb, m, n, k, pad=pad)
    check_both(h, ta, tb, m, n, k, 1.5, A, lda, B, ldb, -0.25, C, ldc)


def test_workspace_slices(h):
    """A long k with few tiles: raw tiles of every slice, then the reduction."""
    m, n, k = 500, 500, 16400
    A, lda, B, ldb, C, ldc = synth.gemm_problem("uniform", 62, "N", "T", m, n, k, pad=4)
    check_both(h, "N", "T", m, n, k, -1.0, A, lda, B, ldb, 0.5, C, ldc, want=2)


def vectors(kind, seed, rows, k, span):
    """rows x k entries whose K-vectors (rows) are badly scaled in a way, by
    at most 2^+-span (60 for op(A) and 40 for op(B): the results stay normal
    FP32 numbers, below which no output could meet the bound)."""
    x = synth.uniform_pm1(synth.draws(seed, 1, rows * k)).reshape(rows, k).astype(np.float64)
    e = synth.int_range(synth.draws(seed, 2, rows), -span, span).astype(np.int64)
    if kind == "rows":      # every vector a scale of its own
        x = np.ldexp(x, e[:, None])
    elif kind == "late":    # zero at first, badly scaled after; some vectors zero throughout
        x = np.ldexp(x, e[:, None])
        x[::3, : k // 2] = 0.0
        x[1::7] = 0.0
    elif kind == "grow":    # far larger after the first steps: exponents of the true maxima
        x = np.ldexp(x, -60)
        x[:, k // 2:] = np.ldexp(x[:, k // 2:], 70)
    elif kind == "shrink":  # the first steps hold the largest entries
        x[:, k // 2:] = np.ldexp(x[:, k // 2:], -70)
    return x.astype(np.float32)


@pytest.mark.parametrize("kind", ["rows", "late", "grow", "shrink"])
@pytest.mark.parametrize("ta,m,n,k,want", [("N", 200, 150, 300, 1), ("T", 200, 150, 700, 1), ("N", 300, 260, 2048, 1),
                                           ("T", 500, 500, 16384, 2)])
def test_badly_scaled_vectors(h, kind, ta, m, n, k, want):
    X = vectors(kind, 63, m, k, 60)
    A = np.ascontiguousarray(X.T if ta == "N" else X).reshape(-1)
    B = np.ascontiguousarray(vectors(kind if kind in ("rows", "late") else "rows", 64, n, k, 40)).reshape(-1)
    C = synth.uniform_matrix(65, 4, m, n, m)
    check_both(h, ta, "N", m, n, k, 1.0, A, m if ta == "N" else k, B, k, 0.0, C, m, want=want)


def test_nonfinite_positions(h):
    m, n, k = 150, 96, 640
    A, lda, B, ldb, C, ldc = synth.gemm_problem("uniform", 66, "T", "N", m, n, k)
    A, B = A.copy(), B.copy()
    A[5 * lda + 7] = np.inf
    A[140 * lda + 600] = np.nan
    B[33 * ldb + 2] = -np.inf
    import torch
    h.set_path(AUTO)
    dC = dev(C)
    h.sgemm("T", "N", m, n, k, 1.0, dev(A), lda, dev(B), ldb, 0.5, dC, ldc)
    torch.cuda.synchronize()
    c64, _ = O.gemm_f64("T", "N", m, n, k, 1.0, A, lda, B, ldb, 0.5, C, ldc)
    assert np.array_equal(np.isfinite(synth.logical(dC.cpu().numpy(), m, n, ldc)), np.isfinite(c64))


@pytest.mark.parametrize("m,n,k,batch,pad", [(192, 256, 700, 9, 0), (70, 100, 200, 33, 1), (130, 60, 1030, 5, 3)])
def test_strided_batch_deterministic_and_beta_zero(h, m, n, k, batch, pad):
    import torch
    lda, ldb, ldc = m + pad, n + pad, m + pad
    sa, sb, sc = lda * k + 5, ldb * k + 3, ldc * n + 7
    draw = lambda s, count: synth.uniform_pm1(synth.draws(67, s, count)).astype(np.float32)
    A, B = draw(0, sa * batch), draw(2, sb * batch)
    dA, dB = dev(A), dev(B)
    h.set_path(AUTO)
    outs = []
    for _ in range(2):
        dC = torch.full((sc * batch,), float("nan"), device="cuda")  # beta = 0 does not read C
        call = lambda: h.sgemm_strided_batched("N", "T", m, n, k, 2.0, dA, lda, sa, dB, ldb, sb, 0.0, dC, ldc, sc, batch)
        assert launches(h, call)[1] == 1
        outs.append(dC.cpu().numpy())
    assert h.get_device_status() == 0
    assert np.array_equal(outs[0].view(np.uint32), outs[1].view(np.uint32))
    zero = np.zeros(ldc * n, dtype=np.float32)
    for z in range(batch):
        c64, bnd = O.gemm_f64("N", "T", m, n, k, 2.0, A[z * sa:], lda, B[z * sb:], ldb, 0.0, zero, ldc)
        full = outs[0][z * sc: z * sc + ldc * n].reshape(n, ldc)
        assert O.error_ratio(full[:, :m].T, c64, bnd) <= 1.0
        assert np.all(np.isnan(full[:, m:])) and np.all(np.isnan(outs[0][z * sc + ldc * n:(z + 1) * sc]))
