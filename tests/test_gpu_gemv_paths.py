"""The sgemv kernels' variants (16-byte loads where every column is aligned,
4-byte loads else; rows per block by the length of y) at the sizes where they
change and at ragged ends: rows that end inside a thread's four, columns that
end inside a step, slices of a few columns or rows, an A that starts off a
16-byte boundary."""

import numpy as np
import pytest

from test_gpu_gemv import check_gemv, dev, h  # noqa: F401  (h: the module's handle)
from oracle import oracle as O
from paper_1608_05265_gb300 import synth

pytestmark = pytest.mark.gpu

SIZES = [(1, 9), (3, 130), (255, 33), (256, 1000), (257, 1001), (510, 77), (1023, 640), (1024, 90), (1025, 2049),
         (1027, 35), (2050, 1500), (4099, 4097), (9000, 70), (70, 9000), (2047, 12), (12, 2047)]


@pytest.mark.parametrize("trans", ["N", "T"])
@pytest.mark.parametrize("m,n", SIZES)
def test_aligned_and_unaligned_columns(h, trans, m, n):  # noqa: F811
    up = -m % 4
    for pad in (up, up + 4, up + 1):  # two leading dimensions of whole 16 bytes, one not
        check_gemv(h, trans, m, n, 1.5, -0.25, pad=pad, seed=81)
    check_gemv(h, trans, m, n, 1.0, 0.0, incx=-2, incy=3, pad=up, seed=82)


@pytest.mark.parametrize("trans", ["N", "T"])
@pytest.mark.parametrize("off", [1, 2, 3, 4])
def test_start_off_a_boundary(h, trans, off):  # noqa: F811
    import torch
    m, n, lda = 1500, 900, 1504
    A = synth.uniform_matrix(83, 0, m, n, lda)
    lx, ly = (m, n) if trans == "T" else (n, m)
    x = synth.uniform_pm1(synth.draws(83, 2, lx)).astype(np.float32)
    buf = torch.zeros(A.size + 8, device="cuda")
    buf[off:off + A.size] = dev(np.ravel(A))
    dy = torch.zeros(ly, device="cuda")
    h.sgemv(trans, m, n, 1.0, buf[off:], lda, dev(x), 1, 0.0, dy, 1)
    torch.cuda.synchronize()
    c64, bnd = O.gemm_f64(trans, "N", ly, 1, lx, 1.0, A, lda, x, lx, 0.0, np.zeros(ly, np.float32), ly)
    assert O.error_ratio(dy.cpu().numpy().reshape(ly, 1), c64, bnd) <= 1.0
