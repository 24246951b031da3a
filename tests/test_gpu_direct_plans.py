"""Every instance and cluster shape of the split path without a packing pass,
in the three ways an operand is read, against the FP64 oracle."""

import numpy as np
import pytest

from oracle import oracle as O
from paper_1608_05265_gb300 import synth

from gpu_util import SPLIT, dev
from test_direct_plan import SHAPES

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


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ta,tb,pad", [("N", "T", 0), ("T", "N", 0), ("T", "N", 1)])
def test_against_the_oracle(h, shape, ta, tb, pad):
    import torch
    m, n, k, batch = shape
    (ar, ac), (br, bc) = synth.op_shape(ta, m, k), synth.op_shape(tb, k, n)
    lda, ldb = ar + pad, br + pad
    draw = lambda s, count: synth.uniform_pm1(synth.draws(96, s, count)).astype(np.float32)
    A, B, C = draw(1, batch * lda * ac), draw(2, batch * ldb * bc), draw(3, batch * m * n)
    dC = dev(C)
    h.set_path(0)
    h.profile_begin()
    if batch == 1:
        h.sgemm(ta, tb, m, n, k, 1.5, dev(A), lda, dev(B), ldb, -0.25, dC, m)
    else:
        h.sgemm_strided_batched(ta, tb, m, n, k, 1.5, dev(A), lda, lda * ac, dev(B), ldb, ldb * bc, -0.25, dC, m,
                                m * n, batch)
    torch.cuda.synchronize()
    assert h.get_device_status() == 0 and h.last_path() == SPLIT
    assert h.profile_end()[2] == (1 if SHAPES[shape][3] else 2)
    out = dC.cpu().numpy()
    for z in range(batch):
        c64, bnd = O.gemm_f64(ta, tb, m, n, k, 1.5, A[z * lda * ac:], lda, B[z * ldb * bc:], ldb, -0.25,
                              C[z * m * n:], m, nthreads=4)
        assert O.error_ratio(out[z * m * n:(z + 1) * m * n].reshape(n, m).T, c64, bnd) <= 1.0
