"""The sgemm binding's two ways into the library (plain arguments straight to
ctypes, others converted first) give the same call."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("conv", ["numpy", "float_dims", "pointers", "bytes_flags", "lower"])
def test_converted_arguments_make_the_same_call(conv):
    import torch
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    h = gbgemm.Handle(0)
    h.set_stream(torch.cuda.current_stream())
    m, n, k = 70, 50, 40
    A, B = torch.rand(m, k, device="cuda"), torch.rand(n, k, device="cuda")  # T N, column-major
    want, got = torch.zeros(n, m, device="cuda"), torch.zeros(n, m, device="cuda")
    h.sgemm("T", "N", m, n, k, 1.5, A, k, B, k, 0.0, want, m)
    ta, tb, a, b, c, alpha = "T", "N", A, B, got, 1.5
    if conv == "numpy":
        m, n, k, alpha = np.int64(m), np.int32(n), np.int64(k), np.float32(alpha)
    elif conv == "float_dims":
        m = float(m)
    elif conv == "pointers":
        a, b, c = A.data_ptr(), B.data_ptr(), got.data_ptr()
    elif conv == "bytes_flags":
        ta, tb = b"T", b"N"
    else:
        ta, tb = "t", "n"
    assert h.sgemm(ta, tb, m, n, k, alpha, a, k, b, k, 0.0, c, m) == 0
    assert torch.equal(got, want)
    with pytest.raises(gbgemm.GbgemmError):
        h.sgemm("X", "N", m, n, k, alpha, a, k, b, k, 0.0, c, m)
    assert h.sgemm("X", "N", 1, 1, 1, 1.0, A, 1, B, 1, 0.0, got, 1, check=False) == -1
    h.close()
