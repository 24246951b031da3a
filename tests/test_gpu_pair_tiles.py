"""Tile widths of the pair launch: widths of every multiple of 32 columns that
the launch picks to fill its rounds, last tiles cut into halves (also halves
that lie past n), with two- and three-part panels, single and batched, odd
sizes and a C that is read (a column stored twice would show), against the FP64
oracle under the acceptance bound."""

import numpy as np
import pytest

from gpu_util import SPLIT, check_full, dev
from oracle import oracle as O
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


@pytest.mark.parametrize("m,n,k", [
    (2324, 774, 512), (772, 2562, 600), (771, 2566, 511), (1028, 2404, 512), (1286, 1921, 256), (2057, 2116, 512),
    (2051, 2119, 511), (2051, 2049, 512), (1281, 2315, 512), (1282, 2311, 300), (2561, 1346, 512), (1931, 1207, 877)])
def test_widths_single(h, m, n, k):
    A, lda, B, ldb, C, ldc = synth.gemm_problem("uniform", 61, "N", "T", m, n, k, pad=3)
    check_full(h, SPLIT, "N", "T", m, n, k, 1.5, A, lda, B, ldb, -0.25, C, ldc)


@pytest.mark.parametrize("m,n,k", [(1552, 263, 600), (1549, 263, 256), (1618, 290, 600), (2057, 257, 256),
                                   (258, 2136, 512), (517, 2148, 600), (519, 2113, 256), (257, 2305, 600)])
def test_widths_batched(h, m, n, k):
    import torch
    b = 3
    probs = [synth.gemm_problem("uniform", 62 + z, "T", "N", m, n, k) for z in range(b)]
    lda, ldb, ldc = probs[0][1], probs[0][3], probs[0][5]
    A, B, C = (np.concatenate([np.ravel(p[i]) for p in probs]) for i in (0, 2, 4))
    dA, dB, dC = dev(A), dev(B), dev(C)
    h.set_path(SPLIT)
    h.sgemm_strided_batched("T", "N", m, n, k, 1.0, dA, lda, A.size // b, dB, ldb, B.size // b, 0.5, dC, ldc,
                            C.size // b, b)
    torch.cuda.synchronize()
    assert h.get_device_status() == 0
    out = dC.cpu().numpy().reshape(b, -1)
    for z, (a, _, bb, _, c, _) in enumerate(probs):
        c64, bnd = O.gemm_f64("T", "N", m, n, k, 1.0, a, lda, bb, ldb, 0.5, c, ldc)
        assert O.error_ratio(synth.logical(out[z], m, n, ldc), c64, bnd) <= 1.0
