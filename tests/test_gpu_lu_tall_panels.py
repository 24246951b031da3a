"""LU of more rows than the register-resident panel holds (16384), in blocks of
one panel each: the first panels are factored in shared memory with the
previous block applied in their prologue, the later ones in registers, each
reading the permutation the other kind wrote."""

import numpy as np
import pytest

from test_gpu_lu_panel import pivots_of

pytestmark = pytest.mark.gpu

EPS32 = 2.0 ** -24


@pytest.mark.parametrize("nb", [32, 30])
def test_pivots_fixed_by_construction(nb):
    import torch
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    h = gbgemm.Handle(0)
    h.set_stream(torch.cuda.current_stream())
    n = 16500
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    uni = lambda *s: torch.empty(*s, device="cuda").uniform_(-1.0, 1.0, generator=g)
    s = 1.0 / np.sqrt(n)
    want = torch.tril(uni(n, n) * (0.5 * s), -1)
    up = torch.triu(uni(n, n) * s, 1) + torch.diag(1.5 + 0.5 * uni(n))
    order = torch.randperm(n, device="cuda", generator=g)
    a = torch.empty(n, n, device="cuda")
    a[order] = (want + torch.eye(n, device="cuda")) @ up
    want += up
    del up
    lu = a.T.contiguous()  # column-major
    ipiv = torch.zeros(n, dtype=torch.int32, device="cuda")
    info = torch.full((1,), -7, dtype=torch.int32, device="cuda")
    h.sgetrf(n, lu, n, ipiv, info, nb)
    torch.cuda.synchronize()
    assert h.get_device_status() == 0 and int(info.item()) == 0
    assert np.array_equal(ipiv.cpu().numpy(), pivots_of(order.cpu().numpy()))
    # well conditioned, entries O(1): a few n eps between FP32 and exact factors
    assert float((lu.T - want).abs().max()) <= 16 * n * EPS32
    h.close()
