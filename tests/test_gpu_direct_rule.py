"""Path AUTO on calls whose estimated times on the direct and the packed path
lie close together: no slower than the packed path beyond the estimates' error."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ta,tb,m,n,k,pad", [
    ("N", "T", 109, 2695, 1831, 1), ("T", "N", 281, 1007, 1197, 0), ("T", "N", 558, 1391, 442, 0),
    ("T", "N", 2539, 154, 1645, 0), ("T", "N", 1928, 311, 509, 0)])
def test_near_the_border(ta, tb, m, n, k, pad):
    import torch
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    h = gbgemm.Handle(0)
    h.set_stream(torch.cuda.current_stream())
    (ar, ac), (br, bc) = ((m, k) if ta == "N" else (k, m)), ((k, n) if tb == "N" else (n, k))
    A, B = torch.rand(ac, ar + pad, device="cuda") - 0.5, torch.rand(bc, br + pad, device="cuda") - 0.5
    C = torch.zeros(n, m + pad, device="cuda")
    call = lambda: h.sgemm(ta, tb, m, n, k, 1.0, A, ar + pad, B, br + pad, 0.0, C, m + pad)
    best = {}
    for _ in range(8):  # in turn
        for path in (gbgemm.PATH_AUTO, gbgemm.PATH_SPLIT_BF16):
            h.set_path(path)
            call()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(20):
                call()
            e1.record()
            torch.cuda.synchronize()
            best[path] = min(best.get(path, 1e30), e0.elapsed_time(e1))
    h.close()
    assert best[gbgemm.PATH_AUTO] <= 1.06 * best[gbgemm.PATH_SPLIT_BF16], best
