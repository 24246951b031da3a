"""The rule of the split path without a packing pass (host only): the plan of
shapes that together take every tile, number of k slices and way to sum them,
and the plans that are left when a device cannot place large clusters."""

import ctypes

import pytest

# (m, n, k, batch): (tile columns, pair of CTAs, k slices, summed in the cluster)
SHAPES = {
    # two parts
    (81, 70, 556, 39): (64, 0, 1, 1), (65, 33, 552, 1): (64, 0, 2, 1), (65, 33, 596, 1): (64, 0, 4, 1),
    (66, 36, 944, 1): (64, 0, 8, 1), (65, 33, 968, 1): (64, 0, 16, 1), (219, 71, 568, 39): (128, 1, 1, 1),
    (138, 65, 1008, 23): (128, 1, 2, 1), (154, 65, 1500, 11): (128, 1, 4, 1), (133, 70, 2916, 4): (128, 1, 8, 1),
    (102, 257, 552, 38): (256, 1, 1, 1), (177, 35, 11280, 1): (256, 1, 59, 0),
    # three parts
    (65, 33, 144, 1): (64, 0, 1, 1), (141, 35, 300, 37): (64, 0, 2, 1), (69, 33, 204, 1): (64, 0, 4, 1),
    (66, 33, 244, 1): (64, 0, 8, 1), (436, 65, 152, 39): (128, 1, 1, 1),
}


@pytest.fixture(scope="module")
def plan():
    from paper_1608_05265_gb300 import build
    f = ctypes.CDLL(build.build()).gbgemm_internal_direct_plan
    i64 = ctypes.c_int64
    f.argtypes = [ctypes.c_char, ctypes.c_char, i64, i64, i64, i64, i64, i64, ctypes.c_int, ctypes.c_int,
                  ctypes.POINTER(ctypes.c_int)]

    def query(ta, tb, m, n, k, batch=1, pad=0, max_cluster=16):
        out = (ctypes.c_int * 6)()
        lda, ldb = (m if ta == "N" else k) + pad, (k if tb == "N" else n) + pad
        if not f(ta.encode(), tb.encode(), m, n, k, batch, lda, ldb, 152, max_cluster, out):
            return None
        assert out[4] < out[5]  # estimated faster than the packed path
        return tuple(out[:4])

    return query


def cluster(p):
    return (p[2] if p[3] else 1) * (2 if p[1] else 1)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ta,tb,pad", [("N", "T", 0), ("T", "N", 0), ("T", "N", 1)])
def test_every_kind_of_plan(plan, shape, ta, tb, pad):
    m, n, k, batch = shape
    assert plan(ta, tb, m, n, k, batch, pad) == SHAPES[shape]


@pytest.mark.parametrize("limit", [8, 4, 2, 1])
def test_plans_without_large_clusters(plan, limit):
    """Where a cluster cannot be placed a smaller one serves, or none (the packed path)."""
    smaller = 0
    for (m, n, k, batch), p in SHAPES.items():
        q = plan("N", "T", m, n, k, batch, 0, limit)
        assert q is None or cluster(q) <= limit
        if cluster(p) <= limit:
            assert q == p
        elif q is not None:
            smaller += 1
    assert smaller > 0
