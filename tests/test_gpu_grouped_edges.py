"""Edge tiles of the grouped split path: tiles whose operands fill only part of
the 128 x BN tile copy and multiply only the rows that exist, and several k
chunks then share a slot of the shared-memory ring.  Every problem against the
FP64 oracle under the acceptance bound, on the wide instance (tiles of up to
256 columns) and the narrow one, at the sizes around the tile, MMA and chunk
boundaries, with two- and three-part panels."""

import itertools

import pytest

from test_gpu_grouped import Batch, h, run_plan  # noqa: F401  (h: the module's handle)

pytestmark = pytest.mark.gpu

M = (1, 8, 9, 33, 64, 65, 127, 129, 200)
N = (1, 15, 17, 48, 64, 65, 128, 129, 250, 257)
K = (16, 33, 64, 97, 130, 250, 511, 512, 545)


def specs():
    out = []
    for g, (m, n) in enumerate(itertools.product(M, N)):
        ta, tb = "NT"[g & 1], "NT"[(g >> 1) & 1]
        out.append((ta, tb, m, n, K[(g * 4 + g // len(K)) % len(K)], (1.0, -1.5)[g % 2], (0.0, 1.0, -0.25)[g % 3]))
    return out


@pytest.mark.parametrize("cfg", [None, "SPLIT_BN64", "SPLIT_BN128", "SPLIT_BN256"])
def test_edge_tiles(h, cfg):  # noqa: F811
    from paper_1608_05265_gb300 import gbgemm
    s = specs()
    b = Batch(s, 41)
    kw = {} if cfg is None else {"configs": [getattr(gbgemm, "CFG_" + cfg)] * len(s)}
    if cfg is None:
        kw["config_source"] = gbgemm.CONFIG_DEFAULT
    plan = run_plan(h, b, **kw)
    b.check(nthreads=4)
    plan.close()
