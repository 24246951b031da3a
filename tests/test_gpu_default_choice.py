"""What the predictor's report compares with is the rule the library runs."""

import pytest

pytestmark = pytest.mark.gpu


def test_default_choice_is_the_plans_default():
    import torch
    from paper_1608_05265_gb300 import build, gbgemm, predictor
    build.build()
    h = gbgemm.Handle(0)
    h.set_stream(torch.cuda.current_stream())
    shapes = [(ta, tb, m, n, k, 1, 1, 1) for ta, tb in (("N", "N"), ("T", "N")) for m in (8, 64, 65, 129, 200, 700)
              for n in (8, 64, 65, 128, 129, 192, 257, 600) for k in (8, 15, 16, 100)]
    buf = torch.zeros(700 * 600 * 3, device="cuda")
    p = buf.data_ptr()
    probs = [gbgemm.problem(ta, tb, m, n, k, 1.0, p, m if ta == "N" else k, p, k if tb == "N" else n, 0.0, p, m)
             for (ta, tb, m, n, k, *_) in shapes]
    plan = gbgemm.GroupedPlan(h, probs, config_source=gbgemm.CONFIG_DEFAULT)
    got = list(plan.configs())
    plan.close()
    h.close()
    assert got == predictor.default_choice(shapes).tolist()


@pytest.mark.parametrize("count,widest", [(1, "BN128"), (8, "BN128"), (38, "BN128"), (39, "BN256"), (200, "BN256")])
def test_small_plans_take_narrower_tiles(count, widest):
    """Plans of at most as many 128 x 128 tiles as SMs (four a problem here) stay at 128 columns."""
    import torch
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    h = gbgemm.Handle(0)
    h.set_stream(torch.cuda.current_stream())
    assert torch.cuda.get_device_properties(0).multi_processor_count == 152
    buf = torch.zeros(256 * 200, device="cuda")
    out = torch.empty(count, 200 * 200, device="cuda")
    p = buf.data_ptr()
    plan = gbgemm.GroupedPlan(h, [gbgemm.problem("N", "N", 200, 200, 256, 1.0, p, 200, p, 256, 0.0, out[i].data_ptr(), 200)
                                  for i in range(count)], config_source=gbgemm.CONFIG_DEFAULT)
    assert set(plan.configs()) == {getattr(gbgemm, "CFG_SPLIT_" + widest)}
    plan.run()
    torch.cuda.synchronize()
    assert h.get_device_status() == 0 and float(out.abs().max()) == 0.0
    plan.close()
    h.close()
