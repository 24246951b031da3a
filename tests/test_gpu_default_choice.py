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
