"""Calls without a packing pass under the tuning modes and the schedule report:
modes 1 and 2 run them like mode 0 where they are faster, tuning files carry
their timing, and gbgemm_last_direct says which calls ran so."""

import os

import pytest

from paper_1608_05265_gb300 import synth

from gpu_util import check_full

pytestmark = pytest.mark.gpu

SHAPE = ("N", "T", 256, 256, 512)  # one launch against three or more


@pytest.fixture
def h():
    import torch
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    hd = gbgemm.Handle(0)
    hd.set_stream(torch.cuda.current_stream())
    yield hd
    hd.close()


def launches(h, path=0):
    import torch
    ta, tb, m, n, k = SHAPE
    A, lda, B, ldb, C, ldc = synth.gemm_problem("uniform", 98, ta, tb, m, n, k, pad=4)
    check_full(h, path, ta, tb, m, n, k, 1.0, A, lda, B, ldb, 0.5, C, ldc)  # a tuned shape's first call
    h.profile_begin()
    check_full(h, path, ta, tb, m, n, k, 1.0, A, lda, B, ldb, 0.5, C, ldc)
    torch.cuda.synchronize()
    return h.profile_end()[2]


def load_predictor(h):
    from paper_1608_05265_gb300 import gbgemm, predictor
    h.predictor_select(1)
    h.predictor_set(predictor.load_weights(predictor.DEFAULT_SCHED_WEIGHTS, gbgemm.SCHED_MLP_PARAMS)[0])
    h.predictor_select(0)


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_every_mode_runs_them(h, mode):
    from paper_1608_05265_gb300 import gbgemm
    h.set_tuning(mode)
    if mode == 2:
        load_predictor(h)
    assert launches(h) == 1 and h.last_direct()
    assert launches(h, gbgemm.PATH_SPLIT_BF16) >= 2 and not h.last_direct()
    assert launches(h, gbgemm.PATH_SIMT) == 1 and not h.last_direct()


def test_a_pinned_schedule_is_what_runs(h):
    assert launches(h) == 1 and h.last_direct()
    h.set_schedule(h.last_schedule())
    assert launches(h) >= 2 and not h.last_direct()
    h.set_schedule(-1)
    assert launches(h) == 1 and h.last_direct()


def test_tuning_files(h, tmp_path):
    h.set_tuning(1)
    assert launches(h) == 1
    path = str(tmp_path / "new.txt")
    h.tuning_save(path)
    h.tuning_clear()
    h.tuning_load(path)
    assert launches(h) == 1 and h.last_direct()
    # without the last figure, as older versions wrote it: schedules only
    old = str(tmp_path / "old.txt")
    with open(old, "w") as f:
        for line in open(path):
            f.write(line.rsplit(" ", 1)[0] + "\n" if line.startswith("S ") else line)
    h.tuning_clear()
    h.tuning_load(old)
    launches(h)
    assert not h.last_direct()
    assert os.path.getsize(old) < os.path.getsize(path)
