"""The transpose flags that Handle.sgemm takes (no GPU: a null handle, which the
library reports after it has checked the arguments)."""

import pytest


@pytest.fixture(scope="module")
def handle():
    from paper_1608_05265_gb300 import build, gbgemm
    build.build()
    h = object.__new__(gbgemm.Handle)
    h._h = None
    return h


@pytest.mark.parametrize("flag", ["N", "n", "T", "c", b"N", b"t", bytearray(b"N"), bytearray(b"C"), ord("T")])
def test_accepted(handle, flag):
    from paper_1608_05265_gb300 import gbgemm
    want = gbgemm.lib().gbgemm_sgemm(None, b"N", b"N", 4, 4, 4, 1.0, 16, 4, 16, 4, 0.0, 16, 4)
    for ta, tb in ((flag, "N"), ("N", flag)):
        assert handle.sgemm(ta, tb, 4, 4, 4, 1.0, 16, 4, 16, 4, 0.0, 16, 4, check=False) == want


@pytest.mark.parametrize("flag", ["X", b"x", bytearray(b"Q")])
def test_refused(handle, flag):
    assert handle.sgemm(flag, "N", 4, 4, 4, 1.0, 16, 4, 16, 4, 0.0, 16, 4, check=False) == -1
    assert handle.sgemm("N", flag, 4, 4, 4, 1.0, 16, 4, 16, 4, 0.0, 16, 4, check=False) == -2


@pytest.mark.parametrize("flag", ["", "NT", b"", None])
def test_not_one_character(handle, flag):
    with pytest.raises(Exception):
        handle.sgemm(flag, "N", 4, 4, 4, 1.0, 16, 4, 16, 4, 0.0, 16, 4, check=False)
