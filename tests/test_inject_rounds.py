"""The attempt counter of a warp's shared injection rounds (fte_inject), on the host: it ends at the
attempt limit exactly, for every limit up to the largest int, where a counter that went on by whole
rounds would wrap to a negative number and never reach the limit."""
import ctypes as C

import pytest

INT_MAX = 2 ** 31 - 1


@pytest.fixture(scope="module")
def lib():
    from paper_2404_12164_gb300 import build
    build.build()
    from paper_2404_12164_gb300 import _abi
    return _abi.lib()


def _round(lib, n, t0, limit):
    width, made = C.c_int32(), C.c_int32()
    assert lib.fte_probe_attempt_round(n, t0, limit, C.byref(width), C.byref(made)) == 0
    return width.value, made.value


@pytest.mark.parametrize("limit,start", [(1, 0), (2, 0), (31, 0), (33, 0), (256, 0), (INT_MAX, INT_MAX - 100),
                                         (INT_MAX - 1, INT_MAX - 70), (INT_MAX, INT_MAX - 1)])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 8, 11, 16, 17, 32])
def test_rounds_end_at_the_limit(lib, n, limit, start):
    t = start
    while t < limit:
        width, made = _round(lib, n, t, limit)
        assert width in (1, 2, 4, 8, 16, 32) and width * n <= 32 < 2 * width * n
        assert made == min(width, limit - t) >= 1
        t += made
        assert t <= limit <= INT_MAX
    assert t == limit


def test_refuses_what_the_kernel_never_asks(lib):
    w, m = C.c_int32(), C.c_int32()
    for n, t0, limit in ((0, 0, 4), (33, 0, 4), (1, 4, 4), (1, -1, 4)):
        assert lib.fte_probe_attempt_round(n, t0, limit, C.byref(w), C.byref(m)) != 0
