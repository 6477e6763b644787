"""What a lock-step run's error words mean for each member (host only, no GPU): a bounded wait that ran
out is recorded with the first member and ends every member's run; everything else is a member's own."""
import ctypes

import pytest

from paper_2506_23895_gb300 import build as B
from paper_2506_23895_gb300 import lks

OK, ARG, CUDA, DIVERGED, TIMEOUT = 0, 1, 4, 5, 6


@pytest.fixture(scope="module")
def lib():
    B.build()
    return lks.load()


def statuses(lib, words):
    n = len(words)
    flat = (ctypes.c_int * (4 * n))(*[v for w in words for v in w])
    out = (ctypes.c_int * n)(*([-9] * n))
    assert lib.lks_batch_statuses(flat, n, out) == n
    return list(out)


@pytest.mark.parametrize("words,want", [
    ([(0, 0, 0, 0)], [OK]),
    ([(0, 0, 0, 8)], [TIMEOUT]),
    ([(0, 0, 0, 8), (0, 0, 0, 0), (0, 0, 0, 0)], [TIMEOUT] * 3),
    ([(0, 0, 0, 0), (0, 0, 0, 0), (0, 0, 0, 24)], [TIMEOUT] * 3),
    ([(0, 0, 1, 8), (0, 0, 1, 0), (0, 1, 0, 0)], [TIMEOUT, TIMEOUT, ARG]),
    ([(1, 0, 0, 0), (0, 0, 1, 0), (0, 1, 1, 0), (0, 0, 1, 16)], [OK, DIVERGED, ARG, CUDA]),
])
def test_a_wait_that_ran_out_ends_every_members_run(lib, words, want):
    assert statuses(lib, words) == want


def test_bad_arguments(lib):
    one = (ctypes.c_int * 4)()
    assert lib.lks_batch_statuses(one, 0, one) == -1
    assert lib.lks_batch_statuses(None, 1, one) == -1
    assert lib.lks_batch_statuses(one, 1, None) == -1
