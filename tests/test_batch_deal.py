"""The deal of a batch's items to CTAs: every item goes to one CTA, longest first
to the least loaded (checked against a simulation), the counted span is the fullest
CTA's work, and long lists, which go in turn, come within an item of the mean.
"""
import ctypes
import heapq
import random

import pytest

from paper_1910_05180_gb300 import build as B
from paper_1910_05180_gb300 import spfm as S

START = 3   # planes' worth of an item's halo and start


@pytest.fixture(scope="module")
def lib():
    B.build()
    return S.load()


def _deal(lib, planes, ctas):
    n = len(planes)
    owner, span = (ctypes.c_int * max(n, 1))(), ctypes.c_longlong()
    assert lib.spfm_debug_deal(n, (ctypes.c_int * max(n, 1))(*planes), ctas, owner, ctypes.byref(span)) == 0
    loads, held = [0] * ctas, 0
    for p, c in zip(planes, owner):
        assert 0 <= c < ctas
        loads[c] += p + START
        held += 1
    assert held == n
    return loads, span.value


def _simulated(planes, ctas):
    heap = [0] * ctas
    for p in sorted(planes, reverse=True):
        heapq.heappush(heap, heapq.heappop(heap) + p + START)
    return sorted(heap)


@pytest.mark.parametrize("ctas", [1, 2, 7, 456, 1024])
def test_items_go_longest_first_to_the_least_loaded(lib, ctas):
    rng = random.Random(ctas)
    for n in (0, 1, ctas - 1, ctas, ctas + 1, 5 * ctas + 3, 12 * ctas, 64 * ctas if ctas < 10 else 20 * ctas):
        for most in (1, 8, 64):
            planes = [rng.choice([most, most, rng.randint(1, most)]) for _ in range(n)]
            loads, span = _deal(lib, planes, ctas)
            assert sorted(loads) == _simulated(planes, ctas)
            assert span == max(loads)


@pytest.mark.parametrize("ctas", [3, 456])
@pytest.mark.parametrize("extra", [1, 17])
def test_long_lists_stay_within_an_item_of_the_mean(lib, ctas, extra):
    rng = random.Random(extra)
    planes = [rng.choice([64, 64, 64, rng.randint(1, 64)]) for _ in range(65 * ctas + extra)]
    loads, _ = _deal(lib, planes, ctas)
    mean = sum(p + START for p in planes) / ctas
    assert max(loads) <= mean + 64 + START and min(loads) >= mean - 64 - START


def test_bad_arguments(lib):
    one = (ctypes.c_int * 1)(1)
    zero = (ctypes.c_int * 1)(0)
    assert lib.spfm_debug_deal(-1, one, 1, one, None) == -1
    assert lib.spfm_debug_deal(1, one, 0, one, None) == -1
    assert lib.spfm_debug_deal(1, None, 1, one, None) == -1
    assert lib.spfm_debug_deal(1, zero, 1, one, None) == -1
