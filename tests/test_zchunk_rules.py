"""The chunk length a step launch takes, by the rule of its kernel family: the
streaming kernels' one-round rule and dispatch model, TI_n's and the FP64
kernels' rules, at the ends of their ranges; and the lengths of launches whose
sweeps were measured on 152 SMs.
"""
import random

import pytest

from paper_1910_05180_gb300 import build as B
from paper_1910_05180_gb300 import spfm as S

STREAM, UNEVEN, FP64 = 0, 1, 2
SMS, TARGET = 152, 6 * 4 * 152


@pytest.fixture(scope="module")
def lib():
    B.build()
    return S.load()


def _ceil(a, b):
    return -(-a // b)


def _one_round(tiles, nz, slots):
    """The shortest chunks whose CTAs fit the slots."""
    return next(z for z in range(1, nz + 1) if tiles * _ceil(nz, z) <= slots)


def _shapes(slots, rng):
    for nz in (1, 2, 3, 4, 5, 8, 63, 64, 65, 130, 500):
        for tiles in (1, 2, slots // 7, slots - 1, slots, slots + 1, 3 * slots, 40 * slots):
            yield max(1, tiles), nz
    for _ in range(200):
        yield rng.randint(1, 3 * slots), rng.randint(1, 300)


@pytest.mark.parametrize("per_sm", [1, 2, 3, 4])
def test_streaming_rule(lib, per_sm):
    slots = per_sm * SMS
    for tiles, nz in _shapes(slots, random.Random(per_sm)):
        got = lib.spfm_debug_zchunk(STREAM, tiles, nz, per_sm, SMS, TARGET)
        if tiles * _ceil(nz, 4) <= slots:
            want = _one_round(tiles, nz, slots)
            assert _ceil(nz, got) == _ceil(nz, want) and got <= 4
        else:
            assert got == lib.spfm_debug_pick_zchunk(tiles, nz, per_sm, SMS, TARGET)
        assert 1 <= got <= nz


@pytest.mark.parametrize("per_sm", [1, 2])
def test_uneven_rule(lib, per_sm):
    slots = per_sm * SMS
    for tiles, nz in _shapes(slots, random.Random(per_sm)):
        got = lib.spfm_debug_zchunk(UNEVEN, tiles, nz, per_sm, SMS, TARGET)
        if tiles * _ceil(nz, 4) < slots:
            assert got == _ceil(nz, min(nz, slots // tiles))
            assert tiles * _ceil(nz, got) <= slots
        else:
            assert got == min(16, max(4, _ceil(tiles * nz, 6 * slots)))


def test_fp64_rule(lib):
    """The least work of the fullest SM, over chunks of 1 to 64 planes."""
    def work(tiles, nz, z):
        n = _ceil(tiles * _ceil(nz, z), SMS)
        return n * (100 + {1: 20, 2: 2}.get(n, 0)) * (9 * (z + 2) + 21 * z)

    for tiles, nz in _shapes(3 * SMS, random.Random(9)):
        got = lib.spfm_debug_zchunk(FP64, tiles, nz, 3, SMS, TARGET)
        best = min(work(tiles, nz, z) for z in range(1, min(nz, 64) + 1))
        assert got == max(z for z in range(1, min(nz, 64) + 1) if work(tiles, nz, z) == best), (tiles, nz)


@pytest.mark.parametrize("family,tiles,nz,per_sm,want", [
    (STREAM, 4, 32, 4, 1),       # 32^3 on 64 x 16 tiles (32 wide pads one tile): less than a round
    (STREAM, 64, 3, 4, 1),       # three planes
    (STREAM, 12, 96, 4, 2),      # 96 x 96: 48 chunks of 2 on 608 slots
    (STREAM, 16, 128, 4, 4),     # 128^3
    (STREAM, 64, 256, 4, 28),    # 256^3
    (STREAM, 256, 512, 4, 35),   # 512^3: many rounds
    (UNEVEN, 4, 60, 2, 1),       # 60^3
    (UNEVEN, 64, 256, 2, 9),     # 256^3
    (UNEVEN, 100, 320, 2, 16),   # 320^3 on 32 x 32 tiles
    (FP64, 8, 32, 3, 2),         # 128 x 32 x 32 on 32 x 16 tiles
    (FP64, 128, 256, 3, 37),     # 256^3
])
def test_measured_launches(lib, family, tiles, nz, per_sm, want):
    assert lib.spfm_debug_zchunk(family, tiles, nz, per_sm, SMS, TARGET) == want


def test_bad_arguments(lib):
    for args in [(3, 4, 10, 4, 152, 100), (-1, 4, 10, 4, 152, 100), (0, 0, 10, 4, 152, 100), (1, 4, 0, 2, 152, 100),
                 (2, 4, 10, 0, 152, 100), (0, 4, 10, 4, 0, 100), (0, 4, 10, 4, 152, 0)]:
        assert lib.spfm_debug_zchunk(*args) == -1
