"""The TI potential's sum over the coupling groups (Eqs. 5, 6) in the form the
step kernels evaluate, N(q) / D(q) with q = phi (1 - phi), against the sum
direction by direction in FP64, on the host: every q that a field can hold,
inside [0, 1/4] and outside it, for the orientations and widths of the studies.

Tolerances.  All groups kept: both sides take at most 4 x 13 rounded operations
on positive numbers, and 1 - A loses at most a factor 1 / (1 - A) < 400 of its
digits at lambda >= dx: 100 x 400 x 2^-53 < 5e-12.  Fewer terms (FP32 and BF16
storage): 2^-30 by construction, over its whole range of q.
"""
import ctypes
import math

import numpy as np
import pytest

from paper_1910_05180_gb300 import build as B
from paper_1910_05180_gb300 import spfm as S
from paper_1910_05180_gb300 import workloads as WL

DIRS = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (0, 1, 1), (1, 0, 1), (1, -1, 0), (0, 1, -1), (1, 0, -1),
        (1, 1, 1), (-1, 1, 1), (1, -1, 1), (1, 1, -1)]
GAMMA = {6: (1.0, 0.0, 0.0), 18: (1 / 3, 2 / 3, 0.0), 26: (1 / 2, 1 / 3, 1 / 6)}
COUNT = {6: 3, 18: 9, 26: 13}


@pytest.fixture(scope="module")
def lib():
    B.build()
    return S.load()


def kernel_form(lib, dtype, stencil, u, lam, q):
    arr = (ctypes.c_double * len(q))(*q)
    out = (ctypes.c_double * len(q))()
    lo = ctypes.c_double()
    deg = lib.spfm_debug_potential(dtype, stencil, (ctypes.c_double * 3)(*u), lam, 1.0, len(q), arr, out,
                                   ctypes.byref(lo))
    return deg, lo.value, np.array(out)


def plain_sum(stencil, u, lam, q):
    total = np.zeros(len(q))
    for d in DIRS[:COUNT[stencil]]:
        j = sum(map(abs, d))
        c = GAMMA[stencil][j - 1] * (1.0, 0.5, 0.75)[j - 1] / j
        x = 2.0 * float(np.dot(d, u)) / lam
        A, E = math.tanh(x) ** 2, 1.0 / math.cosh(x) ** 2
        total += 4.0 * c * A / (E + 4.0 * A * q)
    return total


def directions():
    rng = np.random.default_rng(7)
    named = [WL.unit(v) for v in ((1, 0, 0), (1, 1, 0), (1, 1, 1), (1, 2, 0), (0, 1e-4, 1))]
    return named + [WL.random_normal(rng) for _ in range(40)]


@pytest.mark.parametrize("stencil", [6, 18, 26])
@pytest.mark.parametrize("lam", [1.0, 1.3, 2.0, 2.5, 3.0, 4.0, 6.0, 40.0])
@pytest.mark.parametrize("dtype", [S.SPFM_F64, S.SPFM_F32])
def test_ratio_equals_the_sum_over_directions(lib, dtype, lam, stencil):
    for u in directions():
        amax = max(math.tanh(2.0 * float(np.dot(d, u)) / lam) ** 2 for d in DIRS[:COUNT[stencil]])
        # inside [0, 1/4], and outside down to half way to the first pole of the sum
        pole = -0.25 * (1.0 - amax) / amax
        q = np.concatenate([np.linspace(0.0, 0.25, 401), 0.25 * np.logspace(-9, 0, 60),
                            np.linspace(0.5 * max(pole, -1.0), 0.0, 101)])
        deg, lo, got = kernel_form(lib, dtype, stencil, u, lam, q)
        ref = plain_sum(stencil, u, lam, q)
        groups = len({round(math.log(a), 9) for a in
                      (math.tanh(2.0 * float(np.dot(d, u)) / lam) ** 2 for d in DIRS[:COUNT[stencil]]) if a > 1e-25})
        assert 1 <= deg <= 13
        if lo == -math.inf:
            tol = 5e-12
        else:
            tol = 2.0 ** -30
            assert dtype == S.SPFM_F32 and deg < groups and -0.0126 < lo < 0.0
        assert np.abs(got / ref - 1.0).max() <= tol, (u, deg, lo)


def test_degree_falls_with_the_width(lib):
    """A generic normal has 13 groups: FP64 keeps them, FP32 takes 3-4 terms at
    lambda = 6 and no more than 6 at lambda = 2."""
    for u in directions()[5:]:
        assert kernel_form(lib, S.SPFM_F64, 26, u, 3.0, [0.1])[0] >= 7
        assert kernel_form(lib, S.SPFM_F32, 26, u, 6.0, [0.1])[0] <= 4
        assert kernel_form(lib, S.SPFM_F32, 26, u, 2.0, [0.1])[0] <= 6


def test_extreme_widths_keep_a_form_or_the_groups(lib):
    """lambda far below dx drives every A to 1 and the coefficients out of the
    FP32 range: the groups are then summed one by one (degree 0), never a form
    with overflowed coefficients."""
    u = WL.random_normal(np.random.default_rng(3))
    for lam in (1e-3, 0.02, 0.1, 0.3, 0.5, 0.7, 1e4):
        deg, _, got = kernel_form(lib, S.SPFM_F32, 26, u, lam, [0.25, 0.01])
        if deg == -1:
            # some 1 - A is 0 in FP64: no dt is stable and every step is refused
            assert max(math.tanh(2.0 * float(np.dot(d, u)) / lam) ** 2 for d in DIRS) == 1.0
            continue
        assert 0 <= deg <= 13
        if deg:
            assert np.isfinite(got).all() and (got > 0.0).all()
