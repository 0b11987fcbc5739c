"""The N(q) / D(q) form of the TI potential and the unit of length: at a fixed
lambda / dx its degree and range are the same for every dx, and its values go with
1 / dx^2; FP64 grids take it up to widths whose coefficients FP32 could not hold.
"""
import ctypes
import math

import numpy as np
import pytest

from paper_1910_05180_gb300 import build as B
from paper_1910_05180_gb300 import spfm as S
from paper_1910_05180_gb300 import workloads as WL

Q = np.concatenate([np.linspace(0.0, 0.25, 51), [-1e-4, -1e-3]])


@pytest.fixture(scope="module")
def lib():
    B.build()
    return S.load()


def _form(lib, dtype, u, lam, dx):
    arr, out = (ctypes.c_double * len(Q))(*Q), (ctypes.c_double * len(Q))()
    lo = ctypes.c_double()
    deg = lib.spfm_debug_potential(dtype, 26, (ctypes.c_double * 3)(*u), lam * dx, dx, len(Q), arr, out,
                                   ctypes.byref(lo))
    return deg, lo.value, np.array(out)


@pytest.mark.parametrize("dtype", [S.SPFM_F64, S.SPFM_F32, S.SPFM_BF16])
@pytest.mark.parametrize("lam", [1.0, 2.0, 3.0, 6.0])
def test_form_does_not_depend_on_the_unit(lib, dtype, lam):
    rng = np.random.default_rng(5)
    for u in [WL.unit((1, 2, 0))] + [WL.random_normal(rng) for _ in range(4)]:
        deg, lo, val = _form(lib, dtype, u, lam, 1.0)
        assert deg >= 1
        for dx in (1e-12, 1e-9, 1e-6, 3e-3, 7.0, 1e6, 1e12):
            d, l, v = _form(lib, dtype, u, lam, dx)
            assert d == deg
            assert l == lo or abs(l / lo - 1.0) < 1e-9
            # lam * dx rounds: a relative change of 2^-52 of the couplings' arguments
            assert np.abs(v * dx * dx / val - 1.0).max() <= (1e-12 if dtype == S.SPFM_F64 else 2.0 ** -30), dx


def test_fp64_form_at_small_widths(lib):
    """13 groups at lambda = 0.5 dx: the product of the g_k is beyond 1e24."""
    u = WL.random_normal(np.random.default_rng(3))
    deg, lo, val = _form(lib, S.SPFM_F64, u, 0.5, 1.0)
    assert deg == 13 and lo == -math.inf and np.isfinite(val).all() and (val[:51] > 0.0).all()
