"""FP64 CF steps of a field that varies along z alone against the same operations
in exact arithmetic, each rounded once: bit for bit.  The second difference is
(a - c) + (b - c); a form that rounds a + b first differs in one cell of
several.
"""
from fractions import Fraction as F

import numpy as np
import pytest
import torch

from paper_1910_05180_gb300 import spfm as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


def _fma(a, b, c):
    return float(F(a) * F(b) + F(c))


@pytest.mark.parametrize("lam,dt", [(4.0, 0.05), (3.0, 0.1)])
def test_column_steps_are_the_exact_operations(lam, dt):
    nz = 96
    z = np.arange(nz)
    phi = 0.5 * (1.0 - np.tanh(2.0 * (np.abs(z - 47.3) - 20.0) / lam))
    phi += 1e-3 * np.random.default_rng(7).random(nz)
    g = S.Grid(8, 4, nz, dtype=S.SPFM_F64)
    g.set_field(torch.from_numpy(np.broadcast_to(phi[:, None, None], (nz, 4, 8)).copy()).cuda())
    g.step(1, lam=lam, dt=dt, dF=0.0, stencil=6, scheme=S.SPFM_FD)
    got = g.get_field().numpy()
    g.close()
    nkap = -(1.0 / (lam * lam) * (16.0 / 3.0) * 3.0) * dt     # D = c_1 = 1
    for k in range(nz):
        c, a, b = float(phi[k]), float(phi[k - 1]), float(phi[(k + 1) % nz])
        t = (a - c) + (b - c)
        acc = _fma(dt, t, c)                                   # the in-plane sum is 0
        w = _fma(-2.0, c, 1.0) * nkap
        want = _fma(_fma(-c, c, c), w, acc)
        assert (got[k] == want).all(), (k, got[k, 0, 0] - want)
