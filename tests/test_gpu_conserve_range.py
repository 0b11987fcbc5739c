"""Constant-volume steps whose alpha leaves the FP32 range: a field of exact 0
and 1, which take no correction, and one minute cell.  The step's rounding moves
the volume by dsum, and alpha = dsum / q of that cell; the other cells keep
their plain step bit for bit, and the field stays finite.
"""
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


@pytest.mark.parametrize("scheme", [S.SPFM_FD, S.SPFM_TI_GLOBAL])
@pytest.mark.parametrize("shape", [(48, 40, 36), (33, 17, 9)])
def test_minute_cell_takes_the_correction(shape, scheme):
    nx, ny, nz = shape
    phi = np.random.default_rng(1).integers(0, 2, (nz, ny, nx)).astype(np.float32)
    at = (3, 5, 7)
    phi[at] = np.float32(1e-45)
    t = torch.from_numpy(phi).cuda()
    kw = dict(lam=3.0, dt=0.037, stencil=26, scheme=scheme)
    fields = []
    for conserving in (False, True):
        g = S.Grid(nx, ny, nz, dtype=S.SPFM_F32, n=(0.36, 0.48, 0.8))
        g.set_field(t)
        if conserving:
            g.step_conserving(1, **kw)
        else:
            g.step(1, dF=0.0, **kw)
        fields.append(g.get_field().double().numpy())
        g.close()
    plain, got = fields
    x = phi.astype(np.float64)
    q = x * (1.0 - x)
    dsum = float((plain - x).sum())           # exact to 2^-53 of the sum of its terms
    assert abs(dsum) / q.sum() > 3.5e38, "alpha is meant to leave the FP32 range"
    assert np.isfinite(got).all()
    rest = np.ones(x.shape, bool)
    rest[at] = False
    assert (got[rest] == plain[rest]).all()
    want = plain[at] - dsum                   # alpha q of the only cell with q > 0
    assert abs(got[at] - want) <= 2.0 ** -24 * abs(want) + 2.0 ** -50 * np.abs(plain - x).sum()
