"""TI_n in the bulk phases: a thread whose cells and their face neighbours all sit
in the same clamp of the profile inversion takes the CF potential at once; a row
with other cells takes the general form, which falls back to it cell by cell.

Cells of both clamps (phi below 1e-6 and above 1 - 1e-6, negative and above 1
among them) are stepped with every row wholly in its clamp, and again with one cell
of each aligned group of four off it.  The cells two away from those have the same
27 neighbours in both fields, so they must come out bit for bit the same, on both
tile shapes and in FP64 and BF16.
"""
import numpy as np
import pytest
import torch

from paper_1910_05180_gb300 import spfm as S

pytestmark = pytest.mark.gpu

P, C = S.SPFM_PERIODIC, S.SPFM_CONTACT


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


def _step(phi, dtype, bc, lam, stencil):
    nz, ny, nx = phi.shape
    g = S.Grid(nx, ny, nz, dtype=dtype, bc=bc, n=(0.36, 0.48, 0.8))
    g.set_field(torch.from_numpy(phi).to(S.TORCH_DTYPE[dtype]).cuda())
    g.step(1, lam=lam, dt=0.02, dF=0.02, stencil=stencil, scheme=S.SPFM_TI_LOCAL)
    out = g.get_field()
    g.close()
    return out


@pytest.mark.parametrize("dtype", [S.SPFM_F32, S.SPFM_F64, S.SPFM_BF16])
@pytest.mark.parametrize("bc", [(P,) * 6, (C,) * 6])
@pytest.mark.parametrize("stencil", [6, 18, 26])
@pytest.mark.parametrize("lam", [1.5, 6.0])     # extents above and below 32 lambda: both FP32 tiles
def test_rows_in_the_clamp_equal_the_general_form(lam, stencil, bc, dtype):
    nx, ny, nz = 96, 50, 48
    rng = np.random.default_rng(int(lam) + stencil)
    low = rng.choice([0.0, 1e-30, 3e-7, 9e-7, -2e-4, 1e-6], (nz, ny, nx))
    high = 1.0 - rng.choice([0.0, 1e-7, 5e-7, -3e-4, 9e-7], (nz, ny, nx))
    phi = np.where(np.arange(nz)[:, None, None] < nz // 2, low, high)
    mixed = phi.copy()
    group = 8 if dtype == S.SPFM_BF16 else 4     # a thread's cells
    mixed[:, :, ::group] = 0.3 + 0.4 * rng.random(mixed[:, :, ::group].shape)
    a, b = _step(phi, dtype, bc, lam, stencil), _step(mixed, dtype, bc, lam, stencil)
    far = [x for x in range(nx) if x % group not in (0, 1, group - 1)]
    assert torch.equal(a[:, :, far], b[:, :, far])
    assert torch.isfinite(b.double()).all()
