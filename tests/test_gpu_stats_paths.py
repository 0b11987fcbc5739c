"""The stats pass takes a lane's cells of a row as a whole: cells that are not
finite, values at the band's limits and far outside [0, 1], and rows that end
inside a 16-byte piece or a 512-cell sweep, against sums in numpy.

Bars: counts and extrema exactly; the volume and the band sums to 1e-12 of the
sum of their terms' magnitudes (the diagnostics carry 48 bits, 4e-15, a term
and add at most 2^20 of them with error-free pairs and FP64).
"""
import numpy as np
import pytest
import torch

from paper_1910_05180_gb300 import spfm as S

pytestmark = pytest.mark.gpu

LAM = 3.0


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


@pytest.mark.parametrize("dtype", [S.SPFM_F64, S.SPFM_F32, S.SPFM_BF16])
@pytest.mark.parametrize("nx,ny,nz", [(1, 3, 2), (3, 5, 4), (8, 9, 70), (37, 6, 5), (130, 4, 3), (512, 3, 2),
                                      (515, 2, 2), (1030, 2, 3)])
@pytest.mark.parametrize("bad", [False, True])
def test_sums_match_numpy(dtype, nx, ny, nz, bad):
    rng = np.random.default_rng(nx + 10 * ny + (7 if bad else 0))
    phi = rng.random((nz, ny, nx))
    kind = rng.random(phi.shape)
    phi[kind < 0.35] = 0.0                    # mostly bulk, as in a grain
    phi[(kind >= 0.35) & (kind < 0.7)] = 1.0
    phi[(kind >= 0.70) & (kind < 0.74)] = 1e-6
    phi[(kind >= 0.74) & (kind < 0.78)] = 1.0 - 1e-6
    phi[(kind >= 0.78) & (kind < 0.80)] = 1.0000005e-6
    phi[(kind >= 0.80) & (kind < 0.82)] = -3.5
    phi[(kind >= 0.82) & (kind < 0.84)] = 700.25
    if bad:
        pick = rng.random(phi.shape)
        phi[pick < 0.02] = np.nan
        phi[(pick >= 0.02) & (pick < 0.03)] = np.inf
        phi[(pick >= 0.03) & (pick < 0.04)] = -np.inf
        phi.flat[0] = np.nan
    t = torch.from_numpy(phi).to(S.TORCH_DTYPE[dtype])
    v = t.double().numpy()
    n, ctr = (0.36, 0.48, 0.8), (0.4, 1.3, -2.0)
    g = S.Grid(nx, ny, nz, dtype=dtype, n=n, center=ctr)
    g.init_planar(0.0, LAM)
    g.set_field(t.cuda())
    st = g.stats(allow_nonfinite=True)
    fin = np.isfinite(v)
    assert st["nonfinite"] == (~fin).sum()
    if fin.any():
        assert st["phi_min"] == v[fin].min() and st["phi_max"] == v[fin].max()
    assert abs(st["volume"] - v[fin].sum()) <= 1e-12 * np.abs(v[fin]).sum()
    band = fin & (v > 1e-6) & (v < 1 - 1e-6)
    k, j, i = np.nonzero(band)
    p = v[band]
    q, psi = p * (1 - p), 0.25 * LAM * (np.log1p(-p) - np.log(p))
    pn = n[0] * i + n[1] * j + n[2] * k
    r = np.sqrt((i - ctr[0]) ** 2 + (j - ctr[1]) ** 2 + (k - ctr[2]) ** 2)
    for name, term in (("S_w", q), ("S_c", q * (pn - psi)), ("S_r", q * (r + psi))):
        assert abs(st[name] - term.sum()) <= 1e-12 * (np.abs(term).sum() + (q * np.abs(psi)).sum()), name
    g.close()
