"""The stats pass over many rows a warp: the volume's chains run over four sweeps
(a sweep is 512 cells of a row in FP32 and BF16), go to fixed point and, after 32
of those, to FP64; a sweep with cells that are not finite is redone from chains
that hold earlier rows; and band cells queue across rows, whose slots are reused.

Rows go to the warps in turn.  A batch walks a grid with 256 warps, so 40000 rows
are 156 a warp (39 fixed-point steps); a single grid of 30000 rows has eight or
more a warp.

Bars: counts and extrema exactly; the sums to 1e-13 of their terms' magnitudes
(below 2^-43; the chains lose at most 3e-11 per 64 cells of which a row in
three holds values near 1, and typically 1e-14; FP64 adds of 2^21 terms 2^-45).
"""
import math

import numpy as np
import pytest
import torch

from paper_1910_05180_gb300 import spfm as S

pytestmark = pytest.mark.gpu

LAM, N, CTR = 3.0, (0.36, 0.48, 0.8), (0.4, 1.3, -2.0)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


def _field(shape, bad, seed):
    nx, ny, nz = shape
    rng = np.random.default_rng(seed)
    kind = rng.random((nz, ny, nx))
    phi = np.where(kind < 0.5, rng.random(kind.shape) * 1e-7, 1.0 - rng.random(kind.shape) * 1e-7)
    band = rng.random(kind.shape) < 0.03              # sparse, in most rows
    phi[band] = rng.random(int(band.sum()))
    if bad:                                           # rows 2 to 4 of a group of four, in some groups
        rows = phi.reshape(-1, nx)
        pick = rng.integers(0, len(rows), max(8, len(rows) // 300))
        rows[pick, rng.integers(0, nx, len(pick))] = rng.choice([np.nan, np.inf, -np.inf], len(pick))
    return phi


def _check(st, v):
    fin = np.isfinite(v)
    assert st["nonfinite"] == (~fin).sum()
    assert st["phi_min"] == v[fin].min() and st["phi_max"] == v[fin].max()
    vol = math.fsum(v[fin])
    assert abs(st["volume"] - vol) <= 1e-13 * vol
    band = fin & (v > 1e-6) & (v < 1 - 1e-6)
    k, j, i = np.nonzero(band)
    p = v[band]
    q, psi = p * (1 - p), 0.25 * LAM * (np.log1p(-p) - np.log(p))
    pn = N[0] * i + N[1] * j + N[2] * k
    r = np.sqrt((i - CTR[0]) ** 2 + (j - CTR[1]) ** 2 + (k - CTR[2]) ** 2)
    for name, term in (("S_w", q), ("S_c", q * (pn - psi)), ("S_r", q * (r + psi))):
        assert abs(st[name] - math.fsum(term)) <= 1e-13 * (np.abs(term).sum() + (q * np.abs(psi)).sum()), name


def _grid(shape, dtype, phi):
    g = S.Grid(*shape, dtype=dtype, n=N, center=CTR)
    g.init_planar(0.0, LAM)
    t = torch.from_numpy(phi).to(S.TORCH_DTYPE[dtype])
    g.set_field(t.cuda())
    return g, t.double().numpy()


@pytest.mark.parametrize("dtype", [S.SPFM_F64, S.SPFM_F32, S.SPFM_BF16])
@pytest.mark.parametrize("bad", [False, True])
@pytest.mark.parametrize("shape", [(8, 200, 200), (21, 160, 250), (1500, 60, 50)])
def test_batch_grids_of_many_rows(shape, bad, dtype):
    grids, fields = zip(*[_grid(shape, dtype, _field(shape, bad, s)) for s in (1, 2)])
    b = S.Batch(grids)
    for st, v in zip(b.stats(allow_nonfinite=True), fields):
        _check(st, v)
    b.close()


@pytest.mark.parametrize("dtype", [S.SPFM_F32, S.SPFM_BF16])
@pytest.mark.parametrize("bad", [False, True])
@pytest.mark.parametrize("shape", [(24, 150, 220), (600, 130, 240)])
def test_single_grid_of_many_rows(shape, bad, dtype):
    g, v = _grid(shape, dtype, _field(shape, bad, 3))
    _check(g.stats(allow_nonfinite=True), v)
    g.close()
