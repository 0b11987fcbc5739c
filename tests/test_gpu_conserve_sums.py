"""alpha of constant-volume steps against exact sums of the same cells.

The four-cell sums are exact to 2^-70 and enter FP64 in a tree of some 40 adds, so
alpha is off by a few 2^-53 of random sign: at most 16 of them for any one field
(the adds' worst case is 40 for each sum), and 1.5 in the mean of 16 fields, where
an error of one sign in the cells' terms would stand out.
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


def _exact(x):
    """The sum of FP32 or BF16 cells (as FP64) and of their squares, exactly."""
    m = np.round(x * 2.0 ** 40)
    small = m != x * 2.0 ** 40                 # cells with bits below 2^-40: one by one
    m = m[~small].astype(np.int64)
    hi, lo = m >> 20, m & ((1 << 20) - 1)
    sq = (int((hi * hi).sum()) << 40) + (2 * int((hi * lo).sum()) << 20) + int((lo * lo).sum())
    one, two = F(int(m.sum()), 2 ** 40), F(sq, 2 ** 80)
    for v in x[small]:
        one += F(float(v))
        two += F(float(v)) ** 2
    return one, two


@pytest.mark.parametrize("dtype", [S.SPFM_F32, S.SPFM_BF16])
def test_alpha_is_the_exact_ratio_of_sums(dtype):
    lam, dt, errors = 4.0, 0.0625, []
    for seed in range(16):
        rng = np.random.default_rng(seed)
        n = int(rng.integers(40, 72))
        at = [np.abs(np.arange(n) - ((n - 1) / 2 + rng.uniform(-0.5, 0.5))) for _ in range(3)]
        cube = 1.0
        for ax, p in enumerate(at):
            f = 0.5 * (1.0 - np.tanh(2.0 * (p - 0.2 * n) / lam))
            cube = cube * f.reshape([-1 if a == 2 - ax else 1 for a in range(3)])
        t = torch.from_numpy(1.0 - cube).to(S.TORCH_DTYPE[dtype])
        g = S.Grid(n, n, n, dtype=dtype)
        kw = dict(lam=lam, dt=dt, stencil=26, scheme=S.SPFM_FD)
        g.set_field(t.cuda())
        g.step(1, dF=0.0, **kw)
        plain = g.get_field().double().numpy().ravel()
        g.set_field(t.cuda())
        dF = g.step_conserving(1, **kw)        # alpha = dF 4 dt / lam: powers of two
        g.close()
        x = t.double().numpy().ravel()
        sx, sxx = _exact(x)
        alpha = (_exact(plain)[0] - sx) / (sx - sxx)
        errors.append(float((F(dF) * F(4.0 * dt / lam) / alpha - 1) * 2 ** 53))
    assert max(abs(e) for e in errors) <= 16.0, errors
    assert abs(np.mean(errors)) <= 1.5, errors
