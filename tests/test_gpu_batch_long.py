"""Batches of many items a CTA: above 12 a slot the tile policy and depth come
from the mean, above 64 the list goes in turn.  Every grid equals its single-grid
steps bit for bit.
"""
import numpy as np
import pytest
import torch

from paper_1910_05180_gb300 import spfm as S
from paper_1910_05180_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

C = S.SPFM_CONTACT


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


def _grid(shape, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    nx, ny, nz = shape
    g = S.Grid(*shape, dtype=S.SPFM_F32, bc=(C,) * 6, n=tuple(WL.random_normal(np.random.default_rng(seed))))
    g.set_field(0.02 + 0.96 * torch.rand((nz, ny, nx), device="cuda", generator=gen))
    return g


@pytest.mark.parametrize("shapes", [
    [(512, 512, 3)] * 128 + [(100, 70, 9), (33, 40, 5)],     # 32800 items and more
    [(512, 500, 2 + k % 5) for k in range(40)],              # some 10000
])
def test_long_lists_equal_single_grids(shapes):
    args = [S.step_args(lam=3.0, dt=0.04, dF=0.01, stencil=26) for _ in shapes]
    grids = [_grid(s, k) for k, s in enumerate(shapes)]
    b = S.Batch(grids)
    b.step(3, args)
    for k, s in enumerate(shapes):
        g = _grid(s, k)
        g.step(3, lam=3.0, dt=0.04, dF=0.01, stencil=26)
        assert torch.equal(g.current(), grids[k].current()), k
        g.close()
    b.close()
