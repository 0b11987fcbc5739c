"""Ghosts built in staged planes whose ring slot is copied into again.

A chunk of up to four planes stages at most six planes, one per ring slot, so no
slot is filled twice; longer chunks refill slots whose earlier plane carried
ghost stores.  The fields do not depend on the chunk, so both must agree bit for
bit, on every storage type; in a batch the slots also pass from items that build
ghosts to items that do not.
"""
import numpy as np
import pytest
import torch

from paper_1910_05180_gb300 import spfm as S
from paper_1910_05180_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

N, C = S.SPFM_NOFLUX, S.SPFM_CONTACT


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


def _grid(shape, dtype, bc, seed):
    nx, ny, nz = shape
    n = WL.random_normal(np.random.default_rng(seed))
    g = S.Grid(*shape, dtype=dtype, bc=bc, n=tuple(n))
    phi = 0.02 + 0.96 * np.random.default_rng(seed + 1).random((nz, ny, nx))
    g.set_field(torch.from_numpy(phi).to(S.TORCH_DTYPE[dtype]).cuda())
    return g


@pytest.mark.parametrize("dtype", [S.SPFM_F64, S.SPFM_F32, S.SPFM_BF16])
@pytest.mark.parametrize("bc", [(C,) * 6, (C, N, N, C, C, N)])
@pytest.mark.parametrize("shape", [(150, 66, 40), (61, 15, 23)])
def test_refilled_slots_equal_fresh_ones(shape, bc, dtype):
    fields = []
    for zc in (4, 7, shape[2]):
        g = _grid(shape, dtype, bc, 3)
        g.set_zchunk(zc)
        g.step(6, lam=3.0, dt=0.04, dF=0.01, stencil=26)
        fields.append(g.get_field())
        g.close()
    assert torch.equal(fields[0], fields[1]) and torch.equal(fields[0], fields[2])


@pytest.mark.parametrize("dtype", [S.SPFM_F64, S.SPFM_F32, S.SPFM_BF16])
def test_slots_shared_by_items_with_and_without_ghosts(dtype):
    # several items a CTA, inner and face tiles in turn
    shapes = [(200, 200, 40), (260, 120, 33), (33, 17, 9)] + [(200, 130, 64)] * 6
    b = S.Batch([_grid(s, dtype, (C,) * 6, k) for k, s in enumerate(shapes)])
    b.step(5, [S.step_args(lam=3.0, dt=0.04, dF=0.01, stencil=26)] * len(shapes))
    for k, s in enumerate(shapes):
        g = _grid(s, dtype, (C,) * 6, k)
        g.set_zchunk(4)
        g.step(5, lam=3.0, dt=0.04, dF=0.01, stencil=26)
        assert torch.equal(b.grids[k].get_field(), g.get_field()), k
        g.close()
    b.close()
