"""Grids with no periodic face: the tiles that touch a face have their ghosts
built by the producer warp, the others read the staged planes as they land.
Grids with both kinds of tiles, in x, y and z, single (every storage type the
oracle holds) and in batches whose CTAs take items of both kinds in turn.

Bars: the parity bars (FP64 1e-12, FP32 2e-5); batches equal single grids bit for
bit.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_05180_gb300 import spfm as S
from paper_1910_05180_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

N, C = S.SPFM_NOFLUX, S.SPFM_CONTACT


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


def _field(shape, seed):
    nx, ny, nz = shape
    return 0.02 + 0.96 * np.random.default_rng(seed).random((nz, ny, nx))


@pytest.mark.parametrize("dtype,tol", [(S.SPFM_F64, 1e-12), (S.SPFM_F32, 2e-5)])
@pytest.mark.parametrize("scheme,oscheme", [(S.SPFM_TI_GLOBAL, O.TI_GLOBAL), (S.SPFM_TI_LOCAL, O.TI_LOCAL)])
@pytest.mark.parametrize("shape,zc", [((260, 70, 22), 5), ((192, 48, 13), 1), ((200, 65, 9), 4)])
def test_inner_and_face_tiles_match_the_oracle(shape, zc, scheme, oscheme, dtype, tol):
    bc = (C, N, N, C, C, C)
    n = WL.random_normal(np.random.default_rng(5))
    p = O.Params(*shape, bc=bc, n=tuple(n), lam=3.0, dt=0.02, dF=0.02, stencil=26, scheme=oscheme)
    start = torch.from_numpy(_field(shape, 1)).to(S.TORCH_DTYPE[dtype])
    g = S.Grid(*shape, dtype=dtype, bc=bc, n=tuple(n))
    g.set_zchunk(zc)
    g.set_field(start.cuda())
    g.step(3, lam=3.0, dt=0.02, dF=0.02, stencil=26, scheme=scheme)
    ref = O.step(p, start.double().numpy(), 3)
    assert np.abs(g.get_field(to_host=True).double().numpy() - ref).max() <= tol
    g.close()


@pytest.mark.parametrize("policy", [S.SPFM_TILES_WIDE, S.SPFM_TILES_SQUARE, S.SPFM_TILES_FIT])
def test_batches_of_inner_and_face_tiles_equal_single_grids(policy):
    shapes = [(200, 100, 40), (33, 17, 9), (100, 100, 24), (64, 64, 16), (200, 50, 12)]
    sets = []
    for _ in range(2):
        gs = []
        for k, shape in enumerate(shapes):
            n = WL.random_normal(np.random.default_rng(k))
            g = S.Grid(*shape, dtype=S.SPFM_F32, bc=(C,) * 6, n=tuple(n))
            g.set_field(torch.from_numpy(_field(shape, k)).float().cuda())
            gs.append(g)
        sets.append(gs)
    args = [S.step_args(lam=3.0, dt=0.05, dF=0.01, stencil=26) for _ in shapes]
    b = S.Batch(sets[0])
    b.set_tiles(policy)
    b.step(7, args)
    for g, a in zip(sets[1], args):
        g.step(7, lam=a.lam, dt=a.dt, dF=a.dF, stencil=26)
    for gb, ga in zip(*sets):
        assert torch.equal(gb.get_field(), ga.get_field())
    b.close()
