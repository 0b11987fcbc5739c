"""TI_n steps on both of their tiles: grids whose extent reaches 32 lambda run on
32 x 32 cells, others on 64 x 16.  Extents around the tiles' edges, on both sides
of the line, periodic (images) and contact faces (staged ghosts), against the
FP64 oracle within the FP32 parity bar (2e-5), and bit for bit independent of the
z-chunk.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_05180_gb300 import spfm as S
from paper_1910_05180_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

P, C = S.SPFM_PERIODIC, S.SPFM_CONTACT


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


@pytest.mark.parametrize("shape,bc", [((32, 32, 32), (P,) * 6), ((64, 33, 35), (P,) * 6), ((96, 65, 34), (P,) * 6),
                                      ((70, 64, 33), (C,) * 6), ((101, 40, 32), (C,) * 6)])
@pytest.mark.parametrize("lam", [0.99, 1.1])
def test_local_normal_on_both_tiles(shape, bc, lam):
    n = WL.random_normal(np.random.default_rng(3))
    p = O.Params(*shape, bc=bc, n=tuple(n), lam=lam, dF=0.02, stencil=26, scheme=O.TI_LOCAL)
    # a noisy plane kept inside (0.005, 0.999): beyond the clamp FP32 and FP64 may
    # take the fallback on different cells
    phi = 0.005 + 0.99 * O.init_planar(p, float(n @ (np.array(shape) - 1) / 2.0))
    phi += 0.004 * np.random.default_rng(4).random(phi.shape)
    start = torch.from_numpy(phi).float()
    fields = []
    for zc in (0, 1, 5, shape[2]):
        g = S.Grid(*shape, dtype=S.SPFM_F32, bc=bc, n=tuple(n))
        p.dt = dt = 0.4 * g.max_dt(lam=lam, dF=0.02, stencil=26, scheme=S.SPFM_TI_LOCAL)
        g.set_zchunk(zc)
        g.set_field(start.cuda())
        g.step(3, lam=lam, dt=dt, dF=0.02, stencil=26, scheme=S.SPFM_TI_LOCAL)
        fields.append(g.get_field(to_host=True))
        g.close()
    assert all(torch.equal(f, fields[0]) for f in fields[1:])
    ref = O.step(p, start.double().numpy(), 3)
    assert np.abs(fields[0].double().numpy() - ref).max() <= 2e-5
