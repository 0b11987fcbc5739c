"""The constant-volume correction writes the ghost layer of the field it leaves
itself: the layer is the face kernel's bit for bit (rebuilt by it from the
same interior in a second grid), for every boundary mix, storage type and for
sizes around the 16-byte chunks and axes of one cell; and the fields match the
FP64 oracle within the parity bars (FP64 1e-12, FP32 2e-5).
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_05180_gb300 import spfm as S
from paper_1910_05180_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

P, N, C = S.SPFM_PERIODIC, S.SPFM_NOFLUX, S.SPFM_CONTACT
CASES = [((60, 13, 9), (P,) * 6), ((33, 18, 7), (P,) * 6), ((64, 16, 5), (C,) * 6), ((37, 9, 6), (N, C, P, P, C, N)),
         ((1, 8, 9), (P, P, C, C, N, N)), ((5, 1, 3), (C, N, N, N, P, P)), ((130, 3, 1), (N, N, P, P, P, P)),
         ((2, 2, 2), (P,) * 6)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


@pytest.mark.parametrize("dtype", [S.SPFM_F64, S.SPFM_F32, S.SPFM_BF16])
@pytest.mark.parametrize("shape,bc", CASES)
def test_ghosts_and_field_after_conserving_steps(shape, bc, dtype):
    rng = np.random.default_rng(sum(shape))
    n = WL.random_normal(rng)
    lam, dt, steps = 3.0, 0.05, 4
    p = O.Params(*shape, bc=bc, n=tuple(n), lam=lam, dt=dt, stencil=26)
    phi = 0.02 + 0.96 * rng.random(p.shape)
    start = torch.from_numpy(phi).to(S.TORCH_DTYPE[dtype])
    grids = [S.Grid(*shape, dtype=dtype, bc=bc, n=tuple(n)) for _ in range(2)]
    for g in grids:
        g.init_planar(0.0, lam)
        g.set_field(start.cuda())
    grids[0].step_conserving(steps, lam=lam, dt=dt, stencil=26)
    field = grids[0].get_field(to_host=False)
    grids[1].set_field(field)       # the face kernel rebuilds the layer
    assert torch.equal(grids[0].current_with_ghosts(), grids[1].current_with_ghosts())
    if dtype != S.SPFM_BF16:
        ref, _ = O.step_conserving(p, start.double().numpy(), steps)
        assert np.abs(field.double().cpu().numpy() - ref).max() <= (1e-12 if dtype == S.SPFM_F64 else 2e-5)
