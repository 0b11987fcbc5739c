"""Batches whose calls alternate between parameters of different step kernels (the
degree of the potential goes with lambda): each kernel's graph is captured once,
and the fields equal single grids' bit for bit.
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


def test_alternating_parameters_capture_once():
    shapes = [(48, 40, 24), (64, 64, 16), (33, 20, 12)]

    def grids():
        out = []
        for k, (nx, ny, nz) in enumerate(shapes):
            g = S.Grid(nx, ny, nz, dtype=S.SPFM_F32, bc=(C,) * 6,
                       n=tuple(WL.random_normal(np.random.default_rng(k))))
            phi = 0.02 + 0.96 * np.random.default_rng(10 + k).random((nz, ny, nx))
            g.set_field(torch.from_numpy(phi).float().cuda())
            out.append(g)
        return out

    # degrees up to 4, 5 or 6, and above; then CF
    calls = [dict(lam=6.0), dict(lam=2.0), dict(lam=1.0), dict(lam=4.0, scheme=S.SPFM_FD)]
    batch, single = grids(), grids()
    b = S.Batch(batch, stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    counts = []
    for _ in range(3):
        for kw in calls:
            b.step(16, [S.step_args(dt=0.02, **kw) for _ in shapes])
            for g in single:
                g.step(16, dt=0.02, **kw)
        counts.append(S.load().spfm_debug_batch_captures(b.handle))
    torch.cuda.synchronize()
    assert counts[0] == counts[2] and 2 <= counts[0] <= len(calls)
    for x, y in zip(batch, single):
        assert torch.equal(x.current(), y.current())
    # a fifth kernel takes the place of the one used longest ago
    b.step(16, [S.step_args(dt=0.02, lam=6.0, stencil=18) for _ in shapes])
    for g in single:
        g.step(16, dt=0.02, lam=6.0, stencil=18)
    torch.cuda.synchronize()
    for x, y in zip(batch, single):
        assert torch.equal(x.current(), y.current())
    assert S.load().spfm_debug_batch_captures(b.handle) == counts[0] + 1
    b.close()
