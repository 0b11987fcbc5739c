"""The step kernels' forms of the TI potential on the GPU: every degree a grid
can take, cells below the form's range of q (phi outside [0, 1], summed group
by group), and batches that mix degrees.

Bars as in the parity tests: FP64 1e-12, FP32 2e-5 against the FP64 oracle (one
step of a random field: each FP32 update rounds to 2^-23 of values below 1.5,
and the increment, below 0.1, carries the rounding of some 60 operations); a
batch equals its grids stepped alone bit for bit.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_05180_gb300 import spfm as S
from paper_1910_05180_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

C, P = S.SPFM_CONTACT, S.SPFM_PERIODIC
TOL = {S.SPFM_F64: 1e-12, S.SPFM_F32: 2e-5}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


@pytest.mark.parametrize("dtype", [S.SPFM_F64, S.SPFM_F32])
@pytest.mark.parametrize("u", [(1, 0, 0), (1, 1, 1), (1, 2, 0), None])
@pytest.mark.parametrize("lam,dt", [(1.0, 2e-4), (1.5, 5e-3), (2.0, 0.02), (2.5, 0.02), (4.0, 0.05), (6.0, 0.05)])
def test_step_matches_the_oracle_at_every_degree(dtype, u, lam, dt):
    """Random phi reaching past [0, 1] up to half way to the first pole."""
    rng = np.random.default_rng(int(100 * lam) + (0 if u is None else sum(u)))
    n = WL.random_normal(rng)
    uu = tuple(WL.unit(u)) if u else tuple(n)
    amax = max(np.tanh(2 * np.dot(d, uu) / lam) ** 2 for d in ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (0, 1, 1),
               (1, 0, 1), (1, -1, 0), (0, 1, -1), (1, 0, -1), (1, 1, 1), (-1, 1, 1), (1, -1, 1), (1, 1, -1)))
    s_hi = np.sqrt(1 + 0.5 * (1 / amax - 1))          # |1 - 2 phi| below this
    over = min(0.5 * (s_hi - 1), 0.2)
    for shape, bc in (((37, 19, 9), (C,) * 6), ((64, 18, 7), (P,) * 6)):
        p = O.Params(*shape, bc=bc, n=tuple(n), u=uu, lam=lam, dt=dt, dF=0.02, stencil=26)
        phi = rng.random(p.shape)
        wild = rng.random(p.shape) < 0.02              # a few cells a row outside [0, 1]
        phi[wild] = np.where(rng.random(wild.sum()) < 0.5, -over, 1 + over)
        start = torch.from_numpy(phi).to(S.TORCH_DTYPE[dtype])
        g = S.Grid(*shape, dtype=dtype, bc=bc, n=tuple(n), u=uu)
        g.set_field(start.cuda())
        g.step(1, lam=lam, dt=dt, dF=0.02, stencil=26)
        got = g.get_field(to_host=True).double().numpy()
        ref = O.step(p, start.double().numpy(), 1)
        assert np.abs(got - ref).max() <= TOL[dtype]
        g.close()


@pytest.mark.parametrize("dtype", [S.SPFM_F32, S.SPFM_F64])
@pytest.mark.parametrize("lams", [(6.0, 4.0, 6.0), (2.0, 6.0, 3.0), (1.0, 6.0, 2.0)])
def test_mixed_degrees_in_a_batch_equal_single_grids_bitwise(dtype, lams):
    rng = np.random.default_rng(11)
    jobs = [(lam, WL.random_normal(rng), u) for lam, u in zip(lams, (None, (1, 2, 0), None))]
    sets = []
    for _ in range(2):
        gs = []
        for k, (lam, n, u) in enumerate(jobs):
            shape = [(37, 21, 19), (48, 40, 12), (20, 20, 33)][k]
            g = S.Grid(*shape, dtype=dtype, bc=(C,) * 6, n=tuple(n), u=tuple(WL.unit(u)) if u else (0.0, 0.0, 0.0))
            phi = np.random.default_rng(k).random((shape[2], shape[1], shape[0])) * 1.06 - 0.03
            g.set_field(torch.from_numpy(phi).to(S.TORCH_DTYPE[dtype]).cuda())
            gs.append(g)
        sets.append(gs)
    args = [S.step_args(lam=lam, dt=2e-4, dF=0.01, stencil=26) for lam, _, _ in jobs]
    b = S.Batch(sets[0])
    b.step(5, args)
    for g, a in zip(sets[1], args):
        g.step(5, lam=a.lam, dt=a.dt, dF=a.dF, stencil=26)
    for gb, ga in zip(*sets):
        assert torch.equal(gb.get_field(), ga.get_field())
    b.close()
