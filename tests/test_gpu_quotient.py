"""The FP64 step kernels' quotient against the division, which is correctly
rounded: equal bit for bit on normal operands of every size (a quotient that
differs would have to lie within 2^-50 ulp of a tie), and where the operands are
zeros, infinities, NaN, subnormal or leave the range of its exponents.
"""
import pytest
import torch

from paper_1910_05180_gb300 import spfm as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.load()


def _quotient(a, b):
    q = torch.empty_like(a)
    st = torch.cuda.current_stream().cuda_stream
    assert S.load().spfm_debug_quotient(a.numel(), a.data_ptr(), b.data_ptr(), q.data_ptr(), st) == S.SPFM_OK
    return q


def _same(q, want):
    bits = q.view(torch.int64) == want.view(torch.int64)
    assert bool((bits | (q.isnan() & want.isnan())).all())


@pytest.mark.parametrize("spread", [2, 300, 900])
def test_normal_operands(spread):
    gen = torch.Generator("cuda").manual_seed(spread)
    n = 4_000_000
    m = [torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) + 1.0 for _ in range(2)]
    e = [torch.randint(-spread, spread + 1, (n,), device="cuda", generator=gen) for _ in range(2)]
    a, b = (torch.ldexp(x, k) * torch.where(k % 2 == 0, 1.0, -1.0) for x, k in zip(m, e))
    _same(_quotient(a, b), a / b)


def test_special_operands():
    tiny, big = 2.0 ** -1074, 1.7976931348623157e308
    v = [0.0, 1.0, 1.5, 3.0, tiny, 3 * tiny, 2.0 ** -1022, 2.0 ** -400, 2.0 ** -401, 2.0 ** 400, 2.0 ** 399 * 1.999,
         2.0 ** 1023, big, float("inf"), float("nan")]
    v = torch.tensor(v + [-x for x in v], dtype=torch.float64, device="cuda")
    a, b = (x.flatten().contiguous() for x in torch.meshgrid(v, v, indexing="ij"))
    _same(_quotient(a, b), a / b)
