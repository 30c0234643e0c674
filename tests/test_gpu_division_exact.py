"""The kernels' FP64 division rounds as IEEE division does on nearly every operand pair: with one
Newton-Raphson iteration the reciprocal carries about 40 bits, the remainder correction takes
the quotient's error before its last rounding to about 2^-80, and fewer than one quotient in a
million lies that close to a rounding boundary.  The bound of 1e-5 leaves a factor of ten; a
reciprocal of 20 bits (no iteration) leaves an error of 2^-40 and fails on every pair."""
import pytest
import torch

from paper_1407_1309_gb300 import capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")


@pytest.mark.parametrize("exponents", [1, 100], ids=["near_one", "wide"])
def test_quotients_are_correctly_rounded(exponents):
    gen = torch.Generator(device=DEV).manual_seed(4)
    m = 1 << 24

    def operands():
        x = 1 + torch.rand(m, generator=gen, device=DEV, dtype=torch.float64)
        e = torch.randint(-exponents, exponents + 1, (m,), generator=gen, device=DEV).double()
        return torch.ldexp(x, e)

    n, d = operands(), operands()
    q = torch.empty_like(n)
    capi.mpdata_selftest_division(n, d, q)
    torch.cuda.synchronize()
    ref = n / d
    differ = q != ref
    assert differ.double().mean().item() <= 1e-5
    assert (torch.abs(q - ref) <= torch.abs(ref) * 2.0 ** -52).all()
