"""The range of the high-order closure's complex64 matvec.  A is linear, and scaling the operand by a power of two scales
every operation exactly as long as none leaves FP32's range, so upward the output is the scaled output bit for bit.
Downward the second halves of double-float values reach FP32's smallest numbers before the operand does; a ghost may then
round differently (2^-23 of itself), which a row of A multiplies by at most 2/h^2: tolerance 2^-22 max|U|/h^2.

Scaling every length by a power of two, with k^2 and k0 to match, scales A the same way: bit for bit."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_07711_gb300 import HELM_CLOSURE_HIGH_ORDER, Solver


def _apply(n, order, x, ppw=12, length=1.0):
    h = length / (max(n) - 1)
    k0 = 2 * math.pi / (ppw * h)
    S = Solver(n, np.full(n[::-1], k0 * k0, complex), k0, order=order, L=[h * (m - 1) for m in n], staggered=False)
    S.set_closure(HELM_CLOSURE_HIGH_ORDER)
    y = S.apply_A(x)
    S.close()
    return y, h


def _operand(n, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.complex(*(torch.randn(n[::-1], generator=g, device="cuda") for _ in range(2)))


@pytest.mark.parametrize("order", [2, 4, 6])
@pytest.mark.parametrize("n", [(8, 9, 10), (34, 33, 40), (100, 20, 12)])
@pytest.mark.parametrize("exponent", [-90, -60, 60, 90, 104])
def test_scaling_the_operand_scales_the_output(n, order, exponent):
    x = _operand(n, order)
    s = 2.0 ** exponent
    a, h = _apply(n, order, x)
    b, _ = _apply(n, order, (x * s).contiguous())
    a, b = torch.view_as_real(a).double() * s, torch.view_as_real(b).double()
    tol = 2.0 ** -22 * float(x.abs().max()) * s / h ** 2 if exponent < 0 else 0.0
    assert torch.isfinite(b).all() and float((a - b).abs().max()) <= tol


@pytest.mark.parametrize("order, exponent", [(4, -30), (4, 30), (6, 30)])   # (order 6, -30: its field k^4 is beyond FP32)
def test_scaling_the_lengths_scales_the_operator(order, exponent):
    n = (34, 33, 40)
    x = _operand(n, order)
    s = 2.0 ** (-2 * exponent)
    a, _ = _apply(n, order, x)
    b, _ = _apply(n, order, x, length=2.0 ** exponent)
    a, b = torch.view_as_real(a).double() * s, torch.view_as_real(b).double()
    assert torch.isfinite(b).all() and torch.equal(a, b)
