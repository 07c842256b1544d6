"""The FP16 chain's own normalisation (helm_apply_precond) over the range of FP32 inputs.

M^-1 is linear and the chain runs on r / ||r||, so scaling r by a power of two must scale z by the same
power: the sums of squares, which lie outside FP32's range at these scales, are formed on scaled values.  Only
1/||r|| and ||r|| are rounded (to FP32, 6e-8 each), and a changed rounding of 1/||r|| would move FP16 roundings;
powers of two change neither significand, so the result is exact down to 2^-126.  Below that FP32 is subnormal: the
kernel's product and the reference's scaling each round to a multiple of 2^-149.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_07711_gb300 import HELM_PREC_FP16, Solver


@pytest.mark.parametrize("n", [(8, 6, 5), (32, 18, 11), (64, 64, 50)])
@pytest.mark.parametrize("exponent", [-100, -70, 70, 100])
def test_scaling_the_input_scales_the_output(n, exponent):
    nx, ny, nz = n
    k0 = 2 * math.pi / 10 * nx
    S = Solver(n, np.full((nz, ny, nx), k0 * k0, complex), k0, order=4, L=(1.0, ny / nx, nz / nx),
               precision=HELM_PREC_FP16, flexible=True)
    g = torch.Generator("cuda").manual_seed(nx)
    r = torch.complex(*(torch.randn((nz, ny, nx), generator=g, device="cuda") for _ in range(2)))
    s = 2.0 ** exponent
    a = S.apply_precond(r)
    b = S.apply_precond((r * s).contiguous())
    a, b = torch.view_as_real(a).double() * s, torch.view_as_real(b).double()
    assert ((a - b).abs() <= torch.where(a.abs() < 2.0 ** -126, 2.0 ** -149, 0.0)).all()


def test_zero_stays_zero():
    S = Solver((8, 6, 4), np.full((4, 6, 8), 25.0, complex), 5.0, order=4, precision=HELM_PREC_FP16, flexible=True)
    assert not S.apply_precond(torch.zeros((4, 6, 8), dtype=torch.complex64, device="cuda")).abs().any()
