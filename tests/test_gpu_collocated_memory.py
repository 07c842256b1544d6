"""A collocated context holds the real fields of its medium (k^2 and, at order 6, four more floats a point) only while the
high-order closure's matvec reads them: with the three-point closure a real medium takes no more memory than one with
attenuation, whose fields are complex in any case."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_07711_gb300 import HELM_CLOSURE_HIGH_ORDER, HELM_CLOSURE_THREE_POINT, Solver

N = 128
SLACK = 4 << 20     # allocation granularity


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _context(order, loss):
    k0 = 2 * math.pi * (N - 1) / 12
    k2 = torch.full((N, N, N), complex(k0 * k0, loss), dtype=torch.complex128, device="cuda")
    before = _free()
    S = Solver((N, N, N), k2, k0, order=order, staggered=False)
    return S, before - _free()


@pytest.mark.parametrize("order", [4, 6])
def test_real_fields_are_held_for_the_high_order_closure_alone(order):
    warm, _ = _context(order, 1.0)
    warm.close()
    lossy, lossy_bytes = _context(order, 1.0)
    lossy.close()
    S, real_bytes = _context(order, 0.0)
    assert real_bytes <= lossy_bytes + SLACK
    x = torch.randn((N, N, N), dtype=torch.complex64, device="cuda")
    free = _free()
    S.set_closure(HELM_CLOSURE_HIGH_ORDER)
    first = S.apply_A(x)
    S.set_closure(HELM_CLOSURE_THREE_POINT)
    del first
    torch.cuda.empty_cache()
    assert _free() >= free - SLACK
    S.set_closure(HELM_CLOSURE_HIGH_ORDER)
    a, b = S.apply_A(x), S.apply_A(x)
    assert torch.equal(a, b) and torch.isfinite(torch.view_as_real(a)).all()
    S.close()
