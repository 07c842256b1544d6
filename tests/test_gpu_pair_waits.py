"""Expired waits of the 16-bit passes on CTA pairs (sides above 128 points), in a form that faults and hangs nothing: a
limit of one poll makes the bounded waits run out, the two CTAs of a pair give up at different points, the leader settles
the loads that only one of them issued, and the solve reports it.  The context then gives what it gave before."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_07711_gb300 import HELM_PREC_BF16, HELM_PREC_FP16, Solver

HELM_ERR_ITER_LIMIT = 9


@pytest.mark.parametrize("precision", [HELM_PREC_FP16, HELM_PREC_BF16])
@pytest.mark.parametrize("n", [(144, 144, 40), (256, 64, 24), (64, 256, 24), (148, 132, 12)])
def test_solve_reports_expired_waits_and_the_context_stays_usable(n, precision):
    nx, ny, nz = n
    k0 = 2 * math.pi * max(n) / 11
    g = torch.Generator("cuda").manual_seed(nx)
    b = torch.complex(*(torch.randn((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64) for _ in range(2)))
    k2 = torch.full((nz, ny, nx), k0 * k0, dtype=torch.complex128, device="cuda")
    S = Solver(n, k2, k0, order=4, L=[m / max(n) for m in n], precision=precision, flexible=True, max_iter=4)
    y = b.to(torch.complex64)
    ref = S.apply_precond(y)
    for _ in range(3):
        S.set_wait_limit(1)
        _, info = S.solve(b, check=False)
        assert info.status == HELM_ERR_ITER_LIMIT
        S.set_wait_limit(0)
        assert torch.equal(S.apply_precond(y), ref)
    S.close()
