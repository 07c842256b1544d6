"""Batch plans own what their captured launches address.  A plan lives on while its contexts serve other calls: a
second, larger plan of the same contexts, single solves and preconditioner applications between its runs must not
change what it computes, whatever scratch they make the contexts grow.  The kernels, their data and their order are the
same in every run of a plan, so the results are compared bit by bit.

The grids are wide enough (more pairs of lines than the SMs hold whole) for the z-solve's ring form, which keeps its
checkpoints in device memory, and small enough for the right-hand sides to run as independent branches."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_07711_gb300 import HELM_PREC_FP16, HELM_PREC_FP32, HELM_PREC_TF32, Batch, Solver


def _problem(n, nrhs, precision, seed=3):
    nx, ny, nz = n
    k0 = 2 * math.pi * nx / 12
    g = torch.Generator("cuda").manual_seed(seed)
    k2 = (k0 * k0 * (1 + 0.1 * torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64))).to(torch.complex128)
    S = Solver(n, k2, k0, order=4, L=(1.0, ny / nx, nz / nx), precision=precision, flexible=True, rtol=1e-5, max_iter=40)
    B = torch.complex(*(torch.randn((nrhs, nz, ny, nx), generator=g, device="cuda", dtype=torch.float64) for _ in range(2)))
    return S, B.contiguous()


def _run(plan):
    for x in plan.xs:
        x.zero_()
    code, infos = plan.run()
    return [x.clone() for x in plan.xs], [[i.iterations for i in p] for p in infos]


@pytest.mark.parametrize("precision", [HELM_PREC_FP32, HELM_PREC_TF32])
@pytest.mark.parametrize("n", [(48, 40, 20), (208, 192, 20)])
def test_two_plans_of_one_context(n, precision):
    S, B = _problem(n, 3, precision)
    one = Batch([S], [B[:1].contiguous()], [torch.zeros_like(B[:1])])
    x1, it1 = _run(one)
    three = Batch([S], [B], [torch.zeros_like(B)])      # more right-hand sides on the same context
    x3, it3 = _run(three)
    S.solve(B[0].contiguous(), check=False)
    S.apply_precond(B[1].to(torch.complex64))
    again, it = _run(one)
    assert it == it1 and torch.equal(again[0], x1[0])
    again, it = _run(three)
    assert it == it3 and torch.equal(again[0], x3[0])
    # the right-hand side both plans share
    assert it3[0][0] == it1[0][0] and torch.equal(x3[0][0], x1[0][0])
    for r in range(3):
        xs, info = S.solve(B[r].contiguous(), check=False)
        assert info.iterations == it3[0][r]
        assert float((x3[0][r] - xs).norm() / xs.norm()) < 1e-9
    one.close()
    three.close()
    S.close()


@pytest.mark.parametrize("n", [(48, 48, 48), (64, 36, 20), (128, 304, 20)])
def test_concurrent_fp16_lanes_keep_their_stage_norms_apart(n):
    """Four right-hand sides of very different sizes of one FP16 context, as independent branches of one graph: each
    lane is bit for bit what it is alone in a plan (where nothing runs beside it), in every run."""
    S, B = _problem(n, 4, HELM_PREC_FP16, seed=5)
    B[1] *= 1e-3
    B[2, :, :, : n[0] // 4] = 0
    plan = Batch([S], [B], [torch.zeros_like(B)])
    runs = [_run(plan) for _ in range(4)]
    alone = []
    for r in range(4):
        one = Batch([S], [B[r:r + 1].contiguous()], [torch.zeros_like(B[:1])])
        alone.append(_run(one))
        one.close()
    for x, it in runs:
        for r in range(4):
            assert it[0][r] == alone[r][1][0][0]
            assert torch.equal(x[0][r], alone[r][0][0][0])
    plan.close()
    S.close()
