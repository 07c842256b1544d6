"""The 16-bit chain where its z-solve keeps its lines in the ring of six blocks of eight steps (grids with more pairs of
lines than the SMs hold whole), at depths around the ring's and with a ragged last block, and the FP16 chain's norm of
inputs that are not finite.

Input, basis and the grids between the stages carry one rounding u each (2^-11 FP16, 2^-8 BF16), white like the input:
16 u of the whole result against FP32, as in test_gpu_tile_edges.py.  The same slice by slice, so that an error in one
block of eight steps is not diluted by the others: the sixteen roundings of a slice have the whole grid's error within a
factor of 2 where the slice's own norm is an average one, so 32 u of the average slice's norm."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_07711_gb300 import HELM_PREC_BF16, HELM_PREC_FP16, Solver


def _rand(shape, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.complex(*(torch.randn(shape, generator=g, device="cuda") for _ in range(2)))


@pytest.mark.parametrize("precision, u", [(HELM_PREC_FP16, 2.0 ** -11), (HELM_PREC_BF16, 2.0 ** -8)])
@pytest.mark.parametrize("n", [(208, 192, 41), (208, 192, 48), (208, 192, 49), (208, 192, 57), (240, 168, 104), (128, 308, 50)])
def test_chain_slice_by_slice(n, precision, u):
    nx, ny, nz = n
    k0 = 2 * math.pi * nx / 11
    k2 = np.full((nz, ny, nx), k0 * k0, complex)
    L = [m / nx for m in n]
    y = _rand((nz, ny, nx), nz)
    S = Solver(n, k2, k0, order=4, L=L)
    H = Solver(n, k2, k0, order=4, L=L, precision=precision, flexible=True)
    ref, z = S.apply_precond(y).to(torch.complex128), H.apply_precond(y).to(torch.complex128)
    e = (z - ref).flatten(1).norm(dim=1)
    assert float(e.norm() / ref.norm()) < 16 * u
    assert float(e.max() / (ref.norm() / math.sqrt(nz))) < 32 * u


@pytest.mark.parametrize("value", [math.nan, math.inf, -math.inf])
@pytest.mark.parametrize("where", [0, 1, 1031, 64 * 64 * 50 - 1])
def test_an_input_that_is_not_finite_gives_no_finite_output(value, where):
    """||r|| is then not finite either, and the last pass multiplies by it."""
    n = (64, 64, 50)
    k0 = 2 * math.pi / 10 * 64
    S = Solver(n, np.full(n[::-1], k0 * k0, complex), k0, order=4, L=(1.0, 1.0, 50 / 64), precision=HELM_PREC_FP16, flexible=True)
    y = _rand(n[::-1], 1)
    ref = S.apply_precond(y)
    for part in range(2):
        r = y.clone()
        torch.view_as_real(r).view(-1, 2)[where, part] = value
        assert not torch.isfinite(torch.view_as_real(S.apply_precond(r))).all(dim=-1).any()
    assert torch.equal(S.apply_precond(y), ref)
