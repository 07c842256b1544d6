"""PFFT's boundary correction at the edges of its kernels' ranges: the smallest and largest transform lengths
(frame sums in groups of 4096 points, matrix rows in blocks of 64, vectors in blocks of 8) and slice counts that
are no multiple of the z-solve's blocks of 8.  PFFT and EigT invert the same A_p, so the reference is the oracle's
EigT; the bound is the largest FP32 one of the PFFT suite (2.3e-4 in the 2-norm: three chained solves)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.eigt import EigT
from oracle.grid import Grid
from paper_2602_07711_gb300 import HELM_PRECOND_PFFT, Solver


@pytest.mark.parametrize("staggered", [True, False])
@pytest.mark.parametrize("n", [(4, 4, 4), (4, 64, 9), (512, 4, 7), (8, 512, 10), (128, 32, 41)])
def test_matches_the_exact_inverse(n, staggered):
    nx, ny, nz = n
    big = max(n)
    L = tuple((m if staggered else m - 1) / big for m in n)
    g = Grid(*n, *L, staggered=staggered)
    k0 = 2 * math.pi * big / 12
    S = Solver(n, np.full(g.shape, k0 * k0, complex), k0, order=4, L=L, precond=HELM_PRECOND_PFFT, staggered=staggered)
    r = np.random.default_rng(nx + nz)
    y = r.standard_normal(g.shape) + 1j * r.standard_normal(g.shape)
    z = S.apply_precond(torch.from_numpy(y).to("cuda", torch.complex64)).cpu().numpy()
    ref = EigT(g, k0).apply_Minv(y)
    err = np.linalg.norm(z - ref) / np.linalg.norm(ref)
    assert err < 2.3e-4, err
