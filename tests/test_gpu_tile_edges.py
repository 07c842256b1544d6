"""Kernels at the edges of their tilings, against the CPU oracle, through the C-ABI.

FP32 transform passes: lengths on both sides of the GEMM's tile widths (32 .. 64 columns, 32 rows a warp, 128 a
tile) and K blocks (16), odd ones included.  A pass sums K products of FP32 operands in order: 2-norm error a few
times sqrt(K) 2^-24, two passes; bound 8 sqrt(K) 2^-24.
z-solves: depths on both sides of the blocks of 8 steps whose inner ones run without end conditions; bound 1e-4
(the systems amplify FP32 rounding, here by a few hundred at most).  Wide grids: the same where the lines do not fit
the SMs whole and pass through the ring of 6 blocks, and the whole FP16 chain there against FP32 within a few hundred
2^-11.
16-bit transform chain: sides below, at and above the 128 rows and 256 columns at which the passes go to CTA pairs,
ragged blocks, several vectors' worth of rows.  Input, basis entries and the grids between the stages carry one rounding u
(2^-11, 2^-8) each, white like the input, so each adds about u relative to the result: bound 16 u against FP32.
Complex64 matvec: every kernel variant, grids from the smallest to several chunk lengths, real and complex k^2, and
the padded form of the high-order closure (an output that overlaps the operand included).  The terms of A U are up
to 8/h^2 |U| and cancel to k^2 U, each rounded to 2^-24: bound 32 2^-24 / (k0 h)^2.
Wrong indices or weights give errors of order 1 in each."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.eigt import EigT
from oracle.grid import Grid
from oracle.operators import Operator
from oracle.tridiag import thomas
from paper_2602_07711_gb300 import HELM_C64, HELM_CLOSURE_HIGH_ORDER, HELM_PREC_BF16, HELM_PREC_FP16, Solver, helm


def _rand(shape, seed):
    r = np.random.default_rng(seed)
    return r.standard_normal(shape) + 1j * r.standard_normal(shape)


def _rel(a, b):
    return np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel())


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.complex64)


def _grid(n, staggered=True):
    big = max(n)
    return Grid(*n, *[(m if staggered else m - 1) / big for m in n], staggered=staggered)


def _library_basis(S, g, k0):
    """The oracle's EigT in the library's order and scaling of the eigenvectors."""
    e = EigT(g, k0)
    e.Dx, e.Vx, e.Vxi = S.get_eig(0)
    e.Dy, e.Vy, e.Vyi = S.get_eig(1)
    return e


@pytest.mark.parametrize("n", [(5, 33, 4), (16, 17, 6), (40, 56, 4), (57, 65, 4), (64, 129, 5), (130, 48, 7), (199, 100, 4),
                               (256, 31, 16)])
def test_fp32_transform_passes(n):
    g = _grid(n)
    k0 = 2 * math.pi * max(n) / 11
    S = Solver(n, np.full(g.shape, k0 * k0, complex), k0, order=4, L=g.L)
    e = _library_basis(S, g, k0)
    y = _rand(g.shape, n[0])
    bound = 8 * math.sqrt(max(n[:2])) * 2.0 ** -24
    assert _rel(S.precond_step(1, _dev(y)).cpu().numpy(), e.forward(y)) < bound
    assert _rel(S.precond_step(3, _dev(y)).cpu().numpy(), e.inverse(y)) < bound


@pytest.mark.parametrize("nz", [4, 7, 8, 9, 15, 16, 17, 24, 25, 64, 511])
def test_z_solves(nz):
    n = (12, 10, nz)
    g = Grid(*n, 12 / 40, 10 / 40, nz / 40)
    k0 = 2 * math.pi * 40 / 11
    S = Solver(n, np.full(g.shape, k0 * k0, complex), k0, order=4, L=g.L)
    e = _library_basis(S, g, k0)
    y = _rand(g.shape, nz)
    assert _rel(S.precond_step(2, _dev(y)).cpu().numpy(), thomas(*e.z_coefficients(), y)) < 1e-4


@pytest.mark.parametrize("nz", [4, 9, 40, 41, 48, 49, 57])
def test_z_solves_wide(nz):
    n = (208, 192, nz)
    L = [m / 208 for m in n]
    k0 = 2 * math.pi * 208 / 11
    k2 = np.full((nz, 192, 208), k0 * k0, complex)
    S = Solver(n, k2, k0, order=4, L=L)
    e = _library_basis(S, Grid(*n, *L), k0)
    y = _rand(k2.shape, nz)
    assert _rel(S.precond_step(2, _dev(y)).cpu().numpy(), thomas(*e.z_coefficients(), y)) < 1e-4
    H = Solver(n, k2, k0, order=4, L=L, precision=HELM_PREC_FP16, flexible=True)
    assert _rel(H.apply_precond(_dev(y)).cpu().numpy(), S.apply_precond(_dev(y)).cpu().numpy()) < 0.1


PAIR_SIZES = [(128, 128, 5), (132, 129, 4), (160, 250, 7), (148, 200, 33), (256, 256, 9), (260, 257, 4), (64, 192, 20)]


@pytest.mark.parametrize("precision, u", [(HELM_PREC_FP16, 2.0 ** -11), (HELM_PREC_BF16, 2.0 ** -8)])
@pytest.mark.parametrize("n", PAIR_SIZES)
def test_16_bit_passes(n, precision, u):
    big = max(n)
    k0 = 2 * math.pi * big / 11
    k2 = np.full(n[::-1], k0 * k0, complex)
    L = [m / big for m in n]
    y = _dev(_rand(k2.shape, n[2]))
    S = Solver(n, k2, k0, order=4, L=L)
    H = Solver(n, k2, k0, order=4, L=L, precision=precision, flexible=True)
    ref = S.apply_precond(y).cpu().numpy()
    assert _rel(H.apply_precond(y).cpu().numpy(), ref) < 16 * u


def test_expired_waits_of_the_pair_passes_leave_the_context_usable():
    n = (144, 144, 40)
    k0 = 2 * math.pi * 144 / 11
    k2 = np.full(n[::-1], k0 * k0, complex)
    S = Solver(n, k2, k0, order=4, L=(1, 1, 40 / 144), precision=HELM_PREC_FP16, flexible=True)
    y = _dev(_rand(k2.shape, 3))
    ref = S.apply_precond(y)
    S.set_wait_limit(1)      # one poll a wait
    try:
        S.apply_precond(y)
    except RuntimeError:
        pass
    S.set_wait_limit(0)
    assert torch.equal(S.apply_precond(y), ref)


@pytest.mark.parametrize("lossy", [False, True])
@pytest.mark.parametrize("order", [4, 6])
@pytest.mark.parametrize("n", [(4, 4, 4), (33, 9, 6), (31, 18, 40), (66, 41, 33), (96, 64, 80)])
def test_matvec_variants(n, order, lossy):
    g = _grid(n)
    k0 = 2 * math.pi * max(n) / 10
    k2 = k0 * k0 * (1 + 0.2 * np.cos(3 * g.mesh()[0]) * np.sin(2 * g.mesh()[2])).astype(complex)
    if lossy:
        k2 = k2 + 0.02j * k0 * k0
    S = Solver(n, k2, k0, order=order, L=g.L)
    x = _rand(g.shape, n[1])
    ref = Operator(g, k2, k0, order)(x)
    for v in range(5):
        S.set_matvec_variant(v)
        assert _rel(S.apply_A(_dev(x)).cpu().numpy(), ref) < 32 * 2.0 ** -24 / (k0 * g.h[0]) ** 2, v


@pytest.mark.parametrize("order", [2, 4, 6])
@pytest.mark.parametrize("n,ppw", [((8, 8, 8), 10), ((34, 9, 12), 12), ((40, 33, 64), 60), ((64, 10, 9), 25)])
def test_closure_matvec(n, ppw, order):
    g = _grid(n, staggered=False)
    k0 = 2 * math.pi / (ppw * g.h[0])
    k2 = np.full(g.shape, k0 * k0, complex)
    S = Solver(n, k2, k0, order=order, L=g.L, staggered=False)
    S.set_closure(HELM_CLOSURE_HIGH_ORDER)
    X, Y, Z = g.mesh()
    x = np.exp(1j * k0 * (0.6 * X + 0.8 * Z)) + 0.1 * np.exp(-1j * k0 * Y)
    ref = Operator(g, k2, k0, order, rule="collocated_ho")(x)
    bound = 32 * 2.0 ** -24 / (k0 * g.h[0]) ** 2 * np.linalg.norm(x) * k0 ** 2 / np.linalg.norm(ref)
    xd = _dev(x)
    assert _rel(S.apply_A(xd).cpu().numpy(), ref) < bound
    helm.helm_apply_A(S.ctx, xd, xd, HELM_C64)
    assert _rel(xd.cpu().numpy(), ref) < bound


@pytest.mark.parametrize("precision", [helm.HELM_PREC_FP32, helm.HELM_PREC_TF32, helm.HELM_PREC_TF32X3, HELM_PREC_FP16])
@pytest.mark.parametrize("n", [(16, 10, 7), (100, 64, 40), (160, 144, 24)])
def test_passes_started_early_see_their_predecessors_results(n, precision):
    """Back-to-back preconditioners, in place too, against the same with every launch in plain stream order (as it is
    while the passes are timed): the kernels are the same, so the results are."""
    big = max(n)
    k0 = 2 * math.pi * big / 10
    k2 = np.full(n[::-1], k0 * k0, complex)
    S = Solver(n, k2, k0, order=4, L=[m / big for m in n], precision=precision, flexible=True)
    x = [_dev(_rand(k2.shape, v)) for v in range(6)]

    def run():
        r = []
        for _ in range(4):
            r = [S.apply_precond(v) for v in x]
        z = x[0].clone()
        for _ in range(3):
            helm.helm_apply_precond(S.ctx, z, z)
        return r + [z]

    early = run()
    L = helm.lib()
    assert L.helm_profile(S.ctx, 1) == 0
    plain = run()
    assert L.helm_profile(S.ctx, 0) == 0
    for a, b in zip(early, plain):
        assert torch.equal(a, b)
