"""The work a user of this framework has it do, as measured cases: the solver's building blocks (operator,
preconditioner, learned correction) through their public entry points, and two whole calls (one solve, one
batch of solves).  Sizes are those of the paper's tables and of this repository's tests and workloads, with
ragged grids beside the cubes.

Every input is made from the seed alone on the GPU.  `exact` computes what `run` returns in 64 bits with
plain torch: the discretisations written out on padded grids, the preconditioner by full diagonalisation, the
network by shifted matrix products, a solve by iterative refinement to 1e-13.
"""
import math

import numpy as np
import torch

from paper_2602_07711_gb300 import Batch, HELM_CLOSURE_HIGH_ORDER, Net, Solver
from paper_2602_07711_gb300.helm import helm_net_mse

DEV = "cuda"
FP32, TF32, FP16 = 0, 1, 4     # transform precisions (helm.h)
EIGT, PFFT = 1, 2              # preconditioners
RTOL = 1e-10                   # rel-res of the paper's tables (Sec. 5.1)


def _apply(what, n, **kw):
    nx, ny, nz = n
    c = dict(kind=what, nx=nx, ny=ny, nz=nz, order=6, ppw=10.0, medium="bumps", staggered=True, precision=FP32,
             precond=EIGT)
    c.update(kw)
    return c


def listed():
    return [
        # one preconditioner application in the default precision on the smallest workload's grid (fourth order,
        # 8 points per wavelength): launches and latency
        dict(_apply("precond", (32, 32, 32), order=4, ppw=8.0), name="precond_fp32_32"),
        # the default precision on a grid of the paper's tables that no tile divides
        dict(_apply("precond", (200, 200, 200)), name="precond_fp32_200"),
        # tensor-core transforms on a ragged box
        dict(_apply("precond", (150, 100, 75), order=4, precision=TF32), name="precond_tf32_150x100x75"),
        # the preconditioner of the headline solve
        dict(_apply("precond", (256, 256, 256), precision=FP16), name="precond_fp16_256"),
        # PFFT on an FFT-friendly grid (layered medium, 8 points per wavelength)
        dict(_apply("precond", (256, 256, 256), precision=TF32, precond=PFFT, ppw=8.0), name="precond_pfft_256"),
        # the matvec of the headline solve: sixth order, real medium
        dict(_apply("matvec", (256, 256, 256), precision=FP16), name="matvec6_256"),
        # the matvec of the scattering table: an attenuating inclusion, so complex k^2
        dict(_apply("matvec", (200, 200, 200), medium="lossy"), name="matvec6_lossy_200"),
        # the matvec of the paper's high-order tables: collocated grid, high-order closure
        dict(_apply("matvec", (100, 100, 100), medium="constant", staggered=False, precision=TF32, ppw=30.0),
             name="matvec6_closure_100"),
        # inference of the learned correction (the ~200K-parameter network) on one field
        dict(kind="net", width=28, batch=1, nx=160, ny=160, nz=160, grad=False, name="net_forward_160"),
        # one training pass of that network on a minibatch of two 96^3 fields: output, loss, every gradient
        dict(kind="net", width=28, batch=2, nx=96, ny=96, nz=96, grad=True, name="net_train_96"),
        # the headline problem solved: right-hand side and flexible GMRES(30), FP16 chain and basis
        dict(_apply("solve", (256, 256, 256), precision=FP16), name="solve_fp16_256"),
        # a batch of uneven problems, two right-hand sides each, in one prepared plan
        dict(kind="batch", sizes="48,64,96,48,64,96", orders="4,6,6,6,4,4", rhs=2, precision=TF32, ppw=9.0,
             name="batch_48_96"),
    ]


def _size(rng, lo, hi):
    """A size spread over lo..hi by its logarithm, even (the point count of a grid has to be)."""
    return 2 * int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2))


def draw(rng):
    kind = rng.choice(["precond", "precond", "precond", "pfft", "matvec", "matvec", "closure", "net", "net", "solve",
                       "batch"])
    if kind == "net":
        grad = rng.random() < 0.5
        top = 96 if grad else 160
        return dict(kind="net", width=rng.choice([8, 12, 16, 28, 32]), batch=rng.choice([1, 2]) if grad else 1,
                    nx=_size(rng, 16, top), ny=_size(rng, 16, top), nz=_size(rng, 16, top), grad=grad)
    if kind == "batch":
        k = rng.randint(2, 6)
        return dict(kind="batch", sizes=",".join(str(rng.choice([48, 64, 96])) for _ in range(k)),
                    orders=",".join(str(rng.choice([4, 6])) for _ in range(k)), rhs=rng.choice([1, 2]),
                    precision=rng.choice([FP32, TF32]), ppw=round(rng.uniform(8.0, 12.0), 2))
    if kind == "pfft":
        n = [rng.choice([32, 64, 128, 256]) for _ in range(2)]
        return _apply("precond", (n[0], n[1], _size(rng, 20, 256)), precond=PFFT, precision=rng.choice([FP32, TF32]),
                      ppw=round(rng.uniform(8.0, 12.0), 2))
    if kind == "closure":
        n = _size(rng, 32, 200)
        return _apply("matvec", (n, _size(rng, 32, 200), n), medium="constant", staggered=False,
                      order=rng.choice([4, 6]), precision=TF32, ppw=round(rng.uniform(10.0, 60.0), 2))
    precision = rng.choice([FP32, TF32, FP16])
    order = rng.choice([4, 6])
    ppw = round(rng.uniform(8.0, 12.0), 2)
    if kind == "solve":
        n = 4 * int(round(math.exp(rng.uniform(math.log(32), math.log(128))) / 4))
        return _apply("solve", (n, n, n), order=order, ppw=ppw, precision=precision)
    top = 200 if precision == FP32 and kind == "precond" else 256
    nx, ny, nz = (_size(rng, 32, top) for _ in range(3))
    if precision == FP16:
        nx = nx // 4 * 4
    if rng.random() < 0.5:
        ny += 1                    # odd rows and planes
        nz -= 1
    return _apply(kind, (nx, ny, nz), order=order, ppw=ppw, precision=precision,
                  medium=rng.choice(["bumps", "bumps", "lossy"]) if kind == "matvec" else "bumps")


# ---- inputs --------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _geometry(c):
    """Step h (cubic cells, the x edge is 1) and k0 of a case's grid."""
    h = 1.0 / (c["nx"] if c["staggered"] else c["nx"] - 1)
    return h, 2.0 * math.pi / (c["ppw"] * h)


def _mesh(c, h):
    o = 0.5 if c["staggered"] else 0.0
    ax = [(torch.arange(c[k], dtype=torch.float64, device=DEV) + o) * h for k in ("nz", "ny", "nx")]
    return ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]


def _medium(c, seed, h, k0):
    """k^2 samples: 20 Gaussian bumps of contrast up to 30%, a sphere of the paper's scattering contrast with
    attenuation, or the constant of its test problem."""
    Z, Y, X = _mesh(c, h)
    rng = np.random.default_rng(seed)
    L = (X[..., -1].item(), Y[0, -1].item(), Z[-1].item())
    rel = torch.ones((c["nz"], c["ny"], c["nx"]), dtype=torch.complex128, device=DEV)
    if c["medium"] == "bumps":
        for _ in range(20):
            a, s = rng.uniform(-0.3, 0.3), rng.uniform(0.03, 0.08)
            p = [rng.uniform(0.2, 0.8) * v for v in L]
            rel += a * torch.exp(-(X - p[0]) ** 2 / (2 * s * s)) * torch.exp(-(Y - p[1]) ** 2 / (2 * s * s)) * \
                torch.exp(-(Z - p[2]) ** 2 / (2 * s * s))
    elif c["medium"] == "lossy":
        p = [rng.uniform(0.3, 0.7) * v for v in L]
        rel[((X - p[0]) ** 2 + (Y - p[1]) ** 2 + (Z - p[2]) ** 2) <= 0.2 ** 2] = (1050 + 2.26j) / 439.2
    return (k0 * k0 * rel).contiguous()


def _waves(c, g, h, k0, count=4):
    """A sum of plane waves of wavenumber k0 with random directions and amplitudes."""
    Z, Y, X = _mesh(c, h)
    d = torch.randn(count, 3, generator=g, dtype=torch.float64, device=DEV)
    d = (d / d.norm(dim=1, keepdim=True)).tolist()
    a = torch.randn(count, 2, generator=g, dtype=torch.float64, device=DEV).tolist()
    u = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.complex128, device=DEV)
    for (dx, dy, dz), (ar, ai) in zip(d, a):
        u += complex(ar, ai) * torch.exp(1j * k0 * dx * X) * torch.exp(1j * k0 * dy * Y) * torch.exp(1j * k0 * dz * Z)
    return u


def _noise(shape, g):
    return torch.complex(*(torch.randn(shape, generator=g, dtype=torch.float32, device=DEV) for _ in range(2)))


def _grid_inputs(c, seed):
    """k^2, k0, h and the operand: a Krylov vector (broad-band) for M^-1, a preconditioned one (wave-like) for A,
    the source of a plane wave scattered by the medium for a solve."""
    h, k0 = _geometry(c)
    g = _gen(seed)
    k2 = _medium(c, seed, h, k0)
    u = _waves(c, g, h, k0, 1 if c["kind"] == "solve" else 4)
    if c["kind"] == "solve":
        return k2, k0, h, (-(k2 - k0 * k0) * u).contiguous()
    noise = _noise(u.shape, g)
    return k2, k0, h, (u.to(torch.complex64) + (0.02 if c["kind"] == "matvec" else 0.5) * noise).contiguous()


def _solver(c, k2, k0, h):
    n = (c["nx"], c["ny"], c["nz"])
    L = tuple(h * (m if c["staggered"] else m - 1) for m in n)
    S = Solver(n, k2, k0, order=c["order"], L=L, precond=c["precond"], precision=c["precision"], restart=30,
               rtol=RTOL, flexible=c["precision"] != FP32, staggered=c["staggered"])
    if not c["staggered"]:
        S.set_closure(HELM_CLOSURE_HIGH_ORDER)
    return S


def _net_inputs(c, seed):
    """Parameters (He initialisation, small biases, a small last layer), input features and targets."""
    g = _gen(seed)
    w = c["width"]
    layers = [(w, 5), (w, w), (2 * w, w), (2 * w, 2 * w), (w, 3 * w), (2, w)]
    params = []
    for k, (co, ci) in enumerate(layers):
        std = math.sqrt(2.0 / (27 * ci)) * (0.1 if k == 5 else 1.0)
        params.append((std * torch.randn(co, ci, 3, 3, 3, generator=g, device=DEV),
                       0.05 * torch.randn(co, generator=g, device=DEV)))
    field = dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], staggered=True, medium="bumps", kind="net")
    h = 1.0 / c["nx"]
    k0 = 2.0 * math.pi / (8.0 * h)
    xs = []
    for b in range(c["batch"]):
        v = _noise((c["nz"], c["ny"], c["nx"]), g)
        m = _waves(field, g, h, k0)
        m = m / m.abs().square().mean().sqrt()
        xs.append(torch.stack([v.real, v.imag, m.real.float(), m.imag.float(),
                               (_medium(field, seed + 7 * b, h, k0).real / (k0 * k0) - 1.0).float()]))
    x = torch.stack(xs).to(torch.bfloat16).contiguous()
    t = torch.randn((c["batch"], 2) + tuple(x.shape[2:]), generator=g, device=DEV)
    return params, x, t


def _batch_problems(c, seed):
    """Per problem: its case, k^2, k0, h and the sources of its right-hand sides."""
    out = []
    for p, (n, order) in enumerate(zip(c["sizes"].split(","), c["orders"].split(","))):
        n = int(n)
        q = _apply("solve", (n, n, n), order=int(order), precision=c["precision"], ppw=c["ppw"])
        h, k0 = _geometry(q)
        k2 = _medium(q, seed + 31 * p, h, k0)
        g = _gen(seed + 31 * p)
        out.append((q, k2, k0, h, [(-(k2 - k0 * k0) * _waves(q, g, h, k0, 1)).contiguous() for _ in range(c["rhs"])]))
    return out


def prepare(case, seed):
    if case["kind"] == "net":
        params, x, t = _net_inputs(case, seed)
        net = Net(case["width"], seed=0)
        net.set_params(torch.cat([v.reshape(-1) for wb in params for v in wb]).cpu().numpy())
        return dict(kind="net", grad=case["grad"], net=net, x=x, t=t, gy=torch.empty_like(t),
                    loss=torch.zeros(1, dtype=torch.float64, device=DEV))
    if case["kind"] == "batch":
        solvers, bs = [], []
        for q, k2, k0, h, fs in _batch_problems(case, seed):
            S = _solver(q, k2, k0, h)
            solvers.append(S)
            bs.append(torch.stack([S.build_rhs(f) for f in fs]).contiguous())
        xs = [torch.zeros_like(b) for b in bs]
        return dict(kind="batch", plan=Batch(solvers, bs, xs), xs=xs)
    k2, k0, h, v = _grid_inputs(case, seed)
    return dict(kind=case["kind"], solver=_solver(case, k2, k0, h), v=v)


def run(state):
    kind = state["kind"]
    if kind == "precond":
        return state["solver"].apply_precond(state["v"])
    if kind == "matvec":
        return state["solver"].apply_A(state["v"])
    if kind == "solve":
        S = state["solver"]
        return S.solve(S.build_rhs(state["v"]))[0]
    if kind == "batch":
        for x in state["xs"]:
            x.zero_()
        state["plan"].run()
        return state["xs"]
    net = state["net"]
    if not state["grad"]:
        return net.forward(state["x"])
    net.zero_grad()
    y = net.forward(state["x"])
    state["loss"].zero_()
    helm_net_mse(y, state["t"], state["gy"], state["loss"])
    net.backward(state["gy"])
    return {"y": y, "loss": state["loss"], "grads": net.get_grads()}


def _points(c):
    return c["nx"] * c["ny"] * c["nz"]


def _precond_flops(c):
    p = _points(c)
    if c["precond"] == PFFT:   # two sine transforms each way as FFTs of length 2n, three z-solves
        return p * (2 * 5 * 2 * (math.log2(2 * c["nx"]) + math.log2(2 * c["ny"])) + 3 * 20)
    return p * (16.0 * (c["nx"] + c["ny"]) + 20)   # complex products of length nx, ny, both ways; z-solves


def work(case):
    if case["kind"] == "net":
        w, v = case["width"], case["batch"] * _points(case)
        macs = 27 * v * (5 * w + w * w + 3 * w * w + 2 * w + (2 * w * w + 4 * w * w) / 8.0)
        # inputs and outputs; a training pass adds the targets, and a data and a weight gradient per layer
        return {"bytes": v * (5 * 2 + 2 * 4) + (v * 8 if case["grad"] else 0), "flops": 2 * macs * (3 if case["grad"] else 1)}
    if case["kind"] == "batch":
        w = [work(_apply("solve", (int(n),) * 3, precision=case["precision"])) for n in case["sizes"].split(",")]
        return {k: case["rhs"] * sum(v[k] for v in w) for k in ("bytes", "flops")}
    p = _points(case)
    if case["kind"] == "matvec":   # x and k^2 read, y written; 27 points, a complex multiply-add each
        return {"bytes": p * (16 + (8 if case["medium"] == "lossy" else 4)), "flops": p * 27 * 8}
    if case["kind"] == "precond":
        return {"bytes": p * 16, "flops": _precond_flops(case)}
    # a solve: about 40 iterations of preconditioner, matvec and orthogonalisation against 7 vectors on average
    basis = 4 if case["precision"] == FP16 else 8
    return {"bytes": p * (32 + 40 * (16 + 20 + (2 * 7 + 1) * basis + 16)), "flops": 40 * (_precond_flops(case) + p * 400)}


# ---- what run returns, in 64 bits ------------------------------------------------------------------------
def _pad_mirror(k2, staggered, width):
    """Mirror extension about the face (staggered) or about the boundary node (collocated)."""
    for d in range(3):
        n = k2.shape[d]
        i = torch.arange(-width, n + width, device=DEV)
        i = torch.where(i < 0, -1 - i if staggered else -i, i)
        i = torch.where(i >= n, 2 * n - 1 - i if staggered else 2 * n - 2 - i, i)
        k2 = k2.index_select(d, i)
    return k2


def _second_derivative(n, h):
    """Sixth-order second derivative on n nodes, one-sided over eight nodes near the ends."""
    D = np.zeros((n, n))
    for i in range(n):
        idx = np.arange(i - 3, i + 4) if 3 <= i <= n - 4 else (np.arange(8) if i < 3 else np.arange(n - 8, n))
        o = (idx - i).astype(float)
        A = np.stack([o ** q / math.factorial(q) for q in range(len(o))])
        D[i, idx] = np.linalg.solve(A, np.eye(len(o))[2]) / h ** 2
    return torch.from_numpy(D).to(DEV).to(torch.complex128)


class _Operator:
    """The compact schemes of orders 4 and 6 on a padded grid, complex128 (k^2 h^2-scaled weights)."""

    def __init__(self, c, k2, k0, h):
        self.c, self.h, self.k0 = c, h, k0
        self.gamma = (2 + 1j * k0 * h) / (2 - 1j * k0 * h)
        self.K = _pad_mirror(k2, c["staggered"], 1)
        if not c["staggered"]:
            self.D = {n: _second_derivative(n, h) for n in {m + e for m in (c["nx"], c["ny"], c["nz"]) for e in (0, 2)}}
        if c["order"] == 6:
            Q = _pad_mirror(k2, c["staggered"], 2)
            at = lambda d, s: self._cut(Q, d, s, 2)
            self.dk = [(-at(d, 2) + 8 * at(d, 1) - 8 * at(d, -1) + at(d, -2)) / (12 * h) for d in range(3)]
            self.lap = sum((-at(d, 2) + 16 * at(d, 1) - 30 * at(d, 0) + 16 * at(d, -1) - at(d, -2)) / (12 * h * h)
                           for d in range(3))

    @staticmethod
    def _cut(P, d, s, w):
        """The unknowns of an array padded by w, shifted by s along array axis d."""
        for a in range(3):
            P = P.narrow(a, w + (s if a == d else 0), P.shape[a] - 2 * w)
        return P

    def _ghosts(self, U):
        nz, ny, nx = U.shape
        P = torch.zeros((nz + 2, ny + 2, nx + 2), dtype=U.dtype, device=DEV)
        P[1:-1, 1:-1, 1:-1] = U
        for d in (2, 1, 0):     # x, then y, then z; a later face covers the ghosts already filled
            Q = P.movedim(d, 0)
            if self.c["staggered"]:
                Q[0], Q[-1] = self.gamma * Q[1], self.gamma * Q[-2]
                continue
            ext = [slice(None) if t > d else slice(1, -1) for t in range(3) if t != d]
            F = Q[:, ext[0], ext[1]]
            Da, Db = self.D[F.shape[1]], self.D[F.shape[2]]
            for g, b, i in ((0, 1, 2), (-1, -2, -3)):
                V, G = F[b].clone(), F[i].clone()
                for m in range(3):
                    G = G + 2 * self.h ** (2 * m + 1) / math.factorial(2 * m + 1) * (-1) ** m * 1j * self.k0 * V
                    V = self.k0 ** 2 * V + Da @ V + V @ Db.T
                F[g] = G
        return P

    @staticmethod
    def _d2(P, d):
        """Second difference along array axis d, which loses its two end layers."""
        n = P.shape[d]
        return P.narrow(d, 0, n - 2) - 2 * P.narrow(d, 1, n - 2) + P.narrow(d, 2, n - 2)

    @staticmethod
    def _mid(P, axes):
        for a in axes:
            P = P.narrow(a, 1, P.shape[a] - 2)
        return P

    def __call__(self, U):
        P, K, h2 = self._ghosts(U), self.K, self.h ** 2
        d2, mid = self._d2, self._mid
        one = lambda A: sum(mid(d2(A, d), [a for a in range(3) if a != d]) for d in range(3))
        two = lambda A: sum(mid(d2(d2(A, a), b), [3 - a - b]) for a, b in ((0, 1), (0, 2), (1, 2)))
        k, u = mid(K, (0, 1, 2)), mid(P, (0, 1, 2))
        if self.c["order"] == 4:
            KU = K * P
            return one(P) / h2 + two(P) / (6 * h2) + mid(KU, (0, 1, 2)) + one(KU) / 12
        out = one((1 + h2 / 30 * K) * P) / h2 + d2(d2(d2(P, 0), 1), 2) / (30 * h2) + k * u + \
            two((1 + h2 / 15 * K) * P) / (6 * h2) + h2 / 20 * (self.lap - k * k) * u
        P6 = (1 + h2 / 6 * K) * P
        for d in range(3):
            o = [a for a in range(3) if a != d]
            T = sum(mid(d2(P, a), [b for b in o if b != a]) for a in o)   # still padded along d
            W = mid(P6, o) + T / 6
            n = W.shape[d]
            out = out + h2 / 20 * 2 * self.dk[d] * (W.narrow(d, 2, n - 2) - W.narrow(d, 0, n - 2)) / (2 * self.h)
        return out


class _Inverse:
    """h^2 A_p^-1 (Sec. 4.1) by full diagonalisation in complex128."""

    def __init__(self, c, k0, h):
        self.V, lam = [], []
        gamma, zeta = ((2 + 1j * k0 * h) / (2 - 1j * k0 * h), 1.0) if c["staggered"] else (2j * k0 * h, 2.0)
        for n in (c["nz"], c["ny"], c["nx"]):
            A = np.diag(np.ones(n - 1), 1) + np.diag(np.ones(n - 1), -1) + 0j
            A[0, 0] = A[-1, -1] = gamma
            A[0, 1] = A[-1, -2] = zeta
            w, V = np.linalg.eig(A)
            self.V.append([torch.from_numpy(np.ascontiguousarray(M)).to(DEV) for M in (V, np.linalg.inv(V))])
            lam.append(torch.from_numpy(w).to(DEV))
        self.d = h * h / (lam[0][:, None, None] + lam[1][None, :, None] + lam[2][None, None, :] + (h * k0) ** 2 - 6)

    def __call__(self, r):
        V = [[m.to(r.dtype) for m in p] for p in self.V]
        for k in (1, 0):
            if k == 0:
                r = self.d.to(r.dtype) * r
            r = (r.reshape(-1, r.shape[2]) @ V[2][k].T).reshape(r.shape)
            r = V[1][k] @ r
            r = (V[0][k] @ r.reshape(r.shape[0], -1)).reshape(r.shape)
        return r


def _rhs(c, f, k2, op):
    """The schemes' right-hand sides from samples of f with mirror extension."""
    h = op.h
    if c["order"] == 4:
        P = _pad_mirror(f, True, 1)
        return f + sum(op._cut(P, d, 1, 1) - 2 * f + op._cut(P, d, -1, 1) for d in range(3)) / 12
    Q = _pad_mirror(f, True, 2)
    at = lambda d, s: op._cut(Q, d, s, 2)
    lap = sum(-at(d, 2) + 16 * at(d, 1) - 30 * f + 16 * at(d, -1) - at(d, -2) for d in range(3)) / 12
    pure = sum(at(d, 2) - 4 * at(d, 1) + 6 * f - 4 * at(d, -1) + at(d, -2) for d in range(3))
    P = _pad_mirror(f, True, 1)
    mix = sum(op._mid(op._d2(op._d2(P, a), b), [3 - a - b]) for a, b in ((0, 1), (0, 2), (1, 2)))
    grad = sum(op.dk[d] * (at(d, 1) - at(d, -1)) / (2 * h) for d in range(3))
    return f + lap / 12 + pure / 360 + mix / 90 - h * h / 20 * (k2 * f - h * h / 3 * grad)


def _solve(c, k2, k0, h, fs):
    """A^-1 b to a residual of 1e-13 by iterative refinement: complex128 residuals, corrections by flexible
    GMRES in complex64."""
    A, M = _Operator(c, k2, k0, h), _Inverse(c, k0, h)
    A32 = _Operator(c, k2, k0, h)
    A32.K = A32.K.to(torch.complex64)
    if c["order"] == 6:
        A32.dk, A32.lap = [v.to(torch.complex64) for v in A32.dk], A32.lap.to(torch.complex64)
    xs = []
    for f in fs:
        b = _rhs(c, f, k2, A)
        x = torch.zeros_like(b)
        for _ in range(12):
            r = b - A(x)
            if r.norm() <= 1e-13 * b.norm():
                break
            beta = float(r.norm())
            V, Z, H = [(r / beta).to(torch.complex64).reshape(-1)], [], np.zeros((41, 40), complex)
            for j in range(40):
                Z.append(M(V[j].reshape(b.shape)))
                w = A32(Z[j]).reshape(-1)
                for i in range(j + 1):
                    H[i, j] = complex(torch.vdot(V[i], w))
                    w = w - H[i, j] * V[i]
                H[j + 1, j] = float(w.norm())
                V.append(w / H[j + 1, j].real)
                e = np.zeros(j + 2, complex)
                e[0] = beta
                y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
                if np.linalg.norm(e - H[:j + 2, :j + 1] @ y) <= 2e-5 * beta:
                    break
            for yi, z in zip(y, Z):
                x = x + complex(yi) * z.to(torch.complex128)
        xs.append(x)
    return xs


def _conv(x, w, b):
    """3x3x3 convolution with zero padding as 27 shifted matrix products, float64."""
    B, _, Z, Y, X = x.shape
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    out = b[None, :, None].expand(B, -1, Z * Y * X)
    for t in range(27):
        dz, dy, dx = t // 9, t // 3 % 3, t % 3
        out = out + w[:, :, dz, dy, dx] @ xp[:, :, dz:dz + Z, dy:dy + Y, dx:dx + X].reshape(B, x.shape[1], -1)
    return out.reshape(B, -1, Z, Y, X)


def _net_exact(c, seed):
    params, x, t = _net_inputs(c, seed)
    p = [tuple(v.double().requires_grad_(c["grad"]) for v in wb) for wb in params]
    with torch.set_grad_enabled(c["grad"]):
        a1 = _conv(x.double(), *p[0]).relu()
        a2 = _conv(a1, *p[1]).relu()
        b2 = _conv(_conv(torch.nn.functional.avg_pool3d(a2, 2), *p[2]).relu(), *p[3]).relu()
        up = b2.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)
        y = _conv(_conv(torch.cat([up, a2], 1), *p[4]).relu(), *p[5])
        if not c["grad"]:
            return y
        loss = 0.5 * (y - t.double()).square().mean()
    g = torch.autograd.grad(loss, [v for wb in p for v in wb])
    return {"y": y.detach(), "loss": loss.detach().reshape(1), "grads": torch.cat([v.reshape(-1) for v in g])}


def exact(case, seed):
    if case["kind"] == "net":
        return _net_exact(case, seed)
    if case["kind"] == "batch":
        return [torch.stack(_solve(q, k2, k0, h, fs)) for q, k2, k0, h, fs in _batch_problems(case, seed)]
    k2, k0, h, v = _grid_inputs(case, seed)
    if case["kind"] == "precond":
        return _Inverse(case, k0, h)(v.to(torch.complex128))
    if case["kind"] == "matvec":
        return _Operator(case, k2, k0, h)(v.to(torch.complex128))
    return _solve(case, k2, k0, h, [v])[0]
