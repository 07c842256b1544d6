"""The network's convolutions in the forms that grids of real size take: two 128-point blocks a tile, each with its own
issuing warp, and two to eight output planes per MMA at 16, 32, 48 and 64 padded outputs, with ragged last tiles, last
groups of planes and odd channel groups.  (Small grids take one block and one plane; tests of the tiling's other edges
are in test_gpu_learned_cells.py.)  On 152 SMs, per layer (blocks, planes, padded outputs):
  width 28, 36 x 96 x 90           2, 4, 32 (5 -> 28, 28 -> 28, 84 -> 28); data gradient 28 -> 84: 2, 2, 64 and 1, 4, 32
  width 36, two of 20 x 64 x 64    2, 2, 48; 108 outputs: 2, 2, 64
  width 20, 44 x 64 x 260          rows longer than a tile: 2, 4, 32; 2, 8, 16; 2, 2, 64; half resolution 1, 2, 48

The reference is the oracle's network on the roundings that the library stores (every activation, and every gradient that
enters a convolution, to BF16), in float64 torch.  What is left are FP32 sums (1e-6) and what they tip.  Outputs: a value
within 1e-6 of a BF16 rounding boundary moves by 2^-8, one in 2000, 1e-4 in the 2-norm a layer: 2e-3 as in
test_gpu_learned_cells.py.  Gradients: the same per layer, twelve layers of them, and a ReLU at zero that adds or drops a
point of a channel's gradient: one value in a million, at most one or two of the 8e4 to 7e5 points of a channel, each
1/sqrt(8e4) = 3.5e-3 of its norm and less over all channels: 5e-3.  A wrong index, tap, mask or plane gives errors of order 1."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import torch.nn.functional as F

from oracle import learned as OL
from paper_2602_07711_gb300 import Net, helm


def _bf16(t):
    return t.to(torch.bfloat16).to(torch.float64)


def _rel(a, b):
    return float((a - b).norm() / b.norm())


def _conv(x, w, b=None):
    return F.conv3d(x, w, b, padding=1)


def _forward(P, x):
    layer = lambda k, v: _bf16(_conv(v, P[k + ".w"], P[k + ".b"]).clamp(min=0))
    a1 = layer("c1", x)
    a2 = layer("c2", a1)
    p = _bf16(F.avg_pool3d(a2, 2))
    b1 = layer("c3", p)
    b2 = layer("c4", b1)
    u = torch.cat([F.interpolate(b2, scale_factor=2, mode="nearest"), a2], 1)
    d1 = layer("c5", u)
    return _conv(d1, P["c6.w"], P["c6.b"]), dict(x=x, a1=a1, a2=a2, p=p, b1=b1, b2=b2, u=u, d1=d1)


def _backward(P, S, g):
    G = {}

    def through(k, inp, g):
        r, w = _bf16(g), P[k + ".w"]
        G[k + ".w"] = torch.nn.grad.conv3d_weight(inp, w.shape, r, padding=1)
        G[k + ".b"] = g.sum(dim=(0, 2, 3, 4))            # summed before the rounding
        return torch.nn.grad.conv3d_input(inp.shape, w, r, padding=1)

    def children(t):
        return 8 * F.avg_pool3d(t, 2)

    g = through("c6", S["d1"], g) * (S["d1"] > 0)
    gu = through("c5", S["u"], g)
    n = S["b2"].shape[1]
    g = through("c4", S["b1"], children(gu[:, :n]) * (S["b2"] > 0)) * (S["b1"] > 0)
    gp = through("c3", S["p"], g)
    g = (gu[:, n:] + F.interpolate(gp, scale_factor=2, mode="nearest") / 8) * (S["a2"] > 0)
    g = through("c2", S["a1"], g) * (S["a1"] > 0)
    through("c1", S["x"], g)
    return G


@pytest.mark.parametrize("width,shape,batch", [(28, (36, 96, 90), 1), (36, (20, 64, 64), 2), (20, (44, 64, 260), 1)])
def test_large_tiles_match_the_oracle(width, shape, batch):
    rng = np.random.default_rng(width)
    net = Net(width, seed=1)
    P = {k: v + (0.1 * rng.standard_normal(v.shape) if k.endswith(".b") else 0) for k, v in OL.init(width, 5).items()}
    D = {k: _bf16(torch.from_numpy(v).float().cuda()) for k, v in P.items()}
    net.set_params(net.flatten({k: v.cpu().numpy() for k, v in D.items()}))
    g = torch.Generator("cuda").manual_seed(width)
    x = torch.randn((batch, 5) + shape, generator=g, device="cuda").to(torch.bfloat16)
    t = torch.randn((batch, 2) + shape, generator=g, device="cuda")
    net.zero_grad()
    y = net.forward(x)
    yo, saved = _forward(D, x.to(torch.float64))
    assert _rel(y.double(), yo) < 2e-3
    gy = torch.empty_like(y)
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    helm.helm_net_mse(y, t, gy, loss)
    net.backward(gy)
    got = net.unflatten(net.get_grads())
    want = _backward(D, saved, gy.double())
    for k, v in want.items():
        assert _rel(torch.from_numpy(got[k].astype(np.float64)).cuda(), v) < 5e-3, k
    net.close()
