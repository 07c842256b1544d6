"""The learned correction's convolutions at the edges of their tiling, against the CPU oracle's layers
(oracle/learned.py): grids large enough for the largest tile (1024 points) with a ragged last tile, rows longer
than a tile (three staged runs), rows shorter than 14 points (padded pitch), widths whose channels end inside a
cell of 8, and widths with more than 64 outputs (output slices, 128 accumulator rows, two input blocks).

The reference runs the oracle's layers on the roundings the network stores (every activation to BF16, every
gradient that enters a convolution to BF16), so what is left are FP32 sums (about 1e-6) and what they tip: a value
within 1e-6 of a rounding boundary moves by 2^-8, about one in 2000 (1e-4 in the 2-norm per layer: outputs within
2e-3); and a ReLU at zero, which adds or drops one point of a channel's gradient.  On the smallest grid here (96
points) one such point is 1/sqrt(96) of a channel and 1/8 of that in the norm over 64 channels, so gradients are
held to 4e-2.  A wrong index, tap or mask gives errors of order 1."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import learned as OL
from paper_2602_07711_gb300 import Net, helm


def _bf16(a):
    return torch.from_numpy(np.asarray(a, np.float32)).to(torch.bfloat16).to(torch.float64).numpy()


def _rel(a, b):
    return np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel())


def _forward(P, x):
    layer = lambda k, v: _bf16(np.maximum(OL.conv3(v, P[k + ".w"], P[k + ".b"]), 0))
    a1 = layer("c1", x)
    a2 = layer("c2", a1)
    p = _bf16(OL.avgpool2(a2))
    b1 = layer("c3", p)
    b2 = layer("c4", b1)
    u = np.concatenate([OL.upsample2(b2), a2], axis=1)
    d1 = layer("c5", u)
    return OL.conv3(d1, P["c6.w"], P["c6.b"]), dict(x=x, a1=a1, a2=a2, p=p, b1=b1, b2=b2, u=u, d1=d1)


def _backward(P, S, g):
    G = {}

    def through(k, inp, g):
        gx, G[k + ".w"], _ = OL.conv3_backward(inp, P[k + ".w"], _bf16(g))
        G[k + ".b"] = g.sum(axis=(0, 2, 3, 4))      # summed before the rounding
        return gx

    g = through("c6", S["d1"], g) * (S["d1"] > 0)
    gu = through("c5", S["u"], g)
    n = S["b2"].shape[1]
    B, C, Z, Y, X = gu.shape
    gb2 = gu[:, :n].reshape(B, n, Z // 2, 2, Y // 2, 2, X // 2, 2).sum(axis=(3, 5, 7)) * (S["b2"] > 0)
    g = through("c4", S["b1"], gb2) * (S["b1"] > 0)
    gp = through("c3", S["p"], g)
    g = (gu[:, n:] + OL.upsample2(gp) / 8.0) * (S["a2"] > 0)
    g = through("c2", S["a1"], g) * (S["a1"] > 0)
    through("c1", S["x"], g)
    return G


@pytest.mark.parametrize("width,shape,B", [(3, (40, 96, 90), 1), (2, (2, 4, 300), 2), (5, (4, 4, 2), 3), (12, (4, 6, 14), 1),
                                           (33, (2, 4, 22), 1), (64, (2, 4, 6), 2)])
def test_forward_and_backward_match_oracle(width, shape, B):
    rng = np.random.default_rng(width)
    net = Net(width, seed=1)
    P = {k: _bf16(v + (0.1 * rng.standard_normal(v.shape) if k.endswith(".b") else 0)) for k, v in OL.init(width, 5).items()}
    net.set_params(net.flatten(P))
    for again in range(2):          # a second shape in between: the workspace is laid out anew
        x = _bf16(rng.standard_normal((B, 5) + shape))
        t = rng.standard_normal((B, 2) + shape)
        xd = torch.from_numpy(x).to("cuda", torch.bfloat16)
        net.zero_grad()
        y = net.forward(xd)
        yo, saved = _forward(P, x)
        assert _rel(y.cpu().numpy().astype(np.float64), yo) < 2e-3
        gy = torch.empty_like(y)
        loss = torch.zeros(1, dtype=torch.float64, device="cuda")
        helm.helm_net_mse(y, torch.from_numpy(t).to("cuda", torch.float32), gy, loss)
        net.backward(gy)
        g = net.unflatten(net.get_grads())
        go = _backward(P, saved, OL.mse(yo, t)[1])
        for k in go:
            assert _rel(g[k].astype(np.float64), go[k]) < 4e-2, k
        net.forward(torch.zeros((1, 5, 2, 2, 4), dtype=torch.bfloat16, device="cuda"))
