"""Forward and backward passes of the network recorded into CUDA graphs.  The activations live on grids whose halo has to
be zero; another shape in the same workspace puts its values there.  A replay must give what the eager call gives whatever
shape ran before it, and an eager call what it gave before whatever graph was replayed in between.  Outputs are compared
bit by bit; gradients are summed by atomics in FP32, whose order changes the last bits: 1e-4 of the layer's norm, where a
halo left over from another shape is an error of order 0.1 to 1."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_07711_gb300 import Net

BIG, SMALL = (12, 16, 20), (6, 10, 18)


def _inputs(shape, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    x = torch.randn((1, 5) + shape, generator=g, device="cuda").to(torch.bfloat16)
    return x, torch.randn((1, 2) + shape, generator=g, device="cuda")


def _eager(net, x, gy):
    net.zero_grad()
    y = net.forward(x)
    net.backward(gy)
    return y, net.unflatten(net.get_grads())


def _record(net, x, gy):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        net.zero_grad()
        y = net.forward(x)
        net.backward(gy)
    return graph, y


def _same(a, b):
    assert torch.equal(a[0], b[0])
    for k, v in b[1].items():
        assert abs(a[1][k] - v).max() <= 1e-4 * (v.astype("f8") ** 2).sum() ** 0.5, k


@pytest.mark.parametrize("width", [3, 6, 8, 14, 28])
def test_replays_and_eager_calls_of_two_shapes(width):
    net = Net(width, seed=2)
    big, small = _inputs(BIG, 1), _inputs(SMALL, 2)
    ref_big, ref_small = _eager(net, *big), _eager(net, *small)     # (the larger workspace first: no growth later)
    torch.cuda.synchronize()
    for first, second in ((small, big), (big, small)):
        want = ref_small if first is small else ref_big
        other = ref_big if first is small else ref_small
        _same(_eager(net, *first), want)
        graph, y = _record(net, *first)
        for _ in range(2):
            _same(_eager(net, *second), other)
            graph.replay()
            torch.cuda.synchronize()
            _same((y, net.unflatten(net.get_grads())), want)
            _same(_eager(net, *second), other)
            _same(_eager(net, *first), want)
    net.close()
