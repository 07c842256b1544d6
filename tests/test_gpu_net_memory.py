"""The workspace of a forward pass: cells of 8 channels on grids with a halo of one point (rows of at least 16 cells, a
slack of 4096 cells behind each tensor), channel counts rounded up to 8 and no further."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_07711_gb300 import Net

GRANULE = 2 << 20    # allocations are rounded up to this, one for each of nine arrays


def _cells(channels, n):
    return ((channels + 7) // 8 * (n + 2) ** 2 * max(16, n + 2) + 4096) * 16


@pytest.mark.parametrize("width", [1, 4, 8, 20])
def test_workspace_of_a_forward_pass(width):
    n, c = 96, width
    x = torch.zeros((1, 5, n, n, n), dtype=torch.bfloat16, device="cuda")
    y = torch.empty((1, 2, n, n, n), device="cuda")
    net = Net(width)
    from paper_2602_07711_gb300 import helm
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    assert helm.lib().helm_net_forward(net.h, helm._ptr(x), helm._ptr(y), 1, n, n, n, helm._stream(None)) == 0
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    want = n ** 3 * (5 * 2 + 2 * 4) + sum(_cells(k, n) for k in (5, c, 3 * c, c)) + sum(_cells(k, n // 2) for k in (c, 2 * c, 2 * c))
    assert used <= want + 9 * GRANULE
    net.close()
