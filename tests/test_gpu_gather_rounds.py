"""Gather of scattered points around the size from which a block takes two rounds of points: the same
bits as the same chunks in calls below it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(1 << 20) - 1, 1 << 20, (1 << 20) + 1, (1 << 20) + 129, (1 << 20) + 1153])
def test_two_rounds_equal_one(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import api, build
    build.build()
    gen = torch.Generator(device="cuda").manual_seed(n)
    z = np.linspace(-1.0, 0.2, 48).astype(np.float32)
    nodes = torch.randn((1, 48, 256, 512, 4), generator=gen, device="cuda")   # four times the points
    eta = torch.randn((1, 256, 512), generator=gen, device="cuda")
    grid = api.DeviceGrid(nodes, eta, 512, 256, z, np.array([0.0]), 8.0, 4.0, 0)
    pts = torch.rand((n, 3), generator=gen, device="cuda") * torch.tensor([8.0, 4.0, 1.2], device="cuda")
    pts[:, 2] -= 1.0
    got, _ = api.interp(grid, 0.0, pts)
    half = 1 << 19
    a, _ = api.interp(grid, 0.0, pts[:half].contiguous())
    b, _ = api.interp(grid, 0.0, pts[half:].contiguous())
    for k, v in got.items():
        assert torch.equal(v, torch.cat([a[k], b[k]])), k
