"""Binned points around the size from which a block takes two rounds of points in the caller's order: the same
bits as the same chunks, permuted too, in calls below it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(1 << 20) - 1, (1 << 20) + 129, (1 << 20) + 1153])
def test_binned_points_in_calls_of_any_size(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import api, build
    build.build()
    gen = torch.Generator(device="cuda").manual_seed(n)
    z = np.linspace(-1.0, 0.2, 48).astype(np.float32)
    nodes = torch.randn((1, 48, 256, 512, 4), generator=gen, device="cuda")
    eta = torch.randn((1, 256, 512), generator=gen, device="cuda")
    grid = api.DeviceGrid(nodes, eta, 512, 256, z, np.array([0.0]), 8.0, 4.0, 0)
    pts = torch.rand((n, 3), generator=gen, device="cuda") * torch.tensor([8.0, 4.0, 1.2], device="cuda")
    pts[:, 2] -= 1.0
    perm, srt = api.bin_points(grid, pts)
    got, _ = api.interp_permuted(grid, 0.0, srt, perm)
    half = 1 << 19
    ident = [torch.arange(m, device="cuda", dtype=torch.int32) for m in (half, n - half)]
    a, _ = api.interp_permuted(grid, 0.0, srt[:half].contiguous(), ident[0])
    b, _ = api.interp_permuted(grid, 0.0, srt[half:].contiguous(), ident[1])
    for k, v in got.items():
        assert torch.equal(v[perm.long()], torch.cat([a[k], b[k]])), k
