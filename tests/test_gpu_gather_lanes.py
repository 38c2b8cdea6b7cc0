"""Untiled chunks whose points follow the grid's rows (binned points, layers), on grids whose four levels of all
time levels exceed L2: a point a lane, beside chunks by quads, in both routes of many points, over what
reaches them (node counts, schemes, one to four time levels, a permuted order, ragged ends). The same
points some at a time (quads) agree to the rounding of two summation orders of the same FP32 products,
about 1e-6 of a field's maximum; bar 1e-5. The plan's marks are those of the points' order."""
import numpy as np
import pytest

from wavegen import seas

pytestmark = pytest.mark.gpu
ROWS = 1 << 28


@pytest.mark.parametrize("nx,ny,pad,nz,scheme,n_tl,n,order", [
    (512, 512, 4, 9, "lagrange3", 1, 700_003, "binned"),
    (512, 512, 2, 24, "spline3", 4, 600_129, "layers"),
    (256, 512, 3, 24, "lagrange3", 3, 550_001, "layers"),
    (256, 512, 3, 24, "spline3", 2, 550_007, "binned"),
    (512, 512, 2, 24, "lagrange3", 3, (1 << 21) + 77, "layers"),
    (256, 512, 3, 96, "spline3", 2, (1 << 21) + 1025, "mixed"),
    (512, 512, 2, 24, "lagrange3", 2, 600_000, "none"),
])
def test_lanes_match_calls_of_few_points(nx, ny, pad, nz, scheme, n_tl, n, order):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import api
    rng = np.random.default_rng(nx + pad)
    Lx, Ly = nx / 16, ny / 16
    sea = seas.linear_sea(nx, ny, Lx, Ly, seas.random_linear_components(nx, ny, Lx, Ly, 8, 0.01, rng))
    z = np.linspace(-1.0, 0.08, nz).astype(np.float32)
    tl = [0.05 * i for i in range(n_tl)]
    t = 0.4 * tl[-1]
    assert n < 0.25 * pad * nx * pad * ny * nz
    grid = api.fields_on_grid(api.upload_modes(sea), z, pad, tl, scheme=scheme)
    gen = torch.Generator(device="cuda").manual_seed(nx)
    pts = torch.rand((n, 3), generator=gen, device="cuda") * torch.tensor([Lx, Ly, 1.085], device="cuda")
    pts[:, 2] -= 1.0                                            # some above the grid
    perm = None
    if order in ("binned", "mixed"):
        perm, pts = api.bin_points(grid, pts)
    if order == "layers":                                       # rows of points 9 nodes apart, layer by layer
        i = torch.arange(n, device="cuda")
        w = pad * nx // 9
        pts[:, 0] = (i % w + 0.3 * pts[:, 0] / Lx) * Lx / w
        pts[:, 1] = ((i // w) * 0.37 + 0.01 * pts[:, 1]) % Ly
        pts[:, 2] = -0.9 + 0.9 * (i // 30_000).float() / (n / 30_000)
    if order == "mixed":                                        # every other chunk in no order
        i = torch.arange(n, device="cuda")
        odd = (i // 1024) % 2 == 1
        pts[odd] = pts[odd][torch.randperm(int(odd.sum()), generator=gen, device="cuda")]
    if perm is None and order != "none":                        # a caller that permutes says so (below 2^21 points)
        perm = torch.arange(n, device="cuda", dtype=torch.int32)
    plan = api.interp_plan(grid, pts).view(torch.int32).view(-1, 4)
    marked = float((((plan[:, 2] & ROWS) != 0) & (plan[:, 3] < 0)).float().mean())
    assert {"binned": marked > 0.8, "layers": marked > 0.8, "mixed": 0.3 < marked < 0.7, "none": marked < 0.05}[order], marked

    out, oor = (api.interp(grid, t, pts, count_out_of_range=True) if perm is None else
                api.interp_permuted(grid, t, pts, perm, count_out_of_range=True))
    assert oor == int(((pts[:, 2] < float(z[0])) | (pts[:, 2] > float(z[-1]))).sum())
    few = [api.interp(grid, t, pts[i:i + 100_000].contiguous())[0] for i in range(0, n, 100_000)]
    for k in out:
        a, b = out[k], torch.cat([f[k] for f in few])
        if perm is not None:
            a = a[perm.long()]
        assert torch.equal(torch.isnan(a), torch.isnan(b)), k
        a, b = torch.nan_to_num(a), torch.nan_to_num(b)
        assert float((a - b).abs().max()) <= 1e-5 * float(b.abs().max()), k
