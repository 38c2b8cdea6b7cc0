"""The gather of many points on a fine grid from the layers' shared planes, over what reaches it: node counts
that are and are not powers of two, both schemes, one to four time levels, a permuted order, layers above
the grid, points among them that are in no layer, and layers that leave chunks across two z. The same
points some at a time (no planes) agree to the rounding of two summation orders of the same FP32 products,
about 1e-6 of a field's maximum; bar 1e-5."""
import numpy as np
import pytest

from wavegen import seas

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,pad,nz,scheme,n_tl,permuted,per", [
    (64, 32, 8, 90, "lagrange3", 1, False, 104_857),
    (64, 32, 8, 90, "spline3", 4, True, 104_857),
    (256, 128, 3, 40, "lagrange3", 3, True, 131_072),
    (256, 128, 3, 40, "spline3", 2, False, 104_857),
    (256, 128, 3, 40, "lagrange3", 1, False, 300_007),
    (512, 64, 2, 96, "spline3", 3, False, 90_001),
    (32, 256, 6, 40, "lagrange3", 4, True, 104_857),
])
def test_planes_match_calls_of_few_points(nx, ny, pad, nz, scheme, n_tl, permuted, per):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import _swense as S, api
    n = (1 << 21) + 4097
    rng = np.random.default_rng(nx + pad)
    Lx, Ly = nx / 16, ny / 16
    sea = seas.linear_sea(nx, ny, Lx, Ly, seas.random_linear_components(nx, ny, Lx, Ly, 8, 0.01, rng))
    z = np.linspace(-1.0, 0.08, nz).astype(np.float32)
    tl = [0.05 * i for i in range(n_tl)]
    t = 0.4 * tl[-1]
    assert pad * nx * pad * ny * nz > 4 * n                     # the planes' rule
    grid = api.fields_on_grid(api.upload_modes(sea), z, pad, tl, scheme=scheme)
    gen = torch.Generator(device="cuda").manual_seed(nx)
    pts = torch.rand((n, 3), generator=gen, device="cuda") * torch.tensor([1.5 * Lx, Ly, 1.0], device="cuda")
    zs = torch.from_numpy(rng.uniform(-0.99, 0.07, n // per + 1).astype(np.float32)).cuda()
    zs[2], zs[3], zs[4] = float(z[-1]) + 0.01, float(z[-1]), float(z[5])   # above the grid, on levels
    pts[:, 2] = zs[torch.arange(n, device="cuda") // per]
    pts[7 * 1024 + 5, 2] = -0.5                                 # a chunk with a third z
    pts[-300:, 2] = torch.rand(300, generator=gen, device="cuda") - 0.95
    perm = torch.randperm(n, generator=gen, device="cuda").int() if permuted else None

    def gather(p, q):
        if q is not None:
            return api.interp_permuted(grid, t, p, q, count_out_of_range=True)
        return api.interp(grid, t, p, count_out_of_range=True)

    before = S.swense_launches()
    out, oor = gather(pts, perm)
    assert S.swense_launches() - before >= 7                    # plan, register, lists, planes, tiles, gathers
    assert oor == int(((pts[:, 2] < float(z[0])) | (pts[:, 2] > float(z[-1]))).sum())
    few = [api.interp(grid, t, pts[i:i + 100_000].contiguous())[0] for i in range(0, n, 100_000)]
    for k in out:
        a, b = out[k], torch.cat([f[k] for f in few])
        if permuted:
            a = a[perm.long()]
        assert torch.equal(torch.isnan(a), torch.isnan(b)), k
        a, b = torch.nan_to_num(a), torch.nan_to_num(b)
        assert float((a - b).abs().max()) <= 1e-5 * float(b.abs().max()), k
