"""The learned gather of few chunks, in parts of a chunk: the same bits as the same chunks in one large call, which
takes each whole, from one step a warpgroup (16 parts) to two parts a chunk, with last chunks of one point, of a
part and a little, and of all but one point; staged boxes and per-point stencils."""
import numpy as np
import pytest

from wavegen import configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["flat", "box", "scattered"])
def test_parts_of_a_chunk_equal_the_whole(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import api
    cfg = configs.jonswap3d_small()
    grid = api.fields_on_grid(api.upload_modes(cfg["sea"]), cfg["z_levels"], 4, cfg["t_levels"])
    n = 1600 * 1024                                             # more than five waves of two blocks an SM
    rng = np.random.default_rng(4)
    k = np.arange(n) // 1024
    cx, cy, cz = rng.uniform(0, cfg["sea"]["Lx"], k[-1] + 1), rng.uniform(0, cfg["sea"]["Ly"], k[-1] + 1), rng.uniform(-0.5, 0.0, k[-1] + 1)
    w = 0.15 if kind != "scattered" else 4.0
    pts = np.stack([cx[k] + w * rng.uniform(-1, 1, n), cy[k] + w * rng.uniform(-1, 1, n), cz[k]], 1)
    if kind != "flat":
        pts[:, 2] += rng.uniform(-0.02, 0.02, n)
    d = torch.from_numpy(pts.astype(np.float32)).cuda()
    mlp = api.Mlp(api.mlp_init(3))
    want, _ = api.interp_learned(grid, cfg["t_query"], d, mlp)
    at = 0
    for chunks, last in ((1, 1), (1, 63), (2, 65), (40, 513), (100, 1023), (200, 129), (400, 700), (700, 1024)):
        m = (chunks - 1) * 1024 + last
        out, _ = api.interp_learned(grid, cfg["t_query"], d[at:at + m].contiguous(), mlp)
        for f, v in out.items():
            # a chunk that ends early may be planned otherwise (its box, its z), so its points agree to rounding
            full = (chunks - 1) * 1024
            assert torch.equal(torch.nan_to_num(v[:full], 7.0), torch.nan_to_num(want[f][at:at + full], 7.0)), (f, chunks)
            a, b = torch.nan_to_num(v[full:]), torch.nan_to_num(want[f][at + full:at + m])
            assert float((a - b).abs().max()) <= 1e-5 * float(torch.nan_to_num(want[f]).abs().max()), (f, chunks)
        at += chunks * 1024
