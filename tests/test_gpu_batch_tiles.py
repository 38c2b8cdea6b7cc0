"""The batched gather's two kernels: chunks with a staged tile (among them boxes that lap a narrow grid and
boxes between the single call's tile and the batch's) and chunks straight from the grid, each instance
against the same work as individual public calls. Two summation orders of the same FP32 products
differ by about 1e-6 of a field's maximum; bar 1e-5."""
import numpy as np
import pytest

from wavegen import seas

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import api
    return torch, api


@pytest.mark.parametrize("n_tl", [1, 4])
def test_tiles_and_global_chunks_match_individual_calls(env, n_tl):
    torch, api = env
    rng = np.random.default_rng(n_tl)
    # modes, points per instance: dense (whole rows in a box), the tile between, sparse, a ragged few
    items = []
    for nx, ny, n in ((32, 64, 40_001), (128, 64, 150_003), (128, 128, 3_000), (64, 32, 1_025), (16, 16, 7)):
        sea = seas.jonswap_sea(nx, ny, nx / 16, ny / 16, 0.03, 1.0, heading=0.4, seed=nx + ny)
        z = np.linspace(-1.0, 0.05, 12).astype(np.float32)
        tl = 0.05 * np.arange(n_tl)
        pts = np.stack([rng.uniform(-1, nx / 16 + 1, n), rng.uniform(0, ny / 16, n), rng.uniform(-1.02, 0.055, n)], 1)
        items.append({"sea": sea, "z_levels": z, "pad_n": 1, "t_levels": tl, "t": 0.4 * float(tl[-1]),
                      "pts": pts.astype(np.float32), "bin": nx != 64})
    b = api.Batch(items, p_mode="total")
    b.run()
    torch.cuda.synchronize()
    got = [{k: v.clone() for k, v in it["out"].items()} for it in b.items]
    b.run_individual()
    torch.cuda.synchronize()
    for it, g in zip(b.items, got):
        for k, r in it["out"].items():
            assert torch.equal(torch.isnan(g[k]), torch.isnan(r)), k
            a, c = torch.nan_to_num(g[k]), torch.nan_to_num(r)
            assert float((a - c).abs().max()) <= 1e-5 * float(c.abs().max()) + 1e-30, k
