"""The gather of points whose stencils fit no staged tile (four lanes a point), at the edges of its
batches (16 points a warp, 128 a block, 1024 a chunk) and over the grids it meets: power-of-two and
other node counts, one to four time levels, both schemes, a permuted order, and untiled chunks beside
staged ones. Bar 1e-5 of each field's maximum, as for every FP32 gather (about 1e-6 is expected of 64
products accumulated in FP32)."""
import numpy as np
import pytest

from oracle import interp as ointerp, modal
from tests._util import rel_linf, rel_linf_scaled, velocity_scale
from wavegen import seas

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import api as a
    return a


@pytest.mark.parametrize("n", [1, 15, 17, 127, 130, 1025, 2111])
@pytest.mark.parametrize("pad,n_tl", [(2, 1), (3, 2), (2, 4)])
def test_scattered_points_match_the_oracle(api, n, pad, n_tl):
    import torch
    sea = seas.jonswap_sea(64, 32, 8.0, 4.0, 0.05, 1.0, seed=61)
    z = np.linspace(-1.0, 0.08, 14).astype(np.float32)
    tl = 0.05 * np.arange(n_tl)
    t = float(tl[-1]) * 0.4
    rng = np.random.default_rng(n)
    pts = np.stack([rng.uniform(-3.0, 11.0, n), rng.uniform(-2.0, 6.0, n), rng.uniform(-1.05, 0.085, n)], 1).astype(np.float32)
    grid = api.fields_on_grid(api.upload_modes(sea), z, pad, tl)
    perm = torch.from_numpy(rng.permutation(n).astype(np.int32)).cuda()
    d = torch.from_numpy(pts).cuda()
    out, oor = api.interp(grid, t, d, count_out_of_range=True)
    srt = d[perm.long()].contiguous()                # srt[k] is the caller's point perm[k]
    outp, _ = api.interp_permuted(grid, t, srt, perm)
    nodes = np.stack([modal.fields_on_grid(modal.propagate(sea, x), z, pad)[0] for x in tl])
    etas = np.stack([modal.fields_on_grid(modal.propagate(sea, x), z, pad)[1] for x in tl])
    ref = ointerp.interp_points(nodes, etas, sea["Lx"], sea["Ly"], z, tl, pts, t)
    assert oor == int(ref["out_of_range"].sum())
    vs = velocity_scale(ref["u"], ref["v"], ref["w"])
    for o in (out, outp):
        for k in ("eta", "u", "v", "w", "p"):
            got = o[k].cpu().numpy()
            e = rel_linf_scaled(got, ref[k], vs) if k in ("u", "v", "w") else rel_linf(got, ref[k])
            assert e <= 1e-5, (k, e)
