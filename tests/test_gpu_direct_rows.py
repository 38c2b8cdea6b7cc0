"""FP32 direct sums of seas with short rows: a tile of 64 mode pairs holds one row's part (64 modes and more a
row) or several rows, with a last tile that is partly empty, one row alone and more rows than a tile or a
split of the modes takes. Bar 1e-5 of each field's maximum (velocities on their shared scale), as for every
FP32 direct sum."""
import numpy as np
import pytest

from oracle import modal
from tests._util import rel_linf, rel_linf_scaled, velocity_scale
from wavegen import points as P, seas

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(4, 1), (4, 4), (4, 64), (8, 128), (16, 16), (16, 1), (32, 8), (64, 4), (64, 32), (128, 1),
                                   (128, 8), (8, 512)])
@pytest.mark.parametrize("n", [3, 1300])
@pytest.mark.parametrize("depth", [0.0, 0.8])
def test_short_rows_match_the_oracle(nx, ny, n, depth):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import api
    rng = np.random.default_rng(nx + ny)
    # every row and every mode of a row carries something
    comps = [(m, r, 1e-3 * (0.5 + rng.random()), 6.28 * rng.random()) for m in range(nx // 2)
             for r in ({0} if ny == 1 else set(rng.integers(1 - ny // 2, ny // 2, 12)) | {0, 1, ny // 2 - 1, 1 - ny // 2}) if m or r > 0]
    sea = seas.linear_sea(nx, ny, nx / 16, max(ny, 4) / 16, comps, depth)
    pts = P.uniform_points(n, (-1.0, -1.0, -0.7), (2.0, 1.0, 0.0), n)
    ref = modal.fields_at_points(modal.propagate(sea, 0.21), pts.astype(np.float64), p_mode="dyn")
    out = api.direct(api.upload_modes(sea), 0.21, torch.from_numpy(pts).cuda(), p_mode="dyn")
    vs = velocity_scale(ref["u"], ref["v"], ref["w"])
    for k in ("eta", "u", "v", "w", "p"):
        got = out[k].cpu().numpy()
        e = rel_linf_scaled(got, ref[k], vs) if k in ("u", "v", "w") else rel_linf(got, ref[k])
        assert e <= 1e-5, (k, e)
