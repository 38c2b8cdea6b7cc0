"""The FP32 direct sum's paired rows, tiles and mode splits at their edges: one point and points around
a block's 512; rows shorter and longer than a 64-mode tile; one row, a row without a partner, many
rows (so that the modes are split over blocks and the partial sums added). Bar 1e-5 of each field's
maximum (velocities on their shared scale), as for every FP32 direct sum."""
import numpy as np
import pytest

from oracle import modal
from tests._util import rel_linf, rel_linf_scaled, velocity_scale
from wavegen import points as P, seas

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


@pytest.mark.parametrize("nx,ny", [(8, 1), (512, 1), (8, 4), (256, 4), (32, 64)])
@pytest.mark.parametrize("n", [1, 511, 513, 1700])
@pytest.mark.parametrize("depth", [0.0, 0.8])
def test_fp32_direct_edges(api, nx, ny, n, depth):
    import torch
    # the ends of the rows, and rows n and -n with different amplitudes
    m, r = nx // 2 - 1, ny // 2 - 1
    comps = [(1, 0, 0.01, 0.3), (m, 0, 0.004, 1.9)]
    if ny > 1:
        comps += [(m, r, 0.003, 2.2), (m, -r, 0.005, 0.7), (2, r, 0.006, 4.0), (0, r, 0.004, 1.1)]
    sea = seas.linear_sea(nx, ny, nx / 16, max(ny, 4) / 16, comps, depth)
    pts = P.uniform_points(n, (-1.0, -1.0, -0.7), (2.0, 1.0, 0.03), n)
    t = 0.21
    ref = modal.fields_at_points(modal.propagate(sea, t), pts.astype(np.float64), p_mode="total")
    out = api.direct(api.upload_modes(sea), t, torch.from_numpy(pts).cuda(), p_mode="total")
    vs = velocity_scale(ref["u"], ref["v"], ref["w"])
    for k in ("eta", "u", "v", "w", "p"):
        got = out[k].cpu().numpy()
        e = rel_linf_scaled(got, ref[k], vs) if k in ("u", "v", "w") else rel_linf(got, ref[k])
        assert e <= 1e-5, (k, e)
