"""A chunk size that a caller sets is the one that runs: the workspace of a grid grows with it in step, with
no size that stands for another."""
import numpy as np
import pytest

from wavegen import seas

pytestmark = pytest.mark.gpu
MB = 1 << 20


def test_workspace_follows_the_chunk_size():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import _swense as S, api
    nx, ny, nz, tl = 512, 256, 160, [0.0, 0.1]                  # 322 slots of 2 MB
    sea = seas.linear_sea(nx, ny, nx / 16, ny / 16, [(2, 1, 0.01, 0.2)])
    modes = api.upload_modes(sea)
    z = np.linspace(-1.0, 0.05, nz).astype(np.float32)
    slot = 4 * ny * (nx // 2) * 8
    modes_b = 2 * 5 * ny * (nx // 2) * 8
    g = api.alloc_grid(modes, z, 1, tl)
    ref = api.fields_on_grid(modes, z, 1, tl).nodes
    try:
        for mb in (64, 200, 255, 256, 300, 512):
            S.swense_release()
            S.swense_set_grid_tune(nx, ny, 1, nz, 1, mb * MB, 0)
            api.fields_on_grid(modes, z, 1, tl, out=g)
            # a quarter of headroom; eta's intermediate and padding to 256 bytes
            most = 1.25 * (mb * MB + modes_b + ny * (nx // 2) * 8 + 1024)
            n = -(-322 // (mb * MB // slot))                    # chunks
            least = 1.25 * (322 // n) * slot
            assert least <= S.swense_workspace_bytes() <= most, mb
            assert torch.equal(g.nodes, ref), mb
    finally:
        S.swense_set_grid_tune(nx, ny, 1, nz, -1)
        S.swense_release()
