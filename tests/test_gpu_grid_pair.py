"""What the transform pair branches on: rows of 32 to 2048 nodes with one and with two exchange buffers,
columns of 32 to 1024, deep and finite depth, levels given at once and in chunks that end between the
eta slots. The shared-memory path computes the same sums in another order: 2e-6 of the largest value, as
for every other launch shape. Chunks, levels per block and the numbers of earlier row variants do not
change a bit."""
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
    from paper_2005_12716_gb300 import _swense as S, api
    return torch, S, api


def _grid(S, api, modes, z, pad, tl, scheme, lpc, chunk, rowv):
    S.swense_set_grid_tune(modes.nx, modes.ny, pad, len(z), lpc, chunk, rowv)
    try:
        return api.fields_on_grid(modes, z, pad, tl, scheme=scheme)
    finally:
        S.swense_set_grid_tune(modes.nx, modes.ny, pad, len(z), -1)


@pytest.mark.parametrize("depth", [0.0, 0.6])
@pytest.mark.parametrize("nx,ny,pad", [(32, 32, 1), (64, 32, 1), (128, 64, 1), (256, 32, 1), (512, 32, 1), (1024, 32, 1),
                                       (2048, 32, 1), (8, 8, 4), (16, 32, 4), (32, 64, 4), (64, 128, 4), (128, 256, 4),
                                       (256, 16, 4), (512, 8, 4), (32, 128, 1), (32, 256, 1), (32, 512, 1), (32, 1024, 1)])
def test_pair_matches_the_shared_memory_path(env, nx, ny, pad, depth):
    torch, S, api = env
    rng = np.random.default_rng(nx + ny + pad)
    Lx, Ly = nx / 16, ny / 16
    sea = seas.linear_sea(nx, ny, Lx, Ly, seas.random_linear_components(nx, ny, Lx, Ly, 10, 0.01, rng), depth)
    modes = api.upload_modes(sea)
    z, tl = np.linspace(-0.5, 0.04, 5).astype(np.float32), [0.0, 0.13, 0.2]
    scheme = "spline3" if pad == 4 else "lagrange3"
    got = _grid(S, api, modes, z, pad, tl, scheme, 1, 512 << 20, 0)
    ref = _grid(S, api, modes, z, pad, tl, scheme, 0, 64 << 20, 0)
    for q in range(4):
        m = float(ref.nodes[..., :3].abs().max()) if q < 3 else float(ref.nodes[..., 3].abs().max())
        assert float((got.nodes[..., q] - ref.nodes[..., q]).abs().max()) <= 2e-6 * m, q
    assert float((got.eta - ref.eta).abs().max()) <= 2e-6 * float(ref.eta.abs().max())


# slots of 0.5 MB: 3 time levels of 5 levels, then 3 of eta
@pytest.mark.parametrize("lpc,chunk_mb,rowv", [(1, 1, 0), (2, 1, 0), (4, 4, 0), (2, 8, 5), (1, 5, 5), (1, 64, 1), (2, 2, 2), (1, 3, 3),
                                               (1, 64, 16), (4, 1, 17), (1, 2, 21)])
def test_shape_does_not_change_a_bit(env, lpc, chunk_mb, rowv):
    torch, S, api = env
    nx, ny, pad = 128, 64, 2
    rng = np.random.default_rng(3)
    sea = seas.linear_sea(nx, ny, 8.0, 4.0, seas.random_linear_components(nx, ny, 8.0, 4.0, 10, 0.01, rng), 0.6)
    modes = api.upload_modes(sea)
    z, tl = np.linspace(-0.5, 0.04, 5).astype(np.float32), [0.0, 0.13, 0.2]
    ref = _grid(S, api, modes, z, pad, tl, "lagrange3", 1, 512 << 20, 0)
    got = _grid(S, api, modes, z, pad, tl, "lagrange3", lpc, chunk_mb << 20, rowv)
    assert torch.equal(got.nodes, ref.nodes) and torch.equal(got.eta, ref.eta)
