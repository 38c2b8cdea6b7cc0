"""Waits of the learned gather and of the default row pass that run out, by the library's self-test
switches (MMAs or copies withheld, a few polls): the call returns, the status is
SWENSE_ERR_TIMEOUT, the outputs say so, and the next call is the same as ever."""
import numpy as np
import pytest

from wavegen import configs

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


# one point, a step of 32 and one more, both warpgroups, several blocks (more than an SM holds of some)
@pytest.mark.parametrize("n", [1, 33, 700, 50_000])
@pytest.mark.parametrize("flat", [True, False])
def test_learned_gather_wait_that_runs_out(env, n, flat):
    torch, S, api = env
    cfg = configs.jonswap3d_small()
    grid = api.fields_on_grid(api.upload_modes(cfg["sea"]), cfg["z_levels"], 2, cfg["t_levels"])
    rng = np.random.default_rng(n)
    pts = np.stack([rng.uniform(0, cfg["sea"]["Lx"], n), rng.uniform(0, cfg["sea"]["Ly"], n),
                    np.full(n, -0.2) if flat else rng.uniform(-0.5, 0.0, n)], 1).astype(np.float32)
    d = torch.from_numpy(pts).cuda()
    mlp = api.Mlp(api.mlp_init(3))
    want, _ = api.interp_learned(grid, 0.01, d, mlp)
    want = {k: v.clone() for k, v in want.items()}
    assert S.swense_async_status(reset=True) == 0
    S.swense_selftest_learned_wait_timeout(True)
    try:
        out, _ = api.interp_learned(grid, 0.01, d, mlp)
        st = S.swense_async_status(reset=True, raise_on_error=False)
    finally:
        S.swense_selftest_learned_wait_timeout(False)
    assert st == -6 and S.swense_strerror(st) == "SWENSE_ERR_TIMEOUT"
    for k in ("u", "v", "w", "p"):
        assert bool(torch.isnan(out[k]).all()), k
    assert torch.equal(out["eta"], want["eta"])
    again, _ = api.interp_learned(grid, 0.01, d, mlp)
    assert S.swense_async_status(reset=True) == 0
    for k, v in want.items():
        assert torch.equal(again[k], v), k


# rows of one thread's exchange up to a block a row; one and two exchange buffers; one chunk and several
@pytest.mark.parametrize("nx,ny,pad,rowv,chunk", [(32, 32, 1, 0, 512), (64, 32, 4, 0, 1), (256, 64, 1, 0, 1), (256, 64, 2, 5, 1),
                                                  (2048, 32, 1, 0, 4), (512, 32, 4, 0, 512), (512, 64, 1, 4, 1)])
def test_row_pass_wait_that_runs_out(env, nx, ny, pad, rowv, chunk):
    torch, S, api = env
    from wavegen import seas
    rng = np.random.default_rng(nx)
    sea = seas.linear_sea(nx, ny, nx / 16, ny / 16, seas.random_linear_components(nx, ny, nx / 16, ny / 16, 6, 0.01, rng))
    z, tl = np.linspace(-1.0, 0.05, 7).astype(np.float32), [0.0, 0.1]
    modes = api.upload_modes(sea)
    S.swense_set_grid_tune(nx, ny, pad, len(z), 1, chunk << 20, rowv)
    try:
        want = api.fields_on_grid(modes, z, pad, tl)
        g = api.alloc_grid(modes, z, pad, tl)
        g.nodes.fill_(7.0)
        assert S.swense_async_status(reset=True) == 0
        S.swense_selftest_grid_wait_timeout(True)
        try:
            api.fields_on_grid(modes, z, pad, tl, out=g)
            st = S.swense_async_status(reset=True, raise_on_error=False)
        finally:
            S.swense_selftest_grid_wait_timeout(False)
        assert st == -6 and S.swense_strerror(st) == "SWENSE_ERR_TIMEOUT"
        assert bool((g.nodes == 7.0).all())                    # no row was written
        api.fields_on_grid(modes, z, pad, tl, out=g)
        assert S.swense_async_status(reset=True) == 0
        assert torch.equal(g.nodes, want.nodes) and torch.equal(g.eta, want.eta)
    finally:
        S.swense_set_grid_tune(nx, ny, pad, len(z), -1)
