"""The fused learned gather at the edges of its steps: 32 points a tile, 64 (staged box) or 32
(per-point stencils) a step of a warpgroup, 512 a warpgroup, 1024 a block; against the library's own
features and an FP64 network on the BF16-rounded weights.

Bar, per value: every layer's inputs are exact to u = 2^-16 (two BF16 halves 2^-17, FP32 sums of 80
terms), an error grows by |W| through a layer and by at most 1.13 through GELU; the plain Lagrange
value is a sum of 64 products of at most 4.4 max |value| in FP32 (2e-5 of the maximum)."""
import numpy as np
import pytest

from oracle import mlp as omlp
from wavegen import configs

pytestmark = pytest.mark.gpu
U = 2.0 ** -16


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import api, build
    build.build()
    cfg = configs.jonswap3d_small()
    grid = api.fields_on_grid(api.upload_modes(cfg["sea"]), cfg["z_levels"], 2, cfg["t_levels"])
    p = omlp.init_params(5)
    rng = np.random.default_rng(6)
    for k in ("b1", "b2", "b3"):
        p[k] = rng.standard_normal(p[k].shape) * 0.3
    return torch, api, cfg, grid, p, api.Mlp(torch.from_numpy(api.mlp_flatten(p)), out_scale=1.0)


def _bf16(a):
    u = np.asarray(a, np.float32).view(np.uint32).astype(np.uint64)
    return ((u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32).astype(np.float64)


def _gelu(x):
    return 0.5 * x * (1 + np.tanh(np.sqrt(2 / np.pi) * (x + 0.044715 * x ** 3)))


@pytest.mark.parametrize("order", ["mesh", "random"])
@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 511, 513, 577, 1024, 1025, 2047])
def test_learned_rows(env, n, order):
    torch, api, cfg, grid, p, mlp = env
    sea, z, t = cfg["sea"], cfg["z_levels"], cfg["t_query"]
    if order == "mesh":
        pts = configs.mesh_points(cfg["mesh"])[:n]
    else:
        rng = np.random.default_rng(n)
        pts = np.stack([rng.uniform(0, sea["Lx"], n), rng.uniform(0, sea["Ly"], n),
                        rng.uniform(float(z[0]), float(z[-1]), n)], 1).astype(np.float32)
    pd = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
    n = len(pts)
    got, _ = api.interp_learned(grid, t, pd, mlp, p_mode="phit")
    x, sc, lag, eta = (v.cpu().numpy().astype(np.float64) for v in api.mlp_features(grid, t, pd))
    x = x[:, :67]
    W = [_bf16(p[k]) for k in ("W1", "W2", "W3")]
    b = [np.asarray(p[k], np.float32).astype(np.float64) for k in ("b1", "b2", "b3")]
    W = [w if w.shape[1] == m else w.T for w, m in zip(W, (67, 64, 64))]
    a, err = x, np.zeros_like(x)
    for i in range(3):
        err = (err + U * np.abs(a)) @ np.abs(W[i]).T + U * np.abs(b[i])
        a = a @ W[i].T + b[i]
        if i < 2:
            a, err = _gelu(a), 1.13 * err
    f = np.arange(4 * n) % 4
    sc, lag = sc.reshape(-1), lag.reshape(-1)
    ref = lag + sc * a[np.arange(4 * n), f]
    tol = sc * (2e-5 + err[np.arange(4 * n), f])
    out = np.stack([got[k].cpu().numpy() for k in ("u", "v", "w", "p")], 1).reshape(-1)
    assert np.all(np.abs(out - ref) <= tol), float(np.max(np.abs(out - ref) / tol))
    np.testing.assert_allclose(got["eta"].cpu().numpy(), eta.reshape(-1), rtol=0, atol=2e-5 * np.max(np.abs(eta)))
