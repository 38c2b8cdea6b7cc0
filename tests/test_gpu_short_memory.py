"""Calls on a device short of memory (swense_selftest_workspace_limit makes larger workspaces fail): a
request for faster scratch that cannot be had leaves the workspace as it is and the call does with less,
with the same results, also when it is captured after it was made once outside a capture."""
import numpy as np
import pytest

from wavegen import seas

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import _swense as S, api
    S.swense_release()
    yield torch, S, api
    S.swense_selftest_workspace_limit(0)
    S.swense_release()


def _modes(api, nx, ny, snapshots=0):
    rng = np.random.default_rng(nx + ny)
    sea = seas.linear_sea(nx, ny, nx / 16, ny / 16, seas.random_linear_components(nx, ny, nx / 16, ny / 16, 8, 0.01, rng))
    return api.upload_modes(sea, snapshots=[sea] * snapshots if snapshots else None)


# per slot 2 MB (512 x 256) or 0.5 MB; the limits leave chunks of a quarter, of a few slots, of one, and only the
# shared-memory path (64 snapshots of 256 x 128 modes: 42 MB of formed modes that it does without)
@pytest.mark.parametrize("nx,ny,pad,nz,n_tl,snap,limit", [(512, 256, 1, 130, 2, 0, 200 * MB), (512, 256, 1, 130, 2, 0, 24 * MB),
                                                          (256, 128, 2, 24, 2, 0, 6 * MB), (256, 128, 3, 24, 1, 0, 24 * MB),
                                                          (256, 128, 1, 12, 64, 64, 8 * MB)])
def test_grid_with_less_scratch(env, nx, ny, pad, nz, n_tl, snap, limit):
    torch, S, api = env
    modes = _modes(api, nx, ny, snap)
    z, tl = np.linspace(-1.0, 0.05, nz).astype(np.float32), [0.1 * i for i in range(n_tl)]
    want = api.fields_on_grid(modes, z, pad, tl)
    S.swense_release()
    S.swense_selftest_workspace_limit(limit)
    g = api.alloc_grid(modes, z, pad, tl)
    held = []
    for _ in range(3):
        g.nodes.fill_(float("nan"))
        api.fields_on_grid(modes, z, pad, tl, out=g)
        held.append(S.swense_workspace_bytes())
    assert 0 < held[0] <= limit and held == held[:1] * 3
    if snap:                                                   # the other transform path
        assert float((g.nodes - want.nodes).abs().max()) <= 2e-6 * float(want.nodes.abs().max())
    else:
        assert torch.equal(g.nodes, want.nodes) and torch.equal(g.eta, want.eta)
    ref = g.nodes.clone()
    g.nodes.fill_(float("nan"))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        api.fields_on_grid(modes, z, pad, tl, out=g)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(g.nodes, ref)


def test_gather_without_planes_keeps_the_workspace(env):
    torch, S, api = env
    modes = _modes(api, 64, 32)
    z = np.linspace(-1.0, 0.08, 90).astype(np.float32)
    grid = api.fields_on_grid(modes, z, 8, [0.0])
    n = (1 << 21) + 1501
    gen = torch.Generator(device="cuda").manual_seed(1)
    pts = torch.rand((n, 3), generator=gen, device="cuda") * torch.tensor([4.0, 2.0, 0.0], device="cuda")
    pts[:, 2] = torch.from_numpy(z).cuda()[(torch.arange(n, device="cuda") // 30_000) % 80 + 2] - 0.003
    want, _ = api.interp(grid, 0.0, pts)
    want = {k: v.clone() for k, v in want.items()}
    S.swense_release()
    S.swense_selftest_workspace_limit(40 * MB)                  # the planes' scratch is 84 MB
    api.fields_on_grid(modes, z, 1, [0.0])
    held = S.swense_workspace_bytes()
    for _ in range(2):
        out, _ = api.interp(grid, 0.0, pts)
        assert S.swense_workspace_bytes() == held
        for k, v in want.items():
            assert float((out[k] - v).abs().max()) <= 1e-5 * float(v.abs().max()), k


@pytest.mark.parametrize("limit", [80 * MB, 30 * MB, 8 * MB])
def test_batch_with_less_scratch(env, limit):
    torch, S, api = env
    rng = np.random.default_rng(5)
    items = []
    for nx, ny, n in ((256, 128, 5000), (128, 128, 3000), (64, 32, 900)):
        sea = seas.linear_sea(nx, ny, nx / 16, ny / 16, seas.random_linear_components(nx, ny, nx / 16, ny / 16, 8, 0.01, rng))
        pts = np.stack([rng.uniform(0, nx / 16, n), rng.uniform(0, ny / 16, n), rng.uniform(-0.9, 0.0, n)], 1)
        items.append({"sea": sea, "z_levels": np.linspace(-1.0, 0.05, 40).astype(np.float32), "pad_n": 1,
                      "t_levels": [0.0, 0.1], "t": 0.04, "pts": pts.astype(np.float32)})
    b = api.Batch(items)
    b.run()                                                     # 4 streams' parts of 42 MB
    want = [{k: v.clone() for k, v in it["out"].items()} for it in b.items]
    S.swense_release()
    S.swense_selftest_workspace_limit(limit)
    held = []
    for _ in range(3):
        b.run()
        held.append(S.swense_workspace_bytes())
    assert 0 < held[0] <= limit and held == held[:1] * 3
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        b.run()
    for it in b.items:
        for v in it["out"].values():
            v.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    # the smallest limit leaves the other transform path: equal to rounding
    for it, w in zip(b.items, want):
        for k, v in w.items():
            assert float((it["out"][k] - v).abs().max()) <= 1e-5 * float(v.abs().max()), k


def test_growth_keeps_the_workspace_of_a_captured_graph(env):
    import gc
    import time
    torch, S, api = env
    modes = _modes(api, 64, 32)
    z = np.linspace(-1.0, 0.08, 12).astype(np.float32)
    want = api.fields_on_grid(modes, z, 2, [0.0])
    g = api.alloc_grid(modes, z, 2, [0.0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        api.fields_on_grid(modes, z, 2, [0.0], out=g)
    held = S.swense_workspace_bytes()
    big = _modes(api, 256, 128)
    api.fields_on_grid(big, z, 1, [0.0])                        # outgrows it
    grown = S.swense_workspace_bytes()
    assert grown > 2 * held
    fill = [torch.full((held // 4,), float("nan"), device="cuda") for _ in range(8)]
    g.nodes.fill_(float("nan"))
    g.eta.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(g.nodes, want.nodes) and torch.equal(g.eta, want.eta)
    assert all(bool(torch.isnan(f).all()) for f in fill)
    del graph
    gc.collect()
    torch.cuda.synchronize()
    time.sleep(0.5)                                             # the graph lets go on a thread of the runtime's
    api.fields_on_grid(_modes(api, 512, 256), z, 1, [0.0])
    now = S.swense_workspace_bytes()
    S.swense_release()
    assert S.swense_workspace_bytes() == 0
    api.fields_on_grid(_modes(api, 512, 256), z, 1, [0.0])
    assert S.swense_workspace_bytes() == now                    # both outgrown ones had been given back
