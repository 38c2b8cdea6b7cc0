"""Staged tiles (3-D box, one and two z-collapsed planes) beside untiled chunks, with enough points that
the planned gather runs (a chunk per SM and more); from 2^21 points on and on a grid of more than four
times as many nodes the gather by kinds of chunks, whose layers share collapsed planes; and the unplanned gather of fewer points: the same points taken
in two calls, many and few at a time, agree to rounding, and sampled points match the oracle. Bar 1e-5 of each field's maximum; two summation orders of the same FP32 products differ by
about 1e-6."""
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


@pytest.mark.parametrize("n", [175_321, (1 << 21) + 1501])
@pytest.mark.parametrize("kind", ["flat", "two", "box", "scattered", "mixed", "layers"])
@pytest.mark.parametrize("pad,scheme,n_tl", [(1, "lagrange3", 2), (4, "spline3", 1), (3, "lagrange3", 3),
                                             (8, "lagrange3", 2)])
def test_planned_gather_matches_few_points_and_oracle(api, n, kind, pad, scheme, n_tl):
    import torch
    sea = seas.jonswap_sea(64, 32, 8.0, 4.0, 0.05, 1.0, seed=62)
    # padded eight-fold, 90 levels: 11.8 M nodes per time level (and no oracle for so many)
    z = np.linspace(-1.0, 0.08, 90 if pad == 8 else 14).astype(np.float32)
    tl = 0.05 * np.arange(n_tl)
    t = float(tl[-1]) * 0.4
    rng = np.random.default_rng(5)
    per = {"flat": 4096, "two": 1500, "box": 1024, "scattered": 1 << 30, "mixed": 2048, "layers": 3001}[kind]
    k = np.arange(n) // per
    zs = rng.uniform(-1.0, 0.08, k[-1] + 1)
    if kind == "layers":                             # few z values, met again and again
        zs = zs[:9][rng.integers(0, 9, len(zs))]
        zs[0], zs[-1] = z[-1] + np.float32(0.01), z[3]
    cx, cy = rng.uniform(0.0, 8.0, k[-1] + 1), rng.uniform(0.0, 4.0, k[-1] + 1)
    wide = np.where(rng.random(k[-1] + 1) < {"mixed": 0.5, "layers": 0.5}.get(kind, 0.0), 8.0, 2.5 if pad == 8 else 0.6)
    pts = np.stack([cx[k] + wide[k] * rng.uniform(-0.5, 0.5, n), cy[k] + wide[k] * rng.uniform(-0.5, 0.5, n), zs[k]], 1)
    if kind == "box":
        pts[:, 2] += rng.uniform(-0.01, 0.01, n)
    if kind == "scattered":
        pts = np.stack([rng.uniform(0, 8, n), rng.uniform(0, 4, n), rng.uniform(-1.01, 0.085, n)], 1)
    pts = pts.astype(np.float32)
    grid = api.fields_on_grid(api.upload_modes(sea), z, pad, tl, scheme=scheme)
    d = torch.from_numpy(pts).cuda()
    out, oor = api.interp(grid, t, d, count_out_of_range=True)
    plan = api.interp_plan(grid, d)
    outp, _ = api.interp_with_plan(grid, t, d, plan)
    few = [api.interp(grid, t, d[i:i + 50_000].contiguous())[0] for i in range(0, n, 50_000)]
    assert oor == int(((pts[:, 2] < z[0]) | (pts[:, 2] > z[-1])).sum())
    for f in out:
        a, b = out[f], torch.cat([q[f] for q in few])
        assert torch.equal(torch.nan_to_num(a, 7.0), torch.nan_to_num(outp[f], 7.0)), f
        assert torch.equal(torch.isnan(a), torch.isnan(b)), f
        a, b = torch.nan_to_num(a), torch.nan_to_num(b)
        assert float((a - b).abs().max()) <= 1e-5 * float(b.abs().max()) + 1e-30, f
    if scheme != "lagrange3" or pad == 8:
        return
    sel = rng.choice(n, 400, replace=False)
    g = [modal.fields_on_grid(modal.propagate(sea, x), z, pad) for x in tl]
    ref = ointerp.interp_points(np.stack([q[0] for q in g]), np.stack([q[1] for q in g]), sea["Lx"], sea["Ly"], z, tl,
                                pts[sel], t)
    vs = velocity_scale(ref["u"], ref["v"], ref["w"])
    for f in ("eta", "u", "v", "w", "p"):
        got = out[f][torch.from_numpy(sel).cuda()].cpu().numpy()
        e = rel_linf_scaled(got, ref[f], vs) if f in ("u", "v", "w") else rel_linf(got, ref[f])
        assert e <= 1e-5, (f, e)
