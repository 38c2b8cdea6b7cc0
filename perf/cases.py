"""Performance cases: what a user of this framework has it do at every CFD time step, through
``paper_2005_12716_gb300.api``.

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU from a seed, ``run`` is one
pass through the public entry points, ``exact`` the same outputs in 64 bits by plain torch. Lengths
are in peak wavelengths, g = 9.81, rho = 1000. The seas are JONSWAP (gamma 3.3, cos^2 spreading,
random phases) or third-order Stokes waves, the meshes O-grids around a vertical cylinder whose
cell and face centres are graded towards the cylinder and the free surface.
"""
import math

import numpy as np
import torch

from paper_2005_12716_gb300 import api

G, RHO = 9.81, 1000.0
FIELDS = ("eta", "u", "v", "w", "p")
DEV = "cuda"


# ------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # 2-D regular wave in deep water, reconstruction and gather of 50,000 scattered points: the
        # smallest step a user makes, a few launches long
        {"name": "stokes2d_step", "kind": "step2d", "nx": 256, "nz": 33, "pad": 1, "n_tl": 2, "points": 50_000,
         "scheme": "lagrange3"},
        # the whole incident-wave step of a 3-D sea on a cylinder mesh: modes -> grid -> 2,048,000 cell and
        # 6,177,280 face centres
        {"name": "jonswap_mesh_step", "kind": "step3d", "nx": 512, "ny": 256, "nz": 64, "pad": 1, "n_tl": 2,
         "nr": 160, "nth": 128, "nlay": 100, "scheme": "lagrange3", "depth": 0.0},
        # the same sea reconstructed at four-fold zero-padding for cubic splines, the paper's own setting
        {"name": "grid_pad4_spline", "kind": "grid", "nx": 512, "ny": 256, "nz": 64, "pad": 4, "n_tl": 2,
         "scheme": "spline3", "depth": 0.0},
        # reconstruction of a large steep sea (8.6 GB of grid)
        {"name": "grid_large", "kind": "grid", "nx": 2048, "ny": 1024, "nz": 128, "pad": 1, "n_tl": 2,
         "scheme": "lagrange3", "depth": 0.0},
        # gather of the cylinder mesh from the four-fold padded spline grid
        {"name": "mesh_gather_pad4_spline", "kind": "gather_mesh", "nx": 512, "ny": 256, "nz": 64, "pad": 4, "n_tl": 2,
         "nr": 160, "nth": 128, "nlay": 100, "scheme": "spline3"},
        # gather of 16 M points scattered over the large sea's whole domain, in Morton order
        {"name": "scattered_gather_large", "kind": "gather_cloud", "nx": 2048, "ny": 1024, "nz": 128, "pad": 1, "n_tl": 2,
         "points": 16_000_000, "order": "morton", "scheme": "lagrange3"},
        # eight uneven sea states at four time levels in one call, points binned once
        {"name": "batch_uneven", "kind": "batch", "instances": 8, "nz": 32, "n_tl": 4, "lo": 7, "hi": 10,
         "points_hi": 4_000_000, "sizes": 3},
        # near-body points of the large sea summed over all its two million modes on the tensor cores
        {"name": "direct_split_large", "kind": "direct", "nx": 2048, "ny": 1024, "points": 1_000_000,
         "precision": "split_bf16", "depth": 0.0},
        # near-body points of a modest sea summed in FP32 (the default precision), finite depth
        {"name": "direct_fp32", "kind": "direct", "nx": 128, "ny": 64, "points": 100_003, "precision": "fp32",
         "depth": 0.7},
        # the learned gather of the cylinder mesh
        {"name": "learned_mesh_gather", "kind": "learned", "nx": 512, "ny": 256, "nz": 64, "n_tl": 2, "nr": 160,
         "nth": 128, "nlay": 100},
        # one training step (forward, backward, Adam) of the learned correction
        {"name": "mlp_train_step", "kind": "train", "rows": 1 << 20, "batch": 8192},
        # per-cell work at the end of a CFD step: relaxation-zone blending and the divergence of the face velocity
        {"name": "cells_relax_divergence", "kind": "cells", "nr": 160, "nth": 128, "nlay": 100, "zones": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step2d", "step3d", "grid", "gather_mesh", "gather_cloud", "batch", "direct", "learned", "train",
                       "cells"])
    scheme = rng.choice(["lagrange3", "spline3"])
    depth = rng.choice([0.0, round(rng.uniform(0.3, 1.5), 3)])
    mesh = {"nr": rng.randint(40, 160), "nth": rng.randint(24, 128), "nlay": rng.randint(16, 100)}
    # mode counts of a sea and a padding factor whose padded grid stays within the listed ones
    nx, ny = 1 << rng.randint(6, 10), 1 << rng.randint(5, 9)
    pad = rng.choice([p for p in (1, 2, 3, 4) if p * nx <= 2048 and p * ny <= 1024])
    sea = {"nx": nx, "ny": ny, "nz": rng.randint(12, 64), "pad": pad, "n_tl": rng.randint(1, 4), "scheme": scheme}
    if kind == "step2d":
        nx = 1 << rng.randint(6, 11)
        return {"kind": kind, "nx": nx, "nz": rng.randint(9, 64), "pad": rng.choice([1, 2, 3, 4]),
                "n_tl": rng.randint(1, 4), "points": _log_int(rng, 2_000, 400_000), "scheme": scheme}
    if kind == "step3d":
        return {"kind": kind, **sea, **mesh, "depth": depth and depth + 0.7}
    if kind == "grid":
        return {"kind": kind, **sea, "depth": depth}
    if kind == "gather_mesh":
        return {"kind": kind, **sea, **mesh}
    if kind == "gather_cloud":
        return {"kind": kind, **sea, "points": _log_int(rng, 20_000, 8_000_000), "order": rng.choice(["morton", "binned"])}
    if kind == "batch":
        return {"kind": kind, "instances": rng.randint(2, 8), "nz": rng.randint(12, 32), "n_tl": rng.randint(2, 4),
                "lo": rng.randint(5, 7), "hi": rng.randint(8, 9), "points_hi": _log_int(rng, 50_000, 4_000_000),
                "sizes": rng.randint(0, 1 << 20)}
    if kind == "direct":
        return {"kind": kind, "nx": 1 << rng.randint(6, 9), "ny": 1 << rng.randint(5, 8),
                "points": _log_int(rng, 5_000, 200_000), "precision": rng.choice(["fp32", "split_bf16"]), "depth": depth}
    if kind == "learned":
        return {"kind": kind, "nx": nx, "ny": ny, "nz": sea["nz"], "n_tl": rng.randint(2, 4), **mesh}
    if kind == "train":
        return {"kind": kind, "rows": _log_int(rng, 20_000, 1 << 20), "batch": _log_int(rng, 1_000, 32_768)}
    return {"kind": "cells", **mesh, "zones": rng.randint(1, 8)}


# ------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _wavenumbers(s):
    nx, ny = s["nx"], s["ny"]
    m = torch.arange(nx // 2 + 1, device=DEV, dtype=torch.float64)
    n = torch.arange(ny, device=DEV, dtype=torch.float64)
    n = torch.where(n < ny / 2, n, n - ny) if ny > 1 else n
    kx, ky = 2 * math.pi / s["Lx"] * m, 2 * math.pi / s["Ly"] * n
    return kx[None, :], ky[:, None], torch.sqrt(kx[None, :] ** 2 + ky[:, None] ** 2)


def _sea(g, nx, ny, Hs, depth=0.0):
    """One-sided half spectrum [ny][nx/2+1] of a JONSWAP sea, 16 nodes per peak wavelength."""
    s = {"nx": nx, "ny": ny, "Lx": nx / 16, "Ly": ny / 16 if ny > 1 else 1.0, "depth": depth}
    kx, ky, k = _wavenumbers(s)
    kk = k.clamp_min(1e-9)
    om = torch.sqrt(G * k * (torch.tanh(k * depth) if depth > 0 else 1.0))
    kp = torch.tensor(2 * math.pi, device=DEV, dtype=torch.float64)
    wp = torch.sqrt(G * kp * (torch.tanh(kp * depth) if depth > 0 else 1.0))
    wr = om.clamp_min(1e-3) / wp
    sig = torch.where(wr <= 1, 0.07, 0.09)
    S = wr ** -5 * torch.exp(-1.25 * wr ** -4) * 3.3 ** torch.exp(-((wr - 1) ** 2) / (2 * sig ** 2))
    a = torch.sqrt(S / (om.clamp_min(1e-3) * kk)) * (kx / kk)          # cos^2 spreading about +x
    a[:, -1] = 0
    a[:, 0] = 0
    if ny > 1:
        a[ny // 2] = 0
    a *= Hs / (4 * torch.sqrt((a * a).sum() / 2))
    return _linear(g, s, a, om)


def _linear(g, s, a, om):
    ph = 2 * math.pi * _rand(g, *a.shape)
    e = 0.5 * torch.polar(a, ph)
    s["A_eta"], s["omega"] = e.to(torch.complex64), om
    s["A_phi"] = (-1j * (G / om.clamp_min(1e-3)) * e).to(torch.complex64)
    s["A_phit"] = (-G * e).to(torch.complex64)
    return s


def _stokes(g, nx):
    """Third-order deep-water Stokes wave, ka about 0.1, 16 nodes per wavelength."""
    s = {"nx": nx, "ny": 1, "Lx": nx / 16, "Ly": 1.0, "depth": 0.0}
    m = nx // 16
    ka, phase = 0.08 + 0.04 * float(_rand(g, 1)), 2 * math.pi * float(_rand(g, 1))
    k = 2 * math.pi
    a, om = ka / k, math.sqrt(G * k * (1 + ka * ka))
    A = {q: torch.zeros(1, nx // 2 + 1, dtype=torch.complex128, device=DEV) for q in ("A_eta", "A_phi", "A_phit")}
    w = torch.zeros(1, nx // 2 + 1, dtype=torch.float64, device=DEV)
    for j, c in enumerate((a, 0.5 * k * a * a, 0.375 * k * k * a ** 3), 1):
        A["A_eta"][0, m * j] = 0.5 * c * complex(math.cos(j * phase), math.sin(j * phase))
        w[0, m * j] = j * om
    e = complex(math.cos(phase), math.sin(phase))
    A["A_phi"][0, m] = -0.5j * (om / k) * a * e
    A["A_phit"][0, m] = -0.5 * (om * om / k) * a * e
    return {**s, **{q: v.to(torch.complex64) for q, v in A.items()}, "omega": w}


def _modes(s):
    pair = {q: torch.view_as_real(s[q]).contiguous() for q in ("A_eta", "A_phi", "A_phit")}
    return api.DeviceModes(s["nx"], s["ny"], s["Lx"], s["Ly"], s["depth"], 1, pair["A_eta"], pair["A_phi"],
                           pair["A_phit"], s["omega"], 0.0)


def _levels(nz, bot, top):
    """Uniform levels in a band about the surface (three eighths of them), geometric below."""
    n_band = max(4, 3 * nz // 8)
    up = np.linspace(-top, top, n_band)
    d, n, span = up[1] - up[0], nz - n_band, -top - bot
    lo, hi = 1.0, 3.0
    for _ in range(100):
        q = 0.5 * (lo + hi)
        lo, hi = (lo, q) if d * (q ** np.arange(1, n + 1)).sum() > span else (q, hi)
    steps = d * q ** np.arange(1, n + 1)
    return np.concatenate([(-top - np.cumsum(steps * span / steps.sum()))[::-1], up]).astype(np.float32)


def _times(n_tl, wave_period):
    t = np.arange(n_tl) * (wave_period / 16)
    return t, float(t[(n_tl - 1) // 2] + 0.37 * wave_period / 16) if n_tl > 1 else 0.0


PERIOD = math.sqrt(2 * math.pi / G)                                     # of a deep-water wave of unit length


def _edges(nr, nlay, z_lo, z_hi, band):
    ratio = 1.02 ** (160.0 / nr)
    w = torch.cumsum(ratio ** torch.arange(nr, device=DEV, dtype=torch.float64), 0)
    r = 0.039 + (2.0 - 0.039) * torch.cat([w.new_zeros(1), w / w[-1]])
    nb = max(2, round(0.6 * nlay))
    dz = (z_hi + band) / nb
    zb = -band + dz * torch.arange(nb + 1, device=DEV, dtype=torch.float64)
    st = torch.cumsum(1.03 ** torch.arange(1, nlay - nb + 1, device=DEV, dtype=torch.float64), 0)
    return r, torch.cat([(-band - st * ((-band - z_lo) / st[-1])).flip(0), zb])


def _mesh(c, xc, yc):
    """Edges of an O-grid of radius 0.039 .. 2 about (xc, yc) and its cell and face centres, float32, in mesh
    order (radial fastest, then angular, then the layers; cells, then faces by kind)."""
    r, z = _edges(c["nr"], c["nlay"], -0.9, 0.07, 0.075)
    th = 2 * math.pi / c["nth"] * torch.arange(c["nth"], device=DEV, dtype=torch.float64)
    half = math.pi / c["nth"]
    rm, zm = 0.5 * (r[1:] + r[:-1]) * math.cos(half), 0.5 * (z[1:] + z[:-1])

    def block(zz, tt, rr):
        Z, T, R = torch.meshgrid(zz, tt, rr, indexing="ij")
        return torch.stack([xc + R * torch.cos(T), yc + R * torch.sin(T), Z], -1).reshape(-1, 3)

    pts = [block(zm, th + half, rm), block(zm, th + half, r * math.cos(half)), block(zm, th, rm), block(z, th + half, rm)]
    return r, th, z, torch.cat(pts).to(torch.float32).contiguous()


def _cloud(g, n, lo, hi, order=None):
    lo, hi = (torch.tensor(v, device=DEV, dtype=torch.float64) for v in (lo, hi))
    f = _rand(g, n, 3)
    if order == "morton":
        q = (f * 1024).long()
        code = torch.zeros(n, dtype=torch.long, device=DEV)
        for b in range(10):
            for d in range(3):
                code |= ((q[:, d] >> b) & 1) << (3 * b + d)
        f = f[torch.argsort(code)]
    return (lo + (hi - lo) * f).to(torch.float32).contiguous()


def _near_body(g, s, n, z_lo, z_hi):
    """Points uniform in the annulus 0.039 < r < 0.25 about the domain's centre."""
    r = torch.sqrt(0.039 ** 2 + (0.25 ** 2 - 0.039 ** 2) * _rand(g, n))
    th = 2 * math.pi * _rand(g, n)
    z = z_lo + (z_hi - z_lo) * _rand(g, n)
    return torch.stack([0.5 * s["Lx"] + r * torch.cos(th), 0.5 * s["Ly"] + r * torch.sin(th), z], 1).to(torch.float32).contiguous()


def _out(n, keys=FIELDS):
    return {k: torch.empty(n, dtype=torch.float32, device=DEV) for k in keys}


def _empty_grid(c, s, z, t):
    return api.alloc_grid(_modes(s), z, c["pad"], t, scheme=c["scheme"])


def _filled_grid(c, s, z, t):
    """A grid with its node values in place, as a gather finds it."""
    grid = _empty_grid(c, s, z, t)
    _fields(s, z, c["pad"], t, c["scheme"], grid.nodes, grid.eta)
    return grid


def _mlp_params(g):
    shapes = ((64, 67), (64,), (64, 64), (64,), (4, 64), (4,))
    parts = [torch.randn(*h, generator=g, device=DEV) / math.sqrt(h[-1]) if len(h) == 2 else 0.02 * torch.randn(*h, generator=g, device=DEV)
             for h in shapes]
    return torch.cat([p.reshape(-1) for p in parts])


def _batch_items(case, seed):
    r = np.random.default_rng(case["sizes"])
    items = []
    for i in range(case["instances"]):
        nx, ny = (1 << int(r.integers(case["lo"], case["hi"] + 1)) for _ in "xy")
        n = int(10 ** r.uniform(4, math.log10(case["points_hi"])))
        g = _gen(1000 * seed + i)
        Hs = float(0.02 + 0.03 * _rand(g, 1))
        s = _sea(g, nx, ny, Hs)
        z = _levels(case["nz"], -1.0, 1.5 * Hs)
        t, tq = _times(case["n_tl"], PERIOD)
        pts = _cloud(g, n, (0, 0, float(z[0])), (s["Lx"], s["Ly"], float(z[-1])))
        items.append((s, z, t, tq, pts))
    return items


def _train_data(case, seed):
    g = _gen(seed)
    n = case["rows"]
    x = torch.empty(n, 68, device=DEV)
    x[:, :64].normal_(generator=g)
    x[:, :64] = torch.cumsum(x[:, :64], 1)                              # neighbouring nodes are alike
    x[:, :64] /= x[:, :64].abs().amax(1, keepdim=True)
    x[:, 64:67].uniform_(generator=g)
    x[:, 67] = 0
    field = torch.arange(n, device=DEV, dtype=torch.int32) % 4
    target = torch.randn(n, generator=g, device=DEV)
    batch = torch.randint(0, n, (case["batch"],), generator=g, device=DEV, dtype=torch.int32)
    return _mlp_params(g), x, field, target, batch


def _cells(case, seed):
    g = _gen(seed)
    nr, nth, nlay = case["nr"], case["nth"], case["nlay"]
    r, th, z, pts = _mesh(case, 0.0, 0.0)
    half, nc = math.pi / nth, nr * nth * nlay
    nrf, ntf = nlay * nth * (nr + 1), nc
    dz, dr = z[1:] - z[:-1], r[1:] - r[:-1]
    chord = 2 * math.sin(half) * r

    def area(zz, tt, rr, direction):
        A = (zz[:, None, None] * rr).expand(len(zz), len(tt), -1)
        d = torch.stack([torch.cos(tt), torch.sin(tt)], -1) if direction == "r" else torch.stack([-torch.sin(tt), torch.cos(tt)], -1)
        return torch.cat([A[..., None] * d[None, :, None, :], torch.zeros_like(A)[..., None]], -1).reshape(-1, 3)

    base = 0.5 * (chord[1:] + chord[:-1]) * dr * math.cos(half)
    top = torch.stack([torch.zeros(nr, device=DEV, dtype=torch.float64)] * 2 + [base], -1).repeat((nlay + 1) * nth, 1)
    areas = torch.cat([area(dz, th + half, chord, "r"), area(dz, th, dr, "t"), top]).to(torch.float32).contiguous()
    L, J, I = torch.meshgrid(*(torch.arange(k, device=DEV) for k in (nlay, nth, nr)), indexing="ij")
    fr = (L * nth + J) * (nr + 1) + I
    ft, fz = nrf + (L * nth + J) * nr + I, nrf + ntf + (L * nth + J) * nr + I
    ft2 = nrf + (L * nth + (J + 1) % nth) * nr + I
    faces = torch.stack([-(fr + 1), fr + 2, -(ft + 1), ft2 + 1, -(fz + 1), fz + nth * nr + 1], -1)
    lay = torch.arange(nc, device=DEV) // (nr * nth)
    vel = 0.3 * torch.sin(3.1 * pts[nc:] + 6.28 * torch.rand(3, generator=g, device=DEV)) + 0.02 * torch.randn(len(pts) - nc, 3, generator=g, device=DEV)
    eta = 0.03 * torch.sin(6.28 * pts[:nc, 0] + 6.28 * torch.rand(1, generator=g, device=DEV))
    zones = [(api.S.ZONE_RADIAL, 1.5, 2.0, 0.0, 0.0), (api.S.ZONE_X, -1.2, -2.0, 0.0, 0.0), (api.S.ZONE_X, 1.2, 2.0, 0.0, 0.0),
             (api.S.ZONE_Y, 1.4, 2.0, 0.0, 0.0), (api.S.ZONE_Y, -1.4, -2.0, 0.0, 0.0), (api.S.ZONE_RADIAL, 1.6, 2.0, 0.3, 0.0),
             (api.S.ZONE_X, 1.7, 2.0, 0.0, 0.0), (api.S.ZONE_Y, 1.8, 2.0, 0.0, 0.0)][:case["zones"]]
    return {"xyz": pts[:nc].contiguous(), "zext": torch.stack([z[lay], z[lay + 1]], -1).to(torch.float32).contiguous(),
            "eta": eta.contiguous(), "alpha": torch.rand(nc, generator=g, device=DEV),
            "uc": 0.1 * torch.randn(nc, 3, generator=g, device=DEV), "zones": zones,
            "vel": [vel[:, d].contiguous() for d in range(3)], "area": areas,
            "faces": faces.reshape(-1, 6).to(torch.int32).contiguous(),
            "vol": (dz[:, None, None] * base).expand(nlay, nth, nr).reshape(-1).to(torch.float32).contiguous()}


def _inputs(c, seed):
    """What prepare and exact share: the sea, levels, times and points of a case."""
    g = _gen(seed)
    kind = c["kind"]
    if kind == "step2d":
        s = _stokes(g, c["nx"])
        nb = max(2, round(0.75 * c["nz"]))
        dz = 1.6 / (c["nz"] - nb)
        st = np.geomspace(1.0, 40.0, nb - 1)
        z = np.concatenate([-np.cumsum(st * 8.0 / st.sum())[::-1], [0.0], dz * np.arange(1, c["nz"] - nb + 1)]).astype(np.float32)
        t, tq = _times(c["n_tl"], PERIOD)
        return s, z, t, tq, _cloud(g, c["points"], (0, 0, -8.0), (s["Lx"], 0, 1.6))
    large = c["nx"] >= 2048
    Hs = 0.0382 if large or kind == "direct" else 0.05
    s = _sea(g, c["nx"], c["ny"], Hs, c.get("depth", 0.0))
    if kind == "direct":
        z_lo = -1.0 if s["depth"] <= 0 else max(-1.0, -0.95 * s["depth"])
        return s, None, None, 0.31, _near_body(g, s, c["points"], z_lo, 1.5 * Hs)
    z = _levels(c["nz"], -1.0 if s["depth"] <= 0 else -min(1.0, s["depth"]), 1.5 * Hs)
    t, tq = _times(c["n_tl"], PERIOD)
    if kind in ("step3d", "gather_mesh", "learned"):
        shift = _rand(g, 2) * 0.1
        pts = _mesh(c, 0.5 * s["Lx"] + float(shift[0]), 0.5 * s["Ly"] + float(shift[1]))[3]
    elif kind == "gather_cloud":
        pts = _cloud(g, c["points"], (0, 0, float(z[0])), (s["Lx"], s["Ly"], float(z[-1])), c["order"])
    else:
        pts = None
    return s, z, t, tq, pts


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind == "batch":
        items = []
        for s, z, t, tq, pts in _batch_items(case, seed):
            sea = {k: (v.cpu().numpy() if torch.is_tensor(v) else v) for k, v in s.items()}
            items.append({"sea": sea, "z_levels": z, "pad_n": 1, "t_levels": t, "t": tq, "pts": pts.cpu().numpy(), "bin": True})
        return {**st, "batch": api.Batch(items)}
    if kind == "train":
        params, x, field, target, batch = _train_data(case, seed)
        return {**st, "mlp": api.Mlp(params, DEV), "x": x, "field": field, "target": target, "batch": batch,
                "loss": torch.zeros(1, device=DEV)}
    if kind == "cells":
        c = _cells(case, seed)
        n = len(c["vol"])
        return {**st, **c, "ai": torch.empty(n, device=DEV), "wt": torch.empty(n, device=DEV), "div": torch.empty(n, device=DEV)}
    s, z, t, tq, pts = _inputs(case, seed)
    st.update(z=z, t=t, tq=tq, pts=pts, out=_out(len(pts)) if pts is not None else None)
    if kind in ("step2d", "step3d", "grid"):
        st.update(modes=_modes(s), grid=_empty_grid(case, s, z, t))
    elif kind == "direct":
        st.update(modes=_modes(s))
    elif kind == "learned":
        st.update(grid=_filled_grid({**case, "pad": 1, "scheme": "lagrange3"}, s, z, t),
                  mlp=api.Mlp(_mlp_params(_gen(seed + 7)), DEV, out_scale=0.01))
    else:
        st.update(grid=_filled_grid(case, s, z, t))
        if case.get("order") == "binned":
            st["perm"], st["sorted"] = api.bin_points(st["grid"], pts)
    return st


def run(st):
    kind = st["kind"]
    if kind in ("step2d", "step3d", "grid"):
        c, grid = st["case"], st["grid"]
        api.fields_on_grid(st["modes"], st["z"], c["pad"], st["t"], out=grid, scheme=c["scheme"])
        res = {"nodes": grid.nodes, "grid_eta": grid.eta}
        if st["pts"] is not None:
            res.update(api.interp(grid, st["tq"], st["pts"], out=st["out"])[0])
        return res
    if kind in ("gather_mesh", "gather_cloud"):
        if "perm" in st:
            return api.interp_permuted(st["grid"], st["tq"], st["sorted"], st["perm"], out=st["out"])[0]
        return api.interp(st["grid"], st["tq"], st["pts"], out=st["out"])[0]
    if kind == "batch":
        st["batch"].run()
        return [{**it["out"], "nodes": it["grid"].nodes, "grid_eta": it["grid"].eta} for it in st["batch"].items]
    if kind == "direct":
        return api.direct(st["modes"], st["tq"], st["pts"], precision=st["case"]["precision"], out=st["out"])
    if kind == "learned":
        return api.interp_learned(st["grid"], st["tq"], st["pts"], st["mlp"], out=st["out"])[0]
    if kind == "train":
        mlp = st["mlp"]
        mlp.train_step(st["x"], st["field"], st["target"], st["batch"], loss=st["loss"])
        return {"params": mlp.params, "m": mlp.m, "v": mlp.v, "loss": st["loss"]}
    ai, wt = api.relax_cells(st["xyz"], st["zext"], st["eta"], st["zones"], alpha=st["alpha"], u_c=st["uc"],
                             out_alpha_i=st["ai"], out_weight=st["wt"])
    div = api.fv_divergence(*st["vel"], st["area"], st["faces"], st["vol"], out=st["div"])
    return {"alpha_i": ai, "weight": wt, "alpha": st["alpha"], "u_c": st["uc"], "div": div}


# ------------------------------------------------------------------------------------ work
def _grid_work(nx, ny, nz, pad, n_tl):
    nxr, nyr = pad * nx, pad * ny if ny > 1 else 1
    n = n_tl * nz * nyr * nxr
    # modes and frequencies in; nodes and eta out; two complex transforms per level
    return (4 * 8 * ny * (nx // 2 + 1) + 16 * n + 4 * n_tl * nyr * nxr, 2 * 5 * n * math.log2(max(2, nxr * nyr)))


def _gather_work(n, grid_nodes, touched):
    return 32 * n + 16 * min(grid_nodes, touched), n * (64 * 8 + 16 * 2 + 40)


def _mesh_count(c):
    nr, nth, nl = c["nr"], c["nth"], c["nlay"]
    return nl * nth * nr + nl * nth * (nr + 1) + nl * nth * nr + (nl + 1) * nth * nr


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0
        r = np.random.default_rng(case["sizes"])
        for _ in range(case["instances"]):
            nx, ny = (1 << int(r.integers(case["lo"], case["hi"] + 1)) for _ in "xy")
            n = int(10 ** r.uniform(4, math.log10(case["points_hi"])))
            nodes = case["n_tl"] * case["nz"] * nx * ny
            for x in (_grid_work(nx, ny, case["nz"], 1, case["n_tl"]), _gather_work(n, nodes, 64 * case["n_tl"] * n)):
                b, f = b + x[0], f + x[1]
        return {"bytes": b, "flops": f}
    if kind == "train":
        B, p = case["batch"], 8772
        return {"bytes": B * (68 * 4 + 12) + 6 * 4 * p, "flops": 3 * 2 * B * (67 * 64 + 64 * 64 + 64 * 4)}
    if kind == "cells":
        nc = case["nr"] * case["nth"] * case["nlay"]
        return {"bytes": nc * (32 + 8 + 28 + 8) + 24 * (_mesh_count(case) - nc), "flops": nc * (60 + 12 * case["zones"])}
    if kind == "direct":
        modes, n = case["nx"] // 2 * max(1, case["ny"] - 1), case["points"]
        return {"bytes": 32 * modes + 32 * n, "flops": 20 * modes * n}
    pad = case.get("pad", 1)
    nx, ny, nz, n_tl = case["nx"], case.get("ny", 1), case["nz"], case["n_tl"]
    b = f = 0
    if kind in ("step2d", "step3d", "grid"):
        b, f = _grid_work(nx, ny, nz, pad, n_tl)
    if kind != "grid":
        n = case["points"] if "points" in case else _mesh_count(case)
        nodes = n_tl * nz * nx * pad * (ny * pad if ny > 1 else 1)
        # a mesh reaches two peak wavelengths (16 modes' nodes each) from its centre
        reach = n_tl * nz * (4 * 16 * pad + 4) ** 2 if "nr" in case else 64 * n_tl * n
        x = _gather_work(n, nodes, reach)
        b, f = b + x[0], f + x[1]
        if kind == "learned":
            f += 8 * n * (67 * 64 + 64 * 64 + 64 * 4)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------------------ 64 bits
def _depth_factors(k, z, h):
    if h <= 0:
        e = torch.exp(k * z)
        return e, e
    d = 1 + torch.exp(-2 * k * h)
    e1, e2 = torch.exp(k * z), torch.exp(-k * (z + 2 * h))
    return (e1 + e2) / d, (e1 - e2) / d


def _fields(s, z, pad, times, scheme, nodes, eta):
    """The grid of a sea by 64-bit transforms, into nodes [tl][nz][nyr][nxr][4] and eta [tl][nyr][nxr]."""
    nx, ny = s["nx"], s["ny"]
    nxr, nyr = pad * nx, pad * ny if ny > 1 else 1
    kx, ky, k = _wavenumbers(s)
    live = torch.ones(ny, nx // 2 + 1, device=DEV, dtype=torch.float64)
    live[:, -1] = 0
    if ny > 1:
        live[ny // 2] = 0
    if scheme == "spline3":
        m = torch.arange(nx // 2 + 1, device=DEV, dtype=torch.float64)
        live = live * 3 / (2 + torch.cos(2 * math.pi * m / nxr))[None, :]
        if ny > 1:
            n = torch.arange(ny, device=DEV, dtype=torch.float64)
            live = live * (3 / (2 + torch.cos(2 * math.pi * torch.where(n < ny / 2, n, n - ny) / nyr)))[:, None]

    def inverse(spec):                                                  # [..., ny, nx/2+1] -> [..., nyr, nxr]
        full = spec.new_zeros(*spec.shape[:-2], nyr, nxr // 2 + 1)
        if ny > 1:
            full[..., :ny // 2, :nx // 2 + 1] = spec[..., :ny // 2, :]
            full[..., nyr - ny // 2 + 1:, :nx // 2 + 1] = spec[..., ny // 2 + 1:, :]
            full = torch.fft.ifft(full, dim=-2, norm="forward")
        else:
            full[..., :nx // 2 + 1] = spec
        return torch.fft.irfft(full, n=nxr, dim=-1, norm="forward")

    zz = torch.tensor(np.asarray(z, np.float64), device=DEV)
    step = max(1, min(len(z), (1 << 24) // (nxr * nyr)))
    for l, t in enumerate(times):
        turn = torch.polar(live, -s["omega"] * float(t))
        Ae, Ap, At = (s[q].to(torch.complex128) * turn for q in ("A_eta", "A_phi", "A_phit"))
        eta[l] = inverse(Ae)
        for a in range(0, len(z), step):
            F, S = _depth_factors(k, zz[a:a + step, None, None], s["depth"])
            nodes[l, a:a + step, ..., 0] = inverse(1j * kx * Ap * F)
            nodes[l, a:a + step, ..., 1] = inverse(1j * ky * Ap * F) if ny > 1 else 0
            nodes[l, a:a + step, ..., 2] = inverse(k * Ap * S)
            nodes[l, a:a + step, ..., 3] = inverse(At * F)


def _exact_grid(c, s, z, t):
    nxr, nyr = c["pad"] * c["nx"], c["pad"] * c.get("ny", 1) if c.get("ny", 1) > 1 else 1
    nodes = torch.empty(len(t), len(z), nyr, nxr, 4, device=DEV, dtype=torch.float64)
    eta = torch.empty(len(t), nyr, nxr, device=DEV, dtype=torch.float64)
    _fields(s, z, c["pad"], t, c["scheme"], nodes, eta)
    return nodes, eta


def _lagrange(nodes, x):
    k = nodes.shape[-1]
    w = []
    for a in range(k):
        v = torch.ones_like(x)
        for b in range(k):
            if b != a:
                v = v * (x - nodes[..., b]) / (nodes[..., a] - nodes[..., b])
        w.append(v)
    return torch.stack(w, -1)


def _axis(x, L, n, scheme):
    q = x * (n / L)
    i = torch.floor(q)
    f = q - i
    if scheme == "spline3":
        w = torch.stack([(1 - f) ** 3, 3 * f ** 3 - 6 * f ** 2 + 4, -3 * f ** 3 + 3 * f ** 2 + 3 * f + 1, f ** 3], -1) / 6
    else:
        w = _lagrange(torch.arange(-1, 3, device=DEV, dtype=torch.float64).expand(len(x), 4), f)
    return (i.long()[:, None] + torch.arange(-1, 3, device=DEV)) % n, w, f


def _stencils(s, scheme, z, times, tq, nodes, eta, pts):
    """Chunks of points with their time-blended stencils: indices, weights, offsets, values."""
    nyr, nxr = eta.shape[1:]
    zz = torch.tensor(np.asarray(z, np.float64), device=DEV)
    wt = _lagrange(torch.tensor(np.asarray(times, np.float64), device=DEV), torch.tensor(float(tq), device=DEV, dtype=torch.float64))
    flat, ef = nodes.reshape(len(times), -1, 4), eta.reshape(len(times), -1)
    for a in range(0, len(pts), 1 << 18):
        p = pts[a:a + (1 << 18)].double()
        ix, wx, fx = _axis(p[:, 0], s["Lx"], nxr, scheme)
        if nyr > 1:
            iy, wy, fy = _axis(p[:, 1], s["Ly"], nyr, scheme)
        else:
            iy, wy, fy = torch.zeros(len(p), 1, dtype=torch.long, device=DEV), torch.ones(len(p), 1, dtype=torch.float64, device=DEV), None
        pz = p[:, 2].contiguous()
        j = (torch.searchsorted(zz, pz, right=True) - 1).clamp(0, len(z) - 2)
        j0 = (j - 1).clamp(0, len(z) - 4)
        iz = j0[:, None] + torch.arange(4, device=DEV)
        wz = _lagrange(zz[iz], pz)
        inside = (pz >= zz[0]) & (pz <= zz[-1])
        fz = (pz - zz[j0 + 1]) / (zz[j0 + 2] - zz[j0 + 1])
        col = (iy[:, :, None] * nxr + ix[:, None, :])                    # [n][by][4]
        idx = iz[:, :, None, None] * (nyr * nxr) + col[:, None]          # [n][4][by][4]
        val = sum(wt[l] * flat[l][idx].double() for l in range(len(times)))
        e = sum(wt[l] * (ef[l][col].double() * wy[:, :, None] * wx[:, None, :]).sum((1, 2)) for l in range(len(times)))
        w = wz[:, :, None, None] * wy[:, None, :, None] * wx[:, None, None, :]
        yield p, val, w, e, inside, (fx, fy, fz)


def _bernoulli(f, inside, e):
    f = torch.where(inside[:, None], f, float("nan"))
    return {"eta": e, "u": f[:, 0], "v": f[:, 1], "w": f[:, 2], "p": -RHO * (f[:, 3] + 0.5 * (f[:, :3] ** 2).sum(1))}


def _join(parts):
    return {k: torch.cat([p[k] for p in parts]) for k in FIELDS}


def _exact_gather(s, scheme, z, t, tq, nodes, eta, pts):
    return _join([_bernoulli((w[..., None] * val).sum((1, 2, 3)), inside, e)
                  for _, val, w, e, inside, _ in _stencils(s, scheme, z, t, tq, nodes, eta, pts)])


def _net(params, x):
    i, P = 0, []
    for h in ((64, 67), (64,), (64, 64), (64,), (4, 64), (4,)):
        n = math.prod(h)
        P.append(params[i:i + n].reshape(h))
        i += n
    gelu = torch.nn.functional.gelu
    h1 = gelu(x @ P[0].T + P[1], approximate="tanh")
    return gelu(h1 @ P[2].T + P[3], approximate="tanh") @ P[4].T + P[5]


def _bf16_weights(params):
    """The network's weights as they are held for inference: matrices in BF16, biases in FP32."""
    p, i = params.clone(), 0
    for h in ((64, 67), (64,), (64, 64), (64,), (4, 64), (4,)):
        n = math.prod(h)
        if len(h) == 2:
            p[i:i + n] = p[i:i + n].bfloat16().float()
        i += n
    return p.double()


def _exact_learned(s, z, t, tq, grid, pts, params):
    parts = []
    P = _bf16_weights(params)
    for p, val, w, e, inside, (fx, fy, fz) in _stencils(s, "lagrange3", z, t, tq, grid.nodes, grid.eta, pts):
        lag = (w[..., None] * val).sum((1, 2, 3))
        v = val.reshape(len(p), 64, 4).transpose(1, 2)                  # [n][4 fields][64]
        sc = v.abs().amax(2) + 1e-30
        off = torch.stack([fx, fy, fz], -1)[:, None].expand(-1, 4, -1)
        y = _net(P, torch.cat([v / sc[..., None], off], -1).reshape(-1, 67)).reshape(-1, 4, 4)
        parts.append(_bernoulli(lag + sc * 0.01 * torch.diagonal(y, dim1=1, dim2=2), inside, e))
    return _join(parts)


def _exact_direct(s, t, pts):
    nx, ny = s["nx"], s["ny"]
    kx, ky, k = _wavenumbers(s)
    M = nx // 2
    turn = torch.polar(torch.ones_like(k), -s["omega"] * t)
    Ae, Ap, At = (s[q].to(torch.complex128) * turn for q in ("A_eta", "A_phi", "A_phit"))
    c = torch.full((M,), 2.0, device=DEV, dtype=torch.float64)
    c[0] = 1
    parts = []
    for a in range(0, len(pts), 1 << 15):
        p = pts[a:a + (1 << 15)].double()
        X = torch.polar(torch.ones(len(p), M, device=DEV, dtype=torch.float64), p[:, :1] * kx[:, :M]) * c
        Y = torch.polar(torch.ones(len(p), ny, device=DEV, dtype=torch.float64), p[:, 1:2] * ky[:, 0])
        f, e = torch.zeros(len(p), 4, device=DEV, dtype=torch.float64), torch.zeros(len(p), device=DEV, dtype=torch.float64)
        for r in range(ny):
            if ny > 1 and r == ny // 2:
                continue
            F, S = _depth_factors(k[r, :M], p[:, 2:], s["depth"])
            h = Ap[r, :M]
            E = torch.stack([1j * kx[0, :M] * h, 1j * ky[r, 0] * h, At[r, :M]], 1)
            q = (X * F) @ E
            f[:, [0, 1, 3]] += (q * Y[:, r:r + 1]).real
            f[:, 2] += (((X * S) @ (k[r, :M] * h)) * Y[:, r]).real
            e += ((X @ Ae[r, :M]) * Y[:, r]).real
        parts.append(_bernoulli(f, torch.ones(len(p), dtype=torch.bool, device=DEV), e))
    return _join(parts)


def _exact_train(case, seed):
    params, x, field, target, batch = _train_data(case, seed)
    P = params.double().requires_grad_()
    b = batch.long()
    y = _net(P, x[b, :67].double()).gather(1, field[b].long()[:, None])[:, 0]
    loss = ((y - target[b].double()) ** 2).mean()
    g, = torch.autograd.grad(loss, P)
    m, v = 0.1 * g, 0.001 * g * g
    return {"params": P.detach() - 1e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8), "m": m, "v": v,
            "loss": loss.detach().reshape(1)}


def _exact_cells(case, seed):
    c = _cells(case, seed)
    x, y = c["xyz"][:, 0].double(), c["xyz"][:, 1].double()
    w = torch.zeros_like(x)
    for kind, inner, outer, cx, cy in c["zones"]:
        q = x if kind == api.S.ZONE_X else y if kind == api.S.ZONE_Y else torch.hypot(x - cx, y - cy)
        f = ((q - inner) / (outer - inner)).clamp(0, 1)
        w = torch.maximum(w, f * f * (3 - 2 * f))
    lo, hi = c["zext"].double().unbind(1)
    ai = ((c["eta"].double() - lo) / (hi - lo)).clamp(0, 1)
    flux = sum(v.double() * c["area"][:, d].double() for d, v in enumerate(c["vel"]))
    i = c["faces"].long()
    div = (flux[i.abs() - 1] * i.sign()).sum(1) / c["vol"].double()
    return {"alpha_i": ai, "weight": w, "alpha": w * ai + (1 - w) * c["alpha"].double(),
            "u_c": (1 - w)[:, None] * c["uc"].double(), "div": div}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        res = []
        for s, z, t, tq, pts in _batch_items(case, seed):
            nodes, eta = _exact_grid({"pad": 1, "nx": s["nx"], "ny": s["ny"], "scheme": "lagrange3"}, s, z, t)
            res.append({**_exact_gather(s, "lagrange3", z, t, tq, nodes, eta, pts), "nodes": nodes, "grid_eta": eta})
        return res
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "cells":
        return _exact_cells(case, seed)
    if kind == "direct" and case["nx"] * case["ny"] * case["points"] > 1 << 36:
        return None                                                     # 10^12 terms: minutes in 64 bits
    s, z, t, tq, pts = _inputs(case, seed)
    if kind == "direct":
        return _exact_direct(s, tq, pts)
    if kind == "learned":
        grid = _filled_grid({**case, "pad": 1, "scheme": "lagrange3"}, s, z, t)
        return _exact_learned(s, z, t, tq, grid, pts, _mlp_params(_gen(seed + 7)))
    if kind in ("gather_mesh", "gather_cloud"):
        grid = _filled_grid(case, s, z, t)
        return _exact_gather(s, case["scheme"], z, t, tq, grid.nodes, grid.eta, pts)
    nodes, eta = _exact_grid(case, s, z, t)
    res = {"nodes": nodes, "grid_eta": eta}
    if pts is not None:
        res.update(_exact_gather(s, case["scheme"], z, t, tq, nodes, eta, pts))
    return res
