"""The relaxation kernel's four-cell words at their edges: cell counts around four and a block, and arrays
that are not 16-byte aligned (which take cells one by one), both bit for bit the same as each other and
within 1e-6 of the formula in FP64."""
import numpy as np
import pytest


pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 1025, 70_001])
def test_word_and_single_cells_agree(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import api, _swense as S
    rng = np.random.default_rng(n)
    xyz = rng.uniform(-2, 2, (n + 1, 3)).astype(np.float32)
    zl = rng.uniform(-0.1, 0.0, n + 1).astype(np.float32)
    zext = np.stack([zl, zl + np.float32(0.05)], 1)
    eta = rng.uniform(-0.1, 0.05, n + 1).astype(np.float32)
    alpha, uc = rng.random(n + 1).astype(np.float32), rng.standard_normal((n + 1, 3)).astype(np.float32)
    zones = [(S.ZONE_X, 1.0, 2.0, 0.0, 0.0), (S.ZONE_RADIAL, 1.5, 2.0, 0.1, 0.0)]
    got = []
    for shift in (0, 1):                             # one cell on: 12, 8 and 4 bytes off
        bufs = []
        for a in (xyz, zext, eta, alpha, uc):
            b = torch.empty((n + 2, *a.shape[1:]), device="cuda")
            b[shift:shift + n] = torch.from_numpy(a[:n]).cuda()
            bufs.append(b[shift:shift + n])
        out = [torch.empty(n + 1, device="cuda")[shift:shift + n] for _ in range(2)]
        api.relax_cells(bufs[0], bufs[1], bufs[2], zones, alpha=bufs[3], u_c=bufs[4], out_alpha_i=out[0], out_weight=out[1])
        got.append([t.cpu().numpy() for t in (out[0], out[1], bufs[3], bufs[4])])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    x = xyz[:n].astype(np.float64)
    s = [np.clip(x[:, 0] - 1.0, 0, 1), np.clip((np.hypot(x[:, 0] - np.float64(np.float32(0.1)), x[:, 1]) - 1.5) / 0.5, 0, 1)]
    w = np.max([-2 * q ** 3 + 3 * q ** 2 for q in s], axis=0)
    ai = np.clip((eta[:n].astype(np.float64) - zext[:n, 0]) / (zext[:n, 1].astype(np.float64) - zext[:n, 0]), 0, 1)
    assert np.allclose(got[0][1], w, atol=1e-6) and np.allclose(got[0][0], ai, atol=1e-6)
    assert np.allclose(got[0][2], w * ai + (1 - w) * alpha[:n], atol=1e-6)
    assert np.allclose(got[0][3], (1 - w)[:, None] * uc[:n], atol=4e-6)
