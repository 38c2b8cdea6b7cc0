"""The relaxation kernel's blends of four cells at a time: groups with no, some and all cells in a zone, counts
around a group and a block, alpha or u_c or both or neither given, arrays of any alignment; cells outside
the zones keep their bits, and every form gives the bits of the cell-by-cell formula in FP32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4, 7, 1023, 1028, 50_003])
@pytest.mark.parametrize("share", [0.1, 0.5, 0.97])
@pytest.mark.parametrize("which", ["both", "alpha", "u", "none"])
def test_blends_of_four(n, share, which):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import api, _swense as S
    rng = np.random.default_rng(n)
    xyz = rng.uniform(0, 1, (n, 3)).astype(np.float32)
    xyz[:, 0] = np.where(rng.random(n) < share, 1.0 + rng.uniform(0.0, 1.1, n), 0.5)   # in the zone, or well outside
    zl = rng.uniform(-0.1, 0.0, n).astype(np.float32)
    zext = np.stack([zl, zl + np.float32(0.05)], 1)
    eta = rng.uniform(-0.1, 0.05, n).astype(np.float32)
    alpha, uc = rng.random(n).astype(np.float32), rng.standard_normal((n, 3)).astype(np.float32)
    uc[rng.random(n) < 0.1] = -0.0
    got = []
    for shift in (0, 1):
        def put(a, s):
            b = torch.empty((n + 1, *a.shape[1:]), device="cuda")
            b[s:s + n] = torch.from_numpy(a).cuda()
            return b[s:s + n]
        ins = [put(a, shift) for a in (xyz, zext, eta)]
        al = put(alpha, shift) if which in ("both", "alpha") else None
        u = put(uc, 0 if shift else 0) if which in ("both", "u") else None
        ai, w = api.relax_cells(*ins, [(S.ZONE_X, 1.0, 2.0, 0.0, 0.0)], alpha=al, u_c=u)
        got.append([t.cpu().numpy() for t in (ai, w, al, u) if t is not None])
    for a, b in zip(*got):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
    ai, w = got[0][:2]
    out = w == 0
    assert out.sum() == (xyz[:, 0] <= 1).sum()
    keep = np.float32(1) - w
    rest = got[0][2:]
    if which in ("both", "alpha"):
        a = rest.pop(0)
        assert np.array_equal(a[out].view(np.uint32), alpha[out].view(np.uint32))
        # one rounding of keep alpha, one of the fused sum
        want = (w.astype(np.float64) * ai + (keep * alpha).astype(np.float64)).astype(np.float32)
        assert np.array_equal(a[~out], want[~out])
    if which in ("both", "u"):
        v = rest.pop(0)
        assert np.array_equal(v[out].view(np.uint32), uc[out].view(np.uint32))
        assert np.array_equal(v[~out], (uc * keep[:, None])[~out])
