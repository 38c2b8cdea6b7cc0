"""The training kernel's row tiles at their edges: one row, rows around a tile's 64, and more tiles than
blocks (152 x 64 rows), so that a block adds several tiles' gradients. Gradients against the FP64
oracle on the same BF16-rounded weights: <= 1e-2 of each tensor's largest entry (BF16 operands, FP32
sums: 2^-9 per operand); a training step moves exactly the parameters that its own gradient and the
Adam rule give."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_12716_gb300 import build
    build.build()
    from paper_2005_12716_gb300 import api
    return torch, api


@pytest.mark.parametrize("B", [1, 63, 65, 152 * 64, 152 * 64 + 1, 20000])
def test_gradients_and_step_at_tile_edges(env, B):
    torch, api = env
    rng = np.random.default_rng(B)
    p = omlp.init_params(3)
    for k in p:
        p[k] = torch.from_numpy((p[k] + 0.05 * rng.standard_normal(p[k].shape)).astype(np.float32)).bfloat16().double().numpy()
    n = 6000
    x = np.zeros((n, 68), np.float32)
    x[:, :64] = rng.uniform(-1, 1, (n, 64))
    x[:, 64:67] = rng.random((n, 3))
    field = rng.integers(0, 4, n).astype(np.int32)
    target = rng.standard_normal(n).astype(np.float32)
    batch = rng.integers(0, n, B).astype(np.int32)
    cu = lambda a: torch.from_numpy(a).cuda()   # noqa: E731
    mlp = api.Mlp(torch.from_numpy(api.mlp_flatten(p)))
    g, loss = mlp.grad(cu(x), cu(field), cu(target), cu(batch))
    ref_loss, ref = omlp.loss_and_grad(p, x[batch, :67].astype(np.float64), field[batch], target[batch].astype(np.float64))
    got = api.mlp_unflatten(g.cpu().numpy())
    assert abs(float(loss) - ref_loss) <= 1e-2 * ref_loss
    for k in ref:
        assert np.max(np.abs(got[k] - ref[k])) <= 1e-2 * np.max(np.abs(ref[k])) + 1e-12, k
    before = mlp.params.clone()
    out = torch.zeros(1, device="cuda")
    mlp.train_step(cu(x), cu(field), cu(target), cu(batch), loss=out)
    assert float(out) == float(loss)
    # the decays are FP32 numbers: 1 - 0.999f is 0.99998713e-3
    c1, c2 = float(np.float32(1) - np.float32(0.9)), float(np.float32(1) - np.float32(0.999))
    assert torch.allclose(mlp.m, c1 * g, rtol=1e-6, atol=0) and torch.allclose(mlp.v, c2 * g * g, rtol=1e-5, atol=1e-30)
    step = 1e-3 * (mlp.m / c1) / (torch.sqrt(mlp.v / c2) + 1e-8)
    assert torch.allclose(mlp.params, before - step, rtol=0, atol=2e-6)
