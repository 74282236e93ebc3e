"""Gradient of the threshold network around the sizes where the kernel
changes: parts of a tile, whole tiles, the largest batch whose tiles are
shared by clusters; against 64-bit autograd of the same network."""
import numpy as np
import pytest

from paper_2607_18541_gb300 import aclz

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 11, 16])
@pytest.mark.parametrize("B", [1, 3, 4, 5, 31, 32, 33, 65, 2047, 2048, 2049, 2081])
def test_gradient(B, K):
    r = np.random.RandomState(B * 17 + K)
    P = aclz.aclz_mlp_param_count(K)
    p = (r.randn(P) * 0.2).astype(np.float32)
    x, y = r.randn(B, 24).astype(np.float32), r.randint(0, K, B).astype(np.int32)
    d = [torch.from_numpy(a).cuda() for a in (p, x, y)]
    g = torch.full((P + 8,), 7.0, device="cuda")
    loss = torch.empty(1, device="cuda")
    scratch = torch.empty(aclz.aclz_mlp_scratch_bytes(K, B), dtype=torch.uint8, device="cuda")
    aclz.aclz_mlp_grad(d[0], K, d[1], d[2], B, g, loss, scratch)
    t = torch.from_numpy(p.astype(np.float64)).requires_grad_(True)
    at, w = 0, []
    for shape in ((24, 64), (64,), (64, 64), (64,), (64, K), (K,)):
        n = int(np.prod(shape))
        w.append(t[at:at + n].reshape(shape))
        at += n
    h = torch.relu(torch.from_numpy(x.astype(np.float64)) @ w[0] + w[1])
    z = torch.relu(h @ w[2] + w[3]) @ w[4] + w[5]
    want = torch.nn.functional.cross_entropy(z, torch.from_numpy(y.astype(np.int64)))
    want.backward()
    got = g.cpu().numpy()
    assert (got[P:] == 7.0).all()
    # 32-bit sums of at most 2081 terms of the gradient's own size
    assert np.abs(got[:P] - t.grad.numpy()).max() <= 1e-4 * np.abs(t.grad.numpy()).max()
    assert abs(loss.item() - want.item()) <= 1e-5 * max(1.0, abs(want.item()))
