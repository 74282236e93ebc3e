"""GPU tile decode at the edges of a tile and of the word registers: lengths
around a step and around a tile, streams that take no word, and ones that
take two for almost every byte."""
import numpy as np
import pytest

from paper_2607_18541_gb300 import aclz

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _bytes(kind, n):
    r = np.random.RandomState(n + 7)
    if kind == "one":
        return np.full(n, 9)
    if kind == "flat":
        return r.randint(0, 256, n)
    if kind == "rare":  # one symbol almost always: a few bytes cost 12 bits each
        return np.where(r.rand(n) < 0.002, r.randint(0, 256, n), 65)
    if kind == "bursts":  # runs of cheap and of dear bytes
        return np.where((np.arange(n) // 500) % 2, r.randint(0, 256, n), 65)
    return r.geometric(0.3, n) % 256


@pytest.mark.parametrize("kind", ["one", "flat", "rare", "bursts", "skewed"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 2047, 65535, 65536, 65537, 65536 + 33, 3 * 65536 + 5])
def test_tile_edges(kind, n):
    x = _bytes(kind, n).astype(np.uint8)
    runs = np.array([min(1 << 17, n - p) for p in range(0, n, 1 << 17)], np.uint32)  # one literal run a block
    none = np.zeros(runs.size, np.uint32)
    c = aclz.aclz_pack(n, 1 << 17, (4, 4, 4, 4), none + 1, runs, none, none.astype(np.uint64), x)
    e = aclz.aclz_acle_encode(c)
    h = aclz.aclz_upload_acle(e)
    try:
        out = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
        aclz.aclz_decode_all(h, out, cap=n)
        assert aclz.aclz_device_status(h) == 0
        assert np.array_equal(out[:n].cpu().numpy(), x)
    finally:
        aclz.aclz_free(h)
