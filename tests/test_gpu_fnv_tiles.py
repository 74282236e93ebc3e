"""The tiled GPU hash against the oracle at the edges of its tiling: runs of
64 bytes a thread, tiles of 64 KiB, and hash lists of one tile and more."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

CHUNK = 65536


def _check(x):
    import torch
    from paper_2607_18541_gb300 import aclz
    d = torch.zeros(x.size + 16, dtype=torch.uint8, device="cuda")
    d[:x.size] = torch.from_numpy(x)
    want = oracle.fnv_chunked(x)
    assert aclz.aclz_fnv(d, x.size) == want
    assert aclz.aclz_fnv_noalloc(d, x.size) == want


@pytest.mark.parametrize("n", [0, 1, 31, 32, 33, 63, 64, 65, 2047, 2048, 2049, 32767, 65472, 65535, 65536, 65537,
                               65536 + 63, 3 * 65536 - 1, 3 * 65536, 40 * 65536 + 12345])
@pytest.mark.parametrize("fill", ["random", "zeros", "ones"])
def test_tile_edges(n, fill):
    x = {"random": lambda: np.random.RandomState(n + 1).randint(0, 256, n),
         "zeros": lambda: np.zeros(n), "ones": lambda: np.full(n, 255)}[fill]().astype(np.uint8)
    _check(x)


@pytest.mark.parametrize("chunks", [8190, 8191, 8192, 16385])
def test_hash_list_of_several_tiles(chunks):
    # 8191 hashes and the length fill one tile; the last chunk is short
    tile = np.random.RandomState(chunks).randint(0, 256, 7 * CHUNK + 5).astype(np.uint8)
    _check(np.resize(tile, chunks * CHUNK - 17))
