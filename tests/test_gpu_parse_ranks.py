"""The GPU parse where a position's rank lies near 0, so that a round of
candidates reaches past the first rank: inputs that hold a prefix and its
complement with few ranks between them, against the host encoder and by
decoding the container."""
import numpy as np
import pytest

import oracle
from paper_2607_18541_gb300 import aclz

pytestmark = pytest.mark.gpu

PRESETS = [(4, 4, 4, 4), (6, 8, 10, 12), (12, 16, 24, 32)]


def _check(x, mm, depth, block=1 << 16):
    x = np.frombuffer(bytes(x), dtype=np.uint8)
    p = aclz.aclz_encode_params_default(aclz.ACLZ_PRESET_BASE)
    for i in range(4):
        p.min_match[i] = mm[i]
    p.block_size, p.chain_depth = block, depth
    want = aclz.aclz_encode(x, p, threads=2)
    got = aclz.aclz_encode_gpu(x, p)
    assert got.size == want.size and np.array_equal(got, want)
    assert np.array_equal(oracle.decode(got), x)


@pytest.mark.parametrize("n", [20, 100, 5000, 70000])
@pytest.mark.parametrize("mm", PRESETS)
def test_header_and_fill(n, mm):
    for head in (4, 8, 40):
        _check(bytes(head) + b"\xff" * n, mm, 64)


@pytest.mark.parametrize("a", [0x01, 0x20, 0x55, 0x7f])
@pytest.mark.parametrize("depth", [1, 8, 64, 65, 200])
def test_complement_pairs(a, depth):
    # the smallest prefix is a's, the complement's comes within the first
    # ranks, and more ranks than a round follow
    r = np.random.RandomState(a + depth)
    mid = bytes(range(a + 1, min(a + 30, 255 - a)))
    _check(bytes([a] * 4) + mid + bytes([255 - a]) * 300, (4, 4, 4, 4), depth)
    _check(bytes([255 - a] * 90) + bytes([a] * 12) + bytes([255 - a]) * 90, (6, 8, 10, 12), depth, 64)
    # a prefix of four different bytes and its complement, over and over
    w = bytes([a, a + 1, a + 2, a + 3])
    c = bytes(255 - b for b in w)
    x = w + b"".join(c + bytes(r.randint(200, 255, int(r.randint(0, 6))).astype(np.uint8)) for _ in range(150))
    _check(x, (4, 4, 4, 4), depth)


@pytest.mark.parametrize("depth", [1, 8, 64, 65, 200])
def test_runs_of_two_bytes(depth):
    r = np.random.RandomState(depth)
    for k in range(40):
        n, x = int(r.randint(20, 300)), b""
        a = [0x00, 0x55][k % 2]
        while len(x) < n:
            x += bytes([[a, 255 - a][r.randint(2)]]) * int(r.randint(1, 13))
        _check(x, PRESETS[k % 3], depth)
