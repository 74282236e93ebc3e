"""The GPU parse against the host encoder where its tiling can go wrong:
chain depths around one round of candidates, match lengths around the staged
and the capped comparison, blocks smaller and larger than a window of
lengths, chains reaching rank 0, short inputs."""
import numpy as np
import pytest

from paper_2607_18541_gb300 import aclz

pytestmark = pytest.mark.gpu


def _params(mm, block, depth, window=1 << 40):
    p = aclz.aclz_encode_params_default(aclz.ACLZ_PRESET_BASE)
    for i in range(4):
        p.min_match[i] = mm[i]
    p.block_size, p.chain_depth, p.window = block, depth, window
    return p


def _same(x, p, bmm=None):
    want = aclz.aclz_encode(x, p, block_min_match=bmm, threads=2)
    got = aclz.aclz_encode_gpu(x, p, block_min_match=bmm)
    assert got.size == want.size and np.array_equal(got, want)


def _repeats(n, lengths, seed):
    """Random bytes of a small alphabet with copies of the given lengths."""
    r = np.random.RandomState(seed)
    x = r.randint(0, 40, n).astype(np.uint8)
    p = 300
    while p + max(lengths) < n:
        k = int(r.choice(lengths))
        s = int(r.randint(0, p - k)) if p > k else 0
        x[p:p + k] = x[s:s + k]
        p += k + int(r.randint(0, 40))
    return x


@pytest.mark.parametrize("depth", [1, 31, 32, 63, 64, 65, 127, 128, 129, 1000])
@pytest.mark.parametrize("mm", [(4, 4, 4, 4), (6, 8, 10, 12), (12, 16, 24, 32)])
def test_depths(depth, mm):
    r = np.random.RandomState(depth)
    x = r.randint(0, 3, 20000).astype(np.uint8)  # long chains of few prefixes
    _same(x, _params(mm, 1024, depth))


@pytest.mark.parametrize("mm", [(4, 4, 4, 4), (12, 16, 24, 32), (19, 20, 21, 63), (64, 65, 100, 255)])
@pytest.mark.parametrize("block", [64, 512, 4096, 65536])
def test_lengths_around_the_caps(mm, block):
    x = _repeats(60000, [5, 11, 12, 13, 19, 20, 21, 31, 62, 63, 64, 65, 66, 127, 200, 900], block)
    _same(x, _params(mm, block, 64))
    _same(x, _params(mm, block, 8, window=5000))


@pytest.mark.parametrize("n", [0, 1, 3, 4, 5, 20, 63, 64, 65, 511, 512, 513, 1023, 1025, 4097])
def test_short_inputs(n):
    for fill in (np.zeros(n), np.arange(n) % 7, np.random.RandomState(n).randint(0, 256, n)):
        _same(fill.astype(np.uint8), _params((4, 6, 8, 10), 256, 64))


def test_block_thresholds():
    x = _repeats(50000, [8, 24, 70], 3)
    nb = (x.size + 1023) // 1024
    bmm = np.random.RandomState(4).randint(4, 80, (nb, 4)).astype(np.uint8)
    _same(x, _params((6, 8, 10, 12), 1024, 64), bmm)


@pytest.mark.parametrize("depth", [64, 65, 200])
def test_staged_bytes(depth):
    # many candidates that agree for 35, 36, 37 and more bytes, the longest
    # among the first round's or a later round's
    r = np.random.RandomState(depth)
    stem = r.randint(0, 256, 80).astype(np.uint8)
    parts = []
    for k in range(180):
        n = int(r.choice([34, 35, 36, 37, 38, 60, 63, 64, 65, 80]))
        parts += [stem[:n], r.randint(0, 256, int(r.randint(1, 9))).astype(np.uint8)]
    _same(np.concatenate(parts), _params((6, 8, 10, 12), 4096, depth))
    _same(np.concatenate(parts), _params((30, 36, 37, 40), 65536, depth))
