"""Wave 0 and the small steps where their tiling can go wrong: literal units
around block and unit boundaries, in-order chains of more levels than one
sort digit and of more matches than one window of the level pass, levels on
both sides of the sizes that change the matches per group, matches around
the size of a group's stage and of a piece."""
import numpy as np
import pytest

import oracle
from paper_2607_18541_gb300 import aclz

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _decode_all_ways(c, flatten=True):
    exp = oracle.decode(c)
    s = torch.cuda.current_stream()
    for flags in (0, aclz.ACLZ_UPLOAD_FLATTEN) if flatten else (0,):
        h = aclz.aclz_upload(c, s, flags=flags)
        try:
            for G in (32, 16, 8):
                for mode in (aclz.ACLZ_MODE_AUTO, aclz.ACLZ_MODE_WAVES, aclz.ACLZ_MODE_PERSISTENT):
                    out = torch.full((exp.size + 32,), 0xA5, dtype=torch.uint8, device="cuda")
                    aclz.aclz_decode_all(h, out, cap=exp.size, G=G, mode=mode, stream=s)
                    assert aclz.aclz_device_status(h, s) == 0
                    got = out.cpu().numpy()
                    assert np.array_equal(got[:exp.size], exp), (flags, G, mode)
                    assert (got[exp.size:] == 0xA5).all()
        finally:
            aclz.aclz_free(h)


def _pack(total, bs, blocks, lits):
    """blocks: per block a list of (lit_len, match_len, src)."""
    ll = np.array([t[0] for b in blocks for t in b], dtype=np.uint32)
    ml = np.array([t[1] for b in blocks for t in b], dtype=np.uint32)
    sr = np.array([t[2] for b in blocks for t in b], dtype=np.uint64)
    n = np.array([len(b) for b in blocks], dtype=np.uint32)
    return aclz.aclz_pack(total, bs, (4, 4, 4, 4), n, ll, ml, sr, lits[:int(ll.sum())])


LITS = np.random.RandomState(1).randint(0, 256, 1 << 22).astype(np.uint8)


@pytest.mark.parametrize("bs", [64, 256, 1024, 4096])
@pytest.mark.parametrize("total", [63, 64, 255, 256, 257, 2048, 4095, 4096, 4097, 70000])
def test_all_literal_blocks(bs, total):
    # units end where blocks end, blocks end where units end, short last block
    blocks = [[(min(bs, total - p), 0, 0)] for p in range(0, total, bs)]
    _decode_all_ways(_pack(total, bs, blocks, LITS))


@pytest.mark.parametrize("seed", range(6))
def test_blocks_with_and_without_literals(seed):
    r = np.random.RandomState(seed)
    bs, nb = int(r.choice([64, 128, 512, 2048])), 60
    blocks = [[(bs, 0, 0)]]
    for b in range(1, nb):
        p, toks = b * bs, []
        end = p + bs
        while p < end:
            lit = int(r.choice([0, 0, 0, 1, 3, 17, 300])) if b % 3 else 0
            lit = min(lit, end - p)
            p += lit
            m = min(int(r.randint(1, 90)), end - p, p)
            if m == 0:
                toks.append((lit, 0, 0))
                break
            toks.append((lit, m, int(r.randint(0, p - m + 1))))
            p += m
        blocks.append(toks)
    _decode_all_ways(_pack(nb * bs, bs, blocks, LITS))


@pytest.mark.parametrize("chain", [1, 2, 255, 256, 257, 700])
@pytest.mark.parametrize("width", [1, 5])
def test_in_order_chains(chain, width):
    # each match copies the match `width` tokens before it: `chain` levels
    bs = 1 << 14
    blocks = []
    for b in range(3):
        p = b * bs
        toks, ends = [(40, 0, 0)], []
        pos, lit = p + 40, 40
        toks = []
        starts = []
        for k in range(chain * width):
            ln = 7
            src = starts[k - width] if k >= width else p + (k % 8)
            toks.append((lit if k == 0 else k % 2, ln, src))
            pos = pos + (0 if k == 0 else k % 2)
            starts.append(pos)
            pos += ln
            if pos + 10 > p + bs:
                break
        toks.append((p + bs - pos, 0, 0))
        blocks.append(toks)
    c = _pack(3 * bs, bs, blocks, LITS)
    assert oracle.validate(c) == 0
    _decode_all_ways(c)


@pytest.mark.parametrize("n", [5000, 5001, 20000, 20001, 40000, 40001])
def test_levels_around_the_sizes_per_group(n):
    # levels 1 and 3 of n matches, levels 2 and 4 of a few
    bs, ln = 1 << 17, 8
    blocks, pos = [[(bs, 0, 0)]], bs
    src, readable = 0, bs  # what the wave before wrote at the start of its first block
    for cnt in (n, 40, n, 3):
        start, left = pos, cnt
        while left:
            k = min(left, bs // ln)
            toks = [(0, ln, src + (ln * i) % readable) for i in range(k)]
            if k * ln < bs:
                toks.append((bs - k * ln, 0, 0))
            blocks.append(toks)
            left -= k
            pos += bs
        src, readable = start, min(cnt, bs // ln) * ln
    c = _pack(pos, bs, blocks, LITS)
    assert oracle.validate(c) == 0
    s = torch.cuda.current_stream()
    h = aclz.aclz_upload(c, s)
    try:
        counts = aclz.aclz_wave_counts(h)
        assert counts[1:].tolist() == [n, 40, n, 3]
        assert aclz.aclz_decode_plan(h, mode=aclz.ACLZ_MODE_WAVES)[1] == 5
        assert aclz.aclz_decode_plan(h)[1] == 5
    finally:
        aclz.aclz_free(h)
    _decode_all_ways(c)


@pytest.mark.parametrize("ln", [1, 15, 16, 17, 31, 33, 176, 177, 192, 200, 208, 224, 900, 1023, 1024, 1025, 2049, 5000])
def test_match_lengths_around_the_stage(ln):
    # every source alignment, matches that leave the stage room for 16 and
    # for fewer, and matches that go into the list in pieces
    bs = 1 << 15
    blocks = [[(bs, 0, 0)]]
    for b in range(1, 5):
        toks, p = [], b * bs
        k = 0
        while p + ln + 3 <= (b + 1) * bs:
            toks.append((k % 3, ln, (b - 1) * bs + (k * 37 + b) % (bs - ln)))
            p += k % 3 + ln
            k += 1
        toks.append(((b + 1) * bs - p, 0, 0))
        blocks.append(toks)
    c = _pack(5 * bs, bs, blocks, LITS)
    assert oracle.validate(c) == 0
    _decode_all_ways(c)


@pytest.mark.parametrize("bs,width,levels,ln,lit", [
    (256, 1, 4, 16, 40), (256, 2, 3, 17, 40), (1024, 3, 5, 15, 40), (4096, 40, 6, 7, 40), (1 << 14, 255, 4, 9, 40),
    (1 << 14, 256, 4, 9, 40), (1 << 14, 257, 5, 9, 40), (1 << 14, 6, 8, 63, 40), (1 << 14, 6, 8, 64, 40),
    (1 << 14, 6, 8, 65, 40), (1 << 16, 3, 7, 1025, 40), (1 << 17, 600, 12, 13, 40), (1 << 18, 300, 6, 33, 40),
    (1 << 14, 6, 8, 63, 80), (1 << 14, 6, 8, 64, 80), (1 << 14, 6, 8, 65, 80), (1 << 14, 6, 8, 81, 90),
    (1 << 16, 3, 7, 1025, 1100), (1 << 17, 40, 5, 513, 600), (256, 2, 4, 17, 40)])
def test_in_order_levels_by_block(bs, width, levels, ln, lit):
    # levels of `width` matches of ln bytes in every other block, every source
    # alignment, matches that read the block before among them and after them
    # (they are deferred, and what reads them); a short last block
    r = np.random.RandomState(bs + width + ln)
    nb = 7
    total = nb * bs - 5
    blocks = [[(bs, 0, 0)]]
    for b in range(1, nb):
        toks, at, p, end = [], b * bs, b * bs + lit, min((b + 1) * bs, total)
        before = None
        for _ in range(levels if b % 2 else 0):
            starts = []
            for k in range(width):
                if before is not None:
                    src = before[int(r.randint(width))]
                elif ln <= lit:
                    src = at - 7 if k == 0 else at + k % (lit - ln + 1)
                else:
                    src = k % 8
                toks.append((0 if toks else lit, ln, src))
                starts.append(p)
                p += ln
            before = starts
        if b % 2 and b > 2:
            toks.append((3, 11, (b - 2) * bs + lit + 2))
            p += 14
        if not toks:
            p = at
        assert p <= end
        toks.append((end - p, 0, 0))
        blocks.append(toks)
    c = _pack(total, bs, blocks, LITS)
    assert oracle.validate(c) == 0
    _decode_all_ways(c)
    s = torch.cuda.current_stream()
    h = aclz.aclz_upload(c, s, flags=aclz.ACLZ_UPLOAD_FLATTEN)
    try:
        n = levels if levels < 4 or bs > 1 << 17 else 1
        if ln > lit or width == 1:
            n = 0  # all of them start from another block's bytes
        assert aclz.aclz_decode_plan(h, mode=aclz.ACLZ_MODE_WAVES)[1] == 1 + n + 1
    finally:
        aclz.aclz_free(h)
