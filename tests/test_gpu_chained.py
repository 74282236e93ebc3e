"""Streams whose matches read the ones just before them (runs, short
periods) and in-order chains of more levels than are listed: the in-order
matches are walked block by block in one launch, in every mode, and the
bytes are the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2607_18541_gb300 import aclz, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WAVES, PERSISTENT, AUTO = aclz.ACLZ_MODE_WAVES, aclz.ACLZ_MODE_PERSISTENT, aclz.ACLZ_MODE_AUTO


def _encode(x, block, mm=(4, 4, 4, 4)):
    p = aclz.aclz_encode_params_default(aclz.ACLZ_PRESET_BASE)
    for i in range(4):
        p.min_match[i] = mm[i]
    p.block_size = block
    return aclz.aclz_encode(x, p)


def _chains(nb, bs, ln, width, short=0):
    """Every block: `width` chains of matches of ln bytes side by side, each
    match reading the one `width` before it; the last block `short` bytes less."""
    r = np.random.RandomState(bs + ln + width)
    ll, ml, sr, nt = [], [], [], []
    for b in range(nb):
        size = bs - (short if b == nb - 1 else 0)
        per = (size - ln * width) // ln
        for k in range(per):
            ll.append(ln * width if k == 0 else 0)
            ml.append(ln)
            sr.append(b * bs + k * ln)
        nt.append(per + 1)
        ll.append(size - ln * width - per * ln)
        ml.append(0)
        sr.append(0)
    ll = np.array(ll, dtype=np.uint32)
    lits = r.randint(0, 256, int(ll.sum())).astype(np.uint8)
    return aclz.aclz_pack(nb * bs - short, bs, (4, 4, 4, 4), np.array(nt, dtype=np.uint32), ll,
                          np.array(ml, dtype=np.uint32), np.array(sr, dtype=np.uint64), lits)


def _decode_all_ways(c, order):
    """order: kernels that copy in-order matches of the plain, of the
    flattened handle."""
    exp = oracle.decode(c)
    s = torch.cuda.current_stream()
    for flags, tagged in ((0, False), (0, True), (aclz.ACLZ_UPLOAD_FLATTEN, False)):
        src = c
        if tagged:
            h = aclz.aclz_upload(c, s)
            src = aclz.aclz_export(h)
            aclz.aclz_free(h)
        h = aclz.aclz_upload(src, s, flags=flags)
        try:
            n = order[1 if flags else 0]
            waves = aclz.aclz_handle_info(h).n_waves
            if n is not None:
                assert aclz.aclz_decode_plan(h, mode=WAVES)[1] == 1 + n + (waves - 1)
                assert aclz.aclz_decode_plan(h)[1] <= 1 + n + (waves - 1)
                assert aclz.aclz_decode_plan(h, mode=PERSISTENT)[1] == 1 + n + (waves > 1)
            for G in (32, 16, 8):
                for mode, fl in ((AUTO, 0), (WAVES, 0), (PERSISTENT, 0), (PERSISTENT, aclz.ACLZ_FLAG_STAGED),
                                 (PERSISTENT, aclz.ACLZ_FLAG_REGISTERS)):
                    out = torch.full((exp.size + 32,), 0xA5, dtype=torch.uint8, device="cuda")
                    aclz.aclz_decode_all(h, out, cap=exp.size, G=G, mode=mode, flags=fl, stream=s)
                    assert aclz.aclz_device_status(h, s) == 0
                    got = out.cpu().numpy()
                    assert np.array_equal(got[:exp.size], exp), (flags, tagged, G, mode, fl)
                    assert (got[exp.size:] == 0xA5).all()
        finally:
            aclz.aclz_free(h)


@pytest.mark.parametrize("n,block", [(8 << 10, 16 << 10), (24 << 10, 16 << 10), (33 << 10, 32 << 10),
                                     (300000, 16 << 10), (1 << 20, 1 << 20), ((1 << 20) + 777, 1 << 19), (5000, 64)])
def test_runs(n, block):
    # blocks of 64 bytes hold two matches at most: nothing to tell them by
    order = (None, None) if block == 64 else (1, 1)
    _decode_all_ways(_encode(np.zeros(n, dtype=np.uint8), block), order)
    x = np.tile(np.frombuffer(b"abcdefg", dtype=np.uint8), n // 7 + 1)[:n]
    _decode_all_ways(_encode(x, block), (None, None))


@pytest.mark.parametrize("nb,bs,ln,width,short", [(3, 4096, 5, 1, 0), (5, 4096, 31, 1, 100), (40, 16384, 20, 1, 3),
                                                  (2, 1 << 18, 17, 1, 9), (1, 1 << 20, 16, 1, 0)])
def test_chains_of_neighbours(nb, bs, ln, width, short):
    _decode_all_ways(_chains(nb, bs, ln, width, short), (1, 1))


@pytest.mark.parametrize("nb,bs,ln,width", [(1, 1 << 18, 16, 8), (3, 1 << 18, 23, 9), (2, 1 << 19, 16, 20)])
def test_more_levels_than_are_listed(nb, bs, ln, width):
    # 1137 to 2047 levels, no match near the one it reads
    _decode_all_ways(_chains(nb, bs, ln, width), (1, 1))


@pytest.mark.parametrize("top", [17, 40, 300, 1100])
@pytest.mark.parametrize("cross", [False, True])
def test_chain_of_all_lengths(top, cross):
    # one match after another, each reading bytes of the one before it (or,
    # across, of the block before and then of the one before it): every length
    # up to `top`, at every alignment of source and output
    r = np.random.RandomState(top)
    bs, nb, lit0 = 1 << 15, 3, top + 64
    ll, ml, sr, nt = [], [], [], []
    for b in range(nb):
        at, end = b * bs, (b + 1) * bs
        p, toks = at + lit0, 0
        if cross and b:
            ll.append(0), ml.append(lit0), sr.append(at - lit0 - 3)
            toks = 1
        while p + 2 * top <= end:
            n = int(r.randint(1, top + 1)) if toks % 3 else top
            ll.append(lit0 if toks == 0 else 0), ml.append(n), sr.append(p - n - int(r.randint(0, 20)))
            p += n
            toks += 1
        ll.append(end - p), ml.append(0), sr.append(0)
        nt.append(toks + 1)
    ll = np.array(ll, dtype=np.uint32)
    c = aclz.aclz_pack(nb * bs, bs, (4, 4, 4, 4), np.array(nt, dtype=np.uint32), ll, np.array(ml, dtype=np.uint32),
                       np.array(sr, dtype=np.uint64), r.randint(0, 256, int(ll.sum())).astype(np.uint8))
    assert oracle.validate(c) == 0
    _decode_all_ways(c, (None, None))


@pytest.mark.parametrize("nb,bs,ln,width", [(9, 4096, 20, 8), (300, 16384, 20, 8), (4, 1 << 16, 16, 64), (5, 1024, 16, 12)])
def test_in_order_levels_without_deferred_matches(nb, bs, ln, width):
    # 4 to 102 levels: by block in one launch, in the plain handle too
    _decode_all_ways(_chains(nb, bs, ln, width, 5), (1, 1))


def _narrow(runs, seed):
    """Levels of the given numbers of matches, each match reading one of the
    level before: in-order chains in blocks of their own and, from block to
    block, deferred ones.  Many literal blocks with far matches go first, so
    that most matches are not near what they read."""
    r = np.random.RandomState(seed)
    bs, blocks, lits = 1 << 12, [[(1 << 12, 0, 0)]], 0
    for _ in range(12):
        at = len(blocks) * bs
        blocks.append([(8, 8, int(r.randint(0, bs - 8))) for _ in range(bs // 16)])
    prev = [(0, bs)]  # (place, bytes) of what the next level may read
    for w in runs:
        place, toks, here = len(blocks) * bs, [], []
        for k in range(w):
            n = int(r.choice([1 if k else 9, 7, 16, 33, 64, 130]))
            a, m = prev[int(r.randint(len(prev)))]
            n = min(n, m)
            p = place + sum(t[0] + t[1] for t in toks)
            if p + n + 8 > place + bs:
                break
            toks.append((int(r.randint(0, 3)), n, a + int(r.randint(0, m - n + 1))))
            here.append((p + toks[-1][0], n))
        toks.append((place + bs - place - sum(t[0] + t[1] for t in toks), 0, 0))
        blocks.append(toks)
        prev = [x for x in here if x[1] > 6]
    ll = np.array([t[0] for b in blocks for t in b], dtype=np.uint32)
    ml = np.array([t[1] for b in blocks for t in b], dtype=np.uint32)
    sr = np.array([t[2] for b in blocks for t in b], dtype=np.uint64)
    return aclz.aclz_pack(len(blocks) * bs, bs, (4, 4, 4, 4), np.array([len(b) for b in blocks], dtype=np.uint32), ll, ml,
                          sr, r.randint(0, 256, int(ll.sum())).astype(np.uint8))


@pytest.mark.parametrize("seed,runs", [(1, [1] * 7), (2, [1] * 8), (3, [1, 2, 3, 64, 64, 1, 63, 5, 40, 17]),
                                       (4, [65] * 3 + [1] * 40 + [70] * 2 + [33] * 9 + [66] + [16] * 7)])
def test_runs_of_narrow_levels(seed, runs):
    c = _narrow(runs, seed)
    assert oracle.validate(c) == 0
    _decode_all_ways(c, (None, None))


def test_launches_of_a_narrow_run():
    # a run of zeros in text: hundreds of levels of a match or two
    x = synth.wordtext(1 << 20, seed=3)
    x[300000:300000 + (20 << 10)] = 0
    c = _encode(x, 16 << 10, (6, 8, 10, 12))
    h = aclz.aclz_upload(c, torch.cuda.current_stream())
    try:
        assert 2 < aclz.aclz_decode_plan(h)[1] < 130
        assert aclz.aclz_decode_plan(h, mode=WAVES)[1] < 200
    finally:
        aclz.aclz_free(h)
    _decode_all_ways(c, (None, None))


def test_staged_launch_with_mostly_narrow_levels():
    # it goes by ranges, after the in-order levels in launches of their own
    x = synth.fastq(4 << 20, seed=3)
    x[300000:300000 + (20 << 10)] = 0
    c = _encode(x, 16 << 10, (12, 16, 24, 32))
    h = aclz.aclz_upload(c, torch.cuda.current_stream())
    try:
        assert aclz.aclz_decode_plan(h, mode=PERSISTENT, flags=aclz.ACLZ_FLAG_STAGED)[1] > 2
    finally:
        aclz.aclz_free(h)
    _decode_all_ways(c, (None, None))


@pytest.mark.parametrize("width", [1, 2, 3, 4, 33])
@pytest.mark.parametrize("ln", [15, 16, 17, 47, 64, 65])
def test_few_matches_of_a_level_by_block(width, ln):
    # levels of `width` matches in a block held in shared memory, one warp's
    # matches or several warps', short and longer ones among them; a match
    # reads two levels back, so that most are not near what they read
    r = np.random.RandomState(width + ln)
    bs, nb = 1 << 14, 4
    lit0 = 3 * ln * width + 40
    ll, ml, sr, nt = [], [], [], []
    for b in range(nb):
        at = b * bs
        p, k = at + lit0, 0
        while p + 200 < at + bs:
            n = ln if k % 3 else int(r.randint(1, ln + 1))
            back = ln * (width + 1) + int(r.randint(0, ln))
            ll.append(lit0 if k == 0 else 0), ml.append(n), sr.append(p - back - n)
            p += n
            k += 1
        ll.append(at + bs - p), ml.append(0), sr.append(0)
        nt.append(k + 1)
    ll = np.array(ll, dtype=np.uint32)
    c = aclz.aclz_pack(nb * bs, bs, (4, 4, 4, 4), np.array(nt, dtype=np.uint32), ll, np.array(ml, dtype=np.uint32),
                       np.array(sr, dtype=np.uint64), r.randint(0, 256, int(ll.sum())).astype(np.uint8))
    assert oracle.validate(c) == 0
    _decode_all_ways(c, (1, 1))
