"""Streams whose matches read the ones just before them (runs, short
periods) and in-order chains of more levels than are listed: the in-order
matches are walked block by block in one launch, in every mode, and the
bytes are the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2607_18541_gb300 import aclz

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
