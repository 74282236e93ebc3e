"""Minimal wave tags of streams whose chains are deeper than the relaxation
passes: chains inside blocks (settled by passes over blocks), chains from
block to block and short streams (the ordered pass)."""
import numpy as np
import pytest

import oracle
from paper_2607_18541_gb300 import aclz

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _stream(nb, bs, ln, width, cross):
    """Blocks of `width` chains of matches of ln bytes; the first matches of
    every `cross`-th block read the block before."""
    r = np.random.RandomState(nb + bs + width)
    ll, ml, sr, nt = [], [], [], []
    for b in range(nb):
        at, far = b * bs, b > 0 and b % cross == 0
        per = bs // ln - width if not far else bs // ln
        for k in range(per):
            ll.append(ln * width if k == 0 and not far else 0)
            ml.append(ln)
            sr.append(at - ln * (width - k) - 5 if far and k < width else at + (k - (width if far else 0)) * ln)
        left = bs - per * ln - (0 if far else ln * width)
        if left:
            ll.append(left), ml.append(0), sr.append(0)
        nt.append(per + (1 if left else 0))
    ll = np.array(ll, dtype=np.uint32)
    return aclz.aclz_pack(nb * bs, bs, (4, 4, 4, 4), np.array(nt, dtype=np.uint32), ll, np.array(ml, dtype=np.uint32),
                          np.array(sr, dtype=np.uint64), r.randint(0, 256, int(ll.sum())).astype(np.uint8))


@pytest.mark.parametrize("nb,bs,ln,width,cross", [(20, 1 << 17, 16, 8, 1), (40, 1 << 16, 15, 3, 2), (9, 1 << 18, 13, 20, 3),
                                                  (700, 2048, 64, 2, 1), (12, 1 << 14, 20, 2, 1)])
def test_tags_and_bytes(nb, bs, ln, width, cross):
    c = _stream(nb, bs, ln, width, cross)
    assert oracle.validate(c) == 0
    tags = oracle.min_tags(c)
    exp = oracle.decode(c)
    s = torch.cuda.current_stream()
    h = aclz.aclz_upload(c, s)
    try:
        got = aclz.aclz_tags(h)
        assert np.array_equal(got, tags[0] if isinstance(tags, tuple) else tags)
        out = torch.zeros(exp.size, dtype=torch.uint8, device="cuda")
        for mode in (aclz.ACLZ_MODE_AUTO, aclz.ACLZ_MODE_WAVES, aclz.ACLZ_MODE_PERSISTENT):
            out.zero_()
            aclz.aclz_decode_all(h, out, mode=mode, stream=s)
            assert aclz.aclz_device_status(h, s) == 0
            assert np.array_equal(out.cpu().numpy(), exp)
    finally:
        aclz.aclz_free(h)
