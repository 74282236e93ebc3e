"""The schedule ACLZ_MODE_AUTO takes where the upload found no dependency
levels, and where an event goes between the phases."""
import numpy as np
import pytest

import oracle
from paper_2607_18541_gb300 import aclz, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _deep(nb, bs, L):
    """Every block a copy of the one before, in matches of L bytes."""
    r = np.random.RandomState(L)
    per = bs // L
    ll, ml, sr, nt = [bs], [0], [0], [1]
    for b in range(1, nb):
        for k in range(per):
            one = 1 if k == 0 else 0  # a literal, so that blocks differ
            ll.append(one), ml.append(L - one), sr.append((b - 1) * bs + k * L)
        nt.append(per)
    ll = np.array(ll, dtype=np.uint32)
    return aclz.aclz_pack(nb * bs, bs, (4, 4, 4, 4), np.array(nt, dtype=np.uint32), ll, np.array(ml, dtype=np.uint32),
                          np.array(sr, dtype=np.uint64), r.randint(0, 256, int(ll.sum())).astype(np.uint8))


@pytest.mark.parametrize("L,persistent", [(64, False), (128, False), (256, True), (1024, True)])
def test_chains_deeper_than_the_levels(L, persistent):
    # 600 levels: by waves up to 192 bytes a match, by ranges from there on
    c = _deep(600, 4096, L)
    exp = oracle.decode(c)
    s = torch.cuda.current_stream()
    h = aclz.aclz_upload(c, s)
    try:
        assert aclz.aclz_handle_info(h).n_waves == 600
        plan, n = aclz.aclz_decode_plan(h)
        if persistent:
            assert plan["mode"] == aclz.ACLZ_MODE_PERSISTENT and plan["flags"] == aclz.ACLZ_FLAG_STAGED and n == 2
        else:
            assert plan["mode"] == aclz.ACLZ_MODE_WAVES and n == 600
        # the container with its tags: the same, without passes for levels
        t = aclz.aclz_upload(aclz.aclz_export(h), s)
        assert aclz.aclz_decode_plan(t) == (plan, n)
        assert np.array_equal(aclz.aclz_tags(t), aclz.aclz_tags(h))
        aclz.aclz_free(t)
        for G in (32, 16, 8):
            out = torch.zeros(exp.size, dtype=torch.uint8, device="cuda")
            aclz.aclz_decode_all(h, out, G=G, stream=s)
            assert aclz.aclz_device_status(h, s) == 0
            assert np.array_equal(out.cpu().numpy(), exp)
    finally:
        aclz.aclz_free(h)


@pytest.mark.parametrize("L", [100, 192, 500, 1100])
def test_event_between_the_phases(L):
    # with levels the event takes AUTO to the schedule of streams without them
    sw = synth.copy_sweep(4 << 20, 1 << 15, L, seed=L)
    c = aclz.aclz_pack(sw.total, sw.block_size, (4, 4, 4, 4), sw.blk_ntok, sw.lit_len, sw.match_len, sw.src, sw.literals)
    exp = oracle.decode(c)
    s = torch.cuda.current_stream()
    h = aclz.aclz_upload(c, s)
    try:
        plan, _ = aclz.aclz_decode_plan(h)
        assert plan["mode"] == (aclz.ACLZ_MODE_PERSISTENT if L >= 1024 else aclz.ACLZ_MODE_WAVES)
        for G in (32, 16, 8):
            out = torch.zeros(exp.size, dtype=torch.uint8, device="cuda")
            a, m, b = (torch.cuda.Event(enable_timing=True) for _ in range(3))
            m.record(s)
            a.record(s)
            aclz.aclz_decode_all_ev(h, out, m, G=G, stream=s)
            b.record(s)
            b.synchronize()
            assert aclz.aclz_device_status(h, s) == 0
            assert a.elapsed_time(m) >= 0 and m.elapsed_time(b) > 0
            assert np.array_equal(out.cpu().numpy(), exp)
    finally:
        aclz.aclz_free(h)
