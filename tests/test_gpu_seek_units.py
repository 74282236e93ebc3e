"""Range decode at the edges of its units, cells and request table, on plain
and flattened handles, against slices of the oracle's decode."""
import numpy as np
import pytest

import oracle
from paper_2607_18541_gb300 import aclz, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _streams():
    sw = synth.copy_sweep((2 << 20) + 77, 1 << 13, 300, seed=5)
    yield "sweep", oracle.pack_sweep(sw, tags=False)
    yield "text_base", oracle.encode(synth.wordtext(1 << 20, seed=6), 1 << 16, oracle.PRESET_BASE)
    yield "fastq", oracle.encode(synth.fastq(1 << 20, seed=7), 1 << 12, oracle.PRESET_TUNED)
    yield "tiny_blocks", oracle.encode(synth.markov2(60_001, seed=8), 64, (4, 4, 4, 4))
    yield "random", oracle.encode(np.random.RandomState(9).randint(0, 256, 300_001).astype(np.uint8), 1 << 14,
                                  oracle.PRESET_TUNED)
    yield "constant", oracle.encode(np.zeros(70_000, dtype=np.uint8), 1 << 14, (4, 4, 4, 4))


@pytest.mark.parametrize("flags", [0, aclz.ACLZ_UPLOAD_FLATTEN])
@pytest.mark.parametrize("name,c", list(_streams()), ids=lambda v: v if isinstance(v, str) else "")
def test_ranges(name, c, flags):
    full = oracle.decode(c)
    n = full.size
    r = np.random.RandomState(3)
    lo, hi = [0, 0, n - 1, n // 2], [1, n, n, n // 2]
    for size in (1, 2, 255, 256, 257, 1023, 1024, 1025, 5000):
        for at in (0, 255, 256, 1023, int(r.randint(0, n))):
            lo.append(min(at, n))
            hi.append(min(at + size, n))
    s = torch.cuda.current_stream()
    h = aclz.aclz_upload(c, s, flags=flags)
    try:
        for a, b in zip(lo, hi):
            out = torch.full((b - a + 48,), 0xA5, dtype=torch.uint8, device="cuda")
            aclz.aclz_decode_range(h, a, b, out, stream=s)
            got = out.cpu().numpy()
            assert np.array_equal(got[:b - a], full[a:b]), (a, b)
            assert (got[b - a:] == 0xA5).all()
    finally:
        aclz.aclz_free(h)


@pytest.mark.parametrize("flags", [0, aclz.ACLZ_UPLOAD_FLATTEN])
@pytest.mark.parametrize("k", [2, 255, 256, 257, 600])
def test_request_tables(k, flags):
    c = dict(_streams())["text_base"]
    full = oracle.decode(c)
    n = full.size
    r = np.random.RandomState(k)
    size = np.exp(r.uniform(0, np.log(9000), k)).astype(np.int64) - 1
    lo = (r.rand(k) * (n - size)).astype(np.int64)
    off = np.concatenate([[0], np.cumsum((size + 31) // 16 * 16)]).astype(np.int64)
    s = torch.cuda.current_stream()
    h = aclz.aclz_upload(c, s, flags=flags)
    try:
        for asynchronous in (False, True):
            out = torch.full((int(off[-1]),), 0xA5, dtype=torch.uint8, device="cuda")
            ptr = [int(out.data_ptr() + o) for o in off[:-1]]
            if asynchronous:
                table = torch.zeros(32 * k, dtype=torch.uint8).pin_memory()
                t = table.numpy().view(np.uint64).reshape(k, 4)
                t[:, 0], t[:, 1], t[:, 2] = lo, lo + size, ptr
                aclz.aclz_decode_ranges_async(h, k, table.data_ptr(), s)
            else:
                scratch = torch.empty(aclz.aclz_ranges_scratch_bytes(k), dtype=torch.uint8, device="cuda")
                aclz.aclz_decode_ranges(h, lo, lo + size, ptr, scratch, stream=s)
            assert aclz.aclz_device_status(h, s) == 0
            got = out.cpu().numpy()
            for i in range(k):
                o, m = int(off[i]), int(size[i])
                assert np.array_equal(got[o:o + m], full[lo[i]:lo[i] + m]), i
                assert (got[o + m:int(off[i + 1])] == 0xA5).all()
    finally:
        aclz.aclz_free(h)
