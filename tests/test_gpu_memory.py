"""Uploads and flattening with little device memory left: an upload that does not fit
reports it, one that fits without the level list decodes by waves and the
walk, and every upload that succeeds decodes to the input."""
import pytest

import oracle
from paper_2607_18541_gb300 import aclz, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MIB = 1 << 20


def _fill(left):
    """All device memory but about `left` MiB."""
    torch.cuda.empty_cache()
    for spare in (0, 64, 256, 1024):
        free, _ = torch.cuda.mem_get_info()
        try:
            return torch.empty(max(1, free - (left + spare) * MIB), dtype=torch.uint8, device="cuda")
        except torch.OutOfMemoryError:
            torch.cuda.empty_cache()
    raise AssertionError("no allocation near the free memory succeeds")


def test_upload_as_memory_runs_out():
    # 20 million matches in some 40 levels; the library keeps up to 512 MiB of
    # what it freed, which an upload uses first
    sw = synth.copy_sweep(384 * MIB, 32 << 10, 16, seed=11)
    c = aclz.aclz_pack(sw.total, sw.block_size, (4, 4, 4, 4), sw.blk_ntok, sw.lit_len, sw.match_len, sw.src, sw.literals)
    s = torch.cuda.current_stream()
    want = torch.from_numpy(oracle.decode(c)).cuda()
    out = torch.empty(sw.total, dtype=torch.uint8, device="cuda")
    h = aclz.aclz_upload(c, s)
    full = aclz.aclz_decode_plan(h)
    waves = aclz.aclz_handle_info(h).n_waves
    aclz.aclz_free(h)
    walked, refused = 0, 0
    for left in range(128, 2900, 128):
        fill = _fill(left)
        try:
            h = aclz.aclz_upload(c, s)
        except aclz.AclzError as e:
            assert e.code == aclz.ACLZ_E_NOMEM
            refused += 1
            continue
        finally:
            del fill
        try:
            plan = aclz.aclz_decode_plan(h)
            if plan != full:
                # the walk, then a launch for every wave
                assert plan[1] == 2 + waves - 1
                walked += 1
            out.zero_()
            aclz.aclz_decode_all(h, out, stream=s)
            assert aclz.aclz_device_status(h, s) == 0
            assert torch.equal(out, want)
        finally:
            aclz.aclz_free(h)
    assert walked and refused, (walked, refused)
    assert plan == full  # enough memory at the end


def test_flatten_as_memory_runs_out():
    # however far a flattening comes, the handle decodes in every mode after
    # it, and flattens once there is memory
    sw = synth.copy_sweep(128 * MIB, 32 << 10, 16, seed=12)
    c = aclz.aclz_pack(sw.total, sw.block_size, (4, 4, 4, 4), sw.blk_ntok, sw.lit_len, sw.match_len, sw.src, sw.literals)
    s = torch.cuda.current_stream()
    want = torch.from_numpy(oracle.decode(c)).cuda()
    out = torch.empty(sw.total, dtype=torch.uint8, device="cuda")
    refused = 0
    for left in range(128, 1000, 48):
        h = aclz.aclz_upload(c, s)
        try:
            fill = _fill(left)
            try:
                aclz.aclz_flatten(h, s)
                ok = True
            except aclz.AclzError as e:
                assert e.code == aclz.ACLZ_E_NOMEM
                refused += 1
                ok = False
            del fill
            for mode, flags in ((aclz.ACLZ_MODE_AUTO, 0), (aclz.ACLZ_MODE_WAVES, 0), (aclz.ACLZ_MODE_PERSISTENT, 0),
                                (aclz.ACLZ_MODE_PERSISTENT, aclz.ACLZ_FLAG_STAGED)):
                out.zero_()
                aclz.aclz_decode_all(h, out, mode=mode, flags=flags, stream=s)
                assert aclz.aclz_device_status(h, s) == 0
                assert torch.equal(out, want), (left, ok, mode, flags)
            if not ok:
                torch.cuda.empty_cache()
                aclz.aclz_flatten(h, s)
                assert aclz.aclz_handle_info(h).n_waves == 2
                out.zero_()
                aclz.aclz_decode_all(h, out, stream=s)
                assert torch.equal(out, want)
        finally:
            aclz.aclz_free(h)
    assert refused
