"""The autotuner times what the chosen schedule reads: resident CTAs and range
sizes only for streams that decode in the persistent launch."""
from types import SimpleNamespace

import pytest

from paper_2607_18541_gb300 import aclz, autotune

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mode", [aclz.ACLZ_MODE_WAVES, aclz.ACLZ_MODE_PERSISTENT])
def test_parameters_that_are_read(monkeypatch, mode):
    timed = []
    monkeypatch.setattr(aclz, "aclz_upload", lambda c, st: 1)
    monkeypatch.setattr(aclz, "aclz_free", lambda h: None)
    monkeypatch.setattr(aclz, "aclz_handle_info", lambda h: SimpleNamespace(total_len=1000, n_blocks=4))
    monkeypatch.setattr(aclz, "aclz_set_range_bytes", lambda h, rb, st: None)
    monkeypatch.setattr(aclz, "aclz_decode_plan", lambda h, **kw: ({"mode": mode}, 2))
    monkeypatch.setattr(torch, "empty", lambda n, **kw: SimpleNamespace(numel=lambda: n))

    def measure(h, out, reps, stream, **cfg):
        timed.append(cfg)
        return 1.0 + 0.1 * len(timed)

    monkeypatch.setattr(autotune, "measure", measure)
    r = autotune.tune(lambda bs: b"", 1000, block_sizes=(8192,), Gs=(32,), ctas=(0, 2), range_bytes=(8192, 20480),
                      stream=object())
    assert len(r["trials"]) == len(timed) == (4 if mode == aclz.ACLZ_MODE_PERSISTENT else 1)
    assert r["best"] == r["trials"][0] and r["best"]["block_size"] == 8192
