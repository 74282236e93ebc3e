"""Host side of the GPU encode: the array it returns holds the container and
nothing more, and where there is no room for the largest possible container
it is asked for its size first."""
import ctypes

import numpy as np
import pytest

from paper_2607_18541_gb300 import aclz

N, BLOCK, SIZE = 1 << 20, 1 << 16, 12345


class _Fake:
    """aclz_encode_gpu of a library that writes SIZE bytes."""

    def __init__(self):
        self.caps = []

    def aclz_encode_gpu(self, src, n, params, bmm, stream, out, cap, size):
        self.caps.append(cap if out is not None else None)
        size._obj.value = SIZE
        if out is not None:
            assert cap >= SIZE
            ctypes.memset(out, 0x5A, SIZE)
        return 0


@pytest.fixture
def fake(monkeypatch):
    f = _Fake()
    bound = aclz.aclz_encode_bound(N, BLOCK)
    monkeypatch.setattr(aclz, "lib", lambda: f)
    monkeypatch.setattr(aclz, "aclz_encode_bound", lambda n, block: bound)
    f.bound = bound
    return f


def _params():
    p = aclz.aclz_encode_params()
    p.block_size = BLOCK
    return p


def test_returns_the_container_alone(fake):
    c = aclz.aclz_encode_gpu(np.zeros(N, dtype=np.uint8), _params())
    assert c.size == SIZE and c.base is None and c.nbytes == SIZE and (c == 0x5A).all()
    assert fake.caps == [fake.bound]


def test_without_room_for_the_bound(fake, monkeypatch):
    empty = np.empty

    def limited(n, **kw):
        if n > 2 * SIZE:
            raise MemoryError
        return empty(n, **kw)

    x = np.zeros(N, dtype=np.uint8)
    monkeypatch.setattr(np, "empty", limited)
    c = aclz.aclz_encode_gpu(x, _params())
    assert c.size == SIZE and (c == 0x5A).all()
    assert fake.caps == [None, SIZE]
