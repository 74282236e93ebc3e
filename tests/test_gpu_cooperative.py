"""Uploads where the cooperative launch of the relaxation passes is refused
as too large: with fewer CTAs, or by the passes and the ordered pass that
need none.  The refusal is a fake: the library's upload is compiled once
more with a launch call that answers like a device with room for so many
CTAs."""
import os
import subprocess
import sys

import pytest

from paper_2607_18541_gb300 import build

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <cstdio>
#include <cstdlib>
#include <cuda_runtime.h>
static cudaError_t launch_with_room(const void *f, dim3 g, dim3 b, void **a, size_t s, cudaStream_t st) {
    std::fprintf(stderr, "cooperative %u\n", g.x);
    if (g.x > (unsigned)std::atoi(std::getenv("ROOM"))) return cudaErrorCooperativeLaunchTooLarge;
    return cudaLaunchCooperativeKernel(f, g, b, a, s, st);
}
#define cudaLaunchCooperativeKernel launch_with_room
"""

RUN = r"""
import sys
import numpy as np, torch
sys.path.insert(0, sys.argv[2])
import oracle
from paper_2607_18541_gb300 import aclz, synth
aclz.LIB_PATH = sys.argv[1]
s = torch.cuda.current_stream()
for x, mm, block in ((synth.markov2(1 << 18, seed=2), (6, 8, 10, 12), 1 << 14),
                     (synth.wordtext(1 << 22, seed=2), (6, 8, 10, 12), 1 << 14)):
    p = aclz.aclz_encode_params_default(0)
    for i in range(4):
        p.min_match[i] = mm[i]
    p.block_size = block
    c = aclz.aclz_encode(x, p)
    tags = oracle.min_tags(c)
    tags = tags[0] if isinstance(tags, tuple) else tags
    for _ in range(2):
        h = aclz.aclz_upload(c, s)
        assert np.array_equal(aclz.aclz_tags(h), tags)
        out = torch.zeros(x.size + 16, dtype=torch.uint8, device="cuda")
        for mode in (2, 0, 1):
            out.zero_()
            aclz.aclz_decode_all(h, out, cap=x.size, mode=mode, stream=s)
            assert aclz.aclz_device_status(h, s) == 0
            assert np.array_equal(out[:x.size].cpu().numpy(), x)
        c = aclz.aclz_export(h)  # once more with its tags
        aclz.aclz_free(h)
print("done")
"""


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    d = tmp_path_factory.mktemp("cooperative")
    (d / "fake.h").write_text(FAKE)
    build.build()
    obj, so = str(d / "aclz_index.o"), str(d / "libaclz_fake.so")
    src = os.path.join(build.CSRC, "aclz_index.cu")
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-include", str(d / "fake.h"), "-c", src, "-o", obj],
                   check=True, capture_output=True)
    others = [os.path.join(build.BUILD, os.path.basename(s) + ".o") for s in build.sources() if s != src]
    subprocess.run([build._nvcc(), *build.ARCH, "-shared", "-o", so, obj, *others, "-lpthread"], check=True,
                   capture_output=True)
    return so


@pytest.mark.parametrize("room", [0, 100, 200, 1000])
def test_upload_with_room_for_fewer_ctas(library, room):
    r = subprocess.run([sys.executable, "-c", RUN, library, ROOT], capture_output=True, text=True, timeout=300,
                       env={**os.environ, "ROOM": str(room)})
    assert r.returncode == 0 and "done" in r.stdout, r.stderr[-2000:]
    assert "cooperative" in r.stderr
