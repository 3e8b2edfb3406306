"""The filtered phase's shares of a graph's unsampled chunks (cc_chunks.h): every
chunk of a segment goes to exactly one warp, and no warp gets more than one
chunk more than another. Plain integer code, compiled for the host.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2507_03695_gb300 import build

SOURCE = """
#include "cc_chunks.h"
extern "C" unsigned share(unsigned c0, unsigned c1, unsigned stride, unsigned w, unsigned nw, unsigned *out) {
  unsigned n = 0;
  for (cc::UnsampledChunks mine(c0, stride, w, nw); mine.chunk() < c1; mine.next()) out[n++] = mine.chunk();
  return n;
}
"""


@pytest.fixture(scope="module")
def share(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no compiler")
    d = tmp_path_factory.mktemp("chunks")
    (d / "share.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", build.CSRC, str(d / "share.cpp"), "-o",
                    str(d / "share.so")], check=True)
    f = ctypes.CDLL(os.fspath(d / "share.so")).share

    def call(c0, c1, stride, w, nw):
        out = (ctypes.c_uint * (c1 - c0 + 1))()
        return list(out[:f(c0, c1, stride, w, nw, out)])
    return call


@pytest.mark.parametrize("stride", [2, 3, 4, 5, 7, 8, 15, 16, 17, 33, 63, 64])
@pytest.mark.parametrize("nw", [8, 16])
def test_every_warp_has_its_share(share, stride, nw):
    for c0, c1 in ((0, 1), (0, 2), (0, 64), (1, 64), (63, 130), (64, 1000), (127, 128), (4096, 4096 + 37)):
        parts = [share(c0, c1, stride, w, nw) for w in range(nw)]
        assert sorted(sum(parts, [])) == [c for c in range(c0, c1) if c % stride]
        assert max(map(len, parts)) - min(map(len, parts)) <= 1


def test_large_chunk_numbers(share):
    c0 = 1 << 30
    parts = [share(c0, c0 + 500, 2, w, 16) for w in range(16)]
    assert sorted(sum(parts, [])) == [c for c in range(c0, c0 + 500) if c % 2]
