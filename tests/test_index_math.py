"""Index arithmetic of the kernels, compiled for the host (csrc/index_math.h)
and checked without a GPU."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_25852_gb300", "csrc")
SOURCE = r"""
#include "index_math.h"
extern "C" {
int stream_wave() { return spec::kStreamWave; }
void stream_prefetch(int packed, int has_depth, int block, int i, int j, int c, int B, int K, long long V,
                     long long chunk, long long per_cta, long long* out) {
  const spec::PrefetchSpan s =
      spec::stream_prefetch(packed, has_depth, block, i, j, c, B, K, V, chunk, per_cta);
  out[0] = s.first;
  out[1] = s.end;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("index_math")
    src, out = d / "index_math.cpp", d / "index_math.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(out)], check=True)
    return ctypes.CDLL(str(out))


@pytest.mark.parametrize("B,K,V,chunk", [(3, 2, 5000, 5000), (64, 16, 201088, 212992), (16, 16, 128256, 65536),
                                         (5, 4, 40000, 16384)])
@pytest.mark.parametrize("packed,has_depth", [(False, False), (False, True), (True, True), (True, False)])
def test_prefetched_entries_are_kept_rows(lib, B, K, V, chunk, packed, has_depth):
    """Before the depths are known only rows that every depth keeps are
    fetched: row 0 of each request, or any row of a call without depths.  In
    the packed layout, B of them whatever the depths are, and only by CTAs
    that can run ahead of the grid wait."""
    LL = ctypes.c_longlong
    per, nc = 256 * 64, -(-V // chunk)
    wave = lib.stream_wave()
    span = (LL * 2)()
    for block in range(B * (K + 1) * nc):
        i, rem = divmod(block, (K + 1) * nc)
        j, c = divmod(rem, nc)
        lib.stream_prefetch(packed, has_depth, block, i, j, c, B, K, LL(V), LL(chunk), LL(per), span)
        first, end = span[0], min(span[1], span[0] + per)
        if packed:
            assert first >= end or (block < wave and 0 <= first and end <= B * V)
            assert block >= min(wave, B * V // per) or end - first == per  # the wave's part is fetched
        elif has_depth and j > 0:
            assert first >= end  # a shallower request drops the row
        else:
            row = (i * (K + 1) + j) * V
            assert first == row + c * chunk and end == min(row + V, row + (c + 1) * chunk, first + per)
