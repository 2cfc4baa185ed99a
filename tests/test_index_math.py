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
void unit_of_u(int dup, int halves, int depth, int u, int* out) {
  const spec::UnitsOfU x{dup != 0, halves, depth};
  out[0] = x.tile(u);
  out[1] = x.m(u);
  out[2] = x.stage(u);
  out[3] = (int)x.parity(u);
}
int unit_drains(int dup, int halves, int depth, int u, int issued) {
  return spec::UnitsOfU{dup != 0, halves, depth}.drains(u, issued);
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


@pytest.mark.parametrize("dup", [True, False])
@pytest.mark.parametrize("depth", [1, 2, 3])
def test_units_of_u_wait_on_the_last_phase_of_a_stage(lib, dup, depth):
    """A stage's barrier completes one phase a unit, and a parity wait sees only
    the last one: the producer's waits must each be for a stage's last unit
    (an earlier one would never be seen), and all of them for every stage in
    use.  Units before the ring wraps have parity 0, and tiles go to the two
    epilogue groups in turn."""
    halves = 2
    unit = (ctypes.c_int * 4)()
    for issued in range(0, 12 * halves * depth + 3):
        phases, waits = {}, []
        for u in range(issued):
            lib.unit_of_u(int(dup), halves, depth, u, unit)
            tile, m, stage, parity = unit
            assert tile == (u if dup else u // 2) and stage % halves == tile % halves
            assert parity == phases.get(stage, 0) % 2 and 0 <= stage < halves * depth
            phases[stage] = phases.get(stage, 0) + 1
            if lib.unit_drains(int(dup), halves, depth, u, issued):
                waits.append((stage, parity))
        assert sorted(s for s, _ in waits) == sorted(phases)
        assert all(parity == (phases[stage] - 1) % 2 for stage, parity in waits)
