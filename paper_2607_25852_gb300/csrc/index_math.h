// index_math.h -- index arithmetic of the kernels that a plain host compiler
// takes too (nothing here needs CUDA), so that it is checked without a GPU.
#pragma once

#ifdef __CUDACC__
#define SPEC_HD __host__ __device__ __forceinline__
#else
#define SPEC_HD inline
#endif

namespace spec {

// CTAs of the streaming pass that are resident at once: four per SM, 152 SMs.
constexpr int kStreamWave = 152 * 4;

// The part of the logits that a streaming CTA prefetches before its grid wait:
// one line a thread from entry `first`, below `end` (nothing if first >= end).
struct PrefetchSpan {
  long long first, end;
};

// CTA `block` works on entries [c * chunk, (c + 1) * chunk) of row j of request
// i; `per_cta` entries are a line for each of its threads.  The depths are not
// known yet, so only rows that every depth keeps are fetched:
//   without row offsets the CTA's own first load round, unless the call gives
//   depths and the row is not its request's row 0.  A dropped row's round is
//   read by nothing (33 MB at B=64, K=16, V=201088, all depths 0), and over the
//   CPU-GPU link it is not free: pinned logits, B=64, K=16, V=50048, depths 0,
//   80.6 us a call with every row fetched, 74.2 so, 76.6 without any prefetch.
//   In device memory the rows that are kept start later for it: B=64, K=16,
//   V=201088, depths uniform in 0..16, one chunk a row 45.4 -> 47.5 us (50.8
//   before there was a prefetch, with four chunks).
//   With row offsets rows 0 .. B-1 in order, which every packing holds, by the
//   CTAs of the first wave.  Later CTAs start when others have ended, past the
//   grid wait, and would fetch again what the stream has passed: B=256, K=3,
//   V=128256, every row kept, 64.8 us a call with every CTA fetching, 63.2 so.
SPEC_HD PrefetchSpan stream_prefetch(bool packed, bool has_depth, int block, int i, int j, int c, int B, int K,
                                     long long V, long long chunk, long long per_cta) {
  PrefetchSpan s;
  if (packed) {
    const long long wave = kStreamWave * per_cta;
    s.first = block * per_cta;
    s.end = B * V < wave ? B * V : wave;
  } else {
    const long long row = ((long long)i * (K + 1) + j) * V, last = (c + 1) * chunk;
    s.first = row + c * chunk;
    s.end = has_depth && j > 0 ? 0 : row + (V < last ? V : last);
  }
  return s;
}

// The units of U that the Markov head's U producer loads, in its order of issue
// u = 0, 1, ..: a tile's 64 rows x 128 columns when the operand's rows are
// repeated (dup), else one 64-column half of a tile, the halves in turn.  Tile t
// belongs to epilogue group t % halves; unit m of a group uses one of the group's
// `depth` stages in turn, so that a stage's phases are seen one after another.
struct UnitsOfU {
  bool dup;
  int halves, depth;
  SPEC_HD int per_tile() const { return dup ? 1 : 2; }
  SPEC_HD int tile(int u) const { return dup ? u : u >> 1; }
  SPEC_HD int m(int u) const { return tile(u) / halves * per_tile() + (dup ? 0 : (u & 1)); }
  SPEC_HD int stage(int u) const { return tile(u) % halves + halves * (m(u) % depth); }
  SPEC_HD unsigned parity(int u) const { return (unsigned)(m(u) / depth) & 1u; }
  // The unit that takes u's stage after it.
  SPEC_HD int next(int u) const {
    const int later = m(u) + depth, t = tile(u) % halves + halves * (later / per_tile());
    return per_tile() * t + (dup ? 0 : (later & 1));
  }
  // Giving up after `issued` units: does the producer wait for unit u to land?
  // Only for the last one of its stage, whose parity the barrier still shows; a
  // wait for an earlier one would run to its limit.
  SPEC_HD bool drains(int u, int issued) const { return u < issued && next(u) >= issued; }
};

}  // namespace spec
