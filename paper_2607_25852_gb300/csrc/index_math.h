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
  if (packed) return PrefetchSpan{block * per_cta, block < kStreamWave ? B * V : 0};
  if (has_depth && j > 0) return PrefetchSpan{0, 0};
  const long long row = ((long long)i * (K + 1) + j) * V;
  const long long last = (c + 1) * chunk;
  return PrefetchSpan{row + c * chunk, row + (last < V ? last : V)};
}

}  // namespace spec
