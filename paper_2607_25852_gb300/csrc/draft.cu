// draft.cu -- the drafter's producer step on sm_103a: drafts, token-level
// confidences and D-cut scores from the drafter's logits in one streaming
// pass (arxiv 2607.25852, Section 4.2: D-cut ranks positions by the prefix
// products s_{i,k} of the drafter's confidences c_{i,t}, Eq. dcut-score).
//
// Row k of request i holds the drafter's logits for draft z_{k+1}:
//   q_k = softmax(l_k / tau)                     (tau' = tau, or 1 at tau = 0)
//   z_{k+1} ~ q_k by the two-level exponential race at position
//             pos_base_i + k + 1, purposes DRAFT / DRAFT_IN_BLOCK
//             (argmax, lowest index, at tau = 0)
//   c_{k+1} = q_k(z_{k+1}) at tau'
//   s_0 = 1, s_k = fl32(s_{k-1} * c_k)
//
// draft_rows_kernel: one warp per (row, segment of race blocks), warps
// independent of one another.  A warp takes a round of 8 consecutive race
// blocks (256 entries each; 4 for fp32) at a time: a group of 8 lanes reads
// whole 128-byte lines of one block, so a block's sum of
// 2^(l*c2 - fl(M_r*c2)) needs three shuffles inside its lane group; the
// round's max M_r comes from one redux over order-preserving integer keys.
// Level 1 of the race compares blocks in the log2 domain,
//   log2 key_b = log2 E_b - log2 sum_b - fl(M_r*c2)   (see BlockKey),
// so no pass over the row is needed before the draw.  Each lane keeps the sum
// of one block of every 32, forms that block's key once, and holds its own
// best block and its own part of the softmax sum until the segment ends: no
// other exchange sits between a round's loads and the next.  The last warp of
// a row to arrive merges the segments, draws the entry inside the winning
// block (level 2; at tau = 0 finds the first maximum inside the round that
// holds it) and writes z, c and the row statistics; the last row of a request
// to finish writes the scores.
#include <float.h>
#include <math.h>

#include <algorithm>

#include "verify_common.cuh"

namespace spec {

constexpr int kDraftThreads = 128;
constexpr int kDraftCtas = 8;       // resident CTAs per SM (32 warps, 64 registers a thread)
constexpr int kDraftSlots = 152 * kDraftCtas * kDraftThreads / 32;  // warps in one wave
constexpr int kSegmentBlocks = 64;  // race blocks per warp unit, at most
constexpr int kGroup = 32;          // race blocks whose level-1 words one warp-wide Philox call gives

// A level-1 candidate: block idx with L = log2 E_b - log2 sum_b and P =
// fl(M_r*c2), to which sum_b is relative: log2 key = L - P.  Two candidates
// compare by L_a - L_b < P_a - P_b: the rounding of |M*c2|, which reaches
// thousands at small tau, is in the sum and in P alike and cancels, and the
// difference of two P rounds with the gap between them.
struct BlockKey {
  float L, P;
  int32_t idx;  // INT_MAX: none
};
__device__ __forceinline__ bool block_key_better(const BlockKey& a, const BlockKey& b) {
  if (a.idx == INT_MAX) return false;
  if (b.idx == INT_MAX) return true;
  const float lhs = a.L - b.L, rhs = a.P - b.P;
  return lhs < rhs || (lhs == rhs && a.idx < b.idx);
}

struct alignas(16) DraftPartial {
  float m;        // max logit of the chunk
  float s;        // sum of 2^(l*c2 - fl(m*c2))
  float key;      // tau > 0: L of the best block; tau = 0: the max (= m)
  int32_t idx;    // tau > 0: the best block; tau = 0: first block of the first round that holds the max (INT_MAX: none)
  int32_t flags;  // bit0: NaN or +inf seen
  float keyP;     // tau > 0: P of the best block
  int32_t pad[2];
};

struct DraftLaunch {
  const void* logits;  // [B*K, V]
  int B, K, V;
  float tau, c2, inv_t;  // c2 = log2(e) / tau'
  const uint64_t* seeds;
  const uint64_t* request_ids;
  const int64_t* pos_base;
  int32_t* drafts;     // [B, K]
  float* conf;         // [B, K]
  float* scores;       // [B, K+1] or null
  float* row_stats;    // [B*K, 2] or null
  int32_t* status;
  DraftPartial* part;  // [B*K*NC]
  uint32_t* row_count; // [B*K]
  uint32_t* req_count; // [B]
  uint32_t* req_bad;   // [B]
  int NC, chunk;       // segments per row (one warp each), entries per segment (a multiple of 2048)
};

struct DraftGeometry {
  int NC, chunk;
  size_t part_off, counters_off, bytes;
};

static inline long long ceil_div_ll(long long a, long long b) { return (a + b - 1) / b; }

static DraftGeometry draft_geometry(int B, int K, int V) {
  DraftGeometry g{};
  const long long R = (long long)B * K;
  // one warp per (row, segment): segments of a whole number of 8 blocks, as
  // many as fill one wave of warps (B = 16, K = 16, V = 128256: 17.5 us; twice
  // and four times as many 18.2 and 20.6 us), or of at most kSegmentBlocks when
  // the rows fill several (32 or 64 blocks: the same time at the stress size)
  const long long nb = ceil_div_ll(V, 256);
  const long long want = std::max(8LL, std::min<long long>(kSegmentBlocks, ceil_div_ll(ceil_div_ll(R * nb, kDraftSlots), 8) * 8));
  const long long ns = ceil_div_ll(nb, want);
  const long long bps = ceil_div_ll(ceil_div_ll(nb, ns), 8) * 8;
  g.NC = (int)ceil_div_ll(nb, bps);
  g.chunk = (int)(bps * 256);
  g.part_off = 0;
  g.counters_off = ((size_t)sizeof(DraftPartial) * R * g.NC + 255) / 256 * 256;
  g.bytes = g.counters_off + ((size_t)sizeof(uint32_t) * (R + 2 * (size_t)B) + 255) / 256 * 256;
  return g;
}

// Bytes that hold a call of this shape and of every smaller one.  What a shape
// needs does not grow with each of its sizes (V = 201088, K = 1: 156,160 bytes at
// B = 49, 103,168 at B = 64), so a workspace is asked for by a bound that does: the
// segments of R rows are at most a wave of warps and one more a row, or as many
// as the longest segments make of the rows, and never more than the shortest do.
static size_t draft_workspace_bytes(int B, int K, int V) {
  const long long R = (long long)B * K, nb = ceil_div_ll(V, 256);
  const long long parts = std::min(R * ceil_div_ll(nb, 8),
                                   std::max(kDraftSlots + R, R * ceil_div_ll(nb, kSegmentBlocks)));
  const size_t bytes = ((size_t)sizeof(DraftPartial) * parts + 255) / 256 * 256 +
                       ((size_t)sizeof(uint32_t) * (R + 2 * (size_t)B) + 255) / 256 * 256;
  return std::max(bytes, draft_geometry(B, K, V).bytes);
}

__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// A round's 16-byte words: lane l reads, for each of the round's kHalf sets of
// four blocks, word l & 7 of every 128-byte line of block 4h + (l >> 3): 8
// loads in flight, each of four whole lines over the warp.
template <typename T>
struct Round;
template <>
struct Round<__nv_bfloat16> {
  static constexpr int kBlocks = 8;  // race blocks per round
  static constexpr int kHalf = 2;    // sets of four
  static constexpr int kLines = 4;   // 128-byte lines per block
  static constexpr int kPer = 8;     // entries per word
  static constexpr uint32_t kPad = 0xFF80FF80u;
};
template <>
struct Round<float> {
  static constexpr int kBlocks = 4;
  static constexpr int kHalf = 1;
  static constexpr int kLines = 8;
  static constexpr int kPer = 4;
  static constexpr uint32_t kPad = 0xFF800000u;
};

// First entry of word u of lane l in the round that starts at block b0.
template <typename T>
__device__ __forceinline__ int word_entry(int b0, int u, int lane) {
  using R = Round<T>;
  return (b0 + 4 * (u / R::kLines) + (lane >> 3)) * kRaceBlock + (u % R::kLines) * (8 * R::kPer) + (lane & 7) * R::kPer;
}

// 16 bytes of a row at entry v from any alignment: the two aligned words that
// hold them, shifted together.  A word is read only if it lies inside the
// logits [lo, hi); at their two ends, and where fewer than a word's entries
// are left, the entries are read one by one (past vend: -inf).
template <typename T>
__device__ __forceinline__ uint4 load_shifted(const T* row, int v, int vend, uintptr_t lo, uintptr_t hi) {
  using R = Round<T>;
  const uint32_t pad = R::kPad;
  if (v >= vend) return make_uint4(pad, pad, pad, pad);
  const uintptr_t a = reinterpret_cast<uintptr_t>(row + v);
  const uintptr_t w0 = a & ~(uintptr_t)15;
  if (v + R::kPer <= vend && w0 >= lo && w0 + 32 <= hi) {
    const uint4 x = __ldg(reinterpret_cast<const uint4*>(w0)), y = __ldg(reinterpret_cast<const uint4*>(w0) + 1);
    const uint32_t s = (uint32_t)(a & 15u), bits = 8u * (s & 3u);
    // drop s bytes of the 32: whole words by selection, the rest by a funnel shift
    const uint32_t in[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    uint32_t t[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const uint32_t p = s < 4 ? in[k] : in[k + 1], q = s < 12 ? in[k + 2] : in[k + 3 > 7 ? 7 : k + 3];
      t[k] = s < 8 ? p : q;
    }
    return make_uint4(__funnelshift_r(t[0], t[1], bits), __funnelshift_r(t[1], t[2], bits),
                      __funnelshift_r(t[2], t[3], bits), __funnelshift_r(t[3], t[4], bits));
  }
  uint32_t h[8];
#pragma unroll
  for (int e = 0; e < R::kPer; ++e) {
    if (sizeof(T) == 4)
      h[e] = v + e < vend ? __float_as_uint(__ldg(reinterpret_cast<const float*>(row) + v + e)) : pad;
    else
      h[e] = v + e < vend ? (uint32_t)__ldg(reinterpret_cast<const unsigned short*>(row) + v + e) : 0xFF80u;
  }
  if (sizeof(T) == 4) return make_uint4(h[0], h[1], h[2], h[3]);
  return make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
}

// The round's words (entries at or past vend read -inf).
template <typename T, bool kVec>
__device__ __forceinline__ void load_round(uint4 (&w)[8], const T* row, int b0, int vend, int lane, uintptr_t lo,
                                           uintptr_t hi) {
  using R = Round<T>;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int v = word_entry<T>(b0, u, lane);
    if (kVec) w[u] = v < vend ? ldg_stream(row + v) : make_uint4(R::kPad, R::kPad, R::kPad, R::kPad);
    else w[u] = load_shifted(row, v, vend, lo, hi);
  }
}

// Max over a lane's words (a NaN loses to any number here; the sums catch it).
__device__ __forceinline__ float words_max(const uint4 (&w)[8], __nv_bfloat16) {
  __nv_bfloat162 m[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&w[u]);
    m[u] = __hmax2(__hmax2(h[0], h[1]), __hmax2(h[2], h[3]));
  }
#pragma unroll
  for (int n = 4; n > 0; n >>= 1)
#pragma unroll
    for (int u = 0; u < n; ++u) m[u] = __hmax2(m[u], m[u + n]);
  return fmaxf(__low2float(m[0]), __high2float(m[0]));
}
__device__ __forceinline__ float words_max(const uint4 (&w)[8], float) {
  float m[8];
#pragma unroll
  for (int u = 0; u < 8; ++u)
    m[u] = fmaxf(fmaxf(__uint_as_float(w[u].x), __uint_as_float(w[u].y)),
                 fmaxf(__uint_as_float(w[u].z), __uint_as_float(w[u].w)));
#pragma unroll
  for (int n = 4; n > 0; n >>= 1)
#pragma unroll
    for (int u = 0; u < n; ++u) m[u] = fmaxf(m[u], m[u + n]);
  return m[0];
}

// A warp's running state over its segment.  m (and at tau = 0 first) is the
// same in every lane; s and best are the lane's own parts.
struct WarpDraftState {
  float m = -INFINITY, s = 0.0f;           // max, and the lane's sum of 2^(l*c2 - fl(m*c2)); NaN once a NaN or +inf was read
  BlockKey best{INFINITY, 0.0f, INT_MAX};  // tau > 0: the best of the lane's blocks
  int32_t first = INT_MAX;                 // tau = 0: first block of the first round that reaches m
  float keep_s = 0.0f, keep_p = 0.0f;      // tau > 0: the lane's block of the current 32: its sum, and P
};

// The lane's block among each 32 (level 1 of the race): the round whose index
// in the 32 equals owned_round(), and in it the block whose sum block_sum()
// leaves in the lane.
template <typename T>
__device__ __forceinline__ int owned_round(int lane) { return lane & (Round<T>::kHalf == 2 ? 3 : 7); }
template <typename T>
__device__ __forceinline__ int owned_block(int lane) {
  return Round<T>::kHalf == 2 ? 8 * (lane & 3) + (lane & 4) + (lane >> 3) : 4 * (lane & 7) + (lane >> 3);
}
// Sum over the block's 8 lanes: with two blocks per lane group, lanes with bit
// 2 set end with the second one's.
__device__ __forceinline__ float block_sum(const float (&acc)[2], int lane) {
  const bool hi = (lane & 4) != 0;
  float v = (hi ? acc[1] : acc[0]) + __shfl_xor_sync(0xFFFFFFFFu, hi ? acc[0] : acc[1], 4);
  v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
  return v + __shfl_xor_sync(0xFFFFFFFFu, v, 1);
}
__device__ __forceinline__ float block_sum(const float (&acc)[1], int) {
  float v = acc[0] + __shfl_xor_sync(0xFFFFFFFFu, acc[0], 4);
  v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
  return v + __shfl_xor_sync(0xFFFFFFFFu, v, 1);
}

// The level-1 race word of the lane's block among blocks g0 .. g0+31 (g0 a
// multiple of 32): word l >> 3 of the Philox quad of blocks
// g0 + (owned_block & ~3) .. +3.
template <typename T>
__device__ __forceinline__ uint32_t race_word(int g0, int lane, uint32_t position, uint64_t req, uint32_t k0,
                                              uint32_t k1) {
  const uint4 rq =
      philox(draw_counter(position, req, SPEC_PURPOSE_DRAFT, (uint32_t)((g0 + owned_block<T>(lane)) >> 2)), k0, k1);
  const int e = lane >> 3;
  return e == 0 ? rq.x : e == 1 ? rq.y : e == 2 ? rq.z : rq.w;
}

// One round of consecutive race blocks from b0.  Every value is taken relative
// to the round's max M_r: a block whose weight underflows against M_r is more
// than 2^-126 below the round's best and cannot win the race.  A NaN or a +inf
// entry makes the lane's sum NaN, which stays; a round of -inf adds 0.
template <typename T, bool kGreedy>
__device__ __forceinline__ void draft_round(WarpDraftState& ws, const uint4 (&w)[8], int b0, int lane, float c2) {
  using R = Round<T>;
  const float Mr = from_orderable(__reduce_max_sync(0xFFFFFFFFu, orderable(words_max(w, T()))));
  const float M2 = Mr > -INFINITY ? __fmul_rn(Mr, c2) : 0.0f;
  const float2 c2v = make_float2(c2, c2), nM2 = make_float2(-M2, -M2);
  float acc[R::kHalf];
#pragma unroll
  for (int h = 0; h < R::kHalf; ++h) {
    float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
#pragma unroll
    for (int l = 0; l < R::kLines; ++l) {
#pragma unroll
      for (int e = 0; e < R::kPer; e += 4) {
        const uint4& x = w[h * R::kLines + l];
        const float2 y0 = __ffma2_rn(make_float2(Vec<T>::get(x, e), Vec<T>::get(x, e + 1)), c2v, nM2);
        const float2 y1 = __ffma2_rn(make_float2(Vec<T>::get(x, e + 2), Vec<T>::get(x, e + 3)), c2v, nM2);
        a0 = __fadd2_rn(a0, make_float2(ex2_approx(y0.x), ex2_approx(y0.y)));
        a1 = __fadd2_rn(a1, make_float2(ex2_approx(y1.x), ex2_approx(y1.y)));
      }
    }
    acc[h] = (a0.x + a0.y) + (a1.x + a1.y);
  }
  // the softmax state: the lane's part, scaled to the larger max
  const float own = R::kHalf == 2 ? acc[0] + acc[R::kHalf - 1] : acc[0];
  if (Mr > ws.m) {
    ws.s = fmaf(ws.s, ex2_approx(__fmul_rn(ws.m, c2) - M2), own);
    ws.m = Mr;
    if (kGreedy) ws.first = b0;
  } else {
    ws.s = Mr > -INFINITY ? fmaf(own, ex2_approx(M2 - __fmul_rn(ws.m, c2)), ws.s) : ws.s + own;
  }
  if (kGreedy) return;
  const float sb = block_sum(acc, lane);
  if (((b0 & (kGroup - 1)) / R::kBlocks) == owned_round<T>(lane)) {
    ws.keep_s = sb;
    ws.keep_p = M2;
  }
}

// Level-1 key of the lane's block `b` once its round is in (b < b_hi).
__device__ __forceinline__ void draft_candidate(WarpDraftState& ws, int b, uint32_t word) {
  // E near 0 needs log1pf; log2 of E and of the sum go to lg2.approx: its error,
  // 2^-22 of the result (absolute next to 1), is at most 6e-6 at E = 2^-24, the
  // least there is, and 2e-6 at the E of a typical winner
  if (!(ws.keep_s > 0.0f)) return;
  const float E = -log1pf(-((float)race_m(word) * 0x1p-24f));
  const BlockKey k{lg2_approx(E) - lg2_approx(ws.keep_s), ws.keep_p, b};
  if (block_key_better(k, ws.best)) ws.best = k;
}

// One warp per (row, segment of blocks); the warps of a CTA are independent
// (no CTA barrier).  The last warp of a row to arrive merges the row's segment
// partials, draws inside the winning block and writes the row's outputs; the
// last row of a request writes the scores.
template <typename T, bool kGreedy, bool kVec>
__global__ void __launch_bounds__(kDraftThreads, kDraftCtas) draft_rows_kernel(const DraftLaunch p) {
  using R = Round<T>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long unit = (long long)blockIdx.x * (kDraftThreads / 32) + warp;
  if (unit >= (long long)p.B * p.K * p.NC) return;
  const int r = (int)(unit / p.NC);
  const int c = (int)(unit - (long long)r * p.NC);
  const int i = r / p.K;
  const int k = r - i * p.K;
  const T* row = static_cast<const T*>(p.logits) + (size_t)r * (size_t)p.V;
  const uintptr_t lo = reinterpret_cast<uintptr_t>(p.logits);
  const uintptr_t hi = lo + (size_t)p.B * p.K * (size_t)p.V * sizeof(T);

  // ---- this segment's blocks, a round of consecutive ones at a time ----
  const int nb = (p.V + kRaceBlock - 1) / kRaceBlock;
  const int bps = p.chunk / kRaceBlock;
  const int b_lo = c * bps, b_hi = min(nb, b_lo + bps);
  const int vend = (int)min((long long)p.V, (long long)b_hi * kRaceBlock);
  // The segment's first round starts towards L2 (a line a lane) while the
  // previous kernel on the stream drains: a prefetch returns no data, and L2
  // is where that kernel's writes arrive, so nothing is read early.
  const int v_pre = b_lo * kRaceBlock + lane * (128 / (int)sizeof(T));
  if (v_pre < vend) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + v_pre));
  pdl_wait_prerequisites();
  pdl_launch_dependents();
  uint4 w[8];
  load_round<T, kVec>(w, row, b_lo, vend, lane, lo, hi);  // the first loads ahead of the request's scalars
  const long long pos = __ldg(reinterpret_cast<const long long*>(p.pos_base) + i);
  const uint32_t position = (uint32_t)(pos + k + 1);
  const uint64_t req = __ldg(reinterpret_cast<const unsigned long long*>(p.request_ids) + i);
  const uint64_t seed = __ldg(reinterpret_cast<const unsigned long long*>(p.seeds) + i);
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  WarpDraftState ws;
  uint32_t word = 0;
  for (int b0 = b_lo; b0 < b_hi; b0 += R::kBlocks) {
    if (b0 != b_lo) load_round<T, kVec>(w, row, b0, vend, lane, lo, hi);
    // the group's race words, drawn while the loads are in flight
    if (!kGreedy && (b0 == b_lo || (b0 & (kGroup - 1)) == 0)) {
      word = race_word<T>(b0 & ~(kGroup - 1), lane, position, req, k0, k1);
      ws.keep_s = 0.0f;
    }
    draft_round<T, kGreedy>(ws, w, b0, lane, p.c2);
    const int bn = b0 + R::kBlocks;
    if (!kGreedy && (bn >= b_hi || (bn & (kGroup - 1)) == 0))
      draft_candidate(ws, (b0 & ~(kGroup - 1)) + owned_block<T>(lane), word);
  }

  // ---- the segment's partial over the lanes; the last warp of the row goes on ----
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ws.s += __shfl_xor_sync(0xFFFFFFFFu, ws.s, o);
    if (!kGreedy) {
      const BlockKey ob{__shfl_xor_sync(0xFFFFFFFFu, ws.best.L, o), __shfl_xor_sync(0xFFFFFFFFu, ws.best.P, o),
                        __shfl_xor_sync(0xFFFFFFFFu, ws.best.idx, o)};
      if (block_key_better(ob, ws.best)) ws.best = ob;
    }
  }
  int last = 0;
  if (lane == 0) {
    DraftPartial d{};
    d.m = ws.m;
    d.s = ws.s;
    d.key = kGreedy ? ws.m : ws.best.L;
    d.keyP = kGreedy ? 0.0f : ws.best.P;
    d.idx = kGreedy ? ws.first : ws.best.idx;
    d.flags = ws.s != ws.s;
    p.part[(size_t)r * p.NC + c] = d;
    __threadfence();  // the partial before the count
    last = atomicAdd(p.row_count + r, 1u) == (uint32_t)(p.NC - 1);
  }
  if (!__shfl_sync(0xFFFFFFFFu, last, 0)) return;
  __threadfence();  // the other segments' partials after their counts
  const bool pos_ok = pos >= 0 && pos + p.K <= 0xFFFFFFFFLL;

  // ---- merge the row's segments (lanes over segments) ----
  SoftState st{-INFINITY, 0.0f};
  BlockKey best{INFINITY, 0.0f, INT_MAX};
  ArgState g{-INFINITY, INT_MAX};
  int32_t f = 0;
  for (int cc = lane; cc < p.NC; cc += 32) {
    const uint4* src = reinterpret_cast<const uint4*>(p.part + (size_t)r * p.NC + cc);
    const uint4 a = __ldcg(src), b2 = __ldcg(src + 1);
    st = soft_merge(st, SoftState{__uint_as_float(a.x), __uint_as_float(a.y)}, p.c2);
    if (kGreedy) {
      const ArgState o{__uint_as_float(a.z), (int32_t)a.w};
      if (arg_better(o, g)) g = o;
    } else {
      const BlockKey o{__uint_as_float(a.z), __uint_as_float(b2.y), (int32_t)a.w};
      if (block_key_better(o, best)) best = o;
    }
    f |= (int32_t)b2.x;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    st = soft_merge(st, SoftState{__shfl_xor_sync(0xFFFFFFFFu, st.m, o), __shfl_xor_sync(0xFFFFFFFFu, st.s, o)},
                    p.c2);
    const BlockKey ob{__shfl_xor_sync(0xFFFFFFFFu, best.L, o), __shfl_xor_sync(0xFFFFFFFFu, best.P, o),
                      __shfl_xor_sync(0xFFFFFFFFu, best.idx, o)};
    if (block_key_better(ob, best)) best = ob;
    const ArgState og{__shfl_xor_sync(0xFFFFFFFFu, g.v, o), __shfl_xor_sync(0xFFFFFFFFu, g.idx, o)};
    if (arg_better(og, g)) g = og;
  }
  f = (int32_t)__reduce_or_sync(0xFFFFFFFFu, (unsigned)f);
  if (lane == 0) p.row_count[r] = 0u;  // leave the workspace zeroed for the next call
  const int idx = kGreedy ? g.idx : best.idx;
  const bool bad = f || !pos_ok || !(st.m > -INFINITY) || !(st.s > 0.0f) || !isfinite(st.s) || idx == INT_MAX;
  const float M2 = st.m * p.c2;
  int z = -1;
  if (!bad) {
    if (kGreedy) {
      // the first entry of the round from block idx that equals the max
      load_round<T, kVec>(w, row, idx, p.V, lane, lo, hi);
      unsigned first = 0xFFFFFFFFu;
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int e = 0; e < R::kPer; ++e)
          if (Vec<T>::get(w[u], e) == st.m) first = min(first, (unsigned)(word_entry<T>(idx, u, lane) + e));
      first = __reduce_min_sync(0xFFFFFFFFu, first);
      z = first == 0xFFFFFFFFu ? -1 : (int)first;
    } else {
      // level 2 in the winning block (8 entries per lane), weights relative
      // to the row max
      KeyState e{INFINITY, INT_MAX};
      const int v0 = idx * kRaceBlock + 8 * lane;
      uint4 rw[2];
      rw[0] = philox(draw_counter(position, req, SPEC_PURPOSE_DRAFT_IN_BLOCK, (uint32_t)(v0 >> 2)), k0, k1);
      rw[1] = philox(draw_counter(position, req, SPEC_PURPOSE_DRAFT_IN_BLOCK, (uint32_t)(v0 >> 2) + 1u), k0, k1);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int v = v0 + j;
        if (v < p.V) {
          const float wv = ex2_approx(__fmaf_rn(load_elem(row + v), p.c2, -M2));
          const uint4& q4 = rw[j >> 2];
          const uint32_t word = (j & 3) == 0 ? q4.x : (j & 3) == 1 ? q4.y : (j & 3) == 2 ? q4.z : q4.w;
          if (wv > 0.0f) {
            const KeyState kv{race_key(race_m(word), wv), v};
            if (key_better(kv, e)) e = kv;
          }
        }
      }
      e = warp_min_key(e);
      z = e.idx == INT_MAX ? -1 : e.idx;
    }
  }
  int last_row = 0;
  if (lane == 0) {
    const size_t o = (size_t)i * p.K + k;
    if (bad || z < 0) {
      p.drafts[o] = -1;
      p.conf[o] = 0.0f;
      if (p.row_stats) reinterpret_cast<float2*>(p.row_stats)[o] = make_float2(0.0f, 0.0f);
      atomicOr(p.req_bad + i, 1u);
    } else {
      p.drafts[o] = z;
      // c = q(z) = 2^(l_z*c2 - fl(m*c2)) / S, with one rounding in the exponent
      p.conf[o] = exp2f(fmaf(load_elem(row + z), p.c2, -M2)) / st.s;
      if (p.row_stats) {
        const float resid = fmaf(st.m, p.c2, -M2);
        reinterpret_cast<float2*>(p.row_stats)[o] = make_float2(st.m * p.inv_t, (log2f(st.s) - resid) * 0.69314718055994531f);
      }
    }
    __threadfence();  // this row's outputs before the count
    last_row = atomicAdd(p.req_count + i, 1u) == (uint32_t)(p.K - 1);
  }
  // ---- the last row of the request: the scores, the warp loading 32
  // confidences at a time and multiplying them in order ----
  if (!__shfl_sync(0xFFFFFFFFu, last_row, 0)) return;
  __threadfence();
  const bool req_bad = __ldcg(p.req_bad + i) != 0u;
  __syncwarp();  // every lane has read the flag
  if (lane == 0) {
    p.req_count[i] = 0u;
    if (req_bad) {
      p.req_bad[i] = 0u;
      report(p.status, SPEC_ERR_BAD_INPUT);
    }
  }
  float run = 1.0f;
  if (p.scores && lane == 0) p.scores[(size_t)i * (p.K + 1)] = run;
  for (int base = 0; base < p.K; base += 32) {
    const int kk = base + lane;
    const size_t o = (size_t)i * p.K + kk;
    float cf = 0.0f, mine = 0.0f;
    if (kk < p.K) {
      if (req_bad) {
        p.drafts[o] = -1;
        p.conf[o] = 0.0f;
        if (p.row_stats) reinterpret_cast<float2*>(p.row_stats)[o] = make_float2(0.0f, 0.0f);
      } else {
        cf = __ldcg(p.conf + o);
      }
    }
    const int n = min(32, p.K - base);
    for (int j = 0; j < n; ++j) {
      run = __fmul_rn(run, __shfl_sync(0xFFFFFFFFu, cf, j));
      if (lane == j) mine = run;
    }
    if (p.scores && kk < p.K) p.scores[(size_t)i * (p.K + 1) + kk + 1] = mine;
  }
}

template <typename T>
static cudaError_t launch_draft_typed(const DraftLaunch& p, bool vec, cudaStream_t stream) {
  const long long units = (long long)p.B * p.K * p.NC;  // one warp each
  const dim3 grid((unsigned)((units + kDraftThreads / 32 - 1) / (kDraftThreads / 32))), block(kDraftThreads);
  const bool greedy = p.tau == 0.0f;
  if (vec)
    return greedy ? launch_after_previous(draft_rows_kernel<T, true, true>, grid, block, 0, stream, p)
                  : launch_after_previous(draft_rows_kernel<T, false, true>, grid, block, 0, stream, p);
  return greedy ? launch_after_previous(draft_rows_kernel<T, true, false>, grid, block, 0, stream, p)
                : launch_after_previous(draft_rows_kernel<T, false, false>, grid, block, 0, stream, p);
}

}  // namespace spec

extern "C" size_t spec_draft_workspace(int B, int K, int V) {
  if (B < 1 || K < 1 || K > SPEC_MAX_DRAFTS || V < 1 || V >= SPEC_MAX_VOCAB || (long long)B * K > (1LL << 28))
    return 0;
  return spec::draft_workspace_bytes(B, K, V);
}

extern "C" int spec_draft(const void* logits, int logits_dtype, int B, int K, int V, float tau,
                          const uint64_t* seeds, const uint64_t* request_ids, const int64_t* pos_base,
                          int32_t* drafts_out, float* conf_out, float* scores_out, float* row_stats_out,
                          int32_t* status, void* ws, size_t ws_bytes, cudaStream_t stream) {
  spec::NvtxRange range("spec_draft");
  if (B < 1 || K < 1 || K > SPEC_MAX_DRAFTS || V < 1 || V >= SPEC_MAX_VOCAB || (long long)B * K > (1LL << 28))
    return SPEC_ERR_INVALID_ARG;
  if ((logits_dtype != SPEC_BF16 && logits_dtype != SPEC_F32) || !(tau >= 0.0f) || isinf(tau))
    return SPEC_ERR_INVALID_ARG;
  if (!logits || !seeds || !request_ids || !pos_base || !drafts_out || !conf_out) return SPEC_ERR_INVALID_ARG;
  if (row_stats_out && (reinterpret_cast<uintptr_t>(row_stats_out) & 7u) != 0) return SPEC_ERR_INVALID_ARG;
  const spec::DraftGeometry g = spec::draft_geometry(B, K, V);
  if (!ws || ws_bytes < g.bytes || (reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return SPEC_ERR_WORKSPACE;
  spec::DraftLaunch p{};
  p.logits = logits;
  p.B = B;
  p.K = K;
  p.V = V;
  p.tau = tau;
  const double tc = tau > 0.0f ? (double)tau : 1.0;
  p.c2 = (float)(1.4426950408889634 / tc);
  p.inv_t = (float)(1.0 / tc);
  p.seeds = seeds;
  p.request_ids = request_ids;
  p.pos_base = pos_base;
  p.drafts = drafts_out;
  p.conf = conf_out;
  p.scores = scores_out;
  p.row_stats = row_stats_out;
  p.status = status;
  char* base = static_cast<char*>(ws);
  p.part = reinterpret_cast<spec::DraftPartial*>(base + g.part_off);
  const size_t R = (size_t)B * K;
  p.row_count = reinterpret_cast<uint32_t*>(base + g.counters_off);
  p.req_count = p.row_count + R;
  p.req_bad = p.req_count + B;
  p.NC = g.NC;
  p.chunk = g.chunk;
  const size_t esize = logits_dtype == SPEC_F32 ? 4 : 2;
  // 16-byte loads: rows on the 16-byte grid, of whole groups of 8 entries.  (fp32
  // rows of V % 8 == 4 lie on the grid too, but take the shifted words.)
  const bool vec = (reinterpret_cast<uintptr_t>(logits) & 15u) == 0 && ((size_t)V * esize) % 16 == 0 && V % 8 == 0;
  const cudaError_t err = logits_dtype == SPEC_F32 ? spec::launch_draft_typed<float>(p, vec, stream)
                                                   : spec::launch_draft_typed<__nv_bfloat16>(p, vec, stream);
  if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return SPEC_ERR_CUDA;
  return SPEC_OK;
}
