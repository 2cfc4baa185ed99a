// allocate.cu -- D-cut verification-depth allocation (Section 4.2 of arxiv
// 2607.25852) in one CTA, or one thread-block cluster, on sm_103a.
//
// At most SPEC_MAX_ALLOC_POSITIONS = 8192 positions, so the whole problem fits
// in shared memory.  Every position (i, k) becomes one 64-bit key
//   bits(s_{i,k}) << 32 | (0xFFFF - k) << 16 | (0xFFFF - i)
// whose descending order is the allocator's total order: s >= +0 (a -0
// confidence is taken as +0), so the fp32 bit pattern is monotone in s; then
// shallower k first (the paper's tie rule);
// then lower request index.  Keys are unique.
//
// Batches of at most 1024 requests and 1024 draft positions take
// allocate_small_kernel (below), which sorts the draft keys alone: a merge
// tree over the per-request runs padded to a power of two when they fit in
// 1024 slots, else a bitonic sort.  Larger batches take
// allocate_cluster_kernel: up to eight CTAs sort 1024 draft keys each and rank
// them against one another through distributed shared memory.  Sums of
// floor(s * 2^40) over the top positions give every candidate's utility U(T)
// exactly; the first maximiser of U / cost is chosen and the kept prefixes are
// packed densely.
#include <float.h>
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "spec_internal.cuh"

namespace spec {

constexpr int kAllocThreads = 1024;

__device__ __forceinline__ unsigned long long position_key(float s, int k, int i) {
  return ((unsigned long long)__float_as_uint(s) << 32) |
         ((unsigned long long)(0xFFFFu - (unsigned)k) << 16) | (unsigned long long)(0xFFFFu - (unsigned)i);
}

__device__ __forceinline__ unsigned long long lds_u64(uint32_t addr) {
  unsigned long long v;
  asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_u64(uint32_t addr, unsigned long long v) {
  asm volatile("st.shared.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

// Inclusive block scan of one int64 value per thread (kAllocThreads threads).
__device__ __forceinline__ long long block_inclusive_scan(long long x, long long* warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[warp] = x;
  __syncthreads();
  if (warp == 0) {
    long long t = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xFFFFFFFFu, t, o);
      if (lane >= o) t += y;
    }
    warp_tot[lane] = t;
  }
  __syncthreads();
  const long long before = warp > 0 ? warp_tot[warp - 1] : 0;
  __syncthreads();  // warp_tot reusable after return
  return x + before;
}

// units * 2^-40 as a double, for 0 < units < 2^53 (exact), with integer
// operations only: the product's exponent and mantissa fields are set directly.
__device__ __forceinline__ double units_to_double(long long units) {
  const int msb = 63 - __clzll(units);
  const unsigned long long mant = ((unsigned long long)units << (63 - msb)) << 1 >> 12;  // the bits below the msb
  const unsigned long long expo = (unsigned long long)(msb - 40 + 1023);
  return __longlong_as_double((long long)((expo << 52) | mant));
}

// ---------------------------------------------------------------------------
// Batches of more than 1024 draft positions or 1024 requests
// ---------------------------------------------------------------------------
// One thread-block cluster of C = 2, 4 or 8 CTAs, the least with
// max(B * K, B) <= 1024 C, one draft key per thread: CTA c owns the draft slots
// e = i * K + (k - 1) in [1024 c, 1024 c + 1024) and the requests of that index
// range.  A single CTA is bound by its serial searches (eight keys a thread) and
// by shared-memory bank conflicts; eight CTAs take one key a thread and exchange
// through distributed shared memory, which one GPC's SMs reach without a trip
// to L2.
//   1. scores and keys of the CTA's slots; a merge tree over the per-request
//      runs (already descending) sorts them locally;
//   2. every CTA copies the others' sorted keys and finds each of its keys'
//      rank among all draft keys (C - 1 interleaved binary searches);
//   3. U(T_m) is the sum of the CTAs' local prefixes at rank T_m - B, exact
//      in integers in any order; every CTA gets all parts and picks the same T;
//   4. the last kept draft of each request gives its depth, sent to every
//      CTA; each scans all depths and packs its own slots.
// Three cluster barriers in all.  Measured at B = 256, K = 31, M = 16, calls
// replayed from a graph: 69.4 us a call with a one-CTA merge tree over all
// keys, 15.2 us with the cluster.  The line to allocate_small_kernel is 1024
// draft keys because that kernel's single CTA has one key a thread up to
// there: its sort needs no cluster barrier and no second search (7.5 us at
// B = 64, K = 16).
constexpr int kClusterMax = 8;
constexpr int kSlots = kAllocThreads;  // draft slots, and requests, per CTA
// Floats that stage the confidences of the requests a CTA's slots touch, a row
// of K | 1 each: at most 1024 / K + 2 rows, (1024 / K + 2)(K + 1) <= 2052.
constexpr int kConfStage = 2080;

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// The address of `local` (a shared-memory address of this CTA) in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  return a;
}
__device__ __forceinline__ unsigned long long ldc_u64(uint32_t addr) {
  unsigned long long v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ int ldc_s32(uint32_t addr) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void stc_u64(uint32_t addr, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void stc_s32(uint32_t addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

struct ClusterSmem {
  unsigned long long all[kClusterMax][kSlots];  // every CTA's sorted keys
  unsigned long long keys[2][kSlots];           // local merge tree; then the prefix sums
  long long contrib[kClusterMax][SPEC_MAX_CANDIDATES];
  long long warp_tot[32];
  float conf[kConfStage];                       // [i - i0][k - 1] at (i - i0) * (K | 1) + k - 1, then the scores
  int rank[kSlots];                             // rank of the sorted keys, ascending
  int slot_rank[kSlots];                        // rank of slot 1024 c + t
  int depth[SPEC_MAX_ALLOC_POSITIONS];          // n_i of every request, then the row offsets
  int best_c;
};

template <int C>
__global__ void __launch_bounds__(kAllocThreads, 1) allocate_cluster_kernel(const AllocLaunch p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  static_assert(C > 1, "one CTA's worth of keys is allocate_small_kernel's");
  ClusterSmem& sm = *reinterpret_cast<ClusterSmem*>(smem_raw);
  const int B = p.B, K = p.K, NK = B * K, CS = K | 1;
  const int tid = threadIdx.x, c = blockIdx.x;
  const int e0 = c * kSlots;                              // first slot, and first request, of this CTA
  const int nloc = max(0, min(kSlots, NK - e0));          // draft slots here
  const int i0 = nloc > 0 ? e0 / K : 0;                   // requests the slots touch: i0 ..
  const int nreq = nloc > 0 ? (e0 + nloc - 1) / K - i0 + 1 : 0;
  // The next kernel (the streaming pass) may launch now: it waits for this
  // one's completion before it reads the depths and row offsets.
  pdl_launch_dependents();
  // This kernel starts while the previous one on the stream drains; it reads
  // its inputs, and overwrites the arrays the previous round's kernels read,
  // only once that kernel has completed.
  pdl_wait_prerequisites();

  // ---- every global input in one round trip ----
  const int nconf = nreq > 0 ? e0 + nloc - i0 * K : 0;  // <= 1024 + K - 1
  for (int x = tid; x < nconf; x += kAllocThreads) sm.conf[x / K * CS + x % K] = p.conf[i0 * K + x];
  const int e = e0 + tid;                               // this thread's slot ...
  const int si = tid < nloc ? e / K : 0;                // ... of request si,
  const int sk = tid < nloc ? e - si * K + 1 : 0;       // draft sk
  const int draft = tid < nloc ? p.drafts[e] : 0;
  const long long spos = tid < nloc ? p.pos_base[si] : 0;
  const int last = e < B ? p.last_tokens[e] : 0;        // and the request e0 + tid
  const long long rpos = e < B ? p.pos_base[e] : 0;
  for (int i = tid; i < B; i += kAllocThreads) sm.depth[i] = 0;
  __syncthreads();

  // ---- Eq. (dcut-score): fp32 prefix products in order, a request a thread ----
  for (int rr = tid; rr < nreq; rr += kAllocThreads) {
    float* row = sm.conf + rr * CS;
    const int kend = min(K, nconf - rr * K);
    float s = 1.0f;
    bool bad = false;
#pragma unroll 4
    for (int k = 0; k < kend; ++k) {
      float cf = row[k];
      if (!(cf >= 0.0f && cf <= 1.0f)) {
        bad = true;
        cf = 0.0f;
      }
      // -0 passes the range check and equals 0, but its sign bit would put
      // its key above every positive score: -0 + 0 = +0 drops the sign.
      cf = __fadd_rn(cf, 0.0f);
      s = __fmul_rn(s, cf);
      row[k] = s;
    }
    if (bad) report(p.status, SPEC_ERR_BAD_INPUT);
  }
  __syncthreads();

  // ---- local merge tree (descending).  At level l the groups of 2^l runs
  // merge in pairs; the first and the last run may be cut by the CTA's range.
  // A key's place is its index in its group plus the number of the partner
  // group's keys above it (keys are unique). ----
  unsigned long long x = tid < nloc ? position_key(sm.conf[(si - i0) * CS + sk - 1], sk, si) : 0ull;
  const uint32_t kbuf0 = (uint32_t)__cvta_generic_to_shared(sm.keys[0]);
  const uint32_t kbuf1 = (uint32_t)__cvta_generic_to_shared(sm.keys[1]);
  uint32_t src = kbuf0, dst = kbuf1;
  sts_u64(src + 8u * (uint32_t)tid, x);  // pad slots hold key 0, below every real key
  sts_u64(dst + 8u * (uint32_t)tid, x);
  __syncthreads();
  const int cut = i0 * K - e0;  // <= 0: local slot of request i0's first draft
  for (int lev = 0; (1 << lev) < nreq; ++lev) {
    if (tid < nloc) {
      // the request of the key now at slot tid: groups are contiguous, so the
      // slot's own group is found from its position
      const int group = ((tid - cut) / K) >> lev, pg = group ^ 1;
      const int start = max(0, cut + (group << lev) * K);
      const int pstart = max(0, cut + (pg << lev) * K);
      const int pend = min(nloc, cut + ((pg + 1) << lev) * K);
      int lo = pstart, n = max(0, pend - pstart);
      while (n > 0) {
        const int half = n >> 1;
        const bool above = lds_u64(src + 8u * (uint32_t)(lo + half)) > x;
        lo = above ? lo + half + 1 : lo;
        n = above ? n - half - 1 : half;
      }
      sts_u64(dst + 8u * (uint32_t)(min(start, pstart) + (tid - start) + (lo - pstart)), x);
    }
    __syncthreads();
    const uint32_t t = src;
    src = dst;
    dst = t;
    x = lds_u64(src + 8u * (uint32_t)tid);
  }
  sm.all[c][tid] = x;
  cluster_sync_all();
  // ---- the other CTAs' sorted keys, then this key's rank among them ----
#pragma unroll
  for (int o = 1; o < C; ++o) {
    const int cc = (c + o) & (C - 1);
    sm.all[cc][tid] = ldc_u64(cluster_addr((uint32_t)__cvta_generic_to_shared(&sm.all[cc][tid]), cc));
  }
  __syncthreads();
  int rank = tid;
  uint32_t base[C];
  int cnt[C];
#pragma unroll
  for (int o = 1; o < C; ++o) {
    base[o] = (uint32_t)__cvta_generic_to_shared(sm.all[(c + o) & (C - 1)]);
    cnt[o] = 0;
  }
#pragma unroll
  for (int step = kSlots >> 1; step > 0; step >>= 1)
#pragma unroll
    for (int o = 1; o < C; ++o)
      if (lds_u64(base[o] + 8u * (uint32_t)(cnt[o] + step - 1)) > x) cnt[o] += step;
#pragma unroll
  for (int o = 1; o < C; ++o) {
    if (lds_u64(base[o] + 8u * (uint32_t)cnt[o]) > x) ++cnt[o];
    rank += cnt[o];
  }
  const int xi = 0xFFFF - (int)(x & 0xFFFFull);
  const int xk = 0xFFFF - (int)((x >> 16) & 0xFFFFull);
  sm.rank[tid] = tid < nloc ? rank : INT_MAX;  // ascending along the local order
  if (tid < nloc) sm.slot_rank[xi * K + (xk - 1) - e0] = rank;

  // ---- inclusive scan of floor(s * 2^40) in the local order; the CTA's part
  // of every U(T_m), sent to all CTAs ----
  const long long q40 =
      tid < nloc ? (long long)__float2ll_rd(__uint_as_float((unsigned)(x >> 32)) * 0x1p40f) : 0;
  const long long incl = block_inclusive_scan(q40, sm.warp_tot);
  long long* prefix = reinterpret_cast<long long*>(sm.keys[0]);
  prefix[tid] = incl;
  __syncthreads();
  if (tid < p.M) {
    const int td = p.cand_T[tid] - B;  // draft positions kept at this budget
    int lo = 0, n = nloc;              // local keys of rank < td
    while (n > 0) {
      const int half = n >> 1;
      const bool below = sm.rank[lo + half] < td;
      lo = below ? lo + half + 1 : lo;
      n = below ? n - half - 1 : half;
    }
    const long long part = lo > 0 ? prefix[lo - 1] : 0;
    const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&sm.contrib[c][tid]);
#pragma unroll
    for (int o = 0; o < C; ++o) stc_u64(cluster_addr(mine, o), (unsigned long long)part);
  }
  cluster_sync_all();

  // ---- Eq. (dcut-select): first maximiser of U / cost, in every CTA ----
  if (tid < 32) {
    long long best_key = -1;
    int best_c = INT_MAX;
    for (int m = tid; m < p.M; m += 32) {
      long long Uq = (long long)B << 40;
#pragma unroll
      for (int o = 0; o < C; ++o) Uq += sm.contrib[o][m];
      const double U = units_to_double(Uq);
      if (p.utility_out && c == 0) p.utility_out[m] = U;
      // U > 0 and cost > 0: the quotients order as their bit patterns do
      const long long obj = __double_as_longlong(U / p.cand_cost[m]);
      if (obj > best_key) {  // m increases along the lane's loop
        best_key = obj;
        best_c = m;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ob = __shfl_xor_sync(0xFFFFFFFFu, best_key, o);
      const int cb = __shfl_xor_sync(0xFFFFFFFFu, best_c, o);
      if (ob > best_key || (ob == best_key && cb < best_c)) {
        best_key = ob;
        best_c = cb;
      }
    }
    if (tid == 0) sm.best_c = best_c == INT_MAX ? 0 : best_c;
  }
  __syncthreads();
  const int T = p.cand_T[sm.best_c];
  const int TD = T - B;

  // ---- keep depths: the last kept draft of each request, to every CTA ----
  const bool kept = tid < nloc && sm.slot_rank[tid] < TD;
  if (kept) {
    bool next = false;
    if (sk < K) {  // slot e + 1, in the next CTA past this one's last slot
      if (tid + 1 < kSlots) next = sm.slot_rank[tid + 1] < TD;
      else next = ldc_s32(cluster_addr((uint32_t)__cvta_generic_to_shared(&sm.slot_rank[0]), c + 1)) < TD;
    }
    if (!next) {
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(&sm.depth[si]);
#pragma unroll
      for (int o = 0; o < C; ++o) stc_s32(cluster_addr(d, o), sk);
    }
  }
  cluster_sync_all();

  // ---- row offsets: exclusive scan of (n_i + 1) over all requests, in every
  // CTA; each writes its requests' outputs ----
  const int per = (B + kAllocThreads - 1) / kAllocThreads;  // <= 8, consecutive requests a thread
  const int b0 = min(B, tid * per), b1 = min(B, b0 + per);
  int sum = 0;
  for (int i = b0; i < b1; ++i) sum += sm.depth[i] + 1;
  int off = (int)block_inclusive_scan(sum, sm.warp_tot) - sum;
  for (int i = b0; i < b1; ++i) {
    const int n = sm.depth[i];
    if (i / kSlots == c) {
      p.row_offsets_out[i] = off;
      p.depth_out[i] = n;
    }
    sm.depth[i] = off;  // the offsets from here on
    off += n + 1;
  }
  if (c == 0 && tid == 0) {
    p.row_offsets_out[B] = T;  // sum of (n_i + 1): the T kept positions
    *p.chosen_T_out = T;
  }
  __syncthreads();

  // ---- dense packing of the kept prefixes ----
  if (e < B) {
    p.packed_tokens_out[sm.depth[e]] = last;
    p.packed_pos_out[sm.depth[e]] = rpos;
  }
  if (kept) {
    const int row = sm.depth[si] + sk;
    p.packed_tokens_out[row] = draft;
    p.packed_pos_out[row] = spos + sk;
  }
  for (int r = T + e; r < B * (K + 1); r += C * kAllocThreads) {
    p.packed_tokens_out[r] = -1;
    p.packed_pos_out[r] = -1;
  }
}

// ---------------------------------------------------------------------------
// Batches of at most 1024 requests and 1024 draft positions (B * K)
// ---------------------------------------------------------------------------
// Every bonus position (k = 0) has the largest score (s = 1) and the smallest
// k, so it ranks above every draft position, and the bonus positions rank
// among themselves by request index.  The global order is therefore the B
// bonus positions, then the B * K draft keys sorted; only the latter need a
// sort.  One draft key per thread, sorted by a bitonic network over 1024 slots
// (padding key 0 ranks below every real key, whose k field is nonzero):
// partners within a warp exchange by shuffles, others through shared memory,
// one barrier per such stage.  The keep depths then follow from the sorted
// ranks without atomics: draft (i, k) in the top T - B, with (i, k + 1) not,
// ends request i's kept prefix.
constexpr int kSmallSlots = kAllocThreads;

__device__ __forceinline__ unsigned long long shfl_xor_u64(unsigned long long x, int o) {
  const unsigned lo = __shfl_xor_sync(0xFFFFFFFFu, (unsigned)x, o);
  const unsigned hi = __shfl_xor_sync(0xFFFFFFFFu, (unsigned)(x >> 32), o);
  return ((unsigned long long)hi << 32) | lo;
}

// One level of the small kernel's merge tree over kSmallSlots keys in shared
// memory (src), runs of L keys merged in pairs into dst; x is the calling
// thread's key at slot tid, and on return the key at slot tid of the merged
// order (src and dst swapped).
template <int L>
__device__ __forceinline__ void merge_level(unsigned long long& x, int tid, uint32_t& src, uint32_t& dst) {
  const uint32_t partner = src + 8u * (uint32_t)((tid ^ L) & ~(L - 1));
  int c = 0;
#pragma unroll
  for (int step = L >> 1; step > 0; step >>= 1)
    if (lds_u64(partner + 8u * (uint32_t)(c + step - 1)) > x) c += step;
  if (lds_u64(partner + 8u * (uint32_t)c) > x) ++c;
  sts_u64(dst + 8u * (uint32_t)((tid & ~(2 * L - 1)) + (tid & (L - 1)) + c), x);
  __syncthreads();
  const uint32_t t = src;
  src = dst;
  dst = t;
  x = lds_u64(src + 8u * (uint32_t)tid);
}

__global__ void __launch_bounds__(kAllocThreads) allocate_small_kernel(const AllocLaunch p) {
  __shared__ float sh_conf[2 * kSmallSlots];               // [i][k] at i * (K | 1) + k
  __shared__ int32_t sh_drafts[kSmallSlots];
  __shared__ int32_t sh_last[kSmallSlots];
  __shared__ long long sh_pos[kSmallSlots];
  __shared__ unsigned long long sh_x[2][kSmallSlots];      // sort exchanges, then prefix sums / depths
  __shared__ int32_t sh_rank[kSmallSlots];                 // sorted rank of draft (i, k) at i * K + k - 1
  __shared__ long long warp_tot[32];
  __shared__ int sh_best_c, sh_bad;
  const int B = p.B, K = p.K, NK = B * K, CS = K | 1;
  const int tid = threadIdx.x;
  if (tid == 0) sh_bad = 0;
  // The next kernel (the streaming pass) may launch now: it waits for this
  // one's completion before it reads the depths and row offsets.
  pdl_launch_dependents();
  // This kernel starts while the previous one on the stream drains; it reads
  // its inputs, and overwrites the arrays the previous round's kernels read,
  // only once that kernel has completed.
  pdl_wait_prerequisites();

  // ---- every global input in one round trip ----
  if (tid < NK) {
    const int i = tid / K;
    sh_conf[tid + i * (CS - K)] = p.conf[tid];
    sh_drafts[tid] = p.drafts[tid];
  }
  if (tid < B) {
    sh_last[tid] = p.last_tokens[tid];
    sh_pos[tid] = p.pos_base[tid];
  }
  __syncthreads();

  // ---- Eq. (dcut-score): fp32 prefix products, request i in thread i ----
  // When B * KP <= 1024 (KP = the next power of two >= K), request i's keys
  // fill run i of KP slots in descending order (s is non-increasing in k),
  // and the slots past K, and the runs past B, hold pad keys: unique, below
  // every real key, descending within a run.  A merge tree then sorts the
  // 1024 slots.  Otherwise the keys are staged unsorted for a bitonic sort.
  const int KP = K <= 1 ? 1 : 1 << (32 - __clz(K - 1));
  const bool runs = B * KP <= kSmallSlots;
  // Keys are staged with a row of RL slots per request at the odd stride
  // RS = RL + 1 (in 8-byte words), so that the threads of a half-warp, one
  // request each, store to distinct banks.
  const int RL = runs ? KP : (K > 0 ? K : 1), RS = RL + 1;
  unsigned long long* stage = &sh_x[0][0];  // B * RS <= 2048 words over both buffers
  if (tid < B) {
    const float* ci = sh_conf + tid * CS;
    float s = 1.0f;
    for (int k0 = 1; k0 <= K; k0 += 4) {
      float c4[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) c4[u] = k0 + u <= K ? ci[k0 + u - 1] : 1.0f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = k0 + u;
        if (k > K) break;
        float c = c4[u];
        if (!(c >= 0.0f && c <= 1.0f)) {
          sh_bad = 1;
          c = 0.0f;
        }
        c = __fadd_rn(c, 0.0f);  // -0 counts as +0 (its sign bit would break the key order)
        s = __fmul_rn(s, c);
        stage[tid * RS + k - 1] = position_key(s, k, tid);
      }
    }
  }
  __syncthreads();

  unsigned long long x;
  if (runs) {
    // slot u = i * KP + (k - 1); a pad key is 1024 - u (real keys are above
    // 0xFBFF0000 even at s = 0)
    x = (tid / KP < B && tid % KP < K) ? stage[(tid / KP) * RS + tid % KP] : (unsigned long long)(kSmallSlots - tid);
    __syncthreads();  // the staging area holds the merge buffers from here on
    // ---- merge tree, descending: at the level of runs of L keys, a key's
    // place in the merged pair is its index in its run plus the number of
    // keys of the partner run above it (keys are unique), found by a
    // branch-free binary search of log2(L) + 1 shared-memory probes ----
    uint32_t src = (uint32_t)__cvta_generic_to_shared(&sh_x[0][0]);
    uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sh_x[1][0]);
    sts_u64(src + 8u * (uint32_t)tid, x);
    __syncthreads();
    // the levels from runs of KP on, each unrolled for its L, until one run
    // holds every request's keys: the pads past it are in order and below them
    // (B = K = 4 needs 2 of its 8 levels: 4.7 us from the grid wait to the last
    // store, 6.7 with all)
    const int end = B * KP;
    if (KP <= 1 && 1 < end) merge_level<1>(x, tid, src, dst);
    if (KP <= 2 && 2 < end) merge_level<2>(x, tid, src, dst);
    if (KP <= 4 && 4 < end) merge_level<4>(x, tid, src, dst);
    if (KP <= 8 && 8 < end) merge_level<8>(x, tid, src, dst);
    if (KP <= 16 && 16 < end) merge_level<16>(x, tid, src, dst);
    if (KP <= 32 && 32 < end) merge_level<32>(x, tid, src, dst);
    if (KP <= 64 && 64 < end) merge_level<64>(x, tid, src, dst);
    if (KP <= 128 && 128 < end) merge_level<128>(x, tid, src, dst);
    if (KP <= 256 && 256 < end) merge_level<256>(x, tid, src, dst);
    if (KP <= 512 && 512 < end) merge_level<512>(x, tid, src, dst);
  } else {
    // ---- bitonic sort of the draft keys, descending ----
    x = tid < NK ? stage[(tid / RL) * RS + tid % RL] : 0ull;
    __syncthreads();  // the staging area is the exchange buffer from here on
    int buf = 1;
#pragma unroll
    for (int k = 2; k <= kSmallSlots; k <<= 1) {
#pragma unroll
      for (int j = k >> 1; j > 0; j >>= 1) {
        unsigned long long y;
        if (j >= 32) {
          sh_x[buf][tid] = x;
          __syncthreads();
          y = sh_x[buf][tid ^ j];
          buf ^= 1;
        } else {
          y = shfl_xor_u64(x, j);
        }
        // blocks of k alternate direction (descending first); the lower
        // index of a pair keeps the larger key in a descending block
        const bool take_max = ((tid & k) == 0) == ((tid & j) == 0);
        x = take_max ? (x > y ? x : y) : (x < y ? x : y);
      }
    }
  }
  // x: the draft key of rank tid (tid < NK)
  const int xi = 0xFFFF - (int)(x & 0xFFFFull);
  const int xk = 0xFFFF - (int)((x >> 16) & 0xFFFFull);
  if (tid < NK) sh_rank[xi * K + (xk - 1)] = tid;

  // ---- inclusive scan of floor(s * 2^40) over the sorted draft keys ----
  const long long q40 = tid < NK ? (long long)__float2ll_rd(__uint_as_float((unsigned)(x >> 32)) * 0x1p40f) : 0;
  const long long incl = block_inclusive_scan(q40, warp_tot);  // its barriers also end the sort's reads
  long long* prefix = reinterpret_cast<long long*>(sh_x[0]);
  prefix[tid] = incl;
  __syncthreads();

  // ---- Eq. (dcut-select): first maximiser of U / cost ----
  if (tid < 32) {
    long long best_key = -1;
    int best_c = INT_MAX;
    for (int c = tid; c < p.M; c += 32) {
      const int td = p.cand_T[c] - B;  // draft positions kept at this budget
      const long long Uq = ((long long)B << 40) + (td > 0 ? prefix[td - 1] : 0);
      const double U = units_to_double(Uq);
      if (p.utility_out) p.utility_out[c] = U;
      // U > 0 and cost > 0: the bit patterns of the quotients order as the
      // quotients do, so the comparisons below are integer ones
      const long long obj = __double_as_longlong(U / p.cand_cost[c]);
      if (obj > best_key) {  // c increases along the lane's loop
        best_key = obj;
        best_c = c;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ob = __shfl_xor_sync(0xFFFFFFFFu, best_key, o);
      const int cb = __shfl_xor_sync(0xFFFFFFFFu, best_c, o);
      if (ob > best_key || (ob == best_key && cb < best_c)) {
        best_key = ob;
        best_c = cb;
      }
    }
    if (tid == 0) sh_best_c = best_c == INT_MAX ? 0 : best_c;
  }
  int* depth = reinterpret_cast<int*>(sh_x[1]);
  int* offsets = depth + kSmallSlots;
  if (tid < B) depth[tid] = 0;
  __syncthreads();
  const int T = p.cand_T[sh_best_c];
  const int TD = T - B;

  // ---- keep depths: the last kept draft of each request ----
  if (tid < NK && tid < TD) {
    const bool next_kept = xk < K && sh_rank[xi * K + xk] < TD;
    if (!next_kept) depth[xi] = xk;
  }
  __syncthreads();

  // ---- row offsets: exclusive scan of (n_i + 1), one warp: lane l takes
  // the requests [l * m, (l + 1) * m) in order, m = ceil(B / 32) ----
  if (tid < 32) {
    const int m = (B + 31) >> 5;
    const int i0 = min(B, tid * m), i1 = min(B, i0 + m);
    int sum = 0;
    for (int i = i0; i < i1; ++i) sum += depth[i] + 1;
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (tid >= o) incl += y;
    }
    int off = incl - sum;
    for (int i = i0; i < i1; ++i) {
      const int n = depth[i];
      offsets[i] = off;
      p.row_offsets_out[i] = off;
      p.depth_out[i] = n;
      off += n + 1;
    }
    if (tid == 0) {
      p.row_offsets_out[B] = T;  // sum of (n_i + 1): the T kept positions
      *p.chosen_T_out = T;
    }
  }
  __syncthreads();

  // ---- dense packing of the kept prefixes ----
  if (tid < B) {
    p.packed_tokens_out[offsets[tid]] = sh_last[tid];
    p.packed_pos_out[offsets[tid]] = sh_pos[tid];
  }
  if (tid < NK && tid < TD) {
    const int row = offsets[xi] + xk;
    p.packed_tokens_out[row] = sh_drafts[xi * K + (xk - 1)];
    p.packed_pos_out[row] = sh_pos[xi] + xk;
  }
  for (int r = T + tid; r < B * (K + 1); r += kAllocThreads) {
    p.packed_tokens_out[r] = -1;
    p.packed_pos_out[r] = -1;
  }
  if (tid == 0 && sh_bad) report(p.status, SPEC_ERR_BAD_INPUT);
}

bool allocate_is_small(int B, int K) { return B <= kSmallSlots && (long long)B * K <= kSmallSlots; }

// One cluster of C CTAs (B and B * K are at most 1024 C), launched behind the
// previous kernel as launch_after_previous does.  The shared-memory limit is
// raised on every call (it and the cluster attribute: at most 0.3 us of an 8.5 us
// call): a note per device that it has been would be stale after a device reset.
template <int C>
static cudaError_t launch_cluster(const AllocLaunch& p, cudaStream_t stream) {
  cudaError_t err = cudaFuncSetAttribute(allocate_cluster_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(ClusterSmem));
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(kAllocThreads);
  cfg.dynamicSmemBytes = sizeof(ClusterSmem);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim = {C, 1, 1};
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  err = cudaLaunchKernelEx(&cfg, allocate_cluster_kernel<C>, p);
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_allocate(const AllocLaunch& p, cudaStream_t stream) {
  cudaError_t err;
  if (allocate_is_small(p.B, p.K)) {
    err = launch_after_previous(allocate_small_kernel, dim3(1), dim3(kAllocThreads), 0, stream, p);
    return err != cudaSuccess ? err : cudaGetLastError();
  }
  const int slots = std::max(p.B * p.K, p.B);  // > kSlots here
  if (slots <= 2 * kSlots) return launch_cluster<2>(p, stream);
  if (slots <= 4 * kSlots) return launch_cluster<4>(p, stream);
  return launch_cluster<8>(p, stream);
}

}  // namespace spec
