// adt_tree_expand: one layer of EAGLE-2-style dynamic draft-tree growth
// (Sec. 3.1, last paragraph; Fig. 5; node score Eq. 4 in the log domain), and
// adt_tree_rerank: the final top-N tree (Eq. 4 and the sentence after it).
//
// Expand is one launch of F thread-block clusters, one per frontier row; the
// C <= 8 CTAs of a cluster split the row's vocabulary.  Each CTA loads its
// share into registers, eight logits a thread, or stages it in shared memory
// with one bulk copy where it has more (x / T in fp32, round-to-nearest
// division).  A first pass keeps each thread's largest value; the k-th
// largest of the 32 warp maxima (64 half-warp maxima for k > 32) bounds the
// CTA's top k from below; a second pass sums the exponentials against the
// CTA's maximum and gathers the few selection keys (value order, then lower
// index) at or above the bound, which are ranked by counting.  The CTAs push
// their lists into the cluster's first CTA (asynchronous stores that complete
// on its mbarrier); it ranks them, forms the row's log-sum-exp and writes the
// row's children (log-probability against it in double-float, rounded once).
// The first CTA of the last row to finish (atomic ticket) ranks the next
// frontier across all rows.  Every selection of more than 128 keys first
// bounds them the same way (64 group maxima), so that only about as many as
// are wanted get ranked.
//
// A call is bound by the latency of that chain of phases, not by its bytes
// (2.1 MB at F = 8, V = 65536: 0.3 us of HBM time).  Back-to-back calls in a
// graph: 5.6 us at F = 8, V = 65536, k = 8 and 4.0 us at F = 1; 10.4 us at
// F = 39, V = 16384, k = 39 under guidance.  (With a bound that let half of a
// CTA's logits through for k > 32, each of them inserted in sorted lists, the
// last took 221.7 us.)
#include "adt_common.cuh"
#include "dfloat.cuh"
#include "sm100.cuh"

namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxK = 64;
constexpr int kMaxKeep = 1024;
constexpr int kMaxCluster = 8;
constexpr int kTile = 32768;            // logits staged in shared memory at a time
constexpr int kTileGuided = kTile / 2;  // under guidance (two rows)
constexpr int kRegValues = 8;           // logits a thread of the register path holds
constexpr uint32_t kWaitLimit = 1u << 22;
constexpr int kCandCap = 1024;          // a CTA's candidate buffer (also the cross-row keys)
constexpr float kLog2e = 1.44269504088896340736f;
constexpr float kLargeRow = 1048576.f;  // see pass 2 of expand_kernel

struct ExpandParams {
  const float* logits;
  const float* logits_u;  // classifier-free guidance: unconditional rows (same ld), else NULL
  float cfg;              // guidance scale
  int64_t ld;
  const float* fscore;
  const int32_t* fid;
  int F, V, k, k_keep;
  float T;
  int use_T;
  int32_t id_base;
  int32_t* ctok;
  float* clogp;
  float* cscore;
  int32_t* cpar;
  int32_t* keep;
  float* nscore;
  int32_t* nid;
  uint64_t* cross_keys;   // [F*k]
  unsigned* all_ticket;   // [1]
  unsigned* err;
  int tile;               // kTile or kTileGuided
};

// Entries greater than key in a descending list of n keys.
__device__ __forceinline__ int count_greater(const uint64_t* list, int n, uint64_t key) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (list[mid] > key)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// Top k of nl descending lists (list l at lists + l * stride, its first len
// entries; 0 pads) into out[0..k), which the caller zeroed.  Keys are
// distinct, so an entry's rank is its index plus the entries greater than it
// in the other lists.
__device__ void merge_topk(const uint64_t* lists, int nl, int stride, int len, int k, uint64_t* out) {
  const int lk = min(len, k);
  for (int c = threadIdx.x; c < nl * lk; c += kThreads) {
    const int l = c / lk, j = c % lk;
    const uint64_t key = lists[l * stride + j];
    if (key == 0ull) continue;
    int rank = j;
    for (int l2 = 0; l2 < nl && rank < k; ++l2)
      if (l2 != l) rank += count_greater(lists + l2 * stride, lk, key);
    if (rank < k) out[rank] = key;
  }
}

// Collects the keys >= thr (exactly `count` of them) into sel[] and sorts
// them in descending order (padding with 0 up to a power of two).
template <class KeyAt>
__device__ void collect_sorted(KeyAt key_at, int n, uint64_t thr, int count, uint64_t* sel,
                               unsigned* s_cnt) {
  const int P = adt::next_pow2(count);
  for (int i = threadIdx.x; i < P; i += kThreads) sel[i] = 0ull;
  if (threadIdx.x == 0) *s_cnt = 0u;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += kThreads) {
    const uint64_t key = key_at(i);
    if (key >= thr && key != 0ull) {
      const unsigned slot = atomicAdd(s_cnt, 1u);
      if (slot < static_cast<unsigned>(P)) sel[slot] = key;
    }
  }
  __syncthreads();
  adt::block_bitonic_sort_desc<kThreads>(sel, P);
}

// The k (<= 64) largest keys a warp is offered, kept sorted by insertion:
// lane i holds entries i (a) and i + 32 (b); 0 marks an empty entry.  Used
// only when a warp's candidate buffer overflows (inputs with very many keys
// at or above the warp's bound).
struct WarpTopK {
  uint64_t a = 0, b = 0;
  __device__ __forceinline__ uint64_t threshold(int k) const {
    const int i = k - 1;
    return __shfl_sync(adt::kFullMask, i < 32 ? a : b, i & 31);
  }
  __device__ __forceinline__ void insert(uint64_t key, int k, int lane) {
    const int pos = __popc(__ballot_sync(adt::kFullMask, a > key)) + __popc(__ballot_sync(adt::kFullMask, b > key));
    if (pos >= k) return;
    const uint64_t up_a = __shfl_up_sync(adt::kFullMask, a, 1);
    const uint64_t up_b = __shfl_up_sync(adt::kFullMask, b, 1);
    const uint64_t a31 = __shfl_sync(adt::kFullMask, a, 31);
    const int ia = lane, ib = lane + 32;
    const uint64_t na = ia < pos ? a : (ia == pos ? key : up_a);
    const uint64_t nb = ib < pos ? b : (ib == pos ? key : (lane == 0 ? a31 : up_b));
    a = ia < k ? na : 0ull;
    b = ib < k ? nb : 0ull;
  }
  __device__ __forceinline__ void offer(uint64_t key, int k, int lane, uint64_t& thr) {
    unsigned m = __ballot_sync(adt::kFullMask, key > thr);
    while (m) {
      const int src = __ffs(m) - 1;
      insert(__shfl_sync(adt::kFullMask, key, src), k, lane);
      thr = threshold(k);
      m &= m - 1;
      m &= __ballot_sync(adt::kFullMask, key > thr);
    }
  }
};

// Stages logits [t0, t1) of a row (t0 a multiple of 4; rows start 16-byte
// aligned and ld is a multiple of 4) in shared memory with one bulk copy
// (two with guidance: the unconditional row goes to vals_u), waiting with a
// bound; then forms u + s (c - u) under guidance and divides by the
// temperature, in place (kPlain: neither).  Block-wide.
template <bool kPlain>
__device__ __forceinline__ bool stage_tile(float* vals, float* vals_u, const float* row, const float* row_u, int t0, int t1,
                           const ExpandParams& p, uint64_t* bar, uint32_t& phase) {
  const int n = t1 - t0;
  if (threadIdx.x == 0 && n > 0) {
    const uint32_t bytes = static_cast<uint32_t>((n + 3) / 4 * 16);
    sm100::mbar_arrive_expect_tx(sm100::smem_addr(bar), !kPlain && row_u ? 2 * bytes : bytes);
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
            sm100::smem_addr(vals)),
        "l"(row + t0), "r"(bytes), "r"(sm100::smem_addr(bar))
        : "memory");
    if (!kPlain && row_u)
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
              sm100::smem_addr(vals_u)),
          "l"(row_u + t0), "r"(bytes), "r"(sm100::smem_addr(bar))
          : "memory");
  }
  bool ok = true;
  if (n > 0) {
    ok = sm100::mbar_wait_bounded(sm100::smem_addr(bar), phase, kWaitLimit);
    phase ^= 1u;
  }
  if (!kPlain && (row_u || p.use_T)) {
    for (int i = threadIdx.x; i < n; i += kThreads) {
      float x = vals[i];
      if (row_u) x = adt::cfg_combine(x, vals_u[i], p.cfg);
      if (p.use_T) x = __fdiv_rn(x, p.T);
      vals[i] = x;
    }
  }
  __syncthreads();
  return ok;
}

// 2^x with the hardware approximation (flush-to-zero); 2^-inf = 0.
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}

// out[rank] = key for the k largest of the n (<= kThreads / T) distinct
// nonzero keys in keys[0..n) (0 entries skipped); out[] zeroed by the caller.
// Block-wide: T threads per key, each counting the keys above it among every
// T-th of the others, the counts summed by shuffles within the group.
template <int T>
__device__ __forceinline__ void rank_select_by(const uint64_t* keys, int n, int k, uint64_t* out) {
  const int i = threadIdx.x / T, s = threadIdx.x % T;
  const uint64_t key = i < n ? keys[i] : 0ull;
  int c = 0;
  if constexpr (T == 16) {  // n <= 64
#pragma unroll
    for (int j = 0; j < 4; ++j) c += (s + 16 * j < n && keys[s + 16 * j] > key) ? 1 : 0;
  } else {
#pragma unroll 4
    for (int o = s; o < n; o += T) c += keys[o] > key ? 1 : 0;
  }
#pragma unroll
  for (int off = T / 2; off > 0; off >>= 1) c += __shfl_xor_sync(adt::kFullMask, c, off);
  if (s == 0 && key != 0ull && c < k) out[c] = key;
}

// The largest power of two of threads per key that covers all n <= kThreads
// keys at once (64 keys: 4 comparisons a thread, 128: 16, 256: 64).  Not
// inlined, nor is the bounded selection: the calls with few keys (k = 8) run
// past one copy of this code instead of three (an expansion call is too short
// to hide the instruction fetches).
__device__ __noinline__ void rank_select(const uint64_t* keys, int n, int k, uint64_t* out) {
  if (n <= kThreads / 8)
    rank_select_by<8>(keys, n, k, out);
  else if (n <= kThreads / 4)
    rank_select_by<4>(keys, n, k, out);
  else if (n <= kThreads / 2)
    rank_select_by<2>(keys, n, k, out);
  else
    rank_select_by<1>(keys, n, k, out);
}

// Sixty-four groups of 16 threads hold one value each; the rank of a group's
// value among them (the groups with a larger one, ties to the lower group
// when `ties`), in every thread of the group.
template <bool ties, class T>
__device__ __noinline__ int rank_of_64(const T* v) {
  static_assert(kThreads == 64 * 16, "16 threads for each of 64 values");
  const int g = threadIdx.x >> 4, s = threadIdx.x & 15;
  const T mine = v[g];
  int c = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int o = s + 16 * j;
    const T x = v[o];
    c += (x > mine || (ties && x == mine && o < g)) ? 1 : 0;
  }
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) c += __shfl_xor_sync(adt::kFullMask, c, off);
  return c;
}

struct SelectScratch {
  uint64_t group[64];
  uint64_t bound;
  unsigned count;
};

// out[rank] = key for the k (<= 64) largest of the distinct keys key_at(0..n)
// (0 entries skipped); out[] zeroed by the caller.  The k-th largest of 64
// group maxima (key i belongs to group i % 64, so that runs of large keys
// spread over the groups) bounds the k largest from below; the keys at or
// above it, about 64 ln(64 / (64 - k)) of n in no particular order, are
// gathered in list[kCandCap] and ranked against each other.  False, and
// nothing written, when more than kCandCap keys reach the bound.  Block-wide.
template <class KeyAt>
__device__ bool bound_select(KeyAt key_at, int n, int k, SelectScratch* sc, uint64_t* list, uint64_t* out) {
  const int tid = threadIdx.x;
  uint64_t mx = 0ull;
  for (int i = (tid >> 4) + 64 * (tid & 15); i < n; i += kThreads) {
    const uint64_t key = key_at(i);
    mx = key > mx ? key : mx;
  }
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) {
    const uint64_t o = __shfl_xor_sync(adt::kFullMask, mx, off);
    mx = o > mx ? o : mx;
  }
  if ((tid & 15) == 0) sc->group[tid >> 4] = mx;
  if (tid == 0) {
    sc->bound = 0ull;  // kept when fewer than k groups hold a key
    sc->count = 0u;
  }
  __syncthreads();
  const int rk = rank_of_64<false>(sc->group);
  if ((tid & 15) == 0 && rk == k - 1 && mx != 0ull) sc->bound = mx;
  __syncthreads();
  const uint64_t bound = sc->bound;
  for (int i = tid; i < n; i += kThreads) {
    const uint64_t key = key_at(i);
    if (key >= bound && key != 0ull) {
      const unsigned pos = atomicAdd(&sc->count, 1u);
      if (pos < static_cast<unsigned>(kCandCap)) list[pos] = key;
    }
  }
  __syncthreads();
  const int cnt = static_cast<int>(sc->count);
  if (cnt > kCandCap) return false;
  rank_select(list, cnt, k, out);
  return true;
}

// The same for n <= kCandCap keys in shared memory: up to kDirectRank of them
// are ranked as they are (two barriers less).
constexpr int kDirectRank = 128;

__device__ __noinline__ void select_many(const uint64_t* keys, int n, int k, SelectScratch* sc, uint64_t* list,
                                         uint64_t* out) {
  if (n <= kDirectRank)
    rank_select(keys, n, k, out);
  else
    (void)bound_select([&](int i) { return keys[i]; }, n, k, sc, list, out);
}

__device__ __forceinline__ void select_shared(const uint64_t* keys, int n, int k, SelectScratch* sc, uint64_t* list,
                                              uint64_t* out) {
  if (n <= kThreads / 16)
    rank_select_by<16>(keys, n, k, out);
  else
    select_many(keys, n, k, sc, list, out);
}

// kNarrow: at most 8 children per row, a CTA's share of the row in one tile,
// and at most 64 cross-row keys or no next frontier (the 7B-shape draft).
// kPlain: no guidance, temperature 1.
// The paths it leaves out are only code there, but a call is a chain of short
// phases and each one fetched past them: with all of them a call at F = 8,
// V = 65536, k = 8 took 0.4 us longer.
// kRegs: the CTA's share is held in registers, from coalesced loads.  Staged in
// shared memory instead (a bulk copy, its mbarrier, two passes of loads) the
// calls took 6.3 against 5.6 us (F = 8, V = 65536, k = 8), 4.6 / 4.0 (F = 1),
// 9.7 / 8.1 (F = 13, k = 13) and 12.3 / 10.4 (F = 39, V = 16384, k = 39,
// guided).  A thread takes pairs: with vectors of four a share of 2048 logits
// lies in half the warps, and their maxima bound a large k by nothing.
template <bool kNarrow, bool kPlain, bool kRegs>
__global__ void __launch_bounds__(kThreads, 1) expand_kernel(const ExpandParams p) {
  extern __shared__ __align__(16) float vals[];    // [min(per, tile)] staged logits (x2 with guidance)
  __shared__ uint64_t cand[kCandCap];              // keys at or above the CTA's bound
  __shared__ uint64_t wl[kWarps][kMaxK];           // overflow path: each warp's top k
  __shared__ float s_mw[kWarps], s_sw[kWarps];
  __shared__ float s_hw[2 * kWarps];               // half-warp maxima (k > 32)
  __shared__ SelectScratch sel_s;
  __shared__ float s_B, s_M;
  __shared__ unsigned s_cnt;
  __shared__ uint64_t ctl[kMaxK];                  // this CTA's top k
  __shared__ uint64_t cl_keys[kMaxCluster * kMaxK];  // first CTA of the cluster: every CTA's k keys
  __shared__ float2 cl_ms[kMaxCluster];
  __shared__ uint64_t rowl[kMaxK];
  __shared__ adt::RadixScratch rs;
  __shared__ __align__(8) uint64_t s_bar, s_push;
  __shared__ int s_last;
  __shared__ float2 s_lse;  // hi, lo
  uint64_t* cross_s = cand;  // cross-row keys (reuses the candidate buffer)
  uint64_t* sel = cand;      // radix path [kMaxKeep]

  const int rank = blockIdx.x, C = gridDim.x, r = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = p.k;
  // Shared-memory set-up before the dependency wait (it reads nothing an
  // earlier kernel writes): after the wait the first bulk copy goes out at once.
  for (int i = tid; i < kMaxK; i += kThreads) ctl[i] = 0ull;
  if (tid == 0) {
    s_cnt = 0u;
    if (!kRegs) sm100::mbar_init(sm100::smem_addr(&s_bar), 1);
    sm100::mbar_init(sm100::smem_addr(&s_push), 1);
    sm100::fence_mbar_init();
  }
  __syncthreads();
  sm100::cluster_arrive_release();  // the mbarriers are there: waited for before the push
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  // This CTA's share of the row: [c0, c1), c0 a multiple of 4.
  const int per = (((p.V + C - 1) / C) + 3) & ~3;
  const int c0 = min(p.V, rank * per), c1 = min(p.V, c0 + per);
  const int tile = kNarrow || kRegs ? per : p.tile;
  const int ntiles = kNarrow || kRegs ? 1 : (c1 - c0 + tile - 1) / tile;
  const float* row = p.logits + static_cast<int64_t>(r) * p.ld;
  const float* row_u = p.logits_u ? p.logits_u + static_cast<int64_t>(r) * p.ld : nullptr;
  float xr[kRegs ? kRegValues : 1];
  auto reg_index = [&](int e) { return 2 * (tid + kThreads * (e / 2)) + e % 2; };  // of xr[e] in the share
  if constexpr (kRegs) {
    auto load = [&](const float* src, float* dst) {
#pragma unroll
      for (int u = 0; u < kRegValues / 2; ++u) {
        const int i = reg_index(2 * u);
        const float2 x = i < c1 - c0 ? __ldcg(reinterpret_cast<const float2*>(src + c0 + i))
                                     : make_float2(-INFINITY, -INFINITY);
        dst[2 * u] = x.x;
        dst[2 * u + 1] = x.y;
      }
    };
    load(row, xr);
    if constexpr (!kPlain) {
      if (row_u) {
        float xu[kRegValues];
        load(row_u, xu);
#pragma unroll
        for (int e = 0; e < kRegValues; ++e) xr[e] = adt::cfg_combine(xr[e], xu[e], p.cfg);
      }
      if (p.use_T) {
#pragma unroll
        for (int e = 0; e < kRegValues; ++e) xr[e] = __fdiv_rn(xr[e], p.T);
      }
    }
    // Past the share's end (its last pair may hold one logit): no value.
#pragma unroll
    for (int e = 0; e < kRegValues; ++e)
      if (reg_index(e) >= c1 - c0) xr[e] = -INFINITY;
  }
  float* vals_u = vals + min(per, tile);  // used only with guidance

  // The row's frontier score and id, read now by the threads that write the
  // children at the end: the loads' latency hides behind the passes.
  const bool writer = rank == 0 && tid < K;
  const float f_score = writer ? p.fscore[r] : 0.f;
  const int32_t f_id = writer ? (p.fid ? p.fid[r] : r) : 0;
  uint32_t phase = 0;
  bool ok = true;

  // Pass 1: each thread's largest value.  Thread tid takes elements tid,
  // tid + 1024, ... of every tile.
  float v1 = -INFINITY;
  if constexpr (kRegs) {
#pragma unroll
    for (int e = 0; e < kRegValues; ++e) v1 = fmaxf(v1, xr[e]);
  }
  for (int tt = 0; !kRegs && tt < ntiles; ++tt) {
    const int t0 = c0 + tt * tile, t1 = min(c1, t0 + tile);
    if (tt > 0) __syncthreads();  // the previous tile is consumed
    ok &= stage_tile<kPlain>(vals, vals_u, row, row_u, t0, t1, p, &s_bar, phase);
#pragma unroll 8
    for (int i = tid; i < t1 - t0; i += kThreads) v1 = fmaxf(v1, vals[i]);
  }
  if (!ok && tid == 0) adt::raise_error(p.err, ADT_DEVERR_TIMEOUT);
  // The bound B: a value with at least k of the CTA's logits at or above it,
  // so that its k best are among those >= B.  For k <= 32 the k-th largest of
  // the 32 warp maxima (a warp ranks each), for larger k the k-th largest of
  // the 64 half-warp maxima (16 threads rank each): about
  // 32 ln(32 / (32 - k)) or 64 ln(64 / (64 - k)) logits reach it, 60 for
  // k = 39 of a 2048-logit share.
  {
    float hw = v1;
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) hw = fmaxf(hw, __shfl_xor_sync(adt::kFullMask, hw, off));
    const float mw = fmaxf(hw, __shfl_xor_sync(adt::kFullMask, hw, 16));
    if (!kNarrow && (lane & 15) == 0) s_hw[tid >> 4] = hw;
    if (lane == 0) s_mw[warp] = mw;
  }
  __syncthreads();
  if (!kNarrow && K > 32) {
    const int rk = rank_of_64<true>(s_hw);
    if ((tid & 15) == 0 && rk == K - 1) s_B = s_hw[tid >> 4];
  }
  {
    // Warp w ranks the warp maximum w among all (ties to the lower warp).
    const float mine = s_mw[warp], o = s_mw[lane];
    const int rk = __popc(__ballot_sync(adt::kFullMask, o > mine || (o == mine && lane < warp)));
    if (lane == 0 && rk == 0) s_M = mine;
    if (lane == 0 && (kNarrow || K <= 32) && rk == K - 1) s_B = mine;
  }
  __syncthreads();
  const float B = s_B, M = s_M;
  // Pass 2: sum of exp(x - M) as 2^(x log2 e - Ml), Ml = M log2 e rounded (the
  // rounding, common to the CTA's terms, is taken out of the sum: 0.06 at
  // most).  Of a share whose maximum is 2^20 or more in magnitude, as 2^((x -
  // M) log2 e), the difference exact near the maximum: its M log2 e can leave
  // fp32, and its rounding the range of 2^x.  (That form for every share,
  // log2 e in two words: the 7B draft 36.8 us against 36.2, its scores' error
  // 4.7e-8 against 3.6e-8.)  Gather the keys of values >= B (few: shared-memory
  // atomics, no per-element vote).
  const bool large = fabsf(M) >= kLargeRow;
  const float Ml = large ? 0.f : M * kLog2e;
  const float Ms = large && M != -INFINITY ? M : 0.f;
  auto term = [&](float x) { return ex2_approx(fmaf(x, kLog2e, -Ml)); };
  auto term_any = [&](float x) { return ex2_approx(fmaf(x - Ms, kLog2e, -Ml)); };  // of any share
  float sa[4] = {0.f, 0.f, 0.f, 0.f};
  if constexpr (kRegs) {
    if (large) {
#pragma unroll
      for (int e = 0; e < kRegValues; ++e) sa[e % 4] += term_any(xr[e]);
    } else {
#pragma unroll
      for (int e = 0; e < kRegValues; ++e) sa[e % 4] += term(xr[e]);
    }
#pragma unroll
    for (int e = 0; e < kRegValues; ++e) {
      const int i = reg_index(e);
      if (xr[e] >= B && i < c1 - c0) {
        const unsigned pos = atomicAdd(&s_cnt, 1u);
        if (pos < static_cast<unsigned>(kCandCap)) cand[pos] = adt::select_key(xr[e], static_cast<uint32_t>(c0 + i));
      }
    }
  }
  for (int tt = 0; !kRegs && tt < ntiles; ++tt) {
    const int t0 = c0 + tt * tile, t1 = min(c1, t0 + tile);
    if (ntiles > 1) {
      __syncthreads();
      ok &= stage_tile<kPlain>(vals, vals_u, row, row_u, t0, t1, p, &s_bar, phase);
    }
    const int n = t1 - t0;
    for (int i0 = tid; i0 < n; i0 += 4 * kThreads) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * kThreads;
        if (i < n) {
          const float x = vals[i];
          sa[u] += term_any(x);
          if (x >= B) {
            const unsigned pos = atomicAdd(&s_cnt, 1u);
            if (pos < static_cast<unsigned>(kCandCap)) cand[pos] = adt::select_key(x, static_cast<uint32_t>(t0 + i));
          }
        }
      }
    }
  }
  {
    const float sw = adt::warp_sum((sa[0] + sa[1]) + (sa[2] + sa[3]));
    if (lane == 0) s_sw[warp] = sw;
  }
  __syncthreads();
  const int cnt = static_cast<int>(s_cnt);
  if (cnt <= kCandCap) {
    select_shared(cand, cnt, K, &sel_s, &wl[0][0], ctl);
  } else {
    // Overflow (very many values at or above B): each warp keeps its k
    // largest by insertion in a third pass, then the lists merge.
    for (int i = tid; i < kWarps * kMaxK; i += kThreads) (&wl[0][0])[i] = 0ull;
    const uint64_t kb = B == -INFINITY ? 1ull : adt::select_key(B, 0xffffffffu);  // lowest key of value B
    WarpTopK tk;
    uint64_t thr = 0ull;
    if constexpr (kRegs) {
#pragma unroll
      for (int e = 0; e < kRegValues; ++e) {
        const int i = reg_index(e);
        if (i < c1 - c0) vals[i] = xr[e];
      }
      __syncthreads();
    }
    for (int tt = 0; tt < ntiles; ++tt) {
      const int t0 = c0 + tt * tile, t1 = min(c1, t0 + tile);
      if (ntiles > 1) {
        __syncthreads();
        ok &= stage_tile<kPlain>(vals, vals_u, row, row_u, t0, t1, p, &s_bar, phase);
      }
      const int n = t1 - t0;
      for (int base = warp * 32; base < n; base += kThreads) {
        const int i = base + lane;
        const uint64_t key = i < n ? adt::select_key(vals[i], static_cast<uint32_t>(t0 + i)) : 0ull;
        tk.offer(key >= kb ? key : 0ull, K, lane, thr);
      }
    }
    __syncthreads();
    wl[warp][lane] = tk.a;
    wl[warp][lane + 32] = tk.b;
    __syncthreads();
    merge_topk(&wl[0][0], kWarps, kMaxK, K, K, ctl);
  }
  __syncthreads();
  if (!ok && tid == 0) adt::raise_error(p.err, ADT_DEVERR_TIMEOUT);  // a restaged tile's wait
  // This CTA's top k and (max, sum of exponentials), to the cluster's first
  // CTA: asynchronous stores that complete on its mbarrier, one way.  (With a
  // cluster barrier in their place, the bound ranked by one warp and the
  // scores in fp64, the 7B draft, six calls and the rerank, took 42.2 us
  // against 40.4 us.)
  __syncwarp();
  sm100::cluster_wait_acquire();
  if (warp == 0) {
    const uint32_t bar = sm100::mapa_shared(sm100::smem_addr(&s_push), 0);
    auto push = [&](const void* local, uint64_t v) {
      asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];\n" ::"r"(
                       sm100::mapa_shared(sm100::smem_addr(local), 0)),
                   "l"(v), "r"(bar)
                   : "memory");
    };
    if (lane < K) push(&cl_keys[rank * K + lane], ctl[lane]);
    if (lane + 32 < K) push(&cl_keys[rank * K + lane + 32], ctl[lane + 32]);
    const float S = adt::warp_sum(s_sw[lane]);  // kWarps == 32
    const float off = large ? 0.f : fmaf(M, kLog2e, -Ml);  // exact: every term is 2^off too large
    if (lane == 0)
      push(&cl_ms[rank], static_cast<uint64_t>(__float_as_uint(S * ex2_approx(-off))) << 32 | __float_as_uint(M));
  }
  // The next kernel in the stream may launch now.  (Released right after the
  // wait, a graph of six calls, F = 1, then 8; V = 65536, k = 8, and the rerank
  // took 33.9 us against 33.5; released with the children, 33.7.)
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  if (rank != 0) return;

  // ---- first CTA of row r: the row's top k and log-sum-exp, its children.
  for (int i = tid; i < kMaxK; i += kThreads) rowl[i] = 0ull;
  if (tid == 0)
    sm100::mbar_arrive_expect_tx(sm100::smem_addr(&s_push), static_cast<uint32_t>(C * (K + 1) * sizeof(uint64_t)));
  const bool pushed = sm100::mbar_wait_bounded(sm100::smem_addr(&s_push), 0, kWaitLimit);
  if (warp == 0) {  // lane c takes CTA c's (max, sum); C <= 8
    const float2 ms = lane < C ? cl_ms[lane] : make_float2(-INFINITY, 0.f);
    const float Mr = adt::warp_max(ms.x);
    const float S = adt::warp_sum(ms.x == -INFINITY ? 0.f : ms.y * ex2_approx((ms.x - Mr) * kLog2e));
    if (lane == 0) {
      const dfl::df t = dfl::two_sum(Mr, logf(S));
      s_lse = make_float2(t.hi, t.lo);
    }
  }
  if (__syncthreads_or(!pushed)) {  // late pushes still need this CTA: it stays until every peer has left
    if (tid == 0) adt::raise_error(p.err, ADT_DEVERR_TIMEOUT);
    sm100::cluster_arrive_release();
    sm100::cluster_wait_acquire();
  }
  if constexpr (kNarrow)
    rank_select_by<16>(cl_keys, C * K, K, rowl);
  else
    select_shared(cl_keys, C * K, K, &sel_s, cand, rowl);
  __syncthreads();
  if (writer) {
    const uint64_t key = rowl[tid];
    // x - log-sum-exp and the score in double-float (an fp64 operation takes
    // as long as dozens of these), each rounded to fp32 once; in fp64 where
    // that leaves fp32's range (infinities, masks of fp32's lowest value).
    const float x = adt::select_key_value(key);
    const dfl::df lpd = dfl::df_add(dfl::df{x, 0.f}, dfl::df{-s_lse.x, -s_lse.y});
    float lp = lpd.hi, score = dfl::df_add(dfl::df{f_score, 0.f}, lpd).hi;
    if (!isfinite(lp) || !isfinite(score)) {
      const double l = static_cast<double>(x) - (isfinite(s_lse.y) ? static_cast<double>(s_lse.x) + s_lse.y : s_lse.x);
      lp = static_cast<float>(l);
      score = static_cast<float>(f_score + l);
    }
    const int64_t c = static_cast<int64_t>(r) * K + tid;
    p.ctok[c] = static_cast<int32_t>(adt::select_key_index(key));
    if (p.clogp) p.clogp[c] = lp;
    p.cscore[c] = score;
    p.cpar[c] = f_id;
    if (!p.keep) {
      // No next frontier wanted (the tree's last layer).
    } else if (p.F == 1) {
      // One row: its children are already in score order (the score grows
      // with the log-probability; ties keep the lower index, as the
      // cross-row ranking would), so the next frontier is their first k_keep.
      if (tid < p.k_keep) {
        p.keep[tid] = static_cast<int32_t>(c);
        if (p.nscore) p.nscore[tid] = score;
        if (p.nid) p.nid[tid] = p.id_base + static_cast<int32_t>(c);
      }
    } else {
      p.cross_keys[c] = adt::select_key(score, static_cast<uint32_t>(c));
    }
  }
  if (p.F == 1 || !p.keep) return;
  // The row's cross keys are written (CTA order); the ticket's release
  // publishes them at device scope and its acquire, in the last row, makes
  // every row's keys visible.
  __syncthreads();
  if (tid == 0) s_last = adt::atomic_add_acq_rel_gpu(p.all_ticket, 1u) == static_cast<unsigned>(p.F - 1);
  __syncthreads();
  if (!s_last) return;

  // ---- last row: next frontier across all rows.
  const int nc = p.F * K;
  auto cross_key = [&](int i) { return __ldcg(p.cross_keys + i); };
  bool done = kNarrow;
  if (kNarrow || p.k_keep <= kMaxK) {
    for (int i = tid; i < kMaxK; i += kThreads) rowl[i] = 0ull;
    if constexpr (kNarrow) {
      if (tid < nc) cross_s[tid] = cross_key(tid);
      __syncthreads();
      rank_select_by<16>(cross_s, nc, p.k_keep, rowl);
    } else if (nc <= kCandCap) {
      for (int i = tid; i < nc; i += kThreads) cross_s[i] = cross_key(i);
      __syncthreads();
      select_shared(cross_s, nc, p.k_keep, &sel_s, &wl[0][0], rowl);
      done = true;
    } else {
      __syncthreads();
      done = bound_select(cross_key, nc, p.k_keep, &sel_s, cross_s, rowl);
    }
    __syncthreads();
    if (done && tid < p.k_keep) {
      const uint64_t key = rowl[tid];
      const int32_t c = static_cast<int32_t>(adt::select_key_index(key));
      p.keep[tid] = c;
      if (p.nscore) p.nscore[tid] = adt::select_key_value(key);
      if (p.nid) p.nid[tid] = p.id_base + c;
    }
  }
  if (!kNarrow && !done) {
    const uint64_t thr3 = adt::block_topk_threshold<kThreads>(cross_key, nc, p.k_keep, &rs);
    collect_sorted(cross_key, nc, thr3, p.k_keep, sel, &s_cnt);
    for (int j = tid; j < p.k_keep; j += kThreads) {
      const uint64_t key = sel[j];
      const int32_t c = static_cast<int32_t>(adt::select_key_index(key));
      p.keep[j] = c;
      if (p.nscore) p.nscore[j] = adt::select_key_value(key);
      if (p.nid) p.nid[j] = p.id_base + c;
    }
  }
  if (tid == 0) *p.all_ticket = 0u;
}

// CTAs per row (the cluster size).  A share of 8192 logits is the most that
// registers hold; with up to 8 children half of that is a little faster, with
// more of them every CTA more means a longer list to rank (us with 8, 4 and 2
// CTAs at V = 16384: F = 8, k = 8 5.6, 5.7, 5.7; F = 13, k = 13 8.0, 7.5, 7.5; F =
// 1, k = 39, guided 6.6, 6.3, 5.5; F = 20, k = 20, no next frontier 8.3, 4.6,
// 4.3).  All rows' clusters run at once: a CTA fills an SM (1024 threads) and
// the GPCs leave a part of the SMs out of a larger cluster's reach, so the
// limit is four fifths of the SMs for those, and all of them for pairs; beyond
// it the rows take two waves (F = 20, V = 65536, 8, 6 and 4 CTAs: 8.8, 6.9, 7.2;
// F = 39 with 4, 3 and 2: 15.0, 9.9, 10.2; F = 76, V = 32768 with 2 and 1: 5.8,
// 7.1, F = 90 11.0, 7.7).  Sizes cut down stay even (F = 39, V = 16384, guided,
// 3 and 2: 12.2 and 10.5).
int expand_cluster(int F, int V, int k, int sm_count) {
  const int share = k <= 8 ? kRegValues * kThreads / 2 : kRegValues * kThreads;
  int c = (V + share - 1) / share;
  const int pairs = V / (2 * kThreads);  // shares that still have a pair of logits for each thread
  if (c < 2) c = pairs < 2 ? 1 : 2;
  if (c > kMaxCluster) c = kMaxCluster;
  const int most = 4 * sm_count / (5 * F);
  if (c > most) c = most >= 2 ? most / 2 * 2 : c > 1 && 2 * F <= sm_count ? 2 : 1;
  return c;
}

// Workspace layout.  The completion counter sits at a fixed offset at the
// start, after a zeroed region kept for layout stability, so calls of any
// shape can share one workspace; the keys after it are rewritten before use.
constexpr int kMaxRows = 4096;

struct ExpandWs {
  size_t all_ticket, cross_keys, total;
};

ExpandWs expand_ws(int F, int V, int k) {
  (void)V;
  ExpandWs w{};
  w.all_ticket = kMaxRows * sizeof(unsigned);
  w.cross_keys = adt::align_up(w.all_ticket + sizeof(unsigned), 256);
  w.total = adt::align_up(w.cross_keys + static_cast<size_t>(F) * k * sizeof(uint64_t), 256);
  return w;
}

// ------------------------------------------------------------------ rerank

constexpr int kRerankThreads = 1024;

struct RerankParams {
  const int32_t* ctok;
  const float* cscore;
  const int32_t* cpar;
  int C;
  const int32_t* root;
  int n_nodes;
  int32_t* tokens;
  int32_t* parents;
  int32_t* cand_index;
  int32_t* depth;
  unsigned* err;
};

// Rerank of any pool.  The scores are mapped, order kept, to kRerankBins
// bins over their range; a histogram gives the bin that holds the
// (n_nodes - 1)-th best, every candidate of a better bin is selected, and the
// few of that bin are ranked against each other.  More than kRerankFew there
// -- equal scores, or a few far from the rest that stretch the range -- are
// binned again over the range of their order keys, as often as it takes (a
// binning narrows it 1024 times), and by index once they are all equal; in
// pools too large for registers a radix select finds the threshold key instead,
// unless all scores are equal.  Pools of up to kRerankDirect are ranked as they
// are, and a pool that is selected whole is not ranked at all.  Node ids follow
// ascending candidate index (one scan over the warps' counts of all tiles), and
// node maps, parents and depths stay in shared memory.
//
// Bound by latency.  Scores as grown, us: 2.4 at C = 4 to 40 (3.2 by bins), 2.9
// at C = 100, n = 20 and at C = 328, n = 64 (4.4 when every warp's two largest
// keys gave the bound), 3.4 at C = 858, n = 256 (46 with all keys ranked against
// each other), 4.4 at C = 2000, n = 64, 5.8 at C = 3924, n = 256 (6.1 with eight
// scores a thread), 7.3 at C = 6123, 13.4 at C = 12207 and 38 at C = 40000, n = 64
// (5.1, 7.6, 9.4, 14.8 and 37.6 with radix passes over the keys in memory).  With
// one score at fp32's lowest value C = 328, 858, 2000, 6123 and 12207 take 3.8,
// 4.4, 5.4, 8.8 and 13.2, all equal 3.8, 3.9, 5.3, 8.7 and 18 (the crowded bin
// ranked at once, by a warp a key: 9.0, 29, 7.1, 8.3 and 13.8, all equal 8.9, 29,
// 11, 15.7 and 26; before there were bins: 4.4, 46, 6.3, 9.4 and 14.8, all equal
// 3.6, 46, 10, 15.9 and 24.7).  M: scores a thread keeps in registers (1, 2, 4 or
// 8; C <= 1024 M), with M = 1 tokens and parents too; 0: they are read again where
// needed.
constexpr int kRerankBins = 1024;
constexpr int kRerankFew = 256;        // candidates of the threshold bin ranked by counting
constexpr int kRerankDirect = 128;     // pools ranked by counting as they are
constexpr int kRerankMaxC = 65536;
constexpr int kRerankMaxNodes = 4096;
constexpr int kRerankMaxTiles = kRerankMaxC / kRerankThreads;
constexpr int kRerankRegs = 8;

struct RerankShared {
  int par[kRerankMaxNodes];              // a node's candidate index, then its parent's node id
  uint64_t list[kRerankFew], nth;
  int hist[kRerankBins];
  int tot[kRerankMaxTiles * 32];         // selected per (tile, warp), then their exclusive prefix
  float fmax[32], fmin[32];
  uint32_t kmax[32], kmin[32];
  int wsum[32];
  int bin, need, count, nlist, bad;
  adt::RadixScratch rs;
};

// *nth = the want-th best of the n <= kRerankThreads / T distinct keys: T threads
// per key, as in rank_select_by.
template <int T>
__device__ __forceinline__ void rank_nth_by(const uint64_t* keys, int n, int want, uint64_t* nth) {
  const int i = threadIdx.x / T, s = threadIdx.x % T;
  const uint64_t key = i < n ? keys[i] : 0ull;
  int c = 0;
#pragma unroll 4
  for (int o = s; o < n; o += T) c += keys[o] > key ? 1 : 0;
#pragma unroll
  for (int off = T / 2; off > 0; off >>= 1) c += __shfl_xor_sync(adt::kFullMask, c, off);
  if (s == 0 && i < n && c == want - 1) *nth = key;
}

// n <= kRerankFew.
__device__ __noinline__ void rank_nth(const uint64_t* keys, int n, int want, uint64_t* nth) {
  if (n <= kRerankThreads / 8)
    rank_nth_by<8>(keys, n, want, nth);
  else
    rank_nth_by<4>(keys, n, want, nth);
}

// The want-th best of the n keys in the list.  Block-wide.
__device__ __forceinline__ uint64_t rerank_list_threshold(RerankShared& sh, int n, int want) {
  __syncthreads();
  if (n <= kRerankThreads / 16)
    rank_nth_by<16>(sh.list, n, want, &sh.nth);
  else
    rank_nth(sh.list, n, want, &sh.nth);
  __syncthreads();
  return sh.nth;
}

// Inclusive prefix over the warp.
__device__ __forceinline__ int warp_inclusive(int v) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(adt::kFullMask, v, o);
    if ((threadIdx.x & 31) >= o) v += y;
  }
  return v;
}

// Exclusive prefix of one value per thread over the block.
__device__ __forceinline__ int rerank_block_scan(int v, int* wsum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int incl = warp_inclusive(v);
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  const int w = wsum[lane];
  return __shfl_sync(adt::kFullMask, warp_inclusive(w) - w, warp) + incl - v;
}

// The n_nodes - 1 best by score bins: bit m of the result is candidate tid + 1024 m.
// each(f) calls f(m, candidate, score) for every candidate of the thread.
template <int M, class Each>
__device__ __forceinline__ uint64_t rerank_by_bins(Each each, const float* cscore, int C, int need, RerankShared& sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float mx = -INFINITY, mn = INFINITY;
  each([&](int, int, float v) {
    mx = fmaxf(mx, v);
    mn = v > -INFINITY ? fminf(mn, v) : mn;
  });
  mx = adt::warp_max(mx);
  mn = -adt::warp_max(-mn);
  if (lane == 0) {
    sh.fmax[warp] = mx;
    sh.fmin[warp] = mn;
  }
  __syncthreads();
  mx = adt::warp_max(sh.fmax[lane]);
  mn = -adt::warp_max(-sh.fmin[lane]);
  // Non-increasing in the score (each operation rounds monotonically), so a
  // better bin holds better scores only; equal scores (and +0, -0) share one.
  // -inf comes last; a NaN, as in the selection keys, first (last with its sign
  // set).
  const float span = mx - mn;
  const float scale = span > 0.f && span < INFINITY ? (kRerankBins - 1) / span : 0.f;
  auto bin_of = [&](float v) -> int {
    if (v > -INFINITY) return min(kRerankBins - 1, static_cast<int>((mx - v) * scale));
    return __float_as_int(v) < 0 ? kRerankBins - 1 : 0;
  };
  auto find_bin = [&](int want) {  // the bin with the want-th best, from the histogram
    __syncthreads();
    const int h = sh.hist[tid];
    const int before = rerank_block_scan(h, sh.wsum);
    if (before < want && want <= before + h) {
      sh.bin = tid;
      sh.need = want - before;
      sh.count = h;
    }
    __syncthreads();
  };
  each([&](int, int i, float v) {
    if (i < C) atomicAdd(&sh.hist[bin_of(v)], 1);
  });
  find_bin(need);
  const int tbin = sh.bin, tneed = sh.need, tcount = sh.count;
  uint64_t sel = 0ull;
  if (tcount == tneed) {
    each([&](int m, int i, float v) {
      if (i < C && bin_of(v) <= tbin) sel |= 1ull << m;
    });
  } else if (tcount <= kRerankFew) {
    each([&](int m, int i, float v) {
      if (i >= C) return;
      const int bn = bin_of(v);
      if (bn < tbin) sel |= 1ull << m;
      if (bn == tbin) sh.list[atomicAdd(&sh.nlist, 1)] = adt::select_key(v, static_cast<uint32_t>(i));
    });
    const uint64_t thr = rerank_list_threshold(sh, tcount, tneed);
    each([&](int m, int i, float v) {
      if (i < C && bin_of(v) == tbin && adt::select_key(v, static_cast<uint32_t>(i)) >= thr) sel |= 1ull << m;
    });
  } else if (M > 0 || scale == 0.f) {
    // Bit m of `in`: the candidate is in the threshold bin.
    uint64_t in = 0ull;
    each([&](int m, int i, float v) {
      if (i >= C) return;
      const int bn = bin_of(v);
      if (bn < tbin) sel |= 1ull << m;
      if (bn == tbin) in |= 1ull << m;
    });
    auto each_in = [&](auto f) {
      each([&](int m, int i, float v) {
        if ((in >> m) & 1ull) f(m, i, adt::float_order_key(v));
      });
    };
    int want = tneed, count = tcount;
    do {
      uint32_t hi = 0u, lo = ~0u;
      each_in([&](int, int, uint32_t key) {
        hi = max(hi, key);
        lo = min(lo, key);
      });
      hi = __reduce_max_sync(adt::kFullMask, hi);
      lo = __reduce_min_sync(adt::kFullMask, lo);
      if (lane == 0) {
        sh.kmax[warp] = hi;
        sh.kmin[warp] = lo;
      }
      sh.hist[tid] = 0;
      __syncthreads();
      hi = __reduce_max_sync(adt::kFullMask, sh.kmax[lane]);
      lo = __reduce_min_sync(adt::kFullMask, sh.kmin[lane]);
      // Equal keys: bins of consecutive indices, one of at most 64 (C <= 65536).
      const uint32_t range = hi > lo ? hi - lo : static_cast<uint32_t>(C - 1);
      const int shift = max(0, 22 - __clz(range));
      auto key_bin = [&](int i, uint32_t key) -> int {
        return static_cast<int>((hi > lo ? hi - key : static_cast<uint32_t>(i)) >> shift);
      };
      each_in([&](int, int i, uint32_t key) { atomicAdd(&sh.hist[key_bin(i, key)], 1); });
      find_bin(want);
      const int at = sh.bin;
      want = sh.need;
      count = sh.count;
      each_in([&](int m, int i, uint32_t key) {
        const int bn = key_bin(i, key);
        if (bn < at) sel |= 1ull << m;
        if (bn != at) in &= ~(1ull << m);
      });
    } while (count > want && count > kRerankFew);
    uint64_t thr = 0ull;
    if (count > want) {
      each_in([&](int, int i, uint32_t key) {
        sh.list[atomicAdd(&sh.nlist, 1)] = static_cast<uint64_t>(key) << 32 | (0xffffffffu - static_cast<uint32_t>(i));
      });
      thr = rerank_list_threshold(sh, count, want);
    }
    each_in([&](int m, int i, uint32_t key) {
      if ((static_cast<uint64_t>(key) << 32 | (0xffffffffu - static_cast<uint32_t>(i))) >= thr) sel |= 1ull << m;
    });
  } else {
    const uint64_t thr = adt::block_topk_threshold<kRerankThreads>(
        [&](int i) { return adt::select_key(cscore[i], static_cast<uint32_t>(i)); }, C, need, &sh.rs);
    each([&](int m, int i, float v) {
      if (i < C && adt::select_key(v, static_cast<uint32_t>(i)) >= thr) sel |= 1ull << m;
    });
  }
  return sel;
}

template <int M>
__global__ void __launch_bounds__(kRerankThreads, 1) rerank_kernel(const RerankParams p) {
  extern __shared__ uint16_t node_of[];  // [C]: a candidate's node id, 0xFFFF if not selected
  __shared__ RerankShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int need = p.n_nodes - 1, C = p.C;
  const int tiles = (C + kRerankThreads - 1) / kRerankThreads;
  sh.hist[tid] = 0;
  if (tid == 0) {
    sh.nlist = 0;
    sh.bad = 0;
  }
  adt::pdl_wait_then_release();
  if (tid == 0) {
    p.tokens[0] = *p.root;
    p.parents[0] = -1;
    if (p.cand_index) p.cand_index[0] = -1;
    if (p.depth) p.depth[0] = 0;
    sh.par[0] = -1;
  }
  if (need == 0) return;
  float x[M ? M : 1];
  if constexpr (M > 0) {
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const int i = tid + m * kRerankThreads;
      x[m] = i < C ? p.cscore[i] : -INFINITY;
    }
  }
  int tok = 0, parent = 0;  // M = 1: the thread's candidate's, loaded with its score
  if (M == 1 && tid < C) {
    tok = p.ctok[tid];
    parent = p.cpar[tid];
  }
  // f(m, candidate, score) for every candidate of this thread, tile by tile.
  auto each = [&](auto f) {
    if constexpr (M > 0) {
#pragma unroll
      for (int m = 0; m < M; ++m)
        if (m < tiles) f(m, tid + m * kRerankThreads, x[m]);
    } else {
      for (int m = 0; m < tiles; ++m) {
        const int i = tid + m * kRerankThreads;
        f(m, i, i < C ? p.cscore[i] : -INFINITY);
      }
    }
  };
  // Bit m of `sel`: candidate tid + 1024 m is selected.
  uint64_t sel = 0ull;
  if (need == C) {
    each([&](int m, int i, float) {
      if (i < C) sel |= 1ull << m;
    });
  } else if (M == 1 && C <= kRerankDirect) {
    const uint64_t key = adt::select_key(x[0], static_cast<uint32_t>(tid));
    if (tid < C) sh.list[tid] = key;
    const uint64_t thr = rerank_list_threshold(sh, C, need);
    if (tid < C && key >= thr) sel = 1ull;
  } else {
    sel = rerank_by_bins<M>(each, p.cscore, C, need, sh);
  }
  // Node ids in ascending candidate order.
  for (int m = 0; m < tiles; ++m) {
    const unsigned bal = __ballot_sync(adt::kFullMask, (sel >> m) & 1ull);
    if (lane == 0) sh.tot[m * 32 + warp] = __popc(bal);
  }
  __syncthreads();
  int base = 0;  // M = 1: selected in the warps before this one
  if constexpr (M == 1) {
    const int t = sh.tot[lane];
    base = __shfl_sync(adt::kFullMask, warp_inclusive(t) - t, warp);
  } else {
    const int nt = tiles * 32;  // <= 2 kRerankThreads
    const int a = 2 * tid < nt ? sh.tot[2 * tid] : 0, b = 2 * tid + 1 < nt ? sh.tot[2 * tid + 1] : 0;
    const int before = rerank_block_scan(a + b, sh.wsum);
    if (2 * tid < nt) sh.tot[2 * tid] = before;
    if (2 * tid + 1 < nt) sh.tot[2 * tid + 1] = before + a;
    __syncthreads();
  }
  for (int m = 0; m < tiles; ++m) {
    const int i = tid + m * kRerankThreads;
    const bool mine = (sel >> m) & 1ull;
    const unsigned bal = __ballot_sync(adt::kFullMask, mine);
    const int node = 1 + (M == 1 ? base : sh.tot[m * 32 + warp]) + __popc(bal & ((1u << lane) - 1u));
    if (i < C) node_of[i] = mine ? static_cast<uint16_t>(node) : 0xFFFFu;
    if (mine) sh.par[node] = M == 1 ? parent : i;
    if (M == 1 && mine) {
      p.tokens[node] = tok;
      if (p.cand_index) p.cand_index[node] = i;
    }
  }
  __syncthreads();
  for (int node = 1 + tid; node <= need; node += kRerankThreads) {
    int pc = sh.par[node];
    if constexpr (M != 1) {
      const int c = pc;
      pc = p.cpar[c];
      p.tokens[node] = p.ctok[c];
      if (p.cand_index) p.cand_index[node] = c;
    }
    int pr = 0;
    if (pc >= 0) {
      const int of = pc < C ? node_of[pc] : 0xFFFF;
      pr = of;
      if (of == 0xFFFF || of >= node) {
        sh.bad = 1;
        pr = 0;
      }
    }
    sh.par[node] = pr;
    p.parents[node] = pr;
  }
  __syncthreads();
  if (sh.bad && tid == 0) adt::raise_error(p.err, ADT_DEVERR_BAD_TREE);
  if (p.depth) {
    for (int node = 1 + tid; node <= need; node += kRerankThreads) {
      int d = 0, j = node;
      while (j > 0 && d <= need) {
        j = sh.par[j];
        ++d;
      }
      p.depth[node] = d;
    }
  }
}

}  // namespace

static adt_status expand_impl(const float* logits, const float* logits_u, float cfg_scale, int64_t ld,
                              const float* frontier_score, const int32_t* frontier_id, int32_t F, int32_t V,
                              int32_t k_child, int32_t k_keep, float temperature, int32_t child_id_base,
                              int32_t* child_token, float* child_logp, float* child_score,
                              int32_t* child_parent, int32_t* keep_idx, float* next_score, int32_t* next_id,
                              void* workspace, size_t workspace_bytes, void* stream) {
  ADT_REQUIRE(logits && frontier_score && child_token && child_score && child_parent);
  ADT_REQUIRE(keep_idx || (!next_score && !next_id));
  if (logits_u) ADT_REQUIRE(adt::aligned16(logits_u) && cfg_scale > -1e30f && cfg_scale < 1e30f);
  ADT_REQUIRE(F >= 1 && F <= kMaxRows && V >= 1 && V <= (1 << 24));
  ADT_REQUIRE(k_child >= 1 && k_child <= kMaxK && k_child <= V);
  ADT_REQUIRE(k_keep >= 1 && k_keep <= F * k_child && k_keep <= kMaxKeep);
  ADT_REQUIRE(ld >= V && ld % 4 == 0 && adt::aligned16(logits));
  ADT_REQUIRE(temperature > 0.f && temperature < 1e30f);
  const ExpandWs w = expand_ws(F, V, k_child);
  if (!workspace || workspace_bytes < w.total || !adt::aligned16(workspace)) return ADT_ERR_WORKSPACE;
  adt::DeviceInfo info;
  adt_status st = adt::device_info(&info);
  if (st != ADT_OK) return st;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  ExpandParams p;
  p.logits = logits;
  p.logits_u = logits_u;
  p.cfg = cfg_scale;
  p.ld = ld;
  p.fscore = frontier_score;
  p.fid = frontier_id;
  p.F = F;
  p.V = V;
  p.k = k_child;
  p.k_keep = k_keep;
  p.T = temperature;
  p.use_T = temperature != 1.0f;
  p.id_base = child_id_base;
  p.ctok = child_token;
  p.clogp = child_logp;
  p.cscore = child_score;
  p.cpar = child_parent;
  p.keep = keep_idx;
  p.nscore = next_score;
  p.nid = next_id;
  p.cross_keys = reinterpret_cast<uint64_t*>(ws + w.cross_keys);
  p.all_ticket = reinterpret_cast<unsigned*>(ws + w.all_ticket);
  p.err = info.error_word;
  const int C = expand_cluster(F, V, k_child, info.sm_count);
  const int per = ((V + C - 1) / C + 3) & ~3;
  p.tile = logits_u ? kTileGuided : kTile;
  const size_t dyn = static_cast<size_t>(per < p.tile ? per : p.tile) * sizeof(float) * (logits_u ? 2 : 1);
  static unsigned configured[2] = {0u, 0u};  // bit per device (< 64)
  unsigned& word = configured[(info.device >> 5) & 1];
  const unsigned bit = 1u << (info.device & 31);
  if (!(__atomic_load_n(&word, __ATOMIC_ACQUIRE) & bit)) {
    for (auto k : {expand_kernel<true, true, true>, expand_kernel<true, false, true>, expand_kernel<true, true, false>,
                   expand_kernel<true, false, false>, expand_kernel<false, false, true>,
                   expand_kernel<false, false, false>})
      ADT_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        static_cast<int>(kTile * sizeof(float))));
    __atomic_fetch_or(&word, bit, __ATOMIC_ACQ_REL);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.dynamicSmemBytes = dyn;
  cfg.gridDim = dim3(static_cast<unsigned>(C), static_cast<unsigned>(F), 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.stream = adt::as_stream(stream);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(C);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = adt::pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const bool narrow = k_child <= kThreads / 16 / kMaxCluster && per <= p.tile &&
                      (!keep_idx || F * k_child <= kThreads / 16);
  const bool plain = !logits_u && !p.use_T;
  // A pair in every thread (the bound needs values in all warps) up to eight
  // logits a thread.
  const bool regs = per >= 2 * kThreads && per <= kRegValues * kThreads;
  auto kernel = narrow ? (plain ? expand_kernel<true, true, false> : expand_kernel<true, false, false>)
                       : expand_kernel<false, false, false>;
  if (regs)
    kernel = narrow ? (plain ? expand_kernel<true, true, true> : expand_kernel<true, false, true>)
                    : expand_kernel<false, false, true>;
  ADT_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, p));
  return adt::launch_status();
}

extern "C" {

size_t adt_tree_expand_workspace_size(int32_t F, int32_t V, int32_t k_child) {
  if (F < 1 || V < 1 || k_child < 1) return 0;
  return expand_ws(F, V, k_child).total;
}

adt_status adt_tree_expand(const float* logits, int64_t ld, const float* frontier_score,
                           const int32_t* frontier_id, int32_t F, int32_t V, int32_t k_child,
                           int32_t k_keep, float temperature, int32_t child_id_base,
                           int32_t* child_token, float* child_logp, float* child_score,
                           int32_t* child_parent, int32_t* keep_idx, float* next_score,
                           int32_t* next_id, void* workspace, size_t workspace_bytes,
                           void* stream) {
  adt::TraceRange trace_("adt_tree_expand");
  return expand_impl(logits, nullptr, 0.f, ld, frontier_score, frontier_id, F, V, k_child, k_keep, temperature,
                     child_id_base, child_token, child_logp, child_score, child_parent, keep_idx, next_score,
                     next_id, workspace, workspace_bytes, stream);
}

adt_status adt_tree_expand_cfg(const float* logits_cond, const float* logits_uncond, int64_t ld,
                               float cfg_scale, const float* frontier_score, const int32_t* frontier_id,
                               int32_t F, int32_t V, int32_t k_child, int32_t k_keep, float temperature,
                               int32_t child_id_base, int32_t* child_token, float* child_logp,
                               float* child_score, int32_t* child_parent, int32_t* keep_idx,
                               float* next_score, int32_t* next_id, void* workspace,
                               size_t workspace_bytes, void* stream) {
  adt::TraceRange trace_("adt_tree_expand_cfg");
  ADT_REQUIRE(logits_uncond);
  return expand_impl(logits_cond, logits_uncond, cfg_scale, ld, frontier_score, frontier_id, F, V, k_child,
                     k_keep, temperature, child_id_base, child_token, child_logp, child_score, child_parent,
                     keep_idx, next_score, next_id, workspace, workspace_bytes, stream);
}

// The kernel keeps its scratch in shared memory; callers go on passing what the
// ABI asks for.
size_t adt_tree_rerank_workspace_size(int32_t C) {
  if (C < 1) return 0;
  return adt::align_up(static_cast<size_t>(C) * sizeof(int32_t), 256) +
         adt::align_up(4097 * sizeof(int32_t), 256);
}

adt_status adt_tree_rerank(const int32_t* cand_token, const float* cand_score,
                           const int32_t* cand_parent, int32_t C, const int32_t* root_token,
                           int32_t n_nodes, int32_t* tokens, int32_t* parents,
                           int32_t* cand_index, int32_t* depth, void* workspace,
                           size_t workspace_bytes, void* stream) {
  adt::TraceRange trace_("adt_tree_rerank");
  ADT_REQUIRE(cand_token && cand_score && cand_parent && root_token && tokens && parents);
  ADT_REQUIRE(C >= 1 && C <= kRerankMaxC && n_nodes >= 1 && n_nodes <= C + 1 && n_nodes <= kRerankMaxNodes);
  const size_t need = adt_tree_rerank_workspace_size(C);
  if (!workspace || workspace_bytes < need || !adt::aligned16(workspace)) return ADT_ERR_WORKSPACE;
  adt::DeviceInfo info;
  adt_status st = adt::device_info(&info);
  if (st != ADT_OK) return st;
  RerankParams p;
  p.ctok = cand_token;
  p.cscore = cand_score;
  p.cpar = cand_parent;
  p.C = C;
  p.root = root_token;
  p.n_nodes = n_nodes;
  p.tokens = tokens;
  p.parents = parents;
  p.cand_index = cand_index;
  p.depth = depth;
  p.err = info.error_word;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1, 1, 1);
  cfg.blockDim = dim3(kRerankThreads, 1, 1);
  cfg.stream = adt::as_stream(stream);
  cudaLaunchAttribute attr[1] = {adt::pdl_attribute()};
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  static unsigned configured[2] = {0u, 0u};  // bit per device (< 64)
  unsigned& word = configured[(info.device >> 5) & 1];
  const unsigned bit = 1u << (info.device & 31);
  if (!(__atomic_load_n(&word, __ATOMIC_ACQUIRE) & bit)) {
    ADT_CUDA_TRY(cudaFuncSetAttribute(rerank_kernel<kRerankRegs>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      kRerankRegs * kRerankThreads * static_cast<int>(sizeof(uint16_t))));
    ADT_CUDA_TRY(cudaFuncSetAttribute(rerank_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      kRerankMaxC * static_cast<int>(sizeof(uint16_t))));
    __atomic_fetch_or(&word, bit, __ATOMIC_ACQ_REL);
  }
  cfg.dynamicSmemBytes = static_cast<size_t>(C) * sizeof(uint16_t);
  if (C <= kRerankThreads)
    ADT_CUDA_TRY(cudaLaunchKernelEx(&cfg, rerank_kernel<1>, p));
  else if (C <= 2 * kRerankThreads)
    ADT_CUDA_TRY(cudaLaunchKernelEx(&cfg, rerank_kernel<2>, p));
  else if (C <= 4 * kRerankThreads)
    ADT_CUDA_TRY(cudaLaunchKernelEx(&cfg, rerank_kernel<4>, p));
  else if (C <= kRerankRegs * kRerankThreads)
    ADT_CUDA_TRY(cudaLaunchKernelEx(&cfg, rerank_kernel<kRerankRegs>, p));
  else
    ADT_CUDA_TRY(cudaLaunchKernelEx(&cfg, rerank_kernel<0>, p));
  return adt::launch_status();
}

}  // extern "C"
