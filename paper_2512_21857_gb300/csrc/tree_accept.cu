// adt_tree_accept: the verification walk (Sec. 3.1, Eq. 1; greedy T = 0 and
// sampling T = 1 as in Sec. 5.1).
//
// One thread-block cluster per tree.  The vocabulary is split into equal
// slices, one per CTA of the cluster; a CTA of a sampling walk keeps its slice
// of the current node's target (and draft) row in shared memory.  Every CTA
// takes the walk's decisions itself, from the same values combined in the same
// order, so all take the same ones.  The walk (children in ascending index,
// one accept test each) is sequential, as the method defines it: a chain of
// short phases, bound by their latency and, for the exponentials of the
// sampling modes, by the few SMs of one cluster.
//
// Greedy: the argmax of a slice is published in shared memory and read by
// every CTA after a cluster barrier.
//
// Sampling: vocabulary-wide values (maxima, sums, the CDF's totals) go out
// from every warp straight into all CTAs' shared memory with asynchronous
// stores that complete on the receivers' mbarriers, one way and without a
// barrier.  The children's tokens leave the slices before the exponentials
// are summed: their owners hand e_p and e_q of each to every CTA, so that the
// tests need no further reads.
//
// One tree of 64 nodes, ten children of the root, in a graph, before and now:
// SPEC, all rejected, V = 65536 93.2 -> 40.5 us, V = 16384 51.2 -> 29.5 us;
// SPEC_DET 23.1 -> 13.9 and 17.6 -> 9.9 us; greedy, four nodes visited, 14.5
// -> 11.5 and 13.0 -> 9.9 us (one kernel held all three modes and passed
// every value by a cluster barrier and remote reads).  Of the first, ten
// rejections are 20.5 us, a root without children (one row's exponentials, the
// draw) takes 13.8 us and the draft row with its exponentials the rest.
#include <cooperative_groups.h>

#include "adt_common.cuh"
#include "dfloat.cuh"
#include "sm100.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxNodes = 1024;
constexpr int kMostCtas = 16;      // per tree
constexpr int kBatch = 64;         // children of a node taken out of the slices together
constexpr uint32_t kWaitLimit = 1u << 22;   // polls
constexpr uint32_t kLandLimit = 1u << 12;   // polls (of 10 ns and more) for stores on their way

struct AcceptParams {
  const float* target;
  int64_t ldt;
  const float* draft;
  int64_t ldd;
  const float* target_u;  // classifier-free guidance: unconditional rows (same layout), else NULL
  const float* draft_u;
  float cfg;              // guidance scale
  const int32_t* drow;
  const int32_t* tokens;
  const int32_t* parents;
  const int32_t* offs;
  int V, max_nodes;
  const float* ua;
  const float* us;
  float T;
  int use_T;
  int32_t* path;
  int max_path;
  int32_t* alen;
  int32_t* bonus;
  unsigned* err;
  uint32_t wait_limit;  // polls before a wait gives up
  int Vs;  // vocabulary slice per CTA (multiple of 4)
};

__device__ __forceinline__ bool better(float v, int i, float bv, int bi) {
  return v > bv || (v == bv && i < bi);
}

struct Tree {
  int16_t par[kMaxNodes];
  int tok[kMaxNodes];
  int16_t kids[kMaxNodes];
  int16_t path[kMaxNodes];
  int nkids;
  int bad;
};

// What a tree that is skipped gets: the root alone.  One thread.
__device__ void write_skipped(const AcceptParams& p, int b) {
  p.alen[b] = 0;
  p.bonus[b] = 0;
  for (int i = 0; i < p.max_path; ++i) p.path[static_cast<int64_t>(b) * p.max_path + i] = i == 0 ? 0 : -1;
}

// Parents and tokens of tree b into shared memory; false, with the error
// raised and the outputs set (by the cluster's first CTA), for a malformed
// one.  Block-wide.
__device__ bool load_tree(Tree* t, const AcceptParams& p, int b, int node0, int n, bool first) {
  const int tid = threadIdx.x;
  if (tid == 0) t->bad = (n < 1 || n > p.max_nodes) ? 1 : 0;
  __syncthreads();
  if (!t->bad) {
    for (int i = tid; i < n; i += kThreads) {
      const int pr = p.parents[node0 + i];
      t->tok[i] = p.tokens[node0 + i];
      if ((i == 0) != (pr < 0) || pr >= i) t->bad = 1;
      t->par[i] = static_cast<int16_t>(pr < 0 ? -1 : pr);
    }
  }
  if (tid == 0) t->path[0] = 0;
  __syncthreads();
  if (!t->bad) return true;
  if (first && tid == 0) {
    adt::raise_error(p.err, ADT_DEVERR_BAD_TREE);
    write_skipped(p, b);
  }
  return false;
}

// The children of node v in ascending index, by one warp.
__device__ void find_kids(Tree* t, int n, int v) {
  const int lane = threadIdx.x & 31;
  int cnt = 0;
  for (int base = 0; base < n; base += 32) {
    const int i = base + lane;
    const bool f = i < n && t->par[i] == v;
    const unsigned bal = __ballot_sync(adt::kFullMask, f);
    if (f) t->kids[cnt + __popc(bal & ((1u << lane) - 1u))] = static_cast<int16_t>(i);
    cnt += __popc(bal);
  }
  if (lane == 0) t->nkids = cnt;
}

__device__ void write_path(const Tree* t, const AcceptParams& p, int b, int plen) {
  const int64_t o = static_cast<int64_t>(b) * p.max_path;
  if (plen > p.max_path && threadIdx.x == 0) adt::raise_error(p.err, ADT_DEVERR_BAD_PATH);
  for (int i = threadIdx.x; i < p.max_path; i += kThreads) p.path[o + i] = i < plen ? t->path[i] : -1;
  if (threadIdx.x == 0) p.alen[b] = min(plen, p.max_path) - 1;
}

// ---------------------------------------------------------------- greedy

// What a CTA publishes to its cluster; two copies alternate so that one
// barrier per exchange suffices.
struct GreedyShared {
  Tree tree;
  float best[2];
  int at[2];
  float fred[32];
  int ired[32];
};

// Block argmax over (value desc, index asc); all threads get the result.
__device__ void block_argmax(float& v, int& idx, GreedyShared* sh) {
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(adt::kFullMask, v, o);
    const int oi = __shfl_xor_sync(adt::kFullMask, idx, o);
    if (better(ov, oi, v, idx)) {
      v = ov;
      idx = oi;
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) {
    sh->fred[warp] = v;
    sh->ired[warp] = idx;
  }
  __syncthreads();
  v = lane < kThreads / 32 ? sh->fred[lane] : -INFINITY;
  idx = lane < kThreads / 32 ? sh->ired[lane] : 0x7fffffff;
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(adt::kFullMask, v, o);
    const int oi = __shfl_xor_sync(adt::kFullMask, idx, o);
    if (better(ov, oi, v, idx)) {
      v = ov;
      idx = oi;
    }
  }
}

__global__ void __launch_bounds__(kThreads) accept_greedy_kernel(const AcceptParams p) {
  __shared__ GreedyShared sh;
  adt::pdl_wait_then_release();
  cg::cluster_group cl = cg::this_cluster();
  const int rank = static_cast<int>(cl.block_rank()), csize = static_cast<int>(cl.num_blocks());
  const int b = blockIdx.x / csize;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lo = rank * p.Vs;
  const int cnt = max(0, min(p.Vs, p.V - lo));
  const int node0 = p.offs[b];
  const int n = p.offs[b + 1] - node0;
  if (!load_tree(&sh.tree, p, b, node0, n, rank == 0)) return;  // the same in every CTA of the cluster

  int v = 0, plen = 1, bonus = 0, parity = 0;
  for (int step = 0; step < n; ++step) {
    if (warp == 0) find_kids(&sh.tree, n, v);  // read after the argmax's barriers
    const int gv = node0 + v;
    const float* trow = p.target + static_cast<int64_t>(gv) * p.ldt;
    const float* trow_u = p.target_u ? p.target_u + static_cast<int64_t>(gv) * p.ldt : nullptr;
    float bv = -INFINITY;
    int bi = 0x7fffffff;
    // 16-byte loads (the row start and lo are multiples of 4 floats), a
    // thread's kU loads all issued before any value is compared.
    constexpr int kU = 4;
    const int c4 = cnt >> 2;
    const float4* t4 = reinterpret_cast<const float4*>(trow + lo);
    const float4* u4 = trow_u ? reinterpret_cast<const float4*>(trow_u + lo) : nullptr;
    for (int g0 = tid; g0 < c4; g0 += kU * kThreads) {
      float4 x[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int g = g0 + u * kThreads;
        x[u] = g < c4 ? __ldg(t4 + g) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      }
      if (u4) {
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const int g = g0 + u * kThreads;
          if (g < c4) {
            const float4 y = __ldg(u4 + g);
            x[u].x = adt::cfg_combine(x[u].x, y.x, p.cfg);
            x[u].y = adt::cfg_combine(x[u].y, y.y, p.cfg);
            x[u].z = adt::cfg_combine(x[u].z, y.z, p.cfg);
            x[u].w = adt::cfg_combine(x[u].w, y.w, p.cfg);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int g = g0 + u * kThreads;
        if (g >= c4) continue;
        const int i = lo + 4 * g;
        const float e[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (better(e[j], i + j, bv, bi)) {
            bv = e[j];
            bi = i + j;
          }
      }
    }
    for (int i = 4 * c4 + tid; i < cnt; i += kThreads) {  // the last slice's final cnt % 4 values
      float x = __ldg(trow + lo + i);
      if (trow_u) x = adt::cfg_combine(x, __ldg(trow_u + lo + i), p.cfg);
      if (better(x, lo + i, bv, bi)) {
        bv = x;
        bi = lo + i;
      }
    }
    block_argmax(bv, bi, &sh);
    if (tid == 0) {
      sh.best[parity] = bv;
      sh.at[parity] = bi;
    }
    cl.sync();
    // lane c reads CTA c's candidate; the warp's argmax over the lanes
    float gvv = -INFINITY;
    int g = 0x7fffffff;
    if (lane < csize) {
      const GreedyShared* s = cl.map_shared_rank(&sh, lane);
      gvv = s->best[parity];
      g = s->at[parity];
    }
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(adt::kFullMask, gvv, o);
      const int oi = __shfl_xor_sync(adt::kFullMask, g, o);
      if (better(ov, oi, gvv, g)) {
        gvv = ov;
        g = oi;
      }
    }
    parity ^= 1;
    // the first child whose token it is (a lane per child)
    int nxt = -1;
    for (int j0 = 0; j0 < sh.tree.nkids && nxt < 0; j0 += 32) {
      const int k = j0 + lane < sh.tree.nkids ? sh.tree.kids[j0 + lane] : -1;
      const unsigned hit = __ballot_sync(adt::kFullMask, k >= 0 && sh.tree.tok[k] == g);
      if (hit) nxt = __shfl_sync(adt::kFullMask, k, __ffs(hit) - 1);
    }
    if (nxt < 0) {
      bonus = g;
      break;
    }
    if (tid == 0) sh.tree.path[plen] = static_cast<int16_t>(nxt);
    ++plen;
    v = nxt;
    __syncthreads();  // the node's list is rewritten
  }
  __syncthreads();
  if (rank == 0) {
    write_path(&sh.tree, p, b, plen);
    if (tid == 0) p.bonus[b] = bonus;
  }
  cl.sync();  // no CTA leaves while a peer may still read its shared memory
}

// ---------------------------------------------------------------- sampling

// The slices of e_p and e_q.  Slice<true>: double-float entries (hi, lo) and
// exponentials, so the decisions the walk takes from them (u q(x) < p(x), the
// inverse-CDF draw) agree with fp64 arithmetic to about 1e-11 relative; used
// where the slices fit in shared memory.  Slice<false>: fp32 entries and fp32
// exponentials (relative error about 1e-7), for larger vocabularies.  All
// arithmetic on the entries is double-float either way.
template <bool kDF>
struct Slice;

template <>
struct Slice<false> {
  using E = float;
  static __device__ __forceinline__ E logit(float x) { return x; }
  static __device__ __forceinline__ float value_hi(E v) { return v; }
  static __device__ __forceinline__ dfl::df exp_diff(float x, float M, const float2*) {
    return dfl::df{expf(x - M), 0.f};
  }
  static __device__ __forceinline__ dfl::df as_df(E v) { return dfl::df{v, 0.f}; }
  static __device__ __forceinline__ E from_df(dfl::df v) { return v.hi; }
};

template <>
struct Slice<true> {
  using E = float2;
  static __device__ __forceinline__ E logit(float x) { return make_float2(x, 0.f); }
  static __device__ __forceinline__ float value_hi(E v) { return v.x; }
  static __device__ __forceinline__ dfl::df exp_diff(float x, float M, const float2* tab) {
    return dfl::df_exp_diff(x, M, tab);
  }
  static __device__ __forceinline__ dfl::df as_df(E v) { return dfl::df{v.x, v.y}; }
  static __device__ __forceinline__ E from_df(dfl::df v) { return make_float2(v.hi, v.lo); }
};

struct SampleShared {
  // One entry per warp of the cluster and round (two rounds alternate), and
  // e_p, e_q of the batch's children: pushed by their owners.
  float4 part[2][kMostCtas * kWarps];
  float4 kid_e[kBatch];
  float2 exptab[64];  // 2^(j/64) as double-floats (the double-float exponential's table)
  uint64_t bar[2];
  Tree tree;
  int kid_tok[kBatch];
  uint8_t kid_state[kBatch];  // 0 a child of its own, 2 the token of an earlier one, 4 no token of the vocabulary
  int16_t kid_rep[kBatch];    // 2: that earlier child
  float2 bf[2];               // scalars that warp 0 hands to the block
  int bi[2];
  int late[3];                // thread 0's, at a batch's start, before the draw and at the end
  int tree_own;               // children of state 0
};

__device__ __forceinline__ dfl::df shfl_xor_df(dfl::df v, int o) {
  return dfl::df{__shfl_xor_sync(adt::kFullMask, v.hi, o), __shfl_xor_sync(adt::kFullMask, v.lo, o)};
}
__device__ __forceinline__ dfl::df shfl_df(dfl::df v, int src) {
  return dfl::df{__shfl_sync(adt::kFullMask, v.hi, src), __shfl_sync(adt::kFullMask, v.lo, src)};
}
// Sum over the warp of non-negative terms, in every lane.
__device__ __forceinline__ dfl::df warp_sum_df(dfl::df v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = dfl::df_add_pos(v, shfl_xor_df(v, o));
  return v;
}
// Inclusive sum over the lanes from this one on, of non-negative terms.
__device__ __forceinline__ dfl::df warp_suffix_df(dfl::df v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const dfl::df y{__shfl_down_sync(adt::kFullMask, v.hi, o), __shfl_down_sync(adt::kFullMask, v.lo, o)};
    if (lane + o < 32) v = dfl::df_add_pos(v, y);
  }
  return v;
}
__device__ __forceinline__ dfl::df warp_prefix_df(dfl::df v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const dfl::df y{__shfl_up_sync(adt::kFullMask, v.hi, o), __shfl_up_sync(adt::kFullMask, v.lo, o)};
    if (lane >= o) v = dfl::df_add_pos(v, y);
  }
  return v;
}

// max(0, e_p - B e_q).
__device__ __forceinline__ dfl::df resid(dfl::df ep, dfl::df eq, dfl::df B) {
  return dfl::df_max0(dfl::df_add(ep, dfl::df_neg(dfl::df_mul(B, eq))));
}

// The rounds of the cluster: in a round every warp pushes one entry to every
// CTA of the cluster, and a CTA that has all of them (and `extra` bytes more:
// the children's) goes on.  Two rounds' entries are kept apart by the round's
// parity: a warp pushes for round r + 2 only once round r + 1 is complete, for
// which every warp of the cluster has pushed after it was done with round r.
//
// A wait that runs out raises the error and sets `late` in its thread.  Thread
// 0 tells the others across the block barrier that follows every wait, before
// anything else is pushed: the walk ends there, and the CTA pushes no more.
// (That thread 0 is not late says that the round is complete.  A vote of the
// barrier took 0.05 us each.)
struct Rounds {
  SampleShared* sh;
  unsigned* err;
  uint32_t limit;
  int rank, csize, r;
  int late;
  __device__ __forceinline__ void send(float4 v, const void* local, int c) {
    asm volatile(
        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];\n" ::"r"(
            sm100::mapa_shared(sm100::smem_addr(local), c)),
        "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(sm100::mapa_shared(sm100::smem_addr(&sh->bar[r & 1]), c))
        : "memory");
  }
  // v: the warp's entry, in every lane.
  __device__ __forceinline__ void push(float4 v, int extra = 0) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane < csize) send(v, &sh->part[r & 1][rank * kWarps + warp], lane);
    if (threadIdx.x == 0)
      sm100::mbar_arrive_expect_tx(sm100::smem_addr(&sh->bar[r & 1]),
                                   static_cast<uint32_t>(csize * kWarps * sizeof(float4) + extra));
  }
  __device__ __forceinline__ bool poll(uint32_t polls) {
    return sm100::mbar_wait_bounded(sm100::smem_addr(&sh->bar[r & 1]), (r >> 1) & 1, polls);
  }
  __device__ __forceinline__ void wait() {
    if (!poll(limit)) {
      adt::raise_error(err, ADT_DEVERR_TIMEOUT);
      late = 1;
    }
  }
  // The end of a CTA with a late wait: peers may still push to it (those that
  // are not late have all they wait for and may be gone).  It stays until every
  // peer has ended or come here too, so that none pushes any more, and for the
  // stores that are on their way.
  __device__ __forceinline__ void stay() {
    sm100::cluster_arrive_release();
    sm100::cluster_wait_acquire();
    (void)poll(kLandLimit);
  }
  __device__ __forceinline__ const float4* entries() const { return sh->part[r & 1]; }
  __device__ __forceinline__ int count() const { return csize * kWarps; }
};

// Loads this CTA's slices of the target row and (kQ) the draft row -- under
// guidance u + s (c - u) with the unconditional rows; then divided by T --
// into pbuf and qbuf (entries past V are -inf); a thread's loads of both rows
// go out before any is used.  Returns the largest logits this thread loaded.
template <bool kDF, bool kQ>
__device__ float2 load_rows(const float* trow, const float* trow_u, const float* drow, const float* drow_u, int lo,
                            int cnt, typename Slice<kDF>::E* pbuf, typename Slice<kDF>::E* qbuf,
                            const AcceptParams& p) {
  constexpr int kU = 4, kRows = kQ ? 2 : 1;
  const float* rows[2] = {trow + lo, drow + lo};
  const float* rows_u[2] = {trow_u + lo, drow_u + lo};
  float mx[2] = {-INFINITY, -INFINITY};
  for (int g0 = threadIdx.x * 4; g0 < p.Vs; g0 += kU * kThreads * 4) {
    float4 x[kRows][kU], y[kRows][kU];
#pragma unroll
    for (int r = 0; r < kRows; ++r)
#pragma unroll
      for (int k = 0; k < kU; ++k) {
        const int i = g0 + k * kThreads * 4;
        if (i + 3 < cnt) {
          x[r][k] = __ldg(reinterpret_cast<const float4*>(rows[r] + i));
          if (trow_u) y[r][k] = __ldg(reinterpret_cast<const float4*>(rows_u[r] + i));
        } else {
          float e[4], f[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            e[c] = i + c < cnt ? __ldg(rows[r] + i + c) : -INFINITY;
            f[c] = trow_u && i + c < cnt ? __ldg(rows_u[r] + i + c) : 0.f;
          }
          x[r][k] = make_float4(e[0], e[1], e[2], e[3]);
          y[r][k] = make_float4(f[0], f[1], f[2], f[3]);
        }
      }
#pragma unroll
    for (int r = 0; r < kRows; ++r)
#pragma unroll
      for (int k = 0; k < kU; ++k) {
        const int i = g0 + k * kThreads * 4;
        if (i >= p.Vs) continue;
        const float e[4] = {x[r][k].x, x[r][k].y, x[r][k].z, x[r][k].w};
        const float f[4] = {y[r][k].x, y[r][k].y, y[r][k].z, y[r][k].w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float v = e[c];
          if (i + c < cnt) {
            if (trow_u) v = adt::cfg_combine(v, f[c], p.cfg);
            if (p.use_T) v = __fdiv_rn(v, p.T);
          }
          mx[r] = fmaxf(mx[r], v);
          (r ? qbuf : pbuf)[i + c] = Slice<kDF>::logit(v);
        }
      }
  }
  return make_float2(mx[0], mx[1]);
}

// The walk under SPEC (Eq. 1 with recursive rejection sampling) or SPEC_DET.
//
// SPEC in closed form.  With e_p, e_q the exponentials of the target and draft
// rows, p after any number of rejections is max(0, e_p - B e_q) / N at every
// token not rejected yet: a rejection takes p <- max(0, p - q) / Z with q = e_q
// / Q, which is B <- B + N / Q and N <- the new sum, and B only grows, so a
// token that was cut off stays so.  A rejected token's q is 0, so its e_p
// becomes its part of that sum, once, and its e_q 0.  A rejection therefore
// costs one pass that only reads the slices and one round, no division (the Q
// left after each child do not depend on the walk: their reciprocals are
// formed at once), and the test u q(x) < p(x) reads u e_q N < (e_p - B e_q) Q.
// A rejection at V = 16384 / 65536 with 8 CTAs, updating p and q in place with
// two passes and two exchanges: 3.9 / 7.0 us; this way 1.6 / 2.5 us (2.05 us with
// 16 CTAs).
template <bool kDF, bool kSpec>
__global__ void __launch_bounds__(kThreads) accept_sample_kernel(const AcceptParams p) {
  using SL = Slice<kDF>;
  using E = typename SL::E;
  extern __shared__ __align__(16) float dyn[];
  __shared__ __align__(16) SampleShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (kDF) dfl::exp_table_to_smem(sh.exptab);  // read after the block barriers below
  if (tid == 0) {
    sm100::mbar_init(sm100::smem_addr(&sh.bar[0]), 1);
    sm100::mbar_init(sm100::smem_addr(&sh.bar[1]), 1);
    sm100::fence_mbar_init();
  }
  __syncwarp();
  sm100::cluster_arrive_release();  // the mbarriers are there: waited for before the first push
  adt::pdl_wait_then_release();
  cg::cluster_group cl = cg::this_cluster();
  Rounds rd{&sh, p.err, p.wait_limit, static_cast<int>(cl.block_rank()), static_cast<int>(cl.num_blocks()), 0, 0};
  const int b = blockIdx.x / rd.csize;
  E* pbuf = reinterpret_cast<E*>(dyn);
  E* qbuf = pbuf + p.Vs;
  const int lo = rd.rank * p.Vs;
  const int cnt = max(0, min(p.Vs, p.V - lo));
  const int node0 = p.offs[b];
  const int n = p.offs[b + 1] - node0;
  Tree& tree = sh.tree;
  if (!load_tree(&tree, p, b, node0, n, rd.rank == 0)) {  // the same in every CTA of the cluster
    sm100::cluster_wait_acquire();
    return;
  }

  int v = 0, plen = 1;
  for (int step = 0; step < n; ++step) {
    if (warp == 0) find_kids(&tree, n, v);
    __syncthreads();
    int nk = tree.nkids;
    const int gv = node0 + v;
    const float* trow = p.target + static_cast<int64_t>(gv) * p.ldt;
    const float* trow_u = p.target_u ? p.target_u + static_cast<int64_t>(gv) * p.ldt : nullptr;
    const float us = p.us[gv];
    // The draft row of v (the same value in every thread of the cluster).  A
    // node with children but no draft row (negative index) is an error; its
    // children are then not considered and the bonus comes from p.
    const int64_t dr = kSpec && nk > 0 && p.drow ? static_cast<int64_t>(p.drow[gv]) : gv;
    if (dr < 0) {
      if (rd.rank == 0 && tid == 0) adt::raise_error(p.err, ADT_DEVERR_BAD_INDEX);
      nk = 0;
    }
    const bool need_q = kSpec && nk > 0;
    float2 mx;
    if (need_q)
      mx = load_rows<kDF, true>(trow, trow_u, p.draft + dr * p.ldd, p.draft_u ? p.draft_u + dr * p.ldd : nullptr, lo,
                                cnt, pbuf, qbuf, p);
    else
      mx = load_rows<kDF, false>(trow, trow_u, nullptr, nullptr, lo, cnt, pbuf, qbuf, p);
    mx.x = adt::warp_max(mx.x);
    mx.y = adt::warp_max(mx.y);
    __syncwarp();
    if (step == 0) sm100::cluster_wait_acquire();  // every peer's mbarriers are initialised
    rd.push(make_float4(mx.x, mx.y, 0.f, 0.f));
    rd.wait();
    float Mp = -INFINITY, Mq = -INFINITY;
    for (int e = lane; e < rd.count(); e += 32) {
      Mp = fmaxf(Mp, rd.entries()[e].x);
      Mq = fmaxf(Mq, rd.entries()[e].y);
    }
    Mp = adt::warp_max(Mp);
    Mq = adt::warp_max(Mq);
    ++rd.r;

    int nxt = -1;
    dfl::df N{0.f, 0.f}, B{0.f, 0.f};  // SPEC, warp 0 (N = 0: not set yet)
    bool exps = false;                 // the slices hold exponentials
    int late = 0;                      // the same in every thread
    for (int base = 0; nxt < 0 && (base < nk || !exps); base += kBatch) {
      const int nb = min(kBatch, max(0, nk - base));
      // The batch's tokens leave the slices.
      if (base > 0) {  // no push reaches a peer that still decides on the batch before
        rd.push(make_float4(0.f, 0.f, 0.f, 0.f));
        rd.wait();
        ++rd.r;
      }
      if (tid < nb) sh.kid_tok[tid] = tree.tok[tree.kids[base + tid]];
      if (tid == 0) {
        sh.tree_own = 0;
        sh.late[0] = rd.late;
      }
      __syncthreads();  // also: this CTA's slices are written
      late = sh.late[0];
      if (late) break;
      if (tid < nb) {
        const int x = sh.kid_tok[tid];
        int rep = tid;
        for (int i = tid - 1; i >= 0; --i) rep = sh.kid_tok[i] == x ? i : rep;
        const bool out = x < 0 || x >= p.V;
        sh.kid_rep[tid] = static_cast<int16_t>(rep);
        sh.kid_state[tid] = out ? 4 : rep != tid ? 2 : 0;
        if (!out && rep == tid) {
          atomicAdd(&sh.tree_own, 1);
          if (x / p.Vs == rd.rank) {
            const int off = x - lo;
            dfl::df ep, eq{0.f, 0.f};
            if (exps) {
              ep = SL::as_df(pbuf[off]);
              if (need_q) eq = SL::as_df(qbuf[off]);
              pbuf[off] = SL::logit(0.f);
              if (need_q) qbuf[off] = SL::logit(0.f);
            } else {
              ep = SL::exp_diff(SL::value_hi(pbuf[off]), Mp, sh.exptab);
              if (need_q) eq = SL::exp_diff(SL::value_hi(qbuf[off]), Mq, sh.exptab);
              pbuf[off] = SL::logit(-INFINITY);
              if (need_q) qbuf[off] = SL::logit(-INFINITY);
            }
            for (int c = 0; c < rd.csize; ++c) rd.send(make_float4(ep.hi, ep.lo, eq.hi, eq.lo), &sh.kid_e[tid], c);
          }
        }
      }
      __syncthreads();
      // Exponentials in place (first batch), and the sums of the rest.
      dfl::Acc ap, aq;
#pragma unroll 2
      for (int i = tid; i < p.Vs; i += kThreads) {
        dfl::df e;
        if (exps) {
          e = SL::as_df(pbuf[i]);
        } else {
          e = SL::exp_diff(SL::value_hi(pbuf[i]), Mp, sh.exptab);
          pbuf[i] = SL::from_df(e);
        }
        ap.add(e);
        if (kSpec && need_q) {
          if (exps) {
            e = SL::as_df(qbuf[i]);
          } else {
            e = SL::exp_diff(SL::value_hi(qbuf[i]), Mq, sh.exptab);
            qbuf[i] = SL::from_df(e);
          }
          aq.add(e);
        }
      }
      exps = true;
      {
        const dfl::df sp = warp_sum_df(ap.value_df());
        const dfl::df sq = kSpec ? warp_sum_df(aq.value_df()) : dfl::df{0.f, 0.f};
        rd.push(make_float4(sp.hi, sp.lo, sq.hi, sq.lo), sh.tree_own * static_cast<int>(sizeof(float4)));
      }
      // Warp 0: the cluster's sums over the tokens of no child, and the
      // children: lane i holds child i (c0) and i + 32 (c1).
      dfl::df Rp{0.f, 0.f}, Rq{0.f, 0.f};
      dfl::df p0{0.f, 0.f}, p1{0.f, 0.f}, q0{0.f, 0.f}, q1{0.f, 0.f};
      float u0 = 0.f, u1 = 0.f;
      if (warp == 0) {
        if (lane < nb) u0 = p.ua[node0 + tree.kids[base + lane]];
        if (lane + 32 < nb) u1 = p.ua[node0 + tree.kids[base + lane + 32]];
        rd.wait();
        for (int e = lane; e < rd.count(); e += 32) {
          const float4 t = rd.entries()[e];
          Rp = dfl::df_add_pos(Rp, dfl::df{t.x, t.y});
          Rq = dfl::df_add_pos(Rq, dfl::df{t.z, t.w});
        }
        Rp = warp_sum_df(Rp);
        if (kSpec) Rq = warp_sum_df(Rq);
        if (lane < nb && sh.kid_state[lane] == 0) {
          const float4 t = sh.kid_e[lane];
          p0 = dfl::df{t.x, t.y};
          q0 = dfl::df{t.z, t.w};
        }
        if (lane + 32 < nb && sh.kid_state[lane + 32] == 0) {
          const float4 t = sh.kid_e[lane + 32];
          p1 = dfl::df{t.x, t.y};
          q1 = dfl::df{t.z, t.w};
        }
      }
      ++rd.r;
      if (nb == 0) break;

      if constexpr (!kSpec) {
        // Child j is tried once 0 .. j-1 are rejected: p(x_j) = e_j / (R + sum
        // of e_i, i >= j).  The tests do not depend on each other; the first
        // one accepted counts.  u < e / denom is taken as u denom < e: no
        // division.
        if (warp == 0) {
          const dfl::df s1 = dfl::df_add_pos(Rp, warp_suffix_df(p1));
          const dfl::df s0 = dfl::df_add_pos(shfl_df(s1, 0), warp_suffix_df(p0));
          const unsigned a0 = __ballot_sync(adt::kFullMask, p0.hi > 0.f && dfl::df_less(dfl::df_mul_f(s0, u0), p0));
          const unsigned a1 = __ballot_sync(adt::kFullMask, p1.hi > 0.f && dfl::df_less(dfl::df_mul_f(s1, u1), p1));
          const int at = a0 ? __ffs(a0) - 1 : a1 ? 31 + __ffs(a1) : nb;
          if (rd.rank == 0)
            for (int j = lane; j < at; j += 32)
              if (sh.kid_state[j] == 4) adt::raise_error(p.err, ADT_DEVERR_BAD_INDEX);
          if (lane == 0) sh.bi[0] = rd.late ? -1 : at;
        }
        __syncthreads();
        late = sh.bi[0] < 0;
        if (late) break;
        if (sh.bi[0] < nb) nxt = tree.kids[base + sh.bi[0]];
      } else {
        // Q and 1 / Q once the children before this one are gone.
        dfl::df Q0{0.f, 0.f}, Q1{0.f, 0.f}, iQ0{0.f, 0.f}, iQ1{0.f, 0.f};
        if (warp == 0) {
          Q1 = dfl::df_add_pos(Rq, warp_suffix_df(q1));
          Q0 = dfl::df_add_pos(shfl_df(Q1, 0), warp_suffix_df(q0));
          if (Q0.hi > 0.f) iQ0 = dfl::df_recip(Q0);
          if (Q1.hi > 0.f) iQ1 = dfl::df_recip(Q1);
          if (N.hi == 0.f) {  // in the order of Q: equal rows have equal sums
            const dfl::df t1 = dfl::df_add_pos(Rp, warp_suffix_df(p1));
            N = shfl_df(dfl::df_add_pos(shfl_df(t1, 0), warp_suffix_df(p0)), 0);
          }
        }
        int j = 0;
        for (;;) {
          // Warp 0 tries children until one is accepted or a rejection needs
          // its residual mass.
          dfl::df nB{0.f, 0.f};
          if (warp == 0) {
            int verdict = 0;
            const dfl::df v0 = resid(p0, q0, B), v1 = resid(p1, q1, B);  // p(x) N
            for (; j < nb; ++j) {
              const int st = sh.kid_state[j];
              if (st == 4) {
                if (lane == 0 && rd.rank == 0) adt::raise_error(p.err, ADT_DEVERR_BAD_INDEX);
                continue;
              }
              const bool hi = j >= 32;
              const dfl::df Qj = shfl_df(hi ? Q1 : Q0, j & 31);
              bool ok;
              if (st == 2) {  // an earlier child's token: rejected, q is 0
                const int r = sh.kid_rep[j];
                ok = shfl_df(r >= 32 ? v1 : v0, r & 31).hi > 0.f;
              } else {
                const bool mine = dfl::df_less(dfl::df_mul_f(dfl::df_mul(hi ? q1 : q0, N), hi ? u1 : u0),
                                               dfl::df_mul(hi ? v1 : v0, Qj));
                // no draft mass left: q(x) is 0
                ok = __shfl_sync(adt::kFullMask, Qj.hi > 0.f ? mine : (hi ? v1 : v0).hi > 0.f, j & 31);
              }
              verdict = ok ? 1 : 2;
              const dfl::df iq = shfl_df(hi ? iQ1 : iQ0, j & 31);
              const bool same = N.hi == Qj.hi && N.lo == Qj.lo;
              nB = dfl::df_add_pos(B, same ? dfl::df{1.f, 0.f} : dfl::df_mul(N, iq));
              break;
            }
            if (lane == 0) {
              sh.bi[0] = rd.late ? -1 : verdict;
              sh.bi[1] = j;
              sh.bf[0] = make_float2(nB.hi, nB.lo);
            }
          }
          __syncthreads();
          const int verdict = sh.bi[0];
          late = verdict < 0;
          if (verdict == 1) nxt = tree.kids[base + sh.bi[1]];
          if (verdict != 2) break;
          // The residual mass of the slices at the new B: sum of max(0, e_p -
          // B e_q), the product exact in its leading words (two_prod) and
          // every difference taken with its error.
          const dfl::df cB{sh.bf[0].x, sh.bf[0].y};
          float zs = 0.f, zc = 0.f;
#pragma unroll 4
          for (int i = tid; i < p.Vs; i += kThreads) {
            const dfl::df ep = SL::as_df(pbuf[i]), eq = SL::as_df(qbuf[i]);
            const dfl::df c = dfl::two_prod(cB.hi, eq.hi);
            const float cl = __fmaf_rn(cB.hi, eq.lo, __fmaf_rn(cB.lo, eq.hi, c.lo));
            const dfl::df d = dfl::two_sum(ep.hi, -c.hi);
            const float dl = __fadd_rn(d.lo, __fsub_rn(ep.lo, cl));
            const bool pos = __fadd_rn(d.hi, dl) > 0.f;
            const dfl::df t = dfl::two_sum(zs, pos ? d.hi : 0.f);
            zs = t.hi;
            zc = __fadd_rn(zc, __fadd_rn(t.lo, pos ? dl : 0.f));
          }
          const dfl::df z = warp_sum_df(dfl::df_max0(dfl::fast_two_sum(zs, zc)));
          rd.push(make_float4(z.hi, z.lo, 0.f, 0.f));
          if (warp == 0) {
            // The batch's tokens follow the closed form, rejected ones with
            // e_q = 0.
            const dfl::df v0 = resid(p0, q0, nB), v1 = resid(p1, q1, nB);
            dfl::df Z = dfl::df_add_pos(v0, v1);
            rd.wait();
            for (int e = lane; e < rd.count(); e += 32) {
              const float4 t = rd.entries()[e];
              Z = dfl::df_add_pos(Z, dfl::df{t.x, t.y});
            }
            Z = warp_sum_df(Z);
            const bool zpos = Z.hi > 0.f;  // no mass left: p stays as it is
            const bool own = sh.kid_state[j] == 0;
            if (own && lane == (j & 31)) {
              if (j >= 32) {
                p1 = zpos ? v1 : resid(p1, q1, B);
                q1 = dfl::df{0.f, 0.f};
              } else {
                p0 = zpos ? v0 : resid(p0, q0, B);
                q0 = dfl::df{0.f, 0.f};
              }
            }
            if (zpos) {
              N = Z;
              B = nB;
            }
            ++j;
          }
          ++rd.r;
        }
        if (late) break;
        if (nxt < 0) {
          // All of the batch rejected: their tokens return to the slices.
          if (warp == 0) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int i = lane + 32 * h;
              if (i < nb && sh.kid_state[i] == 0 && sh.kid_tok[i] / p.Vs == rd.rank) {
                pbuf[sh.kid_tok[i] - lo] = SL::from_df(h ? p1 : p0);
                qbuf[sh.kid_tok[i] - lo] = SL::logit(0.f);
              }
            }
            if (lane == 0) sh.bf[1] = make_float2(B.hi, B.lo);
          }
          __syncthreads();
        }
      }
    }

    if (nxt < 0) {
      // The bonus: the smallest t with sum_{j<=t} w_j > u sum_j w_j over the
      // (unnormalised) current p.  Thread t owns a contiguous run of the
      // slice and reads it starting at offset t mod its length, wrapping
      // around: at the same step the threads of a half-warp then touch
      // different banks.
      if (tid == 0) sh.late[1] = rd.late;
      __syncthreads();
      if (late || sh.late[1]) break;
      const dfl::df fB{sh.bf[1].x, sh.bf[1].y};
      const int per = (cnt + kThreads - 1) / kThreads;
      const int b0 = min(cnt, tid * per), b1 = min(cnt, b0 + per), len = b1 - b0;
      dfl::Acc racc;
      int last_pos = -1;
      int jr = len > 0 ? tid % len : 0;
      for (int k = 0; k < len; ++k) {
        const int i = b0 + jr;
        dfl::df w = SL::as_df(pbuf[i]);
        if (kSpec && need_q) {
          w = resid(w, SL::as_df(qbuf[i]), fB);
          pbuf[i] = SL::from_df(w);
        }
        racc.add(w);
        if (w.hi > 0.f) last_pos = max(last_pos, i);
        if (++jr == len) jr = 0;
      }
      const dfl::df run = racc.value_df();
      const dfl::df incl = warp_prefix_df(run);
      const dfl::df tot = shfl_df(incl, 31);
      rd.push(make_float4(tot.hi, tot.lo, 0.f, 0.f));
      rd.wait();
      // The warps' totals in index order: a lane scans count / 32 of them.
      // The draw lies in the first warp whose cumulative total passes the
      // target, else in the last one with mass.  (Every warp does this.)
      const int ne = rd.count() / 32;  // csize * kWarps: 1 to 8
      dfl::df mine{0.f, 0.f};
      for (int k = 0; k < ne; ++k) {
        const float4 t = rd.entries()[lane * ne + k];
        mine = dfl::df_add_pos(mine, dfl::df{t.x, t.y});
      }
      const dfl::df pre = warp_prefix_df(mine);
      const dfl::df grand = shfl_df(pre, 31);
      const dfl::df target = dfl::df_mul_f(grand, us);
      const dfl::df prev{__shfl_up_sync(adt::kFullMask, pre.hi, 1), __shfl_up_sync(adt::kFullMask, pre.lo, 1)};
      dfl::df acc = lane == 0 ? dfl::df{0.f, 0.f} : prev, at{0.f, 0.f};
      int pass = -1, mass = -1;
      for (int k = 0; k < ne; ++k) {
        const float4 t = rd.entries()[lane * ne + k];
        if (t.x > 0.f) mass = lane * ne + k;
        const dfl::df nx = dfl::df_add_pos(acc, dfl::df{t.x, t.y});
        if (pass < 0 && dfl::df_less(target, nx)) {
          pass = lane * ne + k;
          at = acc;
        }
        acc = nx;
      }
      const unsigned pm = __ballot_sync(adt::kFullMask, pass >= 0);
      const unsigned mm = __ballot_sync(adt::kFullMask, mass >= 0);
      int owner = 0;
      if (pm)
        owner = __shfl_sync(adt::kFullMask, pass, __ffs(pm) - 1);
      else if (mm)
        owner = __shfl_sync(adt::kFullMask, mass, 31 - __clz(mm));
      if (owner == rd.rank * kWarps + warp) {
        // The running CDF over the warp's runs, compared with the target
        // through the sign of their difference.
        const dfl::df ntgt = dfl::df_neg(target);
        const dfl::df before{__shfl_up_sync(adt::kFullMask, incl.hi, 1), __shfl_up_sync(adt::kFullMask, incl.lo, 1)};
        dfl::df c = pm ? shfl_df(at, __ffs(pm) - 1) : grand;
        if (lane > 0) c = dfl::df_add_pos(c, before);
        int found = 0x7fffffff;
        if (dfl::df_add(dfl::df_add_pos(c, run), ntgt).hi > 0.f) {
          for (int i = b0; i < b1; ++i) {
            const dfl::df w = SL::as_df(pbuf[i]);
            c = dfl::df_add_pos(c, w);
            if (w.hi > 0.f && dfl::df_add(c, ntgt).hi > 0.f) {
              found = i;
              break;
            }
          }
        }
        __syncwarp();
        found = static_cast<int>(__reduce_min_sync(adt::kFullMask, static_cast<unsigned>(found)));
        last_pos = __reduce_max_sync(adt::kFullMask, last_pos);
        if (lane == 0) p.bonus[b] = lo + (found != 0x7fffffff ? found : last_pos < 0 ? 0 : last_pos);
      }
      break;
    }
    if (tid == 0) tree.path[plen] = static_cast<int16_t>(nxt);
    ++plen;
    v = nxt;
    __syncthreads();  // the node's lists are rewritten
  }
  if (tid == 0) sh.late[2] = rd.late;
  __syncthreads();
  if (sh.late[2]) {
    if (rd.rank == 0 && tid == 0) write_skipped(p, b);
    rd.stay();
    return;
  }
  if (rd.rank == 0) write_path(&tree, p, b, plen);
  // Every warp has waited for the last round, so all pushes to this CTA have
  // landed; a peer its own pushes are for stays until it has them.
}

// CTAs per tree.  Greedy (no slices; a node costs one read of its row and one
// exchange): 4 up to 32768 entries, 8 up to 131072 (a walk of four nodes, 4 / 8
// / 16 CTAs, us: 10.0 / 10.6 / 15.8 at V = 16384, 10.7 / 10.9 / 15.9 at 32768,
// 13.0 / 11.6 / 16.2 at 65536).  Sampling: 8; 16 past 65536 entries, where the
// double-float slices of fewer would not fit, and for SPEC past 32768 with few
// trees (its exponentials and passes are bound by a cluster's SMs; ten
// rejections, 8 / 16 CTAs, us: 34.5 / 35.5 at V = 32768, 47.7 / 40.6 at 65536;
// clusters of 16 for more than about seven trees do not run at once: 49.2 /
// 68.6 with eight).  A SPEC CTA fills its SM's registers: fewer a tree where
// the clusters of more do not all run at once and fewer hold the slices (8 / 4
// / 2 CTAs, ten rejections, us: 32 trees at V = 4096 75 / 27 / 30, 16 at 16384
// 59 / 37 / 45, 64 at 16384 144 / 68 / 47, 64 at 32768 168 / 89).  fit[i]: the SPEC
// clusters of 2 << i that run at once; where a process may use only some of the
// SMs that can be none of 16.
constexpr int kSlice = 8192;  // the most entries of a slice of p and one of q in double-floats

int cluster_size_for(int V, int B, adt_accept_mode mode, const int* fit) {
  if (mode == ADT_ACCEPT_GREEDY) return V <= 32768 ? 4 : V <= 131072 ? 8 : 16;
  if (V > 8 * kSlice) return 16;
  if (mode == ADT_ACCEPT_SPEC_DET) return 8;
  if (V > 32768 && B <= 4 && B <= fit[3]) return 16;
  int cs = 8;
  for (int i = 2; cs > 2 && B > fit[i] && V <= cs / 2 * kSlice; --i) cs /= 2;
  return cs;
}

// The launch limits of instantiation `inst`, once per device and the same
// whatever call comes first: all the dynamic shared memory a block can have
// beside the static part, and clusters of 16.
adt_status configure(void (*kern)(AcceptParams), int inst, const adt::DeviceInfo& info) {
  static unsigned configured[6][2];  // bit per device (< 64)
  unsigned& word = configured[inst][(info.device >> 5) & 1];
  const unsigned bit = 1u << (info.device & 31);
  if (__atomic_load_n(&word, __ATOMIC_ACQUIRE) & bit) return ADT_OK;
  cudaFuncAttributes attr;
  ADT_CUDA_TRY(cudaFuncGetAttributes(&attr, kern));
  ADT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    info.max_smem_optin - static_cast<int>(attr.sharedSizeBytes)));
  ADT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  __atomic_fetch_or(&word, bit, __ATOMIC_ACQ_REL);
  return ADT_OK;
}

int slice_for(int V, int cs) {
  int vs = (V + cs - 1) / cs;
  return (vs + 3) / 4 * 4;
}

// Clusters of cs CTAs of the SPEC walk that run on the device at once (with the
// largest slices: a CTA has its SM to itself with smaller ones too).
int spec_clusters(const adt::DeviceInfo& info, int cs) {
  static int cache[64][17];  // 0 = not queried yet
  int& slot = cache[info.device & 63][cs];
  const int v = __atomic_load_n(&slot, __ATOMIC_ACQUIRE);
  if (v) return v - 1;
  int num = 0;
  const auto kern = accept_sample_kernel<true, true>;
  if (configure(kern, 2 * ADT_ACCEPT_SPEC + 1, info) == ADT_OK) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(cs), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = 2 * sizeof(float2) * kSlice;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cs);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&num, kern, &cfg) != cudaSuccess) num = 0;
  }
  if (num == 0) (void)cudaGetLastError();
  __atomic_store_n(&slot, num + 1, __ATOMIC_RELEASE);
  return num;
}

}  // namespace

static adt_status accept_impl(const float* target_logits, const float* target_u, int64_t ld_target,
                              const float* draft_logits, const float* draft_u, int64_t ld_draft,
                              const int32_t* draft_row, float cfg_scale, const int32_t* tokens,
                              const int32_t* parents, const int32_t* node_offsets, int32_t B, int32_t V,
                              int32_t max_nodes, const float* u_accept, const float* u_sample,
                              adt_accept_mode mode, float temperature, int32_t* path, int32_t max_path,
                              int32_t* accept_len, int32_t* bonus_token, void* workspace,
                              size_t workspace_bytes, void* stream) {
  (void)workspace;
  (void)workspace_bytes;
  ADT_REQUIRE(target_logits && tokens && parents && node_offsets && path && accept_len && bonus_token);
  ADT_REQUIRE(mode == ADT_ACCEPT_GREEDY || mode == ADT_ACCEPT_SPEC || mode == ADT_ACCEPT_SPEC_DET);
  ADT_REQUIRE(B >= 1 && V >= 1 && V <= 262144 && max_nodes >= 1 && max_path >= 1);
  if (max_nodes > kMaxNodes) return ADT_ERR_UNSUPPORTED;
  ADT_REQUIRE(ld_target >= V && ld_target % 4 == 0 && adt::aligned16(target_logits));
  if (mode != ADT_ACCEPT_GREEDY) {
    ADT_REQUIRE(u_accept && u_sample);
    ADT_REQUIRE(temperature > 0.f && temperature < 1e30f);
  }
  if (mode == ADT_ACCEPT_SPEC) {
    ADT_REQUIRE(draft_logits && ld_draft >= V && ld_draft % 4 == 0 && adt::aligned16(draft_logits));
  }
  if (target_u) {
    ADT_REQUIRE(adt::aligned16(target_u) && cfg_scale > -1e30f && cfg_scale < 1e30f);
    if (mode == ADT_ACCEPT_SPEC) ADT_REQUIRE(draft_u && adt::aligned16(draft_u));
  }
  adt::DeviceInfo info;
  adt_status st = adt::device_info(&info);
  if (st != ADT_OK) return st;
  int fit[4] = {0, 0, 0, 0};
  for (int i = 0; mode == ADT_ACCEPT_SPEC && i < 4; ++i) fit[i] = spec_clusters(info, 2 << i);
  const int cs = cluster_size_for(V, B, mode, fit);
  const int vs = slice_for(V, cs);
  const int nbuf = mode == ADT_ACCEPT_SPEC ? 2 : 1;
  // Double-float slices where they fit, fp32 slices otherwise.
  const size_t smem_df = static_cast<size_t>(vs) * sizeof(float2) * nbuf;
  const bool use_df = mode != ADT_ACCEPT_GREEDY && smem_df + sizeof(SampleShared) <= static_cast<size_t>(info.max_smem_optin);
  const size_t smem = mode == ADT_ACCEPT_GREEDY ? 0 : use_df ? smem_df : static_cast<size_t>(vs) * sizeof(float) * nbuf;
  if (smem + sizeof(SampleShared) > static_cast<size_t>(info.max_smem_optin)) return ADT_ERR_UNSUPPORTED;
  auto kern = mode == ADT_ACCEPT_GREEDY ? accept_greedy_kernel
              : mode == ADT_ACCEPT_SPEC
                  ? (use_df ? accept_sample_kernel<true, true> : accept_sample_kernel<false, true>)
                  : (use_df ? accept_sample_kernel<true, false> : accept_sample_kernel<false, false>);
  st = configure(kern, 2 * static_cast<int>(mode) + (use_df ? 1 : 0), info);
  if (st != ADT_OK) return st;
  AcceptParams p;
  p.target = target_logits;
  p.ldt = ld_target;
  p.draft = draft_logits;
  p.ldd = ld_draft;
  p.drow = draft_row;
  p.target_u = target_u;
  p.draft_u = target_u ? draft_u : nullptr;
  p.cfg = cfg_scale;
  p.tokens = tokens;
  p.parents = parents;
  p.offs = node_offsets;
  p.V = V;
  p.max_nodes = max_nodes;
  p.ua = u_accept;
  p.us = u_sample;
  p.T = temperature;
  p.use_T = mode != ADT_ACCEPT_GREEDY && temperature != 1.0f;
  p.path = path;
  p.max_path = max_path;
  p.alen = accept_len;
  p.bonus = bonus_token;
  p.err = info.error_word;
  p.wait_limit = adt::wait_limit(kWaitLimit) - 1;  // of 1: none (a poll lasts longer than a round)
  p.Vs = vs;

  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(cs * B), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = adt::as_stream(stream);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = adt::pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  ADT_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, p));
  return adt::launch_status();
}

namespace {

__global__ void exp_diff_probe_kernel(const float* a, const float* b, int n, double* out) {
  __shared__ float2 tab[64];
  dfl::exp_table_to_smem(tab);
  __syncthreads();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = dfl::to_double(dfl::df_exp_diff(a[i], b[i], tab));
}

}  // namespace

extern "C" {

adt_status adt_testing_exp_diff(const float* a, const float* b, int32_t n, double* out, void* stream) {
  ADT_REQUIRE(a && b && out && n >= 0);
  if (n == 0) return ADT_OK;
  exp_diff_probe_kernel<<<(n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024, 256, 0, adt::as_stream(stream)>>>(a, b, n,
                                                                                                         out);
  return adt::launch_status();
}

int32_t adt_testing_accept_cluster(int32_t V, int32_t B, adt_accept_mode mode, const int32_t* fit) {
  return cluster_size_for(V, B, mode, fit);
}

size_t adt_tree_accept_workspace_size(int32_t B, int32_t V) {
  (void)B;
  (void)V;
  return 0;
}

adt_status adt_tree_accept(const float* target_logits, int64_t ld_target,
                           const float* draft_logits, int64_t ld_draft, const int32_t* draft_row,
                           const int32_t* tokens, const int32_t* parents,
                           const int32_t* node_offsets, int32_t B, int32_t V, int32_t max_nodes,
                           const float* u_accept, const float* u_sample, adt_accept_mode mode,
                           float temperature, int32_t* path, int32_t max_path,
                           int32_t* accept_len, int32_t* bonus_token, void* workspace,
                           size_t workspace_bytes, void* stream) {
  adt::TraceRange trace_("adt_tree_accept");
  return accept_impl(target_logits, nullptr, ld_target, draft_logits, nullptr, ld_draft, draft_row, 0.f, tokens,
                     parents, node_offsets, B, V, max_nodes, u_accept, u_sample, mode, temperature, path, max_path,
                     accept_len, bonus_token, workspace, workspace_bytes, stream);
}

adt_status adt_tree_accept_cfg(const float* target_cond, const float* target_uncond, int64_t ld_target,
                               const float* draft_cond, const float* draft_uncond, int64_t ld_draft,
                               const int32_t* draft_row, float cfg_scale, const int32_t* tokens,
                               const int32_t* parents, const int32_t* node_offsets, int32_t B, int32_t V,
                               int32_t max_nodes, const float* u_accept, const float* u_sample,
                               adt_accept_mode mode, float temperature, int32_t* path, int32_t max_path,
                               int32_t* accept_len, int32_t* bonus_token, void* workspace,
                               size_t workspace_bytes, void* stream) {
  adt::TraceRange trace_("adt_tree_accept_cfg");
  ADT_REQUIRE(target_uncond);
  return accept_impl(target_cond, target_uncond, ld_target, draft_cond, draft_uncond, ld_draft, draft_row,
                     cfg_scale, tokens, parents, node_offsets, B, V, max_nodes, u_accept, u_sample, mode,
                     temperature, path, max_path, accept_len, bonus_token, workspace, workspace_bytes, stream);
}

}  // extern "C"
