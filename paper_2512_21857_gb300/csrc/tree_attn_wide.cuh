// Tree attention over 128 query rows at a time: trees of more than 64 nodes,
// and grouped query heads (two heads of one kv head share a CTA, so that each K
// and V tile is read once for both).  Included by tree_attn.cu,
// which holds the 64-row kernel and the shared helpers.
//
// A CTA's rows are either 128 consecutive nodes of one head (row_stride 128), or
// two heads of one kv head with 64 rows each (row_stride 64).  The CTAs of one
// (tree, head group) form a cluster; a tree's node count, known on the device
// only, decides how many tiles it has, and the cluster's CTAs are dealt to the
// tiles as key splits: a call sized for 256 nodes (two tiles) whose tree has 41
// spends all its CTAs on one tile.
//
// Warp roles (384 threads): warps 0-3 and 4-7 are two softmax groups that take
// the chunks of 128 keys in turn, each with its own S and P tile in tensor
// memory: while one group exponentiates a chunk, the tensor core makes the
// other's scores and adds the chunk before to O.  A thread owns one row
// (tensor-memory lane = row for M = 128), so row maxima and sums need no
// exchange within a chunk; the running maximum that P and O are scaled by
// passes from each chunk's warp to the next chunk's through shared memory.  P
// is the PV product's A operand in tensor memory; nothing of it goes through
// shared memory.  Warps 8-11 as in the 64-row kernel: K loads, S products, V
// loads, PV products.
//
// Bound by: the fixed cost of a launch (5000 cycles to the first scores, 4000
// to 7000 from the last PV product to the exit, the merge with it), and per
// chunk the latency of a group's turn (2600 cycles for scores to
// probabilities, two groups at a time) beside 64 KB of K and V a CTA (11 TB/s
// from L2 over all CTAs).  Per layer, the 64-row kernel before: 256 nodes, 32
// heads x 128, 2400 keys 29.9 -> 18.6 us; four trees of 33 to 64 nodes, 32 / 8
// heads x 128, 3500 to 6001 keys 54.1 -> 30.0 us; two trees of 192 nodes, 20 heads x 64,
// 693 and 577 keys 15.1 -> 12.3 us; 41 nodes in a call sized for 256, 32 heads
// x 128, 1203 keys 18.2 -> 10.2 us.  One accumulator and P apart from S (so
// that the next scores do not wait for the PV product) took the first from
// 22.2 to 19.0 us; K in half tiles with deeper rings and two N = 64 products a
// chunk 20.6 us.
#pragma once

#include <type_traits>

template <int D>
struct WideCfg {
  static constexpr int kRows = 128;
  static constexpr int kBlocks = D / 64;
  static constexpr int kBlock = kRows * 128;             // one column block of 128 rows
  static constexpr int kTile = kBlocks * kBlock;         // 128 rows x D
  static constexpr int kStageBytes = 2 * kTile;          // K tile, then V tile
  static constexpr int kStages = D == 128 ? 2 : 4;
  // A partial row of the merge, in 32-bit words: D = 128: D fp16 values, then
  // m, l and one exponent per half row; D = 64: D fp32 values, m, l, padding.
  // (17 times 16 bytes: 16-byte accesses of consecutive rows do not conflict.)
  static constexpr bool kHalfRows = D == 128;
  static constexpr int kRowStride = (kHalfRows ? D / 2 : D) + 4;
  static constexpr int kStageOff = kTile;                // after Q
  static constexpr int kDynSmem = kStageOff + kStages * kStageBytes + 1024;  // + alignment slack
  static constexpr uint32_t kOCol = 256;                 // after the two S tiles
  static constexpr uint32_t kPCol = 384;                 // two P tiles of 64 columns (128 bf16)
  static constexpr uint32_t kIdescS = sm100::idesc_bf16_f32(128, 128, 0, 0);
  static constexpr uint32_t kIdescO = sm100::idesc_bf16_f32(128, D, 0, 1);
  static_assert(kOCol + D <= kPCol && kPCol + 2 * 64 <= kTmemCols, "tensor memory");
  static_assert(kRows * kRowStride * 4 <= kStages * kStageBytes, "partial rows fit the idle ring");
};

constexpr int kWideThreads = 12 * 32;
constexpr int kWideSoftmax = 8 * 32;
constexpr int kWideRows = 128;

struct WideBarriers {
  uint64_t q_full;                 // Q and the tree chunks are in shared memory
  uint64_t k_full[kMaxStages], v_full[kMaxStages];
  uint64_t k_free[kMaxStages];     // the S product of the chunk in that slot finished
  uint64_t done[4];                // the PV product of chunk j finished (barrier j % 4)
  uint64_t s_full[2], s_free[2], p_full[2];  // per group
  uint64_t mu[2][4];               // the running maxima after a chunk are in shared memory, per group and warp
  uint64_t drain[2];
};

// tcgen05.ld / st, shape 32x32b: thread t of a warp reads or writes lane
// 32 (warp % 4) + t, consecutive columns.
__device__ __forceinline__ void tmem_ld_32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st_32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
      "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
      "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

// Waits for this thread's tensor-memory loads; r, their destination, is an
// operand so that no use of it moves above the wait.
__device__ __forceinline__ void tmem_wait_ld_into(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15])::"memory");
  asm volatile(""
               : "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]),
                 "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                 "+r"(r[30]), "+r"(r[31])::"memory");
}

// Two fp32 values in a 64-bit register pair, and the packed operations on them.
__device__ __forceinline__ uint64_t pack_u32x2(uint32_t lo, uint32_t hi) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(v) : "r"(lo), "r"(hi));
  return v;
}
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  return pack_u32x2(__float_as_uint(lo), __float_as_uint(hi));
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;\n" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void wide_softmax_sync() { asm volatile("bar.sync 1, 256;\n" ::: "memory"); }

// The owner's side of the merge: rows r_lo .. r_lo + rows_mine - 1 of the
// tile, from the S (<= kMost) splits' partial rows at rows_addr in their
// shared memory.  A thread combines 8 columns of kItems rows at a time: all
// their loads go out before any is used.  Weights 2^(m_c - M), times l_c where
// the partial is normalised.  Bound by the bytes between SMs (about 8 a
// cycle), so the owner's own split is read locally.
template <int D, int kMost>
__device__ __forceinline__ void wide_merge(const TcParams& p, const uint8_t* rows, int S, int split, int tiles, int qt,
                                           int rows_mine, int r_lo, int shift, int row0, int n, int node0, int h0) {
  using C = WideCfg<D>;
  constexpr int kC8 = D / 8, kVec = C::kHalfRows ? 1 : 2, kMlOff = C::kHalfRows ? D * 2 : D * 4;
  constexpr int kItems = kMost * kVec <= 4 ? 2 : 1;
  const uint32_t rows_addr = sm100::smem_addr(rows);
  const int items = rows_mine * kC8;
  for (int idx0 = threadIdx.x; idx0 < items; idx0 += kItems * kWideThreads) {
    uint4 ml[kItems][kMost], v[kItems][kMost][kVec];
#pragma unroll
    for (int t = 0; t < kItems; ++t) {
      const int idx = idx0 + t * kWideThreads, r = r_lo + idx / kC8, c8 = idx % kC8;
      if (idx >= items || row0 + (r & ((1 << shift) - 1)) >= n) continue;
#pragma unroll
      for (int c = 0; c < kMost; ++c) {
        if (c >= S) continue;
        const uint32_t off = r * C::kRowStride * 4;
        if (c == split) {
          ml[t][c] = *reinterpret_cast<const uint4*>(rows + off + kMlOff);
#pragma unroll
          for (int k = 0; k < kVec; ++k)
            v[t][c][k] = *reinterpret_cast<const uint4*>(rows + off + (c8 * kVec + k) * 16);
        } else {
          const uint32_t src = sm100::mapa_shared(rows_addr + off, c * tiles + qt);
          ml[t][c] = sm100::ld_cluster_v4(src + kMlOff);
#pragma unroll
          for (int k = 0; k < kVec; ++k) v[t][c][k] = sm100::ld_cluster_v4(src + (c8 * kVec + k) * 16);
        }
      }
    }
#pragma unroll
    for (int t = 0; t < kItems; ++t) {
      const int idx = idx0 + t * kWideThreads, r = r_lo + idx / kC8, c8 = idx % kC8;
      const int head = h0 + (r >> shift), nd = row0 + (r & ((1 << shift) - 1));
      if (idx >= items || nd >= n) continue;  // past the rows, or a gap between two heads' rows
      float M = -INFINITY;
#pragma unroll
      for (int c = 0; c < kMost; ++c)
        if (c < S) M = fmaxf(M, __uint_as_float(ml[t][c].x));
      float lt = 0.f;
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c = 0; c < kMost; ++c) {
        if (c >= S) continue;
        const float mc = __uint_as_float(ml[t][c].x), lc = __uint_as_float(ml[t][c].y);
        float w = mc == -INFINITY ? 0.f : ex2_approx(mc - M);
        lt += w * lc;
        if constexpr (C::kHalfRows) {
          w *= lc * __uint_as_float((127u + (c8 >= kC8 / 2 ? ml[t][c].w : ml[t][c].z)) << 23);
          const __half2* hv = reinterpret_cast<const __half2*>(&v[t][c][0]);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 f = __half22float2(hv[e]);
            acc[2 * e] += w * f.x;
            acc[2 * e + 1] += w * f.y;
          }
        } else {
          const float* f = reinterpret_cast<const float*>(&v[t][c][0]);
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[e] += w * f[e];
        }
      }
      const float inv = __fdividef(1.f, lt);
      uint4 pk;
      pk.x = pack_bf16x2(acc[0] * inv, acc[1] * inv);
      pk.y = pack_bf16x2(acc[2] * inv, acc[3] * inv);
      pk.z = pack_bf16x2(acc[4] * inv, acc[5] * inv);
      pk.w = pack_bf16x2(acc[6] * inv, acc[7] * inv);
      const int64_t o = static_cast<int64_t>(node0 + nd) * p.H + head;
      *reinterpret_cast<uint4*>(p.out + o * D + c8 * 8) = pk;
      if (c8 == 0 && p.lse) p.lse[o] = (M + __log2f(lt)) * kLn2;
    }
  }
}

template <int D>
__global__ void __launch_bounds__(kWideThreads, 1)
    tree_attn_wide_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                          const TcParams p) {
  using C = WideCfg<D>;
  constexpr int NS = C::kStages;
  constexpr int RS = C::kRowStride;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (sm100::smem_addr(smem_raw) & 1023u)) & 1023u);
  __shared__ WideBarriers bars;
  __shared__ __align__(16) uint32_t anc[kWideRows][2 * kMaxTreeUnits];  // ancestor bits of the tile's nodes
  __shared__ int s_par[kMaxTreeNodes];
  __shared__ float s_mu[kWideRows];
  __shared__ float2 s_ml[2][kWideRows];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  __shared__ int s_bad;

  const int rank = blockIdx.x;         // in the cluster, which spans the grid's x extent
  const int h0 = (static_cast<int>(blockIdx.y) - p.prefetch) * p.heads;  // first head of the group
  const int g = h0 / p.group;
  // Slot of the tree and, without a cluster, the tile: all first tiles come
  // before the second ones.
  const int slot = static_cast<int>(blockIdx.z) % p.B, tile_z = static_cast<int>(blockIdx.z) / p.B;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int kKLoad = 8, kSMma = 9, kVLoad = 10, kPvMma = 11;

  constexpr bool kPrefetch = D == 128;
  if (kPrefetch && h0 < 0) {
    if (tile_z == 0) {
      const int nodes = __ldcg(p.offs + slot + 1) - __ldcg(p.offs + slot);  // a hint, like the prefix length
      const int tiles = p.heads > 1 || gridDim.x == 1 ? 1 : min(max((nodes + kWideRows - 1) / kWideRows, 1), 2);
      const int S = static_cast<int>(gridDim.x) / tiles;
      // (Four chunks a split: with 2.75, H = 32, KV 1203, 41 nodes, a layer took 1.4 % longer.)
      if (__ldcg(p.kv_len + slot) >= 4 * S * kChunk) prefetch_stream<C::kBlocks>(&tm_k, &tm_v, p, slot, S, 2);
    }
    return;
  }
  // Set-up that touches no memory the previous kernel writes (see the 64-row
  // kernel).
  if (tid == 0) {
    s_abort = 0;
    s_bad = 0;
    sm100::mbar_init(sm100::smem_addr(&bars.q_full), 8);
    for (int s = 0; s < NS; ++s) {
      sm100::mbar_init(sm100::smem_addr(&bars.k_full[s]), 1);
      sm100::mbar_init(sm100::smem_addr(&bars.v_full[s]), 1);
      sm100::mbar_init(sm100::smem_addr(&bars.k_free[s]), 1);
    }
    for (int s = 0; s < 4; ++s) sm100::mbar_init(sm100::smem_addr(&bars.done[s]), 1);
    for (int s = 0; s < 2; ++s) {
      sm100::mbar_init(sm100::smem_addr(&bars.s_full[s]), 1);
      sm100::mbar_init(sm100::smem_addr(&bars.s_free[s]), 4);
      sm100::mbar_init(sm100::smem_addr(&bars.p_full[s]), 4);
      for (int w = 0; w < 4; ++w) sm100::mbar_init(sm100::smem_addr(&bars.mu[s][w]), 1);
      sm100::mbar_init(sm100::smem_addr(&bars.drain[s]), 1);
    }
    sm100::fence_mbar_init();
  }
  if (warp == 0) {
    sm100::tmem_alloc(sm100::smem_addr(&tmem_slot), kTmemCols);
    sm100::tmem_relinquish();
  }
  if (lane == 0 && (warp == kKLoad || warp == kVLoad)) sm100::prefetch_tensormap(warp == kKLoad ? &tm_k : &tm_v);
  sm100::tc_fence_before();
  __syncthreads();
  sm100::tc_fence_after();
  const uint32_t tmem = tmem_slot;

  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const TreeSlot ts = tree_of_slot(p, slot, lane);
  const int b = ts.b, node0 = ts.node0, n = ts.n, L = ts.L;
  const bool bad_tree = n < 1 || n > p.max_tree || node0 < 0 || node0 + n > ts.total_nodes;
  const bool bad_kv = L < 0 || L > p.max_kv;
  if (bad_tree || bad_kv) {
    if (rank == 0 && h0 == 0 && tile_z == 0 && tid == 0)
      adt::raise_error(p.err, bad_tree ? ADT_DEVERR_BAD_TREE : ADT_DEVERR_KV_RANGE);
    if (warp == 0) sm100::tmem_dealloc(tmem, kTmemCols);
    return;
  }

  // A cluster of several CTAs is dealt to the tree's tiles: CTA `rank` is
  // split rank / tiles of tile rank % tiles (it is sized for one or two tiles
  // with an equal number of splits each, so the tiles divide it).  Clusters of
  // one CTA each have a tile of their own; one past the tree's last ends here.
  const int tiles = p.heads > 1 ? 1 : (n + kWideRows - 1) / kWideRows;
  const bool dealt = gridDim.x > 1;
  const int S = dealt ? static_cast<int>(gridDim.x) / tiles : 1;
  const int qt = dealt ? rank % tiles : tile_z, split = dealt ? rank / tiles : 0;
  if (qt >= tiles) {
    if (warp == 0) sm100::tmem_dealloc(tmem, kTmemCols);
    return;
  }
  const int row0 = qt * kWideRows;
  const int stride = p.row_stride;  // rows of one head: 128 (one head) or 64 (two)
  const int shift = stride == kWideRows ? 7 : 6;
  const int nrows = p.heads > 1 ? (p.heads - 1) * stride + n : min(n - row0, kWideRows);
  // Chunks of 128 keys: ceil(L / 128) of the prefix, then tree chunks 0 .. qt
  // (a node's ancestors come before it).
  const int Pc = (L + kChunk - 1) / kChunk;
  // Split s takes a contiguous share; a tree chunk (ancestor bits, masks)
  // counts for two.
  const int W = Pc + 2 * (qt + 1);
  auto chunk_at = [&](int w) { return w <= Pc ? w : Pc + (w - Pc) / 2; };
  const int c_begin = chunk_at(split * W / S);
  const int c_end = chunk_at((split + 1) * W / S);
  const int nch = c_end - c_begin;
  const int tc0 = max(c_begin, Pc) - Pc;
  const int n_tc = max(0, c_end - max(c_begin, Pc));  // tree chunks, in slots 0 .. n_tc-1 (at most two)

  // Keys from chunk j's first one on (128 or more: the chunk is full).
  auto chunk_keys = [&](int j) -> int {
    return j < n_tc ? n - (tc0 + j) * kChunk : L - (c_begin + j - n_tc) * kChunk;
  };

  uint8_t* sQ = smem;
  uint8_t* sStage = smem + C::kStageOff;

  const bool is_loader = (warp == kKLoad || warp == kVLoad) && lane == 0;
  const bool load_v = warp == kVLoad;
  auto issue_tile = [&](int j) {
    const int st = j % NS;
    const uint32_t bar = sm100::smem_addr(load_v ? &bars.v_full[st] : &bars.k_full[st]);
    if (j < n_tc) {
      sm100::mbar_arrive(bar);
      return;
    }
    const uint32_t dst = sm100::smem_addr(sStage) + st * C::kStageBytes + (load_v ? C::kTile : 0);
    sm100::mbar_arrive_expect_tx(bar, C::kTile);
    for (int blk = 0; blk < C::kBlocks; ++blk)
      sm100::tma_load_4d(dst + blk * C::kBlock, load_v ? &tm_v : &tm_k, blk * 64, (c_begin + j - n_tc) * kChunk, g, b,
                         bar);
  };
  const int first_issue = nch < NS ? nch : NS;
  // The first K tile goes out at once, the other stages after Q (queued
  // behind all of them, Q would hold back the first S product).
  if (is_loader && !load_v && nch > 0) issue_tile(0);
  if (tid < kWideSoftmax) {
    // The parent pointers, Q (rows without a node zero-filled), the tree
    // chunks' K and V: thread t copies 16-byte column t % (D / 8) of every
    // kRowsPass-th row.
    if (tid < n) cp_async4(sm100::smem_addr(&s_par[tid]), p.parents + node0 + tid);
    constexpr int kCh = D / 8, kRowsPass = kWideSoftmax / kCh;
    const int ch = tid % kCh, r0 = tid / kCh;
    if (nch > 0) {
      const __nv_bfloat16* q = p.q + (static_cast<int64_t>(node0) * p.H + h0) * D + ch * 8;
      const uint32_t dq = sm100::smem_addr(sQ);
#pragma unroll
      for (int r = r0; r < kWideRows; r += kRowsPass) {
        const int hh = r >> shift, node = row0 + (r & (stride - 1));
        const bool valid = hh < p.heads && node < n;
        cp_async16(dq + sw128_off(r, ch, kWideRows), q + (valid ? (static_cast<int64_t>(node) * p.H + hh) * D : 0),
                   valid ? 16 : 0);
      }
    }
    for (int jt = 0; jt < n_tc; ++jt) {
      const int64_t step = static_cast<int64_t>(p.Hkv) * D;
      const int64_t off = (static_cast<int64_t>(node0) * p.Hkv + g) * D + ch * 8;
      const uint32_t dk = sm100::smem_addr(sStage) + jt * C::kStageBytes;
#pragma unroll 4
      for (int r = r0; r < kChunk; r += kRowsPass) {
        const int t = (tc0 + jt) * kChunk + r;
        const int64_t o = off + (t < n ? t * step : 0);
        cp_async16(dk + sw128_off(r, ch, kChunk), p.kt + o, t < n ? 16 : 0);
        cp_async16(dk + C::kTile + sw128_off(r, ch, kChunk), p.vt + o, t < n ? 16 : 0);
      }
    }
  }
  __syncthreads();  // Q's copies are requested
  if (is_loader) {
    for (int j = load_v ? 0 : 1; j < first_issue; ++j) issue_tile(j);
  }

  auto wait = [&](uint64_t* bar, int phase) { return wait_bar(bar, phase & 1, &s_abort, p.err, p.wait_limit); };
  // PV(j) done.  A wait on a barrier's parity is only meaningful once the
  // phase before is complete, so no one waits for PV(j) without knowing PV(j -
  // 4) done: the loader's slots, and a softmax group's own last P tile, see to
  // that (with the two barriers that the two slots of D = 128 would need, a
  // group could ask for PV(j - 1) while PV(j - 3) was still running).
  auto wait_done = [&](int j) { return wait(&bars.done[j & 3], j >> 2); };

  if (warp == kKLoad || warp == kVLoad) {
    // ------------------------------------------------------------ K / V loads
    if (lane == 0) {
      int issued = first_issue;
      for (int j = first_issue; j < nch; ++j) {
        if (load_v ? !wait_done(j - NS) : !wait(&bars.k_free[j % NS], j / NS - 1)) break;
        issue_tile(j);
        ++issued;
      }
      if (kPrefetch && p.prefetch && !load_v) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
      // Every copy issued lands before the CTA goes on (also after an abort).
      for (int j = (issued > NS ? issued - NS : 0); j < issued; ++j)
        (void)sm100::mbar_wait_bounded(sm100::smem_addr(load_v ? &bars.v_full[j % NS] : &bars.k_full[j % NS]),
                                       (j / NS) & 1, kWaitLimit);
    }
    __syncwarp();
  } else if (warp == kSMma) {
    // ------------------------------------------------------------ S = Q K^T
    if (lane == 0) {
      const uint32_t q_addr = sm100::smem_addr(sQ);
      bool ok = nch == 0 || wait(&bars.q_full, 0);
      for (int j = 0; ok && j < nch; ++j) {
        if (!wait(&bars.k_full[j % NS], j / NS) || (j >= 2 && !wait(&bars.s_free[j & 1], (j >> 1) - 1))) break;
        sm100::tc_fence_after();
        const uint32_t k_addr = sm100::smem_addr(sStage) + (j % NS) * C::kStageBytes;
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t off = (kk >> 2) * C::kBlock + (kk & 3) * 32;
          sm100::mma_bf16_ss(tmem + (j & 1) * kSCols, sm100::smem_desc_sw128(q_addr + off, 16, 1024),
                             sm100::smem_desc_sw128(k_addr + off, 16, 1024), C::kIdescS, kk > 0 ? 1u : 0u);
        }
        sm100::mma_commit(sm100::smem_addr(&bars.s_full[j & 1]));
      }
      sm100::mma_commit(sm100::smem_addr(&bars.drain[0]));
      (void)sm100::mbar_wait_bounded(sm100::smem_addr(&bars.drain[0]), 0, kWaitLimit);
    }
    __syncwarp();
  } else if (warp == kPvMma) {
    // ------------------------------------------------------------ O += P V
    if (lane == 0) {
      bool ok = nch == 0 || wait(&bars.q_full, 0);
      for (int j = 0; ok && j < nch; ++j) {
        if (!wait(&bars.p_full[j & 1], j >> 1) || !wait(&bars.v_full[j % NS], j / NS)) break;
        sm100::tc_fence_after();
        const uint32_t v_addr = sm100::smem_addr(sStage) + (j % NS) * C::kStageBytes + C::kTile;
        const uint32_t a = tmem + C::kPCol + (j & 1) * 64;
        // Keys past the prefix need no product (the rest of the last 16 are
        // zero in P and in V).
        const int ksteps = min(kChunk / 16, (chunk_keys(j) + 15) / 16);
        // (Whole chunks unrolled: 30.8 against 31.0 us at H = 32, Hkv = 8, KV
        // 3500-6001.  Unrolled with a condition on every product: 32.7 us.)
        const uint64_t vd = sm100::smem_desc_sw128(v_addr, C::kBlock, 1024);
        sm100::mma_bf16_ts(tmem + C::kOCol, a, vd, C::kIdescO, j > 0 ? 1u : 0u);
        if (ksteps == kChunk / 16) {
#pragma unroll
          for (int kk = 1; kk < kChunk / 16; ++kk)
            sm100::mma_bf16_ts(tmem + C::kOCol, a + kk * 8, vd + kk * 128, C::kIdescO, 1u);
        } else {
          for (int kk = 1; kk < ksteps; ++kk)
            sm100::mma_bf16_ts(tmem + C::kOCol, a + kk * 8, vd + kk * 128, C::kIdescO, 1u);
        }
        sm100::mma_commit(sm100::smem_addr(&bars.done[j & 3]));
      }
      sm100::mma_commit(sm100::smem_addr(&bars.drain[1]));
      (void)sm100::mbar_wait_bounded(sm100::smem_addr(&bars.drain[1]), 0, kWaitLimit);
    }
    __syncwarp();
  }

  // The softmax warps' row and the state of their group.
  const int stream = warp >> 2;
  const int row = (warp & 3) * 32 + lane;
  const uint32_t lanes = static_cast<uint32_t>((warp & 3) * 32) << 16;
  const int hh = row >> shift, node = row0 + (row & (stride - 1));
  const bool valid = hh < p.heads && node < n;
  if (tid < kWideSoftmax) {
    // ------------------------------------------------------------ softmax warps
    const bool active = __any_sync(adt::kFullMask, valid);  // a warp without rows only keeps the barriers moving
    cp_async_wait_all();
    sm100::fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.q_full));
    // Parents precede their children; anything else marks the tree malformed:
    // every CTA of it sees all its nodes (a thread its own copy), and none
    // writes a row.
    static_assert(kMaxTreeNodes <= kWideSoftmax, "a thread checks a node");
    if (tid < n) {
      const int par = s_par[tid];
      if ((tid == 0) != (par < 0) || par >= tid) {
        s_bad = 1;
        adt::raise_error(p.err, ADT_DEVERR_BAD_TREE);
      }
    }
    // While the first products run, where this split has a tree chunk: the
    // ancestor bits of the tile's nodes (of a malformed tree, to where a
    // parent does not precede its child).
    if (n_tc > 0) {
      static_assert(kWideRows * 2 == kWideSoftmax, "two threads clear a node's bits");
      reinterpret_cast<uint4*>(anc)[tid] = make_uint4(0u, 0u, 0u, 0u);
      wide_softmax_sync();
      if (tid < kWideRows && row0 + tid < n) {
        int j = row0 + tid;
        for (;;) {
          atomicOr(&anc[tid][j >> 5], 1u << (j & 31));
          const int par = s_par[j];
          if (par < 0 || par >= j) break;
          j = par;
        }
      }
      wide_softmax_sync();
    }
    const uint32_t s_col = tmem + lanes + stream * kSCols;
    const uint32_t o_col = tmem + lanes + C::kOCol, p_col = tmem + lanes + C::kPCol + stream * 64;
    const int w4 = warp & 3;
    const float scale = p.scale_log2;
    float mu = -INFINITY, l = 0.f;
    for (int j = stream; j < nch; j += 2) {
      if (!__all_sync(adt::kFullMask, wait(&bars.s_full[stream], j >> 1))) break;
      // S(j) is complete, so its K tile can be refilled.
      if ((warp & 3) == 0 && lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.k_free[j % NS]));
      sm100::tc_fence_after();
      const bool tree_j = j < n_tc;
      const int kl = chunk_keys(j);
      const int quarters = min(4, (kl + 31) / 32);  // of 32 keys
      if (active) {
        if (tree_j || kl < kChunk) {
          // -inf where the row does not see the key, in place.
          const uint32_t* bits = anc[valid ? node - row0 : 0] + (tree_j ? 4 * (tc0 + j) : 0);
#pragma unroll 1
          for (int s = 0; s < quarters; ++s) {
            const int k = kl - 32 * s;
            const uint32_t keep = tree_j ? bits[s] : k >= 32 ? ~0u : (1u << k) - 1u;
            uint32_t r[32];
            tmem_ld_32(s_col + 32 * s, r);
            tmem_wait_ld_into(r);
#pragma unroll
            for (int e = 0; e < 32; ++e) r[e] = (keep >> e) & 1u ? r[e] : 0xFF800000u;
            tmem_st_32(s_col + 32 * s, r);
          }
          sm100::tmem_wait_st();
        }
        uint32_t x[32], y[32];
        float mq[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        auto largest = [&](const uint32_t (&r)[32]) {
#pragma unroll
          for (int e = 0; e < 32; e += 2)
            mq[(e >> 1) & 3] = fmaxf(fmaxf(mq[(e >> 1) & 3], __uint_as_float(r[e])), __uint_as_float(r[e + 1]));
        };
        // The quarters in turn, each loaded while the one before is used; at
        // the end the first one again, for the exponentials.
        tmem_ld_32(s_col, x);
        tmem_wait_ld_into(x);
        if (quarters == 4) {
#pragma unroll
          for (int s = 0; s < 4; s += 2) {
            tmem_ld_32(s_col + 32 * s + 32, y);
            largest(x);
            tmem_wait_ld_into(y);
            tmem_ld_32(s_col + (s == 0 ? 64 : 0), x);
            largest(y);
            tmem_wait_ld_into(x);
          }
        } else {
          largest(x);
#pragma unroll 1
          for (int s = 1; s < quarters; ++s) {
            tmem_ld_32(s_col + 32 * s, y);
            tmem_wait_ld_into(y);
            largest(y);
          }
        }
        const float mx = fmaxf(fmaxf(mq[0], mq[1]), fmaxf(mq[2], mq[3])) * scale;  // scale > 0
        // The running maximum after the chunk before (the other group's).
        float prev = -INFINITY;
        if (j > 0) {
          if (!__all_sync(adt::kFullMask, wait(&bars.mu[stream ^ 1][w4], (j - 1) >> 1))) break;
          prev = s_mu[row];
        }
        // It is raised only when a row grows by more than 2^8; then O (once
        // the chunks before are in it) is scaled.
        const float nm = mx > prev + kRescaleThreshold ? mx : prev;
        s_mu[row] = nm;
        __syncwarp();
        if (lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.mu[stream][w4]));
        if (nm != mu) l *= ex2_approx(mu - nm);
        // P's tile was last read by the PV product of chunk j - 2.
        if (j >= 2 && !__all_sync(adt::kFullMask, wait_done(j - 2))) break;
        if (j > 0 && __any_sync(adt::kFullMask, nm != prev)) {
          if (!__all_sync(adt::kFullMask, wait_done(j - 1))) break;
          sm100::tc_fence_after();
          const float alpha = nm == prev ? 1.f : ex2_approx(prev - nm);
#pragma unroll 1
          for (int c = 0; c < D; c += 32) {
            uint32_t r[32];
            tmem_ld_32(o_col + c, r);
            tmem_wait_ld_into(r);
#pragma unroll
            for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * alpha);
            tmem_st_32(o_col + c, r);
          }
        }
        mu = nm;
        sm100::tc_fence_after();
        const float base = mu == -INFINITY ? 0.f : mu;
        const uint64_t scale2 = pack_f32x2(scale, scale), base2 = pack_f32x2(-base, -base);
        uint64_t l2[2] = {0ull, 0ull};  // two pairs of partial sums
        // 32 scores -> 16 pairs of bf16 probabilities; the row sum adds the
        // rounded values, the ones V is weighted with.  Scaling and sums take
        // two fp32 values an instruction.
        auto quarter = [&](const uint32_t (&r)[32], int s) {
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            float a0, a1;
            unpack_f32x2(fma_f32x2(pack_u32x2(r[2 * e], r[2 * e + 1]), scale2, base2), a0, a1);
            pk[e] = pack_bf16x2(ex2_approx(a0), ex2_approx(a1));
            l2[e & 1] = add_f32x2(l2[e & 1], pack_u32x2(pk[e] << 16, pk[e] & 0xFFFF0000u));
          }
          tmem_st_16(p_col + 16 * s, pk);
        };
        auto release_s = [&]() {  // S is in registers: its tile may be written again
          sm100::tc_fence_before();
          __syncwarp();
          if (lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.s_free[stream]));
        };
        if (quarters == 4) {
#pragma unroll 1
          for (int s = 0; s < 4; s += 2) {
            tmem_ld_32(s_col + 32 * s + 32, y);
            quarter(x, s);
            tmem_wait_ld_into(y);
            if (s == 0)
              tmem_ld_32(s_col + 64, x);
            else
              release_s();
            quarter(y, s + 1);
            tmem_wait_ld_into(x);
          }
        } else {
#pragma unroll 1
          for (int s = 0; s < quarters; ++s) {
            if (s > 0) {
              tmem_ld_32(s_col + 32 * s, x);
              tmem_wait_ld_into(x);
            }
            quarter(x, s);
          }
          release_s();
        }
        float la, lb, lc, ld;
        unpack_f32x2(l2[0], la, lb);
        unpack_f32x2(l2[1], lc, ld);
        l += (la + lb) + (lc + ld);
        sm100::tmem_wait_st();
      } else {
        // A warp without rows has nothing to do for the chunk, but stays
        // within it as the others do: its arrival for P(j) must not fall into
        // the phase of P(j - 2), nor may it touch a V slot that PV(j - 2) reads.
        if (lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.s_free[stream]));
        if (j >= 2 && !__all_sync(adt::kFullMask, wait_done(j - 2))) break;
      }
      // Cache rows past the prefix can hold anything: zero those the last
      // 16-key product step still reads.
      if (!tree_j && (kl & 15) != 0 && kl < kChunk) {
        if (!__all_sync(adt::kFullMask, wait(&bars.v_full[j % NS], j / NS))) break;
        uint8_t* vt = sStage + (j % NS) * C::kStageBytes + C::kTile;
        const int per_row = C::kBlocks * 8, end = (kl + 15) & ~15;
        for (int i = (tid & 127); i < (end - kl) * per_row; i += 128) {
          const int rr = kl + i / per_row, rem = i % per_row;
          *reinterpret_cast<uint4*>(vt + (rem >> 3) * C::kBlock + rr * 128 + (rem & 7) * 16) =
              make_uint4(0u, 0u, 0u, 0u);
        }
        sm100::fence_proxy_async_smem();
      }
      sm100::tc_fence_before();
      __syncwarp();
      if (lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.p_full[stream]));
    }
    s_ml[stream][row] = make_float2(mu, l);
  }

  // ------------------------------------------------------------ epilogue
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  // A thread takes half of its row's columns of O (group 0 the lower half);
  // the row sum is the two groups' sums at the last maximum.
  constexpr int kHalf = D / 2;
  float o[kHalf];
  float m = -INFINITY, l = 0.f;
  if (tid < kWideSoftmax) {
    bool have = __all_sync(adt::kFullMask, nch > 0 && !s_abort);
    for (int j = max(0, nch - 2); have && j < nch; ++j) have = __all_sync(adt::kFullMask, wait_done(j));
    wide_softmax_sync();
    sm100::tc_fence_after();
#pragma unroll
    for (int s = 0; s < kHalf; s += 32) {
      uint32_t x[32];
      if (have) {
        tmem_ld_32(tmem + lanes + C::kOCol + stream * kHalf + s, x);
        tmem_wait_ld_into(x);
      }
#pragma unroll
      for (int e = 0; e < 32; ++e) o[s + e] = have ? __uint_as_float(x[e]) : 0.f;
    }
    if (have) {
      const float2 a = s_ml[0][row], c = s_ml[1][row];
      m = fmaxf(a.x, c.x);
      l = (a.x > -INFINITY ? ex2_approx(a.x - m) * a.y : 0.f) + (c.x > -INFINITY ? ex2_approx(c.x - m) * c.y : 0.f);
      if (!(l > 0.f)) m = -INFINITY;  // no key of this split is visible to the row
    }
  }
  sm100::tc_fence_before();

  if (S == 1) {
    // No other split: the row is final.
    if (tid < kWideSoftmax && valid && !s_bad) {
      const float inv = __fdividef(1.f, l);
      __nv_bfloat16* dst = p.out + (static_cast<int64_t>(node0 + node) * p.H + h0 + hh) * D + stream * kHalf;
#pragma unroll
      for (int e = 0; e < kHalf; e += 8) {
        uint4 pk;
        pk.x = pack_bf16x2(o[e] * inv, o[e + 1] * inv);
        pk.y = pack_bf16x2(o[e + 2] * inv, o[e + 3] * inv);
        pk.z = pack_bf16x2(o[e + 4] * inv, o[e + 5] * inv);
        pk.w = pack_bf16x2(o[e + 6] * inv, o[e + 7] * inv);
        *reinterpret_cast<uint4*>(dst + e) = pk;
      }
      if (stream == 0 && p.lse)
        p.lse[static_cast<int64_t>(node0 + node) * p.H + h0 + hh] = (m + __log2f(l)) * kLn2;
    }
    __syncthreads();
    sm100::tc_fence_after();
    if (warp == 0) sm100::tmem_dealloc(tmem, kTmemCols);
    return;
  }

  // Row r of the tile is merged by split r / rows_per, its owner: every split
  // leaves its partial rows in its idle ring, and the owners read them there
  // through distributed shared memory.
  const int rows_per = (nrows + S - 1) / S;
  const int r_lo = split * rows_per;
  const int rows_mine = max(0, min(nrows, r_lo + rows_per) - r_lo);
  float* rows_out = reinterpret_cast<float*>(sStage);
  if (tid < kWideSoftmax) {
    if (row < nrows) {
      float* dst = rows_out + row * RS;
      if (stream == 0) *reinterpret_cast<float2*>(dst + (C::kHalfRows ? D / 2 : D)) = make_float2(m, l);
      if constexpr (C::kHalfRows) {
        // O / l in fp16 scaled by a power of two that puts the half row's largest
        // magnitude in [2^14, 2^15) (see the 64-row kernel).
        const float inv = l > 0.f ? __fdividef(1.f, l) : 0.f;
        float amax = 0.f;
#pragma unroll
        for (int e = 0; e < kHalf; ++e) amax = fmaxf(amax, fabsf(o[e]));
        amax *= inv;
        const int ex = static_cast<int>((__float_as_uint(amax) >> 23) & 0xFFu);
        const int e2 = amax > 0.f ? min(max(ex - 127 - 14, -110), 110) : 0;
        const float sc = inv * __uint_as_float(static_cast<uint32_t>(127 - e2) << 23);
        reinterpret_cast<int*>(dst)[D / 2 + 2 + stream] = e2;
        uint32_t* hv = reinterpret_cast<uint32_t*>(dst) + stream * (kHalf / 2);
#pragma unroll
        for (int e = 0; e < kHalf; e += 8) {
          uint4 pk;
          pk.x = pack_half2(o[e] * sc, o[e + 1] * sc);
          pk.y = pack_half2(o[e + 2] * sc, o[e + 3] * sc);
          pk.z = pack_half2(o[e + 4] * sc, o[e + 5] * sc);
          pk.w = pack_half2(o[e + 6] * sc, o[e + 7] * sc);
          *reinterpret_cast<uint4*>(hv + e / 2) = pk;
        }
      } else {
#pragma unroll
        for (int e = 0; e < kHalf; e += 4)
          *reinterpret_cast<float4*>(dst + stream * kHalf + e) = make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]);
      }
    }
  }
  __syncwarp();
  sm100::cluster_arrive_release();
  sm100::cluster_wait_acquire();
  auto merge = [&](auto most) {
    wide_merge<D, decltype(most)::value>(p, reinterpret_cast<const uint8_t*>(rows_out), S, split, tiles, qt,
                                         s_bad ? 0 : rows_mine, r_lo, shift, row0, n, node0, h0);
  };
  if (S <= 2)
    merge(std::integral_constant<int, 2>());
  else if (S <= 4)
    merge(std::integral_constant<int, 4>());
  else
    merge(std::integral_constant<int, kMaxClusterSplits>());
  __syncwarp();
  sm100::cluster_arrive_relaxed();
  sm100::cluster_wait_acquire();  // every owner has read this CTA's rows
  sm100::tc_fence_after();
  if (warp == 0) sm100::tmem_dealloc(tmem, kTmemCols);
}
