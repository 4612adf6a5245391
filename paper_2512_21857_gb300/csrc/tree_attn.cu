// adt_tree_attn: tree-masked attention of the draft-tree nodes over the
// prefix KV cache and their own ancestors (Sec. 3.1: every node is verified
// conditioned on s_{1:t} and ans(t) under the tree mask; the mask is the
// T_N term of Eq. 5).
//
// Split-KV flash decoding on the 5th-generation tensor cores.  A tree's
// nodes (<= 256) are cut into query tiles of 64 rows; the keys a tile sees
// are cut into units of 64: ceil(L/64) prefix units plus the tree units up
// to its own (a node's ancestors come before it), masked per query row by an
// ancestor bitmask, one 64-bit word per tree unit, built from the parent
// pointers.  Grid = (splits, H, B x tiles), one CTA per SM; a CTA handles one
// (tree, head, tile) and a contiguous share of the units, which it walks in
// chunks of two units (128 keys): its tree chunks first (their K/V are
// loaded with Q), then its prefix chunks.
//
// Warp roles inside a CTA (256 threads; one thread of each of warps 4-7):
//   warp 4    TMA tensor loads of prefix K (boxes of 128 keys x 64 columns,
//             128-byte swizzle) into a ring of 128-key stages;
//   warp 5    tcgen05.mma S = Q K^T into one of two tensor-memory tiles
//             (M = 64 queries, N = 128 keys), back to back (softmax warp 0
//             frees each K tile once it sees its S product done);
//   warp 6    TMA loads of prefix V into the same stages;
//   warp 7    tcgen05.mma O += P V (N = head_dim, V read MN-major);
//   warps 0-3 softmax: warp w owns query rows 16w .. 16w+15 (tensor-memory
//             lanes 32w .. 32w+15 for M = 64), read with the 16x256b shape so
//             that each thread holds two rows; exponentiates against a lazily
//             raised running maximum (O is rescaled only when a row maximum
//             grows by more than 2^8), writes P (bf16) with stmatrix for the
//             PV product, and at the end reads O and l for the merge.
// K and V of a stage are released separately (K when S is done, V and the P
// buffer when PV is done), and S and PV are issued by different threads, so
// loads of later chunks never queue behind the softmax of earlier ones.
// Every mbarrier wait is bounded; a timeout sets ADT_DEVERR_TIMEOUT.
//
// The splits of one (tree, head) form a thread-block cluster (<= 8).  Each
// split pushes its partial rows (O, running max, row sum) into the shared
// memory of the split that owns those rows, which then merges them locally;
// at D = 128 a row travels as O / l in fp16 with a power-of-two scale (half
// the bytes of fp32, which the copies between SMs are bound by).  With more
// splits they merge through the workspace.
//
// Back-to-back launches at the 7B shape (four splits, 41.4 MB, 6.1 us at the
// measured HBM rate) take 11.3 to 11.8 us, at the LlamaGen shape (six splits,
// from L2) 7.1 us: the chain from the dependency wait through the first loads
// to the merge, whose instructions come cold for each launch.  So one copy of
// the softmax serves every chunk, masks are bit tests on one word per row, the
// merge is unrolled for the split count's range, and paths off the common one
// lie behind it (7.4 us at the LlamaGen shape with two softmax copies, 64-bit
// masks and an eight-way merge inline).  The first S product follows the block
// barrier after the ancestor walk, but not what the softmax warps do next (the V
// rows past the tree zeroed, their arrival), and four threads send the merge's
// rows (7.3 us without these two).  One split writes its rows directly (eight
// ragged trees, 41.9 -> 38.4 us a layer).
//
// Where the 7B launch's 11 us from the dependency wait to the end went before
// its first chunks were prefetched (cycles at 1.93 GHz): 1500 to the first load,
// 4000 to the first K tile (every CTA's first 128 KB at once), 8800 for the
// stream (6.3 TB/s), then 1700 for the last softmax, 1800 for its PV product,
// 1000 to write the partial rows, 1900 to move them, 800 to merge.  Spare
// clusters now prefetch during those last phases of the launch before (see
// prefetch_stream, 12.5 -> 11.3 us); prefetches by the CTAs that compute made it
// slower or no faster (12.5-13.5 us): they delay the tiles that are needed
// first.
//
// Launches with long key ranges per CTA whose tiles can hold more than 64 rows
// (trees of more than 64 nodes, grouped query heads) take the 128-row kernel
// of tree_attn_wide.cuh instead (see wide_heads).
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_fp16.h>

#include <mutex>
#include <type_traits>

#include "adt_common.cuh"
#include "sm100.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kUnit = 64;               // keys per split unit; the tree unit
constexpr int kChunk = 128;             // keys per pipeline chunk
constexpr int kMaxNodes = 64;           // query rows per CTA: one tile of a tree's nodes
constexpr int kMaxTreeNodes = 256;      // nodes per tree: up to four query tiles
constexpr int kMaxTreeUnits = kMaxTreeNodes / kUnit;
static_assert(kMaxTreeUnits == 4, "the ancestor walk keeps four mask words");
constexpr int kSoftmaxWarps = 4;
constexpr int kKLoadWarp = 4;
constexpr int kSMmaWarp = 5;
constexpr int kVLoadWarp = 6;
constexpr int kPvMmaWarp = 7;
constexpr int kThreads = 8 * 32;
constexpr int kMaxClusterSplits = 8;    // portable cluster size
constexpr int kMaxSplits = 96;          // workspace merge: weights fit in shared memory
constexpr int kMaxStages = 4;
constexpr uint32_t kWaitLimit = 1u << 20;
constexpr int kTmaRows = 1 << 24;       // node extent of the Q / tree tensor maps (boxes are kept inside the buffers)
constexpr uint32_t kTmemCols = 512;     // two S tiles of 128 columns, O (<= 128 columns), row sums
constexpr uint32_t kSCols = 128;
constexpr uint32_t kOCol = 256;
constexpr uint32_t kLCols = 16;         // P times a tile of ones: every column holds the row sum
constexpr float kLn2 = 0.69314718055994530942f;
constexpr float kLog2e = 1.44269504088896340736f;
constexpr float kRescaleThreshold = 8.0f;  // log2 units

template <int D>
struct Cfg {
  static constexpr int kBlocks = D / 64;                 // 128-byte column blocks per row
  static constexpr int kBlock64 = kUnit * 128;           // one column block of 64 rows
  static constexpr int kBlock128 = kChunk * 128;         // one column block of 128 rows
  static constexpr int kTreeTile = kBlocks * kBlock64;   // 64 rows x D
  static constexpr int kStageTile = kBlocks * kBlock128; // 128 rows x D
  static constexpr int kStageBytes = 2 * kStageTile;     // K tile, then V tile
  static constexpr int kPBytes = 2 * kBlock64;           // 64 query rows x 128 keys
  static constexpr int kStages = D == 128 ? 2 : 4;
  // A partial row of the cluster merge, in 32-bit words.  D = 128: D fp16
  // values (O / l scaled by 2^-e), then m, l (fp32) and e (int32), padded to
  // 16 bytes; D = 64: D fp32 values (O), m, l, padding (distributed shared
  // memory moves its rows fast enough that the conversions would cost more
  // than the halved bytes save).
  static constexpr bool kHalfRows = D == 128;
  static constexpr int kRowStride = kHalfRows ? D / 2 + 4 : D + 8;
  static constexpr int kQOff = 0;
  static constexpr int kPOff = kTreeTile;                // Q is 64 rows x D, like a tree tile
  static constexpr int kStageOff = kPOff + 2 * kPBytes;  // the tree unit's K/V go to slot 0
  static constexpr int kSlotOff = kStageOff + kStages * kStageBytes;  // incoming rows of the merge
  static constexpr int kSlotBytes = (kMaxNodes + kMaxClusterSplits) * kRowStride * 4;
  static constexpr int kOnesOff = (kSlotOff + kSlotBytes + 1023) / 1024 * 1024;  // 16 rows of ones (bf16)
  static constexpr int kOnesBytes = 16 * 128;
  static constexpr int kDynSmem = kOnesOff + kOnesBytes + 1024;  // + alignment slack
  static constexpr uint32_t kLCol = kOCol + D;
  static constexpr uint32_t kIdescS128 = sm100::idesc_bf16_f32(64, 128, 0, 0);
  static constexpr uint32_t kIdescS64 = sm100::idesc_bf16_f32(64, 64, 0, 0);
  static constexpr uint32_t kIdescO = sm100::idesc_bf16_f32(64, D, 0, 1);
  static constexpr uint32_t kIdescL = sm100::idesc_bf16_f32(64, kLCols, 0, 1);
  static_assert(kLCol + kLCols <= kTmemCols, "tensor memory");
  static_assert(kStages <= kMaxStages, "stage ring");
};

struct TcParams {
  const __nv_bfloat16* q;
  const __nv_bfloat16* kt;
  const __nv_bfloat16* vt;
  const int32_t* kv_len;
  const int32_t* parents;
  const int32_t* offs;
  int B, H, Hkv, group, max_kv, splits;
  int prefetch;       // leading blockIdx.y rows of clusters that only prefetch (see prefetch_stream)
  int qtiles;         // 64-row query tiles per tree: ceil(max_nodes / 64)
  int cluster_merge;
  int max_tree;       // largest tree accepted: 64 * qtiles
  int heads, row_stride;  // 128-row kernel: heads per CTA and rows per head
  float scale_log2;
  __nv_bfloat16* out;
  float* lse;
  float* part_o;      // [B][H][splits][64][D]   (workspace merge only)
  float2* part_ml;    // [B][H][splits][64]
  unsigned* tickets;  // [B][H]
  unsigned* err;
  uint32_t wait_limit;  // polls before a pipeline wait gives up (kWaitLimit unless a test lowers it)
};

// Byte offset of 16-byte chunk `ch` (0 .. D/8-1) of row `row` in a tile of
// 128-byte column blocks of `block_rows` rows with the 128-byte swizzle (the
// layout TMA writes).
__device__ __forceinline__ uint32_t sw128_off(int row, int ch, int block_rows) {
  return static_cast<uint32_t>((ch >> 3) * block_rows * 128 + row * 128 + (((ch & 7) ^ (row & 7)) << 4));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Named barrier over the four softmax warps.
__device__ __forceinline__ void softmax_warps_sync() { asm volatile("bar.sync 1, 128;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// 2^x with the hardware approximation (flush-to-zero); 2^-inf = 0.
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}

// Four 8x8 bf16 tiles to shared memory; thread l supplies the address of row
// l % 8 of tile l / 8 and holds, in register i, row lane / 4, columns
// 2 (lane % 4) .. +1 of tile i.
__device__ __forceinline__ void stmatrix_x4(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "r"(r0), "r"(r1),
               "r"(r2), "r"(r3)
               : "memory");
}

// tcgen05.ld / st, shape 16x256b, 8 repetitions: for an M = 64 accumulator
// (rows 16w .. 16w+15 in lanes 32w .. 32w+15), thread (g = lane / 4,
// t = lane % 4) of warp w gets, for each 8-column block b = 0..7 starting at
// the address's column: r[4b + 0, 1] = row 16w + g, columns 8b + 2t, 8b + 2t + 1
// and r[4b + 2, 3] = the same columns of row 16w + g + 8.
__device__ __forceinline__ void tmem_ld_16x256b_x8(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st_16x256b_x8(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
      "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
      "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

// The same shape, one 8-column block: r[0, 1] row 16w + g, r[2, 3] row 16w + g + 8.
__device__ __forceinline__ void tmem_ld_16x256b_x1(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st_16x256b_x1(uint32_t taddr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.16x256b.x1.b32 [%0], {%1,%2,%3,%4};\n" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3])
               : "memory");
}

// The keep bits of the 32 columns a thread holds of a row (columns 8b + 2t + e
// of every 8-column block b < 16, t = lane % 4; bit 2b + e): of a tree chunk,
// from the ancestor words of its two units, and of a prefix chunk that ends
// after kl keys.
__device__ __forceinline__ uint32_t unit_bits(uint64_t w, int t4) {
  uint64_t x = (w >> (2 * t4)) & 0x0303030303030303ull;
  x = (x | (x >> 6)) & 0x000F000F000F000Full;
  x = (x | (x >> 12)) & 0x000000FF000000FFull;
  return static_cast<uint32_t>(x | (x >> 24)) & 0xFFFFu;
}
__device__ __forceinline__ uint32_t prefix_bits(int kl, int t4) {
  uint32_t bits = 0u;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int nb = min(max((kl - 2 * t4 - e + 7) >> 3, 0), 16);  // blocks whose column e is in the prefix
    bits |= (nb == 16 ? 0x55555555u : 0x55555555u & ((1u << (2 * nb)) - 1u)) << e;
  }
  return bits;
}

// Softmax of one chunk for the two rows (a, b) a thread holds: scores in sa /
// sb (raw Q.K), keep bits applied only when `masked` (a chunk of one 64-key
// unit is one whose upper half is masked: one copy of this code is fetched
// instead of two).  Updates the lazily raised maxima mu (log2 units), returns
// the rescale factors of O (and of the row sums, which the tensor core
// accumulates from the same bf16 probabilities) and the probabilities packed
// in column pairs.
__device__ __forceinline__ void chunk_softmax(float (&sa)[32], float (&sb)[32], bool masked, uint32_t ka, uint32_t kb,
                                              float scale, float& mu_a, float& mu_b, float& alpha_a, float& alpha_b,
                                              uint32_t (&pa)[16], uint32_t (&pb)[16]) {
  constexpr int NB = 16;
  if (masked) {
#pragma unroll
    for (int i = 0; i < 2 * NB; ++i) {  // a NaN score at a masked position also becomes -inf
      sa[i] = ka & (1u << i) ? sa[i] : -INFINITY;
      sb[i] = kb & (1u << i) ? sb[i] : -INFINITY;
    }
  }
  float mxa = sa[0], mxb = sb[0];
#pragma unroll
  for (int i = 1; i < 2 * NB; ++i) {
    mxa = fmaxf(mxa, sa[i]);
    mxb = fmaxf(mxb, sb[i]);
  }
  mxa = fmaxf(mxa, __shfl_xor_sync(adt::kFullMask, mxa, 1));
  mxa = fmaxf(mxa, __shfl_xor_sync(adt::kFullMask, mxa, 2));
  mxb = fmaxf(mxb, __shfl_xor_sync(adt::kFullMask, mxb, 1));
  mxb = fmaxf(mxb, __shfl_xor_sync(adt::kFullMask, mxb, 2));
  mxa *= scale;  // scale > 0: the maximum of the scaled scores
  mxb *= scale;
  const bool needa = mxa > mu_a + kRescaleThreshold, needb = mxb > mu_b + kRescaleThreshold;
  const float nma = needa ? mxa : mu_a, nmb = needb ? mxb : mu_b;
  alpha_a = needa ? ex2_approx(mu_a - nma) : 1.f;
  alpha_b = needb ? ex2_approx(mu_b - nmb) : 1.f;
  const float base_a = nma == -INFINITY ? 0.f : nma, base_b = nmb == -INFINITY ? 0.f : nmb;
#pragma unroll
  for (int bk = 0; bk < NB; ++bk) {
    pa[bk] = pack_bf16x2(ex2_approx(fmaf(sa[2 * bk], scale, -base_a)), ex2_approx(fmaf(sa[2 * bk + 1], scale, -base_a)));
    pb[bk] = pack_bf16x2(ex2_approx(fmaf(sb[2 * bk], scale, -base_b)), ex2_approx(fmaf(sb[2 * bk + 1], scale, -base_b)));
  }
  mu_a = nma;
  mu_b = nmb;
}

struct Barriers {
  uint64_t q_full;                 // Q and the tree unit's K/V are in shared memory (softmax warps' copies)
  uint64_t q_tma;                  // the same, when they come as tensor copies: those copies landed
  uint64_t k_full[kMaxStages];     // a stage's K tile has landed
  uint64_t v_full[kMaxStages];     // a stage's V tile has landed
  uint64_t k_free[kMaxStages];     // the S product of the chunk in that slot finished
  uint64_t done[kMaxStages];       // the PV product of the chunk in that slot finished
  uint64_t s_full[2];
  uint64_t s_free[2];
  uint64_t p_full[2];
  uint64_t drain[2];               // abort path: every MMA a thread issued finished
  uint64_t recv;                   // cluster merge: every split's rows for this owner landed
};

// Bounded wait of the pipeline that also gives up when another role has
// aborted.  (The waits that let in-flight copies and products land before a
// CTA leaves always keep the full kWaitLimit.)
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                         unsigned* err, uint32_t limit) {
  const uint32_t a = sm100::smem_addr(bar);
  for (uint32_t i = 0; i < limit; ++i) {
    if (sm100::mbar_try_wait(a, parity)) return true;
    if ((i & 255u) == 255u && *abort_flag) return false;
  }
  *abort_flag = 1;
  adt::raise_error(err, ADT_DEVERR_TIMEOUT);
  return false;
}

// The tree of a launch slot.  With several trees (up to 32) the launch slots
// go to the trees by decreasing prefix length (ties: lower index): the CTAs
// are dispatched in slot order, so the longest streams start first and the
// short ones fill in behind them instead of a late long tree ending the
// launch.  Every warp ranks the trees itself (one lane per tree), from the
// same single round of loads the one-tree path makes.
struct TreeSlot {
  int b, node0, n, total_nodes, L;
};

__device__ __forceinline__ TreeSlot tree_of_slot(const TcParams& p, int slot, int lane) {
  TreeSlot t;
  if (p.B > 1 && p.B <= 32) {
    const bool mine = lane < p.B;
    const int kl = mine ? p.kv_len[lane] : 0;
    const int off = mine ? p.offs[lane] : 0;
    t.total_nodes = p.offs[p.B];
    int rank = 0;
    for (int i = 0; i < p.B; ++i) {
      const int o = __shfl_sync(adt::kFullMask, kl, i);
      rank += (o > kl || (o == kl && i < lane)) ? 1 : 0;
    }
    const unsigned hit = __ballot_sync(adt::kFullMask, mine && rank == slot);
    t.b = hit ? __ffs(hit) - 1 : slot;
    t.L = __shfl_sync(adt::kFullMask, kl, t.b);
    t.node0 = __shfl_sync(adt::kFullMask, off, t.b);
    const int next = __shfl_sync(adt::kFullMask, off, (t.b + 1) & 31);
    t.n = (t.b + 1 < p.B ? next : t.total_nodes) - t.node0;
  } else {
    t.b = slot;
    t.node0 = p.offs[t.b];
    t.n = p.offs[t.b + 1] - t.node0;
    t.total_nodes = p.offs[p.B];
    t.L = p.kv_len[t.b];
  }
  return t;
}

// A launch whose clusters leave SMs free puts further clusters on them, which
// bring the first kPrefetchChunks chunks of every split into L2 and end.  They
// run ahead of the dependency wait, while the launch before finishes (its
// merge leaves the memory idle), so what they read are hints: kv_len may be
// about to change, and the lines they touch lie in the cache tensor whatever
// it says (the tensor map bounds them; later writes go through the same L2).
// A thread asks for one box of 128 keys x 64 columns, chunk by chunk over the
// CTAs; an SM's requests go out at about 115 GB/s, so a CTA takes at most 1.5
// MB.  The launch before lets them start once it has requested its last K
// tiles (started at once, they take bandwidth from its own stream).
//
// us a layer back to back, D = 128, without and with: H = 32, KV 2400 12.5 and
// 11.3, KV 1200 9.8 and 9.2, KV 4096 16.5 and 15.9; H = 16, KV 2400 10.3 and 9.8;
// H = 24 11.3 and 11.2; four trees of KV 2320 30.5 and 30.2; in the 128-row
// kernel 256 nodes, KV 2400 19.2 and 18.6, four trees, Hkv = 8, KV 3500-6001
// 30.6 and 30.0.  One or two chunks gave half of it, all chunks took longer
// than none (14.6 us for the first).
constexpr int kPrefetchChunks = 3;
constexpr int kPrefetchBoxes = 96;  // a CTA's share: 1.5 MB

// Tree b's prefix of L keys: split s of S takes chunks s W / S and on of the W
// (tree chunks, which the kernels count as tree_chunks, follow the prefix).
template <int kBlocks>
__device__ __noinline__ void prefetch_stream(const CUtensorMap* tm_k, const CUtensorMap* tm_v, const TcParams& p, int b,
                                             int S, int tree_chunks) {
  const int L = min(max(__ldcg(p.kv_len + b), 0), p.max_kv);
  const int Pc = (L + kChunk - 1) / kChunk, W = Pc + tree_chunks;
  const int per = p.Hkv * S * 2 * kBlocks;  // column blocks of one chunk of every split, K and V
  const int w = (static_cast<int>(threadIdx.x) * p.prefetch + static_cast<int>(blockIdx.y)) *
                    static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x);
  if (threadIdx.x >= kPrefetchBoxes || w >= per * kPrefetchChunks) return;
  const int blk = w % kBlocks, v = w / kBlocks % 2, pair = w % per / (2 * kBlocks);
  const int split = pair % S, c = split * W / S + w / per;
  if (c < min((split + 1) * W / S, Pc))
    sm100::tma_prefetch_4d(v ? tm_v : tm_k, blk * 64, c * kChunk, pair / S, b);
}

// Clusters that prefetch: what the compute clusters of a launch leave of the
// clusters that fit at once, evenly over its trees, up to eight a tree.
int prefetch_clusters(int fit, int compute, int per_tree) {
  const int room = (fit - compute) / per_tree;
  return room < 0 ? 0 : room > 8 ? 8 : room;
}

// kLarge: trees of more than 64 nodes (query tiles, one mask word per tree
// unit); otherwise one tile and one word, kept in registers.

template <int D, bool kLarge>
__global__ void __launch_bounds__(kThreads, 1)
    tree_attn_tc_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                        const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kt,
                        const __grid_constant__ CUtensorMap tm_vt, const TcParams p) {
  using C = Cfg<D>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // 1024-byte aligned for the 128-byte swizzle; pointer arithmetic on the
  // shared array keeps accesses in the shared address space.
  uint8_t* smem = smem_raw + ((1024u - (sm100::smem_addr(smem_raw) & 1023u)) & 1023u);
  __shared__ Barriers bars;
  constexpr int kUnits = kLarge ? kMaxTreeUnits : 1;
  __shared__ uint64_t anc[kMaxNodes][kUnits];
  __shared__ int s_par[kLarge ? kMaxTreeNodes : kMaxNodes];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_bad;
  __shared__ int s_last;
  __shared__ volatile int s_abort;

  constexpr bool kPrefetch = D == 128 && !kLarge;
  const int split = blockIdx.x, h = static_cast<int>(blockIdx.y) - (kPrefetch ? p.prefetch : 0);
  const int slot = kLarge ? static_cast<int>(blockIdx.z) / p.qtiles : static_cast<int>(blockIdx.z);
  const int qt = kLarge ? static_cast<int>(blockIdx.z) % p.qtiles : 0;
  const int g = h / p.group;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NS = C::kStages;

  if (kPrefetch && h < 0) {
    prefetch_stream<C::kBlocks>(&tm_k, &tm_v, p, static_cast<int>(blockIdx.z), p.splits, 1);
    return;
  }
  // Set-up that touches no memory the previous kernel writes: the
  // mbarriers, the tensor memory and the tensor maps' descriptors.  It runs
  // before the dependency wait, so a CTA that is resident early (on an SM
  // the previous launch leaves idle) has it done when the wait releases.
  if (tid == 0) {
    s_bad = 0;
    s_abort = 0;
    sm100::mbar_init(sm100::smem_addr(&bars.q_full), kSoftmaxWarps);
    sm100::mbar_init(sm100::smem_addr(&bars.q_tma), 1);
    for (int s = 0; s < NS; ++s) {
      sm100::mbar_init(sm100::smem_addr(&bars.k_full[s]), 1);
      sm100::mbar_init(sm100::smem_addr(&bars.v_full[s]), 1);
      sm100::mbar_init(sm100::smem_addr(&bars.k_free[s]), 1);
      sm100::mbar_init(sm100::smem_addr(&bars.done[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      sm100::mbar_init(sm100::smem_addr(&bars.s_full[s]), 1);
      sm100::mbar_init(sm100::smem_addr(&bars.s_free[s]), kSoftmaxWarps);
      sm100::mbar_init(sm100::smem_addr(&bars.p_full[s]), kSoftmaxWarps);
    }
    sm100::mbar_init(sm100::smem_addr(&bars.drain[0]), 1);
    sm100::mbar_init(sm100::smem_addr(&bars.drain[1]), 1);
    sm100::mbar_init(sm100::smem_addr(&bars.recv), 1);
    sm100::fence_mbar_init();
  }
  if (warp == 0) {
    sm100::tmem_alloc(sm100::smem_addr(&tmem_slot), kTmemCols);
    sm100::tmem_relinquish();
  }
  if (warp == kKLoadWarp && lane < 4)
    sm100::prefetch_tensormap(lane == 0 ? &tm_k : lane == 1 ? &tm_q : lane == 2 ? &tm_kt : &tm_vt);
  if (warp == kVLoadWarp && lane == 0) sm100::prefetch_tensormap(&tm_v);
  sm100::tc_fence_before();
  __syncthreads();
  sm100::tc_fence_after();
  const uint32_t tmem = tmem_slot;

  // Programmatic dependent launch: every global-memory access that a result
  // depends on comes after the previous kernel in the stream has completed
  // (immediate when this launch does not overlap one).
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const TreeSlot ts = tree_of_slot(p, slot, lane);
  const int b = ts.b, node0 = ts.node0, n = ts.n, total_nodes = ts.total_nodes, L = ts.L;

  // Conditions that hold for every CTA of this (tree, head, tile): all
  // leave here, handing back the tensor memory.  A tile past the end of its
  // tree has no rows.
  const int row0 = qt * kMaxNodes;  // first node (query row) of this tile
  const bool bad_tree = n < 1 || n > kMaxNodes * (kLarge ? p.qtiles : 1) || node0 < 0 || node0 + n > total_nodes;
  const bool bad_kv = L < 0 || L > p.max_kv;
  if (bad_tree || bad_kv || n - row0 <= 0) {
    if (split == 0 && h == 0 && qt == 0 && tid == 0 && (bad_tree || bad_kv))
      adt::raise_error(p.err, bad_tree ? ADT_DEVERR_BAD_TREE : ADT_DEVERR_KV_RANGE);
    if (warp == 0) sm100::tmem_dealloc(tmem, kTmemCols);
    return;
  }
  const int nq = min(n - row0, kMaxNodes);

  // The keys are cut into chunks of two 64-key units: ceil(P / 2) prefix
  // chunks (P = ceil(L / 64); the last holds one unit when P is odd), then
  // the tree units the tile's rows can see, 0 .. qt (a node's ancestors come
  // before it), two to a chunk.  Split s takes chunks [s T / S, (s + 1) T / S)
  // of the T and processes its tree chunks first.
  const int P = (L + kUnit - 1) / kUnit;
  const int Pc = (P + 1) / 2;
  const int Tc = kLarge ? (qt + 2) / 2 : 1;  // tree chunks of this tile
  const int T = Pc + Tc;
  const int S = p.splits;
  // (32-bit: T < 2^24 chunks and S <= 96 splits; 64-bit division is slow)
  const int c_begin = split * T / S;
  const int c_end = (split + 1) * T / S;
  const int nch = c_end - c_begin;
  const int tc0 = max(c_begin, Pc) - Pc;         // first tree chunk of this split
  const int n_tc = max(0, c_end - max(c_begin, Pc));  // its tree chunks, in slots 0 .. n_tc-1
  auto chunk_keys = [&](int j) -> int {
    if (j < n_tc) return (kLarge && 2 * (tc0 + j) + 1 <= qt ? 2 : 1) * kUnit;
    const int pc = c_begin + j - n_tc;
    return (2 * pc + 1 < P ? 2 : 1) * kUnit;
  };
  auto chunk_key0 = [&](int j) -> int { return (c_begin + j - n_tc) * kChunk; };

  // Q (and the one tree unit's K/V) as 64-row tensor copies when the whole
  // box lies inside the node_offsets[B] rows the caller's buffers hold;
  // otherwise (the last tree of a batch with fewer than 64 nodes after its
  // first, or trees of more than 64 nodes) the softmax warps copy the rows
  // of the tree alone, 16 bytes at a time.
  const bool q_tma = !kLarge && node0 + kMaxNodes <= total_nodes && total_nodes < kTmaRows;
  uint8_t* sQ = smem + C::kQOff;
  uint8_t* sP = smem + C::kPOff;
  uint8_t* sStage = smem + C::kStageOff;
  float* slots = reinterpret_cast<float*>(smem + C::kSlotOff);  // merge: [S][rows_per][kRowStride]

  if (warp < kSoftmaxWarps) {
    // Q tile: rows row0 .. row0+63 of the tree (rows past it zero-filled);
    // this split's tree chunks (K/V of kv head g, nodes past the tree
    // zero-filled) into stage slots 0 .. n_tc-1; the parent pointers.
    for (int i = tid; !q_tma && i < kUnit * (D / 8); i += kSoftmaxWarps * 32) {
      const int r = i / (D / 8), ch = i % (D / 8);
      const bool valid = r < nq;
      const int row = node0 + row0 + (valid ? r : 0);
      cp_async16(sm100::smem_addr(sQ) + sw128_off(r, ch, kUnit),
                 p.q + (static_cast<int64_t>(row) * p.H + h) * D + ch * 8, valid ? 16 : 0);
      if (!kLarge && n_tc) {  // the one tree unit: the same rows
        const int64_t off = (static_cast<int64_t>(row) * p.Hkv + g) * D + ch * 8;
        cp_async16(sm100::smem_addr(sStage) + sw128_off(r, ch, kChunk), p.kt + off, valid ? 16 : 0);
        cp_async16(sm100::smem_addr(sStage + C::kStageTile) + sw128_off(r, ch, kChunk), p.vt + off, valid ? 16 : 0);
      }
    }
    for (int jt = 0; kLarge && jt < n_tc; ++jt) {
      uint8_t* st = sStage + jt * C::kStageBytes;
      for (int i = tid; i < chunk_keys(jt) * (D / 8); i += kSoftmaxWarps * 32) {
        const int r = i / (D / 8), ch = i % (D / 8);
        const int t = (tc0 + jt) * kChunk + r;  // tree node
        const bool valid = t < n;
        const int64_t off = (static_cast<int64_t>(node0 + (valid ? t : 0)) * p.Hkv + g) * D + ch * 8;
        cp_async16(sm100::smem_addr(st) + sw128_off(r, ch, kChunk), p.kt + off, valid ? 16 : 0);
        cp_async16(sm100::smem_addr(st + C::kStageTile) + sw128_off(r, ch, kChunk), p.vt + off, valid ? 16 : 0);
      }
    }
    for (int t = tid; t < n; t += kSoftmaxWarps * 32) cp_async4(sm100::smem_addr(&s_par[t]), p.parents + node0 + t);
    // The ones tile (bf16 1.0) of the row-sum product.
    static_assert(C::kOnesBytes == kSoftmaxWarps * 32 * 16, "one 16-byte store per softmax thread");
    reinterpret_cast<uint4*>(smem + C::kOnesOff)[tid] = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
  }
  // Stage loads: chunk j goes to slot j % NS, K tile by warp 4 and V tile by
  // warp 6.  A tree chunk loads nothing (its K/V came with Q) but still
  // completes its slot's phases, so that every slot's phases advance once
  // per chunk.
  const bool is_loader = (warp == kKLoadWarp || warp == kVLoadWarp) && lane == 0;
  const bool load_v = warp == kVLoadWarp;
  auto issue_tile = [&](int j) {
    const int st = j % NS;
    const uint32_t bar = sm100::smem_addr(load_v ? &bars.v_full[st] : &bars.k_full[st]);
    if (j < n_tc) {
      sm100::mbar_arrive(bar);
      return;
    }
    // One 128-key box per column block (a chunk of one unit loads the next
    // 64 rows too; nothing reads them: its products stop at 64 keys).
    const int key0 = chunk_key0(j);
    uint8_t* dst = sStage + st * C::kStageBytes + (load_v ? C::kStageTile : 0);
    const CUtensorMap* map = load_v ? &tm_v : &tm_k;
    sm100::mbar_arrive_expect_tx(bar, C::kBlocks * C::kBlock128);
    for (int blk = 0; blk < C::kBlocks; ++blk)
      sm100::tma_load_4d(sm100::smem_addr(dst + blk * C::kBlock128), map, blk * 64, key0, g, b, bar);
  };
  const int first_issue = nch < NS ? nch : NS;
  if (q_tma) {
    // Q and the tree unit go out first, from the thread that then requests
    // the first K stages; nothing waits for the softmax warps' set-up.
    if (warp == kKLoadWarp && lane == 0) {
      const uint32_t bar = sm100::smem_addr(&bars.q_tma);
      sm100::mbar_arrive_expect_tx(bar, C::kBlocks * C::kBlock64 * (n_tc ? 3 : 1));
      for (int blk = 0; blk < C::kBlocks; ++blk)
        sm100::tma_load_3d(sm100::smem_addr(sQ + blk * C::kBlock64), &tm_q, blk * 64, h, node0, bar);
      for (int blk = 0; n_tc && blk < C::kBlocks; ++blk) {
        sm100::tma_load_3d(sm100::smem_addr(sStage + blk * C::kBlock128), &tm_kt, blk * 64, g, node0, bar);
        sm100::tma_load_3d(sm100::smem_addr(sStage + C::kStageTile + blk * C::kBlock128), &tm_vt, blk * 64, g, node0,
                           bar);
      }
    }
    if (is_loader) {
      for (int j = 0; j < first_issue; ++j) issue_tile(j);
    }
  }
  // Q's copies (when the softmax warps make them) are requested before the
  // stage loads: a CTA's first stages are 128 KB, and Q queued behind them
  // would hold back the first S.
  __syncthreads();
  // The mbarriers are initialised: tell the cluster (the merge's bulk copies
  // complete on a peer's barrier; every thread waits on this before one).
  sm100::cluster_arrive_relaxed();
  if (!q_tma && is_loader) {
    for (int j = 0; j < first_issue; ++j) issue_tile(j);
  }
  if (warp < kSoftmaxWarps) {
    cp_async_wait_all();
    softmax_warps_sync();
    // Ancestor bitmask of every row r of the tile (node t = row0 + r), one
    // 64-bit word per tree unit: bit j of anc[r][u] <=> node 64u + j is in
    // ans(t) or is t.  Parents precede their children, so the walk visits
    // decreasing indices; anything else marks the tree malformed.
    if (!kLarge && tid < kMaxNodes) {
      uint64_t m = 0;
      if (tid < nq) {
        int j = tid;
        int par = s_par[j];
        m = 1ull << j;
        bool bad = (j == 0) != (par < 0);
        while (!bad && par >= 0) {
          if (par >= j) {
            bad = true;
            break;
          }
          m |= 1ull << par;
          j = par;
          par = s_par[j];
          bad = (j == 0) != (par < 0);
        }
        if (bad) s_bad = 1;
      }
      anc[tid][0] = m;
    }
    if (kLarge && tid < kMaxNodes) {
      uint64_t m0 = 0, m1 = 0, m2 = 0, m3 = 0;
      auto set_bit = [&](int j) {
        const uint64_t bit = 1ull << (j & 63);
        const int u = j >> 6;
        m0 |= u == 0 ? bit : 0ull;
        m1 |= u == 1 ? bit : 0ull;
        m2 |= u == 2 ? bit : 0ull;
        m3 |= u == 3 ? bit : 0ull;
      };
      if (tid < nq) {
        int j = row0 + tid;
        int par = s_par[j];
        set_bit(j);
        bool bad = (j == 0) != (par < 0);
        while (!bad && par >= 0) {
          if (par >= j) {
            bad = true;
            break;
          }
          set_bit(par);
          j = par;
          par = s_par[j];
          bad = (j == 0) != (par < 0);
        }
        if (bad) s_bad = 1;
      }
      uint64_t* w = anc[tid];
      w[0] = m0;
      if constexpr (kUnits > 1) {
        w[1] = m1;
        w[2] = m2;
        w[3] = m3;
      }
    }
  }
  __syncthreads();
  if (s_bad) {
    // Same tree for every CTA of the cluster: all leave here, after the
    // loads already issued have landed.
    if (split == 0 && h == 0 && tid == 0) adt::raise_error(p.err, ADT_DEVERR_BAD_TREE);
    if (is_loader) {
      for (int j = 0; j < first_issue; ++j)
        (void)sm100::mbar_wait_bounded(sm100::smem_addr(load_v ? &bars.v_full[j % NS] : &bars.k_full[j % NS]), 0,
                                       kWaitLimit);
      if (q_tma && !load_v) (void)sm100::mbar_wait_bounded(sm100::smem_addr(&bars.q_tma), 0, kWaitLimit);
    }
    sm100::tc_fence_before();
    __syncthreads();
    if (warp == 0) sm100::tmem_dealloc(tmem, kTmemCols);
    return;
  }

  // Final row statistics of the softmax threads' two rows (a, b).
  float m_ra = -INFINITY, l_ra = 0.f, m_rb = -INFINITY, l_rb = 0.f;

  if (warp == kKLoadWarp || warp == kVLoadWarp) {
    // ------------------------------------------------------------ K / V loads
    if (lane == 0) {
      int issued = first_issue;
      for (int j = first_issue; j < nch; ++j) {
        const int st = j % NS;
        // slot st was last used by chunk j - NS: its K is free once its S is
        // done, its V once its PV is done
        if (!wait_bar(load_v ? &bars.done[st] : &bars.k_free[st], ((j / NS) - 1) & 1, &s_abort, p.err, p.wait_limit)) break;
        issue_tile(j);
        ++issued;
      }
      // With its last K tile requested, a next launch may start to prefetch.
      if (kPrefetch && p.prefetch && !load_v) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
      // Every copy issued lands before the CTA goes on: after an abort
      // elsewhere its consumer may never have waited for it (on the normal
      // path these waits return at once).
      for (int j = (issued > NS ? issued - NS : 0); j < issued; ++j)
        (void)sm100::mbar_wait_bounded(sm100::smem_addr(load_v ? &bars.v_full[j % NS] : &bars.k_full[j % NS]),
                                       (j / NS) & 1, kWaitLimit);
      if (q_tma && !load_v) (void)sm100::mbar_wait_bounded(sm100::smem_addr(&bars.q_tma), 0, kWaitLimit);
    }
    __syncwarp();
  } else if (warp == kSMmaWarp) {
    // ------------------------------------------------------------ S = Q K^T
    if (lane == 0) {
      // (Q's copies by the softmax warps end in q_full, which also follows
      // their zeroing of V rows; after a tensor copy the first product needs
      // neither.)
      bool ok = wait_bar(q_tma ? &bars.q_tma : &bars.q_full, 0, &s_abort, p.err, p.wait_limit);
      const uint32_t q_addr = sm100::smem_addr(sQ);
      for (int j = 0; ok && j < nch; ++j) {
        const int st = j % NS, sb = j & 1;
        if (!wait_bar(&bars.k_full[st], (j / NS) & 1, &s_abort, p.err, p.wait_limit) ||
            (j >= 2 && !wait_bar(&bars.s_free[sb], ((j >> 1) - 1) & 1, &s_abort, p.err, p.wait_limit)))
          break;
        sm100::tc_fence_after();
        const uint32_t k_addr = sm100::smem_addr(sStage + st * C::kStageBytes);
        const uint32_t idesc = chunk_keys(j) == kChunk ? C::kIdescS128 : C::kIdescS64;
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint64_t da = sm100::smem_desc_sw128(q_addr + (kk >> 2) * C::kBlock64 + (kk & 3) * 32, 16, 1024);
          const uint64_t db = sm100::smem_desc_sw128(k_addr + (kk >> 2) * C::kBlock128 + (kk & 3) * 32, 16, 1024);
          sm100::mma_bf16_ss(tmem + sb * kSCols, da, db, idesc, kk > 0 ? 1u : 0u);
        }
        sm100::mma_commit(sm100::smem_addr(&bars.s_full[sb]));
      }
      // The tensor core finishes whatever was issued before this thread goes
      // on, also when a consumer aborted after the last product was issued.
      sm100::mma_commit(sm100::smem_addr(&bars.drain[0]));
      (void)sm100::mbar_wait_bounded(sm100::smem_addr(&bars.drain[0]), 0, kWaitLimit);
    }
    __syncwarp();
  } else if (warp == kPvMmaWarp) {
    // ------------------------------------------------------------ O += P V
    if (lane == 0) {
      const uint32_t p_addr = sm100::smem_addr(sP);
      // Any 16 K-rows of the ones tile are the same: one descriptor serves
      // every k step.
      const uint64_t ones_desc = sm100::smem_desc_sw128(sm100::smem_addr(smem + C::kOnesOff), C::kBlock128, 1024);
      for (int i = 0; i < nch; ++i) {
        if (!wait_bar(&bars.p_full[i & 1], (i >> 1) & 1, &s_abort, p.err, p.wait_limit) ||
            !wait_bar(&bars.v_full[i % NS], (i / NS) & 1, &s_abort, p.err, p.wait_limit))
          break;
        sm100::tc_fence_after();
        const uint32_t v_addr = sm100::smem_addr(sStage + (i % NS) * C::kStageBytes + C::kStageTile);
        const uint32_t pb = p_addr + (i & 1) * C::kPBytes;
        const bool whole = chunk_keys(i) == kChunk;
        // Unrolled: one thread issues the products, and a loop's address
        // arithmetic is a serial chain between them (the 16 of a chunk took
        // 985 cycles to issue).
#pragma unroll
        for (int kk = 0; kk < kChunk / 16; ++kk) {
          if (kk == kUnit / 16 && !whole) break;
          const uint64_t da = sm100::smem_desc_sw128(pb + (kk >> 2) * C::kBlock64 + (kk & 3) * 32, 16, 1024);
          const uint64_t db = sm100::smem_desc_sw128(v_addr + kk * 2048, C::kBlock128, 1024);  // LBO: d blocks
          sm100::mma_bf16_ss(tmem + kOCol, da, db, C::kIdescO, (i > 0 || kk > 0) ? 1u : 0u);
          // row sums of the same bf16 P: P times a 16-column tile of ones
          sm100::mma_bf16_ss(tmem + C::kLCol, da, ones_desc, C::kIdescL, (i > 0 || kk > 0) ? 1u : 0u);
        }
        sm100::mma_commit(sm100::smem_addr(&bars.done[i % NS]));
      }
      sm100::mma_commit(sm100::smem_addr(&bars.drain[1]));
      (void)sm100::mbar_wait_bounded(sm100::smem_addr(&bars.drain[1]), 0, kWaitLimit);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ softmax warps 0-3
    if (q_tma && n_tc && n < kUnit) {
      // The tree unit came as a 64-row box: V rows past the tree (another
      // tree's nodes) are zeroed, so that P = 0 there meets finite values.
      if (__all_sync(adt::kFullMask, wait_bar(&bars.q_tma, 0, &s_abort, p.err, p.wait_limit))) {
        uint8_t* vt = sStage + C::kStageTile;
        const int per_row = C::kBlocks * 8;
        for (int i = tid; i < (kUnit - n) * per_row; i += kSoftmaxWarps * 32) {
          const int rr = n + i / per_row, rem = i % per_row;
          *reinterpret_cast<uint4*>(vt + (rem >> 3) * C::kBlock128 + rr * 128 + (rem & 7) * 16) =
              make_uint4(0u, 0u, 0u, 0u);
        }
      }
    }
    sm100::fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.q_full));

    // Thread (g, t) = (lane / 4, lane % 4) of warp w owns rows ra = 16w + g
    // and rb = ra + 8 of the tile, columns 8b + 2t, 8b + 2t + 1 of every
    // 8-column block b (the 16x256b tensor-memory layout); the four threads
    // of a quad share a row and combine row statistics with two shuffles.
    const int g8 = lane >> 2, t4 = lane & 3;
    const int ra = warp * 16 + g8, rb = ra + 8;
    const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
    // stmatrix addressing: lane l writes row (l / 8 odd ? 8 : 0) + l % 8 of
    // the warp's rows, in column block (l / 16) of each pair of blocks.
    const int st_row = warp * 16 + ((lane >> 3) & 1) * 8 + (lane & 7);
    const int st_blk = lane >> 4;
    const float scale = p.scale_log2;
    const uint64_t ama = anc[ra][0], amb = anc[rb][0];  // the one tree unit (kLarge: unused)
    float mua = -INFINITY, mub = -INFINITY;  // running maxima used for the exponentials
    for (int j = 0; j < nch; ++j) {
      const int sb = j & 1;
      if (!__all_sync(adt::kFullMask, wait_bar(&bars.s_full[sb], (j >> 1) & 1, &s_abort, p.err, p.wait_limit))) break;
      // S(j) is complete, so its K tile can be refilled (the S issuer goes
      // straight on to the next S product).
      if (warp == 0 && lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.k_free[j % NS]));
      sm100::tc_fence_after();
      const int keys = chunk_keys(j);
      uint32_t r0[32], r1[32];
      tmem_ld_16x256b_x8(tmem + lane_base + sb * kSCols, r0);
      tmem_ld_16x256b_x8(tmem + lane_base + sb * kSCols + 64, r1);  // a one-unit chunk: stale, masked below
      sm100::tmem_wait_ld();
      // S is in registers: hand the tensor-memory tile back to the MMA warp.
      sm100::tc_fence_before();
      __syncwarp();
      if (lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.s_free[sb]));

      // Which keys a row sees: its ancestors and itself in the tree unit,
      // the prefix up to L otherwise.  Only the tree chunk and a chunk that
      // holds the end of the prefix need a mask.
      const bool tree_j = j < n_tc;
      const int kl = tree_j ? keys : L - chunk_key0(j);
      const bool masked = tree_j || kl < kChunk;
      uint32_t ka = ~0u, kb = ~0u;
      if (tree_j) {
        if constexpr (kLarge) {
          // units 2u and 2u + 1 of the tree (rows past the tile have no bits)
          const int u = 2 * (tc0 + j);
          ka = unit_bits(anc[ra][u], t4);
          kb = unit_bits(anc[rb][u], t4);
          if (keys == kChunk) {
            ka |= unit_bits(anc[ra][u + 1], t4) << 16;
            kb |= unit_bits(anc[rb][u + 1], t4) << 16;
          }
        } else {
          ka = unit_bits(ama, t4);
          kb = unit_bits(amb, t4);
        }
      } else if (kl < kChunk) {
        ka = kb = prefix_bits(kl, t4);
      }
      float sa[32], sbv[32];
#pragma unroll
      for (int bk = 0; bk < 8; ++bk) {
        sa[2 * bk] = __uint_as_float(r0[4 * bk]);
        sa[2 * bk + 1] = __uint_as_float(r0[4 * bk + 1]);
        sbv[2 * bk] = __uint_as_float(r0[4 * bk + 2]);
        sbv[2 * bk + 1] = __uint_as_float(r0[4 * bk + 3]);
        sa[16 + 2 * bk] = __uint_as_float(r1[4 * bk]);
        sa[16 + 2 * bk + 1] = __uint_as_float(r1[4 * bk + 1]);
        sbv[16 + 2 * bk] = __uint_as_float(r1[4 * bk + 2]);
        sbv[16 + 2 * bk + 1] = __uint_as_float(r1[4 * bk + 3]);
      }
      uint32_t pa[16], pb[16];
      float alpha_a, alpha_b;
      chunk_softmax(sa, sbv, masked, ka, kb, scale, mua, mub, alpha_a, alpha_b, pa, pb);

      // P buffer sb was last read by the PV product of chunk j - 2.
      if (j >= 2 && !__all_sync(adt::kFullMask,
                                wait_bar(&bars.done[(j - 2) % NS], ((j - 2) / NS) & 1, &s_abort, p.err, p.wait_limit)))
        break;
      {
        const uint32_t pbase = sm100::smem_addr(sP) + sb * C::kPBytes + st_row * 128;
        const int nb = keys / 8;
#pragma unroll
        for (int bb = 0; bb < 16; bb += 2) {
          if (bb < nb) {
            const int blk = bb + st_blk;
            const uint32_t addr = pbase + (blk >> 3) * C::kBlock64 + (((blk & 7) ^ (st_row & 7)) << 4);
            stmatrix_x4(addr, pa[bb], pb[bb], pa[bb + 1], pb[bb + 1]);
          }
        }
      }
      // Cache rows at or past L in this chunk (the end of the prefix) can
      // hold anything, NaN included, and P is 0 there: zero their V rows.
      if (!tree_j && kl < keys) {
        if (!__all_sync(adt::kFullMask, wait_bar(&bars.v_full[j % NS], (j / NS) & 1, &s_abort, p.err, p.wait_limit))) break;
        uint8_t* vt = sStage + (j % NS) * C::kStageBytes + C::kStageTile;
        const int per_row = C::kBlocks * 8;
        for (int i = tid; i < (keys - kl) * per_row; i += kSoftmaxWarps * 32) {
          const int rr = kl + i / per_row, rem = i % per_row;
          *reinterpret_cast<uint4*>(vt + (rem >> 3) * C::kBlock128 + rr * 128 + (rem & 7) * 16) =
              make_uint4(0u, 0u, 0u, 0u);
        }
      }
      sm100::fence_proxy_async_smem();
      // Raise O to the new maxima (rare): needs the previous PV product done.
      if (j > 0 && __any_sync(adt::kFullMask, alpha_a != 1.f || alpha_b != 1.f)) {
        if (!__all_sync(adt::kFullMask,
                        wait_bar(&bars.done[(j - 1) % NS], ((j - 1) / NS) & 1, &s_abort, p.err, p.wait_limit)))
          break;
        sm100::tc_fence_after();
#pragma unroll 1
        for (int c0 = 0; c0 < D; c0 += 64) {
          uint32_t o[32];
          tmem_ld_16x256b_x8(tmem + lane_base + kOCol + c0, o);
          sm100::tmem_wait_ld();
#pragma unroll
          for (int bk = 0; bk < 8; ++bk) {
            o[4 * bk + 0] = __float_as_uint(__uint_as_float(o[4 * bk + 0]) * alpha_a);
            o[4 * bk + 1] = __float_as_uint(__uint_as_float(o[4 * bk + 1]) * alpha_a);
            o[4 * bk + 2] = __float_as_uint(__uint_as_float(o[4 * bk + 2]) * alpha_b);
            o[4 * bk + 3] = __float_as_uint(__uint_as_float(o[4 * bk + 3]) * alpha_b);
          }
          tmem_st_16x256b_x8(tmem + lane_base + kOCol + c0, o);
        }
        {
          uint32_t l4[4];
          tmem_ld_16x256b_x1(tmem + lane_base + C::kLCol, l4);
          sm100::tmem_wait_ld();
          l4[0] = __float_as_uint(__uint_as_float(l4[0]) * alpha_a);
          l4[1] = __float_as_uint(__uint_as_float(l4[1]) * alpha_a);
          l4[2] = __float_as_uint(__uint_as_float(l4[2]) * alpha_b);
          l4[3] = __float_as_uint(__uint_as_float(l4[3]) * alpha_b);
          tmem_st_16x256b_x1(tmem + lane_base + C::kLCol, l4);
        }
        sm100::tmem_wait_st();
      }
      sm100::tc_fence_before();
      __syncwarp();
      if (lane == 0) sm100::mbar_arrive(sm100::smem_addr(&bars.p_full[sb]));
    }
    m_ra = mua;
    m_rb = mub;
  }

  // ------------------------------------------------------------ epilogue
  // The next kernel in the stream may start its set-up now.
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  // The softmax threads take their rows of O (unnormalised) into registers.
  constexpr int kOB = D / 64;
  uint32_t o[kOB][32];
  bool have_o = false;
  if (warp < kSoftmaxWarps) {
    const int last = nch - 1;
    // s_abort can change under the warp: decide once, by a vote.
    if (__all_sync(adt::kFullMask, nch > 0 && !s_abort))
      have_o = __all_sync(adt::kFullMask, wait_bar(&bars.done[last % NS], (last / NS) & 1, &s_abort, p.err, p.wait_limit));
    if (have_o) {
      sm100::tc_fence_after();
      const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
#pragma unroll
      for (int c = 0; c < kOB; ++c) tmem_ld_16x256b_x8(tmem + lane_base + kOCol + c * 64, o[c]);
      uint32_t l4[4];
      tmem_ld_16x256b_x1(tmem + lane_base + C::kLCol, l4);  // every column holds the row sum
      sm100::tmem_wait_ld();
      l_ra = __uint_as_float(l4[0]);
      l_rb = __uint_as_float(l4[2]);
    } else {
      // A split without key units (kv_len shorter than max_kv) contributes
      // nothing: weight 0.
      m_ra = m_rb = -INFINITY;
      l_ra = l_rb = 0.f;
#pragma unroll
      for (int c = 0; c < kOB; ++c)
#pragma unroll
        for (int e = 0; e < 32; ++e) o[c][e] = 0u;
    }
  }
  sm100::tc_fence_before();

  const int g8 = lane >> 2, t4 = lane & 3;
  const int ra = warp * 16 + g8, rb = ra + 8;
  const int64_t bh = static_cast<int64_t>(blockIdx.z) * p.H + h;  // (tree, tile, head)
  constexpr int kC4 = D / 4;
  if (p.cluster_merge && S > 1) {
    // Row r of the (tree, head, tile) is merged by split r / rows_per, its owner.
    // Each split writes its partial rows (O unnormalised, then m and l) into
    // its own stage ring, idle now, in row order; one thread sends every
    // owner its rows with bulk shared-to-shared copies into the owner's slot
    // region, completing on the owner's mbarrier; each owner merges locally.
    constexpr int RS = C::kRowStride;
    const int rows_per = (nq + S - 1) / S;
    const int r_lo = split * rows_per;
    const int rows_mine = max(0, min(nq, r_lo + rows_per) - r_lo);
    float* rows_out = reinterpret_cast<float*>(sStage);
    if (tid == 0)
      sm100::mbar_arrive_expect_tx(sm100::smem_addr(&bars.recv), static_cast<uint32_t>(S * rows_mine * RS * 4));
    if (warp < kSoftmaxWarps) {
      if constexpr (C::kHalfRows) {
        // The row normalised by its sum, O / l, goes out in fp16: half the
        // bytes through distributed shared memory.  It is a convex
        // combination of V rows, scaled by 2^-e (e from the row's largest
        // magnitude, over the quad) into [2^14, 2^15): no overflow, and full
        // fp16 precision relative to that magnitude whatever V's range; the
        // owner undoes the scale.
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int r = half ? rb : ra;
          const float l = half ? l_rb : l_ra;
          const float inv = l > 0.f ? __fdividef(1.f, l) : 0.f;
          float amax = 0.f;
#pragma unroll
          for (int c = 0; c < kOB; ++c)
#pragma unroll
            for (int bk = 0; bk < 8; ++bk)
              amax = fmaxf(amax, fmaxf(fabsf(__uint_as_float(o[c][4 * bk + 2 * half])),
                                         fabsf(__uint_as_float(o[c][4 * bk + 2 * half + 1]))));
          amax = fmaxf(amax, __shfl_xor_sync(adt::kFullMask, amax, 1));
          amax = fmaxf(amax, __shfl_xor_sync(adt::kFullMask, amax, 2));
          amax *= inv;
          const int ex = static_cast<int>((__float_as_uint(amax) >> 23) & 0xFFu);  // biased exponent
          const int e = amax > 0.f ? min(max(ex - 127 - 14, -110), 110) : 0;
          const float sc = inv * __uint_as_float(static_cast<uint32_t>(127 - e) << 23);  // inv * 2^-e
          if (r < nq) {
            float* dst = rows_out + r * RS;
            if (t4 == 0) {
              *reinterpret_cast<float2*>(dst + D / 2) =
                  make_float2(half ? m_rb : m_ra, l);
              reinterpret_cast<int*>(dst)[D / 2 + 2] = e;
            }
#pragma unroll
            for (int c = 0; c < kOB; ++c) {
#pragma unroll
              for (int bk = 0; bk < 8; ++bk)
                reinterpret_cast<__half2*>(dst)[(c * 64 + 8 * bk + 2 * t4) / 2] =
                    __floats2half2_rn(__uint_as_float(o[c][4 * bk + 2 * half]) * sc,
                                      __uint_as_float(o[c][4 * bk + 2 * half + 1]) * sc);
            }
          }
        }
      } else {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int r = half ? rb : ra;
          if (r < nq) {
            float* dst = rows_out + r * RS;
            if (t4 == 0) *reinterpret_cast<float2*>(dst + D) = half ? make_float2(m_rb, l_rb) : make_float2(m_ra, l_ra);
#pragma unroll
            for (int c = 0; c < kOB; ++c) {
#pragma unroll
              for (int bk = 0; bk < 8; ++bk)
                *reinterpret_cast<float2*>(dst + c * 64 + 8 * bk + 2 * t4) =
                    make_float2(__uint_as_float(o[c][4 * bk + 2 * half]), __uint_as_float(o[c][4 * bk + 2 * half + 1]));
            }
          }
        }
      }
      sm100::fence_proxy_async_smem();
      softmax_warps_sync();
    }
    // Pairs with the arrive after the prologue: every peer's receive barrier
    // is initialised.
    sm100::cluster_wait_acquire();
    // (Four threads share the copies: one thread took about 100 cycles each.)
    if (warp < kSoftmaxWarps && lane == 0) {
      for (int c = warp; c < S; c += kSoftmaxWarps) {
        const int rc = max(0, min(nq, (c + 1) * rows_per) - c * rows_per);
        if (rc > 0)
          sm100::bulk_copy_to_cluster(sm100::mapa_shared(sm100::smem_addr(slots + split * rows_per * RS), c),
                                      sm100::smem_addr(rows_out + c * rows_per * RS),
                                      static_cast<uint32_t>(rc * RS * 4),
                                      sm100::mapa_shared(sm100::smem_addr(&bars.recv), c));
      }
    }
    // Not abandoned on an abort elsewhere: copies into this CTA's shared
    // memory must have landed before it exits.
    if (!sm100::mbar_wait_bounded(sm100::smem_addr(&bars.recv), 0, kWaitLimit) && tid == 0)
      adt::raise_error(p.err, ADT_DEVERR_TIMEOUT);
    // This owner has its rows, so the copies it was sent are complete.
    sm100::cluster_arrive_relaxed();
    if constexpr (C::kHalfRows) {
      // Thread (row i, 8-column group c8) combines the S normalised partials
      // of that row: weights 2^(m_c - M) l_c / sum (times 2^e_c, the scale the
      // partial was stored at).  A split without keys sent m = -inf (weight 0).
      // (Unrolled for the split count's range: the code of splits that are not
      // there would be fetched all the same.)
      constexpr int kC8 = D / 8;
      auto merge = [&](auto range) {
        constexpr int kMost = decltype(range)::value;
        for (int idx = tid; idx < rows_mine * kC8; idx += kThreads) {
          const int i = idx / kC8, c8 = idx % kC8;
          float2 ml[kMost];
          int ec[kMost];
          uint4 v[kMost];
#pragma unroll
          for (int c = 0; c < kMost; ++c) {
            if (c < S) {
              const float* row = slots + (c * rows_per + i) * RS;
              ml[c] = *reinterpret_cast<const float2*>(row + D / 2);
              ec[c] = reinterpret_cast<const int*>(row)[D / 2 + 2];
              v[c] = *reinterpret_cast<const uint4*>(row + c8 * 4);
            }
          }
          float M = -INFINITY;
#pragma unroll
          for (int c = 0; c < kMost; ++c)
            if (c < S) M = fmaxf(M, ml[c].x);
          float lt = 0.f;
          float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int c = 0; c < kMost; ++c) {
            if (c < S) {
              const float w = ml[c].x == -INFINITY ? 0.f : ex2_approx(ml[c].x - M) * ml[c].y;
              lt += w;
              const float ws = w * __uint_as_float(static_cast<uint32_t>(127 + ec[c]) << 23);  // w * 2^e_c
              const __half2* hv = reinterpret_cast<const __half2*>(&v[c]);
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float2 f = __half22float2(hv[e]);
                acc[2 * e] += ws * f.x;
                acc[2 * e + 1] += ws * f.y;
              }
            }
          }
          const float inv = __fdividef(1.f, lt);
          __nv_bfloat16* dst = p.out + (static_cast<int64_t>(node0 + row0 + r_lo + i) * p.H + h) * D + c8 * 8;
          uint4 pk;
          pk.x = pack_bf16x2(acc[0] * inv, acc[1] * inv);
          pk.y = pack_bf16x2(acc[2] * inv, acc[3] * inv);
          pk.z = pack_bf16x2(acc[4] * inv, acc[5] * inv);
          pk.w = pack_bf16x2(acc[6] * inv, acc[7] * inv);
          *reinterpret_cast<uint4*>(dst) = pk;
          if (c8 == 0 && p.lse) p.lse[static_cast<int64_t>(node0 + row0 + r_lo + i) * p.H + h] = (M + __log2f(lt)) * kLn2;
        }
      };
      if (S <= 4)
        merge(std::integral_constant<int, 4>());
      else
        merge(std::integral_constant<int, kMaxClusterSplits>());
    } else {
      // Thread (row i, column group c4) combines the S partials of that row:
      // weights 2^(m_c - M) l_c / sum.  A split without keys sent zeros with m
      // = -inf (weight 0).
      auto merge = [&](auto range) {
        constexpr int kMost = decltype(range)::value;
        for (int idx = tid; idx < rows_mine * kC4; idx += kThreads) {
          const int i = idx / kC4, c4 = idx % kC4;
          float2 ml[kMost];
          float4 v[kMost];
#pragma unroll
          for (int c = 0; c < kMost; ++c) {
            if (c < S) {
              const float* row = slots + (c * rows_per + i) * RS;
              ml[c] = *reinterpret_cast<const float2*>(row + D);
              v[c] = *reinterpret_cast<const float4*>(row + c4 * 4);
            }
          }
          float M = -INFINITY;
#pragma unroll
          for (int c = 0; c < kMost; ++c)
            if (c < S) M = fmaxf(M, ml[c].x);
          float lt = 0.f;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int c = 0; c < kMost; ++c) {
            if (c >= S) continue;
            const float w = ml[c].x == -INFINITY ? 0.f : ex2_approx(ml[c].x - M);
            lt += w * ml[c].y;
            acc.x += w * v[c].x;
            acc.y += w * v[c].y;
            acc.z += w * v[c].z;
            acc.w += w * v[c].w;
          }
          const float inv = __fdividef(1.f, lt);
          __nv_bfloat16* dst = p.out + (static_cast<int64_t>(node0 + row0 + r_lo + i) * p.H + h) * D + c4 * 4;
          uint2 pk;
          pk.x = pack_bf16x2(acc.x * inv, acc.y * inv);
          pk.y = pack_bf16x2(acc.z * inv, acc.w * inv);
          *reinterpret_cast<uint2*>(dst) = pk;
          if (c4 == 0 && p.lse) p.lse[static_cast<int64_t>(node0 + row0 + r_lo + i) * p.H + h] = (M + __log2f(lt)) * kLn2;
        }
      };
      if (S <= 4)
        merge(std::integral_constant<int, 4>());
      else
        merge(std::integral_constant<int, kMaxClusterSplits>());
    }
    // Every owner has its rows: this CTA's outgoing copies are complete.
    sm100::cluster_wait_acquire();
    sm100::tc_fence_after();
    if (warp == 0) sm100::tmem_dealloc(tmem, kTmemCols);
    return;
  }

  if (p.cluster_merge) {
    // One split: the rows are final.  Normalised, they go through the idle
    // ring (rows of 16 bytes more than D, so that neither side's accesses
    // conflict) to be written out 16 bytes at a time.
    constexpr int kPitch = D * 2 + 16;
    if (warp < kSoftmaxWarps && have_o) {
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int r = half ? rb : ra;
        const float l = half ? l_rb : l_ra;
        const float inv = __fdividef(1.f, l);
        uint8_t* dst = sStage + r * kPitch + t4 * 4;
#pragma unroll
        for (int c = 0; c < kOB; ++c)
#pragma unroll
          for (int bk = 0; bk < 8; ++bk)
            *reinterpret_cast<uint32_t*>(dst + c * 128 + bk * 16) =
                pack_bf16x2(__uint_as_float(o[c][4 * bk + 2 * half]) * inv,
                            __uint_as_float(o[c][4 * bk + 2 * half + 1]) * inv);
        if (t4 == 0 && r < nq && p.lse)
          p.lse[static_cast<int64_t>(node0 + row0 + r) * p.H + h] = ((half ? m_rb : m_ra) + __log2f(l)) * kLn2;
      }
      __syncwarp();  // a warp writes out its own 16 rows
      constexpr int kC8 = D / 8;
      for (int i = lane; i < 16 * kC8; i += 32) {
        const int r = warp * 16 + i / kC8, c8 = i % kC8;
        if (r < nq)
          *reinterpret_cast<uint4*>(p.out + (static_cast<int64_t>(node0 + row0 + r) * p.H + h) * D + c8 * 8) =
              *reinterpret_cast<const uint4*>(sStage + r * kPitch + c8 * 16);
      }
    }
    __syncthreads();
    sm100::tc_fence_after();
    if (warp == 0) sm100::tmem_dealloc(tmem, kTmemCols);
    return;
  }
  // More splits than a portable cluster holds: partials go to the workspace
  // and the CTA that finishes a (tree, head) last merges them.
  float* po = p.part_o + (bh * S + split) * kMaxNodes * D;
  float2* pml = p.part_ml + (bh * S + split) * kMaxNodes;
  if (warp < kSoftmaxWarps) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int r = half ? rb : ra;
      if (r < nq) {
        if (t4 == 0) pml[r] = half ? make_float2(m_rb, l_rb) : make_float2(m_ra, l_ra);
#pragma unroll
        for (int c = 0; c < kOB; ++c) {
#pragma unroll
          for (int bk = 0; bk < 8; ++bk) {
            const float2 v = have_o ? make_float2(__uint_as_float(o[c][4 * bk + 2 * half]),
                                                  __uint_as_float(o[c][4 * bk + 2 * half + 1]))
                                    : make_float2(0.f, 0.f);
            *reinterpret_cast<float2*>(po + r * D + c * 64 + 8 * bk + 2 * t4) = v;
          }
        }
      }
    }
  }
  sm100::cluster_wait_acquire();  // pairs with the prologue's arrive (a cluster of one CTA here)
  __syncthreads();
  sm100::tc_fence_after();
  if (warp == 0) sm100::tmem_dealloc(tmem, kTmemCols);
  // The ticket's release publishes this split's partials (ordered before it
  // by the barrier); its acquire, in the last split, makes all of them visible.
  if (tid == 0) s_last = adt::atomic_add_acq_rel_gpu(p.tickets + bh, 1u) == static_cast<unsigned>(S - 1);
  __syncthreads();
  if (!s_last) return;
  const float* po_bh = p.part_o + bh * S * kMaxNodes * D;
  const float2* pml_bh = p.part_ml + bh * S * kMaxNodes;
  float* wsm = reinterpret_cast<float*>(sStage);  // [64][S]
  if (tid < nq) {
    float M = -INFINITY;
    for (int sp = 0; sp < S; ++sp) M = fmaxf(M, __ldcg(&pml_bh[sp * kMaxNodes + tid]).x);
    float lt = 0.f;
    for (int sp = 0; sp < S; ++sp) {
      const float2 ml = __ldcg(&pml_bh[sp * kMaxNodes + tid]);
      const float w = ml.x == -INFINITY ? 0.f : exp2f(ml.x - M);
      wsm[tid * S + sp] = w;
      lt += w * ml.y;
    }
    const float inv = 1.f / lt;
    for (int sp = 0; sp < S; ++sp) wsm[tid * S + sp] *= inv;
    if (p.lse) p.lse[static_cast<int64_t>(node0 + row0 + tid) * p.H + h] = (M + log2f(lt)) * kLn2;
  }
  __syncthreads();
  constexpr int kStride4 = kMaxNodes * D / 4;
  for (int idx = tid; idx < nq * kC4; idx += kThreads) {
    const int rr = idx / kC4, c4 = idx % kC4;
    const float4* src = reinterpret_cast<const float4*>(po_bh + rr * D) + c4;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    int sp = 0;
    for (; sp + 4 <= S; sp += 4) {
      float4 v[4];
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) v[q4] = __ldcg(src + (sp + q4) * kStride4);
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) {
        const float w = wsm[rr * S + sp + q4];
        acc.x += w * v[q4].x;
        acc.y += w * v[q4].y;
        acc.z += w * v[q4].z;
        acc.w += w * v[q4].w;
      }
    }
    for (; sp < S; ++sp) {
      const float4 v = __ldcg(src + sp * kStride4);
      const float w = wsm[rr * S + sp];
      acc.x += w * v.x;
      acc.y += w * v.y;
      acc.z += w * v.z;
      acc.w += w * v.w;
    }
    __nv_bfloat16* dst = p.out + (static_cast<int64_t>(node0 + row0 + rr) * p.H + h) * D + c4 * 4;
    uint2 pk;
    pk.x = pack_bf16x2(acc.x, acc.y);
    pk.y = pack_bf16x2(acc.z, acc.w);
    *reinterpret_cast<uint2*>(dst) = pk;
  }
  if (tid == 0) p.tickets[bh] = 0u;
}

#include "tree_attn_wide.cuh"

// ---------------------------------------------------------------- host side

// Splits per (tree, head): about one CTA per SM, at most one split per chunk
// of keys.  Up to kMaxClusterSplits splits form a cluster; the count is
// lowered until all B*H clusters are co-resident (GPC sizes decide how many
// clusters of a given size fit at once).  Many splits (small B*H, long
// prefixes) merge through the workspace instead.
int max_active_clusters(int D, bool large, int cluster, int dev);

int qtiles_for(int max_nodes) { return (max_nodes + kMaxNodes - 1) / kMaxNodes; }

// Bq = trees x query tiles.
int choose_splits(int sm_count, int Bq, int H, int D, int max_kv, int dev, bool large) {
  const int units = ((max_kv + kUnit - 1) / kUnit + 1) / 2 + 1;  // chunks, the tree unit included
  const int bh = Bq * H;
  int s = sm_count / bh;
  if (s < 1) s = 1;
  if (s > units) s = units;
  if (s >= 2 * kMaxClusterSplits) return s > kMaxSplits ? kMaxSplits : s;
  if (s > kMaxClusterSplits) s = kMaxClusterSplits;
  while (s > 1 && max_active_clusters(D, large, s, dev) < bh) --s;
  return s;
}

// Workspace layout.  The per-(tree, head) completion tickets sit at fixed
// offsets at the start (room for kMaxBH pairs), so calls of any shape can
// share one workspace; the partials after them are rewritten before use.
constexpr int kMaxBH = 65536;

struct WsLayout {
  size_t tickets, part_ml, part_o, total;
};

WsLayout ws_layout(int B, int H, int D, int splits) {
  WsLayout w{};
  const size_t bhs = static_cast<size_t>(B) * H * splits;
  w.tickets = 0;
  w.part_ml = adt::align_up(static_cast<size_t>(kMaxBH) * sizeof(unsigned), 256);
  w.part_o = adt::align_up(w.part_ml + bhs * kMaxNodes * sizeof(float2), 256);
  w.total = adt::align_up(w.part_o + bhs * kMaxNodes * D * sizeof(float), 256);
  return w;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

std::once_flag g_encode_once;
EncodeTiledFn g_encode = nullptr;

void load_encode() {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
          cudaSuccess &&
      q == cudaDriverEntryPointSuccess)
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
}

// 4-D map of a cache (d, pos, kv head, tree) with the 128-byte swizzle and
// boxes of 64 columns x box_keys positions; positions at or past max_kv read
// as zero.
adt_status make_cache_map(CUtensorMap* map, const void* base, int D, int max_kv, int Hkv, int B, int64_t sh,
                          int64_t sb, int box_keys = kChunk) {
  std::call_once(g_encode_once, load_encode);
  if (!g_encode) return ADT_ERR_CUDA;
  const int64_t span = static_cast<int64_t>(max_kv > 0 ? max_kv : 1);
  cuuint64_t dims[4] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(span), static_cast<cuuint64_t>(Hkv),
                        static_cast<cuuint64_t>(B)};
  cuuint64_t strides[3] = {static_cast<cuuint64_t>(D) * 2, static_cast<cuuint64_t>(sh > 0 ? sh : span * D) * 2,
                           static_cast<cuuint64_t>(sb > 0 ? sb : span * D * Hkv) * 2};
  cuuint32_t box[4] = {64, static_cast<cuuint32_t>(box_keys), 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? ADT_OK : ADT_ERR_INVALID_ARG;
}

// 3-D map of a node-major tensor [nodes][heads][D] (Q or the tree's K / V)
// with the 128-byte swizzle and boxes of 64 nodes x 64 columns of one head.
// The node extent is nominal: the kernel only requests boxes that lie inside
// the node_offsets[B] rows the caller's buffer holds.
adt_status make_rows_map(CUtensorMap* map, const void* base, int D, int heads) {
  std::call_once(g_encode_once, load_encode);
  if (!g_encode) return ADT_ERR_CUDA;
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(heads), static_cast<cuuint64_t>(kTmaRows)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(D) * 2, static_cast<cuuint64_t>(heads) * D * 2};
  cuuint32_t box[3] = {64, 1, kUnit};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? ADT_OK : ADT_ERR_INVALID_ARG;
}

template <int D, bool kLarge>
int occupancy_clusters(cudaLaunchConfig_t* cfg) {
  int num = 0;
  cudaFuncSetAttribute(tree_attn_tc_kernel<D, kLarge>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kDynSmem);
  cfg->dynamicSmemBytes = Cfg<D>::kDynSmem;
  if (cudaOccupancyMaxActiveClusters(&num, tree_attn_tc_kernel<D, kLarge>, cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    num = 0;
  }
  return num;
}

int max_active_clusters(int D, bool large, int cluster, int dev) {
  static int cache[64][2][2][kMaxClusterSplits + 1];  // 0 = not queried yet
  int& slot = cache[dev & 63][D == 128 ? 1 : 0][large ? 1 : 0][cluster];
  int v = __atomic_load_n(&slot, __ATOMIC_ACQUIRE);
  if (v) return v - 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(cluster), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const int num = D == 128 ? (large ? occupancy_clusters<128, true>(&cfg) : occupancy_clusters<128, false>(&cfg))
                           : (large ? occupancy_clusters<64, true>(&cfg) : occupancy_clusters<64, false>(&cfg));
  __atomic_store_n(&slot, num + 1, __ATOMIC_RELEASE);
  return num;
}

template <int D>
int wide_active_clusters(int cluster, int dev) {
  static int cache[64][kMaxClusterSplits + 1];  // 0 = not queried yet
  int& slot = cache[dev & 63][cluster];
  const int v = __atomic_load_n(&slot, __ATOMIC_ACQUIRE);
  if (v) return v - 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(cluster), 1, 1);
  cfg.blockDim = dim3(kWideThreads, 1, 1);
  cfg.dynamicSmemBytes = WideCfg<D>::kDynSmem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int num = 0;
  cudaFuncSetAttribute(tree_attn_wide_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, WideCfg<D>::kDynSmem);
  if (cudaOccupancyMaxActiveClusters(&num, tree_attn_wide_kernel<D>, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    num = 0;
  }
  __atomic_store_n(&slot, num + 1, __ATOMIC_RELEASE);
  return num;
}

// The 64-row kernel's prefetching clusters.  At least 2.5 chunks a split: a
// launch of less is mostly latency.  At D = 64, where a chunk is half the bytes,
// there is no gain (H = 20, KV 2400: 9.8 and 9.8 us; in the 128-row kernel 12.4
// and 12.4 us, 192 nodes, KV 693 and 577).
int tc_prefetch(const TcParams& prm, int D, bool large, bool overlap_previous, int dev) {
  if (D != 128 || large || !overlap_previous || prm.splits > kMaxClusterSplits) return 0;
  if (2 * ((prm.max_kv + kChunk - 1) / kChunk + 1) < 5 * prm.splits) return 0;
  return prefetch_clusters(max_active_clusters(D, large, prm.splits, dev), prm.B * prm.H, prm.B);
}

template <int D, bool kLarge>
adt_status launch(TcParams prm, const void* k_cache, const void* v_cache, int64_t sb, int64_t sh, cudaStream_t st,
                  int dev, bool overlap_previous) {
  static unsigned configured[2] = {0u, 0u};  // bit per device (< 64), per instantiation
  const unsigned bit = 1u << (dev & 31);
  unsigned& word = configured[dev >> 5];
  if (!(__atomic_load_n(&word, __ATOMIC_ACQUIRE) & bit)) {
    ADT_CUDA_TRY(cudaFuncSetAttribute(tree_attn_tc_kernel<D, kLarge>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      Cfg<D>::kDynSmem));
    __atomic_fetch_or(&word, bit, __ATOMIC_ACQ_REL);
  }
  CUtensorMap tm_k, tm_v, tm_q, tm_kt, tm_vt;
  adt_status s1 = make_cache_map(&tm_k, k_cache, D, prm.max_kv, prm.Hkv, prm.B, sh, sb);
  if (s1 != ADT_OK) return s1;
  s1 = make_cache_map(&tm_v, v_cache, D, prm.max_kv, prm.Hkv, prm.B, sh, sb);
  if (s1 != ADT_OK) return s1;
  if ((s1 = make_rows_map(&tm_q, prm.q, D, prm.H)) != ADT_OK) return s1;
  if ((s1 = make_rows_map(&tm_kt, prm.kt, D, prm.Hkv)) != ADT_OK) return s1;
  if ((s1 = make_rows_map(&tm_vt, prm.vt, D, prm.Hkv)) != ADT_OK) return s1;
  prm.cluster_merge = prm.splits <= kMaxClusterSplits ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  prm.prefetch = tc_prefetch(prm, D, kLarge, overlap_previous, dev);
  cfg.gridDim = dim3(static_cast<unsigned>(prm.splits), static_cast<unsigned>(prm.H + prm.prefetch),
                     static_cast<unsigned>(prm.B * prm.qtiles));
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = Cfg<D>::kDynSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = prm.cluster_merge ? static_cast<unsigned>(prm.splits) : 1u;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // Programmatic dependent launch: the launch and the set-up before the
  // kernel's griddepcontrol.wait may overlap the tail of the previous kernel.
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = overlap_previous ? 2 : 1;
  ADT_CUDA_TRY(cudaLaunchKernelEx(&cfg, tree_attn_tc_kernel<D, kLarge>, tm_k, tm_v, tm_q, tm_kt, tm_vt, prm));
  return adt::launch_status();
}

// CTAs per (tree, head group) of the 128-row kernel: `tiles` tiles with as many
// key splits as fit the SMs and a portable cluster, all clusters co-resident;
// 1 where even one split a tile takes more CTAs than there are SMs (the tiles
// are then CTAs of their own, and those a smaller tree lacks end at once --
// within a cluster they would hold their SM until its last CTA ends).
template <int D>
int wide_cluster(int sm_count, int groups, int tiles, int max_kv, int dev) {
  const int chunks = (max_kv + kChunk - 1) / kChunk + tiles;
  int s = sm_count / (groups * tiles);
  if (s > chunks) s = chunks;
  if (s > kMaxClusterSplits / tiles) s = kMaxClusterSplits / tiles;
  while (s > 0 && wide_active_clusters<D>(s * tiles, dev) < groups) --s;
  return s > 0 ? s * tiles : 1;
}

// Which calls take the 128-row kernel: heads per CTA (0: the 64-row kernel).
// A chunk of 128 keys costs it 0.9 us for 128 rows, against 1.1 to 1.2 us for
// 64, but its fixed cost is 1 to 2 us higher (twice the rows to merge, one
// thread per row): it pays from about kWideChunks chunks per CTA of the 64-row
// kernel on.  64-row / 128-row kernel, us: two chunks (H = 8 / 2, D = 64, four
// trees over 600 keys) 8.8 / 9.6, three (20 / 5 heads, D = 64, 2400 keys)
// 10.6 / 11.1, nine (32 / 8, D = 128, 4000 keys) 15.3 / 13.1, 20 (256 nodes,
// 32 heads, D = 128, 2400 keys) 29.9 / 18.6.
constexpr int kWideChunks = 6;

int wide_heads(const TcParams& prm, int sm_count) {
  const int heads = prm.qtiles > 1 ? 1 : prm.group % 2 == 0 ? 2 : 0;
  const int chunks = (prm.max_kv + kChunk - 1) / kChunk + (prm.qtiles + 1) / 2;
  const int ctas = prm.B * prm.qtiles * prm.H * prm.splits;
  const int waves = (ctas + sm_count - 1) / sm_count;
  // (More splits than a cluster holds merge in fp32 through the workspace.)
  return prm.splits <= kMaxClusterSplits && chunks * waves >= kWideChunks * prm.splits ? heads : 0;
}

// A launch of the 128-row kernel: `heads` (1 or 2) query heads of a kv head per
// CTA, trees of `tiles` tiles, `groups` (tree, head group) pairs.
struct WidePlan {
  int heads, tiles, groups, cluster, prefetch;
};

template <int D>
WidePlan wide_plan(const TcParams& prm, int heads, bool overlap_previous, int dev, int sm_count) {
  WidePlan w;
  w.heads = heads;
  w.tiles = (prm.max_tree + kWideRows - 1) / kWideRows;
  w.groups = prm.B * (prm.H / heads);
  w.cluster = wide_cluster<D>(sm_count, w.groups, w.tiles, prm.max_kv, dev);
  w.prefetch = 0;
  if (D == 128 && overlap_previous) {
    const int z = w.cluster > 1 ? 1 : w.tiles;  // clusters of one CTA: a tile each
    w.prefetch = prefetch_clusters(wide_active_clusters<D>(w.cluster, dev), w.groups * z, prm.B * z);
  }
  return w;
}

template <int D>
adt_status launch_wide(TcParams prm, int heads, const void* k_cache, const void* v_cache, int64_t sb, int64_t sh,
                       cudaStream_t st, int dev, int sm_count, bool overlap_previous) {
  static unsigned configured[2] = {0u, 0u};  // bit per device (< 64)
  const unsigned bit = 1u << (dev & 31);
  unsigned& word = configured[dev >> 5];
  if (!(__atomic_load_n(&word, __ATOMIC_ACQUIRE) & bit)) {
    ADT_CUDA_TRY(cudaFuncSetAttribute(tree_attn_wide_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      WideCfg<D>::kDynSmem));
    __atomic_fetch_or(&word, bit, __ATOMIC_ACQ_REL);
  }
  CUtensorMap tm_k, tm_v;
  adt_status s1 = make_cache_map(&tm_k, k_cache, D, prm.max_kv, prm.Hkv, prm.B, sh, sb);
  if (s1 != ADT_OK) return s1;
  s1 = make_cache_map(&tm_v, v_cache, D, prm.max_kv, prm.Hkv, prm.B, sh, sb);
  if (s1 != ADT_OK) return s1;
  ADT_REQUIRE(heads == 1 || heads == 2);  // the kernel's row strides
  const WidePlan w = wide_plan<D>(prm, heads, overlap_previous, dev, sm_count);
  prm.heads = heads;
  prm.row_stride = kWideRows / heads;
  prm.prefetch = w.prefetch;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(w.cluster), static_cast<unsigned>(prm.H / heads + w.prefetch),
                     static_cast<unsigned>(w.cluster > 1 ? prm.B : prm.B * w.tiles));
  cfg.blockDim = dim3(kWideThreads, 1, 1);
  cfg.dynamicSmemBytes = WideCfg<D>::kDynSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(w.cluster);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = adt::pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = overlap_previous ? 2 : 1;
  ADT_CUDA_TRY(cudaLaunchKernelEx(&cfg, tree_attn_wide_kernel<D>, tm_k, tm_v, prm));
  return adt::launch_status();
}

adt_status launch_any(const TcParams& prm, int D, const void* k_cache, const void* v_cache, int64_t sb, int64_t sh,
                      cudaStream_t st, int dev, int sm_count, bool overlap_previous) {
  const int heads = wide_heads(prm, sm_count);
  if (heads)
    return D == 128 ? launch_wide<128>(prm, heads, k_cache, v_cache, sb, sh, st, dev, sm_count, overlap_previous)
                    : launch_wide<64>(prm, heads, k_cache, v_cache, sb, sh, st, dev, sm_count, overlap_previous);
  const bool large = prm.qtiles > 1;
  if (D == 128)
    return large ? launch<128, true>(prm, k_cache, v_cache, sb, sh, st, dev, overlap_previous)
                 : launch<128, false>(prm, k_cache, v_cache, sb, sh, st, dev, overlap_previous);
  return large ? launch<64, true>(prm, k_cache, v_cache, sb, sh, st, dev, overlap_previous)
               : launch<64, false>(prm, k_cache, v_cache, sb, sh, st, dev, overlap_previous);
}

// Shared host checks of both entry points.
adt_status check_args(const adt_bf16* q, const adt_bf16* k_cache, const adt_bf16* v_cache, const int32_t* kv_len,
                      int64_t sb, int64_t sh, const adt_bf16* k_tree, const adt_bf16* v_tree,
                      const int32_t* parents, const int32_t* node_offsets, int32_t B, int32_t H, int32_t Hkv,
                      int32_t D, int32_t max_nodes, int32_t max_kv, float scale, const adt_bf16* out) {
  ADT_REQUIRE(q && k_cache && v_cache && kv_len && k_tree && v_tree && parents && node_offsets && out);
  ADT_REQUIRE(B >= 1 && H >= 1 && Hkv >= 1 && H % Hkv == 0);
  ADT_REQUIRE(max_nodes >= 1 && max_kv >= 0 && max_kv < (1 << 30));
  if (max_nodes > kMaxTreeNodes) return ADT_ERR_UNSUPPORTED;
  const int64_t bq = static_cast<int64_t>(B) * qtiles_for(max_nodes);
  ADT_REQUIRE(bq * H <= kMaxBH && bq <= 65535 && H <= 65535);
  ADT_REQUIRE(scale > 0.f && scale < 1e30f);
  if (D != 64 && D != 128) return ADT_ERR_UNSUPPORTED;
  ADT_REQUIRE(sb >= 0 && sh >= 0 && sb % 8 == 0 && sh % 8 == 0);
  ADT_REQUIRE(Hkv == 1 || sh >= static_cast<int64_t>(max_kv) * D);
  ADT_REQUIRE(B == 1 || sb >= static_cast<int64_t>(max_kv) * D);
  ADT_REQUIRE(adt::aligned16(q) && adt::aligned16(k_cache) && adt::aligned16(v_cache) && adt::aligned16(k_tree) &&
              adt::aligned16(v_tree) && adt::aligned16(out));
  return ADT_OK;
}

TcParams make_params(const adt_bf16* q, const int32_t* kv_len, const adt_bf16* k_tree, const adt_bf16* v_tree,
                     const int32_t* parents, const int32_t* node_offsets, int B, int H, int Hkv, int max_kv,
                     int max_nodes, int splits, float scale, adt_bf16* out, float* lse, unsigned* err) {
  TcParams prm{};
  prm.q = reinterpret_cast<const __nv_bfloat16*>(q);
  prm.kt = reinterpret_cast<const __nv_bfloat16*>(k_tree);
  prm.vt = reinterpret_cast<const __nv_bfloat16*>(v_tree);
  prm.kv_len = kv_len;
  prm.parents = parents;
  prm.offs = node_offsets;
  prm.B = B;
  prm.H = H;
  prm.Hkv = Hkv;
  prm.group = H / Hkv;
  prm.max_kv = max_kv;
  prm.splits = splits;
  prm.qtiles = qtiles_for(max_nodes);
  prm.max_tree = kMaxNodes * prm.qtiles;
  prm.scale_log2 = scale * kLog2e;
  prm.out = reinterpret_cast<__nv_bfloat16*>(out);
  prm.lse = lse;
  prm.err = err;
  prm.wait_limit = adt::wait_limit(kWaitLimit);
  return prm;
}

}  // namespace

extern "C" {

adt_status adt_testing_attn_plan(int32_t B, int32_t H, int32_t Hkv, int32_t D, int32_t max_nodes, int32_t max_kv,
                                 int32_t* plan) {
  ADT_REQUIRE(plan && B >= 1 && Hkv >= 1 && H >= 1 && H % Hkv == 0 && max_kv >= 0);
  ADT_REQUIRE(max_nodes >= 1 && max_nodes <= kMaxTreeNodes && (D == 64 || D == 128));
  adt::DeviceInfo info;
  const adt_status st = adt::device_info(&info);
  if (st != ADT_OK) return st;
  const int dev = info.device, Bq = B * qtiles_for(max_nodes);
  const bool large = max_nodes > kMaxNodes;
  const int splits = choose_splits(info.sm_count, Bq, H, D, max_kv, dev, large);
  const TcParams prm = make_params(nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, B, H, Hkv, max_kv, max_nodes,
                                   splits, 1.f, nullptr, nullptr, nullptr);
  const int heads = wide_heads(prm, info.sm_count);
  if (heads) {
    const WidePlan w = D == 128 ? wide_plan<128>(prm, heads, true, dev, info.sm_count)
                                : wide_plan<64>(prm, heads, true, dev, info.sm_count);
    plan[0] = kWideRows;
    plan[1] = w.cluster;
    plan[2] = w.prefetch;
  } else {
    plan[0] = kMaxNodes;
    plan[1] = splits;
    plan[2] = tc_prefetch(prm, D, large, true, dev);
  }
  return ADT_OK;
}

size_t adt_tree_attn_workspace_size(int32_t B, int32_t H, int32_t D, int32_t max_nodes,
                                    int32_t max_kv) {
  if (B < 1 || H < 1 || (D != 64 && D != 128) || max_kv < 0 || max_nodes < 1 || max_nodes > kMaxTreeNodes) return 0;
  const int Bq = B * qtiles_for(max_nodes);
  if (static_cast<int64_t>(Bq) * H > kMaxBH) return 0;
  adt::DeviceInfo info;
  if (adt::device_info(&info) != ADT_OK) return 0;
  return ws_layout(Bq, H, D, choose_splits(info.sm_count, Bq, H, D, max_kv, info.device, max_nodes > kMaxNodes)).total;
}

adt_status adt_tree_attn(const adt_bf16* q, const adt_bf16* k_cache, const adt_bf16* v_cache,
                         const int32_t* kv_len, int64_t cache_stride_b, int64_t cache_stride_h,
                         const adt_bf16* k_tree, const adt_bf16* v_tree, const int32_t* parents,
                         const int32_t* node_offsets, int32_t B, int32_t H, int32_t Hkv, int32_t D,
                         int32_t max_nodes, int32_t max_kv, float softmax_scale, adt_bf16* out,
                         float* lse, void* workspace, size_t workspace_bytes, void* stream) {
  adt::TraceRange trace_("adt_tree_attn");
  adt_status st = check_args(q, k_cache, v_cache, kv_len, cache_stride_b, cache_stride_h, k_tree, v_tree, parents,
                             node_offsets, B, H, Hkv, D, max_nodes, max_kv, softmax_scale, out);
  if (st != ADT_OK) return st;
  adt::DeviceInfo info;
  st = adt::device_info(&info);
  if (st != ADT_OK) return st;
  const int Bq = B * qtiles_for(max_nodes);
  const int splits = choose_splits(info.sm_count, Bq, H, D, max_kv, info.device, max_nodes > kMaxNodes);
  const WsLayout w = ws_layout(Bq, H, D, splits);
  if (!workspace || workspace_bytes < w.total || !adt::aligned16(workspace)) return ADT_ERR_WORKSPACE;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  TcParams prm = make_params(q, kv_len, k_tree, v_tree, parents, node_offsets, B, H, Hkv, max_kv, max_nodes, splits,
                             softmax_scale, out, lse, info.error_word);
  prm.part_o = reinterpret_cast<float*>(ws + w.part_o);
  prm.part_ml = reinterpret_cast<float2*>(ws + w.part_ml);
  prm.tickets = reinterpret_cast<unsigned*>(ws + w.tickets);
  cudaStream_t s = adt::as_stream(stream);
  return launch_any(prm, D, k_cache, v_cache, cache_stride_b, cache_stride_h, s, info.device, info.sm_count, true);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// adt_tree_attn_noalloc: the same tree attention for callers that cannot
// allocate device memory themselves, for example a plugin inside a serving
// engine whose host owns every device allocation, or code on a latency-
// critical thread that must not call cudaMalloc (it can synchronise the
// device).  The scratch that adt_tree_attn takes as a workspace (split
// partials and completion tickets) lives in one fixed, per-device static
// array instead.
// ---------------------------------------------------------------------------

// 4 MiB of scratch, held by every GPU that loads the library until the
// process exits.  Shared by all calls on a device: calls that overlap on the
// GPU (different streams, or different host threads) race on it.
static constexpr size_t kNoAllocScratchBytes = size_t(4) << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

namespace {

constexpr int kNoAllocMaxDevices = 64;
std::once_flag g_noalloc_once[kNoAllocMaxDevices];
void* g_noalloc_ptr[kNoAllocMaxDevices];
cudaError_t g_noalloc_status[kNoAllocMaxDevices];

// Runs once per device, with that device current: the array's name is a
// host-side stand-in in host code, so the kernel needs its device address.
void noalloc_setup(int dev) {
  void* p = nullptr;
  g_noalloc_status[dev] = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  g_noalloc_ptr[dev] = p;
}

// What a launch with `splits` key splits uses: nothing when the splits merge
// inside their cluster (splits <= kMaxClusterSplits, the kernel returns
// before it touches tickets or partials); otherwise Bq*H tickets, then
// Bq*H*splits partial rows (m, l) and partial outputs of 64 rows x D.
struct NoAllocLayout {
  size_t tickets, part_ml, part_o, total;
};

NoAllocLayout noalloc_layout(int Bq, int H, int D, int splits) {
  NoAllocLayout w{};
  if (splits <= kMaxClusterSplits) return w;
  const size_t bh = static_cast<size_t>(Bq) * H;
  const size_t bhs = bh * splits;
  w.tickets = 0;
  w.part_ml = adt::align_up(bh * sizeof(unsigned), 256);
  w.part_o = adt::align_up(w.part_ml + bhs * kMaxNodes * sizeof(float2), 256);
  w.total = adt::align_up(w.part_o + bhs * kMaxNodes * D * sizeof(float), 256);
  return w;
}

// The split count of a no-allocation launch: the usual heuristic's, lowered
// while a workspace merge's partials would not fit the scratch; once it is
// down to a cluster's size the splits merge in their cluster and need no
// scratch, and the count is lowered further until all clusters are
// co-resident, as the heuristic does for its own cluster-sized counts.
int noalloc_splits(int sm_count, int Bq, int H, int D, int max_kv, int dev, bool large) {
  int s = choose_splits(sm_count, Bq, H, D, max_kv, dev, large);
  while (s > kMaxClusterSplits && noalloc_layout(Bq, H, D, s).total > kNoAllocScratchBytes) --s;
  if (s <= kMaxClusterSplits) {
    const int bh = Bq * H;
    while (s > 1 && max_active_clusters(D, large, s, dev) < bh) --s;
  }
  return s;
}

}  // namespace

extern "C" adt_status adt_tree_attn_noalloc(const adt_bf16* q, const adt_bf16* k_cache,
                                            const adt_bf16* v_cache, const int32_t* kv_len,
                                            int64_t cache_stride_b, int64_t cache_stride_h,
                                            const adt_bf16* k_tree, const adt_bf16* v_tree,
                                            const int32_t* parents, const int32_t* node_offsets,
                                            int32_t B, int32_t H, int32_t Hkv, int32_t D,
                                            int32_t max_nodes, int32_t max_kv, float softmax_scale,
                                            adt_bf16* out, float* lse, void* stream) {
  adt::TraceRange trace_("adt_tree_attn_noalloc");
  adt_status st = check_args(q, k_cache, v_cache, kv_len, cache_stride_b, cache_stride_h, k_tree, v_tree, parents,
                             node_offsets, B, H, Hkv, D, max_nodes, max_kv, softmax_scale, out);
  if (st != ADT_OK) return st;
  adt::DeviceInfo info;
  st = adt::device_info(&info);
  if (st != ADT_OK) return st;
  if (info.device < 0 || info.device >= kNoAllocMaxDevices) return ADT_ERR_UNSUPPORTED;
  std::call_once(g_noalloc_once[info.device], noalloc_setup, info.device);
  if (g_noalloc_status[info.device] != cudaSuccess || !g_noalloc_ptr[info.device]) return ADT_ERR_CUDA;
  const int Bq = B * qtiles_for(max_nodes);
  const int splits = noalloc_splits(info.sm_count, Bq, H, D, max_kv, info.device, max_nodes > kMaxNodes);
  const NoAllocLayout w = noalloc_layout(Bq, H, D, splits);
  // Unreachable for the shapes check_args accepts (a workspace merge is
  // chosen only when its partials fit); kept as the guard of the array.
  if (w.total > kNoAllocScratchBytes) return ADT_ERR_WORKSPACE;
  uint8_t* ws = static_cast<uint8_t*>(g_noalloc_ptr[info.device]);
  cudaStream_t s = adt::as_stream(stream);
  // A workspace merge counts finished splits in tickets that start at zero.
  // A completed call leaves them at zero, but one that a bounded wait ended
  // (ADT_DEVERR_TIMEOUT) can leave them set, so they are cleared here, on
  // the caller's stream.  Cluster merges use no tickets.
  if (splits > kMaxClusterSplits)
    ADT_CUDA_TRY(cudaMemsetAsync(ws + w.tickets, 0, static_cast<size_t>(Bq) * H * sizeof(unsigned), s));
  TcParams prm = make_params(q, kv_len, k_tree, v_tree, parents, node_offsets, B, H, Hkv, max_kv, max_nodes, splits,
                             softmax_scale, out, lse, info.error_word);
  prm.part_o = reinterpret_cast<float*>(ws + w.part_o);
  prm.part_ml = reinterpret_cast<float2*>(ws + w.part_ml);
  prm.tickets = reinterpret_cast<unsigned*>(ws + w.tickets);
  return launch_any(prm, D, k_cache, v_cache, cache_stride_b, cache_stride_h, s, info.device, info.sm_count, false);
}

