// Step 3: block-causal GQA verify attention on GB300 (split-KV, Stream-K,
// warp-specialised persistent CTAs, 5th-generation tensor cores, all layers
// of a round in one launch).
//
// Work decomposition. For sequence b the verified block has M_b = (L_b+1)*g
// query rows per kv head (g = Hq/Hkv; row r is block position t = r / g of
// query head kvh*g + r % g) and N_b = kv_len_b + L_b + 1 visible keys. Rows
// are cut into groups of R = g * floor(128/g) (whole block positions, at most
// 128: one tcgen05 M=128 tile) and keys into 64-key tiles. All (row group, key
// tile) pairs of the batch form one tile sequence (sequence-major, then kv
// head, row group, key tile); CTA c of the persistent grid (one CTA per SM)
// takes a contiguous range of it: with equal groups its part of one group
// (aligned_ctas), else a range cut by cost (each row group weighs its tiles
// plus an item's fixed cost; find_tile), so that CTAs finish together
// whatever the ragged lengths. The plan is derived on the device from L[] and
// kv_len[] by every CTA, and it is the same for every layer (all layers share
// L and kv_len).
//
// Two streams per CTA. An item (a run of tiles of one row group) is worked on
// in steps of 128 keys by two streams in turn, each with its own softmax
// warpgroup, scores and O accumulator, so that one stream's MMAs run beside
// the other's softmax; the epilogue combines the streams' (O, m, l). One
// softmax warpgroup over 64-key tiles was the limit before: with few rows one
// warp holds them all, and its 1150 cycles per 64-key tile did not keep up
// with HBM, and large trees left the tensor cores idle three quarters of the
// time. 8 sequences of 131072 keys (64/8 heads): 771 -> 602 us (105% of the
// copy rate); B = 64 ragged: 326 -> 286; 32 layers at B = 1: 302 -> 234; a
// 512-node tree, 4 layers: 367 -> 220 (with what is said below).
//
// Roles in a CTA (384 threads):
//  * producer warp: walks the CTA's range layer after layer in items; loads
//    the group's Q rows (one 3-D TMA box per 64-column half: R/g positions x g
//    heads) and K and V of the tiles (3-D TMA, 128-byte swizzle) into a ring
//    of chunks (K or V of 128 keys), in the order in which the MMA warp uses
//    them;
//  * MMA warp: one thread issues S = Q K^T (tcgen05.mma, A and B K-major from
//    shared memory, fp32 accumulator in tensor memory) and O += P V (A = P
//    from tensor memory, B = V MN-major from shared memory), and signals
//    completions with tcgen05.commit;
//  * softmax warpgroups (thread i <-> tensor-memory lane i = row i of the
//    group): read S, mask keys beyond kv_len_b + t, keep the online softmax in
//    the log2 domain, write P (bf16) over the scores they have read, and at
//    the end of an item normalise O and store it (or a split partial);
//  * two merge warps: merge the split groups of earlier layers; every warp
//    helps with the last layer's.
// Registers are what the roles' code must fit: with the merge's calls in the
// softmax path 120 bytes of spills made every wait and epilogue wait for
// local memory behind the K/V stream (B = 1: 361 us instead of 268), so the
// merge is one inline copy outside the roles and holds 12 loads per lane.
// Scores are read once: the reference max of a row is that of its first 32
// keys in the item, raised only when a later key exceeds it by more than 8 (a
// factor 2^8), so O is rescaled in tensor memory rarely; p <= 2^8 keeps bf16
// P and fp32 O in range, and O / l is unchanged by the choice of reference.
// (A pass for the tile's max before the one that forms P: the 512-node tree 332
// us instead of 320, all else equal. Two copies of the 32-key step, the second
// chunk's loads issued ahead, were slower, 337 and B = 1 290 instead of 265:
// the role loops are bound by instruction fetches as soon as they are long.)
//
// Layers. Layer l+1 may read Q, the block's own keys (positions >= kv_len_b)
// and layer l's partials only after every CTA has finished layer l: a
// grid-wide barrier (one counter per layer; the launch is cooperative, so all
// CTAs are resident and the bounded waits end). The cache prefix
// (keys < kv_len_b) is state from earlier rounds, so the producer streams the
// next layer's prefix tiles while the softmax warps still finish the current
// layer.
//
// Split groups. A row group covered by one CTA is written directly. A group
// spread over CTAs c0..c1 leaves one fp32 partial (O, m, l) per CTA, in slot
// 2c+1 for c0 (its last item) and 2c for the others (their first item), in a
// buffer chosen by the layer (l mod 3). After the barrier that ends layer
// l, each of those CTAs merges its share of the group's rows from all parts
// in CTA order (deterministic, spread over every contributing SM); the merge
// of layer l runs beside the CTA's items of layer l+1. The last layer waits
// for no grid barrier: a group's parts are counted in as they are written,
// and its CTAs merge it once all are in.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cstdio>
#include <cstdlib>
#include <memory>

#include "common.cuh"
#include "tc.cuh"

namespace libraspec {

constexpr int kStreams = 2;                    // softmax warpgroups (tile streams) per CTA
constexpr int kSoftmaxWarps = 4 * kStreams;
constexpr int kProducerWarp = kSoftmaxWarps;
constexpr int kMmaWarp = kSoftmaxWarps + 1;
constexpr int kMergeWarp = kSoftmaxWarps + 2;  // the first of two
constexpr int kAttnThreads = (kSoftmaxWarps + 4) * 32;
constexpr int kMaxWaitIters = 1 << 24;
constexpr int kSoftmaxBar = 1;  // named barrier of the softmax warpgroups
constexpr float kRescaleLog2 = 8.f;
constexpr int kTmemCols = 512;

__device__ __forceinline__ void softmax_sync() {
  asm volatile("bar.sync %0, %1;" ::"n"(kSoftmaxBar), "n"(kSoftmaxWarps * 32) : "memory");
}
// Barrier of the softmax warpgroups that also tells whether any of their threads holds `pred`.
__device__ __forceinline__ bool softmax_any(bool pred) { return bar_any<kSoftmaxBar, kSoftmaxWarps * 32>(pred); }

// (d0, d1) = (a0, a1) * b + c, and (d0, d1) += (a0, a1): one instruction for two elements
__device__ __forceinline__ void fma2(float& d0, float& d1, float a0, float a1, float b, float c) {
  asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %4};\n\tmov.b64 c, {%5, %5};\n\t"
      "fma.rn.f32x2 a, a, b, c;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b), "f"(c));
}
__device__ __forceinline__ void add2(float& d0, float& d1, float a0, float a1) {
  asm("{\n\t.reg .b64 a, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 d, {%0, %1};\n\t"
      "add.rn.f32x2 d, d, a;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "+f"(d0), "+f"(d1)
      : "f"(a0), "f"(a1));
}

// bits [0, n) set (n clamped to [0, 64])
__device__ __forceinline__ uint64_t low_bits(int n) {
  return n <= 0 ? 0ull : (n >= 64 ? ~0ull : ((1ull << n) - 1ull));
}

// Bits [o, o + 64) of the bit set row[0 .. words) (bits outside read as 0;
// o may be negative).
__device__ __forceinline__ uint64_t bit_window(const uint64_t* __restrict__ row, int words, int o) {
  const int q = o >> 6, r = o & 63;  // floor division
  const uint64_t lo = (q >= 0 && q < words) ? __ldg(row + q) : 0ull;
  const uint64_t hi = (q + 1 >= 0 && q + 1 < words) ? __ldg(row + q + 1) : 0ull;
  return r == 0 ? lo : (lo >> r) | (hi << (64 - r));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// ---------------------------------------------------------------------------
// Device-side plan.
// ---------------------------------------------------------------------------
struct SeqPlan {
  int M, n_mg, N, n_tiles;  // rows, row groups, visible keys, key tiles
  bool ok;
};

__device__ __forceinline__ SeqPlan seq_plan(int b, int B, const int32_t* kv_len, const int32_t* Ls, int K, int g,
                                            int R, int S_cap) {
  SeqPlan p{0, 0, 0, 0, false};
  if (b >= B) return p;
  const int Lb = Ls[b], kv = kv_len[b];
  if (Lb < 0 || Lb > K || kv < 0 || (long)kv + Lb + 1 > S_cap) return p;
  p.ok = true;
  p.M = (Lb + 1) * g;
  p.n_mg = (p.M + R - 1) / R;
  p.N = kv + Lb + 1;
  p.n_tiles = (p.N + kAttnTileKeys - 1) / kAttnTileKeys;
  return p;
}

// Warp-wide: total tiles T of the batch, its row groups (*groups) and the tiles
// of every group if they have the same (*equal, else 0); flags invalid sequences.
__device__ long long total_tiles(int B, const int32_t* kv_len, const int32_t* Ls, int K, int g, int R, int Hkv,
                                 int S_cap, int* status, bool report, long long* groups, int* equal) {
  const int lane = threadIdx.x & 31;
  long long tot = 0, ng = 0;
  int t_min = 0x7fffffff, t_max = 0;
  bool bad = false;
  for (int b = lane; b < B; b += 32) {
    const SeqPlan p = seq_plan(b, B, kv_len, Ls, K, g, R, S_cap);
    if (!p.ok) bad = true;
    else {
      tot += (long long)Hkv * p.n_mg * p.n_tiles;
      ng += (long long)Hkv * p.n_mg;
      t_min = min(t_min, p.n_tiles);
      t_max = max(t_max, p.n_tiles);
    }
  }
  t_min = __reduce_min_sync(0xffffffffu, t_min);
  t_max = __reduce_max_sync(0xffffffffu, t_max);
  *equal = t_min == t_max ? t_max : 0;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    tot += __shfl_xor_sync(0xffffffffu, tot, off);
    ng += __shfl_xor_sync(0xffffffffu, ng, off);
  }
  *groups = ng;
  if (report && __any_sync(0xffffffffu, bad) && lane == 0) {
    int bits = 0;
    for (int b = 0; b < B; ++b) {
      const int Lb = Ls[b], kv = kv_len[b];
      if (Lb < 0 || Lb > K) bits |= LIBRASPEC_ST_BAD_LENGTH;
      else if (kv < 0 || (long)kv + Lb + 1 > S_cap) bits |= LIBRASPEC_ST_KV_OVERFLOW;
    }
    raise_status(status, bits);
  }
  return tot;
}

// a / b for a >= 0, b > 0: 32-bit when both fit (a 64-bit division is a
// long software sequence, and the plan runs on one warp before any copy)
__device__ __forceinline__ long long div_nn(long long a, long long b) {
  if ((((unsigned long long)a | (unsigned long long)b) >> 32) == 0) return (long long)((uint32_t)a / (uint32_t)b);
  return a / b;
}

__device__ __forceinline__ long long range_lo(int c, long long T, int G) { return div_nn((long long)c * T, G); }

// CTA whose range holds tile t: the largest c with c*T/G <= t.
__device__ __forceinline__ int cta_of(long long t, long long T, int G) {
  return (int)div_nn((t + 1) * (long long)G - 1, T);
}

// Cost-weighted Stream-K. A row group costs its key tiles plus C (an item's
// fixed cost: the Q load the first S waits for, the epilogue, a partial's
// merge, in tile-equivalents), placed before its tiles; the batch weighs
// W = T + C * groups, and CTA c takes the tiles of the weighted range
// [c W / G, (c+1) W / G). A boundary inside a group's C falls on the
// group's first tile. C = 0 is the plain split by tiles. C is 4, or a quarter
// of a CTA's tiles if that is less (a cost of several tiles would leave CTAs
// with few tiles without any): 16 paged sequences 110 -> 102 us (2 layers), a
// tree of 512 nodes 352 -> 339 (4 layers), ragged B = 64 312 -> 296; C = 8 and
// 12 gave ragged 298 and 301, the tree 332.
struct TileLoc {
  long long tile;       // the tile (T: past the end)
  int b;                // its sequence
  long long seq_start;  // first tile of sequence b
  int group0;           // global index of b's first row group
  SeqPlan p;
};

// The tile at weighted position x (at C = 0: tile x), and where it lies (warp-wide).
__device__ TileLoc find_tile(long long x, int C, long long T, int B, const int32_t* kv_len, const int32_t* Ls, int K,
                             int g, int R, int Hkv, int S_cap) {
  const int lane = threadIdx.x & 31;
  TileLoc loc{T, 0, 0, 0, {}};
  long long carry_t = 0;
  int carry_g = 0;
  for (int base = 0; base < B; base += 32) {
    const SeqPlan p = seq_plan(base + lane, B, kv_len, Ls, K, g, R, S_cap);
    const int ng = p.ok ? Hkv * p.n_mg : 0;
    const long long nt = (long long)ng * p.n_tiles;
    long long inc_t = nt;
    int inc_g = ng;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const long long a = __shfl_up_sync(0xffffffffu, inc_t, off);
      const int c = __shfl_up_sync(0xffffffffu, inc_g, off);
      if (lane >= off) { inc_t += a; inc_g += c; }
    }
    const long long st = carry_t + inc_t - nt;  // the sequence's first tile and row group
    const int sg = carry_g + inc_g - ng;
    const long long sw = st + (long long)C * sg;
    const unsigned ball = __ballot_sync(0xffffffffu, nt > 0 && x >= sw && x < sw + nt + (long long)C * ng);
    if (ball) {
      const int src = __ffs(ball) - 1;
      loc.b = base + src;
      loc.seq_start = __shfl_sync(0xffffffffu, st, src);
      loc.group0 = __shfl_sync(0xffffffffu, sg, src);
      loc.p = seq_plan(loc.b, B, kv_len, Ls, K, g, R, S_cap);
      const long long o = x - (loc.seq_start + (long long)C * loc.group0);
      const long long gib = div_nn(o, loc.p.n_tiles + C), r = o - gib * (loc.p.n_tiles + C);
      loc.tile = loc.seq_start + gib * loc.p.n_tiles + (r > C ? r - C : 0);
      return loc;
    }
    carry_t += __shfl_sync(0xffffffffu, inc_t, 31);
    carry_g += __shfl_sync(0xffffffffu, inc_g, 31);
  }
  return loc;
}

// Equal groups. Where every row group has the same number nt of tiles (one
// sequence, or equal caches) and the NG groups fit the grid, each group may
// get p = G / NG CTAs of its own: no CTA has two items, and a group of p = 1
// is never split nor merged. Taken when the longest range, nt / p tiles, is
// at most kAlignTiles above the even split's T / G: what a group cut at any
// tile costs is an extra item per CTA and a merge of parts of unequal length,
// the more the more rows it has. Over 56 shapes of equal groups (trees of 64
// to 512 nodes, 1 to 36 sequences of 500 to 32000 keys, graphs of 2 to 8
// layers) the rule gains 1 to 48% where it applies against the cut by cost
// and loses nowhere: 512 nodes (136 groups of 128 rows, 4 layers) 213 us
// against 245, 100 nodes 89 against 121, 16 sequences of 1500 keys 46 against
// 56, 8 of 4096 (5.6 tiles above) 61 against 63. Between 10 and 20 tiles above
// it would still gain mostly (500 nodes 209 against 241, 20 sequences of 28/4
// heads 61.7 against 60.6), from 24 on it loses (10 sequences of 4096: 84
// against 72).
constexpr int kAlignTiles = 10;
__device__ __forceinline__ int aligned_ctas(long long T, long long NG, int nt, int G) {
  if (nt <= 0 || NG > G) return 0;
  const int p = min((int)(G / NG), nt);
  const long long longest = (nt + p - 1) / p;
  return longest * G <= T + (long long)kAlignTiles * G ? p : 0;
}

// Weighted position of tile t of global row group `group` (the groups up to
// and including it each put C before their tiles).
__device__ __forceinline__ long long weighted_pos(long long t, long long group, int C) {
  return t + (long long)C * (group + 1);
}

// Bounded poll of a grid-barrier counter (acquire).
__device__ __forceinline__ bool wait_counter(const uint32_t* ctr, uint32_t target) {
  for (int i = 0; i < kMaxWaitIters; ++i) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
    if (v >= target) return true;
    __nanosleep(32);
  }
  return false;
}

// One item handed from the producer to the MMA and softmax warps.
struct ItemInfo {
  int b, kvh, mg, rows, kv;
  int key0, key1;  // keys [key0, key1)
  int partial;     // 1: write a partial, else write O
  int slot;        // partial slot
  int grp;         // global row group index
  int last;        // 1: the CTA's last item of the layer; 2: no item, in any layer
  int pad[5];
};
static_assert(sizeof(ItemInfo) == 64, "items lie in 64-byte slots");

// A split row group this CTA helps merge (the same for every layer).
struct MergeTask {
  int b, kvh, mg, rows, c0, np;
  int grp;  // global row group index
  int pad;
};
static_assert(2 * sizeof(MergeTask) <= 64, "two merge tasks fit their shared-memory slot");

constexpr int kMaxLayers = kAttnMaxLayers;

struct LayerPtrs {
  const __nv_bfloat16* Q;
  __nv_bfloat16* O;
  float* lse;
};

// Everything a launch needs per layer, passed by value as one kernel
// parameter (< 32 KB).
struct LayerSet {
  CUtensorMap K[kMaxLayers];
  CUtensorMap V[kMaxLayers];
  CUtensorMap Q[kMaxLayers];
  LayerPtrs p[kMaxLayers];
  int n;
};
static_assert(sizeof(LayerSet) <= 32000, "kernel parameters are limited to 32764 bytes");

template <int D>
struct AttnSmem {
  static constexpr int kBoxes = D / 64;
  static constexpr int kChunkBytes = kBoxes * 16384;     // K or V of one 128-key tile
  static constexpr int kChunks = D == 128 ? 5 : 10;      // in the ring
  static constexpr int kQ = 0;
  static constexpr int kRing = kQ + kBoxes * 16384;      // (Q: per 64 columns 128 rows)
  // mbarriers: full[chunks], empty[chunks], ifull[2], iempty[2], sfull[2], pfull[2], pvdone[2], qfull, qempty,
  // ofree, drain
  static constexpr int kBar = kRing + kChunks * kChunkBytes;
  static constexpr int kNumBars = 2 * kChunks + 5 * 2 + 4;
  static constexpr int kInfo = kBar + ((8 * kNumBars + 63) / 64) * 64;
  static constexpr int kTasks = kInfo + 2 * 64;
  static constexpr int kTmem = kTasks + 64;
  // [0] abort, [1] merge tasks, [2] the tasks are set, [3] merge chunks per
  // layer, [4] chunks claimed, [5] the last layer's merges may start, [6..8]
  // chunks done of the layers in each buffer of partials
  static constexpr int kMisc = kTmem + 16;
  // (m, l) of each stream's rows, for the epilogue of an item whose streams are combined
  static constexpr int kStat = kMisc + 48;
  // kv_len and L of up to kPlanCap sequences, read once from global memory
  // for the CTA's tile plan (a larger batch plans from global memory)
  static constexpr int kPlanCap = 1024;
  static constexpr int kPlan = kStat + kStreams * 128 * 8;
  static constexpr int kBytes = kPlan + 2 * 4 * kPlanCap;
  static constexpr int kAlloc = kBytes + 1024;           // room to align the base to 1024
  // tensor-memory columns: per stream S of a tile (128 fp32, its P as 64
  // columns of bf16 pairs in the same place) and O (D fp32); lane = row
  static constexpr int kColS = 0, kColO = 256;
  static_assert(kStat % 16 == 0 && kInfo % 16 == 0, "alignment");
  static_assert(kAlloc <= 227 * 1024, "shared memory per CTA");
  // paged caches: the page of each of the CTA's tiles, after everything else
  static constexpr int kPageCap = 4096;
  static constexpr int kAllocPaged = kAlloc + kPageCap * 4;
  static_assert(kAllocPaged <= 227 * 1024, "shared memory per CTA (paged)");
};

// Merging a layer's split groups. This CTA merges its share of rows
// [rows*k/np, rows*(k+1)/np) of each group it contributed to (k = its index
// among the group's np CTAs): O = sum_p w_p O_p / sum_p w_p l_p with
// w_p = 2^(m_p - M), M = max m_p, parts in CTA order. The share is cut into
// chunks of (row, 4-column) items that a warp claims once the layer's grid
// barrier has passed: the two merge warps, beside the next layer's items; the
// last layer's any warp whose role is done. A lane
// loads (m_p, l_p) and its 4 columns of O_p for a batch of parts at once and
// folds the batch in with a running maximum, so a chunk costs one memory
// round trip per batch and no weights are staged in shared memory.

// This CTA's share [u0, u0 + nr) of task t's rows.
__device__ __forceinline__ int merge_share(const MergeTask& t, int& u0) {
  const int k_me = (int)blockIdx.x - t.c0;
  u0 = (int)((long long)t.rows * k_me / t.np);
  return (int)((long long)t.rows * (k_me + 1) / t.np) - u0;
}

constexpr int kMergeLoads = 12;  // of a lane in flight (with 16, registers spill)

// Items per lane in a chunk of a group of np parts: J items x 12/J parts are
// in flight per batch, and a share of `items` items costs ceil(items / 32J)
// chunks x ceil(np / (12/J)) batches, one memory round trip each. J = 4 wins
// for many rows over few parts (tree and long blocks), J = 1 for one row
// over many parts (short blocks at B = 1); ties go to J = 1 (more chunks to
// share among helping warps).
__device__ __forceinline__ int merge_j(int np, int items) {
  const int trips1 = ((items + 31) / 32) * ((np + kMergeLoads - 1) / kMergeLoads);
  const int trips4 = ((items + 127) / 128) * ((np + kMergeLoads / 4 - 1) / (kMergeLoads / 4));
  return trips4 < trips1 ? 4 : 1;
}

template <int D>
__device__ __forceinline__ int merge_chunk_count(const MergeTask* tasks, int n_tasks) {
  int n = 0;
  for (int ti = 0; ti < n_tasks; ++ti) {
    int u0;
    const int items = merge_share(tasks[ti], u0) * (D / 4);
    const int ci = 32 * merge_j(tasks[ti].np, items);
    n += (items + ci - 1) / ci;
  }
  return n;
}

// Chunk lc of task t: items (lc*J + j)*32 + lane, j < J.
template <int J, int D>
__device__ __forceinline__ void merge_chunk(const MergeTask& t, int u0, int nr, int lc, const float* __restrict__ part_o,
                                            const float* __restrict__ part_ml, int K, int Hq, int g, int R,
                                            __nv_bfloat16* __restrict__ O, float* __restrict__ lse) {
  constexpr int PB = kMergeLoads / J, C4 = D / 4;
  const int lane = threadIdx.x & 31;
  const int np = t.np, c0 = t.c0, items = nr * C4;
  float M[J], Ls[J];
  float4 acc[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    M[j] = -INFINITY;
    Ls[j] = 0.f;
    acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  for (int p0 = 0; p0 < np; p0 += PB) {
    float2 ml[J][PB];
    float4 v[J][PB];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int i = (lc * J + j) * 32 + lane;
      const int r = i / C4, c = i - r * C4;
#pragma unroll
      for (int k = 0; k < PB; ++k) {
        const int p = p0 + k;
        if (i < items && p < np) {
          const size_t at = (size_t)(p == 0 ? 2 * c0 + 1 : 2 * (c0 + p)) * kAttnRows + u0 + r;
          ml[j][k] = __ldcg(reinterpret_cast<const float2*>(part_ml + at * 2));
          v[j][k] = __ldcg(reinterpret_cast<const float4*>(part_o + at * D) + c);
        } else {
          ml[j][k] = make_float2(-INFINITY, 0.f);
          v[j][k] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
      float bm = -INFINITY;
#pragma unroll
      for (int k = 0; k < PB; ++k) bm = fmaxf(bm, ml[j][k].x);
      const float Mn = fmaxf(M[j], bm);
      if (Mn == -INFINITY) continue;  // no visible key in these parts yet
      const float f = ex2_approx(M[j] - Mn);  // 0 while M is still -inf
      acc[j].x *= f;
      acc[j].y *= f;
      acc[j].z *= f;
      acc[j].w *= f;
      Ls[j] *= f;
      M[j] = Mn;
#pragma unroll
      for (int k = 0; k < PB; ++k) {
        const float w = ex2_approx(ml[j][k].x - Mn);  // 0 for a part with no visible key
        acc[j].x += w * v[j][k].x;
        acc[j].y += w * v[j][k].y;
        acc[j].z += w * v[j][k].z;
        acc[j].w += w * v[j][k].w;
        Ls[j] += w * ml[j][k].y;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int i = (lc * J + j) * 32 + lane;
    if (i >= items) continue;
    const int r = i / C4, c = i - r * C4;
    const float inv = 1.f / Ls[j];
    const int rr = t.mg * R + u0 + r;
    const int tt = rr / g, hq = t.kvh * g + rr % g;
    uint2 o;
    o.x = pack_bf16(acc[j].x * inv, acc[j].y * inv);
    o.y = pack_bf16(acc[j].z * inv, acc[j].w * inv);
    *reinterpret_cast<uint2*>(O + (((size_t)t.b * (K + 1) + tt) * Hq + hq) * D + c * 4) = o;
    if (lse && c == 0) lse[((size_t)t.b * (K + 1) + tt) * Hq + hq] = (M[j] + __log2f(Ls[j])) * kLn2;
  }
}

// Claims and merges chunks of layers up to `last_layer` until none is left,
// oldest first. Chunks are numbered [l * C, (l + 1) * C) for layer l on the
// CTA's monotonic counter; ctr_done counts the chunks merged (stores done) of
// the layers in each buffer of partials.
template <int D>
__device__ __forceinline__ void merge_chunks(int last_layer, const LayerSet& set, const MergeTask* tasks, int n_tasks, int C,
                             int* ctr_claim, int* ctr_done, int K, int Hq, int Hkv, int R,
                             const float* __restrict__ part_buf_o, const float* __restrict__ part_buf_ml,
                             size_t part_o_stride, size_t part_ml_stride) {
  const int lane = threadIdx.x & 31;
  const int g = Hq / Hkv;
  const int hi = (last_layer + 1) * C;
  for (;;) {
    int u = 0;
    if (lane == 0) {
      u = *reinterpret_cast<volatile int*>(ctr_claim);
      while (u < hi) {
        const int prev = atomicCAS(ctr_claim, u, u + 1);
        if (prev == u) break;
        u = prev;
      }
    }
    u = __shfl_sync(0xffffffffu, u, 0);
    if (u >= hi) return;
    // the chunk's layer, task and index within the task
    const int layer = u / C;
    const float* part_o = part_buf_o + (layer % kAttnPartBufs) * part_o_stride;
    const float* part_ml = part_buf_ml + (layer % kAttnPartBufs) * part_ml_stride;
    __nv_bfloat16* O = set.p[layer].O;
    float* lse = set.p[layer].lse;
    int lc = u - layer * C, ti = 0, u0 = 0, nr = 0;
    for (; ti < n_tasks; ++ti) {
      nr = merge_share(tasks[ti], u0);
      const int ci = 32 * merge_j(tasks[ti].np, nr * (D / 4));
      const int nc = (nr * (D / 4) + ci - 1) / ci;
      if (lc < nc) break;
      lc -= nc;
    }
    if (ti < n_tasks) {
      const MergeTask& t = tasks[ti];
      if (merge_j(t.np, nr * (D / 4)) == 1) merge_chunk<1, D>(t, u0, nr, lc, part_o, part_ml, K, Hq, g, R, O, lse);
      else merge_chunk<4, D>(t, u0, nr, lc, part_o, part_ml, K, Hq, g, R, O, lse);
    }
    __syncwarp();
    if (lane == 0) {
      __threadfence_block();  // (the warp's reads lie before the count)
      atomicAdd(ctr_done + layer % kAttnPartBufs, 1);
    }
  }
}

// PAGED: the caches are page pools [n_pages, Hkv, page_size, d] and key s of
// sequence b lives at page block_table[b * max_pages + s / page_size], row
// s % page_size (page_size a multiple of 64, so a key tile lies in one page);
// S_cap is then max_pages * page_size.
// tree_vis (optional, [B, K+1, tree_words]): the block is a draft tree and
// row t sees the block keys of the set bits (bit j <-> block position j + 1)
// besides the root and the prefix; nullptr: the chain draft (block-causal).
template <int D, bool PAGED>
__global__ void __launch_bounds__(kAttnThreads, 1) verify_attn_kernel(
    const __grid_constant__ LayerSet set, const int32_t* __restrict__ kv_len, const int32_t* __restrict__ Ls,
    const uint64_t* __restrict__ tree_vis, int tree_words,
    const int32_t* __restrict__ block_table, int max_pages, int page_size, int n_pages, int page_cache,
    int B, int K, int Hq, int Hkv, int S_cap, float scale_log2, int min_tiles, int item_tiles,
    float* __restrict__ part_buf_o,
    float* __restrict__ part_buf_ml, size_t part_o_stride, size_t part_ml_stride, uint32_t* __restrict__ bar_cnt,
    uint32_t* __restrict__ grp_cnt, int* __restrict__ status) {
  using SM = AttnSmem<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sQ = smem_u32(smem + SM::kQ);
  const uint32_t sRing = smem_u32(smem + SM::kRing);
  const uint32_t bFull = smem_u32(smem + SM::kBar);
  const uint32_t bEmpty = bFull + 8 * SM::kChunks;
  const uint32_t bIFull = bEmpty + 8 * SM::kChunks;
  const uint32_t bIEmpty = bIFull + 16;
  const uint32_t bSFull = bIEmpty + 16;   // [stream]
  const uint32_t bPFull = bSFull + 16;    // [stream]
  const uint32_t bPVDone = bPFull + 16;   // [stream]
  const uint32_t bQFull = bPVDone + 16;
  const uint32_t bQEmpty = bQFull + 8;
  const uint32_t bOFree = bQEmpty + 8;
  const uint32_t bDrain = bOFree + 8;
  ItemInfo* info = reinterpret_cast<ItemInfo*>(smem + SM::kInfo);
  MergeTask* tasks = reinterpret_cast<MergeTask*>(smem + SM::kTasks);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + SM::kTmem);
  volatile int* misc = reinterpret_cast<int*>(smem + SM::kMisc);
  uint32_t* exit_cnt = bar_cnt + kMaxLayers;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = Hq / Hkv;
  const int R = g * (kAttnRows / g);  // rows per group: whole block positions
  const int n_layers = set.n;
  const uint32_t n_ctas = gridDim.x;
  // the tensor maps' first use then finds them on chip
  if (warp == kProducerWarp)
    for (int l = lane; l < n_layers; l += 32) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&set.Q[l])) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&set.K[l])) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&set.V[l])) : "memory");
    }
  // the plan reads kv_len and L from shared memory when the batch fits
  const bool plan_cached = B <= SM::kPlanCap;
  int32_t* plan_kv = reinterpret_cast<int32_t*>(smem + SM::kPlan);
  int32_t* plan_L = plan_kv + SM::kPlanCap;
  const int32_t* kvs = plan_cached ? plan_kv : kv_len;
  const int32_t* Lss = plan_cached ? plan_L : Ls;

  if (plan_cached)
    for (int b = tid; b < B; b += kAttnThreads) {
      plan_kv[b] = kv_len[b];
      plan_L[b] = Ls[b];
    }
  if (tid == 0) {
    for (int s = 0; s < SM::kChunks; ++s) {
      mbar_init(bFull + 8 * s, 1);
      mbar_init(bEmpty + 8 * s, 1);  // the MMA warp's commit after the chunk's last use
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(bIFull + 8 * q, 1);
      mbar_init(bIEmpty + 8 * q, 1 + kSoftmaxWarps);  // the item has been read
      mbar_init(bPFull + 8 * q, 4);
      mbar_init(bPVDone + 8 * q, 1);
      mbar_init(bSFull + 8 * q, 1);
    }
    mbar_init(bQFull, 1);   // the producer's arrive; Q bytes as transactions
    mbar_init(bQEmpty, 1);  // the MMA warp's commit after the item's last S
    mbar_init(bOFree, kSoftmaxWarps);
    mbar_init(bDrain, 1);
    misc[0] = 0;
    misc[2] = 0;
    misc[4] = 0;
    misc[5] = 0;
    for (int i = 0; i < kAttnPartBufs; ++i) misc[6 + i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    // one CTA per SM: the whole tensor memory
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(const_cast<uint32_t*>(tmem_slot))),
                 "n"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  int* merge_claimed = const_cast<int*>(misc) + 4;
  int* merge_done = const_cast<int*>(misc) + 6;
  // The plan (identical for every layer) is worked out by the warps that need
  // it, in one copy of code that runs while the others already wait for their
  // first item: the producer needs the CTA's first and last tile, the first
  // merge warp the split groups the CTA contributes to. (One warp planning for
  // all before a block barrier, and the producer locating every item again:
  // 16 paged sequences, 2 layers, 98 us instead of 96.)
  struct {
    long long lo, hi;  // the CTA's tiles
    TileLoc first;     // where tile lo lies
  } plan{};
  if (warp == kProducerWarp || warp == kMergeWarp) {
    long long NG = 0;
    int equal = 0;
    const long long T = total_tiles(B, kvs, Lss, K, g, R, Hkv, S_cap, status,
                                    blockIdx.x == 0 && warp == kProducerWarp, &NG, &equal);
    int G = (int)n_ctas;
    if (T > 0) {
      const long long g_cap = div_nn(T + min_tiles - 1, min_tiles);
      if ((long long)G > g_cap) G = (int)g_cap;
    }
    const int c = blockIdx.x;
    const int p_cta = aligned_ctas(T, NG, equal, G);  // > 0: CTAs of each group
    // an item's fixed cost in tiles, less where a CTA has few
    const int C = T > 0 && p_cta == 0 ? (int)min((long long)item_tiles, div_nn(T, 4 * (long long)G)) : 0;
    const long long W = T + (long long)C * NG;  // weighted length
    long long x0 = 0, x1 = 0;                   // the CTA's range in weighted positions
    if (p_cta > 0) {
      const int grp = c / p_cta, k = c - grp * p_cta;
      if (grp < NG) {
        x0 = (long long)grp * equal + group_part(equal, k, p_cta);
        x1 = (long long)grp * equal + group_part(equal, k + 1, p_cta);
      }
    } else if (T > 0 && c < G) {
      x0 = range_lo(c, W, G);
      x1 = range_lo(c + 1, W, G);
    }
    if (x0 < x1) {
      int n_tasks = 0, group_lo = 0;
      // e = 0: the first tile; 1: the end; 2 (merges): the last tile
#pragma unroll 1
      for (int e = 0; e < (warp == kMergeWarp ? 3 : 2); ++e) {
        if (e == 2 && plan.lo >= plan.hi) break;
        const TileLoc loc = find_tile(e == 0 ? x0 : e == 1 ? x1 : plan.hi - 1, e == 2 ? 0 : C, T, B, kvs, Lss, K, g, R,
                                      Hkv, S_cap);
        if (e == 0) {
          plan.lo = loc.tile;
          plan.first = loc;
        }
        if (e == 1) plan.hi = loc.tile;
        if (e == 1 || warp == kProducerWarp) continue;
        // a group at either end of the range that other CTAs share
        const int nt = loc.p.n_tiles;
        const int gib = (int)div_nn(loc.tile - loc.seq_start, nt), group = loc.group0 + gib;
        const long long gstart = loc.seq_start + (long long)gib * nt, gend = gstart + nt;
        MergeTask t;
        t.b = loc.b;
        t.kvh = gib / loc.p.n_mg;
        t.mg = gib % loc.p.n_mg;
        t.rows = min(R, loc.p.M - t.mg * R);
        t.c0 = p_cta > 0 ? group * p_cta : cta_of(weighted_pos(gstart, group, C), W, G);
        t.np = p_cta > 0 ? p_cta : cta_of(weighted_pos(gend - 1, group, C), W, G) - t.c0 + 1;
        t.grp = group;
        if (t.np > 1 && !(e == 2 && group == group_lo)) {
          if (lane == 0) tasks[n_tasks] = t;
          ++n_tasks;
        }
        if (e == 0) group_lo = group;
      }
      if (plan.lo >= plan.hi) n_tasks = 0;  // (the range lies in a group's fixed cost)
      if (warp == kMergeWarp && lane == 0) {
        misc[1] = n_tasks;
        misc[3] = merge_chunk_count<D>(tasks, n_tasks);  // merge chunks per layer
      }
    } else if (warp == kMergeWarp && lane == 0) {
      misc[1] = 0;
      misc[3] = 0;
    }
    if (warp == kMergeWarp && lane == 0) {
      __threadfence_block();
      misc[2] = 1;  // the merge tasks may be read
    }
    __syncwarp();
  }
  // bounded wait (one lane) for the merge tasks
  auto tasks_ready = [&]() {
    for (int i = 0; i < kMaxWaitIters; ++i) {
      if (misc[2]) {
        __threadfence_block();
        return true;
      }
      if (misc[0]) return false;
      __nanosleep(64);
    }
    return false;
  };
  // bounded wait until every CTA has finished `layer` (lane 0 polls)
  auto layer_done = [&](int layer) {
    bool ok = false;
    if ((threadIdx.x & 31) == 0) ok = wait_counter(bar_cnt + layer, n_ctas) && !misc[0];
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
  };
  // bounded wait (warp-wide) until the merge warp has seen every split group
  // of the last layer complete
  auto last_groups_ready = [&]() {
    bool ok = false;
    if ((threadIdx.x & 31) == 0) {
      for (int i = 0; i < kMaxWaitIters; ++i) {
        if (misc[5]) { ok = true; break; }
        if (misc[0]) break;
        __nanosleep(64);
      }
    }
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
  };
  // bounded wait (one lane) until the next layer may write its partials
  auto next_buf_free = [&](int layer) {
    for (int i = 0; i < kMaxWaitIters; ++i) {
      if (part_buf_free(merge_done, layer, misc[3])) {
        __threadfence_block();  // (the merges' reads lie before what this thread releases)
        return true;
      }
      if (misc[0]) return false;
      __nanosleep(64);
    }
    return false;
  };
  const uint32_t tmem = *tmem_slot;

  if (warp == kProducerWarp) {
    // ======================= producer =======================
    const int c = blockIdx.x;
    const long long lo = plan.lo, hi = plan.hi;
    // lane 0 reads the abort flag for the whole warp (the loop body has warp-wide steps)
    auto aborted = [&]() { return __shfl_sync(0xffffffffu, misc[0], 0) != 0; };
    // paged: the page of every tile of the range, read once for all layers
    // (they share the block table); a range beyond the cache reads the
    // table tile by tile
    int32_t* tile_page = reinterpret_cast<int32_t*>(smem + SM::kBytes);
    const bool pages_cached = PAGED && hi - lo <= page_cache;
    auto page_of = [&](int b, int key) {
      int id = __ldg(block_table + (size_t)b * max_pages + key / page_size);
      if (id < 0 || id >= n_pages) {
        raise_status(status, LIBRASPEC_ST_BAD_PAGE);
        id = 0;  // read a valid page; the sequence's output is then meaningless
      }
      return id;
    };
    // the item at hand: row group gib of sequence loc.b, from its first tile gstart
    TileLoc loc = plan.first;
    int gib = 0;
    long long gstart = 0;
    auto first_item = [&]() {
      loc = plan.first;
      gib = lo < hi ? (int)div_nn(lo - loc.seq_start, loc.p.n_tiles) : 0;
      gstart = loc.seq_start + (long long)gib * loc.p.n_tiles;
    };
    auto next_item = [&]() {  // (there is one: the range goes on)
      gstart += loc.p.n_tiles;
      if (++gib < Hkv * loc.p.n_mg) return;
      loc.group0 += gib;
      loc.seq_start = gstart;
      gib = 0;
      do {
        loc.p = seq_plan(++loc.b, B, kvs, Lss, K, g, R, S_cap);
      } while (!loc.p.ok && loc.b < B);
    };
    if (pages_cached) {
      first_item();
      for (long long pos = lo; pos < hi;) {
        const long long iend = gstart + loc.p.n_tiles < hi ? gstart + loc.p.n_tiles : hi;
        const int key0 = (int)(pos - gstart) * kAttnTileKeys;
        for (int i = lane; i < (int)(iend - pos); i += 32)
          tile_page[pos - lo + i] = page_of(loc.b, key0 + i * kAttnTileKeys);
        pos = iend;
        if (pos < hi) next_item();
      }
      __syncwarp();
    }
    if (lo >= hi && lane == 0) {  // nothing to do in any layer
      info[0].last = 2;
      mbar_arrive(bIFull);
    }
    uint32_t item_ctr = 0, chunk_ctr = 0;           // items; chunks filled
    // K and V are read once and pass through L2 first in, first out: a stream
    // larger than L2 otherwise pushes out the kernel's own code, and a role's
    // first instructions then wait behind the copies in flight (the first
    // MMA of the ragged batch issued 4000 cycles after its operands had landed,
    // with the hint 600): 16 paged sequences, 2 layers, 96 -> 88 us, 32 layers
    // at B = 1 248 -> 240, ragged B = 64 295 -> 291.
    const uint64_t policy = evict_first_policy();
    // the next chunk may be filled
    auto chunk_free = [&]() { return bEmpty + 8 * (chunk_ctr % SM::kChunks); };
    auto chunk_parity = [&]() { return ((chunk_ctr / SM::kChunks) & 1) ^ 1; };
    for (int layer = 0; layer < n_layers && !aborted(); ++layer) {
      // layer's dependent data (Q, the block's keys) is readable once every
      // CTA has finished the previous layer
      bool ready = layer == 0;
      first_item();
      for (long long pos = lo; pos < hi && !aborted();) {
        ItemInfo it{};
        const long long gend = gstart + loc.p.n_tiles;
        const long long iend = gend < hi ? gend : hi;
        it.b = loc.b;
        it.kvh = gib / loc.p.n_mg;
        it.mg = gib % loc.p.n_mg;
        it.rows = min(R, loc.p.M - it.mg * R);
        it.kv = kvs[loc.b];
        it.key0 = (int)(pos - gstart) * kAttnTileKeys;
        it.key1 = min(loc.p.N, (int)(iend - gstart) * kAttnTileKeys);
        it.partial = ((pos == gstart) && (gend <= hi)) ? 0 : 1;
        it.slot = (pos == gstart) ? 2 * c + 1 : 2 * c;
        it.grp = loc.group0 + gib;
        it.last = iend >= hi ? 1 : 0;
        const int n_half = (int)(iend - pos), n_tiles = (n_half + 1) >> 1;
        const int zc = loc.b * Hkv + it.kvh;
        const long long item_pos = pos;  // the item's first 64-key tile in the tile sequence
        pos = iend;
        if (lane == 0) {
          // The ring is filled in the order in which the MMA warp uses it: K of
          // tile t, then V of tile t - lag.
          constexpr int lag = 2;
          int kt = 0, vt = 0;  // the next K and V tile
          auto next_is_k = [&]() { return kt < n_tiles && kt < vt + lag; };
          auto key_tile = [&](int key_half, int& y, int& z) {  // TMA row and plane of the item's 64-key tile
            y = it.key0 + key_half * kAttnTileKeys;
            z = zc;
            if (PAGED) {
              const int page = pages_cached ? tile_page[item_pos - lo + key_half] : page_of(it.b, y);
              z = page * Hkv + it.kvh;
              y %= page_size;
            }
          };
          auto fill_chunk = [&]() {
            const uint32_t ch = chunk_ctr % SM::kChunks;
            const uint32_t bar = bFull + 8 * ch, dst = sRing + ch * SM::kChunkBytes;
            const bool is_k = next_is_k();
            const int tt = is_k ? kt++ : vt++, nh = min(2, n_half - 2 * tt);
            mbar_expect_tx(bar, nh * SM::kBoxes * 8192);
            for (int h = 0; h < nh; ++h) {
              int y, z;
              key_tile(2 * tt + h, y, z);
              // K: per 64 dims 128 keys; V: per 64 keys all dims (boxes of 64 keys x 64 dims)
#pragma unroll
              for (int hb = 0; hb < SM::kBoxes; ++hb) {
                if (is_k) tma_load_3d_hint(dst + hb * 16384 + h * 8192, &set.K[layer], bar, hb * 64, y, z, policy);
                else tma_load_3d_hint(dst + (h * SM::kBoxes + hb) * 8192, &set.V[layer], bar, hb * 64, y, z, policy);
              }
            }
            ++chunk_ctr;
          };
          const int q_head = it.kvh * g, q_pos = it.b * (K + 1) + it.mg * (R / g);
          // Chunks are filled as they free, before the item's Q slot is free
          // (an earlier item's last S), so the ring does not drain between
          // items; before the layer barrier only tiles that lie wholly in
          // the cache prefix (the block's keys are the previous layer's
          // output).
          if (!ready) {
            // Q is read once the layer barrier passes; bring it into L2 now
            for (int hb = 0; hb < SM::kBoxes; ++hb) tma_prefetch_3d(&set.Q[layer], hb * 64, q_head, q_pos);
          }
          bool ok = true, q_done = false;
          // a layer's first item: its prefix tiles go out once the previous
          // layer's last S has read its Q slot (earlier copies only slow the
          // previous layer, whose barrier this layer waits for)
          const uint32_t q_par = (item_ctr & 1) ^ 1;  // of the previous item's last S
          if (!ready) ok = mbar_wait(bQEmpty, q_par);
          for (int spin = 0; ok && !q_done; ++spin) {
            if (ready && mbar_test_wait(bIEmpty + 8 * (item_ctr & 1), ((item_ctr >> 1) & 1) ^ 1) &&
                mbar_test_wait(bQEmpty, q_par)) {
              // Q: R/g positions x g heads of kv head kvh, one box per 64-column half
              info[item_ctr & 1] = it;
              mbar_arrive(bIFull + 8 * (item_ctr & 1));
              mbar_expect_tx(bQFull, (uint32_t)R * D * 2);
              for (int hb = 0; hb < SM::kBoxes; ++hb)
                tma_load_3d(sQ + hb * 16384, &set.Q[layer], bQFull, hb * 64, q_head, q_pos);
              q_done = true;
              break;
            }
            while (vt < n_tiles) {
              // the chunk's last key lies before the block
              const int tt = next_is_k() ? kt : vt;
              if (!ready && it.key0 + min(2 * tt + 2, n_half) * kAttnTileKeys > it.kv) break;
              if (!mbar_test_wait(chunk_free(), chunk_parity())) break;
              fill_chunk();
            }
            if (!ready) {
              uint32_t v;
              asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar_cnt + (layer - 1)) : "memory");
              if (v >= n_ctas) {
                ready = true;
                continue;
              }
            }
            if (spin >= kMaxWaitIters) ok = false;
            else __nanosleep(32);
          }
          while (ok && vt < n_tiles) {
            ok = mbar_wait(chunk_free(), chunk_parity());
            if (ok) fill_chunk();
          }
          if (!ok) {
            raise_status(status, LIBRASPEC_ST_TIMEOUT);
            misc[0] = 1;
          }
        }
        ready = true;
        ++item_ctr;
        if (pos < hi) next_item();
        __syncwarp();
      }
    }
    // before leaving, wait (bounded) for this CTA's copies still in flight
    if (lane == 0) {
      for (uint32_t k = 0; k < (uint32_t)SM::kChunks && k < chunk_ctr; ++k) {
        const uint32_t i = chunk_ctr - 1 - k;
        mbar_wait(bFull + 8 * (i % SM::kChunks), (i / SM::kChunks) & 1);
      }
      if (item_ctr > 0) mbar_wait(bQFull, (item_ctr - 1) & 1);
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // ======================= MMA issue =======================
    if (lane == 0) {
      uint32_t item_ctr = 0, chunk_ctr = 0;
      uint32_t p_par = 0;  // bit s: parity of P steps of stream s
      bool ok = true;
      auto take = [&]() {  // the next chunk, once it is filled
        const uint32_t ch = chunk_ctr % SM::kChunks;
        ok = ok && mbar_wait(bFull + 8 * ch, (chunk_ctr / SM::kChunks) & 1);
        ++chunk_ctr;
        return ch;
      };
      bool none = false;  // the CTA has no item
      for (int layer = 0; layer < n_layers && ok && !none; ++layer) {
        for (int last = 0; !last && ok; ++item_ctr) {
          ok = mbar_wait(bIFull + 8 * (item_ctr & 1), (item_ctr >> 1) & 1);
          if (!ok) break;
          const ItemInfo it = info[item_ctr & 1];
          mbar_arrive(bIEmpty + 8 * (item_ctr & 1));
          last = it.last;
          if (last == 2) {
            none = true;
            break;
          }
          const int n_half = (it.key1 - it.key0 + kAttnTileKeys - 1) / kAttnTileKeys, n_tiles = (n_half + 1) >> 1;
          // Step j: tile j, stream j & 1. S of a step goes where P of the
          // stream's last step lies, so its PV is issued first.
          for (int j = 0; j < n_tiles + 2 && ok; ++j) {
            const int st = j & 1;
            const uint32_t ts = tmem + SM::kColS + st * 128;
            if (j >= 2) {  // O += P V of step j - 2
              const uint32_t ch = take();
              ok = ok && mbar_wait(bPFull + 8 * st, (p_par >> st) & 1u);
              p_par ^= 1u << st;
              if (j == 2) ok = ok && mbar_wait(bOFree, (item_ctr & 1) ^ 1);
              if (!ok) break;
              tc_fence_after();
              constexpr uint32_t idesc = mma_idesc(128, D, 1);
              const uint32_t va = desc_lo(sRing + ch * SM::kChunkBytes, 8192);
              const uint32_t d = tmem + SM::kColO + st * 128;
              mma_ts4<2048>(d, ts, va, idesc, j < 4 ? 0u : 1u);
              if (n_half - 2 * (j - 2) >= 2) mma_ts4<2048>(d, ts + 32, va + SM::kBoxes * 512, idesc, 1u);
              mma_commit(bPVDone + 8 * st);
              mma_commit(bEmpty + 8 * ch);
            }
            if (j < n_tiles) {  // S = Q K^T of step j: the group's rows x up to 128 keys
              const uint32_t ch = take();
              if (j == 0) ok = ok && mbar_wait(bQFull, item_ctr & 1);
              if (!ok) break;
              tc_fence_after();
              const uint32_t idesc = mma_idesc(128, n_half - 2 * j >= 2 ? 128 : 64, 0);
              const uint32_t qa = desc_lo(sQ, 16), ka = desc_lo(sRing + ch * SM::kChunkBytes, 16);
#pragma unroll
              for (int hb = 0; hb < SM::kBoxes; ++hb)
                mma_ss4<32, 32>(ts, qa + hb * 1024, ka + hb * 1024, idesc, hb != 0 ? 1u : 0u);
              mma_commit(bSFull + 8 * st);
              mma_commit(bEmpty + 8 * ch);
              if (j == n_tiles - 1) mma_commit(bQEmpty);
            }
          }
        }
      }
      if (!ok) {
        raise_status(status, LIBRASPEC_ST_TIMEOUT);
        misc[0] = 1;
      }
      // every MMA issued has completed before the tensor memory is released
      mma_commit(bDrain);
      mbar_wait(bDrain, 0);
    }
    __syncwarp();
  } else if (warp < kSoftmaxWarps) {
    // ======================= softmax warpgroups =======================
    const int st = warp >> 2, wq = warp & 3;       // stream; quarter of the tensor-memory lanes
    const int row = wq * 32 + lane;                // tensor-memory lane: the unit's row
    const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
    const uint32_t ts = tmem + lane_off + SM::kColS + st * 128;
    float2* stat = reinterpret_cast<float2*>(smem + SM::kStat);  // [stream][128]
    uint32_t item_ctr = 0, done0 = 0, done1 = 0;   // steps of streams 0 and 1 in the items before this one
    bool ok = true, none = false;  // none: the CTA has no item
    // A wait that fails leaves `ok` false; the item is then finished without
    // further waits, so that every thread still reaches every named barrier.
    auto wait = [&](uint32_t bar, uint32_t parity) { ok = ok && warp_wait(bar, parity); };
    for (int layer = 0; layer < n_layers; ++layer) {
      float* part_o = part_buf_o + (layer % kAttnPartBufs) * part_o_stride;
      float* part_ml = part_buf_ml + (layer % kAttnPartBufs) * part_ml_stride;
      if (layer > 0) {
        // layer's inputs are ready once every CTA is done with the previous layer
        if (tid == 0 && !wait_counter(bar_cnt + (layer - 1), n_ctas)) ok = false;
        if (softmax_any(!ok)) {
          ok = false;
          break;
        }
      }
      __nv_bfloat16* O = set.p[layer].O;
      float* lse = set.p[layer].lse;
      bool failed = false;  // (of a wait for an item)
      for (int last = none ? 1 : 0; !last;) {
        wait(bIFull + 8 * (item_ctr & 1), (item_ctr >> 1) & 1);
        if (softmax_any(!ok)) {
          failed = true;
          break;
        }
        const ItemInfo& it = info[item_ctr & 1];
        last = it.last;
        if (last == 2) {
          none = true;
          break;
        }
        const int n_half = (it.key1 - it.key0 + kAttnTileKeys - 1) / kAttnTileKeys, n_tiles = (n_half + 1) >> 1;
        const int steps0 = (n_tiles + 1) >> 1, steps1 = n_tiles >> 1;
        const int my_steps = st ? steps1 : steps0;
        const int rows = it.rows;
        const bool valid = row < rows;
        // a warp without valid rows only keeps the barrier counts in step
        const bool warp_live = wq * 32 < rows;
        const int rr = it.mg * R + row;  // row of the (sequence, kv head)
        const int t_row = rr / g;
        float m_run = -INFINITY, l_run = 0.f;
        // (a lane past the group's rows holds scores of whatever its Q row is: at 0 they ask for no raise)
        const float scale_row = valid ? scale_log2 : 0.f;
        {
          // Keys seen by this row: the cache prefix and the root (keys <= kv),
          // then chain: the block positions up to t_row (keys <= kv + t_row);
          // tree: the ancestors of node t_row and itself, bit j of its
          // visibility row <-> key kv + 1 + j.
          const int kv = it.kv, key1 = it.key1;
          const uint64_t* vrow =
              (tree_vis && valid) ? tree_vis + ((size_t)it.b * (K + 1) + t_row) * tree_words : nullptr;
          // tiles past this key need the mask; rows past the group compute on whatever their lanes hold, seen by no
          // other row and never stored
          const int mask_from = valid ? min(tree_vis ? kv : kv + t_row, key1 - 1) : 0x7fffffff;
          int kt0 = it.key0 + st * 128;
          for (int i = 0; i < my_steps; ++i, kt0 += 256) {
            const uint32_t n = (st ? done1 : done0) + i;
            wait(bSFull + 8 * st, n & 1);
            if (!warp_live) {
              __syncwarp();
              if (lane == 0) mbar_arrive(bPFull + 8 * st);
              continue;
            }
            tc_fence_after();
            const bool two = key1 - kt0 > 64;  // the tile's second 64 keys exist
            // (the whole warp masks or none of it: the loops below hold warp-wide tensor-memory instructions)
            const bool need_mask = __any_sync(0xffffffffu, kt0 + 127 > mask_from);
            float la[2] = {0.f, 0.f}, lb[2] = {0.f, 0.f};
            // The reference max of a row is the max of its first 32 keys; it
            // is raised, by a power of two, when a later key exceeds it by
            // more than 2^8 (rare): what was computed against the old one (l,
            // O, the tile's P so far) is scaled, P exactly.
            auto raise_to = [&](float cmax, int c0) {
              const bool raise = cmax > m_run + kRescaleLog2;
              const bool unset = m_run == -INFINITY;
              const float up = unset ? cmax : m_run + ceilf(cmax - m_run);
              const float f = !raise ? 1.f : unset ? 0.f : ex2_approx(m_run - up);
              m_run = raise ? up : m_run;
              l_run *= f;
              la[0] *= f;
              la[1] *= f;
              lb[0] *= f;
              lb[1] *= f;
              // the P read back here was stored by this thread, chunk by chunk; a load is ordered behind a store of the
              // same thread by the wait alone
              tmem_wait_st();
#pragma unroll 1
              for (int c = 0; c < c0 / 2; c += 16) {
                uint32_t q[16];
                tmem_ld16(ts + c, q);
                tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < 16; ++k) q[k] = pack_bf16(bf16_lo(q[k]) * f, bf16_hi(q[k]) * f);
                tmem_st16(ts + c, q);
              }
              if (i > 0) {
                // O holds the stream's earlier tiles of this item: its last PV has landed
                wait(bPVDone + 8 * st, (n - 1) & 1);
                tc_fence_after();
#pragma unroll 1
                for (int d0 = 0; d0 < D; d0 += 32) {
                  uint32_t o[32];
                  const uint32_t oa = tmem + lane_off + SM::kColO + st * 128 + d0;
                  tmem_ld32(oa, o);
                  tmem_wait_ld();
#pragma unroll
                  for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * f);
                  tmem_st32(oa, o);
                }
              }
              tmem_wait_st();
            };
            // keys c0 .. c0 + 31 of the tile, their scores in x: P of them in place of scores already read
            auto softmax_32 = [&](int c0, uint32_t (&x)[32]) {
              if (need_mask) {  // keys this row does not see count as -inf
                const int k0 = kt0 + c0;
                uint32_t bits = (uint32_t)(!vrow ? low_bits(kv + t_row + 1 - k0)
                                                 : low_bits(kv + 1 - k0) | bit_window(vrow, tree_words, k0 - kv - 1));
                bits &= (uint32_t)low_bits(key1 - k0);
                if (!valid) bits = ~0u;
#pragma unroll
                for (int c = 0; c < 32; ++c)
                  if (!((bits >> c) & 1u)) x[c] = __float_as_uint(-INFINITY);
              }
              float a = -INFINITY, b = -INFINITY;
#pragma unroll
              for (int c = 0; c < 32; c += 4) {
                a = fmaxf(fmaxf(a, __uint_as_float(x[c])), __uint_as_float(x[c + 1]));
                b = fmaxf(fmaxf(b, __uint_as_float(x[c + 2])), __uint_as_float(x[c + 3]));
              }
              const float cmax = fmaxf(a, b) * scale_row;
              if (i == 0 && c0 == 0) m_run = cmax;
              else if (__any_sync(0xffffffffu, cmax > m_run + kRescaleLog2)) raise_to(cmax, c0);
              const float neg_m = (m_run == -INFINITY) ? 0.f : -m_run;
              uint32_t pk[16];
#pragma unroll
              for (int c = 0; c < 32; c += 4) {
                float y0, y1, y2, y3;
                fma2(y0, y1, __uint_as_float(x[c]), __uint_as_float(x[c + 1]), scale_row, neg_m);
                fma2(y2, y3, __uint_as_float(x[c + 2]), __uint_as_float(x[c + 3]), scale_row, neg_m);
                y0 = ex2_approx(y0);
                y1 = ex2_approx(y1);
                y2 = ex2_approx(y2);
                y3 = ex2_approx(y3);
                add2(la[0], la[1], y0, y1);
                add2(lb[0], lb[1], y2, y3);
                pk[c >> 1] = pack_bf16(y0, y1);
                pk[(c >> 1) + 1] = pack_bf16(y2, y3);
              }
              tmem_st16(ts + c0 / 2, pk);
            };
            // (one rolled copy of the code: two, with the next 32 keys loaded ahead, were slower)
            const int n_cols = two ? 128 : 64;
#pragma unroll 1
            for (int c0 = 0; c0 < n_cols; c0 += 32) {
              uint32_t x[32];
              tmem_ld32(ts + c0, x);
              tmem_wait_ld();
              softmax_32(c0, x);
            }
            l_run += (la[0] + la[1]) + (lb[0] + lb[1]);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bPFull + 8 * st);
          }
        }
        // ---- epilogue: O of this item is complete once the last PVs have landed ----
        float f0 = 1.f, f1 = 0.f;  // factors of the streams' O
        const bool second = steps1 > 0;
        if (second) {  // the streams hold keys of the same rows: exchange (m, l)
          if (warp_live) stat[st * 128 + row] = make_float2(m_run, l_run);
          softmax_sync();
          if (warp_live) {
            const float2 a = stat[row], b = stat[128 + row];
            const float M = fmaxf(a.x, b.x);
            f0 = M == -INFINITY ? 0.f : ex2_approx(a.x - M);
            f1 = M == -INFINITY ? 0.f : ex2_approx(b.x - M);
            m_run = M;
            l_run = f0 * a.y + f1 * b.y;
          }
        }
        wait(bPVDone, (done0 + steps0 - 1) & 1);
        if (second) wait(bPVDone + 8, (done1 + steps1 - 1) & 1);
        tc_fence_after();
        // the warpgroups share out the columns; a single step leaves all to the first
        if (warp_live && (second || st == 0)) {
          const int hq = it.kvh * g + rr % g;
          const size_t prow = (size_t)it.slot * kAttnRows + row;
          const bool partial = it.partial;
          if (!partial) {
            const float inv = 1.f / l_run;
            f0 *= inv;
            f1 *= inv;
          }
          const int cb = second ? st * (D / 2) : 0, ce = second ? cb + D / 2 : D;
          __nv_bfloat16* orow = O + (((size_t)it.b * (K + 1) + t_row) * Hq + hq) * D;
          const uint32_t oa = tmem + lane_off + SM::kColO;
#pragma unroll 1
          for (int c0 = cb; c0 < ce; c0 += 32) {
            uint32_t o[32];
            tmem_ld32(oa + c0, o);
            if (second) {
              uint32_t o1[32];
              tmem_ld32(oa + 128 + c0, o1);
              tmem_wait_ld();
#pragma unroll
              for (int c = 0; c < 32; ++c)
                o[c] = __float_as_uint(fmaf(__uint_as_float(o1[c]), f1, __uint_as_float(o[c]) * f0));
            } else {
              tmem_wait_ld();
#pragma unroll
              for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * f0);
            }
            if (valid) {
              if (!partial) {
                uint4* dst = reinterpret_cast<uint4*>(orow + c0);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                  dst[i] = make_uint4(pack_bf16(__uint_as_float(o[8 * i]), __uint_as_float(o[8 * i + 1])),
                                      pack_bf16(__uint_as_float(o[8 * i + 2]), __uint_as_float(o[8 * i + 3])),
                                      pack_bf16(__uint_as_float(o[8 * i + 4]), __uint_as_float(o[8 * i + 5])),
                                      pack_bf16(__uint_as_float(o[8 * i + 6]), __uint_as_float(o[8 * i + 7])));
              } else {
                uint4* dst = reinterpret_cast<uint4*>(part_o + prow * D + c0);
#pragma unroll
                for (int i = 0; i < 8; ++i) dst[i] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
              }
            }
          }
          if (valid && st == 0) {
            if (partial) {
              *reinterpret_cast<float2*>(part_ml + prow * 2) = make_float2(m_run, l_run);
            } else if (lse) {
              lse[((size_t)it.b * (K + 1) + t_row) * Hq + hq] = (m_run + __log2f(l_run)) * kLn2;
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bOFree);
        if (it.partial && layer == n_layers - 1) {
          // The last layer's split groups need no grid barrier: each part is
          // counted in as written (the named barrier orders the warpgroups'
          // writes before the release).
          softmax_sync();
          if (tid == 0)
            asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(grp_cnt + 2 * it.grp), "r"(1u) : "memory");
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bIEmpty + 8 * (item_ctr & 1));  // `it` has been read
        done0 += steps0;
        done1 += steps1;
        ++item_ctr;
      }
      if (failed) {
        ok = false;
        break;
      }
      // This CTA is done with the layer's items. Once its grid barrier
      // passes, CTAs write layer + 1's partials into the buffer of layer - 2,
      // whose merge must be done first.
      if (layer >= kAttnPartBufs - 1 && tid == 0 && !(tasks_ready() && next_buf_free(layer))) ok = false;
      if (softmax_any(!ok || misc[0])) {
        ok = false;
        break;
      }
      if (tid == 0)
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar_cnt + layer), "r"(1u) : "memory");
    }
    if (!ok) {
      if (lane == 0) raise_status(status, LIBRASPEC_ST_TIMEOUT);
      misc[0] = 1;
    }
  }
  // ======================= merges =======================
  // The two merge warps come here at once and merge layer l's split groups
  // once every CTA has finished layer l (its grid barrier), beside the next
  // layers' items; the other warps come when their roles are done and help
  // with the last layer's. One copy of the code for all of them, outside the
  // roles: a second one in the softmax warps' path cost fetches of cold
  // instructions and their registers.
  __syncwarp();
  {
    bool ok = lane != 0 || tasks_ready();
    ok = __all_sync(0xffffffffu, ok);
    const int n_tasks = misc[1], merge_n = misc[3];
    // (with more parts than rows some CTAs have a share of no rows: their first merge warp still passes the groups'
    // counters, which the last of the np CTAs resets)
    const bool merging = warp == kMergeWarp ? n_tasks > 0 : merge_n > 0;
    for (int layer = warp >= kMergeWarp && merge_n > 0 ? 0 : n_layers - 1; layer < n_layers && ok && merging; ++layer) {
      if (layer < n_layers - 1) {
        ok = layer_done(layer);
      } else if (warp == kMergeWarp) {
        // the last layer: each split group once its np parts are counted in
        // (no grid barrier); the last CTA past a group's wait resets its
        // counters for the next launch
        if (lane == 0) {
          for (int ti = 0; ti < n_tasks && ok; ++ti) ok = wait_counter(grp_cnt + 2 * tasks[ti].grp, tasks[ti].np);
          if (ok) {
            misc[5] = 1;  // the other warps may start
            for (int ti = 0; ti < n_tasks; ++ti) {
              uint32_t* gc = grp_cnt + 2 * tasks[ti].grp;
              if (atomicAdd(gc + 1, 1u) == (uint32_t)tasks[ti].np - 1) {
                gc[0] = 0u;
                gc[1] = 0u;
              }
            }
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0) != 0 && !misc[0];
      } else {
        ok = last_groups_ready();
      }
      if (ok)
        merge_chunks<D>(layer, set, tasks, n_tasks, merge_n, merge_claimed, merge_done, K, Hq, Hkv, R,
                        part_buf_o, part_buf_ml, part_o_stride, part_ml_stride);
    }
    if (!ok && lane == 0 && !misc[0]) {
      raise_status(status, LIBRASPEC_ST_TIMEOUT);
      misc[0] = 1;
    }
    __syncwarp();
  }
  // every role is done with the tensor memory
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0 && !misc[0] && n_layers > 0) {
    // the last CTA out resets the barrier counters for the next launch (each
    // CTA has arrived at every layer's barrier by now)
    __threadfence();
    const uint32_t done = atomicAdd(exit_cnt, 1u);
    if (done == n_ctas - 1) {
      for (int l = 0; l < n_layers; ++l) bar_cnt[l] = 0u;
      *exit_cnt = 0u;
      __threadfence();
    }
  }
  if (warp == kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmemCols) : "memory");
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
int num_sms_current();

// Q [B*(K+1), Hq, D] as 3-D; box = 64 columns x g heads x R/g positions (one
// row group of one kv head), 128-byte swizzle.
static bool make_q_map(CUtensorMap* map, const void* base, int D, int Hq, int BT, int g, int R) {
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)Hq, (cuuint64_t)BT};
  cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)Hq * D * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)g, (cuuint32_t)(R / g)};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

static bool make_kv_map(CUtensorMap* map, const void* base, int D, int S_cap, int BH) {
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)S_cap, (cuuint64_t)BH};
  cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)S_cap * D * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)kAttnTileKeys, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Smallest tile range per CTA (1: as many CTAs as there are tiles; at 2, half
// the CTAs work on 3 sequences of 900 keys and 32 layers take 319 us instead
// of 235); the LIBRASPEC_ATTN_MIN_TILES environment variable overrides the
// default, read once per process.
static int attn_min_tiles() {
  static int t = [] {
    int v = 1;
    if (const char* e = getenv("LIBRASPEC_ATTN_MIN_TILES")) {
      int a = 0;
      if (sscanf(e, "%d", &a) == 1 && a >= 1 && a <= 4096) v = a;
    }
    return v;
  }();
  return t;
}

// Tile-equivalents an item costs at most in the split by cost (see find_tile);
// the LIBRASPEC_ATTN_ITEM_TILES environment variable overrides the default,
// read once per process. 0 / 4 / 6 / 8 / 12: 16 paged sequences, 2 layers 110 /
// 102 / 102 / 102 / 102 us, ragged B = 64 312 / 296 / 299 / 298 / 301.
static int attn_item_tiles() {
  static int t = [] {
    int v = 4;
    if (const char* e = getenv("LIBRASPEC_ATTN_ITEM_TILES")) {
      int a = 0;
      if (sscanf(e, "%d", &a) == 1 && a >= 0 && a <= 64) v = a;
    }
    return v;
  }();
  return t;
}

// Ancestor sets of a draft tree, one CTA per sequence, by pointer jumping:
// after round r, m[t] holds the nodes on the path from t up to (not
// including) up[t], the ancestor at distance 2^r (the root absorbs: m[0] =
// 0, up[0] = 0); rounds stop once every up[] is the root (depth <= 2^r).
// vis[b, t] = m[t] as `words` 64-bit words, bit j <-> block position j + 1;
// rows t > L_b get 0. A parent outside [0, t) raises LIBRASPEC_ST_BAD_TREE
// and is read as the root. Each round reads all (node, word) pairs into
// registers before any is written.
constexpr int kTreeThreads = 256;
constexpr int kTreeWords = (LIBRASPEC_MAX_TREE_NODES + 63) / 64;
constexpr int kTreePer = ((LIBRASPEC_MAX_TREE_NODES + 1) * kTreeWords + kTreeThreads - 1) / kTreeThreads;

__global__ void __launch_bounds__(kTreeThreads) tree_vis_kernel(const int32_t* __restrict__ parent,
                                                                 const int32_t* __restrict__ Ls, int K, int words,
                                                                 uint64_t* __restrict__ vis,
                                                                 int* __restrict__ status) {
  __shared__ int up[LIBRASPEC_MAX_TREE_NODES + 1];
  __shared__ uint64_t m[(LIBRASPEC_MAX_TREE_NODES + 1) * kTreeWords];
  const int b = blockIdx.x, tid = threadIdx.x;
  int Lb = Ls[b];
  if (Lb < 0 || Lb > K) Lb = 0;  // the attention kernel reports the bad length
  const int pairs = (K + 1) * words;
  for (int t = tid; t <= K; t += kTreeThreads) {
    int p = 0;
    if (t >= 1 && t <= Lb) {
      p = parent[(size_t)b * (K + 1) + t];
      if (p < 0 || p >= t) {
        raise_status(status, LIBRASPEC_ST_BAD_TREE);
        p = 0;
      }
    }
    up[t] = p;
  }
  for (int i = tid; i < pairs; i += kTreeThreads) {
    const int t = i / words, w = i % words;
    m[i] = (t >= 1 && t <= Lb && (t - 1) / 64 == w) ? 1ull << ((t - 1) % 64) : 0ull;
  }
  __syncthreads();
  for (int r = 0; r < 16; ++r) {  // depth <= 512 needs at most 10 rounds
    uint64_t nm[kTreePer];
    int nu[kTreePer];
    bool more = false;
#pragma unroll
    for (int k = 0; k < kTreePer; ++k) {
      const int i = tid + k * kTreeThreads;
      if (i < pairs) {
        const int t = i / words, w = i % words;
        const int u = up[t];
        nm[k] = m[i] | m[u * words + w];
        nu[k] = up[u];
        more |= nu[k] != 0;
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kTreePer; ++k) {
      const int i = tid + k * kTreeThreads;
      if (i < pairs) {
        m[i] = nm[k];
        if (i % words == 0) up[i / words] = nu[k];
      }
    }
    if (!__syncthreads_or(more)) break;
  }
  for (int i = tid; i < pairs; i += kTreeThreads) vis[(size_t)b * pairs + i] = m[i];
}

inline int tree_words(int K) { return K <= 64 ? 1 : (K + 63) / 64; }

// parent != nullptr: fill the tree visibility masks of the workspace first.
static cudaError_t tree_vis(const int32_t* parent, const int32_t* L, int B, int K, char* ws, const WsLayout& lay,
                            cudaStream_t stream, const uint64_t** out) {
  *out = nullptr;
  if (!parent) return cudaSuccess;
  auto* vis = reinterpret_cast<uint64_t*>(ws + lay.tree_vis);
  tree_vis_kernel<<<B, kTreeThreads, 0, stream>>>(parent, L, K, tree_words(K), vis,
                                                  reinterpret_cast<int*>(ws + lay.status));
  *out = vis;
  return cudaGetLastError();
}

// Paged caches (block_table != nullptr): Kc / Vc are page pools of n_pages
// pages of page_size keys and S_cap = max_pages * page_size.
// Tiles per CTA whose page ids are cached in shared memory (at most cap);
// the LIBRASPEC_ATTN_PAGE_CACHE environment variable lowers it (0: read the
// block table tile by tile). Read once per process.
static int attn_page_cache(int cap) {
  static int v = [] {
    int a = -1;
    if (const char* e = getenv("LIBRASPEC_ATTN_PAGE_CACHE")) {
      if (sscanf(e, "%d", &a) != 1 || a < 0) a = -1;
    }
    return a;
  }();
  return v < 0 || v > cap ? cap : v;
}

// The tensor maps of a launch cost the host about a microsecond each (3 per
// layer); a caller that runs round after round on the same buffers (the
// staged round) gets them from this per-thread cache of the last launch of
// each chunk of layers, keyed by every pointer and shape they encode.
struct LayerSetCache {
  bool valid = false;
  int rows = 0, planes = 0, Hq = 0, BT = 0, g = 0, R = 0;
  const void* Kp[kMaxLayers];
  const void* Vp[kMaxLayers];
  LayerSet set;
};
constexpr int kCachedChunks = 4;

template <int D, bool PAGED>
static cudaError_t launch_layers_t(const uint16_t* const* Q, const uint16_t* const* Kc, const uint16_t* const* Vc,
                                   int n_layers, const int32_t* kv_len, const int32_t* L, const uint64_t* tree_vis,
                                   const int32_t* block_table,
                                   int max_pages, int page_size, int n_pages, int B, int K, int Hq, int Hkv, int S_cap,
                                   float scale, uint16_t* const* O, float* const* lse, char* ws, const WsLayout& lay,
                                   cudaStream_t stream) {
  using SM = AttnSmem<D>;
  constexpr int kSmem = PAGED ? SM::kAllocPaged : SM::kAlloc;
  static bool configured = false;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(verify_attn_kernel<D, PAGED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kSmem);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  int grid = num_sms_current();  // one CTA per SM (it holds all 512 tensor-memory columns)
  if (grid > kAttnMaxCtas) grid = kAttnMaxCtas;
  auto kern = verify_attn_kernel<D, PAGED>;
  const int g = Hq / Hkv;
  const int R = g * (kAttnRows / g);
  // layers beyond kMaxLayers go in further launches of the same kernel
  for (int l0 = 0; l0 < n_layers; l0 += kMaxLayers) {
    const int n = n_layers - l0 < kMaxLayers ? n_layers - l0 : kMaxLayers;
    // dense: [B*Hkv, S_cap, D]; paged: [n_pages*Hkv, page_size, D]
    const int rows = PAGED ? page_size : S_cap;
    const int planes = PAGED ? n_pages * Hkv : B * Hkv;
    const int BT = B * (K + 1);
    static thread_local std::unique_ptr<LayerSetCache[]> caches;
    const int ci = l0 / kMaxLayers;
    LayerSetCache* c = nullptr;
    if (ci < kCachedChunks) {
      if (!caches) caches.reset(new (std::nothrow) LayerSetCache[kCachedChunks]);
      if (caches) c = &caches[ci];
    }
    bool hit = c && c->valid && c->set.n == n && c->rows == rows && c->planes == planes && c->Hq == Hq &&
               c->BT == BT && c->g == g && c->R == R;
    for (int i = 0; i < n && hit; ++i) {
      const int l = l0 + i;
      hit = c->Kp[i] == Kc[l] && c->Vp[i] == Vc[l] && c->set.p[i].Q == reinterpret_cast<const __nv_bfloat16*>(Q[l]) &&
            c->set.p[i].O == reinterpret_cast<__nv_bfloat16*>(O[l]) && c->set.p[i].lse == (lse ? lse[l] : nullptr);
    }
    LayerSet local;
    LayerSet& set = c ? c->set : local;  // ~26 KB: built on the host, copied into the launch parameters
    if (!hit) {
      if (c) c->valid = false;
      set.n = n;
      for (int i = 0; i < n; ++i) {
        const int l = l0 + i;
        if (!make_kv_map(&set.K[i], Kc[l], D, rows, planes) || !make_kv_map(&set.V[i], Vc[l], D, rows, planes) ||
            !make_q_map(&set.Q[i], Q[l], D, Hq, BT, g, R))
          return cudaErrorInvalidValue;
        set.p[i].Q = reinterpret_cast<const __nv_bfloat16*>(Q[l]);
        set.p[i].O = reinterpret_cast<__nv_bfloat16*>(O[l]);
        set.p[i].lse = lse ? lse[l] : nullptr;
        if (c) {
          c->Kp[i] = Kc[l];
          c->Vp[i] = Vc[l];
        }
      }
      if (c) {
        c->rows = rows;
        c->planes = planes;
        c->Hq = Hq;
        c->BT = BT;
        c->g = g;
        c->R = R;
        c->valid = true;
      }
    }
    // one partial buffer's share, kept 256-byte aligned
    const size_t o_part = ((lay.attn_ml - lay.attn_o) / kAttnPartBufs) & ~size_t(255);
    const size_t ml_part = ((lay.attn_cnt - lay.attn_ml) / kAttnPartBufs) & ~size_t(255);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kAttnThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = stream;
    // cooperative: every CTA is resident at once, which the layer barriers rely on
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(
        &cfg, kern, set, kv_len, L, tree_vis, tree_words(K), block_table, max_pages, page_size, n_pages,
        attn_page_cache(SM::kPageCap), B, K, Hq, Hkv, S_cap, scale * kLog2e, attn_min_tiles(), attn_item_tiles(),
        reinterpret_cast<float*>(ws + lay.attn_o), reinterpret_cast<float*>(ws + lay.attn_ml), o_part / sizeof(float),
        ml_part / sizeof(float), reinterpret_cast<uint32_t*>(ws + lay.attn_cnt),
        reinterpret_cast<uint32_t*>(ws + lay.attn_grp), reinterpret_cast<int*>(ws + lay.status));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// parent (optional, [B, K+1]): the block is a draft tree (nullptr: the chain).
cudaError_t launch_verify_attn_layers(const uint16_t* const* Q, const uint16_t* const* Kc,
                                      const uint16_t* const* Vc, int n_layers, const int32_t* parent,
                                      const int32_t* kv_len, const int32_t* L, int B, int K, int Hq, int Hkv, int D,
                                      int S_cap, float scale, uint16_t* const* O, float* const* lse, char* ws,
                                      const WsLayout& lay, cudaStream_t stream) {
  if (B == 0 || n_layers == 0) return cudaSuccess;
  const uint64_t* vis = nullptr;
  cudaError_t e = tree_vis(parent, L, B, K, ws, lay, stream, &vis);
  if (e != cudaSuccess) return e;
  auto* launch = D == 128 ? launch_layers_t<128, false> : launch_layers_t<64, false>;
  return launch(Q, Kc, Vc, n_layers, kv_len, L, vis, nullptr, 0, 0, 0, B, K, Hq, Hkv, S_cap, scale, O, lse, ws, lay,
                stream);
}

cudaError_t launch_verify_attn_paged_layers(const uint16_t* const* Q, const uint16_t* const* Kp,
                                            const uint16_t* const* Vp, int n_layers, const int32_t* parent,
                                            const int32_t* block_table, int max_pages, int page_size, int n_pages,
                                            const int32_t* kv_len, const int32_t* L, int B, int K, int Hq, int Hkv,
                                            int D, float scale, uint16_t* const* O, float* const* lse, char* ws,
                                            const WsLayout& lay, cudaStream_t stream) {
  if (B == 0 || n_layers == 0) return cudaSuccess;
  const int S_cap = max_pages * page_size;
  const uint64_t* vis = nullptr;
  cudaError_t e = tree_vis(parent, L, B, K, ws, lay, stream, &vis);
  if (e != cudaSuccess) return e;
  auto* launch = D == 128 ? launch_layers_t<128, true> : launch_layers_t<64, true>;
  return launch(Q, Kp, Vp, n_layers, kv_len, L, vis, block_table, max_pages, page_size, n_pages, B, K, Hq, Hkv, S_cap,
                scale, O, lse, ws, lay, stream);
}

cudaError_t launch_verify_attn(const uint16_t* Q, const uint16_t* Kc, const uint16_t* Vc, const int32_t* kv_len,
                               const int32_t* L, int B, int K, int Hq, int Hkv, int D, int S_cap, float scale,
                               uint16_t* O, float* lse, char* ws, const WsLayout& lay, cudaStream_t stream) {
  float* lse_arr[1] = {lse};
  return launch_verify_attn_layers(&Q, &Kc, &Vc, 1, nullptr, kv_len, L, B, K, Hq, Hkv, D, S_cap, scale, &O,
                                   lse ? lse_arr : nullptr, ws, lay, stream);
}

}  // namespace libraspec
