// The LM head with the confidence / acceptance row statistics in its
// epilogue: logits x = H W^T (H [M, Dm] hidden states, W [V, Dm] the head,
// bf16) are accumulated by the 5th-generation tensor cores in tensor memory
// and reduced there to per-row (max, sum of exp, argmax, logit of one token)
// partials, so the logits never reach HBM; a second kernel merges each row's
// partials (Assumption 1's confidence q = softmax(x / T)[token], and the max /
// argmax / Z of the acceptance rows, Sec. 3.1).
//
// Work: CTA pairs (cta_group::2), one pair per two SMs. The vocabulary lies
// on the MMA's M side (256 head rows over the pair, 128 per CTA) and the rows
// of H on its N side (up to 256, split between the two CTAs), so a k-slab of
// 64 brings 16 KB of W and N x 64 bytes of H into each CTA. At N = 256 that
// is 64 bytes per cycle and SM at the tensor peak, which L2 sustains (2112 rows
// over V = 128256, Dm = 4096: 1160 us in 20 calls, 1.91 PFLOP/s; 1335 to 1385
// over seconds of calls, at the power limit); single-CTA tiles of 128 x 128
// need twice the bytes and were bound by them (1920 us over seconds). The time
// of a tile follows its operand bytes, 256 + N (N = 64: 96 us per row tile
// of that head, 128: 103, 192: 119, 256: 141), so rows are cut into as few
// tiles as 256 allows, of sizes that differ by 32 at most.
//  * Several row tiles: items (vocabulary tile, row tile) with the row tile
//    innermost, item i to pair i mod pairs: the pairs at work share the same
//    few tiles of W through L2. One partial per (row, 128 vocabulary columns).
//  * One row tile (M <= 256, decode: bound by the head's bytes): each pair
//    walks its own contiguous V / pairs columns, whose last tile is cut short,
//    so no pair streams more than its share (whole tiles of 256 leave 6.6
//    tiles per pair, a loss of 6%); its rows' statistics stay in registers
//    from tile to tile, the sum as two floats, and leave one partial per
//    (row, CTA).
//
// Roles (192 threads): warp 4 streams W and H k-slabs (128-byte swizzle) by
// TMA into a ring of stages, each CTA its half, counted on the leader's
// barrier; warp 5 of the leader issues tcgen05.mma into one of two
// accumulators (lane = head column, column = row of H); warps 0-3 turn 32 x 32
// blocks of an accumulator through shared memory, so that a thread holds one
// row's 32 logits, reduce them, and combine the four warps' shares (a wait
// that runs out is the verdict of all four: they meet at named barriers). Rows past
// M and columns past V come from the TMA's zero fill (or are never loaded)
// and are left out of the statistics.
#include <cmath>
#include <cstdio>

#include "tc.cuh"

namespace libraspec {

constexpr int kLmBK = 64, kLmMaxStages = 12;
constexpr int kLmEpiWarps = 4, kLmProducer = 4, kLmMma = 5, kLmThreads = 6 * 32;
constexpr int kLmHalf = 128;                           // head rows per CTA and tile
constexpr int kLmTile = 2 * kLmHalf;                   // head rows per tile
constexpr int kLmRows = 256;                           // rows of H per row tile (at most)
constexpr int kLmSub = 2;                              // k-slabs per stage (1 if Dm / 64 is odd)
constexpr uint32_t kLmATile = kLmHalf * kLmBK * 2;     // 16 KB
constexpr int kLmBarBytes = (2 * kLmMaxStages + 5) * 8 + 16;  // barriers and the tensor-memory slot
constexpr int kLmTurn = kLmEpiWarps * 32 * 33 * 4;     // a padded 32 x 32 block per epilogue warp
constexpr int kLmShares = kLmEpiWarps * kLmRows;       // the warps' (max, sum, argmax) per row
// shared memory besides the ring (with log2(e)/T and the token of each row of the item, and the table of powers)
constexpr int kLmFixed = 1024 + 1024 + kLmTurn + 3 * kLmShares * 4 + 2 * kLmRows * 4 + 32 * 8;
constexpr int kLmSmemMax = 227 * 1024;
static_assert(kLmBarBytes <= 1024, "barriers before the ring");

struct LmPartial {
  float m, zh, zl;  // max of the logits, sum of 2^((x - m) c) as two floats
  int arg;          // first column of the max
};

// 2^(j / 32) as a sum of two floats.
struct LmExpTable {
  float2 t[32];
};

// (m - mx) c as a sum of two floats, its error at most 2^-46 of it.
__device__ __forceinline__ void lm_exponent(float m, float mx, float c, float& xh, float& xl) {
  const float d = __fsub_rn(m, mx), b = __fsub_rn(d, m);
  const float dl = __fsub_rn(__fsub_rn(m, __fsub_rn(d, b)), __fadd_rn(mx, b));  // the difference's rounding error
  xh = __fmul_rn(d, c);
  xl = __fmaf_rn(dl, c, __fmaf_rn(d, c, -xh));
}

// (h + l) 2^n = 2^(xh + xl) for xh in [-1000, 0] (below, h = l = 0), within 2^-39 of it, by Tang's table-driven method
// (ACM Trans. Math. Softw. 15, 1989): the argument is cut at the nearest multiple of 1/32, whose power comes from the
// table, and the rest g = f ln 2, |g| < 0.011, goes through the Taylor series of e^g, whose first three terms are
// carried in two floats.
__device__ __forceinline__ void lm_exp2(float xh, float xl, const float2* table, float& h, float& l, int& n) {
  if (xh < -1000.f) {
    h = l = 0.f;
    n = 0;
    return;
  }
  constexpr float kLn2 = 0x1.62e43p-1f, kLn2Lo = -0x1.05c61p-29f;  // ln 2 to 48 bits
  const float kf = rintf(xh * 32.f);
  const int k = (int)kf;
  const float f0 = __fsub_rn(xh, kf * 0.03125f);  // exact
  const float f = __fadd_rn(f0, xl), fb = __fsub_rn(f, f0);
  const float fl = __fadd_rn(__fsub_rn(f0, __fsub_rn(f, fb)), __fsub_rn(xl, fb));
  const float g = __fmul_rn(f, kLn2);
  const float gl = __fadd_rn(__fmaf_rn(f, kLn2, -g), __fmaf_rn(f, kLn2Lo, __fmul_rn(fl, kLn2)));
  const float q = __fmul_rn(g, g);  // g^2 = q + ql
  const float ql = __fmaf_rn(2.f * g, gl, __fmaf_rn(g, g, -q));
  const float rest = __fmul_rn(__fmul_rn(q, g), __fmaf_rn(__fmaf_rn(g, 1.f / 120.f, 1.f / 24.f), g, 1.f / 6.f));
  const float a = __fadd_rn(1.f, g), al = __fsub_rn(g, __fsub_rn(a, 1.f));
  const float e = __fadd_rn(a, 0.5f * q), el0 = __fsub_rn(0.5f * q, __fsub_rn(e, a));
  const float el = __fadd_rn(__fadd_rn(al, el0), __fadd_rn(__fmaf_rn(0.5f, ql, gl), rest));
  const float2 t = table[k & 31];
  h = __fmul_rn(e, t.x);
  l = __fadd_rn(__fmaf_rn(e, t.x, -h), __fmaf_rn(e, t.y, __fmul_rn(el, t.x)));
  n = k >> 5;
}

// (zh + zl) += t + tl, |t| >= |tl|
__device__ __forceinline__ void two_add(float& zh, float& zl, float t, float tl) {
  const float sum = __fadd_rn(zh, t), b = __fsub_rn(sum, zh);
  zl = __fadd_rn(zl, __fadd_rn(__fadd_rn(__fsub_rn(zh, __fsub_rn(sum, b)), __fsub_rn(t, b)), tl));
  zh = sum;
}

// (zh + zl) += (vh + vl) 2^((m - mx) c), in two floats; a sum whose maximum is -inf is 0, or NaN.
__device__ __forceinline__ void lm_add(float& zh, float& zl, float vh, float vl, float m, float mx, float c,
                                       const float2* table) {
  if (!(m > -INFINITY)) {
    zh += vh;
    return;
  }
  float xh, xl, h, l;
  int e;
  lm_exponent(m, mx, c, xh, xl);
  lm_exp2(xh, xl, table, h, l, e);
  // (below 2^-126 nothing: the sum has a term of at least 1)
  const float s = e < -126 ? 0.f : __int_as_float((e + 127) << 23);
  const float z = vh * s, t = __fmul_rn(h, z);
  two_add(zh, zl, t, __fmaf_rn(l, z, __fmaf_rn(h, vl * s, __fmaf_rn(h, z, -t))));
}

// How the work is cut. The vocabulary: ranges of `range` columns, each in
// `tiles` tiles of which the last gives each CTA `tail` head rows (a multiple
// of 8), the others 128. The rows of H: row_tiles tiles, the first n_big of
// `big` rows (a multiple of 32, the MMA's N), the others of 32 fewer.
struct LmCut {
  int range, tiles, tail;
  int row_tiles, n_big, big;
};

constexpr int kEpiBar = 1;  // named barrier of the epilogue warps
__device__ __forceinline__ void epi_sync() {
  asm volatile("bar.sync %0, %1;" ::"n"(kEpiBar), "n"(kLmEpiWarps * 32) : "memory");
}

// One item of a pair: head rows [v0, v0 + rows) of this CTA, rows [h0, h0 + nrow) of H, the partial's slot.
struct LmItem {
  int v0, rows, h0, nrow, slot;
};

__device__ __forceinline__ LmItem lm_item(int it, int pair, int pairs, int rank, const LmCut& cut) {
  LmItem x;
  if (cut.row_tiles == 1) {  // tile `it` of the pair's own range
    x.rows = it == cut.tiles - 1 ? cut.tail : kLmHalf;
    x.v0 = pair * cut.range + it * kLmTile + rank * x.rows;
    x.h0 = 0;
    x.nrow = cut.big;
    x.slot = 2 * pair + rank;
  } else {
    const int i = pair + it * pairs, v = i / cut.row_tiles, n = i - v * cut.row_tiles;
    x.rows = kLmHalf;
    x.v0 = v * kLmTile + rank * kLmHalf;
    x.h0 = n * cut.big - 32 * max(n - cut.n_big, 0);
    x.nrow = n < cut.n_big ? cut.big : cut.big - 32;
    x.slot = 2 * v + rank;
  }
  return x;
}

// mapH / mapHs: boxes of cut.big / 2 rows / 16 fewer; mapW / mapWt: boxes of 128 / cut.tail head rows.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kLmThreads, 1) lm_head_stats_kernel(
    const __grid_constant__ CUtensorMap mapH, const __grid_constant__ CUtensorMap mapHs,
    const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapWt,
    const float* __restrict__ temperature, int rows_per_seq, const int32_t* __restrict__ tokens, int M, int V, int Dm,
    LmCut cut, int stages, int sub, int n_part, const __grid_constant__ LmExpTable exp_table,
    LmPartial* __restrict__ part, float* __restrict__ token_logit, int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // a stage holds `sub` consecutive k-slabs (W slab, then H slab), so every row is read `sub` * 128 contiguous
  // bytes at a time
  const uint32_t slab_bytes = kLmATile + (uint32_t)cut.big * kLmBK;
  const uint32_t stage_bytes = sub * slab_bytes;
  const uint32_t sbase = smem_u32(smem) + 1024;
  const uint32_t bFull = smem_u32(smem), bEmpty = bFull + 8 * kLmMaxStages;
  const uint32_t bAccFull = bEmpty + 8 * kLmMaxStages, bAccEmpty = bAccFull + 16, bDrain = bAccEmpty + 16;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + (2 * kLmMaxStages + 5) * 8);
  float* turn = reinterpret_cast<float*>(smem + 1024 + stages * stage_bytes);
  float* sh_m = turn + kLmEpiWarps * 32 * 33;
  float* sh_z = sh_m + kLmShares;
  int* sh_arg = reinterpret_cast<int*>(sh_z + kLmShares);
  float* sh_c = reinterpret_cast<float*>(sh_arg + kLmShares);
  int* sh_tok = reinterpret_cast<int*>(sh_c + kLmRows);
  float2* table = reinterpret_cast<float2*>(sh_tok + kLmRows);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  // items of this pair, stages per item
  const int n_items = cut.row_tiles == 1 ? cut.tiles : (cut.row_tiles * cut.tiles - pair + pairs - 1) / pairs;
  const int nk = Dm / kLmBK / sub;
  auto item_at = [&](int it) { return lm_item(it, pair, pairs, (int)rank, cut); };

  if (threadIdx.x < 32) table[threadIdx.x] = exp_table.t[threadIdx.x];
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(bFull + 8 * s, 1);   // (the leader's) its expect_tx; both CTAs' bytes as transactions
      mbar_init(bEmpty + 8 * s, 1);  // the leader's commit
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(bAccFull + 8 * a, 1);
      mbar_init(bAccEmpty + 8 * a, 2 * kLmEpiWarps);  // (the leader's) both CTAs' epilogue warps
    }
    mbar_init(bDrain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kLmMma) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(const_cast<uint32_t*>(tmem_slot))),
                 "n"(2 * kLmRows)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers are initialised
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;

  if (warp == kLmProducer) {
    if (lane == 0) {
      // One row tile: the head passes through L2 once, ahead of H and the code (64 rows over V = 32896, Dm = 2048:
      // 39.8 -> 34.1 us). Several: its tiles are read again by the other row tiles, so they keep the usual priority
      // (2112 rows, over seconds of calls: 1277 us, evict first 1597).
      const uint64_t policy = cut.row_tiles == 1 ? evict_first_policy() : evict_normal_policy();
      const uint64_t keep = cut.row_tiles == 1 ? evict_last_policy() : evict_normal_policy();
      uint32_t s = 0, ph = 0;
      for (int it = 0; it < n_items && ok; ++it) {
        const LmItem x = item_at(it);
        const CUtensorMap* mh = x.nrow < cut.big ? &mapHs : &mapH;
        const CUtensorMap* mw = x.rows < kLmHalf ? &mapWt : &mapW;
        const int hrow = x.h0 + (int)rank * (x.nrow >> 1);
        const uint32_t bytes = (uint32_t)(x.rows * 128 + x.nrow * kLmBK) * sub;  // this CTA's of a stage
        for (int k = 0; k < nk; ++k) {
          if (!(ok = mbar_wait(bEmpty + 8 * s, ph ^ 1))) break;
          const uint32_t a = sbase + s * stage_bytes;
          const uint32_t bar = map_rank(bFull + 8 * s, 0);
          if (rank == 0) mbar_expect_tx(bFull + 8 * s, 2 * bytes);
          for (int j = 0; j < sub; ++j) {
            const int kc = (k * sub + j) * kLmBK;
            tma_load_2d_pair(a + j * slab_bytes, mw, bar, kc, x.v0, policy);
            tma_load_2d_pair(a + j * slab_bytes + kLmATile, mh, bar, kc, hrow, keep);
          }
          if (++s == (uint32_t)stages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok) raise_status(status, LIBRASPEC_ST_TIMEOUT);
    }
    __syncwarp();
  } else if (warp == kLmMma) {
    if (lane == 0) {
      if (rank == 0) {
        uint32_t s = 0, ph = 0;
        for (int it = 0; it < n_items && ok; ++it) {
          const uint32_t ab = it & 1, aph = (it >> 1) & 1;
          if (!(ok = mbar_wait(bAccEmpty + 8 * ab, aph ^ 1))) break;
          tc_fence_after();
          const uint32_t idesc = mma_idesc(kLmTile, item_at(it).nrow, 0);
          const uint32_t d = tmem + ab * kLmRows;
          for (int k = 0; k < nk; ++k) {
            if (!(ok = mbar_wait(bFull + 8 * s, ph))) break;
            tc_fence_after();
            for (int j = 0; j < sub; ++j) {
              const uint32_t a = sbase + s * stage_bytes + j * slab_bytes;
#pragma unroll
              for (int kk = 0; kk < kLmBK / 16; ++kk)
                mma_ss_pair(d, smem_desc(a + kk * 32, 16, 1024), smem_desc(a + kLmATile + kk * 32, 16, 1024), idesc,
                            (k | j | kk) != 0 ? 1u : 0u);
            }
            mma_commit_pair(bEmpty + 8 * s);  // the stage is free, in both CTAs, once these MMAs have read it
            if (++s == (uint32_t)stages) {
              s = 0;
              ph ^= 1;
            }
          }
          if (ok) mma_commit_pair(bAccFull + 8 * ab);
        }
        if (!ok) raise_status(status, LIBRASPEC_ST_TIMEOUT);
        mma_commit_pair(bDrain);
      } else {  // item by item, so that each bounded wait covers one item
        for (int it = 0; it < n_items && ok; ++it) ok = mbar_wait(bAccFull + 8 * (it & 1), (it >> 1) & 1);
      }
      // every MMA has completed, and its signals have landed in both CTAs, before the tensor memory is released
      if (!mbar_wait(bDrain, 0)) raise_status(status, LIBRASPEC_ST_TIMEOUT);
    }
    __syncwarp();
  } else {
    // ===== epilogue: accumulator lane = head row v0 + warp * 32 + lane, column = row of H =====
    const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
    float* tw = turn + warp * 32 * 33;
    // one row tile: the statistics so far of rows threadIdx.x and threadIdx.x + 128
    float run_m[2] = {-INFINITY, -INFINITY}, run_zh[2] = {0.f, 0.f}, run_zl[2] = {0.f, 0.f};
    int run_arg[2] = {0x7fffffff, 0x7fffffff};
    for (int it = 0; it < n_items; ++it) {
      const LmItem x = item_at(it);
      const uint32_t ab = it & 1, aph = (it >> 1) & 1;
      const int vw = x.v0 + warp * 32;
      int nvalid = min(min(32, x.rows - warp * 32), V - vw);
      if (cut.row_tiles == 1) nvalid = min(nvalid, (pair + 1) * cut.range - vw);  // the next range's columns
      // log2(e) / T and the token of the item's rows, read while its MMAs run (a load from global memory takes
      // thousands of cycles beside the stream of the head: read block by block below, 128 rows over V = 32896, Dm =
      // 2048 took 70 us)
      if (it == 0 || cut.row_tiles > 1) {
        for (int j = threadIdx.x; j < x.nrow; j += kLmEpiWarps * 32) {
          const int grow = min(x.h0 + j, M - 1);
          const float T = temperature ? temperature[grow / rows_per_seq] : 1.f;
          sh_c[j] = log2e_over(T > 0.f ? T : 1.f);
          sh_tok[j] = tokens && x.h0 + j < M ? tokens[grow] : -1;
        }
        epi_sync();
      }
      // (one verdict of the four warps: they meet at the barriers below)
      if (!(ok = group_wait<kEpiBar, kLmEpiWarps * 32>(bAccFull + 8 * ab, aph))) break;
      tc_fence_after();
#pragma unroll 1
      for (int ch = 0; ch < x.nrow / 32; ++ch) {
        const int grow = x.h0 + ch * 32 + lane;  // this thread's row of H
        const int tok = sh_tok[ch * 32 + lane];
        const float c = sh_c[ch * 32 + lane];
        uint32_t r[32];
        tmem_ld32(tmem + lane_off + ab * kLmRows + ch * 32, r);
        tmem_wait_ld();
        __syncwarp();  // the last block has been read
#pragma unroll
        for (int i = 0; i < 32; ++i) tw[lane * 33 + i] = __uint_as_float(r[i]);
        __syncwarp();
        float y[32];
        float cm = -INFINITY;
        int ca = 0x7fffffff;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          y[i] = tw[i * 33 + lane];
          if (i < nvalid && y[i] > cm) {
            cm = y[i];
            ca = vw + i;
          }
        }
        const float ref = cm == -INFINITY ? 0.f : cm;
        float zs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (i < nvalid) zs[i & 3] += ex2_approx((y[i] - ref) * c);
        const int at = warp * kLmRows + ch * 32 + lane;
        sh_m[at] = cm;
        sh_z[at] = (zs[0] + zs[1]) + (zs[2] + zs[3]);
        sh_arg[at] = ca;
        if (tok >= vw && tok - vw < nvalid && token_logit) token_logit[grow] = tw[(tok - vw) * 33 + lane];
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(map_rank(bAccEmpty + 8 * ab, 0));
      epi_sync();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = threadIdx.x + h * kLmEpiWarps * 32, grow = x.h0 + j;
        if (j >= x.nrow || grow >= M) continue;
        const float c = sh_c[j];
        float m = run_m[h];
        int arg = run_arg[h];
#pragma unroll
        for (int w = 0; w < kLmEpiWarps; ++w)  // (columns in ascending order: the first of equal maxima stays)
          if (sh_m[w * kLmRows + j] > m) {
            m = sh_m[w * kLmRows + j];
            arg = sh_arg[w * kLmRows + j];
          }
        // the tile's sum, then the pair's range so far, in two floats (a sum over the range in one, rescaled by
        // ex2.approx: rms error of Z against 64 bits 9.5e-8 for 33 rows over V = 128256, with exact logits; so 5.6e-8,
        // and 6.4e-8 for 128-column partials in one float merged in binary64)
        const float mt = fmaxf(fmaxf(sh_m[j], sh_m[kLmRows + j]), fmaxf(sh_m[2 * kLmRows + j], sh_m[3 * kLmRows + j]));
        float zh = 0.f, zl = 0.f;
#pragma unroll
        for (int w = 0; w < kLmEpiWarps; ++w) {
          const float v = sh_z[w * kLmRows + j], mw = sh_m[w * kLmRows + j];
          const float f = mw > -INFINITY ? ex2_approx((mw - mt) * c) : 0.f;
          const float t = __fmul_rn(v, f);
          two_add(zh, zl, t, __fmaf_rn(v, f, -t));
        }
        if (cut.row_tiles == 1 && it > 0) {
          const bool up = mt > run_m[h];
          float ah = up ? zh : run_zh[h], al = up ? zl : run_zl[h];
          lm_add(ah, al, up ? run_zh[h] : zh, up ? run_zl[h] : zl, up ? run_m[h] : mt, m, c, table);
          zh = ah;
          zl = al;
        }
        if (cut.row_tiles == 1) {
          run_m[h] = m;
          run_zh[h] = zh;
          run_zl[h] = zl;
          run_arg[h] = arg;
        }
        if ((cut.row_tiles > 1 || it == n_items - 1) && x.slot < n_part)
          *reinterpret_cast<float4*>(part + (size_t)grow * n_part + x.slot) =
              make_float4(m, zh, zl, __int_as_float(arg));
      }
      epi_sync();  // the shares are read before the next item's are written
    }
    if (!ok && lane == 0) raise_status(status, LIBRASPEC_ST_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // neither CTA leaves while the other may still signal it
  tc_fence_after();
  if (warp == kLmMma)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(2 * kLmRows) : "memory");
}

// One CTA per row, a programmatic dependent launch: Z = sum_n z_n 2^((m_n - m) c); the argmax is the first column
// of the largest max; the token probability is 2^((x_tok - m) c) / Z, x_tok left in its place by the tiles. What
// bounds it: the powers. In binary64 (a sixty-fourth of the rate), a warp per row, this launch took 9 us of 37 (128
// rows over V = 32896, Dm = 2048) and 100 of 1320 (2112 rows over V = 128256, Dm = 4096), so terms and sum are carried
// in two floats each (2^-39, against the 2^-22 of the terms within z_n) and the last steps in binary64: both launches
// then took 31 and 1270 us. The launch of the tiles gives no early signal: a merge that may start beside the tiles
// puts all of its CTAs on the few SMs without one and took 66 us for those 128 rows.
// A token outside [-1, V) sets LIBRASPEC_ST_BAD_TOKEN (probability NaN).
constexpr int kMergeThreads = 128;
__global__ void __launch_bounds__(kMergeThreads) lm_head_merge_kernel(
    const LmPartial* __restrict__ part, int V, int n_part, const float* __restrict__ temperature, int rows_per_seq,
    const int32_t* __restrict__ tokens, const __grid_constant__ LmExpTable exp_table, float* __restrict__ row_stat,
    int32_t* __restrict__ row_argmax, float* __restrict__ token_prob, int* __restrict__ status) {
  __shared__ float2 table[32];
  __shared__ float sh_m[kMergeThreads / 32];
  __shared__ int sh_arg[kMergeThreads / 32];
  __shared__ double sh_z[kMergeThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = blockIdx.x;
  const LmPartial* p = part + (size_t)r * n_part;
  float T = temperature ? temperature[r / rows_per_seq] : 1.f;
  if (!(T > 0.f)) T = 1.f;
  const float c = log2e_over(T);
  if (warp == 0) table[lane] = exp_table.t[lane];
  asm volatile("griddepcontrol.wait;" ::: "memory");  // every partial is written
  float mx = -INFINITY;
  int arg = 0x7fffffff;
#pragma unroll 4
  for (int n = threadIdx.x; n < n_part; n += kMergeThreads) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(p + n));
    argmax_combine(mx, arg, v.x, __float_as_int(v.w));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, mx, off);
    const int a2 = __shfl_xor_sync(0xffffffffu, arg, off);
    argmax_combine(mx, arg, m2, a2);
  }
  if (lane == 0) {
    sh_m[warp] = mx;
    sh_arg[warp] = arg;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kMergeThreads / 32; ++w) argmax_combine(mx, arg, sh_m[w], sh_arg[w]);
  float zh = 0.f, zl = 0.f;
#pragma unroll 4
  for (int n = threadIdx.x; n < n_part; n += kMergeThreads) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(p + n));
    if (v.x > -INFINITY) lm_add(zh, zl, v.y, v.z, v.x, mx, c, table);
  }
  double Z = (double)zh + (double)zl;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, off);
  if (lane == 0) sh_z[warp] = Z;
  __syncthreads();
  if (threadIdx.x != 0) return;
  Z = (sh_z[0] + sh_z[1]) + (sh_z[2] + sh_z[3]);
  if (row_stat) {
    row_stat[2 * (size_t)r] = mx;
    row_stat[2 * (size_t)r + 1] = (float)Z;
  }
  if (row_argmax) row_argmax[r] = arg;
  if (token_prob) {
    const int tok = tokens ? tokens[r] : -1;
    if (tok >= V || tok < -1) {
      raise_status(status, LIBRASPEC_ST_BAD_TOKEN);
      token_prob[r] = __int_as_float(0x7fc00000);
    } else if (tok < 0) {
      token_prob[r] = 0.f;
    } else {
      float xh, xl, h, l;
      int e;
      lm_exponent(__ldcg(token_prob + r), mx, c, xh, xl);  // (the token's logit, left there by the tiles)
      lm_exp2(xh, xl, table, h, l, e);
      const double scale = __hiloint2double((e + 1023) << 20, 0);  // 2^e, e >= -1000
      token_prob[r] = (float)(((double)h + (double)l) * scale / Z);
    }
  }
}
static_assert(sizeof(LmPartial) == 16, "a partial is one float4");
static_assert(kMergeThreads == 128, "four warps' sums");

int num_sms_current();

// Partials per row: one per 128 columns, or one per CTA of the pairs that share the vocabulary (at least one pair).
static int lm_parts(int V) { return std::max((V + kLmHalf - 1) / kLmHalf, 2); }

size_t lm_head_workspace_bytes(int M, int V) { return 256 + align256((size_t)M * lm_parts(V) * sizeof(LmPartial)); }

static bool make_2d_map(CUtensorMap* map, const void* base, int cols, int rows, int box_rows) {
  // box_rows <= 256 (TMA), a multiple of 8 (whole 1024-byte swizzle atoms)
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)kLmBK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

static const LmExpTable& exp_table() {
  static const LmExpTable table = [] {
    LmExpTable t;
    for (int j = 0; j < 32; ++j) {
      const double v = std::exp2(j / 32.0);
      t.t[j].x = (float)v;
      t.t[j].y = (float)(v - (double)t.t[j].x);
    }
    return t;
  }();
  return table;
}

// Workspace: the status word, then the partials [M, n_part].
cudaError_t launch_lm_head_stats(const uint16_t* H, const uint16_t* W, const float* temperature, int rows_per_seq,
                                 const int32_t* tokens, int M, int V, int Dm, float* row_stat, int32_t* row_argmax,
                                 float* token_prob, char* ws, cudaStream_t stream) {
  if (M == 0) return cudaSuccess;
  const int max_pairs = std::max(num_sms_current() / 2, 1);
  const int units = (M + 31) / 32;
  LmCut cut;
  cut.row_tiles = (M + kLmRows - 1) / kLmRows;
  cut.big = (units + cut.row_tiles - 1) / cut.row_tiles * 32;
  cut.n_big = cut.row_tiles - (cut.row_tiles * (cut.big / 32) - units);
  int pairs, n_part;
  if (cut.row_tiles == 1) {
    // one range per pair, at most lm_parts(V) / 2 of them, each a multiple of 16 columns
    pairs = std::min(max_pairs, lm_parts(V) / 2);
    cut.range = ((V + pairs - 1) / pairs + 15) / 16 * 16;
    pairs = (V + cut.range - 1) / cut.range;
    cut.tiles = (cut.range + kLmTile - 1) / kLmTile;
    cut.tail = ((cut.range - (cut.tiles - 1) * kLmTile) / 2 + 7) / 8 * 8;
    n_part = 2 * pairs;
  } else {
    cut.range = V;
    cut.tiles = (V + kLmTile - 1) / kLmTile;
    cut.tail = kLmHalf;
    pairs = (int)std::min<long long>((long long)cut.row_tiles * cut.tiles, max_pairs);
    n_part = (V + kLmHalf - 1) / kLmHalf;
  }
  const int slab_bytes = (int)kLmATile + cut.big * kLmBK;
  const int sub = Dm / kLmBK % kLmSub == 0 ? kLmSub : 1;
  const int stage_bytes = sub * slab_bytes;
  const int stages = std::min((kLmSmemMax - kLmFixed) / stage_bytes, kLmMaxStages);
  CUtensorMap mapH, mapHs, mapW, mapWt;
  if (!make_2d_map(&mapH, H, Dm, M, cut.big / 2) ||
      !make_2d_map(&mapHs, H, Dm, M, std::max(cut.big / 2 - 16, 16)) ||
      !make_2d_map(&mapW, W, Dm, V, kLmHalf) || !make_2d_map(&mapWt, W, Dm, V, cut.tail))
    return cudaErrorInvalidValue;
  static bool configured = false;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(lm_head_stats_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kLmSmemMax);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  auto* part = reinterpret_cast<LmPartial*>(ws + 256);
  auto* status = reinterpret_cast<int*>(ws);
  lm_head_stats_kernel<<<2 * pairs, kLmThreads, kLmFixed + stages * stage_bytes, stream>>>(
      mapH, mapHs, mapW, mapWt, temperature, rows_per_seq, tokens, M, V, Dm, cut, stages, sub,
      n_part, exp_table(), part, token_prob, status);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // the merge launch is prepared while the tiles run (2.5 us less than a plain launch)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(M);
  cfg.blockDim = dim3(kMergeThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lm_head_merge_kernel, (const LmPartial*)part, V, n_part, temperature, rows_per_seq,
                            tokens, exp_table(), row_stat, row_argmax, token_prob, status);
}

}  // namespace libraspec
