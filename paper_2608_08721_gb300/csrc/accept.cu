// Step 4: acceptance (greedy argmax match / rejection sampling).
#include "rowpass.cuh"

namespace libraspec {

// ---------------------------------------------------------------------------
// Node rows of a draft tree: grid (nsplit, K+1, B), rows j > L_b exit at once.
// A row's slices each leave (value, token), and the CTA that completes the row
// (atomic ticket) takes the token of the largest value (the lowest on ties)
// into node_arg[b, j], which the walk reads.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tree_row_finish(float m, int arg, int row, int split, int nsplit,
                                                RowPartial* __restrict__ part, uint32_t* __restrict__ cnt,
                                                int32_t* __restrict__ node_arg) {
  __shared__ float smf[32];
  __shared__ int smi[32];
  __shared__ int last;
  cta_reduce_arg(m, arg, smf, smi);
  if (nsplit == 1) {
    if (threadIdx.x == 0) node_arg[row] = arg;
    return;
  }
  if (threadIdx.x == 0) {
    RowPartial p;
    p.m = m;
    p.arg = arg;
    p.s = 0.0;
    part[(size_t)row * kRowMaxSplits + split] = p;
    __threadfence();
    const uint32_t ticket = atomicAdd(&cnt[row], 1u);
    last = (ticket == (uint32_t)(nsplit - 1));
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return;
  __threadfence();
  float M;
  int A;
  double Z;
  warp_merge_partials(part + (size_t)row * kRowMaxSplits, nsplit, 0.f, true, M, A, Z);
  if (threadIdx.x == 0) {
    node_arg[row] = A;
    cnt[row] = 0u;
  }
}

// Every sequence greedy: the rows' argmaxes.
template <bool VEC, typename E>
__global__ void __launch_bounds__(kRowThreads) tree_argmax_kernel(
    const E* __restrict__ target, const int32_t* __restrict__ Ls, int K, int V, int nsplit, int chunk,
    RowPartial* __restrict__ part, uint32_t* __restrict__ cnt, int32_t* __restrict__ node_arg,
    int* __restrict__ status) {
  const int split = blockIdx.x, j = blockIdx.y, b = blockIdx.z;
  const int Lb = Ls[b];
  if (Lb < 0 || Lb > K) {
    if (split == 0 && j == 0 && threadIdx.x == 0) raise_status(status, LIBRASPEC_ST_BAD_LENGTH);
    return;
  }
  if (j > Lb) return;
  const int row = b * (K + 1) + j;
  const int c0 = split * chunk, c1 = min(V, c0 + chunk);
  SumAcc sa;
  ArgAcc aa;
  sa.init();
  aa.init();
  row_slice_pass<false, true, VEC, E>(target + (size_t)row * V, c0, c1, 1.f, sa, aa);
  tree_row_finish(aa.m, aa.arg, row, split, nsplit, part, cnt, node_arg);
}

// ---------------------------------------------------------------------------
// Acceptance of a chain draft (Sec. 3.1: the target verifies every drafted
// position; the rule is the rejection sampler of Leviathan et al. at T > 0
// and the argmax match at T = 0), in two launches (three above 256
// sequences):
//
// The plan. From L[] and the temperatures, the rows the decisions read:
//   j <= L_b of a greedy sequence (the argmax of row L_b is its bonus token),
//   j < L_b of a sampling one; cut into S slices, S chosen so that the units
//   fill the rows grid (one unit per CTA). A sampling sequence with L_b = 0
//   is decided here (its bonus draw). Up to 256 sequences every rows CTA
//   makes the plan by itself, a sequence per thread (a prefix sum over the
//   CTA, less than a microsecond); above, accept_plan_kernel (one CTA) writes
//   one 8-byte descriptor per unit (sequence, row, slice, L_b, and log2(e)/T
//   of a sampling sequence), in a whole round before the attention layers.
//   As a launch of its own for every batch the plan cost 4 us (64 ragged
//   sequences: 49.4 us, now 45.1).
// accept_rows_kernel. CTA u works on unit u: a greedy row's slice yields
//   (max, argmax); a sampling row's slice (max, sum of exp((y - max) / T))
//   and, from the slice that holds the drafted token x_j, y_{j, x_j}. The CTA
//   completing a sequence's last slice merges its rows and takes the
//   decisions (binary64 p/q against the Philox uniform, or the argmax
//   match): a greedy sequence writes its result; a sampling one records its
//   draw, the bonus draw from row L_b when all drafts were accepted, else the
//   residual draw max(0, p_n - q_n) after the rejection at n.
// accept_race_kernel (a programmatic dependent launch). Grid (slices, B):
//   every recorded draw is an exponential race over the vocabulary, split
//   into slices; the CTA completing a sequence's last slice merges it and
//   writes the result. The bonus race's winner argmin_v E_v / exp((y_v -
//   m) / T) does not depend on the row's max m or normaliser, so its
//   candidates are carried as (E_v, y_v) and compared pairwise and the row
//   needs no statistics pass.
// ---------------------------------------------------------------------------
constexpr int kAccMaxRows = LIBRASPEC_MAX_K + 1;
constexpr int kPlanThreads = 1024;

struct AccPlanHeader {
  int R;      // rows
  int S;      // slices per row
  int chunk;  // logits per slice
  int U;      // units (R * S)
};

// descriptor: b | j << 12 | s << 19 | L_b << 25 (b < 4096, j, L_b <= 64,
// s < 64), and log2(e)/T as float bits (0: a greedy sequence)
__device__ __forceinline__ uint32_t pack_unit(int b, int j, int s, int Lb) {
  return (uint32_t)b | ((uint32_t)j << 12) | ((uint32_t)s << 19) | ((uint32_t)Lb << 25);
}

template <typename E>
struct AcceptArgs {
  const E* target;          // [B, K+1, V]
  const E* draft;           // [B, K, V]
  const int32_t* tokens;    // [B, K]
  const float* conf;        // [B, K] q_j(x_j)
  const float* dstat;       // [B, K, 2] drafter (max, Z)
  const float* temperature; // [B]
  const int32_t* L;         // [B]
  int B, K, V;
  int have_q;               // conf and dstat are given
  int chunkB, SB;           // race slices: length and count per row
  uint64_t seed, round_offset;
  uint32_t seq_offset;
  const uint64_t* rng;      // optional {seed, round_offset, seq_offset} in device memory
  const AccPlanHeader* hdr;
  const uint2* desc;        // [max(kAccMaxGrid, B*(K+1))]
  RowPartial* part;         // [B*(K+1), kRowMaxSplits]
  float* yx;                // [B*(K+1)]
  uint32_t* seq_cnt;        // [B]
  ResEntry* res;            // [B]
  uint32_t* ready;          // [B] res[b] published (reset by the draw's last CTA)
  RaceCand* rpart;          // [B, kRaceMaxSplits]
  uint32_t* rcnt;           // [B]
  int32_t* n_accepted;
  int32_t* bonus;
  int* status;
};

// (E, y, idx) candidates of a race whose key is E * 2^(-y c): candidate 2
// replaces 1 iff E2 < E1 * 2^((y2 - y1) c), or on equality at a lower index.
__device__ __forceinline__ void race_combine(float& E, float& y, int& i, float E2, float y2, int i2, float c) {
  if (!(E2 < INFINITY)) return;
  if (!(E < INFINITY)) {
    E = E2; y = y2; i = i2;
    return;
  }
  const float X = E * ex2_approx((y2 - y) * c);
  if (E2 < X || (E2 == X && i2 < i)) {
    E = E2; y = y2; i = i2;
  }
}

// Order-preserving map of floats to ints (for atomicMin on shared memory) and back.
__device__ __forceinline__ int float_order(float f) {
  const int i = __float_as_int(f);
  return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float order_float(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }

// The smallest value any lane of the warp holds (all 32 lanes take part).
__device__ __forceinline__ float warp_fmin(float x) {
  float r;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}

// A race over logits [c0, c1) of one row: token v's key is E_v / w_v with
// E_v = -ln u_v, u_v the uniform of word v & 3 of the Philox block (v >> 2, j,
// seq, purpose), and log2 w_v <= y_v c + off. The smallest key wins.
//
// Bound by issue (a Philox block alone is about 60 instructions per four
// tokens), so almost no token is worked out: since -ln u >= 1 - u, a token
// can only beat the best log2 key `thr` known so far if
//   1 - u_v < 2^(thr + off + y_v c),
// and the eight tokens of two Philox blocks are dismissed by one such test on
// their largest uniform and their largest logit. If it passes, they are tested one
// by one, and eval(y, u, v) takes those that pass exactly. `thr` is the best
// key of any lane of the CTA: the lanes' own() keys (log2, a fast logarithm
// is enough) by warp minimum, the warps' through s_thr, refreshed after the
// first token of each lane and whenever a test of the warp has passed. The
// margins (2^0.004, and 2^-21 of |y c| in the exponent) are far above the
// rounding of the test, so every possible winner passes.
// Before (each token tested with two exponentials, exact steps whenever a
// lane of the warp passed): 70 instructions per token; 2 trees of 257 nodes,
// V = 152064, bf16: 148 us; now 23 instructions, 87 us (the Philox blocks by
// themselves: 50 us).
// Loads run two trips ahead of the eight logits in use (two Philox blocks and
// one copy of the exact step per trip: short code, and two chains to
// interleave); the trip counts are the warp's, so that every lane joins the
// votes.
template <bool VEC, typename E, typename Own, typename Eval>
__device__ __forceinline__ void race_slice(const E* __restrict__ yr, int c0, int c1, int V, float c, float off,
                                           uint64_t seed, uint32_t j, uint32_t seq, uint32_t purpose,
                                           uint64_t round_offset, int* s_thr, Own own, Eval eval) {
  const int g1 = (c1 + 3) >> 2;
  const int lane = threadIdx.x & 31;
  const float slack = c * 4.76837158203125e-7f;
  const float add = off + 0.004f;
  float thr = INFINITY;
  auto bound = [&](float y) { return ex2_approx(thr + (fmaf(fabsf(y), slack, add) + y * c)); };
  auto refresh = [&]() {
    const float m = warp_fmin(own());
    if (lane == 0 && m < thr) atomicMin(s_thr, float_order(m));
    thr = fminf(thr, m);
  };
  using Raw4 = typename Logit<E>::Raw4;
  auto load = [&](int g, Raw4 (&raw)[2]) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int gg = g + k * kRowThreads;
      if (VEC) raw[k] = gg < g1 ? Logit<E>::load4(yr + 4 * gg) : Logit<E>::none4();
      else raw[k] = Logit<E>::gather4(yr + 4 * (size_t)gg, gg < g1 ? V - 4 * gg : 0);
    }
  };
  const int gw0 = (c0 >> 2) + (int)(threadIdx.x & ~31u);
  Raw4 next[2], after[2];
  load(gw0 + lane, next);
  load(gw0 + 2 * kRowThreads + lane, after);
#pragma unroll 1
  for (int gw = gw0; gw < g1; gw += 2 * kRowThreads) {
    const int g = gw + lane;
    float y[8];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      float y4[4];
      Logit<E>::unpack4(next[k], y4);
#pragma unroll
      for (int t = 0; t < 4; ++t) y[4 * k + t] = y4[t];
      next[k] = after[k];
    }
    load(g + 4 * kRowThreads, after);
    const uint4 wa = philox_block(seed, (uint32_t)g, j, seq, purpose, round_offset);
    const uint4 wb = philox_block(seed, (uint32_t)(g + kRowThreads), j, seq, purpose, round_offset);
    const uint32_t ws[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
    if (gw == gw0) {
      if (4 * g < c1 && y[0] > -INFINITY) eval(y[0], word_to_uniform(ws[0]), 4 * g);
      refresh();
    }
    thr = fminf(thr, order_float(*reinterpret_cast<volatile int*>(s_thr)));
    const float ym = fmaxf(fmaxf(fmaxf(y[0], y[1]), fmaxf(y[2], y[3])), fmaxf(fmaxf(y[4], y[5]), fmaxf(y[6], y[7])));
    const uint32_t wm = max(max(max(ws[0], ws[1]), max(ws[2], ws[3])), max(max(ws[4], ws[5]), max(ws[6], ws[7])));
    const bool pass = word_to_uniform(~wm) < bound(ym);  // word ~w: exactly 1 - u
    if (__any_sync(0xffffffffu, pass)) {
      if (pass) {
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int v = 4 * (g + (t >> 2) * kRowThreads) + (t & 3);
          if (v < c1 && y[t] > -INFINITY && word_to_uniform(~ws[t]) < bound(y[t])) eval(y[t], word_to_uniform(ws[t]), v);
        }
      }
      __syncwarp();
      refresh();
    }
  }
}

// CTA reduction of race candidates; result in thread 0.
__device__ __forceinline__ void cta_reduce_race(float& E, float& y, int& i, float c, float* smE /*[32]*/,
                                                float* smy /*[32]*/, int* smi /*[32]*/) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float E2 = __shfl_xor_sync(0xffffffffu, E, off);
    const float y2 = __shfl_xor_sync(0xffffffffu, y, off);
    const int i2 = __shfl_xor_sync(0xffffffffu, i, off);
    race_combine(E, y, i, E2, y2, i2, c);
  }
  if (lane == 0) { smE[warp] = E; smy[warp] = y; smi[warp] = i; }
  __syncthreads();
  if (threadIdx.x == 0) {
    E = smE[0]; y = smy[0]; i = smi[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) race_combine(E, y, i, smE[w], smy[w], smi[w], c);
  }
}

// Largest b with start[b] <= r (rows of empty sequences are skipped).
__device__ __forceinline__ int seq_of_row(const int* start, int B, int r) {
  int lo = 0, hi = B - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= r) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// CTA argmin of (key, index); result in thread 0.
__device__ __forceinline__ void cta_reduce_min(float& best, int& besti, float* smk, int* smi) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float k2 = __shfl_xor_sync(0xffffffffu, best, off);
    const int i2 = __shfl_xor_sync(0xffffffffu, besti, off);
    argmin_combine(best, besti, k2, i2);
  }
  if (lane == 0) { smk[warp] = best; smi[warp] = besti; }
  __syncthreads();
  if (threadIdx.x == 0) {
    best = smk[0];
    besti = smi[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) argmin_combine(best, besti, smk[w], smi[w]);
  }
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Publish sequence b's draw (release: the entry is visible before the flag).
__device__ __forceinline__ void publish_draw(ResEntry* res, uint32_t* ready, int b, const ResEntry& en) {
  res[b] = en;
  __threadfence();
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ready + b), "r"(1u) : "memory");
}

// Bounded wait for a published flag: false after limit_ns (LIBRASPEC_ST_TIMEOUT).
__device__ bool wait_published(const uint32_t* flag, int* status, uint64_t limit_ns = 2000000000ull) {
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (ld_acquire_u32(flag) != 0u) return true;
    if (it == 0) {
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    } else if ((it & 7u) == 0u) {
      uint64_t t;
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
      if (t - t0 > limit_ns) {
        raise_status(status, LIBRASPEC_ST_TIMEOUT);
        return false;
      }
    }
    __nanosleep(it < 8 ? 128u : 1024u);
  }
}

// The rows that sequence b's decisions read. A sequence whose L_b lies
// outside [0, K], or that samples without q, has none and gets its result at
// once (written where `write` holds).
__device__ __forceinline__ int planned_rows(int b, int Lb, bool sampling, int K, int have_q, bool write,
                                            int32_t* __restrict__ n_accepted, int32_t* __restrict__ bonus,
                                            ResEntry* __restrict__ res, uint32_t* __restrict__ ready,
                                            int* __restrict__ status) {
  const bool bad_len = Lb < 0 || Lb > K;
  const bool bad = bad_len || (sampling && !have_q);
  if (!bad && !sampling) return Lb + 1;
  if (!bad && Lb > 0) return Lb;
  if (!write) return 0;
  ResEntry en;
  en.n = bad ? -1 : 0;
  en.mode = bad ? 0 : 1;  // (no draft to verify: the bonus draw from row 0)
  en.mp = 0.f;
  en.invZp = 0.f;
  if (bad) {
    n_accepted[b] = 0;
    bonus[b] = 0;
    raise_status(status, bad_len ? LIBRASPEC_ST_BAD_LENGTH : LIBRASPEC_ST_MISSING_INPUT);
  }
  if (sampling) publish_draw(res, ready, b, en);  // its draw CTAs wait for it
  return 0;
}

// Slices per row: as many as the grid of G CTAs holds (one unit per CTA),
// each of at least 2048 logits.
__device__ __forceinline__ void plan_slices(int R, int G, int V, int& S, int& chunk) {
  const int smax = max(1, min(kRowMaxSplits, (V + 2047) / 2048));
  S = R > 0 ? G / R : 1;
  S = max(1, min(S, smax));
  chunk = (((V + S - 1) / S) + kRowAlign - 1) & ~(kRowAlign - 1);
  S = (V + chunk - 1) / chunk;
}

// The plan of the rows grid (G CTAs) above kPlanInline sequences.
__global__ void __launch_bounds__(kPlanThreads) accept_plan_kernel(const int32_t* __restrict__ Ls,
                                                                   const float* __restrict__ temperature,
                                                                   int have_q, int B, int K, int V, int G,
                                                                   AccPlanHeader* __restrict__ hdr,
                                                                   uint2* __restrict__ desc,
                                                                   int32_t* __restrict__ n_accepted,
                                                                   int32_t* __restrict__ bonus,
                                                                   ResEntry* __restrict__ res,
                                                                   uint32_t* __restrict__ ready,
                                                                   int* __restrict__ status) {
  __shared__ int s_start[LIBRASPEC_MAX_B + 1];
  __shared__ float s_c[LIBRASPEC_MAX_B];
  __shared__ int s_L[LIBRASPEC_MAX_B];
  __shared__ int smi[32];
  __shared__ int s_tot;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (B + kPlanThreads - 1) / kPlanThreads;
  int loc = 0;
  for (int i = 0; i < per; ++i) {
    const int b = tid * per + i;
    if (b >= B) break;
    const int Lb = Ls[b];
    const float tb = temperature[b];
    const bool sampling = tb > 0.f;
    const int r = planned_rows(b, Lb, sampling, K, have_q, true, n_accepted, bonus, res, ready, status);
    s_start[b] = r;  // rows for now, turned into the prefix below
    s_c[b] = sampling ? log2e_over(tb) : 0.f;
    s_L[b] = Lb;
    loc += r;
  }
  int incl = loc;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += o;
  }
  if (lane == 31) smi[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int t = smi[lane];
    int ti = t;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, ti, off);
      if (lane >= off) ti += o;
    }
    smi[lane] = ti - t;  // exclusive prefix of the warp totals
    if (lane == 31) s_tot = ti;
  }
  __syncthreads();
  {
    int run = smi[warp] + incl - loc;
    for (int i = 0; i < per; ++i) {
      const int b = tid * per + i;
      if (b >= B) break;
      const int r = s_start[b];
      s_start[b] = run;
      run += r;
    }
  }
  const int R = s_tot;
  int S, chunk;
  plan_slices(R, G, V, S, chunk);
  const int U = R * S;
  if (tid == 0) {
    s_start[B] = R;
    AccPlanHeader h;
    h.R = R;
    h.S = S;
    h.chunk = chunk;
    h.U = U;
    *hdr = h;
  }
  __syncthreads();
  for (int u = tid; u < U; u += kPlanThreads) {
    const int r = u / S, s = u - r * S;
    const int b = seq_of_row(s_start, B, r);
    desc[u] = make_uint2(pack_unit(b, r - s_start[b], s, s_L[b]), __float_as_uint(s_c[b]));
  }
}

// PLAN: at most kPlanInline sequences, the plan made here.
constexpr int kPlanInline = kRowThreads;
template <bool VEC, typename E, bool PLAN>
__global__ void __launch_bounds__(kRowThreads, 6) accept_rows_kernel(const AcceptArgs<E> a) {
  __shared__ float s_m[kAccMaxRows];
  __shared__ double s_Z[kAccMaxRows];
  __shared__ int s_arg[kAccMaxRows];
  __shared__ float smf[64];
  __shared__ int smi[32];
  __shared__ int sh[1];
  __shared__ float s_yx;
  __shared__ int4 s_unit;  // this unit's sequence, row, L_b, log2(e)/T
  // the race launch may start its CTAs (each waits for its own sequence)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // after the attention layers of a round: a programmatic dependent launch
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x;
  const int K = a.K, V = a.V;
  int S, chunk, U;
  uint2 d = make_uint2(0, 0);
  int my_rows = 0, my_first = 0, my_L = 0;  // PLAN: of sequence tid
  float my_c = 0.f;
  if constexpr (PLAN) {
    if (tid < a.B) {
      my_L = a.L[tid];
      const float tb = a.temperature[tid];
      my_rows = planned_rows(tid, my_L, tb > 0.f, K, a.have_q, blockIdx.x == 0, a.n_accepted, a.bonus, a.res, a.ready,
                             a.status);
      my_c = tb > 0.f ? log2e_over(tb) : 0.f;
    }
    int incl = my_rows;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) smi[warp] = incl;
    __syncthreads();
    int R = 0;
    my_first = incl - my_rows;
#pragma unroll
    for (int w = 0; w < kRowThreads / 32; ++w) {
      if (w < warp) my_first += smi[w];
      R += smi[w];
    }
    plan_slices(R, G, V, S, chunk);
    U = R * S;
  } else {
    const AccPlanHeader h = *a.hdr;
    d = a.desc[blockIdx.x];  // read beside the header (stale beyond the plan's units)
    S = h.S;
    chunk = h.chunk;
    U = h.U;
  }

  for (int u = blockIdx.x; u < U; u += G) {
    int b, j, s, Lb;
    float c;
    if constexpr (PLAN) {
      const int r = u / S;
      s = u - r * S;
      if (r >= my_first && r < my_first + my_rows)
        s_unit = make_int4(tid, r - my_first, my_L, __float_as_int(my_c));
      __syncthreads();  // (and smi has been read)
      b = s_unit.x;
      j = s_unit.y;
      Lb = s_unit.z;
      c = __int_as_float(s_unit.w);
    } else {
      if (u != (int)blockIdx.x) d = a.desc[u];
      b = (int)(d.x & 0xfffu);
      j = (int)((d.x >> 12) & 0x7fu);
      s = (int)((d.x >> 19) & 0x3fu);
      Lb = (int)(d.x >> 25);
      c = __uint_as_float(d.y);
    }
    const bool sampling = c > 0.f;
    const int rows_b = sampling ? Lb : Lb + 1;
    const size_t row = (size_t)b * (K + 1) + j;
    const E* yr = a.target + row * V;
    const int c0 = s * chunk, c1 = min(V, c0 + chunk);
    RowPartial* pp = a.part + row * kRowMaxSplits + s;
    if (!sampling) {
      SumAcc sa;
      ArgAcc aa;
      sa.init();
      aa.init();
      row_slice_pass<false, true, VEC, E>(yr, c0, c1, 1.f, sa, aa);
      float m = aa.m;
      int arg = aa.arg;
      cta_reduce_arg(m, arg, smf, smi);
      if (tid == 0) {
        RowPartial p;
        p.m = m;
        p.arg = arg;
        p.s = 0.0;
        *pp = p;
      }
    } else {
      // the drafted token's logit: kept by the thread that streams it
      const int x = a.tokens[(size_t)b * K + j];
      SumAcc sa;
      ArgAcc aa;
      sa.init();
      row_slice_pass<true, false, VEC, E, true>(yr, c0, c1, c, sa, aa, x, &s_yx);
      float m = sa.m, sum = sa.value();
      cta_reduce_sum(m, sum, c, smf);  // its barrier also publishes s_yx
      if (tid == 0) {
        RowPartial p;
        p.m = m;
        p.arg = 0;
        p.s = (double)sum;
        *pp = p;
        if (x >= c0 && x < c1) a.yx[row] = s_yx;
      }
    }
    if (tid == 0) {
      __threadfence();
      sh[0] = atomicAdd(&a.seq_cnt[b], 1u) == (uint32_t)(rows_b * S - 1);
    }
    __syncthreads();
    if (!sh[0]) continue;

    // ---- decision for sequence b (this CTA completed its last slice) ----
    __threadfence();
    const size_t row0 = (size_t)b * (K + 1);
    // the first 32 decisions' inputs, loaded beside the merges
    int xj = 0;
    float yj = 0.f, qj = 0.f;
    if (warp == 0 && lane < Lb) {
      xj = a.tokens[(size_t)b * K + lane];
      if (sampling) {
        yj = __ldcg(&a.yx[row0 + lane]);
        qj = a.conf[(size_t)b * K + lane];
      }
    }
    for (int jj = warp; jj < rows_b; jj += kRowThreads / 32) {
      const RowPartial* p = a.part + (row0 + jj) * kRowMaxSplits;
      float M;
      int A;
      double Z;
      if (!sampling) {
        warp_merge_partials(p, S, 0.f, true, M, A, Z);
        if (lane == 0) s_arg[jj] = A;
      } else {
        warp_merge_partials(p, S, c, false, M, A, Z);
        if (lane == 0) { s_m[jj] = M; s_Z[jj] = Z; }
      }
    }
    __syncthreads();
    if (warp == 0) {
      uint64_t seed = a.seed, round_offset = a.round_offset;
      uint32_t seq_offset = a.seq_offset;
      if (a.rng) {  // the generator's arguments from device memory (a replayed graph of a staged round)
        seed = a.rng[0];
        round_offset = a.rng[1];
        seq_offset = (uint32_t)a.rng[2];
      }
      int n = Lb;
      for (int base = 0; base < Lb; base += 32) {
        const int jj = base + lane;
        bool reject = false;
        if (jj < Lb) {
          const int x = base == 0 ? xj : a.tokens[(size_t)b * K + jj];
          if (x < 0 || x >= V) {
            raise_status(a.status, LIBRASPEC_ST_BAD_TOKEN);
            reject = true;
          } else if (!sampling) {
            reject = s_arg[jj] != x;
          } else {
            const float y = base == 0 ? yj : __ldcg(&a.yx[row0 + jj]);
            const double p = (double)exp2f((y - s_m[jj]) * c) / s_Z[jj];
            const double q = (double)(base == 0 ? qj : a.conf[(size_t)b * K + jj]);
            const double ratio = (q <= p) ? 1.0 : p / q;
            const uint4 w = philox_block(seed, 0u, (uint32_t)jj, seq_offset + (uint32_t)b, 0u, round_offset);
            reject = !((double)word_to_uniform(w.x) < ratio);
          }
        }
        const unsigned ball = __ballot_sync(0xffffffffu, reject);
        if (ball) {
          n = base + __ffs(ball) - 1;
          break;
        }
      }
      if (lane == 0) {
        a.seq_cnt[b] = 0u;  // ready for the next call
        ResEntry en;
        en.n = n;
        en.mode = 0;
        en.mp = 0.f;
        en.invZp = 0.f;
        if (!sampling) {
          const int w = s_arg[n];
          a.n_accepted[b] = n;
          a.bonus[b] = w == 0x7fffffff ? 0 : w;  // a row without a finite logit
        } else {
          if (n == Lb) {
            en.mode = 1;  // all drafts accepted: the bonus draw from row L_b
          } else {
            en.mode = 2;  // rejected at n: the residual draw
            en.mp = s_m[n];
            en.invZp = (float)(1.0 / s_Z[n]);
          }
          publish_draw(a.res, a.ready, b, en);
        }
      }
    }
    __syncthreads();
  }
}

// The draws: CTA (s, b) runs slice s of sequence b's race, if b recorded
// one; the CTA completing the last slice merges the race and writes
// (n, the drawn token). A programmatic dependent launch of the rows grid:
// it starts once every rows CTA has started, and each CTA waits (bounded)
// only for its own sequence's decision, so a sequence's race overlaps the
// rows still streaming for the others.
template <bool VEC, typename E>
__global__ void __launch_bounds__(kRowThreads, 4) accept_race_kernel(const AcceptArgs<E> a) {
  __shared__ float smk[32];
  __shared__ float smy[32];
  __shared__ int smi[32];
  __shared__ int sh[2];
  __shared__ ResEntry s_en;
  __shared__ float s_c;
  __shared__ int s_thr;
  const int s = blockIdx.x, b = blockIdx.y;
  // a greedy sequence has no draw (and publishes none): its CTAs leave at
  // once, so they hold no slot while the sampling races wait and run
  if (!(a.temperature[b] > 0.f)) return;
  if (threadIdx.x == 0) {
    sh[0] = wait_published(a.ready + b, a.status);
    s_en = a.res[b];
    s_c = log2e_over(a.temperature[b]);  // once per CTA: a binary32 division and reciprocal
    s_thr = float_order(INFINITY);
  }
  __syncthreads();
  if (!sh[0]) return;
  const ResEntry en = s_en;
  if (en.mode == 0) {  // nothing to draw: the last CTA of b resets the flag
    if (threadIdx.x == 0 && atomicAdd(&a.rcnt[b], 1u) == (uint32_t)(a.SB - 1)) {
      a.rcnt[b] = 0u;
      a.ready[b] = 0u;
    }
    return;
  }
  const int n = en.n;
  uint64_t seed = a.seed, round_offset = a.round_offset;
  uint32_t seq_offset = a.seq_offset;
  if (a.rng) {
    seed = a.rng[0];
    round_offset = a.rng[1];
    seq_offset = (uint32_t)a.rng[2];
  }
  const int K = a.K, V = a.V;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float c = s_c;
  const E* yr = a.target + ((size_t)b * (K + 1) + n) * V;
  const uint32_t seq = seq_offset + (uint32_t)b;
  const int c0 = s * a.chunkB, c1 = min(V, c0 + a.chunkB);
  const bool residual = en.mode == 2;
  float bE = INFINITY, by = 0.f;
  int bi = 0x7fffffff;
  if (residual) {
    const E* dr = a.draft + ((size_t)b * K + n) * V;
    const float mq = a.dstat[2 * ((size_t)b * K + n)];
    const float invZq = 1.0f / a.dstat[2 * ((size_t)b * K + n) + 1];
    // weight max(0, p - q): at most p, which bounds the key; the drafter's
    // logit is read for the tokens that pass
    race_slice<VEC, E>(
        yr, c0, c1, V, c, __log2f(en.invZp) - en.mp * c, seed, (uint32_t)n, seq, 1u, round_offset, &s_thr,
        [&]() { return bi == 0x7fffffff ? INFINITY : __log2f(bE); },
        [&](float y, float u, int v) {
          // exponents are <= 0 (below the row maxima), so the fast base-2
          // exponential is exact to a few ulp
          const float w = ex2_approx((y - en.mp) * c) * en.invZp - ex2_approx((Logit<E>::at(dr, v) - mq) * c) * invZq;
          if (w > 0.f) argmin_combine(bE, bi, __fdividef(-logf(u), w), v);
        });
    cta_reduce_min(bE, bi, smk, smi);
  } else {
    race_slice<VEC, E>(
        yr, c0, c1, V, c, 0.f, seed, (uint32_t)n, seq, 1u, round_offset, &s_thr,
        [&]() { return bE < INFINITY ? __log2f(bE) - by * c : INFINITY; },
        [&](float y, float u, int v) {
          const float Ev = -logf(u);
          if (!(bE < INFINITY) || Ev < bE * ex2_approx((y - by) * c)) {
            bE = Ev;
            by = y;
            bi = v;
          }
        });
    cta_reduce_race(bE, by, bi, c, smk, smy, smi);
  }
  if (tid == 0) {
    RaceCand p;
    p.E = bE;
    p.y = by;
    p.idx = bi;
    p.pad = 0;
    a.rpart[(size_t)b * kRaceMaxSplits + s] = p;
    __threadfence();
    sh[0] = atomicAdd(&a.rcnt[b], 1u) == (uint32_t)(a.SB - 1);
  }
  __syncthreads();
  if (!sh[0]) return;
  __threadfence();
  if (warp == 0) {
    float kb = INFINITY, ky = 0.f;
    int ib = 0x7fffffff;
    const RaceCand* rp = a.rpart + (size_t)b * kRaceMaxSplits;
    for (int i = lane; i < a.SB; i += 32) {
      if (residual) argmin_combine(kb, ib, __ldcg(&rp[i].E), __ldcg(&rp[i].idx));
      else race_combine(kb, ky, ib, __ldcg(&rp[i].E), __ldcg(&rp[i].y), __ldcg(&rp[i].idx), c);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float k2 = __shfl_xor_sync(0xffffffffu, kb, off);
      const float y2 = __shfl_xor_sync(0xffffffffu, ky, off);
      const int i2 = __shfl_xor_sync(0xffffffffu, ib, off);
      if (residual) argmin_combine(kb, ib, k2, i2);
      else race_combine(kb, ky, ib, k2, y2, i2, c);
    }
    if (lane == 0) {
      a.rcnt[b] = 0u;  // ready for the next call
      a.ready[b] = 0u;
      sh[1] = kb < INFINITY ? ib : (residual ? -1 : 0);  // a bonus row without a finite logit: token 0
    }
  }
  __syncthreads();
  int win = sh[1];
  if (win < 0) {
    // residual identically zero (p_n == q_n to rounding): draw from p_n
    // instead, in this CTA alone (rare)
    float bk = INFINITY;
    int bkI = 0x7fffffff;
    for (int v = tid; v < V; v += kRowThreads) {
      const uint4 w4 = philox_block(seed, (uint32_t)(v >> 2), (uint32_t)n, seq, 1u, round_offset);
      const uint32_t wsel = (v & 3) == 0 ? w4.x : (v & 3) == 1 ? w4.y : (v & 3) == 2 ? w4.z : w4.w;
      const float wv = exp2f((Logit<E>::at(yr, v) - en.mp) * c);
      if (wv > 0.f) argmin_combine(bk, bkI, -logf(word_to_uniform(wsel)) / wv, v);
    }
    cta_reduce_min(bk, bkI, smk, smi);
    win = bkI == 0x7fffffff ? 0 : bkI;
  }
  if (tid == 0) {
    a.n_accepted[b] = n;
    a.bonus[b] = win;
  }
}

// Failure-detection self-test: the draws' bounded wait on a device flag with
// a caller-given limit; observed = 1 if the flag was seen, 0 if the wait
// gave up (and raised LIBRASPEC_ST_TIMEOUT).
__global__ void selftest_wait_kernel(const uint32_t* __restrict__ flag, uint64_t limit_ns,
                                     int32_t* __restrict__ observed, int* __restrict__ status) {
  if (threadIdx.x == 0) *observed = wait_published(flag, status, limit_ns) ? 1 : 0;
}

// ---------------------------------------------------------------------------
// Per-node draws of a draft tree (the same grid). A greedy sequence
// (temperature 0) takes the argmax of the node's target row; a sampling one
// draws from softmax(row / T) by the exponential race x = argmin_v key_v,
// key_v = log2(E_v) - y_v log2(e) / T, E_v = -ln u_v, u_v from Philox at
// (v >> 2, node t, sequence, purpose 2), word v & 3 (race_slice). The race is
// carried as an argmax of -key so the partials merge like argmaxes (lowest
// index on ties).
// ---------------------------------------------------------------------------
template <bool VEC, typename E>
__global__ void __launch_bounds__(kRowThreads, 4) tree_rows_kernel(
    const E* __restrict__ target, const int32_t* __restrict__ Ls, const float* __restrict__ temperature, int K,
    int V, int nsplit, int chunk, uint64_t seed, uint64_t round_offset, uint32_t seq_offset,
    RowPartial* __restrict__ part, uint32_t* __restrict__ cnt, int32_t* __restrict__ node_arg,
    int* __restrict__ status) {
  __shared__ int s_thr;
  const int split = blockIdx.x, j = blockIdx.y, b = blockIdx.z;
  const int Lb = Ls[b];
  if (Lb < 0 || Lb > K) {
    if (split == 0 && j == 0 && threadIdx.x == 0) raise_status(status, LIBRASPEC_ST_BAD_LENGTH);
    return;
  }
  if (j > Lb) return;
  const int row = b * (K + 1) + j;
  const float tb = temperature[b];
  const E* xr = target + (size_t)row * V;
  const int c0 = split * chunk, c1 = min(V, c0 + chunk);
  float m;
  int arg;
  if (!(tb > 0.f)) {
    SumAcc sa;
    ArgAcc aa;
    sa.init();
    aa.init();
    row_slice_pass<false, true, VEC, E>(xr, c0, c1, 1.f, sa, aa);
    m = aa.m;
    arg = aa.arg;
  } else {
    const float c = log2e_over(tb);
    const uint32_t seq = seq_offset + (uint32_t)b;
    float best = INFINITY;
    int besti = 0x7fffffff;
    if (threadIdx.x == 0) s_thr = float_order(INFINITY);
    __syncthreads();
    race_slice<VEC, E>(
        xr, c0, c1, V, c, 0.f, seed, (uint32_t)j, seq, 2u, round_offset, &s_thr, [&]() { return best; },
        [&](float y, float u, int v) { argmin_combine(best, besti, log2f(-logf(u)) - y * c, v); });
    m = -best;
    arg = besti;
  }
  tree_row_finish(m, arg, row, split, nsplit, part, cnt, node_arg);
}

// ---------------------------------------------------------------------------
// Walk of a draft tree, one warp per sequence. Node t in [1, L_b] has parent
// parent[b, t] < t and token tokens[b, t-1]. The warp first finds, for every
// node p, its matching child next[p]: the lowest-numbered child whose token is
// p's (node_arg: its target row's argmax, or the draw of a sampling sequence),
// by shared-memory atomicMin over the nodes; then it follows next[] from the
// root. n = nodes walked, last = the final node, bonus = its token. A parent
// outside [0, t) or a token outside [0, V) never matches and raises its
// status bit.
// ---------------------------------------------------------------------------
constexpr int kWalkWarps = 4;
constexpr int kWalkNodes = LIBRASPEC_MAX_TREE_NODES + 1;

__global__ void __launch_bounds__(kWalkWarps * 32) tree_walk_kernel(
    const int32_t* __restrict__ tokens, const int32_t* __restrict__ parent, const int32_t* __restrict__ Ls, int B,
    int K, int V, const int32_t* __restrict__ node_arg, int32_t* __restrict__ n_accepted,
    int32_t* __restrict__ last_node, int32_t* __restrict__ bonus, int* __restrict__ status) {
  __shared__ int arg_s[kWalkWarps][kWalkNodes];
  __shared__ int next_s[kWalkWarps][kWalkNodes];
  asm volatile("griddepcontrol.wait;" ::: "memory");  // every node's token is written
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * kWalkWarps + w;
  if (b >= B) return;
  const int Lb = Ls[b];
  if (Lb < 0 || Lb > K) {  // the rows' kernel raised the status
    if (lane == 0) {
      n_accepted[b] = 0;
      if (last_node) last_node[b] = 0;
      bonus[b] = 0;
    }
    return;
  }
  int* arg = arg_s[w];
  int* next = next_s[w];
  constexpr int kNone = 0x7fffffff;
  for (int t = lane; t <= Lb; t += 32) {
    const int a = __ldcg(node_arg + (size_t)b * (K + 1) + t);
    arg[t] = a == 0x7fffffff ? 0 : a;  // a row without a finite logit
    next[t] = kNone;
  }
  __syncwarp();
  for (int t = lane + 1; t <= Lb; t += 32) {
    const int p = parent[(size_t)b * (K + 1) + t];
    const int x = tokens[(size_t)b * K + t - 1];
    if (p < 0 || p >= t) raise_status(status, LIBRASPEC_ST_BAD_TREE);
    else if (x < 0 || x >= V) raise_status(status, LIBRASPEC_ST_BAD_TOKEN);
    else if (x == arg[p]) atomicMin(&next[p], t);
  }
  __syncwarp();
  if (lane == 0) {
    int cur = 0, n = 0;
    while (n < Lb && next[cur] != kNone) {  // next[] only points to higher nodes
      cur = next[cur];
      ++n;
    }
    n_accepted[b] = n;
    if (last_node) last_node[b] = cur;
    bonus[b] = arg[cur];
  }
}

// ---------------------------------------------------------------------------
// Host launchers.
// ---------------------------------------------------------------------------
int num_sms_current();

// temperature == nullptr: every sequence greedy (argmax rows); else per
// sequence, greedy at 0 and drawing at T > 0 (tree_rows_kernel).
template <typename T>
cudaError_t launch_accept_tree(const T* target, const int32_t* tokens, const int32_t* parent, const int32_t* L,
                               const float* temperature, int B, int K, int V, uint64_t seed, uint64_t round_offset,
                               uint32_t seq_offset, int32_t* n_accepted, int32_t* last_node, int32_t* bonus,
                               char* ws, const WsLayout& lay, cudaStream_t stream) {
  if (B == 0) return cudaSuccess;
  const int sms = num_sms_current();
  auto* st = reinterpret_cast<int*>(ws + lay.status);
  auto* node_arg = reinterpret_cast<int32_t*>(ws + lay.node_arg);
  const long rows = (long)B * (K + 1);
  // The draws' rows: as few slices as make one wave of resident CTAs (4 per SM), since a race settles its threshold
  // anew in each (2 trees of 257 nodes: 100 us at 16 CTAs per SM, 94 at 8, 90 at 4, 99 at 2); the argmax rows: more,
  // for the loads.
  const int nsplit0 = temperature == nullptr ? row_splits(rows, V, sms, kRowMaxSplits, 4096)
                                             : wave_splits(rows, V, 4L * sms, kRowMaxSplits, 4096);
  const int chunk = row_chunk(V, nsplit0);
  const int nsplit = (V + chunk - 1) / chunk;
  dim3 grid(nsplit, K + 1, B);
  auto* part = reinterpret_cast<RowPartial*>(ws + lay.row_part);
  auto* cnt = reinterpret_cast<uint32_t*>(ws + lay.row_cnt);
  const bool vec = rows_vectorizable(target, V);
  if (temperature == nullptr) {
    if (vec)
      tree_argmax_kernel<true, T><<<grid, kRowThreads, 0, stream>>>(target, L, K, V, nsplit, chunk, part, cnt,
                                                                     node_arg, st);
    else
      tree_argmax_kernel<false, T><<<grid, kRowThreads, 0, stream>>>(target, L, K, V, nsplit, chunk, part, cnt,
                                                                      node_arg, st);
  } else if (vec) {
    tree_rows_kernel<true, T><<<grid, kRowThreads, 0, stream>>>(target, L, temperature, K, V, nsplit, chunk, seed,
                                                                 round_offset, seq_offset, part, cnt, node_arg, st);
  } else {
    tree_rows_kernel<false, T><<<grid, kRowThreads, 0, stream>>>(target, L, temperature, K, V, nsplit, chunk, seed,
                                                                  round_offset, seq_offset, part, cnt, node_arg, st);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // the walk's launch is prepared while the rows run (2 trees of 257 nodes: 88.7 -> 86.7 us)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((B + kWalkWarps - 1) / kWalkWarps);
  cfg.blockDim = dim3(kWalkWarps * 32);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, tree_walk_kernel, tokens, parent, L, B, K, V, (const int32_t*)node_arg, n_accepted,
                            last_node, bonus, st);
}
template cudaError_t launch_accept_tree<float>(const float*, const int32_t*, const int32_t*, const int32_t*,
                                               const float*, int, int, int, uint64_t, uint64_t, uint32_t, int32_t*,
                                               int32_t*, int32_t*, char*, const WsLayout&, cudaStream_t);
template cudaError_t launch_accept_tree<uint16_t>(const uint16_t*, const int32_t*, const int32_t*, const int32_t*,
                                                  const float*, int, int, int, uint64_t, uint64_t, uint32_t, int32_t*,
                                                  int32_t*, int32_t*, char*, const WsLayout&, cudaStream_t);

// CTAs of the acceptance rows kernel resident at once on the current device;
// its grid is two waves of them (at most kAccMaxGrid; measured on the ragged
// batch: 51.5 us back to back against 54.3 with four waves, 53.0 with three).
template <bool VEC, typename T>
int accept_grid() {
  static int cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int g = cached[dev];
  if (g == 0) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, accept_rows_kernel<VEC, T, true>, kRowThreads, 0) !=
            cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
    g = std::min(2 * per_sm * num_sms_current(), kAccMaxGrid);
    cached[dev] = g;
  }
  return g;
}

template <typename T>
bool accept_vec(const T* target, const T* draft, int V) {
  // the races read groups of 4 logits: both rows must allow those loads too
  return rows_vectorizable(target, V) && (draft == nullptr || rows_vectorizable(draft, V));
}

// The acceptance plan for the rows grid of launch_accept<T> with the same
// pointers' alignment (one CTA; needs only L and the temperatures); nothing
// up to kPlanInline sequences, whose rows CTAs make it.
template <typename T>
cudaError_t launch_accept_plan(const T* target, const T* draft, const float* conf, const float* dstat,
                               const int32_t* L, const float* temperature, int B, int K, int V, int32_t* n_accepted,
                               int32_t* bonus, char* ws, const WsLayout& lay, cudaStream_t stream) {
  if (B <= kPlanInline) return cudaSuccess;
  const int G = accept_vec(target, draft, V) ? accept_grid<true, T>() : accept_grid<false, T>();
  if (G <= 0) return cudaErrorInvalidConfiguration;
  accept_plan_kernel<<<1, kPlanThreads, 0, stream>>>(
      L, temperature, conf != nullptr && dstat != nullptr, B, K, V, G,
      reinterpret_cast<AccPlanHeader*>(ws + lay.acc_plan), reinterpret_cast<uint2*>(ws + lay.acc_plan + 16),
      n_accepted, bonus, reinterpret_cast<ResEntry*>(ws + lay.acc_res),
      reinterpret_cast<uint32_t*>(ws + lay.acc_ready), reinterpret_cast<int*>(ws + lay.status));
  return cudaGetLastError();
}

// rng (optional, device): {seed, round_offset, seq_offset} read by the
// kernels in place of the three arguments. plan_ready: launch_accept_plan
// already ran for these inputs on this stream. after_own: the launch before
// this one on the stream is one of this call's, without a programmatic
// trigger, so that the rows may be launched dependent on it (the rows after a
// round's layers: with the plan 91.5 -> 84.8 us, 16 sampling sequences). A
// launch behind a draw never is: draws may end before their rows.
template <typename T>
cudaError_t launch_accept(const T* target, const T* draft, const int32_t* tokens, const float* conf,
                          const float* dstat, const int32_t* L, const float* temperature, int B, int K, int V,
                          uint64_t seed, uint64_t round_offset, uint32_t seq_offset, int32_t* n_accepted,
                          int32_t* bonus, char* ws, const WsLayout& lay, cudaStream_t stream,
                          const uint64_t* rng, bool plan_ready, bool after_own) {
  if (B == 0) return cudaSuccess;
  if (!plan_ready) {
    const cudaError_t e = launch_accept_plan<T>(target, draft, conf, dstat, L, temperature, B, K, V, n_accepted,
                                                bonus, ws, lay, stream);
    if (e != cudaSuccess) return e;
  }
  const bool vec = accept_vec(target, draft, V);
  AcceptArgs<T> a;
  a.target = target;
  a.draft = draft;
  a.tokens = tokens;
  a.conf = conf;
  a.dstat = dstat;
  a.temperature = temperature;
  a.L = L;
  a.have_q = conf != nullptr && dstat != nullptr;
  a.B = B;
  a.K = K;
  a.V = V;
  // race slices of about 4096 logits of each row
  int SB = (V + 4095) / 4096;
  if (SB > kRaceMaxSplits) SB = kRaceMaxSplits;
  const int chunkB = row_chunk(V, SB);
  a.SB = (V + chunkB - 1) / chunkB;
  a.chunkB = chunkB;
  a.seed = seed;
  a.round_offset = round_offset;
  a.seq_offset = seq_offset;
  a.rng = rng;
  a.hdr = reinterpret_cast<const AccPlanHeader*>(ws + lay.acc_plan);
  a.desc = reinterpret_cast<const uint2*>(ws + lay.acc_plan + 16);
  a.part = reinterpret_cast<RowPartial*>(ws + lay.row_part);
  a.yx = reinterpret_cast<float*>(ws + lay.acc_yx);
  a.seq_cnt = reinterpret_cast<uint32_t*>(ws + lay.acc_seq);
  a.res = reinterpret_cast<ResEntry*>(ws + lay.acc_res);
  a.ready = reinterpret_cast<uint32_t*>(ws + lay.acc_ready);
  a.rpart = reinterpret_cast<RaceCand*>(ws + lay.race_part);
  a.rcnt = reinterpret_cast<uint32_t*>(ws + lay.race_cnt);
  a.n_accepted = n_accepted;
  a.bonus = bonus;
  a.status = reinterpret_cast<int*>(ws + lay.status);
  const int G = vec ? accept_grid<true, T>() : accept_grid<false, T>();
  if (G <= 0) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(kRowThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = after_own || (!plan_ready && B > kPlanInline) ? 1 : 0;
  auto* rows = vec ? (B <= kPlanInline ? accept_rows_kernel<true, T, true> : accept_rows_kernel<true, T, false>)
                   : (B <= kPlanInline ? accept_rows_kernel<false, T, true> : accept_rows_kernel<false, T, false>);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, rows, a);
  if (e != cudaSuccess) return e;
  // the draws: launched once every rows CTA has started (each waits for its sequence)
  cfg.gridDim = dim3(a.SB, B);
  cfg.numAttrs = 1;
  if (vec) return cudaLaunchKernelEx(&cfg, accept_race_kernel<true, T>, a);
  return cudaLaunchKernelEx(&cfg, accept_race_kernel<false, T>, a);
}
template cudaError_t launch_accept<float>(const float*, const float*, const int32_t*, const float*, const float*,
                                          const int32_t*, const float*, int, int, int, uint64_t, uint64_t, uint32_t,
                                          int32_t*, int32_t*, char*, const WsLayout&, cudaStream_t,
                                          const uint64_t*, bool, bool);
template cudaError_t launch_accept_plan<float>(const float*, const float*, const float*, const float*,
                                               const int32_t*, const float*, int, int, int, int32_t*, int32_t*,
                                               char*, const WsLayout&, cudaStream_t);
template cudaError_t launch_accept_plan<uint16_t>(const uint16_t*, const uint16_t*, const float*, const float*,
                                                  const int32_t*, const float*, int, int, int, int32_t*, int32_t*,
                                                  char*, const WsLayout&, cudaStream_t);
cudaError_t launch_selftest_wait(const uint32_t* flag, uint64_t limit_ns, int32_t* observed, int* status,
                                 cudaStream_t stream) {
  selftest_wait_kernel<<<1, 32, 0, stream>>>(flag, limit_ns, observed, status);
  return cudaGetLastError();
}

template cudaError_t launch_accept<uint16_t>(const uint16_t*, const uint16_t*, const int32_t*, const float*,
                                             const float*, const int32_t*, const float*, int, int, int, uint64_t,
                                             uint64_t, uint32_t, int32_t*, int32_t*, char*, const WsLayout&,
                                             cudaStream_t, const uint64_t*, bool, bool);

}  // namespace libraspec
