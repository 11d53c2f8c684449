// The quantile-summary + MLP aggregator on the GPU (Pro-Router, Section 4.2,
// Table 2: the verifier-architecture ablation's alternative to the
// transformer head).  Per request: for each of the four Eq. 3 features (l, m,
// h, rho) over its T rows, the quantiles at levels a/b (q_level_a / q_level_b; linear
// interpolation between order statistics), a 28-number summary, then a
// 28 -> 64 -> 64 -> 1 ReLU MLP and a sigmoid.
//
// One CTA per request.  Up to Q_SMALL rows two warps per feature sort its
// column's order-preserving 32-bit keys (padded to 256) in registers, four
// per lane (a bitonic network inside the lanes, across them by shfl.xor, and
// one stage between the two warps).  Up to Q_MID rows the four columns are
// bitonic-sorted together, each thread holding a run of keys in registers
// (register and warp-shuffle stages, one stage through shared memory).  Longer
// requests select: histograms of the keys find the few keys around each needed
// rank, and only those are sorted (q_select).  All three give the exact order
// statistics.  The MLP runs in the same CTA with fixed-order sums (four
// threads per hidden unit, quarters added in a fixed butterfly).
#pragma once

#include "pr_device.cuh"

namespace prk {

constexpr int Q_NT = 256;
constexpr int Q_NQ = 7;             // quantile levels
constexpr int Q_NS = 4 * Q_NQ;      // summary length
constexpr int Q_H = 64;             // hidden width
constexpr int Q_SMALL = 256;        // rows sorted in registers, two warps per column
// Rows sorted whole: 12.4 us for a lone request of 513 to 1,024 rows whatever its
// values (graph replay).  From 1,025 rows, where 2,048 keys per column no longer
// fit the registers and the sort through shared memory took 62 us, the selection
// takes 10.3 us, 22 to 32 us when its bins are crowded, which is why shorter
// requests keep the sort (2,048 rows: 11.7 against 62.5 us, crowded 30 to 49;
// 4,000 rows: 17.6 against 360 us by a radix selection of one rank at a time).
constexpr int Q_MID = 1024;
__constant__ int32_t q_level_a[Q_NQ] = {0, 1, 1, 1, 3, 9, 1};
__constant__ int32_t q_level_b[Q_NQ] = {1, 10, 4, 2, 4, 10, 1};

// weight offsets (floats)
constexpr int QW_W1 = 0, QW_B1 = QW_W1 + Q_H * Q_NS, QW_W2 = QW_B1 + Q_H,
              QW_B2 = QW_W2 + Q_H * Q_H, QW_W3 = QW_B2 + Q_H, QW_B3 = QW_W3 + Q_H,
              QW_SIZE = QW_B3 + 1;

// the MLP's weights in shared memory once the keys are done with (they reuse
// the key buffer): rows padded to an odd stride, so that the 64 threads of a
// layer, one output each, read 64 different banks
constexpr int QS_W1 = 0, QS_B1 = Q_H * (Q_NS + 1), QS_W2 = QS_B1 + Q_H,
              QS_B2 = QS_W2 + Q_H * (Q_H + 1), QS_W3 = QS_B2 + Q_H, QS_B3 = QS_W3 + Q_H,
              QS_SIZE = QS_B3 + 1;
constexpr int QW_PER_T = (QW_SIZE + Q_NT - 1) / Q_NT;  // weights each thread fetches

// q_select: histograms of Q_BINS bins per feature, scanned by 64 threads in runs
// of Q_RUN bins (one word of padding per run, so that the runs lie in different
// banks), then of Q_SUB bins for each crowded bin
constexpr int Q_BINS = 2048, Q_SUB = 64, Q_RUN = Q_BINS / 64;
constexpr int Q_HW = Q_BINS + Q_BINS / Q_RUN;  // words of a feature's histogram
constexpr int Q_NR = 2 * Q_NQ;              // ranks per feature (12 distinct ones)
constexpr int Q_FEW = 42;                   // most keys of a bin that are collected
constexpr int Q_CAND = 512;                 // collected keys per feature
constexpr int Q_REC = 8;                    // records a thread holds in registers
static_assert(12 * Q_FEW <= Q_CAND, "the bins of all needed ranks fit");
constexpr int Q_SUB_WORDS = 4 * 12 * (Q_SUB + 1);  // counts of up to 12 crowded bins per feature
static_assert(Q_SUB_WORDS + 12 * Q_SUB <= 4 * Q_HW, "in the place of the histograms");
// dynamic shared memory (words): the MLP's weights, in whose place q_select
// keeps its histograms and marks before, and the keys of a column set
constexpr int Q_HM_WORDS = 4 * Q_HW + Q_BINS;  // histograms, a byte of marks per bin
constexpr int Q_W_WORDS = (QS_SIZE > Q_HM_WORDS ? QS_SIZE : Q_HM_WORDS) + 3 & ~3;
constexpr int Q_DYN = Q_W_WORDS + 4 * Q_CAND;
static_assert(4 * Q_MID <= Q_DYN && 4 * Q_SMALL + QS_SIZE <= Q_DYN, "whole columns");
static_assert(Q_SMALL == 256 && Q_NT == 256, "two warps per column sort 256 keys");
static_assert(Q_NT == 4 * Q_H && Q_NS % 4 == 0 && Q_H % 4 == 0, "four threads per hidden unit");

// shared-memory position of flat weight g
__device__ __forceinline__ int q_wpos(int g) {
  if (g < QW_B1) return QS_W1 + (g / Q_NS) * (Q_NS + 1) + g % Q_NS;
  if (g < QW_W2) return QS_B1 + (g - QW_B1);
  if (g < QW_B2) return QS_W2 + ((g - QW_W2) / Q_H) * (Q_H + 1) + (g - QW_W2) % Q_H;
  if (g < QW_W3) return QS_B2 + (g - QW_B2);
  if (g < QW_B3) return QS_W3 + (g - QW_W3);
  return QS_B3;
}

struct QArgs {
  const float* feat;
  const uint32_t* row_flags;
  int64_t n_rows;
  const int64_t* offsets;
  int32_t n_req;
  const float* w;
  float zthr;
  float* summary;  // [n_req][28] or null
  float* score;
  uint8_t* ship;
  uint32_t* req_flags;
  uint32_t* ctx_flags;
  int32_t full;  // the launch fills the GPU: the next one may be set up at once
};

__device__ __forceinline__ uint32_t q_key(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float q_unkey(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// record slot of feature f: l, m, h, rho
__device__ __forceinline__ int q_slot(int f) { return f == 0 ? 0 : f == 1 ? 1 : f == 2 ? 4 : 5; }

// Ascending bitonic sort of the 256 keys of one column held by two warps:
// lane l of warp `half` holds keys c = 128 half + 4 l .. + 3 in v.  Stages of
// partner distance below 4 run inside the lane's registers, 4..64 between
// lanes (shfl.xor), 128 between the two warps through xbuf (128 keys per
// warp) and the named barrier `bar` of the pair's 64 threads.
__device__ __forceinline__ void q_sort256_pair(uint32_t (&v)[4], int half, int lane,
                                               uint32_t* xbuf, int bar) {
#pragma unroll
  for (int k = 2; k <= 256; k <<= 1) {
    if (k == 256) {  // partner distance 128: the other warp
#pragma unroll
      for (int e = 0; e < 4; ++e) xbuf[half * 128 + lane * 4 + e] = v[e];
      asm volatile("bar.sync %0, 64;" ::"r"(bar) : "memory");
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t p = xbuf[(half ^ 1) * 128 + lane * 4 + e];
        v[e] = half == 0 ? min(v[e], p) : max(v[e], p);  // one ascending block
      }
    }
#pragma unroll
    for (int j = (k >> 1) < 64 ? (k >> 1) : 64; j >= 4; j >>= 1) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int c = half * 128 + lane * 4 + e;
        const uint32_t p = __shfl_xor_sync(FULL, v[e], j >> 2);
        const bool keep_min = ((c & j) == 0) == ((c & k) == 0);
        v[e] = keep_min ? min(v[e], p) : max(v[e], p);
      }
    }
#pragma unroll
    for (int j = (k >> 1) < 2 ? (k >> 1) : 2; j >= 1; j >>= 1) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if ((e & j) == 0) {
          const uint32_t x = v[e], y = v[e + j];
          const bool up = ((half * 128 + lane * 4 + e) & k) == 0;
          const uint32_t lo = min(x, y), hi = max(x, y);
          v[e] = up ? lo : hi;
          v[e + j] = up ? hi : lo;
        }
      }
    }
  }
}

// Ascending bitonic sort of the four columns col f = qs + (f << ln2) of n2 =
// 2^ln2 keys each, n2 = 64 E (512 or 1,024), by the whole CTA: thread t
// holds the E consecutive keys c0 .. c0 + E - 1 of one column (two warps per
// column).  A compare-exchange stage of partner distance j runs in registers
// for j < E, between the lanes of a warp (shfl.xor) for j < 32 E, and through
// shared memory only for j = n2 / 2.
template <int E>
__device__ void q_bitonic(uint32_t* qs, int ln2) {
  const int n2 = 1 << ln2, tid = threadIdx.x;
  const int per_col = n2 / E;  // threads per column
  const int c0 = (tid % per_col) * E;
  uint32_t* col = qs + ((tid / per_col) << ln2);
  uint32_t v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = col[c0 + e];
  for (int k = 2; k <= n2; k <<= 1) {
    for (int j = k >> 1; j >= E; j >>= 1) {
      if (j >= 32 * E) {  // the other warp of the column
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; ++e) col[c0 + e] = v[e];
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int c = c0 + e;
          const uint32_t p = col[c ^ j];
          const bool keep_min = ((c & j) == 0) == ((c & k) == 0);
          v[e] = keep_min ? min(v[e], p) : max(v[e], p);
        }
      } else {
        const int lm = j / E;  // lane distance
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int c = c0 + e;
          const uint32_t p = __shfl_xor_sync(FULL, v[e], lm);
          const bool keep_min = ((c & j) == 0) == ((c & k) == 0);
          v[e] = keep_min ? min(v[e], p) : max(v[e], p);
        }
      }
    }
#pragma unroll
    for (int jj = E / 2; jj >= 1; jj >>= 1) {  // inside the thread's keys
      if (jj < k) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if ((e & jj) == 0) {
            const uint32_t x = v[e], y = v[e + jj];
            const bool up = ((c0 + e) & k) == 0;
            const uint32_t lo = min(x, y), hi = max(x, y);
            v[e] = up ? lo : hi;
            v[e + jj] = up ? hi : lo;
          }
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < E; ++e) col[c0 + e] = v[e];
}

// keys [lo, lo + range] in `bins` equal steps: step of a key at distance d from
// lo is umulhi(d, mul), or d itself when mul is 0 (at most `bins` keys).  The
// multiplier is rounded down, so the last step stays below `bins`.
__device__ __forceinline__ uint32_t q_mul(uint32_t range, int bins) {
  if (range < (uint32_t)bins) return 0u;
  return (uint32_t)__fdiv_rz((float)bins * 4294963200.f, (float)range + 1.f);
}
__device__ __forceinline__ uint32_t q_step(uint32_t d, uint32_t mul) {
  return mul ? __umulhi(d, mul) : d;
}

// The order statistics of a request of T > Q_MID rows, by selection: whole
// CTA, quantile tid of the summary in *out for tid < Q_NS.
//   1. every feature's smallest and largest key (up to Q_REC * Q_NT rows the
//      records stay in registers, more rows are read again in each pass)
//   2. a histogram of Q_BINS equal steps of key between the two (key space is
//      about logarithmic in the value, which suits log-probabilities,
//      probabilities and position fractions alike)
//   3. the bin of every needed rank and the count of keys before it
//   4. the keys of those bins: bins of up to Q_FEW keys are collected, of a
//      crowded bin the smallest and largest key are kept
//   5. crowded bins whose keys differ are divided again, by Q_SUB, until the
//      ranks' bins hold few keys or one key many times (at most five rounds
//      for 32-bit keys; none on data without clusters)
//   6. the collected keys, about 150 per feature, are sorted; bins are
//      disjoint and ascending, so a rank's key stands at a known place
// Bound by the latency of this chain and, for long requests, of the passes.
// `idle` runs before the sort (loads that the caller wants in flight).
template <typename F>
__device__ __forceinline__ void q_select(const float* feat, int64_t lo, int T,
                                         uint32_t* dyn, uint32_t (*qx)[Q_SMALL], float* out,
                                         F idle) {
  __shared__ uint32_t s_red[8][Q_NT / 32], s_rank[Q_NR], s_pre[4][64], s_half[4], s_n[4];
  __shared__ uint32_t s_base[4][Q_NR], s_cnt[4][Q_NR], s_lo[4][Q_NR], s_hi[4][Q_NR];
  __shared__ uint32_t s_glo[4][Q_NR], s_ghi[4][Q_NR], s_gmul[4][Q_NR], s_bin0[4][Q_NR];
  __shared__ int s_grp[4][Q_NR], s_gend[4][Q_NR], s_off[4][Q_NR];
  uint32_t* hist = dyn;                                     // [4][Q_HW]
  uint8_t* mark = reinterpret_cast<uint8_t*>(dyn + 4 * Q_HW);  // [4][Q_BINS]
  // of the crowded bins: [4][12][Q_SUB + 1] counts and [4][12][Q_SUB] marks
  uint8_t* sub_mark = reinterpret_cast<uint8_t*>(dyn + Q_SUB_WORDS);
  uint32_t* cand = dyn + Q_W_WORDS;                         // [4][Q_CAND]
  constexpr uint8_t COLLECT = 0xff;  // a mark: collect the bin's keys; r + 1: extremes to rank r
  constexpr int CHUNK = Q_REC * Q_NT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool once = T <= CHUNK;
  uint32_t k[Q_REC][4];
  auto load = [&](uint32_t c0) {
#pragma unroll
    for (int i = 0; i < Q_REC; ++i) {
      const uint32_t t = c0 + (uint32_t)(i * Q_NT + tid);
      if (t < (uint32_t)T) {
        const float4* rec = reinterpret_cast<const float4*>(feat + (lo + t) * NFEAT);
        const float4 r0 = rec[0], r1 = rec[1];
        k[i][0] = q_key(r0.x);  // l
        k[i][1] = q_key(r0.y);  // m
        k[i][2] = q_key(r1.x);  // h
        k[i][3] = q_key(r1.y);  // rho
      }
    }
  };
  // body(f, key) for every key of the request
  auto each_key = [&](bool held, auto body) {
    for (uint32_t c0 = 0; c0 < (uint32_t)T; c0 += CHUNK) {
      if (!held) load(c0);
#pragma unroll
      for (int i = 0; i < Q_REC; ++i)
        if (c0 + (uint32_t)(i * Q_NT + tid) < (uint32_t)T) {
#pragma unroll
          for (int f = 0; f < 4; ++f) body(f, k[i][f]);
        }
    }
  };

  auto clear = [&](int words) {
    for (int i = tid; i < words / 4; i += Q_NT)
      reinterpret_cast<uint4*>(dyn)[i] = make_uint4(0u, 0u, 0u, 0u);
  };
  static_assert(Q_HM_WORDS % 4 == 0 && Q_SUB_WORDS % 4 == 0 && Q_SUB % 4 == 0, "16-byte stores");
  clear(Q_HM_WORDS);
  if (tid < Q_NR) {  // rank 2 j: the lower order statistic of level j; 2 j + 1: the upper
    const int64_t num = (int64_t)q_level_a[tid >> 1] * (T - 1);
    const int b = q_level_b[tid >> 1];
    const int64_t i = num / b;
    s_rank[tid] = (uint32_t)((tid & 1) && num != i * b ? i + 1 : i);
  }
  if (tid < 4) s_n[tid] = 0u;
  uint32_t kmin[4] = {~0u, ~0u, ~0u, ~0u}, kmax[4] = {0u, 0u, 0u, 0u}, mul[4];
  each_key(false, [&](int f, uint32_t key) {
    kmin[f] = min(kmin[f], key);
    kmax[f] = max(kmax[f], key);
  });
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const uint32_t a = __reduce_min_sync(FULL, kmin[f]), b = __reduce_max_sync(FULL, kmax[f]);
    if (lane == 0) {
      s_red[f][warp] = a;
      s_red[4 + f][warp] = b;
    }
  }
  __syncthreads();
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    kmin[f] = s_red[f][0];
    kmax[f] = s_red[4 + f][0];
#pragma unroll
    for (int w = 1; w < Q_NT / 32; ++w) {
      kmin[f] = min(kmin[f], s_red[f][w]);
      kmax[f] = max(kmax[f], s_red[4 + f][w]);
    }
    mul[f] = q_mul(kmax[f] - kmin[f], Q_BINS);
  }
  each_key(once, [&](int f, uint32_t key) {
    const uint32_t b = q_step(key - kmin[f], mul[f]);
    atomicAdd(hist + f * Q_HW + b + b / Q_RUN, 1u);
  });
  __syncthreads();

  {  // 64 threads per feature: the counts before each run of bins
    const int f = tid >> 6, u = tid & 63;
    const uint32_t* h = hist + f * Q_HW + (Q_RUN + 1) * u;
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < Q_RUN; ++i) sum += h[i];
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += y;
    }
    s_pre[f][u] = x - sum;
    if (u == 31) s_half[f] = x;
  }
  __syncthreads();
  // the bin of each rank (one warp per feature, one lane per rank), marked by
  // its first rank: collect its keys, or keep their extremes at that rank
  const int f_of = warp >> 1, j_of = min(lane, Q_NR - 1);
  auto settle = [&](uint32_t base, uint32_t cnt, uint8_t* m) {
    const uint32_t prev = __shfl_up_sync(FULL, base, 1);
    if (lane >= Q_NR || !m) return;
    s_base[f_of][lane] = base;
    s_cnt[f_of][lane] = cnt;
    s_lo[f_of][lane] = ~0u;
    s_hi[f_of][lane] = 0u;
    if (lane == 0 || base != prev) *m = cnt <= (uint32_t)Q_FEW ? COLLECT : (uint8_t)(lane + 1);
  };
  if ((warp & 1) == 0) {
    const uint32_t r = s_rank[j_of];
    int u = 0;
#pragma unroll
    for (int o = 32; o > 0; o >>= 1) {  // the last run whose count before is <= r
      const int v = u + o;
      if (s_pre[f_of][v] + (v >= 32 ? s_half[f_of] : 0u) <= r) u = v;
    }
    const uint32_t* h = hist + f_of * Q_HW + (Q_RUN + 1) * u;
    uint32_t c = s_pre[f_of][u] + (u >= 32 ? s_half[f_of] : 0u), base = c, cnt = 0;
    int at = 0;
#pragma unroll
    for (int i = 0; i < Q_RUN; ++i) {
      const uint32_t n = h[i];
      if (r >= c && r < c + n) {
        at = i;
        base = c;
        cnt = n;
      }
      c += n;
    }
    settle(base, cnt, mark + f_of * Q_BINS + Q_RUN * u + at);
    if (lane < Q_NR) s_bin0[f_of][lane] = base;
  }
  __syncthreads();
  auto take = [&](int f, uint32_t key, uint32_t m) {
    if (m == COLLECT) {
      cand[f * Q_CAND + atomicAdd(&s_n[f], 1u)] = key;
    } else if (m) {  // most keys of a bin lie inside the extremes seen so far
      if (key < *(volatile uint32_t*)&s_lo[f][m - 1]) atomicMin(&s_lo[f][m - 1], key);
      if (key > *(volatile uint32_t*)&s_hi[f][m - 1]) atomicMax(&s_hi[f][m - 1], key);
    }
  };
  auto mark_of = [&](int f, uint32_t key) -> uint32_t {
    return mark[f * Q_BINS + (int)q_step(key - kmin[f], mul[f])];
  };
  each_key(once, [&](int f, uint32_t key) { take(f, key, mark_of(f, key)); });

  // crowded bins with different keys: divided again between their extremes
  for (;;) {
    __syncthreads();
    bool mixed = false;
    if ((warp & 1) == 0) {
      const uint32_t base = s_base[f_of][j_of], bin0 = s_bin0[f_of][j_of];
      const uint32_t prev = __shfl_up_sync(FULL, base, 1);
      const uint32_t prev0 = __shfl_up_sync(FULL, bin0, 1);
      const uint32_t a = s_lo[f_of][j_of], b = s_hi[f_of][j_of];
      mixed = lane < Q_NR && (lane == 0 || base != prev) && a < b;
      const unsigned bal = __ballot_sync(FULL, mixed);
      // a rank's group is the one that its bin's first rank opens; the groups of
      // a bin of the first histogram end where those of the next one start
      const unsigned upto = 0xffffffffu >> (31 - lane);
      const unsigned firsts = __ballot_sync(FULL, lane == 0 || base != prev);
      const unsigned firsts0 = __ballot_sync(FULL, lane == 0 || bin0 != prev0);
      const int head = 31 - __clz(firsts & upto);
      const int g = __popc(bal & ((1u << head) - 1u));
      const unsigned later = firsts0 & ~upto;
      const int next = later ? __ffs(later) - 1 : 31;
      if (lane < Q_NR) {
        s_grp[f_of][lane] = g;
        s_gend[f_of][lane] = __popc(bal & ((1u << next) - 1u));
        s_off[f_of][lane] = (bal >> head) & 1u;  // whether the rank is in a group
      }
      if (mixed) {
        s_glo[f_of][g] = a;
        s_ghi[f_of][g] = b;
        s_gmul[f_of][g] = q_mul(b - a, Q_SUB);
      }
    }
    if (!__syncthreads_or(mixed)) break;
    clear(Q_SUB_WORDS + 12 * Q_SUB);
    __syncthreads();
    // group and step of a key, as f * 12 + group and 0 .. Q_SUB - 1; -1: none
    auto sub_of = [&](int f, uint32_t key, int& at) -> int {
      const uint32_t m = mark_of(f, key);
      if (m == 0u || m == COLLECT) return -1;
      for (int g = s_grp[f][m - 1]; g < s_gend[f][m - 1]; ++g)
        if (key >= s_glo[f][g] && key <= s_ghi[f][g]) {
          at = f * 12 + g;
          return (int)q_step(key - s_glo[f][g], s_gmul[f][g]);
        }
      return -1;
    };
    each_key(once, [&](int f, uint32_t key) {
      int at;
      const int s = sub_of(f, key, at);
      if (s >= 0) atomicAdd(dyn + at * (Q_SUB + 1) + s, 1u);
    });
    __syncthreads();
    if ((warp & 1) == 0) {
      const int at = f_of * 12 + s_grp[f_of][j_of];
      const bool in = s_off[f_of][j_of] != 0;
      const uint32_t r = s_rank[j_of];
      uint32_t c = s_base[f_of][j_of], base = c, cnt = 0;
      uint8_t* m = nullptr;
      if (in)
        for (int i = 0; i < Q_SUB; ++i) {
          const uint32_t n = dyn[at * (Q_SUB + 1) + i];
          if (r >= c && r < c + n) {
            m = sub_mark + at * Q_SUB + i;
            base = c;
            cnt = n;
          }
          c += n;
        }
      __syncwarp();
      settle(base, cnt, m);
    }
    __syncthreads();
    each_key(once, [&](int f, uint32_t key) {
      int at;
      const int s = sub_of(f, key, at);
      if (s >= 0) take(f, key, sub_mark[at * Q_SUB + s]);
    });
  }

  idle();
  if ((warp & 1) == 0) {  // where the collected keys of each rank's bin start
    const uint32_t base = s_base[f_of][j_of], cnt = s_cnt[f_of][j_of];
    const uint32_t prev = __shfl_up_sync(FULL, base, 1);
    const bool few = cnt <= (uint32_t)Q_FEW;
    uint32_t x = few && lane < Q_NR && (lane == 0 || base != prev) ? cnt : 0u;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += y;
    }
    if (lane < Q_NR) s_off[f_of][lane] = few ? (int)(x - cnt) : -1;
  }
  const uint32_t nmax = max(max(s_n[0], s_n[1]), max(s_n[2], s_n[3]));
  if (nmax <= (uint32_t)Q_SMALL) {
    const int f = warp >> 1, half = warp & 1;
    uint32_t* col = cand + f * Q_CAND + half * 128 + lane * 4;
    uint32_t v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      v[e] = (uint32_t)(half * 128 + lane * 4 + e) < s_n[f] ? col[e] : 0xffffffffu;
    q_sort256_pair(v, half, lane, qx[f], 1 + f);
#pragma unroll
    for (int e = 0; e < 4; ++e) col[e] = v[e];
  } else {
    for (int i = tid; i < 4 * Q_CAND; i += Q_NT)
      if ((uint32_t)(i % Q_CAND) >= s_n[i / Q_CAND]) cand[i] = 0xffffffffu;
    __syncthreads();
    q_bitonic<Q_CAND / 64>(cand, 9);
  }
  __syncthreads();
  if (tid < Q_NS) {
    const int f = tid / Q_NQ, lv = tid - f * Q_NQ;
    float x[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      int j = 2 * lv + e;
      if (s_off[f][j] >= 0) {
        x[e] = q_unkey(cand[f * Q_CAND + s_off[f][j] + (int)(s_rank[j] - s_base[f][j])]);
      } else {
        while (j > 0 && s_base[f][j - 1] == s_base[f][j]) --j;
        x[e] = q_unkey(s_lo[f][j]);
      }
    }
    const int64_t num = (int64_t)q_level_a[lv] * (T - 1);
    const int b = q_level_b[lv], rem = (int)(num % b);
    *out = rem ? x[0] + ((float)rem / (float)b) * (x[1] - x[0]) : x[0];
  }
}

__global__ void __launch_bounds__(Q_NT, 3) qmlp_requests(const QArgs a) {
  extern __shared__ __align__(16) uint32_t qs[];  // Q_DYN words
  __shared__ float qv[Q_NS];
  __shared__ float h1[Q_H], h2[Q_H];
  __shared__ uint32_t wfl[Q_NT / 32];
  __shared__ uint32_t qx[4][Q_SMALL];  // exchange between the two warps of a column
  __shared__ float zpart[2];
  pdl_wait();
  if (a.full) pdl_trigger();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r = blockIdx.x;
  const int64_t lo = a.offsets[r], hi = a.offsets[r + 1];
  if (lo < 0 || hi < lo || hi > a.n_rows) {
    if (tid == 0) {
      a.score[r] = NAN;
      a.ship[r] = 0;
      a.req_flags[r] = FLAG_BAD_OFFSETS;
      atomicOr(a.ctx_flags, FLAG_BAD_OFFSETS);
    }
    return;
  }
  const int T = (int)(hi - lo);
  // the MLP's weights, fetched now (coalesced) so that their latency overlaps
  // the offsets', the key loads and the sort; a selection, whose records take the
  // registers, fetches them again before it sorts
  float wr[QW_PER_T];
  auto fetch_w = [&]() {
#pragma unroll
    for (int i = 0; i < QW_PER_T; ++i) {
      const int g = tid + i * Q_NT;
      wr[i] = 0.f;
      if (g < QW_SIZE)  // (volatile: not to be moved behind the request's offsets)
        asm volatile("ld.global.f32 %0, [%1];" : "=f"(wr[i]) : "l"(a.w + g));
    }
  };
  fetch_w();
  if (T == 0) {
    if (tid == 0) {
      a.score[r] = 0.f;
      a.ship[r] = 0;
      a.req_flags[r] = FLAG_EMPTY_REQ;
    }
    return;
  }
  // the rows' flags: read now, decided after the order statistics (a flagged
  // request is rare, and its loads then overlap the key loads)
  uint32_t fl = 0;
  if (a.row_flags)
    for (int t = tid; t < T; t += Q_NT) fl |= a.row_flags[lo + t];
  fl = __reduce_or_sync(FULL, fl);
  if (lane == 0) wfl[warp] = fl;

  float* W = reinterpret_cast<float*>(qs);  // the MLP's weights in shared memory
  if (T <= Q_SMALL) {
    // the weights go beside the keys at once (their loads were issued at the
    // top), so that staging them is off the request's critical path
    W = reinterpret_cast<float*>(qs + 4 * Q_SMALL);
#pragma unroll
    for (int i = 0; i < QW_PER_T; ++i) {
      const int g = tid + i * Q_NT;
      if (g < QW_SIZE) W[q_wpos(g)] = wr[i];
    }
    // two warps per feature column: its keys (padded with the largest key to
    // 256) sorted in registers, then stored in order for the interpolation
    {
      const int f = warp >> 1, half = warp & 1;
      const int slot = q_slot(f);
      uint32_t v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int t = half * 128 + lane * 4 + e;
        v[e] = t < T ? q_key(a.feat[(lo + t) * NFEAT + slot]) : 0xffffffffu;
      }
      q_sort256_pair(v, half, lane, qx[f], 1 + f);
#pragma unroll
      for (int e = 0; e < 4; ++e) qs[f * Q_SMALL + half * 128 + lane * 4 + e] = v[e];
    }
    __syncthreads();
    if (tid < Q_NS) {
      const int f = tid / Q_NQ, lv = tid - f * Q_NQ;
      const uint32_t num = (uint32_t)q_level_a[lv] * (uint32_t)(T - 1);  // T <= 256
      const uint32_t b = (uint32_t)q_level_b[lv];
      const uint32_t lo_i = num / b, rem = num - lo_i * b;
      const uint32_t* col = qs + f * Q_SMALL;
      const float xl = q_unkey(col[lo_i]);
      float q = xl;
      if (rem) q = xl + ((float)rem / (float)b) * (q_unkey(col[lo_i + 1]) - xl);
      qv[tid] = q;
    }
  } else if (T <= Q_MID) {
    int ln2 = 9;  // n2 = 2^ln2 >= T, at least 512
    while ((1 << ln2) < T) ++ln2;
    const int n2 = 1 << ln2;
    // each thread reads whole records (two 16-byte loads give the four
    // features), several rows in flight at once
#pragma unroll 4
    for (int t = tid; t < n2; t += Q_NT) {
      uint32_t k0 = 0xffffffffu, k1 = 0xffffffffu, k2 = 0xffffffffu, k3 = 0xffffffffu;
      if (t < T) {
        const float4* rec = reinterpret_cast<const float4*>(a.feat + (lo + t) * NFEAT);
        const float4 r0 = rec[0], r1 = rec[1];
        k0 = q_key(r0.x);  // l
        k1 = q_key(r0.y);  // m
        k2 = q_key(r1.x);  // h
        k3 = q_key(r1.y);  // rho
      }
      qs[t] = k0;
      qs[n2 + t] = k1;
      qs[2 * n2 + t] = k2;
      qs[3 * n2 + t] = k3;
    }
    __syncthreads();
    if (ln2 == 9) q_bitonic<8>(qs, 9);
    else q_bitonic<16>(qs, 10);
    __syncthreads();
    if (tid < Q_NS) {
      const int f = tid / Q_NQ, j = tid - f * Q_NQ;
      const int64_t num = (int64_t)q_level_a[j] * (T - 1);
      const int b = q_level_b[j];
      const int lo_i = (int)(num / b), rem = (int)(num - (int64_t)lo_i * b);
      const uint32_t* col = qs + (f << ln2);
      const float xl = q_unkey(col[lo_i]);
      float q = xl;
      if (rem) {
        const float xh = q_unkey(col[min(lo_i + 1, T - 1)]);
        q = xl + ((float)rem / (float)b) * (xh - xl);
      }
      qv[tid] = q;
    }
  } else {
    q_select(a.feat, lo, T, qs, qx, qv + min(tid, Q_NS - 1), fetch_w);
  }
  __syncthreads();

  fl = 0;
#pragma unroll
  for (int w2 = 0; w2 < Q_NT / 32; ++w2) fl |= wfl[w2];
  if (fl & (FLAG_NONFINITE | FLAG_BAD_CHOSEN)) {
    if (tid == 0) {
      a.score[r] = NAN;
      a.ship[r] = 0;
      a.req_flags[r] = fl;
    }
    return;
  }

  // MLP 28 -> 64 -> 64 -> 1, weights from shared memory (longer requests
  // stage them now, in the key buffer)
  if (T > Q_SMALL) {
#pragma unroll
    for (int i = 0; i < QW_PER_T; ++i) {
      const int g = tid + i * Q_NT;
      if (g < QW_SIZE) W[q_wpos(g)] = wr[i];
    }
  }
  __syncthreads();
  // four threads per hidden unit: each sums a quarter of the inputs in order,
  // then the quarters are added in a fixed butterfly (lanes 4o .. 4o + 3)
  {
    const int o = tid >> 2, part = tid & 3;
    constexpr int P1 = Q_NS / 4, P2 = Q_H / 4;
    float s1 = 0.f;
#pragma unroll
    for (int i = 0; i < P1; ++i)
      s1 = fmaf(W[QS_W1 + o * (Q_NS + 1) + part * P1 + i], qv[part * P1 + i], s1);
    s1 += __shfl_xor_sync(FULL, s1, 1);
    s1 += __shfl_xor_sync(FULL, s1, 2);
    if (part == 0) h1[o] = fmaxf(s1 + W[QS_B1 + o], 0.f);
    __syncthreads();
    float s2 = 0.f;
#pragma unroll
    for (int i = 0; i < P2; ++i)
      s2 = fmaf(W[QS_W2 + o * (Q_H + 1) + part * P2 + i], h1[part * P2 + i], s2);
    s2 += __shfl_xor_sync(FULL, s2, 1);
    s2 += __shfl_xor_sync(FULL, s2, 2);
    if (part == 0) h2[o] = fmaxf(s2 + W[QS_B2 + o], 0.f);
  }
  __syncthreads();
  if (warp < 2) {
    float z = W[QS_W3 + tid] * h2[tid];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(FULL, z, o);
    if (lane == 0) zpart[warp] = z;
  }
  if (a.summary && tid < Q_NS) a.summary[r * Q_NS + tid] = qv[tid];
  __syncthreads();
  if (tid == 0) {
    const float z = (zpart[0] + zpart[1]) + W[QS_B3];
    a.score[r] = 1.f / (1.f + expf(-z));
    a.ship[r] = (z >= a.zthr) ? 1 : 0;
    a.req_flags[r] = fl;
  }
}

}  // namespace prk
