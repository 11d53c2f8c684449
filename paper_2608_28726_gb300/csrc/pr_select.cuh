// Operating-point calibration and selective-prediction metrics on the GPU
// (Pro-Router, Section 3.1: tau fixed on a validation pool; Section 4.1: the
// coverage rule with ship fraction q, AUROC and AUARC, the area under the
// accuracy of what ships against the fraction shipped).
//
// Everything follows from the scores' ascending order, in which the finite
// scores' order-preserving 32-bit keys form tie groups (runs of equal keys); a
// group of c items, p of them correct, with a items and Pa correct ones below
// it, contributes
//   to AUROC  p (2 (a - Pa) + (c - p)), twice its correct items' count of
//             incorrect items below plus half the tied ones (exact integers),
//   to AUARC  sum over its descending ranks k of C_k / k, C_k spreading its
//             correct answers evenly over its ranks; each term as a float pair
//             (about 44 bits), summed with compensation per thread, then in
//             fp64 in a fixed order (a long group in closed form, in fp64),
// and tau is the key of the group that holds ascending rank n_f - k, k =
// min(floor(q n + 1/2), n_f), n_f the number of finite scores.
//
// No pass sorts the pool.  The keys are partitioned into buckets of consecutive
// keys, and each bucket is resolved in shared memory:
//   sel_coarse   a histogram of the keys' 12 leading bits
//   sel_plan     each such bin is cut into 1 to 64 equal buckets, enough for
//                about `target` items each: at most SB_NB buckets
//   sel_count    items and correct items per bucket; each share of the pool
//                learns its place in every bucket from the atomic that adds it
//   sel_offsets  prefix sums over the buckets
//   sel_scatter  the items, as (key's offset in its bucket, label) in one word,
//                into their buckets (the order inside a bucket does not matter)
//   sel_heavy    buckets of more than SB_HEAVY items counted per key by many CTAs
//   sel_bucket   one bucket at a time: a crowded one by counting items and labels
//                for each of its keys, a light one by sorting it; then its groups
//   sel_finish   the buckets' sums in bucket order
// Results do not depend on the order in which items reach their buckets, so
// they are deterministic.  2^24 scores (sigmoids of normals): 468 us; a radix
// sort of keys and labels with scans and a pass over the sorted items took 787, of
// which the ranking of equal digits alone 425.  100,000 scores: 62 us against 130.
// sel_bucket takes 246 of the 468, bound by the issue of the groups' arithmetic
// (two CTAs with twice the registers per SM instead of three: the same within 2%
// either way, by the spread of the keys); sel_scatter 143, bound by its partly
// filled 32-byte sectors (a share has some 70 bytes for each bucket).  Scores of
// random bits in pools of a million, some 250 items in each of 4,095 coarse bins,
// stay the weakest pool: 157 us against 153.
#pragma once

#include "pr_device.cuh"

namespace prk {

constexpr int SB_NT = 512;            // threads per CTA
constexpr int SB_SHIFT = 20;          // a coarse bin: 2^20 consecutive keys
constexpr int SB_BINS = 1 << (32 - SB_SHIFT);
constexpr int SB_MAXB = 6;            // a bin has at most 2^6 buckets
constexpr int SB_TARGET = 1024;       // items per bucket aimed at, where the pool is large
constexpr int SB_FEW_TARGET = 256;    //   enough for 64 buckets of that many; at least
constexpr int SB_NB = SB_BINS + 2 * 8192 + 1;  // most buckets (a bin of c items over the
                                      //   target has fewer than 2 c / target; n / target <= 8192)
constexpr int SB_SHARE = 61440;       // most items of a share (16-bit counts)
constexpr int SB_VBITS = SB_SHIFT - SB_MAXB;  // keys counted at once: 2^14
constexpr int SB_SMALL = 128;         // most items of a bucket resolved by one warp (10,000
                                      //   random bit patterns: 70 us, by CTAs 143; with 256
                                      //   here a million of them 296 us instead of 158)
constexpr int SB_LIGHT = 4096;        // most items sorted in shared memory
constexpr int SB_HEAVY = 65535;       // more items than this: counted by several CTAs, in
constexpr int SB_CHUNK = 32768;       //   chunks of this many
constexpr int SB_RADIX = 4096;        // first step of sorting a light bucket
constexpr int SB_RUN = 24;            // most items of a sub-bin sorted by its thread
constexpr int SB_LONG = 64;           // most near groups: in closed form from here on
constexpr uint32_t SEL_NONFINITE = 0xffffffffu;
static_assert(SB_NB < 65536 && SB_SHARE <= 65535, "16-bit bucket numbers and counts");

struct SelResult {        // written by sel_bucket and sel_finish, copied to the host
  float tau;
  int32_t pad;
  int64_t n_finite, k, n_ship, n_pos;
  double auroc, auarc, acc_shipped;
};

struct SelArgs {
  const float* scores;
  const uint8_t* labels;       // or null
  uint32_t n, share, target, nbcap;
  double q;
  uint32_t* coarse;            // [SB_BINS] items per coarse bin       (zeroed)
  unsigned long long* total;   // [nbcap] items | correct << 32        (zeroed)
  uint32_t* info;              // buckets, finite, correct, next of the list, heavy buckets,
                               //   their chunks, crowded and light buckets (zeroed)
  uint32_t* plan;              // [SB_BINS] first bucket | log2 buckets << 16
  uint32_t* bkey;              // [nbcap] first key | log2 keys
  uint32_t* start;             // [nbcap + 1] items before the bucket
  uint32_t* pstart;            // [nbcap + 1] correct items before it
  uint32_t* rel;               // [shares][nbcap] a share's place in each bucket
  uint32_t* items;             // [n] offset in the bucket << 1 | label
  uint32_t* list;              // [nbcap] crowded buckets from the front, light from the back
  uint32_t* hidx;              // [nbcap] a heavy bucket's number
  uint2* hchunk;               // bucket and chunk of each chunk of the heavy buckets
  unsigned long long* hcnt;    // [heavy][2^SB_VBITS] items | correct << 32 per key
  unsigned long long* proc;    // [nbcap] AUROC and
  double* parc;                // [nbcap] AUARC sums of a bucket
  SelResult* out;
};

// finite score -> order-preserving key (-0 and +0 share one key)
__device__ __forceinline__ uint32_t sel_key(float s) {
  if (!isfinite(s)) return SEL_NONFINITE;
  const uint32_t u = __float_as_uint(s + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float sel_unkey(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// C / k for integers 0 <= C <= k < 2^32 as an unevaluated sum hi + lo of two floats
// without fp64: a correctly rounded fp32 reciprocal gives the first quotient q,
// fmaf gives the remainder C - q k, and the remainder times the reciprocal is
// the correction (about 46 correct bits).  Below 2^24 both integers are floats and
// the remainder is exact; from there on they are split by bit masks into parts
// that floats hold.
__device__ __forceinline__ float2 sel_ratio(uint32_t C, uint32_t k, float r) {  // r = 1 / k
  const float q = __fmul_rn((float)C, r);
  float rem;
  if (k < 1u << 24) {
    rem = fmaf(-q, (float)k, (float)C);
  } else {
    const float kh = (float)(k & ~0xffu), kl = (float)(k & 0xffu);
    const float ch = (float)(C & ~0xffu), cl = (float)(C & 0xffu);
    rem = fmaf(-q, kh, ch) + fmaf(-q, kl, cl);
  }
  return make_float2(q, rem * r);
}
__device__ __forceinline__ float2 sel_ratio(uint32_t C, uint32_t k) {
  return sel_ratio(C, k, __frcp_rn((float)k));
}

// body(key, label) for the scores i, i + 1, .. of [lo, hi) that this thread takes;
// vector loads when the pointers allow (lo is a multiple of 4)
template <typename F>
__device__ __forceinline__ void sel_each(const SelArgs& a, uint32_t lo, uint32_t hi, uint32_t first,
                                         uint32_t step, bool labels, F body) {
  const bool vec = ((reinterpret_cast<uintptr_t>(a.scores) |
                     reinterpret_cast<uintptr_t>(a.labels)) & 15u) == 0;
  auto one = [&](float s, uint32_t lab) {
    const uint32_t k = sel_key(s);
    if (k != SEL_NONFINITE) body(k, lab);
  };
  if (vec) {
#pragma unroll 4
    for (uint64_t i = (uint64_t)lo + 4ull * first; i + 3 < hi; i += 4ull * step) {
      const float4 f = *reinterpret_cast<const float4*>(a.scores + i);
      const uint32_t l = labels ? *reinterpret_cast<const uint32_t*>(a.labels + i) : 0u;
      one(f.x, (l & 0xffu) ? 1u : 0u);
      one(f.y, (l & 0xff00u) ? 1u : 0u);
      one(f.z, (l & 0xff0000u) ? 1u : 0u);
      one(f.w, (l & 0xff000000u) ? 1u : 0u);
    }
    const uint32_t rest = lo + ((hi - lo) & ~3u);
    if (rest + first < hi && first < 4u)
      one(a.scores[rest + first], labels && a.labels[rest + first] ? 1u : 0u);
  } else {
    for (uint64_t i = (uint64_t)lo + first; i < hi; i += step)
      one(a.scores[i], labels && a.labels[i] ? 1u : 0u);
  }
}

__global__ void __launch_bounds__(SB_NT) sel_coarse(const SelArgs a) {
  __shared__ uint32_t h[SB_BINS];
  pdl_enter(false);
  for (int i = threadIdx.x; i < SB_BINS; i += SB_NT) h[i] = 0u;
  __syncthreads();
  sel_each(a, 0u, a.n, blockIdx.x * SB_NT + threadIdx.x, gridDim.x * SB_NT, false,
           [&](uint32_t k, uint32_t) { atomicAdd(&h[k >> SB_SHIFT], 1u); });
  __syncthreads();
  for (int i = threadIdx.x; i < SB_BINS; i += SB_NT)
    if (h[i]) atomicAdd(a.coarse + i, h[i]);
}

// exclusive prefix of two counts over the CTA's threads (NT of them), and the totals
template <int NT>
__device__ __forceinline__ void sel_scan2(uint32_t& x, uint32_t& y, uint32_t& xall, uint32_t& yall,
                                          uint32_t (*ws)[NT / 32]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t ix = x, iy = y;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t xx = __shfl_up_sync(FULL, ix, o), yy = __shfl_up_sync(FULL, iy, o);
    if (lane >= o) {
      ix += xx;
      iy += yy;
    }
  }
  __syncthreads();  // ws may still be read from the scan before
  if (lane == 31) {
    ws[0][warp] = ix;
    ws[1][warp] = iy;
  }
  __syncthreads();
  uint32_t bx = 0, by = 0;
  xall = yall = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    if (w == warp) {
      bx = xall;
      by = yall;
    }
    xall += ws[0][w];
    yall += ws[1][w];
  }
  x = bx + ix - x;
  y = by + iy - y;
}

__global__ void __launch_bounds__(1024) sel_plan(const SelArgs a) {
  __shared__ uint32_t ws[2][32];
  pdl_enter(false);
  constexpr int PER = SB_BINS / 1024;
  uint32_t c[PER], b[PER], nb = 0, nf = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    c[j] = a.coarse[threadIdx.x * PER + j];
    b[j] = 0;
    while (b[j] < (uint32_t)SB_MAXB && (c[j] >> b[j]) > a.target) ++b[j];
    nb += c[j] ? 1u << b[j] : 0u;
    nf += c[j];
  }
  uint32_t at = nb, dummy = nf, nball, nfall;
  sel_scan2<1024>(at, dummy, nball, nfall, ws);
  if (threadIdx.x == 0) {
    a.info[0] = nball;
    a.info[1] = nfall;
  }
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    if (!c[j]) continue;
    const uint32_t bin = threadIdx.x * PER + j, r = SB_SHIFT - b[j];
    a.plan[bin] = at | b[j] << 16;
    for (uint32_t s = 0; s < 1u << b[j]; ++s)  // the low SB_VBITS bits of a first key are 0
      a.bkey[at + s] = bin << SB_SHIFT | s << r | r;
    at += 1u << b[j];
  }
}

// bucket of a key, and its offset there
__device__ __forceinline__ uint32_t sel_bucket_of(uint32_t key, const uint32_t* plan, uint32_t& off) {
  const uint32_t p = plan[key >> SB_SHIFT], r = SB_SHIFT - (p >> 16);
  off = key & ((1u << r) - 1u);
  return (p & 0xffffu) + ((key & ((1u << SB_SHIFT) - 1u)) >> r);
}

// share s: items and correct items per bucket, added to the buckets' totals
__global__ void __launch_bounds__(SB_NT, 2) sel_count(const SelArgs a) {
  extern __shared__ __align__(16) uint32_t sb_dyn[];  // [SB_BINS] plan, [buckets] counts
  uint32_t *plan = sb_dyn, *cnt = sb_dyn + SB_BINS;
  pdl_enter(false);
  const uint32_t nb = a.info[0];
  for (int i = threadIdx.x; i < SB_BINS; i += SB_NT) plan[i] = a.plan[i];
  for (uint32_t i = threadIdx.x; i < nb; i += SB_NT) cnt[i] = 0u;
  __syncthreads();
  const uint32_t lo = blockIdx.x * a.share, hi = min(a.n - lo, a.share) + lo;
  sel_each(a, lo, hi, threadIdx.x, SB_NT, a.labels != nullptr, [&](uint32_t k, uint32_t lab) {
    uint32_t off;
    atomicAdd(cnt + sel_bucket_of(k, plan, off), 1u + (lab << 16));
  });
  __syncthreads();
  uint32_t* rel = a.rel + (size_t)blockIdx.x * a.nbcap;
  for (uint32_t i = threadIdx.x; i < nb; i += SB_NT) {
    const uint32_t c = cnt[i];
    if (c)
      rel[i] = (uint32_t)atomicAdd(a.total + i, (unsigned long long)(c & 0xffffu) |
                                                    (unsigned long long)(c >> 16) << 32);
  }
}

// ascending rank of tau's item (the k-th largest finite score), and k
__device__ __forceinline__ uint32_t sel_tau_rank(const SelArgs& a, uint32_t nf, int64_t& k) {
  k = (int64_t)floor(a.q * (double)a.n + 0.5);
  k = k < 0 ? 0 : (k > (int64_t)nf ? (int64_t)nf : k);
  return nf - (uint32_t)k;
}

__global__ void __launch_bounds__(1024) sel_offsets(const SelArgs a) {
  __shared__ uint32_t ws[2][32], listed[2];
  pdl_enter(false);
  if (threadIdx.x < 2) listed[threadIdx.x] = 0u;  // (the scan synchronises)
  int64_t kk;
  const uint32_t itau = sel_tau_rank(a, a.info[1], kk);
  const uint32_t nb = a.info[0], per = (nb + 1023u) / 1024u, i0 = threadIdx.x * per;
  uint32_t x = 0, y = 0, xall, yall;
  for (uint32_t i = i0; i < min(i0 + per, nb); ++i) {
    const unsigned long long t = a.total[i];
    x += (uint32_t)t;
    y += (uint32_t)(t >> 32);
  }
  sel_scan2<1024>(x, y, xall, yall, ws);
  for (uint32_t i = i0; i < min(i0 + per, nb); ++i) {
    const unsigned long long t = a.total[i];
    a.start[i] = x;
    a.pstart[i] = y;
    // to be resolved by a CTA; without labels only tau's bucket counts
    if ((uint32_t)t > (uint32_t)SB_SMALL && (a.labels || (kk > 0 && itau - x < (uint32_t)t))) {
      if ((uint32_t)t > (uint32_t)SB_LIGHT) a.list[atomicAdd(listed, 1u)] = i;
      else a.list[a.nbcap - 1u - atomicAdd(listed + 1, 1u)] = i;
    }
    if ((uint32_t)t > (uint32_t)SB_HEAVY && (a.bkey[i] & 31u) == (uint32_t)SB_VBITS) {
      a.hidx[i] = atomicAdd(a.info + 4, 1u);
      const uint32_t chunks = ((uint32_t)t + SB_CHUNK - 1) / SB_CHUNK;
      const uint32_t at = atomicAdd(a.info + 5, chunks);
      for (uint32_t j = 0; j < chunks; ++j) a.hchunk[at + j] = make_uint2(i, j);
    }
    x += (uint32_t)t;
    y += (uint32_t)(t >> 32);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a.info[6] = listed[0];
    a.info[7] = listed[1];
    a.start[nb] = xall;
    a.pstart[nb] = yall;
    a.info[2] = yall;
  }
}

__global__ void __launch_bounds__(SB_NT, 2) sel_scatter(const SelArgs a) {
  extern __shared__ __align__(16) uint32_t sb_dyn[];  // [SB_BINS] plan, [buckets] next places
  uint32_t *plan = sb_dyn, *pos = sb_dyn + SB_BINS;
  pdl_enter(false);
  const uint32_t nb = a.info[0];
  const uint32_t* rel = a.rel + (size_t)blockIdx.x * a.nbcap;
  for (int i = threadIdx.x; i < SB_BINS; i += SB_NT) plan[i] = a.plan[i];
  // (a bucket that the share has no item of has no place; it is not used)
  for (uint32_t i = threadIdx.x; i < nb; i += SB_NT) pos[i] = a.start[i] + rel[i];
  const uint64_t hwords = (uint64_t)a.info[4] << SB_VBITS;  // the heavy buckets' counters
  for (uint64_t i = (uint64_t)blockIdx.x * SB_NT + threadIdx.x; i < hwords;
       i += (uint64_t)gridDim.x * SB_NT)
    a.hcnt[i] = 0ull;
  __syncthreads();
  const uint32_t lo = blockIdx.x * a.share, hi = min(a.n - lo, a.share) + lo;
  sel_each(a, lo, hi, threadIdx.x, SB_NT, a.labels != nullptr, [&](uint32_t k, uint32_t lab) {
    uint32_t off;
    const uint32_t b = sel_bucket_of(k, plan, off);
    a.items[atomicAdd(pos + b, 1u)] = off << 1 | lab;
  });
}

constexpr int SB_WORDS = 1 << SB_VBITS;  // the counters of sel_heavy and sel_bucket
constexpr size_t SB_BUCKET_SMEM = SB_WORDS * sizeof(uint32_t);

// The heavy buckets (scores piled up on few keys, as those of a confident
// scorer just below 1): their items counted chunk by chunk on all SMs
__global__ void __launch_bounds__(SB_NT, 3) sel_heavy(const SelArgs a) {
  extern __shared__ __align__(16) uint32_t sb_dyn[];
  pdl_enter(false);
  const uint32_t chunks = a.info[5];
  for (uint32_t q = blockIdx.x; q < chunks; q += gridDim.x) {
    const uint2 bc = a.hchunk[q];
    const uint32_t s0 = a.start[bc.x], m = a.start[bc.x + 1] - s0;
    const uint32_t lo = bc.y * SB_CHUNK, hi = min(lo + SB_CHUNK, m);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < (uint32_t)SB_WORDS; i += SB_NT) sb_dyn[i] = 0u;
    __syncthreads();
    for (uint32_t i = lo + threadIdx.x; i < hi; i += SB_NT) {
      const uint32_t it = a.items[s0 + i];
      atomicAdd(sb_dyn + (it >> 1), 1u + ((it & 1u) << 16));
    }
    __syncthreads();
    unsigned long long* out = a.hcnt + ((size_t)a.hidx[bc.x] << SB_VBITS);
    for (uint32_t w = threadIdx.x; w < 1u << SB_VBITS; w += SB_NT) {
      const uint32_t u = sb_dyn[w];
      if (u)
        atomicAdd(out + w, (unsigned long long)(u & 0xffffu) | (unsigned long long)(u >> 16) << 32);
    }
  }
}

// H(x + c) - H(x), the harmonic numbers' difference: summed up to 64, then by
// the asymptotic series of H (its next term is below 2e-17 there)
__device__ __forceinline__ double sel_harmonic(uint32_t x, uint32_t c) {
  double s = 0.0;
  while (x < 64u && c > 0u) {
    ++x;
    --c;
    s += 1.0 / (double)x;
  }
  if (c == 0u) return s;
  const double A = (double)x, N = A + (double)c;
  const double u = 1.0 / A, v = 1.0 / N;
  auto tail = [](double w) {  // 1/2n - 1/12n^2 + 1/120n^4 - 1/252n^6
    const double w2 = w * w;
    return w * 0.5 - w2 * (1.0 / 12.0 - w2 * (1.0 / 120.0 - w2 * (1.0 / 252.0)));
  };
  return s + (log1p((double)c * u) + (tail(v) - tail(u)));
}

// A thread's sums over tie groups
struct SelSums {
  float fs, fc;              // compensated float-float sum of AUARC terms
  double ds;                 // long groups
  unsigned long long roc2;   // twice the AUROC numerator
  __device__ __forceinline__ void add(float th, float tl) {
    const float u = fs + th;  // two-sum into the running pair (fs, fc)
    const float bv = u - fs;
    fc += ((fs - (u - bv)) + (th - bv)) + tl;
    fs = u;
  }
  // this lane's group (if `on`) of c items, p correct, with lo items and plo
  // correct ones below it; whole warp
  __device__ __forceinline__ void group(bool on, uint32_t lo, uint32_t plo, uint32_t c, uint32_t p,
                                        uint32_t nf, uint32_t ptot, int lane) {
    const uint32_t above = nf - lo - c, cab = ptot - plo - p;
    if (on) roc2 += (unsigned long long)p * (2u * (lo - plo) + (c - p));  // (below 2^32)
    // sum over j = 1 .. c of (cab + p j / c) / (above + j)
    const bool one = c == 1u, near = !one && (above >> 6 < c || c >> 23 != 0u);
    if (on && !near) {
      // one item: its ratio.  More: ranks M + d around their mean M = D / 2, D =
      // 2 above + c + 1, c / M < 2^-6, 1 / (M + d) expanded to d^4.  The leading term
      // (2 c cab + p (c + 1)) / D as float pairs; the correction (Cm / M - p / c)
      // (S2 / M^2 + S4 / M^4), S2 and S4 = sums of d^2 and d^4, Cm the mean of the
      // numerators, in fp32 without S4 for c / M < 2^-10, else in fp64.  Where the
      // answers above are as often correct as the group's, Cm / M and p / c cancel; the
      // worst case is no correct answer above: the correction is c / 6M of the sum,
      // in fp32 good to 2^-35.6 of it, S4 left out is 2^-35.3 of it, and in fp64 what
      // is left 2 (c / M)^5 / 448 < 2^-37.8.  So a group's sum is good to 2^-34 at the
      // least (measured 3.4e-11; rank by rank in float pairs it was 3.1e-8)
      const uint32_t D = one ? nf - lo : 2u * above + c + 1u;
      const float rD = __frcp_rn((float)D);
      const float2 t1 = sel_ratio(one ? ptot - plo : cab, D, rD);
      const float cf = (float)c, c2 = one ? 1.f : 2.f * cf;  // exact (c < 2^23)
      const float x = __fmul_rn(t1.x, c2), xl = fmaf(t1.x, c2, -x) + t1.y * c2;
      add(x, xl);
      if (!one) {
        const float2 t2 = sel_ratio(p, D, rD);
        const float c1 = cf + 1.f;
        const float y = __fmul_rn(t2.x, c1), yl = fmaf(t2.x, c1, -y) + t2.y * c1;
        const float r = 2.f * rD, lead = x + y;  // c Cm / M
        float corr = 0.f;
        if (above >> 10 >= c) {
          corr = cf * (cf * cf - 1.f) * (1.f / 12.f) * r * r * __fdividef(lead - (float)p, cf);
        } else {
          const double cd = (double)c, rd = (double)r, im = rd * (2.0 - 0.5 * (double)D * rd);
          const double im2 = im * im, cc = cd * cd, ri = (double)__frcp_rn(cf);
          const double w = (((double)x + (double)y) + ((double)xl + (double)yl)) - (double)p;
          ds += (cc - 1.0) * (1.0 / 12.0) * im2 * (1.0 + (3.0 * cc - 7.0) * 0.05 * im2) *
                (w * (cd * ri * (2.0 - cd * ri)));
        }
        add(y, yl + corr);
      }
    }
    // groups at the top ranks: long ones in closed form, of the others the warp
    // takes one by one, a lane every 32nd rank
    if (on && near && c >= (uint32_t)SB_LONG) {
      const double dh = sel_harmonic(above, c);
      ds += (double)cab * dh + ((double)p / (double)c) * ((double)c - (double)above * dh);
    }
    unsigned todo = __ballot_sync(FULL, on && near && c < (uint32_t)SB_LONG);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1u;
      ranks(__shfl_sync(FULL, above, src), __shfl_sync(FULL, cab, src), __shfl_sync(FULL, c, src),
            __shfl_sync(FULL, p, src), lane);
    }
  }
  __device__ __forceinline__ void ranks(uint32_t above, uint32_t cab, uint32_t c, uint32_t p,
                                        int lane) {
    // rank k = above + j: (correct answers above) / k + (j / c)(p / k) as
    // float-float ratios and one float-float product, the roundings carried
    for (uint32_t j = 1u + lane; j <= c; j += 32u) {
      const uint32_t k = above + j;
      const float2 t1 = sel_ratio(cab, k);
      const float2 u1 = sel_ratio(j, c), u2 = sel_ratio(p, k);
      const float pr = __fmul_rn(u1.x, u2.x);  // (not to be fused into the sum below)
      const float pl = fmaf(u1.x, u2.x, -pr) + fmaf(u1.x, u2.y, u1.y * u2.x);
      const float th = t1.x + pr;  // two-sum of the high parts
      const float bv = th - t1.x;
      add(th, ((t1.x - (th - bv)) + (pr - bv)) + (t1.y + pl));
    }
  }
};

// word of sub-bin w: one word of padding per 32, so that the runs of 8 that
// threads scan lie in different banks
__device__ __forceinline__ uint32_t sel_at(uint32_t w) { return w + (w >> 5); }
static_assert(SB_SMALL < 256 && 3 * SB_SMALL * SB_NT / 32 <= SB_WORDS, "three arrays per warp");
static_assert(2 * SB_LIGHT + SB_RADIX + SB_RADIX / 32 <= SB_WORDS,
              "a light bucket, its label prefix and the sub-bins");
static_assert(2 * SB_LIGHT + SB_RADIX + SB_RADIX / 32 + SB_RADIX / 2 <= SB_WORDS,
              "and the sub-bins' prefix counts in 16 bits");
static_assert(SB_SHIFT - 12 <= 8, "at most 256 keys in a sub-bin");
static_assert(1 << SB_VBITS == 32 * SB_NT, "a strip of 32 keys per thread");
static_assert(SB_RADIX == 8 * SB_NT && SB_LIGHT == 8 * SB_NT, "eight per thread");

// LARGE: for pools in which buckets of more than SB_LIGHT items over more keys than
// are counted at once are the rule, not the exception (target above SB_LIGHT, from
// 3.4e7 scores on).  Apart, as its registers would cost the other pools 3%.
template <bool LARGE>
__global__ void __launch_bounds__(SB_NT, 3) sel_bucket(const SelArgs a) {
  extern __shared__ __align__(16) uint32_t sb_dyn[];
  __shared__ uint32_t ws[2][SB_NT / 32], next, ranges[4], strip[2][SB_NT];
  __shared__ double sd[SB_NT / 32];
  __shared__ unsigned long long su[SB_NT / 32];
  pdl_enter(false);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t nb = a.info[0], nf = a.info[1], ptot = a.info[2];
  int64_t kk;
  const uint32_t itau = sel_tau_rank(a, nf, kk);
  const bool metrics = a.labels != nullptr;
  // a warp's group of keys at key0 + off; every lane of the warp calls
  auto visit = [&](SelSums& S, bool has_tau, uint32_t key, uint32_t lo, uint32_t plo, uint32_t c,
                   uint32_t p) {
    if (metrics) S.group(c != 0u, lo, plo, c, p, nf, ptot, lane);
    if (has_tau && itau - lo < c) {
      a.out->tau = sel_unkey(key);
      a.out->n_ship = (int64_t)(nf - lo);
      a.out->acc_shipped = metrics ? (double)(ptot - plo) / (double)(nf - lo)
                                   : __longlong_as_double(0x7ff8000000000000ll);
    }
  };
  // ---- buckets of a few items (those of a pool spread over many coarse bins), a
  // warp each: a lane counts the items below and equal to its own, and the first of
  // each group leaves it at its rank, so that the sums' order is the groups' and not
  // that in which the items came
  uint32_t* mine = sb_dyn + warp * 3 * SB_SMALL;
  uint32_t *goff = mine + SB_SMALL, *gcnt = goff + SB_SMALL;  // c | p << 8 | correct below << 16
  for (uint32_t b = blockIdx.x * (SB_NT / 32) + warp; b < nb; b += gridDim.x * (SB_NT / 32)) {
    const uint32_t s0 = a.start[b], m = a.start[b + 1] - s0, p0 = a.pstart[b];
    const bool has_tau = kk > 0 && itau - s0 < m;
    if (m > (uint32_t)SB_SMALL || !(metrics || has_tau)) continue;
    SelSums S = {0.f, 0.f, 0.0, 0ull};
    __syncwarp();
    for (uint32_t i = lane; i < ((m + 3u) & ~3u); i += 32u) {
      mine[i] = i < m ? a.items[s0 + i] : ~0u;  // no item's offset
      gcnt[i] = 0u;
    }
    __syncwarp();
    for (uint32_t base = 0; base < m; base += 32u) {
      const uint32_t i = base + lane, v = i < m ? mine[i] : ~0u, key = v & ~1u;
      uint32_t below = 0u, same = 0u, first = i;  // items | correct << 16
#pragma unroll 2
      for (uint32_t j = 0; j < m; j += 4u) {
        const uint4 q = *reinterpret_cast<const uint4*>(mine + j);
        const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (uint32_t e = 0; e < 4u; ++e) {
          const uint32_t add = 1u | (u[e] & 1u) << 16;
          if (u[e] < key) below += add;
          if ((u[e] ^ v) < 2u) {
            same += add;
            first = min(first, j + e);
          }
        }
      }
      if (i < m && first == i) {
        goff[below & 0xffffu] = v >> 1;
        gcnt[below & 0xffffu] = (same & 0xffffu) | (same >> 16) << 8 | (below >> 16) << 16;
      }
    }
    __syncwarp();
    for (uint32_t base = 0; base < m; base += 32u) {
      const uint32_t i = base + lane, g = i < m ? gcnt[i] : 0u;
      visit(S, has_tau, (a.bkey[b] & ~31u) + (g ? goff[i] : 0u), s0 + i, p0 + (g >> 16), g & 0xffu,
            (g >> 8) & 0xffu);
    }
    double d = ((double)S.fs + (double)S.fc) + S.ds;
    unsigned long long u = S.roc2;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      d += __shfl_xor_sync(FULL, d, o);
      u += __shfl_xor_sync(FULL, u, o);
    }
    if (lane == 0) {
      a.parc[b] = d;
      a.proc[b] = u;
    }
  }
  // ---- the others, the crowded ones first, a CTA each
  const uint32_t crowds = a.info[6], listed = crowds + a.info[7];
  for (;;) {
    __syncthreads();
    if (tid == 0) next = atomicAdd(a.info + 3, 1u);
    __syncthreads();
    if (next >= listed) return;
    const uint32_t b = a.list[next < crowds ? next : a.nbcap - 1u - (next - crowds)];
    const uint32_t s0 = a.start[b], m = a.start[b + 1] - s0, p0 = a.pstart[b];
    const bool has_tau = kk > 0 && itau - s0 < m;
    const uint32_t bk = a.bkey[b], r = bk & 31u, key0 = bk & ~31u;
    const uint32_t* items = a.items + s0;
    SelSums S = {0.f, 0.f, 0.0, 0ull};
    // the groups of `vals` consecutive keys from key0 + first on, with a0 items and
    // q0 correct ones below; count(w, c, p) gives key w's.  The keys go by strips
    // of 32, a lane per key, to the warps in turn: long tie groups come in
    // neighbouring keys, and all warps share them.  `small`: the counts are the
    // 16-bit halves of sb_dyn's words.  Returns the totals.
    auto walk = [&](uint32_t first, uint32_t vals, uint32_t a0, uint32_t q0, bool small, auto count,
                    uint32_t& xall, uint32_t& yall) {
      const uint32_t strips = vals / 32u;  // at most one per thread
      if (small)  // four strips at a time, both counts in one sum
        for (uint32_t s = 4u * warp; s < strips; s += SB_NT / 8) {
          const uint4 u = *reinterpret_cast<const uint4*>(sb_dyn + 32u * s + 4u * lane);
          uint32_t c = (u.x + u.y) + (u.z + u.w);
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) c += __shfl_xor_sync(FULL, c, o);
          if ((lane & 7) == 0) {
            strip[0][s + (lane >> 3)] = c & 0xffffu;
            strip[1][s + (lane >> 3)] = c >> 16;
          }
        }
      else
        for (uint32_t s = warp; s < strips; s += SB_NT / 32) {
          uint32_t c, p;
          count(32u * s + lane, c, p);
          c = __reduce_add_sync(FULL, c);
          p = __reduce_add_sync(FULL, p);
          if (lane == 0) {
            strip[0][s] = c;
            strip[1][s] = p;
          }
        }
      __syncthreads();
      uint32_t x = (uint32_t)tid < strips ? strip[0][tid] : 0u,
               y = (uint32_t)tid < strips ? strip[1][tid] : 0u;
      sel_scan2<SB_NT>(x, y, xall, yall, ws);
      strip[0][tid] = x;
      strip[1][tid] = y;
      __syncthreads();
      for (uint32_t s = warp; s < strips; s += SB_NT / 32) {
        uint32_t c, p;
        count(32u * s + lane, c, p);
        if (!__any_sync(FULL, c != 0u)) continue;
        uint32_t ic = small ? c | p << 16 : c, ip = p;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t cc = __shfl_up_sync(FULL, ic, o);
          if (lane >= o) ic += cc;
        }
        if (small) {
          ip = ic >> 16;
          ic &= 0xffffu;
        } else {
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t pp = __shfl_up_sync(FULL, ip, o);
            if (lane >= o) ip += pp;
          }
        }
        visit(S, has_tau, key0 + first + 32u * s + lane, a0 + strip[0][s] + ic - c, q0 + strip[1][s] + ip - p, c, p);
      }
    };
    // ---- up to SB_LIGHT items it[] (e * SB_NT + tid: offset from `base` << 1 | label;
    // offsets below 2^(sh + 12)), a0 items and q0 correct ones below them: sorted,
    // then a group per run of equal offsets.  The items go to sub-bins of the
    // offset's leading bits (about one item in each), a thread sorts each sub-bin;
    // piled-up offsets take a bitonic sort of the whole.  Returns the correct ones.
    auto light = [&](uint32_t (&it)[8], uint32_t m, uint32_t sh, uint32_t base, uint32_t a0,
                     uint32_t q0) -> uint32_t {
      uint32_t *v = sb_dyn, *pre = sb_dyn + SB_LIGHT, *sub = pre + SB_LIGHT;
      for (uint32_t i = tid; i < SB_RADIX + SB_RADIX / 32; i += SB_NT) sub[i] = 0u;
      __syncthreads();
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (e * SB_NT + tid < m) atomicAdd(sub + sel_at(it[e] >> 1 >> sh), 1u);
      __syncthreads();
      uint32_t c8[8], sx = 0, sy = 0, sxall, syall;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        c8[e] = sub[sel_at(8 * tid + e)];
        sx += c8[e];
      }
      sel_scan2<SB_NT>(sx, sy, sxall, syall, ws);
      bool crowded = false;
      uint32_t at8 = sx;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        sub[sel_at(8 * tid + e)] = at8;
        at8 += c8[e];
        crowded = crowded || c8[e] > (uint32_t)SB_RUN;
      }
      uint32_t n2 = SB_NT;
      while (n2 < m) n2 <<= 1;
      if (!__syncthreads_or(crowded)) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (e * SB_NT + tid < m) v[atomicAdd(sub + sel_at(it[e] >> 1 >> sh), 1u)] = it[e];
        __syncthreads();
        at8 = sx;
#pragma unroll 1
        for (int e = 0; e < 8; ++e) {
          for (uint32_t i = at8 + 1; i < at8 + c8[e]; ++i) {  // insertion sort
            const uint32_t x = v[i];
            uint32_t j = i;
            for (; j > at8 && v[j - 1] > x; --j) v[j] = v[j - 1];
            v[j] = x;
          }
          at8 += c8[e];
        }
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (e * SB_NT + tid < n2) v[e * SB_NT + tid] = it[e];  // ~0 past the items
        for (uint32_t k = 2; k <= n2; k <<= 1)
          for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            __syncthreads();
            for (uint32_t q = tid; q < n2 >> 1; q += SB_NT) {
              const uint32_t i = ((q & ~(j - 1u)) << 1) | (q & (j - 1u)), l = i + j;
              const uint32_t x = v[i], y = v[l];
              if ((x > y) == ((i & k) == 0u)) {
                v[i] = y;
                v[l] = x;
              }
            }
          }
      }
      __syncthreads();
      const uint32_t per = n2 / SB_NT, i0 = tid * per;
      uint32_t x = 0, y = 0, xall, yall;
      for (uint32_t i = i0; i < min(i0 + per, m); ++i) x += v[i] & 1u;
      sel_scan2<SB_NT>(x, y, xall, yall, ws);
      for (uint32_t i = i0; i < min(i0 + per, m); ++i) {
        pre[i] = x;  // correct items before item i
        x += v[i] & 1u;
      }
      __syncthreads();
      for (uint32_t i0 = 0; i0 < m; i0 += SB_NT) {
        const uint32_t i = i0 + tid;
        uint32_t off = 0u, pi = 0u, c = 0u, p = 0u;
        if (i < m) {
          off = v[i] >> 1;
          pi = pre[i];
          if (i == 0 || v[i - 1] >> 1 != off) {
            uint32_t e = i + 1, hi = m;  // the group's end
            if (e < m && v[e] >> 1 == off) {
              while (e < hi) {
                const uint32_t mid = (e + hi) >> 1;
                if (v[mid] >> 1 <= off) e = mid + 1;
                else hi = mid;
              }
            }
            c = e - i;
            p = (e < m ? pre[e] : xall) - pi;
          }
        }
        visit(S, has_tau, key0 + base + off, a0 + i, q0 + pi, c, p);
      }
      return xall;
    };
    if (m <= (uint32_t)SB_LIGHT) {
      uint32_t it[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) it[e] = e * SB_NT + tid < m ? items[e * SB_NT + tid] : ~0u;
      light(it, m, r - 12u, 0u, s0, p0);  // 2^r keys, SB_RADIX = 2^12 sub-bins
    } else if (m > (uint32_t)SB_HEAVY && r == (uint32_t)SB_VBITS) {
      // ---- a heavy bucket: already counted (sel_heavy)
      const unsigned long long* hc = a.hcnt + ((size_t)a.hidx[b] << SB_VBITS);
      uint32_t xall, yall;
      walk(0u, 1u << SB_VBITS, s0, p0, false, [&](uint32_t w, uint32_t& c, uint32_t& p) {
        const unsigned long long u = __ldcg(hc + w);
        c = (uint32_t)u;
        p = (uint32_t)(u >> 32);
      }, xall, yall);
    } else {
      // ---- counted: 2^14 keys at a time (16-bit counts of items and labels), or
      // 2^13 with 32-bit counts for a bucket of more items than 16 bits hold
      const bool wide = m > (uint32_t)SB_HEAVY;
      const int vb = wide ? SB_VBITS - 1 : SB_VBITS;
      const uint32_t vals = 1u << vb;
      uint32_t* lab = sb_dyn + vals;  // wide only
      uint32_t a0 = s0, q0 = p0;
      // which of the (up to 128) key ranges hold items: piled-up scores fill few
      uint32_t used[4] = {r == (uint32_t)vb ? 1u : 0u, 0u, 0u, 0u};
      for (uint32_t i = r == (uint32_t)vb ? m : tid; i < m; i += SB_NT) {
        const uint32_t ps = items[i] >> 1 >> vb;
#pragma unroll
        for (int e = 0; e < 4; ++e) used[e] |= ps >> 5 == (uint32_t)e ? 1u << (ps & 31u) : 0u;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) used[e] = __reduce_or_sync(FULL, used[e]);
      if (tid < 4) ranges[tid] = 0u;
      __syncthreads();
      if (lane < 4)
        atomicOr(ranges + lane, lane == 0 ? used[0] : lane == 1 ? used[1] : lane == 2 ? used[2] : used[3]);
      __syncthreads();
      uint32_t ps = 0u;  // first range
      const uint32_t filled =
          LARGE ? __popc(ranges[0]) + __popc(ranges[1]) + __popc(ranges[2]) + __popc(ranges[3]) : 0u;
      if (LARGE && !wide && filled > m / 2048u + 2u) {
        // spread over more ranges than it takes chunks of up to SB_LIGHT items (a pool
        // of tens of millions over many coarse bins; 4e7 random bit patterns 7.3 ms
        // range by range, 1.36 now): chunk by chunk, whole sub-bins of the offset's 12
        // leading bits, their prefix counts in 16 bits behind what `light` uses
        uint16_t* pre16 = reinterpret_cast<uint16_t*>(sb_dyn + SB_WORDS - SB_RADIX / 2);
        const uint32_t sb = r - 12u;  // bits of a sub-bin
        for (uint32_t i = tid; i < SB_RADIX; i += SB_NT) sb_dyn[i] = 0u;
        __syncthreads();
        for (uint32_t i = tid; i < m; i += SB_NT) atomicAdd(sb_dyn + (items[i] >> 1 >> sb), 1u);
        __syncthreads();
        uint32_t c8[8], x = 0, y = 0, xall, yall;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          c8[e] = sb_dyn[8 * tid + e];
          x += c8[e];
        }
        sel_scan2<SB_NT>(x, y, xall, yall, ws);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          pre16[8 * tid + e] = (uint16_t)x;
          x += c8[e];
        }
        auto before = [&](uint32_t sub) { return sub < (uint32_t)SB_RADIX ? (uint32_t)pre16[sub] : m; };
        for (uint32_t b0 = 0; b0 < (uint32_t)SB_RADIX;) {
          __syncthreads();
          const uint32_t i0 = before(b0);
          if (i0 == m) break;
          uint32_t b1 = b0, step = SB_RADIX;  // the most sub-bins of up to SB_LIGHT items
          for (; step; step >>= 1)
            if (b1 + step <= (uint32_t)SB_RADIX && before(b1 + step) - i0 <= (uint32_t)SB_LIGHT)
              b1 += step;
          const bool dense = b1 == b0;  // more of them in one sub-bin (at most 256 keys)
          if (dense) ++b1;
          const uint32_t n = before(b1) - i0, low = b0 << sb;
          if (tid == 0) ranges[0] = 0u;
          if (dense)
            for (uint32_t i = tid; i < 256u; i += SB_NT) sb_dyn[i] = 0u;
          __syncthreads();
          for (uint32_t i = tid; i < m; i += SB_NT) {
            const uint32_t it = items[i], off = it >> 1, sub = off >> sb;
            if (sub < b0 || sub >= b1) continue;
            if (dense) atomicAdd(sb_dyn + (off - low), 1u + ((it & 1u) << 16));
            else sb_dyn[atomicAdd(ranges, 1u)] = it - (low << 1);
          }
          __syncthreads();
          if (dense) {
            walk(low, 256u, a0, q0, true, [&](uint32_t w, uint32_t& c, uint32_t& p) {
              c = sb_dyn[w] & 0xffffu;
              p = sb_dyn[w] >> 16;
            }, xall, yall);
            q0 += yall;
          } else {
            uint32_t it[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) it[e] = e * SB_NT + tid < n ? sb_dyn[e * SB_NT + tid] : ~0u;
            __syncthreads();
            const int bits = 32 - __clz(((b1 - b0) << sb) - 1u);  // offsets below 2^bits
            q0 += light(it, n, (uint32_t)max(bits - 12, 0), low, a0, q0);
          }
          a0 += n;
          b0 = b1;
        }
        ps = 1u << (r - vb);
      }
      for (; ps < 1u << (r - vb); ++ps) {
        if (!(ranges[ps >> 5] >> (ps & 31u) & 1u)) continue;
        __syncthreads();
        for (uint32_t i = tid; i < (uint32_t)SB_WORDS; i += SB_NT) sb_dyn[i] = 0u;
        __syncthreads();
        for (uint32_t i = tid; i < m; i += SB_NT) {
          const uint32_t it = items[i], off = it >> 1;
          if (off >> vb != ps) continue;
          const uint32_t at = off & (vals - 1u);
          if (!wide) {
            atomicAdd(sb_dyn + at, 1u + ((it & 1u) << 16));
          } else {
            atomicAdd(sb_dyn + at, 1u);
            if (it & 1u) atomicAdd(lab + at, 1u);
          }
        }
        __syncthreads();
        uint32_t xall, yall;
        walk(ps << vb, vals, a0, q0, !wide, [&](uint32_t w, uint32_t& c, uint32_t& p) {
          const uint32_t u = sb_dyn[w];
          c = wide ? u : u & 0xffffu;
          p = wide ? lab[w] : u >> 16;
        }, xall, yall);
        a0 += xall;
        q0 += yall;
      }
    }
    // the bucket's sums, in a fixed order
    double d = ((double)S.fs + (double)S.fc) + S.ds;
    unsigned long long u = S.roc2;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      d += __shfl_xor_sync(FULL, d, o);
      u += __shfl_xor_sync(FULL, u, o);
    }
    if (lane == 0) {
      sd[warp] = d;
      su[warp] = u;
    }
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < SB_NT / 32; ++w) {
        d += sd[w];
        u += su[w];
      }
      a.parc[b] = d;
      a.proc[b] = u;
    }
  }
}

// One CTA: the buckets' sums in a fixed order, and the counts.
__global__ void __launch_bounds__(SB_NT) sel_finish(const SelArgs a) {
  __shared__ double sd[SB_NT];
  __shared__ unsigned long long su[SB_NT];
  pdl_enter(false);
  const int tid = threadIdx.x;
  const uint32_t nb = a.info[0], nf = a.info[1];
  double arc = 0.0;
  unsigned long long roc2 = 0;
  if (a.labels)
    for (uint32_t t = tid; t < nb; t += SB_NT) {  // each thread in bucket order
      arc += a.parc[t];
      roc2 += a.proc[t];
    }
  sd[tid] = arc;
  su[tid] = roc2;
  __syncthreads();
  for (int h = SB_NT / 2; h > 0; h >>= 1) {
    if (tid < h) {
      sd[tid] += sd[tid + h];
      su[tid] += su[tid + h];
    }
    __syncthreads();
  }
  if (tid != 0) return;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  SelResult* out = a.out;
  int64_t k;
  sel_tau_rank(a, nf, k);
  out->pad = 0;
  out->n_finite = nf;
  out->k = k;
  const int64_t P = a.labels ? (int64_t)a.info[2] : 0, N = (int64_t)nf - P;
  out->n_pos = P;
  if (k == 0) {
    out->tau = __int_as_float(0x7f800000);  // +inf: nothing ships
    out->n_ship = 0;
    out->acc_shipped = nan;
  }
  out->auroc = (a.labels && P > 0 && N > 0) ? (double)su[0] / (2.0 * (double)P * (double)N) : nan;
  out->auarc = (a.labels && nf > 0) ? sd[0] / (double)nf : nan;
}

}  // namespace prk
