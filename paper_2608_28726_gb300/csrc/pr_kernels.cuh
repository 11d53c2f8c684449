// Kernels of the verifier data path: the row kernels (Eq. 3 features, with a
// fused pooling / scoring / ship-rule epilogue in route and decode modes) and
// the standalone pooling kernel.  Algorithm notes are in pr_device.cuh.
//   verify_rows_ws  persistent, warp-specialised: one CTA streams one row at a
//                   time (used whenever a row needs no split)
//   verify_rows     one thread-block cluster of C CTAs per row (C = 2, 4, 8:
//                   batches too small to fill the GPU, e.g. decode steps)
#pragma once

#include "pr_device.cuh"

namespace prk {

// A scattered 16-byte re-read of a row already streamed: without the 256-byte
// L2 prefetch of ld_stream, a load that misses L2 fetches one 32-byte sector
// from DRAM instead of a 256-byte block.
__device__ __forceinline__ uint4 ld_reread(const void* p) {
  uint4 r;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// ---- pooling, scoring, ship rule (Section 3.1) -------------------------------------

template <int N>
struct Const {
  static constexpr int value = N;
};

struct Pooled {
  float agg[NAGG];
  float score;
  uint8_t ship;
  uint32_t flags;
};

// Warp-parallel pool of rows [lo, hi) of a [rows][8] feature array.  Lane j
// sums rows lo + j, lo + j + 32, ... in order, then a fixed butterfly combines
// the lanes, so the result depends only on T.  All lanes return the result.
// AHEAD rows of a lane are loaded at once: 4 where registers are short (the row
// kernels' epilogue), more where a long request's latency counts (4 all the same in
// a request of up to 128 rows: the loads past its end take issue slots).
template <int AHEAD>
__device__ __forceinline__ Pooled pool_rows(const float* feat, const uint32_t* flags, int64_t lo,
                                            int64_t hi, const float* w, float b, float zthr,
                                            int lane) {
  float s[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  float mn[5] = {INFINITY, INFINITY, INFINITY, INFINITY, INFINITY};
  uint32_t fl = 0;
  auto add = [&](const float4& a, float h, uint32_t rf) {
    const float v[5] = {a.x, a.y, a.z, -a.w, h};  // l, m, margin, -H, h
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      s[f] += v[f];
      mn[f] = fminf(mn[f], v[f]);
    }
    fl |= rf;
  };
  int64_t i = lo + lane;
  // the last fewer than N rows of a lane
  auto rest = [&](auto n) {
    constexpr int N = decltype(n)::value;
    if (i >= hi) return;
    float4 a[N];
    float h[N];
    uint32_t rf[N];
#pragma unroll
    for (int k = 0; k < N; ++k)
      if (i + 32 * k < hi) {
        a[k] = __ldcg(reinterpret_cast<const float4*>(feat + (i + 32 * k) * NFEAT));
        h[k] = __ldcg(feat + (i + 32 * k) * NFEAT + 4);
        rf[k] = flags ? __ldcg(flags + i + 32 * k) : 0u;
      }
#pragma unroll
    for (int k = 0; k < N; ++k)
      if (i + 32 * k < hi) add(a[k], h[k], rf[k]);
  };
  for (; i + 32 * (AHEAD - 1) < hi; i += 32 * AHEAD) {
    float4 a[AHEAD];
    float h[AHEAD];
    uint32_t rf[AHEAD];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
      a[k] = __ldcg(reinterpret_cast<const float4*>(feat + (i + 32 * k) * NFEAT));
      h[k] = __ldcg(feat + (i + 32 * k) * NFEAT + 4);
      rf[k] = flags ? __ldcg(flags + i + 32 * k) : 0u;
    }
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) add(a[k], h[k], rf[k]);
  }
  if (AHEAD > 4 && hi - lo <= 128) rest(Const<4>());
  else rest(Const<AHEAD>());
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      s[f] += __shfl_xor_sync(FULL, s[f], o);
      mn[f] = fminf(mn[f], __shfl_xor_sync(FULL, mn[f], o));
    }
    fl |= __shfl_xor_sync(FULL, fl, o);
  }
  Pooled p;
  const int64_t T = hi - lo;
  p.flags = fl;
  if (fl & (FLAG_NONFINITE | FLAG_BAD_CHOSEN)) {
#pragma unroll
    for (int j = 0; j < NAGG; ++j) p.agg[j] = NAN;
    p.score = NAN;
    p.ship = 0;
    return p;
  }
  const float Tf = (float)T;
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    p.agg[2 * f] = s[f] / Tf;
    p.agg[2 * f + 1] = mn[f];
  }
  p.agg[10] = (float)(T + 1) / (float)(2 * T);  // mean of t/T over t = 1..T
  float z = b;
#pragma unroll
  for (int j = 0; j < NAGG; ++j) z = fmaf(w[j], p.agg[j], z);
  p.score = 1.f / (1.f + expf(-z));
  p.ship = (z >= zthr) ? 1 : 0;
  return p;
}

__device__ __forceinline__ void write_pooled(const Pooled& p, int64_t r, float* agg, float* score,
                                             uint8_t* ship, uint32_t* req_flags, int lane) {
  if (agg && lane < NAGG) {
    float v = p.agg[0];
#pragma unroll
    for (int j = 1; j < NAGG; ++j)
      if (lane == j) v = p.agg[j];
    agg[r * NAGG + lane] = v;
  }
  if (lane == 0) {
    score[r] = p.score;
    ship[r] = p.ship;
    req_flags[r] = p.flags;
  }
}

__device__ __forceinline__ void write_special(int64_t r, float sc, uint32_t fl, float* agg,
                                              float* score, uint8_t* ship, uint32_t* req_flags) {
  if (agg)
    for (int j = 0; j < NAGG; ++j) agg[r * NAGG + j] = NAN;
  score[r] = sc;
  ship[r] = 0;
  req_flags[r] = fl;
}

// Request that owns global row gr: the r with offsets[r] <= gr < offsets[r+1],
// by a 32-way search (two dependent loads for up to 1,024 requests).
// Returns -1 when the offsets are inconsistent with gr.  Whole warp.
__device__ __forceinline__ int32_t find_request(const int64_t* off, int32_t n_req, int64_t gr,
                                                int lane) {
  if (n_req <= 0) return -1;
  int64_t lo = 0, hi = n_req - 1;  // answer: largest r in [lo, hi] with off[r] <= gr
  while (hi > lo) {
    const int64_t step = (hi - lo + 32) / 32;
    const int64_t pos = lo + (int64_t)lane * step;
    const bool ok = pos <= hi && off[pos] <= gr;
    const unsigned bal = __ballot_sync(FULL, ok);
    if (bal == 0) return -1;
    const int L = 31 - __clz(bal);
    lo = lo + (int64_t)L * step;
    hi = min(hi, lo + step - 1);
  }
  const int64_t a = off[lo], c = off[lo + 1];
  return (a <= gr && gr < c) ? (int32_t)lo : -1;
}

// Route mode: whether request r's rows [lo, hi) are inconsistent with the
// batch.  A whole-batch call also needs the last request to end at the last row.
__device__ __forceinline__ bool route_bad_request(const Args& a, int64_t r, int64_t lo,
                                                  int64_t hi) {
  return lo < 0 || hi < lo || hi > a.max_rows ||
         (a.whole && r == (int64_t)a.n_req - 1 && hi != a.max_rows);
}

// Route mode: the results of empty requests touching this launch's row range
// and of requests whose offsets are inconsistent (requests start, start +
// stride, ...).  Written by every launch; idempotent.
__device__ __forceinline__ void route_special_requests(const Args& a, int64_t start,
                                                       int64_t stride) {
  for (int64_t r = start; r < a.n_req; r += stride) {
    const int64_t lo = a.offsets[r], hi = a.offsets[r + 1];
    if (route_bad_request(a, r, lo, hi)) {
      write_special(r, NAN, FLAG_BAD_OFFSETS, a.agg, a.score, a.ship, a.req_flags);
      atomicOr(a.ctx_flags, FLAG_BAD_OFFSETS);
    } else if (lo == hi && lo >= a.row_base && lo <= a.row_base + a.n_rows) {
      write_special(r, 0.f, FLAG_EMPTY_REQ, a.agg, a.score, a.ship, a.req_flags);
    }
  }
}


// ---- cluster helpers ------------------------------------------------------------------

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// the same in two halves; no memory is handed over between them
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t dsmem_addr(const void* p, uint32_t rank) {
  uint32_t local = (uint32_t)__cvta_generic_to_shared(p), remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
  return remote;
}
__device__ __forceinline__ void dsmem_st_u32(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dsmem_st_u64(uint32_t a, uint64_t v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

// ---- block reduction of the (m, S, U, bad) state ------------------------------------

__device__ __forceinline__ void block_reduce_state(Smem& sm, float& m, float& S, float& U,
                                                   bool& bad, int warp, int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float mo = __shfl_xor_sync(FULL, m, o);
    const float So = __shfl_xor_sync(FULL, S, o);
    const float Uo = __shfl_xor_sync(FULL, U, o);
    lse_merge(m, S, U, mo, So, Uo);
  }
  bad = __any_sync(FULL, bad);
  if (lane == 0) {
    sm.pm[warp] = m;
    sm.pS[warp] = S;
    sm.pU[warp] = U;
    sm.pbad[warp] = bad;
  }
  __syncthreads();
  if (warp == 0) {
    m = lane < NWARP ? sm.pm[lane] : M2_INIT;
    S = lane < NWARP ? sm.pS[lane] : 0.f;
    U = lane < NWARP ? sm.pU[lane] : 0.f;
    bad = lane < NWARP ? (sm.pbad[lane] != 0) : false;
#pragma unroll
    for (int o = NWARP / 2; o > 0; o >>= 1) {
      const float mo = __shfl_xor_sync(FULL, m, o);
      const float So = __shfl_xor_sync(FULL, S, o);
      const float Uo = __shfl_xor_sync(FULL, U, o);
      lse_merge(m, S, U, mo, So, Uo);
    }
    bad = __any_sync(FULL, bad);
    // only lanes 0..NWARP-1 took part in the last butterfly: give every lane the total
    m = __shfl_sync(FULL, m, 0);
    S = __shfl_sync(FULL, S, 0);
    U = __shfl_sync(FULL, U, 0);
  }
}

// ---- row geometry -----------------------------------------------------------------------
//
// A row is cut into 16-byte groups of VEC elements from its first element on; the
// nedge < VEC elements after the last full group are read one by one by the
// lanes of a warp.  A tile is TILE groups, of which warp w of a CTA takes the
// UNR x 32 consecutive ones from 32 UNR w on, lane l the groups 32 k + l (2 KB in
// a row per warp: 3,214 rows of V = 262,144 fp32 take 506 us, 520 us with the
// warps' loads interleaved).
struct RowGeom {
  int32_t gfull, nedge;       // full groups, elements after them
  int32_t nfull, rem, ntiles; // tiles of TILE groups: full ones, groups of the last, all
  __device__ __forceinline__ RowGeom(int64_t V, int vec) {
    gfull = (int32_t)(V / vec);
    nedge = (int32_t)(V - (int64_t)gfull * vec);
    nfull = gfull / TILE;
    rem = gfull - nfull * TILE;
    ntiles = nfull + (rem > 0 ? 1 : 0);
  }
};
// index in its tile of thread tid's group k
__device__ __forceinline__ int32_t tile_pos(int tid, int k) {
  return (tid >> 5) * (32 * UNR) + 32 * k + (tid & 31);
}

// Rows that start off the 16-byte grid (rows of an odd vocabulary stored side
// by side): a group starts s bytes (a multiple of the element size) into a
// 16-byte word of the grid and is read with the widest aligned loads that cover
// it, two or three; a bf16 group that starts inside a 4-byte word takes five such
// words (the fifth in x) and cut_groups shifts them into place.  Loads that
// share a sector meet in L1.  The groups, and with them every sum, are those of
// an aligned row.  (The split kernel's way; the persistent kernel has a ring, see
// RingWS.)  350 rows of V = 70,001 bf16: 20.3 us per launch in a CUDA graph, 27.3
// with every group loaded by its elements.
__device__ __forceinline__ uint32_t ld_l1_32(const char* p) {
  uint32_t r;
  asm volatile("ld.global.L2::256B.u32 %0, [%1];" : "=r"(r) : "l"(p));
  return r;
}
__device__ __forceinline__ void ld_l1_64(const char* p, uint32_t& x, uint32_t& y) {
  asm volatile("ld.global.L2::256B.v2.u32 {%0,%1}, [%2];" : "=r"(x), "=r"(y) : "l"(p));
}
__device__ __forceinline__ void ld_l1_128(const char* p, uint32_t& x, uint32_t& y, uint32_t& z,
                                          uint32_t& w) {
  asm volatile("ld.global.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(x), "=r"(y), "=r"(z), "=r"(w)
               : "l"(p));
}
// the group S bytes into the grid word at p
template <int S>
__device__ __forceinline__ void ld_group(const char* p, uint4& w, uint32_t& x) {
  uint32_t unused;
  if (S == 0) {
    ld_l1_128(p, w.x, w.y, w.z, w.w);
  } else if (S == 2) {
    ld_l1_128(p, w.x, w.y, w.z, w.w);
    x = ld_l1_32(p + 16);
  } else if (S == 4) {
    w.x = ld_l1_32(p + 4);
    ld_l1_64(p + 8, w.y, w.z);
    w.w = ld_l1_32(p + 16);
  } else if (S == 6) {
    w.x = ld_l1_32(p + 4);
    ld_l1_64(p + 8, w.y, w.z);
    ld_l1_64(p + 16, w.w, x);
  } else if (S == 8) {
    ld_l1_64(p + 8, w.x, w.y);
    ld_l1_64(p + 16, w.z, w.w);
  } else if (S == 10) {
    ld_l1_64(p + 8, w.x, w.y);
    ld_l1_128(p + 16, w.z, w.w, x, unused);
  } else if (S == 12) {
    w.x = ld_l1_32(p + 12);
    ld_l1_64(p + 16, w.y, w.z);
    w.w = ld_l1_32(p + 24);
  } else {
    w.x = ld_l1_32(p + 12);
    ld_l1_128(p + 16, w.y, w.z, w.w, x);
  }
}
// groups n0 + tile_pos(tid, k) < n of the row whose group 0 starts s bytes into
// the grid word at p
template <int S>
__device__ __forceinline__ void ld_groups(const char* p, int32_t n0, int32_t n, int tid,
                                          uint4 (&w)[UNR], uint32_t (&x)[UNR], const uint4& none) {
  const char* q = p + 16 * (int64_t)(n0 + tile_pos(tid, 0));
  if (n0 + TILE <= n) {
#pragma unroll
    for (int k = 0; k < UNR; ++k) ld_group<S>(q + 512 * k, w[k], x[k]);
  } else {
#pragma unroll
    for (int k = 0; k < UNR; ++k) {
      w[k] = none;
      x[k] = none.x;
      if (n0 + tile_pos(tid, k) < n) ld_group<S>(q + 512 * k, w[k], x[k]);
    }
  }
}
template <typename T>
__device__ __forceinline__ void ld_tile_off_grid(const T* rowt, int32_t n0, int32_t n, bool rim,
                                                 int tid, uint4 (&w)[UNR], uint32_t (&x)[UNR],
                                                 const uint4& none) {
  const int s = (int)(reinterpret_cast<uintptr_t>(rowt) & 15u);
  const char* p = reinterpret_cast<const char*>(rowt) - s;
  if (rim) {  // the first or last tile of the call's buffer: no byte outside it
#pragma unroll
    for (int k = 0; k < UNR; ++k) {
      const int32_t g = n0 + tile_pos(tid, k);
      w[k] = g < n ? Traits<T>::load_elems(rowt, g) : none;
      x[k] = none.x;
      if (s & 2) {  // as cut_group expects it
        x[k] = w[k].w >> 16;
        w[k] = make_uint4(w[k].x << 16, __funnelshift_l(w[k].x, w[k].y, 16),
                          __funnelshift_l(w[k].y, w[k].z, 16), __funnelshift_l(w[k].z, w[k].w, 16));
      }
    }
    return;
  }
  if (sizeof(T) == 4 || (s & 2) == 0) {
    if (s == 0) ld_groups<0>(p, n0, n, tid, w, x, none);
    else if (s == 4) ld_groups<4>(p, n0, n, tid, w, x, none);
    else if (s == 8) ld_groups<8>(p, n0, n, tid, w, x, none);
    else ld_groups<12>(p, n0, n, tid, w, x, none);
  } else {
    if (s == 2) ld_groups<2>(p, n0, n, tid, w, x, none);
    else if (s == 6) ld_groups<6>(p, n0, n, tid, w, x, none);
    else if (s == 10) ld_groups<10>(p, n0, n, tid, w, x, none);
    else ld_groups<14>(p, n0, n, tid, w, x, none);
  }
}
template <typename T>
__device__ __forceinline__ void cut_groups(const T* rowt, uint4 (&w)[UNR], const uint32_t (&x)[UNR]) {
  if constexpr (sizeof(T) == 2) {
    if ((reinterpret_cast<uintptr_t>(rowt) & 2u) == 0) return;
#pragma unroll
    for (int k = 0; k < UNR; ++k)
      w[k] = make_uint4(__funnelshift_r(w[k].x, w[k].y, 16), __funnelshift_r(w[k].y, w[k].z, 16),
                        __funnelshift_r(w[k].z, w[k].w, 16), __funnelshift_r(w[k].w, x[k], 16));
  }
}

// ---- one row's features and the mode's epilogue (one warp) ------------------------------

// Whole warp (the request search is warp-collective).
template <typename T, int MODE>
__device__ __forceinline__ RowPre load_pre(const Args& a, int64_t row, int32_t y, const char* rowp,
                                           int lane) {
  using Tr = Traits<T>;
  RowPre p;
  p.y = y;
  p.xy = (p.y >= 0 && (int64_t)p.y < a.vocab) ? Tr::elem(rowp, p.y) : NAN;
  p.r = -1;
  p.lo = p.hi = 0;
  p.eos = 0;
  if (MODE == MODE_FEATURES && a.offsets) {
    p.r = find_request(a.offsets, a.n_req, row, lane);
  } else if (MODE == MODE_ROUTE) {
    p.r = find_request(a.offsets, a.n_req, a.row_base + row, lane);
  } else if (MODE == MODE_DECODE) {
    p.r = a.slot[row];
    p.eos = a.eos[row];
  }
  if (MODE != MODE_DECODE && p.r >= 0) {
    p.lo = a.offsets[p.r];
    p.hi = a.offsets[p.r + 1];
  }
  return p;
}

__device__ __forceinline__ int atom_add_acq_rel(int* p, int v) {
  int old;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}

// Eq. 3 features of the row from its (m, S, U) state and its top-32 element keys
// E (lane 0 = largest), then, by mode: write the record; or fold it into the
// request and, for the request's last row, pool / score / threshold; or fold it
// into its decode slot.  Whole warp.
template <typename T, int MODE>
__device__ __forceinline__ void row_finish(const Args& a, int64_t row, float m, float S, float U,
                                           bool bad, uint64_t E, const RowPre& pre, int lane) {
  const int64_t V = a.vocab;
  const int kc = a.kc, K = a.topk;
  const int32_t y = pre.y;
  uint32_t flags = 0;
  if (y < 0 || (int64_t)y >= V) flags |= FLAG_BAD_CHOSEN;
  const bool nonfinite = bad || !(S > 0.f) || !isfinite(S) || !isfinite(U);
  if (nonfinite) flags |= FLAG_NONFINITE;

  const float log2S = log2f(S);
  const bool hasE = lane < kc && E != 0ull;
  const float xk = hasE ? key_val(E) : -INFINITY;
  const float lp2 = fmaf(xk, L2E, -m) - log2S;  // log2 p of this lane's token
  const float pk = hasE ? exp2f(lp2) : 0.f;
  float term = (lane < K && pk > 0.f) ? pk * lp2 : 0.f;
  float pmass = lane < K ? pk : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    term += __shfl_xor_sync(FULL, term, o);
    pmass += __shfl_xor_sync(FULL, pmass, o);
  }
  const float hraw = term * LN2;  // sum over top-K of p ln p = -H^K
  const float h = a.renorm ? (pmass > 0.f ? hraw / pmass - logf(pmass) : 0.f) : hraw;
  const float x1 = __shfl_sync(FULL, xk, 0);
  const float p1 = __shfl_sync(FULL, pk, 0);
  const float p2 = V >= 2 ? __shfl_sync(FULL, pk, 1) : 0.f;
  const uint64_t e1 = shfl64(E, 0), e2 = shfl64(E, 1);
  float logp = NAN;
  if (!(flags & FLAG_BAD_CHOSEN)) logp = (fmaf(pre.xy, L2E, -m) - log2S) * LN2;
  float fv[NFEAT];
  fv[0] = logp;
  fv[1] = p1;
  fv[2] = p1 - p2;
  fv[3] = (log2S - U / S) * LN2;
  fv[4] = h;
  fv[5] = 0.f;
  fv[6] = (m + log2S) * LN2;
  fv[7] = x1;
  int32_t i1 = (int32_t)key_idx(e1), i2 = V >= 2 ? (int32_t)key_idx(e2) : -1;
  if (nonfinite) {
#pragma unroll
    for (int j = 0; j < NFEAT; ++j) fv[j] = NAN;
    i1 = i2 = -1;
  }

  if (MODE == MODE_FEATURES) {
    if (a.offsets && !nonfinite && pre.r >= 0)
      fv[5] = (float)(row - pre.lo + 1) / (float)(pre.hi - pre.lo);
    if (lane < NFEAT) {
      float v = fv[0];
#pragma unroll
      for (int j = 1; j < NFEAT; ++j)
        if (lane == j) v = fv[j];
      a.feat[row * NFEAT + lane] = v;
    }
    if (lane == 0) {
      a.top2[2 * row] = i1;
      a.top2[2 * row + 1] = i2;
      a.row_flags[row] = flags;
    }
    return;
  }

  if (MODE == MODE_ROUTE) {
    const int64_t gr = a.row_base + row;
    const int32_t r = pre.r;
    const int64_t lo = pre.lo, hi = pre.hi;
    if (r < 0 || route_bad_request(a, r, lo, hi)) {
      if (lane == 0) atomicOr(a.ctx_flags, FLAG_BAD_OFFSETS);
      return;
    }
    if (!nonfinite) fv[5] = (float)(gr - lo + 1) / (float)(hi - lo);
    int last = 0;
    if (lane == 0) {
      // the record, then one acquire-release increment: the request's last row
      // sees every other row's record
      float4* rp = reinterpret_cast<float4*>(a.rec + gr * NFEAT);
      rp[0] = make_float4(fv[0], fv[1], fv[2], fv[3]);
      rp[1] = make_float4(fv[4], fv[5], fv[6], fv[7]);
      a.rec_flags[gr] = flags;
      last = (atom_add_acq_rel(a.req_cnt + r, 1) == (int)(hi - lo) - 1);
    }
    last = __shfl_sync(FULL, last, 0);
    if (last) {
      const Pooled p = pool_rows<4>(a.rec, a.rec_flags, lo, hi, a.w, a.b, a.zthr, lane);
      write_pooled(p, r, a.agg, a.score, a.ship, a.req_flags, lane);
      if (lane == 0) a.req_cnt[r] = 0;
    }
    return;
  }

  if (MODE == MODE_DECODE) {
    const int32_t s = pre.r;
    if (s < 0 || s >= a.n_slots) {
      if (lane == 0) atomicOr(a.ctx_flags, FLAG_BAD_SLOT);
      return;
    }
    // lane f < 5 keeps statistic f (l, m, margin, -H, h)
    float* A = a.acc + (int64_t)s * ACC_WORDS;
    const int f = lane < 5 ? lane : 0;
    const int32_t n = __float_as_int(A[0]) + 1;
    const uint32_t fl = __float_as_uint(A[1]) | flags;
    const float sum0 = A[2 + f], comp0 = A[7 + f], mn0 = A[12 + f];
    const float v = f == 0 ? fv[0] : f == 1 ? fv[1] : f == 2 ? fv[2] : f == 3 ? -fv[3] : fv[4];
    float sum = v, comp = 0.f, mn = v;
    if (n != 1) {  // compensated (Kahan) running sum in step order
      const float yv = v - comp0;
      sum = sum0 + yv;
      comp = (sum - sum0) - yv;
      mn = fminf(mn0, v);
    }
    __syncwarp();  // every lane has read the slot
    if (!pre.eos) {
      if (lane < 5) {
        A[2 + f] = sum;
        A[7 + f] = comp;
        A[12 + f] = mn;
      }
      if (lane == 0) {
        A[0] = __int_as_float(n);
        A[1] = __uint_as_float(fl);
      }
      return;
    }
    // the request ends with this row: pool, score, ship rule, clear the slot
    const bool none = (fl & (FLAG_NONFINITE | FLAG_BAD_CHOSEN)) != 0;
    const float mean = sum / (float)n;
    float z = a.b, mine = NAN, sc = NAN;
    uint8_t sh = 0;
    if (!none) {
      float ag[NAGG];
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        ag[2 * j] = __shfl_sync(FULL, mean, j);
        ag[2 * j + 1] = __shfl_sync(FULL, mn, j);
      }
      ag[10] = (float)(n + 1) / (float)(2 * n);
#pragma unroll
      for (int j = 0; j < NAGG; ++j) {
        z = fmaf(a.w[j], ag[j], z);
        if (lane == j) mine = ag[j];
      }
      sc = 1.f / (1.f + expf(-z));
      sh = (z >= a.zthr) ? 1 : 0;
    }
    if (a.agg && lane < NAGG) a.agg[(int64_t)s * NAGG + lane] = mine;
    if (lane == 0) {
      a.score[s] = sc;
      a.ship[s] = sh;
      a.req_flags[s] = fl;
    }
    if (lane < ACC_WORDS) A[lane] = 0.f;
  }
}

// What theta1 comes from.  pub[0 .. 31]: 32 of a CTA's largest thread maxima, every
// warp's PUB largest ones; of a range of less than a tile, whose first warps hold
// all of it, the 32 / A largest ones of A warps, A the largest power of two up to the
// number of warps with a group in every lane.  low[warp] (unless null): a code that
// at least kc of the warp's maxima reach, for rows whose largest values lie side by
// side in one warp's share (a range of allowed tokens, sorted logits).
__device__ __forceinline__ void publish_max(uint32_t cur, uint32_t* pub, uint32_t* low,
                                            int32_t groups, int kc, int warp, int lane) {
  if (groups >= TILE) {
    if (low) {
      const uint32_t least = __reduce_min_sync(FULL, cur);
      if (lane == 0) low[warp] = least;
    }
#pragma unroll
    for (int i = 0; i < PUB; ++i) {
      const uint32_t w = __reduce_max_sync(FULL, cur);
      const unsigned eq = __ballot_sync(FULL, cur == w);
      if (lane == 0) pub[warp * PUB + i] = w;
      if (lane == __ffs(eq) - 1) cur = 0u;
    }
    return;
  }
  const int full = max(1, (groups + 32 * (UNR - 1)) / (32 * UNR));  // warps with 32 groups or more
  const int A = full >= 8 ? 8 : full >= 4 ? 4 : full >= 2 ? 2 : 1, n = 32 / A;
  if (warp >= A) {
    if (low && lane == 0) low[warp] = 0u;
    return;
  }
  cur = warp_sort_desc<uint32_t>(cur, lane);
  if (lane < n) pub[warp * n + lane] = cur;
  if (low && lane == kc - 1) low[warp] = cur;
}

// A better bound where theta1 lets too many tiles or elements pass (values side by
// side in the shares of few warps), by bisection of the ord() codes of all thread
// maxima (code(j): this lane's j-th, N per lane) from th1, which at least kc of them
// reach, to the smallest of kc to kc + 4 of them (of more where they tie).
// With 1,000 neighbouring tokens 10 above the others: 256 rows of V = 151,936 bf16
// 781 us when the published maxima alone decided and such rows went on to the scan,
// 21 now; 1,500 rows 3,594 us, 95 now.
template <int N, typename F>
__device__ __forceinline__ float raise_bound(F code, float th1, int kc) {
  uint32_t v[N], lo = ord(th1);
#pragma unroll
  for (int j = 0; j < N; ++j) v[j] = code(j);
  auto reach = [&](uint32_t from) {
    int c = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) c += v[j] >= from ? 1 : 0;
    return __reduce_add_sync(FULL, c);
  };
  if (reach(lo + 1u) < kc) return th1;  // ties, or too few unmasked tokens
  uint32_t hi = v[0];
#pragma unroll
  for (int j = 1; j < N; ++j) hi = max(hi, v[j]);
  hi = __reduce_max_sync(FULL, hi) + 1u;
#pragma unroll 1
  while (hi - lo > 1u) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    const int c = reach(mid);
    if (c < kc) {
      hi = mid;
    } else {
      lo = mid;
      if (c <= kc + 4) break;
    }
  }
  uint32_t least = 0xffffffffu;  // the least of those that reach lo: nothing lies between
#pragma unroll
  for (int j = 0; j < N; ++j) least = v[j] >= lo ? min(least, v[j]) : least;
  return unord(__reduce_min_sync(FULL, least));
}
static __device__ __noinline__ float raise_cta(const uint32_t* all, float th1, int kc, int lane) {
  return raise_bound<NWARP>([&](int j) { return all[32 * j + lane]; }, th1, kc);
}
__device__ __forceinline__ float raise_ws(const float4* tinfo, uint32_t edge, float th1, int kc,
                                              int lane) {
  return raise_bound<NWARP + 1>(
      [&](int j) { return j < NWARP ? ord(tinfo[j * 32 + lane].x) : edge; }, th1, kc);
}
// Candidate tiles from which on it is tried.  Of values in no order about kc + 3 reach
// theta1, up to twice as many in a range of less than a tile (of which not every
// warp publishes) or where kc is most of what is published.
__device__ __forceinline__ int many_tiles(int kc) { return 2 * kc + 24; }

// The guarded pass over a range's groups first, first + step, .. below last: NaN and
// +inf mark the row, -inf is a masked token.  A group at a time, rescaled once, with
// AHEAD groups' loads in flight (token by token, 256 rows of V = 151,936 bf16 whose
// padding is -inf took 266 us, now 50; 1,500 of V = 32,000 1,550, now 138).
template <typename T, bool ALIGNED, int AHEAD>
__device__ __forceinline__ void careful_groups(const char* rowp, int32_t first, int32_t last,
                                               int32_t step, float& m, float& S, float& U,
                                               bool& bad) {
  using Tr = Traits<T>;
  const uint4 NEG = make_uint4(Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD);
#pragma unroll 1
  for (int32_t g0 = first; g0 < last; g0 += AHEAD * step) {
    uint4 w[AHEAD];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
      const int32_t g = g0 + k * step;
      w[k] = NEG;
      if (g < last)
        w[k] = ALIGNED ? ld_stream(reinterpret_cast<const uint4*>(rowp) + g)
                       : Tr::load_elems(rowp, g);
    }
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
#pragma unroll
      for (int e = 0; e < Tr::VEC; ++e) bad = bad || !(Tr::at(w[k], e) < INFINITY);
      const float most = Tr::gmax(w[k]);
      if (!(most > -INFINITY && most < INFINITY)) continue;
      const float mn = fmaxf(m, most * L2E);
      if (S != 0.f) {
        const float dl = m - mn, f = ex2(dl);
        U = f * fmaf(dl, S, U);
        S *= f;
      }
      m = mn;
#pragma unroll
      for (int e = 0; e < Tr::VEC; ++e) {
        const float d = fmaf(Tr::at(w[k], e), L2E, -m), p = ex2(d);
        S += p;
        U = fmaf(p, p != 0.f ? d : 0.f, U);
      }
    }
  }
}

// The exact scan, of groups [ga, gb) by one warp: rows whose ties overflow the
// buffers, or with fewer than kc unmasked tokens.  Elements from thr on go to the
// list; once that is full, only those that beat its last entry: an element of a
// later round has a higher index, so that its equals no longer count.  (A round's
// elements come by their place in the group, not by index: the bound moves
// between rounds.)  AHEAD rounds' loads are in flight.
template <typename T, bool ALIGNED, int AHEAD>
__device__ __forceinline__ void scan_groups(const char* rowp, int32_t ga, int32_t gb, float thr,
                                            WarpTopK& ek, int lane) {
  using Tr = Traits<T>;
  const uint4 NEG = make_uint4(Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD);
  uint32_t least = 0u;  // ord() code
#pragma unroll 1
  for (int32_t g0 = ga; g0 < gb; g0 += 32 * AHEAD) {
    uint4 w[AHEAD];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
      const int32_t g = g0 + 32 * k + lane;
      w[k] = NEG;
      if (g < gb)
        w[k] = ALIGNED ? ld_stream(reinterpret_cast<const uint4*>(rowp) + g)
                       : Tr::load_elems(rowp, g);
    }
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
      const int32_t g = g0 + 32 * k + lane;
      const float most = Tr::gmax(w[k]);
      if (!__any_sync(FULL, g < gb && most >= thr && ord(most) >= least)) continue;
#pragma unroll 1
      for (int e = 0; e < Tr::VEC; ++e) {
        const float x = Tr::at(w[k], e);
        const bool c = g < gb && x >= thr && ord(x) >= least;
        ek.push(c, c ? make_key(x, (uint32_t)(g * Tr::VEC + e)) : 0ull, lane);
        ek.drain(lane);
      }
      const uint64_t last = shfl64(ek.list, 31);
      if (last != 0ull) least = (uint32_t)(last >> 32) + 1u;
    }
  }
}

// ---- the row kernel for split rows: one thread-block cluster of C CTAs per row ----------------

// Resident CTAs per SM the compiler sizes registers for: five for fp32 rows
// (48 registers), four for bf16.  Measured in CUDA graphs with one CTA per
// row: 354-row batches of V = 32,000 fp32 10.0 us per batch with five
// against 11.5 us with four (two consecutive launches then fit on the GPU
// together), 256-row decode steps of V = 151,936 bf16 11.1 against 10.7 us.
// Off the 16-byte grid, where a group's loads need more registers, four.
template <typename T, bool ALIGNED>
constexpr int rows_min_blocks() {
  return sizeof(T) == 4 && ALIGNED ? 5 : 4;
}

// What a CTA of the split kernel works on.  Read from the special registers each time
// it is built: the stream and the selection after it build their own, so that
// nothing of the latter takes registers from the former (kept alive together, fp32
// batches of V = 151,936 took up to 9% longer).
template <typename T>
struct SplitPlace {
  uint32_t C, rank, cid;  // CTAs of the row, this one's, the row
  int32_t gfull, g0, g1, ng, ntiles, shift;
  __device__ __forceinline__ explicit SplitPlace(const Args& a) {
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(cid));
    gfull = (int32_t)((uint32_t)a.vocab / Traits<T>::VEC);
    const int lc = __ffs(C) - 1;  // C is 1, 2, 4 or 8
    g0 = (int32_t)(((int64_t)gfull * rank) >> lc);
    g1 = (int32_t)(((int64_t)gfull * (rank + 1)) >> lc);
    ng = g1 - g0;
    ntiles = (int32_t)((uint32_t)(ng + TILE - 1) / TILE);
    shift = 0;
    while (((ntiles + (1 << shift) - 1) >> shift) > MAX_SLOTS) ++shift;
  }
  __device__ __forceinline__ const T* row(const Args& a) const {
    return reinterpret_cast<const T*>(a.logits) + (int64_t)cid * a.row_stride;
  }
};

template <typename T, int MODE, bool ALIGNED>
__global__ void __launch_bounds__(NT, rows_min_blocks<T, ALIGNED>()) verify_rows(const Args a) {
  __shared__ Smem sm;
  using Tr = Traits<T>;
  constexpr int VEC = Tr::VEC;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint4 NEG = make_uint4(Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD);

  pdl_enter(a.early);

  float m = M2_INIT;
  float2 S2 = make_float2(0.f, 0.f), U2 = make_float2(0.f, 0.f);
  float thr_max = -INFINITY;
  bool bad = false;

  // ---- stream the groups [g0, g1): tile t holds groups t*TILE + k*NT + tid ------------
  {
    const SplitPlace<T> pl(a);
    const uint32_t C = pl.C;
    const int32_t g0 = pl.g0, g1 = pl.g1, ng = pl.ng, ntiles = pl.ntiles, shift = pl.shift;
    const int32_t nfull = (int32_t)((uint32_t)ng / TILE), rem = ng & (TILE - 1), smask = (1 << shift) - 1;
    const T* rowt = pl.row(a);
    const uint4* vp = reinterpret_cast<const uint4*>(rowt);
    float racc = -INFINITY;
    if (C > 1) cluster_arrive();  // every CTA of the cluster has started (waited for below)
  if (tid == 0) {
    sm.ncand[0] = sm.ncand[1] = 0;
    sm.nelem[0] = sm.nelem[1] = 0;
    // the row's inputs beside the logits, on their way into L2 while it streams
    if (pl.rank == 0) {
      prefetch_line(a.chosen + pl.cid);
      if (MODE == MODE_DECODE) {
        prefetch_line(a.slot + pl.cid);
        prefetch_line(a.eos + pl.cid);
      }
    }
  }
  if (tid < 32) sm.top[tid] = 0ull;

    // the groups of tile t (off the grid: uncut), nothing past the range
    auto load_tile = [&](uint4 (&dst)[UNR], uint32_t (&ext)[UNR], int32_t t) {
      const int32_t nb = t * TILE;
      if (ALIGNED) {
        // one pointer per tile for bf16 (16 decode steps of 256 rows 341 us, 360 with
        // an index per load); fp32 at 48 registers spills less with the indices
        // (353 rows of V = 32,000 16.6 us against 16.8)
        const uint4* q = vp + (g0 + nb + tile_pos(tid, 0));
        auto load = [&](int k) {
          return ld_stream(sizeof(T) == 2 ? q + 32 * k : vp + g0 + nb + tile_pos(tid, k));
        };
        if (t < nfull) {
#pragma unroll
          for (int k = 0; k < UNR; ++k) dst[k] = load(k);
        } else {
#pragma unroll
          for (int k = 0; k < UNR; ++k) dst[k] = tile_pos(tid, k) < rem ? load(k) : NEG;
        }
      } else {
        // (a row of fewer groups than CTAs has its first group in a later CTA)
        const bool rim = (pl.cid == 0 && g0 + nb == 0) ||
                         (pl.cid == a.n_rows - 1 && g1 == pl.gfull && t == ntiles - 1);
        ld_tile_off_grid(rowt, g0 + nb, g1, rim, tid, dst, ext, NEG);
      }
    };
    // one CTA per row: one thread keeps the tiles PF_TILES ahead on their way
    // into L2 (bulk prefetches need no registers, so the CTA has more bytes in
    // flight than its two register tiles; measured on 256-row decode steps:
    // 24.9 us isolated and 11.2 us in a CUDA graph against 27.0 and 12.8 us
    // without; with clusters, whose CTAs already keep HBM busy, it slowed
    // the step)
    auto prefetch_tile = [&](int32_t t) {
      if (PF_TILES > 0 && C == 1 && tid == 0 && t < ntiles) {
        const int32_t gs = t * TILE;
        // (off the grid: the 16-byte words below the groups; t > 0)
        prefetch_l2(reinterpret_cast<const uint4*>(reinterpret_cast<uintptr_t>(vp + g0 + gs) &
                                                   ~(uintptr_t)15),
                    (uint32_t)min(TILE, ng - gs) * 16u);
      }
    };
#pragma unroll
    for (int32_t p = 1; p <= PF_TILES; ++p) prefetch_tile(p);
    uint4 cur[UNR], nxt[UNR];
    uint32_t ext[UNR], ext_n[UNR];  // off the grid: the groups' fifth words
    load_tile(cur, ext, 0);
    for (int32_t t = 0; t < ntiles; ++t) {
      prefetch_tile(t + 1 + PF_TILES);
      if (t + 1 < ntiles) load_tile(nxt, ext_n, t + 1);
      if (!ALIGNED) cut_groups(rowt, cur, ext);
      const float tmax = Tr::tile_max(cur);
      thr_max = fmaxf(thr_max, tmax);
      racc = fmaxf(racc, tmax);
      if ((t & smask) == smask || t == ntiles - 1) {
        sm.tm[t >> shift][tid] = racc;
        racc = -INFINITY;
      }
      // online rescale, branch-free (a no-op when the maximum did not move)
      const float mn = fmaxf(m, tmax * L2E);
      const float dl = m - mn;
      const float f = ex2(dl);
      U2 = __fmul2_rn(make_float2(f, f), __ffma2_rn(make_float2(dl, dl), S2, U2));
      S2 = __fmul2_rn(make_float2(f, f), S2);
      m = mn;
      const float2 nm = make_float2(-m, -m);
      if (t < nfull) {
#pragma unroll
        for (int k = 0; k < UNR; ++k) Tr::accum(cur[k], nm, S2, U2);
      } else {
#pragma unroll
        for (int k = 0; k < UNR; ++k)
          if (tile_pos(tid, k) < rem) Tr::accum(cur[k], nm, S2, U2);
      }
#pragma unroll
      for (int k = 0; k < UNR; ++k) {
        cur[k] = nxt[k];
        if (!ALIGNED) ext[k] = ext_n[k];
      }
    }
  }
  float S = S2.x + S2.y, U = U2.x + U2.y;

  const SplitPlace<T> pl(a);
  const uint32_t C = pl.C, rank = pl.rank, cid = pl.cid;
  const int64_t row = cid, V = a.vocab;
  const int32_t g0 = pl.g0, g1 = pl.g1, ng = pl.ng, ntiles = pl.ntiles, shift = pl.shift;
  const int32_t nslots = (ntiles + (1 << shift) - 1) >> shift;
  const char* rowp = reinterpret_cast<const char*>(pl.row(a));
  const uint4* vp = reinterpret_cast<const uint4*>(rowp);
  // cluster rank 0 takes the last elements
  const int32_t nedge = rank == 0 ? (int32_t)V & (VEC - 1) : 0;

  // What follows the stream is a chain of latencies that a lone launch cannot
  // hide; it is kept short: four block barriers, no sort, every global load
  // issued as early as its address is known (see the phases' comments).
  // Measured against sorted maxima, a serial merge and a pull-style cluster merge
  // (CUDA graphs, per launch): 256 rows of V = 151,936 bf16 21.6 -> 19.5 us, 8 rows
  // 11.3 -> 8.4 us, 256 rows of V = 32,000 fp32 13.9 -> 12.5 us.

  // ---- the elements after the last group: warp 0 of cluster rank 0, one per lane
  float xe = -INFINITY;
  const int64_t ve = (int64_t)pl.gfull * VEC + lane;  // this lane's
  if (warp == 0 && lane < nedge) {
    const float x = Tr::elem(rowp, ve);
    careful_add(x, m, S, U, bad);
    if (!isnan(x)) xe = x;
    thr_max = fmaxf(thr_max, xe);
  }

  // ---- theta1: the kc-th largest of the published thread maxima
  // (kc <= 32 distinct elements reach it, so it bounds the kc-th element from
  // below).  Against the kc-th largest of all thread maxima, which takes a sort
  // per warp and seven merges, about one candidate more passes it (22 for 21 of
  // 151,936 normal values and kc = 20).
  const int kc = a.kc;
  publish_max(ord(thr_max), sm.pub, nullptr, ng, kc, warp, lane);
  sm.all_max[tid] = ord(thr_max);
  int32_t y = 0;
  if (rank == 0 && warp == 1) y = a.chosen[row];  // used after the next barrier
  __syncthreads();
  float th1;
  {
    const uint32_t mine = sm.pub[lane];
    int rk = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const uint32_t q = sm.pub[j];
      rk += (q > mine || (q == mine && j < lane)) ? 1 : 0;
    }
    th1 = unord(__shfl_sync(FULL, mine, __ffs(__ballot_sync(FULL, rk == kc - 1)) - 1));
  }
  // the warp's state
  lse_warp(m, S, U);
  bad = __any_sync(FULL, bad);
  if (lane == 0) {
    sm.pm[warp] = m;
    sm.pS[warp] = S;
    sm.pU[warp] = U;
    sm.pbad[warp] = bad;
  }

  // ---- candidates and their elements by theta1; once more by a bound from all
  // thread maxima if too many reach theta1, or fewer than kc maxima are published (all
  // but a few neighbouring tokens masked; one warp's share has published all it has)
  bool more = ng > 32 * UNR, merged = false;
  int ncand, at = 0;  // counters of this attempt
#pragma unroll 1
  for (;;) {
    // candidate super-groups: this thread's stored tile maxima >= theta1
    if (th1 > -INFINITY && thr_max >= th1) {
      uint32_t mask = 0u;
#pragma unroll
      for (int32_t s = 0; s < MAX_SLOTS; ++s)
        if (s < nslots) mask |= sm.tm[s][tid] >= th1 ? 1u << s : 0u;
      if (mask) {
        int i = atomicAdd(&sm.ncand[at], __popc(mask));
        for (; mask; mask &= mask - 1u, ++i)
          if (i < CCAP) sm.cand_id[i] = ((uint32_t)(__ffs(mask) - 1) << 8) | (uint32_t)tid;
      }
      if (xe >= th1) {  // an edge element is a candidate by itself
        const int e = atomicAdd(&sm.nelem[at], 1);
        if (e < ECAP) sm.ebuf[e] = make_key(xe, (uint32_t)ve);
      }
    }
    __syncthreads();
    ncand = sm.ncand[at];
    if (!more || (th1 > -INFINITY && ncand <= many_tiles(kc))) {
      // re-read the candidates (a 16-byte group per thread, all in flight at
      // once); their elements >= theta1 become keys: kc distinct elements reach
      // theta1, so the CTA's top kc are among them
      const int total = ncand <= CCAP ? ncand * (UNR << shift) : 0;  // the super-groups' groups
      int32_t g = -1;
      uint4 wv = NEG;
      auto fetch = [&](int i) {
        const int c = i / UNR >> shift, j = i - (c << shift) * UNR;
        const uint32_t id = sm.cand_id[c];
        const int32_t t = (int32_t)((id >> 8) << shift) + j / UNR;
        const int32_t gi = t * TILE + tile_pos((int)(id & 255u), j % UNR);
        g = t < ntiles && gi < ng ? g0 + gi : -1;
        if (g >= 0) wv = ALIGNED ? ld_reread(vp + g) : Tr::load_elems(rowp, g);
      };
      if (tid < total) fetch(tid);
      // while they arrive: warp 0 merges the CTA's state, warp 1 of cluster rank 0
      // finds what the row's epilogue needs besides the reduction
      if (warp == 0 && !merged) {
        m = lane < NWARP ? sm.pm[lane] : M2_INIT;
        S = lane < NWARP ? sm.pS[lane] : 0.f;
        U = lane < NWARP ? sm.pU[lane] : 0.f;
        bad = __any_sync(FULL, lane < NWARP && sm.pbad[lane] != 0);
#pragma unroll
        for (int o = NWARP / 2; o > 0; o >>= 1) {
          const float mo = __shfl_xor_sync(FULL, m, o);
          const float So = __shfl_xor_sync(FULL, S, o);
          const float Uo = __shfl_xor_sync(FULL, U, o);
          lse_merge(m, S, U, mo, So, Uo);
        }
        // only lanes 0..NWARP-1 took part in the last butterfly: give every lane the total
        m = __shfl_sync(FULL, m, 0);
        S = __shfl_sync(FULL, S, 0);
        U = __shfl_sync(FULL, U, 0);
        // a masked (-inf), NaN or infinite logit made the CTA's fast accumulators
        // non-finite: it re-streams its range with guards (the row's merged state
        // is non-finite exactly when a CTA's is)
        if (lane == 0) sm.careful = (!bad && !(isfinite(S) && isfinite(U))) ? 1 : 0;
      } else if (warp == 1 && rank == 0 && !merged) {
        const RowPre p = load_pre<T, MODE>(a, row, y, rowp, lane);
        if (lane == 0) sm.pre = p;
      }
      merged = true;
      for (int i = tid; i < total;) {
        if (g >= 0) {
          uint32_t hits = 0u;
#pragma unroll
          for (int e = 0; e < VEC; ++e) hits |= Tr::at(wv, e) >= th1 ? 1u << e : 0u;
          if (hits) {
            int k = atomicAdd(&sm.nelem[at], __popc(hits));
            for (; hits; hits &= hits - 1u, ++k) {
              const int e = __ffs(hits) - 1;
              if (k < ECAP)
                sm.ebuf[k] = make_key(Tr::at(wv, e), (uint32_t)(g * VEC + e));
            }
          }
        }
        i += NT;
        if (i < total) fetch(i);
      }
      __syncthreads();
      if (!more || sm.nelem[at] <= NT) break;
    }
    more = false;
    at = 1;
    th1 = raise_cta(sm.all_max, th1, kc, lane);
  }
  const bool fb_cand = !(th1 > -INFINITY) || ncand > CCAP;
  if (sm.careful) {
    float cm = M2_INIT, cS = 0.f, cU = 0.f;
    bool cbad = false;
    careful_groups<T, ALIGNED, 2>(rowp, g0 + tid, g1, NT, cm, cS, cU, cbad);
    if (tid < nedge) careful_add(Tr::elem(rowp, ve), cm, cS, cU, cbad);
    block_reduce_state(sm, cm, cS, cU, cbad, warp, lane);  // warp 0 holds the CTA's state
    m = cm;
    S = cS;
    U = cU;
    bad = cbad;
  }

  // ---- the CTA's exact top-32 elements: up to NT candidate keys are ranked
  // by counting (keys are distinct: the index is part of the key; up to NT / 2
  // keys with two threads each), more by warp 0's sorting network; the exact
  // scan when the buffers overflowed
  uint64_t E = 0ull;
  const int ne = sm.nelem[at];
  const bool fb = fb_cand || ne > ECAP;
  if (!fb && ne <= NT) {
    if (ne <= NT / 2) {
      const int i = tid >> 1;
      uint64_t key = 0ull;
      int rk = 0;
      if (i < ne) {
        key = sm.ebuf[i];
        for (int q = tid & 1; q < ne; q += 2) rk += sm.ebuf[q] > key ? 1 : 0;
      }
      rk += __shfl_xor_sync(FULL, rk, 1);
      if (i < ne && rk < 32) sm.top[rk] = key;
    } else if (tid < ne) {
      const uint64_t key = sm.ebuf[tid];
      int rk = 0;
      for (int q = 0; q < ne; ++q) rk += sm.ebuf[q] > key ? 1 : 0;
      if (rk < 32) sm.top[rk] = key;
    }
    __syncthreads();
    if (warp == 0) E = sm.top[lane];
  } else if (!fb) {
    if (warp == 0)
      for (int b0 = 0; b0 < ne; b0 += 32) {
        uint64_t k = b0 + lane < ne ? sm.ebuf[b0 + lane] : 0ull;
        k = warp_sort_desc<uint64_t>(k, lane);
        E = warp_merge_desc<uint64_t>(E, k, lane);
      }
  } else {
    // exact scan of the whole range, an eighth of it per warp (256 equal rows of
    // V = 151,936 bf16: 3,760 us with one warp and no rising bound, 50 now)
    WarpTopK ek;
    ek.buf = sm.ebuf + warp * (ECAP / NWARP);
    ek.cnt = 0;
    ek.list = 0ull;
    scan_groups<T, ALIGNED, 2>(rowp, g0 + (int32_t)((int64_t)ng * warp / NWARP),
                               g0 + (int32_t)((int64_t)ng * (warp + 1) / NWARP), th1, ek, lane);
    if (warp == 0 && nedge > 0) {
      const bool c = lane < nedge && xe >= th1;
      ek.push(c, c ? make_key(xe, (uint32_t)ve) : 0ull, lane);
      ek.drain(lane);
    }
    ek.drain_all(lane);
    __syncthreads();
    sm.ebuf[32 * warp + lane] = ek.list;
    __syncthreads();
    if (warp == 0) {
      E = ek.list;
      for (int w = 1; w < NWARP; ++w)
        E = warp_merge_desc<uint64_t>(E, sm.ebuf[32 * w + lane], lane);
    }
  }

  // ---- split-vocab merge across the cluster (distributed shared memory): the
  // other CTAs leave their state and list in rank 0's shared memory, one lane
  // per 8 bytes of list, and one cluster barrier hands them over
  if (C > 1) {
    cluster_wait();  // the arrivals at the start: rank 0 runs, its memory may be written
    if (warp == 0 && rank != 0) {
      dsmem_st_u64(dsmem_addr(&sm.peer_list[rank][lane], 0), E);
      if (lane < 4) {
        const uint32_t v = lane == 0   ? __float_as_uint(m)
                           : lane == 1 ? __float_as_uint(S)
                           : lane == 2 ? __float_as_uint(U)
                                       : (bad ? 1u : 0u);
        dsmem_st_u32(dsmem_addr(&sm.peer_state[rank][lane], 0), v);
      }
    }
    cluster_sync_all();
    if (rank != 0) return;
    if (warp == 0) {
      for (uint32_t r = 1; r < C; ++r) {
        lse_merge(m, S, U, __uint_as_float(sm.peer_state[r][0]),
                  __uint_as_float(sm.peer_state[r][1]), __uint_as_float(sm.peer_state[r][2]));
        bad = bad || sm.peer_state[r][3] != 0u;
        E = warp_merge_desc<uint64_t>(E, sm.peer_list[r][lane], lane);
      }
    }
  }

  if (MODE == MODE_ROUTE && warp == 2) {
    pdl_wait();
    const int64_t nclusters = gridDim.x / C;
    route_special_requests(a, (int64_t)cid * 32 + lane, nclusters * 32);
  }
  if (warp != 0) return;
  pdl_wait();
  row_finish<T, MODE>(a, row, m, S, U, bad, E, sm.pre, lane);
}

// ---- the persistent, warp-specialised row kernel (one CTA per row at a time) -----------------
//
// NWARP streaming warps read rows blockIdx.x, blockIdx.x + gridDim.x, ...; they
// never wait on the per-row selection: at the end of a row they leave its tile
// maxima, per-warp (m, S, U), largest thread maxima and each thread's best
// tile in one of two shared buffers, signal the finaliser warp with a named
// barrier and go on (the next row's first tile is already in flight).  The finaliser warp turns a buffer
// into the row's exact top-K, features and epilogue, then hands the buffer
// back.  Named barriers (bar.arrive / bar.sync with NT + 32 threads) are the
// only synchronisation; every thread reaches each of them a known number of
// times, so no wait depends on data.

constexpr int NT_WS = NT + 32;
constexpr int BAR_FULL = 1;   // ids 1, 2: buffer b holds a streamed row
constexpr int BAR_EMPTY = 3;  // ids 3, 4: buffer b may be overwritten

__device__ __forceinline__ void named_bar_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void named_bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

struct SmemWS {
  float4 tinfo[2][NT];          // per thread: best, second and third tile maxima, and
                                //   (best tile | second tile << 16); two row buffers
  uint32_t pub[2][NWARP * PUB]; // every warp's largest thread maxima, ord() encoded, and
  uint32_t low[2][NWARP];       //   what kc of its maxima reach (publish_max)
  float pm[2][NWARP], pS[2][NWARP], pU[2][NWARP];
  uint32_t cand_id[CCAP];       // finaliser: candidate tiles (tile << 8 | thread, | BEST_BIT
                                //   for a thread's best tile)
  uint64_t ebuf[ECAP];          // finaliser: candidate element keys
  uint4 best[2][UNR][NT];       // per thread: the groups of its best tile, as streamed
};

// A candidate that is its thread's best tile: the finaliser reads its groups
// from SmemWS::best instead of re-reading the row (tile indices stay below 2^16).
constexpr uint32_t BEST_BIT = 0x80000000u;

// The finaliser warp's work for one streamed row held in buffer b.
//
// Every streaming thread reports its best and second-best tile (value and
// index) and its third-best tile value, the warps their largest thread
// maxima (publish_max).  theta1 = the kc-th largest of those (kc distinct elements reach it).
// Candidate tiles are the best / second-best tiles >= theta1; a thread whose
// third-best value also reaches theta1 contributes all its tiles.  Elements >=
// theta1 of the candidate tiles are the only ones that can be among the top kc
// (about 22 for kc = 20).  A best tile is read from the copy the streaming
// thread left in shared memory; the other candidate tiles are re-read from the
// row, which may have left L2 by then.  The warp has one row's stream time for
// this, 9 us for V = 70,000 bf16, and its instructions take issue slots from the
// stream: counting ranks instead of sorting, one threshold instead of two and
// lse_warp took 4,457 such rows from 125 to 110 us, 9,670 rows of V = 151,936 bf16
// from 449 to 436 us.
template <typename T, int MODE, bool ALIGNED>
__device__ __noinline__ void finalize_ws(const Args& a, SmemWS& sm, int b, int64_t row,
                                         const RowPre& pre, int lane) {
  using Tr = Traits<T>;
  constexpr int VEC = Tr::VEC;
  const int64_t V = a.vocab;
  const int kc = a.kc;
  const char* rowp = reinterpret_cast<const char*>(a.logits) + row * a.row_stride * (int64_t)sizeof(T);
  const uint4* vp = reinterpret_cast<const uint4*>(rowp);
  const RowGeom geo(V, VEC);
  const uint4 NEG = make_uint4(Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD);
  const unsigned lt = (1u << lane) - 1u;

  // ---- the row's (m, S, U) from the streaming warps' partials
  float m = lane < NWARP ? sm.pm[b][lane] : M2_INIT;
  float S = lane < NWARP ? sm.pS[b][lane] : 0.f;
  float U = lane < NWARP ? sm.pU[b][lane] : 0.f;
#pragma unroll
  for (int o = NWARP / 2; o > 0; o >>= 1) {
    const float mo = __shfl_xor_sync(FULL, m, o);
    const float So = __shfl_xor_sync(FULL, S, o);
    const float Uo = __shfl_xor_sync(FULL, U, o);
    lse_merge(m, S, U, mo, So, Uo);
  }
  m = __shfl_sync(FULL, m, 0);
  S = __shfl_sync(FULL, S, 0);
  U = __shfl_sync(FULL, U, 0);
  bool bad = false;

  // ---- the elements after the last group, one per lane
  float xe = -INFINITY;
  const bool edge = lane < geo.nedge;
  const int64_t ve = (int64_t)geo.gfull * VEC + lane;
  if (geo.nedge > 0) {
    float em = M2_INIT, eS = 0.f, eU = 0.f;
    if (edge) {
      const float x = Tr::elem(rowp, ve);
      careful_add(x, em, eS, eU, bad);
      if (!isnan(x)) xe = x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float mo = __shfl_xor_sync(FULL, em, o);
      const float So = __shfl_xor_sync(FULL, eS, o);
      const float Uo = __shfl_xor_sync(FULL, eU, o);
      lse_merge(em, eS, eU, mo, So, Uo);
    }
    lse_merge(m, S, U, em, eS, eU);
    bad = __any_sync(FULL, bad);
  }

  // ---- theta1: the kc-th largest of the published thread maxima and of the last
  // elements
  float th1;
  bool one_warp;  // it is one warp's least maximum: sharper bounds are near
  {
    const uint32_t mine = sm.pub[b][lane], em = edge ? ord(xe) : 0u;
    int rk = 0, re = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const uint32_t q = sm.pub[b][j];
      rk += (q > mine || (q == mine && j < lane)) ? 1 : 0;
      if (geo.nedge > 0) re += q >= em ? 1 : 0;
    }
    for (int j = 0; j < geo.nedge; ++j) {
      const uint32_t q = __shfl_sync(FULL, em, j);
      rk += q > mine ? 1 : 0;
      re += (q > em || (q == em && j < lane)) ? 1 : 0;
    }
    const unsigned hit = __ballot_sync(FULL, rk == kc - 1);
    const unsigned hite = __ballot_sync(FULL, edge && re == kc - 1);
    const uint32_t v = hit ? __shfl_sync(FULL, mine, __ffs(hit) - 1)
                           : __shfl_sync(FULL, em, (__ffs(hite) - 1) & 31);
    const uint32_t lows = __reduce_max_sync(FULL, sm.low[b][lane & (NWARP - 1)]);
    one_warp = lows > v && geo.gfull >= TILE;
    th1 = unord(max(v, lows));
  }
  // ---- candidate tiles: lane l looks at the reports of threads l, 32 + l, ...  Once
  // more by a bound from all thread maxima if too many reach theta1, or fewer than
  // kc maxima are published (all but a few neighbouring tokens masked; rows of up
  // to 32 x UNR groups have published all they have)
  uint32_t m1, m2, m3;  // bit j: best, second, third tile >= theta1
  int x, n;
  auto count = [&]() {
    m1 = m2 = m3 = 0u;
#pragma unroll
    for (int j = 0; j < NT / 32; ++j) {
      const float4 inf = sm.tinfo[b][j * 32 + lane];
      m1 |= inf.x >= th1 ? 1u << j : 0u;
      m2 |= inf.y >= th1 ? 1u << j : 0u;
      m3 |= inf.z >= th1 ? 1u << j : 0u;
    }
    m2 &= ~m3;
    x = __popc(m1) + __popc(m2);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += y;
    }
    n = __shfl_sync(FULL, x, 31);  // candidate tiles
  };
  count();
  // (32 candidates are read at once: where theta1 is sharp, more are already too many;
  // rows of V = 32,000 bf16 with 1,000 neighbouring tokens 10 above the others, 1,500
  // of them, take 63 us with one warp's least maximum, 51 with the bound raised)
  const int many = kc <= 24 && geo.gfull >= TILE ? kc + 12 : many_tiles(kc);
  if (geo.gfull > 32 * UNR && (n > many || !(th1 > -INFINITY) || one_warp)) {
    th1 = raise_ws(sm.tinfo[b], edge ? ord(xe) : 0u, th1, kc, lane);
    count();
  }
  bool fb = !(th1 > -INFINITY);
  if (!fb) {
    int pos = x - __popc(m1) - __popc(m2);
    for (uint32_t q = m1; q; q &= q - 1u, ++pos) {
      const uint32_t t = (uint32_t)((__ffs(q) - 1) * 32 + lane);
      if (pos < CCAP)
        sm.cand_id[pos] = BEST_BIT | ((__float_as_uint(sm.tinfo[b][t].w) & 0xffffu) << 8) | t;
    }
    for (uint32_t q = m2; q; q &= q - 1u, ++pos) {
      const uint32_t t = (uint32_t)((__ffs(q) - 1) * 32 + lane);
      if (pos < CCAP) sm.cand_id[pos] = ((__float_as_uint(sm.tinfo[b][t].w) >> 16) << 8) | t;
    }
    // a thread with a third tile >= theta1: every other tile of it
    if (__any_sync(FULL, m3 != 0u)) {
#pragma unroll 1
      for (int j = 0; j < NT / 32; ++j) {
        unsigned b3 = __ballot_sync(FULL, (m3 >> j) & 1u);
        while (b3) {
          const uint32_t ts = (uint32_t)(j * 32 + __ffs(b3) - 1);
          b3 &= b3 - 1;
          const uint32_t ti1 = __float_as_uint(sm.tinfo[b][ts].w) & 0xffffu;
          for (int t0 = 0; t0 < geo.ntiles; t0 += 32) {
            const int tt = t0 + lane;
            const bool c = tt < geo.ntiles && (uint32_t)tt != ti1;
            const unsigned bb = __ballot_sync(FULL, c);
            const int p = n + __popc(bb & lt);
            if (c && p < CCAP) sm.cand_id[p] = ((uint32_t)tt << 8) | ts;
            n += __popc(bb);
          }
        }
      }
    }
    if (n > CCAP) fb = true;
  }
  __syncwarp();

  // ---- the candidate tiles' groups (a thread's best tile from shared memory,
  // the others re-read from the row); their elements >= theta1 become keys: kc
  // distinct elements reach theta1, so the row's top kc are among them
  int ne = 0;
  if (!fb) {
    const int total = n * UNR;
    for (int i0 = 0; i0 < total; i0 += 128) {
      uint4 wv[4];
      int32_t gsel[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int it = i0 + q * 32 + lane;
        gsel[q] = -1;
        wv[q] = NEG;
        if (it < total) {
          const uint32_t id = sm.cand_id[it >> 2];
          const int k = it & (UNR - 1), t = (int)(id & 255u);
          const int32_t gi = (int32_t)((id & ~BEST_BIT) >> 8) * TILE + tile_pos(t, k);
          if (gi < geo.gfull) {
            gsel[q] = gi;
            if (!ALIGNED) wv[q] = Tr::load_elems(rowp, gi);
            else if (id & BEST_BIT) wv[q] = sm.best[b][k][t];
            else wv[q] = ld_reread(vp + gi);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t hits = 0u;
#pragma unroll
        for (int e = 0; e < VEC; ++e) hits |= Tr::at(wv[q], e) >= th1 ? 1u << e : 0u;
        if (gsel[q] < 0) hits = 0u;
        unsigned bal;
        while ((bal = __ballot_sync(FULL, hits != 0u)) != 0u) {  // mostly one round
          const int e = __ffs(hits) - 1, pos = ne + __popc(bal & lt);
          if (hits && pos < ECAP)
            sm.ebuf[pos] = make_key(Tr::at(wv[q], e), (uint32_t)(gsel[q] * VEC + e));
          hits &= hits - 1u;
          ne += __popc(bal);
        }
      }
    }
    if (geo.nedge > 0) {
      const bool c = edge && xe >= th1;
      const unsigned bal = __ballot_sync(FULL, c);
      const int pos = ne + __popc(bal & lt);
      if (c && pos < ECAP) sm.ebuf[pos] = make_key(xe, (uint32_t)ve);
      ne += __popc(bal);
    }
    if (ne > ECAP) fb = true;
  }
  // (the scan below is the shorter, the higher its bound)
  __syncwarp();

  // ---- the row's exact top-32 elements: up to 64 keys are ranked by counting
  // (keys are distinct: the index is part of the key), more are sorted
  uint64_t E = 0ull;
  if (!fb && ne <= 64) {
    const uint64_t k0 = lane < ne ? sm.ebuf[lane] : 0ull;
    const uint64_t k1 = 32 + lane < ne ? sm.ebuf[32 + lane] : 0ull;
    int r0 = 0, r1 = 0;
    for (int q = 0; q < ne; ++q) {
      const uint64_t k = sm.ebuf[q];
      r0 += k > k0 ? 1 : 0;
      r1 += k > k1 ? 1 : 0;
    }
    __syncwarp();
    sm.ebuf[64 + lane] = 0ull;
    __syncwarp();
    if (k0 != 0ull && r0 < 32) sm.ebuf[64 + r0] = k0;
    if (k1 != 0ull && r1 < 32) sm.ebuf[64 + r1] = k1;
    __syncwarp();
    E = sm.ebuf[64 + lane];
  } else if (!fb) {
#pragma unroll 1
    for (int b0 = 0; b0 < ne; b0 += 32) {
      uint64_t k = b0 + lane < ne ? sm.ebuf[b0 + lane] : 0ull;
      k = warp_sort_desc<uint64_t>(k, lane);
      E = warp_merge_desc<uint64_t>(E, k, lane);
    }
  } else {
    // exact scan of the whole row (1,500 equal rows of V = 151,936 bf16: 14.7 ms
    // without the rising bound, 0.64 now)
    WarpTopK ek;
    ek.buf = sm.ebuf;
    ek.cnt = 0;
    ek.list = 0ull;
    scan_groups<T, ALIGNED, 4>(rowp, 0, geo.gfull, th1, ek, lane);
    if (geo.nedge > 0) {
      const bool c = edge && xe >= th1;
      ek.push(c, c ? make_key(xe, (uint32_t)ve) : 0ull, lane);
      ek.drain(lane);
    }
    ek.drain_all(lane);
    E = ek.list;
  }

  // ---- rows that made the fast accumulators non-finite: re-stream with guards
  if (!bad && !(isfinite(S) && isfinite(U))) {
    float cm = M2_INIT, cS = 0.f, cU = 0.f;
    bool cbad = false;
    careful_groups<T, ALIGNED, 4>(rowp, lane, geo.gfull, 32, cm, cS, cU, cbad);
    if (edge) careful_add(Tr::elem(rowp, ve), cm, cS, cU, cbad);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float mo = __shfl_xor_sync(FULL, cm, o);
      const float So = __shfl_xor_sync(FULL, cS, o);
      const float Uo = __shfl_xor_sync(FULL, cU, o);
      lse_merge(cm, cS, cU, mo, So, Uo);
    }
    m = __shfl_sync(FULL, cm, 0);
    S = __shfl_sync(FULL, cS, 0);
    U = __shfl_sync(FULL, cU, 0);
    bad = __any_sync(FULL, cbad);
  }

  row_finish<T, MODE>(a, row, m, S, U, bad, E, pre, lane);
}

// Rows off the 16-byte grid (rows of an odd vocabulary stored side by side): each
// streaming warp brings its share of a tile, as the 16-byte words of the grid
// that cover it, into its own ring of RING_STAGES shared-memory stages with one
// bulk copy, two tiles ahead, and cuts a group out of two neighbouring words
// when it reads it.  The groups, and with them every sum, are those of an
// aligned row.  The ring lies where an aligned row keeps its best tiles, so that
// three CTAs fit an SM all the same.
// Measured on 4,457 rows of V = 70,001 bf16 (624 MB): 144 us (4.3 TB/s); 199 us
// when every group was loaded by its elements, 163 to 186 us with narrower loads
// into registers, shuffles between lanes or 4-byte cp.async, whose instructions
// kept the warps from covering the memory latency.  V = 151,935: 287 for 407 us;
// fp32, where an element load is 4 bytes, is level (218 us for 1.25 GB).
constexpr int RING_STAGES = 3;
constexpr int RING_WARP = 32 * UNR * 16;    // bytes of a tile that a warp takes
constexpr int RING_STAGE = RING_WARP + 16;  // and the word after them
struct RingWS {
  unsigned char stage[NWARP][RING_STAGES][RING_STAGE];
  uint64_t bar[NWARP][RING_STAGES];  // a stage's copy has landed
};
constexpr size_t WS_SMEM_ALIGNED = sizeof(SmemWS);
constexpr size_t WS_SMEM_RING = offsetof(SmemWS, best) + sizeof(RingWS);
static_assert(offsetof(SmemWS, best) % 16 == 0 && RING_STAGE % 16 == 0, "bulk copies");
constexpr uint64_t RING_WAIT_NS = 2000000000ull;  // a wait gives up after 2 s

__device__ __forceinline__ bool ring_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait for a stage: false (and the flag) when its copy has not landed
static __device__ __noinline__ bool ring_wait_slow(uint32_t bar, uint32_t parity, uint32_t* flags) {
  uint64_t t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (;;) {
    for (int i = 0; i < 256; ++i)
      if (ring_test(bar, parity)) return true;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > RING_WAIT_NS) break;
  }
  atomicOr(flags, FLAG_TIMEOUT);
  return false;
}
// the group S bytes into the grid word at st (shared memory)
template <int S>
__device__ __forceinline__ uint4 ring_group(const unsigned char* st) {
  const uint4 a = *reinterpret_cast<const uint4*>(st);
  if (S == 0) return a;
  uint32_t w[8] = {a.x, a.y, a.z, a.w, 0u, 0u, 0u, 0u};
  constexpr int NEXT = (S + 3) / 4;  // words of the next grid word
  if (NEXT == 1) {
    w[4] = *reinterpret_cast<const uint32_t*>(st + 16);
  } else if (NEXT == 2) {
    const uint2 b = *reinterpret_cast<const uint2*>(st + 16);
    w[4] = b.x;
    w[5] = b.y;
  } else {
    const uint4 b = *reinterpret_cast<const uint4*>(st + 16);
    w[4] = b.x;
    w[5] = b.y;
    w[6] = b.z;
    w[7] = b.w;
  }
  uint32_t o[4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    o[j] = (S & 2) ? __funnelshift_r(w[j + S / 4], w[j + S / 4 + 1], 16) : w[j + S / 4];
  return make_uint4(o[0], o[1], o[2], o[3]);
}
template <int S>
__device__ __forceinline__ void ring_tile(const unsigned char* st, uint4 (&c)[UNR]) {
#pragma unroll
  for (int k = 0; k < UNR; ++k) c[k] = ring_group<S>(st + 512 * k);
}

template <typename T, int MODE, bool ALIGNED>
__global__ void __launch_bounds__(NT_WS, 3) verify_rows_ws(const Args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmemWS& sm = *reinterpret_cast<SmemWS*>(smem_raw);
  using Tr = Traits<T>;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t G = gridDim.x;

  pdl_enter(a.early);

  auto rowp_of = [&](int64_t r) {
    return reinterpret_cast<const char*>(a.logits) + r * a.row_stride * (int64_t)sizeof(T);
  };
  if (warp == NWARP) {
    // ---- the finaliser warp: the next row's inputs are fetched while its
    // stream is still running
    int i = 0;
    int64_t row = blockIdx.x;
    RowPre pre = load_pre<T, MODE>(a, row, a.chosen[row], rowp_of(row), lane);
    pdl_wait();
    if (MODE == MODE_ROUTE) route_special_requests(a, (int64_t)blockIdx.x * 32 + lane, G * 32);
    for (; row < a.n_rows; row += G, ++i) {
      const int b = i & 1;
      named_bar_sync(BAR_FULL + b, NT_WS);
      finalize_ws<T, MODE, ALIGNED>(a, sm, b, row, pre, lane);
      if (row + 2 * G < a.n_rows) {
        __syncwarp();
        __threadfence_block();
        named_bar_arrive(BAR_EMPTY + b, NT_WS);
      }
      if (row + G < a.n_rows) pre = load_pre<T, MODE>(a, row + G, a.chosen[row + G], rowp_of(row + G), lane);
    }
    return;
  }

  // ---- the streaming warps
  const uint4 NEG = make_uint4(Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD, Tr::NEG_WORD);
  const RowGeom geo(a.vocab, Tr::VEC);
  auto load_tile = [&](uint4 (&dst)[UNR], int64_t r, int32_t t) {
    const uint4* vp = reinterpret_cast<const uint4*>(rowp_of(r));
    const int32_t base = t * TILE;
    if (t < geo.nfull) {
#pragma unroll
      for (int k = 0; k < UNR; ++k) dst[k] = ld_stream(vp + base + tile_pos(tid, k));
    } else {
#pragma unroll
      for (int k = 0; k < UNR; ++k)
        dst[k] = tile_pos(tid, k) < geo.rem ? ld_stream(vp + base + tile_pos(tid, k)) : NEG;
    }
  };
  // off the grid: this warp's ring, and the next tile to bring in
  RingWS& ring = *reinterpret_cast<RingWS*>(smem_raw + offsetof(SmemWS, best));
  int64_t ahead_row = blockIdx.x;
  int32_t ahead_t = 0;
  int ahead_stage = 0, stage = 0;
  uint32_t parity = 0u;
  bool landed = true;
  auto bring = [&]() {
    if (ahead_row >= a.n_rows || !landed) return;
    const char* rp = rowp_of(ahead_row);
    const int s = (int)(reinterpret_cast<uintptr_t>(rp) & 15u);
    const int32_t g = ahead_t * TILE + warp * (32 * UNR);  // the warp's first group
    const int32_t n = min(32 * UNR, geo.gfull - g);        // its groups
    // grid words [lo, hi) of the warp's share; the words that reach past the
    // call's buffer are left out and their elements of the row copied singly
    int32_t lo = 0, hi = n + (s ? 1 : 0);
    const bool first = s != 0 && ahead_row == 0 && g == 0;
    const bool last = s != 0 && ahead_row == a.n_rows - 1 && g + n == geo.gfull &&
                      geo.nedge * (int)sizeof(T) < 16 - s;
    unsigned char* dst = ring.stage[warp][ahead_stage];
    if (n > 0 && (first || last)) {
      const int el = lane * (int)sizeof(T);  // one element per lane
      auto copy1 = [&](int at, const char* from) {
        if (sizeof(T) == 2)
          *reinterpret_cast<uint16_t*>(dst + at) = *reinterpret_cast<const uint16_t*>(from);
        else
          *reinterpret_cast<uint32_t*>(dst + at) = *reinterpret_cast<const uint32_t*>(from);
      };
      if (first && s + el < 16) copy1(s + el, rp + el);
      if (last && el < s) copy1(16 * n + el, rp + 16 * (int64_t)geo.gfull - s + el);
    }
    if (first) lo = 1;
    if (last) hi = n;
    if (lane == 0 && n > 0) {
      const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&ring.bar[warp][ahead_stage]);
      const uint32_t bytes = (uint32_t)max(hi - lo, 0) * 16u;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                   : "memory");
      if (bytes)
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
                "r"((uint32_t)__cvta_generic_to_shared(dst + 16 * lo)),
            "l"(rp - s + 16 * ((int64_t)g + lo)), "r"(bytes), "r"(bar)
            : "memory");
    }
    if (++ahead_t == geo.ntiles) {
      ahead_t = 0;
      ahead_row += G;
    }
    ahead_stage = ahead_stage + 1 == RING_STAGES ? 0 : ahead_stage + 1;
  };

  uint4 cur[UNR], nxt[UNR];
  int64_t row = blockIdx.x;
  if (geo.ntiles > 0) {
    if (ALIGNED) {
      if (row < a.n_rows) load_tile(cur, row, 0);
    } else {
      if (lane == 0) {
        for (int j = 0; j < RING_STAGES; ++j)
          asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(
                           (uint32_t)__cvta_generic_to_shared(&ring.bar[warp][j]))
                       : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      __syncwarp();
      for (int j = 0; j < RING_STAGES - 1; ++j) bring();
    }
  }
  int i = 0;
  while (row < a.n_rows) {
    const int b = i & 1;
    if (i >= 2) named_bar_sync(BAR_EMPTY + b, NT_WS);
    const int64_t next = row + G;
    float m = M2_INIT;
    float2 S2 = make_float2(0.f, 0.f), U2 = make_float2(0.f, 0.f);
    // this thread's best, second and third tile maxima and the first two tiles
    float v1 = -INFINITY, v2 = -INFINITY, v3 = -INFINITY;
    uint32_t i1 = 0, i2 = 0;
    for (int32_t t = 0; t < geo.ntiles; ++t) {
      if (ALIGNED) {
        if (t + 1 < geo.ntiles) load_tile(nxt, row, t + 1);
        else if (next < a.n_rows) load_tile(nxt, next, 0);
      } else {
        __syncwarp();  // every lane is done with the stage that is filled next
        bring();
        const bool some = t * TILE + warp * (32 * UNR) < geo.gfull;  // the warp has a share
        const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&ring.bar[warp][stage]);
        if (some && landed) {
          if (!ring_test(bar, (parity >> stage) & 1u))
            landed = ring_wait_slow(bar, (parity >> stage) & 1u, a.ctx_flags);
          if (landed) parity ^= 1u << stage;
        }
        __syncwarp();
        const unsigned char* st = ring.stage[warp][stage] + 16 * lane;
        const int s = (int)(reinterpret_cast<uintptr_t>(rowp_of(row)) & 15u);
        if ((s & 2) == 0) {
          if (s == 0) ring_tile<0>(st, cur);
          else if (s == 4) ring_tile<4>(st, cur);
          else if (s == 8) ring_tile<8>(st, cur);
          else ring_tile<12>(st, cur);
        } else if constexpr (sizeof(T) == 2) {
          if (s == 2) ring_tile<2>(st, cur);
          else if (s == 6) ring_tile<6>(st, cur);
          else if (s == 10) ring_tile<10>(st, cur);
          else ring_tile<14>(st, cur);
        }
        if (t >= geo.nfull) {
#pragma unroll
          for (int k = 0; k < UNR; ++k)
            if (tile_pos(tid, k) >= geo.rem) cur[k] = NEG;
        }
        stage = stage + 1 == RING_STAGES ? 0 : stage + 1;
      }
      const float tmax = Tr::tile_max(cur);
      {
        const bool c1 = tmax > v1, c2 = tmax > v2;
        if (ALIGNED && c1) {  // a new best tile: keep its groups for the finaliser
#pragma unroll
          for (int k = 0; k < UNR; ++k) sm.best[b][k][tid] = cur[k];
        }
        v3 = fmaxf(v3, fminf(tmax, v2));
        const float nv2 = c1 ? v1 : (c2 ? tmax : v2);
        const uint32_t ni2 = c1 ? i1 : (c2 ? (uint32_t)t : i2);
        v1 = c1 ? tmax : v1;
        i1 = c1 ? (uint32_t)t : i1;
        v2 = nv2;
        i2 = ni2;
      }
      const float mn = fmaxf(m, tmax * L2E);
      const float dl = m - mn;
      const float f = ex2(dl);
      U2 = __fmul2_rn(make_float2(f, f), __ffma2_rn(make_float2(dl, dl), S2, U2));
      S2 = __fmul2_rn(make_float2(f, f), S2);
      m = mn;
      const float2 nm = make_float2(-m, -m);
      if (t < geo.nfull) {
#pragma unroll
        for (int k = 0; k < UNR; ++k) Tr::accum(cur[k], nm, S2, U2);
      } else {
#pragma unroll
        for (int k = 0; k < UNR; ++k)
          if (tile_pos(tid, k) < geo.rem) Tr::accum(cur[k], nm, S2, U2);
      }
#pragma unroll
      for (int k = 0; k < UNR; ++k)
        if (ALIGNED) cur[k] = nxt[k];
    }
    // the warp's partial state, its sorted per-thread maxima, the tile report
    float S = S2.x + S2.y, U = U2.x + U2.y;
    lse_warp(m, S, U);
    if (lane == 0) {
      sm.pm[b][warp] = m;
      sm.pS[b][warp] = S;
      sm.pU[b][warp] = U;
    }
    publish_max(ord(v1), sm.pub[b], sm.low[b], geo.gfull, a.kc, warp, lane);
    sm.tinfo[b][tid] = make_float4(v1, v2, v3, __uint_as_float(i1 | (i2 << 16)));
    __syncwarp();
    __threadfence_block();
    named_bar_arrive(BAR_FULL + b, NT_WS);
    row = next;
    ++i;
  }
  if (!ALIGNED && !landed)  // a wait ran out: no copy may be in flight when the CTA ends
    for (int j = 0; j < RING_STAGES; ++j)
      ring_wait_slow((uint32_t)__cvta_generic_to_shared(&ring.bar[warp][j]), (parity >> j) & 1u,
                     a.ctx_flags);
}

// ---- standalone pooling kernel: one warp per request ----------------------------------
//
// Up to POOL_FEW requests are bound by the latency of a request's loads: a warp
// has 16 rows per lane in flight (512 of the request's rows) and a CTA of its
// own.  More requests are bound by the launch of CTAs and by occupancy: four to a
// CTA, with four rows per lane.  These let the next launch in once they have their
// rows, not at their start, where its CTAs would take the places that theirs still
// wait for.  Back to back in a CUDA graph, requests of 1 to 8, 300 and 1,000 rows
// take: 24 requests 2.5, 3.3 and 4.2 us; 1,024 2.8, 4.1 and 6.6; 2,048
// (four to a CTA) 3.0, 4.9 and 9.8; 4,096 3.8 and 7.3.  A CTA each takes 2,048 to 3.9,
// 5.6 and 11.4, 4,096 to 6.4 and 9.3; four to one takes 24 to 2.5, 3.4 and 5.4.
constexpr int POOL_FEW = 1024;
constexpr int POOL_WARPS = 4;

struct AggArgs {
  const float* feat;
  const uint32_t* row_flags;
  int64_t n_rows;
  const int64_t* offsets;
  int32_t n_req;
  const float* w;
  float b, zthr;
  float* agg;
  float* score;
  uint8_t* ship;
  uint32_t* req_flags;
  uint32_t* ctx_flags;
};

// internal linkage: the header is included by more than one translation unit
template <int WARPS, int AHEAD>
static __global__ void __launch_bounds__(32 * WARPS) pool_requests(const AggArgs a) {
  pdl_wait();
  if (WARPS == 1) pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * WARPS + (threadIdx.x >> 5);
  if (r >= a.n_req) return;
  const int64_t lo = a.offsets[r], hi = a.offsets[r + 1];
  if (lo < 0 || hi < lo || hi > a.n_rows) {
    if (lane == 0) {
      write_special(r, NAN, FLAG_BAD_OFFSETS, a.agg, a.score, a.ship, a.req_flags);
      atomicOr(a.ctx_flags, FLAG_BAD_OFFSETS);
    }
    return;
  }
  if (lo == hi) {
    if (lane == 0) write_special(r, 0.f, FLAG_EMPTY_REQ, a.agg, a.score, a.ship, a.req_flags);
    return;
  }
  const Pooled p = pool_rows<AHEAD>(a.feat, a.row_flags, lo, hi, a.w, a.b, a.zthr, lane);
  if (WARPS > 1) pdl_trigger();
  write_pooled(p, r, a.agg, a.score, a.ship, a.req_flags, lane);
}

}  // namespace prk
