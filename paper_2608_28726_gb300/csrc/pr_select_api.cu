// Host side of pr_selective_metrics: argument checks, the context's sort
// workspace and the launch sequence of the kernels in pr_select.cuh.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>

#include "pr_ctx.h"
#include "pr_select.cuh"

using namespace prh;

static_assert(sizeof(prk::SelResult) == sizeof(pr_selective), "result layout");
static_assert(offsetof(prk::SelResult, n_finite) == offsetof(pr_selective, n_finite), "layout");
static_assert(offsetof(prk::SelResult, auroc) == offsetof(pr_selective, auroc), "layout");
static_assert(offsetof(prk::SelResult, acc_shipped) == offsetof(pr_selective, acc_shipped),
              "layout");

namespace {

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// shares of the pool and most buckets of a pool of n scores
struct SelShape {
  uint32_t share, shares, target, nbcap, rows;
  SelShape(int64_t n, int num_sms) {
    // two shares per SM, or as many rounds of those as a share's counts need (4e7
    // uniform scores 2.2 ms with shares of SB_SHARE, whose last round was nearly empty,
    // now 1.0), not below 4,096 items (a share pays for every bucket); a multiple of 4
    // for the vector loads
    const int64_t round = 2 * (int64_t)num_sms, rounds = (n + round * prk::SB_SHARE - 1) / (round * prk::SB_SHARE);
    const int64_t even = ((n + round * rounds - 1) / (round * rounds) + 3) & ~(int64_t)3;
    share = (uint32_t)std::min<int64_t>(prk::SB_SHARE, std::max<int64_t>(4096, even));
    shares = (uint32_t)((n + share - 1) / share);
    // a bin that holds most of a small pool is still cut into 64 buckets, whose keys
    // are counted in one go (33,000 scores just below 1: 118 us, at 1,024 a bucket 151)
    target = (uint32_t)std::max<int64_t>(
        std::min<int64_t>(prk::SB_TARGET, std::max<int64_t>(prk::SB_FEW_TARGET, n / 64)),
        (n + 8191) / 8192);
    // the workspace's bounds do not fall when n grows: n / target buckets over the
    // coarse bins', twice, and the shares
    nbcap = (uint32_t)(std::min<int64_t>(n, prk::SB_BINS) + 1 +
                       2 * std::max(std::min<int64_t>(n / prk::SB_FEW_TARGET, 65),
                                    std::min<int64_t>(n / prk::SB_TARGET, 8192)));
    rows = (uint32_t)std::min<int64_t>((n + 4095) / 4096, round * rounds);
  }
};

// byte offsets of the workspace pieces
struct SelLayout {
  size_t coarse, total, info, zeroed, plan, bkey, start, pstart, proc, parc, out, items, list, hidx, hchunk, hcnt, rel, bytes;
  SelLayout(int64_t n, const SelShape& g) {
    size_t o = 0;
    auto take = [&](size_t b) {
      const size_t at = o;
      o += align256(b);
      return at;
    };
    coarse = take(prk::SB_BINS * 4);
    total = take((size_t)g.nbcap * 8);
    info = take(32);
    zeroed = o;  // zeroed at the start of a call
    plan = take(prk::SB_BINS * 4);
    bkey = take((size_t)g.nbcap * 4);
    start = take(((size_t)g.nbcap + 1) * 4);
    pstart = take(((size_t)g.nbcap + 1) * 4);
    proc = take((size_t)g.nbcap * 8);
    parc = take((size_t)g.nbcap * 8);
    out = take(sizeof(prk::SelResult));
    items = take((size_t)n * 4);
    const size_t heavy = (size_t)(n / (prk::SB_HEAVY + 1));  // buckets with more than SB_HEAVY items
    list = take((size_t)g.nbcap * 4);
    hidx = take((size_t)g.nbcap * 4);
    hchunk = take(((size_t)(n / prk::SB_CHUNK) + heavy + 1) * 8);
    hcnt = take((heavy << prk::SB_VBITS) * 8);
    rel = take((size_t)g.rows * g.nbcap * 4);
    bytes = o;
  }
};

}  // namespace

extern "C" {

pr_status pr_selective_metrics(pr_ctx* c, const float* scores, const uint8_t* labels, int64_t n,
                               double q, pr_selective* out, void* stream) {
  if (!c || !out || n < 0 || n > 0x7fffffffLL) return PR_ERR_INVALID_ARG;
  if (!(q >= 0.0 && q <= 1.0)) return PR_ERR_INVALID_ARG;
  if (n > 0 && !scores) return PR_ERR_INVALID_ARG;
  const double nan = __builtin_nan("");
  if (n == 0) {
    memset(out, 0, sizeof *out);
    out->tau = __builtin_inff();
    out->auroc = out->auarc = out->acc_shipped = nan;
    return PR_OK;
  }
  pr_status st = set_device(c);
  if (st != PR_OK) return st;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const SelShape g(n, c->num_sms);
  const SelLayout L(n, g);
  if ((int64_t)L.bytes > c->sel_cap) {
    PR_CUDA(cudaDeviceSynchronize());  // the old workspace may still be in use
    cudaFree(c->sel_ws);
    c->sel_ws = nullptr;
    c->sel_cap = 0;
    if (cudaMalloc(&c->sel_ws, L.bytes) != cudaSuccess) {
      cudaGetLastError();
      c->sel_ws = nullptr;
      return PR_ERR_NO_MEMORY;
    }
    c->sel_cap = (int64_t)L.bytes;
  }
  const size_t share_smem = (size_t)(prk::SB_BINS + g.nbcap) * sizeof(uint32_t);
  if (!c->sel_ready) {
    const int most = (prk::SB_BINS + prk::SB_NB) * (int)sizeof(uint32_t);
    PR_CUDA(cudaFuncSetAttribute(prk::sel_count, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    PR_CUDA(cudaFuncSetAttribute(prk::sel_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    PR_CUDA(cudaFuncSetAttribute(prk::sel_heavy, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)prk::SB_BUCKET_SMEM));
    PR_CUDA(cudaFuncSetAttribute(prk::sel_bucket<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)prk::SB_BUCKET_SMEM));
    PR_CUDA(cudaFuncSetAttribute(prk::sel_bucket<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)prk::SB_BUCKET_SMEM));
    c->sel_ready = true;
  }
  char* w = static_cast<char*>(c->sel_ws);
  prk::SelArgs a;
  memset(&a, 0, sizeof a);
  a.scores = scores;
  a.labels = labels;
  a.n = (uint32_t)n;
  a.share = g.share;
  a.target = g.target;
  a.nbcap = g.nbcap;
  a.q = q;
  a.coarse = reinterpret_cast<uint32_t*>(w + L.coarse);
  a.total = reinterpret_cast<unsigned long long*>(w + L.total);
  a.info = reinterpret_cast<uint32_t*>(w + L.info);
  a.plan = reinterpret_cast<uint32_t*>(w + L.plan);
  a.bkey = reinterpret_cast<uint32_t*>(w + L.bkey);
  a.start = reinterpret_cast<uint32_t*>(w + L.start);
  a.pstart = reinterpret_cast<uint32_t*>(w + L.pstart);
  a.rel = reinterpret_cast<uint32_t*>(w + L.rel);
  a.items = reinterpret_cast<uint32_t*>(w + L.items);
  a.list = reinterpret_cast<uint32_t*>(w + L.list);
  a.hidx = reinterpret_cast<uint32_t*>(w + L.hidx);
  a.hchunk = reinterpret_cast<uint2*>(w + L.hchunk);
  a.hcnt = reinterpret_cast<unsigned long long*>(w + L.hcnt);
  a.proc = reinterpret_cast<unsigned long long*>(w + L.proc);
  a.parc = reinterpret_cast<double*>(w + L.parc);
  a.out = reinterpret_cast<prk::SelResult*>(w + L.out);
  int launches = 0;
  // one kernel of the chain, set up behind the one before it
  auto launch = [&](void (*kernel)(prk::SelArgs), unsigned grid, unsigned block,
                    size_t smem) -> pr_status {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[] = {&a};
    PR_CUDA(cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kernel), args));
    ++launches;
    return timing_mark(c, s);
  };
#define PR_LAUNCH(...)                                   \
  do {                                                   \
    if ((st = launch(__VA_ARGS__)) != PR_OK) return st; \
  } while (0)

  PR_CUDA(cudaMemsetAsync(w, 0, L.zeroed, s));
  if ((st = timing_begin(c, s)) != PR_OK) return st;
  const unsigned g_coarse =
      (unsigned)std::min<int64_t>((n + 16 * prk::SB_NT - 1) / (16 * prk::SB_NT), 4 * c->num_sms);
  PR_LAUNCH(prk::sel_coarse, g_coarse, prk::SB_NT, 0);
  PR_LAUNCH(prk::sel_plan, 1, 1024, 0);
  PR_LAUNCH(prk::sel_count, g.shares, prk::SB_NT, share_smem);
  PR_LAUNCH(prk::sel_offsets, 1, 1024, 0);
  PR_LAUNCH(prk::sel_scatter, g.shares, prk::SB_NT, share_smem);
  if (n > prk::SB_HEAVY)
    PR_LAUNCH(prk::sel_heavy,
              (unsigned)std::min<int64_t>(n / prk::SB_CHUNK + 1, 3 * c->num_sms), prk::SB_NT,
              prk::SB_BUCKET_SMEM);
  PR_LAUNCH(g.target > (uint32_t)prk::SB_LIGHT ? prk::sel_bucket<true> : prk::sel_bucket<false>,
            (unsigned)std::min<int64_t>(g.nbcap, 3 * c->num_sms), prk::SB_NT,
            prk::SB_BUCKET_SMEM);
  PR_LAUNCH(prk::sel_finish, 1, prk::SB_NT, 0);
#undef PR_LAUNCH
  g_launches.fetch_add((uint64_t)launches, std::memory_order_relaxed);
  PR_CUDA(cudaMemcpyAsync(out, a.out, sizeof *out, cudaMemcpyDeviceToHost, s));
  PR_CUDA(cudaStreamSynchronize(s));
  return PR_OK;
}

}  // extern "C"
