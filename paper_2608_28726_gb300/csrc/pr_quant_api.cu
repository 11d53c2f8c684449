// Host side of pr_quantile_score: argument checks and the launch of the
// kernel in pr_quant.cuh.
#include <cuda_runtime.h>

#include <cstring>

#include "pr_ctx.h"
#include "pr_quant.cuh"

using namespace prh;

static_assert(prk::QW_SIZE == PR_QMLP_PARAMS, "weight layout");

extern "C" {

pr_status pr_quantile_score(pr_ctx* c, const float* feat, const uint32_t* row_flags,
                            int64_t n_rows, const int64_t* offsets, int32_t n_req, const float* w,
                            float tau, float* summary, float* score, uint8_t* ship,
                            uint32_t* req_flags, void* stream) {
  if (!c || n_req < 0 || n_rows < 0 || n_rows > 0x7fffffffLL) return PR_ERR_INVALID_ARG;
  if (n_req == 0) return PR_OK;
  if (!offsets || !w || !score || !ship || !req_flags) return PR_ERR_INVALID_ARG;
  if (n_rows > 0 && !feat) return PR_ERR_INVALID_ARG;
  if (!aligned16(feat)) return PR_ERR_INVALID_ARG;  // records are read as 16-byte words
  pr_status st = set_device(c);
  if (st != PR_OK) return st;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if ((st = timing_begin(c, s)) != PR_OK) return st;
  prk::QArgs a;
  memset(&a, 0, sizeof a);
  a.feat = feat;
  a.row_flags = row_flags;
  a.n_rows = n_rows;
  a.offsets = offsets;
  a.n_req = n_req;
  a.w = w;
  a.zthr = zthreshold(tau);
  a.summary = summary;
  a.score = score;
  a.ship = ship;
  a.req_flags = req_flags;
  a.ctx_flags = c->flags;
  // Three CTAs fit an SM.  A launch of fewer than fill the GPU does not let the next
  // one in before its CTAs end: that one's would take the free places, and its last
  // ones go together on the SMs that end first (300 requests of 700 rows back to back
  // 21.0 us, 27.0 with the early set-up; of 1 to 8 rows 6.7 and 8.1; 512 ragged ones
  // 24.4 and 23.3).
  a.full = n_req >= 3 * c->num_sms ? 1 : 0;
  if (!c->qmlp_ready) {
    PR_CUDA(cudaFuncSetAttribute(prk::qmlp_requests, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(prk::Q_DYN * sizeof(uint32_t))));
    c->qmlp_ready = true;
  }
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3((unsigned)n_req);
  cfg.blockDim = dim3(prk::Q_NT);
  cfg.dynamicSmemBytes = prk::Q_DYN * sizeof(uint32_t);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[] = {&a};
  PR_CUDA(cudaLaunchKernelExC(&cfg, reinterpret_cast<void*>(&prk::qmlp_requests), args));
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return timing_mark(c, s);
}

}  // extern "C"
