// sw_selftest_wait, sw_selftest_trace: the library's bounded device waits, made
// to run out.
// Every wait between warps or CTAs in the kernels gives up after a clock
// budget, reports SW_ETIMEOUT and returns, so that a failure leaves the CUDA
// context usable.  This entry point runs the two wait helpers the kernels use
// against a condition that nothing fulfils, so that a test can check that
// they give up and report it, without faulting or hanging a GPU.
#include <cstdio>

#include "devutil.cuh"
#include "host_pool.h"
#include "internal.h"
#include "../../include/swgb.h"

namespace swgb {
namespace {

__global__ void wait_selftest_kernel(int which, long long budget, const int32_t *flag, int32_t *status) {
  __shared__ uint64_t bar;
  if (which == 0) {
    // a progress counter that nothing raises (the pair-band kernel's waits)
    const int32_t v = wait_flag_value(flag, 1, budget);
    *status = v >= 1 ? SW_OK : SW_ETIMEOUT;
  } else {
    // an mbarrier phase that nothing completes (the profile-chunk waits of
    // the inter- and intra-task kernels; their fixed budget of ~1 s)
    mbar_init(&bar, 1);
    fence_mbar_init();
    *status = mbar_wait_bounded(&bar, 0u) ? SW_OK : SW_ETIMEOUT;
  }
}

int st_fail(int code, const char *msg) { return set_last_error(code, msg); }

int st_cuda(cudaError_t e, const char *what, const char *call = "sw_selftest_wait") {
  char buf[256];
  snprintf(buf, sizeof buf, "%s: %s: %s", call, what, cudaGetErrorString(e));
  return set_last_error(e == cudaErrorMemoryAllocation ? SW_ENOMEM : SW_ECUDA, buf);
}

}  // namespace
}  // namespace swgb

using namespace swgb;

extern "C" int sw_selftest_wait(int32_t which, int64_t budget_cycles, int32_t *status_out, void *stream) {
  clear_last_error();
  if (!status_out) return st_fail(SW_EINVAL, "sw_selftest_wait: null status_out");
  if (which != 0 && which != 1) return st_fail(SW_EINVAL, "sw_selftest_wait: which must be 0 or 1");
  if (which == 0 && (budget_cycles <= 0 || budget_cycles > ((int64_t)1 << 32)))
    return st_fail(SW_EINVAL, "sw_selftest_wait: budget_cycles must lie in (0, 2^32]");
  cudaStream_t s = (cudaStream_t)stream;
  int32_t *d = nullptr;  // [0] the flag, [1] the status
  cudaError_t e = cudaMallocAsync((void **)&d, 2 * sizeof(int32_t), s);
  if (e != cudaSuccess) return st_cuda(e, "device allocation");
  e = cudaMemsetAsync(d, 0, 2 * sizeof(int32_t), s);
  if (e == cudaSuccess) {
    wait_selftest_kernel<<<1, 1, 0, s>>>(which, (long long)budget_cycles, d, d + 1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(status_out, d + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(d, s);
  const cudaError_t e2 = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) return st_cuda(e, "run");
  return SW_OK;
}

extern "C" int sw_selftest_trace(int64_t budget_cycles, int32_t *status_out, int32_t *score_out, void *stream) {
  clear_last_error();
  if (!status_out || !score_out) return st_fail(SW_EINVAL, "sw_selftest_trace: null output");
  if (budget_cycles <= 0 || budget_cycles > ((int64_t)1 << 36))
    return st_fail(SW_EINVAL, "sw_selftest_trace: budget_cycles must lie in (0, 2^36]");
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0, sms = 1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return st_cuda(e, "device", "sw_selftest_trace");
  TraceHit hit{};
  hit.nb = 64 * sms + 1;  // (one more than an SM's 64 warps, on every SM)
  hit.m = hit.nb * trace_rows_per_band();
  hit.n = hit.npad = kColBlock;
  const int64_t dir_words = (int64_t)hit.nb * (hit.npad + 32) * 32;
  // one block, 256-byte aligned parts
  size_t bytes = 0;
  auto part = [&](size_t n) {
    const size_t at = bytes;
    bytes += (n + 255) / 256 * 256;
    return at;
  };
  const size_t o_q = part((size_t)hit.m), o_t = part((size_t)hit.npad), o_sub = part(kAlphabet * kAlphabet),
               o_hit = part(sizeof hit), o_bandhit = part(4 * (size_t)hit.nb), o_words = part(8);
  const size_t o_left = bytes;  // from here on: what other work left
  const size_t o_best = part(sizeof(int4) * (size_t)hit.nb), o_ops = part((size_t)hit.m + hit.n),
               o_res = part(sizeof(TraceResult)), o_dirs = part(4 * (size_t)dir_words);
  void *block = nullptr;
  if ((e = pool_alloc(&block, bytes, s)) != cudaSuccess) return st_cuda(e, "device allocation", "sw_selftest_trace");
  uint8_t *p = (uint8_t *)block;
  int8_t sub[kAlphabet * kAlphabet];
  for (int i = 0; i < kAlphabet * kAlphabet; ++i) sub[i] = i % (kAlphabet + 1) ? -1 : 1;
  TraceArgs a{};
  a.qres = p + o_q;
  a.tres = p + o_t;
  a.tres_bytes = hit.npad;
  a.submat = (const int8_t *)(p + o_sub);
  a.hits = (const TraceHit *)(p + o_hit);
  a.band_hit = (const int32_t *)(p + o_bandhit);
  a.nhits = 1;
  a.nbands = hit.nb;
  a.band_counter = (int32_t *)(p + o_words);
  a.status = a.band_counter + 1;
  a.wait_cycles = budget_cycles;
  a.best = (int4 *)(p + o_best);
  a.ops = p + o_ops;
  a.results = (TraceResult *)(p + o_res);
  a.dirs = (uint32_t *)(p + o_dirs);
  a.dir_words = dir_words;
  a.sc.go = 2;
  a.sc.ge = 1;
  a.sc.pad = -1;
  e = cudaMemsetAsync(p, 0, o_left, s);  // (both sequences: residue 0 only; every band belongs to hit 0)
  if (e == cudaSuccess) e = cudaMemsetAsync(p + o_left, 0x41, bytes - o_left, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.results, 0xff, sizeof(TraceResult), s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(p + o_sub, sub, sizeof sub, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(p + o_hit, &hit, sizeof hit, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = launch_trace(a, sms, s);
  TraceResult res{};
  int32_t words[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpyAsync(&res, a.results, sizeof res, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(words, a.band_counter, sizeof words, cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(block, s);
  const cudaError_t e2 = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) return st_cuda(e, "run", "sw_selftest_trace");
  *status_out = words[1];
  *score_out = res.score;
  return SW_OK;
}
