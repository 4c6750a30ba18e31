// sw_traceback: one optimal local alignment per hit, on the traceback kernels
// (k_trace.cu).
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <numeric>
#include <vector>

#include "host_pool.h"
#include "internal.h"
#include "../../include/swgb.h"

namespace swgb {
namespace {

inline int64_t tr_round_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

int tr_fail(int code, const char *fmt, long long a = 0, long long b = 0) {
  char buf[256];
  snprintf(buf, sizeof buf, fmt, a, b);
  return set_last_error(code, buf);
}

int tr_cuda(cudaError_t e, const char *what) {
  char buf[256];
  snprintf(buf, sizeof buf, "sw_traceback: %s: %s", what, cudaGetErrorString(e));
  return set_last_error(e == cudaErrorMemoryAllocation ? SW_ENOMEM : SW_ECUDA, buf);
}

struct TraceScratch {
  void *block = nullptr;
  cudaStream_t s = nullptr;
  ~TraceScratch() {
    if (block) {
      cudaFreeAsync(block, s);
      cudaStreamSynchronize(s);
    }
  }
};

}  // namespace
}  // namespace swgb

using namespace swgb;

extern "C" int sw_traceback(const sw_db *db, const uint8_t *queries, const int64_t *q_offsets, int64_t n_queries,
                            const sw_hit *hits, int64_t n_hits, const int8_t *submat, int32_t gap_open,
                            int32_t gap_extend, sw_alignment *out, uint8_t *ops, int64_t ops_capacity,
                            void *stream) {
  clear_last_error();
  if (!db) return tr_fail(SW_EINVAL, "sw_traceback: null database");
  if (n_hits < 0 || n_queries < 0) return tr_fail(SW_EINVAL, "sw_traceback: negative count");
  if (n_hits == 0) return SW_OK;
  if (!hits || !out || !q_offsets || !submat) return tr_fail(SW_EINVAL, "sw_traceback: null argument");
  if (q_offsets[0] != 0) return tr_fail(SW_EINVAL, "sw_traceback: q_offsets[0] must be 0");
  for (int64_t i = 0; i < n_queries; ++i)
    if (q_offsets[i + 1] < q_offsets[i]) return tr_fail(SW_EINVAL, "sw_traceback: offsets decrease at %lld", i);
  if (q_offsets[n_queries] > 0 && !queries) return tr_fail(SW_EINVAL, "sw_traceback: null queries");
  for (int64_t i = 0; i < q_offsets[n_queries]; ++i)
    if (queries[i] >= kAlphabet) return tr_fail(SW_EINVAL, "sw_traceback: residue code %lld >= 20", queries[i]);
  int smin = 127, smax = -128;
  for (int i = 0; i < kAlphabet * kAlphabet; ++i) {
    smin = std::min<int>(smin, submat[i]);
    smax = std::max<int>(smax, submat[i]);
  }
  if (smin < -64 || smax > 63) return tr_fail(SW_EINVAL, "sw_traceback: submat entries must lie in [-64, 63]");
  if (gap_open < 0 || gap_extend < 0 || (int64_t)gap_open + 2 * (int64_t)gap_extend > 1024)
    return tr_fail(SW_EINVAL, "sw_traceback: gap penalties out of range (%lld, %lld)", gap_open, gap_extend);
  const int64_t ndb = db_view(db).n;

  // per-hit layout: bands, direction words, operations
  const int band_rows = trace_rows_per_band();
  std::vector<TraceHit> th((size_t)n_hits);
  int64_t dir_words = 0, ops_bytes = 0, nbands = 0;
  for (int64_t h = 0; h < n_hits; ++h) {
    const int32_t qi = hits[h].query, ti = hits[h].target;
    if (qi < 0 || qi >= n_queries) return tr_fail(SW_EINVAL, "sw_traceback: hit %lld: query index %lld out of range", h, qi);
    if (ti < 0 || ti >= ndb) return tr_fail(SW_EINVAL, "sw_traceback: hit %lld: target index %lld out of range", h, ti);
    const int64_t pos = db_sorted_pos(db, ti);
    TraceHit &x = th[h];
    x.qoff = q_offsets[qi];
    x.m = (int32_t)(q_offsets[qi + 1] - q_offsets[qi]);
    x.toff = db_sorted_off(db, pos);
    x.n = db_sorted_len(db, pos);
    x.npad = db_sorted_npad(db, pos);
    x.nb = std::max(1, (x.m + band_rows - 1) / band_rows);
    x.dir0 = dir_words;
    x.ops_off = ops_bytes;
    dir_words += (int64_t)x.nb * (x.npad + 32) * 32;
    ops_bytes += (int64_t)x.m + x.n;
    nbands += x.nb;
  }
  if (nbands >= ((int64_t)1 << 31)) return tr_fail(SW_EINVAL, "sw_traceback: too many bands");
  if (ops_bytes > ops_capacity)
    return tr_fail(SW_EINVAL, "sw_traceback: ops buffer holds %lld bytes, the hits need %lld", ops_capacity,
                   ops_bytes);
  if (ops_bytes > 0 && !ops) return tr_fail(SW_EINVAL, "sw_traceback: null ops");

  // the bands of all hits, the hits that take longest first
  std::vector<int32_t> order((size_t)n_hits), band_hit((size_t)nbands);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
    return (int64_t)th[x].npad + 64 * (int64_t)th[x].nb > (int64_t)th[y].npad + 64 * (int64_t)th[y].nb;
  });
  int32_t next_band = 0;
  for (int32_t h : order) {
    th[h].band0 = next_band;
    for (int32_t b = 0; b < th[h].nb; ++b) band_hit[next_band++] = h;
  }

  const int64_t b_q = tr_round_up(std::max<int64_t>(q_offsets[n_queries], 1), 256);
  const int64_t b_sub = 512, b_hits = tr_round_up((int64_t)sizeof(TraceHit) * n_hits, 256);
  const int64_t b_res = tr_round_up((int64_t)sizeof(TraceResult) * n_hits, 256);
  const int64_t b_ops = tr_round_up(std::max<int64_t>(ops_bytes, 1), 256);
  const int64_t b_bandhit = tr_round_up(4 * nbands, 256), b_best = tr_round_up((int64_t)sizeof(int4) * nbands, 256);
  const int64_t b_words = 256;
  const int64_t bytes = b_q + b_sub + b_hits + b_bandhit + b_best + b_res + b_words + b_ops + 4 * dir_words;
  cudaStream_t s = (cudaStream_t)stream;
  TraceScratch sc;
  sc.s = s;
  cudaError_t e = pool_alloc(&sc.block, (size_t)bytes, s);
  if (e != cudaSuccess) {
    sc.block = nullptr;
    // (short hits take whole bands of 256 rows and 32 columns more: in two calls they need half at a time)
    if (e == cudaErrorMemoryAllocation && n_hits > 1) {
      cudaGetLastError();
      const int64_t first = n_hits / 2, used = th[first].ops_off;
      int rc = sw_traceback(db, queries, q_offsets, n_queries, hits, first, submat, gap_open, gap_extend, out, ops,
                            ops_capacity, stream);
      if (rc != SW_OK) return rc;
      rc = sw_traceback(db, queries, q_offsets, n_queries, hits + first, n_hits - first, submat, gap_open, gap_extend,
                        out + first, ops + used, ops_capacity - used, stream);
      for (int64_t h = first; rc == SW_OK && h < n_hits; ++h) out[h].ops_offset += used;
      return rc;
    }
    return tr_cuda(e, "device allocation");
  }
  uint8_t *p = (uint8_t *)sc.block;
  TraceArgs a{};
  uint8_t *d_q = p;
  int8_t *d_sub = (int8_t *)(d_q + b_q);
  TraceHit *d_hits = (TraceHit *)((uint8_t *)d_sub + b_sub);
  TraceResult *d_res = (TraceResult *)((uint8_t *)d_hits + b_hits);
  int32_t *d_bandhit = (int32_t *)((uint8_t *)d_res + b_res);
  int4 *d_best = (int4 *)((uint8_t *)d_bandhit + b_bandhit);
  int32_t *d_words = (int32_t *)((uint8_t *)d_best + b_best);  // [0] band counter, [1] status
  uint8_t *d_ops = (uint8_t *)d_words + b_words;
  a.qres = d_q;
  a.tres = db_view(db).res;
  a.tres_bytes = db_view(db).res_bytes;
  a.submat = d_sub;
  a.hits = d_hits;
  a.band_hit = d_bandhit;
  a.nhits = (int32_t)n_hits;
  a.nbands = (int32_t)nbands;
  a.band_counter = d_words;
  a.status = d_words + 1;
  a.wait_cycles = kTraceWaitCycles;
  a.dirs = (uint32_t *)(d_ops + b_ops);
  a.dir_words = dir_words;
  a.best = d_best;
  a.ops = d_ops;
  a.results = d_res;
  a.sc.go = gap_open + gap_extend;
  a.sc.ge = gap_extend;
  a.sc.pad = std::min(0, smin);
  a.sc.maxp = std::max(0, smax);
  a.sc.thresh = 32767 - a.sc.maxp;

  if (q_offsets[n_queries] > 0) e = cudaMemcpyAsync(d_q, queries, q_offsets[n_queries], cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_sub, submat, 400, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_hits, th.data(), sizeof(TraceHit) * n_hits, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return tr_cuda(e, "upload");
  if ((e = cudaMemcpyAsync(d_bandhit, band_hit.data(), 4 * (size_t)nbands, cudaMemcpyHostToDevice, s)) != cudaSuccess)
    return tr_cuda(e, "upload");
  int dev = 0, sms = 1;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return tr_cuda(e, "cudaGetDevice");
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if ((e = launch_trace(a, sms, s)) != cudaSuccess) return tr_cuda(e, "traceback kernels");
  std::vector<TraceResult> res((size_t)n_hits);
  int32_t words[2] = {0, 0};
  e = cudaMemcpyAsync(res.data(), d_res, sizeof(TraceResult) * n_hits, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(words, d_words, sizeof words, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && ops_bytes > 0) e = cudaMemcpyAsync(ops, d_ops, ops_bytes, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return tr_cuda(e, "results");
  if (words[1] == SW_ETIMEOUT) return tr_fail(SW_ETIMEOUT, "sw_traceback: a bounded device wait expired");
  if (words[1]) return tr_fail(SW_ECUDA, "sw_traceback: internal error: an index left its buffer (checked build)");
  for (int64_t h = 0; h < n_hits; ++h) {
    sw_alignment &o = out[h];
    o.score = res[h].score;
    o.q_begin = res[h].begin_i;
    o.q_end = res[h].end_i;
    o.t_begin = res[h].begin_j;
    o.t_end = res[h].end_j;
    o.n_ops = res[h].n_ops;
    o.ops_offset = th[h].ops_off;
  }
  return SW_OK;
}
