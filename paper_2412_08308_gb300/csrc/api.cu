// C-ABI entry points (include/swgb.h): database packing, query planning and the
// search pipeline (profile -> DP kernels -> overflow rescue), all on one GPU.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <limits>
#include <memory>
#include <mutex>
#include <tuple>
#include <numeric>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/swgb.h"
#include "host_pool.h"
#include "internal.h"

using namespace swgb;

namespace {

// NVTX range around the host-side enqueue of one stage of a search (profile,
// DP kernels, rescue), for timeline tools; free when no tool is attached.
struct StageRange {
  explicit StageRange(const char *name) { nvtxRangePushA(name); }
  ~StageRange() { nvtxRangePop(); }
};

thread_local std::string g_err;

int fail(int code, const char *fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_err = buf;
  return code;
}

int cuda_fail(cudaError_t e, const char *what) {
  if (e == cudaErrorMemoryAllocation) return fail(SW_ENOMEM, "%s: %s", what, cudaGetErrorString(e));
  return fail(SW_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define SW_CUDA(call, what)                   \
  do {                                        \
    cudaError_t e_ = (call);                  \
    if (e_ != cudaSuccess) return cuda_fail(e_, what); \
  } while (0)

inline int64_t round_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

// Rows per lane of the transposed jobs (heights whose kernels exist), and the
// cycles of one step (two columns) of a band that has its SM sub-partition to
// itself, or per band where two or more share it: from timings of 500 to
// 20,000 proteins at every height.
struct TrackHeight {
  int rows;
  double packed1, packed2, int1, int2;
};
constexpr TrackHeight kTrackHeights[] = {{8, 290, 245, 229, 183},
                                         {12, 351, 356, 290, 264},
                                         {16, 460, 445, 353, 324},
                                         {20, 585, 538, 511, 395},
                                         {24, 685, 680, 560, 509}};
double track_step_cycles(bool packed, int rows, int w) {
  for (const TrackHeight &h : kTrackHeights)
    if (h.rows == rows) return w <= 1 ? (packed ? h.packed1 : h.int1) : w * (packed ? h.packed2 : h.int2);
  return 1e9;
}

// Cycles of one step of an inter-task warp with w warps on its SM
// sub-partition: its share of the sub-partition's rate (row, step), or, with
// few warps, its own latency (row1, step1).  From 1,850 timings of one query
// of 60 to 6,000 residues x 500 to 160,000 proteins at 8, 16 and 24 rows and 4
// to 32 lanes: the lanes and rows that the model picks measure within 5 % of
// the best ones in 9 of 10 cases.
double chain_step_cycles(int form, int R, int w) {
  const bool i32 = form == kFormInt32;
  const double row = i32 ? 8.0 : form == kFormPacked ? 10.2 : 8.5, step = i32 ? 26 : 22;
  const double row1 = i32 ? 14.0 : 12.5, step1 = i32 ? 171 : 110;
  return std::max(step1 + row1 * R, w * (row * R + step));
}

int sm_count(int dev) {
  int n = 0;
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

// Launch occupancies depend only on the device, the kernel and its launch
// shape, so each is asked of the runtime once per process (the query, and the
// shared-memory attribute it sets, cost tens of microseconds per plan).
// kind: 0 inter-task (a = R, b = form), 1 band-stream (a = R), 2 transposed
// (a = R); gaps: GapSet.  Failures (0) are not kept.
int cached_occupancy(int kind, int a, int b, int gaps, int threads, size_t smem) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int, int, int, int, size_t>, int> memo;
  int dev = 0;
  cudaGetDevice(&dev);
  const auto key = std::make_tuple(dev, kind, a, b, gaps, threads, smem);
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = memo.find(key);
    if (it != memo.end()) return it->second;
  }
  const int n = kind == 0 ? inter_max_ctas_per_sm(a, b, gaps, threads, smem)
                : kind == 1 ? band_max_ctas_per_sm(a, gaps)
                            : track_max_ctas_per_sm(a, gaps);
  if (n > 0) {
    std::lock_guard<std::mutex> lock(mu);
    memo[key] = n;
  }
  return n;
}

// The stream-ordered pool that every query batch's device block comes from,
// one per device, created on first use: freed blocks stay reserved up to
// 1 GiB, so that planning a batch after another does not map fresh memory
// (the default pool returns it at every synchronisation: ~0.1-0.2 ms per
// plan).  Its own pool, so that the process's default pool keeps its settings.
cudaError_t batch_pool(cudaMemPool_t *pool) {
  static std::mutex mu;
  static std::map<int, cudaMemPool_t> pools;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  auto it = pools.find(dev);
  if (it != pools.end()) {
    *pool = it->second;
    return cudaSuccess;
  }
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t p = nullptr;
  e = cudaMemPoolCreate(&p, &props);
  if (e != cudaSuccess) return e;
  uint64_t keep = (uint64_t)1 << 30;
  e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
  if (e != cudaSuccess) {
    cudaMemPoolDestroy(p);
    return e;
  }
  pools[dev] = p;
  *pool = p;
  return cudaSuccess;
}

int check_seqs(const uint8_t *res, const int64_t *off, int64_t n, const char *what) {
  if (n < 0) return fail(SW_EINVAL, "%s: negative sequence count", what);
  if (!off) return fail(SW_EINVAL, "%s: null offsets", what);
  if (off[0] != 0) return fail(SW_EINVAL, "%s: offsets[0] must be 0", what);
  for (int64_t i = 0; i < n; ++i)
    if (off[i + 1] < off[i]) return fail(SW_EINVAL, "%s: offsets decrease at %lld", what, (long long)i);
  const int64_t total = off[n];
  if (total > 0 && !res) return fail(SW_EINVAL, "%s: null residues", what);
  for (int64_t i = 0; i < total; ++i)
    if (res[i] >= kAlphabet) return fail(SW_EINVAL, "%s: residue code %d >= 20 at %lld", what, (int)res[i], (long long)i);
  return SW_OK;
}

bool is_device_ptr(const void *p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// --- the database in row tracks (transposed jobs, k_band.cu) ----------------
// Sequences (sorted order, longest first) go to the 16-bit tracks (f = 0; two
// tracks share each word) when their length is at most `cut`, else to int32
// tracks (f = 1).  A sequence that fits a band (32 lanes of tR rows) takes
// whole lanes of the fullest band that has room, so these bands depend on no
// other band.  A longer one gets a track of its own, in lanes of
// track_long_rows(tR) rows, whose bands run as a pipeline: its last band
// starts about 50 steps per band above it late, and the shorter lanes' steps
// make up for that (one 144-residue query x 2,000 proteins: the few proteins
// past 768 rows cost 15 of 58 us in 24-row lanes).  Lanes that it leaves free
// in its last band take short sequences too.  Empty sequences score 0 without
// a lane.
struct TrackSeg {
  int32_t pos, bin, lane0, lanes;  // sequence, track, first lane in the track, lanes
};
struct TrackBins {
  std::vector<TrackSeg> seg[2];
  std::vector<int32_t> used[2];  // lanes of each track
  std::vector<char> tall[2];     // 1: tR rows per lane (one band), 0: track_long_rows(tR)
};
// a pipeline of bands: one int32 track, or two 16-bit tracks sharing words
struct TrackPipe {
  int32_t packed, nb, lane0, rows;  // rows per lane
};

// What the transposed jobs of one query cost a launch: bands over all
// pipelines and the most bands of one, of the 16-bit [0] and int32 [1] tracks.
struct TrackLoad {
  double bands[2] = {0, 0};
  int64_t deepest[2] = {1, 1};
};

void bin_tracks(const std::vector<int32_t> &len, int tR, int32_t cut, TrackBins &b) {
  const int tL = track_long_rows(tR);
  // tracks by the lanes free in their last band, per height
  std::vector<int32_t> room[2][2][33];
  for (int f = 0; f < 2; ++f) {
    b.seg[f].clear();
    b.used[f].clear();
    b.tall[f].clear();
  }
  for (size_t k = 0; k < len.size(); ++k) {
    if (len[k] == 0) continue;
    const int f = len[k] <= cut ? 0 : 1;
    const int32_t lanes_t = (len[k] + tR - 1) / tR, lanes_l = (len[k] + tL - 1) / tL;
    int32_t bin = -1, tall = lanes_t <= 32 ? 1 : 0, lanes = tall ? lanes_t : lanes_l;
    if (tall) {  // the track with room whose free rows it leaves fewest of
      int32_t best = 32 * tR + 1;
      for (int h = 0; h < 2; ++h)
        for (int32_t r = h ? lanes_t : lanes_l; r <= 32; ++r)
          if (!room[f][h][r].empty()) {
            const int32_t left = (r - (h ? lanes_t : lanes_l)) * (h ? tR : tL);
            if (left < best) {
              best = left;
              tall = h;
              lanes = h ? lanes_t : lanes_l;
              bin = room[f][h][r].back();
            }
            break;
          }
    }
    if (bin < 0) {
      bin = (int32_t)b.used[f].size();
      b.used[f].push_back(0);
      b.tall[f].push_back((char)tall);
    } else {
      room[f][tall][32 - (b.used[f][bin] + 31) % 32 - 1].pop_back();
    }
    b.seg[f].push_back({(int32_t)k, bin, b.used[f][bin], lanes});
    b.used[f][bin] += lanes;
    room[f][tall][32 - (b.used[f][bin] + 31) % 32 - 1].push_back(bin);
  }
}

// The pipelines (deeper first; 16-bit ones pair consecutive tracks of the same
// height in that order) and their lane table: band b, lane l of a pipeline
// covers the rows of lane 32 b + l of its track(s); each segment writes its
// own lanes, the others stay idle.
void lay_tracks(const TrackBins &b, int tR, std::vector<TrackPipe> &pipes, std::vector<TrackLane> &lanes) {
  pipes.clear();
  lanes.clear();
  const int rows_of[2] = {track_long_rows(tR), tR};
  for (int f = 0; f < 2; ++f) {
    const std::vector<int32_t> &U = b.used[f];
    const int32_t B = (int32_t)U.size();
    auto bands = [&](int32_t t) { return (U[t] + 31) / 32; };
    std::vector<int32_t> order(B), base(B), high(B);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
      return b.tall[f][x] != b.tall[f][y] ? b.tall[f][x] < b.tall[f][y] : bands(x) > bands(y);
    });
    for (int32_t i = 0; i < B; ++i) {
      const int32_t ta = order[i];
      const bool pair = f == 0 && i + 1 < B && b.tall[f][order[i + 1]] == b.tall[f][ta];
      TrackPipe pp{f == 0 ? 1 : 0, bands(ta), (int32_t)lanes.size(), rows_of[(int)b.tall[f][ta]]};
      base[ta] = pp.lane0;
      high[ta] = 0;
      if (pair) {  // (bands(order[i + 1]) <= bands(ta): sorted)
        ++i;
        base[order[i]] = pp.lane0;
        high[order[i]] = 1;
      }
      lanes.resize(lanes.size() + 32 * (size_t)pp.nb, TrackLane{-1, 0, -1, 0});
      pipes.push_back(pp);
    }
    for (const TrackSeg &g : b.seg[f]) {
      const int32_t rows = rows_of[(int)b.tall[f][g.bin]];
      TrackLane *L = lanes.data() + base[g.bin] + g.lane0;
      for (int32_t k = 0; k < g.lanes; ++k) {
        if (high[g.bin]) {
          L[k].pb = g.pos;
          L[k].rb = k * rows;
        } else {
          L[k].pa = g.pos;
          L[k].ra = k * rows;
        }
      }
    }
  }
  std::stable_sort(pipes.begin(), pipes.end(), [](const TrackPipe &x, const TrackPipe &y) { return x.nb > y.nb; });
}

// Row-track layouts a database keeps (built on first use, its lane table on
// the device): at most this many, each with at most this many bytes of lanes;
// other layouts are built for every plan.
constexpr size_t kTrackLayouts = 8;
constexpr int64_t kTrackLayoutBytes = (int64_t)64 << 20;

}  // namespace

struct sw_db {
  int device = 0;
  int64_t n = 0, total = 0;
  DbView view{};
  void *block = nullptr;
  size_t bytes = 0;
  int32_t max_npad = 0;
  double mean_npad = 0;
  std::vector<int32_t> h_npad;  // padded lengths in sorted order
  std::vector<int32_t> h_len;   // true lengths in sorted order
  std::vector<int32_t> h_pos;   // sorted position of each sequence, caller order
  std::vector<int64_t> h_off;   // residue offsets in sorted order
  // device [0, 1, ..., n - 1, n - 1]: the sorted positions of the database
  // units (one sequence, or two consecutive ones in packed mode, the last
  // repeated when n is odd), shared by every query batch
  const int32_t *d_ident = nullptr;
  // per mode (0 int32: one sequence per unit; 1 packed: two), built on first
  // use: the count of units of each padded length / 16 and the prefix sums
  // of the units' lengths, so that planning a batch does not walk every unit
  struct UnitStats {
    std::vector<int64_t> hist, prefix;
  };
  mutable std::mutex stats_mu;
  mutable std::unique_ptr<UnitStats> unit_stats[2];
  const UnitStats &units(bool packed) const {
    std::lock_guard<std::mutex> lock(stats_mu);
    std::unique_ptr<UnitStats> &u = unit_stats[packed ? 1 : 0];
    if (!u) {
      u.reset(new UnitStats());
      const int64_t nu = packed ? (n + 1) / 2 : n;
      u->hist.assign((size_t)max_npad / 16 + 1, 0);
      u->prefix.assign((size_t)nu + 1, 0);
      for (int64_t k = 0; k < nu; ++k) {
        const int32_t len = h_npad[(size_t)std::min<int64_t>(packed ? 2 * k : k, n - 1)];
        ++u->hist[(size_t)len / 16];
        u->prefix[(size_t)k + 1] = u->prefix[(size_t)k] + len;
      }
    }
    return *u;
  }
  // transposed jobs: the database's row tracks for one lane height and one
  // 16-bit / int32 routing (cut), with the lane table on the device, shared
  // by every query batch that plans them
  struct TrackLayout {
    int32_t tR = 0, cut = 0;
    TrackLoad load;
    int64_t n_lanes = 0;
    std::vector<TrackPipe> pipes;
    TrackLane *d_lanes = nullptr;
  };
  mutable std::mutex track_mu;
  mutable std::vector<std::unique_ptr<TrackLayout>> track_layouts;
  // whether its row tracks can be kept in lanes of 16 rows or more (a large
  // database's bands fill the GPU at those)
  bool keeps_tracks() const { return (total / 16 + n) * (int64_t)sizeof(TrackLane) <= kTrackLayoutBytes; }
  // the layout for (tR, cut), built and uploaded on stream s on first use
  // (synchronising s), or nullptr: not kept (too large, too many, called on
  // another device, or a CUDA error) -- the caller then builds it itself
  const TrackLayout *track_layout(int tR, int32_t cut, cudaStream_t s) const {
    std::lock_guard<std::mutex> lock(track_mu);
    for (const std::unique_ptr<TrackLayout> &t : track_layouts)
      if (t->tR == tR && t->cut == cut) return t.get();
    int dev = -1;
    if (track_layouts.size() >= kTrackLayouts || cudaGetDevice(&dev) != cudaSuccess || dev != device) {
      cudaGetLastError();
      return nullptr;
    }
    // at most one lane per track_long_rows(tR) residues and one more per sequence
    if ((total / track_long_rows(tR) + n) * (int64_t)sizeof(TrackLane) > kTrackLayoutBytes) return nullptr;
    TrackBins b;
    bin_tracks(h_len, tR, cut, b);
    std::unique_ptr<TrackLayout> t(new TrackLayout());
    t->tR = tR;
    t->cut = cut;
    std::vector<TrackLane> lanes;
    lay_tracks(b, tR, t->pipes, lanes);
    if ((int64_t)(lanes.size() * sizeof(TrackLane)) > kTrackLayoutBytes) return nullptr;
    for (const TrackPipe &p : t->pipes) {
      const int f = p.packed ? 0 : 1;
      t->load.bands[f] += p.nb;
      t->load.deepest[f] = std::max<int64_t>(t->load.deepest[f], p.nb);
    }
    t->n_lanes = (int64_t)lanes.size();
    if (!lanes.empty()) {
      void *d = nullptr;
      cudaError_t e = cudaMalloc(&d, sizeof(TrackLane) * lanes.size());
      if (e == cudaSuccess) e = cudaMemcpyAsync(d, lanes.data(), sizeof(TrackLane) * lanes.size(), cudaMemcpyHostToDevice, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) {
        if (d) cudaFree(d);
        cudaGetLastError();
        return nullptr;
      }
      t->d_lanes = (TrackLane *)d;
    }
    track_layouts.push_back(std::move(t));
    return track_layouts.back().get();
  }
};

struct sw_queries {
  const sw_db *db = nullptr;
  int64_t nq = 0;
  int mode = SW_MODE_PACKED;
  int R = 16, Ri = 16;
  Scoring sc{};
  std::vector<QDesc> qd, qdi;  // inter-task and intra-task plans per query
  std::vector<QDesc> qdp;      // query-track plans (packed mode, inter-task kernel)
  std::vector<TrackChunk> track;  // their chunk descriptors
  int64_t n_units = 0, n_long = 0, n_upos = 0, n_ipos32 = 0;
  int64_t n_tasks = 0, n_itasks = 0, n_itasks32 = 0, n_rtask_cap = 0;
  int64_t npairs = 0, n_ptasks = 0, n_solo = 0, n_single = 0;
  bool inter_may_flag = false;  // some packed inter-task pair can exceed the 16-bit threshold
  int grid = 1, rgrid = 1, igrid = 1, pgrid = 1, threads = 256;
  int pbuf_bytes = 0, ipbuf_bytes = 0, ppbuf_bytes = 0;
  int pbuf_count = 2, ppbuf_count = 2;  // profile buffers of the two inter-task launches
  size_t smem = 0, ismem = 0, psmem = 0;
  int32_t gbuf_stride = 0, igbuf_stride = 0;
  int64_t long_stride = 1;
  // device memory (one stream-ordered allocation)
  void *block = nullptr;
  size_t bytes = 0;
  cudaStream_t alloc_stream = nullptr;
  cudaStream_t side = nullptr;  // second stream for the intra-task kernel
  cudaEvent_t fork = nullptr, join = nullptr;
  // third stream: the int32 intra-task launch beside the packed one
  cudaStream_t side2 = nullptr;
  cudaEvent_t join2 = nullptr;
  uint8_t *d_qres = nullptr;
  int8_t *d_submat = nullptr;
  QDesc *d_qd = nullptr, *d_qdi = nullptr, *d_qdp = nullptr;
  TrackChunk *d_track = nullptr;
  Task *d_tasks = nullptr, *d_itasks = nullptr, *d_itasks32 = nullptr, *d_rtasks = nullptr, *d_ptasks = nullptr;
  int32_t *d_ipos32 = nullptr, *d_upos = nullptr;
  uint8_t *d_prof = nullptr;
  int64_t prof_bytes = 0;
  uint2 *d_gbuf = nullptr, *d_igbuf = nullptr;
  int32_t *d_words = nullptr;
  // sw_search to host memory: the scores, directly after the words' b_words bytes and before the row tracks' rings
  int32_t *d_scores = nullptr;
  size_t b_words = 0, b_scores = 0;
  int32_t *d_flag_pos = nullptr, *d_iflag_pos = nullptr;
  // band-stream jobs (small batches): long queries against every unit, the
  // other queries against the long units
  int64_t n_bjobs = 0, n_bands = 0, n_btargets = 0, band_ring_bytes = 0;
  int bgrid = 1, bR = 8;
  bool bone = false;  // band-stream launch limited to one CTA per SM
  // transposed jobs (small batches): database row tracks against each short query
  int64_t n_tjobs = 0, n_tbands = 0, n_tlanes = 0, track_ring_bytes = 0, qt_bytes = 16;
  int tgrid = 1, tR = 16;
  int n_tgroups = 0;
  TrackJob *d_tjobs = nullptr;
  TrackGroup *d_tgroups = nullptr;
  TrackLane *d_tlanes = nullptr;
  bool tlanes_shared = false;  // d_tlanes is the database's kept lane table, not in the block
  uint8_t *d_qt = nullptr;
  int64_t *d_qt_off = nullptr;
  int32_t *d_qt_npad = nullptr;
  unsigned long long *d_trings = nullptr;
  BandJob *d_bjobs = nullptr;
  int32_t *d_bjob_of = nullptr;
  int2 *d_btpos = nullptr;
  unsigned long long *d_brings = nullptr;
  int64_t h2d_bytes = 0;
  bool timing = false, timed = false;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  cudaGraphExec_t gexec = nullptr;  // captured search (sw_search_graph)
  const sw_db *gdb = nullptr;
  int32_t *gscores = nullptr;
  // word layout: [0] inter counter, [1] inter rescue counter, [2] status, [3] inter rescue tasks,
  // [4] intra (packed) counter, [5] intra (int32) counter, [6] query-pair counter, [7] band counter,
  // (the transposed jobs' counter is word [1], the inter rescue counter, unused in small batches)
  // [8, 8+nq) inter flag counts, [8+nq, 8+2nq) intra flag counts   -- zeroed every search
  // [8+2nq] inter tasks, [9+2nq] intra packed tasks, [10+2nq] intra int32 tasks,
  // [11+2nq] query-pair tasks -- constants
  int64_t zero_words() const { return 8 + 2 * nq; }
};

namespace {

// Lanes per chain for one query at R rows per lane: minimise padded rows x
// steps per column (fill[L], below) x idle lanes, with a small charge per
// chunk for the boundary strip and the CTA barrier.  (Against the measured
// time of the 20-query benchmark with L forced to 4..32, this model is
// proportional to within 1.5 %.)  At least Lmin lanes.
double lanes_cost(int m, int R, const double *fill, int L) {
  const int LR = L * R;
  const int C = std::max(1, (m + LR - 1) / LR);
  const double rows = (double)C * LR;
  const int G = 32 / L;
  const double lane_eff = (double)(G * L) / 32.0;
  return rows * fill[L] / lane_eff * (1.0 + 0.001 * C);
}

// The lanes with the least cost(L), at least Lmin of them.  Where the costs are
// kept from one floor to the next (null: not), each is formed once.
struct LaneCosts {
  double c[33];
  bool have = false;
};
template <class Cost>
int choose_lanes(int Lmin, LaneCosts *kept, const Cost &cost) {
  if (kept && !kept->have) {
    for (int L = 4; L <= 32; ++L) kept->c[L] = cost(L);
    kept->have = true;
  }
  int bestL = Lmin;
  double best = 1e300;
  for (int L = Lmin; L <= 32; ++L) {
    const double c = kept ? kept->c[L] : cost(L);
    if (c < best - 1e-9) {
      best = c;
      bestL = L;
    }
  }
  return bestL;
}

void free_queries(sw_queries *q) {
  if (!q) return;
  if (q->block) {
    cudaFreeAsync(q->block, q->alloc_stream);
    cudaStreamSynchronize(q->alloc_stream);
  }
  if (q->ev0) cudaEventDestroy(q->ev0);
  if (q->ev1) cudaEventDestroy(q->ev1);
  if (q->gexec) cudaGraphExecDestroy(q->gexec);
  if (q->fork) cudaEventDestroy(q->fork);
  if (q->join) cudaEventDestroy(q->join);
  if (q->side) cudaStreamDestroy(q->side);
  if (q->join2) cudaEventDestroy(q->join2);
  if (q->side2) cudaStreamDestroy(q->side2);
  delete q;
}

}  // namespace

namespace swgb {
const DbView &db_view(const sw_db *db) { return db->view; }
int db_device(const sw_db *db) { return db->device; }
const int32_t *db_ident(const sw_db *db) { return db->d_ident; }
int64_t db_sorted_pos(const sw_db *db, int64_t caller_index) { return db->h_pos[caller_index]; }
int32_t db_sorted_len(const sw_db *db, int64_t pos) { return db->h_len[pos]; }
int32_t db_sorted_npad(const sw_db *db, int64_t pos) { return db->h_npad[pos]; }
int64_t db_sorted_off(const sw_db *db, int64_t pos) { return db->h_off[pos]; }
cudaError_t pool_alloc(void **ptr, size_t bytes, cudaStream_t s) {
  cudaMemPool_t pool = nullptr;
  cudaError_t e = batch_pool(&pool);
  return e == cudaSuccess ? cudaMallocFromPoolAsync(ptr, bytes, pool, s) : e;
}
int set_last_error(int code, const char *msg) { return fail(code, "%s", msg); }
void clear_last_error() { g_err.clear(); }
}  // namespace swgb

extern "C" {

const char *sw_last_error(void) { return g_err.c_str(); }

int sw_db_prepare(const uint8_t *residues, const int64_t *offsets, int64_t n_seqs, void *stream, sw_db **out) {
  g_err.clear();
  if (!out) return fail(SW_EINVAL, "sw_db_prepare: null output handle");
  *out = nullptr;
  if (int rc = check_seqs(residues, offsets, n_seqs, "sw_db_prepare")) return rc;
  if (n_seqs >= (int64_t)1 << 30) return fail(SW_EINVAL, "sw_db_prepare: too many sequences");
  cudaStream_t s = (cudaStream_t)stream;
  sw_db *db = new sw_db();
  SW_CUDA(cudaGetDevice(&db->device), "cudaGetDevice");
  db->n = n_seqs;
  db->total = n_seqs ? offsets[n_seqs] : 0;

  std::vector<int32_t> order(n_seqs), len(n_seqs), npad(n_seqs);
  std::vector<int64_t> off(n_seqs);
  for (int64_t i = 0; i < n_seqs; ++i) {
    const int64_t L = offsets[i + 1] - offsets[i];
    if (L > (int64_t)1 << 28) {
      delete db;
      return fail(SW_EINVAL, "sw_db_prepare: sequence %lld too long", (long long)i);
    }
    len[i] = (int32_t)L;
  }
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return len[a] > len[b]; });
  int64_t padded = 0;
  std::vector<int32_t> slen(n_seqs);
  for (int64_t k = 0; k < n_seqs; ++k) {
    slen[k] = len[order[k]];
    npad[k] = (int32_t)std::max<int64_t>(kColBlock, round_up(slen[k], kColBlock));
    off[k] = padded;
    padded += npad[k];
    db->max_npad = std::max(db->max_npad, npad[k]);
  }
  db->mean_npad = n_seqs ? (double)padded / n_seqs : 0;
  db->h_npad = npad;
  db->h_len = slen;
  db->h_off = off;
  db->h_pos.assign(n_seqs, 0);
  for (int64_t k = 0; k < n_seqs; ++k) db->h_pos[order[k]] = (int32_t)k;
  std::vector<uint8_t> packed((size_t)std::max<int64_t>(padded, 16), (uint8_t)kPadCode);
  for (int64_t k = 0; k < n_seqs; ++k)
    if (slen[k]) memcpy(&packed[off[k]], residues + offsets[order[k]], (size_t)slen[k]);

  const size_t b_res = round_up((int64_t)packed.size(), 256);
  const size_t b_off = round_up(8 * std::max<int64_t>(n_seqs, 1), 256);
  const size_t b_i32 = round_up(4 * std::max<int64_t>(n_seqs, 1), 256);
  const size_t b_ident = round_up(4 * (n_seqs + 1), 256);
  db->bytes = b_res + b_off + 3 * b_i32 + b_ident;
  cudaError_t e = cudaMalloc(&db->block, db->bytes);
  if (e != cudaSuccess) {
    delete db;
    return cuda_fail(e, "sw_db_prepare: device allocation");
  }
  uint8_t *p = (uint8_t *)db->block;
  db->view.res = p;
  db->view.off = (const int64_t *)(p + b_res);
  db->view.npad = (const int32_t *)(p + b_res + b_off);
  db->view.len = (const int32_t *)(p + b_res + b_off + b_i32);
  db->view.perm = (const int32_t *)(p + b_res + b_off + 2 * b_i32);
  db->view.n = n_seqs;
  db->view.res_bytes = (int64_t)packed.size();
  db->d_ident = (const int32_t *)(p + b_res + b_off + 3 * b_i32);
  std::vector<int32_t> ident((size_t)n_seqs + 1);
  for (int64_t k = 0; k <= n_seqs; ++k) ident[k] = (int32_t)std::max<int64_t>(0, std::min<int64_t>(k, n_seqs - 1));
  e = cudaMemcpyAsync((void *)db->view.res, packed.data(), packed.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && n_seqs) {
    e = cudaMemcpyAsync((void *)db->view.off, off.data(), 8 * n_seqs, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync((void *)db->view.npad, npad.data(), 4 * n_seqs, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync((void *)db->view.len, slen.data(), 4 * n_seqs, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync((void *)db->view.perm, order.data(), 4 * n_seqs, cudaMemcpyHostToDevice, s);
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync((void *)db->d_ident, ident.data(), 4 * ident.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cudaFree(db->block);
    delete db;
    return cuda_fail(e, "sw_db_prepare: upload");
  }
  *out = db;
  return SW_OK;
}

int sw_db_free(sw_db *db) {
  g_err.clear();
  if (!db) return SW_OK;
  if (db->block) cudaFree(db->block);
  for (const std::unique_ptr<sw_db::TrackLayout> &t : db->track_layouts)
    if (t->d_lanes) cudaFree(t->d_lanes);
  delete db;
  return SW_OK;
}

int sw_db_stats(const sw_db *db, int64_t *n_seqs, int64_t *residues, int64_t *device_bytes) {
  g_err.clear();
  if (!db) return fail(SW_EINVAL, "sw_db_stats: null handle");
  if (n_seqs) *n_seqs = db->n;
  if (residues) *residues = db->total;
  if (device_bytes) {
    int64_t b = (int64_t)db->bytes;
    std::lock_guard<std::mutex> lock(db->track_mu);
    for (const std::unique_ptr<sw_db::TrackLayout> &t : db->track_layouts)
      b += t->n_lanes * (int64_t)sizeof(TrackLane);
    *device_bytes = b;
  }
  return SW_OK;
}

namespace {

// a DP task and its modelled cost (tasks are sorted longest first)
struct TW {
  Task t;
  double w;
};

// The planner's large host tables, one set per thread, emptied at the start
// of each plan but keeping their memory.
struct PlanScratch {
  std::vector<BandJob> bjobs;
  std::vector<int32_t> bjob_of;
  std::vector<int2> btpos;
  std::vector<TrackJob> tjobs;
  std::vector<TrackGroup> tgroups;
  std::vector<TrackLane> tlanes;
  std::vector<TrackPipe> tpipes;
  TrackBins bins;
  std::vector<uint8_t> stage;  // the plan's upload, laid out like its device block
  std::vector<TW> tw;
  std::vector<Task> tasks;
  std::vector<uint8_t> back;  // a search's words and scores on their way to the caller
};
constexpr int64_t kSearchStage = 64 << 10;

PlanScratch &plan_scratch() {
  static thread_local PlanScratch ps;
  ps.bjobs.clear();
  ps.bjob_of.clear();
  ps.btpos.clear();
  ps.tjobs.clear();
  ps.tgroups.clear();
  ps.tlanes.clear();
  ps.tpipes.clear();
  ps.tw.clear();
  ps.tasks.clear();
  return ps;
}

}  // namespace

// The plan of a batch, its device block and its upload.  one_search: for a
// single search that reads its results back and frees the batch (sw_search):
// the upload is not waited for (the caller's thread synchronises the stream
// before it returns or plans again), and score_bytes of the block, if not 0,
// hold its scores.
static int prepare_queries(const sw_db *db, const uint8_t *queries, const int64_t *q_offsets, int64_t n_queries,
                           const int8_t *submat, int32_t gap_open, int32_t gap_extend, int32_t mode,
                           const sw_options *opts, void *stream, bool one_search, int64_t score_bytes,
                           sw_queries **out) {
  g_err.clear();
  if (!out) return fail(SW_EINVAL, "sw_queries_prepare: null output handle");
  *out = nullptr;
  if (!db) return fail(SW_EINVAL, "sw_queries_prepare: null database");
  if (!submat) return fail(SW_EINVAL, "sw_queries_prepare: null submat");
  if (mode != SW_MODE_INT32 && mode != SW_MODE_PACKED) return fail(SW_EINVAL, "sw_queries_prepare: bad mode %d", mode);
  if (gap_open < 0 || gap_extend < 0 || (int64_t)gap_open + 2 * (int64_t)gap_extend > 1024)
    return fail(SW_EINVAL, "sw_queries_prepare: gap penalties out of range (%d, %d)", gap_open, gap_extend);
  sw_options o{};
  if (opts) o = *opts;
  if (o.reserved[0]) return fail(SW_EINVAL, "sw_queries_prepare: reserved option fields must be 0");
  const int bR = o.band_rows ? o.band_rows : 16;
  if (!band_supported_R(bR)) return fail(SW_EINVAL, "sw_queries_prepare: band_rows must be 8 or 16");
  if (o.band_stream < 0 || o.band_stream > 2) return fail(SW_EINVAL, "sw_queries_prepare: band_stream must be 0, 1 or 2");
  if (o.query_pairs != 0 && o.query_pairs != 1) return fail(SW_EINVAL, "sw_queries_prepare: query_pairs must be 0 or 1");
  int R = o.rows_per_lane ? o.rows_per_lane : 24;
  const int Ri = o.intra_rows ? o.intra_rows : 16;
  const int forceL = o.lanes_per_chain;
  const int cutover = o.cutover > 0 ? o.cutover : 2048;
  if (!inter_supported_R(R)) return fail(SW_EINVAL, "sw_queries_prepare: rows_per_lane must be 4, 8, 12, 16 or 24");
  if (Ri != 8 && Ri != 16) return fail(SW_EINVAL, "sw_queries_prepare: intra_rows must be 8 or 16");
  if (forceL && (forceL < 4 || forceL > 32)) return fail(SW_EINVAL, "sw_queries_prepare: lanes_per_chain must be 4..32");
  if (o.cutover < 0) return fail(SW_EINVAL, "sw_queries_prepare: negative cutover");
  if (int rc = check_seqs(queries, q_offsets, n_queries, "sw_queries_prepare")) return rc;
  int smin = 127, smax = -128;
  for (int i = 0; i < kAlphabet * kAlphabet; ++i) {
    smin = std::min<int>(smin, submat[i]);
    smax = std::max<int>(smax, submat[i]);
  }
  if (smin < -64 || smax > 63) return fail(SW_EINVAL, "sw_queries_prepare: submat entries must lie in [-64, 63]");
  if (n_queries * std::max<int64_t>(db->n, 1) >= ((int64_t)1 << 31))
    return fail(SW_EINVAL, "sw_queries_prepare: n_queries * n_db must be < 2^31");
  for (int64_t i = 0; i < n_queries; ++i)
    if (q_offsets[i + 1] - q_offsets[i] > (1 << 24)) return fail(SW_EINVAL, "sw_queries_prepare: query too long");

  cudaStream_t s = (cudaStream_t)stream;
  sw_queries *Q = new sw_queries();
  Q->db = db;
  Q->nq = n_queries;
  Q->mode = mode;
  Q->alloc_stream = s;
  Q->Ri = Ri;
  const bool packed = mode == SW_MODE_PACKED;
  Scoring &sc = Q->sc;
  sc.go = gap_open + gap_extend;
  sc.ge = gap_extend;
  sc.pad = std::min(0, smin);
  sc.maxp = std::max(0, smax);
  sc.thresh = 32767 - sc.maxp;
  const int gaps = gap_set(sc);

  const int sms = sm_count(db->device);
  const int64_t n = db->n;
  const std::vector<int32_t> &npad = db->h_npad;

  // --- units (sorted positions); a unit is long when its first (longest) sequence reaches the cutover
  // (unit u: sorted positions 2u and min(2u + 1, n - 1) in packed mode, u in
  // int32 mode; the database's identity array holds them on the device)
  Q->n_units = packed ? (n + 1) / 2 : n;
  auto unit_seq = [&](int64_t i) { return (int32_t)std::min<int64_t>(i, n - 1); };
  auto unit_len = [&](int64_t u) { return npad[unit_seq(packed ? 2 * u : u)]; };
  // (units are sorted by length, longest first: the long ones are a prefix)
  int64_t n_long = 0, hi = Q->n_units;
  while (n_long < hi) {
    const int64_t mid = (n_long + hi) / 2;
    if (unit_len(mid) >= cutover) n_long = mid + 1;
    else hi = mid;
  }
  Q->n_long = n_long;
  static const sw_db::UnitStats kNoUnits{{0}, {0}};
  const sw_db::UnitStats &ust = n > 0 ? db->units(packed) : kNoUnits;
  int32_t max_short = 16, max_long = 16;
  const double sum_short = n > 0 ? (double)(ust.prefix[(size_t)Q->n_units] - ust.prefix[(size_t)n_long]) : 0.0;
  if (n_long < Q->n_units) max_short = unit_len(n_long);
  if (n_long) max_long = unit_len(0);
  // fill[L]: steps a chain of L lanes spends per real column of a short unit.
  // A pass over a unit of n padded columns takes n + lag steps (lag = L - 1,
  // or 2 L - 1 for the split lanes of the 16-bit forms) rounded up to whole
  // 16-column blocks.
  // (padded lengths are multiples of 16 and every long unit is longer than
  // every short one, so the short units' counts are the first bins)
  std::vector<int64_t> len_hist(max_short / kColBlock + 1, 0);
  if (n_long < Q->n_units)
    std::copy(ust.hist.begin(), ust.hist.begin() + std::min(len_hist.size(), ust.hist.size()), len_hist.begin());
  // (the lag does not depend on the rows beyond whether they split)
  double fills[2][33];
  bool have_fill[2] = {false, false};
  auto fill_of = [&](int form, int rows) -> const double * {
    const int k = inter_chain_lag(rows, form, 4) > 3;
    double *out = fills[k];
    if (!have_fill[k])
      for (int L = 0; L <= 32; ++L) {
        const int lag = L > 0 ? inter_chain_lag(rows, form, L) : 0;
        double steps = 0;
        for (size_t b = 1; b < len_hist.size(); ++b)
          steps += (double)len_hist[b] * (double)((b * kColBlock + lag + kColBlock - 1) / kColBlock * kColBlock);
        out[L] = sum_short > 0 ? steps / sum_short : 1.0;
      }
    have_fill[k] = true;
    return out;
  };
  const int64_t n_short = Q->n_units - n_long;
  auto qlen = [&](int64_t q) { return (int32_t)(q_offsets[q + 1] - q_offsets[q]); };
  auto may_flag = [&](int64_t q, int32_t n_upper) {
    return packed && (int64_t)sc.maxp * std::min<int64_t>(qlen(q), n_upper) > sc.thresh;
  };

  // --- the inter-task kernel's plan: rows per lane, lanes per chain, CTA size,
  // and (packed mode) query tracks.
  // Query tracks: two queries share one chain, one per
  // 16-bit half: the database residue of a column is common to both, so one
  // 32-bit profile word per row feeds both halves and the residue-pair byte
  // shuffle of the two-sequence form disappears.  Each half runs a track of
  // queries laid end to end chunk by chunk, so queries of different lengths
  // share chains without idle rows (greedy longest-first packing into
  // balanced tracks).  Only queries that cannot pass the 16-bit threshold
  // against the short database units join tracks (the form has no rescue
  // pass); the others keep the two-sequence form.
  const int64_t s0 = packed ? std::min<int64_t>(n, 2 * n_long) : n_long;  // first short sequence
  Q->n_single = n - s0;
  std::vector<int32_t> elig;
  if (packed && o.query_pairs == 0 && n_queries >= 2 && Q->n_single > 0) {
    for (int64_t q = 0; q < n_queries; ++q)
      if (!may_flag(q, max_short)) elig.push_back((int32_t)q);
    if (elig.size() < 2) elig.clear();
    std::stable_sort(elig.begin(), elig.end(), [&](int32_t x, int32_t y) { return qlen(x) > qlen(y); });
  }
  struct InterPlan {
    int R = 24, warps = 8;
    std::vector<int> L;                        // lanes per chain of each query's own plan
    std::vector<char> in_track;                // query runs in a track plan
    std::vector<std::vector<int32_t>> tracks;  // two per track plan
    std::vector<int> plan_L;
    double time = 0;       // modelled cycles
    bool even = false;     // many tasks per CTA: no task sets the time
    int floor_to = 32;     // up to this floor of lanes the plan stays the same
  };
  struct Part {
    int C, L;  // chunks and lanes per chain of a query's (a track plan's) chains
  };
  // Modelled cycles of one launch of `parts` over nu units, longest first:
  // the average work of a CTA, and what list scheduling cannot split -- the
  // longest task, and j + 1 tasks on some CTA as long as there are more than j
  // per CTA.  *even: the average is many times the longest task.
  auto launch_time = [&](int form, int rows, int W, const std::vector<Part> &parts, int64_t nu, double sum_len,
                         int32_t max_len, const std::vector<int64_t> &at_least, const double *fl, bool *even) {
    const double slots = (double)sms * 16 / W;
    double tasks = 0, work = 0, longest = 0;
    for (const Part &p : parts) {
      const int chains = W * (32 / p.L);
      tasks += (double)((nu + chains - 1) / chains);
      work += (double)p.C * std::max(fl[p.L] * sum_len / chains, (double)max_len);
      longest = std::max(longest, (double)p.C * (double)round_up(max_len + inter_chain_lag(rows, form, p.L), kColBlock));
    }
    if (tasks <= 0) return 0.0;
    const int w = (int)std::max(1.0, std::min(4.0, std::ceil(tasks * W / (4.0 * sms))));
    const double cyc = chain_step_cycles(form, rows, w);
    if (tasks <= slots) {
      *even = false;
      return longest * cyc;
    }
    double bound = std::max(work / slots, longest);
    if (work / slots < 8 * longest) {
      *even = false;
      // x: the largest length with more than j * slots tasks at least that long
      auto longer = [&](double x) {  // tasks at least x long
        double cnt = 0;
        for (const Part &p : parts) {
          const double len = x / p.C - inter_chain_lag(rows, form, p.L);
          const size_t bin = len <= 0 ? 0 : (size_t)std::ceil(len / kColBlock);
          cnt += bin < at_least.size() ? std::ceil((double)at_least[bin] / (W * (32 / p.L))) : 0.0;
        }
        return cnt;
      };
      for (int j = 1; j <= 3 && tasks > j * slots; ++j) {
        if (longer(bound / (j + 1)) <= j * slots) continue;  // (x is no more than that)
        double lo = 0, hi = longest;
        for (int it = 0; it < 10; ++it) {
          const double x = 0.5 * (lo + hi);
          (longer(x) > j * slots ? lo : hi) = x;
        }
        bound = std::max(bound, (j + 1) * lo);
      }
    }
    return bound * cyc;
  };
  // counts of short units (of this mode; single sequences) at least 16 b long
  auto suffix_counts = [&](const std::vector<int64_t> &hist, size_t bins) {
    std::vector<int64_t> c(std::min(hist.size(), bins), 0);
    int64_t acc = 0;
    for (size_t b = c.size(); b-- > 0;) c[b] = acc += hist[b];
    return c;
  };
  const std::vector<int64_t> units_ge = suffix_counts(ust.hist, len_hist.size());
  std::vector<int64_t> singles_ge;
  double sum_single = 0;
  if (!elig.empty()) {
    const sw_db::UnitStats &single = db->units(false);
    singles_ge = suffix_counts(single.hist, len_hist.size());
    sum_single = (double)(single.prefix[(size_t)n] - single.prefix[(size_t)s0]);
  }
  // The plan at `rows` rows per lane with at least Lfloor lanes per chain
  // (where the query has that many): more lanes mean fewer chunks, so shorter
  // tasks, at the price of idle lanes and longer pipeline fill.
  // (the same queries are planned at many floors: costs that do not depend on the
  // floor are kept, and a floor that changes no choice is not planned.  31 queries
  // of 19 to 674 residues x 266 sequences: preparing 397 -> 219 us; four of 56 to
  // 68 x 615 95 -> 51)
  auto floor_of_any = [](int m, int rows) { return std::min(32, std::max(4, (m + rows - 1) / rows)); };
  std::vector<LaneCosts> kept_costs[7];  // by rows / 4: of each query, then of each group
  auto make_plan = [&](int rows, int Lfloor) {
    InterPlan P;
    P.R = rows;
    std::vector<LaneCosts> &kept = kept_costs[rows / 4];
    if (kept.empty() && n_queries <= 256) kept.resize((size_t)n_queries + 2 * elig.size());
    auto kept_of = [&](size_t k) { return kept.empty() ? nullptr : &kept[k]; };
    const double *fl = fill_of(packed ? kFormPacked : kFormInt32, rows), *flq = fill_of(kFormQPair, rows);
    auto floor_of = [&](int m) { return std::min(Lfloor, floor_of_any(m, rows)); };
    auto chunks_of = [&](int32_t q, int L) { return std::max(1, (qlen(q) + L * rows - 1) / (L * rows)); };
    // (a choice of L stays while the floor is at most L, or is bound by the length)
    auto chosen = [&](int m, int L) {
      if (L < floor_of_any(m, rows)) P.floor_to = std::min(P.floor_to, L);
      return L;
    };
    P.L.resize((size_t)n_queries);
    for (int64_t q = 0; q < n_queries; ++q) {
      const int m = std::max(1, qlen(q));
      P.L[q] = forceL ? forceL
               : q > 0 && qlen(q) == qlen(q - 1)
                   ? P.L[q - 1]  // (batches of one length: chosen once)
                   : chosen(m, choose_lanes(floor_of(m), kept_of((size_t)q),
                                            [&](int L) { return lanes_cost(m, rows, fl, L); }));
    }
    P.in_track.assign((size_t)n_queries, 0);
    if (!elig.empty()) {
      // Two ways to lay the eligible queries out, priced with the same model as
      // choose_lanes (padded rows x steps per column / lane use, the two halves of
      // a plan running max(track) chunks), the cheaper one kept:
      //  - grouped tracks: the queries sorted by length and cut into K consecutive
      //    groups, each packed longest first into two balanced tracks.  K grows
      //    with the query count (at least 8 queries per plan keep the tracks
      //    balanced) and so that every resident CTA sees several tiles;
      //  - pairs: neighbours in length order whose shorter one has at least 3/4
      //    of the longer one's rows share a plan (one query per track); the
      //    others keep the two-sequence form (two database sequences per chain;
      //    pairing their scores costs a byte shuffle per word, priced as 6/5 of
      //    the query-pair form's time per cell).
      // Each plan has its own lanes per chain.  (Many queries of similar length
      // favour pairs: each pair's L fits its length; few queries of spread-out
      // lengths favour tracks: no idle half.)
      // best L for a group packed into two tracks, and its modelled cost
      int last_a = -1, last_b = -1, last_L = 4;
      double last_cost = 0;
      auto pack = [&](const int32_t *g0, const int32_t *g1, int L, std::vector<int32_t> *out) {
        int64_t load[2] = {0, 0};
        for (const int32_t *q = g0; q < g1; ++q) {
          const int t = load[1] < load[0] ? 1 : 0;
          if (out) out[t].push_back(*q);
          load[t] += chunks_of(*q, L);
        }
        return std::max(load[0], load[1]);
      };
      auto plan_group = [&](const int32_t *g0, const int32_t *g1, size_t key, int *Lout) {
        auto cost_of = [&](int L) {
          const double eff = (double)((32 / L) * L) / 32.0, chunks = (double)pack(g0, g1, L, nullptr);
          return chunks * L * rows * flq[L] / eff * (1.0 + 0.002 * chunks / std::max<double>(1.0, (double)(g1 - g0)));
        };
        int Lp = forceL ? forceL : 4;
        // (neighbouring pairs of the same two lengths: chosen once)
        const bool again = g1 - g0 == 2 && last_a == qlen(g0[0]) && last_b == qlen(g0[1]);
        if (again) {
          *Lout = last_L;
          return last_cost;
        }
        if (!forceL)
          Lp = chosen(qlen(*g0), choose_lanes(floor_of(qlen(*g0)), kept_of((size_t)n_queries + key), cost_of));
        *Lout = Lp;
        const double cost = cost_of(Lp);
        if (g1 - g0 == 2) {
          last_a = qlen(g0[0]);
          last_b = qlen(g0[1]);
          last_L = Lp;
          last_cost = cost;
        }
        return cost;
      };
      auto solo_cost = [&](int32_t q) {  // two-sequence form: half the columns, 6/5 the time per word
        const int L = P.L[q];
        const double C = chunks_of(q, L), eff = (double)((32 / L) * L) / 32.0;
        return C * L * rows * fl[L] / eff * (1.0 + 0.001 * C) * 0.6;
      };
      const int64_t ne = (int64_t)elig.size();
      // grouped tracks
      struct Group {
        int64_t i0, i1;  // of elig
        int L;
      };
      std::vector<Group> gA, gB;
      double costA = 0, costB = 0;
      const int64_t tiles8 = std::max<int64_t>(1, (Q->n_single + 31) / 32);
      int64_t K = std::max<int64_t>((8 * 2 * (int64_t)sms + tiles8 - 1) / tiles8, std::min<int64_t>(8, ne / 8));
      K = std::max<int64_t>(1, std::min<int64_t>(K, ne / 2));
      gA.reserve((size_t)K);
      gB.reserve((size_t)(ne / 2));
      // (key: groups from 0, pairs from the count of eligible queries)
      auto add = [&](int64_t i0, int64_t i1, int64_t key, std::vector<Group> &g) {
        int Lp = 4;
        const double c = plan_group(elig.data() + i0, elig.data() + i1, (size_t)key, &Lp);
        g.push_back({i0, i1, Lp});
        return c;
      };
      for (int64_t k = 0; k < K; ++k) costA += add(ne * k / K, ne * (k + 1) / K, k, gA);
      // pairs
      std::vector<int32_t> soloB;
      for (int64_t i = 0; i < ne; ++i) {
        if (i + 1 < ne && 4 * (int64_t)qlen(elig[i + 1]) >= 3 * (int64_t)qlen(elig[i])) {
          costB += add(i, i + 2, ne + i, gB);
          ++i;
        } else {
          soloB.push_back(elig[i]);
          costB += solo_cost(elig[i]);
        }
      }
      for (int32_t q : elig) P.in_track[q] = 1;
      if (costB < costA)
        for (int32_t q : soloB) P.in_track[q] = 0;
      const std::vector<Group> &groups = costB < costA ? gB : gA;
      P.tracks.resize(2 * groups.size());
      for (size_t k = 0; k < groups.size(); ++k) {
        pack(elig.data() + groups[k].i0, elig.data() + groups[k].i1, groups[k].L, &P.tracks[2 * k]);
        P.plan_L.push_back(groups[k].L);
      }
    }
    std::vector<Part> solo, pairs;
    for (int64_t q = 0; q < n_queries; ++q)
      if (!P.in_track[q]) solo.push_back({chunks_of((int32_t)q, P.L[q]), P.L[q]});
    for (size_t k = 0; k < P.plan_L.size(); ++k) {
      int64_t load[2] = {0, 0};
      for (int h = 0; h < 2; ++h)
        for (int32_t q : P.tracks[2 * k + h]) load[h] += chunks_of(q, P.plan_L[k]);
      pairs.push_back({(int)std::max<int64_t>({1, load[0], load[1]}), P.plan_L[k]});
    }
    // CTAs shrink until the tasks cover every SM twice
    for (P.warps = inter_threads() / 32; P.warps > 2; P.warps /= 2) {
      int64_t tasks = 0;
      for (const Part &p : solo) tasks += (n_short + P.warps * (32 / p.L) - 1) / (P.warps * (32 / p.L));
      for (const Part &p : pairs) tasks += (Q->n_single + P.warps * (32 / p.L) - 1) / (P.warps * (32 / p.L));
      if (tasks >= 2 * sms) break;
    }
    P.even = true;
    P.time = launch_time(packed ? kFormPacked : kFormInt32, rows, P.warps, solo, n_short, sum_short, max_short,
                         units_ge, fl, &P.even);
    if (!pairs.empty())
      P.time += launch_time(kFormQPair, rows, P.warps, pairs, Q->n_single, sum_single, max_short, singles_ge, flq,
                            &P.even);
    return P;
  };
  // The plan with the least modelled time over the rows per lane and the
  // fewest lanes.  (Measured, GCUPS: one 1,301-residue query x 80,000 proteins
  // 24 rows x 8 lanes 5,783, x 4 5,050; 20 queries x 40,000 proteins 8 lanes
  // 6,745, 4 lanes 5,908; one 60-residue query x 80,000 16 rows x 4 lanes
  // 4,759, 24 rows x 4 2,982.)
  auto best_plan = [&]() {
    static const int kRows[] = {24, 16, 8};
    static const int kFloors[] = {5, 6, 8, 10, 12, 16, 20, 24, 32};
    InterPlan best;
    bool first = true;
    int floor_to[7] = {0};  // by rows / 4: floors up to it give the plan seen last
    int32_t m_max = 1;
    for (int64_t q = 0; q < n_queries; ++q) m_max = std::max(m_max, qlen(q));
    // the least a plan can take: the longest query's chunks over the longest
    // short unit, in either form, with the warp alone on its SM sub-partition
    auto at_least = [&](int rows, int Lfloor) {
      double t = 1e300;
      for (int form : {(int)kFormPacked, (int)kFormQPair, (int)kFormInt32}) {
        if (packed == (form == kFormInt32)) continue;
        double steps = 1e300;
        for (int L = std::min(Lfloor, floor_of_any(m_max, rows)); L <= 32; ++L)
          steps = std::min(steps, (double)((m_max + L * rows - 1) / (L * rows)) *
                                      (double)round_up(max_short + inter_chain_lag(rows, form, L), kColBlock));
        t = std::min(t, steps * chain_step_cycles(form, rows, 1));
      }
      return t;
    };
    auto consider = [&](int rows, int Lfloor) {
      if (Lfloor <= floor_to[rows / 4]) return false;
      if (!first && !forceL && n_queries > 1 && n_short > 0 && at_least(rows, Lfloor) >= best.time) return false;
      InterPlan P = make_plan(rows, Lfloor);
      floor_to[rows / 4] = P.floor_to;
      const bool even = P.even;
      if (first || P.time < best.time * (1 - 1e-9)) best = std::move(P);
      first = false;
      return even;
    };
    bool even = true;
    for (int rows : kRows)
      if (o.rows_per_lane ? rows == o.rows_per_lane : rows > 8 || n_queries <= 32) even &= consider(rows, 4);
    if (first) even = consider(R, 4);  // (4 or 12 rows, by option)
    if (even || forceL) return best;
    if (n_queries > 32) {  // (many queries: each plan costs more, and the choice matters less)
      const int rows = best.R;
      for (int Lfloor : {8, 16, 32}) consider(rows, Lfloor);
      return best;
    }
    for (int Lfloor : kFloors)
      if (o.rows_per_lane) consider(o.rows_per_lane, Lfloor);
      else
        for (int rows : kRows) consider(rows, Lfloor);
    return best;
  };
  InterPlan plan;

  // --- small batches: band-stream jobs and transposed jobs (k_band.cu).  In
  // a batch too small to fill the GPU, the longest chains of the inter-task
  // kernel set the time while most SMs idle, so:
  //  - a query of at least two bands (2 x 32 x band_rows rows; 1,024 with the
  //    default 16 rows per lane) runs against every database unit as
  //    pipelines of bands, one warp each: a job is one query and a stream of
  //    units, all its bands sweeping the stream together.  A unit whose pair
  //    with the query could pass the 16-bit range is split into its
  //    sequences in int32; the others keep two sequences per word.  Streams
  //    are cut so that every warp of one launch gets about one and a half
  //    jobs' worth of columns (one unit at least);
  //  - every shorter query runs transposed: the database sequences are the
  //    rows, stacked in row tracks of whole lanes (8 to 24 rows, the height
  //    with the least modelled time), and the query the columns; each band of
  //    a track is one warp, several short sequences share a band, and the
  //    bands of a longer one run as a pipeline.  In packed mode two tracks
  //    share each word (their substitution bytes paired per row), except
  //    sequences whose pair with the longest of these queries could pass the
  //    16-bit range (int32 tracks).
  // The inter- and intra-task kernels are then not used.  If the rings (one
  // entry per column between consecutive bands) do not fit a memory budget,
  // the batch takes the regular plan.
  std::vector<char> band_q(n_queries, 0), track_q(n_queries, 0), small_q(n_queries, 0);
  // (the planner's large tables live in per-thread buffers that keep their
  // memory from one plan to the next: fresh allocations of a few hundred KB
  // each cost their page faults again, ~0.2-0.8 ms per plan)
  PlanScratch &scratch = plan_scratch();
  std::vector<BandJob> &bjobs = scratch.bjobs;
  std::vector<int32_t> &bjob_of = scratch.bjob_of;
  std::vector<int2> &btpos = scratch.btpos;
  std::vector<TrackJob> &tjobs = scratch.tjobs;
  std::vector<TrackGroup> &tgroups = scratch.tgroups;
  std::vector<TrackLane> &tlanes = scratch.tlanes;
  std::vector<int64_t> qt_off(std::max<int64_t>(n_queries, 1), 0);
  std::vector<int32_t> qt_npad(std::max<int64_t>(n_queries, 1), 16);
  bool band_mode = false;
  // The load of one query in lanes of tR rows, estimated from the length
  // histogram (lengths up to cut take the 16-bit tracks).
  auto track_estimate = [&](int tR, const sw_db::UnitStats &single, int32_t cut) {
    const int tL = track_long_rows(tR);
    TrackLoad e;
    double lanes[2] = {0, 0};
    for (size_t h = 1; h < single.hist.size(); ++h) {
      if (!single.hist[h]) continue;
      const int64_t len = (int64_t)h * kColBlock - 7;  // (the middle of the bin)
      const int f = len > cut ? 1 : 0;
      if (len <= 32 * tR) {
        lanes[f] += (double)single.hist[h] * (double)((len + tR - 1) / tR);
      } else {
        const int64_t nb = (len + 32 * tL - 1) / (32 * tL);
        e.bands[f] += (double)(single.hist[h] * nb);
        e.deepest[f] = std::max(e.deepest[f], nb);
        // (short sequences fill most of what the last band leaves)
        lanes[f] -= 0.8 * (double)single.hist[h] * (double)(32 * tL * nb - len) / tR;
      }
    }
    for (int f = 0; f < 2; ++f)  // (two 16-bit tracks share a band)
      e.bands[f] = std::ceil((e.bands[f] + std::max(0.0, lanes[f]) / 32 / 0.98) * (f == 0 ? 0.5 : 1.0));
    return e;
  };
  // Modelled time (cycles) of the transposed jobs: their bands over the SM
  // sub-partitions, up to the launch's residency at a time; at least the
  // longest pipeline, whose bands start about 50 steps after one another.
  auto track_time = [&](int tR, int occ, const TrackLoad &load) {
    double steps_sum = 0, steps_max = 0, n_q = 0;
    for (int64_t q = 0; q < n_queries; ++q) {
      if (!track_q[q]) continue;
      const double steps = (double)(round_up(std::max(1, qlen(q)), kColBlock) + 64) / 2;
      steps_sum += steps;
      steps_max = std::max(steps_max, steps);
      ++n_q;
    }
    const double parts = 4.0 * sms, nb = n_q * (load.bands[0] + load.bands[1]);
    const int w = (int)std::max(1.0, std::min((double)occ, std::ceil(nb / parts)));
    double work = 0, step_max = 0, chain = 0;
    for (int f = 0; f < 2; ++f) {
      if (load.bands[f] <= 0) continue;
      const double step = track_step_cycles(f == 0, tR, w);
      work += load.bands[f] * steps_sum * step;
      step_max = std::max(step_max, step);
      if (load.deepest[f] > 1)
        chain = std::max(chain, (steps_max + 50.0 * (double)(load.deepest[f] - 1)) *
                                    track_step_cycles(f == 0, track_long_rows(tR), w));
    }
    const double all = nb > parts * w ? work / (parts * w) + 0.5 * steps_max * step_max : steps_max * step_max;
    return std::max(all, chain);
  };
  // a sequence takes the 16-bit tracks (packed mode) unless its pair with the
  // longest of these queries could pass the 16-bit range: a length cut that
  // depends on the queries only through that longest one
  auto track_cut = [&]() {
    int32_t mtq = 0;
    for (int64_t q = 0; q < n_queries; ++q)
      if (track_q[q]) mtq = std::max(mtq, qlen(q));
    return !packed ? -1
           : (int64_t)sc.maxp * mtq <= sc.thresh ? std::numeric_limits<int32_t>::max()
                                                 : sc.thresh / sc.maxp;
  };
  // rows per lane and cut of the transposed jobs, in order of the modelled
  // time.  A deep pipeline's time is its bands' steps one after the other, and
  // an int32 step is the shorter one (16 rows: 353 against 460 cycles), so
  // sequences past kDeepCut may take int32 tracks where there are few of them
  // (144 residues, packed, x one sequence of 35,000: 765 -> 605 us; x 4,000
  // proteins and one of 9,000: 236 -> 203).
  constexpr int32_t kDeepCut = 2048;
  struct TrackChoice {
    double time;
    int tR, occ;
    int32_t cut;
  };
  std::vector<TrackChoice> heights;
  auto rank_heights = [&]() {
    heights.clear();
    const sw_db::UnitStats &single = db->units(false);
    const int32_t cut = track_cut();
    // (beside band-stream jobs, which take longer, the fewer bands are the better)
    const bool alone = std::find(band_q.begin(), band_q.end(), (char)1) == band_q.end();
    for (const TrackHeight &h : kTrackHeights) {
      const int occ = cached_occupancy(2, h.rows, 0, gaps, 0, 0);
      if (occ <= 0) continue;
      heights.push_back({track_time(h.rows, occ, track_estimate(h.rows, single, cut)), h.rows, occ, cut});
      if (alone && cut > kDeepCut && db->max_npad > kDeepCut)
        heights.push_back({track_time(h.rows, occ, track_estimate(h.rows, single, kDeepCut)), h.rows, occ, kDeepCut});
    }
    std::stable_sort(heights.begin(), heights.end(),
                     [](const TrackChoice &x, const TrackChoice &y) { return x.time < y.time; });
    // (the deep sequences in int32 only where that is clearly the faster: the
    // chains' part of the model is within 20 %)
    const auto plain = std::find_if(heights.begin(), heights.end(), [&](const TrackChoice &c) { return c.cut == cut; });
    if (plain != heights.end()) {
      const int32_t keep = heights[0].time < 0.8 * plain->time ? heights[0].cut : cut;
      heights.erase(std::remove_if(heights.begin(), heights.end(), [&](const TrackChoice &c) { return c.cut != keep; }),
                    heights.end());
    }
    return heights.empty() ? 1e300 : heights[0].time;
  };
  auto rank_heights_of = [&]() {
    for (int64_t q = 0; q < n_queries; ++q)
      if (track_q[q]) return rank_heights();
    return 0.0;
  };
  // Modelled time (cycles) of the band-stream jobs of the queries in band_q:
  // cells at the kernel's rate, or one stream's columns and the bands'
  // hand-offs one after another (from timings of one query of 1,301 to 6,000
  // residues x 500 to 40,000 proteins, within 20 %).  A band's last lane ends a
  // unit 31 columns after its first, which is a tenth of a protein and more
  // than a peptide: 4,852 residues x 58,000 of about 20, int32, 7.3 ms (2.5 by the
  // sequences' own cells; 3.4 inter-task, 2.2 transposed).
  auto band_time = [&]() {
    double thr = 0, lat = 0;
    const int brows = 32 * bR;
    const double columns = (double)db->units(false).prefix[(size_t)n] + 32.0 * (double)n;
    const double widest = Q->n_units > 0 ? (double)unit_len(0) : 0.0;
    for (int64_t q = 0; q < n_queries; ++q) {
      if (!band_q[q]) continue;
      const double nb = (double)((qlen(q) + brows - 1) / brows), rows = nb * brows;
      const bool i32 = !packed || may_flag(q, (int32_t)widest);  // (some units in int32: their columns set the pace)
      thr += rows * columns / (packed ? 2510 : 1485);
      lat = std::max(lat, packed && !i32 ? 528 * widest + 24800 * nb : (packed ? 180 : 310) * widest + 27000 * nb);
    }
    return 0.95 * std::max(thr, lat) + 0.15 * std::min(thr, lat);
  };
  // A lower bound of the inter-task plan's modelled time: the longest query's
  // chunks over the longest short unit, in the plan's rows or any of them,
  // with the warp alone on its SM sub-partition.
  auto inter_at_least = [&]() {
    if (n_short <= 0) return 0.0;
    double m = 1, best = 1e300;
    for (int64_t q = 0; q < n_queries; ++q) m = std::max<double>(m, qlen(q));
    for (int rows : {24, 16, 12, 8, 4})
      if (!o.rows_per_lane || rows == o.rows_per_lane)
        best = std::min(best, std::ceil(m / (32 * rows)) * max_short *
                                  chain_step_cycles(packed ? kFormQPair : kFormInt32, rows, 1));
    return best;
  };
  // Modelled time (cycles) of the intra-task launches, one CTA (and matrix) per
  // SM: the longest matrix, or all of them over the SMs.  A chain sweeps a
  // unit's columns one after the other, however few rows it has: 550 cycles a
  // column for a query of one warp (500 with 32-bit cells), 1,000 + 32 per warp
  // where its warps pass the rows on (60 to 5,000 residues against sequences of
  // up to 35,000: 8.6 to 23 ms, within 6 %).
  auto intra_time = [&]() {
    double longest = 0, work = 0;
    for (int64_t q = 0; q < n_queries; ++q) {
      const int w = std::max(1, std::min(intra_threads() / 32, (qlen(q) + 32 * Ri - 1) / (32 * Ri)));
      const double chunks = std::ceil(std::max(1, qlen(q)) / (32.0 * w * Ri));
      const double column = chunks * (w > 1 ? 1000 + 32 * w : packed ? 550 : 500) * Ri / 16;
      longest = std::max(longest, column * max_long);
      // (pairs of sequences that could pass the 16-bit range run one by one)
      work += column * (double)ust.prefix[(size_t)n_long] * (may_flag(q, max_long) ? 2 : 1);
    }
    return std::max(longest, work / sms);
  };
  // Which kernels: the small-batch ones (band-stream jobs for the long queries
  // and transposed ones for the others, or all transposed), or the inter- and
  // intra-task ones, by modelled time.
  //  - Where the database has units past the cutover, at any size whose row
  //    tracks it can keep: the intra-task kernel takes one such unit far longer
  //    than bands do (35,000 residues: 9.4 against 0.78 ms for a 144-residue
  //    query, 18.1 against 2.1 ms for 1,301).  The model picks within 5 % of the
  //    faster side up to 40,000 proteins; above 16,384 the small-batch kernels
  //    have to be modelled a tenth faster (3,000 residues x 150,000 proteins,
  //    less than that apart: 25.7 against 24.1 ms).
  //  - Else up to 16,384 sequences, or of 200 residues on average at most (and
  //    10 million together): longer ones are laid in row tracks too slowly for a
  //    new database, for sides that differ little (17,000 to 40,000 proteins,
  //    packed: transposed jobs 0.78 to 1.2 of the inter-task time at 144
  //    residues, 0.85 to 0.88 at 400, 0.95 to 1.0 at 1,000, 1.05 to 1.2 at
  //    1,301, 1.0 to 1.6 at 60), but the shorter the sequences the more of the
  //    inter-task kernel's steps are fill (144 residues, packed, x 17,000 of
  //    about 60: 102 us transposed, 172 inter-task; 1,000 x 60,000 of about 20
  //    449 and 945).  Its model is low there by up to a half where the sequences
  //    are the shortest or the query has 200 residues or more, and the transposed
  //    jobs' is for a query of 60 or less: a factor weighs them (17,000 to 80,000
  //    sequences of 10 to 200 on average x 40 to 1,000 residues, both modes).  Not
  //    above 1 for packed batches that fill the query tracks (256 queries of 30 to
  //    285 x 60,000 of about 30: 20.0 ms inter-task, 23.9 transposed).
  bool small = o.band_stream == 2;
  if (n > 0 && n_queries > 0 && o.band_stream != 1) {
    bool any_band = false;
    for (int64_t q = 0; q < n_queries; ++q) {
      band_q[q] = qlen(q) >= 2 * 32 * bR;
      track_q[q] = !band_q[q];
      any_band |= band_q[q] != 0;
    }
    int32_t m_max = 0;
    for (int64_t q = 0; q < n_queries; ++q) m_max = std::max(m_max, qlen(q));
    const bool peptides = !n_long && n > 16384 && db->total <= std::min<int64_t>(200 * n, 10000000);
    const auto ramp = [](double x, double lo, double hi) { return std::min(1.0, std::max(0.0, (x - lo) / (hi - lo))); };
    double peptide_factor =
        (0.75 + 0.4 * ramp(m_max, 60, 300)) * (1.2 - 0.2 * ramp((double)db->total / (double)n, 30, 100));
    if (packed && n_queries >= 16) peptide_factor = std::min(1.0, peptide_factor);
    if (o.band_stream == 0 && (n <= 16384 || (n_long && db->keeps_tracks()) || peptides)) {
      const double tracks_a = rank_heights_of(), bands_a = any_band ? band_time() : 0.0;
      double best_small = std::max(tracks_a, bands_a) + 0.5 * std::min(tracks_a, bands_a);
      if (any_band) {  // all transposed?
        std::vector<char> bq = band_q, tq = track_q;
        std::fill(band_q.begin(), band_q.end(), 0);
        std::fill(track_q.begin(), track_q.end(), 1);
        const double all = rank_heights_of();
        if (all < best_small) {
          best_small = all;
        } else {
          band_q.swap(bq);
          track_q.swap(tq);
        }
      }
      // (the plan is left out where its longest chain alone would take longer:
      // one 144-residue query x 2,000 proteins, 7.6 of 130 us)
      if (best_small < inter_at_least()) {
        small = true;
      } else {
        plan = best_plan();
        double inter = plan.time;
        if (n_long) {  // the intra-task kernel beside it
          const double intra = intra_time();
          inter = std::max(inter, intra) + 0.3 * std::min(inter, intra);
        }
        const bool bands = std::find(band_q.begin(), band_q.end(), (char)1) != band_q.end();
        small = best_small < (peptides && !bands ? peptide_factor : n_long && n > 16384 ? 0.9 : 1.0) * inter;
      }
    }
  }
  if (small) {
    const int brows = 32 * bR;
    bool any_band = false, any_track = false;
    for (int64_t q = 0; q < n_queries; ++q) {
      any_band |= band_q[q] != 0;
      any_track |= track_q[q] != 0;
    }
    const int bmax = any_band ? cached_occupancy(1, bR, 0, gaps, 0, 0) : 1;
    int bocc = bmax;
    if (any_track) rank_heights();
    int tocc = !any_track ? 1 : heights.empty() ? 0 : heights[0].occ;
    int64_t ring = 0, band = 0, tring = 0, tband = 0, n_tlanes = 0;
    if (bocc > 0 && tocc > 0) {
      // band jobs: each band query against every unit
      struct BList {
        int32_t q, packed, nb;
        std::vector<int2> t;
        std::vector<int32_t> w;  // columns of each unit
        int64_t cols = 0, widest = 0;
      };
      std::vector<BList> lists;
      double total = 0;
      for (int64_t q = 0; q < n_queries; ++q) {
        if (!band_q[q]) continue;
        const int32_t nb = std::max(1, (qlen(q) + brows - 1) / brows);
        BList lp{(int32_t)q, 1, nb, {}, {}, 0}, li{(int32_t)q, 0, nb, {}, {}, 0};
        for (int64_t u = 0; u < Q->n_units; ++u) {
          const int32_t a = unit_seq(packed ? 2 * u : u), b = packed ? unit_seq(2 * u + 1) : a;
          if (packed && !may_flag(q, unit_len(u))) {
            lp.t.push_back(make_int2(a, b));
            lp.w.push_back(std::max(npad[a], npad[b]));
            lp.cols += lp.w.back();
          } else {
            li.t.push_back(make_int2(a, a));
            li.w.push_back(npad[a]);
            li.cols += npad[a];
            if (b != a) {
              li.t.push_back(make_int2(b, b));
              li.w.push_back(npad[b]);
              li.cols += npad[b];
            }
          }
        }
        for (BList *L : {&lp, &li})
          if (!L->t.empty()) {
            total += (double)L->nb * (double)L->cols;
            for (int32_t x : L->w) L->widest = std::max<int64_t>(L->widest, x);
            lists.push_back(std::move(*L));
          }
      }
      // Streams are cut into jobs of about per_warp columns, three jobs per two
      // warps of the launch (a warp that finishes early takes a band of the
      // second wave, whose pipeline fill overlaps the first wave's drain; one,
      // two and three jobs per warp: 663, 564, 559 against 528 us for a
      // 1,301-residue query x 5,000 proteins).  Units
      // are not cut, so an int32 unit wider than per_warp makes a job that
      // sets the pace of the launch: it runs in bands of half the height
      // (half the work per step; its steps run one after the other), and if
      // its steps, slowed by the other warps that share its SM sub-partition
      // (those of every CTA on the SM, all computing), would outlast the
      // launch's average load, the launch keeps one CTA per SM (a choice
      // only for band heights whose CTAs fit twice on an SM).
      constexpr double kWaves = 1.5;
      const int wpc = band_threads() / 32;  // warps per CTA
      auto per_warp_at = [&](int occ) {
        return std::max<int64_t>(1, (int64_t)std::ceil(total / ((double)sms * occ * wpc * kWaves)));
      };
      if (bocc > 1) {
        const int64_t pw = per_warp_at(bocc);
        double crit = 0;  // steps of the widest oversized int32 unit, in full-height band steps
        for (const BList &L : lists)
          if (!L.packed && L.widest > pw) crit = std::max(crit, 0.5 * (double)L.widest);
        const double warps_per_smsp = (double)bocc * wpc / 4.0;
        const double load = total / ((double)sms * 4.0);  // full-height band steps per SM sub-partition
        if (crit * warps_per_smsp > 1.3 * load) bocc = 1;
      }
      const int64_t per_warp = per_warp_at(bocc);
      for (const BList &L : lists) {
        size_t i = 0;
        while (i < L.t.size()) {
          BandJob j{};
          j.q = L.q;
          j.form = L.packed ? kBandPacked : kBandInt32;
          j.nb = L.nb;
          j.t_begin = (int32_t)btpos.size();
          int64_t cols = 0;
          while (i < L.t.size() && (cols == 0 || cols + L.w[i] <= per_warp)) {
            btpos.push_back(L.t[i]);
            cols += L.w[i];
            ++i;
          }
          j.t_count = (int32_t)(btpos.size() - j.t_begin);
          j.cols = cols;
          // an int32 unit wider than the budget (a long query against a long
          // sequence whose pair could pass the 16-bit range) makes the job
          // that sets the pace of the launch: bands of half the height halve
          // the work of each of its steps, which run one after the other
          if (!L.packed && cols > per_warp) {
            j.form = kBandInt32Half;
            j.nb = std::max(1, (qlen(L.q) + brows / 2 - 1) / (brows / 2));
          }
          bjobs.push_back(j);
        }
      }
      // longest streams first: their bands are handed out first
      std::stable_sort(bjobs.begin(), bjobs.end(), [](const BandJob &x, const BandJob &y) {
        return (int64_t)x.nb * x.cols > (int64_t)y.nb * y.cols;
      });
      for (size_t k = 0; k < bjobs.size(); ++k) {
        bjobs[k].band0 = (int32_t)band;
        bjobs[k].ring0 = ring;
        ring += (int64_t)(bjobs[k].nb - 1) * bjobs[k].cols;
        for (int b = 0; b < bjobs[k].nb; ++b) bjob_of.push_back((int32_t)k);
        band += bjobs[k].nb;
      }

      // transposed jobs: the database in row tracks, each short query as columns
      int64_t qt = 0;
      int64_t n_track_q = 0;
      for (int64_t q = 0; q < n_queries; ++q) {
        if (!track_q[q]) continue;
        ++n_track_q;
        qt_npad[q] = (int32_t)std::max<int64_t>(kColBlock, round_up(qlen(q), kColBlock));
        qt_off[q] = qt;
        qt += qt_npad[q];
      }
      Q->qt_bytes = std::max<int64_t>(qt, 16);
      // the jobs: each pipeline once per query, deeper pipelines first, and the
      // order of their bands.  Job by job, the warps in flight hold a few
      // pipelines, whose bands run about 50 steps apart and wait on one another;
      // by level (bands with more of their job below them first) a band follows
      // the one above it with the other jobs' bands of that depth between them.
      // By level where those 50 steps a band outlast a band's own or the bands
      // fill the warps twice (40 queries of 144 residues x 5 sequences of 30,000:
      // 4.25 ms job by job, 0.69 by level; four of 100 to 400 x 1,200 of 2,500: 1.02
      // and 0.73); else the hand-off to a neighbour on the same SM is the faster
      // (400 residues x 4,000 proteins and 400 of 2,500: 301 and 321 us).
      auto make_jobs = [&](const std::vector<TrackPipe> &pipes, int occ) {
        tjobs.clear();
        tgroups.clear();
        tring = 0;
        tband = 0;
        int32_t steps = 0;
        for (const TrackPipe &pp : pipes)
          for (int64_t q = 0; q < n_queries; ++q) {
            if (!track_q[q]) continue;
            TrackJob j{};
            j.q = (int32_t)q;
            j.packed = pp.packed;
            j.nb = pp.nb;
            j.rows = pp.rows;
            j.lane0 = pp.lane0;
            j.ring0 = tring;
            tring += (int64_t)(pp.nb - 1) * qt_npad[q];
            tband += pp.nb;
            steps = std::max(steps, (qt_npad[q] + 64) / 2);
            tjobs.push_back(j);
          }
        if (tband >= ((int64_t)1 << 30)) return;  // (the plan is refused below)
        const int32_t deepest = tjobs.empty() ? 0 : tjobs[0].nb;
        int32_t start = 0;
        if (deepest > 2 && (50 * (int64_t)(deepest - 1) > steps ||
                            tband > 2 * (int64_t)sms * occ * (track_threads() / 32))) {
          size_t k = 0;
          for (int32_t below = deepest; below > 0; --below) {
            while (k < tjobs.size() && tjobs[k].nb >= below) ++k;
            tgroups.push_back({start, 0, 0, below});
            start += (int32_t)k;
          }
        } else {
          for (size_t k = 0; k < tjobs.size(); ++k) {
            if (k == 0 || tjobs[k].nb != tjobs[k - 1].nb) tgroups.push_back({start, (int32_t)k, tjobs[k].nb, 0});
            start += tjobs[k].nb;
          }
        }
      };
      if (any_track) {
        // the height with the least modelled time; one that its packed bands
        // make slower than the next one's estimate gives way to that.  The
        // layouts come from the database's kept ones where it keeps them, so
        // that repeated searches skip the binning and the lane upload.
        TrackBins &bins = scratch.bins;
        TrackChoice c = heights[0];
        const sw_db::TrackLayout *lay = db->track_layout(c.tR, c.cut, s);
        if (lay) c.time = track_time(c.tR, c.occ, lay->load);
        for (size_t k = 1; lay && k < heights.size() && heights[k].time < c.time; ++k) {
          const TrackChoice &h = heights[k];
          const sw_db::TrackLayout *other = db->track_layout(h.tR, h.cut, s);
          if (!other) break;
          const double t = track_time(h.tR, h.occ, other->load);
          if (t < c.time) {
            c = {t, h.tR, h.occ, h.cut};
            lay = other;
          }
        }
        if (!lay) bin_tracks(db->h_len, c.tR, c.cut, bins);
        const int tR = c.tR;
        tocc = c.occ;
        if (lay) {
          make_jobs(lay->pipes, tocc);
          Q->d_tlanes = lay->d_lanes;  // the database's (not the batch's block)
          n_tlanes = lay->n_lanes;
        } else {
          lay_tracks(bins, tR, scratch.tpipes, tlanes);
          make_jobs(scratch.tpipes, tocc);
          n_tlanes = (int64_t)tlanes.size();
        }
        Q->tR = tR;
      }
      const int64_t kBandRingBudget = (int64_t)4 << 30;
      band_mode = 8 * (ring + tring) <= kBandRingBudget && band + tband < ((int64_t)1 << 30) &&
                  n_tlanes < ((int64_t)1 << 31);
      if (band_mode) {
        Q->n_bjobs = (int64_t)bjobs.size();
        Q->n_bands = band;
        Q->n_btargets = (int64_t)btpos.size();
        Q->band_ring_bytes = 8 * ring;
        Q->bR = bR;
        Q->bgrid = (int)std::max<int64_t>(1, std::min<int64_t>((band + band_threads() / 32 - 1) / (band_threads() / 32),
                                                               (int64_t)sms * bocc));
        Q->bone = bocc == 1 && bmax > 1;
        Q->n_tjobs = (int64_t)tjobs.size();
        Q->n_tbands = tband;
        Q->n_tgroups = (int)tgroups.size();
        Q->n_tlanes = n_tlanes;
        Q->tlanes_shared = Q->d_tlanes != nullptr;
        Q->track_ring_bytes = 8 * tring;
        Q->tgrid = (int)std::max<int64_t>(1, std::min<int64_t>((tband + track_threads() / 32 - 1) / (track_threads() / 32),
                                                               (int64_t)sms * tocc));
        for (int64_t q = 0; q < n_queries; ++q) small_q[q] = band_q[q] || track_q[q];
      }
    }
    if (!band_mode) {
      bjobs.clear();
      bjob_of.clear();
      btpos.clear();
      tjobs.clear();
      tgroups.clear();
      tlanes.clear();
      Q->d_tlanes = nullptr;
    }
  }
  if (!band_mode) {
    std::fill(band_q.begin(), band_q.end(), 0);
    std::fill(track_q.begin(), track_q.end(), 0);
  }

  // --- the inter-task plan, unless the batch takes the small-batch kernels
  if (band_mode) plan = InterPlan();
  else if (plan.L.empty()) plan = best_plan();
  R = plan.R;
  Q->R = R;
  const int warps = plan.warps, threads = warps * 32;
  Q->threads = threads;
  std::vector<char> &in_track = plan.in_track;
  std::vector<std::vector<int32_t>> &tracks = plan.tracks;
  std::vector<int> &plan_L = plan.plan_L;
  in_track.resize((size_t)n_queries, 0);
  plan.L.resize((size_t)n_queries, 32);
  Q->n_solo = 0;  // queries with a profile of their own (not in query-pair tracks, not band-stream jobs)
  for (int64_t q = 0; q < n_queries; ++q) Q->n_solo += (in_track[q] || small_q[q]) ? 0 : 1;
  Q->npairs = (int64_t)plan_L.size();  // track plans

  // --- per-query plans and profile layout (queries in a pair get no solo profile)
  Q->qd.resize(n_queries);
  Q->qdi.resize(n_queries);
  int64_t prof = 0;
  int maxc = 16, maxci = 16, maxcp = 16;
  bool chunked = false, ichunked = false;
  for (int64_t q = 0; q < n_queries; ++q) {
    QDesc &d = Q->qd[q];
    d.m = qlen(q);
    d.R = R;
    d.L = plan.L[q];
    const int LR = d.L * R;
    d.nchunks = std::max(1, (d.m + LR - 1) / LR);
    d.chunk_stride = (int32_t)round_up((int64_t)profile_slots(d.L) * R, 128);
    d.chunk_bytes = (in_track[q] || small_q[q]) ? 0 : kProfRows * d.chunk_stride;
    d.prof_off = prof;
    d.qoff = q_offsets[q];
    prof += (int64_t)d.nchunks * d.chunk_bytes;
    maxc = std::max(maxc, d.chunk_bytes);
    chunked |= d.chunk_bytes > 0 && d.nchunks > 1;
  }
  // track plans: 4-byte entries; every plan uses the chunk layout of 32 lane
  // slots of R words (the most any L needs), so one kernel builds all of
  // them; chunks of all plans in table order, plan p's from track_off
  Q->qdp.resize(Q->npairs);
  Q->track.clear();
  {
    const int32_t stride = (int32_t)round_up(4 * (int64_t)32 * R, 128);
    for (int64_t p = 0; p < Q->npairs; ++p) {
      QDesc &d = Q->qdp[p];
      const int LR = plan_L[p] * R;
      std::vector<TrackChunk> half[2];
      for (int h = 0; h < 2; ++h)
        for (int32_t q : tracks[2 * p + h]) {
          const int C = std::max(1, (qlen(q) + LR - 1) / LR);
          for (int k = 0; k < C; ++k) {
            TrackChunk t{};
            t.qa = q;
            t.ka = k;
            t.flags = (k == 0 ? kStartA : 0) | (k == C - 1 ? kEndA : 0);
            half[h].push_back(t);
          }
        }
      const size_t nc = std::max(half[0].size(), half[1].size());
      d.track_off = (int32_t)Q->track.size();
      for (size_t c = 0; c < nc; ++c) {
        TrackChunk t{};
        t.qa = c < half[0].size() ? half[0][c].qa : -1;
        t.ka = c < half[0].size() ? half[0][c].ka : 0;
        t.qb = c < half[1].size() ? half[1][c].qa : -1;
        t.kb = c < half[1].size() ? half[1][c].ka : 0;
        t.flags = (c < half[0].size() ? half[0][c].flags : 0) | (c < half[1].size() ? half[1][c].flags * 2 : 0);
        t.L = plan_L[p];
        Q->track.push_back(t);
      }
      d.m = (int32_t)nc * LR;
      d.L = plan_L[p];
      d.R = R;
      d.nchunks = (int32_t)nc;
      d.chunk_stride = stride;
      d.chunk_bytes = kProfRows * stride;
      d.prof_off = prof;
      d.qoff = 0;
      prof += (int64_t)nc * d.chunk_bytes;
      maxcp = std::max(maxcp, d.chunk_bytes);
      chunked |= nc > 1;
    }
  }
  if (n_long && !band_mode) {
    const int wmax = intra_threads() / 32;
    for (int64_t q = 0; q < n_queries; ++q) {
      QDesc &d = Q->qdi[q];
      d.m = Q->qd[q].m;
      d.R = Ri;
      const int w = (int)std::min<int64_t>(wmax, std::max<int64_t>(1, (d.m + 32 * Ri - 1) / (32 * Ri)));
      d.L = 32 * w;
      const int LR = d.L * Ri;
      d.nchunks = std::max(1, (d.m + LR - 1) / LR);
      d.chunk_stride = (int32_t)round_up((int64_t)profile_slots(d.L) * Ri, 128);
      d.chunk_bytes = kProfRows * d.chunk_stride;
      d.prof_off = prof;
      d.qoff = q_offsets[q];
      prof += (int64_t)d.nchunks * d.chunk_bytes;
      maxci = std::max(maxci, d.chunk_bytes);
      ichunked |= d.nchunks > 1;
    }
  }
  Q->prof_bytes = std::max<int64_t>(prof, 16);
  Q->pbuf_bytes = (int)round_up(maxc, 128);
  Q->ipbuf_bytes = (int)round_up(maxci, 128);
  Q->ppbuf_bytes = (int)round_up(maxcp, 128);

  // --- tasks, longest first
  std::vector<TW> twi, twi32, twp;
  std::vector<TW> &tw = scratch.tw;
  std::vector<int32_t> ipos32;  // database positions of the int32 intra-task units
  int64_t rcap = 0;
  // (a pair of sequences scores at most max(SM) * min(m, n): a packed lane
  // that cannot pass the threshold needs no rescue pass)
  for (int64_t p = 0; p < Q->npairs; ++p) {  // query pairs x single short sequences
    const QDesc &d = Q->qdp[p];
    const int chains = warps * (32 / d.L);
    for (int64_t i0 = 0; i0 < Q->n_single; i0 += chains) {
      Task t{(int32_t)p, (int32_t)i0, (int32_t)std::min<int64_t>(chains, Q->n_single - i0), 0};
      twp.push_back({t, (double)d.nchunks * d.L * d.R * (npad[s0 + i0] + d.L + 8)});
    }
  }
  std::vector<size_t> tw_runs;  // start of each query's tiles in tw (each run is longest first already)
  for (int64_t q = 0; q < n_queries && Q->n_units > n_long; ++q) {
    if (in_track[q] || small_q[q]) continue;
    const QDesc &d = Q->qd[q];
    const int chains = warps * (32 / d.L);
    tw_runs.push_back(tw.size());
    tw.reserve(tw.size() + (size_t)((Q->n_units - n_long + chains - 1) / chains));
    for (int64_t u0 = n_long; u0 < Q->n_units; u0 += chains) {
      Task t{(int32_t)q, (int32_t)u0, (int32_t)std::min<int64_t>(chains, Q->n_units - u0), 0};
      tw.push_back({t, (double)d.nchunks * d.L * d.R * (unit_len(u0) + d.L + 8)});
    }
    rcap += (n + chains - 1) / chains;
    Q->inter_may_flag |= may_flag(q, max_short);
  }
  // long units: packed intra-task kernel where no lane can saturate, int32
  // otherwise (recomputing a saturated long matrix would cost more than
  // computing it once in int32)
  for (int64_t q = 0; q < n_queries && n_long && !band_mode; ++q) {
    const QDesc &d = Q->qdi[q];
    for (int64_t u = 0; u < n_long; ++u) {
      const double w = (double)d.nchunks * d.L * d.R * (unit_len(u) + d.L);
      if (packed && !may_flag(q, unit_len(u))) {
        twi.push_back({Task{(int32_t)q, (int32_t)u, 1, 0}, w});
        continue;
      }
      const int32_t a = unit_seq(packed ? 2 * u : u);
      const int32_t b = packed ? unit_seq(2 * u + 1) : a;
      twi32.push_back({Task{(int32_t)q, (int32_t)ipos32.size(), 1, 0}, 2 * w});
      ipos32.push_back(a);
      if (b != a) {
        twi32.push_back({Task{(int32_t)q, (int32_t)ipos32.size(), 1, 0}, 2 * w});
        ipos32.push_back(b);
      }
    }
  }
  // all tiles longest first (ties in query order): the stable merge of the
  // queries' runs, each already longest first (units are sorted), in place
  // of a full sort of up to a few hundred thousand tiles
  {
    auto longer = [](const TW &a, const TW &b) { return a.w > b.w; };
    tw_runs.push_back(tw.size());
    while (tw_runs.size() > 2) {
      std::vector<size_t> next;
      for (size_t i = 0; i + 2 < tw_runs.size(); i += 2) {
        std::inplace_merge(tw.begin() + tw_runs[i], tw.begin() + tw_runs[i + 1], tw.begin() + tw_runs[i + 2], longer);
        next.push_back(tw_runs[i]);
      }
      if (tw_runs.size() % 2 == 0) next.push_back(tw_runs[tw_runs.size() - 2]);
      next.push_back(tw_runs.back());
      tw_runs.swap(next);
    }
  }
  std::stable_sort(twi.begin(), twi.end(), [](const TW &a, const TW &b) { return a.w > b.w; });
  std::stable_sort(twi32.begin(), twi32.end(), [](const TW &a, const TW &b) { return a.w > b.w; });
  // track tiles plan by plan (each plan's profile stays hot in L2 while the
  // CTAs stream it), longest tiles first within a plan; where single tasks set
  // the time, longest first over all plans
  std::stable_sort(twp.begin(), twp.end(), [&](const TW &a, const TW &b) {
    return plan.even && a.t.q != b.t.q ? a.t.q < b.t.q : a.w > b.w;
  });
  Q->n_ptasks = (int64_t)twp.size();
  Q->n_tasks = (int64_t)tw.size();
  Q->n_itasks = (int64_t)twi.size();
  Q->n_itasks32 = (int64_t)twi32.size();
  Q->n_ipos32 = (int64_t)ipos32.size();
  Q->long_stride = std::max<int64_t>(1, packed ? 2 * n_long : n_long);
  Q->n_rtask_cap = Q->inter_may_flag ? rcap : 0;

  // --- launch geometry
  // two CTAs per SM need at most (228 KB - 2 x 1 KB reserved) / 2 of shared
  // memory each: drop to one profile buffer where two would not fit
  const size_t kTwoCtaSmem = 113 * 1024;
  Q->pbuf_count = inter_smem_bytes(Q->pbuf_bytes, 2, threads) <= kTwoCtaSmem ? 2 : 1;
  Q->ppbuf_count = inter_smem_bytes(Q->ppbuf_bytes, 2, threads) <= kTwoCtaSmem ? 2 : 1;
  Q->smem = inter_smem_bytes(Q->pbuf_bytes, Q->pbuf_count, threads);
  Q->psmem = inter_smem_bytes(Q->ppbuf_bytes, Q->ppbuf_count, threads);
  Q->ismem = intra_smem_bytes(Q->ipbuf_bytes);
  if (Q->smem > 200 * 1024 || Q->psmem > 200 * 1024 || (n_long && Q->ismem > 220 * 1024)) {
    delete Q;
    return fail(SW_EINVAL, "sw_queries_prepare: profile chunk too large for shared memory");
  }
  const int occ = cached_occupancy(0, R, packed ? kFormPacked : kFormInt32, gaps, threads, Q->smem);
  const int occ32 = cached_occupancy(0, R, kFormInt32, gaps, threads, Q->smem);
  const int occp = Q->n_ptasks ? cached_occupancy(0, R, kFormQPair, gaps, threads, Q->psmem) : 1;
  if (occ <= 0 || occ32 <= 0 || occp <= 0) {
    delete Q;
    return fail(SW_ECUDA, "sw_queries_prepare: cannot configure the inter-task kernel");
  }
  if (n_long) {
    cudaError_t ce = configure_intra(Ri, packed);
    if (ce == cudaSuccess && packed) ce = configure_intra(Ri, false);
    if (ce != cudaSuccess) {
      delete Q;
      return cuda_fail(ce, "sw_queries_prepare: cannot configure the intra-task kernel");
    }
  }
  Q->grid = (int)std::max<int64_t>(1, std::min<int64_t>(Q->n_tasks, (int64_t)sms * occ));
  Q->rgrid = std::max(1, sms * occ32);
  Q->pgrid = (int)std::max<int64_t>(1, std::min<int64_t>(Q->n_ptasks, (int64_t)sms * occp));
  Q->igrid = (int)std::max<int64_t>(1, std::min<int64_t>(std::max(Q->n_itasks, Q->n_itasks32), sms));
  const int gslots = std::max(std::max(Q->grid, Q->rgrid), Q->pgrid);
  Q->gbuf_stride = chunked ? (int32_t)round_up(std::max<int32_t>(16, max_short), 16) : 2;
  Q->igbuf_stride = ichunked ? (int32_t)round_up(std::max<int32_t>(16, max_long), 16) : 2;

  // --- device allocation (stream ordered)
  const int64_t nqm = std::max<int64_t>(n_queries, 1);
  const size_t b_qres = round_up(std::max<int64_t>(q_offsets[n_queries], 16), 256);
  const size_t b_sub = 512;
  const size_t b_qd = round_up(sizeof(QDesc) * nqm, 256);
  const size_t b_tasks = round_up(sizeof(Task) * std::max<int64_t>(Q->n_tasks, 1), 256);
  const size_t b_itasks = round_up(sizeof(Task) * std::max<int64_t>(Q->n_itasks, 1), 256);
  const size_t b_itasks32 = round_up(sizeof(Task) * std::max<int64_t>(Q->n_itasks32, 1), 256);
  const size_t b_ipos32 = round_up(4 * std::max<int64_t>((int64_t)ipos32.size(), 1), 256);
  const size_t b_rtasks = round_up(sizeof(Task) * std::max<int64_t>(Q->n_rtask_cap, 1), 256);
  const size_t b_qdp = round_up(sizeof(QDesc) * std::max<int64_t>(Q->npairs, 1), 256);
  const size_t b_track = round_up(sizeof(TrackChunk) * std::max<int64_t>((int64_t)Q->track.size(), 1), 256);
  const size_t b_ptasks = round_up(sizeof(Task) * std::max<int64_t>(Q->n_ptasks, 1), 256);
  const size_t b_prof = round_up(Q->prof_bytes, 256);
  const size_t b_gbuf = round_up((int64_t)gslots * warps * 8 * (int64_t)Q->gbuf_stride * 8, 256);
  // (two intra-task launches at once, packed and int32, each with its strips)
  const int ilaunches = Q->n_itasks && Q->n_itasks32 ? 2 : 1;
  const size_t b_igbuf = round_up((int64_t)ilaunches * Q->igrid * (int64_t)Q->igbuf_stride * 8, 256);
  const size_t b_words = round_up(4 * (12 + 2 * nqm), 256);  // zeroed words + 3 constants
  const size_t b_flag = Q->inter_may_flag ? round_up(4 * nqm * std::max<int64_t>(n, 1), 256) : 0;
  const size_t b_iflag = packed ? round_up(4 * nqm * Q->long_stride, 256) : 0;
  const size_t b_bjobs = round_up((int64_t)sizeof(BandJob) * std::max<int64_t>(Q->n_bjobs, 1), 256);
  const size_t b_bjobof = round_up(4 * std::max<int64_t>(Q->n_bands, 1), 256);
  const size_t b_btpos = round_up((int64_t)sizeof(int2) * std::max<int64_t>(Q->n_btargets, 1), 256);
  const size_t b_brings = Q->n_bjobs ? round_up(std::max<int64_t>(Q->band_ring_bytes, 8), 256) : 0;
  const bool tmode = Q->n_tjobs > 0;
  const size_t b_tjobs = tmode ? round_up((int64_t)sizeof(TrackJob) * Q->n_tjobs, 256) : 0;
  const size_t b_tgroups = tmode ? round_up(sizeof(TrackGroup) * tgroups.size(), 256) : 0;
  const size_t b_tlanes = tmode && !Q->tlanes_shared ? round_up((int64_t)sizeof(TrackLane) * Q->n_tlanes, 256) : 0;
  const size_t b_qt = tmode ? round_up(Q->qt_bytes, 256) : 0;
  const size_t b_qtoff = tmode ? round_up(8 * nqm, 256) : 0;
  const size_t b_qtnpad = tmode ? round_up(4 * nqm, 256) : 0;
  const size_t b_trings = tmode ? round_up(std::max<int64_t>(Q->track_ring_bytes, 8), 256) : 0;
  const size_t b_scores = round_up(score_bytes, 256);
  Q->bytes = b_scores + b_tjobs + b_tgroups + b_tlanes + b_qt + b_qtoff + b_qtnpad + b_trings + b_qres + b_sub + 2 * b_qd + b_tasks + b_itasks + b_itasks32 + b_ipos32 + b_rtasks + b_prof +
             b_gbuf + b_igbuf + b_words + b_flag + b_iflag + b_qdp + b_ptasks + b_track + b_bjobs + b_bjobof +
             b_btpos + b_brings;
  cudaMemPool_t pool = nullptr;
  cudaError_t e = batch_pool(&pool);
  if (e == cudaSuccess) e = cudaMallocFromPoolAsync(&Q->block, Q->bytes, pool, s);
  if (e != cudaSuccess) {
    delete Q;
    return cuda_fail(e, "sw_queries_prepare: device allocation");
  }
  uint8_t *p = (uint8_t *)Q->block;
  auto take = [&](size_t b) {
    uint8_t *r = p;
    p += b;
    return r;
  };
  // the regions the host fills come first, back to back, so that one copy
  // uploads them (with the zeroed status words and their constants)
  Q->d_qres = take(b_qres);
  Q->d_submat = (int8_t *)take(b_sub);
  Q->d_qd = (QDesc *)take(b_qd);
  Q->d_qdi = (QDesc *)take(b_qd);
  Q->d_tasks = (Task *)take(b_tasks);
  Q->d_itasks = (Task *)take(b_itasks);
  Q->d_itasks32 = (Task *)take(b_itasks32);
  Q->d_ipos32 = (int32_t *)take(b_ipos32);
  Q->d_qdp = (QDesc *)take(b_qdp);
  Q->d_track = (TrackChunk *)take(b_track);
  Q->d_ptasks = (Task *)take(b_ptasks);
  Q->d_bjobs = (BandJob *)take(b_bjobs);
  Q->d_bjob_of = (int32_t *)take(b_bjobof);
  Q->d_btpos = (int2 *)take(b_btpos);
  if (tmode) {
    Q->d_tjobs = (TrackJob *)take(b_tjobs);
    Q->d_tgroups = (TrackGroup *)take(b_tgroups);
    if (!Q->tlanes_shared) Q->d_tlanes = (TrackLane *)take(b_tlanes);
    Q->d_qt = take(b_qt);
    Q->d_qt_off = (int64_t *)take(b_qtoff);
    Q->d_qt_npad = (int32_t *)take(b_qtnpad);
  }
  Q->d_words = (int32_t *)take(b_words);
  Q->b_words = b_words;
  const size_t up_bytes = (size_t)(p - (uint8_t *)Q->block);
  // device-only regions
  if (b_scores) Q->d_scores = (int32_t *)take(b_scores);
  Q->b_scores = b_scores;
  if (tmode) Q->d_trings = (unsigned long long *)take(b_trings);
  Q->d_rtasks = (Task *)take(b_rtasks);
  Q->d_prof = take(b_prof);
  Q->d_gbuf = (uint2 *)take(b_gbuf);
  Q->d_igbuf = (uint2 *)take(b_igbuf);
  Q->d_flag_pos = Q->inter_may_flag ? (int32_t *)take(b_flag) : nullptr;
  Q->d_iflag_pos = packed ? (int32_t *)take(b_iflag) : nullptr;
  Q->d_brings = Q->n_bjobs ? (unsigned long long *)take(b_brings) : nullptr;
  Q->d_upos = const_cast<int32_t *>(db->d_ident) + s0;  // the short sequences, in sorted order
  Q->n_upos = n + 1 - s0;

  std::vector<Task> &tasks = scratch.tasks;
  tasks.resize((size_t)Q->n_tasks);
  std::vector<Task> itasks(Q->n_itasks), itasks32(Q->n_itasks32), ptasks(Q->n_ptasks);
  for (int64_t i = 0; i < Q->n_ptasks; ++i) ptasks[i] = twp[i].t;
  for (int64_t i = 0; i < Q->n_tasks; ++i) tasks[i] = tw[i].t;
  for (int64_t i = 0; i < Q->n_itasks; ++i) itasks[i] = twi[i].t;
  for (int64_t i = 0; i < Q->n_itasks32; ++i) itasks32[i] = twi32[i].t;
  const int32_t consts[4] = {(int32_t)Q->n_tasks, (int32_t)Q->n_itasks, (int32_t)Q->n_itasks32,
                             (int32_t)Q->n_ptasks};
  Q->h2d_bytes = q_offsets[n_queries] + 400 + 2 * (int64_t)sizeof(QDesc) * n_queries +
                 (int64_t)sizeof(QDesc) * Q->npairs + (int64_t)sizeof(TrackChunk) * (int64_t)Q->track.size() +
                 (int64_t)sizeof(Task) * (Q->n_tasks + Q->n_itasks + Q->n_itasks32 + Q->n_ptasks) +
                 4 * (int64_t)ipos32.size() + 16 + (int64_t)sizeof(BandJob) * Q->n_bjobs + 4 * Q->n_bands +
                 (int64_t)sizeof(int2) * Q->n_btargets + (int64_t)sizeof(TrackJob) * Q->n_tjobs +
                 (int64_t)(sizeof(TrackGroup) * tgroups.size()) +
                 (Q->tlanes_shared ? 0 : (int64_t)sizeof(TrackLane) * Q->n_tlanes) +
                 (tmode ? Q->qt_bytes + 12 * n_queries : 0);
  // stage the host tables at their offsets in the block (the rest zero:
  // padding and the status words) and upload them with one copy
  std::vector<uint8_t> &stage = scratch.stage;
  stage.assign(up_bytes, 0);
  auto put = [&](const void *dst, const void *src, size_t bytes) {
    if (bytes) memcpy(stage.data() + ((const uint8_t *)dst - (const uint8_t *)Q->block), src, bytes);
  };
  put(Q->d_qres, queries, (size_t)q_offsets[n_queries]);
  put(Q->d_submat, submat, 400);
  if (n_queries) put(Q->d_qd, Q->qd.data(), sizeof(QDesc) * n_queries);
  if (n_queries && n_long) put(Q->d_qdi, Q->qdi.data(), sizeof(QDesc) * n_queries);
  put(Q->d_tasks, tasks.data(), sizeof(Task) * Q->n_tasks);
  put(Q->d_itasks, itasks.data(), sizeof(Task) * Q->n_itasks);
  if (Q->n_itasks32) {
    put(Q->d_itasks32, itasks32.data(), sizeof(Task) * Q->n_itasks32);
    put(Q->d_ipos32, ipos32.data(), 4 * ipos32.size());
  }
  if (Q->npairs) {
    put(Q->d_qdp, Q->qdp.data(), sizeof(QDesc) * Q->npairs);
    put(Q->d_track, Q->track.data(), sizeof(TrackChunk) * Q->track.size());
    put(Q->d_ptasks, ptasks.data(), sizeof(Task) * Q->n_ptasks);
  }
  if (Q->n_bjobs) {
    put(Q->d_bjobs, bjobs.data(), sizeof(BandJob) * Q->n_bjobs);
    put(Q->d_bjob_of, bjob_of.data(), 4 * Q->n_bands);
    put(Q->d_btpos, btpos.data(), sizeof(int2) * Q->n_btargets);
  }
  if (tmode) {
    put(Q->d_tjobs, tjobs.data(), sizeof(TrackJob) * Q->n_tjobs);
    put(Q->d_tgroups, tgroups.data(), sizeof(TrackGroup) * tgroups.size());
    if (!Q->tlanes_shared) put(Q->d_tlanes, tlanes.data(), sizeof(TrackLane) * Q->n_tlanes);
    uint8_t *qtp = stage.data() + (Q->d_qt - (uint8_t *)Q->block);
    memset(qtp, kPadCode, (size_t)Q->qt_bytes);
    for (int64_t q = 0; q < n_queries; ++q)
      if (track_q[q] && qlen(q) > 0) memcpy(qtp + qt_off[q], queries + q_offsets[q], (size_t)qlen(q));
    put(Q->d_qt_off, qt_off.data(), 8 * n_queries);
    put(Q->d_qt_npad, qt_npad.data(), 4 * n_queries);
  }
  put(Q->d_words + Q->zero_words(), consts, sizeof consts);
  e = cudaMemcpyAsync(Q->block, stage.data(), up_bytes, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && ((n_long && !band_mode) || Q->n_bjobs)) {
    e = cudaStreamCreateWithFlags(&Q->side, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&Q->fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&Q->join, cudaEventDisableTiming);
    if (e == cudaSuccess && Q->n_itasks && Q->n_itasks32) {
      e = cudaStreamCreateWithFlags(&Q->side2, cudaStreamNonBlocking);
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&Q->join2, cudaEventDisableTiming);
    }
  }
  if (e == cudaSuccess && !one_search) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    free_queries(Q);
    return cuda_fail(e, "sw_queries_prepare: upload");
  }
  *out = Q;
  return SW_OK;
}

int sw_queries_prepare(const sw_db *db, const uint8_t *queries, const int64_t *q_offsets, int64_t n_queries,
                       const int8_t *submat, int32_t gap_open, int32_t gap_extend, int32_t mode,
                       const sw_options *opts, void *stream, sw_queries **out) {
  return prepare_queries(db, queries, q_offsets, n_queries, submat, gap_open, gap_extend, mode, opts, stream, false, 0,
                         out);
}

int sw_queries_free(sw_queries *q) {
  g_err.clear();
  free_queries(q);
  return SW_OK;
}

// fresh: the batch has just been uploaded (its words are zero)
static int search_prepared(const sw_db *db, const sw_queries *Q, int32_t *scores_dev, void *stream, bool fresh) {
  g_err.clear();
  if (!db || !Q) return fail(SW_EINVAL, "sw_search_prepared: null handle");
  if (Q->db != db) return fail(SW_EINVAL, "sw_search_prepared: query batch prepared for another database");
  if (Q->nq == 0 || db->n == 0) return SW_OK;
  if (!scores_dev) return fail(SW_EINVAL, "sw_search_prepared: null scores");
  cudaStream_t s = (cudaStream_t)stream;
  const bool packed = Q->mode == SW_MODE_PACKED;
  const int threads = Q->threads;
  const int nq = (int)Q->nq;
  int32_t *w = Q->d_words;

  if (!fresh) SW_CUDA(cudaMemsetAsync(w, 0, 4 * Q->zero_words(), s), "memset");
  std::unique_ptr<StageRange> stage(new StageRange("swgb: query profiles"));
  if (Q->n_solo)
    SW_CUDA(launch_build_profiles(Q->d_qres, Q->d_qd, nq, Q->d_submat, Q->sc.pad, Q->d_prof, s), "profile kernel");
  if (Q->npairs)
    SW_CUDA(launch_build_track_profiles(Q->d_qres, Q->d_qd, Q->d_qdp, Q->d_track, (int32_t)Q->track.size(),
                                        Q->d_submat, Q->sc.pad, Q->d_prof, s),
            "track profile kernel");
  if (Q->n_itasks || Q->n_itasks32)
    SW_CUDA(launch_build_profiles(Q->d_qres, Q->d_qdi, nq, Q->d_submat, Q->sc.pad, Q->d_prof, s),
            "profile kernel");

  stage.reset(new StageRange("swgb: dynamic programming"));
  // band-stream and transposed jobs add their scores with atomicMax: every score starts at 0
  const bool small = Q->n_bjobs || Q->n_tjobs;
  // (the block's own scores lie before the row tracks' rings: one memset for both)
  const bool with_rings = Q->n_tjobs && scores_dev == Q->d_scores;
  if (small)
    SW_CUDA(cudaMemsetAsync(scores_dev, 0,
                            with_rings ? Q->b_scores + (size_t)Q->track_ring_bytes
                                       : 4 * (size_t)Q->nq * (size_t)db->n,
                            s),
            "memset");
  const bool band_timing = Q->timing && small;
  if (band_timing) SW_CUDA(cudaEventRecord(Q->ev0, s), "event");

  InterArgs a{};
  a.db = db->view;
  a.unit_pos = db->d_ident;
  a.n_unit_pos = db->n + 1;
  a.prof = Q->d_prof;
  a.prof_bytes = Q->prof_bytes;
  a.out = scores_dev;
  a.out_stride = db->n;
  a.out_size = Q->nq * db->n;
  a.sc = Q->sc;
  a.status = w + 2;

  // long database units: intra-task kernel on the side stream, concurrently;
  // int32 matrices (those that could saturate 16 bits) on a third stream
  // when packed ones exist too, so that neither waits for the other.  In
  // small batches the band-stream jobs take the side stream instead.
  if (Q->side) {
    SW_CUDA(cudaEventRecord(Q->fork, s), "event");
    SW_CUDA(cudaStreamWaitEvent(Q->side, Q->fork, 0), "event");
    if (Q->side2) SW_CUDA(cudaStreamWaitEvent(Q->side2, Q->fork, 0), "event");
    if (Q->n_bjobs) {
      SW_CUDA(cudaMemsetAsync(Q->d_brings, 0, (size_t)Q->band_ring_bytes, Q->side), "memset");
      BandArgs ba{};
      ba.db = db->view;
      ba.tpos = Q->d_btpos;
      ba.jobs = Q->d_bjobs;
      ba.band_job = Q->d_bjob_of;
      ba.nbands = (int32_t)Q->n_bands;
      ba.band_counter = w + 7;
      ba.qres = Q->d_qres;
      ba.qd = Q->d_qd;
      ba.submat = Q->d_submat;
      ba.rings = Q->d_brings;
      ba.out = scores_dev;
      ba.out_stride = db->n;
      ba.out_size = Q->nq * db->n;
      ba.ring_entries = Q->band_ring_bytes / 8;
      ba.n_tpos = Q->n_btargets;
      ba.sc = Q->sc;
      ba.status = w + 2;
      SW_CUDA(launch_band(ba, Q->bR, Q->bgrid, Q->bone, Q->side), "band-stream kernel");
    }
    InterArgs b = a;
    b.qd = Q->d_qdi;
    b.pbuf_bytes = Q->ipbuf_bytes;
    b.gbuf = Q->d_igbuf;
    b.gbuf_stride = Q->igbuf_stride;
    b.flag_count = w + 8 + nq;
    b.flag_pos = Q->d_iflag_pos;
    b.flag_stride = Q->long_stride;
    b.flag_size = Q->nq * Q->long_stride;
    if (Q->n_itasks) {  // packed units that cannot saturate
      b.tasks = Q->d_itasks;
      b.n_tasks = w + Q->zero_words() + 1;
      b.task_counter = w + 4;
      SW_CUDA(launch_intra(b, Q->Ri, true, Q->igrid, Q->ismem, Q->side), "intra-task kernel");
    }
    if (Q->n_itasks32) {  // single sequences in int32
      b.unit_pos = Q->d_ipos32;
      b.n_unit_pos = Q->n_ipos32;
      b.tasks = Q->d_itasks32;
      b.n_tasks = w + Q->zero_words() + 2;
      b.task_counter = w + 5;
      cudaStream_t st = Q->side;
      if (Q->side2) {
        st = Q->side2;
        b.gbuf = Q->d_igbuf + (size_t)Q->igrid * Q->igbuf_stride;
      }
      SW_CUDA(launch_intra(b, Q->Ri, false, Q->igrid, Q->ismem, st), "intra-task kernel (int32)");
      if (Q->side2) SW_CUDA(cudaEventRecord(Q->join2, Q->side2), "event");
    }
    SW_CUDA(cudaEventRecord(Q->join, Q->side), "event");
  }

  if (Q->n_tjobs) {  // transposed jobs, on the caller's stream beside the band-stream ones
    if (!with_rings) SW_CUDA(cudaMemsetAsync(Q->d_trings, 0, (size_t)Q->track_ring_bytes, s), "memset");
    TrackArgs ta{};
    ta.db = db->view;
    ta.lanes = Q->d_tlanes;
    ta.jobs = Q->d_tjobs;
    ta.groups = Q->d_tgroups;
    ta.n_groups = Q->n_tgroups;
    ta.nbands = (int32_t)Q->n_tbands;
    ta.band_counter = w + 1;
    ta.qt = Q->d_qt;
    ta.qt_off = Q->d_qt_off;
    ta.qt_npad = Q->d_qt_npad;
    ta.submat = Q->d_submat;
    ta.rings = Q->d_trings;
    ta.out = scores_dev;
    ta.out_stride = db->n;
    ta.sc = Q->sc;
    ta.status = w + 2;
    ta.n_lanes = Q->n_tlanes;
    ta.ring_entries = Q->track_ring_bytes / 8;
    ta.out_size = Q->nq * db->n;
    ta.qt_bytes = Q->qt_bytes;
    SW_CUDA(launch_track(ta, Q->tR, Q->tgrid, s), "band-stream kernel (transposed jobs)");
  }
  if (Q->timing && !band_timing && (Q->n_tasks || Q->n_ptasks)) SW_CUDA(cudaEventRecord(Q->ev0, s), "event");
  if (Q->n_ptasks) {  // query pairs, one short database sequence per chain
    InterArgs p = a;
    p.qd = Q->d_qdp;
    p.track = Q->d_track;
    p.unit_pos = Q->d_upos;
    p.n_unit_pos = Q->n_upos;
    p.tasks = Q->d_ptasks;
    p.n_tasks = w + Q->zero_words() + 3;
    p.task_counter = w + 6;
    p.pbuf_bytes = Q->ppbuf_bytes;
    p.pbuf_count = Q->ppbuf_count;
    p.gbuf = Q->d_gbuf;
    p.gbuf_stride = Q->gbuf_stride;
    p.flag_count = nullptr;
    p.flag_pos = nullptr;
    p.flag_stride = 0;
    SW_CUDA(launch_inter(p, Q->R, kFormQPair, Q->pgrid, threads, Q->psmem, s), "inter-task kernel (query pairs)");
  }
  if (Q->n_tasks) {
    a.qd = Q->d_qd;
    a.tasks = Q->d_tasks;
    a.n_tasks = w + Q->zero_words();
    a.task_counter = w + 0;
    a.pbuf_bytes = Q->pbuf_bytes;
    a.pbuf_count = Q->pbuf_count;
    a.gbuf = Q->d_gbuf;
    a.gbuf_stride = Q->gbuf_stride;
    a.flag_count = w + 8;
    a.flag_pos = Q->d_flag_pos;
    a.flag_stride = db->n;
    a.flag_size = Q->inter_may_flag ? Q->nq * db->n : 0;
    SW_CUDA(launch_inter(a, Q->R, packed ? kFormPacked : kFormInt32, Q->grid, threads, Q->smem, s), "inter-task kernel");
  }
  if (Q->timing && !band_timing && (Q->n_tasks || Q->n_ptasks)) {
    SW_CUDA(cudaEventRecord(Q->ev1, s), "event");
    const_cast<sw_queries *>(Q)->timed = true;
  }
  if (Q->n_tasks) {
    if (Q->inter_may_flag) {
      stage.reset(new StageRange("swgb: int32 rescue"));
      SW_CUDA(launch_rescue_tasks(w + 8, Q->d_qd, nq, db->n, threads / 32, 0, Q->d_rtasks, w + 3, w + 1, s),
              "rescue task kernel");
      InterArgs r = a;
      r.unit_pos = Q->d_flag_pos;
      r.n_unit_pos = Q->nq * db->n;
      r.tasks = Q->d_rtasks;
      r.n_tasks = w + 3;
      r.task_counter = w + 1;
      r.flag_count = nullptr;
      r.flag_pos = nullptr;
      SW_CUDA(launch_inter(r, Q->R, kFormInt32, Q->rgrid, threads, Q->smem, s), "inter-task rescue kernel");
    }
  }
  if (Q->side) SW_CUDA(cudaStreamWaitEvent(s, Q->join, 0), "event");
  if (Q->side2) SW_CUDA(cudaStreamWaitEvent(s, Q->join2, 0), "event");
  if (band_timing) {
    SW_CUDA(cudaEventRecord(Q->ev1, s), "event");
    const_cast<sw_queries *>(Q)->timed = true;
  }
  return SW_OK;
}

int sw_search_prepared(const sw_db *db, const sw_queries *Q, int32_t *scores_dev, void *stream) {
  return search_prepared(db, Q, scores_dev, stream, false);
}

int sw_search_graph(const sw_db *db, sw_queries *Q, int32_t *scores_dev, void *stream) {
  g_err.clear();
  if (!db || !Q) return fail(SW_EINVAL, "sw_search_graph: null handle");
  if (!stream) return fail(SW_EINVAL, "sw_search_graph: stream capture needs a non-default stream");
  if (Q->nq == 0 || db->n == 0) return SW_OK;
  cudaStream_t s = (cudaStream_t)stream;
  if (!Q->gexec || Q->gdb != db || Q->gscores != scores_dev) {
    if (Q->gexec) {
      cudaGraphExecDestroy(Q->gexec);
      Q->gexec = nullptr;
    }
    SW_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal), "cudaStreamBeginCapture");
    const bool timing = Q->timing;
    Q->timing = false;
    int rc = sw_search_prepared(db, Q, scores_dev, stream);
    Q->timing = timing;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(s, &graph);
    if (rc != SW_OK) {
      if (graph) cudaGraphDestroy(graph);
      return rc;
    }
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
    e = cudaGraphInstantiate(&Q->gexec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
      Q->gexec = nullptr;
      return cuda_fail(e, "cudaGraphInstantiate");
    }
    Q->gdb = db;
    Q->gscores = scores_dev;
  }
  SW_CUDA(cudaGraphLaunch(Q->gexec, s), "cudaGraphLaunch");
  return SW_OK;
}

// what the words of a finished search say
static int words_status(const sw_queries *Q, const int32_t *w, int64_t *rescued) {
  int64_t inter_flags = 0, intra_flags = 0;
  for (int64_t q = 0; q < Q->nq; ++q) {
    inter_flags += w[8 + q];
    intra_flags += w[8 + Q->nq + q];
  }
  if (rescued) *rescued = inter_flags;
  if (w[2] == SW_ETIMEOUT) return fail(SW_ETIMEOUT, "a bounded device wait expired");
  if (w[2] == kStatusSaturated) return fail(SW_ECUDA, "internal error: a query-pair lane passed its bound");
  if (w[2] == kStatusBounds) return fail(SW_ECUDA, "internal error: an index left its buffer (checked build)");
  if (intra_flags) return fail(SW_ECUDA, "internal error: a packed intra-task lane passed its bound");
  return SW_OK;
}

int sw_queries_status(const sw_queries *Q, void *stream, int64_t *rescued) {
  g_err.clear();
  if (!Q) return fail(SW_EINVAL, "sw_queries_status: null handle");
  cudaStream_t s = (cudaStream_t)stream;
  std::vector<int32_t> w(Q->zero_words());
  SW_CUDA(cudaMemcpyAsync(w.data(), Q->d_words, 4 * w.size(), cudaMemcpyDeviceToHost, s), "status read");
  SW_CUDA(cudaStreamSynchronize(s), "status sync");
  return words_status(Q, w.data(), rescued);
}

int sw_queries_set_timing(sw_queries *q, int32_t enable) {
  g_err.clear();
  if (!q) return fail(SW_EINVAL, "sw_queries_set_timing: null handle");
  if (enable && !q->ev0) {
    SW_CUDA(cudaEventCreate(&q->ev0), "cudaEventCreate");
    SW_CUDA(cudaEventCreate(&q->ev1), "cudaEventCreate");
  }
  q->timing = enable != 0;
  q->timed = false;
  return SW_OK;
}

int sw_queries_kernel_ms(const sw_queries *q, void *stream, float *ms) {
  g_err.clear();
  if (!q || !ms) return fail(SW_EINVAL, "sw_queries_kernel_ms: null argument");
  if (!q->timing || !q->timed) return fail(SW_EINVAL, "sw_queries_kernel_ms: no timed search");
  SW_CUDA(cudaStreamSynchronize((cudaStream_t)stream), "sync");
  SW_CUDA(cudaEventElapsedTime(ms, q->ev0, q->ev1), "cudaEventElapsedTime");
  return SW_OK;
}

int sw_queries_info(const sw_queries *q, int64_t *h2d_bytes, int64_t *device_bytes, int64_t *n_tasks,
                    int64_t *launches) {
  g_err.clear();
  if (!q) return fail(SW_EINVAL, "sw_queries_info: null handle");
  if (launches) {
    int64_t k = 0;
    if (q->nq > 0 && q->db->n > 0) {
      k = (q->n_solo ? 1 : 0) + (q->npairs ? 1 : 0) + ((q->n_itasks || q->n_itasks32) ? 1 : 0);  // profile builds
      k += (q->n_tasks ? 1 : 0) + (q->n_ptasks ? 1 : 0);  // inter-task kernels
      k += (q->n_tasks && q->inter_may_flag) ? 2 : 0;     // rescue tasks + int32 rescue
      k += (q->n_itasks ? 1 : 0) + (q->n_itasks32 ? 1 : 0);
      k += q->n_bjobs ? 1 : 0;  // band-stream kernel
      k += q->n_tjobs ? 1 : 0;  // transposed jobs
    }
    *launches = k;
  }
  if (h2d_bytes) *h2d_bytes = q->h2d_bytes;
  if (device_bytes) *device_bytes = (int64_t)q->bytes;
  if (n_tasks) *n_tasks = q->n_tasks + q->n_itasks + q->n_itasks32 + q->n_ptasks;
  return SW_OK;
}

int sw_search(const sw_db *db, const uint8_t *queries, const int64_t *q_offsets, int64_t n_queries,
              const int8_t *submat, int32_t gap_open, int32_t gap_extend, int32_t mode, int32_t *scores_out,
              void *stream) {
  g_err.clear();
  if (!db) return fail(SW_EINVAL, "sw_search: null database");
  if (n_queries > 0 && db->n > 0 && !scores_out) return fail(SW_EINVAL, "sw_search: null scores");
  const int64_t count = n_queries > 0 && n_queries <= std::numeric_limits<int32_t>::max() ? n_queries * db->n : 0;
  const bool host = count > 0 && !is_device_ptr(scores_out);
  sw_queries *Q = nullptr;
  int rc = prepare_queries(db, queries, q_offsets, n_queries, submat, gap_open, gap_extend, mode, nullptr, stream, true,
                           host ? 4 * count : 0, &Q);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  if (count > 0) rc = search_prepared(db, Q, host ? Q->d_scores : scores_out, stream, true);
  // The words (status, flag counts) and, up to 64 KB, the scores after them
  // come back in one copy: a copy to pageable memory waits for the device and
  // then for its own staging, 11 us each for a search of 130 us.
  const size_t words = 4 * (size_t)Q->zero_words();
  const bool together = host && 4 * count <= kSearchStage;
  std::vector<uint8_t> &back = plan_scratch().back;
  back.resize(together ? Q->b_words + 4 * (size_t)count : words);
  if (rc == SW_OK && host && !together) {
    cudaError_t e = cudaMemcpyAsync(scores_out, Q->d_scores, 4 * count, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) rc = cuda_fail(e, "sw_search: score copy");
  }
  if (rc == SW_OK) {
    cudaError_t e = cudaMemcpyAsync(back.data(), Q->d_words, back.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) rc = cuda_fail(e, "sw_search: results");
  }
  if (rc == SW_OK) {
    if (together) memcpy(scores_out, back.data() + Q->b_words, 4 * (size_t)count);
    rc = words_status(Q, (const int32_t *)back.data(), nullptr);
  }
  std::string keep = g_err;
  free_queries(Q);
  g_err = keep;
  return rc;
}

}  // extern "C"
