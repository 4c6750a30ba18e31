// Traceback of selected hits: one optimal local alignment per (query,
// database sequence) pair, the alignment output the paper's score-only search
// leaves out (Sec. 2.2: H records the best score of an alignment ending at
// each cell; the alignment itself is the path that produced it).
//
// Fill: every hit's query rows are cut into bands of 32 lanes x 8 rows, one
// warp each, which sweep the target's columns as a pipeline (band_core.cuh):
// the bottom row of a band reaches the next one through the part of the
// direction buffer that the next band writes later (see below).  The bands of all hits are handed out by one counter, the longest
// hits first, so a long hit is spread over as many SMs as it has bands and
// short ones fill in.  (One CTA of 8 warps per hit, 512-row chunks in turn:
// 19.5 ms for 200 hits of 144 to 5,478 residues, the ten longest alone on
// their SMs for most of it.)  Per cell the fill records four bits of
// provenance: whether E and F extend a gap (else they open one), and whether H
// is not the diagonal's, not E's value; each is the sign of a difference,
// shifted into one of four bytes by a funnel shift (compared and selected per
// cell, 29 instructions instead of 14: 910 cycles per step of 8 rows).  The
// zero floor needs no bit: the walk knows the score that is left.  A lane's 8
// rows of a column are one word, and a step's words of the 32 lanes (32
// columns of the wavefront) are stored side by side: one 128-byte line per
// step.  The 16 boundary entries of a block of columns take the line of the
// block's first step in the band that reads them: it has read them when it
// gets to that step, and stores its words over them.  (So the boundaries need no memory of
// their own: rings would add 1/16.)  The fill also keeps the first cell (row-major) holding the best
// score.
//
// Walk: one warp per hit follows the bits back from that cell to a cell whose
// H is 0, ties in the order floor, diagonal, E, F, through tiles of 144 steps x
// 16 lanes staged in shared memory; up to 32 cells of a diagonal run at a time,
// their scores summed by shuffles.  (One thread per hit on the words in global
// memory: a dependent load of ~0.8 us per cell of the path.)
#include <algorithm>

#include "band_core.cuh"

namespace swgb {
namespace {

constexpr int kTraceR = 8;  // rows per lane
constexpr int kTraceRows = 32 * kTraceR;
constexpr int kTraceThreads = 128;
constexpr int kTraceProfBytes = kProfRows * 32 * kTraceR;
constexpr int kTraceWarpBytes = kTraceProfBytes + 2 * kResChunk + 2 * kColBlock * 8;  // profile, residues, slots

constexpr int kBlockWords = kColBlock * 32;  // direction words of a block of steps

// Clears the lines that hold boundary entries first (an entry is there when
// its tag bit is set) and the counter and status words.
__global__ void trace_clear_kernel(const TraceArgs a) {
  const int64_t n = a.dir_words / kBlockWords * 8;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    reinterpret_cast<uint4 *>(a.dirs + i / 8 * kBlockWords)[i % 8] = make_uint4(0u, 0u, 0u, 0u);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *a.band_counter = 0;
    *a.status = 0;
  }
}

__device__ __forceinline__ bool earlier(int32_t s, int32_t i, int32_t j, int32_t bs, int32_t bi, int32_t bj) {
  // better score, or the same score at a cell earlier in row-major order
  return s > bs || (s == bs && (i < bi || (i == bi && j < bj)));
}

// bit r of a flag byte is row 7 - r's
constexpr int kExtE = 0, kExtF = 8, kNotDiag = 16, kNotE = 24;
__device__ __forceinline__ uint32_t trace_flag(uint32_t w, int flag, int r) { return (w >> (flag + 7 - r)) & 1u; }

// A lane's 8 rows, a column per step (the lane type of band_sweep).  Passes H
// and F of its last row; the row below forms its own F and the bit of it.
struct TraceLane {
  static constexpr int R = kTraceR;
  int32_t Hl[R], El[R];        // H and E of each row at the previous column
  int32_t outH[1], outF[1];    // of the last row
  int32_t hdiag;
  int32_t bs, bi, bj;          // best score and its cell (1-based)
  int32_t top;                 // the warp's best score, at least 1
  int32_t col, row0, n;        // this lane's column (0-based), its first row (0-based); the target's length
  uint32_t real_rows;          // bit r: row0 + r is a row of the query
  uint32_t *dir;               // this step's word
  const uint32_t *dirs;        // the direction buffer and its words (checked build)
  int64_t dir_words;
  int32_t *status;

  template <class Prof>
  __device__ __forceinline__ void step(const Prof &p, const int32_t (&inH)[1], const int32_t (&inF)[1],
                                       const Consts &cs) {
    int32_t x[R];
#pragma unroll
    for (int r = R - 1; r >= 0; --r) x[r] = p.add(0, r, r > 0 ? Hl[r - 1] : hdiag);
    int32_t f_open = inH[0] - cs.go, f = inF[0], best = 0;
    uint32_t xe = 0u, xf = 0u, nd = 0u, ne = 0u;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int32_t e_open = Hl[r] - cs.go;
      const int32_t e = max(El[r] - cs.ge, e_open);
      f = max(f - cs.ge, f_open);
      const int32_t h = __vimax3_s32_relu(x[r], e, f);
      xe = __funnelshift_l((uint32_t)(e_open - e), xe, 1);  // 1: E extends (opening is less)
      xf = __funnelshift_l((uint32_t)(f_open - f), xf, 1);
      nd = __funnelshift_l((uint32_t)(x[r] - h), nd, 1);
      ne = __funnelshift_l((uint32_t)(e - h), ne, 1);
      if (r & 1) best = __vimax3_s32(best, Hl[r - 1], h);
      Hl[r] = h;
      El[r] = e;
      f_open = h - cs.go;
    }
    // the best cell: only a step whose maximum reaches the warp's best so far
    // needs the rows.  (Cells past the query or the target are left out: they
    // add no positive score, so a real cell before them holds as much.)
    // (Against each lane's own best, row by row: 0.94 against 0.88 ms a call for
    // 200 hits of 100 to 1,000 residues.)
    const bool reach = col >= 0 && col < n && best >= top;
    if (__any_sync(0xffffffffu, reach)) {
      uint32_t eq = 0u;
#pragma unroll
      for (int r = 0; r < R; ++r) eq |= Hl[r] == best ? 1u << r : 0u;
      eq &= real_rows;
      const int32_t i = row0 + __ffs(eq);
      if (reach && eq && earlier(best, i, col + 1, bs, bi, bj)) {
        bs = best;
        bi = i;
        bj = col + 1;
      }
      top = max(1, __reduce_max_sync(0xffffffffu, bs));
    }
    hdiag = inH[0];
    outH[0] = Hl[R - 1];
    outF[0] = f;
    const uint32_t word = prmt(prmt(xe, xf, 0x0040u), prmt(nd, ne, 0x0040u), 0x5410u);
    if (in_range(dir - dirs, dir_words, status)) *dir = word;
    dir += 32;
    ++col;
  }
};

__global__ void __launch_bounds__(kTraceThreads, 4) trace_fill_kernel(const TraceArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint8_t *prof = smem + kScoreBytes + (size_t)warp * kTraceWarpBytes;
  uint8_t *io = prof + kTraceProfBytes;
  uint2 *rgb = reinterpret_cast<uint2 *>(io + 2 * kResChunk);
  build_scores<false>(smem, a.submat, a.sc.pad);
  __syncthreads();
  const Consts cs = make_consts(a.sc);
  for (;;) {
    int g = 0;
    if (lane == 0) {
      const int32_t gave_up = *(const volatile int32_t *)a.status;
      g = atomicAdd(a.band_counter, 1);
      if (gave_up) g = a.nbands;  // (a wait has expired: the entries of the bands below it never come)
    }
    g = __shfl_sync(0xffffffffu, g, 0);
    if (g >= a.nbands) break;
    const TraceHit hit = a.hits[a.band_hit[g]];
    const int b = g - hit.band0;
    __syncwarp();  // (the band before this one has read its profile, residues and slots)
    ResidueStage<1> rs{io, a.tres + hit.toff, nullptr, hit.npad, 0, lane, a.tres, a.tres_bytes, a.status};
    rs.stage(0);
    const int row0 = b * kTraceRows + lane * kTraceR;
    uint32_t code[kTraceR / 4];
#pragma unroll
    for (int i = 0; i < kTraceR / 4; ++i) {
      uint32_t v = 0u;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int row = row0 + 4 * i + j;
        v |= (uint32_t)(row < hit.m ? a.qres[hit.qoff + row] : (uint8_t)kPadCode) << (8 * j);
      }
      code[i] = v;
    }
    profile_from_scores<kTraceR>(prof + lane * kTraceR, 32 * kTraceR, smem, code);
    clear_slots(rgb, lane, 0u);
    const int64_t band_words = (int64_t)(hit.npad + 32) * 32;
    uint32_t *dirs = a.dirs + hit.dir0 + b * band_words;
    unsigned long long *ring = reinterpret_cast<unsigned long long *>(dirs);
    OnceRing<kBlockWords / 2> x{ring, ring + band_words / 2, rgb, lane,
                                reinterpret_cast<const unsigned long long *>(a.dirs), a.dir_words / 2, a.status, b > 0,
                                b + 1 < hit.nb};
    x.budget = a.wait_cycles;
    TraceLane ln{};
    ln.row0 = row0;
    ln.n = hit.n;
    ln.top = 1;
    ln.real_rows = (1u << min(max(hit.m - row0, 0), kTraceR)) - 1u;
    ln.col = -lane;
    ln.dir = dirs + lane;
    ln.dirs = a.dirs;
    ln.dir_words = a.dir_words;
    ln.status = a.status;
    const bool ok = band_sweep<kFormInt32, 1, 4, false, IntProfile<kTraceR, 1>>(
        ln, rs, x, rgb, prof + lane * kTraceR, 32 * kTraceR, lane, hit.npad / kColBlock, -1, 0, cs, a.status);
    cp_async_wait<0>();
    int32_t bs = ln.bs, bi = ln.bi, bj = ln.bj;
    for (int d = 16; d > 0; d >>= 1) {
      const int32_t os = __shfl_xor_sync(0xffffffffu, bs, d);
      const int32_t oi = __shfl_xor_sync(0xffffffffu, bi, d);
      const int32_t oj = __shfl_xor_sync(0xffffffffu, bj, d);
      if (earlier(os, oi, oj, bs, bi, bj)) {
        bs = os;
        bi = oi;
        bj = oj;
      }
    }
    if (lane == 0) a.best[g] = make_int4(bs, bi, bj, 0);
    if (!ok) break;
  }
}

// Walk back from the best cell: in H, a score of 0 left ends the alignment,
// the diagonal aligns Q[i] with D[j] ('M'), E and F switch state; in E a
// target residue faces a gap ('D'), in F a query residue ('I'); the extension
// bit keeps the state, else the walk returns to H.  Operations are written
// from the end of the hit's part of the buffer to the front, then moved to its
// beginning.
// Steps x lanes of a tile: a diagonal crosses 16 lanes' rows in 144 steps, so a
// tile serves four runs of 32 cells and its load's latency is paid once for
// them (64 x 8: two runs, 302 against 265 us for 200 hits).
constexpr int kWalkSteps = 144, kWalkLanes = 16;
__global__ void __launch_bounds__(128) trace_walk_kernel(const TraceArgs a) {
  if (*a.status != 0) return;  // the fill gave up: bands not taken have left no best cell
  __shared__ __align__(16) uint32_t tiles[4][kWalkSteps * kWalkLanes];
  __shared__ int8_t sm[kAlphabet * kAlphabet];
  for (int x = threadIdx.x; x < kAlphabet * kAlphabet; x += blockDim.x) sm[x] = a.submat[x];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  uint32_t *tile = tiles[threadIdx.x >> 5];
  const int h = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (h >= a.nhits) return;
  const TraceHit hit = a.hits[h];
  int32_t bs = 0, bi = 0, bj = 0;
  for (int b = lane; b < hit.nb; b += 32) {
    const int4 v = a.best[hit.band0 + b];
    if (earlier(v.x, v.y, v.z, bs, bi, bj)) {
      bs = v.x;
      bi = v.y;
      bj = v.z;
    }
  }
  for (int d = 16; d > 0; d >>= 1) {
    const int32_t os = __shfl_xor_sync(0xffffffffu, bs, d);
    const int32_t oi = __shfl_xor_sync(0xffffffffu, bi, d);
    const int32_t oj = __shfl_xor_sync(0xffffffffu, bj, d);
    if (earlier(os, oi, oj, bs, bi, bj)) {
      bs = os;
      bi = oi;
      bj = oj;
    }
  }
  // (every index below follows from the cell)
  if (!in_range(bi, (int64_t)hit.m + 1, a.status) || !in_range(bj, (int64_t)hit.n + 1, a.status)) return;
  const uint32_t *dirs = a.dirs + hit.dir0;
  const uint8_t *q = a.qres + hit.qoff, *t = a.tres + hit.toff;
  const int steps = hit.npad + 32;
  uint8_t *ops = a.ops + hit.ops_off;
  const int64_t cap = (int64_t)hit.m + hit.n;
  int i = bi, j = bj, state = 0, left = bs;  // left: the value of H (of E, F in their states) at the cell
  int64_t k = 0;
  int tb = -1, tg = -1, t_lo = 0, t_hi = -1;  // the tile: band, group of lanes, steps
  while (i > 0 && j > 0 && k < cap && (state != 0 || left > 0)) {
    {
      const int b = (i - 1) / kTraceRows, l = (i - 1) % kTraceRows / kTraceR, s = j - 1 + l;
      if (b != tb || l / kWalkLanes != tg || s < t_lo || s > t_hi) {
        tb = b;
        tg = l / kWalkLanes;
        t_hi = s;
        t_lo = max(0, s - (kWalkSteps - 1));
        __syncwarp();
        // (four 16-byte loads per step, all in flight at once)
        static_assert(kWalkSteps * kWalkLanes % 128 == 0, "whole loads");
        constexpr int kLoads = kWalkSteps * kWalkLanes / 4 / 32;
        uint4 v[kLoads];
#pragma unroll
        for (int p = 0; p < kLoads; ++p) {
          const int e = p * 32 + lane, x = min(t_lo + e / (kWalkLanes / 4), t_hi);
          v[p] = __ldg(reinterpret_cast<const uint4 *>(dirs + ((int64_t)b * steps + x) * 32 + tg * kWalkLanes) +
                       e % (kWalkLanes / 4));
        }
#pragma unroll
        for (int p = 0; p < kLoads; ++p) reinterpret_cast<uint4 *>(tile)[p * 32 + lane] = v[p];
        __syncwarp();
      }
    }
    // this lane's cell of the diagonal (the other states use lane 0's)
    const int ci = i - lane, cj = j - lane;
    uint32_t w = 0u;
    int r = 0;
    bool in_tile = false;
    if (ci > 0 && cj > 0) {
      const int row = (ci - 1) % kTraceRows, l = row / kTraceR, s = cj - 1 + l;
      r = row % kTraceR;
      in_tile = (ci - 1) / kTraceRows == tb && l / kWalkLanes == tg && s >= t_lo && s <= t_hi;
      if (in_tile) w = tile[(s - t_lo) * kWalkLanes + l % kWalkLanes];
    }
    if (state == 0) {
      const bool diag = in_tile && !trace_flag(w, kNotDiag, r);
      const int32_t score = diag ? sm[q[ci - 1] * kAlphabet + t[cj - 1]] : 0;
      int32_t sum = score;  // inclusive, then exclusive
      for (int d = 1; d < 32; d <<= 1) {
        const int32_t o = __shfl_up_sync(0xffffffffu, sum, d);
        if (lane >= d) sum += o;
      }
      const int32_t here = left - (sum - score);  // H at this lane's cell
      const uint32_t stop = __ballot_sync(0xffffffffu, !diag || here == 0);
      const int run = stop ? __ffs(stop) - 1 : 32;
      if (lane < run) ops[cap - 1 - k - lane] = 'M';
      left = run < 32 ? __shfl_sync(0xffffffffu, here, run) : left - __shfl_sync(0xffffffffu, sum, 31);
      // the cell that ends the run: the floor, another tile's (or none), E or F
      const uint32_t end = run < 32 ? __shfl_sync(0xffffffffu, w, run) : 0u;
      const int end_r = __shfl_sync(0xffffffffu, r, run & 31);
      const bool end_in = run < 32 && __shfl_sync(0xffffffffu, (int)in_tile, run & 31) != 0;
      i -= run;
      j -= run;
      k += run;
      if (end_in && left > 0) state = trace_flag(end, kNotE, end_r) ? 2 : 1;
    } else {
      const uint32_t w0 = __shfl_sync(0xffffffffu, w, 0);
      const int r0 = __shfl_sync(0xffffffffu, r, 0);
      const bool ext = trace_flag(w0, state == 1 ? kExtE : kExtF, r0) != 0;
      if (lane == 0) ops[cap - 1 - k] = state == 1 ? 'D' : 'I';
      ++k;
      left += ext ? a.sc.ge : a.sc.go;
      if (state == 1) --j;
      else --i;
      if (!ext) state = 0;
    }
  }
  // move the operations to the front (the source lies behind the destination:
  // a round's stores touch nothing that a later round loads)
  __syncwarp();
  const int64_t shift = cap - k;
  if (shift > 0)
    for (int64_t base = 0; base < k; base += 256) {
      uint8_t v[8];
#pragma unroll
      for (int x = 0; x < 8; ++x) v[x] = base + 32 * x + lane < k ? ops[shift + base + 32 * x + lane] : 0;
      __syncwarp();
#pragma unroll
      for (int x = 0; x < 8; ++x)
        if (base + 32 * x + lane < k) ops[base + 32 * x + lane] = v[x];
      __syncwarp();
    }
  if (lane == 0) {
    TraceResult res{};
    res.score = bs;
    res.end_i = bs > 0 ? bi : 0;
    res.end_j = bs > 0 ? bj : 0;
    res.begin_i = bs > 0 ? i : 0;
    res.begin_j = bs > 0 ? j : 0;
    res.n_ops = (int32_t)k;
    a.results[h] = res;
  }
}

}  // namespace

int trace_rows_per_band() { return kTraceRows; }

cudaError_t launch_trace(const TraceArgs &a, int sms, cudaStream_t s) {
  if (a.nhits <= 0) return cudaSuccess;
  constexpr int wpc = kTraceThreads / 32;
  const size_t smem = kScoreBytes + (size_t)wpc * kTraceWarpBytes;
  // one warp per SM sub-partition: the longest hits' bands, which set the time,
  // then have theirs to themselves (200 hits: 2.7 ms a call; two warps 3.35,
  // four 3.75).  Also slower: lanes of 4 rows and two columns a step 3.06-3.4.
  const int grid = std::min((a.nbands + wpc - 1) / wpc, sms);
  const int64_t clear = a.dir_words / kBlockWords * 8;
  trace_clear_kernel<<<(int)std::min<int64_t>((clear + 255) / 256, 8 * sms), 256, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  trace_fill_kernel<<<grid, kTraceThreads, smem, s>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  trace_walk_kernel<<<(a.nhits + 3) / 4, 128, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace swgb
