// Band-stream kernel: long queries, and long database sequences, of small
// batches (Sec. 2.2 Eqs. 1-3; Sec. 3.1 "long kernel"; Fig. 1 intra-sequence
// parallelism), for sm_103a.
//
// In a small batch a long query (thousands of rows) against a few thousand
// database sequences leaves the inter-task kernel one chain per database
// unit, each chain sweeping its unit once per chunk of query rows, chunk
// after chunk: the longest chains set the time while most SMs idle.  Here the
// query's rows are cut into bands of 32 lanes x R rows, one warp each, and
// all bands of a *job* -- a query and a stream of database units -- run as a
// pipeline: the warp of band b sweeps the units of the stream one after the
// other, and reads the bottom row of band b - 1 for each column from a ring
// in global memory as soon as band b - 1 has written it.  A job's stream is
// short enough (a few thousand columns) that many jobs run at once, and every
// unit's cells are spread over all the job's warps instead of one.
//
// Forms: int32 cells, one database sequence per unit (in 16-bit batches for
// the pairs that could pass the 16-bit range), or two sequences per unit in
// the 16-bit halves of a word (only for pairs that cannot pass the 16-bit
// range, so no rescue is needed).  One column per step (band_core.cuh): every
// unit is a matrix of its own, and a band's last lane finishes it 32 columns
// after its first; two columns per step would make that 64.
//
// Rings and progress.  Each ring holds one 64-bit entry per column of the
// job's whole stream, zeroed before the launch, and is written once: the
// writer (band b's last lane) stores (H | 1 << 31, F) with one relaxed 64-bit
// store, and the reader (band b + 1, lanes 0..15, a block of 16 columns ahead)
// reloads until bit 31 is set.  H is below 2^31 (int32: bounded by the host;
// 16-bit halves: both halves non-negative, so bit 31 is the high half's sign
// bit, 0).  No band ever waits for a band below it (the rings never wrap), and
// warps take their bands from an atomic counter in order, so every band a
// warp waits on was taken earlier by a warp that is running: the pipeline
// cannot deadlock whatever the launch's residency.  Every wait is bounded.
//
// Scores: each band keeps its running best per unit and adds it to the
// caller-order output with atomicMax (the host zeroes the jobs' output rows
// first); the maximum over the bands is the unit's score.
#include <algorithm>
#include "band_core.cuh"

namespace swgb {
namespace {

// 12 warps, one band at a time each, one CTA per SM with up to 168
// registers a thread (the 512-row bands' profiles and residues take 157 KB of
// shared memory).  Homolog search, ms (packed / int32): 8 warps 1.82 / 3.19;
// 10 warps 1.91 / 2.88; 12 warps 1.68 / 2.52; 14 warps 1.82 / 2.52; 16 warps
// 1.83 / 2.41.  (Before the steps of band_core.cuh: 1.89 / 2.71 at 12.)
constexpr int kBandStreamThreads = 384;
// Steps unrolled (4 -> 8: homolog search 1,747 -> 1,719 us packed, 2,570 ->
// 2,528 int32).
constexpr int kBandUnroll = 8;
constexpr int kSubmatBytes = 512;
// R rows per lane: bands of 32 R query rows; a band's profile is [21][32 lanes
// x R] bytes, followed by its residues (two sequences, two chunks) and
// boundary slots (2 x 16 x 8 B)
template <int R>
constexpr int kProfBytes = kProfRows * 32 * R;
constexpr int kBandIoBytes = 4 * kResChunk + 2 * kColBlock * 8;
template <int R>
constexpr int kWarpBytes = (kProfBytes<R> + kBandIoBytes + 127) / 128 * 128;

// A band's profile in the warp's shared-memory block: byte [c][lane * R + r]
// = SM(Q[row], c) for row = band * 32 R + lane * R + r, the pad value for the
// pad residue (c = 20) and rows past the query's end.
template <int R>
__device__ __forceinline__ void build_band_profile(uint8_t *prof, const int8_t *sm, const uint8_t *q, int m,
                                                   int row0, int lane, int32_t pad) {
  uint8_t codes[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int row = row0 + lane * R + r;
    codes[r] = row < m ? q[row] : (uint8_t)kPadCode;
  }
  for (int c = 0; c < kProfRows; ++c) {
#pragma unroll
    for (int w = 0; w < R / 4; ++w) {
      uint32_t v = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int code = codes[4 * w + b];
        const int32_t s = (c < kAlphabet && code < kAlphabet) ? (int32_t)sm[code * kAlphabet + c] : pad;
        v |= ((uint32_t)s & 0xffu) << (8 * b);
      }
      *reinterpret_cast<uint32_t *>(prof + c * 32 * R + lane * R + 4 * w) = v;
    }
  }
}

// One band over one database unit (columns sbase .. of the job's stream, its
// padded length); io: the warp's residues and boundary slots.  Returns false
// when a wait expired.
template <int R, int FORM>
__device__ __forceinline__ bool band_unit(const BandArgs &a, const uint8_t *__restrict__ prof, uint8_t *io,
                                          const int lane, const int posA, const int posB, const int64_t sbase,
                                          const unsigned long long *ring_in, unsigned long long *ring_out,
                                          const Consts &cs, Word<FORM> &Sout) {
  constexpr bool PACKED = FORM == kFormPacked;
  using Prof = std::conditional_t<PACKED, SeqPairProfile<R, 1>, IntProfile<R, 1>>;
  const int npa = a.db.npad[posA];
  const int npb = PACKED ? a.db.npad[posB] : 0;
  const int npad = max(npa, npb);
  ResidueStage<PACKED ? 2 : 1> rs{io,   a.db.res + a.db.off[posA], a.db.res + a.db.off[posB], npa, npb, lane,
                                  a.db.res, a.db.res_bytes, a.status};
  uint2 *rgb = reinterpret_cast<uint2 *>(io + 4 * kResChunk);
  __syncwarp();  // (the unit before this one has read its residues and slots)
  rs.stage(0);
  clear_slots(rgb, lane, PACKED ? cs.F0W : 0u);
  OnceRing<> x{ring_in ? ring_in + sbase : nullptr, ring_out ? ring_out + sbase : nullptr, rgb, lane, a.rings,
             a.ring_entries, a.status, ring_in != nullptr, ring_out != nullptr};
  BandLane<R, FORM, 1> ln;
  ln.reset(cs);
  const bool ok = band_sweep<FORM, 1, kBandUnroll, false, Prof>(ln, rs, x, rgb, prof + lane * R, 32 * R, lane,
                                                      npad / kColBlock, (Word<FORM>)-1, (Word<FORM>)0, cs, a.status);
  cp_async_wait<0>();
  Sout = ln.S;
  return ok;
}

template <int R, int GAPS>
__global__ void __launch_bounds__(kBandStreamThreads, 1) band_stream_kernel(const BandArgs a) {
  constexpr int RH = R / 2;  // rows per lane of kBandInt32Half jobs
  extern __shared__ __align__(128) uint8_t smem[];
  int8_t *sm = reinterpret_cast<int8_t *>(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint8_t *prof = smem + kSubmatBytes + (size_t)warp * kWarpBytes<R>;
  uint8_t *io = prof + kProfBytes<R>;
  for (int i = threadIdx.x; i < kAlphabet * kAlphabet; i += blockDim.x) sm[i] = a.submat[i];
  __syncthreads();
  const Consts cs = make_consts<GAPS>(a.sc);

  for (;;) {
    int g = 0;
    if (lane == 0) g = atomicAdd(a.band_counter, 1);
    g = __shfl_sync(0xffffffffu, g, 0);
    if (g >= a.nbands) break;
    const BandJob job = a.jobs[a.band_job[g]];
    const int b = g - job.band0;
    const QDesc qd = a.qd[job.q];
    const bool half = job.form == kBandInt32Half;
    __syncwarp();
    if (half) build_band_profile<RH>(prof, sm, a.qres + qd.qoff, qd.m, b * 32 * RH, lane, a.sc.pad);
    else build_band_profile<R>(prof, sm, a.qres + qd.qoff, qd.m, b * 32 * R, lane, a.sc.pad);
    __syncwarp();
    const unsigned long long *ring_in = b > 0 ? a.rings + job.ring0 + (int64_t)(b - 1) * job.cols : nullptr;
    unsigned long long *ring_out = b + 1 < job.nb ? a.rings + job.ring0 + (int64_t)b * job.cols : nullptr;
    int32_t *orow = a.out + (int64_t)job.q * a.out_stride;
    int64_t sbase = 0;
    bool ok = true;
    for (int t = 0; t < job.t_count && ok; ++t) {
      int2 p = make_int2(0, 0);
      if (in_range(job.t_begin + t, a.n_tpos, a.status)) p = a.tpos[job.t_begin + t];
      if (!in_range(p.x, a.db.n, a.status) || !in_range(p.y, a.db.n, a.status)) p = make_int2(0, 0);
      if (job.form == kBandPacked) {
        uint32_t S = 0u;
        ok = band_unit<R, kFormPacked>(a, prof, io, lane, p.x, p.y, sbase, ring_in, ring_out, cs, S);
        for (int d = 16; d > 0; d >>= 1) S = __vmaxs2(S, __shfl_xor_sync(0xffffffffu, S, d));
        if (ok && lane == 0) {
          if (in_range(job.q * a.out_stride + a.db.perm[p.x], a.out_size, a.status))
            atomicMax(&orow[a.db.perm[p.x]], (int32_t)(S & 0xffffu));
          if (p.y != p.x && in_range(job.q * a.out_stride + a.db.perm[p.y], a.out_size, a.status))
            atomicMax(&orow[a.db.perm[p.y]], (int32_t)(S >> 16));
        }
        sbase += max(a.db.npad[p.x], a.db.npad[p.y]);
      } else {
        int32_t S = 0;
        if (half) ok = band_unit<RH, kFormInt32>(a, prof, io, lane, p.x, p.x, sbase, ring_in, ring_out, cs, S);
        else ok = band_unit<R, kFormInt32>(a, prof, io, lane, p.x, p.x, sbase, ring_in, ring_out, cs, S);
        for (int d = 16; d > 0; d >>= 1) S = max(S, __shfl_xor_sync(0xffffffffu, S, d));
        if (ok && lane == 0 && in_range(job.q * a.out_stride + a.db.perm[p.x], a.out_size, a.status))
          atomicMax(&orow[a.db.perm[p.x]], S);
        sbase += a.db.npad[p.x];
      }
    }
    __syncwarp();
    if (!ok) break;
  }
}

// ---------------------------------------------------------------------------
// Transposed jobs: database row tracks against one query (see TrackArgs in
// internal.h).  The query residues are the columns; the bands' rows are
// database sequences stacked in row tracks.
//
// Two row tracks share a word in the 16-bit forms; their substitution scores
// come from two byte tables, one per track (rows [0, 21) and [21, 42) of the
// band's profile), both read at the column's residue code and paired into the
// two halves by a byte shuffle (TablePairProfile).  (One table of query-pair
// words would save the shuffle but take twice the shared memory, and so half
// the resident warps.)
// ---------------------------------------------------------------------------

// 4 warps, one per SM sub-partition: a small batch has few bands, and CTAs
// of 8 warps put two on each sub-partition of half the SMs while the others
// idle
constexpr int kTrackThreads = 128;
constexpr int kTrackCols = 2;  // columns per step (band_core.cuh)
template <int R>
constexpr int kTrackStride = 32 * R;                                // bytes per residue row of one table
template <int R>
constexpr int kTrackProfBytes = 2 * kProfRows * kTrackStride<R>;    // two tables of [21][32 lanes x R] bytes
constexpr int kTrackIoBytes = 2 * kResChunk + 2 * kColBlock * 8;    // residues, boundary slots
template <int R>
constexpr int kTrackWarpBytes = (kTrackProfBytes<R> + kTrackIoBytes + 127) / 128 * 128;

// Profile of a band's rows: the substitution score of query residue c
// (column) against each database row, SM(c, D[row]) (the query residue is
// the matrix's row index): table t, byte (c, lane, r) at (21 t + c) * stride
// + lane * R + r, for the low (t = 0) and high (t = 1) track.  Rows past a
// sequence's end, idle lanes and the pad residue (c = 20) hold the pad value.
// (R = 24: 10.4 -> 3.4 us of a small search against a byte lookup per score.)
template <int R, bool TWO>
__device__ __forceinline__ void build_track_profile(uint8_t *prof, const uint8_t *score, const DbView &db,
                                                    const TrackLane &L, int lane, int32_t *status) {
#pragma unroll 1
  for (int t = 0; t < (TWO ? 2 : 1); ++t) {
    const int32_t pos = t ? L.pb : L.pa, r0 = t ? L.rb : L.ra;
    const bool ok = pos >= 0 && in_range(pos, db.n, status);
    const int32_t npad = ok ? db.npad[pos] : 0;
    const uint8_t *res = db.res + (ok ? db.off[pos] : 0);
    uint32_t code[R / 4];  // (a sequence's padding up to npad, a multiple of 16, holds the pad code)
#pragma unroll
    for (int i = 0; i < R / 4; ++i) {
      const int32_t row = r0 + 4 * i;
      code[i] = (row < npad && in_range(res + row + 3 - db.res, db.res_bytes, status))
                    ? *reinterpret_cast<const uint32_t *>(res + row) : 0x14141414u;
    }
    profile_from_scores<R>(prof + t * kProfRows * kTrackStride<R> + lane * R, kTrackStride<R>, score, code);
  }
}

// One band of a row track over all columns of its query.  keepH / addF: the
// lane's restart masks (a half whose rows start a sequence takes the matrix
// top boundary (0, F0) instead of the row above).  io: the warp's residues
// and boundary slots, the first chunk of residues staged.  Returns false when
// a wait expired.
template <int R, int FORM, int U>
__device__ __forceinline__ bool track_pass(const TrackArgs &a, const uint8_t *__restrict__ prof, ResidueStage<1> &rs,
                                           uint2 *rgb, const int lane, const int npad,
                                           const unsigned long long *ring_in, unsigned long long *ring_out,
                                           const Word<FORM> keepH, const Word<FORM> addF, const Consts &cs,
                                           Word<FORM> &Sout) {
  constexpr bool PACKED = FORM != kFormInt32;
  using Prof = std::conditional_t<PACKED, TablePairProfile<R, kTrackCols>, IntProfile<R, kTrackCols>>;
  clear_slots(rgb, lane, PACKED ? cs.F0W : 0u);
  OnceRing<> x{ring_in, ring_out, rgb, lane, a.rings, a.ring_entries, a.status, ring_in != nullptr, ring_out != nullptr};
  BandLane<R, FORM, kTrackCols> ln;
  ln.reset(cs);
  const bool ok = band_sweep<FORM, kTrackCols, U, true, Prof>(ln, rs, x, rgb, prof + lane * R, kTrackStride<R>, lane,
                                                              npad / kColBlock, keepH, addF, cs, a.status);
  cp_async_wait<0>();
  Sout = ln.S;
  return ok;
}

// The best score of each sequence among a band's lanes (its rows are
// contiguous lanes): a segmented maximum down the lanes, keyed by the
// sequence; the last lane of each segment adds it to the caller-order score
// with atomicMax (a sequence spanning several bands gets one per band).
__device__ __forceinline__ void track_scores(const TrackArgs &a, int32_t q, int32_t key, int32_t v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int32_t ov = __shfl_up_sync(0xffffffffu, v, d);
    const int32_t ok = __shfl_up_sync(0xffffffffu, key, d);
    if (lane >= d && ok == key) v = max(v, ov);
  }
  const int32_t nk = __shfl_down_sync(0xffffffffu, key, 1);
  if ((lane == 31 || nk != key) && key >= 0 && in_range(key, a.db.n, a.status)) {
    const int64_t i = (int64_t)q * a.out_stride + a.db.perm[key];
    if (in_range(i, a.out_size, a.status)) atomicMax(&a.out[i], v);
  }
}

// The job of band g of the launch, and its band or (negative) how many of the
// job's bands are left from it on.
__device__ __forceinline__ int2 track_band_of(const TrackArgs &a, int g, int lane) {
  int4 e = make_int4(0, 0, 1, 0);
  for (int k = 0; k < a.n_groups; k += 32) {  // the last group that starts at or before g
    const int4 v = k + lane < a.n_groups ? reinterpret_cast<const int4 *>(a.groups)[k + lane]
                                         : make_int4(0x7fffffff, 0, 1, 0);
    const uint32_t m = __ballot_sync(0xffffffffu, v.x <= g);
    if (m == 0u) break;
    const int src = 31 - __clz(m);
    e = make_int4(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src),
                  __shfl_sync(0xffffffffu, v.z, src), __shfl_sync(0xffffffffu, v.w, src));
    if (m != 0xffffffffu) break;
  }
  const int i = g - e.x;
  return e.z == 0 ? make_int2(e.y + i, -e.w) : make_int2(e.y + i / e.z, i % e.z);
}

// One band: its rows' profile, the sweep, and the scores of its sequences.
template <int R, int UP, int UI>
__device__ __forceinline__ bool track_band(const TrackArgs &a, uint8_t *prof, const uint8_t *score,
                                           ResidueStage<1> &rs, uint2 *rgb, const int32_t q, const bool packed,
                                           const TrackLane &L, const int lane, const int npad,
                                           const unsigned long long *ring_in, unsigned long long *ring_out,
                                           const Consts &cs) {
  const bool ra0 = L.pa < 0 || L.ra == 0, rb0 = L.pb < 0 || L.rb == 0;  // halves that restart
  bool ok;
  if (packed) {
    build_track_profile<R, true>(prof, score, a.db, L, lane, a.status);
    __syncwarp();
    const uint32_t mask = (ra0 ? 0x0000ffffu : 0u) | (rb0 ? 0xffff0000u : 0u);
    uint32_t S = 0u;
    ok = track_pass<R, kFormPacked, UP>(a, prof, rs, rgb, lane, npad, ring_in, ring_out, ~mask, cs.F0W & mask, cs, S);
    track_scores(a, q, L.pa, (int32_t)(S & 0xffffu), lane);
    track_scores(a, q, L.pb, (int32_t)(S >> 16), lane);
  } else {
    build_track_profile<R, false>(prof, score, a.db, L, lane, a.status);
    __syncwarp();
    int32_t S = 0;
    ok = track_pass<R, kFormInt32, UI>(a, prof, rs, rgb, lane, npad, ring_in, ring_out, ra0 ? 0 : -1, 0, cs, S);
    track_scores(a, q, L.pa, S, lane);
  }
  return ok;
}

template <int R, int GAPS>
__global__ void __launch_bounds__(kTrackThreads, R <= 8 ? 4 : R <= 20 ? 2 : 1) band_track_kernel(const TrackArgs a) {
  constexpr int RL = track_long_rows(R);  // sequences longer than a band
  // steps unrolled (16-bit words, int32): what fits the instruction cache,
  // together with the longer sequences' height where that is another one (one
  // query x 2,000 proteins, 20-row words beside 16-row ones: 4 -> 2 steps 54.5
  // -> 47.7 us at 144 residues, 210 -> 171 us at 1,000)
  constexpr int UP = R == RL ? (R <= 12 ? 8 : 4) : 2, UI = R == RL ? 8 : 4;
  extern __shared__ __align__(128) uint8_t smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint8_t *prof = smem + kScoreBytes + (size_t)warp * kTrackWarpBytes<R>;
  uint8_t *io = prof + kTrackProfBytes<R>;
  uint2 *rgb = reinterpret_cast<uint2 *>(io + 2 * kResChunk);
  build_scores<true>(smem, a.submat, a.sc.pad);
  __syncthreads();
  const Consts cs = make_consts<GAPS>(a.sc);
  const TrackLane idle{-1, 0, -1, 0};
  // a lane continues the sequence of the row above (in at least one used half)
  auto continues = [](const TrackLane &L, bool packed) {
    return (L.pa >= 0 && L.ra > 0) || (packed && L.pb >= 0 && L.rb > 0);
  };

  for (;;) {
    int g = 0;
    if (lane == 0) g = atomicAdd(a.band_counter, 1);
    g = __shfl_sync(0xffffffffu, g, 0);
    if (g >= a.nbands) break;
    const int2 jb = track_band_of(a, g, lane);
    const TrackJob job = a.jobs[jb.x];
    const int b = jb.y < 0 ? job.nb + jb.y : jb.y;
    const bool packed = job.packed != 0;
    const int64_t li = (int64_t)job.lane0 + 32 * (int64_t)b + lane;
    const TrackLane L = in_range(li, a.n_lanes, a.status) ? a.lanes[li] : idle;
    // the band reads the band above when its first lane continues a sequence;
    // it writes for the band below when that one's first lane does
    const bool prev = b > 0 && __shfl_sync(0xffffffffu, (int)continues(L, packed), 0) != 0;
    int nxt = 0;
    if (lane == 0 && b + 1 < job.nb) {
      const int64_t ln = (int64_t)job.lane0 + 32 * (int64_t)(b + 1);
      nxt = in_range(ln, a.n_lanes, a.status) && continues(a.lanes[ln], packed) ? 1 : 0;
    }
    const bool next = __shfl_sync(0xffffffffu, nxt, 0) != 0;
    const int32_t npad = a.qt_npad[job.q];
    const uint8_t *resQ = a.qt + a.qt_off[job.q];
    __syncwarp();  // (the band before this one has read its profile, residues and slots)
    ResidueStage<1> rs{io, resQ, nullptr, npad, 0, lane, a.qt, a.qt_bytes, a.status};
    rs.stage(0);
    const unsigned long long *ring_in = prev ? a.rings + job.ring0 + (int64_t)(b - 1) * npad : nullptr;
    unsigned long long *ring_out = next ? a.rings + job.ring0 + (int64_t)b * npad : nullptr;
    bool ok;
    if (R == RL || job.rows == R)
      ok = track_band<R, UP, UI>(a, prof, smem, rs, rgb, job.q, packed, L, lane, npad, ring_in, ring_out, cs);
    else
      ok = track_band<RL, UP, UI>(a, prof, smem, rs, rgb, job.q, packed, L, lane, npad, ring_in, ring_out, cs);
    __syncwarp();
    if (!ok) break;
  }
}

template <int R>
size_t smem_of() {
  return kSubmatBytes + (size_t)(kBandStreamThreads / 32) * kWarpBytes<R>;
}

// Dynamic shared memory that leaves room for only one band-stream CTA per SM
// (more than half of an SM's shared memory), or 0 if a block may not take it.
size_t one_cta_smem() {
  int dev = 0, per_sm = 0, per_block = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const size_t want = ((size_t)per_sm / 2 + 1024 + 127) / 128 * 128;
  return want <= (size_t)per_block ? want : 0;
}

// The kernels with the protein penalties compiled in (see GapSet), or general.
using BandKernel = void (*)(const BandArgs);
BandKernel band_kernel(int R, int gaps) {
  const bool p = gaps == kGapsProtein;
  if (R == 8) return p ? band_stream_kernel<8, kGapsProtein> : band_stream_kernel<8, kGapsAny>;
  if (R == 16) return p ? band_stream_kernel<16, kGapsProtein> : band_stream_kernel<16, kGapsAny>;
  return nullptr;
}
using TrackKernel = void (*)(const TrackArgs);
template <int R>
TrackKernel track_kernel_of(int gaps) {
  return gaps == kGapsProtein ? band_track_kernel<R, kGapsProtein> : band_track_kernel<R, kGapsAny>;
}
#define SWGB_TRACK_R_LIST(X) X(8) X(12) X(16) X(20) X(24)
TrackKernel track_kernel(int R, int gaps) {
#define SWGB_CASE(RR) \
  if (R == RR) return track_kernel_of<RR>(gaps);
  SWGB_TRACK_R_LIST(SWGB_CASE)
#undef SWGB_CASE
  return nullptr;
}

template <class Kernel>
int occupancy_of(Kernel kern, int threads, size_t smem, size_t limit) {
  int n = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

size_t track_smem_of(int R) {
  size_t warp_bytes = 0;
#define SWGB_CASE(RR) \
  if (R == RR) warp_bytes = kTrackWarpBytes<RR>;
  SWGB_TRACK_R_LIST(SWGB_CASE)
#undef SWGB_CASE
  return kScoreBytes + (kTrackThreads / 32) * warp_bytes;
}

}  // namespace

int track_threads() { return kTrackThreads; }

int track_max_ctas_per_sm(int R, int gaps) {
  const TrackKernel kern = track_kernel(R, gaps);
  return kern ? occupancy_of(kern, kTrackThreads, track_smem_of(R), track_smem_of(R)) : 0;
}

cudaError_t launch_track(const TrackArgs &a, int R, int grid, cudaStream_t s) {
  const TrackKernel kern = track_kernel(R, gap_set(a.sc));
  if (!kern) return cudaErrorInvalidValue;
  kern<<<grid, kTrackThreads, track_smem_of(R), s>>>(a);
  return cudaGetLastError();
}

int band_threads() { return kBandStreamThreads; }
bool band_supported_R(int R) { return R == 8 || R == 16; }
size_t band_smem_bytes(int R) { return R == 16 ? smem_of<16>() : smem_of<8>(); }
int band_max_ctas_per_sm(int R, int gaps) {
  const BandKernel kern = band_kernel(R, gaps);
  // (the limit admits the one-CTA-per-SM reservation as well)
  return kern ? occupancy_of(kern, kBandStreamThreads, band_smem_bytes(R), std::max(band_smem_bytes(R), one_cta_smem()))
              : 0;
}

cudaError_t launch_band(const BandArgs &a, int R, int grid, bool one_per_sm, cudaStream_t s) {
  // one CTA per SM: the launch takes more than half of an SM's shared memory,
  // so that the hardware never places two on an SM, whatever else (the
  // transposed jobs beside it, a kernel finishing before it) holds the SMs
  // when its CTAs are placed
  const BandKernel kern = band_kernel(R, gap_set(a.sc));
  if (!kern) return cudaErrorInvalidValue;
  kern<<<grid, kBandStreamThreads, std::max(one_per_sm ? one_cta_smem() : 0, band_smem_bytes(R)), s>>>(a);
  return cudaGetLastError();
}

}  // namespace swgb
