// The sweep shared by the pipelines of one-warp bands (long pairs, band-stream
// jobs, transposed jobs, tracebacks): 32 lanes of R rows, an anti-diagonal wavefront down
// the lanes, the bottom row handed to the band below through a ring of 64-bit
// entries in global memory.
//
// A band often has its SM sub-partition to itself, so a step is laid out for
// one warp's latency: what a step needs besides the row above it -- residue
// codes, profile words, boundary entries -- is fetched during the step before;
// H_diag + SM of all rows is formed while the shuffles are on their way; the
// bottom row is stored by one predicated instruction at the start of the next
// step.  (With the store as a branch of the last lane, and the residue and
// profile loads behind the shuffle, a step of the pair kernel took 190 cycles
// beside its cells, of 287 at R = 8.)
#pragma once

#include "devutil.cuh"
#include "dp_common.cuh"
#include "internal.h"
#include "../../include/swgb.h"

namespace swgb {

// Profile bytes of a lane's R rows, rounded up to whole words.
template <int R>
constexpr int kSlotBytes = (R + 3) / 4 * 4;
template <int R>
__device__ __forceinline__ void load_rows(const uint8_t *p, uint32_t (&w)[kSlotBytes<R> / 4]) {
  if constexpr (R % 4 == 0) {
    load_prof<R>(p, w);
  } else {
#pragma unroll
    for (int i = 0; i < kSlotBytes<R> / 4; ++i) w[i] = reinterpret_cast<const uint32_t *>(p)[i];
  }
}

// N words to byte p (as aligned as load_prof reads them).
template <int N>
__device__ __forceinline__ void store_words(uint8_t *p, const uint32_t (&w)[N]) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N / 4; ++i)
      reinterpret_cast<uint4 *>(p)[i] = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
  } else if constexpr (N % 2 == 0) {
#pragma unroll
    for (int i = 0; i < N / 2; ++i) reinterpret_cast<uint2 *>(p)[i] = make_uint2(w[2 * i], w[2 * i + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) reinterpret_cast<uint32_t *>(p)[i] = w[i];
  }
}

// Score table in shared memory: row k holds the scores of residue k (of the
// bands' rows) against the columns' residues c = 0..20 (pad), one byte each;
// rows are 28 bytes apart (seven words: the 21 rows' words of a lookup fall in
// different banks).  TARGET_ROWS: the bands' rows are database residues and
// the columns the query's (SM's row index), else the other way round.
constexpr int kScoreRow = 28;
constexpr int kScoreBytes = 640;
template <bool TARGET_ROWS>
__device__ __forceinline__ void build_scores(uint8_t *score, const int8_t *submat, int32_t pad) {
  for (int i = threadIdx.x; i < kProfRows * kScoreRow; i += blockDim.x) {
    const int k = i / kScoreRow, c = i - k * kScoreRow;
    score[i] = (uint8_t)(k < kAlphabet && c < kAlphabet ? submat[TARGET_ROWS ? c * kAlphabet + k : k * kAlphabet + c]
                                                        : pad);
  }
}

// A lane's profile bytes from its rows' residue codes (four per word): row r
// at residue c to p[c * stride + r].  Four rows against four residues are four
// words of the score table, transposed by byte shuffles.
template <int R>
__device__ __forceinline__ void profile_from_scores(uint8_t *p, int stride, const uint8_t *score,
                                                    const uint32_t (&code)[R / 4]) {
#pragma unroll 1
  for (int w = 0; w < (kProfRows + 3) / 4; ++w) {
    uint32_t out[4][R / 4];
#pragma unroll
    for (int i = 0; i < R / 4; ++i) {
      uint32_t v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        v[j] = *reinterpret_cast<const uint32_t *>(score + prmt(code[i], 0u, sel_one(j)) * kScoreRow + 4 * w);
      const uint32_t a = prmt(v[0], v[1], 0x5140u), b = prmt(v[2], v[3], 0x5140u);
      const uint32_t c = prmt(v[0], v[1], 0x7362u), d = prmt(v[2], v[3], 0x7362u);
      out[0][i] = prmt(a, b, 0x5410u);
      out[1][i] = prmt(a, b, 0x7632u);
      out[2][i] = prmt(c, d, 0x5410u);
      out[3][i] = prmt(c, d, 0x7632u);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (4 * w + j < kProfRows) store_words(p + (4 * w + j) * stride, out[j]);
  }
}

// The profile words of one step, COLS columns: add(c, r, h) is h plus the
// substitution score of row r at column c.  load() takes the step's residue
// codes (the layout is the sweep's `res` word).
template <int R, int COLS>
struct IntProfile {  // int32 cells: one byte table, a code per column
  static constexpr int kBits = 8;
  uint32_t w[COLS][kSlotBytes<R> / 4];
  __device__ __forceinline__ void load(const uint8_t *prow, int stride, uint32_t res) {
#pragma unroll
    for (int c = 0; c < COLS; ++c) load_rows<R>(prow + (res >> (8 * c) & 0xffu) * stride, w[c]);
  }
  __device__ __forceinline__ int32_t add(int c, int r, int32_t h) const { return add_byte(w[c], r, h); }
  static __device__ __forceinline__ uint32_t checked(uint32_t res, int32_t *status) {
    if constexpr (kChecked)
      for (int c = 0; c < COLS; ++c)
        if ((res >> (8 * c) & 0xffu) > (uint32_t)kPadCode) {
          atomicExch(status, kStatusBounds);
          return kPadCode * 0x0101u;
        }
    return res;
  }
};
template <int R, int COLS>
struct SeqPairProfile {  // 16-bit halves, two sequences: one byte table, two codes per column
  static_assert(COLS == 1, "one column per step");
  uint32_t a[kSlotBytes<R> / 4], b[kSlotBytes<R> / 4];
  __device__ __forceinline__ void load(const uint8_t *prow, int stride, uint32_t res) {
    load_rows<R>(prow + (res & 0xffu) * stride, a);
    load_rows<R>(prow + (res >> 8) * stride, b);
  }
  __device__ __forceinline__ uint32_t add(int, int r, uint32_t h) const {
    return __vadd2(h, prmt(a[r >> 2], b[r >> 2], sel_pair(r & 3)));
  }
  static __device__ __forceinline__ uint32_t checked(uint32_t res, int32_t *status) {
    if constexpr (kChecked)
      if ((res & 0xffu) > (uint32_t)kPadCode || (res >> 8) > (uint32_t)kPadCode) {
        atomicExch(status, kStatusBounds);
        return kPadCode * 0x0101u;
      }
    return res;
  }
};
template <int R, int COLS>
struct TablePairProfile {  // 16-bit halves, two byte tables of 21 rows each, a code per column
  uint32_t a[COLS][kSlotBytes<R> / 4], b[COLS][kSlotBytes<R> / 4];
  __device__ __forceinline__ void load(const uint8_t *prow, int stride, uint32_t res) {
#pragma unroll
    for (int c = 0; c < COLS; ++c) {
      const uint8_t *p = prow + (res >> (8 * c) & 0xffu) * stride;
      load_rows<R>(p, a[c]);
      load_rows<R>(p + kProfRows * stride, b[c]);
    }
  }
  __device__ __forceinline__ uint32_t add(int c, int r, uint32_t h) const {
    return __vadd2(h, prmt(a[c][r >> 2], b[c][r >> 2], sel_pair(r & 3)));
  }
  static __device__ __forceinline__ uint32_t checked(uint32_t res, int32_t *status) {
    return IntProfile<R, COLS>::checked(res, status);
  }
};

// A lane's rows: one step computes COLS columns.  With two, the second
// column's chain down the rows runs one row behind the first one's, so a warp
// has two chains to interleave, and the step's fixed cost is paid once for
// both; the lanes then work two columns apart.
template <int R, int FORM, int COLS>
struct BandLane {
  using W = Word<FORM>;
  W Hl[R], E[R];
  W outH[COLS], outF[COLS];  // the bottom row of the last step: H, and F of the row below
  W hdiag;                   // H of the row above at the last column of the step before
  W S;                       // best so far

  __device__ __forceinline__ void reset(const Consts &cs) {
    const W E0 = FORM != kFormInt32 ? (W)cs.F0W : (W)0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      Hl[r] = (W)0;
      E[r] = E0;
    }
#pragma unroll
    for (int c = 0; c < COLS; ++c) {
      outH[c] = (W)0;
      outF[c] = E0;
    }
    hdiag = S = (W)0;
  }

  template <class Prof>
  __device__ __forceinline__ void step(const Prof &p, const W (&inH)[COLS], const W (&inF)[COLS], const Consts &cs) {
    W x[R];  // H_diag + SM of the first column
#pragma unroll
    for (int r = R - 1; r >= 0; --r) x[r] = (W)p.add(0, r, r > 0 ? Hl[r - 1] : hdiag);
    W f[COLS];
#pragma unroll
    for (int c = 0; c < COLS; ++c) f[c] = inF[c];
    W d = inH[0];  // H of the row above at the first column
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const W h = cell(x[r], E[r], f[0], cs);
      if constexpr (COLS == 2) {
        const W h2 = cell((W)p.add(1, r, d), E[r], f[1], cs);
        S = max3(S, h, h2);
        Hl[r] = h2;
        d = h;
      } else {
        Hl[r] = h;
      }
    }
    if constexpr (COLS == 1) {  // (as in word_rows: after the rows, as two chains)
      constexpr int R2 = R / 2;
      static_assert(R % 4 == 0, "two halves of whole pairs");
      W a = Hl[R2 - 1], b = Hl[R - 1];
#pragma unroll
      for (int r = 0; r + 1 < R2; r += 2) {
        a = max3(a, Hl[r], Hl[r + 1]);
        b = max3(b, Hl[R2 + r], Hl[R2 + r + 1]);
      }
      S = max3(S, a, b);
    }
    outH[0] = COLS == 2 ? d : Hl[R - 1];
    if constexpr (COLS == 2) outH[1] = Hl[R - 1];
#pragma unroll
    for (int c = 0; c < COLS; ++c) outF[c] = f[c];
    hdiag = inH[COLS - 1];
  }

 private:
  static __device__ __forceinline__ W max3(W a, W b, W c) {
    if constexpr (FORM != kFormInt32) return __vimax3_s16x2(a, b, c);
    else return __vimax3_s32(a, b, c);
  }
  // H = max(x, E, F, 0) (Eq. 1); E of the next column and F of the row below (Eqs. 2, 3)
  static __device__ __forceinline__ W cell(W x, W &e, W &f, const Consts &cs) {
    if constexpr (FORM != kFormInt32) {
      const uint32_t h = __vimax3_s16x2_relu(x, e, f);
      const uint32_t hgo = __vsub2(h, cs.goW);
      e = __vmaxs2(__vsub2(e, cs.geW), hgo);
      f = __vmaxs2(__vsub2(f, cs.geW), hgo);
      return h;
    } else {
      const int32_t h = __vimax3_s32_relu(x, e, f);
      const int32_t hgo = h - cs.go;
      e = max(e - cs.ge, hgo);
      f = max(f - cs.ge, hgo);
      return h;
    }
  }
};

// Residues of the columns, staged in shared memory kResChunk columns at a time
// by the whole warp, a chunk ahead.  SEQS sequences of na, nb real (padded)
// columns; the pad code past them.  ring: 2 * SEQS * kResChunk bytes.
constexpr int kResChunk = 512;  // 16 columns per lane
template <int SEQS>
struct ResidueStage {
  uint8_t *ring;
  const uint8_t *a, *b;
  int na, nb, lane;
  const uint8_t *base;  // the residue buffer and its size (checked build)
  int64_t bytes;
  int32_t *status;

  __device__ __forceinline__ void put(uint8_t *d, const uint8_t *s, int col, int n) {
    if (col < n && in_range(s + col + 15 - base, bytes, status)) cp_async16(d, s + col);
    else *reinterpret_cast<uint4 *>(d) = make_uint4(0x14141414u, 0x14141414u, 0x14141414u, 0x14141414u);
  }
  __device__ __forceinline__ void stage(int chunk) {
    uint8_t *d = ring + (chunk & 1) * kResChunk + lane * 16;
    const int64_t col = (int64_t)chunk * kResChunk + lane * 16;
    const int c = (int)min(col, (int64_t)0x7fffffff);
    put(d, a, c, na);
    if constexpr (SEQS == 2) put(d + 2 * kResChunk, b, c, nb);
    cp_async_commit();
  }
  // the codes of columns [col, col + COLS), 8 bits each (two sequences: A's and B's code of one column)
  template <int COLS>
  __device__ __forceinline__ uint32_t at(int col) const {
    const uint8_t *p = ring + (col & (2 * kResChunk - 1));
    if constexpr (SEQS == 2) return (uint32_t)p[0] | ((uint32_t)p[2 * kResChunk] << 8);
    else if constexpr (COLS == 2) return *reinterpret_cast<const uint16_t *>(p);
    else return p[0];
  }
};

// Columns between the first lane computing one and the last lane storing it,
// in blocks of 16 (the store is one step behind the last lane's).
template <int COLS>
constexpr int kStoreLagBlocks = 32 * COLS / kColBlock;

// Sweep a band over nreal blocks of columns.  ln: the lane's rows (BandLane, or
// a class with its step(), outH and outF).  rgb: the two slots of 16 (H, F)
// entries of the band above, both holding the matrix top boundary (0, F0) on
// entry.  Io passes the rows between bands:
//   prev, next      a band above / below
//   load()          start loading the next block's entries (lanes 0..15)
//   land(slot)      wait for them and unpack them into rgb slot; false: timed out
//   room(wblk)      wait until block wblk of the own ring may be written; false: timed out
//   out(wblk), lo_bias, hi_bias   where block wblk goes; what an entry's words
//                   are on top of H and F
//   done(wblk)      block wblk has been written
// U: steps unrolled.  MASK: a lane whose rows start a sequence takes (in & keepH) and (in & keepH)
// | addF in place of the row above.  Returns false when a wait expired.
template <int FORM, int COLS, int U, bool MASK, class Prof, class Lane, class Res, class Io>
__device__ __forceinline__ bool band_sweep(Lane &ln, Res &rs, Io &io, uint2 *rgb,
                                           const uint8_t *prow, const int stride, const int lane, const int nreal,
                                           const Word<FORM> keepH, const Word<FORM> addF, const Consts &cs,
                                           int32_t *status) {
  using W = Word<FORM>;
  constexpr int kSteps = kColBlock / COLS;
  static_assert(kSteps % U == 0, "whole blocks");
  constexpr int kChunkBlocks = kResChunk / kColBlock;
  const uint32_t F0 = FORM != kFormInt32 ? cs.F0W : 0u;
  const int src = lane > 0 ? lane - 1 : lane;
  const bool lead = lane == 0;
  const int nblk = nreal + kStoreLagBlocks<COLS>;
  if (io.prev && nreal > 0) {
    io.load();
    if (!io.land(0)) return false;
  }
  cp_async_wait<0>();  // the first chunk of residues, staged by the caller
  __syncwarp();
  uint32_t res = Prof::checked(lead ? rs.template at<COLS>(0) : (uint32_t)kPadCode * 0x0101u, status);
  Prof pw;
  pw.load(prow, stride, res);
  for (int blk = 0; blk < nblk; ++blk) {
    // the block of the ring that this block's steps store
    const int wblk = blk - kStoreLagBlocks<COLS>;
    const bool writes = io.next && wblk >= 0;  // (and below nreal: nblk ends there)
    if (writes && !io.room(wblk)) return false;
    // the next chunk of residues: staged half-way through this one, waited
    // for before its last block (whose last step takes the next chunk's first)
    if (blk % kChunkBlocks == kChunkBlocks / 2) rs.stage(blk / kChunkBlocks + 1);
    if (blk % kChunkBlocks == kChunkBlocks - 1) {
      cp_async_wait<0>();
      __syncwarp();
    }
    const uint2 *gslot = rgb + (blk & 1) * kColBlock;
    const bool more = io.prev && blk + 1 < nreal;
    unsigned long long *wp = io.out(writes ? wblk : 0);
    const bool tail = writes && lane == 31;
    uint2 g[COLS];
    auto entry = [&](int s, uint2 (&e)[COLS]) {
      if constexpr (COLS == 2) {
        const uint4 v = reinterpret_cast<const uint4 *>(gslot)[s & (kSteps - 1)];
        e[0] = make_uint2(v.x, v.y);
        e[1] = make_uint2(v.z, v.w);
      } else {
        e[0] = gslot[s & (kSteps - 1)];
      }
    };
    entry(0, g);
    if (more) io.load();
#pragma unroll 1
    for (int part = 0; part < kSteps / U; ++part) {
#pragma unroll
      for (int s4 = 0; s4 < U; ++s4) {
        const int s = part * U + s4;
        const int col = blk * kColBlock + s * COLS;
        // the last step's bottom row (lane 31: a column of the ring's block wblk)
        if (tail) {
          if constexpr (COLS == 2)
            st_relaxed_2xu64(wp + 2 * s, (uint32_t)ln.outH[0] + io.lo_bias, (uint32_t)ln.outF[0] + io.hi_bias,
                             (uint32_t)ln.outH[1] + io.lo_bias, (uint32_t)ln.outF[1] + io.hi_bias);
          else
            st_relaxed_u64(wp + s, ((unsigned long long)((uint32_t)ln.outF[0] + io.hi_bias) << 32) |
                                       ((uint32_t)ln.outH[0] + io.lo_bias));
        }
        W inH[COLS], inF[COLS];
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
          inH[c] = (W)__shfl_sync(0xffffffffu, ln.outH[c], src);
          inF[c] = (W)__shfl_sync(0xffffffffu, ln.outF[c], src);
        }
        uint32_t resN = __shfl_sync(0xffffffffu, res, src);
        const uint32_t res0 = rs.template at<COLS>(col + COLS);
        uint2 gN[COLS];
        entry(s + 1, gN);
        if (lead) resN = res0;
        resN = Prof::checked(resN, status);
        Prof pwN;
        pwN.load(prow, stride, resN);
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
          inH[c] = lead ? (W)g[c].x : inH[c];
          inF[c] = lead ? (W)g[c].y : inF[c];
          if constexpr (MASK) {
            inH[c] = (W)((uint32_t)inH[c] & (uint32_t)keepH);
            inF[c] = (W)(((uint32_t)inF[c] & (uint32_t)keepH) | (uint32_t)addF);
          }
        }
        ln.step(pw, inH, inF, cs);
        res = resN;
        pw = pwN;
#pragma unroll
        for (int c = 0; c < COLS; ++c) g[c] = gN[c];
      }
    }
    if (writes) io.done(wblk);
    if (more) {
      if (!io.land((blk + 1) & 1)) return false;
    } else if (io.prev && blk + 1 < nblk) {
      // the padding blocks after the last real one: the top boundary again
      if (lane < kColBlock) rgb[((blk + 1) & 1) * kColBlock + lane] = make_uint2(0u, F0);
      __syncwarp();
    }
  }
  return true;
}

// Both boundary slots as the matrix top boundary (a band without a band above
// keeps it, the others overwrite them block by block).
__device__ __forceinline__ void clear_slots(uint2 *rgb, int lane, uint32_t F0) {
  rgb[lane] = make_uint2(0u, F0);  // 2 x 16 entries, one per lane
  __syncwarp();
}

// Rings written once (band-stream and transposed jobs): one entry per column,
// zeroed before the launch, (H | 1 << 31, F).  H is below 2^31 (int32: bounded
// by the host; 16-bit halves: both non-negative), so bit 31 tells a written
// entry, and entries need no other flag or fence.
// STRIDE: entries from one block of 16 columns to the next.
template <int STRIDE = kColBlock>
struct OnceRing {
  const unsigned long long *in;  // at the first column, or nullptr
  unsigned long long *own;       // at the first column, or nullptr
  uint2 *rgb;
  int lane;
  const unsigned long long *base;  // the ring buffer and its size (checked build)
  int64_t entries;
  int32_t *status;
  bool prev, next;
  uint32_t lo_bias = 0x80000000u, hi_bias = 0u;
  unsigned long long pend = 0ull;
  long long budget = kWaitBudgetCycles;  // of a wait

  __device__ __forceinline__ bool fresh() const { return (pend >> 31 & 1ull) != 0ull; }
  __device__ __forceinline__ void load() {
    if (lane < kColBlock && in_range(in - base + lane, entries, status)) pend = ld_relaxed_u64(in + lane);
  }
  __device__ __forceinline__ bool land(int slot) {
    bool ok = lane >= kColBlock || fresh();
    if (!__all_sync(0xffffffffu, ok)) {
      const long long t0 = clock64();
      do {
        if (__any_sync(0xffffffffu, clock64() - t0 > budget)) {
          if (lane == 0) atomicExch(status, SW_ETIMEOUT);
          return false;
        }
        if (!ok) {
          __nanosleep(32);  // (a waiting band leaves the issue slots to the bands that compute)
          load();
          ok = fresh();
        }
      } while (!__all_sync(0xffffffffu, ok));
    }
    if (lane < kColBlock)
      rgb[slot * kColBlock + lane] = make_uint2((uint32_t)pend & 0x7fffffffu, (uint32_t)(pend >> 32));
    in += STRIDE;
    pend = 0ull;
    __syncwarp();
    return true;
  }
  __device__ __forceinline__ bool room(int wblk) {
    // (every column has a place of its own; the checked build tests that)
    return in_range(own - base + (int64_t)wblk * STRIDE + kColBlock - 1, entries, status);
  }
  __device__ __forceinline__ unsigned long long *out(int wblk) const { return own + (int64_t)wblk * STRIDE; }
  __device__ __forceinline__ void done(int) {}
};

}  // namespace swgb
