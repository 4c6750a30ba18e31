// Cell arithmetic shared by the inter-task and intra-task kernels:
// one column step of R query rows owned by one lane (Sec. 2.2 Eqs. 1-3), or,
// with split lanes, the lane's two halves of R/2 rows a column apart.
//
// int32 form: one cell per lane op.
// packed form: two cells per 32-bit word, each 16-bit half a signed cell value.
// On sm_103 the integer ALU pipe (which executes every maximum and PRMT)
// issues a warp instruction every second cycle, whether a maximum has two
// inputs, three, or an addition fused to it; the FMA pipe is a second pipe
// that executes the per-half 16x2 adds (__vadd2 / __vsub2) and the byte dot
// products, also every second cycle.  So a cell's cost is its instructions on
// the ALU pipe: 3.5 (one three-input maximum for H, the zero floor of Eq. 1
// free in it, an add-maximum each for E and F, half a three-input maximum for
// the running best).  Per-half adds never carry into the other half; a half
// whose running score exceeds 32767 - max(SM) may have wrapped and is
// recomputed in int32.
#pragma once

#include <cstdint>
#include <type_traits>

#include "internal.h"

namespace swgb {

constexpr uint32_t kPadPair = 20u | (20u << 16);

// Checked build (-DSW_CHECK): every index into a packed residue buffer, a
// profile, a boundary strip or ring, or an output is tested before the
// access; an index outside its buffer records kStatusBounds in the status
// word and the access is skipped (no trap, no assert).  The regular build
// compiles the tests away.
#ifdef SW_CHECK
constexpr bool kChecked = true;
#else
constexpr bool kChecked = false;
#endif

__device__ __forceinline__ bool in_range(int64_t i, int64_t n, int32_t *status) {
  if constexpr (kChecked) {
    if (i < 0 || i >= n) {
      atomicExch(status, kStatusBounds);
      return false;
    }
  }
  return true;
}

// Profile row codes of a column (0..20, 20 = pad), as the form reads them:
// the low byte (int32 forms), the two 16-bit halves (two sequences per word)
// or the whole word (query pairs, one bare code).  A code past the pad row is
// reported and replaced by the pad code.
template <int FORM>
__device__ __forceinline__ uint32_t checked_codes(uint32_t res, int32_t *status) {
  if constexpr (kChecked) {
    bool bad;
    if constexpr (FORM == kFormPacked) bad = (res & 0xffffu) > (uint32_t)kPadCode || (res >> 16) > (uint32_t)kPadCode;
    else if constexpr (FORM == kFormQPair) bad = res > (uint32_t)kPadCode;
    else bad = (res & 0xffu) > (uint32_t)kPadCode;
    if (bad) {
      atomicExch(status, kStatusBounds);
      return FORM == kFormPacked ? kPadPair : (uint32_t)kPadCode;
    }
  }
  return res;
}

struct Consts {
  // packed: (x, x) in both 16-bit halves; F0W: E and F of the boundaries
  uint32_t goW, geW, F0W;
  // int32
  int32_t go, ge;
};

template <int GAPS = kGapsAny>
__device__ __forceinline__ Consts make_consts(const Scoring &sc) {
  const int32_t go = GAPS == kGapsProtein ? kProteinGo : GAPS == kGapsDna ? kDnaGo : sc.go;
  const int32_t ge = GAPS == kGapsProtein ? kProteinGe : GAPS == kGapsDna ? kDnaGe : sc.ge;
  Consts c;
  c.goW = (uint32_t)go * 0x10001u;
  c.geW = (uint32_t)ge * 0x10001u;
  const uint32_t ngo = (uint32_t)(-go) & 0xffffu;  // E, F start at -Go (any value <= 0 works)
  c.F0W = ngo | (ngo << 16);
  c.go = go;
  c.ge = ge;
  return c;
}

// PTX prmt.b32 (default mode): each selector nibble picks one of the 8 bytes
// {b, a}; a set nibble msb replicates the sign of the picked byte instead.
// (CUDA's __byte_perm masks the nibbles to 3 bits, so it cannot express the
// sign-replicate form used here.)
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

// Selectors.  pair(i) -> (byte i of a, its sign, byte i of b, its sign): the two
// bytes sign-extended into the 16-bit halves (residue codes < 128 come out
// zero-extended).  one(i) -> byte i of a, zero-extended from b = 0.
__host__ __device__ constexpr uint32_t sel_pair(int i) {
  return (uint32_t)i | ((uint32_t)(i | 8) << 4) | ((uint32_t)(4 + i) << 8) | ((uint32_t)((4 + i) | 8) << 12);
}
__host__ __device__ constexpr uint32_t sel_one(int i) { return 0x4440u | (uint32_t)i; }

template <int R>
__device__ __forceinline__ void load_prof(const uint8_t *p, uint32_t (&w)[R / 4]) {
  static_assert(R % 4 == 0, "rows per lane must be a multiple of 4");
  if constexpr (R % 16 == 0) {
#pragma unroll
    for (int i = 0; i < R / 16; ++i) {
      const uint4 v = reinterpret_cast<const uint4 *>(p)[i];
      w[4 * i + 0] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
    }
  } else if constexpr (R % 8 == 0) {
#pragma unroll
    for (int i = 0; i < R / 8; ++i) {
      const uint2 v = reinterpret_cast<const uint2 *>(p)[i];
      w[2 * i + 0] = v.x; w[2 * i + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < R / 4; ++i) w[i] = reinterpret_cast<const uint32_t *>(p)[i];
  }
}

// N profile bytes at byte OFF of an 8-byte-aligned slot, as N/4 words, by the
// widest aligned loads (the halves of a 24-byte slot start at 0 and 12).
template <int N, int OFF, int W = 0>
__device__ __forceinline__ void load_prof_at(const uint8_t *p, uint32_t (&w)[N / 4]) {
  static_assert(N % 4 == 0 && OFF % 4 == 0, "whole words");
  constexpr int b = 4 * W;
  if constexpr (b < N) {
    if constexpr ((OFF + b) % 8 == 0 && b + 8 <= N) {
      const uint2 v = *reinterpret_cast<const uint2 *>(p + OFF + b);
      w[W] = v.x;
      w[W + 1] = v.y;
      load_prof_at<N, OFF, W + 2>(p, w);
    } else {
      w[W] = *reinterpret_cast<const uint32_t *>(p + OFF + b);
      load_prof_at<N, OFF, W + 1>(p, w);
    }
  }
}

__device__ __forceinline__ uint32_t word_of(const uint4 &v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

// N rows [R0, R0 + N) of one column, 32-bit words of two 16-bit cells
// (Eqs. 1-3 per half).  hd0 is H of the row above R0 at the previous column,
// p the rows' substitution words; E (per row, this column) and f (passed down
// the column) are updated in place, S keeps the running best.
//
// Per word: H = max(H_diag + SM, E, F, 0) is one three-input maximum with the
// zero floor, the E and F updates one add-maximum each, and the running best
// one three-input maximum per two rows: 3.5 instructions on the ALU pipe
// (each a warp instruction every second cycle, three-input or not); H_diag +
// SM and H - Go (shared by E and F) are per-half adds on the FMA pipe.  All
// H_diag + SM are formed first: the previous column's H is then dead before
// any row is rewritten (forming them row by row costs a register copy each).
// Two-input maxima throughout (5 on the ALU pipe) took 10.3 cycles per word
// and SM sub-partition in a loop over 24 rows and four warps, this 9.1 (the
// ALU pipe 79 % busy; register operands, up to three per instruction, are the
// rest; 8.4-8.7 with the penalties as immediates), and the same formed row by
// row 10.2-10.6.  The running best is taken after the rows, as two chains:
// inside the row loop the two-sequence form took 71.5 ms instead of 67.0 (20
// queries x 40,000 proteins), query pairs the same.
template <int R0, int N, int R>
__device__ __forceinline__ void word_rows(uint32_t hd0, const uint32_t (&p)[N], uint32_t (&E)[R],
                                          uint32_t (&Hl)[R], uint32_t &f, uint32_t &S, const Consts &cs) {
  static_assert(R0 + N <= R && N % 2 == 0, "rows in range, whole pairs of rows");
  uint32_t x[N];
#pragma unroll
  for (int r = 0; r < N; ++r) x[r] = __vadd2(r > 0 ? Hl[R0 + r - 1] : hd0, p[r]);
#pragma unroll
  for (int r = 0; r < N; ++r) {
    const uint32_t h = __vimax3_s16x2_relu(x[r], E[R0 + r], f);  // max(H_diag + SM, E, F, 0)
    const uint32_t hgo = __vsub2(h, cs.goW);
    E[R0 + r] = __vmaxs2(__vsub2(E[R0 + r], cs.geW), hgo);
    f = __vmaxs2(__vsub2(f, cs.geW), hgo);
    Hl[R0 + r] = h;
  }
  constexpr int N2 = N / 2;
  uint32_t a = Hl[R0], b = Hl[R0 + N2];
#pragma unroll
  for (int r = 1; r + 1 < N2; r += 2) {
    a = __vimax3_s16x2(a, Hl[R0 + r], Hl[R0 + r + 1]);
    b = __vimax3_s16x2(b, Hl[R0 + N2 + r], Hl[R0 + N2 + r + 1]);
  }
  if constexpr (N2 % 2 == 0) a = __vimax3_s16x2(a, Hl[R0 + N2 - 1], Hl[R0 + N - 1]);
  S = __vimax3_s16x2(S, a, b);
}

template <int FORM>
using Word = typename std::conditional<FORM != kFormInt32, uint32_t, int32_t>::type;

// The rows of word_rows in int32 cells (Algorithm 1, one cell per lane op).
// add(r, h): h plus the substitution score of row R0 + r.
// Per cell 3.5 instructions on the ALU pipe like a word of word_rows; the
// score is added by a byte dot product (FMA pipe), which sign-extends it on
// the way.  Statement by statement with two-input maxima and a byte
// extraction on the ALU pipe: 11.3 cycles per cell and SM sub-partition in a
// loop over 24 rows and four warps; three-input maxima 9.45; with the dot
// product 7.9 (the ALU pipe 89 % busy).
template <int R0, int N, int R, class Add>
__device__ __forceinline__ void int_rows_of(int32_t hd0, Add add, int32_t (&E)[R], int32_t (&Hl)[R], int32_t &f,
                                            int32_t &S, const Consts &cs) {
  static_assert(R0 + N <= R && N % 2 == 0, "rows in range, whole pairs of rows");
  int32_t x[N];
#pragma unroll
  for (int r = N - 1; r >= 0; --r) x[r] = add(r, r > 0 ? Hl[R0 + r - 1] : hd0);
#pragma unroll
  for (int r = 0; r < N; ++r) {
    const int32_t h = __vimax3_s32_relu(x[r], E[R0 + r], f);  // max(H_diag + SM, E, F, 0)
    const int32_t hgo = h - cs.go;
    E[R0 + r] = max(E[R0 + r] - cs.ge, hgo);
    f = max(f - cs.ge, hgo);
    Hl[R0 + r] = h;
    if (r & 1) S = __vimax3_s32(S, Hl[R0 + r - 1], h);
  }
}

// h plus profile byte r (signed) of pb: the dot product with a one in that byte
template <int W>
__device__ __forceinline__ int32_t add_byte(const uint32_t (&pb)[W], int r, int32_t h) {
  return __dp4a((int32_t)pb[r >> 2], 1 << (8 * (r & 3)), h);
}


// Per-lane DP state of R rows.
template <int R, int FORM>
struct LaneState {
  Word<FORM> Hl[R];  // H of each row at the previous column
  Word<FORM> E[R];   // E of each row at the current column
  Word<FORM> hdiag;  // H of the row above this lane's first row, previous column
};

template <int R, int FORM>
__device__ __forceinline__ void lane_reset(LaneState<R, FORM> &st, const Consts &cs) {
  using W = Word<FORM>;
  constexpr bool PACKED = FORM != kFormInt32;
  const W E0 = PACKED ? (W)cs.F0W : (W)0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    st.Hl[r] = (W)0;
    st.E[r] = E0;
  }
  st.hdiag = (W)0;
}

// One column: inputs are the (H, F) pair passed down from the row above this
// lane's rows and the residue code(s) of the column; prow points at this
// lane's R profile entries of residue row 0 (rows are `stride` bytes apart).
// Query-pair form: res is the bare residue code (no second code in the high
// half); prow points at this lane's first 16-byte group of four words; its
// R/4 groups are `gstride` bytes apart (lanes interleaved, so the
// 32 lanes of a warp read 32 consecutive 16-byte groups: no bank conflict).
// Outputs the (H, F) pair for the row below: H of the last row, F of the row
// below it.
template <int R, int FORM>
__device__ __forceinline__ void column_step(LaneState<R, FORM> &st, const uint8_t *prow, int stride,
                                            uint32_t res, Word<FORM> inH, Word<FORM> inF, const Consts &cs,
                                            Word<FORM> &S, Word<FORM> &outH, Word<FORM> &outF, int gstride = 0) {
  using W = Word<FORM>;
  if constexpr (FORM == kFormQPair) {
    // the two queries' scores for this column's residue, one word per row
    uint32_t pw[R];
#pragma unroll
    for (int i = 0; i < R / 4; ++i) {
      const uint4 v = *reinterpret_cast<const uint4 *>(prow + res * stride + i * gstride);
      pw[4 * i + 0] = v.x; pw[4 * i + 1] = v.y; pw[4 * i + 2] = v.z; pw[4 * i + 3] = v.w;
    }
    uint32_t f = (uint32_t)inF, s = (uint32_t)S;
    word_rows<0, R>((uint32_t)st.hdiag, pw, st.E, st.Hl, f, s, cs);
    S = (W)s;
    outH = st.Hl[R - 1];
    outF = (W)f;
  } else if constexpr (FORM == kFormPacked) {
    uint32_t pw[R];
    uint32_t pa[R / 4], pb[R / 4];
    load_prof<R>(prow + (res & 0xffu) * stride, pa);
    load_prof<R>(prow + (res >> 16) * stride, pb);
#pragma unroll
    for (int r = 0; r < R; ++r) pw[r] = prmt(pa[r >> 2], pb[r >> 2], sel_pair(r & 3));  // (SM_a, SM_b), signed halves
    uint32_t f = (uint32_t)inF, s = (uint32_t)S;
    word_rows<0, R>((uint32_t)st.hdiag, pw, st.E, st.Hl, f, s, cs);
    S = (W)s;
    outH = st.Hl[R - 1];
    outF = (W)f;
  } else {
    int32_t f = inF, s = S;
    uint32_t pa[R / 4];
    load_prof<R>(prow + (res & 0xffu) * stride, pa);
    int_rows_of<0, R, R>(st.hdiag, [&](int r, int32_t h) { return add_byte(pa, r, h); }, st.E, st.Hl, f, s, cs);
    S = (W)s;
    outH = st.Hl[R - 1];
    outF = (W)f;
  }
  st.hdiag = inH;
}

// 16-bit forms with two independent half-chains per lane: rows [0, R/2) at
// column c and rows [R/2, R) at column c - 1, one step behind, so that the
// two F/H dependency chains down the rows interleave.  The upper half's F
// output and its bottom H feed the lower half one step later (midF, hdiagB);
// the lane passes on the lower half's bottom row, of column c - 1, so lane
// k + 1 works two columns behind lane k.  resA / resB: the residue code(s) of
// column c / c - 1.  S and S2 keep the halves' running best.
template <int R, int FORM>
__device__ __forceinline__ void column_step_split(LaneState<R, FORM> &st, uint32_t &hdiagB, uint32_t &midF,
                                                  const uint8_t *prow, int stride, uint32_t resA, uint32_t resB,
                                                  uint32_t inH, uint32_t inF, const Consts &cs, uint32_t &S,
                                                  uint32_t &S2, uint32_t &outH, uint32_t &outF, int gstride) {
  static_assert(FORM != kFormInt32 && R % 8 == 0, "16-bit forms, halves of whole 4-row groups");
  constexpr int H2 = R / 2;
  // substitution words of the upper half (column c) and the lower half (column c - 1)
  uint32_t pa[H2], pb[H2];
  if constexpr (FORM == kFormQPair) {
#pragma unroll
    for (int i = 0; i < H2 / 4; ++i) {
      const uint4 v = *reinterpret_cast<const uint4 *>(prow + resA * stride + i * gstride);
      pa[4 * i + 0] = v.x; pa[4 * i + 1] = v.y; pa[4 * i + 2] = v.z; pa[4 * i + 3] = v.w;
      const uint4 w = *reinterpret_cast<const uint4 *>(prow + resB * stride + (H2 / 4 + i) * gstride);
      pb[4 * i + 0] = w.x; pb[4 * i + 1] = w.y; pb[4 * i + 2] = w.z; pb[4 * i + 3] = w.w;
    }
  } else {
    // two database sequences: each word pairs their profile bytes by a byte
    // shuffle (ALU pipe).  32-bit entries paired by a multiply-add on the FMA
    // pipe take two shared-memory wavefronts per word, of the one per cycle
    // that an SM has for its four sub-partitions, and measured slower: 4,974
    // against 5,242 GCUPS, one 400-residue query x 200,000 proteins.
    uint32_t a0[H2 / 4], a1[H2 / 4], b0[H2 / 4], b1[H2 / 4];
    load_prof_at<H2, 0>(prow + (resA & 0xffu) * stride, a0);
    load_prof_at<H2, 0>(prow + (resA >> 16) * stride, a1);
    load_prof_at<H2, H2>(prow + (resB & 0xffu) * stride, b0);
    load_prof_at<H2, H2>(prow + (resB >> 16) * stride, b1);
#pragma unroll
    for (int r = 0; r < H2; ++r) {
      pa[r] = prmt(a0[r >> 2], a1[r >> 2], sel_pair(r & 3));
      pb[r] = prmt(b0[r >> 2], b1[r >> 2], sel_pair(r & 3));
    }
  }
  const uint32_t diagB_next = st.Hl[H2 - 1];  // H of the upper half's last row at column c - 1
  // lower half first in program order (its inputs are ready), then the upper
  uint32_t f = midF, s2 = S2;
  word_rows<H2, H2>(hdiagB, pb, st.E, st.Hl, f, s2, cs);
  outH = st.Hl[R - 1];
  outF = f;
  S2 = s2;
  f = inF;
  uint32_t s = S;
  word_rows<0, H2>(st.hdiag, pa, st.E, st.Hl, f, s, cs);
  S = s;
  midF = f;
  hdiagB = diagB_next;
  st.hdiag = inH;
}

// int32 form with split lanes (the intra-task kernel): as
// column_step_split, with byte profiles.
template <int R>
__device__ __forceinline__ void column_step_split_int(LaneState<R, kFormInt32> &st, int32_t &hdiagB, int32_t &midF,
                                                      const uint8_t *prow, int stride, uint32_t resA, uint32_t resB,
                                                      int32_t inH, int32_t inF, const Consts &cs, int32_t &S,
                                                      int32_t &S2, int32_t &outH, int32_t &outF) {
  static_assert(R % 8 == 0, "halves of whole profile words");
  constexpr int H2 = R / 2;
  uint32_t pa[H2 / 4], pb[H2 / 4];
  load_prof_at<H2, 0>(prow + (resA & 0xffu) * stride, pa);
  load_prof_at<H2, H2>(prow + (resB & 0xffu) * stride, pb);
  const int32_t diagB_next = st.Hl[H2 - 1];  // H of the upper half's last row at column c - 1
  // lower half first in program order (its inputs are ready), then the upper
  int32_t f = midF, s2 = S2;
  int_rows_of<H2, H2, R>(hdiagB, [&](int r, int32_t h) { return add_byte(pb, r, h); }, st.E, st.Hl, f, s2, cs);
  outH = st.Hl[R - 1];
  outF = f;
  S2 = s2;
  f = inF;
  int32_t s = S;
  int_rows_of<0, H2, R>(st.hdiag, [&](int r, int32_t h) { return add_byte(pa, r, h); }, st.E, st.Hl, f, s, cs);
  S = s;
  midF = f;
  hdiagB = diagB_next;
  st.hdiag = inH;
}

template <int FORM>
__device__ __forceinline__ Word<FORM> score_max(Word<FORM> a, Word<FORM> b) {
  if constexpr (FORM != kFormInt32) return (Word<FORM>)__vmaxs2((uint32_t)a, (uint32_t)b);
  else return max(a, b);
}

// Epilogue for one database unit: flag possible overflows (packed) and scatter
// to caller order.  (The query-pair form writes its scores per query-track
// chunk, in the inter-task kernel.)
template <int FORM>
__device__ __forceinline__ void write_scores(Word<FORM> S, int posA, int posB, int q, const QDesc &qd,
                                             const InterArgs &a) {
  static_assert(FORM != kFormQPair, "query-pair scores are written per track chunk");
  constexpr bool PACKED = FORM == kFormPacked;
  const DbView &db = a.db;
  const Scoring &sc = a.sc;
  int32_t *out = a.out;
  int32_t *flag_count = a.flag_count;
  int32_t *flag_pos = a.flag_pos;
  const int64_t row = (int64_t)q * a.out_stride;
  const int64_t frow = (int64_t)q * a.flag_stride;
  if (!in_range(posA, db.n, a.status) || !in_range(posB, db.n, a.status)) return;
  if constexpr (PACKED) {
    const int32_t sa = (int32_t)((uint32_t)S & 0xffffu), sb = (int32_t)((uint32_t)S >> 16);
    if (sa > sc.thresh) {
      const int i = atomicAdd(&flag_count[q], 1);
      if (in_range(frow + i, a.flag_size, a.status)) flag_pos[frow + i] = posA;
    }
    if (in_range(row + db.perm[posA], a.out_size, a.status)) out[row + db.perm[posA]] = sa;
    if (posB != posA) {
      if (sb > sc.thresh) {
        const int i = atomicAdd(&flag_count[q], 1);
        if (in_range(frow + i, a.flag_size, a.status)) flag_pos[frow + i] = posB;
      }
      if (in_range(row + db.perm[posB], a.out_size, a.status)) out[row + db.perm[posB]] = sb;
    }
  } else {
    if (in_range(row + db.perm[posA], a.out_size, a.status)) out[row + db.perm[posA]] = (int32_t)S;
  }
}

}  // namespace swgb
