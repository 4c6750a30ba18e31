// Pair-band kernel: one long (query, target) pair, int32 cells (the pairwise
// alignment of two long sequences, Sec. 2.2 case (a); Fig. 1 intra-sequence
// parallelism).  Band b is query rows [32 R b, 32 R (b+1)): one warp is a
// chain of 32 lanes of R rows (the inter-task chain of k_inter.cu) that sweeps
// every target column.  Warp w of the grid takes bands w, w + warps, ... in
// order (warps numbered across the SMs first, so that even a few bands per SM
// land on every SM); a band's top boundary is the bottom row of the band
// above, read from that band's ring as soon as the entries are there, so the
// bands run as a pipeline over every warp of every SM.  All warps are resident (cooperative
// launch), a band waits only on the band above (data) and on the band below
// (room in its ring), and every wait is bounded.
//
// Boundary rings
// --------------
// Band b writes its bottom row to ring b mod nslots, `window` columns long
// (column j at j mod window).  An entry is one 64-bit word written by one
// relaxed store, so the band below can tell a fresh entry from the one it
// replaces by two tag bits, with no flag and no fence on the producer's side:
//   low word  = H | (lap parity << 31)            lap = j / window
//   high word = (F + Go) | (generation bit << 31)  generation = b / nslots,
//                                                  bit = its parity inverted
// A location holds either the entry the reader waits for or the one written
// before it there: the previous lap of the same band (other lap parity) or the
// last lap of the band that used the ring before (other generation parity), or
// zeros (generation bit 0, which no band of generation 0 writes).  The reader
// hands consumed columns back through a counter (release/acquire), so a band
// never overwrites an entry that the band below has not read.  H lies in
// [0, 2^31 - Go) (the host bounds the scores) and F, that of the row below, in
// [-Go, H] (max(F - Ge, H - Go) with F <= H and H >= 0), so both fields fit 31
// bits.
#include "devutil.cuh"
#include "dp_common.cuh"
#include "internal.h"
#include "../../include/swgb.h"

namespace swgb {
namespace {

// Columns per step.  A lane computes two columns of its R rows in one step:
// the step's fixed cost (the shuffles' latency, the first lane's selects, the
// hand-off to the band below) is paid once for both, and the second column's
// chain down the rows runs one row behind the first one's, so that a warp
// that has its SM sub-partition to itself has two chains to interleave.  In a
// loop over one warp per sub-partition a two-column step takes 180 cycles at R
// = 8 and 316 at R = 16, in a band between two others 244 and 378.
constexpr int kStepCols = 2;
constexpr int kBlockSteps = kColBlock / kStepCols;
// A band's last lane works on columns 62 and 63 behind the first lane's and
// stores them one step later, at the start of its next step: 64 columns, four
// blocks, so that the columns it stores in one block are a block of the ring.
constexpr int kBandLagBlocks = 4;
constexpr int kResChunk = 512;                              // target residues staged at a time (16 per lane)
constexpr int kBandRingBytes = 2 * kResChunk + 2 * kColBlock * 8;  // per warp: residues, boundary entries
// At most this many warps per CTA, one CTA per SM: two per SM sub-partition,
// with up to 255 registers a thread.  (Sixteen warps of 128 registers: 473
// against 380 cycles per step at R = 16; a pair long enough for more warps
// gets taller bands instead, which measured faster: 1M x 1M 273 ms at R = 28
// and two warps, 283 at R = 20 and three, 284 at R = 14 and four.)
constexpr int kPairWarps = 8;
// Steps unrolled: a whole block where its code fits the instruction cache, half
// of one above (R = 8: 269 -> 244 cycles per step, R = 20: 478 -> 660).
template <int R>
constexpr int kUnrolled = R <= 16 ? kBlockSteps : kBlockSteps / 2;
template <int R>
constexpr int kSlotBytes = (R + 3) / 4 * 4;  // profile bytes of a lane

struct BandIO {
  const unsigned long long *in;  // ring of the band above
  unsigned long long *out;       // this band's ring
  int32_t *cons_in;              // columns of `in` consumed, published for the band above
  const int32_t *cons_out;       // columns of `out` consumed by the band below
  int32_t window;
  uint32_t gen_in, gen_out;      // generation tag bits of the two rings (0 or 1)
  int32_t cons_every;            // blocks between publications of cons_in
  int32_t *status;
};

__device__ __forceinline__ uint32_t band_gen(int b, int nslots) { return ((uint32_t)(b / nslots) & 1u) ^ 1u; }

// The profile bytes of a lane's R rows, as words.
template <int R>
__device__ __forceinline__ void load_rows(const uint8_t *p, uint32_t (&w)[kSlotBytes<R> / 4]) {
  if constexpr (R % 4 == 0) {
    load_prof<R>(p, w);
  } else {
#pragma unroll
    for (int i = 0; i < kSlotBytes<R> / 4; ++i) w[i] = reinterpret_cast<const uint32_t *>(p)[i];
  }
}

// One band over all target columns.  Each lane passes its bottom row (H and F
// of both columns) and the residues to the next lane by shuffle; the first
// lane takes the residues from shared memory (staged 512 at a time, a chunk
// ahead, by the whole warp) and the band above's entries from its slot there.
// Residues, profile words and boundary entries of a step are fetched during
// the step before, off the chain.  Lanes 0..15 load the next block's entries
// during a block and check their tags at its end (loading again until they
// are fresh).  Lane 31 stores its two columns with one 128-bit store at the
// start of the next step, each 64-bit half an entry of its own.
// (Per block instead, 16 entries through shared memory, residues two blocks
// ahead by the first lane and a vote on the room in the ring: 326 against 244
// cycles per step of a band between two others, R = 8.)
// Returns false when a wait expired.
template <int R>
__device__ __forceinline__ bool band_pass(const uint8_t *__restrict__ pch, const int stride, const int lane,
                                          const int npad, const uint8_t *__restrict__ target, uint8_t *ring,
                                          const bool prev, const bool next, const Consts &cs, int32_t &Sout,
                                          const BandIO &x) {
  constexpr int PW = kSlotBytes<R> / 4;
  int32_t Hl[R], E[R];
#pragma unroll
  for (int r = 0; r < R; ++r) Hl[r] = E[r] = 0;
  int32_t outHA = 0, outFA = 0, outHB = 0, outFB = 0, hdiag = 0, S = 0;
  const int src = lane > 0 ? lane - 1 : lane;
  const bool lead = lane == 0;
  const int nreal = npad / kColBlock;  // blocks of real columns
  const int nblk = nreal + kBandLagBlocks;
  uint8_t *rres = ring;                                           // [2][512] residue codes
  uint2 *rgb = reinterpret_cast<uint2 *>(ring + 2 * kResChunk);  // [2 slots][16] (H, F) of the band above
  const uint8_t *prow = pch + lane * kSlotBytes<R>;
  bool failed = false;

  constexpr int kChunkBlocks = kResChunk / kColBlock;
  auto stage = [&](int chunk) {
    uint8_t *d = rres + (chunk & 1) * kResChunk + lane * 16;
    const int64_t col = (int64_t)chunk * kResChunk + lane * 16;
    if (col < npad) cp_async16(d, target + col);
    else *reinterpret_cast<uint4 *>(d) = make_uint4(0x14141414u, 0x14141414u, 0x14141414u, 0x14141414u);
    cp_async_commit();
  };
  __syncwarp();  // (the band before this one on the warp has read its residues)
  stage(0);

  // reading side: ring position and lap parity of the next block to load
  int rpos = 0, consumed = 0, since = 0;
  uint32_t rlap = 0u;
  unsigned long long pend = 0ull;
  auto load = [&]() {
    if (lane < kColBlock) pend = ld_relaxed_u64(x.in + rpos + lane);
  };
  auto fresh = [&](unsigned long long v) {
    return ((uint32_t)v >> 31) == rlap && (uint32_t)(v >> 63) == x.gen_in;
  };
  // wait until the loaded entries are fresh, unpack them into `slot`, advance
  auto land = [&](int slot) {
    bool ok = lane >= kColBlock || fresh(pend);
    long long t0 = 0;
    bool waited = false;
    while (!__all_sync(0xffffffffu, ok)) {
      if (!waited) {
        t0 = clock64();
        waited = true;
      }
      if (__any_sync(0xffffffffu, clock64() - t0 > kLongWaitBudgetCycles)) {
        failed = true;
        if (lead) atomicExch(x.status, SW_ETIMEOUT);
        return;
      }
      if (!ok) {
        pend = ld_relaxed_u64(x.in + rpos + lane);
        ok = fresh(pend);
      }
    }
    if (lane < kColBlock) {
      const int32_t h = (int32_t)((uint32_t)pend & 0x7fffffffu);
      const int32_t f = (int32_t)((uint32_t)(pend >> 32) & 0x7fffffffu) - cs.go;
      rgb[slot * kColBlock + lane] = make_uint2((uint32_t)h, (uint32_t)f);
    }
    consumed += kColBlock;
    rpos += kColBlock;
    if (rpos == x.window) {
      rpos = 0;
      rlap ^= 1u;
    }
    __syncwarp();
    // hand the columns back every few blocks and at the end (the release orders
    // the loads of lanes 0..15, which the warp barrier above ordered first)
    if (++since == x.cons_every || consumed == npad) {
      since = 0;
      if (lead) st_release(x.cons_in, consumed);
    }
  };
  // both boundary slots start as the matrix top boundary (the band without
  // a band above keeps it; the others overwrite block by block, and the
  // padding blocks at the end get it back below)
  if (lane < kColBlock) {
    rgb[lane] = make_uint2(0u, 0u);
    rgb[kColBlock + lane] = make_uint2(0u, 0u);
  }
  __syncwarp();
  if (prev) {
    load();
    land(0);
  }
  cp_async_wait<0>();
  __syncwarp();

  // writing side: this band's ring at the block being stored, its lap bit,
  // and the columns there is room for, as last read
  int wpos = 0, room = x.window;
  uint32_t lap_bit = 0u;
  const uint32_t f_bias = (uint32_t)cs.go + (x.gen_out << 31);

  // this step's residues (two codes) and profile words
  uint32_t res = lead ? (uint32_t)*reinterpret_cast<const uint16_t *>(rres)
                      : (uint32_t)(kPadCode | (kPadCode << 8));
  uint32_t pwA[PW], pwB[PW];
  load_rows<R>(prow + (res & 0xffu) * stride, pwA);
  load_rows<R>(prow + (res >> 8) * stride, pwB);

  for (int blk = 0; blk < nblk && !failed; ++blk) {
    // the block of the ring that this block stores (columns 64 behind)
    const int wblk = blk - kBandLagBlocks;
    const bool writes = next && wblk >= 0;  // (wblk < nreal: nblk is nreal + 4)
    if (writes && (wblk + 1) * kColBlock > room) {
      const int need = (wblk + 1) * kColBlock - x.window;
      int seen = 0;
      if (lead) seen = wait_flag_value(x.cons_out, need, kLongWaitBudgetCycles);
      seen = __shfl_sync(0xffffffffu, seen, 0);
      if (seen < need) {
        failed = true;
        if (lead) atomicExch(x.status, SW_ETIMEOUT);
        break;
      }
      // (no farther than the columns themselves: both terms stay in 32 bits)
      room = seen > npad - x.window ? npad : seen + x.window;
    }
    // the next chunk of residues: staged half-way through this one, waited
    // for before its last block (whose last step takes the next chunk's first)
    if (blk % kChunkBlocks == kChunkBlocks / 2) stage(blk / kChunkBlocks + 1);
    if (blk % kChunkBlocks == kChunkBlocks - 1) {
      cp_async_wait<0>();
      __syncwarp();
    }
    const uint4 *gslot = reinterpret_cast<const uint4 *>(rgb + (blk & 1) * kColBlock);
    const bool more = prev && blk + 1 < nreal;
    unsigned long long *wp = x.out + wpos;
    const bool tail = writes && lane == 31;
    uint4 g = gslot[0];
    if (more) load();
#pragma unroll 1
    for (int part = 0; part < kBlockSteps / kUnrolled<R>; ++part) {
#pragma unroll
      for (int s4 = 0; s4 < kUnrolled<R>; ++s4) {
        const int s = part * kUnrolled<R> + s4;
        const int t = blk * kBlockSteps + s;
        if (tail)
          st_relaxed_2xu64(wp + kStepCols * s, (uint32_t)outHA + lap_bit, (uint32_t)outFA + f_bias,
                           (uint32_t)outHB + lap_bit, (uint32_t)outFB + f_bias);
        const int32_t shHA = __shfl_sync(0xffffffffu, outHA, src);
        const int32_t shFA = __shfl_sync(0xffffffffu, outFA, src);
        const int32_t shHB = __shfl_sync(0xffffffffu, outHB, src);
        const int32_t shFB = __shfl_sync(0xffffffffu, outFB, src);
        uint32_t resN = __shfl_sync(0xffffffffu, res, src);
        const uint32_t res0 =
            *reinterpret_cast<const uint16_t *>(rres + ((kStepCols * t + kStepCols) & (2 * kResChunk - 1)));
        const uint4 gN = gslot[(s + 1) & (kBlockSteps - 1)];
        if (lead) resN = res0;
        uint32_t pwAN[PW], pwBN[PW];
        load_rows<R>(prow + (resN & 0xffu) * stride, pwAN);
        load_rows<R>(prow + (resN >> 8) * stride, pwBN);
        int32_t xA[R];  // H_diag + SM of the first column
#pragma unroll
        for (int r = R - 1; r >= 0; --r) xA[r] = add_byte(pwA, r, r > 0 ? Hl[r - 1] : hdiag);
        const int32_t inHA = lead ? (int32_t)g.x : shHA;
        int32_t fA = lead ? (int32_t)g.y : shFA;
        const int32_t inHB = lead ? (int32_t)g.z : shHB;
        int32_t fB = lead ? (int32_t)g.w : shFB;
        int32_t dB = inHA;  // H of the row above at the first column
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int32_t hA = __vimax3_s32_relu(xA[r], E[r], fA);  // Eq. 1, floor included
          const int32_t gA = hA - cs.go;
          const int32_t e = max(E[r] - cs.ge, gA);  // Eq. 2, the second column's E
          fA = max(fA - cs.ge, gA);                 // Eq. 3, the row below's F
          const int32_t hB = __vimax3_s32_relu(add_byte(pwB, r, dB), e, fB);
          const int32_t gB = hB - cs.go;
          E[r] = max(e - cs.ge, gB);
          fB = max(fB - cs.ge, gB);
          S = __vimax3_s32(S, hA, hB);
          Hl[r] = hB;
          dB = hA;
        }
        outHA = dB;
        outFA = fA;
        outHB = Hl[R - 1];
        outFB = fB;
        hdiag = inHB;
        res = resN;
        g = gN;
#pragma unroll
        for (int i = 0; i < PW; ++i) {
          pwA[i] = pwAN[i];
          pwB[i] = pwBN[i];
        }
      }
    }
    if (writes) {
      wpos += kColBlock;
      if (wpos == x.window) {
        wpos = 0;
        lap_bit ^= 0x80000000u;
      }
    }
    if (more) {
      land((blk + 1) & 1);
    } else if (prev && blk + 1 < nblk) {
      // the padding blocks after the last real one: top boundary again
      if (lane < kColBlock) rgb[((blk + 1) & 1) * kColBlock + lane] = make_uint2(0u, 0u);
      __syncwarp();
    }
  }
  cp_async_wait<0>();
  Sout = max(Sout, S);
  return !failed;
}

template <int R, int GAPS>
__global__ void __launch_bounds__(32 * kPairWarps, 1) pair_band_kernel(const PairBandArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  uint8_t *pbuf = smem + (size_t)warp * (a.pbuf_bytes + kBandRingBytes);
  uint8_t *ring = pbuf + a.pbuf_bytes;
  const Consts cs = make_consts<GAPS>(a.sc);
  int32_t S = 0;
  // global warp g = warp * grid + CTA: bands spread over the SMs first
  for (int b = warp * gridDim.x + blockIdx.x; b < a.nbands; b += gridDim.x * nw) {
    const uint4 *src = reinterpret_cast<const uint4 *>(a.prof + (int64_t)b * a.band_bytes);
    for (int i = lane; i < a.band_bytes / 16; i += 32) reinterpret_cast<uint4 *>(pbuf)[i] = __ldg(src + i);
    __syncwarp();
    BandIO x;
    x.in = a.strips + (size_t)((b + a.nslots - 1) % a.nslots) * a.window;
    x.out = a.strips + (size_t)(b % a.nslots) * a.window;
    x.cons_in = a.cons + (b > 0 ? b - 1 : 0);
    x.cons_out = a.cons + b;
    x.window = a.window;
    x.gen_in = band_gen(b > 0 ? b - 1 : 0, a.nslots);
    x.gen_out = band_gen(b, a.nslots);
    x.cons_every = a.cons_every;
    x.status = a.status;
    const bool ok = band_pass<R>(pbuf, a.stride, lane, a.npad, a.target, ring, b > 0, b + 1 < a.nbands,
                                 cs, S, x);
    __syncwarp();
    if (!ok) break;
  }
  for (int d = 16; d > 0; d >>= 1) S = max(S, __shfl_xor_sync(0xffffffffu, S, d));
  if (lane == 0) atomicMax(a.best, S);
}

// The kernel of a band height: with the DNA penalties compiled in at the
// heights the planner picks (see GapSet), else the general one.
using PairKernel = void (*)(const PairBandArgs);
template <int R>
PairKernel pair_kernel_of(int gaps) {
  return gaps == kGapsDna ? pair_band_kernel<R, kGapsDna> : pair_band_kernel<R, kGapsAny>;
}
#define SWGB_PAIR_R_LIST(X) X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(20) X(24) X(28)
PairKernel pair_kernel(int R, int gaps) {
#define SWGB_CASE(RR) \
  if (R == RR) return pair_kernel_of<RR>(gaps);
  SWGB_PAIR_R_LIST(SWGB_CASE)
#undef SWGB_CASE
  return nullptr;
}

}  // namespace

int pair_max_warps() { return kPairWarps; }
int pair_slot_bytes(int R) { return (R + 3) / 4 * 4; }

size_t pair_smem_bytes(int pbuf_bytes, int warps) { return (size_t)warps * (pbuf_bytes + kBandRingBytes); }

int pair_max_ctas_per_sm(int R, int gaps, int threads, size_t smem) {
  const PairKernel kern = pair_kernel(R, gaps);
  int n = 0;
  if (!kern ||
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_pair(const PairBandArgs &a, int R, int grid, int threads, size_t smem, cudaStream_t s) {
  const PairKernel kern = pair_kernel(R, gap_set(a.sc));
  if (!kern) return cudaErrorInvalidValue;
  void *args[] = {(void *)&a};
  return cudaLaunchCooperativeKernel((const void *)kern, dim3(grid), dim3(threads), args, smem, s);
}

}  // namespace swgb
