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
#include "band_core.cuh"

namespace swgb {
namespace {

// Two columns per step (band_core.cuh).  In a loop over one warp per
// sub-partition a two-column step takes 180 cycles at R = 8 and 316 at R = 16,
// in a band between two others 244 and 378.
constexpr int kPairCols = 2;
constexpr int kBandRingBytes = 2 * kResChunk + 2 * kColBlock * 8;  // per warp: residues, boundary entries
// Steps unrolled: a whole block where its code fits the instruction cache (R =
// 8: 269 -> 244 cycles per step, R = 20: 478 -> 660).
template <int R>
constexpr int kPairUnroll = R <= 16 ? 8 : 4;
// At most this many warps per CTA, one CTA per SM: two per SM sub-partition,
// with up to 255 registers a thread.  (Sixteen warps of 128 registers: 473
// against 380 cycles per step at R = 16; a pair long enough for more warps
// gets taller bands instead, which measured faster: 1M x 1M 273 ms at R = 28
// and two warps, 283 at R = 20 and three, 284 at R = 14 and four.)
constexpr int kPairWarps = 8;

__device__ __forceinline__ uint32_t band_gen(int b, int nslots) { return ((uint32_t)(b / nslots) & 1u) ^ 1u; }

// The tagged, wrapping rings of this kernel.  Lanes 0..15 load the next
// block's entries during a block and check their tags at its end (loading
// again until they are fresh).
struct WrapRing {
  const unsigned long long *in;  // ring of the band above
  unsigned long long *own;       // this band's ring
  int32_t *cons_in;              // columns of `in` consumed, published for the band above
  const int32_t *cons_out;       // columns of `own` consumed by the band below
  int32_t window, npad;
  uint32_t gen_in;               // generation tag bit of `in` (0 or 1)
  int32_t cons_every;            // blocks between publications of cons_in
  int32_t *status;
  int32_t go;
  uint2 *rgb;
  int lane;
  const unsigned long long *base;  // the rings and their entries (checked build)
  int64_t entries;
  bool prev, next;
  uint32_t lo_bias, hi_bias;     // this lap's tag in H's word; Go and the generation tag in F's
  // reading: ring position and lap parity of the next block, columns consumed
  int rpos = 0, consumed = 0, since = 0;
  uint32_t rlap = 0u;
  unsigned long long pend = 0ull;
  // writing: ring position of the block being written, columns there is room for
  int wpos = 0, room_end = 0;

  __device__ __forceinline__ bool fresh() const {
    return ((uint32_t)pend >> 31) == rlap && (uint32_t)(pend >> 63) == gen_in;
  }
  __device__ __forceinline__ void load() {
    if (lane < kColBlock && in_range(in - base + rpos + lane, entries, status)) pend = ld_relaxed_u64(in + rpos + lane);
  }
  __device__ __forceinline__ bool land(int slot) {
    bool ok = lane >= kColBlock || fresh();
    if (!__all_sync(0xffffffffu, ok)) {
      const long long t0 = clock64();
      do {
        if (__any_sync(0xffffffffu, clock64() - t0 > kLongWaitBudgetCycles)) {
          if (lane == 0) atomicExch(status, SW_ETIMEOUT);
          return false;
        }
        if (!ok) {
          load();
          ok = fresh();
        }
      } while (!__all_sync(0xffffffffu, ok));
    }
    if (lane < kColBlock) {
      const int32_t h = (int32_t)((uint32_t)pend & 0x7fffffffu);
      const int32_t f = (int32_t)((uint32_t)(pend >> 32) & 0x7fffffffu) - go;
      rgb[slot * kColBlock + lane] = make_uint2((uint32_t)h, (uint32_t)f);
    }
    consumed += kColBlock;
    rpos += kColBlock;
    if (rpos == window) {
      rpos = 0;
      rlap ^= 1u;
    }
    __syncwarp();
    // hand the columns back every few blocks and at the end (the release orders
    // the loads of lanes 0..15, which the warp barrier above ordered first)
    if (++since == cons_every || consumed == npad) {
      since = 0;
      if (lane == 0) st_release(cons_in, consumed);
    }
    return true;
  }
  __device__ __forceinline__ bool room(int wblk) {
    if (!in_range(own - base + wpos, entries, status) || !in_range(own - base + wpos + kColBlock - 1, entries, status))
      return false;
    if ((wblk + 1) * kColBlock <= room_end) return true;
    const int need = (wblk + 1) * kColBlock - window;
    int seen = 0;
    if (lane == 0) seen = wait_flag_value(cons_out, need, kLongWaitBudgetCycles);
    seen = __shfl_sync(0xffffffffu, seen, 0);
    if (seen < need) {
      if (lane == 0) atomicExch(status, SW_ETIMEOUT);
      return false;
    }
    // (no farther than the columns themselves: both terms stay in 32 bits)
    room_end = seen > npad - window ? npad : seen + window;
    return true;
  }
  __device__ __forceinline__ unsigned long long *out(int) const { return own + wpos; }
  __device__ __forceinline__ void done(int) {
    wpos += kColBlock;
    if (wpos == window) {
      wpos = 0;
      lo_bias ^= 0x80000000u;
    }
  }
};

template <int R, int GAPS>
__global__ void __launch_bounds__(32 * kPairWarps, 1) pair_band_kernel(const PairBandArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  uint8_t *pbuf = smem + (size_t)warp * (a.pbuf_bytes + kBandRingBytes);
  uint8_t *ring = pbuf + a.pbuf_bytes;                        // residues, then the boundary slots
  uint2 *rgb = reinterpret_cast<uint2 *>(ring + 2 * kResChunk);
  const Consts cs = make_consts<GAPS>(a.sc);
  int32_t S = 0;
  // global warp g = warp * grid + CTA: bands spread over the SMs first
  for (int b = warp * gridDim.x + blockIdx.x; b < a.nbands; b += gridDim.x * nw) {
    __syncwarp();  // (the band before this one has read its profile, residues and slots)
    ResidueStage<1> rs{ring, a.target, nullptr, a.npad, 0, lane, a.target, a.npad, a.status};
    rs.stage(0);
    const uint4 *src = reinterpret_cast<const uint4 *>(a.prof + (int64_t)b * a.band_bytes);
    for (int i = lane; i < a.band_bytes / 16; i += 32) reinterpret_cast<uint4 *>(pbuf)[i] = __ldg(src + i);
    clear_slots(rgb, lane, 0u);
    WrapRing x;
    x.in = a.strips + (size_t)((b + a.nslots - 1) % a.nslots) * a.window;
    x.own = a.strips + (size_t)(b % a.nslots) * a.window;
    x.cons_in = a.cons + (b > 0 ? b - 1 : 0);
    x.cons_out = a.cons + b;
    x.window = x.room_end = a.window;
    x.npad = a.npad;
    x.gen_in = band_gen(b > 0 ? b - 1 : 0, a.nslots);
    x.cons_every = a.cons_every;
    x.status = a.status;
    x.go = cs.go;
    x.rgb = rgb;
    x.lane = lane;
    x.base = a.strips;
    x.entries = a.ring_entries;
    x.prev = b > 0;
    x.next = b + 1 < a.nbands;
    x.lo_bias = 0u;
    x.hi_bias = (uint32_t)cs.go + (band_gen(b, a.nslots) << 31);
    BandLane<R, kFormInt32, kPairCols> ln;
    ln.reset(cs);
    const bool ok = band_sweep<kFormInt32, kPairCols, kPairUnroll<R>, false, IntProfile<R, kPairCols>>(
        ln, rs, x, rgb, pbuf + lane * kSlotBytes<R>, a.stride, lane, a.npad / kColBlock, -1, 0, cs, a.status);
    cp_async_wait<0>();
    S = max(S, ln.S);
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
