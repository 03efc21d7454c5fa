// Tensor-core path of LPConvolution / LPInnerProduct (paper Sec. 2) for sm_100a.
//
// The layer is an exact integer GEMM  acc[m][n] = sum_k A[m][k] * B[n][k]  with
//   A = activations (implicit im2col of the NHWC planes for a convolution, [B][K] rows for an
//       inner product), B = weights [N][K] (K ordered tap-major, channel-minor).
// Operands of more than 8 bits live as two byte planes (q = 256*hi + lo, hi signed, lo
// unsigned); the product of two such numbers is four int8 products
//   q_a*q_b = 2^16 hi_a*hi_b + 2^8 (hi_a*lo_b + lo_a*hi_b) + lo_a*lo_b
// each accumulated exactly in int32 by tcgen05.mma kind::i8 into its own TMEM accumulator
// (the two middle terms share one) and recombined exactly in the epilogue.  8-bit operands
// take a single product.
//
// One persistent CTA per SM walks over output tiles (128 rows x BN columns):
//   warps 0-2  : TMA producers, spread over the operand planes (im2col / tiled loads into a ring
//                of shared-memory stages; a single warp issues bulk-tensor copies too slowly)
//   warp  3    : MMA issue; also owns the TMEM allocation (with one product a step and one copy for all taps
//                warp 2 issues every other tile's MMAs, and two warps copy: kIssuers)
//   warps 4-19 : epilogue (tcgen05.ld -> 64-bit recombination -> bias, ReLU, requantize with
//                saturation, zero / saturation counters; byte planes staged in shared memory and
//                written by bulk-tensor stores; or range / split-K)
// Every device-side wait is bounded; on expiry the kernel flags ADAPTION_ERR_TIMEOUT in the
// caller's stats word, drains what it has in flight, frees its TMEM and returns.
#include <cuda.h>

#include <atomic>
#include <cstdlib>
#include <cstring>

#include "common.cuh"
#include "knobs.cuh"
#include "tc_ptx.cuh"
#include "tensor_maps.cuh"

namespace adaption {

int num_sms();

namespace {

constexpr int kBM = 128;
constexpr int kMaxStages = 12;
constexpr int kMaxAccBufs = 4;
constexpr int kEpiWarps = 16;                // four per TMEM lane quarter, each takes a quarter of the columns
constexpr int kProducerWarps = 3;            // spread over the operand planes: TMA issue is slow per warp
// One MMA-issuing warp of its own (a second one, alternating stages of a tile, measured no faster; see kIssuers for the loops
// in which a copying warp issues every other tile).
constexpr int kMmaWarps = 1;
constexpr int kMmaWarp = kProducerWarps;
constexpr int kFirstEpiWarp = kProducerWarps + kMmaWarps;
constexpr int kThreads = 32 * (kFirstEpiWarp + kEpiWarps);
// int32 accumulators: the shared middle accumulator takes two products of magnitude
// <= 128*255 per k, so a reduction of up to 32768 stays below 2^31.
constexpr int64_t kMaxKPerAccumulation = 32768;
// epilogue variants (a template parameter of the kernel): generic 64-bit, the 32-bit fast path of
// ReLU layers, generic with stochastic rounding, 32-bit with stochastic rounding (16 images, us: 3 -> 64 channels at
// 224 x 224 243 -> 166, 128 -> 128 at 112 x 112 158 -> 103, the same at 8 bits 167 -> 51)
constexpr int kEpiGeneric = 0, kEpiFast = 1, kEpiStochastic = 2, kEpiFastStochastic = 3;
// main-loop variants: one full k-block per stage; several k-blocks per stage and / or resident weights; one
// k-block per stage of which the last one of a tap has fewer steps (channel pitch no multiple of 128).  (Variants,
// because the issuing warp's code decides the main loop's speed: with the bookkeeping of the third in the second
// 64 x 224 x 224 x 64 -> 64 took 595 us against 515.)
// kLoopPixels: neighbouring output pixels share a row of the GEMM, see PixelPlan.
// kLoopHalo, kLoopTaps: the activations of a tile are copied once for all filter taps, see HaloPlan.
constexpr int kLoopPlain = 0, kLoopGrouped = 1, kLoopPartial = 2, kLoopPixels = 3, kLoopHalo = 4, kLoopTaps = 5;
// Added to the first three: tiles are boxes of pixels whose epilogue stores whole pooled windows, see BoxPlan.  (The last two
// are always boxes, pooled or not.  Kernels of their own, because the box's coordinates stay live beside the 64-bit
// epilogue's accumulators: with them in the kernels of all other layers too, 16 x 112 x 112, 64 -> 64, took 21.6 us instead of
// 18.0 (1x1, 16 bits) and 28.6 instead of 23.5 (3x3, 8 by 16 bits); 126 random layers 3 % on average, at most 18.)
// Partial blocks with the 32-bit epilogue are an exception: their kernel for boxes takes other tiles of 128 columns too, which
// the compiler schedules better in it (12 x 45 x 37, 96 -> 168, 12 bits 24.3 us, 25.2 in the kernel without boxes; seven others
// within 1 %), but not narrower ones (16 x 56 x 56, 96 -> 32, 16 bits 18.1 us, 17.2 without).
constexpr int kLoopBoxes = 8;

// Division by a number fixed for the launch: q = (n * mul >> 32) >> shift for 0 <= n < 2^31 (mul =
// ceil(2^(32 + shift) / d) with 2^(shift + 1) >= d > 2^shift; mul = 0 stands for d = 1).  An integer division costs a
// warp twenty to thirty instructions, and the copying and issuing warps share their schedulers with the epilogue's.
struct FastDiv {
  uint32_t mul, shift;
  int d;
  __device__ __forceinline__ int quot(int n) const { return mul == 0u ? n : (int)(__umulhi((uint32_t)n, mul) >> shift); }
};
FastDiv fast_div(int d) {
  FastDiv f;
  f.d = d;
  f.mul = 0;
  f.shift = 0;
  if (d > 1) {
    while ((2ll << f.shift) < d) ++f.shift;
    f.mul = (uint32_t)(((1ull << (32 + f.shift)) + (unsigned)d - 1) / (unsigned)d);
  }
  return f;
}

// Pixel grouping (kLoopPixels), for convolutions of stride 1 over a pitch of 32 channels.  With G neighbouring pixels
// taken as one of 32 G channels (the tensor is the same bytes) a row of the GEMM covers G output pixels, its G * ys
// columns are (pixel p, output channel), and one copy of 128 rows of 32 G bytes serves what took up to 2 G copies of
// 32-byte rows: copies deliver one row per two cycles whatever its length, and an MMA reads its 128 rows of activations
// from shared memory whatever its columns.  The step of input pixel u (from the first output pixel's position, before
// padding) meets output pixel p under tap u + pad - p: it runs for the pixels p where that is a tap, a range, on the
// accumulator columns of that range.  The weights stay in shared memory as rows of one 32-byte step, taps in
// descending order, so the B operand of such a range is a contiguous run of rows.
// 16 bits, us: 16 x 112 x 112 x 16 -> 16, 7x7 112 -> 55 (G = 2); 16 x 112 x 112 x 32 -> 64, 5x5 72 -> 42; 64 x 56 x 56 x 32
// -> 32, 3x3 27.6 -> 19.4.  (With 64-byte pixels in pairs 64 x 224 x 224 x 64 -> 64 gained nothing, 457 -> 452 us: there
// the operand bytes that the MMAs read bound both.)
constexpr int kMaxPixelBlocks = 8;
struct PixelPlan {
  int G;                      // pixels per row (1: not grouped)
  int ys, ys_shift;           // columns per pixel (pitch of the output), a power of two
  int n_valid;                // of which real output channels
  int S;                      // filter taps per row
  int blocks, first;          // groups of input pixels that a row of taps reaches; the one to begin with
  uint32_t b_plane;           // bytes of one resident weight plane
  uint32_t row_u;             // one filter row of it, in 16-byte units
  // per block and 32-byte step: bits 17-22 columns / 8 (0: the step meets no pixel), below them the first column
  uint32_t step[kMaxPixelBlocks][4];
  uint32_t b_row[kMaxPixelBlocks][4];   // where its weights start in a filter row, in 16-byte units
};

// Tiles whose 128 rows are a box of 2^w x 2^h x 2^n pixels (columns fastest, then rows, then images) instead of
// consecutive pixels: whole 2x2 windows of a max-pool lie in one tile, even in one warp, so the epilogue stores their
// maxima, a quarter of the bytes, and no pooling pass reads the layer back.
// Against storing pair maxima and pooling them vertically, us: 16 bits, 64 x 224 x 224 x 64 -> 64 531 -> 439, 64 x 112 x 112 x
// 128 -> 128 345 -> 312, 64 x 56 x 56 x 256 -> 256 287 -> 270, 64 x 28 x 28 x 512 -> 512 263 -> 251; 8 bits, 128 images 448 ->
// 435, 221 -> 174, 160 -> 131, 145 -> 129; one image 18 -> 15, 15 -> 13.
struct BoxPlan {
  int on, pool;
  int w, h, n;                // powers of two, as exponents
  int tiles_w, tiles_h, images;
  FastDiv div_w, div_h;
};

// One copy of a tile's activations for all filter taps (kLoopHalo, kLoopTaps), for convolutions of stride 1 on boxes of 8
// columns x 16 rows: the copied box has the filter's margin around it, `w` pixels per row of it, and the operand of a tap is
// the same rows of shared memory begun (r w + s) pixels further on: the eight rows of a swizzle group are eight pixels of
// an image row, and the groups lie `w` pixels apart whatever the tap.  (The swizzle is a function of the address, so rows
// may begin anywhere in its pattern.)  Copies deliver one row per two cycles whatever its length, and they write shared
// memory while the MMAs read it: 3x3 filters take 180 rows per tile this way, 1152 before.  us, before -> now: 16 bits, 64 x
// 224 x 224 x 64 -> 64 488 -> 322 (pooled 441 -> 329), 64 x 112 x 112 x 64 -> 128 185 -> 161; 8 bits, 128 images 385 -> 338
// (439 -> 342), 128 x 112 x 112 x 128 -> 128 192 -> 169 (173 -> 146).
// kLoopTaps is the same for the pixels of 16 bytes of a first layer, unswizzled: a step of 32 bytes is two taps, whose
// distance is the operand's leading offset.  No packed copy of the image is written and read back.
constexpr int kHaloW = 8, kHaloH = 16, kMaxTapSteps = 5;
struct HaloPlan {
  int w, R, S;
  int steps;                       // kLoopTaps: steps of 32 bytes (0: kLoopHalo)
  uint32_t px_u;                   // a pixel in 16-byte units
  uint32_t b_row_u;                // kLoopTaps: weights of a step in 16-byte units
  uint32_t a_lo[kMaxTapSteps];     // kLoopTaps: low descriptor word of a step relative to the tile's first pixel
};

struct TcParams {
  int M, N;
  int tile_m;                 // rows per tile: 128, or 256 for a CTA pair
  int tiles_m, tiles_n, splits, total_tiles;
  int num_kb, kb_per_split;
  int BN, BK;
  int ksteps, ksteps_last;    // 32-byte steps of a k-block, of the last channel block of a tap
  uint32_t sbo, layout_type;
  int stages;
  uint32_t a_bytes, b_bytes, stage_bytes;
  // a stage holds `kps` consecutive k-blocks of `kb_bytes` each (short k-blocks are grouped so
  // that the per-stage hand-shake is amortised over enough MMAs)
  int kps;
  uint32_t kb_bytes, tx_bytes;     // tx_bytes: what the copies of a k-block deliver
  // weights resident in shared memory (one column tile, short reduction): the ring then holds
  // only activation planes and all weight k-blocks are loaded once per CTA at this offset
  int b_resident, b_blocks;        // b_blocks: weight k-blocks (kLoopTaps: slabs of a tap) that are resident
  uint32_t b_res_off;
  int acc_bufs, acc_shift;    // 1, 2 or 4 accumulator sets, and the power of two
  FastDiv div_tiles_n, div_splits, div_ow, div_oh, div_s, div_cblks;
  // Three accumulators of 128 columns leave one quarter of TMEM free: the high accumulator then
  // alternates between the first and the last quarter from tile to tile (the other two stay put),
  // and the epilogue hands the low and middle accumulators back before it reads the high one, so
  // that the next tile's MMAs start while this tile's high accumulator is still being read.
  int split_hh;
  // With the split release: the last two k-blocks of a tile are issued product by product (all low
  // products, then the middle ones, then the high ones) with a completion signal after each group,
  // so that the epilogue pulls the low and the middle accumulator into registers while the
  // remaining MMAs of the tile still run, and the next tile's MMAs can follow almost at once.
  int tail_stagger;
  uint32_t tmem_cols;
  int is_conv, OH, OW, S, cblks, w_pitch, stride_h, stride_w, pad_h, pad_w;
  const int16_t* bias;
  int bias_shift;
  RequantParams rq;
  StochasticParams st;         // stochastic rounding in the requantization
  int mode;
  int8_t* y_hi;
  uint8_t* y_lo;
  int16_t* y_q16;
  long long y_stride;
  long long* ws;
  long long ws_ld;
  adaption_stats* stats;
  unsigned long long timeout_ns;
  // test aid (adaption_debug_set "stall_at"): every producer warp stops, with nothing in flight for
  // that stage, before its stage number `stall_at` (counted per CTA from 0); -1 = never.  The waits
  // of the other roles then run out and the kernel reports ADAPTION_ERR_TIMEOUT.
  int stall_at;
  // epilogue variants chosen on the host
  int fast_relu;              // launch the FAST kernel variant (paired 16-bit epilogue)
  int fast_stochastic;        // ... the 32-bit one with stochastic rounding
  int byte_out;               // ... with one accumulator: staged 8-bit outputs, four to a word
  int fast_range;             // range mode: 32-bit keys decide what is worth the exact 64-bit value
  int pool_w;                 // store max(row 2j, row 2j+1) of the tile: half of a 2x2 max-pool (staged only)
  int epi_groups;             // 1, 2 or 4 groups of epilogue warps that take turns tile by tile
  // One copy for all taps, four groups: every warp makes, stages and stores 32 whole rows of a tile by itself, with no
  // barrier among the warps (8 bits, 128 x 224 x 224, 3 -> 64 230 -> 214 us; 128 x 112 x 112, us with two groups and four: 64
  // -> 128 146 and 114, 128 -> 128 174 and 140), and in the one kernel that takes box tiles and others.  Not in the other
  // loops, whose kernels spilled for it: 48 x 62 x 137, 38 -> 92,
  // 3x3 at 12 bits 164 us with it and 148 without, 61 x 36 x 197, 8 -> 72, 1x1 63 and 61, 51 x 200 x 158, 41 -> 22 at 8 bits 43.5
  // and 40.3.
  int own_rows;
  int staged;                 // outputs leave through shared memory and bulk-tensor stores
  int stage_bufs;             // staging buffers per epilogue group: 1, or 2 used in turn (narrow tiles)
  uint32_t stage_off;         // offset of the staging planes from the ring base
  uint32_t const_off;         // offset of the per-column epilogue constants (8 bytes per column and group)
  PixelPlan px;
  BoxPlan box;
  HaloPlan halo;
};

// Optional per-role time stamps of CTA 0 (development builds only: -DADAPTION_TIMELINE).
#ifdef ADAPTION_TIMELINE
__device__ long long g_timeline[8192];
#define TL_STAMP(role, tile, slot)                                                        \
  do {                                                                                    \
    if (blockIdx.x == 0 && (tile) < 32u) g_timeline[((role) * 32 + (tile)) * 8 + (slot)] = clock64(); \
  } while (0)
#else
#define TL_STAMP(role, tile, slot) do { } while (0)
#endif

struct Ctrl {
  // A slot's copies report to the barrier of the warp that issues the MMAs on them (the first kMaxStages, or the second
  // where there are two issuing warps).  A wait on an mbarrier tells phases apart only modulo two: a warp that waits may
  // be at most one fill behind.  With one barrier per slot, counted in laps of the ring, a warp waiting for a fill whose
  // predecessor was the other warp's, and had not landed yet, was let through by the one before that.  A barrier of its
  // own, whose fills it counts itself, cannot run ahead: its next fill needs the slot that this warp hands back.
  unsigned long long full[2 * kMaxStages];
  unsigned long long empty[kMaxStages];
  unsigned long long tmem_full[kMaxAccBufs];
  unsigned long long tmem_empty[kMaxAccBufs];
  unsigned long long part_full[2];   // staggered tail: low accumulator complete, middle accumulator complete
  unsigned long long drain[2];  // an issuing warp's last commit before an early exit
  unsigned long long b_ready;   // resident weights have landed
  uint32_t tmem_base;
  volatile uint32_t abort;
};

// Bounded wait on an mbarrier phase.  Returns false once the time limit is hit (or another
// role already gave up); the caller then leaves its loop.
// `relaxed` waiters (producers, epilogue) let the hardware suspend them while the phase is
// incomplete, so that their polling neither takes issue slots from the MMA-issuing thread, whose
// instruction stream is the critical path, nor burns power during the long mainloops.
__device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, Ctrl* ctrl, const TcParams& p,
                                       bool relaxed) {
  const unsigned long long t0 = global_ns();
  uint32_t spins = 0;
  while (!(relaxed ? mbar_try_wait_suspend(bar, parity, 1000u) : mbar_try_wait(bar, parity))) {
    if (relaxed || (++spins & 127u) == 0) {
      if (ctrl->abort) return false;
      if (global_ns() - t0 > p.timeout_ns) {
        ctrl->abort = 1;
        atomicExch(&p.stats->status, (int)ADAPTION_ERR_TIMEOUT);
        return false;
      }
    }
  }
  return true;
}
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, Ctrl* ctrl, const TcParams& p,
                                         bool relaxed = true) {
  if (mbar_try_wait(bar, parity)) return true;
  return wait_slow(bar, parity, ctrl, p, relaxed);
}

// The same bounded wait without a function call, for waits that sit between TMEM loads whose
// results are live in registers (a call there would make the compiler save and restore them).
__device__ __forceinline__ bool wait_bar_inline(uint32_t bar, uint32_t parity, Ctrl* ctrl, const TcParams& p) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_try_wait_suspend(bar, parity, 1000u)) {
    if (ctrl->abort) return false;
    if (global_ns() - t0 > p.timeout_ns) {
      ctrl->abort = 1;
      atomicExch(&p.stats->status, (int)ADAPTION_ERR_TIMEOUT);
      return false;
    }
  }
  return true;
}

// Two issuing warps: which barrier of its slot fill number `j` of the ring reports to, and with which parity (the tile's
// warp, and how many of that warp's fills the slot had before).
struct Fill {
  uint32_t bar, parity;
};
__device__ __noinline__ Fill fill_of(uint32_t j, uint32_t stages, uint32_t num_kb) {
  Fill f{(j / num_kb) & 1u, 0u};
  for (uint32_t i = j % stages; i < j; i += stages) f.parity ^= ((i / num_kb) & 1u) == f.bar ? 1u : 0u;
  f.bar = j % stages + f.bar * (uint32_t)kMaxStages;
  return f;
}

struct TileCoord {
  int m0, n0, kb_begin, kb_end;
};
__device__ __forceinline__ TileCoord decode_tile(int t, const TcParams& p) {
  TileCoord tc;
  const int rest = p.div_tiles_n.quot(t);
  const int tn = t - rest * p.tiles_n;
  const int tm = p.div_splits.quot(rest);
  const int split = rest - tm * p.splits;
  tc.m0 = tm * p.tile_m;
  tc.n0 = tn * p.BN;
  tc.kb_begin = split * p.kb_per_split;
  tc.kb_end = min(p.num_kb, tc.kb_begin + p.kb_per_split);
  return tc;
}

// First pixel of box `b`.
struct BoxCoord {
  int ow, oh, img;
};
__device__ __forceinline__ BoxCoord decode_box(int b, const BoxPlan& x) {
  BoxCoord c;
  const int rest = x.div_w.quot(b);
  const int ib = x.div_h.quot(rest);
  c.ow = (b - rest * x.tiles_w) << x.w;
  c.oh = (rest - ib * x.tiles_h) << x.h;
  c.img = ib << x.n;
  return c;
}

template <int NACC>
__device__ __forceinline__ long long combine(int32_t a0, int32_t a1, int32_t a2) {
  if (NACC == 3) return (long long)a0 * 65536ll + (long long)a1 * 256ll + (long long)a2;
  if (NACC == 2) return (long long)a0 * 256ll + (long long)a1;
  return (long long)a0;
}

// Requantization of one pre-activation value for the common case of a rounding right shift
// (shift >= 1): v / 2^shift rounded half away from zero, saturated to [qmin, qmax].  The shifted
// value is narrowed to 32 bits with saturation first, so clamping and counting are 32-bit work.
// With ReLU the value is non-negative and the lower bound cannot be crossed.
template <bool RELU>
__device__ __forceinline__ int32_t requant_shift_right(long long v, long long half, int shift, int32_t qmin,
                                                       int32_t qmax, bool counted, Counts& c) {
  if (RELU) v = v < 0 ? 0ll : v;
  long long t = v + half;
  if (!RELU) t += (v >> 63);
  const long long r = t >> shift;
  const int32_t r32 = (int32_t)r;
  const int32_t rh = (int32_t)(r >> 32);
  const int32_t rs = (rh == (r32 >> 31)) ? r32 : (rh < 0 ? (int32_t)0x80000000 : 0x7fffffff);
  const int32_t q = min(max(rs, qmin), qmax);
  c.sat_pos += (counted && rs > qmax);
  if (!RELU) c.sat_neg += (counted && rs < qmin);
  c.zeros += (counted && q == 0);
  return q;
}


// Fast requantization for ReLU layers with a rounding right shift 9 <= shift <= 31, in 32-bit
// arithmetic.  Wanted: floor((v + C) / 2^shift) with v = 2^16 hh + 2^8 mid + ll and the per-column
// constant C = bias * 2^bias_shift + 2^(shift-1) (ReLU maps negative values to zero, so rounding
// half away from zero is this floor).  With C = 2^16 Ch + Cl, 0 <= Cl < 2^16:
//   T = mid + floor((ll + Cl) / 2^8),  H = hh + Ch,   v + C = 2^8 (2^8 H + T) + (a remainder below 2^8)
// and because shift >= 8 the remainder cannot change the floor:
//   shift >= 16:  floor((H + floor(T / 2^8)) / 2^(shift-16))
//   shift <  16:  H * 2^(16-shift) + floor(T / 2^(shift-8))
// The host checks from the reduction length that none of these 32-bit quantities can overflow
// (otherwise the layer takes the generic 64-bit epilogue).
__device__ __forceinline__ int32_t mad_lo(int32_t a, int32_t b, int32_t c) {
  int32_t d;
  asm("mad.lo.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
// two 32-bit values -> two 16-bit values saturated to [-32768, 32767]; `lo` lands in the low half
__device__ __forceinline__ uint32_t pack_sat_s16x2(int32_t hi, int32_t lo) {
  uint32_t d;
  asm("cvt.pack.sat.s16.s32 %0, %1, %2;" : "=r"(d) : "r"(hi), "r"(lo));
  return d;
}
__device__ __forceinline__ uint32_t max_s16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.s16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t min_s16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("min.s16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// Fast path, accumulator by accumulator over thirty-two columns of one row.  With T and H as derived
// above, `t` holds T (with a mixed 16 x 8-bit layer hh is absent and H = Ch) or, with 8-bit
// operands on both sides, the single accumulator (the whole sum: one 32-bit add, any shift >= 0);
// `h` holds hh.  Outputs are handled as pairs of 16-bit lanes (saturating pack, ReLU, upper bound,
// zero count).  Saturation is only detected here (some lane reached the bound); the exact count of
// that group of eight is then redone from the 32-bit results, which is rare.  Every group of eight
// columns is either entirely real or entirely padding (N is a multiple of 8).
template <int NACC, bool WIDE>
__device__ __forceinline__ int32_t fast_result(int32_t t, int32_t h, int shift) {
  if (NACC == 1) return t >> shift;
  if (WIDE) return (h + (t >> 8)) >> (shift - 16);
  return mad_lo(h, 1 << (16 - shift), t >> (shift - 8));
}
// real columns of the eight that begin at column `col` (0, or all eight where N is a multiple of 8)
template <bool PIX>
__device__ __forceinline__ int real_columns8(int col, const TcParams& p) {
  const int n = PIX ? p.px.n_valid - (col & (p.px.ys - 1)) : p.N - col;
  return min(max(n, 0), 8);
}
// index of an output element among the real ones, row-major over pixels and channels
template <bool PIX>
__device__ __forceinline__ uint64_t element_index(int m, int col, const TcParams& p) {
  if (PIX)
    return ((uint64_t)m * (uint64_t)p.px.G + (uint64_t)(col >> p.px.ys_shift)) * (uint64_t)p.px.n_valid +
           (uint64_t)(col & (p.px.ys - 1));
  return (uint64_t)m * (uint64_t)p.N + (uint64_t)col;
}

// sixteen of the thirty-two columns (`half` = 0 or 1; they begin at column `col`) -> eight packed words; `t` and `h`
// hold T and H (or, with a single accumulator, t holds the sum plus its constant)
template <int NACC, bool WIDE, bool PIX>
__device__ __forceinline__ void fast_outputs16(const int32_t (&t)[32], const int32_t (&h)[32], int half, int shift,
                                               int32_t qmax, bool row_ok, int col, const TcParams& p,
                                               Counts& cnt, uint32_t (&w)[8]) {
  const uint32_t qmax2 = (uint32_t)qmax * 0x00010001u;
  const int32_t bound = qmax == 32767 ? 32767 : qmax + 1;      // a lane that reached this may have been clipped
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const int base = 16 * half + 8 * g;
    const bool counted = row_ok && real_columns8<PIX>(col + 8 * g, p) > 0;
    uint32_t top = 0, nonzero = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = base + 2 * j;
      const int32_t r0 = fast_result<NACC, WIDE>(t[k], h[k], shift);
      const int32_t r1 = fast_result<NACC, WIDE>(t[k + 1], h[k + 1], shift);
      uint32_t v = max_s16x2(pack_sat_s16x2(r1, r0), 0u);
      top = max_s16x2(top, v);
      if (qmax != 32767) v = min_s16x2(v, qmax2);
      nonzero += min_s16x2(v, 0x00010001u);
      w[4 * g + j] = v;
    }
    if (counted) cnt.zeros += 8u - (nonzero & 0xffffu) - (nonzero >> 16);
    if (counted && ((int32_t)(top & 0xffffu) >= bound || (int32_t)(top >> 16) >= bound)) {
#pragma unroll
      for (int j = 0; j < 8; ++j) cnt.sat_pos += (fast_result<NACC, WIDE>(t[base + j], h[base + j], shift) > qmax);
    }
  }
}

// Sixteen 8-bit outputs of a single accumulator (`t` holds the sum plus its constant, shift >= 1, bound 127), four to a
// word: floor(v / 2^(shift-1)) saturated to [0, 255] and halved is floor(v / 2^shift) with ReLU and bound.  Zeros and
// bytes at the bound are found four at a time; possible saturations are recounted exactly, which is rare.
// (4.3 integer operations a value instead of 7.5; 8 bits, batch 128, 3 -> 64 channels at 224 x 224 352 -> 314 us,
// 128 -> 128 at 112 x 112 with pooling 220 -> 213.)
__device__ __forceinline__ uint32_t pack_sat_u8x4(int32_t e0, int32_t e1, int32_t e2, int32_t e3) {
  uint32_t d;
  asm("{\n"
      ".reg .b32 u;\n"
      "cvt.pack.sat.u8.s32.b32 u, %4, %3, 0;\n"
      "cvt.pack.sat.u8.s32.b32 %0, %2, %1, u;\n"
      "}\n"
      : "=r"(d)
      : "r"(e0), "r"(e1), "r"(e2), "r"(e3));
  return d;
}
// larger of two values 0 .. 127, byte by byte
__device__ __forceinline__ uint32_t max_bytes7(uint32_t a, uint32_t b) {
  const uint32_t ge = ((a | 0x80808080u) - b) & 0x80808080u;
  return b ^ ((a ^ b) & (ge - (ge >> 7)));
}
template <bool PIX>
__device__ __forceinline__ void fast_bytes16(const int32_t (&t)[32], int half, int shift, bool row_ok, int col,
                                             const TcParams& p, Counts& cnt, uint32_t (&w)[4]) {
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const int base = 16 * half + 8 * g;
    uint32_t nonzero = 0, bound = 0;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int k = base + 4 * j;
      const uint32_t x = (pack_sat_u8x4(t[k] >> (shift - 1), t[k + 1] >> (shift - 1), t[k + 2] >> (shift - 1),
                                        t[k + 3] >> (shift - 1)) >> 1) & 0x7f7f7f7fu;
      nonzero = __dp4a((x + 0x7f7f7f7fu) & 0x80808080u, 0x01010101u, nonzero);      // 128 for each
      bound |= x + 0x01010101u;
      w[2 * g + j] = x;
    }
    const bool counted = row_ok && real_columns8<PIX>(col + 8 * g, p) > 0;
    if (counted) cnt.zeros += 8u - (nonzero >> 7);
    if (counted && (bound & 0x80808080u) != 0u) {
#pragma unroll
      for (int j = 0; j < 8; ++j) cnt.sat_pos += (t[base + j] >> shift) > 127;
    }
  }
}

// One group of accumulators for eight consecutive columns of one row.
template <int NACC>
struct Acc8 {
  int32_t a[3][8];
};
// sixteen columns as two groups of eight, one load instruction per accumulator
template <int NACC>
__device__ __forceinline__ void load_acc16(uint32_t taddr, uint32_t first_off, int bn, Acc8<NACC>& x, Acc8<NACC>& y) {
  tmem_ld16(taddr + first_off, x.a[0], y.a[0]);
  if (NACC >= 2) tmem_ld16(taddr + (uint32_t)bn, x.a[1], y.a[1]);
  if (NACC == 3) tmem_ld16(taddr + 2u * (uint32_t)bn, x.a[2], y.a[2]);
}
template <int NACC>
__device__ __forceinline__ void load_acc8(uint32_t taddr, uint32_t first_off, int bn, Acc8<NACC>& x) {
  tmem_ld8(taddr + first_off, x.a[0]);
  if (NACC >= 2) tmem_ld8(taddr + (uint32_t)bn, x.a[1]);
  if (NACC == 3) tmem_ld8(taddr + 2u * (uint32_t)bn, x.a[2]);
}
template <int NACC>
__device__ __forceinline__ void pin_acc8(Acc8<NACC>& x) {
  pin_after_wait(x.a[0]);
  if (NACC >= 2) pin_after_wait(x.a[1]);
  if (NACC == 3) pin_after_wait(x.a[2]);
}
template <int NACC>
__device__ __forceinline__ long long acc_value(const Acc8<NACC>& x, int j) {
  return combine<NACC>(x.a[0][j], NACC >= 2 ? x.a[1][j] : 0, NACC == 3 ? x.a[2][j] : 0);
}

// Draws of the eight consecutive elements i0 .. i0 + 7 (two or three generator blocks).
__device__ __forceinline__ void philox_draws8(uint64_t i0, uint32_t k0, uint32_t k1, uint32_t (&R)[8]) {
  const uint64_t b0 = i0 >> 2;
  const uint32_t off = (uint32_t)i0 & 3u;
  const Philox4 a = philox4x32_10((uint32_t)b0, (uint32_t)(b0 >> 32), 0u, 0u, k0, k1);
  const Philox4 b = philox4x32_10((uint32_t)(b0 + 1), (uint32_t)((b0 + 1) >> 32), 0u, 0u, k0, k1);
  if (off == 0) {
#pragma unroll
    for (int j = 0; j < 4; ++j) { R[j] = a.w[j]; R[4 + j] = b.w[j]; }
    return;
  }
  const Philox4 c = philox4x32_10((uint32_t)(b0 + 2), (uint32_t)((b0 + 2) >> 32), 0u, 0u, k0, k1);
  const uint32_t w[12] = {a.w[0], a.w[1], a.w[2], a.w[3], b.w[0], b.w[1], b.w[2], b.w[3], c.w[0], c.w[1], c.w[2], c.w[3]};
#pragma unroll
  for (int j = 0; j < 8; ++j) R[j] = off == 1 ? w[j + 1] : (off == 2 ? w[j + 2] : w[j + 3]);
}

// Eight consecutive outputs with stochastic rounding in 32-bit arithmetic (ReLU layers, 9 <= shift <= 31, with one
// accumulator 1 <= shift <= 31, N a multiple of 8): with C = bias * 2^bias_shift and T, H as in fast_result
// (without the rounding half) q = floor(v / 2^shift) is what fast_result returns, and the threshold
// (v mod 2^shift) 2^(32 - shift) is the low 32 bits of v, v = 2^16 H + 2^8 T + (low byte of ll + Cl), shifted left.
// Negative v give q <= -1, at most 0 after the draw: the packed maximum with zero is the ReLU.  N is a multiple
// of 8, so the eight elements are two whole generator blocks.
template <int NACC, bool PIX>
__device__ __forceinline__ void stochastic8(const Acc8<NACC>& x, const int* cl, const int* ch, const TcParams& p,
                                            bool row_ok, int m, int col, Counts& cnt, uint32_t* w) {
  const bool counted = row_ok && real_columns8<PIX>(col, p) > 0;
  const int shift = p.rq.shift;
  uint32_t R[8];
  if (counted) {
    const uint64_t b = element_index<PIX>(m, col, p) >> 2;
    const Philox4 r0 = philox4x32_10((uint32_t)b, (uint32_t)(b >> 32), 0u, 0u, p.st.key0, p.st.key1);
    const Philox4 r1 = philox4x32_10((uint32_t)(b + 1), (uint32_t)((b + 1) >> 32), 0u, 0u, p.st.key0, p.st.key1);
#pragma unroll
    for (int j = 0; j < 4; ++j) { R[j] = r0.w[j]; R[4 + j] = r1.w[j]; }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) R[j] = 0xffffffffu;
  }
  int32_t q[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    int32_t f;
    uint32_t v_lo;
    if (NACC == 1) {
      const int32_t v = x.a[0][j] + cl[j];
      f = v >> shift;
      v_lo = (uint32_t)v;
    } else {
      const int32_t l = x.a[NACC - 1][j] + cl[j];
      const int32_t T = x.a[NACC - 2][j] + (l >> 8), H = (NACC == 3 ? x.a[0][j] : 0) + ch[j];
      f = shift >= 16 ? (H + (T >> 8)) >> (shift - 16) : mad_lo(H, 1 << (16 - shift), T >> (shift - 8));
      v_lo = ((uint32_t)H << 16) + ((uint32_t)T << 8) + ((uint32_t)l & 255u);
    }
    q[j] = f + (R[j] < (v_lo << (32 - shift)) ? 1 : 0);
  }
  const uint32_t qmax2 = (uint32_t)p.rq.qmax * 0x00010001u;
  uint32_t nonzero = 0;
  bool clipped = false;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t v = max_s16x2(pack_sat_s16x2(q[2 * j + 1], q[2 * j]), 0u);
    const uint32_t c = min_s16x2(v, qmax2);
    clipped |= (c & 0xffffu) == (uint32_t)p.rq.qmax || (c >> 16) == (uint32_t)p.rq.qmax;      // (maybe)
    nonzero += min_s16x2(c, 0x00010001u);
    w[j] = counted ? c : 0u;
  }
  if (counted) {
    cnt.zeros += 8u - (nonzero & 0xffffu) - (nonzero >> 16);
    if (clipped) {
#pragma unroll
      for (int j = 0; j < 8; ++j) cnt.sat_pos += q[j] > p.rq.qmax;
    }
  }
}

template <int NACC, bool RELU, bool STOCH, bool PIX>
__device__ __forceinline__ void requant8(const Acc8<NACC>& x, const long long* c64, const TcParams& p, bool row_ok,
                                         int m, int col, Counts& cnt, uint32_t* w) {
  const int nvalid = row_ok ? real_columns8<PIX>(col, p) : 0;
  int32_t q[8];
  if (STOCH && p.rq.shift > 0) {
    // stochastic rounding: element index = row-major index over the real M x N outputs
    uint32_t R[8];
    if (nvalid > 0) philox_draws8(element_index<PIX>(m, col, p), p.st.key0, p.st.key1, R);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      q[j] = j < nvalid ? requant_value_stochastic(acc_value<NACC>(x, j) + c64[j], p.rq, R[j], true, cnt)
                        : requant_value(0, p.rq, false, cnt);
  } else if (p.rq.shift > 0) {
    const long long half = 1ll << (p.rq.shift - 1);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      q[j] = requant_shift_right<RELU>(acc_value<NACC>(x, j) + c64[j], half, p.rq.shift, p.rq.qmin, p.rq.qmax, j < nvalid,
                                       cnt);
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) q[j] = requant_value(acc_value<NACC>(x, j) + c64[j], p.rq, j < nvalid, cnt);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) w[j] = __byte_perm((uint32_t)q[2 * j], (uint32_t)q[2 * j + 1], 0x5410);
}

// What the epilogue does with eight accumulator columns of one row in the modes that store nothing:
// split-K partial sums go to the int64 workspace, the range mode keeps the largest magnitude.
template <int NACC, bool PIX>
__device__ __forceinline__ void partial_or_range8(const Acc8<NACC>& x, const long long* c64, const TcParams& p,
                                                  bool row_ok, int m, int col, long long& vmax) {
  if (!PIX && p.splits > 1) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const long long v = acc_value<NACC>(x, j);
      if (row_ok && col + j < p.N && v != 0)
        atomicAdd((unsigned long long*)(p.ws + (long long)m * p.ws_ld + col + j), (unsigned long long)v);
    }
  } else {
    const int nvalid = row_ok ? real_columns8<PIX>(col, p) : 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      long long v = acc_value<NACC>(x, j) + c64[j];
      if (p.rq.relu && v < 0) v = 0;
      v = v < 0 ? -v : v;
      if (j < nvalid) vmax = v > vmax ? v : vmax;
    }
  }
}

// The range mode where 32 bits hold the parts (see fast_result; C without a rounding half): floor(v / 2^16) = H + floor(T / 2^8)
// costs six operations a value, the exact 64-bit |v| about fifteen.  `key` is floor(max |v| / 2^16) over what the warp has
// seen; only eight columns in which some lane reaches it are looked at exactly (for a negative v the complement of its
// quotient is compared, at most |v| / 2^16 and never below floor((|v| - 1) / 2^16), so no larger magnitude is missed).
// With a single accumulator v itself is compared.  Columns past N add up to zero; rows past M are left out.
// 16 images, us: 3 -> 64 channels at 224 x 224 117 -> 83, 64 -> 64 149 -> 105; 64 -> 128 at 112 x 112 65 -> 57; 8 bits, 128 ->
// 128 at 112 x 112 41 -> 28.
template <int NACC>
__device__ __forceinline__ void fast_range8(const Acc8<NACC>& x, const int* cl, const int* ch, const TcParams& p, bool row_ok,
                                            long long& vmax, int32_t& key) {
  const int32_t flip = p.rq.relu ? 0 : -1;
  int32_t best = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    int32_t f;
    if (NACC == 1) {
      f = x.a[0][j] + cl[j];
    } else {
      const int32_t T = x.a[NACC - 2][j] + ((x.a[NACC - 1][j] + cl[j]) >> 8);
      f = (NACC == 3 ? x.a[0][j] : 0) + ch[j] + (T >> 8);
    }
    best = max(best, f ^ ((f >> 31) & flip));
  }
  if (__any_sync(0xffffffffu, row_ok && best >= key)) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      long long v = acc_value<NACC>(x, j) + (NACC == 1 ? (long long)cl[j] : (long long)ch[j] * 65536ll + (long long)cl[j]);
      if (v < 0) v = p.rq.relu ? 0 : -v;
      if (row_ok && v > vmax) vmax = v;
    }
    key = __reduce_max_sync(0xffffffffu, (int32_t)min(NACC == 1 ? vmax + 1 + flip : vmax >> 16, 0x7fffffffll));
  }
}

// byte planes of sixteen packed outputs: four low bytes / four high bytes per word
__device__ __forceinline__ uint4 plane_lo(const uint32_t* w) {
  return make_uint4(__byte_perm(w[0], w[1], 0x6420), __byte_perm(w[2], w[3], 0x6420),
                    __byte_perm(w[4], w[5], 0x6420), __byte_perm(w[6], w[7], 0x6420));
}
__device__ __forceinline__ uint4 plane_hi(const uint32_t* w) {
  return make_uint4(__byte_perm(w[0], w[1], 0x7531), __byte_perm(w[2], w[3], 0x7531),
                    __byte_perm(w[4], w[5], 0x7531), __byte_perm(w[6], w[7], 0x7531));
}

// Direct stores of sixteen outputs of one row (16 bytes per plane; optional int16 copy).
__device__ __forceinline__ void store16_global(const uint32_t* w, const TcParams& p, bool row_ok, int m,
                                               int col) {
  if (row_ok && col < p.y_stride) {
    const size_t off = (size_t)m * (size_t)p.y_stride + (size_t)col;
    *reinterpret_cast<uint4*>(p.y_lo + off) = plane_lo(w);
    if (p.rq.out_planes == 2) *reinterpret_cast<uint4*>(p.y_hi + off) = plane_hi(w);
    if (p.y_q16 != nullptr) {
      uint4* dst = reinterpret_cast<uint4*>(p.y_q16 + off);
      dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
      dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
  }
}

// ... of eight outputs (8 bytes per plane)
__device__ __forceinline__ void store8_global(const uint32_t* w, const TcParams& p, bool row_ok, int m, int col) {
  if (row_ok && col < p.y_stride) {
    const size_t off = (size_t)m * (size_t)p.y_stride + (size_t)col;
    *reinterpret_cast<uint2*>(p.y_lo + off) = make_uint2(__byte_perm(w[0], w[1], 0x6420), __byte_perm(w[2], w[3], 0x6420));
    if (p.rq.out_planes == 2)
      *reinterpret_cast<uint2*>(p.y_hi + off) = make_uint2(__byte_perm(w[0], w[1], 0x7531), __byte_perm(w[2], w[3], 0x7531));
    if (p.y_q16 != nullptr) *reinterpret_cast<uint4*>(p.y_q16 + off) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Staged stores: the tile's byte planes are assembled in shared memory (rows of BN bytes, 16-byte
// chunks swizzled the way the bulk-tensor store expects for that row length, which also keeps the
// 16-byte writes of a quarter warp on distinct banks) and leave as one bulk-tensor store per plane.
// (Rows longer than the 128-byte swizzle span are kept as sub-planes of 128 columns, one store each.)
__device__ __forceinline__ uint32_t staged_offset(int row, int chunk, int bn, int rows = kBM) {
  const int sub = chunk >> 3;
  const int w = bn < 128 ? bn : 128;                       // row length of a (sub-)plane
  uint32_t off = (uint32_t)row * (uint32_t)w + (uint32_t)(chunk & 7) * 16u;
  off ^= ((off >> 7) & (uint32_t)((w >> 4) - 1) & 7u) << 4;
  return off + (uint32_t)sub * (uint32_t)(rows * 128);
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}
__device__ __forceinline__ void st_shared_v2(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void st_shared_b32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// 2x2 windows of a box tile: the four lanes of a window (they differ in lane bits 1 and `down`) hold sixteen channels of a
// pixel each.  Every exchange hands over the half that the partner keeps, so each lane ends with the maxima of four
// channels, `first` being the first of them.  16-bit values in pairs (eight words in, two out) or bytes 0 .. 127 (four in,
// one out).
template <bool BYTES, int WORDS>
__device__ __forceinline__ void window_max(uint32_t (&w)[WORDS], int lane, int down, int& first) {
  const bool right = (lane & 1) != 0, lower = (lane & down) != 0;
#pragma unroll
  for (int j = 0; j < WORDS / 2; ++j) {
    const uint32_t other = __shfl_xor_sync(0xffffffffu, right ? w[j] : w[j + WORDS / 2], 1);
    const uint32_t mine = right ? w[j + WORDS / 2] : w[j];
    w[j] = BYTES ? max_bytes7(mine, other) : max_s16x2(mine, other);
  }
#pragma unroll
  for (int j = 0; j < WORDS / 4; ++j) {
    const uint32_t other = __shfl_xor_sync(0xffffffffu, lower ? w[j] : w[j + WORDS / 4], down);
    const uint32_t mine = lower ? w[j + WORDS / 4] : w[j];
    w[j] = BYTES ? max_bytes7(mine, other) : max_s16x2(mine, other);
  }
  first = (right ? 8 : 0) + (lower ? 4 : 0);
}
__device__ __forceinline__ void store_window_max(uint32_t (&wq)[8], int lane, int down, int window, int chunk, const TcParams& p,
                                                 uint32_t stage_lo, uint32_t stage_hi) {
  int first;
  window_max<false>(wq, lane, down, first);
  const uint32_t off = staged_offset(window, chunk, p.BN, kBM / 4) + (uint32_t)first;
  st_shared_b32(stage_lo + off, __byte_perm(wq[0], wq[1], 0x6420));
  if (p.rq.out_planes == 2) st_shared_b32(stage_hi + off, __byte_perm(wq[0], wq[1], 0x7531));
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int x, int y, int z, int w) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(map),
               "r"(src), "r"(x), "r"(y), "r"(z), "r"(w)
               : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(map),
               "r"(src), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// the bulk stores committed so far have read their shared-memory source
__device__ __forceinline__ void bulk_wait_read_all() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// ... all but the most recent group have (two staging buffers in turn)
__device__ __forceinline__ void bulk_wait_read_all_but_one() {
  asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
}
// ... and have completed
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Barriers among the warps of one epilogue group only (barrier 0 belongs to __syncthreads; group g
// uses barriers 1 + 2g and 2 + 2g).
__device__ __forceinline__ void epi_bar_sync(int group, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + 2 * group), "r"(threads) : "memory");
}
// ... that also returns the conjunction of every thread's predicate
__device__ __forceinline__ bool epi_bar_all(int group, int threads, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n"
      ".reg .pred p, q;\n"
      "setp.ne.b32 p, %1, 0;\n"
      "bar.red.and.pred q, %2, %3, p;\n"
      "selp.u32 %0, 1, 0, q;\n"
      "}\n"
      : "=r"(r)
      : "r"((uint32_t)pred), "r"(2 + 2 * group), "r"(threads)
      : "memory");
  return r != 0;
}

// An epilogue warp hands accumulator columns back to the issuing warp (of the leader CTA in a pair).
template <bool PAIR>
__device__ __forceinline__ void release_accumulators(unsigned long long* bar_ptr, int lane) {
  tc_fence_before();
  __syncwarp();
  if (lane == 0) {
    const uint32_t bar = smem_u32(bar_ptr);
    if (PAIR)
      mbar_arrive_cluster(mapa_rank(bar, 0));
    else
      mbar_arrive(bar);
  }
}

// ---------------------------------------------------------------------------------- kernel
// LOOP: the form of the main loop, see kLoopPlain (GROUPED, PARTIAL and PIX below).
// EPI: the epilogue, see kEpiGeneric.  The 32-bit ones (FAST, FASTST) are launched for ReLU layers in requantizing mode whose
// shift lies in [9, 31] ([0, 31] with 8-bit operands on both sides), N a multiple of 8, no split-K, magnitudes within
// their bounds (fast_epilogue), and contain only that path.
// 20 warps: one block per SM, 96 registers per thread.
template <int NAX, int NBW, bool PAIR, int LOOP, int EPI>
__global__ void __launch_bounds__(kThreads, 1)
lp_gemm_kernel(const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_a1,
               const __grid_constant__ CUtensorMap map_b0, const __grid_constant__ CUtensorMap map_b1,
               const __grid_constant__ CUtensorMap map_y_hi, const __grid_constant__ CUtensorMap map_y_lo,
               const __grid_constant__ TcParams p) {
  constexpr int NACC = NAX + NBW - 1;
  constexpr int MAIN = LOOP & (kLoopBoxes - 1);
  constexpr bool GROUPED = MAIN == kLoopGrouped, PARTIAL = MAIN == kLoopPartial, PIX = MAIN == kLoopPixels;
  constexpr bool HALO = MAIN == kLoopHalo, TAPS = MAIN == kLoopTaps, BOX = HALO || TAPS || LOOP != MAIN;
  // (the exception that kLoopBoxes tells of)
  constexpr bool EITHER = LOOP == kLoopPartial + kLoopBoxes && EPI == kEpiFast;
  const bool boxes = BOX && (!EITHER || p.box.on != 0);
  const bool box_pool = boxes && ((LOOP != MAIN && !EITHER) || p.box.pool != 0);
  constexpr bool FAST = EPI == kEpiFast;
  // Where one copy serves all taps and a step is one product, the last copying warp issues MMAs too, every other tile: they
  // take the tensor core less time than one warp needs for its loop (64 channels: 105 cycles an instruction, 40 where
  // nothing else bounds them; 8 bits, 128 x 224 x 224 x 64 -> 64 340 -> 290 us).  With four products a step one warp
  // keeps up, and two tiles' instructions in turn cost the tensor core more (16 bits, 64 images 329 -> 453 us).
  constexpr int kIssuers = (HALO || TAPS) && NAX * NBW == 1 ? 2 : 1, kCopyWarps = kProducerWarps + 1 - kIssuers;
  constexpr bool STOCH = EPI == kEpiStochastic, FASTST = EPI == kEpiFastStochastic;
  extern __shared__ uint8_t smem_raw[];
  __shared__ Ctrl ctrl;

  const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);   // warp-uniform for the compiler too
  const int lane = threadIdx.x & 31;
  // PAIR: two CTAs (a cluster of two) share every tile of 256 rows.  Rank 0 is the leader: it owns
  // the "full" and "tmem_empty" barriers that are in use and issues the MMAs for both.
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
  const int worker = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const int workers = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  // rows of B this CTA stages per k-block, and where they start inside the tile's columns
  const int b_rows = PAIR ? p.BN / 2 : p.BN;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&ctrl.full[s]), 1);
      mbar_init(smem_u32(&ctrl.full[kMaxStages + s]), 1);
      mbar_init(smem_u32(&ctrl.empty[s]), 1);
    }
    for (int b = 0; b < kMaxAccBufs; ++b) {
      mbar_init(smem_u32(&ctrl.tmem_full[b]), 1);
      mbar_init(smem_u32(&ctrl.tmem_empty[b]), (uint32_t)((PAIR ? 2 : 1) * (kEpiWarps / p.epi_groups)));
    }
    mbar_init(smem_u32(&ctrl.part_full[0]), 1);
    mbar_init(smem_u32(&ctrl.part_full[1]), 1);
    mbar_init(smem_u32(&ctrl.drain[0]), 1);
    mbar_init(smem_u32(&ctrl.drain[1]), 1);
    mbar_init(smem_u32(&ctrl.b_ready), 1);
    ctrl.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    tmem_alloc<PAIR>(smem_u32(&ctrl.tmem_base), p.tmem_cols);
    tmem_relinquish<PAIR>();
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();      // the peer's barriers exist before anything signals them
  tc_fence_after();
  const uint32_t tmem_base = ctrl.tmem_base;
  // Everything above touched only this block's shared and tensor memory.  From here on global memory
  // is read (operands) and written (outputs, counters): wait for the previous kernel of the stream.
  pdl_wait();
  pdl_launch_dependents();

  if (warp < kCopyWarps) {
    // ------------------------------------------------------------------ TMA producers
    // Operand planes are numbered A planes first, then B planes.  Every producer warp walks the same
    // sequence of stages and issues only the copies of its own planes (warp w takes planes w and
    // w + 3), so the copies of a stage are in flight side by side.
    constexpr int NPLANES = NAX + NBW;
    // (whole warp in uniform control flow; one elected lane issues the copies)
    // Planes that are streamed through the ring: all of them, or only the activation planes when
    // the weights are resident.  With fewer streamed planes than producer warps, several warps
    // share a plane and take turns stage by stage.
    const bool b_res = PIX || HALO || TAPS || (GROUPED && p.b_resident);
    const int nact = b_res ? NAX : NPLANES;
    const int kps = GROUPED ? p.kps : 1;
    const int nsub = nact >= kCopyWarps ? 1 : kCopyWarps / nact;           // warps per streamed plane
    const int act_plane = nact >= kCopyWarps ? warp : warp % nact;
    const int sub = nact >= kCopyWarps ? 0 : warp / nact;
    const bool two_planes = act_plane + kCopyWarps < nact;                 // this warp also owns a second plane
    {
      const bool is_a = act_plane < NAX;
      const int plane = is_a ? act_plane : act_plane - NAX;
      const CUtensorMap* my_map = is_a ? (plane == 0 ? &map_a0 : &map_a1) : (plane == 0 ? &map_b0 : &map_b1);
      const uint32_t my_off = is_a ? (uint32_t)plane * p.a_bytes : NAX * p.a_bytes + (uint32_t)plane * p.b_bytes;
      // the second plane, if any, is the last B plane (plane index 3 of 4)
      const CUtensorMap* my_map2 = &map_b1;
      const uint32_t my_off2 = NAX * p.a_bytes + (uint32_t)(NBW - 1) * p.b_bytes;
      uint32_t it = 0, ph = 0;
      int s = 0, turn = 0;                     // turn: s modulo nsub
      bool ok = true;
      if (b_res && warp == kCopyWarps - 1) {
        // the whole weight matrix (of the single column tile, or of both that kLoopHalo may have), one copy per
        // k-block and plane, all reporting to one barrier
        // (in a pair each CTA fetches its own half of the weight rows; the bytes of both are counted
        // on the leader's barrier, which the leader arms for both)
        if (TAPS) {
          // a slab of 16-byte rows per tap (the one behind the last tap of an odd number arrives as zeros)
          if (elect_one()) {
            const uint32_t bar = smem_u32(&ctrl.b_ready);
            mbar_expect_tx(bar, NBW * p.b_bytes);
            for (int tap = 0; tap < p.b_blocks; ++tap)
              for (int bplane = 0; bplane < NBW; ++bplane)
                tma_load_3d<false>(ring + p.b_res_off + (uint32_t)bplane * p.b_bytes + (uint32_t)(tap * p.BN * 16),
                                   bplane == 0 ? &map_b0 : &map_b1, bar, 0, tap, 0);
          }
        } else if (PIX) {
          if (elect_one()) {
            const uint32_t bar = smem_u32(&ctrl.b_ready);
            mbar_expect_tx(bar, NBW * p.px.b_plane);
            uint32_t dst = ring + p.b_res_off;
            for (int row = 0; row < p.num_kb; row += p.px.blocks, dst += p.px.row_u * 16u) {
              const int r = p.div_s.quot(row);
              for (int tap = 0; tap < p.px.S; ++tap)
                for (int bplane = 0; bplane < NBW; ++bplane)
                  tma_load_2d<false>(dst + (uint32_t)bplane * p.px.b_plane + (uint32_t)((p.px.S - 1 - tap) * p.px.ys) * 32u,
                                     bplane == 0 ? &map_b0 : &map_b1, bar, (r * p.px.S + tap) * p.w_pitch, 0);
            }
          }
        } else if (elect_one()) {
          uint32_t bar = smem_u32(&ctrl.b_ready);
          const int tiles_n = HALO ? p.tiles_n : 1;
          if (rank == 0) mbar_expect_tx(bar, (PAIR ? 2u : 1u) * (uint32_t)(tiles_n * p.b_blocks) * NBW * p.b_bytes);
          if (PAIR) bar = mapa_rank(bar, 0);
          uint32_t dst = ring + p.b_res_off;
          for (int tn = 0; tn < tiles_n; ++tn)
            for (int kb = 0; kb < p.b_blocks; ++kb) {
              const int kcol = p.is_conv ? (kb / p.cblks) * p.w_pitch + (kb % p.cblks) * p.BK : kb * p.BK;
              for (int bplane = 0; bplane < NBW; ++bplane, dst += p.b_bytes)
                tma_load_2d<PAIR>(dst, bplane == 0 ? &map_b0 : &map_b1, bar, kcol, tn * p.BN + (int)rank * b_rows);
            }
        }
        __syncwarp();
      }
      const bool in_tile_loop = sub < nsub;
      bool stalled = false;
      int to = 0;                              // two issuing warps: the tile's row of barriers
      for (int t = worker; t < p.total_tiles && ok && in_tile_loop && !stalled;
           t += workers, to = kIssuers == 2 ? kMaxStages - to : 0) {
        const TileCoord tc = decode_tile(t, p);
        const int m_begin = tc.m0 + (int)rank * kBM;        // first of the 128 rows this CTA stages
        const int n_begin = tc.n0 + (int)rank * b_rows;     // first weight row this CTA stages
        int img = 0, base_h = 0, base_w = 0;
        int tap = 0, cb = 0, r = 0, sx = 0;       // position of kb in the (tap, channel block) order
        if (lane == 0 && warp == 0) TL_STAMP(0, (uint32_t)((t - worker) / workers), 0);
        if (boxes) {
          const BoxCoord bc = decode_box(m_begin >> 7, p.box);
          img = bc.img;
          base_w = bc.ow - p.pad_w;
          base_h = bc.oh - p.pad_h;
        } else if (p.is_conv) {
          const int rest = p.div_ow.quot(m_begin);
          const int ow = m_begin - rest * p.OW;
          img = p.div_oh.quot(rest);
          const int oh = rest - img * p.OH;
          base_w = ow * p.stride_w - p.pad_w;
          base_h = oh * p.stride_h - p.pad_h;
        }
        if (p.is_conv && !HALO && !TAPS) {
          tap = p.div_cblks.quot(tc.kb_begin);
          cb = tc.kb_begin - tap * p.cblks;
          r = p.div_s.quot(tap);
          sx = tap - r * p.S;
        }
        for (int kb = tc.kb_begin; kb < tc.kb_end; kb += kps, ++it) {
          if (it == (uint32_t)p.stall_at) { stalled = true; break; }
          const int nkb = GROUPED ? min(kps, tc.kb_end - kb) : 1;      // k-blocks in this stage
          const bool my_turn = turn == sub;           // ring slots have fixed owners
          if (++turn == nsub) turn = 0;
          if ((GROUPED || PIX || HALO || TAPS) && !my_turn) {
            if (++s == p.stages) { s = 0; ph ^= 1u; turn = 0; }
            continue;
          }
          if ((GROUPED || PIX) && nsub > 1 && p.is_conv) {     // (the stages in between were another warp's)
            tap = p.div_cblks.quot(kb);
            cb = kb - tap * p.cblks;
            r = p.div_s.quot(tap);
            sx = tap - r * p.S;
          }
          uint32_t full = 0, dst = 0;
          if (my_turn) {                                  // this warp's turn for its plane
            ok = __all_sync(0xffffffffu, wait_bar(smem_u32(&ctrl.empty[s]), ph ^ 1u, &ctrl, p));
            if (!ok) break;
            // bytes are reported to the leader's barrier; the leader arms it for both CTAs' copies
            full = smem_u32(&ctrl.full[s + to]);
            if (PAIR) full = mapa_rank(full, 0);
            dst = ring + (uint32_t)s * p.stage_bytes;
            if (act_plane == 0 && rank == 0 && elect_one())
              mbar_expect_tx(smem_u32(&ctrl.full[s + to]), (PAIR ? 2u : 1u) * (uint32_t)nkb * p.tx_bytes);
          }
          for (int j = 0; j < nkb; ++j) {
            if (my_turn && elect_one()) {
              if (TAPS) {
                tma_load_3d<PAIR>(dst + my_off, my_map, full, 2 * base_w, base_h, img);
              } else if (HALO) {
                tma_load_4d<PAIR>(dst + my_off, my_map, full, kb * p.BK, base_w, base_h, img);
              } else if (p.is_conv) {
                if (PIX) {
                  int d = sx + p.px.first;                     // (the block order begins with a full one)
                  if (d >= p.px.blocks) d -= p.px.blocks;
                  tma_load_im2col<false>(dst + my_off, my_map, full, 0, base_w, base_h, img, (uint16_t)d, (uint16_t)r);
                } else if (is_a && boxes)
                  tma_load_4d<PAIR>(dst + my_off, my_map, full, cb * p.BK, base_w + sx, base_h + r, img);
                else if (is_a)
                  tma_load_im2col<PAIR>(dst + my_off, my_map, full, cb * p.BK, base_w, base_h, img, (uint16_t)sx,
                                        (uint16_t)r);
                else
                  tma_load_2d<PAIR>(dst + my_off, my_map, full, tap * p.w_pitch + cb * p.BK, n_begin);
                if (two_planes)
                  tma_load_2d<PAIR>(dst + my_off2, my_map2, full, tap * p.w_pitch + cb * p.BK, n_begin);
              } else {
                tma_load_2d<PAIR>(dst + my_off, my_map, full, (kb + j) * p.BK, is_a ? m_begin : n_begin);
                if (two_planes) tma_load_2d<PAIR>(dst + my_off2, my_map2, full, (kb + j) * p.BK, n_begin);
              }
            }
            dst += p.kb_bytes;
            if (p.is_conv && !HALO && !TAPS) {
              if (++cb == p.cblks) {
                cb = 0;
                ++tap;
                if (++sx == p.S) { sx = 0; ++r; }
              }
            }
          }
          if (++s == p.stages) { s = 0; ph ^= 1u; turn = 0; }
        }
      }
      const bool is_b_loader = b_res && warp == kCopyWarps - 1;
      if (ctrl.abort && lane == 0 && is_b_loader) {
        // another role gave up: let the resident-weight copies land before the CTA exits (the
        // follower of a pair cannot see the leader's barrier: it waits a fixed time)
        const unsigned long long t0 = global_ns();
        if (PAIR && rank != 0) {
          while (global_ns() - t0 < 2000000ull) {
          }
        } else {
          while (!mbar_try_wait(smem_u32(&ctrl.b_ready), 0) && global_ns() - t0 < 50000000ull) {
          }
        }
      }
      if ((!ok || ctrl.abort) && lane == 0) {
        // gave up: let the copies already issued land before the CTA releases its shared memory.
        // (In a pair the bytes are counted on the leader's barriers, so the follower just waits.)
        const uint32_t n = it < (uint32_t)p.stages ? it : (uint32_t)p.stages;
        for (uint32_t j = it - n; j < it; ++j) {
          Fill f{j % (uint32_t)p.stages, (j / (uint32_t)p.stages) & 1u};
          if (kIssuers == 2) f = fill_of(j, (uint32_t)p.stages, (uint32_t)p.num_kb);
          const unsigned long long t0 = global_ns();
          if (PAIR && rank != 0) {
            while (global_ns() - t0 < 2000000ull) {
            }
            break;
          }
          while (!mbar_try_wait(smem_u32(&ctrl.full[f.bar]), f.parity) && global_ns() - t0 < 50000000ull) {
          }
        }
      }
    }
    __syncwarp();
  } else if (warp < kFirstEpiWarp) {
    // ------------------------------------------------------------------ MMA issuer (leader only)
    // The warp walks the stages in uniform control flow; one elected lane issues.
    if (rank == 0) {
      const int tile_rows = PAIR ? 2 * kBM : kBM;
      const int id_n = PIX ? 0 : p.BN;                              // (PIX: filled in step by step)
      const uint32_t id_ss = make_idesc(true, true, id_n, tile_rows);
      const uint32_t id_su = make_idesc(true, false, id_n, tile_rows);
      const uint32_t id_us = make_idesc(false, true, id_n, tile_rows);
      const uint32_t id_uu = make_idesc(false, false, id_n, tile_rows);
      const uint32_t dhi_b = smem_desc_hi(256, 6);                  // PIX: weight rows of 32 bytes
      const uint32_t dhi = smem_desc_hi(p.sbo, p.layout_type);
      // (weights of a tile that is copied with its margin: rows of their own; kLoopTaps gives leading offsets step by step)
      const uint32_t dhi_rows = TAPS ? smem_desc_hi(128, 0) : smem_desc_hi((uint32_t)(8 * p.BK), p.layout_type);
      const uint32_t ring_lo = TAPS ? smem_desc_lo(ring) - (1u << 16) : smem_desc_lo(ring);
      const uint32_t stage_u = p.stage_bytes >> 4, a_u = p.a_bytes >> 4, b_u = p.b_bytes >> 4;
      const uint32_t kb_u = p.kb_bytes >> 4;
      const uint32_t off_a1 = a_u, off_b0 = NAX * a_u;
      const int ksteps_full = p.ksteps;
      const uint32_t issuer = kIssuers == 2 && warp != kMmaWarp ? 1u : 0u;
      const uint32_t full_bar0 = smem_u32(&ctrl.full[issuer * kMaxStages]), empty_bar0 = smem_u32(&ctrl.empty[0]);
      uint32_t tile_iter = 0, ph = 0;      // (two issuing warps: bit s of ph is the parity of this warp's next fill of slot s)
      uint32_t a0 = ring_lo, full_bar = full_bar0, empty_bar = empty_bar0;
      int s = 0;
      bool ok = true;
      const bool b_res = PIX || HALO || TAPS || (GROUPED && p.b_resident);
      const int kps = GROUPED ? p.kps : 1;
      const uint32_t bres_lo = smem_desc_lo(ring + p.b_res_off) + (TAPS ? (uint32_t)(p.BN - 1) << 16 : 0u), bres_u = NBW * b_u;
      const uint32_t issue = HALO || TAPS ? (elect_one() ? 1u : 0u) : 0u;
      const int halo_r = p.halo.R, halo_s = p.halo.S;
      const uint32_t px_u = p.halo.px_u, row_u = (uint32_t)p.halo.w * px_u, tap_u = (uint32_t)p.cblks * bres_u;
      if (b_res) {
        ok = __all_sync(0xffffffffu, wait_bar(smem_u32(&ctrl.b_ready), 0u, &ctrl, p, false));
        tc_fence_after();
      }
      for (int t = worker; t < p.total_tiles && ok; t += workers, ++tile_iter) {
        if (kIssuers == 2 && (tile_iter & 1u) != issuer) {            // the other warp's tile: pass over its stages
          for (s += p.num_kb; s >= p.stages;) s -= p.stages;
          a0 = ring_lo + (uint32_t)s * stage_u;
          full_bar = full_bar0 + 8u * (uint32_t)s;
          empty_bar = empty_bar0 + 8u * (uint32_t)s;
          continue;
        }
        const TileCoord tc = decode_tile(t, p);
        const uint32_t buf = tile_iter & (uint32_t)(p.acc_bufs - 1);
        const uint32_t bph = (tile_iter >> p.acc_shift) & 1u;
        if (lane == 0) TL_STAMP(1, tile_iter, 0);
        ok = __all_sync(0xffffffffu, wait_bar(smem_u32(&ctrl.tmem_empty[buf]), bph ^ 1u, &ctrl, p, false));
        // split release: barrier 0 above covers the middle and low accumulators, barriers 1 and 2
        // the two places of the high one
        const uint32_t hh_sel = (NACC == 3 && p.split_hh) ? (tile_iter & 1u) : 0u;
        if (ok && NACC == 3 && p.split_hh)
          ok = __all_sync(0xffffffffu, wait_bar(smem_u32(&ctrl.tmem_empty[1u + hh_sel]), ((tile_iter >> 1) & 1u) ^ 1u,
                                                &ctrl, p, false));
        if (!ok) break;
        tc_fence_after();
        if (lane == 0) TL_STAMP(1, tile_iter, 1);
        // accumulator columns of this tile: the set's three (or fewer) consecutive groups of BN
        // columns, except that with the split release the first (high) one may sit in the last quarter
        const uint32_t dset = tmem_base + buf * (uint32_t)(NACC * p.BN);
        const uint32_t d0 = dset + hh_sel * (uint32_t)(3 * p.BN);
        const uint32_t d1 = dset + (uint32_t)p.BN, d2 = dset + 2u * (uint32_t)p.BN;
        uint32_t bres = bres_lo + (uint32_t)tc.kb_begin * bres_u;   // resident weights of this k-block
        if (HALO && tc.n0 != 0) bres += (uint32_t)p.b_blocks * bres_u;
        const bool stagger = !GROUPED && !PIX && !HALO && !TAPS && NAX == 2 && NBW == 2 && p.tail_stagger != 0;
        const int kb_main_end = stagger ? tc.kb_end - 2 : tc.kb_end;
        int cb = PARTIAL ? tc.kb_begin % p.cblks : 0;               // channel block of its tap
        int pb = 0;                                                 // block of input pixels
        uint32_t pb_row = bres_lo;                                  // weights of the filter row
        for (int kb = tc.kb_begin; kb < kb_main_end; kb += kps) {
          const int nkb = GROUPED ? min(kps, tc.kb_end - kb) : 1;
          int ksteps = ksteps_full;                                 // (fixed unless PARTIAL)
          if (PARTIAL) {
            if (cb == p.cblks - 1) ksteps = p.ksteps_last;
            if (++cb == p.cblks) cb = 0;
          }
          {
#ifdef ADAPTION_TIMELINE
          const long long tw0 = clock64();
#endif
          ok = __all_sync(0xffffffffu, wait_bar(full_bar, kIssuers == 2 ? (ph >> s) & 1u : ph, &ctrl, p, false));
          if (kIssuers == 2) ph ^= 1u << s;
#ifdef ADAPTION_TIMELINE
          if (lane == 0 && blockIdx.x == 0 && tile_iter < 32u)
            g_timeline[(1 * 32 + tile_iter) * 8 + 3] += clock64() - tw0;   // time waiting for data
#endif
          if (!ok) break;
          tc_fence_after();
          const uint32_t acc = kb == tc.kb_begin ? 0u : 1u;
          if (HALO) {
            // the taps of this channel block: the same copied rows from different pixels on
            uint32_t a = a0, b = bres + (uint32_t)kb * bres_u, first = acc;
            const int steps = kb == p.cblks - 1 ? p.ksteps_last : ksteps_full;
#pragma unroll 1
            for (int r = 0; r < halo_r; ++r) {
              uint32_t at = a;
#pragma unroll 1
              for (int sx = 0; sx < halo_s; ++sx) {
                mma_kblock_if<NAX, NBW, PAIR>(issue, d0, d1, d2, at, off_a1, b, b_u, dhi, dhi_rows, id_ss, id_su, id_us, id_uu,
                                              steps, first);
                first = 1u;
                at += px_u;
                b += tap_u;
              }
              a += row_u;
            }
            tc_commit_if<PAIR>(issue, empty_bar);              // stage reusable once these MMAs retire
          } else if (TAPS) {
            uint32_t b = bres_lo, first = 0u;
#pragma unroll 1
            for (int i = 0; i < p.halo.steps; ++i) {
              const uint32_t a = a0 + p.halo.a_lo[i];
              mma_kstep_if<NAX, NBW, false>(issue, d0, d1, d2, a, a + off_a1, b, b + b_u, dhi, dhi_rows, id_ss, id_su, id_us,
                                            id_uu, first);
              first = 1u;
              b += p.halo.b_row_u;
            }
            tc_commit_if<PAIR>(issue, empty_bar);
          } else if (elect_one()) {
            // a0 / ak: low descriptor word of the first A plane of a k-block; the other planes and
            // the k-steps are fixed offsets (16-byte units) from it (weights: in the stage or
            // resident).  The first k-block is straight-line code; grouped stages loop over the rest.
            if (PIX) {
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const uint32_t e = p.px.step[pb][i];
                if (e != 0u) {
                  const uint32_t col = e & 0x1ffu, n = e & ~0x1ffu, a = a0 + 2u * (uint32_t)i;
                  const uint32_t b = pb_row + p.px.b_row[pb][i];
                  mma_kstep<NAX, NBW, false>(d0 + col, d1 + col, d2 + col, a, a + off_a1, b, b + (p.px.b_plane >> 4), dhi,
                                             id_ss + n, id_su + n, id_us + n, id_uu + n, i == 0 ? acc : 1u, dhi_b);
                }
              }
            } else {
              mma_kblock<NAX, NBW, PAIR, PARTIAL>(d0, d1, d2, a0, off_a1, b_res ? bres : a0 + off_b0, b_u, dhi, id_ss, id_su,
                                                  id_us, id_uu, ksteps, acc);
            }
            if (GROUPED) {
              // (unrolled: a loop here costs the issuing thread more than the narrow MMAs take)
#pragma unroll
              for (int j = 1; j < 4; ++j)
                if (j < nkb) {
                  const uint32_t ak = a0 + (uint32_t)j * kb_u;
                  mma_kblock<NAX, NBW, PAIR, false>(d0, d1, d2, ak, off_a1, b_res ? bres + (uint32_t)j * bres_u : ak + off_b0,
                                                    b_u, dhi, id_ss, id_su, id_us, id_uu, ksteps, 1u);
                }
            }
            tc_commit<PAIR>(empty_bar);                        // stage reusable once these MMAs retire
          }
          }
          if (GROUPED) bres += (uint32_t)nkb * bres_u;
          if (PIX) {
            if (++pb == p.px.blocks) { pb = 0; pb_row += p.px.row_u; }
          }
          a0 += stage_u;
          full_bar += 8u;
          empty_bar += 8u;
          if (++s == p.stages) {
            s = 0;
            if (kIssuers == 1) ph ^= 1u;
            a0 = ring_lo;
            full_bar = full_bar0;
            empty_bar = empty_bar0;
          }
        }
        if (ok && stagger) {
          // The two last k-blocks together, product by product.  (Integer accumulation: the order of
          // the MMAs does not matter.)  Both stages are handed back at the end.
          uint32_t st_a[2], st_full[2], st_empty[2], st_ph[2];
          int st_ks[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            st_ks[j] = ksteps_full;
            if (PARTIAL) {
              if (cb == p.cblks - 1) st_ks[j] = p.ksteps_last;
              if (++cb == p.cblks) cb = 0;
            }
            st_a[j] = a0; st_full[j] = full_bar; st_empty[j] = empty_bar; st_ph[j] = ph;
            a0 += stage_u;
            full_bar += 8u;
            empty_bar += 8u;
            if (++s == p.stages) {
              s = 0;
              ph ^= 1u;
              a0 = ring_lo;
              full_bar = full_bar0;
              empty_bar = empty_bar0;
            }
          }
          ok = __all_sync(0xffffffffu, wait_bar(st_full[0], st_ph[0], &ctrl, p, false));
          if (ok) ok = __all_sync(0xffffffffu, wait_bar(st_full[1], st_ph[1], &ctrl, p, false));
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint32_t off_b1 = off_b0 + b_u;
#pragma unroll
            for (int j = 0; j < 2; ++j)
              for (int ks = 0; ks < st_ks[j]; ++ks)                     // lo * lo
                mma_i8<PAIR>(d2, st_a[j] + off_a1 + 2u * ks, st_a[j] + off_b1 + 2u * ks, dhi, id_uu, 1u);
            tc_commit<PAIR>(smem_u32(&ctrl.part_full[0]));
#pragma unroll
            for (int j = 0; j < 2; ++j)
              for (int ks = 0; ks < st_ks[j]; ++ks) {                   // hi * lo and lo * hi
                mma_i8<PAIR>(d1, st_a[j] + 2u * ks, st_a[j] + off_b1 + 2u * ks, dhi, id_su, 1u);
                mma_i8<PAIR>(d1, st_a[j] + off_a1 + 2u * ks, st_a[j] + off_b0 + 2u * ks, dhi, id_us, 1u);
              }
            tc_commit<PAIR>(smem_u32(&ctrl.part_full[1]));
#pragma unroll
            for (int j = 0; j < 2; ++j)
              for (int ks = 0; ks < st_ks[j]; ++ks)                     // hi * hi
                mma_i8<PAIR>(d0, st_a[j] + 2u * ks, st_a[j] + off_b0 + 2u * ks, dhi, id_ss, 1u);
            tc_commit<PAIR>(st_empty[0]);
            tc_commit<PAIR>(st_empty[1]);
          }
        }
        if (ok && elect_one()) tc_commit<PAIR>(smem_u32(&ctrl.tmem_full[buf]));   // tile complete
        __syncwarp();
        if (lane == 0) TL_STAMP(1, tile_iter, 2);
      }
      if ((!ok || ctrl.abort) && lane == 0) {
        // make sure no MMA still reads shared memory or writes TMEM when the CTAs tear down
        tc_commit<PAIR>(smem_u32(&ctrl.drain[issuer]));
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(smem_u32(&ctrl.drain[issuer]), 0) && global_ns() - t0 < 50000000ull) {
        }
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue warps
    const int quarter = warp & 3;          // TMEM lanes 32*quarter .. 32*quarter+31
    // With several accumulator sets the warps form groups that take turns tile by tile (each with an
    // accumulator set, barriers, constants and staging planes of its own), so that one group's waits and
    // TMEM loads overlap the others' arithmetic.
    const int groups = p.epi_groups;
    const int gwarps = kEpiWarps / groups, gthreads = 32 * gwarps;
    const int group = (warp - kFirstEpiWarp) / gwarps;
    const int ew = (warp - kFirstEpiWarp) - group * gwarps;      // warp index within its group
    // the warps of a lane quarter split the columns of the tile
    const int cols_per_warp = max(16, p.BN / (gwarps / 4));
    const int col_begin = min(p.BN, (ew >> 2) * cols_per_warp);
    const int col_end = min(p.BN, col_begin + cols_per_warp);
    const int row = quarter * 32 + lane;   // row of the tile (and of this CTA's staging planes)
    const int plane_rows = box_pool ? kBM / 4 : kBM;
    const int plane_bytes = plane_rows * (PIX && p.pool_w ? p.BN >> 1 : p.BN);
    const int planes_bytes = plane_bytes * p.rq.out_planes;
    // box tiles: the lane of the pixel below, and the row of the stored tile that a 2x2 window becomes
    const int down = 1 << p.box.w;
    const int pool = box_pool ? 1 : 0;
    const int window = ((row >> (p.box.w + 1)) << (p.box.w - pool)) | ((row & (down - 1)) >> 1);
    const uint32_t stage_group = ring + p.stage_off + (uint32_t)(group * planes_bytes * p.stage_bufs);
    uint32_t stage_lo = stage_group;
    uint32_t stage_hi = stage_lo + (uint32_t)plane_bytes;
    uint32_t stage_turn = 0;
    // per-column epilogue constants of the current tile, one array per group, behind the staging planes
    // (one per warp where warps work by themselves: then no barrier separates readers and writers)
    const bool own = (HALO || TAPS || EITHER) && p.own_rows != 0;
    long long* colconst = reinterpret_cast<long long*>(smem_raw + (ring - smem_u32(smem_raw)) + p.const_off) +
                          (own ? warp - kFirstEpiWarp : group) * p.BN;
    const bool store_leader = (own || ew == 0) && lane == 0;
    uint32_t tile_iter = (uint32_t)group;
    Counts cnt;
    long long vmax = 0;
    int32_t key = 0;
    bool ok = true;
    int const_n0 = -1;          // first column of the tile whose constants are staged
    for (int t = worker + group * workers; t < p.total_tiles; t += groups * workers, tile_iter += (uint32_t)groups) {
      const TileCoord tc = decode_tile(t, p);
      const uint32_t buf = tile_iter & (uint32_t)(p.acc_bufs - 1);
      const uint32_t bph = (tile_iter >> p.acc_shift) & 1u;
      // per-column constants of this tile (the last barrier of the previous tile separates these
      // writes from its readers): bias aligned to the accumulator, plus the rounding half on the
      // fast path.  Kept when the tile covers the same columns as the previous one.
      if (tc.n0 != const_n0) {
        for (int c = own ? lane : 32 * ew + lane; c < p.BN; c += own ? 32 : gthreads) {
          const int n = tc.n0 + c;
          long long b = 0;
          const int ch = PIX ? n & (p.px.ys - 1) : n;
          if (p.bias != nullptr && ch < (PIX ? p.px.n_valid : p.N) && p.splits == 1)
            b = (long long)p.bias[ch] * (1ll << p.bias_shift);
          if (FAST || FASTST || (EPI == kEpiGeneric && p.fast_range)) {
            // two arrays of BN 32-bit words: C mod 2^16 and C div 2^16 (a single accumulator takes all
            // of C from the first), read four columns per load
            const long long C = b + (FAST && p.rq.shift > 0 ? 1ll << (p.rq.shift - 1) : 0ll);
            int* cw = reinterpret_cast<int*>(colconst);
            cw[c] = NACC == 1 ? (int)C : (int)(C & 0xffff);
            cw[p.BN + c] = (int)(C >> 16);
          } else {
            colconst[c] = b;
          }
        }
        const_n0 = tc.n0;
      }
      // the previous tile's bulk stores must have read the staging planes before they are reused
      // (with two buffers in turn: the store from two tiles ago)
      if (p.stage_bufs == 2) {
        stage_lo = stage_group + stage_turn * (uint32_t)planes_bytes;
        stage_hi = stage_lo + (uint32_t)plane_bytes;
        stage_turn ^= 1u;
        if (p.staged && store_leader) bulk_wait_read_all_but_one();
      } else if (p.staged && store_leader) {
        bulk_wait_read_all();
      }
      if (lane == 0 && (ew & 3) == 0) TL_STAMP(2 + (ew >> 2), tile_iter, 0);
      // (staggered tail: the first thing to wait for is the low accumulator)
      const bool stagger = FAST && NACC == 3 && p.tail_stagger != 0;
      bool w = wait_bar(smem_u32(stagger ? &ctrl.part_full[0] : &ctrl.tmem_full[buf]), bph, &ctrl, p);
      // one decision for all epilogue warps (they meet at barriers below), which also publishes the
      // constants and the free staging planes
      if (own) {
        w = __all_sync(0xffffffffu, w);
        __syncwarp();
      } else {
        w = epi_bar_all(group, gthreads, w);
      }
      if (lane == 0 && (ew & 3) == 0) TL_STAMP(2 + (ew >> 2), tile_iter, 1);
      if (!w) { ok = false; break; }
      tc_fence_after();
      int m = tc.m0 + (int)rank * kBM + row;
      bool row_ok = m < p.M;
      BoxCoord bc{0, 0, 0};
      if (boxes) {
        bc = decode_box(m >> 7, p.box);
        const int ow = bc.ow + (row & (down - 1)), oh = bc.oh + ((row >> p.box.w) & ((1 << p.box.h) - 1));
        const int img = bc.img + (row >> (p.box.w + p.box.h));
        row_ok = ow < p.OW && oh < p.OH && img < p.box.images;
        m = (img * p.OH + oh) * p.OW + ow;
      }
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * (uint32_t)(NACC * p.BN);
      // where this tile's high accumulator lives, and the barrier that hands it back
      const bool split = NACC == 3 && p.split_hh != 0;
      const uint32_t hh_sel = split ? (tile_iter & 1u) : 0u;
      const uint32_t hh_off = hh_sel * (uint32_t)(3 * p.BN);
      unsigned long long* const bar_rest = &ctrl.tmem_empty[buf];
      unsigned long long* const bar_hh = split ? &ctrl.tmem_empty[1u + hh_sel] : bar_rest;
      // Sixteen columns per step.  The accumulators are handed back to the issuing warp as soon as
      // the last step's values are in registers, before the arithmetic on them.
      const bool storing = FAST || FASTST || (p.splits == 1 && p.mode == ADAPTION_MODE_REQUANT);
      bool released = false;
      bool tile_ok = true;        // a later wait of this tile gave up: finish the tile, then leave together
      // Fast path with thirty-two columns per warp step: one TMEM load per accumulator, the low and
      // middle accumulators first (they fold into T), the high one last; the accumulators go back
      // to the issuing warp as soon as the last load has landed.
      // (the host launches the FAST kernels only where every warp owns a multiple of 32 columns)
      if (FAST) {
        if (col_begin >= col_end) {          // a warp without columns only hands the accumulators back
          release_accumulators<PAIR>(bar_rest, lane);
          if (split) release_accumulators<PAIR>(bar_hh, lane);
          released = true;
        }
        for (int cv = col_begin; cv < col_end; cv += 32) {
          int32_t t[32], h[32];
          // two runs of sixteen columns, next to each other; grouped pixels that are pooled in pairs: the same
          // channels of two neighbouring pixels
          int c0 = cv, run = 16;
          const bool pool_px = PIX && p.pool_w != 0;
          if (pool_px) {
            run = p.px.ys;
            c0 = (cv & ~(2 * run - 1)) + ((cv & (2 * run - 1)) >> 1);
          }
          const int4* cl4 = reinterpret_cast<const int4*>(reinterpret_cast<const int*>(colconst) + c0);
          const int4* ch4 = reinterpret_cast<const int4*>(reinterpret_cast<const int*>(colconst) + p.BN + c0);
          const int run4 = (run >> 2) - 4;       // what the second run's constants are further on
          const auto load32 = [&](uint32_t at, int32_t (&r)[32]) {
            if (PIX)
              tmem_ld16x2(at, (uint32_t)run, r);
            else
              tmem_ld32(at, r);
          };
          if (NACC == 3) {
            load32(taddr + (uint32_t)(c0 + 2 * p.BN), t);       // ll
            if (!stagger) load32(taddr + (uint32_t)(c0 + p.BN), h);   // mid
          } else if (NACC == 2) {
            load32(taddr + (uint32_t)(c0 + p.BN), t);           // weight 1
            load32(taddr + (uint32_t)c0, h);                    // weight 2^8
          } else {
            load32(taddr + (uint32_t)c0, t);
          }
          tmem_ld_wait();
          pin_after_wait32(t);
          if (NACC >= 2 && !stagger) pin_after_wait32(h);
          if (NACC == 3 && stagger) {
            // fold the constant into the low accumulator while the middle one completes, then fetch it
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int4 c = cl4[j + (PIX && j >= 4 ? run4 : 0)];
              t[4 * j + 0] = (t[4 * j + 0] + c.x) >> 8;
              t[4 * j + 1] = (t[4 * j + 1] + c.y) >> 8;
              t[4 * j + 2] = (t[4 * j + 2] + c.z) >> 8;
              t[4 * j + 3] = (t[4 * j + 3] + c.w) >> 8;
            }
            tile_ok = wait_bar_inline(smem_u32(&ctrl.part_full[1]), bph, &ctrl, p) && tile_ok;
            tc_fence_after();
            load32(taddr + (uint32_t)(c0 + p.BN), h);           // mid
            tmem_ld_wait();
            pin_after_wait32(h);
#pragma unroll
            for (int j = 0; j < 32; ++j) t[j] += h[j];             // T
          }
          // the low and middle accumulators are in registers: with the split release they go back now
          if (split && cv + 32 >= col_end) {
            release_accumulators<PAIR>(bar_rest, lane);
            if (lane == 0 && (ew & 3) == 0) TL_STAMP(2 + (ew >> 2), tile_iter, 3);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (NACC == 3 && stagger) break;
            const int4 c = cl4[j + (PIX && j >= 4 ? run4 : 0)];
            if (NACC >= 2) {                                       // T = mid + floor((ll + Cl) / 2^8)
              t[4 * j + 0] = h[4 * j + 0] + ((t[4 * j + 0] + c.x) >> 8);
              t[4 * j + 1] = h[4 * j + 1] + ((t[4 * j + 1] + c.y) >> 8);
              t[4 * j + 2] = h[4 * j + 2] + ((t[4 * j + 2] + c.z) >> 8);
              t[4 * j + 3] = h[4 * j + 3] + ((t[4 * j + 3] + c.w) >> 8);
            } else {
              t[4 * j + 0] += c.x; t[4 * j + 1] += c.y; t[4 * j + 2] += c.z; t[4 * j + 3] += c.w;
            }
          }
          if (NACC == 3) {
            if (stagger) {
              tile_ok = wait_bar_inline(smem_u32(&ctrl.tmem_full[buf]), bph, &ctrl, p) && tile_ok;
              tc_fence_after();
            }
            load32(taddr + hh_off + (uint32_t)c0, h);           // hh
            tmem_ld_wait();
            pin_after_wait32(h);
          }
          if (cv + 32 >= col_end) {
            release_accumulators<PAIR>(bar_hh, lane);
            if (lane == 0 && (ew & 3) == 0) TL_STAMP(2 + (ew >> 2), tile_iter, 4);
            released = true;
          }
          if (NACC >= 2) {                                         // H = hh + Ch
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int4 c = ch4[j + (PIX && j >= 4 ? run4 : 0)];
              if (NACC == 3) {
                h[4 * j + 0] += c.x; h[4 * j + 1] += c.y; h[4 * j + 2] += c.z; h[4 * j + 3] += c.w;
              } else {
                h[4 * j + 0] = c.x; h[4 * j + 1] = c.y; h[4 * j + 2] = c.z; h[4 * j + 3] = c.w;
              }
            }
          }
          const bool wide = NACC == 1 || p.rq.shift >= 16;
          uint32_t left[8];
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            uint32_t wq[8];
            const int col = tc.n0 + c0 + half * run;
            if (NACC == 1 && p.byte_out) {
              uint32_t b[4];
              fast_bytes16<PIX>(t, half, p.rq.shift, row_ok, col, p, cnt, b);
              if (box_pool) {
                int first;
                window_max<true>(b, lane, down, first);
                st_shared_b32(stage_lo + staged_offset(window, (c0 >> 4) + half, p.BN, kBM / 4) + (uint32_t)first, b[0]);
                continue;
              }
              uint32_t at = staged_offset(row, (c0 >> 4) + half, p.BN);
              bool mine = true;
              if (pool_px) {
#pragma unroll
                for (int j = 0; j < 4; ++j) left[j] = b[j] = half == 0 ? b[j] : max_bytes7(left[j], b[j]);
                at = staged_offset(row, cv >> 5, p.BN >> 1);
                mine = half == 1;
              } else if (p.pool_w) {
#pragma unroll
                for (int j = 0; j < 4; ++j) b[j] = max_bytes7(b[j], __shfl_xor_sync(0xffffffffu, b[j], 1));
                at = staged_offset(row >> 1, (c0 >> 4) + half, p.BN);
                mine = (lane & 1) == 0;
              }
              if (mine) st_shared_v4(stage_lo + at, make_uint4(b[0], b[1], b[2], b[3]));
              continue;
            }
            if (wide)
              fast_outputs16<NACC, true, PIX>(t, h, half, p.rq.shift, p.rq.qmax, row_ok, col, p, cnt, wq);
            else
              fast_outputs16<NACC, false, PIX>(t, h, half, p.rq.shift, p.rq.qmax, row_ok, col, p, cnt, wq);
            const int chunk = (c0 >> 4) + half;
            if (box_pool) {
              store_window_max(wq, lane, down, window, chunk, p, stage_lo, stage_hi);
            } else if (pool_px) {
              // the right pixel of a pair: its maximum with the left one, one chunk of the pooled row
#pragma unroll
              for (int j = 0; j < 8; ++j) left[j] = half == 0 ? wq[j] : max_s16x2(left[j], wq[j]);
              if (half == 1) {
                const uint32_t off = staged_offset(row, cv >> 5, p.BN >> 1);
                st_shared_v4(stage_lo + off, plane_lo(left));
                if (p.rq.out_planes == 2) st_shared_v4(stage_hi + off, plane_hi(left));
              }
            } else if (p.staged && p.pool_w) {
#pragma unroll
              for (int j = 0; j < 8; ++j) wq[j] = max_s16x2(wq[j], __shfl_xor_sync(0xffffffffu, wq[j], 1));
              if ((lane & 1) == 0) {
                const uint32_t off = staged_offset(row >> 1, chunk, p.BN);
                st_shared_v4(stage_lo + off, plane_lo(wq));
                if (p.rq.out_planes == 2) st_shared_v4(stage_hi + off, plane_hi(wq));
              }
            } else if (p.staged) {
              const uint32_t off = staged_offset(row, chunk, p.BN);
              st_shared_v4(stage_lo + off, plane_lo(wq));
              if (p.rq.out_planes == 2) st_shared_v4(stage_hi + off, plane_hi(wq));
            } else {
              store16_global(wq, p, row_ok, m, col);
            }
          }
        }
      }
      if (STOCH || FASTST) {
        // Stochastic rounding: a rolled loop over eight columns.  The generator's rounds are long straight-line code: with
        // sixteen columns a step (eight blocks of it) the warps waited for instructions (16 images, 3 -> 16 channels at
        // 224 x 224, 1x1: 61 us with sixteen, 48 with eight, 7x7 over 16 channels at 112 x 112 81 and 69, 64 -> 64 47 and 39; the
        // generator's rounds as a loop: 53, 69, 43).
#pragma unroll 1
        for (int c0 = col_begin; c0 < col_end; c0 += 8) {
          const int col = tc.n0 + c0;
          Acc8<NACC> v;
          load_acc8<NACC>(taddr + (uint32_t)c0, hh_off, p.BN, v);
          tmem_ld_wait();
          pin_acc8<NACC>(v);
          if (c0 + 8 >= col_end) {
            release_accumulators<PAIR>(bar_rest, lane);
            if (split) release_accumulators<PAIR>(bar_hh, lane);
            released = true;
          }
          uint32_t wq[4];
          if (FASTST) {
            const int* cl = reinterpret_cast<const int*>(colconst) + c0;
            stochastic8<NACC, PIX>(v, cl, cl + p.BN, p, row_ok, m, col, cnt, wq);
          } else if (p.rq.relu) {
            requant8<NACC, true, true, PIX>(v, colconst + c0, p, row_ok, m, col, cnt, wq);
          } else {
            requant8<NACC, false, true, PIX>(v, colconst + c0, p, row_ok, m, col, cnt, wq);
          }
          if (p.staged) {
            const uint32_t off = staged_offset(row, c0 >> 4, p.BN) + (uint32_t)(c0 & 8);
            st_shared_v2(stage_lo + off, __byte_perm(wq[0], wq[1], 0x6420), __byte_perm(wq[2], wq[3], 0x6420));
            if (p.rq.out_planes == 2)
              st_shared_v2(stage_hi + off, __byte_perm(wq[0], wq[1], 0x7531), __byte_perm(wq[2], wq[3], 0x7531));
          } else {
            store8_global(wq, p, row_ok, m, col);
          }
        }
        if (!released) {                     // a warp without columns only hands the accumulators back
          release_accumulators<PAIR>(bar_rest, lane);
          if (split) release_accumulators<PAIR>(bar_hh, lane);
          released = true;
        }
      }
      for (int c0 = col_begin; !FAST && !STOCH && !FASTST && (c0 < col_end || !released); c0 += 16) {
        const bool have = c0 < col_end;
        Acc8<NACC> xa, xb;
        if (have) {
          load_acc16<NACC>(taddr + c0, hh_off, p.BN, xa, xb);
          tmem_ld_wait();
          pin_acc8<NACC>(xa);
          pin_acc8<NACC>(xb);
        }
        if (c0 + 16 >= col_end) {
          release_accumulators<PAIR>(bar_rest, lane);
          if (split) release_accumulators<PAIR>(bar_hh, lane);
          released = true;
        }
        if (!have) break;
        const int col = tc.n0 + c0;
        const long long* bcol = colconst + c0;
        if (EPI == kEpiGeneric && p.fast_range) {
          const int* cl = reinterpret_cast<const int*>(colconst) + c0;
          fast_range8<NACC>(xa, cl, cl + p.BN, p, row_ok, vmax, key);
          fast_range8<NACC>(xb, cl + 8, cl + p.BN + 8, p, row_ok, vmax, key);
        } else if (!storing) {
          partial_or_range8<NACC, PIX>(xa, bcol, p, row_ok, m, col, vmax);
          partial_or_range8<NACC, PIX>(xb, bcol + 8, p, row_ok, m, col + 8, vmax);
        } else {
          uint32_t wq[8];
          if (p.rq.relu) {
            requant8<NACC, true, false, PIX>(xa, bcol, p, row_ok, m, col, cnt, wq);
            requant8<NACC, true, false, PIX>(xb, bcol + 8, p, row_ok, m, col + 8, cnt, wq + 4);
          } else {
            requant8<NACC, false, false, PIX>(xa, bcol, p, row_ok, m, col, cnt, wq);
            requant8<NACC, false, false, PIX>(xb, bcol + 8, p, row_ok, m, col + 8, cnt, wq + 4);
          }
          if (box_pool) {
            store_window_max(wq, lane, down, window, c0 >> 4, p, stage_lo, stage_hi);
          } else if (p.staged && p.pool_w) {
            // Horizontal half of a 2x2 max-pool: rows 2j and 2j+1 of the tile are neighbouring
            // pixels of one image row (even width, tiles start at even rows) and sit in neighbouring
            // lanes; the maximum of the packed 16-bit values is stored once, as row j.
#pragma unroll
            for (int j = 0; j < 8; ++j) wq[j] = max_s16x2(wq[j], __shfl_xor_sync(0xffffffffu, wq[j], 1));
            if ((lane & 1) == 0) {
              const uint32_t off = staged_offset(row >> 1, c0 >> 4, p.BN);
              st_shared_v4(stage_lo + off, plane_lo(wq));
              if (p.rq.out_planes == 2) st_shared_v4(stage_hi + off, plane_hi(wq));
            }
          } else if (p.staged) {
            const uint32_t off = staged_offset(row, c0 >> 4, p.BN);
            st_shared_v4(stage_lo + off, plane_lo(wq));
            if (p.rq.out_planes == 2) st_shared_v4(stage_hi + off, plane_hi(wq));
          } else {
            store16_global(wq, p, row_ok, m, col);
          }
        }
      }
      // staged planes complete -> one bulk-tensor store per plane (rows beyond M and columns beyond
      // the channel pitch are clipped by the tensor map); the barrier also ends this tile's reads
      // of the per-column constants
      if (p.staged) fence_async_shared();
      if (stagger) {
        // the same barrier also carries the verdict on this tile's later waits, so that all warps
        // of the group leave together if one of them gave up
        if (!epi_bar_all(group, gthreads, tile_ok)) { ok = false; break; }
      } else if (own) {
        __syncwarp();
      } else {
        epi_bar_sync(group, gthreads);
      }
      if (own && p.staged && store_leader) {
        // this warp's rows (a quarter of the tile, whose stored rows are consecutive whatever the pool)
        const int first = 32 * quarter;
        const uint32_t so = (uint32_t)(quarter * (plane_bytes >> (p.pool_w && !PIX ? 3 : 2)));
        if (boxes) {
          const int oh = (bc.oh + ((first >> p.box.w) & ((1 << p.box.h) - 1))) >> pool, ow = bc.ow >> pool;
          const int img = bc.img + (first >> (p.box.w + p.box.h));
          tma_store_4d(&map_y_lo, stage_lo + so, tc.n0, ow, oh, img);
          if (p.rq.out_planes == 2) tma_store_4d(&map_y_hi, stage_hi + so, tc.n0, ow, oh, img);
        } else {
          const int m_first = (tc.m0 + (int)rank * kBM + first) >> (p.pool_w && !PIX ? 1 : 0);
          tma_store_2d(&map_y_lo, stage_lo + so, tc.n0, m_first);
          if (p.rq.out_planes == 2) tma_store_2d(&map_y_hi, stage_hi + so, tc.n0, m_first);
        }
        bulk_commit();
      } else if (boxes && p.staged && store_leader) {
        const int ow = bc.ow >> pool, oh = bc.oh >> pool;
        for (int sub = 0; sub * 128 < p.BN; ++sub) {
          const uint32_t so = (uint32_t)sub * (uint32_t)(plane_rows * 128);
          tma_store_4d(&map_y_lo, stage_lo + so, tc.n0 + sub * 128, ow, oh, bc.img);
          if (p.rq.out_planes == 2) tma_store_4d(&map_y_hi, stage_hi + so, tc.n0 + sub * 128, ow, oh, bc.img);
        }
        bulk_commit();
      } else if (p.staged && store_leader) {
        const int m_first = (tc.m0 + (int)rank * kBM) >> (p.pool_w && !PIX ? 1 : 0);     // row of the stored tensor
        const int y_cols = PIX && p.pool_w ? p.BN >> 1 : p.BN;
        for (int sub = 0; sub * 128 < y_cols; ++sub) {
          const uint32_t so = (uint32_t)sub * (uint32_t)(kBM * 128);
          tma_store_2d(&map_y_lo, stage_lo + so, tc.n0 + sub * 128, m_first);
          if (p.rq.out_planes == 2) tma_store_2d(&map_y_hi, stage_hi + so, tc.n0 + sub * 128, m_first);
        }
        bulk_commit();
      }
      if (lane == 0 && (ew & 3) == 0) TL_STAMP(2 + (ew >> 2), tile_iter, 2);
    }
    (void)ok;
    if (p.staged && store_leader) bulk_wait_all();
    if (p.splits == 1) {
      if (p.mode == ADAPTION_MODE_RANGE)
        flush_max_warp(vmax, p.stats);
      else
        flush_counts_warp(cnt, p.stats);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();      // neither CTA leaves (or frees TMEM) while the other may still signal it
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc<PAIR>(tmem_base, p.tmem_cols);
  }
}

// ---------------------------------------------------------------------------------- host
struct TcConfig {
  bool ok = false;
  int BN = 0, BK = 0;
  CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_NONE;
  uint32_t layout_type = 0;
  int nax = 1, nbw = 1, nacc = 1;
  int stages = 0;
  uint32_t a_bytes = 0, b_bytes = 0, stage_bytes = 0;
  int a_rows = kBM;            // rows of the activation tile that are staged
  int acc_bufs = 1;
  uint32_t tmem_cols = 32;
  int num_kb = 0, splits = 1, kb_per_split = 0;
  int tiles_m = 0, tiles_n = 0;
  int cblks = 1, ksteps_last = 0;
  bool b_resident = false;
  uint32_t b_res_bytes = 0;
  int kps = 1;
  uint32_t kb_bytes = 0;
  bool pair = false;           // two CTAs per 256-row tile (cta_group::2)
  int tile_m = kBM;
  int epi_groups = 1;
  bool own_rows = false;
  bool staged = false;         // outputs staged in shared memory and written by bulk-tensor stores
  uint32_t stage_out_bytes = 0, stage_off = 0, const_bytes = 0;
  int stage_bufs = 1;
  size_t smem_bytes = 0;
  size_t workspace_bytes = 0;
  PixelPlan px{};              // px.G > 1: pixels grouped (make_pixel_config)
  BoxPlan box{};               // box.on: tiles are boxes of pixels
  HaloPlan halo{};             // halo.w > 0: one copy of activations for all taps (make_halo_config)
  int b_blocks = 0;            // weight k-blocks that are resident
  uint32_t a_tx = 0;           // bytes of one copy of activations, where they are not a_bytes
};

// Boxes of 2^w x 2^h x 2^n pixels over OW x OH pixels of `images` images.
BoxPlan box_plan(int w, int h, int n, int OW, int OH, int images, bool pool) {
  BoxPlan b{};
  b.on = 1;
  b.pool = pool ? 1 : 0;
  b.w = w; b.h = h; b.n = n;
  b.images = images;
  b.tiles_w = (OW + (1 << w) - 1) >> w;
  b.tiles_h = (OH + (1 << h) - 1) >> h;
  b.div_w = fast_div(b.tiles_w);
  b.div_h = fast_div(b.tiles_h);
  return b;
}
int64_t box_count(const BoxPlan& b) {
  return (int64_t)b.tiles_w * b.tiles_h * ((b.images + (1 << b.n) - 1) >> b.n);
}
// The boxes of 128 pixels with whole 2x2 windows that cover a layer with the fewest tiles, wide ones before narrow ones.
// A window's rows have to lie in one warp of 32: at most 16 columns.  (box.on = 0: more than one tile in sixteen would be
// margin; the pooling pass that boxes save takes 7 to 20 % of the layer.)
BoxPlan pool_boxes(const GemmProblem& g) {
  BoxPlan best{};
  int64_t fewest = 0;
  for (int w = 4; w >= 1; --w)
    for (int h = 7 - w; h >= 1; --h) {
      const BoxPlan b = box_plan(w, h, 7 - w - h, g.OW, g.OH, g.cs.N, true);
      const int64_t n = box_count(b);
      if (!best.on || n < fewest) {
        best = b;
        fewest = n;
      }
    }
  if (fewest * kBM * 16 > g.M * 17 || fewest > (1 << 23)) best.on = 0;
  return best;
}

TcConfig make_config_impl(const GemmProblem& g, bool allow_wide);

// 256-column tiles only exist as CTA pairs: if the wide attempt does not end up paired (the
// reduction gets split, say), the ordinary configuration is taken.
TcConfig make_config(const GemmProblem& g) {
  TcConfig c = make_config_impl(g, true);
  if (c.BN == 256 && !(c.ok && c.pair)) c = make_config_impl(g, false);
  return c;
}

TcConfig make_config_impl(const GemmProblem& g, bool allow_wide) {
  TcConfig c;
  if (g.M <= 0 || g.N <= 0 || g.M > (int64_t)1 << 30 || g.N > (int64_t)1 << 24) return c;
  c.nax = g.x.fmt.n_bits > 8 ? 2 : 1;
  c.nbw = g.w.fmt.n_bits > 8 ? 2 : 1;
  c.nacc = c.nax + c.nbw - 1;
  int64_t k_padded;
  if (g.is_conv) {
    const int64_t cs = g.x.c_stride;
    if (cs != g.w.c_stride || cs % 32 != 0 || cs > 65536) return c;
    // k-blocks of 128 bytes as soon as there are more than 64: bulk copies deliver one row per two cycles
    // whatever its length, so narrow blocks cost as many rows each.  Where the pitch is no multiple of 128 the
    // last block of a tap reaches past the pitch (the copy fills zeros without reading) and the MMAs skip
    // the steps that are not there (in a grouped main loop they multiply the zeros: those loops wait for copies).
    // 3x3 layers before -> now: 12 x 45 x 37 x 96 -> 168 at 12 bits 29.6 -> 25.0 us, 16 x 56 x 56 x 160 -> 128 at 16
    // bits 44.8 -> 34.0, 16 x 56 x 56 x 96 -> 256 at 8 bits 34.8 -> 20.3.
    c.BK = cs > 64 ? 128 : (int)cs;
    c.cblks = (int)((cs + c.BK - 1) / c.BK);
    c.ksteps_last = (int)(cs - (int64_t)(c.cblks - 1) * c.BK) / 32;
    c.num_kb = g.cs.R * g.cs.S * c.cblks;
    k_padded = (int64_t)g.cs.R * g.cs.S * cs;
    // im2col traversal limits of the tensor map (two spatial dimensions: 8-bit signed corners)
    const int lo_w = -g.cs.pad_w, lo_h = -g.cs.pad_h;
    const int up_w = g.cs.pad_w - (g.cs.S - 1), up_h = g.cs.pad_h - (g.cs.R - 1);
    if (lo_w < -128 || lo_h < -128 || up_w < -128 || up_h < -128 || up_w > 127 || up_h > 127) return c;
    if (g.cs.stride_h > 8 || g.cs.stride_w > 8 || g.cs.R > 255 || g.cs.S > 255) return c;
    // tensors below 128 KiB stay on the direct kernel (tiny problems gain nothing here)
    if ((int64_t)g.cs.N * g.cs.H * g.cs.W * cs < 131072) return c;
    if (k_padded > (int64_t)1 << 30) return c;
  } else {
    if (g.K < 32) return c;
    c.BK = g.K >= 128 ? 128 : (g.K >= 64 ? 64 : 32);
    const int forced_bk = knob(kBK);   // experiment knob: narrower K-blocks
    if ((forced_bk == 32 || forced_bk == 64) && forced_bk < c.BK) c.BK = forced_bk;
    c.num_kb = (int)((g.K + c.BK - 1) / c.BK);
    k_padded = g.K;
    if (g.K > (int64_t)1 << 30) return c;
  }
  c.swizzle = c.BK == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                          : (c.BK == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
  c.layout_type = c.BK == 128 ? 2u : (c.BK == 64 ? 4u : 6u);
  c.BN = g.N <= 32 ? 32 : (g.N <= 64 ? 64 : 128);
  const int forced_bn = knob(kBN);    // experiment knob: narrower tiles
  if ((forced_bn == 32 || forced_bn == 64) && forced_bn < c.BN) c.BN = forced_bn;
  // Single-pass (8-bit) layers with many output channels take 256-column pair tiles: one int32
  // accumulator per tile leaves room for two sets of 256 columns, and a 256 x 256 tile halves the
  // operand bytes per MMA cycle, which is what limits the int8 rate (see make_config's pair notes).
  // (not for short reductions over partial blocks where the channel count is no multiple of 8: the 64-bit epilogue
  // bounds those and pays for every column of the last tile; 45 x 16 x 14 pixels, 3x3, 69 -> 294 24.7 us against 18.7)
  const bool partial = g.is_conv && c.ksteps_last != c.BK / 32;
  const bool wide = allow_wide && c.nacc == 1 && c.BK == 128 && g.N >= 256 && c.num_kb >= 9 && g.M >= 1024 &&
                    (num_sms() % 2) == 0 && forced_bn == 0 && knob(kPair) != 0 &&
                    knob(kWide) != 0 && !(partial && g.N % 8 != 0 && c.num_kb < 16);
  if (wide) c.BN = 256;
  c.tiles_m = (int)((g.M + kBM - 1) / kBM);
  if (g.box_pool) {
    if (!g.is_conv || g.cs.stride_h != 1 || g.cs.stride_w != 1) return c;
    c.box = pool_boxes(g);
    if (!c.box.on) return c;
    c.tiles_m = (int)box_count(c.box);
  }
  c.tiles_n = (int)((g.N + c.BN - 1) / c.BN);
  c.acc_bufs = 512 / (c.nacc * c.BN);
  if (c.acc_bufs > kMaxAccBufs) c.acc_bufs = kMaxAccBufs;
  if (c.acc_bufs == 3) c.acc_bufs = 2;
  if (c.acc_bufs < 1) return c;
  uint32_t cols = (uint32_t)(c.acc_bufs * c.nacc * c.BN);
  c.tmem_cols = 32;
  while (c.tmem_cols < cols) c.tmem_cols <<= 1;
  // split the reduction when one accumulation would exceed the int32-safe length, or when
  // there are too few output tiles to fill the machine and the reduction is long
  const int max_kb_per_acc = (int)(kMaxKPerAccumulation / c.BK);
  int splits = (c.num_kb + max_kb_per_acc - 1) / max_kb_per_acc;
  const int tiles = c.tiles_m * c.tiles_n;
  const int sms = num_sms();
  if (tiles * 2 <= sms && c.num_kb >= 16) {
    int want = sms / tiles;
    int cap = c.num_kb / 8;
    if (want > cap) want = cap;
    if (want > splits) splits = want;
  }
  const int forced = knob(kSplits);
  if (forced > 0) splits = forced > splits ? forced : splits;
  if (splits > c.num_kb) splits = c.num_kb;
  if (splits < 1) splits = 1;
  c.kb_per_split = (c.num_kb + splits - 1) / splits;
  c.splits = (c.num_kb + c.kb_per_split - 1) / c.kb_per_split;
  if ((int64_t)c.kb_per_split * c.BK > kMaxKPerAccumulation) return c;
  if ((int64_t)tiles * c.splits > (int64_t)1 << 30) return c;
  c.workspace_bytes = c.splits > 1 ? (size_t)g.M * (size_t)g.N * sizeof(long long) : 0;
  // Large unsplit problems run as CTA pairs: 256-row tiles, each CTA stages its own 128 rows of A
  // and only half of the weight rows, which cuts the bytes (and TMA rows) per MAC by a quarter.
  const int pair_env = knob(kPair);
  // (measured: pairs win from K = 1152 bytes per plane row on; 256 x 64 pair tiles with two
  // accumulator sets were tried for medium reductions and lost to these once the epilogue hands the
  // accumulators back early)
  const bool pair_ok = c.splits == 1 && g.M >= 1024 && (sms % 2) == 0;
  c.pair = pair_ok && c.BN >= 128 && c.BK == 128 && c.num_kb >= 9;
  // 64-channel convolutions with at most 64 output channels (64-byte k-blocks, one 64-column tile):
  // as a pair each CTA stages half of the weight rows and the MMAs find half of their B operand in
  // the peer's shared memory; with one filter row of taps per stage this measured 0.43 ms against
  // 0.53 ms for 64 x 224 x 224 x 64 -> 64 with the weights resident in a single CTA.
  // (16-bit operands only: with one int8 product per k-step the single CTA with resident weights
  // stays ahead, 0.65 ms against 0.79 ms for the same layer at 8 bits and batch 128)
  const bool narrow_pair = pair_ok && g.is_conv && c.nacc == 3 && c.BK == 64 && c.BN == 64 && c.num_kb >= 9 &&
                           c.num_kb % 3 == 0;
  if (narrow_pair) c.pair = true;
  if (pair_env == 0) c.pair = false;
  if (pair_env == 1 && c.splits == 1 && (sms % 2) == 0) c.pair = true;
  if (c.pair) {
    c.tile_m = 2 * kBM;
    c.tiles_m = g.box_pool ? (c.tiles_m + 1) / 2 : (int)((g.M + c.tile_m - 1) / c.tile_m);
  }
  // Inner products on a small batch: only the rows that exist are staged (the MMA still covers 128
  // rows; the rest reads whatever follows in the stage and lands in accumulator rows nobody stores).
  // Smaller stages mean a deeper ring, i.e. more weight bytes in flight per SM, which is what bounds
  // these weight-streaming layers.
  c.a_rows = (!g.is_conv && !c.pair && g.M <= 64) ? 64 : kBM;
  c.a_bytes = (uint32_t)(c.a_rows * c.BK);
  c.b_bytes = (uint32_t)((c.pair ? c.BN / 2 : c.BN) * c.BK);
  // Output staging: one plane of 128 rows x BN bytes per output byte plane.  Needs a tensor map over
  // the output planes (pitch a multiple of 16 bytes and at least one tile wide) and no int16 copy.
  const int out_planes = g.y.fmt.n_bits > 8 ? 2 : 1;
  c.staged = g.mode == ADAPTION_MODE_REQUANT && c.splits == 1 && g.y.q16 == nullptr && g.y.lo != nullptr &&
             g.y.c_stride >= c.BN && g.y.c_stride % 16 == 0 && knob(kStaged) != 0;
  // As many epilogue groups as tiles can be in flight in TMEM, two for wide tiles: a group's chain per tile (wait,
  // TMEM loads, arithmetic, staging, barrier, store) is mostly latency.  8 bits, batch 128: 3 -> 64 channels at 224 x 224
  // 387 us with two groups, 349 with four; 64 -> 128 at 112 x 112 163 with one, 128 with two, 126 with four;
  // 128 -> 256 at 56 x 56 106 with one, 90 with two; 3 -> 16 at 16 bits, batch 16 91 with two, 62 with four.
  // Stored outputs of a channel count that is no multiple of 8 take the 64-bit epilogue, whose steps of 16 columns four
  // groups do not share: two for those where a tile has the k-blocks to cover a longer chain (60 layers of up to 31
  // channels and at least nine blocks 5 % faster on average, at best 40; 16 bits, 36 x 97 x 139 pixels, 3x3, 23 -> 11 82 us
  // against 67; 8 bits, 14 x 71 x 165, 3x3, 166 -> 9 47 against 34.  One block, 58 x 60 x 176, 3 -> 31 53 with four, 58
  // with two; 64 columns gain 2 to 4 % beyond nine blocks).
  c.epi_groups = c.acc_bufs;
  const bool two_groups = g.is_conv && g.mode == ADAPTION_MODE_REQUANT && g.N % 8 != 0 &&
                          c.num_kb >= (c.BN == 32 ? 9 : 10);
  const int most_groups = c.BN <= 64 && !two_groups ? 4 : 2;
  while (c.epi_groups > 1 && (c.epi_groups > most_groups || c.epi_groups > knob(kEpiGroups))) c.epi_groups /= 2;
  c.stage_out_bytes = c.staged ? (uint32_t)(kBM * c.BN * out_planes * c.epi_groups) / (c.box.pool ? 4u : 1u) : 0u;
  // dynamic shared memory: everything up to the per-block limit except the control block
  // (box tiles over partial blocks with the 32-bit epilogue: launch_tensor)
  c.own_rows = partial && c.box.on && c.epi_groups * 4 == kEpiWarps;
  c.const_bytes = (uint32_t)(c.BN * (c.own_rows ? kEpiWarps : c.epi_groups) * sizeof(long long));
  const size_t budget = 232448 - sizeof(Ctrl) - 256 - c.stage_out_bytes - c.const_bytes;
  // group short k-blocks so that a stage carries roughly 768 tensor-pipe cycles of work or more.  512 with one product
  // per step (128 -> 128 channels at 112 x 112, 8 bits, batch 128 231 us with two k-blocks, 264 with three), but not for
  // convolutions of more than twelve k-blocks on 128 columns, whose weights cannot stay resident beside either ring (18 to
  // 48 blocks 10 % faster with three; 8 x 74 x 194 pixels, 5x5, 112 -> 103 63 us against 56; an inner product of 512 rows,
  // 4096 -> 4096, has 12.1 with two, 13.4 with three).
  // Two accumulators over partial blocks (a pitch that is no multiple of 128): one block per stage, because the grouped
  // loop multiplies the zeros behind the pitch (128 columns 10 to 15 % faster, 64 columns 6 to 9; 19 x 35 x 12 pixels, 5x5,
  // 302 -> 259 70 us against 58; tiles of 32 columns wait for copies either way).
  {
    const int products = c.nax * c.nbw;
    const int cyc_per_kb = (c.BK / 32) * products * (c.BN >= 128 ? c.BN / 2 : 48);
    const int want = c.nacc == 1 && !(g.is_conv && c.BN == 128 && c.num_kb > 12) ? 512 : 768;
    int kps = (want + cyc_per_kb - 1) / cyc_per_kb;
    if (kps > 4) kps = 4;
    if (c.nacc == 2 && partial && c.BN >= 64) kps = 1;
    const int kps_env = knob(kKps);
    if (narrow_pair && c.pair) kps = 3;
    if (kps_env >= 1 && kps_env <= 4) kps = kps_env;
    if (kps > c.kb_per_split) kps = c.kb_per_split;
    if (kps < 1) kps = 1;
    if (kps_env == 0) {                     // as few stages per tile, but even ones
      const int per_tile = (c.kb_per_split + kps - 1) / kps;
      kps = (c.kb_per_split + per_tile - 1) / per_tile;
    }
    c.kps = kps;
  }
  c.kb_bytes = c.nax * c.a_bytes + c.nbw * c.b_bytes;
  // One column tile and a short reduction: keep every weight k-block resident in shared memory and
  // stream only the activation planes (fewer bulk copies per k-block for the 64-channel and
  // 3-channel layers).  Only if at least three activation stages still fit.
  const size_t res_bytes = (size_t)c.num_kb * c.nbw * c.b_bytes;
  if (c.tiles_n == 1 && c.splits == 1 && c.tiles_m >= 4 * sms && (!c.pair || knob(kBres) != 2) &&
      res_bytes + 3 * (size_t)c.kps * c.nax * c.a_bytes + 1024 <= budget && knob(kBres) != 0) {
    c.b_resident = true;
    c.b_blocks = c.num_kb;
    c.b_res_bytes = (uint32_t)res_bytes;
    c.kb_bytes = c.nax * c.a_bytes;
  }
  c.stage_bytes = (uint32_t)c.kps * c.kb_bytes;
  c.stages = (int)((budget - 1024 - c.b_res_bytes) / c.stage_bytes);
  if (c.staged && c.stages < 3) {
    // not enough room for a useful ring beside the staging planes: store directly instead
    c.stages = (int)((budget + c.stage_out_bytes - 1024 - c.b_res_bytes) / c.stage_bytes);
    c.staged = false;
    c.stage_out_bytes = 0;
    c.stage_bufs = 1;
  }
  if (c.stages > kMaxStages) c.stages = kMaxStages;
  // Narrow tiles with two epilogue groups (with four the other groups cover the wait): a second staging buffer per group, so that a group does
  // not wait for its previous tile's bulk store to have read shared memory - where the ring keeps at
  // least four stages beside it (short reductions with small stages, e.g. a packed first layer).
  if (c.staged && c.epi_groups == 2 && c.BN <= 64 && knob(kStageBufs) != 1) {
    const size_t extra = c.stage_out_bytes;
    const size_t used = (size_t)c.stages * c.stage_bytes + c.b_res_bytes + 1024;
    size_t slack = budget > used ? budget - used : 0;
    int stages = c.stages;
    while (slack < extra && stages > 4) {
      --stages;
      slack += c.stage_bytes;
    }
    if (slack >= extra) {
      c.stages = stages;
      c.stage_bufs = 2;
      c.stage_out_bytes = (uint32_t)(2 * extra);
    }
  }
  const int stage_cap = knob(kStages);   // experiment knob: shallower ring
  if (stage_cap >= 2 && stage_cap < c.stages) c.stages = stage_cap;
  if (c.stages < 2) return c;
  c.stage_off = (uint32_t)(((size_t)c.stages * c.stage_bytes + c.b_res_bytes + 1023) & ~(size_t)1023);
  c.smem_bytes = (size_t)c.stage_off + 1024 + c.stage_out_bytes + c.const_bytes;
  c.ok = true;
  return c;
}

// The tile configuration with groups of G pixels (see PixelPlan), or one that is not ok.
TcConfig make_pixel_config(const GemmProblem& g, int G) {
  TcConfig c;
  const int S = g.cs.S, R = g.cs.R, pad = g.cs.pad_w;
  const bool storing = g.mode == ADAPTION_MODE_REQUANT;
  const int64_t ys = storing ? g.y.c_stride : (g.N + 31) / 32 * 32;
  c.nax = g.x.fmt.n_bits > 8 ? 2 : 1;
  c.nbw = g.w.fmt.n_bits > 8 ? 2 : 1;
  c.nacc = c.nax + c.nbw - 1;
  if ((ys != 32 && ys != 64 && ys != 128) || g.N > ys || g.cs.W % G != 0 || g.OW % G != 0 ||
      G * ys > (c.nacc == 1 ? 256 : 128))
    return c;
  PixelPlan& px = c.px;
  px.G = G;
  px.ys = (int)ys;
  px.ys_shift = ys == 32 ? 5 : (ys == 64 ? 6 : 7);
  px.n_valid = (int)g.N;
  px.S = S;
  px.row_u = (uint32_t)(S * ys * 2);
  px.b_plane = (uint32_t)(R * S * 32 * ys);
  const int lead = (pad + G - 1) / G;                       // groups before the first output pixel's
  px.blocks = lead + (S - 1 - pad + 2 * G - 1) / G;         // (pad < S)
  if (px.blocks > kMaxPixelBlocks) return c;
  px.first = -1;
  uint32_t step[kMaxPixelBlocks][4] = {}, b_row[kMaxPixelBlocks][4] = {};
  for (int d = 0; d < px.blocks; ++d)
    for (int i = 0; i < G; ++i) {
      const int u = (d - lead) * G + i;
      int lo = u + pad - (S - 1), hi = u + pad;             // output pixels that see input pixel u under a tap
      if (lo < 0) lo = 0;
      if (hi > G - 1) hi = G - 1;
      if (lo > hi) continue;
      step[d][i] = (uint32_t)((hi - lo + 1) * ys / 8) << 17 | (uint32_t)(lo * ys);
      b_row[d][i] = (uint32_t)((S - 1 - (u + pad - lo)) * ys * 2);
      if (i == 0 && hi - lo + 1 == G && px.first < 0) px.first = d;
    }
  // the first MMA of a tile overwrites the accumulators: it has to cover all their columns
  if (px.first < 0) return c;
  for (int d = 0; d < px.blocks; ++d) {
    const int from = (d + px.first) % px.blocks;
    std::memcpy(px.step[d], step[from], sizeof(step[0]));
    std::memcpy(px.b_row[d], b_row[from], sizeof(b_row[0]));
  }
  c.BK = G * 32;
  c.ksteps_last = G;
  c.swizzle = G == 4 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
  c.layout_type = G == 4 ? 2u : 4u;
  c.BN = G * px.ys;
  c.num_kb = c.kb_per_split = R * px.blocks;
  // (same limits of the tensor map as in make_config_impl)
  const int up_w = g.OW / G - g.cs.W / G - lead, up_h = g.cs.pad_h - (R - 1);
  if (lead > 128 || g.cs.pad_h > 128 || up_w < -128 || up_h < -128 || up_w > 127 || up_h > 127) return c;
  c.tiles_m = (int)((g.M / G + kBM - 1) / kBM);
  c.tiles_n = 1;
  // Too few tiles leave SMs without one: 112 x 112 x 16 -> 16, 7x7, 16 bits, ungrouped against grouped: one image (46 tiles)
  // 14.7 us against 15.6, two 25.0 against 17.6, four 37 against 26; 112 x 112 x 32 -> 64, 5x5: one image (49) 10.5
  // against 12.4, four (196) 22.6 against 18.8.
  if (c.tiles_m < num_sms() / 2 && knob(kPixels) < 2) return c;
  c.acc_bufs = 512 / (c.nacc * c.BN);
  if (c.acc_bufs > kMaxAccBufs) c.acc_bufs = kMaxAccBufs;
  if (c.acc_bufs == 3) c.acc_bufs = 2;
  while (c.tmem_cols < (uint32_t)(c.acc_bufs * c.nacc * c.BN)) c.tmem_cols <<= 1;
  c.a_bytes = (uint32_t)(kBM * c.BK);
  c.kb_bytes = c.stage_bytes = c.nax * c.a_bytes;
  const int out_planes = g.y.fmt.n_bits > 8 ? 2 : 1;
  c.staged = storing && g.y.q16 == nullptr && g.y.lo != nullptr;
  c.epi_groups = c.acc_bufs;
  const int most_groups = c.BN <= 64 ? 4 : 2;
  while (c.epi_groups > 1 && (c.epi_groups > most_groups || c.epi_groups > knob(kEpiGroups))) c.epi_groups /= 2;
  c.stage_out_bytes = c.staged ? (uint32_t)(kBM * c.BN * out_planes * c.epi_groups) / (g.pool_w ? 2u : 1u) : 0u;
  c.const_bytes = (uint32_t)(c.BN * c.epi_groups * sizeof(long long));
  const size_t budget = 232448 - sizeof(Ctrl) - 256 - c.stage_out_bytes - c.const_bytes;
  c.b_resident = true;
  c.b_res_bytes = c.nbw * px.b_plane;
  if (c.b_res_bytes + 3 * c.stage_bytes + 1024 > budget) return c;
  c.stages = (int)((budget - 1024 - c.b_res_bytes) / c.stage_bytes);
  if (c.stages > kMaxStages) c.stages = kMaxStages;
  c.stage_off = (uint32_t)(((size_t)c.stages * c.stage_bytes + c.b_res_bytes + 1023) & ~(size_t)1023);
  c.smem_bytes = (size_t)c.stage_off + 1024 + c.stage_out_bytes + c.const_bytes;
  c.ok = true;
  return c;
}

// Grouped pixels where they apply: the widest groups whose weights and stages fit.
TcConfig make_pixel_config(const GemmProblem& g) {
  if (knob(kPixels) == 0 || !g.is_conv || g.x.c_stride != 32 || g.w.c_stride != 32 || g.N > 128 || g.cs.stride_w != 1 ||
      g.cs.stride_h > 8 || g.cs.R > 255 || g.cs.pad_w >= g.cs.S || g.M > (int64_t)1 << 30 ||
      (int64_t)g.cs.R * g.cs.S * 32 > kMaxKPerAccumulation)
    return TcConfig();
  for (Knob k : {kSplits, kPair, kStaged, kStages, kBK, kBN, kKps, kBres, kWide, kSplitHh, kStageBufs})
    if (knob(k) != kKnobDefaults[k]) return TcConfig();        // an override of the other tiles asks for them
  for (int G = knob(kPixels) > 1 ? knob(kPixels) : 4; G > 1; G /= 2) {
    const TcConfig c = make_pixel_config(g, G);
    if (c.ok) return c;
  }
  return TcConfig();
}

// Whether one copy for all taps beats a copy per tap.  It waits for all of the weights before its first MMA and gains by
// the rows that it does not copy: `bytes` per pixel and plane otherwise.  Ratio of times, streaming / this, over images of 16 to
// 224 columns (T: tiles of a pair of SMs):
//   one tile per pair or fewer: 0.81 to 1.02 whatever the filter;
//   256 to 448 bytes (2x2 over 64 channels): 0.77 to 1.0 up to T = 4800; 512: 0.83 to 1.0 at 100 to 600, 1.02 to 1.1 at 1200;
//   measuring only, with two column tiles 0.83 to 1.05 up to T = 222, 0.97 to 1.1 from 296 on; 512 bytes 1.08 to 1.12 from 600 on;
//   three accumulators: two column tiles, which read the copy twice, 64 -> 128 0.85 to 0.96 up to 600, 0.98 at 1200, 0.99 to 1.06
//     from 2400 on, but 1.12 to 1.6 from 600 on where the streamed tile of 128 columns is wider than the output's pitch and
//     cannot be staged (64 -> 72); the 64-bit epilogue, 64 -> 61 and 100 0.94 to 1.0 (5x5 1.05 to 1.38), 96 -> 50 0.92 to 1.0 up to
//     148, 1.0 to 1.2 beyond; 640 and 768 bytes of wide blocks 0.9 to 1.07 at 100 and 148, 1.06 to 1.3 from 300 on;
//   one accumulator, where a streamed tile is a single CTA's: 64 -> 64 0.95 to 1.06 up to T = 148, 1.05 to 1.3 at 150 to 290, 0.91
//     to 1.06 from 296 on, where the streamed weights stay resident too, 1.03 to 1.25 from 700 on; 64 -> 128 0.81 to 1.06 up to 784,
//     1.0 to 1.08 from 1200 on; 128 -> 128 with 640 bytes 0.92 to 0.97 at 100 to 300, 768 to 1024 0.93 to 0.98 at 100 and 148, 1.02
//     to 1.16 at 300, 1152 and more 1.03 and more; 128 columns through the 64-bit epilogue, whose four groups take a tile each:
//     128 -> 99 and 96 -> 70 0.91 to 1.08 up to 300, 1.02 to 1.13 from 600 on, 64 -> 100 0.97, 1.0 and 1.03 at 600, 1200 and 2400.
// Everything else measured 0.94 to 1.27 at 100 and 148, 0.97 to 2.3 beyond.
bool one_copy_pays(const TcConfig& c, const GemmProblem& g, int taps) {
  const int pairs = num_sms() / 2, T = c.tiles_m, bytes = taps * c.cblks * c.BK;
  const bool wide_sums = g.N % 8 != 0;         // the 64-bit epilogue
  if (T <= pairs) return false;
  if (g.mode != ADAPTION_MODE_REQUANT)
    return bytes < 576 ? bytes >= 512 && T >= 8 * pairs : c.tiles_n == 1 || T >= 4 * pairs;
  if (bytes < 576) return bytes >= 512 && c.tiles_n == 1 && T >= 16 * pairs;
  if (c.nacc == 3) {
    if (wide_sums && c.BK == 64 && bytes < 1024) return false;
    if (c.tiles_n > 1) return T >= (g.y.c_stride < 128 ? 4 : 32) * pairs;
    return c.BK == 64 || (bytes >= 1152 && !wide_sums) || T > 2 * pairs;
  }
  if (c.BN == 128 && wide_sums) return T >= (c.BK == 64 ? 16 : 9) * pairs;
  if (c.BK == 64 && bytes < 1024)
    return c.BN == 128 ? T >= 16 * pairs : T >= 9 * pairs || (T > 2 * pairs && T < 4 * pairs);
  if (c.BK == 128 && bytes < 1152) return T >= (bytes < 768 ? 9 : 4) * pairs;
  return true;
}

// One copy of the activations for all taps (see HaloPlan), where the weights stay resident beside at least two tiles'
// copies of them: operands of one width, 8 x 16 boxes without much margin.
TcConfig make_halo_config(const GemmProblem& g) {
  TcConfig c;
  if (knob(kHalo) == 0 || !g.is_conv || g.pool_w || g.cs.stride_h != 1 || g.cs.stride_w != 1 || g.cs.R > 15 || g.cs.S > 15 ||
      g.M > (int64_t)1 << 30 || g.x.c_stride != g.w.c_stride)
    return c;
  for (Knob k : {kSplits, kPair, kStages, kBK, kBN, kKps, kBres, kWide, kStageBufs})
    if (knob(k) != kKnobDefaults[k]) return TcConfig();        // an override of the other tiles asks for them
  const int sms = num_sms(), taps = g.cs.R * g.cs.S;
  const int64_t cs = g.x.c_stride;
  c.nax = g.x.fmt.n_bits > 8 ? 2 : 1;
  c.nbw = g.w.fmt.n_bits > 8 ? 2 : 1;
  c.nacc = c.nax + c.nbw - 1;
  if (c.nax != c.nbw || g.N > 128) return c;
  c.BN = g.N <= 32 ? 32 : (g.N <= 64 ? 64 : 128);
  c.tiles_n = 1;
  c.box = box_plan(3, 4, 0, g.OW, g.OH, g.cs.N, g.box_pool);
  const int64_t boxes = box_count(c.box);
  if (boxes > (1 << 23) || boxes * kBM * 16 > g.M * 17) return c;
  HaloPlan& h = c.halo;
  h.w = kHaloW + g.cs.S - 1;
  h.R = g.cs.R;
  h.S = g.cs.S;
  if (g.taps) {
    // pixels of 16 bytes: two taps are a step of 32
    h.steps = (taps + 1) / 2;
    if (cs != 16 || h.steps > kMaxTapSteps) return c;
    c.BK = 16;
    h.px_u = 1;
    h.b_row_u = (uint32_t)(2 * c.BN);
    for (int i = 0; i < h.steps; ++i) {
      const int t0 = 2 * i, t1 = 2 * i + 1 < taps ? 2 * i + 1 : 2 * i;     // (behind the last tap the weights are zero)
      const int at0 = t0 / g.cs.S * h.w + t0 % g.cs.S, at1 = t1 / g.cs.S * h.w + t1 % g.cs.S;
      h.a_lo[i] = (uint32_t)at0 | (uint32_t)(at1 - at0) << 16;
    }
    c.num_kb = 1;
    c.ksteps_last = 1;
    c.b_blocks = 2 * h.steps;
    c.b_bytes = (uint32_t)(c.b_blocks * c.BN * 16);
    c.b_res_bytes = (uint32_t)c.nbw * c.b_bytes;
    c.tiles_m = (int)boxes;
  } else {
    if (taps < 4 || cs % 32 != 0 || cs < 64 || c.BN < 64 || (sms & 1) != 0 || taps * cs > kMaxKPerAccumulation) return c;
    c.BK = cs > 64 ? 128 : 64;
    c.cblks = (int)((cs + c.BK - 1) / c.BK);
    c.ksteps_last = (int)(cs - (int64_t)(c.cblks - 1) * c.BK) / 32;
    c.swizzle = c.BK == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    c.layout_type = c.BK == 128 ? 2u : 4u;
    h.px_u = (uint32_t)(c.BK / 16);
    c.pair = true;
    c.tile_m = 2 * kBM;
    c.num_kb = c.cblks;
    c.b_blocks = taps * c.cblks;
    c.b_bytes = (uint32_t)(c.BN / 2 * c.BK);
    // 16-bit operands: two tiles of 64 columns rather than one of 128, whose three accumulators could not be doubled
    // (64 x 112 x 112 x 64 -> 128: 205 us with one, 158 with two)
    if (c.nacc == 3 && c.BN == 128) {
      c.BN = 64;
      c.b_bytes /= 2;
      c.tiles_n = 2;
    }
    c.b_res_bytes = (uint32_t)(c.tiles_n * c.b_blocks * c.nbw) * c.b_bytes;
    c.tiles_m = (int)((boxes + 1) / 2);
    if (!one_copy_pays(c, g, taps) && knob(kHalo) < 2) return c;
  }
  c.kb_per_split = c.num_kb;
  c.a_tx = (uint32_t)(h.w * (kHaloH + g.cs.R - 1) * c.BK);
  c.a_bytes = (c.a_tx + 1023u) & ~1023u;
  c.kb_bytes = c.stage_bytes = (uint32_t)c.nax * c.a_bytes;
  c.acc_bufs = 512 / (c.nacc * c.BN);
  if (c.acc_bufs > kMaxAccBufs) c.acc_bufs = kMaxAccBufs;
  if (c.acc_bufs == 3) c.acc_bufs = 2;
  while (c.tmem_cols < (uint32_t)(c.acc_bufs * c.nacc * c.BN)) c.tmem_cols <<= 1;
  const int out_planes = g.y.fmt.n_bits > 8 ? 2 : 1;
  c.staged = g.mode == ADAPTION_MODE_REQUANT && g.y.q16 == nullptr && g.y.lo != nullptr && g.y.c_stride >= c.BN &&
             g.y.c_stride % 16 == 0 && knob(kStaged) != 0;
  if (g.box_pool && !c.staged) return c;
  c.epi_groups = c.acc_bufs;
  // (first layers through the 64-bit epilogue with up to two tiles per SM: a tile's chain counts, so twice the warps share it;
  // 8 bits, 3 -> 100, us with four groups and two, 76 tiles 11.6 and 10.1, 222 14.8 and 13.6, 300 16.9 and 18.2; 3 -> 61 7.7 and 6.9,
  // 9.6 and 9.1, 10.1 and 11.5)
  const bool two_groups = g.taps && g.N % 8 != 0 && c.tiles_m <= 2 * sms;
  const int most_groups = !two_groups && (c.BN <= 64 || c.nacc == 1) ? 4 : 2;
  while (c.epi_groups > 1 && (c.epi_groups > most_groups || c.epi_groups > knob(kEpiGroups))) c.epi_groups /= 2;
  c.stage_out_bytes = c.staged ? (uint32_t)(kBM * c.BN * out_planes * c.epi_groups) / (g.box_pool ? 4u : 1u) : 0u;
  c.own_rows = c.epi_groups * 4 == kEpiWarps && c.BN <= 128;
  c.const_bytes = (uint32_t)(c.BN * (c.own_rows ? kEpiWarps : c.epi_groups) * sizeof(long long));
  const size_t budget = 232448 - sizeof(Ctrl) - 256 - c.stage_out_bytes - c.const_bytes;
  c.b_resident = true;
  if (c.b_res_bytes + 2 * c.stage_bytes + 1024 > budget) return c;
  c.stages = (int)((budget - 1024 - c.b_res_bytes) / c.stage_bytes);
  if (c.stages > kMaxStages) c.stages = kMaxStages;
  c.stage_off = (uint32_t)(((size_t)c.stages * c.stage_bytes + c.b_res_bytes + 1023) & ~(size_t)1023);
  c.smem_bytes = (size_t)c.stage_off + 1024 + c.stage_out_bytes + c.const_bytes;
  c.ok = true;
  return c;
}

template <int NAX, int NBW, bool PAIR, int LOOP, int EPI>
int launch_kernel(const CUtensorMap* maps, const TcParams& p, int grid, size_t smem, cudaStream_t stream) {
  note_layer(LOOP & (kLoopBoxes - 1), p.stages, p.total_tiles, p.staged);
  // The dynamic shared-memory limit is a per-device attribute of the kernel: remember, per device
  // ordinal, the largest size it has been raised to (a racing thread at worst sets it once more).
  constexpr int kMaxDevices = 64;
  static std::atomic<size_t> attr_size[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return ADAPTION_ERR_CUDA;
  const bool cached = dev >= 0 && dev < kMaxDevices;
  if (!cached || smem > attr_size[dev].load(std::memory_order_acquire)) {
    const cudaError_t ae = cudaFuncSetAttribute(lp_gemm_kernel<NAX, NBW, PAIR, LOOP, EPI>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ae != cudaSuccess) return cuda_failure(ae, "lp_gemm_kernel shared-memory attribute");
    if (cached) {
      size_t seen = attr_size[dev].load(std::memory_order_relaxed);
      while (seen < smem && !attr_size[dev].compare_exchange_weak(seen, smem, std::memory_order_release)) {
      }
    }
  }
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  unsigned n_attr = 0;
  if (PAIR) {
    attr[n_attr].id = cudaLaunchAttributeClusterDimension;
    attr[n_attr].val.clusterDim.x = 2;
    attr[n_attr].val.clusterDim.y = 1;
    attr[n_attr].val.clusterDim.z = 1;
    ++n_attr;
  }
  if (knob(kPdl) != 0) {
    // the kernel waits for its predecessor itself (pdl_wait) before it touches global memory
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
    ++n_attr;
  }
  cfg.attrs = n_attr ? attr : nullptr;
  cfg.numAttrs = n_attr;
  count_launch();
  const cudaError_t le =
      cudaLaunchKernelEx(&cfg, lp_gemm_kernel<NAX, NBW, PAIR, LOOP, EPI>, maps[0], maps[1], maps[2], maps[3], maps[4],
                         maps[5], p);
  if (le != cudaSuccess) {
    (void)cudaGetLastError();
    return cuda_failure(le, "lp_gemm_kernel launch");
  }
  return cuda_status(cudaGetLastError(), "after lp_gemm_kernel launch");
}

template <int NAX, int NBW, bool PAIR, int LOOP>
int launch_epi(const CUtensorMap* maps, const TcParams& p, int grid, size_t smem, cudaStream_t stream) {
  if (p.fast_relu != 0) return launch_kernel<NAX, NBW, PAIR, LOOP, kEpiFast>(maps, p, grid, smem, stream);
  if constexpr ((LOOP & kLoopBoxes) == 0) {                // (the pooling call rounds to nearest)
    if (p.fast_stochastic != 0) return launch_kernel<NAX, NBW, PAIR, LOOP, kEpiFastStochastic>(maps, p, grid, smem, stream);
    if (p.st.enabled != 0) return launch_kernel<NAX, NBW, PAIR, LOOP, kEpiStochastic>(maps, p, grid, smem, stream);
  } else if (p.st.enabled != 0) {
    return ADAPTION_ERR_UNSUPPORTED;
  }
  return launch_kernel<NAX, NBW, PAIR, LOOP, kEpiGeneric>(maps, p, grid, smem, stream);
}

template <int NAX, int NBW, bool PAIR, int BOXES>
int launch_loop(const CUtensorMap* maps, const TcParams& p, int grid, size_t smem, cudaStream_t stream) {
  if (p.kps > 1 || p.b_resident != 0) return launch_epi<NAX, NBW, PAIR, kLoopGrouped + BOXES>(maps, p, grid, smem, stream);
  if (p.ksteps_last != p.ksteps && p.fast_relu != 0 && p.BN == 128)
    return launch_kernel<NAX, NBW, PAIR, kLoopPartial + kLoopBoxes, kEpiFast>(maps, p, grid, smem, stream);
  if (p.ksteps_last != p.ksteps) return launch_epi<NAX, NBW, PAIR, kLoopPartial + BOXES>(maps, p, grid, smem, stream);
  return launch_epi<NAX, NBW, PAIR, kLoopPlain + BOXES>(maps, p, grid, smem, stream);
}

template <int NAX, int NBW>
int launch_either(bool pair, const CUtensorMap* maps, const TcParams& p, int grid, size_t smem,
                  cudaStream_t stream) {
  if (p.px.G > 1) return launch_epi<NAX, NBW, false, kLoopPixels>(maps, p, grid, smem, stream);
  if constexpr (NAX == NBW) {
    if (p.halo.steps > 0) return launch_epi<NAX, NBW, false, kLoopTaps>(maps, p, grid, smem, stream);
    if (p.halo.w > 0) return launch_epi<NAX, NBW, true, kLoopHalo>(maps, p, grid, smem, stream);
  }
  if (p.box.on != 0)
    return pair ? launch_loop<NAX, NBW, true, kLoopBoxes>(maps, p, grid, smem, stream)
                : launch_loop<NAX, NBW, false, kLoopBoxes>(maps, p, grid, smem, stream);
  return pair ? launch_loop<NAX, NBW, true, 0>(maps, p, grid, smem, stream)
              : launch_loop<NAX, NBW, false, 0>(maps, p, grid, smem, stream);
}


// ---------------------------------------------------------------------------------- peak probe
// Issue-rate probe for the roofline denominator: every SM (or SM pair) runs back-to-back
// tcgen05.mma kind::i8 instructions on operand tiles that stay resident in shared memory (no
// loads), so the time per instruction is the tensor pipe's own.
template <bool PAIR>
__global__ void __launch_bounds__(128, 1)
i8_peak_kernel(int bn, int iters, int commit_every, unsigned long long* out_cycles, int* out_status) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ unsigned long long done_bar;
  __shared__ unsigned long long side_bar;      // target of the optional intermediate commits
  __shared__ uint32_t tmem_slot;
  const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
  // A: 128 rows x 128 bytes, B: up to 256 rows x 128 bytes, filled with a fixed byte pattern
  uint32_t* words = reinterpret_cast<uint32_t*>(smem_raw + (ring - smem_u32(smem_raw)));
  for (int i = threadIdx.x; i < (16384 + 32768) / 4; i += blockDim.x) words[i] = 0x9E3779B9u * (uint32_t)(i + 1);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&done_bar), 1);
    mbar_init(smem_u32(&side_bar), (1u << 20) - 1u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if ((threadIdx.x >> 5) == 0) {
    tmem_alloc<PAIR>(smem_u32(&tmem_slot), 512);
    tmem_relinquish<PAIR>();
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  if (threadIdx.x == 0 && rank == 0) {
    const uint32_t idesc = make_idesc(true, true, bn, PAIR ? 256 : 128);
    const uint32_t dhi = smem_desc_hi(1024, 2);
    const uint32_t a_lo = smem_desc_lo(ring), b_lo = smem_desc_lo(ring + 16384);
    const long long t0 = clock64();
    for (int i = 0; i < iters; ++i) {
#pragma unroll
      for (uint32_t ks = 0; ks < 8; ks += 2) mma_i8<PAIR>(tmem_base, a_lo + ks, b_lo + ks, dhi, idesc, 1u);
      // optional: an intermediate commit every `commit_every` groups of four instructions, as a
      // pipelined mainloop issues when it hands a shared-memory stage back
      if (commit_every > 0 && (i + 1) % commit_every == 0) tc_commit<PAIR>(smem_u32(&side_bar));
    }
    tc_commit<PAIR>(smem_u32(&done_bar));
    const unsigned long long w0 = global_ns();
    bool ok = true;
    while (!mbar_try_wait(smem_u32(&done_bar), 0)) {
      if (global_ns() - w0 > 2000000000ull) { ok = false; break; }
    }
    const long long t1 = clock64();
    if (!ok) atomicExch(out_status, (int)ADAPTION_ERR_TIMEOUT);
    out_cycles[blockIdx.x] = (unsigned long long)(t1 - t0);
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();
  if ((threadIdx.x >> 5) == 0) {
    tc_fence_after();
    tmem_dealloc<PAIR>(tmem_base, 512);
  }
}

template <bool PAIR>
int launch_peak(int bn, int iters, int commit_every, unsigned long long* d_cycles, int* d_status, int grid,
                cudaStream_t stream) {
  const size_t smem = 16384 + 32768 + 1024;
  if (cudaFuncSetAttribute(i8_peak_kernel<PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return ADAPTION_ERR_CUDA;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(128, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  if (PAIR) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  if (cudaLaunchKernelEx(&cfg, i8_peak_kernel<PAIR>, bn, iters, commit_every, d_cycles, d_status) != cudaSuccess) {
    (void)cudaGetLastError();
    return ADAPTION_ERR_CUDA;
  }
  return ADAPTION_OK;
}

}  // namespace

int probe_i8_peak(int bn, int pair, int iters, int commit_every, unsigned long long* d_cycles, int* d_status,
                  cudaStream_t stream) {
  const int sms = num_sms();
  const int grid = pair ? (sms / 2) * 2 : sms;
  return pair ? launch_peak<true>(bn, iters, commit_every, d_cycles, d_status, grid, stream)
              : launch_peak<false>(bn, iters, commit_every, d_cycles, d_status, grid, stream);
}

#ifdef ADAPTION_TIMELINE
extern "C" __attribute__((visibility("default"))) int adaption_debug_timeline_reset() {
  static long long zeros[8192];
  return cudaMemcpyToSymbol(g_timeline, zeros, sizeof(zeros)) == cudaSuccess ? 0 : 6;
}
extern "C" __attribute__((visibility("default"))) int adaption_debug_timeline(long long* h_out, int n) {
  return cudaMemcpyFromSymbol(h_out, g_timeline, sizeof(long long) * (size_t)n) == cudaSuccess ? 0 : 6;
}
#endif

bool tensor_path_supported(const GemmProblem& g) { return make_config(g).ok; }

// A first layer whose pixels of 16 bytes are read by the layer kernel itself (`g.taps`).
bool tensor_path_taps(const GemmProblem& g) { return make_halo_config(g).ok; }

// The whole 2x2 max-pool in the layer's epilogue (`g.box_pool`): box tiles.  (The columns of a pitch behind the last tile's
// would stay unwritten.  Layers over 32 channels are grouped by pixels, which gains more than the pooling pass costs.)
bool tensor_path_can_pool_boxes(const GemmProblem& g) {
  if (knob(kBox) == 0) return false;
  GemmProblem half = g;
  half.box_pool = false;
  TcConfig c = make_halo_config(g);
  if (!c.ok && (g.taps || make_pixel_config(half).ok)) return false;
  if (!c.ok) c = make_config(g);
  return c.ok && c.box.on && c.staged && c.splits == 1 && g.y.c_stride <= (int64_t)c.tiles_n * c.BN;
}

// The horizontal half of a 2x2 max-pool can ride on the staged stores of a requantizing layer.
bool tensor_path_can_pool(const GemmProblem& g) {
  const TcConfig c = make_config(g);
  return c.ok && c.staged && g.M % 2 == 0;
}

int tensor_path_tiles(const GemmProblem& g, bool* split) {
  const TcConfig c = make_config(g);
  *split = c.ok && c.splits > 1;
  return c.ok ? c.tiles_m * c.tiles_n : 0;
}

size_t tensor_path_workspace(const GemmProblem& g) { return make_config(g).workspace_bytes; }

// 32-bit bounds of the fast epilogues (see fast_result): with a reduction of kred bytes per plane row
// |hh| <= kred 2^14, |mid| <= kred 65280, |ll| <= kred 65025, and |C| < 2^(15 + bias_shift) + 2^(shift-1).
// Shift 0: no rounding half is added, and the result is floor(v / 2^16) (range mode) or, with one accumulator, v.
bool fits_32_bits(const GemmProblem& g, const TcConfig& c, int shift) {
  const bool single = c.nacc == 1;
  const long long kred = g.is_conv ? (long long)g.cs.R * g.cs.S * g.x.c_stride : (long long)c.num_kb * c.BK;
  const long long cmax = (g.bias != nullptr ? (1ll << (15 + g.bias_shift)) : 0ll) + (shift > 0 ? 1ll << (shift - 1) : 0ll);
  const long long hmax = kred * 16384 + (cmax >> 16) + 1;
  const long long tmax = kred * 65280 + ((kred * 65025 + 65535) >> 8) + 1;
  const long long lim = 1ll << 31;
  // single accumulator: s8 x s8 products only, the constant added in full
  if (single) return kred * 16384 + cmax < lim;
  bool ok = kred * 65025 + 65535 < lim && tmax < lim && hmax + (tmax >> 8) + 1 < lim;
  if (shift > 0 && shift < 16) ok = ok && (hmax << (16 - shift)) + (tmax >> (shift - 8)) + 1 < lim;
  return ok;
}

// The 32-bit epilogues: 1 = rounding to nearest (kEpiFast), 2 = stochastic (kEpiFastStochastic), 0 = neither applies.
int fast_epilogue(const GemmProblem& g, const TcConfig& c, const RequantParams& rq) {
  const bool single = c.nacc == 1;
  // (its steps of 32 columns need that many per warp: tiles of 64 columns need several groups, tiles of 32 take
  // the generic epilogue; the stochastic form takes 16, and with a shift of zero, where nothing is drawn, both do the same)
  const int cols_per_epi_warp = c.BN / (kEpiWarps / c.epi_groups / 4);
  const bool draws = g.stochastic.enabled && rq.shift > 0;
  if (!(g.mode == ADAPTION_MODE_REQUANT && c.splits == 1 && g.relu && rq.shift >= (single ? 0 : 9) && rq.shift <= 31 &&
        g.N % 8 == 0 && (draws ? cols_per_epi_warp % 16 == 0 : cols_per_epi_warp >= 32 && cols_per_epi_warp % 32 == 0) &&
        knob(kFast) != 0))
    return 0;
  return fits_32_bits(g, c, rq.shift) ? (draws ? 2 : 1) : 0;
}

int launch_tensor(const GemmProblem& g) {
  const RequantParams rq = g.mode == ADAPTION_MODE_REQUANT ? make_requant(g.acc_frac_bits, g.y.fmt, g.relu)
                                                           : RequantParams{0, g.relu ? 1 : 0, 0, 0, 1};
  // (with grouped pixels only the rounding 32-bit epilogue pools)
  TcConfig c = make_halo_config(g);
  if (!c.ok && g.taps) return ADAPTION_ERR_UNSUPPORTED;
  if (!c.ok && !g.box_pool) c = make_pixel_config(g);
  if (!c.ok || (g.pool_w && !(c.staged && fast_epilogue(g, c, rq) == 1))) c = make_config(g);
  if (!c.ok) return ADAPTION_ERR_UNSUPPORTED;
  const int G = c.px.G > 1 ? c.px.G : 1;       // output pixels per row
  const int64_t M = g.M / G, N = G > 1 ? c.BN : g.N, y_stride = g.y.c_stride * G;
  // the convolution that the copies of the activations see
  adaption_conv_shape cs = g.cs;
  const int OW = g.OW / G;
  if (G > 1) {
    cs.W /= G;
    cs.pad_w = (g.cs.pad_w + G - 1) / G;
    cs.S = cs.W - OW + 2 * cs.pad_w + 1;        // (the filter width that gives OW)
  }
  if (!load_tensor_map_encoders()) return ADAPTION_ERR_CUDA;
  const int fast = fast_epilogue(g, c, rq);
  // (the kernels that know it)
  c.own_rows = c.own_rows && (c.halo.w > 0 || (fast == 1 && c.kps == 1 && !c.b_resident && c.ksteps_last != c.BK / 32));

  // plane 0 is the high byte plane when there are two, else the single plane
  const void* xa[2] = {c.nax == 2 ? g.x.hi : g.x.lo, g.x.lo};
  const void* wb[2] = {c.nbw == 2 ? g.w.hi : g.w.lo, g.w.lo};
  CUtensorMap maps[6];   // activation planes, weight planes, output planes (hi, lo)
  std::memset(maps, 0, sizeof(maps));
  for (int i = 0; i < 2; ++i) {
    bool ok;
    if (c.box.on) {
      // (with the filter's margin around it where all taps share one copy)
      const uint64_t px = (uint64_t)g.x.c_stride, W = (uint64_t)g.cs.W, H = (uint64_t)g.cs.H;
      const uint32_t bw = c.halo.w > 0 ? (uint32_t)c.halo.w : 1u << c.box.w;
      const uint32_t bh = c.halo.w > 0 ? (uint32_t)(kHaloH + g.cs.R - 1) : 1u << c.box.h;
      if (c.halo.steps > 0) {
        const uint64_t dims[3] = {2 * W, H, (uint64_t)g.cs.N}, strides[2] = {px * W, px * W * H};
        const uint32_t box[3] = {2 * bw, bh, 1u};
        ok = encode_tiled_words(&maps[i], xa[i], 3, dims, strides, box);
      } else {
        const uint64_t dims[4] = {px, W, H, (uint64_t)g.cs.N}, strides[3] = {px, px * W, px * W * H};
        const uint32_t box[4] = {(uint32_t)c.BK, bw, bh, 1u << c.box.n};
        ok = encode_tiled(&maps[i], xa[i], 4, dims, strides, box, nullptr, c.swizzle);
      }
    } else if (g.is_conv)
      ok = encode_im2col_nhwc(&maps[i], xa[i], cs, g.x.c_stride * G, (uint32_t)c.BK, (uint32_t)kBM, c.swizzle);
    else
      ok = encode_tiled_2d(&maps[i], xa[i], (uint64_t)g.K, (uint64_t)g.M, (uint64_t)g.x.c_stride,
                           (uint32_t)c.BK, (uint32_t)c.a_rows, c.swizzle);
    if (!ok) return ADAPTION_ERR_CUDA;
    const uint64_t wk = g.is_conv ? (uint64_t)g.cs.R * g.cs.S * g.w.c_stride : (uint64_t)g.K;
    const uint64_t wpitch = g.is_conv ? wk : (uint64_t)g.w.c_stride;
    if (c.halo.steps > 0) {
      const uint64_t taps = (uint64_t)g.cs.R * g.cs.S;
      const uint64_t dims[3] = {2, taps, (uint64_t)g.N}, strides[2] = {16, 16 * taps};
      const uint32_t box[3] = {2u, 1u, (uint32_t)c.BN};
      if (!encode_tiled_words(&maps[2 + i], wb[i], 3, dims, strides, box)) return ADAPTION_ERR_CUDA;
      continue;
    }
    const bool rows32 = G > 1;                 // grouped pixels: weight rows of one 32-byte step
    if (!encode_tiled_2d(&maps[2 + i], wb[i], wk, (uint64_t)g.N, wpitch, rows32 ? 32u : (uint32_t)c.BK,
                         (uint32_t)(rows32 ? c.px.ys : (c.pair ? c.BN / 2 : c.BN)),
                         rows32 ? CU_TENSOR_MAP_SWIZZLE_32B : c.swizzle))
      return ADAPTION_ERR_CUDA;
  }

  if (c.staged) {
    // rows and columns of a stored tile: pooling halves the rows, or with grouped pixels the columns
    const bool halve_rows = g.pool_w && G == 1, halve_cols = g.pool_w && G > 1;
    const int ycols = halve_cols ? c.BN / 2 : c.BN;
    const int ybox = ycols < 128 ? ycols : 128;     // wider tiles leave as several stores of 128 columns
    const uint64_t ypitch = (uint64_t)(halve_cols ? y_stride / 2 : y_stride);
    const CUtensorMapSwizzle yswz = ybox == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                                : (ybox == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    const void* planes[2] = {g.y.hi, g.y.lo};
    for (int i = 0; i < 2; ++i) {
      if (planes[i] == nullptr) continue;      // single-plane outputs have no high plane
      if (c.box.on) {
        const int half = c.box.pool;
        const uint64_t W = (uint64_t)(g.OW >> half), H = (uint64_t)(g.OH >> half);
        const uint64_t dims[4] = {ypitch, W, H, (uint64_t)g.cs.N}, strides[3] = {ypitch, ypitch * W, ypitch * W * H};
        uint32_t box[4] = {(uint32_t)ybox, 1u << (c.box.w - half), 1u << (c.box.h - half), 1u << c.box.n};
        if (c.own_rows) {        // 32 of the tile's rows
          const int h = c.box.w + c.box.h < 5 ? c.box.h : 5 - c.box.w;
          box[2] = 1u << (h - half);
          box[3] = 1u << (5 - c.box.w - h);
        }
        if (!encode_tiled(&maps[4 + i], planes[i], 4, dims, strides, box, nullptr, yswz)) return ADAPTION_ERR_CUDA;
        continue;
      }
      if (!encode_tiled_2d(&maps[4 + i], planes[i], ypitch, (uint64_t)(halve_rows ? M / 2 : M), ypitch, (uint32_t)ybox,
                           (uint32_t)((halve_rows ? kBM / 2 : kBM) / (c.own_rows ? 4 : 1)), yswz))
        return ADAPTION_ERR_CUDA;
    }
  }

  TcParams p;
  std::memset(&p, 0, sizeof(p));
  p.M = (int)M; p.N = (int)N; p.tile_m = c.tile_m;
  p.tiles_m = c.tiles_m; p.tiles_n = c.tiles_n; p.splits = c.splits;
  p.total_tiles = c.tiles_m * c.tiles_n * c.splits;
  p.num_kb = c.num_kb; p.kb_per_split = c.kb_per_split;
  p.BN = c.BN; p.BK = c.BK; p.ksteps = c.BK / 32;
  p.px = c.px;
  p.box = c.box;
  p.halo = c.halo;
  p.ksteps_last = g.is_conv ? c.ksteps_last : p.ksteps;
  p.sbo = (uint32_t)((c.halo.w > 0 ? c.halo.w : 8) * c.BK); p.layout_type = c.layout_type;
  p.stages = c.stages; p.a_bytes = c.a_bytes; p.b_bytes = c.b_bytes; p.stage_bytes = c.stage_bytes;
  p.kps = c.kps; p.kb_bytes = c.kb_bytes;
  p.tx_bytes = c.a_tx != 0 ? (uint32_t)c.nax * c.a_tx : c.kb_bytes;
  p.b_resident = c.b_resident ? 1 : 0;
  p.b_blocks = c.b_blocks;
  p.b_res_off = (uint32_t)c.stages * c.stage_bytes;
  p.acc_bufs = c.acc_bufs;
  p.acc_shift = c.acc_bufs == 4 ? 2 : (c.acc_bufs == 2 ? 1 : 0);
  p.div_tiles_n = fast_div(c.tiles_n);
  p.div_splits = fast_div(c.splits);
  p.div_ow = fast_div(g.is_conv ? OW : 1);
  p.div_oh = fast_div(g.is_conv ? g.OH : 1);
  const int taps_s = G > 1 ? c.px.blocks : g.cs.S;       // k-blocks per filter row and channel block
  p.div_s = fast_div(g.is_conv ? taps_s : 1);
  p.div_cblks = fast_div(c.cblks);
  p.tmem_cols = c.tmem_cols;
  p.split_hh = (c.nacc == 3 && c.acc_bufs == 1 && 4 * c.BN <= 512 && knob(kSplitHh) != 0) ? 1 : 0;
  if (p.split_hh) p.tmem_cols = 512;
  p.is_conv = g.is_conv ? 1 : 0;
  p.cblks = c.cblks;
  if (g.is_conv) {
    p.OH = g.OH; p.OW = OW; p.S = taps_s; p.w_pitch = (int)g.w.c_stride;
    p.stride_h = g.cs.stride_h; p.stride_w = g.cs.stride_w; p.pad_h = g.cs.pad_h; p.pad_w = cs.pad_w;
  }
  p.bias = g.bias; p.bias_shift = g.bias_shift;
  p.mode = g.mode;
  p.rq = rq;
  if (g.mode == ADAPTION_MODE_REQUANT) {
    p.y_hi = (int8_t*)g.y.hi; p.y_lo = (uint8_t*)g.y.lo; p.y_q16 = g.y.q16; p.y_stride = y_stride;
  }
  if (g.pool_w && !(c.staged && g.M % 2 == 0)) return ADAPTION_ERR_UNSUPPORTED;
  if (g.box_pool && !(c.staged && c.box.pool)) return ADAPTION_ERR_UNSUPPORTED;
  p.pool_w = g.pool_w ? 1 : 0;
  p.epi_groups = c.epi_groups;
  p.own_rows = c.own_rows ? 1 : 0;
  p.staged = c.staged ? 1 : 0;
  p.stage_bufs = c.stage_bufs;
  p.stage_off = c.stage_off;
  p.const_off = c.stage_off + c.stage_out_bytes;
  // stochastic rounding happens where the value is requantized: in this kernel's epilogue, or in the
  // finalize kernel when the reduction is split
  p.st = g.stochastic;
  if (g.mode != ADAPTION_MODE_REQUANT || c.splits > 1) p.st.enabled = 0;
  p.fast_relu = fast == 1 ? 1 : 0;
  p.fast_stochastic = fast == 2 ? 1 : 0;
  p.byte_out = p.fast_relu && c.nacc == 1 && c.staged && rq.shift >= 1 && rq.out_planes == 1 && rq.qmax == 127 ? 1 : 0;
  p.fast_range = g.mode == ADAPTION_MODE_RANGE && c.splits == 1 && knob(kFast) != 0 && fits_32_bits(g, c, 0) ? 1 : 0;
  const bool grouped_kernel = c.kps > 1 || c.b_resident;     // (resident: also the tiles copied with their margin)
  p.tail_stagger = (p.split_hh && p.fast_relu && !grouped_kernel && c.kb_per_split >= 3 && c.stages >= 3 &&
                    c.nax == 2 && c.nbw == 2 && knob(kStagger) != 0) ? 1 : 0;
  p.ws = (long long*)g.workspace; p.ws_ld = g.N;
  p.stats = g.stats;
  p.timeout_ns = wait_limit_ns();
  p.stall_at = knob(kStallAt);

  if (c.splits > 1) {
    const cudaError_t me = cudaMemsetAsync(g.workspace, 0, c.workspace_bytes, g.stream);
    if (me != cudaSuccess) return cuda_failure(me, "split-K workspace memset");
  }
  int grid;
  if (c.pair) {
    const int pairs = num_sms() / 2;
    grid = 2 * (p.total_tiles < pairs ? p.total_tiles : pairs);
  } else {
    grid = p.total_tiles < num_sms() ? p.total_tiles : num_sms();
  }
  int rc;
  if (c.nax == 2 && c.nbw == 2) rc = launch_either<2, 2>(c.pair, maps, p, grid, c.smem_bytes, g.stream);
  else if (c.nax == 2) rc = launch_either<2, 1>(c.pair, maps, p, grid, c.smem_bytes, g.stream);
  else if (c.nbw == 2) rc = launch_either<1, 2>(c.pair, maps, p, grid, c.smem_bytes, g.stream);
  else rc = launch_either<1, 1>(c.pair, maps, p, grid, c.smem_bytes, g.stream);
  if (rc != ADAPTION_OK) return rc;
  if (c.splits > 1) return launch_finalize((const int64_t*)g.workspace, g.N, g);
  return ADAPTION_OK;
}

}  // namespace adaption
