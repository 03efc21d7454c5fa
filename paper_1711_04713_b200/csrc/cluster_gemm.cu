// LPConvolution / LPInnerProduct (paper Sec. 2) for layers with few output tiles: one thread-block
// cluster per output tile.
//
// The persistent kernel (gemm_tc.cu) needs at least about one 128- or 256-row tile per SM.  A layer with
// fewer (a small batch, the deep layers of a network on one image, the inner products) leaves most SMs
// idle unless its reduction is split, and a split there costs a cleared workspace, 64-bit atomics and
// a second kernel.  Here the CTAs of a cluster share one output tile: each reduces its own share of the
// k-blocks on the tensor cores, then sends the columns that the others own to them (bulk copies from
// shared memory to the peers' shared memory), and every CTA finishes (bias, ReLU, requantization, counters,
// optional 2x2 max-pool, stores) the columns it owns.  One launch per layer, no workspace.
//
// Operands:
//   convolution    rows = output pixels: a box of bn images x bh rows x bw columns with
//                  bn * bh * bw <= 128, fetched per filter tap by one tiled copy (zero fill outside the image,
//                  element strides for strided layers), so tensors of few bytes qualify and the tile's
//                  shape can follow the 2x2 windows of a pool; columns = output channels.  A row of outputs is
//                  at most 16 boxes: widths up to 2048, with a pool (boxes of at most 64 columns) up to 1024
//   inner product  rows = 128 output channels, columns = the batch rows: the weights take the
//                  128-row side of the MMA, so a batch of 1 to 16 costs 16 columns instead of 128 rows
// K-blocks are 128 bytes of one tap's channels.  Where the channel pitch is no multiple of 128 the copy's
// box reaches past the pitch: the rest arrives as zeros without being read, and the MMAs skip it.
//
// What bounds it: latency (launch, first copies, the exchange), then for inner products the weight
// stream from HBM.
#include <cuda.h>

#include <cstring>

#include "common.cuh"
#include "knobs.cuh"
#include "tc_ptx.cuh"
#include "tensor_maps.cuh"

namespace adaption {

int num_sms();

namespace {

constexpr int kRows = 128;
constexpr int kMaxClusterStages = 12;
constexpr int kClusterThreads = 384;      // warps 0, 1: copies; 2: MMA; 4-7: tables; then all of them the epilogue
constexpr int kClusterWarps = kClusterThreads / 32;
constexpr int kFirstTableWarp = 4;
// exchange: one 16-byte slot (two columns' 64-bit partial sums) per pair of columns and row
constexpr uint32_t kPairBytes = kRows * 16;

struct CgParams {
  int M, N;                       // logical output: M pixels or batch rows, N channels
  int S;                          // CTAs per tile (cluster size)
  int tiles_c;                    // column tiles (fastest in the block index)
  int BN, BK;
  int num_kb, kb_per_split;
  int ksteps, ksteps_last;        // 32-byte steps of a k-block, of the last channel block of a tap
  uint32_t sbo, layout_type;
  int stages;
  uint32_t a_bytes, b_bytes, a_tx, stage_bytes, tmem_cols;
  int is_conv;
  int cblks, S_w, stride_h, stride_w, pad_h, pad_w, OH, OW, images;
  int bw, bh, bn, tiles_w, tiles_h;
  int pool;                       // store the maxima of 2x2 windows
  const int16_t* bias;
  int bias_shift;
  RequantParams rq;
  StochasticParams st;
  int mode;
  int8_t* y_hi;
  uint8_t* y_lo;
  int16_t* y_q16;
  long long y_stride;
  int y_cols;                     // columns stored per row: N and the padding behind it
  adaption_stats* stats;
  unsigned long long timeout_ns;
  int stall_at;                   // test aid, see adaption_debug_set
};

// Optional time stamps of block 0 (development builds only: -DADAPTION_TIMELINE).
#ifdef ADAPTION_TIMELINE
__device__ long long g_cg_timeline[64];
#define CG_STAMP(slot)                                                    \
  do {                                                                    \
    if (blockIdx.x == 0 && lane == 0) g_cg_timeline[slot] = clock64();     \
  } while (0)
#else
#define CG_STAMP(slot) do { } while (0)
#endif

struct CgCtrl {
  unsigned long long full[kMaxClusterStages];
  unsigned long long empty[kMaxClusterStages];
  unsigned long long done;        // every MMA of this CTA has retired
  unsigned long long recv;        // the peers' partial sums have arrived
  long long bias[kRows];          // aligned to the accumulator: per owned column (convolution) or row (inner product)
  int pix[kRows];                 // convolution: output pixel of a row of the tile (pool: of a window), -1 = outside
  int win_row[kRows / 4];         // pool: first row of a window
  uint32_t tmem_base;
  volatile uint32_t abort;
};

__device__ __noinline__ bool cg_wait_slow(uint32_t bar, uint32_t parity, CgCtrl* ctrl, const CgParams& p) {
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
__device__ __forceinline__ bool cg_wait(uint32_t bar, uint32_t parity, CgCtrl* ctrl, const CgParams& p) {
  if (mbar_try_wait(bar, parity)) return true;
  return cg_wait_slow(bar, parity, ctrl, p);
}

__device__ __forceinline__ void st_shared_pair(uint32_t addr, long long a, long long b) {
  asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(addr), "l"(a), "l"(b) : "memory");
}
// shared memory of this CTA -> shared memory of a peer, reported to a barrier of that peer
__device__ __forceinline__ void bulk_copy_to_peer(uint32_t dst_cluster, uint32_t src, uint32_t bytes, uint32_t bar_cluster) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   dst_cluster),
               "r"(src), "r"(bytes), "r"(bar_cluster)
               : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// Where the partial sums of a CTA's own columns lie: its own share, then one block per peer.
struct Slots {
  const uint8_t* own;
  const uint8_t* in;             // blocks of np pairs
  int peers, np;
};

// sum of the partial sums of `G` owned columns (from pair `pair` on) of one row
template <int G>
__device__ __forceinline__ void slot_sums(const Slots& s, int pair, int row, long long (&v)[G]) {
  const uint32_t off = (uint32_t)pair * kPairBytes + (uint32_t)row * 16u;
#pragma unroll
  for (int j = 0; j < G; j += 2) {
    const longlong2 t = *reinterpret_cast<const longlong2*>(s.own + off + (uint32_t)(j >> 1) * kPairBytes);
    v[j] = t.x;
    v[j + 1] = t.y;
  }
  const uint8_t* q = s.in + off;
  for (int src = 0; src < s.peers; ++src, q += (uint32_t)s.np * kPairBytes) {
#pragma unroll
    for (int j = 0; j < G; j += 2) {
      const longlong2 t = *reinterpret_cast<const longlong2*>(q + (uint32_t)(j >> 1) * kPairBytes);
      v[j] += t.x;
      v[j + 1] += t.y;
    }
  }
}

__device__ __forceinline__ void keep_range(long long v, const CgParams& p, long long& vmax) {
  if (p.rq.relu && v < 0) v = 0;
  v = v < 0 ? -v : v;
  vmax = v > vmax ? v : vmax;
}

__device__ __forceinline__ void store_q2(const CgParams& p, size_t off, int32_t q0, int32_t q1) {
  // (columns are even and the pitch is a multiple of 16: two-byte stores are aligned)
  *reinterpret_cast<uint16_t*>(p.y_lo + off) = (uint16_t)((q0 & 255) | ((q1 & 255) << 8));
  if (p.rq.out_planes == 2)
    *reinterpret_cast<uint16_t*>(p.y_hi + off) = (uint16_t)(((q0 >> 8) & 255) | (q1 & 0xff00));
  if (p.y_q16 != nullptr)
    *reinterpret_cast<uint32_t*>(p.y_q16 + off) = (uint32_t)(q0 & 0xffff) | ((uint32_t)q1 << 16);
}

// `G` consecutive channels of one output pixel
template <int G>
__device__ __forceinline__ void store_group(const CgParams& p, size_t off, const int32_t (&q)[G]) {
  if constexpr (G == 2) {
    store_q2(p, off, q[0], q[1]);
  } else {
    static_assert(G == 8, "groups of two or eight channels");
    uint32_t w[4];                                            // packed pairs of 16-bit values
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = __byte_perm((uint32_t)q[2 * j], (uint32_t)q[2 * j + 1], 0x5410);
    *reinterpret_cast<uint2*>(p.y_lo + off) = make_uint2(__byte_perm(w[0], w[1], 0x6420), __byte_perm(w[2], w[3], 0x6420));
    if (p.rq.out_planes == 2)
      *reinterpret_cast<uint2*>(p.y_hi + off) = make_uint2(__byte_perm(w[0], w[1], 0x7531), __byte_perm(w[2], w[3], 0x7531));
    if (p.y_q16 != nullptr) *reinterpret_cast<uint4*>(p.y_q16 + off) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// What happens to a finished sum.  Each kind has a kernel of its own, so that a launch only fetches the
// instructions it runs: with the generator inlined beside the deterministic path the final stage of a
// 128 x 128 tile took 29 k cycles, nearly all of it instruction fetches.  (Three epilogues in one kernel: 150 registers
// where rounding alone takes 94, and every change of one moved the others; weights not in L2, us, one kernel and three: 5
// rows, 4096 -> 1000, 16 bits 7.33 and 7.18, 8 by 16 bits 6.57 and 6.42; 2 rows, 284 -> 813 4.91 and 4.75.)
constexpr int kFinishRound = 0, kFinishStochastic = 1, kFinishRange = 2;

// `G` finished sums (the first `nreal` are real outputs, the rest padding with sum 0) of the elements `index`,
// `index + step`, ...
template <int G, int KIND>
__device__ __forceinline__ void finish_group(const long long (&v)[G], int nreal, const CgParams& p, uint64_t index, uint64_t step,
                                             int32_t (&q)[G], Counts& cnt, long long& vmax) {
  if constexpr (KIND == kFinishRange) {
#pragma unroll
    for (int j = 0; j < G; ++j) keep_range(v[j], p, vmax);
  } else if constexpr (KIND == kFinishStochastic) {
    if (G == 8) {      // (a convolution of N % 8 = 0 channels, finish_tile: two whole generator blocks, or padding)
      if (nreal == 0) {
#pragma unroll
        for (int j = 0; j < G; ++j) q[j] = 0;
        return;
      }
#pragma unroll
      for (int b = 0; b < G / 4; ++b) {
        const uint64_t blk = (index >> 2) + (uint64_t)b;
        const Philox4 r = philox4x32_10((uint32_t)blk, (uint32_t)(blk >> 32), 0u, 0u, p.st.key0, p.st.key1);
#pragma unroll
        for (int j = 0; j < 4; ++j) q[4 * b + j] = requant_value_stochastic(v[4 * b + j], p.rq, r.w[j], true, cnt);
      }
      return;
    }
#pragma unroll
    for (int j = 0; j < G; ++j) {
      q[j] = 0;
      if (j < nreal)
        q[j] = requant_value_stochastic(v[j], p.rq, philox_draw(index + (uint64_t)j * step, p.st.key0, p.st.key1), true, cnt);
    }
  } else if (p.rq.shift <= 0) {
#pragma unroll
    for (int j = 0; j < G; ++j) q[j] = requant_value(v[j], p.rq, j < nreal, cnt);
  } else {
    // rounding right shift (half away from zero), narrowed to 32 bits with saturation, clamped; zeros are
    // counted per group, clipped values only where a clamp changed something
    const long long half = 1ll << (p.rq.shift - 1);
    int32_t r[G], clipped = 0, nonzero = 0;
#pragma unroll
    for (int j = 0; j < G; ++j) {
      const long long x = p.rq.relu && v[j] < 0 ? 0ll : v[j];
      const long long t = (x + half + (x >> 63)) >> p.rq.shift;
      const int32_t t32 = (int32_t)t, th = (int32_t)(t >> 32);
      r[j] = th == (t32 >> 31) ? t32 : (th < 0 ? (int32_t)0x80000000 : 0x7fffffff);
      q[j] = min(max(r[j], p.rq.qmin), p.rq.qmax);
      clipped |= r[j] ^ q[j];
      nonzero += q[j] != 0 ? 1 : 0;
    }
    cnt.zeros += (uint32_t)(nreal - nonzero);
    if (clipped != 0) {
#pragma unroll
      for (int j = 0; j < G; ++j) {
        cnt.sat_pos += r[j] > p.rq.qmax;
        cnt.sat_neg += r[j] < p.rq.qmin;
      }
    }
  }
}

// Inner product: a thread keeps one output channel (row of the tile; consecutive lanes store consecutive
// bytes) and walks the batch rows this CTA owns, `G` at a time.
template <int G, int KIND>
__device__ __forceinline__ void finish_inner_product(const CgParams& p, const Slots& slots, const CgCtrl& ctrl, int cpo,
                                                     int r0, int col_first) {
  Counts cnt;
  long long vmax = 0;
  const int row = (int)threadIdx.x & (kRows - 1), n = r0 + row;
  if (n < p.y_cols) {
    const bool real = n < p.N;
    const long long bias = ctrl.bias[row];
#pragma unroll 1
    for (int g = (int)threadIdx.x / kRows; g * G < cpo; g += kClusterThreads / kRows) {
      const int m = col_first + g * G;
      if (m >= p.M) break;
      const int rows = min(G, p.M - m);
      long long v[G];
      int32_t q[G];
      slot_sums<G>(slots, g * (G / 2), row, v);
#pragma unroll
      for (int e = 0; e < G; ++e) v[e] = real && e < rows ? v[e] + bias : 0;
      // (element indices of consecutive batch rows are N apart)
      finish_group<G, KIND>(v, real ? rows : 0, p, (uint64_t)m * (uint64_t)p.N + (uint64_t)n, (uint64_t)p.N, q, cnt, vmax);
      if (KIND != kFinishRange) {
#pragma unroll
        for (int e = 0; e < G; ++e)
          if (e < rows)
            store_q(p.rq.out_planes == 2 ? p.y_hi : nullptr, p.y_lo, p.y_q16, (size_t)(m + e) * (size_t)p.y_stride + n, q[e]);
      }
    }
  }
  __syncwarp();
  if (KIND == kFinishRange) flush_max_warp(vmax, p.stats);
  else flush_counts_warp(cnt, p.stats);
}

// Convolution: a thread keeps one pixel (with a pool: one 2x2 window) and walks groups of `G` of the
// channels this CTA owns.
template <int G, int KIND>
__device__ __forceinline__ void finish_conv(const CgParams& p, const Slots& slots, const CgCtrl& ctrl, int cpo,
                                            int col_first) {
  Counts cnt;
  long long vmax = 0;
  const int lanes = p.pool ? kRows / 4 : kRows;
  const int item = (int)threadIdx.x & (lanes - 1);
  const int pix = ctrl.pix[item];
  if (pix >= 0) {
    const int first_row = p.pool ? ctrl.win_row[item] : item;
    const int points = p.pool ? 4 : 1;
#pragma unroll 1
    for (int g = (int)threadIdx.x / lanes; g * G < cpo; g += kClusterThreads / lanes) {
      const int n0 = col_first + g * G;
      if (n0 >= p.y_cols) break;
      const int nreal = min(G, max(0, p.N - n0));
      int32_t best[G];
#pragma unroll 1
      for (int w = 0; w < points; ++w) {
        long long v[G];
        int32_t q[G];
        slot_sums<G>(slots, g * (G / 2), first_row + (w >> 1) * p.bw + (w & 1), v);
#pragma unroll
        for (int j = 0; j < G; ++j) v[j] = j < nreal ? v[j] + ctrl.bias[g * G + j] : 0;
        // (stochastic rounding never comes with a pool: `pix` is the pixel's own index)
        finish_group<G, KIND>(v, nreal, p, (uint64_t)pix * (uint64_t)p.N + (uint64_t)n0, 1, q, cnt, vmax);
#pragma unroll
        for (int j = 0; j < G; ++j) best[j] = w == 0 ? q[j] : max(best[j], q[j]);
      }
      if (KIND != kFinishRange) store_group<G>(p, (size_t)pix * (size_t)p.y_stride + n0, best);
    }
  }
  __syncwarp();
  if (KIND == kFinishRange) flush_max_warp(vmax, p.stats);
  else flush_counts_warp(cnt, p.stats);
}

template <int KIND>
__device__ __forceinline__ void finish_tile(const CgParams& p, const Slots& slots, const CgCtrl& ctrl, int cpo, int r0,
                                            int col_first) {
  // (eight at a time where the owned columns divide: 310 cycles per value and thread against 780)
  const bool wide = (cpo & 7) == 0 && (KIND == kFinishRound || (KIND == kFinishStochastic && p.is_conv && p.N % 8 == 0));
  if (!p.is_conv) {
    if (wide)
      finish_inner_product<8, KIND>(p, slots, ctrl, cpo, r0, col_first);
    else
      finish_inner_product<2, KIND>(p, slots, ctrl, cpo, r0, col_first);
  } else if (wide && (!p.pool || cpo >= 64)) {
    finish_conv<8, KIND>(p, slots, ctrl, cpo, col_first);
  } else {
    finish_conv<2, KIND>(p, slots, ctrl, cpo, col_first);
  }
}

template <int NAX, int NBW, int KIND>
__global__ void __launch_bounds__(kClusterThreads, 1)
lp_cluster_kernel(const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_a1,
                  const __grid_constant__ CUtensorMap map_b0, const __grid_constant__ CUtensorMap map_b1,
                  const CgParams p) {
  constexpr int NACC = NAX + NBW - 1;
  extern __shared__ uint8_t smem_raw[];
  __shared__ CgCtrl ctrl;
  const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* const ring_ptr = smem_raw + (ring - smem_u32(smem_raw));
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const uint32_t rank = p.S > 1 ? cluster_ctarank() : 0u;
  const int tile = (int)blockIdx.x / p.S;
  if (warp == 0) CG_STAMP(0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&ctrl.full[s]), 2);       // one arming arrival per copying warp
      mbar_init(smem_u32(&ctrl.empty[s]), 1);
    }
    mbar_init(smem_u32(&ctrl.done), 1);
    mbar_init(smem_u32(&ctrl.recv), 1);
    ctrl.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1 && lane < 4) prefetch_map(lane == 0 ? &map_a0 : (lane == 1 ? &map_b0 : (lane == 2 ? &map_a1 : &map_b1)));
  if (warp == 2) {
    tmem_alloc<false>(smem_u32(&ctrl.tmem_base), p.tmem_cols);
    tmem_relinquish<false>();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctrl.tmem_base;

  // tile coordinates
  const int tc = tile % p.tiles_c;
  const int tr = tile / p.tiles_c;
  const int c0 = tc * p.BN;                                  // first column of the tile
  int ow0 = 0, oh0 = 0, img0 = 0;
  if (p.is_conv) {
    const int rest = tr / p.tiles_w;
    ow0 = (tr - rest * p.tiles_w) * p.bw;
    const int ib = rest / p.tiles_h;
    oh0 = (rest - ib * p.tiles_h) * p.bh;
    img0 = ib * p.bn;
  }
  const int r0 = tr * kRows;                                 // inner product: first output channel
  const int kb_begin = (int)rank * p.kb_per_split;
  const int kb_end = min(p.num_kb, kb_begin + p.kb_per_split);
  const int cpo = p.BN / p.S;                // columns each CTA owns
  const int np = cpo / 2;                    // ... as pairs
  if (warp == 0) CG_STAMP(1);

  pdl_wait();
  pdl_launch_dependents();
  if (warp == 0) CG_STAMP(2);

  bool ok = true;
  if (warp < 2) {
    // ---- copies: warp 0 the row operand's planes, warp 1 the column operand's
    const bool is_a = warp == 0;
    const CUtensorMap* m0 = is_a ? &map_a0 : &map_b0;
    const CUtensorMap* m1 = is_a ? &map_a1 : &map_b1;
    const int planes = is_a ? NAX : NBW;
    const uint32_t pb = is_a ? p.a_bytes : p.b_bytes;
    const uint32_t tx = (uint32_t)planes * (is_a ? p.a_tx : p.b_bytes);
    const uint32_t off = is_a ? 0u : (uint32_t)NAX * p.a_bytes;
    int s = 0, issued = 0;
    uint32_t ph = 0;
    int tap = 0, cb = 0, r = 0, sx = 0;
    if (p.is_conv) {
      tap = kb_begin / p.cblks;
      cb = kb_begin - tap * p.cblks;
      r = tap / p.S_w;
      sx = tap - r * p.S_w;
    }
    for (int kb = kb_begin; kb < kb_end; ++kb) {
      if (issued == p.stall_at) break;
      ok = __all_sync(0xffffffffu, cg_wait(smem_u32(&ctrl.empty[s]), ph ^ 1u, &ctrl, p));
      if (!ok) break;
      if (elect_one()) {
        const uint32_t full = smem_u32(&ctrl.full[s]);
        const uint32_t dst = ring + (uint32_t)s * p.stage_bytes + off;
        mbar_expect_tx(full, tx);
        if (!p.is_conv) {
          tma_load_2d<false>(dst, m0, full, kb * p.BK, is_a ? r0 : c0);
          if (planes == 2) tma_load_2d<false>(dst + pb, m1, full, kb * p.BK, is_a ? r0 : c0);
        } else if (is_a) {
          const int x = ow0 * p.stride_w - p.pad_w + sx, y = oh0 * p.stride_h - p.pad_h + r;
          tma_load_4d<false>(dst, m0, full, cb * p.BK, x, y, img0);
          if (planes == 2) tma_load_4d<false>(dst + pb, m1, full, cb * p.BK, x, y, img0);
        } else {
          tma_load_3d<false>(dst, m0, full, cb * p.BK, tap, c0);
          if (planes == 2) tma_load_3d<false>(dst + pb, m1, full, cb * p.BK, tap, c0);
        }
      }
      __syncwarp();
      ++issued;
      if (p.is_conv && ++cb == p.cblks) {
        cb = 0;
        ++tap;
        if (++sx == p.S_w) { sx = 0; ++r; }
      }
      if (++s == p.stages) { s = 0; ph ^= 1u; }
    }
    // the ring is given another use only once the MMAs (or the issuing warp, giving up) are through with it
    if (!cg_wait(smem_u32(&ctrl.done), 0, &ctrl, p)) ok = false;
    if ((!ok || ctrl.abort) && lane == 0) {
      // gave up: let the copies in flight land.  (A stage that only one of the two copying warps armed
      // never completes its phase: that wait runs out.)
      const int n = issued < p.stages ? issued : p.stages;
      for (int j = issued - n; j < issued; ++j) {
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(smem_u32(&ctrl.full[j % p.stages]), (uint32_t)(j / p.stages) & 1u) &&
               global_ns() - t0 < 5000000ull) {
        }
      }
    }
    __syncwarp();
  } else if (warp == 2) {
    // ---- MMA issue
    const uint32_t id_ss = make_idesc(true, true, p.BN, kRows), id_su = make_idesc(true, false, p.BN, kRows);
    const uint32_t id_us = make_idesc(false, true, p.BN, kRows), id_uu = make_idesc(false, false, p.BN, kRows);
    const uint32_t dhi = smem_desc_hi(p.sbo, p.layout_type);
    const uint32_t a_u = p.a_bytes >> 4, b_u = p.b_bytes >> 4;
    const uint32_t d0 = tmem_base, d1 = d0 + (uint32_t)p.BN, d2 = d1 + (uint32_t)p.BN;
    int s = 0;
    uint32_t ph = 0;
    int cb = p.is_conv ? kb_begin % p.cblks : 0;
    for (int kb = kb_begin; kb < kb_end; ++kb) {
      ok = __all_sync(0xffffffffu, cg_wait(smem_u32(&ctrl.full[s]), ph, &ctrl, p));
      if (!ok) break;
      tc_fence_after();
      if (kb - kb_begin < 32) CG_STAMP(16 + kb - kb_begin);
      const int ksteps = (p.is_conv && cb == p.cblks - 1) ? p.ksteps_last : p.ksteps;
      // (straight-line code on warp-uniform operands: a loop inside the elected branch costs the issuing
      // thread 68 cycles per MMA, more than a narrow MMA takes)
      const uint32_t a0 = smem_desc_lo(ring) + (uint32_t)s * (p.stage_bytes >> 4);
      const uint32_t a1 = a0 + a_u, b0 = a0 + (uint32_t)NAX * a_u, b1 = b0 + b_u;
      const uint32_t acc = kb == kb_begin ? 0u : 1u;
      if (elect_one()) {
        mma_kstep<NAX, NBW, false>(d0, d1, d2, a0, a1, b0, b1, dhi, id_ss, id_su, id_us, id_uu, acc);
        if (ksteps > 1)
          mma_kstep<NAX, NBW, false>(d0, d1, d2, a0 + 2u, a1 + 2u, b0 + 2u, b1 + 2u, dhi, id_ss, id_su, id_us, id_uu, 1u);
        if (ksteps > 2)
          mma_kstep<NAX, NBW, false>(d0, d1, d2, a0 + 4u, a1 + 4u, b0 + 4u, b1 + 4u, dhi, id_ss, id_su, id_us, id_uu, 1u);
        if (ksteps > 3)
          mma_kstep<NAX, NBW, false>(d0, d1, d2, a0 + 6u, a1 + 6u, b0 + 6u, b1 + 6u, dhi, id_ss, id_su, id_us, id_uu, 1u);
        tc_commit<false>(smem_u32(&ctrl.empty[s]));
      }
      __syncwarp();
      if (p.is_conv && ++cb == p.cblks) cb = 0;
      if (++s == p.stages) { s = 0; ph ^= 1u; }
    }
    CG_STAMP(3);
    if (elect_one()) tc_commit<false>(smem_u32(&ctrl.done));
    __syncwarp();
    if (!ok || ctrl.abort) {
      // no MMA may still read shared memory when the ring is given another use
      const unsigned long long t0 = global_ns();
      while (!mbar_try_wait(smem_u32(&ctrl.done), 0) && global_ns() - t0 < 50000000ull) {
      }
    }
  } else if (warp >= kFirstTableWarp) {
    // ---- while the main loop runs: what the epilogue needs to know about rows and columns
    const int t = (int)threadIdx.x - 32 * kFirstTableWarp;
    if (t < kRows) {
      const int n = p.is_conv ? c0 + (int)rank * cpo + t : r0 + t;
      ctrl.bias[t] = (p.bias != nullptr && n < p.N && (!p.is_conv || t < cpo)) ? (long long)p.bias[n] * (1ll << p.bias_shift) : 0;
      if (p.is_conv) {
        const int step = p.pool ? 2 : 1;
        const int iw = p.bw / step, ih = p.bh / step;
        const int wl = (t % iw) * step, hl = ((t / iw) % ih) * step, nl = t / (iw * ih);
        const int oh = oh0 + hl, ow = ow0 + wl, img = img0 + nl;
        const bool inside = nl < p.bn && oh < p.OH && ow < p.OW && img < p.images;
        ctrl.pix[t] = inside ? (img * (p.OH / step) + oh / step) * (p.OW / step) + ow / step : -1;
        if (p.pool && t < kRows / 4) ctrl.win_row[t] = inside ? (nl * p.bh + hl) * p.bw + wl : 0;
      }
    }
    if (warp == kFirstTableWarp) CG_STAMP(4);
  }
  __syncwarp();

  // The ring turns into exchange buffers once every MMA has retired: this CTA's partial sums, one block of
  // np pairs per owner of columns (its own block stays), behind them the peers' blocks for its columns.
  const uint32_t block_bytes = (uint32_t)np * kPairBytes;
  const uint32_t in_off = (uint32_t)p.S * block_bytes;
  if (threadIdx.x == 0 && p.S > 1) mbar_expect_tx(smem_u32(&ctrl.recv), (uint32_t)(p.S - 1) * block_bytes);
  __syncthreads();
  // (the peers may write here from now on; the wait for theirs comes behind the drain)
  if (p.S > 1) cluster_arrive();
  if (warp == kFirstTableWarp) CG_STAMP(5);
  {
    const int rows_used = p.is_conv ? p.bw * p.bh * p.bn : kRows;
    const int cols_real = min(p.BN, (p.is_conv ? p.N : p.M) - c0);
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const bool row_ok = row < rows_used;
    tc_fence_after();
    if (quarter * 32 < rows_used) {
      for (int c = 16 * (warp >> 2); c < cols_real; c += 16 * (kClusterWarps / 4)) {
        int32_t a[3][16];
        tmem_ld16(taddr + (uint32_t)c, reinterpret_cast<int32_t(&)[8]>(a[0][0]), reinterpret_cast<int32_t(&)[8]>(a[0][8]));
        if (NACC >= 2)
          tmem_ld16(taddr + (uint32_t)(p.BN + c), reinterpret_cast<int32_t(&)[8]>(a[1][0]),
                    reinterpret_cast<int32_t(&)[8]>(a[1][8]));
        if (NACC == 3)
          tmem_ld16(taddr + (uint32_t)(2 * p.BN + c), reinterpret_cast<int32_t(&)[8]>(a[2][0]),
                    reinterpret_cast<int32_t(&)[8]>(a[2][8]));
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < NACC; ++i) {
          pin_after_wait(reinterpret_cast<int32_t(&)[8]>(a[i][0]));
          pin_after_wait(reinterpret_cast<int32_t(&)[8]>(a[i][8]));
        }
        const uint32_t base = ring + (uint32_t)(c >> 1) * kPairBytes + (uint32_t)row * 16u;
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          if (c + j >= cols_real) break;
          long long v[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int32_t x0 = a[0][j + e];
            if (NACC == 3)
              v[e] = (long long)x0 * 65536ll + (long long)a[1][j + e] * 256ll + (long long)a[2][j + e];
            else if (NACC == 2)
              v[e] = (long long)x0 * 256ll + (long long)a[1][j + e];
            else
              v[e] = x0;
          }
          if (row_ok) st_shared_pair(base + (uint32_t)(j >> 1) * kPairBytes, v[0], v[1]);
        }
      }
    }
    tc_fence_before();
    if (warp == kFirstTableWarp) CG_STAMP(6);
  }
  fence_async_shared();
  if (p.S > 1) cluster_wait();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc<false>(tmem_base, p.tmem_cols);
  }
  if (p.S > 1) {
    if (threadIdx.x < (unsigned)p.S && threadIdx.x != rank) {
      // to owner `threadIdx.x`: its block of this CTA's sums (block index: this CTA's place among its peers)
      const uint32_t owner = threadIdx.x, place = rank - (rank > owner ? 1u : 0u);
      bulk_copy_to_peer(mapa_rank(ring + in_off + place * block_bytes, owner), ring + owner * block_bytes, block_bytes,
                        mapa_rank(smem_u32(&ctrl.recv), owner));
    }
    __syncwarp();
    ok = cg_wait(smem_u32(&ctrl.recv), 0, &ctrl, p);
    __syncwarp();
    cluster_arrive();           // (this CTA's shared memory is no longer written; the wait at the end keeps it readable)
  }
  if (warp == kFirstTableWarp) CG_STAMP(7);
  Slots slots;
  slots.own = ring_ptr + rank * block_bytes;
  slots.in = ring_ptr + in_off;
  slots.peers = p.S - 1;
  slots.np = np;

  // ---- the columns this CTA owns: sum over the CTAs, bias, ReLU, requantize, store
  const bool aborted = ctrl.abort != 0;
  const int col_first = c0 + (int)rank * cpo;
  if (!aborted) finish_tile<KIND>(p, slots, ctrl, cpo, r0, col_first);      // (else the status says that nothing was stored)
  if (warp == kFirstTableWarp) CG_STAMP(8);
  // zeros in the padding behind the last column tile (channels), if the pitch reaches that far
  const int pad_first = p.is_conv ? p.tiles_c * p.BN : (p.N + kRows - 1) / kRows * kRows;
  if (!aborted && p.mode == ADAPTION_MODE_REQUANT && p.y_cols > pad_first && (p.is_conv ? tc == p.tiles_c - 1 : r0 + kRows == pad_first)) {
    if (!p.is_conv) {
      for (int m = col_first; m < min(p.M, col_first + cpo); ++m)
        for (int n = pad_first + (int)threadIdx.x; n < p.y_cols; n += kClusterThreads)
          store_q(p.rq.out_planes == 2 ? p.y_hi : nullptr, p.y_lo, p.y_q16, (size_t)m * (size_t)p.y_stride + n, 0);
    } else if (threadIdx.x < (p.pool ? kRows / 4 : kRows) && ctrl.pix[threadIdx.x] >= 0) {
      for (int e = pad_first + 2 * (int)rank; e < p.y_cols; e += 2 * p.S)
        store_q2(p, (size_t)ctrl.pix[threadIdx.x] * (size_t)p.y_stride + e, 0, 0);
    }
  }
  if (warp == kFirstTableWarp) CG_STAMP(9);
  __syncwarp();
  if (p.S > 1) cluster_wait();
}

// ---------------------------------------------------------------------------------- host
struct CgPlan {
  bool ok = false;
  int nax = 1, nbw = 1;              // planes of the row and the column operand
  int BN = 0, BK = 0, S = 1;
  int cblks = 1, num_kb = 0, kb_per_split = 0, ksteps = 4, ksteps_last = 4;
  int bw = 0, bh = 0, bn = 0, tiles_w = 1, tiles_h = 1, tiles_r = 0, tiles_c = 0;
  int stages = 0;
  uint32_t a_bytes = 0, b_bytes = 0, stage_bytes = 0, tmem_cols = 32;
  size_t smem = 0;
  double cost = 0;
};

int ceil_div(int a, int b) { return (a + b - 1) / b; }

// The tile of output pixels with the fewest copies: whole rows if a row fits, several images if an image
// fits; with a pool every tile starts on even coordinates and holds whole 2x2 windows.
bool choose_box(CgPlan& c, int OW, int OH, int images, int stride_w, int stride_h, bool pool) {
  const int unit = pool ? 2 : 1;
  long long best = -1;
  for (int nw = 1; nw <= 16; ++nw) {
    const int bw = ceil_div(ceil_div(OW, nw), unit) * unit;
    if (bw < unit || bw * unit > kRows || (bw - 1) * stride_w + 1 > 256) continue;
    int bh = kRows / bw / unit * unit;
    const int hmax = ((256 - 1) / stride_h + 1) / unit * unit;
    if (bh > hmax) bh = hmax;
    const int oh_pad = ceil_div(OH, unit) * unit;
    if (bh > oh_pad) bh = oh_pad;
    if (bh < unit) continue;
    const int th = ceil_div(OH, bh);
    bh = ceil_div(ceil_div(OH, th), unit) * unit;
    int bn = 1;
    if (th == 1 && nw == 1) {
      bn = kRows / (bw * bh);
      if (bn > images) bn = images;
      if (bn < 1) bn = 1;
      bn = ceil_div(images, ceil_div(images, bn));
    }
    const int tw = ceil_div(OW, bw);
    const long long tiles = (long long)tw * th * ceil_div(images, bn);
    if (best < 0 || tiles < best) {
      best = tiles;
      c.bw = bw; c.bh = bh; c.bn = bn;
      c.tiles_w = tw; c.tiles_h = th;
    }
    if (bw <= 8) break;
  }
  if (best < 0 || best > (1 << 20)) return false;
  c.tiles_r = (int)best;
  return true;
}

// this CTA's sums for every owner of columns, and the peers' sums for its own columns
size_t exchange_bytes(int BN, int S) { return (size_t)(BN / 2 + (S - 1) * (BN / S / 2)) * kPairBytes; }
constexpr size_t kRingLimit = 220 * 1024;

// Estimated SM cycles of a layer with column tiles of `BN` and clusters of `S` (constants from per-role time
// stamps at 16 bits: 57 / 64 / 77 cycles per MMA at 16 / 64 / 128 columns, 12 bytes per cycle between shared
// memories, first data 3.4 k cycles after the start).
double plan_cost(const CgPlan& c, int BN, int S, int columns, int sms) {
  const int products = c.nax * c.nbw;
  const int kb = ceil_div(c.num_kb, S);
  const double mma = (double)c.ksteps * products * (54 + 0.18 * BN);
  const double load = 2.0 * (c.nax * kRows + c.nbw * BN);
  const double main_loop = kb * (mma > load ? mma : load);
  const int cpo = BN / S;
  const double drain = 600 + 15.0 * BN;
  const double exchange = S > 1 ? 1400 + 85.0 * (BN - cpo) : 0;
  const double finish = 800 + (cpo % 8 == 0 ? 310.0 : 780.0) * cpo * kRows / kClusterThreads;
  const long long ctas = (long long)c.tiles_r * ceil_div(columns, BN) * S;
  // (clusters of more than two CTAs do not fill every GPC)
  const int resident = S > 4 ? sms * 6 / 7 : (S > 2 ? sms * 9 / 10 : sms);
  const double waves = (double)((ctas + resident - 1) / resident);
  return waves * (3400 + main_loop + drain + exchange + finish) + (S > 1 && waves > 1 ? 4000.0 * waves : 0.0);
}

CgPlan make_plan(const GemmProblem& g, bool pool) {
  CgPlan c;
  if (g.M <= 0 || g.N <= 0 || g.M > (int64_t)1 << 24 || g.N > (int64_t)1 << 20 || g.K > (int64_t)1 << 30) return c;
  const int px = g.x.fmt.n_bits > 8 ? 2 : 1, pw = g.w.fmt.n_bits > 8 ? 2 : 1;
  int columns;
  if (g.is_conv) {
    const int64_t cs = g.x.c_stride;
    if (cs != g.w.c_stride || cs % 32 != 0 || cs > 65536) return c;
    if (g.cs.stride_h > 8 || g.cs.stride_w > 8 || g.cs.R > 255 || g.cs.S > 255) return c;
    c.nax = px; c.nbw = pw;
    c.BK = cs > 64 ? 128 : (int)cs;
    c.cblks = ceil_div((int)cs, c.BK);
    c.ksteps = c.BK / 32;
    c.ksteps_last = ((int)cs - (c.cblks - 1) * c.BK) / 32;
    c.num_kb = g.cs.R * g.cs.S * c.cblks;
    columns = (int)g.N;
    if (!choose_box(c, g.OW, g.OH, g.cs.N, g.cs.stride_w, g.cs.stride_h, pool)) return c;
  } else {
    if (g.K < 32) return c;
    c.nax = pw; c.nbw = px;
    c.BK = g.K > 64 ? 128 : (g.K > 32 ? 64 : 32);
    c.ksteps = c.ksteps_last = c.BK / 32;
    c.num_kb = (int)((g.K + c.BK - 1) / c.BK);
    columns = (int)g.M;
    c.tiles_r = (int)((g.N + kRows - 1) / kRows);
  }
  const int nacc = c.nax + c.nbw - 1, sms = num_sms();
  const int forced_s = knob(kClusterSize), forced_bn = knob(kClusterBN);
  double best = -1;
  const int bn_max = columns >= 128 ? 128 : ceil_div(columns, 16) * 16;
  for (int bn = 16; bn <= bn_max; bn += 16) {
    // equal tiles: the narrowest width for this number of column tiles
    if (bn != ceil_div(ceil_div(columns, ceil_div(columns, bn)), 16) * 16) continue;
    if (forced_bn > 0 && bn != forced_bn && bn != bn_max) continue;
    for (int s = 1; s <= 8; s *= 2) {
      if (s > c.num_kb || (bn / s) % 2 != 0 || bn / s < 2) continue;
      if (forced_s > 0 && s != forced_s) continue;
      if (ceil_div(c.num_kb, s) > 32768 / c.BK) continue;          // exact 32-bit accumulation
      if (exchange_bytes(bn, s) > kRingLimit) continue;
      const double cost = plan_cost(c, bn, s, columns, sms);
      if (best < 0 || cost < best || (forced_bn > 0 && bn == forced_bn && c.BN != forced_bn)) {
        best = cost;
        c.BN = bn;
        c.S = s;
      }
    }
  }
  if (best < 0) return c;
  c.cost = best;
  c.tiles_c = ceil_div(columns, c.BN);
  if ((long long)c.tiles_r * c.tiles_c * c.S > (1 << 24)) return c;
  c.kb_per_split = ceil_div(c.num_kb, c.S);
  // (every CTA of the cluster needs at least one k-block: its accumulators are read unconditionally)
  while (c.S > 1 && (c.S - 1) * c.kb_per_split >= c.num_kb) {
    c.S /= 2;
    c.kb_per_split = ceil_div(c.num_kb, c.S);
  }
  if (c.kb_per_split * c.BK > 32768) return c;
  c.a_bytes = (uint32_t)(kRows * c.BK);
  c.b_bytes = (uint32_t)(c.BN * c.BK);
  c.stage_bytes = (uint32_t)c.nax * c.a_bytes + (uint32_t)c.nbw * c.b_bytes;
  c.stage_bytes = (c.stage_bytes + 1023u) & ~1023u;
  c.stages = (int)(kRingLimit / c.stage_bytes);
  if (c.stages > c.kb_per_split) c.stages = c.kb_per_split;
  if (c.stages > kMaxClusterStages) c.stages = kMaxClusterStages;
  if (c.stages < 1) return c;
  const size_t exchange = exchange_bytes(c.BN, c.S);
  const size_t bytes = (size_t)c.stages * c.stage_bytes;
  c.smem = (bytes > exchange ? bytes : exchange) + 1024;
  c.tmem_cols = 32;
  while (c.tmem_cols < (uint32_t)(nacc * c.BN)) c.tmem_cols <<= 1;
  c.ok = true;
  return c;
}

template <int NAX, int NBW, int KIND>
int launch_cg(const CUtensorMap* maps, const CgParams& p, int grid, size_t smem, cudaStream_t stream) {
  // (per device ordinal: the largest dynamic shared-memory size the kernel has been allowed)
  constexpr int kMaxDevices = 64;
  static std::atomic<size_t> attr_size[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return ADAPTION_ERR_CUDA;
  const bool cached = dev >= 0 && dev < kMaxDevices;
  if (!cached || smem > attr_size[dev].load(std::memory_order_acquire)) {
    const cudaError_t ae = cudaFuncSetAttribute(lp_cluster_kernel<NAX, NBW, KIND>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ae != cudaSuccess) return cuda_failure(ae, "lp_cluster_kernel shared-memory attribute");
    if (cached) {
      size_t seen = attr_size[dev].load(std::memory_order_relaxed);
      while (seen < smem && !attr_size[dev].compare_exchange_weak(seen, smem, std::memory_order_release)) {
      }
    }
  }
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(kClusterThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  unsigned n_attr = 0;
  if (p.S > 1) {
    attr[n_attr].id = cudaLaunchAttributeClusterDimension;
    attr[n_attr].val.clusterDim.x = (unsigned)p.S;
    attr[n_attr].val.clusterDim.y = 1;
    attr[n_attr].val.clusterDim.z = 1;
    ++n_attr;
  }
  if (pdl_enabled()) {
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
    ++n_attr;
  }
  cfg.attrs = n_attr ? attr : nullptr;
  cfg.numAttrs = n_attr;
  count_launch();
  const cudaError_t le = cudaLaunchKernelEx(&cfg, lp_cluster_kernel<NAX, NBW, KIND>, maps[0], maps[1], maps[2], maps[3], p);
  if (le != cudaSuccess) {
    (void)cudaGetLastError();
    return cuda_failure(le, "lp_cluster_kernel launch");
  }
  return ADAPTION_OK;
}

template <int NAX, int NBW>
int launch_kind(const CUtensorMap* maps, const CgParams& p, int grid, size_t smem, cudaStream_t stream) {
  if (p.mode == ADAPTION_MODE_RANGE) return launch_cg<NAX, NBW, kFinishRange>(maps, p, grid, smem, stream);
  if (p.st.enabled) return launch_cg<NAX, NBW, kFinishStochastic>(maps, p, grid, smem, stream);
  return launch_cg<NAX, NBW, kFinishRound>(maps, p, grid, smem, stream);
}

}  // namespace

// Whether this layer runs here rather than on the persistent kernel.
bool cluster_path_preferred(const GemmProblem& g) {
  const int mode = knob(kCluster);
  // (pair maxima are stored by the persistent kernel alone; a plan with planes of half the rows has chosen it)
  if (mode == 0 || g.pool_w || g.box_pool) return false;
  // an override of the persistent kernel's tiles asks for that kernel
  for (Knob k : {kSplits, kPair, kFast, kStaged, kStages, kBK, kBN, kKps, kBres, kWide, kEpiGroups, kSplitHh, kStagger,
                 kStageBufs})
    if (knob(k) != kKnobDefaults[k]) return false;
  const CgPlan c = make_plan(g, g.pool2x2);
  if (!c.ok) return false;
  if (mode == 2) return true;
  // (a convolution over less than 4 KiB has too few outputs and terms to gain anything over the plain kernel)
  if (g.is_conv && (int64_t)g.cs.N * g.cs.H * g.cs.W * g.x.c_stride < 4096) return false;
  // Where the persistent kernel would have to split the reduction, or cannot run, this one is ahead
  // (16-bit, one image, us: 28x28x512->512 20.5 against 25.5, 14x14x512->512 12 against 5300 on the plain
  // kernel; inner products 4096->4096 on 1 row 8.5 against 15.5, on 64 rows 12.8 against 19.5).  With an
  // unsplit reduction on enough tiles the persistent kernel is (56x56x128->256 12.9 against 17.1).
  bool split = false;
  const int tiles = tensor_path_tiles(g, &split);
  if (tiles > 0 && !split && tiles > num_sms() / (g.is_conv ? 4 : 2)) return false;
  return (long long)c.tiles_r * c.tiles_c * c.S <= 2 * num_sms();
}

int launch_cluster(const GemmProblem& g) {
  if (g.pool_w) return ADAPTION_ERR_UNSUPPORTED;
  const CgPlan c = make_plan(g, g.pool2x2);
  if (!c.ok) return ADAPTION_ERR_UNSUPPORTED;
  note_layer(-1, 0, 0, 0);
  if (!load_tensor_map_encoders()) return ADAPTION_ERR_CUDA;
  const CUtensorMapSwizzle swz = c.BK == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                             : (c.BK == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
  const bool x2 = g.x.fmt.n_bits > 8, w2 = g.w.fmt.n_bits > 8;
  const void* xp[2] = {x2 ? g.x.hi : g.x.lo, g.x.lo};
  const void* wp[2] = {w2 ? g.w.hi : g.w.lo, g.w.lo};
  CUtensorMap maps[4];
  std::memset(maps, 0, sizeof(maps));
  for (int i = 0; i < 2; ++i) {
    bool ok = true;
    if (g.is_conv) {
      const uint64_t cs = (uint64_t)g.x.c_stride;
      if (i == 0 || x2) {
        const uint64_t dims[4] = {cs, (uint64_t)g.cs.W, (uint64_t)g.cs.H, (uint64_t)g.cs.N};
        const uint64_t strides[3] = {cs, cs * g.cs.W, cs * g.cs.W * g.cs.H};
        const uint32_t box[4] = {(uint32_t)c.BK, (uint32_t)((c.bw - 1) * g.cs.stride_w + 1),
                                 (uint32_t)((c.bh - 1) * g.cs.stride_h + 1), (uint32_t)c.bn};
        const uint32_t estr[4] = {1u, (uint32_t)g.cs.stride_w, (uint32_t)g.cs.stride_h, 1u};
        ok = encode_tiled(&maps[i], xp[i], 4, dims, strides, box, estr, swz);
      }
      if (ok && (i == 0 || w2)) {
        const uint64_t taps = (uint64_t)g.cs.R * g.cs.S;
        const uint64_t dims[3] = {cs, taps, (uint64_t)g.N};
        const uint64_t strides[2] = {cs, cs * taps};
        const uint32_t box[3] = {(uint32_t)c.BK, 1u, (uint32_t)c.BN};
        ok = encode_tiled(&maps[2 + i], wp[i], 3, dims, strides, box, nullptr, swz);
      }
    } else {
      if (i == 0 || w2)
        ok = encode_tiled_2d(&maps[i], wp[i], (uint64_t)g.K, (uint64_t)g.N, (uint64_t)g.w.c_stride, (uint32_t)c.BK,
                             (uint32_t)kRows, swz, true);
      if (ok && (i == 0 || x2))
        ok = encode_tiled_2d(&maps[2 + i], xp[i], (uint64_t)g.K, (uint64_t)g.M, (uint64_t)g.x.c_stride, (uint32_t)c.BK,
                             (uint32_t)c.BN, swz);
    }
    if (!ok) return ADAPTION_ERR_CUDA;
  }
  CgParams p;
  std::memset(&p, 0, sizeof(p));
  p.M = (int)g.M; p.N = (int)g.N; p.S = c.S; p.tiles_c = c.tiles_c;
  p.BN = c.BN; p.BK = c.BK; p.num_kb = c.num_kb; p.kb_per_split = c.kb_per_split;
  p.ksteps = c.ksteps; p.ksteps_last = c.ksteps_last;
  p.sbo = (uint32_t)(8 * c.BK);
  p.layout_type = c.BK == 128 ? 2u : (c.BK == 64 ? 4u : 6u);
  p.stages = c.stages; p.a_bytes = c.a_bytes; p.b_bytes = c.b_bytes; p.stage_bytes = c.stage_bytes;
  p.tmem_cols = c.tmem_cols;
  p.is_conv = g.is_conv ? 1 : 0;
  p.a_tx = c.a_bytes;
  if (g.is_conv) {
    p.a_tx = (uint32_t)(c.bw * c.bh * c.bn * c.BK);
    p.cblks = c.cblks; p.S_w = g.cs.S;
    p.stride_h = g.cs.stride_h; p.stride_w = g.cs.stride_w; p.pad_h = g.cs.pad_h; p.pad_w = g.cs.pad_w;
    p.OH = g.OH; p.OW = g.OW; p.images = g.cs.N;
    p.bw = c.bw; p.bh = c.bh; p.bn = c.bn; p.tiles_w = c.tiles_w; p.tiles_h = c.tiles_h;
  }
  p.pool = g.pool2x2 ? 1 : 0;
  p.bias = g.bias; p.bias_shift = g.bias_shift;
  p.mode = g.mode; p.st = g.stochastic; p.stats = g.stats;
  if (g.mode == ADAPTION_MODE_REQUANT) {
    p.rq = make_requant(g.acc_frac_bits, g.y.fmt, g.relu);
    p.y_hi = (int8_t*)g.y.hi; p.y_lo = (uint8_t*)g.y.lo; p.y_q16 = g.y.q16; p.y_stride = g.y.c_stride;
    // (columns are counted in 32 bits, and at most 2^20 are outputs: padding further out than 2^30 is not zeroed)
    p.y_cols = (int)(g.y.c_stride < (1 << 30) ? g.y.c_stride : 1 << 30);
  } else {
    p.rq = RequantParams{0, g.relu ? 1 : 0, 0, 0, 1};
    p.st.enabled = 0;
    p.y_cols = (int)g.N;
  }
  p.timeout_ns = wait_limit_ns();
  p.stall_at = knob(kStallAt);
  const int grid = c.tiles_r * c.tiles_c * c.S;
  if (c.nax == 2 && c.nbw == 2) return launch_kind<2, 2>(maps, p, grid, c.smem, g.stream);
  if (c.nax == 2) return launch_kind<2, 1>(maps, p, grid, c.smem, g.stream);
  if (c.nbw == 2) return launch_kind<1, 2>(maps, p, grid, c.smem, g.stream);
  return launch_kind<1, 1>(maps, p, grid, c.smem, g.stream);
}

}  // namespace adaption

#ifdef ADAPTION_TIMELINE
extern "C" __attribute__((visibility("default"))) int adaption_debug_cluster_timeline(long long* h_out) {
  return cudaMemcpyFromSymbol(h_out, adaption::g_cg_timeline, sizeof(long long) * 64) == cudaSuccess ? 0 : 6;
}
#endif
