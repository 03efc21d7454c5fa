// The quantizer (paper Sec. 2; LPAct with an fp32 input is the same with the ReLU flag), for one tensor or
// for all parameters of a network in one launch (Sec. 2.1: they are quantized anew in every forward pass),
// with deterministic (nearest, ties away from zero) or stochastic rounding (Sec. 2.4).
//
// One kernel walks chunks of one or several tensors; per element it reads 4 bytes and writes 1 or 2, so
// it has to stay below about ten integer instructions per element to be bound by HBM:
//   - outputs are handled as pairs of 16-bit lanes (saturating pack, clamp, zero count on packed bytes), and
//     saturations are only detected on the way and recounted where one occurred;
//   - the generator of the stochastic rounding (one Philox4x32-10 block per four elements) costs ten integer
//     instructions per element, so the rounding itself is single-precision arithmetic with one conversion.
// Dense tensors (pitch == row length) are flat arrays: eight consecutive elements per thread and step.  With
// channel padding a thread makes one 16-byte vector per plane; with a generator it quantizes the aligned blocks
// of four that cover its up to sixteen elements and shifts the bytes into place, or, in large tensors, the lanes of
// a warp share the blocks of several rows and assemble the vectors from shared memory.
//
// Measured (16 bits; before: integer arithmetic on unpacked values, as many blocks as fit walking the tensor
// together): 268 M dense elements 275 -> 239 us (6.74 TB/s), 51 M with ReLU 55.6 -> 48.5; stochastic 558 -> 332 us
// (4.9 TB/s; 385 before the rounding below took five instructions); the parameters of VGG16 157 -> 132 us, stochastic 359 -> 249 (56 M of 2-D weights 97 -> 84 since); 3.2 M pixels
// of 3 channels 27.5 -> 28.4, stochastic 89.5 -> 38; 150001 rows of 50 in a pitch of 64 12.8 -> 12.5, stochastic
// 40 -> 19.2 (rows assembled in shared memory by a whole block took 18.5 and 27).
#include "common.cuh"

namespace adaption {

int num_sms();

namespace {

constexpr int kQThreads = 256;
constexpr int kBatchItems = 40;
constexpr int kFlatBytes = 1024;            // one plane of the rows a warp assembles at a time
// Blocks per SM.  More than fit at a time: blocks then start in address order as others end, which the memory
// system rewards (268 M dense elements, 16 bits: 236 us with 32 blocks of three chunks' worth per SM, 299 us with
// the 6 that fit walking the tensor together).
constexpr int kBlocksPerSm = 32;

struct QuantItem {
  const float* x;
  uint8_t* hi;
  uint8_t* lo;
  int16_t* q16;
  const adaption_qfmt* d_fmt;
  unsigned long long first_chunk;           // chunks of the items before it
  unsigned long long count;                 // dense: groups of eight elements; padded: 16-byte vectors
  unsigned long long numel;
  long long inner;
  uint32_t row_vecs, inv_vecs;              // padded: vectors per row, ceil(2^32 / row_vecs)
  int32_t warp_rows;                        // rows a warp assembles at a time; 0: one vector per thread
  int32_t aligned;                          // x on a boundary of 16 (1) or 32 bytes (2)
  int32_t frac_bits, qmin, qmax, planes;
  uint32_t key0, key1;
};

template <int CAP>
struct QuantArgs {
  QuantItem item[CAP];
  unsigned long long total_chunks;
  adaption_stats* stats;
  int32_t n, relu, chunk;                   // chunk: groups or vectors per chunk
};

struct QuantRule {
  float scale, y_max;                       // y_max: qmax
  int32_t qmin, qmax, relu, counted;
  uint32_t qmin2, qmax2;                    // both lanes
  uint32_t key0, key1;
};

__device__ __forceinline__ uint32_t pack_sat2(int32_t lo, int32_t hi) {
  uint32_t d;
  asm("cvt.pack.sat.s16.s32 %0, %1, %2;" : "=r"(d) : "r"(hi), "r"(lo));
  return d;
}
__device__ __forceinline__ uint32_t vmax2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.s16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t vmin2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("min.s16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// Nearest integer, ties away from zero: trunc(y + copysign(1/2, y)) with the sum rounded toward zero, which
// cannot reach an integer the exact sum does not reach.  The conversion saturates and maps NaN to 0.
__device__ __forceinline__ int32_t round_away(float y) {
  const float h = __int_as_float((__float_as_int(y) & 0x80000000) | 0x3f000000);
  return __float2int_rz(__fadd_rz(y, h));
}

// Stochastic rounding of y, |y| <= 2^15 + 2: floor(y) + 1 iff draw < T, T = floor(frac(y) 2^32), without a branch.
// With d = (draw + 1) 2^-32 the value goes up iff frac(y) >= d, so the result is floor(y - d) + 1, or, the same number,
// floor(y + (1 - d)).  ~draw as a signed integer is -(draw + 1) where d <= 1/2 and 2^32 - (draw + 1) above, one of the
// two summands in units of 2^-32, at most 1/2 in magnitude; it is converted with rounding down, and so is the sum (a
// rounded-down sum has the floor of the exact one).  Rounding the summand changes no decision:
//   d <= 1/2: frac(y) >= d is asked with d rounded up.  frac(y) is a float wherever that can matter (y > 0 or y <= -1/2:
//     a multiple of the last place of y, below 1; for -1/2 < y < 0 it is above 1/2, and rounded d is not).
//   d > 1/2: 1 - frac(y) <= 1 - d is asked with 1 - d rounded down.  1 - frac(y) is a float (y < 0 or y >= 1/2), or above
//     1/2 and so above 1 - d.
// Five instructions a value; bringing frac(y) and the draw to one scale and comparing them took eight where a test of
// all four values allowed it and fourteen elsewhere.  The result is the low half of the returned word (the sum carries
// 1.5 * 2^23).
__device__ __forceinline__ uint32_t round_stochastic(float y, uint32_t draw) {
  const int32_t k = (int32_t)~draw;
  const float m = __fadd_rd(__fmaf_rd(__int2float_rd(k), 2.3283064365386963e-10f, y), 12582912.0f);
  return __float_as_uint(m) + ((uint32_t)k >> 31);
}
// largest of three magnitudes; NaN if one of them is
__device__ __forceinline__ float max_abs_nan(float a, float b, float c) {
  float d;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Four consecutive elements -> two words of two 16-bit lanes.  Elements that are not there are passed as 0
// and left out by the caller's count of real ones.
template <bool STOCH>
__device__ __forceinline__ void quantize4(const float4 v, const QuantRule& r, uint32_t block, uint32_t block_hi, int real,
                                          Counts& c, uint32_t& w0, uint32_t& w1) {
  const float x[4] = {v.x, v.y, v.z, v.w};
  if constexpr (STOCH) {
    const Philox4 rnd = philox4x32_10(block, block_hi, 0u, 0u, r.key0, r.key1);
    float y[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      y[k] = x[k] * r.scale;
      if (r.relu) y[k] = fmaxf(y[k], 0.0f);                // (NaN -> 0)
    }
    const float top = max_abs_nan(max_abs_nan(y[0], y[1], y[2]), y[3], 0.0f);
    uint32_t m[4];
    if (top <= r.y_max) {
#pragma unroll
      for (int k = 0; k < 4; ++k) m[k] = round_stochastic(y[k], rnd.w[k]);
    } else {                                               // something may saturate, or is no number
      const float y_lo = (float)r.qmin - 2.0f, y_hi = r.y_max + 2.0f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float yk = y[k] != y[k] ? 0.0f : fminf(fmaxf(y[k], y_lo), y_hi);
        const int32_t e = (int32_t)round_stochastic(yk, rnd.w[k]) - 0x4B400000;
        m[k] = (uint32_t)min(max(e, r.qmin), r.qmax);
        c.sat_pos += e > r.qmax;
        c.sat_neg += e < r.qmin;
      }
    }
    w0 = __byte_perm(m[0], m[1], 0x5410);
    w1 = __byte_perm(m[2], m[3], 0x5410);
  } else {
    int32_t q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = round_away(x[k] * r.scale);
    w0 = pack_sat2(q[0], q[1]);
    w1 = pack_sat2(q[2], q[3]);
    if (r.relu) {
      w0 = vmax2(w0, 0u);
      w1 = vmax2(w1, 0u);
    }
    bool rare;
    if (r.qmax == 32767) {
      // a lane at a bound of the 16-bit range may have been clipped
      const uint32_t top = vmax2(w0, w1), bot = vmin2(w0, w1);
      rare = (int16_t)(top & 0xffffu) == 32767 || (int16_t)(top >> 16) == 32767 || (int16_t)(bot & 0xffffu) == -32768 ||
             (int16_t)(bot >> 16) == -32768;
    } else {
      const uint32_t c0 = vmin2(vmax2(w0, r.qmin2), r.qmax2), c1 = vmin2(vmax2(w1, r.qmin2), r.qmax2);
      rare = ((c0 ^ w0) | (c1 ^ w1)) != 0u;
      w0 = c0;
      w1 = c1;
    }
    if (rare) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int32_t e = r.relu ? max(q[k], 0) : q[k];
        c.sat_pos += e > r.qmax;
        c.sat_neg += e < r.qmin;
      }
    }
  }
  // zero lanes, counted as bits (parameters are quantized without counters)
  if (!STOCH || r.counted) {
    const uint32_t nz = __vcmpne2(w0, 0u), nz1 = __vcmpne2(w1, 0u);
    c.zeros += (uint32_t)(real - __popc((nz & 0x00010001u) | (nz1 & 0x00020002u)));
  }
}

__device__ __forceinline__ uint32_t low_bytes(uint32_t w0, uint32_t w1) { return __byte_perm(w0, w1, 0x6420); }
__device__ __forceinline__ uint32_t high_bytes(uint32_t w0, uint32_t w1) { return __byte_perm(w0, w1, 0x7531); }

// eight consecutive elements, in one load where they lie on a 32-byte boundary
__device__ __forceinline__ void load8(const float* p, bool aligned32, float4 (&v)[2]) {
  if (aligned32) {
    asm volatile("ld.global.cs.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[0].z), "=f"(v[0].w), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[1].z),
                   "=f"(v[1].w)
                 : "l"(p));
  } else {
    v[0] = __ldcs(reinterpret_cast<const float4*>(p));
    v[1] = __ldcs(reinterpret_cast<const float4*>(p) + 1);
  }
}

__device__ __forceinline__ QuantRule rule_of(const QuantItem& it, int relu, bool counted) {
  QuantRule r;
  const int32_t f = it.d_fmt != nullptr ? it.d_fmt->frac_bits : it.frac_bits;
  r.scale = __int_as_float((127 + f) << 23);
  r.y_max = (float)it.qmax;
  r.qmin = it.qmin;
  r.qmax = it.qmax;
  r.relu = relu;
  r.counted = counted;
  r.qmin2 = (uint32_t)(it.qmin & 0xffff) * 0x00010001u;
  r.qmax2 = (uint32_t)it.qmax * 0x00010001u;
  r.key0 = it.key0;
  r.key1 = it.key1;
  return r;
}

// Eight consecutive elements of a dense tensor per thread and step, two steps in flight.
template <bool STOCH>
__device__ __forceinline__ void quantize_dense_chunk(const QuantItem& it, const QuantRule& rule, unsigned long long base,
                                                     unsigned chunk, Counts& c) {
  const unsigned long long end = min(it.count, base + chunk);
  // (chunks are powers of two: a chunk's generator blocks share the high word, and the first two rounds' work on it)
  const uint32_t block_hi = (uint32_t)(base >> 31);
  float4 v[2][2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const unsigned long long i = base + u * kQThreads + threadIdx.x;
    if (i < end) load8(it.x + 8 * i, it.aligned == 2, v[u]);
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const unsigned long long i = base + u * kQThreads + threadIdx.x;
    if (i < end) {
      uint32_t w[4];
      quantize4<STOCH>(v[u][0], rule, (uint32_t)(2 * i), block_hi, 4, c, w[0], w[1]);
      quantize4<STOCH>(v[u][1], rule, (uint32_t)(2 * i) + 1u, block_hi, 4, c, w[2], w[3]);
      // (streaming stores: the planes are read much later)
      __stcs(reinterpret_cast<uint2*>(it.lo) + i, make_uint2(low_bytes(w[0], w[1]), low_bytes(w[2], w[3])));
      if (it.planes == 2)
        __stcs(reinterpret_cast<uint2*>(it.hi) + i, make_uint2(high_bytes(w[0], w[1]), high_bytes(w[2], w[3])));
      if (it.q16 != nullptr) reinterpret_cast<uint4*>(it.q16)[i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

__device__ __forceinline__ void load_block(const QuantItem& it, unsigned long long i, float4& v) {
  v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (it.aligned && i + 4 <= it.numel) {
    v = __ldg(reinterpret_cast<const float4*>(it.x + i));
  } else {
    if (i < it.numel) v.x = __ldg(it.x + i);
    if (i + 1 < it.numel) v.y = __ldg(it.x + i + 1);
    if (i + 2 < it.numel) v.z = __ldg(it.x + i + 2);
    if (i + 3 < it.numel) v.w = __ldg(it.x + i + 3);
  }
}

// Rows of at most four elements in a pitch of sixteen (the pixels of an input image): the blocks of four that
// four consecutive rows consist of are quantized by the first `inner` of four neighbouring lanes, and
// every lane shuffles its own row's bytes together.  (One generator block per row instead of two.)
template <bool STOCH>
__device__ __forceinline__ void quantize_narrow_rows(const QuantItem& it, const QuantRule& rule, unsigned long long g,
                                                     bool mine, Counts& c) {
  const int sub = threadIdx.x & 3, first = threadIdx.x & 28, inner = (int)it.inner;
  uint32_t w0 = 0u, w1 = 0u;
  const unsigned long long block = (g >> 2) * (unsigned)inner + (unsigned)sub, i = block << 2;
  if (sub < inner && i < it.numel) {
    float4 v;
    load_block(it, i, v);
    quantize4<STOCH>(v, rule, (uint32_t)block, (uint32_t)(block >> 32), (int)min(4ull, it.numel - i), c, w0, w1);
  }
  const uint32_t l = low_bytes(w0, w1), h = high_bytes(w0, w1);
  const int at = inner * sub;                         // place of this row's first byte among the 4 * inner
  const int from = first + (at >> 2), next = first + min((at >> 2) + 1, 3);
  const uint32_t sh = 8u * (uint32_t)(at & 3), keep = 0xffffffffu >> (32 - 8 * inner);
  const uint32_t l0 = __shfl_sync(0xffffffffu, l, from), l1 = __shfl_sync(0xffffffffu, l, next);
  const uint32_t h0 = __shfl_sync(0xffffffffu, h, from), h1 = __shfl_sync(0xffffffffu, h, next);
  if (mine) {
    reinterpret_cast<uint4*>(it.lo)[g] = make_uint4(__funnelshift_r(l0, l1, sh) & keep, 0u, 0u, 0u);
    if (it.planes == 2) reinterpret_cast<uint4*>(it.hi)[g] = make_uint4(__funnelshift_r(h0, h1, sh) & keep, 0u, 0u, 0u);
  }
  if (it.q16 != nullptr) {
    // the same on 16-bit lanes: word k of the string is w0 (even k) or w1 of lane k / 2
    uint32_t word[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int k = min((at >> 1) + j, 7);
      const uint32_t a = __shfl_sync(0xffffffffu, w0, first + (k >> 1)), b = __shfl_sync(0xffffffffu, w1, first + (k >> 1));
      word[j] = (k & 1) ? b : a;
    }
    const uint32_t half = 16u * (uint32_t)(at & 1);
    uint32_t o0 = __funnelshift_r(word[0], word[1], half), o1 = __funnelshift_r(word[1], word[2], half);
    o0 = inner == 1 ? o0 & 0xffffu : o0;
    o1 = inner <= 2 ? 0u : (inner == 3 ? o1 & 0xffffu : o1);
    if (mine) {
      uint4* d = reinterpret_cast<uint4*>(it.q16) + 2 * g;
      d[0] = make_uint4(o0, o1, 0u, 0u);
      d[1] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
}

// sixteen bytes from byte `at` on, the first `real` of them, zeros behind
__device__ __forceinline__ uint4 unaligned16(const uint32_t* words, int at, int real) {
  const uint32_t* w = words + (at >> 2);
  const uint32_t sh = 8u * (uint32_t)(at & 3);
  uint32_t in[5], o[4];
#pragma unroll
  for (int j = 0; j < 5; ++j) in[j] = w[j];               // (the buffer has room for a word behind its end)
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int k = min(max(real - 4 * j, 0), 4);
    o[j] = __funnelshift_r(in[j], in[j + 1], sh);
    if (k < 4) o[j] &= (1u << (8 * k)) - 1u;
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// `warp_rows` rows (a multiple of four, so they start on a block boundary) per warp: the lanes quantize the rows'
// blocks of four in input order, no element twice, and leave the bytes densely in shared memory; then each
// lane picks up whole vectors of the padded rows from there.
template <bool STOCH>
__device__ __forceinline__ void quantize_rows_by_warp(const QuantItem& it, const QuantRule& rule, unsigned long long group,
                                                      uint8_t* flat, Counts& c) {
  const int lane = threadIdx.x & 31;
  const unsigned long long row0 = group * (unsigned)it.warp_rows, outer = it.count;
  if (row0 >= outer) return;
  const int rows = (int)min((unsigned long long)it.warp_rows, outer - row0);
  const int inner = (int)it.inner, n = rows * inner;                    // at most kFlatBytes
  const unsigned long long f0 = row0 * (unsigned)inner;                 // a multiple of four
  uint32_t* const flat_lo = reinterpret_cast<uint32_t*>(flat);
  uint32_t* const flat_hi = reinterpret_cast<uint32_t*>(flat + kFlatBytes + 16);
  __syncwarp();                                                         // (the previous rows have been picked up)
  const int blocks = (n + 3) / 4;
  constexpr int kAhead = 2;                                             // loads in flight per lane
  for (int first = lane; first < blocks; first += 32 * kAhead) {
    float4 v[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (first + 32 * u < blocks) load_block(it, f0 + 4u * (unsigned)(first + 32 * u), v[u]);
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int b = first + 32 * u;
      if (b < blocks) {
        uint32_t w0, w1;
        const unsigned long long blk = (f0 >> 2) + (unsigned)b;
        quantize4<STOCH>(v[u], rule, (uint32_t)blk, (uint32_t)(blk >> 32), min(4, n - 4 * b), c, w0, w1);
        flat_lo[b] = low_bytes(w0, w1);
        if (it.planes == 2) flat_hi[b] = high_bytes(w0, w1);
      }
    }
  }
  __syncwarp();
  const int vecs = rows * (int)it.row_vecs;
  uint4* const out_lo = reinterpret_cast<uint4*>(it.lo) + row0 * it.row_vecs;
  uint4* const out_hi = reinterpret_cast<uint4*>(it.hi) + row0 * it.row_vecs;
  for (int i = lane; i < vecs; i += 32) {
    const int row = it.row_vecs == 1 ? i : (int)__umulhi((uint32_t)i, it.inv_vecs);
    const int c0 = 16 * (i - row * (int)it.row_vecs), real = min(16, max(0, inner - c0));
    uint4 l = make_uint4(0u, 0u, 0u, 0u), h = l;
    if (real > 0) {
      const int at = row * inner + c0;
      l = unaligned16(flat_lo, at, real);
      if (it.planes == 2) h = unaligned16(flat_hi, at, real);
    }
    __stcs(out_lo + i, l);
    if (it.planes == 2) __stcs(out_hi + i, h);
  }
}

// One 16-byte vector of a padded row per thread.
template <bool STOCH>
__device__ __forceinline__ void quantize_padded_chunk(const QuantItem& it, const QuantRule& rule, unsigned long long base,
                                                      unsigned chunk, uint8_t* flat, Counts& c) {
  if (STOCH && it.warp_rows > 0) {
    // (a chunk stands for one run of rows per warp)
    quantize_rows_by_warp<STOCH>(it, rule, base / chunk * (kQThreads / 32) + (threadIdx.x >> 5), flat, c);
    return;
  }
  const unsigned long long g = base + threadIdx.x;
  if (it.row_vecs == 1 && it.inner <= 4) {
    quantize_narrow_rows<STOCH>(it, rule, g, g < it.count, c);
    return;
  }
  if (g >= it.count) return;
  const unsigned long long row = it.count <= 0xffffffffull ? (unsigned long long)((uint32_t)g / it.row_vecs) : g / it.row_vecs;
  const long long c0 = (long long)(g - row * it.row_vecs) * 16;
  const int real = (int)min(16ll, max(0ll, it.inner - c0));               // real elements of this vector
  const unsigned long long i0 = row * (unsigned long long)it.inner + (unsigned long long)c0;
  const int off = (int)(i0 & 3ull);                                        // place of the first one in its block
  const unsigned long long b0 = i0 >> 2;
  if constexpr (!STOCH) {
    // no generator, so no blocks: groups of four from the vector's own first element
    uint32_t wl[4], wh[4], wq[8];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      wl[t] = wh[t] = wq[2 * t] = wq[2 * t + 1] = 0u;
      if (4 * t < real) {
        const float* __restrict__ src = it.x + i0 + 4 * t;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        v.x = __ldg(src);
        if (4 * t + 1 < real) v.y = __ldg(src + 1);
        if (4 * t + 2 < real) v.z = __ldg(src + 2);
        if (4 * t + 3 < real) v.w = __ldg(src + 3);
        quantize4<false>(v, rule, 0u, 0u, min(4, real - 4 * t), c, wq[2 * t], wq[2 * t + 1]);
        wl[t] = low_bytes(wq[2 * t], wq[2 * t + 1]);
        wh[t] = high_bytes(wq[2 * t], wq[2 * t + 1]);
      }
    }
    reinterpret_cast<uint4*>(it.lo)[g] = make_uint4(wl[0], wl[1], wl[2], wl[3]);
    if (it.planes == 2) reinterpret_cast<uint4*>(it.hi)[g] = make_uint4(wh[0], wh[1], wh[2], wh[3]);
    if (it.q16 != nullptr) {
      uint4* d = reinterpret_cast<uint4*>(it.q16) + 2 * g;
      d[0] = make_uint4(wq[0], wq[1], wq[2], wq[3]);
      d[1] = make_uint4(wq[4], wq[5], wq[6], wq[7]);
    }
    return;
  }
  const int blocks = real > 0 ? (off + real + 3) / 4 : 0;                  // at most five
  float4 v[5];
#pragma unroll
  for (int t = 0; t < 5; ++t) {
    v[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t < blocks) load_block(it, (b0 + (unsigned)t) << 2, v[t]);
  }
  uint32_t wl[6], wh[6], wq[11];
#pragma unroll
  for (int t = 0; t < 6; ++t) wl[t] = wh[t] = 0u;
#pragma unroll
  for (int t = 0; t < 11; ++t) wq[t] = 0u;
#pragma unroll
  for (int t = 0; t < 5; ++t) {
    if (t < blocks) {
      // elements before the vector's first and behind its last belong to others
      const int lo = t == 0 ? off : 0, hi = min(4, off + real - 4 * t);
      if (lo > 0) v[t].x = 0.f;
      if (lo > 1 || hi < 2) v[t].y = 0.f;
      if (lo > 2 || hi < 3) v[t].z = 0.f;
      if (hi < 4) v[t].w = 0.f;
      uint32_t w0, w1;
      quantize4<STOCH>(v[t], rule, (uint32_t)(b0 + (unsigned)t), (uint32_t)((b0 + (unsigned)t) >> 32), hi - lo, c, w0, w1);
      wl[t] = low_bytes(w0, w1);
      wh[t] = high_bytes(w0, w1);
      if (it.q16 != nullptr) {
        wq[2 * t] = w0;
        wq[2 * t + 1] = w1;
      }
    }
  }
  const uint32_t sh = 8u * (uint32_t)off;
  reinterpret_cast<uint4*>(it.lo)[g] =
      make_uint4(__funnelshift_r(wl[0], wl[1], sh), __funnelshift_r(wl[1], wl[2], sh), __funnelshift_r(wl[2], wl[3], sh),
                 __funnelshift_r(wl[3], wl[4], sh));
  if (it.planes == 2)
    reinterpret_cast<uint4*>(it.hi)[g] =
        make_uint4(__funnelshift_r(wh[0], wh[1], sh), __funnelshift_r(wh[1], wh[2], sh), __funnelshift_r(wh[2], wh[3], sh),
                   __funnelshift_r(wh[3], wh[4], sh));
  if (it.q16 != nullptr) {
    uint32_t o[8];
    const uint32_t half = 16u * (uint32_t)(off & 1);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t a = off >= 2 ? wq[j + 1] : wq[j], b = off >= 2 ? wq[j + 2] : wq[j + 1];
      o[j] = __funnelshift_r(a, b, half);
    }
    uint4* d = reinterpret_cast<uint4*>(it.q16) + 2 * g;
    d[0] = make_uint4(o[0], o[1], o[2], o[3]);
    d[1] = make_uint4(o[4], o[5], o[6], o[7]);
  }
}

// With a generator three blocks per SM for a single tensor, registers for more independent chains: 268 M elements 345 us with
// four, 331 with three; 2 to 4 % from 2 M elements on, dense or rows of 13 to 1000 in their pitch, equal below (rows of 3: 0.5 %
// slower); a batch 83.6 and 91.
template <bool STOCH, bool PADDED, int CAP>
__global__ void __launch_bounds__(kQThreads, STOCH ? (CAP == 1 ? 3 : 4) : (PADDED ? 6 : 5)) quantize_kernel(const __grid_constant__ QuantArgs<CAP> a) {
  constexpr int kFlat = 2 * (kFlatBytes + 16);
  constexpr bool kByWarp = PADDED && STOCH;
  __shared__ __align__(16) uint8_t flat[kByWarp ? kQThreads / 32 * kFlat : 16];
  uint8_t* const my_flat = kByWarp ? flat + (threadIdx.x >> 5) * kFlat : flat;
  pdl_prologue();
  Counts c;
  // Chunks come in increasing order, so the search for a chunk's tensor only moves forward.
  int t = 0;
  QuantRule rule = rule_of(a.item[0], a.relu, a.stats != nullptr);
  for (unsigned long long chunk = blockIdx.x; chunk < a.total_chunks; chunk += gridDim.x) {
    if (CAP > 1) {
      const int was = t;
      while (t + 1 < a.n && a.item[t + 1].first_chunk <= chunk) ++t;
      if (t != was) rule = rule_of(a.item[t], a.relu, a.stats != nullptr);
    }
    const QuantItem& it = a.item[t];
    const unsigned long long base = (chunk - it.first_chunk) * (unsigned)a.chunk;
    if (PADDED)
      quantize_padded_chunk<STOCH>(it, rule, base, (unsigned)a.chunk, my_flat, c);
    else
      quantize_dense_chunk<STOCH>(it, rule, base, (unsigned)a.chunk, c);
  }
  if (a.stats != nullptr) flush_counts_block(c, a.stats);
}

bool is_dense(const float* x, size_t inner, const adaption_qtensor& q) {
  return (int64_t)inner == q.c_stride && aligned16(x);
}

// Fills one item (the chunk numbering comes with the launch).
void make_item(QuantItem& it, const float* x, size_t outer, size_t inner, const adaption_qtensor& q,
               const adaption_qfmt* d_fmt, uint64_t seed) {
  it.x = x;
  it.planes = q.fmt.n_bits > 8 ? 2 : 1;
  it.hi = it.planes == 2 ? static_cast<uint8_t*>(q.hi) : nullptr;
  it.lo = static_cast<uint8_t*>(q.lo);
  it.q16 = q.q16;
  it.d_fmt = d_fmt;
  it.numel = (unsigned long long)outer * inner;
  it.inner = (long long)inner;
  it.row_vecs = (uint32_t)(q.c_stride / 16);
  it.aligned = !aligned16(x) ? 0 : ((reinterpret_cast<uintptr_t>(x) & 31u) == 0 ? 2 : 1);
  it.frac_bits = q.fmt.frac_bits;
  it.qmin = -(1 << (q.fmt.n_bits - 1));
  it.qmax = (1 << (q.fmt.n_bits - 1)) - 1;
  it.key0 = (uint32_t)seed;
  it.key1 = (uint32_t)(seed >> 32);
  it.inv_vecs = it.row_vecs > 1 ? (uint32_t)(((1ull << 32) + it.row_vecs - 1) / it.row_vecs) : 0u;
  it.warp_rows = 0;
  it.count = is_dense(x, inner, q) ? it.numel / 8 : (unsigned long long)outer * it.row_vecs;   // (pitches are multiples of 16)
}

// Padded tensors that a warp assembles several rows of at a time: with a generator (150001 rows of 50: 25.2 us with
// one vector per thread, 19.4 this way; without one 13.6 and 14.1), where four rows fit, rows do not share
// lanes (quantize_narrow_rows) and the tensor fills the chip with such runs of rows.  The vectors of a run are
// divided by row_vecs through a reciprocal whose error is below row_vecs / 2^32: exact while vectors * row_vecs < 2^32
// (one element per row: pitches up to 32 KB; 256 elements: up to 512 KB).
int rows_by_warp(const QuantItem& it, bool stochastic) {
  if (!stochastic || it.q16 != nullptr || it.inner * 4 > kFlatBytes || (it.row_vecs == 1 && it.inner <= 4) ||
      it.count < (unsigned long long)num_sms() * 1024)
    return 0;
  const int rows = (int)(kFlatBytes / it.inner) & ~3;
  const unsigned long long vecs = it.row_vecs < (1u << 16) ? (unsigned long long)rows * it.row_vecs : 1ull << 32;
  return vecs * it.row_vecs < 1ull << 32 ? rows : 0;
}

template <bool STOCH, bool PADDED, int CAP>
int launch_quantize(QuantArgs<CAP>& a, cudaStream_t stream) {
  if (a.n == 0) return ADAPTION_OK;
  a.chunk = kQThreads;
  if (!PADDED) {
    // two steps per thread, one where the problem is too small to fill the chip that way
    unsigned long long groups = 0;
    for (int k = 0; k < a.n; ++k) groups += a.item[k].count;
    if (groups >= (unsigned long long)num_sms() * 8 * kQThreads) a.chunk = 2 * kQThreads;
  }
  a.total_chunks = 0;
  for (int k = 0; k < a.n; ++k) {
    QuantItem& it = a.item[k];
    it.first_chunk = a.total_chunks;
    if (PADDED) it.warp_rows = rows_by_warp(it, STOCH);
    if (it.warp_rows > 0) {
      it.count /= it.row_vecs;
      const unsigned long long per_chunk = (unsigned long long)it.warp_rows * (kQThreads / 32);
      a.total_chunks += (it.count + per_chunk - 1) / per_chunk;
    } else {
      a.total_chunks += (it.count + (unsigned)a.chunk - 1) / (unsigned)a.chunk;
    }
  }
  // Padded rows without a generator: with few chunks per SM a block of one or two chunks costs more in its start and its
  // counters than the order gives (1 M rows, us, 32 blocks per SM and 12: of 1 element 10.0, 8.5, of 5 13.8, 12.6, of 13
  // 19.2, 18.0; 3 M rows of 13 50.9, 51.4).  Rows that share lanes gain at any size (3 M rows of 3 27.5, 27.0).
  const bool narrow = PADDED && a.n == 1 && a.item[0].row_vecs == 1 && a.item[0].inner <= 4;
  const bool few = PADDED && !STOCH && (narrow || a.total_chunks < (unsigned long long)num_sms() * 64);
  const unsigned long long cap = (unsigned long long)num_sms() * (few ? 12 : kBlocksPerSm);
  const unsigned grid = (unsigned)(a.total_chunks < cap ? a.total_chunks : cap);
  const cudaError_t e = launch_after_predecessor(quantize_kernel<STOCH, PADDED, CAP>, dim3(grid), dim3(kQThreads), stream, a);
  if (e != cudaSuccess) (void)cudaGetLastError();
  return cuda_status(e, "quantize_kernel launch");
}

int check_source(const float* d_x) {
  if (d_x == nullptr) return ADAPTION_ERR_INVALID_ARG;
  return (reinterpret_cast<uintptr_t>(d_x) & 3u) != 0 ? ADAPTION_ERR_ALIGNMENT : ADAPTION_OK;
}

template <bool STOCH>
int quantize_one(const float* d_x, size_t outer, size_t inner, const adaption_qtensor& out, const adaption_qfmt* d_fmt,
                 int32_t relu, uint64_t seed, adaption_stats* d_stats, cudaStream_t stream) {
  int rc = check_qtensor_out(out, (int64_t)inner);
  if (rc != ADAPTION_OK) return rc;
  if (outer == 0 || inner == 0) return ADAPTION_OK;
  rc = check_source(d_x);
  if (rc != ADAPTION_OK) return rc;
  QuantArgs<1> a;
  make_item(a.item[0], d_x, outer, inner, out, d_fmt, seed);
  a.n = 1;
  a.relu = relu;
  a.stats = d_stats;
  return is_dense(d_x, inner, out) ? launch_quantize<STOCH, false, 1>(a, stream) : launch_quantize<STOCH, true, 1>(a, stream);
}

template <bool STOCH>
int quantize_many(const adaption_quantize_item* h_items, const uint64_t* h_seeds, int32_t n_items, cudaStream_t stream) {
  if (n_items < 0 || (n_items > 0 && h_items == nullptr)) return ADAPTION_ERR_INVALID_ARG;
  if (STOCH && n_items > 0 && h_seeds == nullptr) return ADAPTION_ERR_INVALID_ARG;
  // validate everything before the first launch
  for (int32_t k = 0; k < n_items; ++k) {
    const adaption_quantize_item& h = h_items[k];
    if (h.outer < 0 || h.inner < 0) return ADAPTION_ERR_INVALID_ARG;
    int rc = check_qtensor_out(h.q, h.inner);
    if (rc != ADAPTION_OK) return rc;
    if (h.outer == 0 || h.inner == 0) continue;
    rc = check_source(h.d_x);
    if (rc != ADAPTION_OK) return rc;
  }
  // dense tensors in one run of launches, padded ones in another
  QuantArgs<kBatchItems> a;
  a.relu = 0;
  a.stats = nullptr;
  for (const bool dense : {true, false}) {
    a.n = 0;
    for (int32_t k = 0; k < n_items; ++k) {
      const adaption_quantize_item& h = h_items[k];
      if (h.outer == 0 || h.inner == 0 || is_dense(h.d_x, (size_t)h.inner, h.q) != dense) continue;
      make_item(a.item[a.n], h.d_x, (size_t)h.outer, (size_t)h.inner, h.q, h.d_fmt, STOCH ? h_seeds[k] : 0);
      if (++a.n == kBatchItems) {
        const int rc = dense ? launch_quantize<STOCH, false, kBatchItems>(a, stream)
                             : launch_quantize<STOCH, true, kBatchItems>(a, stream);
        if (rc != ADAPTION_OK) return rc;
        a.n = 0;
      }
    }
    const int rc = dense ? launch_quantize<STOCH, false, kBatchItems>(a, stream)
                         : launch_quantize<STOCH, true, kBatchItems>(a, stream);
    if (rc != ADAPTION_OK) return rc;
  }
  return ADAPTION_OK;
}

}  // namespace

int quantize_impl(const float* d_x, size_t outer, size_t inner, const adaption_qtensor& out,
                  const adaption_qfmt* d_fmt, int32_t relu, int32_t rounding, adaption_stats* d_stats,
                  cudaStream_t stream) {
  if (rounding == ADAPTION_ROUND_STOCHASTIC) return ADAPTION_ERR_UNSUPPORTED;
  if (rounding != ADAPTION_ROUND_DETERMINISTIC) return ADAPTION_ERR_INVALID_ARG;
  return quantize_one<false>(d_x, outer, inner, out, d_fmt, relu, 0, d_stats, stream);
}

int quantize_stochastic_impl(const float* d_x, size_t outer, size_t inner, const adaption_qtensor& out,
                             const adaption_qfmt* d_fmt, int32_t relu, uint64_t seed, adaption_stats* d_stats,
                             cudaStream_t stream) {
  return quantize_one<true>(d_x, outer, inner, out, d_fmt, relu ? 1 : 0, seed, d_stats, stream);
}

int quantize_batch_impl(const adaption_quantize_item* h_items, int32_t n_items, cudaStream_t stream) {
  return quantize_many<false>(h_items, nullptr, n_items, stream);
}

int quantize_batch_stochastic_impl(const adaption_quantize_item* h_items, const uint64_t* h_seeds, int32_t n_items,
                                   cudaStream_t stream) {
  return quantize_many<true>(h_items, h_seeds, n_items, stream);
}

}  // namespace adaption
