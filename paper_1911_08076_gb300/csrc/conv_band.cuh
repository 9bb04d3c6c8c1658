// Band path of the quantized convolution (Eq. (1) integer core with the thresholds of Eq. (7) / (8)
// fused as the epilogue): 4-bit tensor-core products on an input band that is expanded once.
//
// GEMM view: D[m][n] = sum_K A[m][K] * B[n][K], m = an anchor (output pixel),
// n = output channel, on tcgen05.mma kind::mxf4 with every block scale 1.
//
// Exact integers on the e2m1 tensor cores:
//   * a 2-bit code c in 0..3 is the e2m1 nibble c, i.e. the value c / 2, and +1 / -1 are the nibbles
//     0x2 / 0xA, so every product is a multiple of 1/2 and D = A / 2;
//   * a 3- or 4-bit code in its 4-bit field is two 2-bit digits (low digit first), so its map is a
//     2-bit map of twice the channels whose odd channels weigh +4 / -4 (nibbles 0x6 / 0xE);
//   * the fp32 accumulation was checked exact on GB300 up to |A| = 196608 with odd addends along all
//     of K = 65536, the bound the planner admits (test_accumulation_exact_at_the_admitted_bound).
// Measured rate of the instruction (M128 x N128 x K64, both operands in shared memory): 9.57 PTOPS on 152 SMs, twice
// the e4m3 rate of the im2col kernel (conv_tc.cuh).  That is 64 cycles; N = 64 takes 48 (6.31 PTOPS) and N = 32 46 (3.31),
// where reading the 4 KB of A takes longer than the products.
//
// A is the input itself.  A slot is 16 bytes: 32 consecutive 2-bit fields of one input pixel (one
// "plane" of it), expanded to nibbles by a mask and a shift.  Slots lie in shared memory in pixel
// order with `P` slots a row and `HP` rows an image (the zero padding of a row's right edge is the
// next row's left edge, and likewise between images), so the A operand of filter tap (dy, dx) for
// 128 consecutive anchors is the same band read dy * P + dx slots further on: the non-swizzled K-major
// layout has 8-row core matrices of 16 bytes a row, so consecutive anchors are consecutive slots and a
// tap is one more descriptor.  Every code is expanded once per tile instead of once per tap and channel
// tile, which is what bounded the im2col kernel.
// A strided 1 x 1 filter reads one pixel in s x s, so its band holds those alone.  (Larger strided filters
// and fused pools would need the s x s phases of the input apart and a pass per window position: they measured
// 1.1 to 1.7 times the im2col and window kernels' times and are not here.)
//
// K order: plane pairs, within a pair the taps (row-major), within a tap the two planes; an MMA
// takes the two 16-byte core columns (plane 2i, plane 2i + 1) of one tap.  An odd last plane pairs
// consecutive taps instead (a lone last tap with a zero column).  The prepared filters are laid
// out in that order, [core column][output channel][16 bytes], so a filter stage is one TMA box, in the
// core-matrix layout already.
//
// Persistent, warp-specialized CTA bound to a group of output-channel tiles (its thresholds are
// loaded once; its filters too where they fit, else they stream through a ring):
//   epilogue warps   two groups of 8 (lane quadrant = warp % 4), groups on alternate accumulators;
//   producer warps   packed codes global -> registers -> nibbles -> band ring (chunks of planes);
//   MMA warps        one elected lane issues; B warp: TMA boxes of filter stages.
// Every wait is bounded (IFQ_ETIMEOUT; the roles then leave their loops).
//
// Threshold epilogue.  The thresholds of a layer are floors of equally spaced values (Eq. (7), (8)),
// so a line g(x) separates them: g(T_i) < i - 1/2 < g(T_i + 1).  Then the code is g rounded and clamped
// to 0..L, two FMA-pipe operations (v = sat(a D + b), v L + 2^23 whose low bits are the code) and one
// shift-add to pack, where a compare per threshold takes six or more (k = 2) or a search (k = 3, 4).
// Each column's line is fitted and then checked at every T_i and T_i + 1 with those same operations
// when the CTA starts; between these the result cannot change because g is monotone in x and so is its
// rounding.  A block of 64 columns with a column whose check fails takes one of two slower forms:
//   * 3- and 4-bit codes whose thresholds are nearly equally spaced (the separated conversion's, floored one by one):
//     a line half a step lower is the code or one below it, and one comparison with the threshold that it names
//     decides;
//   * any others: three comparisons (2-bit codes) or a search of four steps.
// Measured (us; im2col kernel, then here by line, line and comparison, search): 4-bit codes 3x3 384 -> 384 on 14 x 14 x
// 256 images 64.7, 53.4, 60.7, 71.3, 1x1 128 -> 256 on 28 x 28 x 256 93.8, 26.8, 40.9, 62.9; 2-bit codes (line, three
// comparisons) 38.6, 33.3, 37.9 and 37.9, 23.5, 32.8.  A 4-ary search by compares and selects took 78.0 and 79.1 where
// the search takes 71.3 and 62.9, and spilled.  The form is one for all of a warp's channel tiles, in a loop of its own:
// chosen unit by unit the network of 16 small layers took 1 % longer.
// Every comparison is a saturating fma, sat(s A - T), of integers.  All instances fit 80 registers without spilling:
// with the comparisons beside the lines' 32 registers they spilled (and a spill may move around a tensor-memory load).
//
// Measured (us, uniform codes, launches back to back; im2col kernel, this one): 3x3 256 -> 256 on 56 x 56 x 256 images
// 270, 167 (5.7 PTOPS; 59 % of the instruction's rate); 1x1 512 -> 512 on 28 x 28 x 256 92.3, 40.6; 5x5 96 -> 256 on 27 x 27
// x 128 37.6, 23.6; 3x3 1024 -> 1024 on 13 x 13 x 64 64.8, 42.0; the same 5x5 layer with 4-bit codes 60.3, 46.5.  What
// bounds the large layers now is instruction latency beside 24 warps (issue slots 48 to 59 % busy): the MMA warps wait
// for slots that the epilogue takes.
#pragma once
#include "conv_common.cuh"

namespace ifq {

constexpr int kBandMaxTaps = 49;     // filter taps (tables in shared memory)
constexpr int kBandEpi = 16;         // epilogue warps, in two groups
constexpr int kBandProd = 5;         // producer warps
constexpr int kBandThreads = 32 * (kBandEpi + kBandProd + 1 + 2);
constexpr int kBandCols = 512;       // tensor-memory columns: accumulators, then 16 of unit scales
constexpr int kBandBlock = 64;       // output channels whose filter rows are permuted together

// MMAs of an odd last plane: pairs of consecutive taps.
__host__ __device__ inline int band_odd_steps(int taps) { return (taps + 1) / 2; }

// Output channel of accumulator column c (filter row c).  Within a block of 64 columns the order is such that
// the fragment of a thread of quad position q, columns 8 k + 2 q + e, holds 16 consecutive channels: one word of
// 2-bit codes, with no exchange.
__host__ __device__ inline int band_channel(int c) {
  const int p = c & (kBandBlock - 1);
  return c - p + (kBandBlock / 4) * ((p >> 1) & 3) + 2 * (p >> 3) + (p & 1);
}

struct BandArgs {
  const uint8_t* x;        // packed input codes, NHWC
  const int32_t* thr;      // [cout][lvl]
  const int8_t* sign;      // [cout]
  uint8_t* y_codes;        // packed output codes or nullptr
  int32_t* y_acc;          // int32 accumulators or nullptr
  int n, h, w, pb;         // input map, packed bytes per pixel
  int cout, lvl;           // output channels, thresholds per channel
  int bound;               // largest magnitude of an accumulator
  int oh, ow;              // anchors of an image: the output map
  int P, HP;               // slots per row, rows per image
  int pad, kh, kw, s;      // s: stride (1 but for 1 x 1 filters)
  int slots;               // slots of one plane of a chunk
  int planes, cp, nchunk;  // planes per pixel, planes per chunk, chunks
  int linear;              // 1: slot f is input pixel f (1 x 1, stride 1, no padding)
  int gran, glg;           // bytes per load (16: two planes; 8, 4, 2, 1: one plane); log2 of the granule lanes
  int taps, nodd;          // filter taps; MMAs of the odd plane
  int nstep;               // MMAs (K = 64) per pass
  int tab_last, ntab;      // table entries before the last chunk's, and in all
  int ring;                // chunk buffers
  int nst, stages;         // filter stages (four MMAs of a chunk) per channel tile, stages in shared memory
  int resident;            // 1: every stage of the CTA's channel tiles has its own buffer, loaded once
  int ngrp, ngroups, nt;   // channel tiles per CTA, groups of them, channel tiles
  int mt, mtiles;          // 128-anchor subtiles per tile, tiles
  int nacc, ncb;           // accumulator buffers; barrier pairs that their uses take in turn.  ncb is
                           // even, so an epilogue group meets each of its barriers' phases in
                           // order
  uint32_t plane_bytes, chunk_bytes, stage_bytes;
  uint32_t off_b, off_lin, off_thr, off_bad, off_tab, off_bar;
  int early;               // 1: no kernel before this one in the stream writes the filters or thresholds
  FastDiv div_P, div_HP;
};

// D[128][N] (+)= A . B, 4-bit operands in shared memory, unit scales at `sf` for both.
__device__ __forceinline__ void mma_mxf4(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t sf, uint32_t acc) {
  asm volatile(
      "{.reg .pred p; setp.ne.b32 p, %5, 0;"
      " tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%4], [%4], p;}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(sf), "r"(acc));
}
// Instruction descriptor, kind::mxf4: e2m1 x e2m1, ue8m0 scales, both operands K-major.
__host__ __device__ constexpr uint32_t idesc_mxf4(int M, int N) {
  return (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | (1u << 23) | ((uint32_t)(M >> 4) << 24);
}
// Descriptor of a non-swizzled K-major operand at `addr16` (16-byte units): 8-row core matrices 128
// bytes apart along M / N, `lbo16` 16-byte units apart along K.
__device__ __forceinline__ uint64_t band_desc(uint32_t addr16, uint32_t lbo16) {
  return (uint64_t)(addr16 & 0x3FFFu) | ((uint64_t)(lbo16 & 0x3FFFu) << 16) | ((uint64_t)8 << 32) | ((uint64_t)1 << 46);
}

// The same from its low word: address in bits 0..13, the K distance in bits 16..29.
__device__ __forceinline__ uint64_t band_desc_lo(uint32_t lo) { return (uint64_t)lo | ((uint64_t)(8u | (1u << 14)) << 32); }

// 16 lanes x 32 columns of tensor memory as matrix fragments (16x256b): thread t gets, for k = 0..3,
// v[4k], v[4k + 1] = columns 8k + 2 (t % 4), + 1 of lane t / 4 and v[4k + 2], v[4k + 3] the same of lane
// t / 4 + 8.  The wait is in the same statement.
__device__ __forceinline__ void band_ld(uint32_t t0, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(t0)
      : "memory");
}

// The same with 16 columns (k = 0, 1).
__device__ __forceinline__ void band_ld16(uint32_t t0, uint32_t (&v)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
      : "r"(t0)
      : "memory");
}

// 8 packed bytes (32 two-bit fields) -> one slot: nibble i of register 2j holds field 16j + 2i, of
// register 2j + 1 field 16j + 2i + 1.
__device__ __forceinline__ uint4 band_expand(uint32_t w0, uint32_t w1) {
  return make_uint4(w0 & 0x33333333u, (w0 >> 2) & 0x33333333u, w1 & 0x33333333u, (w1 >> 2) & 0x33333333u);
}

// Shared memory at a 32-bit address that a code is part of (tables that do not change after the fit).
__device__ __forceinline__ float lds_f(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ float4 lds_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}

// The code of D against the column's line (a, b), as the low bits of the result: 2^23 + round(L sat(a D + b)).
constexpr float kBandMagic = 8388608.0f;
__device__ __forceinline__ uint32_t band_code(float d, float la, float lb, float fl) {
  return __float_as_uint(fmaf(sat_fma(d, la, lb), fl, kBandMagic));
}

// The codes of D0 and D1 (band_code) with the second step of both as one packed fma.
__device__ __forceinline__ void band_code2(float d0, float d1, float2 l0, float2 l1, uint64_t fl2, uint32_t& c0,
                                           uint32_t& c1) {
  const float v0 = sat_fma(d0, l0.x, l0.y), v1 = sat_fma(d1, l1.x, l1.y);
  uint64_t v, m, r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(v0), "f"(v1));
  asm("mov.b64 %0, {%1, %1};" : "=l"(m) : "f"(kBandMagic));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(v), "l"(fl2), "l"(m));
  asm("mov.b64 {%0, %1}, %2;" : "=r"(c0), "=r"(c1) : "l"(r));
}

// Fits the line of one column: thresholds thr[0..L-1], sign s, |accumulator| <= B (LMAX: 3 or 15, the most that L
// is).  Thresholds at or past the bound (never or always exceeded, as the conversion's saturated ones of a channel
// with a small batch-norm scale) only have to stay past it.  Returns kBandLine where the line gives the exact code of
// every accumulator: with ascending thresholds it does when its code is at most i at x = T_i and at least i + 1
// at x = T_i + 1 (i = 0..L-1, both within the bound), because it cannot decrease with x = s A.  Else, for
// LMAX = 15, the line half a step lower: kBandNear where that is the code or one below it (at most i at T_i, at least
// i at T_i + 1), so that one comparison is left.  Else kBandFar.
// LMAX = 15: the four lanes of a quad share a column, q-th lane thresholds i = q, q + 4, .. against all (105 pairs
// in one thread took 5 us at the start of every launch).
constexpr uint32_t kBandLine = 0, kBandNear = 1, kBandFar = 2;
template <int LMAX>
__device__ __forceinline__ uint32_t band_fit(const int32_t* thr, int L, int s, int B, int q, float2* line) {
  constexpr int NQ = LMAX == 3 ? 1 : 4, NI = (LMAX + NQ - 1) / NQ;
  constexpr float kBig = 3.0e37f;
  const float fb = (float)B, fl = (float)L;
  auto quad = [&](float v, bool mx) {
    if constexpr (NQ == 4) {
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        const float u = __shfl_xor_sync(0xffffffffu, v, o);
        v = mx ? fmaxf(v, u) : fminf(v, u);
      }
    }
    return v;
  };
  float t[LMAX];           // clamped to -B - 1 (always exceeded) .. B (never)
  int below = 0, inside = 0;
  bool ok = true;
#pragma unroll
  for (int j = 0; j < LMAX; ++j) {
    t[j] = j < L ? fminf(fmaxf((float)thr[j], -fb - 1.0f), fb) : fb;
    below += t[j] < -fb ? 1 : 0;
    inside += t[j] >= -fb && t[j] < fb ? 1 : 0;
    if (j > 0) ok = ok && t[j] >= t[j - 1];
  }
  // The separating values m_i = m1 + i w: T_i < m_i < T_i + 1, below -B or above B for a threshold past it.
  // Slopes that leave room for an offset: (T_j - T_i - 1) / (j - i) < w < (T_j - T_i + 1) / (j - i)
  float ti[NI], lo = 0.0f, hi = kBig;
#pragma unroll
  for (int k = 0; k < NI; ++k) {
    const int i = NQ * k + q;
    ti[k] = i < L ? fminf(fmaxf((float)thr[i], -fb - 1.0f), fb) : kBig;
    const bool in = ti[k] >= -fb && ti[k] < fb;
#pragma unroll
    for (int j = NQ * k + 1; j < LMAX; ++j)
      if (j < L) {
        const int c = j - NQ * k;                      // j - i = c - q
        const float r = c > q ? 1.0f / (float)(c - q) : 0.0f;
        lo = fmaxf(lo, fmaf(t[j] - ti[k], r, -r));
        if (in && t[j] < fb && c > q) hi = fminf(hi, fmaf(t[j] - ti[k], r, r));
      }
  }
  lo = quad(lo, true);
  hi = quad(hi, false);
  const float w = hi < kBig ? fmaxf(0.5f * (lo + hi), 1.0f / 32.0f) : lo + 1.0f;
  float mlo = -kBig, mhi = kBig;
#pragma unroll
  for (int k = 0; k < NI; ++k) {
    const int i = NQ * k + q;
    const float v = ti[k] - (float)i * w;
    if (i < L && ti[k] >= -fb) mlo = fmaxf(mlo, v);
    if (i < L && ti[k] < fb) mhi = fminf(mhi, v + 1.0f);
  }
  const float m1 = 0.5f * (quad(mlo, true) + quad(mhi, false));
  // g(x) = (x - m1) / w + 1/2, x = s A = 2 s D;  v = g / L
  const float iw = 1.0f / (w * fl), fs = (float)s;
  const float la = inside ? 2.0f * fs * iw : copysignf(0.0f, fs);   // (the sign is read from it: band_near)
  float lb = inside ? 0.5f / fl - m1 * iw : (float)below / fl;
  // the code at T_i at most i, at T_i + 1 at least i + up
  auto check = [&](uint32_t up) {
    bool good = ok;
#pragma unroll
    for (int k = 0; k < NI; ++k) {
      const int i = NQ * k + q;
      const uint32_t c0 = band_code(0.5f * fs * ti[k], la, lb, fl) & 0xFFu;
      const uint32_t c1 = band_code(0.5f * fs * (ti[k] + 1.0f), la, lb, fl) & 0xFFu;
      if (i < L) good = good && (ti[k] < -fb || c0 <= (uint32_t)i) && (ti[k] >= fb || c1 >= (uint32_t)i + up);
    }
    if constexpr (NQ == 4) {   // all four lanes'
      const uint32_t votes = __ballot_sync(0xffffffffu, good);
      good = (votes >> (threadIdx.x & 28) & 15u) == 15u;
    }
    return good;
  };
  uint32_t kind = check(1u) ? kBandLine : kBandFar;
  if constexpr (LMAX == 15) {
    if (__any_sync(0xffffffffu, kind != kBandLine)) {
      if (kind != kBandLine && inside) lb = -m1 * iw;
      if (check(0u) && kind != kBandLine) kind = kBandNear;
    }
  }
  *line = make_float2(la, lb);
  return kind;
}

// Codes where some column of a block has no line, as band_code's results, two rows (D0, D1) of a column at a time.
// They are sums of saturating fmas, sat(2 s D - T) = [s A > T] (every T is an integer), added in pairs.
__device__ __forceinline__ uint64_t band_pair(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ uint64_t band_add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ void band_split(uint64_t v, uint32_t& a, uint32_t& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v));
}
// A column's thresholds in shared memory: (-T0, -T1, -T2, 2 s) for 2-bit codes, else sixteen -T in a row (-inf past the
// last), then 2 s.
__host__ __device__ constexpr int band_thr_bytes(int sbo) { return sbo == 2 ? 16 : 80; }

// `t`: the column's table.  4-bit codes are searched for in four steps, each one threshold.
template <int SBO>
__device__ __forceinline__ void band_codes_far(float d0, float d1, uint32_t t, uint32_t& c0, uint32_t& c1) {
  uint64_t n = band_pair(kBandMagic, kBandMagic);
  if constexpr (SBO == 2) {
    const float4 h = lds_f4(t);
    n = band_add2(n, band_pair(sat_fma(d0, h.w, h.x), sat_fma(d1, h.w, h.x)));
    n = band_add2(n, band_pair(sat_fma(d0, h.w, h.y), sat_fma(d1, h.w, h.y)));
    n = band_add2(n, band_pair(sat_fma(d0, h.w, h.z), sat_fma(d1, h.w, h.z)));
    band_split(n, c0, c1);
  } else {
    const float s2 = lds_f(t + 64u), m = lds_f(t + 28u);
    c0 = __float_as_uint(fmaf(sat_fma(d0, s2, m), 8.0f, kBandMagic));
    c1 = __float_as_uint(fmaf(sat_fma(d1, s2, m), 8.0f, kBandMagic));
#pragma unroll
    for (int k = 4; k >= 1; k >>= 1) {   // [s A > T_(c + k - 1)]
      const uint32_t tk = t + 4u * (uint32_t)(k - 1) - 4u * 0x4B000000u;
      c0 = __float_as_uint(fmaf(sat_fma(d0, s2, lds_f(tk + 4u * c0)), (float)k, __uint_as_float(c0)));
      c1 = __float_as_uint(fmaf(sat_fma(d1, s2, lds_f(tk + 4u * c1)), (float)k, __uint_as_float(c1)));
    }
  }
}

// From a line that is the code c or one below it: c + [s A > T_c].  (With an exact line s A <= T_c.)
__device__ __forceinline__ void band_codes_near(float d0, float d1, float2 line, uint64_t fl2, uint32_t t, uint32_t& c0,
                                                uint32_t& c1) {
  band_code2(d0, d1, line, line, fl2, c0, c1);
  const float t0 = lds_f(t + 4u * c0 - 4u * 0x4B000000u), t1 = lds_f(t + 4u * c1 - 4u * 0x4B000000u);
  const float s2 = copysignf(2.0f, line.x);
  band_split(band_add2(band_pair(__uint_as_float(c0), __uint_as_float(c1)),
                       band_pair(sat_fma(d0, s2, t0), sat_fma(d1, s2, t1))), c0, c1);
}

// Position in a ring of n buffers and the parity of its pass.
struct BandRing {
  int i = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void add(int k, int n) {
    i += k;
    while (i >= n) {
      i -= n;
      ph ^= 1u;
    }
  }
};

// n / d for 0 <= n < 2^31 as fdiv, in 32-bit arithmetic (umulhi(n, mul) <= n, so the sum fits).
__device__ __forceinline__ int fdiv31(int n, const FastDiv& f) {
  return (int)((__umulhi((uint32_t)n, f.mul) + (uint32_t)n) >> f.shift);
}

// One producer warp: packed codes global -> registers -> nibbles -> band ring.  A batch is kU slots a
// lane; the loads of the next batch (the next chunk's or tile's included) are in flight while a batch is
// expanded and stored, and only the stores wait for a free chunk buffer.  G16: 16-byte granules (two planes).
template <int G16>
__device__ __forceinline__ void band_produce(const BandArgs& a, uint8_t* smem, uint32_t bar, int first, int step,
                                             int n_local, int pw, int lane) {
  constexpr int kU = 4, PW = kBandProd;
  const int sw = 32 >> a.glg;                      // slots a warp takes at once
  const int sl = lane & (sw - 1), gl = lane >> (5 - a.glg);
  const int jstep = kU * PW * sw;
  const int j_own = pw * sw + sl;
  struct Cur { int jt, c, j0; };
  auto advance = [&](Cur& u) {                     // the next batch
    u.j0 += jstep;
    if (u.j0 >= a.slots) {
      u.j0 = 0;
      if (++u.c == a.nchunk) {
        u.c = 0;
        ++u.jt;
      }
    }
  };
  auto granules = [&](int c) {
    const int npl = min(a.cp, a.planes - c * a.cp);
    return G16 ? npl >> 1 : npl;
  };
  auto load = [&](const Cur& u, uint4 (&v)[kU]) {
    const int f0 = (first + u.jt * step) * 128 * a.mt + u.j0 + j_own;
    const int boff = u.c * a.cp * 8 + gl * (G16 ? 16 : 8);   // byte within the pixel
    const bool act = gl < granules(u.c);
    const uint8_t* xb = a.x + boff;
    if (G16 && a.linear) {                           // slot f is input pixel f
      const int last = min(a.slots - u.j0 - j_own, a.n * a.h * a.w - f0);
      const uint8_t* p = xb + (size_t)(uint32_t)f0 * (uint32_t)a.pb;
      const size_t dp = (size_t)(uint32_t)(PW * sw) * (uint32_t)a.pb;
#pragma unroll
      for (int k = 0; k < kU; ++k, p += dp) {
        v[k] = make_uint4(0u, 0u, 0u, 0u);
        if (act && k * PW * sw < last) v[k] = __ldg((const uint4*)p);
      }
      return;
    }
#pragma unroll
    for (int k = 0; k < kU; ++k) {
      v[k] = make_uint4(0u, 0u, 0u, 0u);
      const int f = f0 + k * PW * sw;
      const int r = fdiv31(f, a.div_P), xx = f - r * a.P;
      const int b = fdiv31(r, a.div_HP), yy = r - b * a.HP;
      const int iy = yy * a.s - a.pad, ix = xx * a.s - a.pad;
      const bool in = act && b < a.n && (unsigned)iy < (unsigned)a.h && (unsigned)ix < (unsigned)a.w &&
                      u.j0 + j_own + k * PW * sw < a.slots;
      if (in) {
        const uint8_t* p = xb + (size_t)(uint32_t)((b * a.h + iy) * a.w + ix) * (uint32_t)a.pb;
        if constexpr (G16) {
          v[k] = __ldg((const uint4*)p);
        } else if (a.gran == 8) {
          const uint2 q = __ldg((const uint2*)p);
          v[k].x = q.x;
          v[k].y = q.y;
        } else {
          const int left = a.pb - boff;              // bytes of this pixel from p on
          if (a.gran == 4) {
            v[k].x = __ldg((const uint32_t*)p);
            if (left > 4) v[k].y = __ldg((const uint32_t*)(p + 4));
          } else if (a.gran == 2) {
            v[k].x = __ldg((const uint16_t*)p);
            if (left > 2) v[k].x |= (uint32_t)__ldg((const uint16_t*)(p + 2)) << 16;
            if (left > 4) v[k].y = __ldg((const uint16_t*)(p + 4));
            if (left > 6) v[k].y |= (uint32_t)__ldg((const uint16_t*)(p + 6)) << 16;
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              if (q < left) v[k].x |= (uint32_t)__ldg(p + q) << (8 * q);
              if (q + 4 < left) v[k].y |= (uint32_t)__ldg(p + 4 + q) << (8 * q);
            }
          }
        }
      }
    }
  };
  BandRing cr;
  auto store = [&](const Cur& u, const uint4 (&v)[kU]) {
    const bool act = gl < granules(u.c);
    uint8_t* d = smem + (uint32_t)cr.i * a.chunk_bytes + (uint32_t)(G16 ? 2 * gl : gl) * a.plane_bytes + (uint32_t)(u.j0 + j_own) * 16u;
#pragma unroll
    for (int k = 0; k < kU; ++k, d += PW * sw * 16) {
      if (act && u.j0 + j_own + k * PW * sw < a.slots) {
        *(uint4*)d = band_expand(v[k].x, v[k].y);
        if constexpr (G16) *(uint4*)(d + a.plane_bytes) = band_expand(v[k].z, v[k].w);
      }
    }
  };
  // one batch: false once a wait ran out
  auto put = [&](const Cur& u, const uint4 (&v)[kU]) {
    if (u.j0 == 0 &&
        !__all_sync(0xffffffffu, mbar_wait_backoff(bar + 8u * (uint32_t)(a.ring + cr.i), cr.ph ^ 1u, 32)))
      return false;
    store(u, v);
    if (u.j0 + jstep >= a.slots) {   // the chunk is complete
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar + 8u * (uint32_t)cr.i);
      cr.add(1, a.ring);
    }
    return true;
  };
  if (n_local == 0) return;
  Cur u{0, 0, 0};
  uint4 v0[kU], v1[kU];
  load(u, v0);
#pragma unroll 1
  while (true) {   // two batches a round, so that the register sets need no copy
    Cur n = u;
    advance(n);
    if (n.jt < n_local) load(n, v1);
    if (!put(u, v0) || n.jt >= n_local) break;
    u = n;
    advance(u);
    if (u.jt < n_local) load(u, v0);
    if (!put(n, v1) || u.jt >= n_local) break;
  }
}

// What the MMA warps need (all uniform over a warp).
struct BandMma {
  uint32_t sbase, tmem, bar_a, bar_b, bar_c, done_bar, bar_turn;
  int n_local, ntl;
};

// One MMA warp.  The whole warp runs the loops with uniform values (the descriptors stay in uniform
// registers) and one elected lane issues groups of four MMAs, straight-line: what bounds this warp is its
// instruction count (it gets an issue slot every 10 cycles or so beside the other roles), so RES (resident
// filters) is compile-time.  A loop inside the elected lane's
// branch took about 200 cycles per MMA, run-time branches per MMA 150.  With
// two subtiles per tile, warp mi issues for subtile mi: both take every chunk and filter stage in order, and
// with an even number of accumulators (the planner sees to it) warp mi, epilogue group mi and every other
// accumulator belong together.  So each parity wait can only mean the phase it should.
template <int BN, int RES, int ALT>
__device__ __forceinline__ void band_mma(const BandArgs& a, const BandMma& w, const uint32_t* sTab, int mi, int lane) {
  constexpr uint32_t idesc = idesc_mxf4(128, BN);
  constexpr int kAccMax = (kBandCols - 16) / BN;
  static_assert(RES || !ALT, "the turn goes over with a pass's last chunk");
  const uint32_t sf = w.tmem + kBandCols - 16;
  auto a_full = [&](int i) { return w.bar_a + 8u * (uint32_t)i; };
  auto a_empty = [&](int i) { return w.bar_a + 8u * (uint32_t)(a.ring + i); };
  auto b_full = [&](int i) { return w.bar_b + 8u * (uint32_t)i; };
  auto b_empty = [&](int i) { return w.bar_b + 8u * (uint32_t)(a.stages + i); };
  auto c_full = [&](int i) { return w.bar_c + 8u * (uint32_t)i; };
  auto c_empty = [&](int i) { return w.bar_c + 8u * (uint32_t)(2 * kAccMax + i); };
  const uint32_t sB16 = (w.sbase + a.off_b) >> 4, st16 = a.stage_bytes >> 4;
  const int steps_full = (a.cp >> 1) * a.taps;
  const int npl_last = a.planes - (a.nchunk - 1) * a.cp;
  const int steps_last = (npl_last >> 1) * a.taps + (npl_last & 1 ? a.nodd : 0);
  // ALT: passes (a tile's channel tiles) alternate between the two warps.  A pass's
  // waits come after the ones of the pass before it (the turn barriers), so no parity can mean another
  // phase; its MMAs overlap the other warp's, which hides what lies between two passes (about 700 cycles).
  const int passes = w.ntl;
  const int last_use = ALT && passes > 1 ? passes - 2 : passes - 1;   // passes from here on are a warp's last of a tile
  uint32_t turn_ph = 0;
  BandRing tr, br, ar;   // the tile's first chunk, the next filter stage (streamed), the next accumulator
  BandRing fr, wr;       // its barriers, and those of the accumulator's last use (a.nacc passes before)
  int uses = 0;          // accumulators taken
  auto next_acc = [&](int k) {
    ar.add(k, a.nacc);
    fr.add(k, a.ncb);
    const int past = uses + k - a.nacc;               // how far beyond the first round
    if (past > 0) wr.add(min(past, k), a.ncb);
    uses = min(uses + k, a.nacc);
  };
  if constexpr (!ALT) next_acc(mi);
  bool ok = true, ready = false;   // ready: the next chunk was seen full already
#pragma unroll 1
  for (int jt = 0; jt < w.n_local && ok; ++jt) {
#pragma unroll 1
    for (int p = 0; p < passes; ++p) {
      if (ALT && ((jt * passes + p) & 1) != mi) {   // the other warp's
        ready = false;
      } else {
        bool in = true;
        if (ALT && (jt | p)) {
          in = mbar_wait(w.bar_turn + 8u * (uint32_t)mi, turn_ph);
          turn_ph ^= 1u;
        }
        if (uses == a.nacc) in = mbar_wait(c_empty(wr.i), wr.ph) && in;
        const uint32_t dacc = w.tmem + (uint32_t)(ar.i * BN);
        // filters: resident stages of channel tile p, waited for in the first tiles
        uint32_t b16 = sB16 + (uint32_t)(p * a.nst) * st16, bwait = b_full(p * a.nst);
        const bool wait_res = jt < 2;
        uint32_t acc = 0;
        BandRing cr = tr;
#pragma unroll 1
        for (int c = 0; c < a.nchunk; ++c, cr.add(1, a.ring)) {
          const bool last_c = c == a.nchunk - 1;
          const int steps = last_c ? steps_last : steps_full;
          const uint4* ent = (const uint4*)(sTab + (last_c ? a.tab_last : 0));
          const uint32_t a16 = ((w.sbase + (uint32_t)cr.i * a.chunk_bytes) >> 4) + (ALT ? 0u : (uint32_t)(128 * mi));
          if (p == 0) in = (ready || mbar_wait(a_full(cr.i), cr.ph)) && in;
          if (!__all_sync(0xffffffffu, in)) {
            ok = false;
            break;
          }
          tc_fence_after();
          // the turn goes over as soon as this pass's waits are done: two passes issued side by side beat handing it
          // over with two groups left (179 and 200 us on the 3x3 256 -> 256 layer at batch 256, in an earlier build that
          // differed in nothing else)
          if (ALT && last_c && lane == 0) mbar_arrive(w.bar_turn + 8u * (uint32_t)(mi ^ 1));
          // Shared memory is the busy unit here (an MMA reads 8 KB of it in 64 cycles), so what this warp
          // reads from it is asked for ahead: the next group's entries during this group, and whether the
          // next chunk is there during the last group.
          uint4 en = ent[0];
#pragma unroll 1
          for (int q = 0; q < steps; q += 4) {
            const uint4 e = en;
            en = ent[(q >> 2) + 1];                   // (one past the table at its end: slack behind it)
            if (!ALT && q + 4 >= steps) {
              BandRing nx = cr;
              nx.add(1, a.ring);
              ready = mbar_test(a_full(nx.i), nx.ph);
            }
            if constexpr (!RES) {
              b16 = sB16 + (uint32_t)br.i * st16;
              if (!__all_sync(0xffffffffu, mbar_wait(b_full(br.i), br.ph))) {
                ok = false;
                break;
              }
              tc_fence_after();
            } else if (wait_res) {
              if (!__all_sync(0xffffffffu, mbar_wait(bwait, 0u))) {
                ok = false;
                break;
              }
              bwait += 8u;
              tc_fence_after();
            }
            if (elect_one()) {
              auto mma = [&](uint32_t ee, int k, uint32_t ac) {
                mma_mxf4(dacc, band_desc_lo(a16 + ee), band_desc(b16 + (uint32_t)(2 * BN * k), BN), idesc, sf, ac);
              };
              mma(e.x, 0, acc);
              if (q + 4 <= steps) {
                mma(e.y, 1, 1u);
                mma(e.z, 2, 1u);
                mma(e.w, 3, 1u);
              } else {
                if (q + 1 < steps) mma(e.y, 1, 1u);
                if (q + 2 < steps) mma(e.z, 2, 1u);
              }
              if constexpr (!RES) mma_commit(b_empty(br.i));
            }
            __syncwarp();
            acc = 1;
            if constexpr (RES) b16 += st16;
            else br.add(1, a.stages);
          }
          if (!ok) break;
          if (p >= last_use || last_c) {
            if (elect_one()) {
              if (p >= last_use) mma_commit(a_empty(cr.i));
              if (last_c) mma_commit(c_full(fr.i));
            }
            __syncwarp();
          }
        }
        if (!ok) break;
      }
      next_acc(a.mt);
    }
    tr.add(a.nchunk, a.ring);
  }
  if (elect_one()) mma_commit(w.done_bar);   // fires once every MMA this warp issued has completed
  __syncwarp();
}

// BN: output channels per tile; SBO: bits per output code.  One CTA per SM.  (Two smaller ones, with one epilogue
// group each, were as fast on single layers, but behind another layer of a network both may start on one SM:
// 89.6 against 82.8 us on the ResNet-18 body at batch 1.)
template <int BN, int SBO>
__global__ void __launch_bounds__(kBandThreads, 1)
    conv_band_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ BandArgs a) {
  constexpr int EG = 2, PW = kBandProd, kEW = kBandEpi;
  constexpr int kWarpProd = kEW, kWarpB = kEW + PW, kWarpMma = kEW + PW + 1;
  constexpr uint32_t kCols = kBandCols;
  constexpr int kAccMax = (int)(kCols - 16) / BN;    // accumulator buffers that fit beside the scales
  constexpr uint32_t kSf = kCols - 16;               // scale columns
  constexpr uint32_t kColB = BN * 16;                // bytes of a core column of filters
  extern __shared__ uint8_t smem_raw_[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw_ + 127) & ~(uintptr_t)127);
  const uint32_t sbase = smem_u32(smem);
  float2* sLin = (float2*)(smem + a.off_lin);        // [ngrp * BN] (a, b)
  float4* sThr = (float4*)(smem + a.off_thr);        // their thresholds (band_codes_far)
  uint32_t* sBad = (uint32_t*)(smem + a.off_bad);    // per warp of the fit: the worst kind of its columns
  uint32_t* sTab = (uint32_t*)(smem + a.off_tab);    // A descriptors of the MMAs of a chunk
  uint32_t* tmem_slot = (uint32_t*)(smem + a.off_bad + 128);
  const uint32_t bar = sbase + a.off_bar;
  auto a_full = [&](int i) { return bar + 8u * (uint32_t)i; };
  auto a_empty = [&](int i) { return bar + 8u * (uint32_t)(a.ring + i); };
  const uint32_t bar_b = bar + 16u * (uint32_t)a.ring;
  auto b_full = [&](int i) { return bar_b + 8u * (uint32_t)i; };
  auto b_empty = [&](int i) { return bar_b + 8u * (uint32_t)(a.stages + i); };
  const uint32_t bar_c = bar_b + 16u * (uint32_t)a.stages;
  auto c_full = [&](int i) { return bar_c + 8u * (uint32_t)i; };
  auto c_empty = [&](int i) { return bar_c + 8u * (uint32_t)(2 * kAccMax + i); };
  const uint32_t done_bar = bar_c + 32u * (uint32_t)kAccMax;

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // known to be uniform: the roles' branches are
  // CTA c: channel group c % ngroups, tiles c / ngroups, + gridDim / ngroups, ...
  const int grp = (int)blockIdx.x % a.ngroups;
  const int first = (int)blockIdx.x / a.ngroups, step = (int)gridDim.x / a.ngroups;
  const int nt0 = grp * a.ngrp, ntl = min(a.ngrp, a.nt - nt0);   // its channel tiles
  const int n_local = first < a.mtiles ? (a.mtiles - first + step - 1) / step : 0;

  // ---- setup (reads no global memory, so it may overlap the previous grid)
  if (warp == kWarpB && lane == 0) prefetch_tmap(&tmap_w);
  if (warp == kWarpMma) {
    tmem_alloc(smem_u32(tmem_slot), kCols);
    tmem_relinquish();
  }
  if (tid == 0) {
    // MMA warps that release a chunk (both with a subtile each, or where a tile's passes alternate) and a stage
    const bool alt = a.mt == 1;
    const int rel_a = alt ? min(2, ntl) : 2, rel_b = alt ? 1 : 2;
    for (int i = 0; i < a.ring; ++i) {
      mbar_init(a_full(i), PW);
      mbar_init(a_empty(i), rel_a);
    }
    for (int i = 0; i < a.stages; ++i) {
      mbar_init(b_full(i), 1);
      mbar_init(b_empty(i), rel_b);
    }
    mbar_init(done_bar + 8u, 1);
    mbar_init(done_bar + 16u, 1);
    for (int i = 0; i < 2 * kAccMax; ++i) {
      mbar_init(c_full(i), 1);
      mbar_init(c_empty(i), 8);
    }
    mbar_init(done_bar, 2);
    fence_mbar_init();
  }
  {
    // One entry per MMA of a chunk: the low word of its A descriptor relative to the chunk's first
    // slot.  The table of a full chunk (pairs of planes), then the last chunk's, each a multiple of four
    // entries (a.tab_last, a.ntab).
    auto off16 = [&](int tap) { return (uint32_t)(tap / a.kw * a.P + tap % a.kw); };
    const uint32_t pl16 = a.plane_bytes >> 4;
    const int pairs_last = (a.planes - (a.nchunk - 1) * a.cp) >> 1;
    for (int i = tid; i < a.ntab; i += kBandThreads) {
      const bool last = i >= a.tab_last;
      const int q = last ? i - a.tab_last : i, pairs = last ? pairs_last : a.cp >> 1;
      uint32_t e = 0;
      if (q < pairs * a.taps) {
        const int p = q / a.taps;
        e = (2u * (uint32_t)p * pl16 + off16(q - p * a.taps)) | (pl16 << 16);
      } else if (last && q - pairs * a.taps < a.nodd) {
        const int t0 = 2 * (q - pairs * a.taps);
        const uint32_t o0 = off16(t0), o1 = t0 + 1 < a.taps ? off16(t0 + 1) : o0 + 1u;
        e = (2u * (uint32_t)pairs * pl16 + o0) | ((o1 - o0) << 16);
      }
      sTab[i] = e;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  if (warp < 4) {   // unit scales (ue8m0 1.0) in every lane
    const uint32_t one = 0x7F7F7F7Fu;
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};\n\t"
        "tcgen05.wait::st.sync.aligned;" ::"r"(tmem + kSf + ((uint32_t)(warp * 32) << 16)),
        "r"(one)
        : "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dep_launch();

  if (warp >= kWarpProd && warp < kWarpB) {
    // =================== producers: packed codes -> nibbles -> band ring ===================
    grid_dep_wait();
    if (a.gran == 16) band_produce<1>(a, smem, bar, first, step, n_local, warp - kWarpProd, lane);
    else band_produce<0>(a, smem, bar, first, step, n_local, warp - kWarpProd, lane);
  } else if (warp == kWarpB) {
    // =================== filter stages: TMA boxes ===================
    if (!a.early) grid_dep_wait();
    const int passes = a.resident ? 1 : n_local;
    BandRing br;
    int it = 0;
    bool ok = true;
#pragma unroll 1
    for (int jt = 0; jt < passes && n_local > 0 && ok; ++jt)
#pragma unroll 1
      for (int t = 0; t < ntl && ok; ++t) {
        const int n0 = (nt0 + t) * BN;
        int col = 0, left = 0, c = 0;                 // core column, MMAs left in the chunk, next chunk
#pragma unroll 1
        for (int st = 0; st < a.nst; ++st, ++it, br.add(1, a.stages)) {
          const int buf = br.i;
          if (left == 0) {
            const int npl = min(a.cp, a.planes - c * a.cp);
            left = (npl >> 1) * a.taps + (npl & 1 ? a.nodd : 0);
            ++c;
          }
          if (!a.resident && !__all_sync(0xffffffffu, mbar_wait(b_empty(buf), br.ph ^ 1u))) {
            ok = false;
            break;
          }
          // one box per stage: 8 core columns x BN filter rows (a stage that ends a chunk also brings columns
          // that nothing reads).  One bulk copy per core column took about 97 cycles each whatever its size,
          // 21 bytes a cycle at BN = 128: the 3x3 1024 -> 1024 layer at 13 x 13, b64 took 89 us with streamed
          // filters and one subtile.
          if (elect_one()) {
            mbar_arrive_expect_tx(b_full(buf), 8u * kColB);
            tma_load_2d(sbase + a.off_b + (uint32_t)buf * a.stage_bytes, &tmap_w, b_full(buf), 2 * n0, col);
          }
          __syncwarp();
          const int n = min(4, left);
          col += 2 * n;
          left -= n;
        }
      }
    // after a timeout: every copy issued has landed before the CTA may exit
    if (!ok)
      for (int i = max(0, it - a.stages); i < it; ++i) mbar_wait(b_full(i % a.stages), (uint32_t)(i / a.stages) & 1u);
    if (a.resident)
      for (int i = 0; i < it; ++i) mbar_wait(b_full(i), 0);
    __syncwarp();
  } else if (warp >= kWarpMma) {
    // =================== MMA issue ===================
    const BandMma w{sbase, tmem, bar, bar_b, bar_c, done_bar, done_bar + 8u, n_local, ntl};
    const int mi = warp - kWarpMma;
    if (a.mt == 1) band_mma<BN, 1, 1>(a, w, sTab, mi, lane);   // (with resident filters)
    else if (a.resident) band_mma<BN, 1, 0>(a, w, sTab, mi, lane);
    else band_mma<BN, 0, 0>(a, w, sTab, mi, lane);
  } else {
    // =================== epilogue: thresholds, packing, stores ===================
    if (!a.early) grid_dep_wait();
    const int eg = warp >> 3;                         // group
    const int quarter = warp & 3, sub = (warp >> 2) & 1;
    // A warp's share of an accumulator: a block of KB columns, in 16-lane halves.  BN = 128: warp pair
    // (quarter, sub) takes column block `sub`, both halves of the quarter; else lane half `sub`.
    constexpr int KB = kBandBlock;                    // columns of a block: one word of 2-bit codes per lane quad
    constexpr int NC = KB / 4;                        // channels of a thread: NC consecutive ones (prep_band_kernel)
    constexpr int NH = BN == 128 ? 2 : 1;             // lane halves
    constexpr int NL = KB / 32;                       // loads of 32 columns
    constexpr int kW = NC * SBO / 32;                 // words of codes
    const int cblk = BN == 128 ? sub * KB : 0;
    const int half0 = BN == 128 ? 0 : sub;
    const int quad = lane & 3;
    uint64_t fl2;                                     // the highest code, twice
    {
      const float fl = (float)a.lvl;
      asm("mov.b64 %0, {%1, %1};" : "=l"(fl2) : "f"(fl));
    }
    // lines and thresholds of every column of this CTA, in accumulator-column order
    constexpr int NQ = SBO == 2 ? 1 : 4;              // threads of a column (band_fit)
    for (int c4 = tid; c4 < ntl * BN * NQ; c4 += 32 * kEW) {
      const int c = c4 / NQ, q = c4 % NQ;
      const int nn = band_channel(nt0 * BN + c);
      const bool has = nn < a.cout && a.thr && a.y_codes;
      const int32_t* T = a.thr + (size_t)(has ? nn : 0) * a.lvl;
      const int s = has ? a.sign[nn] : 1, L = has ? a.lvl : 0;
      float2 ln;
      const uint32_t kind = band_fit<SBO == 2 ? 3 : 15>(T, L, s, a.bound, q, &ln);
      if (q == 0) sLin[c] = has ? ln : make_float2(0.f, 0.f);
      auto th = [&](int i) { return i < L ? (float)T[i] : INFINITY; };
      if constexpr (SBO == 2) {
        sThr[c] = make_float4(-th(0), -th(1), -th(2), 2.0f * (float)s);
      } else {
        sThr[5 * c + q] = make_float4(-th(4 * q), -th(4 * q + 1), -th(4 * q + 2), -th(4 * q + 3));
        if (q == 0) sThr[5 * c + 4].x = 2.0f * (float)s;
      }
      // the worst of a warp's columns
      const uint32_t worst = __reduce_max_sync(0xffffffffu, has ? kind : kBandLine);
      if (lane == 0) sBad[c4 >> 5] = worst;
    }
    named_bar(1, 32 * kEW);
    bool ok = true;
    // units (a tile's subtile and channel tile) in order; this group takes every EG-th
    const int per_tile = ntl * a.mt;
    const int rowb = (a.cout * SBO) >> 3;
    BandRing ar, fr;                                  // the unit's accumulator and its barriers
    ar.add(eg, a.nacc);
    fr.add(eg, a.ncb);
    int rest = eg % per_tile;                         // its place in the tile
    int tile = first + eg / per_tile * step;
    const int msh = a.mt >> 1;                        // (one or two subtiles)
    // One unit of channel tile t in the given form; line: with kBandLine, this thread's columns 8 k +
    // 2 quad, + 1 (the other forms read what they need, so that no register holds a line there).  False after a
    // timeout.
    auto unit = [&](auto kind_c, const int t, const float2* line) __attribute__((always_inline)) {
      constexpr uint32_t kind = decltype(kind_c)::value;
      const int m = rest & (a.mt - 1);
      // the output pixel of row `lane` of the quarter, -1 for an anchor that is none
      const int f = (tile * a.mt + m) * 128 + quarter * 32 + lane;
      const int rr = fdiv31(f, a.div_P), xx = f - rr * a.P;
      const int b = fdiv31(rr, a.div_HP), yy = rr - b * a.HP;
      const int pixel = b < a.n && yy < a.oh && xx < a.ow ? (b * a.oh + yy) * a.ow + xx : -1;
      if (!__all_sync(0xffffffffu, mbar_wait_backoff(c_full(fr.i), fr.ph, 32))) return false;
      const uint32_t tacc = tmem + (uint32_t)(ar.i * BN + cblk) + ((uint32_t)(quarter * 32 + 16 * half0) << 16);
      tc_fence_after();
      const int ch0 = (nt0 + t) * BN + cblk + NC * quad;   // this thread's first output channel
      const bool chans = ch0 < a.cout;
#pragma unroll 1
      for (int h = 0; h < NH; ++h) {
        uint32_t packed[2][kW];                       // rows lane / 4 and lane / 4 + 8 of the half
        // the output pixel of row r (asked for where it is used: two registers fewer)
        auto pix_of = [&](int r) {
          return __shfl_sync(0xffffffffu, pixel, 16 * (half0 + h) + 8 * r + (lane >> 2));
        };
        const uint32_t lo16 = (uint32_t)(16 * h) << 16;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int w = 0; w < kW; ++w) packed[r][w] = 0;
#pragma unroll
        for (int ld = NL - 1; ld >= 0; --ld) {        // descending, so that the first code ends up lowest
          uint32_t v[16];
          if constexpr (kind == kBandLine) {
            band_ld(tacc + lo16 + (uint32_t)(32 * ld), v);
            if (a.y_codes) {
#pragma unroll
              for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int j = 6; j >= 0; j -= 2) {     // channels 8 ld + j, + 1 of this thread
                  uint32_t c0, c1;
                  band_code2(__uint_as_float(v[2 * j + 2 * r]), __uint_as_float(v[2 * j + 2 * r + 1]), line[8 * ld + j],
                             line[8 * ld + j + 1], fl2, c0, c1);
                  uint32_t& w = packed[r][(8 * ld + j) * SBO / 32];
                  w = (w << SBO) + c1;
                  w = (w << SBO) + c0;
                }
            }
          } else {
            // thresholds that no line separates: 16 columns at a time, in a loop (the registers of more spill)
#pragma unroll 1
            for (int g = 1; g >= 0; --g) {
              const int c16 = 32 * ld + 16 * g;
              uint32_t u[8];
              band_ld16(tacc + lo16 + (uint32_t)c16, u);
#pragma unroll
              for (int j = 3; j >= 0; --j) {          // channel 8 ld + 4 g + j
                const float d0 = __uint_as_float(u[4 * (j >> 1) + (j & 1)]), d1 = __uint_as_float(u[4 * (j >> 1) + 2 + (j & 1)]);
                const int col = t * BN + cblk + c16 + 2 * quad + 8 * (j >> 1) + (j & 1);
                const uint32_t tab = sbase + a.off_thr + (uint32_t)(col * band_thr_bytes(SBO));
                uint32_t c0, c1;
                if constexpr (kind == kBandNear) band_codes_near(d0, d1, sLin[col], fl2, tab, c0, c1);
                else band_codes_far<SBO>(d0, d1, tab, c0, c1);
                uint32_t& w0 = packed[0][8 * ld * SBO / 32];
                uint32_t& w1 = packed[1][8 * ld * SBO / 32];
                w0 = (w0 << SBO) + c0;
                w1 = (w1 << SBO) + c1;
              }
            }
          }
          if (a.y_acc) {
            if constexpr (kind != kBandLine) band_ld(tacc + lo16 + (uint32_t)(32 * ld), v);
            // A = 2 D as an integer: the low mantissa bits of 2 D + 1.5 * 2^23
            auto ia = [&](int i) { return __float_as_int(fmaf(__uint_as_float(v[i]), 2.0f, 12582912.0f)) - 0x4B400000; };
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              const int pix = pix_of(r);
              if (pix < 0) continue;
              int32_t* dst = a.y_acc + (size_t)pix * a.cout + ch0 + 8 * ld;
              if ((a.cout & 3) == 0) {
#pragma unroll
                for (int j = 0; j < 8; j += 4)
                  if (ch0 + 8 * ld + j < a.cout)
                    *(int4*)(dst + j) = make_int4(ia(2 * j + 2 * r), ia(2 * j + 2 * r + 1), ia(2 * j + 4 + 2 * r),
                                                  ia(2 * j + 5 + 2 * r));
              } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                  if (ch0 + 8 * ld + j < a.cout) dst[j] = ia(4 * (j >> 1) + 2 * r + (j & 1));
              }
            }
          }
        }
        if (a.y_codes) {
          const int pix0 = pix_of(0), pix1 = pix_of(1);
          // what the exponent bits of the terms add up to (0x4B000000 each, shifted)
          constexpr uint32_t kOff = SBO == 2 ? 0xE7000000u : 0xFB000000u;
#pragma unroll
          for (int r = 0; r < 2 && chans; ++r) {
            const int pix = r ? pix1 : pix0;
            if (pix < 0) continue;
            uint8_t* dst = a.y_codes + (size_t)pix * rowb + ((ch0 * SBO) >> 3);
#pragma unroll
            for (int w = 0; w < kW; ++w) packed[r][w] -= kOff;
            if (ch0 + NC <= a.cout && (rowb & (4 * kW - 1)) == 0) {
              if constexpr (kW == 1) *(uint32_t*)dst = packed[r][0];
              else *(uint2*)dst = make_uint2(packed[r][0], packed[r][kW - 1]);
            } else {
              const int nbytes = (min(NC, a.cout - ch0) * SBO) >> 3;
#pragma unroll
              for (int q = 0; q < 4 * kW; ++q)
                if (q < nbytes) dst[q] = (uint8_t)(packed[r][q >> 2] >> (8 * (q & 3)));
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(c_empty(fr.i));
      rest += EG;
      while (rest >= per_tile) {
        rest -= per_tile;
        tile += step;
      }
      ar.add(EG, a.nacc);
      fr.add(EG, a.ncb);
      return true;
    };
    // this warp's blocks (one a channel tile) all take the form that the worst of them needs
    uint32_t kind = kBandLine;
#pragma unroll 1
    for (int t = 0; t < ntl; ++t)
#pragma unroll
      for (int i = 0; i < 2 * NQ; ++i) kind = max(kind, sBad[((t * BN + cblk) * NQ >> 5) + i]);
    if (kind == kBandLine) {
#pragma unroll 1
      while (ok && tile < a.mtiles) {
        const int t = rest >> msh;
        float2 line[NC];                              // a channel tile's lines stay in registers
        const float4* l4 = (const float4*)(sLin + t * BN + cblk + 2 * quad);
#pragma unroll
        for (int k = 0; k < NC / 2; ++k) {
          const float4 l = l4[4 * k];
          line[2 * k] = make_float2(l.x, l.y);
          line[2 * k + 1] = make_float2(l.z, l.w);
        }
#pragma unroll 1
        do {
          ok = unit(std::integral_constant<uint32_t, kBandLine>{}, t, line);
        } while (ok && tile < a.mtiles && rest >> msh == t);
      }
    } else if (SBO == 4 && kind == kBandNear) {
#pragma unroll 1
      while (ok && tile < a.mtiles) ok = unit(std::integral_constant<uint32_t, kBandNear>{}, rest >> msh, nullptr);
    } else {
#pragma unroll 1
      while (ok && tile < a.mtiles) ok = unit(std::integral_constant<uint32_t, kBandFar>{}, rest >> msh, nullptr);
    }
  }

  // ---- teardown: every MMA has completed (done_bar) before tensor memory is released
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    mbar_wait(done_bar, 0);
    tmem_dealloc(tmem, kCols);
  }
}

// Prepared filters of the band path, [core column][crows][16 bytes], from the sign words (rows past cout are
// zero).  dig: 2-bit digits per filter weight (1, or 2 for 4-bit fields: digit 1 weighs 4).  fields: 2-bit
// fields per pixel.
__global__ void prep_band_kernel(const uint32_t* bits, uint4* out, int cout, int crows, int kwords, int fields, int dig,
                                 int taps, int npair, long total) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const int n = band_channel((int)(i % crows)), cc = (int)(i / crows);
    const bool odd = cc >= npair * taps * 2;          // core column of the odd last plane: one tap each
    const int pair = cc / (2 * taps), r = cc - pair * 2 * taps;
    const int plane = odd ? 2 * npair : 2 * pair + (r & 1), tap = odd ? cc - npair * taps * 2 : r >> 1;
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    if (tap < taps && n < cout) {
      const uint32_t* row = bits + (size_t)n * kwords;
      const int cin = fields / dig;
#pragma unroll
      for (int p = 0; p < 32; ++p) {
        const int fld = plane * 32 + 16 * (p >> 4) + 2 * (p & 7) + ((p >> 3) & 1);   // the order of band_expand
        if (fld < fields) {
          const int c = dig == 2 ? fld >> 1 : fld;
          const int k = tap * cin + c;
          const bool plus = (row[k >> 5] >> (k & 31)) & 1u;
          const uint32_t mag = dig == 2 && (fld & 1) ? 0x6u : 0x2u;
          w[p >> 3] |= (plus ? mag : (mag | 0x8u)) << (4 * (p & 7));
        }
      }
    }
    out[i] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

}  // namespace ifq
