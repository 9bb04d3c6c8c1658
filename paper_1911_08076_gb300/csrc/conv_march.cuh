// March path of the quantized convolution for the narrow first layers of a detector: 3 x 3, stride 1, a fused
// 2 x 2 pool, 2-bit codes out, few channels (Eq. (1), the pool of Sec. 2.1 on Y^conv, the thresholds of Eq. (7)).
// Inputs of 4 channels of 8-bit values or of 8 channels of 2-bit codes: at most one 32-bit word a pixel.
//
// These layers have too few channels to fill a tcgen05 tile.  One
// warp takes 8 pooled columns and marches down the pooled rows; a step is two m16n8k16 f16 products chains (the
// two conv rows of the pooled row), whose 16 rows are the 8 pooled columns at window column 0 (rows 0..7) and 1
// (rows 8..15).  So a thread's fragments of the two chains hold all four window positions of its channels, and
// the pool is a maximum in registers.
//
// K is laid out so that a fragment needs no exchange: lane t of a quad holds filter column dx = t (lane 3 has zero
// weights) and K step the filter row, so its A registers are the pixel it loaded itself: bytes (or 2-bit fields)
// moved into f16 halves by a permute or a mask.  The bits are read as f16 subnormals, x * 2^-24 (a field 4^i x
// against a weight of 4^-i), so no conversion is needed, and every product and fp32 sum is an exact integer
// multiple of 2^-24.  A pixel is loaded and expanded once per filter column and window column and kept over the
// rows of the march; the rows are loaded two steps ahead.
//
// Measured (us, batch 64, pooled; the kernel before, this one): 3 x 3 4 -> 8 on 416 x 416 8-bit pixels 64.9 (dp4a, the
// direct kernel), 43.9; 3 x 3 8 -> 16 on 208 x 208 2-bit codes 41.9 (the warp kernel's e4m3 mma.sync, which
// issues as four instructions), 30.3.  Their bytes take 7.5 and 1.25 us: latency bounds both.
// On 16 images issue slots are busy in 41 and 30 % of the cycles; of the 12.2 and 8.4 cycles between two instructions of
// a warp, 2.9 and 1.0 wait for loads, 3.1 and 2.0 for fixed latencies and 1.1 and 1.8 for the product pipe (rows
// loaded one step ahead 45.2 and 32.3 us).
#pragma once
#include "conv_common.cuh"

namespace ifq {

constexpr int kMarchThreads = 128;

// CTAs per SM: as many as their registers allow.
__host__ __device__ constexpr int march_ctas(int in8, int nt) { return in8 ? (nt == 1 ? 8 : 5) : (nt == 1 ? 5 : (nt == 2 ? 4 : 3)); }

struct MarchArgs {
  const void* x;           // 8-bit values, 4 a pixel, or 2-bit codes, 8 a pixel
  const uint32_t* w;       // IN8: [36] bit n: filter n is +1 at (tap, channel); else sign words [cout][kwords]
  const int32_t* thr;      // [cout][3]
  const int8_t* sign;      // [cout]
  uint8_t* y;              // packed 2-bit codes [n][pho][pwo][cout / 4]
  int h, w_in, cout, kwords, pad, pho, pwo;
  int ry;                  // pooled rows of a march
  int units;               // n * ceil(pho / ry) * ceil(pwo / 8)
  FastDiv div_strips, div_blocks;
};

// D (+)= A . B, m16n8k16, f16 operands, fp32 sums.
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}

// IN8: 1 for 8-bit values; NT: tiles of 8 output channels.
template <int IN8, int NT>
__global__ void __launch_bounds__(kMarchThreads, march_ctas(IN8, NT)) conv_march_kernel(const MarchArgs a) {
  constexpr int NR = IN8 ? 2 : 4;                    // f16 pairs of a pixel
  constexpr int KS = NR / 2;                         // K steps of a filter row
  using Word = typename std::conditional<IN8 != 0, uint32_t, uint16_t>::type;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  grid_dep_launch();
  grid_dep_wait();
  // Weights as B fragments: channel 8 j + g, filter column t.
  uint2 b[NT][3 * KS];
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
      for (int q = 0; q < KS; ++q) {
        const int n = 8 * j + g, tap = 3 * dy + t;
        uint32_t r[2] = {0u, 0u};
        if (t < 3 && n < a.cout) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {              // halves of the pairs 2 q and 2 q + 1
            bool plus;
            uint32_t one = 0x3C00u;
            if constexpr (IN8) {
              plus = (__ldg(a.w + 4 * tap + e) >> n) & 1u;
            } else {
              const int i = 2 * q + (e >> 1), k = 8 * tap + i + 4 * (e & 1);   // pair i: channels i and 4 + i
              one -= (uint32_t)(2 * i) << 10;        // 4^-i
              plus = (__ldg(a.w + (size_t)n * a.kwords + (k >> 5)) >> (k & 31)) & 1u;
            }
            r[e >> 1] |= (one | (plus ? 0u : 0x8000u)) << (16 * (e & 1));
          }
        }
        b[j][KS * dy + q] = make_uint2(r[0], r[1]);
      }
  // Thresholds of channels 8 j + 2 t + c, as code3f's (conv_tc.cuh): [s A > T] = sat(2^24 s D - T).
  float4 th[NT][2];
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int n = min(8 * j + 2 * t + c, a.cout - 1);
      th[j][c] = make_float4(-(float)__ldg(a.thr + 3 * n), -(float)__ldg(a.thr + 3 * n + 1),
                             -(float)__ldg(a.thr + 3 * n + 2), 16777216.0f * (float)a.sign[n]);
    }
  const float s0 = (float)(1 << (4 * t)), s1 = 4.0f * s0;   // places of the two codes in a pixel's 16 bits
  const int rowb = a.cout >> 2, w = a.w_in;

  for (int u = (blockIdx.x * kMarchThreads + threadIdx.x) >> 5; u < a.units; u += gridDim.x * (kMarchThreads / 32)) {
    const int ub = (int)fdiv((uint32_t)u, a.div_strips), strips = (a.pwo + 7) >> 3;
    const int x0 = 8 * (u - ub * strips);
    const int img = (int)fdiv((uint32_t)ub, a.div_blocks), blocks = (a.pho + a.ry - 1) / a.ry;
    const int y0 = a.ry * (ub - img * blocks);
    const int ny = min(a.ry, a.pho - y0);
    const int X = x0 + g, ix = 2 * X + t - a.pad;
    const bool c0 = t < 3 && (unsigned)ix < (unsigned)w, c1 = t < 3 && (unsigned)(ix + 1) < (unsigned)w;
    int iy = 2 * y0 - a.pad;                         // the next input row
    const Word* p = (const Word*)a.x + ((long long)img * a.h + iy) * w + ix;
    uint32_t qa[2][2], qb[2][2];                     // the pixels of the next two row pairs, in turn
    auto load = [&](uint32_t (&raw)[2][2]) {                              // two input rows, window columns 0 and 1
#pragma unroll
      for (int r = 0; r < 2; ++r, ++iy, p += w) {
        const bool ok = (unsigned)iy < (unsigned)a.h;
        raw[r][0] = ok && c0 ? (uint32_t)__ldg(p) : 0u;
        raw[r][1] = ok && c1 ? (uint32_t)__ldg(p + 1) : 0u;
      }
    };
    uint32_t ra[2][2][NR], rb[2][2][NR];             // rows 0, 1 and 2, 3 of the window, in turn
    auto expand = [&](const uint32_t (&raw)[2][2], uint32_t (&v)[2][2][NR]) {
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const uint32_t e = __byte_perm(raw[r][c], 0u, 0x4140);
          if constexpr (IN8) {
            v[r][c][0] = e;
            v[r][c][1] = __byte_perm(raw[r][c], 0u, 0x4342);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[r][c][i] = e & (0x00030003u << (2 * i));
          }
        }
    };
    uint8_t* dst = a.y + ((size_t)((size_t)img * a.pho + y0) * a.pwo + X) * rowb;
    // one pooled row: `top` the first two input rows, the next two expanded into `bot`
    auto row = [&](const uint32_t (&top)[2][2][NR], uint32_t (&bot)[2][2][NR], uint32_t (&raw)[2][2], bool more) {
      expand(raw, bot);
      if (more) load(raw);
      float d[2][NT][4];
#pragma unroll
      for (int py = 0; py < 2; ++py)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) d[py][j][i] = 0.0f;
#pragma unroll
      for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int q = 0; q < KS; ++q)
#pragma unroll
          for (int py = 0; py < 2; ++py) {
            const int r = py + dy;
            auto v = [&](int c, int i) { return r < 2 ? top[r & 1][c][i] : bot[r & 1][c][i]; };
#pragma unroll
            for (int j = 0; j < NT; ++j)
              mma_f16(d[py][j], v(0, 2 * q), v(1, 2 * q), v(0, 2 * q + 1), v(1, 2 * q + 1), b[j][KS * dy + q]);
          }
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        float f = 0.0f;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float m = fmaxf(fmaxf(d[0][j][c], d[0][j][c + 2]), fmaxf(d[1][j][c], d[1][j][c + 2]));
          const float4 v = th[j][c];
          const float code = sat_fma(m, v.w, v.x) + sat_fma(m, v.w, v.y) + sat_fma(m, v.w, v.z);
          f = fmaf(code, c ? s1 : s0, f);
        }
        f += __shfl_xor_sync(0xffffffffu, f, 1);
        f += __shfl_xor_sync(0xffffffffu, f, 2);
        const uint32_t bits = __float_as_uint(f + 8388608.0f);   // 8 codes in the low 16 bits
        if (t == 0 && X < a.pwo) {
          if ((a.cout & 7) == 0) {
            *(uint16_t*)(dst + 2 * j) = (uint16_t)bits;
          } else {
            if (2 * j < rowb) dst[2 * j] = (uint8_t)bits;
            if (2 * j + 1 < rowb) dst[2 * j + 1] = (uint8_t)(bits >> 8);
          }
        }
      }
      dst += (size_t)a.pwo * rowb;
    };
    load(qb);
    load(qa);
    expand(qb, ra);
    load(qb);
#pragma unroll 1
    for (int y = 0; y < ny; y += 2) {
      row(ra, rb, qa, y + 2 < ny);
      if (y + 1 < ny) row(rb, ra, qb, y + 3 < ny);
    }
  }
}

}  // namespace ifq
