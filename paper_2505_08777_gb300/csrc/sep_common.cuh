// Separable tile transforms: shared layout, parameter blocks and device pieces.
//
// Over a 32 x 32 pixel tile a basis of total degree <= 4 gives every spot a
// phase that is a polynomial of degree <= 4 in the pixel's offsets
// u = (col - 16) / 16, v = (row - 16) / 16 from the tile's pixel (16, 16):
//
//   C_n . Z = 2 pi (base + px(u) + py(v)) + r(u, v),
//   r(u, v) = u R1(v) + u^2 R2(v) + u^3 R3(v),   R_k(0) = 0.
//
// px and py (tilts, defocus, the pure powers) can be of any size; r holds
// only the mixed terms, which over one tile are small. So the kernel
// factors, exp(-i C.Z) = Y(v) X(u) exp(-i r), and with exp(-i r) as a cubic
// in u (its coefficients Q_k are polynomials of R1 .. R3 per row) the sum
// over a tile's pixels is
//
//   sum_v Y(v) sum_k Q_k(v) [ sum_u X(u) u^k f(u, v) ],
//
// where the bracket is a matrix product over the tile's columns: it runs on
// the tensor cores (tcgen05, kind::f16, fp32 accumulators in TMEM), and a
// (spot, tile) pair costs 32 + 32 sine / cosine pairs instead of 1024.
//
// fp32 accuracy from f16 operands (split-f16): every operand value |x| <= 1
// is x = hi + lo with hi on the grid 2^-11 (exact in f16) and lo = f16(x -
// hi), so that |x - hi - lo| <= 2^-25; the product is hi hi + hi lo + lo hi.
// The nearfield is scaled by a power of two per tile to meet |x| <= 1.
#pragma once

#include "common.cuh"
#include "sep_launch.h"
#include "tc_common.cuh"
#include "tc_launch.h"

namespace ash {

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\t"
      "mov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\t"
      "mov.b64 rb, {%4, %5};\n\t"
      "sub.rn.f32x2 rd, ra, rb;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// hi of the split: x rounded to the grid 2^-11 (adding 1.5 * 2^12 leaves no
// finer bits), for |x| <= 1.
__device__ __forceinline__ float2 split_hi2(float2 x) {
  return sub2(add2(x, dup2(6144.0f)), dup2(6144.0f));
}
// (a, b) as a pair of f16, a in the low half.
__device__ __forceinline__ uint32_t pack_f16(float a, float b) {
  uint32_t d;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
  return d;
}

// mbar_wait with a suspend time (ns) for each poll, so that waiting warps leave
// the issue slots to the others; at most about a second in all.
constexpr uint32_t kSepWaitPolls = 1u << 20, kSepWaitNs = 1000;
__device__ __forceinline__ bool sep_wait(uint64_t* bar, uint32_t parity) {
  uint32_t done = 0;
  for (uint32_t it = 0; it < kSepWaitPolls; ++it) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity), "r"(kSepWaitNs)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Instruction descriptor of kind::f16 with f16 operands and an fp32
// accumulator, both operands K-major, shape M x N.
__host__ __device__ constexpr uint32_t umma_idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate));
}

// 8 consecutive fp32 columns of this thread's TMEM lane, without waiting.
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// Byte offset of the 16-byte chunk c (0..7) of row r in a K-major operand of
// 128-byte rows (64 f16) with the 128-byte swizzle.
__device__ __forceinline__ uint32_t swz_chunk(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

// A (tile, spot)'s phase polynomial as stored by k_sep_params, in the pixel
// offsets mx = col - 16, my = row - 16 from the tile's pixel (16, 16).
struct SepPoly {
  float base;                  // at that pixel, turns, about [-1/2, 1/2]
  float ax, ay;                // turns per pixel along columns and rows,
  float axl, ayl;              // and what their rounding left, radians
  float x2, x3, x4;            // mx^2, mx^3, mx^4, radians
  float y2, y3, y4;            // my^2, my^3, my^4, radians
  // mixed terms u^k my^l (u = mx / 16), radians; n31 negated
  float c11, c21, c12, c22, n31, c13;
};

__device__ __forceinline__ uint32_t pack_bf16_rz(float lo, float hi) {
  return (__float_as_uint(lo) >> 16) | (__float_as_uint(hi) & 0xffff0000u);
}

// Words of a spot's polynomial: word k of the 32 spots of a chunk are 32
// consecutive floats.
enum SepWord : int { kWBase, kWAx, kWAy, kWLow, kWX2, kWX3, kWX4, kWY2, kWY3, kWY4, kWC11, kWC21, kWC12, kWC22, kWN31,
                     kWC13 };
__device__ __forceinline__ SepPoly sep_unpack(const float* w) {
  SepPoly p;
  p.base = w[32 * kWBase];
  p.ax = w[32 * kWAx];
  p.ay = w[32 * kWAy];
  const uint32_t lo = __float_as_uint(w[32 * kWLow]);
  p.axl = __uint_as_float(lo << 16);
  p.ayl = __uint_as_float(lo & 0xffff0000u);
  p.x2 = w[32 * kWX2];
  p.x3 = w[32 * kWX3];
  p.x4 = w[32 * kWX4];
  p.y2 = w[32 * kWY2];
  p.y3 = w[32 * kWY3];
  p.y4 = w[32 * kWY4];
  p.c11 = w[32 * kWC11];
  p.c21 = w[32 * kWC21];
  p.c12 = w[32 * kWC12];
  p.c22 = w[32 * kWC22];
  p.n31 = w[32 * kWN31];
  p.c13 = w[32 * kWC13];
  return p;
}

// sin and cos of two angles through the MUFU. Its error is a phase error of
// -7.5e-8 of the angle (besides the random part). The tilt and the base are
// reduced to [-pi, pi], the pure powers over a tile are not: they are far below
// 1 for ordinary aberrations, and with 1400 rad of defocus on 300^2 (70 rad) the
// forward is 8.8e-7 off, where the kernels of one sine and cosine per term are
// 1.2e-5 (at 20 rad 3.8e-7 and 2.2e-6). FP32 polynomials (rms 3.5e-8) in place of
// the MUFU bring the adjoint from 3.1e-7 to 2.9e-7 and cost it 4 to 12 %.
__device__ __forceinline__ void cis2(float2 x, float2& c, float2& s) {
  s.x = __sinf(x.x);
  c.x = __cosf(x.x);
  s.y = __sinf(x.y);
  c.y = __cosf(x.y);
}

// The angles 2 pi (a m + b) + m (al + q2 m + q3 m^2 + q4 m^3), less whole turns
// of a m + b, for two values each; a m less an integer is exact. b is in
// turns, |b| <= 1.
__device__ __forceinline__ float2 sep_angle(float2 a, float2 al, float2 q2, float2 q3, float2 q4, float2 b, float2 m) {
  const float2 k = sub2(dup2(12582912.0f), add2(fma2(a, m, b), dup2(12582912.0f)));   // -rint(a m + b)
  const float2 r = add2(fma2(a, m, k), b);
  const float2 q = fma2(fma2(fma2(q4, m, q3), m, q2), m, al);
  return fma2(r, dup2(6.283185307179586f), mul2(q, m));
}
// The same with b = 0.
__device__ __forceinline__ float2 sep_angle(float2 a, float2 al, float2 q2, float2 q3, float2 q4, float2 m) {
  const float2 k = sub2(dup2(12582912.0f), fma2(a, m, dup2(12582912.0f)));
  const float2 r = fma2(a, m, k);
  const float2 q = fma2(fma2(fma2(q4, m, q3), m, q2), m, al);
  return fma2(r, dup2(6.283185307179586f), mul2(q, m));
}

// cos and sin of 2 pi r, |r| <= 1/2 and a little, on the FP32 pipe. With the
// zeros taken out, sin = r (1/4 - u) P(u) and cos = (1 - 16 u) Q(u), u = r^2, P
// and Q are polynomials of degree 5 and 6 without cancellation
// (gen_sincos_poly.py): at most 2.2e-7 and rms 4.8e-8 off, and the cosine 5e-10 on
// average over a turn.
__device__ constexpr float kSepSin[6] = {2.513274193e+01f, -6.483582306e+01f, 6.707675934e+01f, -3.849846649e+01f, 1.406576729e+01f,
                                        -3.193897486e+00f};
__device__ constexpr float kSepCos[7] = {1.000000000e+00f, -3.739208698e+00f, 5.112048626e+00f, -3.663868427e+00f, 1.620155334e+00f,
                                        -4.817714989e-01f, 9.075499326e-02f};
__device__ __forceinline__ void cis2_turns(float2 r, float2& c, float2& s) {
  const float2 u = mul2(r, r);
  float2 P = fma2(u, dup2(kSepSin[5]), dup2(kSepSin[4]));
  float2 Q = fma2(fma2(u, dup2(kSepCos[6]), dup2(kSepCos[5])), u, dup2(kSepCos[4]));
#pragma unroll
  for (int k = 3; k >= 0; --k) {
    P = fma2(P, u, dup2(kSepSin[k]));
    Q = fma2(Q, u, dup2(kSepCos[k]));
  }
  s = mul2(mul2(r, sub2(dup2(0.25f), u)), P);
  c = mul2(fma2(u, dup2(-16.0f), dup2(1.0f)), Q);
}

// Offset my of a strip's middle row (0 for the whole tile).
__device__ __forceinline__ float strip_mid(int s, int ls) {
  const int n = 32 >> ls;
  return ls == 0 ? 0.0f : (float)(s * n - 16) + 0.5f * (float)(n - 1);
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Two values split into f16 pairs (hi, lo).
__device__ __forceinline__ void split_pack(float2 v, uint32_t& hi, uint32_t& lo) {
  const float2 h = split_hi2(v), l = sub2(v, h);
  hi = pack_f16(h.x, h.y);
  lo = pack_f16(l.x, l.y);
}

// A spot's column polynomials about a strip's middle row (the mixed terms
// there are phases of the column part).
struct SepColumns {
  float ax, axl, x2, x3, x4;
};
__device__ __forceinline__ SepColumns sep_columns(const SepPoly& q, int s, int ls) {
  SepColumns o{q.ax, q.axl, q.x2, q.x3, q.x4};
  if (ls) {
    const float ms = strip_mid(s, ls);
    const float R1 = ms * (q.c11 + ms * (q.c12 + ms * q.c13)), R2 = ms * (q.c21 + ms * q.c22), n3 = ms * q.n31;
    const float d = R1 * (0.15915494309189535f * 0.0625f);
    const float a = __fadd_rn(q.ax, d), z = __fsub_rn(a, q.ax);
    o.axl = fmaf(__fadd_rn(__fsub_rn(q.ax, __fsub_rn(a, z)), __fsub_rn(d, z)), 6.283185307179586f, q.axl);
    o.ax = a;
    o.x2 = fmaf(R2, 0.0625f * 0.0625f, q.x2);
    o.x3 = fmaf(n3, -0.0625f * 0.0625f * 0.0625f, q.x3);
  }
  return o;
}

// The exponent e by which values are scaled to |x| <= 1: the largest, with the
// bits mx, is below 2^e. Over the whole range of floats (from 2^127 on |x| < 2, the
// split a bit coarser); 2^-127 is the subnormal 0x00400000.
__device__ __forceinline__ int sep_exponent(uint32_t mx) { return min(max((int)(mx >> 23), 0), 253) - 126; }
__device__ __forceinline__ float pow2_up(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }
__device__ __forceinline__ float pow2_down(int e) {
  return __uint_as_float(e == 127 ? 0x00400000u : (uint32_t)(127 - e) << 23);
}

// y of the 32 spots of a chunk divided by a power of two (scale), so that
// |y| <= 1: the 32 real, then the 32 imaginary parts; by one warp.
__device__ __forceinline__ void sep_scale_chunk(const float2* __restrict__ y, int N, int c, float* __restrict__ ys,
                                                float* __restrict__ scale) {
  const int lane = threadIdx.x & 31, n = c * 32 + lane;
  const float2 v = n < N ? __ldg(y + n) : make_float2(0.0f, 0.0f);
  const int e = sep_exponent(__reduce_max_sync(0xffffffffu, __float_as_uint(hypotf(v.x, v.y))));
  const float inv = pow2_down(e);
  ys[c * 64 + lane] = v.x * inv;
  ys[c * 64 + 32 + lane] = v.y * inv;
  if (lane == 0) scale[c] = pow2_up(e);
}

}  // namespace ash
