// Separable forward transform (see sep_common.cuh): the tables it works from,
// the kernel and the sum of its CTAs' partial fields.
#include <type_traits>

#include "sep_common.cuh"

namespace ash {

namespace {

// --- tables ---------------------------------------------------------------------

// One thread per (tile, mode): sum coef x^a y^b about pixel (16, 16) in fp64.
__global__ void k_sep_table(const Geometry G, const MonoTerm* __restrict__ terms, const int* __restrict__ term_off,
                            float* __restrict__ tab) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)G.T * G.D) return;
  const int d = (int)(e % G.D), tile = (int)(e / G.D);
  const double R = grid_radius(G);
  const double xc = grid_x(G, (double)((tile % G.tiles_x) * kTileX) + 16.0);
  const double yc = grid_y(G, (double)((tile / G.tiles_x) * kTileY) + 16.0);
  double b[5][5] = {};
  for (int t = term_off[d]; t < term_off[d + 1]; ++t) {
    const MonoTerm m = terms[t];
    // coefficients of (xc + x)^px and (yc + y)^py
    double fx[5], fy[5];
    auto expand = [](int n, double c, double* f) {
      for (int k = 0; k <= 4; ++k) f[k] = 0.0;
      double binom = 1.0;
      for (int k = 0; k <= n && k <= 4; ++k) {
        double p = binom;
        for (int q = 0; q < n - k; ++q) p *= c;
        f[k] = p;
        binom = binom * (n - k) / (k + 1);
      }
    };
    expand(m.px, xc, fx);
    expand(m.py, yc, fy);
    for (int k = 0; k <= 4; ++k)
      for (int l = 0; k + l <= 4; ++l) b[k][l] += m.coef * fx[k] * fy[l];
  }
  const double turn = 0.15915494309189533576888376337251, s = 16.0 / R;
  double pw[5] = {1.0, s, s * s, s * s * s, s * s * s * s};
  float* o = tab + (size_t)e * kSepTab;
  const double hl[3] = {b[0][0] * turn, b[1][0] * turn / R, b[0][1] * turn / R};
  for (int k = 0; k < 3; ++k) {
    o[2 * k] = (float)hl[k];
    o[2 * k + 1] = (float)(hl[k] - (double)o[2 * k]);
  }
  o[6] = (float)(b[2][0] * pw[2] * turn);
  o[7] = (float)(b[3][0] * pw[3] * turn);
  o[8] = (float)(b[4][0] * pw[4] * turn);
  o[9] = (float)(b[0][2] * pw[2] * turn);
  o[10] = (float)(b[0][3] * pw[3] * turn);
  o[11] = (float)(b[0][4] * pw[4] * turn);
  // mixed terms in radians
  o[12] = (float)(b[1][1] * pw[2]);
  o[13] = (float)(b[2][1] * pw[3]);
  o[14] = (float)(b[1][2] * pw[3]);
  o[15] = (float)(b[2][2] * pw[4]);
  o[16] = (float)(b[3][1] * pw[4]);
  o[17] = (float)(b[1][3] * pw[4]);
}

// acc (hi, lo) += c (bh + bl), with the rounding errors of the product and
// the sum kept in lo.
__device__ __forceinline__ void acc_hl(float& hi, float& lo, float c, float bh, float bl) {
  const float p = __fmul_rn(c, bh);
  const float e = __fmaf_rn(c, bl, __fmaf_rn(c, bh, -p));
  const float s = __fadd_rn(hi, p);
  const float z = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(e, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, z)), __fsub_rn(p, z))));
  hi = s;
}

// CTA (tile, block): thread = spot. Bound: the table is read once per CTA
// from shared memory and 64 B per (tile, spot) are written.
__global__ void __launch_bounds__(kSepSpots) k_sep_params(const Geometry G, const float* __restrict__ tab,
                                                          const float* __restrict__ coeff, float* __restrict__ poly,
                                                          unsigned char* __restrict__ strips, int npad) {
  __shared__ float st[kMaxModes * kSepTab];
  __shared__ int sred[4];
  const int tile = blockIdx.x, b = blockIdx.y, t = threadIdx.x, D = G.D;
  for (int k = t; k < D * kSepTab; k += kSepSpots) st[k] = __ldg(tab + (size_t)tile * D * kSepTab + k);
  __syncthreads();
  const int n = b * kSepSpots + t;
  float base = 0.0f, axh = 0.0f, axl = 0.0f, ayh = 0.0f, ayl = 0.0f;
  float q[12] = {};
  if (n < G.N) {
    for (int d = 0; d < D; ++d) {
      const float c = __ldg(coeff + (size_t)n * D + d);
      const float* o = st + d * kSepTab;
      // base: every product and sum reduced modulo one turn (base_turns)
      const float p = __fmul_rn(c, o[0]);
      const float e = __fmaf_rn(c, o[0], -p);
      const float r = __fsub_rn(p, rint_fma_pipe(p));
      base = __fadd_rn(base, __fadd_rn(r, __fmaf_rn(c, o[1], e)));
      base = __fsub_rn(base, rint_fma_pipe(base));
      acc_hl(axh, axl, c, o[2], o[3]);
      acc_hl(ayh, ayl, c, o[4], o[5]);
#pragma unroll
      for (int k = 0; k < 12; ++k) q[k] = __fmaf_rn(c, o[6 + k], q[k]);
    }
    const float x = __fadd_rn(axh, axl), y = __fadd_rn(ayh, ayl);
    axl = __fsub_rn(axl, __fsub_rn(x, axh));
    ayl = __fsub_rn(ayl, __fsub_rn(y, ayh));
    axh = x;
    ayh = y;
  }
  // per pixel offset (u = mx / 16, v = my / 16); the powers in radians
  constexpr float tp = 6.283185307179586f, h = 0.0625f;
  float* o = poly + ((size_t)tile * (npad / 32) + (n >> 5)) * 512 + (n & 31);
  o[32 * kWBase] = base;
  o[32 * kWAx] = axh;
  o[32 * kWAy] = ayh;
  o[32 * kWLow] = __uint_as_float(pack_bf16_rz(tp * axl, tp * ayl));
  o[32 * kWX2] = tp * q[0] * (h * h);
  o[32 * kWX3] = tp * q[1] * (h * h * h);
  o[32 * kWX4] = tp * q[2] * (h * h * h * h);
  o[32 * kWY2] = tp * q[3] * (h * h);
  o[32 * kWY3] = tp * q[4] * (h * h * h);
  o[32 * kWY4] = tp * q[5] * (h * h * h * h);
  o[32 * kWC11] = q[6] * h;
  o[32 * kWC21] = q[7] * h;
  o[32 * kWC12] = q[8] * (h * h);
  o[32 * kWC22] = q[9] * (h * h);
  o[32 * kWN31] = -q[10] * h;
  o[32 * kWC13] = q[11] * (h * h * h);
  // Row strips: the cubic in u takes u^4 R1^4 / 24 etc. as u^2 (off by at most
  // 1/4) and drops the rest; with 2^k strips R_k about a strip's middle row is
  // at most |dR_k/dv| / 2^k. The fewest strips that drop less than kSepTol.
  auto dropped = [](float R1, float R2, float R3) {
    const float s = R1 * R1;
    const float e4 = s * s * (1.0f / 24.0f) + 0.5f * s * R2 + 0.5f * R2 * R2;
    const float e5 = s * s * R1 * (1.0f / 120.0f) + s * R1 * R2 * (1.0f / 6.0f) + 0.5f * R1 * R2 * R2 + 0.5f * s * R3 +
                     R2 * R3;
    return 0.25f * e4 + R1 * R3 + e5;
  };
  const float a11 = fabsf(q[6]), a21 = fabsf(q[7]), a12 = fabsf(q[8]), a22 = fabsf(q[9]), a31 = fabsf(q[10]),
              a13 = fabsf(q[11]);
  int k = 0;
  if (!(dropped(a11 + a12 + a13, a21 + a22, a31) <= kSepTol)) {
    float f = 0.5f;
    for (k = 1; k < 5; ++k, f *= 0.5f)
      if (dropped(f * (a11 + 2.0f * a12 + 3.0f * a13), f * (a21 + 2.0f * a22), f * a31) <= kSepTol) break;
  }
  k = __reduce_max_sync(0xffffffffu, k);
  if ((t & 31) == 0) sred[t >> 5] = k;
  __syncthreads();
  if (t == 0) strips[(size_t)tile * gridDim.y + b] = (unsigned char)max(max(sred[0], sred[1]), max(sred[2], sred[3]));
}

// Cost prefixes of the (tile, spot block) units, cost[u] .. cost[u + 1]: unit
// u runs 2^strips[u] forward steps (CTA 0), or the chunks of its spots in the
// adjoint (CTA 1; acost[U + 1]: the largest chunk). CTAs of 1024 threads.
__global__ void k_sep_scan(const unsigned char* __restrict__ strips, int U, int N, int nb, int* __restrict__ cost,
                           int* __restrict__ acost) {
  __shared__ int wsum[32], wmax[32];
  const bool adj = blockIdx.x == 1;
  int* out = adj ? acost : cost;
  const int t = threadIdx.x, per = (U + 1023) / 1024;
  const int a = min(U, t * per), b = min(U, a + per);
  auto of = [&](int u) {
    const int ls = strips[u];
    return adj ? sep_chunks(N, u % nb) * sep_chunk_cost(ls) : sep_step_cost(ls) << ls;
  };
  int sum = 0, most = 0;
  for (int u = a; u < b; ++u) {
    sum += of(u);
    most = max(most, (int)strips[u]);
  }
  most = __reduce_max_sync(0xffffffffu, most);
  int inc = sum;
  for (int h = 1; h < 32; h <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, inc, h);
    if ((t & 31) >= h) inc += v;
  }
  if ((t & 31) == 31) {
    wsum[t >> 5] = inc;
    wmax[t >> 5] = most;
  }
  __syncthreads();
  if (t < 32) {
    int v = wsum[t];
    for (int h = 1; h < 32; h <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, v, h);
      if (t >= h) v += x;
    }
    wsum[t] = v;
    most = __reduce_max_sync(0xffffffffu, wmax[t]);
    if (adj && t == 0) out[U + 1] = sep_chunk_cost(most);
  }
  __syncthreads();
  int acc = inc - sum + (t >= 32 ? wsum[(t >> 5) - 1] : 0);
  for (int u = a; u < b; ++u) {
    out[u] = acc;
    acc += of(u);
  }
  if (t == 1023) out[U] = acc;
}

// --- forward --------------------------------------------------------------------

// One CTA per SM, 20 warps in three roles. The generators (warps 8-15)
// prepare the steps' operands, the summers (warps 0-7) read the results, one
// thread (warp 17) lists the steps and fetches their phase polynomials, and
// two (warps 16, 18) issue the MMAs of every second step each (issuing and its
// waits take longer than the MMAs themselves). A step: A = X(u) of 128 spots, rows [Re X(0..31) | Im X(0..31)];
// B = the tile's nearfield times u^k, k = 0..3, rows (k / 2, row pair, k % 2,
// re / im, row of the pair), [Re f | -Im f] and [Im f | Re f]. D[spot][256]
// then holds the four complex sums of every tile row, to which the summers
// apply Q_k(v) and Y(v). The low parts of the operands enter for k = 0, 1
// only: |Q_2|, |Q_3| < 0.01. A, B and D have two buffers each, so the
// generators, the tensor core and the summers work on different steps.
//
// Bound: the FP32 pipe, about 2100 clocks of a 3600-clock step (128 spots of a
// tile, one strip) against 1024 of tensor core and 1400 of shared memory; at
// 1024^2, N = 1024: FMA pipe 58 % busy, issue 56 %, tensor core 27 %, DRAM 9 %.
// The rest is the hand-over between the roles. Kernel times, before (one
// sine and cosine per term) / now: 1024^2 N = 400 252 / 60 us, 1024^2 N = 1024
// 571 / 104, 1920 x 1152 N = 2000 2365 / 430. Two uniform CTAs per SM took 75
// (540), one uniform CTA with lookahead 92 (858), MMAs issued by a generator 74.
constexpr int kFwdThreads = 640;
// Registers: 20 warps launch with 96 a thread; the summers take 120, the
// generators keep 96, the last warpgroup drops to 40.
static_assert(2 * 120 + 2 * 96 + 40 <= 5 * 96);
constexpr uint32_t kFA = 16384, kFB = 32768, kFBlo = 16384, kFSlot = 4 * 2048;
constexpr uint32_t kFwdBuf = kFB + kFBlo;                            // one B buffer
constexpr size_t kFwdB = 4 * kFA, kFwdSlots = kFwdB + 2 * kFwdBuf;   // slots: phase polynomials of 128 spots, 4 steps
constexpr size_t kFwdTail = kFwdSlots + 4 * kFSlot;                  // barriers, TMEM slot, maxima, step records
constexpr size_t kFwdSmem = 1024 + kFwdTail + 256;

// A step: spot block b (-1: no more steps) of a tile, strip s of 2^ls, and the
// B buffer that holds (or is to hold) the tile.
struct SepStep {
  int tile, b, s, ls, bb;
};

// The tensor core's fp32 accumulator truncates: measured over 256^2 to
// 1920 x 1152 pixels, fields came out smaller by 1.9e-7 of themselves whatever
// the input (phases 1.83e-7 to 2.2e-7, random fields 1.6e-7 to 1.8e-7), and by
// 5e-8 at random; 2.8e-7 with the pixel phases of a loop. This makes up for the
// first.
constexpr float kTruncation = 1.9e-7f, kTruncationLoop = 1.0f + 2.4e-7f;

// Sums over row pairs of c Tr, s Ti, c Ti, s Tr, with Y = c - i s.
struct SepSum {
  float2 cr, si, ci, sr;
  __device__ __forceinline__ void zero() { cr = si = ci = sr = make_float2(0.0f, 0.0f); }
};

// acc += Y(v) sum_k Q_k(v) D_k(v) over one pair of rows, offsets m; x and z
// hold D_0, D_1 and D_2, D_3 of the pair (re, im; both rows). `one` >= 0: only
// that row of the pair counts.
__device__ __forceinline__ void sep_sum_pair(const SepPoly& q, float R1s, float R2s, float n3s, const uint32_t* x,
                                             const uint32_t* z, float2 m, int one, SepSum& acc) {
  auto D = [](const uint32_t* a, int i) { return make_float2(__uint_as_float(a[2 * i]), __uint_as_float(a[2 * i + 1])); };
  const float2 R1 = fma2(fma2(fma2(dup2(q.c13), m, dup2(q.c12)), m, dup2(q.c11)), m, dup2(-R1s));
  const float2 R2 = fma2(fma2(dup2(q.c22), m, dup2(q.c21)), m, dup2(-R2s));
  const float2 n3 = fma2(dup2(q.n31), m, dup2(-n3s));   // -R3
  // exp(-i r) = 1 - i R1 u + q2 u^2 + q3 u^3, with the u^4 term taken as u^2
  const float2 n1 = sub2(make_float2(0.0f, 0.0f), R1), s = mul2(R1, R1);
  const float2 q2r = fma2(s, fma2(s, dup2(1.0f / 24.0f), dup2(-0.5f)), mul2(R2, mul2(R2, dup2(-0.5f))));
  const float2 q2i = mul2(R2, fma2(s, dup2(0.5f), dup2(-1.0f)));
  const float2 q3r = mul2(n1, R2), q3i = fma2(mul2(R1, s), dup2(1.0f / 6.0f), n3);
  const float2 ur = fma2(q3i, D(z, 3), mul2(q2i, D(z, 1)));
  float2 Tr = fma2(q3r, D(z, 2), fma2(q2r, D(z, 0), fma2(R1, D(x, 3), D(x, 0))));
  Tr = sub2(Tr, ur);
  float2 Ti = fma2(q2r, D(z, 1), fma2(n1, D(x, 2), D(x, 1)));
  Ti = fma2(q3r, D(z, 3), fma2(q3i, D(z, 2), fma2(q2i, D(z, 0), Ti)));
  float2 c, sn;
  cis2(sep_angle(dup2(q.ay), dup2(q.ayl), dup2(q.y2), dup2(q.y3), dup2(q.y4), dup2(q.base), m), c, sn);
  if (one >= 0) {
    const float2 w = one ? make_float2(0.0f, 1.0f) : make_float2(1.0f, 0.0f);
    c = mul2(c, w);
    sn = mul2(sn, w);
  }
  acc.cr = fma2(c, Tr, acc.cr);
  acc.si = fma2(sn, Ti, acc.si);
  acc.ci = fma2(c, Ti, acc.ci);
  acc.sr = fma2(sn, Tr, acc.sr);
}

// The coefficient gradient runs on the same steps: the summers keep the 14
// moments of degree <= 4 of their spot instead of its field and fold them with
// the modes' tile polynomials once per (spot block, tile), so that its time is
// the summers' (FP32; 1024^2 N = 400 D = 10: 301 -> 146 us, N = 1024: 569 -> 236,
// before: a sine and cosine and 14 multiply-adds per term).
//
// Moments of a tile over its pixels, Im(conj(gE) f K) mx^k my^l summed: m0[l]
// (k = 0), m1, m2, m3.
struct SepMoments {
  float2 m0[5], m1[4], m2[3], m3[2];
  __device__ __forceinline__ void zero() {
    for (float2& v : m0) v = make_float2(0.0f, 0.0f);
    for (float2& v : m1) v = make_float2(0.0f, 0.0f);
    for (float2& v : m2) v = make_float2(0.0f, 0.0f);
    for (float2& v : m3) v = make_float2(0.0f, 0.0f);
  }
};

// The moments' share of one pair of rows (arguments as sep_sum_pair; g is
// dL/dE). u^k exp(-i r) keeps powers up to 3: u^4 counts as u^2 - 1/8, and
// what lies beyond is dropped (its factors b_dk Q_m are below 4e-6 of the
// largest basis values at the sides this serves).
__device__ __forceinline__ void sep_moment_pair(const SepPoly& q, float R1s, float R2s, float n3s, const uint32_t* x,
                                                const uint32_t* z, float2 m, int one, float2 g, SepMoments& acc) {
  auto D = [](const uint32_t* a, int i) { return make_float2(__uint_as_float(a[2 * i]), __uint_as_float(a[2 * i + 1])); };
  const float2 R1 = fma2(fma2(fma2(dup2(q.c13), m, dup2(q.c12)), m, dup2(q.c11)), m, dup2(-R1s));
  const float2 R2 = fma2(fma2(dup2(q.c22), m, dup2(q.c21)), m, dup2(-R2s));
  const float2 n3 = fma2(dup2(q.n31), m, dup2(-n3s));   // -R3
  const float2 n1 = sub2(make_float2(0.0f, 0.0f), R1), s = mul2(R1, R1);
  const float2 q2r = fma2(s, fma2(s, dup2(1.0f / 24.0f), dup2(-0.5f)), mul2(R2, mul2(R2, dup2(-0.5f))));
  const float2 q2i = mul2(R2, fma2(s, dup2(0.5f), dup2(-1.0f))), p2i = sub2(make_float2(0.0f, 0.0f), q2i);
  const float2 q3r = mul2(n1, R2), q3i = fma2(mul2(R1, s), dup2(1.0f / 6.0f), n3), p3i = sub2(make_float2(0.0f, 0.0f), q3i);
  const float2 d4r = fma2(D(x, 0), dup2(-0.125f), D(z, 0)), d4i = fma2(D(x, 1), dup2(-0.125f), D(z, 1));
  // conj(gE) Y
  float2 c, sn;
  cis2(sep_angle(dup2(q.ay), dup2(q.ayl), dup2(q.y2), dup2(q.y3), dup2(q.y4), dup2(q.base), m), c, sn);
  if (one >= 0) {
    const float2 w = one ? make_float2(0.0f, 1.0f) : make_float2(1.0f, 0.0f);
    c = mul2(c, w);
    sn = mul2(sn, w);
  }
  const float2 Gr = fma2(sn, dup2(-g.y), mul2(c, dup2(g.x))), Gi = fma2(sn, dup2(-g.x), mul2(c, dup2(-g.y)));
  const float2 mm = mul2(m, m), m3 = mul2(mm, m), m4 = mul2(mm, mm);
  {
    float2 Sr = fma2(R1, D(x, 3), D(x, 0)), Si = fma2(n1, D(x, 2), D(x, 1));
    Sr = fma2(q2r, D(z, 0), fma2(p2i, D(z, 1), Sr));
    Si = fma2(q2r, D(z, 1), fma2(q2i, D(z, 0), Si));
    Sr = fma2(q3r, D(z, 2), fma2(p3i, D(z, 3), Sr));
    Si = fma2(q3r, D(z, 3), fma2(q3i, D(z, 2), Si));
    const float2 P = fma2(Gr, Si, mul2(Gi, Sr));
    acc.m0[0] = add2(acc.m0[0], P);
    acc.m0[1] = fma2(P, m, acc.m0[1]);
    acc.m0[2] = fma2(P, mm, acc.m0[2]);
    acc.m0[3] = fma2(P, m3, acc.m0[3]);
    acc.m0[4] = fma2(P, m4, acc.m0[4]);
  }
  {
    float2 Sr = fma2(R1, D(z, 1), D(x, 2)), Si = fma2(n1, D(z, 0), D(x, 3));
    Sr = fma2(q2r, D(z, 2), fma2(p2i, D(z, 3), Sr));
    Si = fma2(q2r, D(z, 3), fma2(q2i, D(z, 2), Si));
    Sr = fma2(q3r, d4r, fma2(p3i, d4i, Sr));
    Si = fma2(q3r, d4i, fma2(q3i, d4r, Si));
    const float2 P = fma2(Gr, Si, mul2(Gi, Sr));
    acc.m1[0] = add2(acc.m1[0], P);
    acc.m1[1] = fma2(P, m, acc.m1[1]);
    acc.m1[2] = fma2(P, mm, acc.m1[2]);
    acc.m1[3] = fma2(P, m3, acc.m1[3]);
  }
  {
    float2 Sr = fma2(R1, D(z, 3), D(z, 0)), Si = fma2(n1, D(z, 2), D(z, 1));
    Sr = fma2(q2r, d4r, fma2(p2i, d4i, Sr));
    Si = fma2(q2r, d4i, fma2(q2i, d4r, Si));
    const float2 P = fma2(Gr, Si, mul2(Gi, Sr));
    acc.m2[0] = add2(acc.m2[0], P);
    acc.m2[1] = fma2(P, m, acc.m2[1]);
    acc.m2[2] = fma2(P, mm, acc.m2[2]);
  }
  {
    const float2 Sr = fma2(R1, d4i, D(z, 2)), Si = fma2(n1, d4r, D(z, 3));
    const float2 P = fma2(Gr, Si, mul2(Gi, Sr));
    acc.m3[0] = add2(acc.m3[0], P);
    acc.m3[1] = fma2(P, m, acc.m3[1]);
  }
}

// The row pairs [p0, p0 + np) of D at TMEM address ta.
__device__ __forceinline__ void sep_moment_rows(const SepPoly& q, float ms, uint32_t ta, int p0, int np, int one,
                                                float2 g, SepMoments& acc) {
  const float R1s = ms * (q.c11 + ms * (q.c12 + ms * q.c13)), R2s = ms * (q.c21 + ms * q.c22), n3s = ms * q.n31;
  for (int k = 0; k < np; ++k) {
    uint32_t x[8], z[8];
    tmem_ld8_nowait(ta + (uint32_t)((p0 + k) * 8), x);
    tmem_ld8_nowait(ta + (uint32_t)(128 + (p0 + k) * 8), z);
    tmem_wait();
    const float m0 = (float)(2 * (p0 + k) - 16);
    sep_moment_pair(q, R1s, R2s, n3s, x, z, make_float2(m0, m0 + 1.0f), one, g, acc);
  }
}

// The row pairs [p0, p0 + np) of D at TMEM address ta (np 1 or even).
__device__ __forceinline__ void sep_sum_rows(const SepPoly& q, float ms, uint32_t ta, int p0, int np, int one,
                                             SepSum& acc) {
  const float R1s = ms * (q.c11 + ms * (q.c12 + ms * q.c13)), R2s = ms * (q.c21 + ms * q.c22), n3s = ms * q.n31;
  uint32_t x[16], z[16];
  if (np == 1) {
    tmem_ld8_nowait(ta + (uint32_t)(p0 * 8), x);
    tmem_ld8_nowait(ta + (uint32_t)(128 + p0 * 8), z);
    tmem_wait();
    const float m0 = (float)(2 * p0 - 16);
    sep_sum_pair(q, R1s, R2s, n3s, x, z, make_float2(m0, m0 + 1.0f), one, acc);
    return;
  }
  for (int k = 0; k < np; k += 2) {
    tmem_ld16_nowait(ta + (uint32_t)((p0 + k) * 8), x);
    tmem_ld16_nowait(ta + (uint32_t)(128 + (p0 + k) * 8), z);
    tmem_wait();
    const float m0 = (float)(2 * (p0 + k) - 16);
    sep_sum_pair(q, R1s, R2s, n3s, x, z, make_float2(m0, m0 + 1.0f), -1, acc);
    sep_sum_pair(q, R1s, R2s, n3s, x + 8, z + 8, make_float2(m0 + 2.0f, m0 + 3.0f), -1, acc);
  }
}

__device__ __forceinline__ void put16(uint8_t* base, int r, int c, const uint32_t (&v)[4], uint32_t flip = 0) {
  *reinterpret_cast<uint4*>(base + swz_chunk(r, c)) = make_uint4(v[0] ^ flip, v[1] ^ flip, v[2] ^ flip, v[3] ^ flip);
}

// GRAD: the moment pass dL/dC = Im(conj(gE_n) sum_m Z_dm f_m K_nm): the summers
// take moments of the same row sums over mx, my per tile and contract them with
// the tile's basis polynomials.
template <bool GRAD>
__global__ void __launch_bounds__(kFwdThreads, 1) k_sep_forward(const SepFwdParams p) {
  extern __shared__ uint8_t raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + kFwdTail);   // [2] MMAs of a step done
  uint64_t* empty = full + 2;                                    // [4] its D and slot read
  uint64_t* ready = full + 6;                                    // [4] its operands written
  uint64_t* listed = full + 10;                                  // [4] its record and polynomials written
  uint32_t* slot = reinterpret_cast<uint32_t*>(full + 14);
  uint32_t* smax = slot + 2;                                     // [8]
  float* scales = reinterpret_cast<float*>(smax + 8);            // [4] 2^e of the steps' tiles
  SepStep* steps = reinterpret_cast<SepStep*>(scales + 4);       // [4]
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int row = t & 127, prow = (row >> 5) * 512 + (row & 31);   // the spot's place in a slot
  const int nb = p.nb, npad = nb * kSepSpots, U = p.g.T * nb;
  if (w == 0) tmem_alloc(slot, 512);
  if (t == 0) {
    for (int k = 0; k < 14; ++k) mbar_init(full + k, k >= 2 && k < 6 ? 8 : 1);
    fence_mbar_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  bool ok = true;
  pdl_begin();

  if (w < 8) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 120;");
    // --- summers: spot `row`, half of a step's row pairs ---
    const int half = t >> 7;
    float2* part = p.part + (size_t)(kSepFwdRows * blockIdx.x + half) * npad + row;
    const int D = p.g.D;
    float* dpart = p.dpart + (size_t)(kSepFwdRows * blockIdx.x + half) * D * npad + row;
    // no other thread touches these partial sums
    if constexpr (GRAD) {
      for (int k = 0; k < D * nb; ++k) dpart[(size_t)k * kSepSpots] = 0.0f;
    } else {
      for (int b = 0; b < nb; ++b) part[b * kSepSpots] = make_float2(0.0f, 0.0f);
    }
    const uint32_t tlane = tmem + ((uint32_t)((w & 3) * 32) << 16);
    std::conditional_t<GRAD, SepMoments, SepSum> acc;
    acc.zero();
    int pb = -1, pt = -1;   // block, tile and scale of the sums held
    float psc = 1.0f, pscale = 1.0f;
    float2 g = make_float2(0.0f, 0.0f);
    auto flush = [&]() {
      if constexpr (GRAD) {
        constexpr float tp = 6.283185307179586f, h = 0.0625f;
        auto S = [&](float2 v, float f) { return fmaf(v.x + v.y, kTruncation, v.x + v.y) * (f * pscale); };
        // in the table's units: turns for the pure powers, per pixel for the slopes
        const float a00 = S(acc.m0[0], tp), a01 = S(acc.m0[1], tp), a02 = S(acc.m0[2], tp * h * h),
                    a03 = S(acc.m0[3], tp * h * h * h), a04 = S(acc.m0[4], tp * h * h * h * h);
        const float a10 = S(acc.m1[0], tp * 16.0f), a20 = S(acc.m2[0], tp), a30 = S(acc.m3[0], tp);
        const float a40 = fmaf(a00, -0.125f, a20);
        const float a11 = S(acc.m1[1], h), a21 = S(acc.m2[1], h), a12 = S(acc.m1[2], h * h), a22 = S(acc.m2[2], h * h),
                    a31 = S(acc.m3[1], h), a13 = S(acc.m1[3], h * h * h);
        const float2* tb = reinterpret_cast<const float2*>(p.tab + (size_t)pt * D * kSepTab);
        for (int d = 0; d < D; ++d, tb += kSepTab / 2) {
          const float2 t0 = __ldg(tb), t1 = __ldg(tb + 1), t2 = __ldg(tb + 2), t3 = __ldg(tb + 3), t4 = __ldg(tb + 4),
                       t5 = __ldg(tb + 5), t6 = __ldg(tb + 6), t7 = __ldg(tb + 7), t8 = __ldg(tb + 8);
          float v = fmaf(t0.x, a00, fmaf(t0.y, a00, fmaf(t1.x, a10, t2.x * a01)));
          v = fmaf(t3.x, a20, fmaf(t3.y, a30, fmaf(t4.x, a40, fmaf(t4.y, a02, fmaf(t5.x, a03, fmaf(t5.y, a04, v))))));
          v = fmaf(t6.x, a11, fmaf(t6.y, a21, fmaf(t7.x, a12, fmaf(t7.y, a22, fmaf(t8.x, a31, fmaf(t8.y, a13, v))))));
          atomicAdd(dpart + (size_t)d * npad + pb * kSepSpots, v);
        }
      } else {
        float2* o = part + pb * kSepSpots;
        const float re = (acc.cr.x + acc.cr.y) + (acc.si.x + acc.si.y), im = (acc.ci.x + acc.ci.y) - (acc.sr.x + acc.sr.y);
        atomicAdd(&o->x, (p.exact ? fmaf(re, kTruncation, re) : re) * pscale);
        atomicAdd(&o->y, (p.exact ? fmaf(im, kTruncation, im) : im) * pscale);
      }
    };
    for (uint32_t it = 0;; ++it) {
      ok = ok && sep_wait(&ready[it & 3], (it >> 2) & 1);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const SepStep r = steps[it & 3];
      const float scale = scales[it & 3];
      if (r.b != pb || scale != psc || (GRAD && r.tile != pt)) {
        if (pb >= 0) flush();
        acc.zero();
        if (GRAD && r.b >= 0 && r.b != pb) {
          const int n = r.b * kSepSpots + row;
          g = n < p.g.N ? __ldg(p.gE + n) : make_float2(0.0f, 0.0f);
        }
        pb = r.b;
        pt = r.tile;
        pscale = p.exact ? scale : scale * kTruncationLoop;
        psc = scale;
      }
      if (r.b < 0) break;
      const SepPoly q = sep_unpack(reinterpret_cast<const float*>(sm + kFwdSlots + (it & 3) * kFSlot) + prow);
      const int rows = 32 >> r.ls, pairs = rows >= 2 ? rows >> 1 : 1;
      const int np = pairs >= 2 ? pairs >> 1 : (half ? 0 : 1), p0 = ((r.s * rows) >> 1) + half * np;
      ok = ok && sep_wait(&full[it & 1], (it >> 1) & 1);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const int one = rows == 1 ? (r.s & 1) : -1;
      if constexpr (GRAD) {
        sep_moment_rows(q, strip_mid(r.s, r.ls), tlane + 256u * (it & 1), p0, np, one, g, acc);
      } else {
        if (np > 0) sep_sum_rows(q, strip_mid(r.s, r.ls), tlane + 256u * (it & 1), p0, np, one, acc);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[it & 3]);
    }
  } else if (w >= 16) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if ((w == 16 || w == 18) && lane == 0) {
      // --- MMA issue: even or odd steps, into D buffer d ---
      const int d = (w - 16) >> 1;
      uint32_t it = (uint32_t)d;
      for (;; it += 2) {
        ok = ok && sep_wait(&listed[it & 3], (it >> 2) & 1);
        if (!ok) break;
        const SepStep r = steps[it & 3];
        if (r.b < 0) break;
        ok = ok && sep_wait(&ready[it & 3], (it >> 2) & 1);
        if (it >= 2) ok = ok && sep_wait(&empty[(it - 2) & 3], ((it - 2) >> 2) & 1);
        if (!ok) break;
        tc_fence_after();
        // the columns of the step's rows in each half of D (N >= 16)
        const int rows = 32 >> r.ls, p0 = (r.s * rows) >> 1;
        const int n = rows >= 4 ? rows * 4 : 16, col = (n == 16 ? (p0 & ~1) : p0) * 8;
        const uint32_t dst = tmem + (uint32_t)(256 * d + col), idesc = umma_idesc_f16(128, n);
        // (descriptors count 16-byte units)
        const uint64_t a = umma_desc(smem_u32(sm) + (uint32_t)d * 2 * kFA);
        const uint64_t b = umma_desc(smem_u32(sm + kFwdB) + (uint32_t)r.bb * kFwdBuf + (uint32_t)col * 128);
        // the small products first: the accumulator truncates every sum
        const uint64_t al = a + (kFA >> 4), bl = b + (kFB >> 4), b1 = b + 128 * 8;
#pragma unroll
        for (int ks = 0; ks < 8; ks += 2) {
          umma_f16(dst, al + ks, b + ks, idesc, ks > 0);
          umma_f16(dst, a + ks, bl + ks, idesc, 1u);
        }
        umma_f16(dst, a, b, idesc, 1u);
        umma_f16(dst + 128, a, b1, idesc, 0u);
        if (r.ls == 0) {
#pragma unroll
          for (int ks = 2; ks < 8; ks += 2) umma_f16(dst, a + ks, b + ks, umma_idesc_f16(128, 256), 1u);
        } else {
#pragma unroll
          for (int ks = 2; ks < 8; ks += 2) {
            umma_f16(dst, a + ks, b + ks, idesc, 1u);
            umma_f16(dst + 128, a + ks, b1 + ks, idesc, 1u);
          }
        }
        umma_commit(&full[d]);
      }
      // nothing in flight when the CTA gives up its memory
      if (it >= 2) ok = sep_wait(&full[d], ((it - 2) >> 1) & 1) && ok;
    } else if (w == 17 && lane == 0) {
      // --- steps of this CTA: those whose place in the cost prefix lies in [c0, c1) ---
      const long long W = p.cost[U];
      const int c0 = (int)(W * blockIdx.x / p.G), c1 = (int)(W * (blockIdx.x + 1) / p.G);
      int u = 0, hi = U - 1;
      while (u < hi) {
        const int mid = (u + hi + 1) / 2;
        if (p.cost[mid] <= c0) u = mid;
        else hi = mid - 1;
      }
      SepStep x{u / nb, u % nb, 0, p.strips[u], 0};
      int pos = p.cost[u], c = sep_step_cost(x.ls);
      x.s = (c0 - pos + c - 1) / c;
      pos += x.s * c;
      int ls1 = u + 1 < U ? p.strips[u + 1] : 0;   // of the next unit, fetched early
      uint32_t it = 0;
      for (;; ++it) {
        if (x.s >> x.ls) {
          ++u;
          x.s = 0;
          x.ls = ls1;
          c = sep_step_cost(ls1);
          if (++x.b == nb) {
            x.b = 0;
            ++x.tile;
            x.bb ^= 1;
          }
          if (u + 1 < U) ls1 = p.strips[u + 1];
        }
        const bool more = pos < c1;
        if (!more) {
          // an end for each of the two issuers
          for (uint32_t k = it; k < it + 2; ++k)
            if (k >= 4) ok = ok && sep_wait(&empty[k & 3], ((k >> 2) - 1) & 1);
          for (uint32_t k = it; ok && k < it + 2; ++k) {
            steps[k & 3] = SepStep{0, -1, 0, 0, 0};
            mbar_arrive(&listed[k & 3]);
          }
          break;
        }
        // slot it & 3 was step it - 4's
        if (it >= 4) ok = ok && sep_wait(&empty[it & 3], ((it >> 2) - 1) & 1);
        if (!ok) break;   // the slot may still be read
        steps[it & 3] = x;
        mbar_expect_tx(&listed[it & 3], kFSlot);
        bulk_g2s(sm + kFwdSlots + (it & 3) * kFSlot, p.poly + ((size_t)x.tile * nb + x.b) * (16 * kSepSpots), kFSlot,
                 &listed[it & 3]);
        pos += c;
        ++x.s;
      }
      // every copy has landed when the CTA gives up its memory (after the ends,
      // those of steps up to it - 3 have been read, and others' slots hold the ends)
      const uint32_t open = ok ? 2 : 4;
      for (uint32_t k = it > open ? it - open : 0; k < it; ++k) ok = sep_wait(&listed[k & 3], (k >> 2) & 1) && ok;
    }
    __syncwarp();
  } else {
    // --- generators: spot `row`, half of the columns ---
    const int g = t - 256, half = g >> 7;
    auto gen_sync = [&]() { asm volatile("bar.sync 1, 256;" ::: "memory"); };
    // B of a tile; returns the tile's scale 2^e (the nearfield is divided by it)
    auto build_b = [&](int tile, uint8_t* bh) -> float {
      // thread: tile row j, 8 columns from 8 c, powers u^(2 kh), u^(2 kh + 1)
      const int j = g >> 3, c = g & 3, kh = (g >> 2) & 1;
      const float4* f = p.fimg + ((size_t)tile * kTcChunksPerTile + (j >> 1)) * 32 + (j & 1) * 16 + c * 4;
      float4 v[4];
      float mx = 0.0f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        v[q] = __ldg(f + q);
        mx = fmaxf(mx, fmaxf(fabsf(v[q].x), fabsf(v[q].y)));
      }
      const uint32_t wm = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
      if (lane == 0) smax[g >> 5] = wm;
      gen_sync();
      uint32_t m = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) m = max(m, smax[q]);
      const int e = sep_exponent(m);
      const float inv = pow2_down(e);
      constexpr uint32_t S = 0x80008000u;
      // The pixels' phases, not through the MUFU: its cosine is on average 7.5e-8
      // off over a turn, which all pixels add up in a spot without tilt and
      // aberrations (random field of 1024^2, N = 19, the middle spot among them: 7e-6
      // of the norm, with the phase's turns as exact 4e-7; the times are the same).
      // Loops, whose spots are bright and which multiply any change of rounding,
      // keep it.
      float2 pc[4], ps[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 t = make_float2(v[q].z, v[q].w);
        if (p.exact) cis2_turns(t, pc[q], ps[q]);
        else cis2(mul2(t, dup2(6.283185307179586f)), pc[q], ps[q]);
      }
#pragma unroll
      for (int k2 = 0; k2 < 2; ++k2) {
        uint32_t rh[4], rl[4], ih[4], il[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 u = make_float2((float)(8 * c + 2 * q - 16) * 0.0625f, (float)(8 * c + 2 * q - 15) * 0.0625f);
          float2 a = mul2(make_float2(v[q].x, v[q].y), dup2(inv));
          if (kh) a = mul2(a, mul2(u, u));
          if (k2) a = mul2(a, u);
          split_pack(mul2(a, pc[q]), rh[q], rl[q]);
          split_pack(mul2(a, ps[q]), ih[q], il[q]);
        }
        const int r0 = kh * 128 + (j >> 1) * 8 + k2 * 4 + (j & 1);   // re row; im row is r0 + 2
        put16(bh, r0, c, rh);
        put16(bh, r0, 4 + c, ih, S);
        put16(bh, r0 + 2, c, ih);
        put16(bh, r0 + 2, 4 + c, rh);
        if (kh == 0) {
          put16(bh + kFB, r0, c, rl);
          put16(bh + kFB, r0, 4 + c, il, S);
          put16(bh + kFB, r0 + 2, c, il);
          put16(bh + kFB, r0 + 2, 4 + c, rl);
        }
      }
      return pow2_up(e);
    };

    // A: X(u) of this thread's spot for its 16 columns, about the strip's row
    auto build_a = [&](const float* sq, const SepStep& x, uint8_t* ah) {
      const SepPoly q = sep_unpack(sq);
      const SepColumns o = sep_columns(q, x.s, x.ls);
      // X = exp(-i angle): the negated angle's cosine and sine
#pragma unroll
      for (int c8 = 0; c8 < 2; ++c8) {
        uint32_t rh[4], rl[4], ih[4], il[4];
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) {
          const float m0 = (float)(16 * half - 16 + 8 * c8 + 2 * q2);
          float2 cs, sn;
          cis2(sep_angle(dup2(-o.ax), dup2(-o.axl), dup2(-o.x2), dup2(-o.x3), dup2(-o.x4), make_float2(m0, m0 + 1.0f)),
               cs, sn);
          split_pack(cs, rh[q2], rl[q2]);
          split_pack(sn, ih[q2], il[q2]);
        }
        const int c = 2 * half + c8;
        put16(ah, row, c, rh);
        put16(ah, row, 4 + c, ih);
        put16(ah + kFA, row, c, rl);
        put16(ah + kFA, row, 4 + c, il);
      }
    };

    float scale = 1.0f;
    int tile = -1;
    for (uint32_t it = 0;; ++it) {
      const int d = it & 1;
      ok = ok && sep_wait(&listed[it & 3], (it >> 2) & 1);
      // MMA(it - 2) done: its A, and B of an older tile, are free
      if (it >= 2) ok = ok && sep_wait(&full[d], ((it >> 1) - 1) & 1);
      // every generator goes on or none (they meet at a barrier)
      int stop;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.eq.s32 p, %1, 0;\n\tbarrier.red.or.pred q, 2, 256, p;\n\t"
          "selp.s32 %0, 1, 0, q;\n\t}"
          : "=r"(stop)
          : "r"((int)ok)
          : "memory");
      if (stop) break;
      const SepStep x = steps[it & 3];
      if (x.b < 0) {
        if (g == 0) mbar_arrive(&ready[it & 3]);
        break;
      }
      if (x.tile != tile) {
        tile = x.tile;
        scale = build_b(tile, sm + kFwdB + (uint32_t)x.bb * kFwdBuf);
      }
      build_a(reinterpret_cast<const float*>(sm + kFwdSlots + (it & 3) * kFSlot) + prow, x,
              sm + (uint32_t)d * 2 * kFA);
      fence_async_smem();
      if (g == 0) scales[it & 3] = scale;
      gen_sync();
      if (g == 0) mbar_arrive(&ready[it & 3]);
    }
  }
  if (!ok) atomicOr(p.err, kErrTimeout);
  tc_fence_before();
  __syncthreads();
  if (w == 0) tmem_dealloc(tmem, 512);
}

// dL/dC_nd = the sum of the CTAs' partial rows (as k_sep_forward_reduce).
__global__ void k_sep_gradc_reduce(const float* __restrict__ part, int rows, int npad, int N, int D,
                                   float* __restrict__ dC) {
  __shared__ float acc[16][33];
  pdl_begin();
  const int n = blockIdx.x * 32 + threadIdx.x, d = blockIdx.y, k = threadIdx.y;
  float v = 0.0f;
#pragma unroll 10
  for (int r = k; r < rows; r += 16) v += part[((size_t)r * D + d) * npad + n];
  acc[k][threadIdx.x] = v;
  __syncthreads();
  for (int h = 8; h > 0; h >>= 1) {
    if (k < h) acc[k][threadIdx.x] += acc[k + h][threadIdx.x];
    __syncthreads();
  }
  if (k == 0 && n < N) dC[(size_t)n * D + d] = acc[0][threadIdx.x];
}

// E_n = the sum of the CTAs' partial rows, in a fixed order: row-lane k of the
// 32 x 32 threads adds rows k, k + 32, ..., then a fixed-shape tree. Latency
// bound: 4.4 us for the 304 rows of N = 400 (1.2 MB from L2).
__global__ void k_sep_forward_reduce(const float2* __restrict__ part, int rows, int npad, int N,
                                     float2* __restrict__ E) {
  __shared__ float2 acc[32][33];
  pdl_begin();
  const int n = blockIdx.x * 32 + threadIdx.x, k = threadIdx.y;
  float2 v = make_float2(0.0f, 0.0f);
#pragma unroll 10
  for (int r = k; r < rows; r += 32) {
    const float2 x = part[(size_t)r * npad + n];
    v.x += x.x;
    v.y += x.y;
  }
  acc[k][threadIdx.x] = v;
  __syncthreads();
  for (int h = 16; h > 0; h >>= 1) {
    if (k < h) {
      acc[k][threadIdx.x].x += acc[k + h][threadIdx.x].x;
      acc[k][threadIdx.x].y += acc[k + h][threadIdx.x].y;
    }
    __syncthreads();
  }
  if (k == 0 && n < N) E[n] = acc[0][threadIdx.x];
}

}  // namespace

cudaError_t sep_build_table(const Geometry& g, const MonoTerm* terms, const int* term_off, float* tab,
                            cudaStream_t s) {
  const long long n = (long long)g.T * g.D;
  k_sep_table<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(g, terms, term_off, tab);
  return cudaGetLastError();
}

cudaError_t sep_build_params(const Geometry& g, const float* tab, const float* coeff, float* poly,
                             unsigned char* strips, int* cost, int* acost, cudaStream_t s) {
  const int nb = sep_blocks(g.N);
  k_sep_params<<<dim3(g.T, nb), kSepSpots, 0, s>>>(g, tab, coeff, poly, strips, nb * kSepSpots);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_sep_scan<<<2, 1024, 0, s>>>(strips, g.T * nb, g.N, nb, cost, acost);
  return cudaGetLastError();
}

cudaError_t sep_prepare() {
  cudaError_t e;
  for (const void* k : {(const void*)k_sep_forward<false>, (const void*)k_sep_forward<true>})
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFwdSmem))) return e;
  for (const void* k : {(const void*)k_sep_forward<false>, (const void*)k_sep_forward<true>,
                        (const void*)k_sep_forward_reduce, (const void*)k_sep_gradc_reduce, (const void*)k_sep_params,
                        (const void*)k_sep_scan})
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                  (int)cudaSharedmemCarveoutMaxShared)))
      return e;
  return cudaSuccess;
}

cudaError_t sep_launch_forward(const SepFwdParams& p, cudaStream_t s) {
  return launch_pdl(k_sep_forward<false>, p.G, kFwdThreads, kFwdSmem, s, p);
}

cudaError_t sep_launch_forward_reduce(const SepFwdParams& p, cudaStream_t s) {
  return launch_pdl(k_sep_forward_reduce, (p.g.N + 31) / 32, dim3(32, 32), 0, s, p.part, kSepFwdRows * p.G,
                    p.nb * kSepSpots, p.g.N, p.E);
}

cudaError_t sep_launch_gradc(const SepFwdParams& p, cudaStream_t s) {
  return launch_pdl(k_sep_forward<true>, p.G, kFwdThreads, kFwdSmem, s, p);
}

cudaError_t sep_launch_gradc_reduce(const SepFwdParams& p, cudaStream_t s) {
  return launch_pdl(k_sep_gradc_reduce, dim3((p.g.N + 31) / 32, p.g.D), dim3(32, 16), 0, s, p.dpart,
                    kSepFwdRows * p.G, p.nb * kSepSpots, p.g.N, p.g.D, p.dC);
}

}  // namespace ash
