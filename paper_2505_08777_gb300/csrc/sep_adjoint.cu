// Separable adjoint transform (see sep_common.cuh): over a tile
//
//   g(u, v) = sum_k u^k sum_n [y_n Y_n(v) Q_k,n(v)] X_n(u),
//
// the inner sum a matrix product over the spots. W = y Y Q_k and X are
// written by the warps as split-f16 operands; the tensor core contracts 32
// spots per step, and the partial products are added up in fp32 registers.
#include "sep_common.cuh"
#include "tc_epilogue.cuh"

namespace ash {

namespace {

// One CTA per SM, 28 warps. Warps 0-7 (adders): lane = tile row, warp w adds
// up half of the columns of the plane u^(w % 4); warp 8 lists the steps and
// fetches their spots, warps 9-11 issue the MMAs of every third step each (one
// issuer spent 2400 clocks a step, mostly on its waits: operands were always
// ready); warps 12-19 and 20-27
// (generators, taking turns step by step): two spots (in the halves of the
// packed operations), two tile rows and two tile columns each. A step is 32 spots of a tile and one strip of its
// rows (the strips of a chunk share W). A: rows (k, tile row), (Re W, Im W) of
// the 32 spots; low parts for k = 0, 1 only (|Q_2|, |Q_3| < 0.01). B: rows
// (column, re / im), (Re X, -Im X) and (Im X, Re X), high then low parts.
// D[128][128]: products with the high and with the low parts of X.
//
// Bound: the issue slots (67 % used; FMA pipe 49 %, tensor core 22 %, DRAM 4 % at
// 1024^2, N = 1024): a step, 32 spots of a tile and all its rows, takes the
// generators about 2000 clocks for 8192 values of W and 2048 of X. Kernel
// times, before (one sine and cosine per term) / now: 1024^2 N = 400 276 / 91
// us, 1920 x 1152 N = 2000 2656 / 828 (1024^2 N = 1024: 194). One group of 16
// generator warps took 157 (1266), two groups with one spot a thread 97 (884).
constexpr int kAdjThreads = 896;
// Registers: launched with 72 a thread; the adders keep 72, warps 8-11 drop
// to 40, the generators take 80.
static_assert(2 * 72 + 40 + 4 * 80 <= 7 * 72);
constexpr int kAdjBufs = 3, kAdjSlots = 8;
// Barriers of the steps' MMAs. A wait names a phase by its parity, so a barrier
// may not come round again before every waiter has seen it: the generators of
// step it wait for step it - 3, and nothing of step it holds back step it + 1
// (other generators, another issuer), which with one barrier per D buffer is
// that barrier's next phase. With eight it is step it + 5, whose sums go where
// step it + 1's were, read after step it's.
constexpr int kAdjFull = 8;
constexpr uint32_t kAA = 32768, kAB = 16384, kASlot = 2048 + 256;
constexpr uint32_t kAdjB = kAdjBufs * kAA, kAdjSum = kAdjB + kAdjBufs * kAB;   // sums of the planes: [4][32][33] float2
constexpr uint32_t kAdjSlot0 = kAdjSum + 4 * 32 * 33 * 8, kAdjTail = kAdjSlot0 + kAdjSlots * kASlot;
constexpr size_t kAdjSmem = 1024 + kAdjTail + 512;
static_assert(kAdjFull == 8 && (kAdjFull + 26) * 8 + 16 + kAdjSlots * 16 <= 512 && kAdjTail % 16 == 0);
static_assert(kAdjSum % 16 == 0 && kAdjSlot0 % 16 == 0 && kAdjTail % 8 == 0);

// A step's record, read as one 16-byte word.
struct __align__(16) AdjStep {
  int tile;        // negative: no more steps
  uint32_t bits;   // s | ls << 8 | a << 16 | end << 18: strip s of 2^ls, buffer of W
  int used;        // 2 (the last step that used that buffer before this chunk, or -1) + (that chunk had several strips)
  float scale;     // 2^e: y is divided by it
  __device__ int s() const { return (int)(bits & 255u); }
  __device__ int ls() const { return (int)(bits >> 8 & 255u); }
  __device__ uint32_t a() const { return bits >> 16 & 3u; }
  // bits: 1 the CTA's last step of this tile, 2 other CTAs have part of it, 4
  // it starts here, 8 the CTA's last step
  __device__ int end() const { return (int)(bits >> 18); }
};
__device__ __forceinline__ AdjStep adj_step(const AdjStep* p) {
  const int4 v = *reinterpret_cast<const int4*>(p);
  return AdjStep{v.x, (uint32_t)v.y, v.z, __int_as_float(v.w)};
}
__device__ __forceinline__ void put_step(AdjStep* p, int tile, uint32_t bits, int used, float scale) {
  *reinterpret_cast<int4*>(p) = make_int4(tile, (int)bits, used, __float_as_int(scale));
}

// (see kTruncation of the forward: here -1.5e-7)
constexpr float kAdjTruncation = 1.0f + 1.2e-7f;

template <int V>
struct IntTag {
  static constexpr int value = V;
};
template <int OFF>
__device__ __forceinline__ void sts64(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.u32 [%0 + %1], {%2, %3};" ::"r"(addr), "n"(OFF), "r"(a), "r"(b) : "memory");
}

// CTA whose range [W g / G, W (g + 1) / G) holds position c.
__device__ __forceinline__ int adj_owner(long long W, int G, int c) {
  int g = (int)((long long)c * G / W);
  while (g + 1 < G && W * (g + 1) / G <= c) ++g;
  while (g > 0 && W * g / G > c) --g;
  return g;
}

__global__ void __launch_bounds__(kAdjThreads, 1) k_sep_adjoint(const SepAdjParams p) {
  extern __shared__ uint8_t raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + kAdjTail);   // [8] MMAs of a step done
  uint64_t* empty = full + kAdjFull;                             // [8] its D and record read
  uint64_t* ready = empty + 8;                                   // [8] its operands written
  uint64_t* listed = ready + 8;                                  // [8] its record and spots written
  uint64_t* summed = listed + 8;                                 // the adders' meeting point at a tile's end
  uint32_t* slot = reinterpret_cast<uint32_t*>(summed + 2);
  AdjStep* steps = reinterpret_cast<AdjStep*>(slot + 4);         // [8]
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int N = p.a.g.N, nb = p.nb, npad = nb * kSepSpots, U = p.a.g.T * nb;
  // rows k = 2, 3 of W's low parts stay zero
  for (int k = t; k < kAdjBufs * 512; k += kAdjThreads)
    reinterpret_cast<uint4*>(sm + (k >> 9) * kAA + 16384 + 8192)[k & 511] = make_uint4(0, 0, 0, 0);
  if (w == 0) tmem_alloc(slot, 512);
  if (t == 0) {
    for (uint64_t* b = full; b <= summed; ++b) mbar_init(b, (b >= empty && b < ready) || b == summed ? 8 : 1);
    fence_mbar_init();
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  bool ok = true;
  pdl_begin();
  const long long W = p.cost[U];
  // ranges no shorter than a chunk, so that every CTA of a split tile has one
  const int G = (int)max(1LL, min((long long)p.G, W / p.cost[U + 1]));

  if (w < 8) {
    // --- adders: plane u^pl of tile row `lane`, columns 16 hc .. 16 hc + 15 ---
    const int pl = w & 3, hc = w >> 2;
    const uint32_t ta = tmem + ((uint32_t)(pl * 32) << 16) + 32u * hc;
    float2* sums = reinterpret_cast<float2*>(sm + kAdjSum);
    // (an mbarrier, not a named one: a warp whose wait runs out leaves alone, and
    // so do then the others, before they read what it has not written)
    uint32_t meets = 0;
    auto add_sync = [&]() -> bool {
      __syncwarp();
      if (lane == 0) mbar_arrive(summed);
      ok = ok && sep_wait(summed, meets & 1);
      ++meets;
      return ok = __all_sync(0xffffffffu, ok);
    };
    float2 acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = make_float2(0.0f, 0.0f);
    for (uint32_t it = 0; blockIdx.x < G; ++it) {
      const int sl = it & 7, d = it & 3;
      ok = ok && sep_wait(&full[sl], (it >> 3) & 1);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const AdjStep x = adj_step(steps + sl);
      tc_fence_after();
      const int n = 32 >> x.ls();
      const float f = (lane >= x.s() * n && lane < (x.s() + 1) * n) ? x.scale : 0.0f;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        uint32_t a[8], b[8];
        tmem_ld8_nowait(ta + (uint32_t)(128 * d + 8 * h), a);
        tmem_ld8_nowait(ta + (uint32_t)(128 * d + 64 + 8 * h), b);
        tmem_wait();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 v = add2(make_float2(__uint_as_float(a[2 * i]), __uint_as_float(a[2 * i + 1])),
                                make_float2(__uint_as_float(b[2 * i]), __uint_as_float(b[2 * i + 1])));
          acc[4 * h + i] = fma2(v, dup2(f), acc[4 * h + i]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[sl]);
      if (!x.end()) continue;
      // sum of the planes; then thread: pixels (row q * 8 + w, column lane)
      float2* mine = sums + (size_t)(pl * 32 + lane) * 33 + 16 * hc;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float u = (float)(16 * hc + i - 16) * 0.0625f;
        const float c = (pl & 1 ? u : 1.0f) * (pl & 2 ? u * u : 1.0f) * kAdjTruncation;
        mine[i] = mul2(acc[i], dup2(c));
        acc[i] = make_float2(0.0f, 0.0f);
      }
      if (!add_sync()) break;
      const TcAdjParams& o = p.a;
      const Geometry& g = o.g;
      const int tx = x.tile % g.tiles_x, ty = x.tile / g.tiles_x;
      const int pi = tx * kTileX + lane, pj = ty * kTileY + w;   // pixel of q = 0; rows 8 apart
      float2 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2* s = sums + (size_t)(8 * q + w) * 33 + lane;
        v[q] = add2(add2(s[0], s[32 * 33]), add2(s[2 * 32 * 33], s[3 * 32 * 33]));
      }
      bool out = true;
      if (x.end() & 2) {
        // a split tile: the last of its CTAs adds up the partial sums (a
        // CTA's second buffer is that of the tile that starts in it)
        float2* dst = p.split + ((size_t)blockIdx.x * 2 + (x.end() & 4 ? 1 : 0)) * kTilePix + w * 32 + lane;
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[q * 256] = v[q];
        __threadfence();
        if (!add_sync()) break;
        int* flag = reinterpret_cast<int*>(slot + 1);   // [2]: the tile's first CTA if this is the last to come, its last CTA
        if (t == 0) {
          const int u0 = x.tile * nb, u1 = u0 + nb;
          const int g_lo = adj_owner(W, G, p.cost[u0]);
          const int g_hi = adj_owner(W, G, p.cost[u1] - sep_chunk_cost(p.strips[u1 - 1]));
          const bool last = atomicAdd(&p.tickets[x.tile], 1) == g_hi - g_lo;
          flag[0] = last ? g_lo : -1;
          flag[1] = g_hi;
        }
        if (!add_sync()) break;
        const int g_lo = flag[0], g_hi = flag[1];
        out = g_lo >= 0;
        if (out) {
          __threadfence();
#pragma unroll
          for (int q = 0; q < 4; ++q) v[q] = make_float2(0.0f, 0.0f);
          for (int k = g_lo; k <= g_hi; ++k) {
            const float2* src = p.split + ((size_t)k * 2 + (k == g_lo ? 1 : 0)) * kTilePix + w * 32 + lane;
            float2 r[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) r[q] = __ldcg(src + q * 256);
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = add2(v[q], r[q]);
          }
        }
      }
      if (out && pi < g.nx) {
        float amp[4] = {};
        if (o.out.epilogue & (kEpiGradPhase | kEpiFimg)) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            amp[q] = __ldg(o.amp_img + tc_pixel(g, (long long)x.tile * kTcChunksPerTile + 4 * q + (w >> 1), (w & 1) * 32 + lane).img);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int j = pj + 8 * q;
          if (j >= g.ny) break;
          adjoint_epilogue(o.out, (size_t)j * g.nx + pi, v[q].x, v[q].y, amp[q]);
          if (o.out.epilogue & kEpiFimg) {
            const float ph = (v[q].x == 0.0f && v[q].y == 0.0f) ? 0.0f : atan2f(v[q].y, v[q].x) * 0.15915494309189535f;
            // row 8 q + w of the tile, column lane
            float* f = reinterpret_cast<float*>(o.fimg + ((size_t)x.tile * kTcChunksPerTile + 4 * q + (w >> 1)) * 32 +
                                                (w & 1) * 16 + (lane >> 1)) + (lane & 1);
            f[0] = amp[q];
            f[2] = ph;
          }
        }
      }
      if (x.end() & 8) break;
      if (!add_sync()) break;   // `sums` is rewritten at the next tile's end
    }
  } else if (w < 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (w > 8 && lane == 0) {
      // --- MMA issue: steps w - 9, w - 6, .. (their X is in buffer w - 9) ---
      static_assert(kAdjBufs == 3);
      uint32_t it = (uint32_t)(w - 9);
      for (;; it += 3) {
        const int sl = it & 7, d = it & 3;
        ok = ok && sep_wait(&ready[sl], (it >> 3) & 1);
        if (!ok) break;
        const AdjStep x = adj_step(steps + sl);
        if (x.tile < 0) break;
        // W came with the chunk's first step (for s > 3 this thread's own last
        // step, it - 3, has waited for it)
        if (x.s() >= 1 && x.s() <= 3)
          ok = ok && sep_wait(&ready[(it - x.s()) & 7], ((it - x.s()) >> 3) & 1);
        if (it >= 4) ok = ok && sep_wait(&empty[(it - 4) & 7], ((it - 4) >> 3) & 1);
        if (!ok) break;
        tc_fence_after();
        const uint32_t dst = tmem + 128u * d;
        const uint64_t a = umma_desc(smem_u32(sm) + x.a() * kAA), al = a + (16384 >> 4);
        const uint64_t b = umma_desc(smem_u32(sm + kAdjB) + (uint32_t)(w - 9) * kAB);
#pragma unroll
        for (int ks = 0; ks < 8; ks += 2) umma_f16(dst, a + ks, b + ks, umma_idesc_f16(128, 128), ks > 0);
#pragma unroll
        for (int ks = 0; ks < 8; ks += 2) umma_f16(dst + 64, al + ks, b + ks, umma_idesc_f16(128, 64), 1u);
        umma_commit(&full[sl]);
      }
      // nothing in flight when the CTA gives up its memory
      if (it >= 3) ok = sep_wait(&full[(it - 3) & 7], ((it - 3) >> 3) & 1) && ok;
    } else if (w == 8 && lane == 0) {
      // --- steps of this CTA: the chunks whose place in the cost prefix lies in [c0, c1) ---
      const int c0 = blockIdx.x < G ? (int)(W * blockIdx.x / G) : 0;
      const int c1 = blockIdx.x < G ? (int)(W * (blockIdx.x + 1) / G) : 0;
      int u = 0, hi = U - 1;
      while (u < hi) {
        const int mid = (u + hi + 1) / 2;
        if (p.cost[mid] <= c0) u = mid;
        else hi = mid - 1;
      }
      int tile = u / nb, b = u % nb, ls = p.strips[u], pos = p.cost[u];
      int cc = sep_chunk_cost(ls), c = (c0 - pos + cc - 1) / cc, s = 0, a = 0;
      pos += c * cc;
      int ls1 = u + 1 < U ? p.strips[u + 1] : 0;   // of the next unit, fetched early
      int used[kAdjBufs] = {-2, -2, -2};   // of the last three chunks, as AdjStep::used
      uint32_t it = 0;
      for (;; ++it) {
        const int sl = it & 7;
        if (s == 0 && c == sep_chunks(N, b)) {
          c = 0;
          ++u;
          ls = ls1;
          cc = sep_chunk_cost(ls);
          if (++b == nb) {
            b = 0;
            ++tile;
          }
          if (u + 1 < U) ls1 = p.strips[u + 1];
        }
        const bool more = s > 0 || pos < c1;
        const int chunk = b * (kSepSpots / kSepChunk) + c;
        const float sc = more ? __ldg(p.scale + chunk) : 0.0f;
        if (!more) {
          // an end for each group of generators (-1, -2) and each issuer
          for (uint32_t k = it; k < it + 3; ++k)
            if (k >= 8) ok = ok && sep_wait(&empty[k & 7], ((k >> 3) - 1) & 1);
          if (!ok) break;
          for (uint32_t k = it; k < it + 3; ++k) put_step(steps + (k & 7), -1 - (int)(k - it), 0, -2, 0.0f);
          mbar_arrive(&listed[it & 7]);
          mbar_arrive(&listed[(it + 1) & 7]);
          break;
        }
        if (it >= 8) ok = ok && sep_wait(&empty[sl], ((it >> 3) - 1) & 1);
        if (!ok) break;   // the slot may still be read
        uint8_t* dst = sm + kAdjSlot0 + sl * kASlot;
        uint32_t end = 0;
        if (((s + 1) >> ls) && (pos + cc >= c1 || (c + 1 == sep_chunks(N, b) && b + 1 == nb))) {
          const int t1 = p.cost[(tile + 1) * nb] - sep_chunk_cost(p.strips[(tile + 1) * nb - 1]);
          const bool here = c0 <= p.cost[tile * nb];
          end = 1u | (here && t1 < c1 ? 0u : 2u) | (here ? 4u : 0u) | (pos + cc >= c1 ? 8u : 0u);
        }
        put_step(steps + sl, tile, (uint32_t)s | (uint32_t)ls << 8 | (uint32_t)a << 16 | end << 18, used[0], sc);
        mbar_expect_tx(&listed[sl], kASlot);
        bulk_g2s(dst, p.poly + ((size_t)tile * (npad / kSepChunk) + chunk) * 512, 2048, &listed[sl]);
        bulk_g2s(dst + 2048, p.ys + chunk * 64, 256, &listed[sl]);
        if (++s >> ls) {
          s = 0;
          ++c;
          pos += cc;
          a = a == kAdjBufs - 1 ? 0 : a + 1;
          used[0] = used[1];
          used[1] = used[2];
          used[2] = 2 * (int)it + (ls > 0 ? 1 : 0);
        }
      }
      // every copy has landed when the CTA gives up its memory (after the ends,
      // those of steps up to it - 6 have been read, and others' slots hold the ends)
      const uint32_t open = ok ? 5 : 8;
      for (uint32_t k = it > open ? it - open : 0; k < it; ++k) ok = sep_wait(&listed[k & 7], (k >> 3) & 1) && ok;
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 80;");
    // --- generators: spots 2 sp, 2 sp + 1 (as pairs), tile rows and columns j0, j0 + 1 ---
    const int group = (w - 12) >> 3, gw = (w - 12) & 7, sp = lane & 15, hr = lane >> 4, j0 = 4 * gw + 2 * hr;
    // The spots' 8 bytes in a row r (r = 8 a + e) of a 128-byte-swizzled operand
    // lie at row + (place ^ (e << 4)). W: rows k 32 + j0 + c, X: rows 2 j0 + e.
    const uint32_t place = (uint32_t)sp * 8;
    const uint32_t w0 = smem_u32(sm) + (uint32_t)j0 * 128 + (place ^ ((uint32_t)(j0 & 7) << 4));
    const uint32_t x0 = smem_u32(sm + kAdjB) + (uint32_t)j0 * 256 + (place ^ ((uint32_t)(j0 & 2) << 5));
    uint32_t bi = group;
    for (uint32_t it = group;; it += 2, bi = bi == 0 ? 2 : bi - 1) {
      const int sl = it & 7;
      ok = ok && sep_wait(&listed[sl], (it >> 3) & 1);
      // the MMAs of step it - 3 are done: its X is free
      if (it >= 3) ok = ok && sep_wait(&full[(it - 3) & 7], ((it - 3) >> 3) & 1);
      AdjStep x{-4, 0u, -2, 0.0f};
      if (ok) x = adj_step(steps + sl);
      if (x.tile >= 0) {
        const int xs = x.s(), xl = x.ls();
        const uint8_t* sd = sm + kAdjSlot0 + sl * kASlot;
        auto word = [&](int k) { return *reinterpret_cast<const float2*>(sd + 128 * k + 8 * sp); };
        const float2 lo = word(kWLow);
        const float2 c11 = word(kWC11), c21 = word(kWC21), c12 = word(kWC12), c22 = word(kWC22), n31 = word(kWN31),
                     c13 = word(kWC13);
        if (xs == 0) {
          // W's buffer: the MMAs of all strips of its last user are done. Those of
          // step it - 3: above. More than 7 steps ago: the record's slot was free.
          // Else by its last step's sums having been read, which is after all
          // earlier steps'; the MMAs are issued by three threads, so that another
          // step's being done says nothing.
          const int used = x.used >> 1, ago = (int)it - used;
          if (used >= 0 && ago < 8 && (ago > 3 || (x.used & 1))) ok = ok && sep_wait(&empty[used & 7], (used >> 3) & 1);
          const float2 yr = word(16), yi = word(17), nyi = sub2(make_float2(0.0f, 0.0f), yi);
          const float2 base = word(kWBase), ay = word(kWAy), y2 = word(kWY2), y3 = word(kWY3), y4 = word(kWY4);
          const float2 ayl = make_float2(__uint_as_float(__float_as_uint(lo.x) & 0xffff0000u),
                                         __uint_as_float(__float_as_uint(lo.y) & 0xffff0000u));
          const uint32_t ah = w0 + x.a() * kAA;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const float2 m = dup2((float)(j0 + c - 16));
            float2 R1 = mul2(fma2(fma2(c13, m, c12), m, c11), m);
            float2 R2 = mul2(fma2(c22, m, c21), m);
            float2 n3 = mul2(n31, m);
            if (xl) {
              // about the middle row of the row's strip: the rest is in X
              const float2 v = dup2(strip_mid((j0 + c) / (32 >> xl), xl)), nv = sub2(make_float2(0.0f, 0.0f), v);
              R1 = fma2(fma2(fma2(c13, v, c12), v, c11), nv, R1);
              R2 = fma2(fma2(c22, v, c21), nv, R2);
              n3 = fma2(n31, nv, n3);
            }
            // exp(+i r) = 1 + i R1 u + (q2r + i q2i) u^2 + (q3r + i q3i) u^3
            const float2 s2 = mul2(R1, R1), n1 = sub2(make_float2(0.0f, 0.0f), R1);
            const float2 q2r = fma2(s2, fma2(s2, dup2(1.0f / 24.0f), dup2(-0.5f)), mul2(R2, mul2(R2, dup2(-0.5f))));
            const float2 q2i = mul2(R2, fma2(s2, dup2(-0.5f), dup2(1.0f)));
            const float2 q3r = mul2(n1, R2), n3i = fma2(mul2(R1, s2), dup2(1.0f / 6.0f), n3);   // -q3i
            float2 cs, sn;
            cis2(sep_angle(ay, ayl, y2, y3, y4, base, m), cs, sn);
            // (a complex product: the phase of y, carried from iteration to
            // iteration by a WGS loop, keeps its fp32 accuracy)
            const float2 wr = fma2(sn, nyi, mul2(cs, yr)), wi = fma2(cs, yi, mul2(sn, yr));
            const uint32_t at = (ah ^ (uint32_t)(c << 4)) + 128 * c;
            auto emit = [&](auto kk, float2 re, float2 im) {
              constexpr int k = decltype(kk)::value, o = k * 4096;
              if constexpr (k < 2) {
                const float2 hr2 = split_hi2(re), hi2 = split_hi2(im);
                const float2 lr2 = sub2(re, hr2), li2 = sub2(im, hi2);
                sts64<o>(at, pack_f16(hr2.x, hi2.x), pack_f16(hr2.y, hi2.y));
                sts64<o + 16384>(at, pack_f16(lr2.x, li2.x), pack_f16(lr2.y, li2.y));
              } else {
                sts64<o>(at, pack_f16(re.x, im.x), pack_f16(re.y, im.y));
              }
            };
            const float2 nwi = sub2(make_float2(0.0f, 0.0f), wi), nwr = sub2(make_float2(0.0f, 0.0f), wr);
            emit(IntTag<0>{}, wr, wi);
            emit(IntTag<1>{}, mul2(R1, nwi), mul2(R1, wr));
            emit(IntTag<2>{}, fma2(q2r, wr, mul2(q2i, nwi)), fma2(q2r, wi, mul2(q2i, wr)));
            emit(IntTag<3>{}, fma2(q3r, wr, mul2(n3i, wi)), fma2(q3r, wi, mul2(n3i, nwr)));
          }
        }
        float2 ax = word(kWAx), x2 = word(kWX2), x3 = word(kWX3);
        float2 axl = make_float2(__uint_as_float(__float_as_uint(lo.x) << 16), __uint_as_float(__float_as_uint(lo.y) << 16));
        if (xl) {
          // about the strip's middle row (sep_columns)
          const float2 v = dup2(strip_mid(xs, xl));
          const float2 R1 = mul2(fma2(fma2(c13, v, c12), v, c11), v), R2 = mul2(fma2(c22, v, c21), v);
          const float2 d = mul2(R1, dup2(0.15915494309189535f * 0.0625f));
          const float2 a = add2(ax, d), z = sub2(a, ax);
          const float2 e = add2(fma2(sub2(a, z), dup2(-1.0f), ax), sub2(d, z));
          axl = fma2(e, dup2(6.283185307179586f), axl);
          ax = a;
          x2 = fma2(R2, dup2(0.0625f * 0.0625f), x2);
          x3 = fma2(mul2(n31, v), dup2(-0.0625f * 0.0625f * 0.0625f), x3);
        }
        const float2 x4 = word(kWX4);
        const uint32_t bh = x0 + bi * kAB;
        constexpr uint32_t S = 0x80000000u;   // the sign of the upper half
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float2 cs, sn;
          cis2(sep_angle(ax, axl, x2, x3, x4, dup2((float)(j0 + c - 16))), cs, sn);
          const float2 hc = split_hi2(cs), hs = split_hi2(sn);
          const float2 lc = sub2(cs, hc), lsn = sub2(sn, hs);
          // rows 2 (j0 + c): (re, -im), and the next: (im, re)
          const uint32_t b0 = (bh ^ (uint32_t)(c << 5)) + 256 * c, b1 = (bh ^ (uint32_t)(c << 5 | 16)) + 256 * c;
          sts64<0>(b0, pack_f16(hc.x, hs.x) ^ S, pack_f16(hc.y, hs.y) ^ S);
          sts64<128>(b1, pack_f16(hs.x, hc.x), pack_f16(hs.y, hc.y));
          sts64<8192>(b0, pack_f16(lc.x, lsn.x) ^ S, pack_f16(lc.y, lsn.y) ^ S);
          sts64<8192 + 128>(b1, pack_f16(lsn.x, lc.x), pack_f16(lsn.y, lc.y));
        }
        fence_async_smem();
      }
      // all generators go on or stop together
      int stop;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.lt.s32 p, %1, 0;\n\tbarrier.red.or.pred q, %2, 256, p;\n\t"
          "selp.s32 %0, 1, 0, q;\n\t}"
          : "=r"(stop)
          : "r"(x.tile), "r"(2 + group)
          : "memory");
      if (gw == 0 && lane == 0 && ok) {
        mbar_arrive(&ready[sl]);
        if (x.tile == -1) mbar_arrive(&ready[(it + 2) & 7]);   // the third issuer's end
      }
      if (stop) break;
    }
  }
  if (!ok) atomicOr(p.a.err, kErrTimeout);
  tc_fence_before();
  __syncthreads();
  if (w == 0) tmem_dealloc(tmem, 512);
}

// One warp per chunk of 32 spots (1.4 us, its launch; the adjoint fetches the
// result with the phase polynomials). It also sets the split tiles' counts to
// zero, so that an adjoint whose wait ran out leaves none behind for the next.
__global__ void k_sep_scale(const float2* __restrict__ y, int N, int chunks, float* __restrict__ ys,
                            float* __restrict__ scale, int* __restrict__ tickets, int T) {
  pdl_begin();
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < T; k += gridDim.x * blockDim.x) tickets[k] = 0;
  const int c = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (c < chunks) sep_scale_chunk(y, N, c, ys, scale);
}

}  // namespace

cudaError_t sep_launch_scale(const float2* y, int N, float* ys, float* scale, int* tickets, int T, cudaStream_t s) {
  const int chunks = sep_blocks(N) * (kSepSpots / kSepChunk);
  return launch_pdl(k_sep_scale, (chunks + 3) / 4, 128, 0, s, y, N, chunks, ys, scale, tickets, T);
}

cudaError_t sep_adjoint_prepare() {
  cudaError_t e = cudaFuncSetAttribute(k_sep_adjoint, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAdjSmem);
  if (e != cudaSuccess) return e;
  for (const void* k : {(const void*)k_sep_adjoint, (const void*)k_sep_scale})
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                  (int)cudaSharedmemCarveoutMaxShared)))
      return e;
  return cudaSuccess;
}

cudaError_t sep_launch_adjoint(const SepAdjParams& p, cudaStream_t s) {
  return launch_pdl(k_sep_adjoint, p.G, kAdjThreads, kAdjSmem, s, p);
}

}  // namespace ash
