// The adjoints' per-pixel output in the tensor-core pixel order.
#pragma once

#include "common.cuh"
#include "tc_launch.h"

namespace ash {

// A phase in turns, reduced to [-1/2, 1/2] and a little: the product with
// 1 / 2 pi in two pieces, its rounding kept, so that a phase of any size is right
// to 2^-25 turns and the mean error over a turn vanishes (the single constant is
// 4e-8 too small).
__device__ __forceinline__ float exact_turns(float ph) {
  const float p = __fmul_rn(ph, 0.15915494f), e = __fmaf_rn(ph, 0.15915494f, -p);
  return __fadd_rn(__fsub_rn(p, rintf(p)), __fmaf_rn(ph, 6.4206382e-09f, e));
}

// Adjoint output of row r of chunk qc (in the pixel's user-layout slot and,
// for kEpiFimg, in the tc-layout nearfield f = A exp(i arg g) as (A, arg g / 2 pi)).
__device__ __forceinline__ void tc_adjoint_epilogue(const TcAdjParams& p, long long qc, int r, float gr, float gi) {
  const Geometry& G = p.g;
  const TcPixel px = tc_pixel(G, qc, r);
  if (px.i >= G.nx || px.j >= G.ny) return;
  const bool need_a = (p.out.epilogue & (kEpiGradPhase | kEpiFimg)) != 0;
  const float a = need_a ? __ldg(p.amp_img + px.img) : 0.0f;
  adjoint_epilogue(p.out, (size_t)px.j * G.nx + px.i, gr, gi, a);
  if (p.out.epilogue & kEpiFimg) {
    const float ph = (gr == 0.0f && gi == 0.0f) ? 0.0f : atan2f(gi, gr) * 0.15915494309189535f;
    float* q = reinterpret_cast<float*>(p.fimg + (size_t)qc * 32 + (r >> 1));
    q[r & 1] = a;
    q[2 + (r & 1)] = ph;
  }
}

}  // namespace ash
