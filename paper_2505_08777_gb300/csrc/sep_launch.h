// Separable tile transforms (sep_common.cuh): parameter blocks and launchers.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"
#include "mono.h"

namespace ash {

constexpr int kSepMaxOrd = 4;        // total degree of the basis polynomials
constexpr int kSepTab = 18;          // floats per (tile, mode) of the basis table
constexpr int kSepSpots = 128;       // spots of a block
constexpr int kSepFwdRows = 2;       // rows of partial sums per forward CTA
constexpr float kSepTol = 1e-6f;   // largest part of exp(-i r) the cubic in u may drop

// Estimated time of one step of a unit cut into 2^ls row strips (the whole
// tile: 20): preparing X and the MMAs' latency stay, the sums shrink.
__host__ __device__ constexpr int sep_step_cost(int ls) { return ls == 0 ? 20 : ls == 1 ? 13 : ls == 2 ? 10 : 8; }

inline int sep_blocks(int N) { return (N + kSepSpots - 1) / kSepSpots; }

// Basis polynomials over each tile about its pixel (16, 16), in turns:
// [T][D][kSepTab] = (c00 hi, lo), (c10 hi, lo), (c01 hi, lo) per pixel,
// c20 c30 c40 c02 c03 c04 c11 c21 c12 c22 c31 c13 per u^k v^l.
cudaError_t sep_build_table(const Geometry& g, const MonoTerm* terms, const int* term_off, float* tab, cudaStream_t s);

// Phase polynomials of every (tile, spot), [T][4][npad] float4 (SepPoly), and
// per (tile, spot block) the log2 of the row strips its mixed terms need and
// the prefix of its steps' cost [T nb + 1].
cudaError_t sep_build_params(const Geometry& g, const float* tab, const float* coeff, float4* poly,
                             unsigned char* strips, int* cost, cudaStream_t s);

struct SepFwdParams {
  Geometry g;
  int nb;                        // spot blocks
  const float4* poly;
  const unsigned char* strips;
  const int* cost;
  const float4* fimg;            // nearfield image (tc_launch.h)
  float2* part;                  // [kSepFwdRows G][128 nb] partial sums
  float2* E;                     // [N]
  int G;
  unsigned* err;
};
cudaError_t sep_prepare();
cudaError_t sep_launch_forward(const SepFwdParams& p, cudaStream_t s);   // kernel and reduction

}  // namespace ash
