// Separable tile transforms (sep_common.cuh): parameter blocks and launchers.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"
#include "launch.h"
#include "mono.h"
#include "tc_launch.h"

namespace ash {

constexpr int kSepMaxOrd = 4;        // total degree of the basis polynomials
constexpr int kSepTab = 18;          // floats per (tile, mode) of the basis table
constexpr int kSepSpots = 128;       // spots of a block
constexpr int kSepFwdRows = 2;       // rows of partial sums per forward CTA
constexpr float kSepTol = 1e-6f;   // largest part of exp(-i r) the cubic in u may drop

// Estimated time of one step of a unit cut into 2^ls row strips (the whole
// tile: 20): preparing X and the MMAs' latency stay, the sums shrink.
__host__ __device__ constexpr int sep_step_cost(int ls) { return ls == 0 ? 20 : ls == 1 ? 13 : ls == 2 ? 10 : 8; }

// The same of one chunk (32 spots of a tile) of the adjoint, all its strips.
constexpr int kSepChunk = 32;
__host__ __device__ constexpr int sep_chunk_cost(int ls) { return 20 + 14 * ((1 << ls) - 1); }
__host__ __device__ constexpr int sep_chunks(int N, int b) {
  return (N - b * kSepSpots >= kSepSpots) ? kSepSpots / kSepChunk : (N - b * kSepSpots + kSepChunk - 1) / kSepChunk;
}

inline int sep_blocks(int N) { return (N + kSepSpots - 1) / kSepSpots; }

// Basis polynomials over each tile about its pixel (16, 16), in turns:
// [T][D][kSepTab] = (c00 hi, lo), (c10 hi, lo), (c01 hi, lo) per pixel,
// c20 c30 c40 c02 c03 c04 c11 c21 c12 c22 c31 c13 per u^k v^l.
cudaError_t sep_build_table(const Geometry& g, const MonoTerm* terms, const int* term_off, float* tab, cudaStream_t s);

// Phase polynomials of every (tile, spot), [T][chunk of 32 spots][16 words][32]
// (SepPoly), and
// per (tile, spot block) the log2 of the row strips its mixed terms need and
// the prefixes of their forward steps' cost
// [T nb + 1] and of their adjoint chunks' cost [T nb + 1], then the largest
// chunk cost.
cudaError_t sep_build_params(const Geometry& g, const float* tab, const float* coeff, float* poly,
                             unsigned char* strips, int* cost, int* acost, cudaStream_t s);

struct SepFwdParams {
  Geometry g;
  int nb;                        // spot blocks
  const float* poly;
  const unsigned char* strips;
  const int* cost;
  const float4* fimg;            // nearfield image (tc_launch.h)
  float2* part;                  // [kSepFwdRows G][128 nb] partial sums
  float2* E;                     // [N]
  int G;
  unsigned* err;
  bool exact;                    // pixel phases without a mean error (not inside a loop)
  // the moment pass (dL/dC) instead of E
  const float2* gE;              // [N] dL/dE
  const float* tab;              // basis polynomials per tile
  float* dpart;                  // [kSepFwdRows G][D][128 nb] partial sums
  float* dC;                     // [N][D]
};
cudaError_t sep_launch_gradc(const SepFwdParams& p, cudaStream_t s);            // partial sums
cudaError_t sep_launch_gradc_reduce(const SepFwdParams& p, cudaStream_t s);     // dL/dC from them
struct SepAdjParams {
  TcAdjParams a;                 // geometry, amplitude, y, outputs
  int nb;
  const float* poly;
  const unsigned char* strips;
  const int* cost;               // adjoint prefix
  const float* ys;               // [4 nb][re, im][32] y / scale
  const float* scale;            // [4 nb] power of two per chunk of 32 spots
  float2* split;                 // [G][2][kTilePix] partial sums of tiles split between CTAs
  int* tickets;                  // [T] CTAs done with a split tile (0 at the start)
  int G;
};
cudaError_t sep_prepare();
cudaError_t sep_adjoint_prepare();
// y divided by a power of two (scale) per chunk of 32 spots; the counts of the
// T tiles set to 0. Goes before every adjoint.
cudaError_t sep_launch_scale(const float2* y, int N, float* ys, float* scale, int* tickets, int T, cudaStream_t s);
cudaError_t sep_launch_adjoint(const SepAdjParams& p, cudaStream_t s);
cudaError_t sep_launch_forward(const SepFwdParams& p, cudaStream_t s);          // partial sums
cudaError_t sep_launch_forward_reduce(const SepFwdParams& p, cudaStream_t s);   // E from them

}  // namespace ash
