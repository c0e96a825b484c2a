// Which kernel a SmoothGEMM call takes when the caller leaves the tile size to the library, and how
// the problem is cut for it.  Host arithmetic only.
#pragma once

#include <cstdint>

namespace xy {

constexpr int kSwapMaxSplits = 4;     // pairs per cluster of the weight-major kernel
constexpr int kClusterMaxCtas = 8;

enum GemmKernel : int {
  kGemmTile = 0,    // 128 x tile_n tiles on single CTAs
  kGemmPair = 1,    // 256 x tile_n tiles on CTA pairs
  kGemmSplitK = 2,  // 128 x 128 tiles, K split over a cluster
  kGemmSwap = 3,    // weight-major on CTA pairs
  kGemmSmall = 4    // weight-streaming, up to 128 tokens
};

// What the choice needs to know of a device.
struct GemmDevice {
  int sms = 0;
  int clusters[kClusterMaxCtas] = {0};       // clusters of 1 .. 8 CTAs that fit at once, one CTA per SM
  int pair_clusters[kSwapMaxSplits] = {0};   // clusters of 1 .. 4 pairs of the weight-major kernel
};

// Scratch the kernels can use, in bytes: two slots of a 128 x 256 fp32 tile per SM.  Less is none.
constexpr int64_t gemm_scratch_bytes(int sms) { return static_cast<int64_t>(sms) * 2 * 128 * 256 * 4; }

// How a problem is cut for the weight-major kernel (tok = 0: no cut fits the device).
struct SwapPlan {
  int m_tiles = 0, tok = 0, halves = 1, splits = 1;
  float us = 1e30f;
};

struct GemmChoice {
  GemmKernel kernel = kGemmTile;
  int tile_n = 0, splits = 1;
  SwapPlan swap;
  float us = 0.f;  // what the models expect
};

GemmChoice choose_gemm(int M, int N, int K, int64_t workspace_bytes, const GemmDevice& dev);

}  // namespace xy
