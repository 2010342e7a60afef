// Exact product of sliced matrices in one pass (slice_gemm.cu).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace submat {

constexpr int SG_SLICES = 6;  // most slices of an operand
constexpr int SG_LEVELS = 7;  // levels p + q = 2 .. 8

// Z = sum over p + q <= 8 of 2^(6 (8 - p - q)) X_p Y_q^T in 64-bit integers, with
// slices of at most 63 in magnitude, p = 1 .. nx, q = 1 .. ny.
struct SliceGemmParams {
  const int4* items;         // (s, ti, tj, bucket | slot << 8), 128 x 128 tiles
  int nitems;
  const CUtensorMap* maps;   // device array [set][bucket], boxes of 128 rows and 32 columns
  int nbucket;
  int nx, ny;
  int a_set[SG_SLICES], b_set[SG_SLICES];
  const int64_t* off;
  const int32_t* ld;
  long long* Z;
  int* flags;
  long long timeout_cycles;
};
// whether three pipeline stages of the slices fit
bool slice_gemm_fits(int nx, int ny);
// products a tile of the launch runs
int slice_gemm_products(int nx, int ny);
cudaError_t launch_slice_gemm(const SliceGemmParams& p, int nsm, cudaStream_t st);

}  // namespace submat
