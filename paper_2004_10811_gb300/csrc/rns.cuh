// FP64-accurate products on the tensor cores by residue numbers (rns.cu).
//
// A product C = A B of fixed-point matrices is an integer product, and an
// integer below P / 2 in magnitude is determined by its residues modulo pairwise
// coprime m_1 .. m_14 with product P = 2^109.87 (Chinese remainder theorem).  The
// residues of A and B lie in [-128, 128], exact in BF16, so each modulus costs
// one BF16 tensor-core product whose FP32 accumulator is exact (1024 terms of
// at most 2^14).  Operands with rows of norm 1 or less are rounded to multiples
// of 1 / S, S = sqrt(P / 2.02) = 2^54.43, so that |C| S^2 < P / 2 (Cauchy-Schwarz),
// and C follows from
//     C S^2 / P = frac(sum_i r_i w_i),   w_i = ((P / m_i)^-1 mod m_i) / m_i,
// summed modulo 1 in 64-bit integers.  The absolute error is ~2e-17 an entry:
// on involutions a Newton-Schulz run ends with 0.8 of the error that FP64
// multiply-add chains leave (n = 100 .. 400, against 80-bit arithmetic), while
// the fourteen products run at the BF16 rate, ~1500 times the FP64 one.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace submat {

constexpr int RNS_MODS = 14;
constexpr int RNS_FRAC = 58;   // fraction bits of the iterates
constexpr int RNS_CHUNK = 16;  // k-blocks of 64 per exact FP32 accumulation (1024 terms)

// Residue arrays: per size bucket [count][RNS_MODS][ld][ld] BF16, so submatrix
// s starts at RNS_MODS * off[s] and its modulus i at + i ld^2.
struct RnsGemmParams {
  const int4* items;         // (s, ti, tj, bucket | slot << 8), 128 x 128 tiles
  int nitems;
  const CUtensorMap* map_a;  // device, one per bucket: [count * RNS_MODS][ld][ld], 128-row boxes
  const CUtensorMap* map_b;  // rows of B^T (B itself when symmetric)
  const int64_t* off;
  const int32_t* ld;
  const int* state;          // optional: submatrices with state == skip_state are skipped
  int skip_state;
  int split;                 // parts a tile's moduli are spread over (> 1: F zeroed beforehand, added to)
  long long* F;              // frac(C / P) 2^64 on the listed tiles, [ld][ld] at off
  int* flags;
  long long timeout_cycles;
};
// split for a launch of ntiles tiles: enough CTAs for every SM
int rns_split(int ntiles, int nsm);
cudaError_t launch_rns_gemm(RnsGemmParams p, int nsm, cudaStream_t st);

// Largest row 2-norm squared of X per submatrix (bits of a float) into norm2.
cudaError_t launch_rns_rownorm(const WaveDev& w, const double* X, const int* state, unsigned* norm2, int max_ld,
                               cudaStream_t st);
// Residues of X 2^-sh for a complete FP64 matrix; sh from norm2 (the smallest
// that brings the row norms to 1), or the constant sh_fixed when norm2 is null.
// fixed (optional, may be X's own memory): X as 2^-RNS_FRAC fixed point.
cudaError_t launch_rns_convert(const WaveDev& w, const double* X, const int* state, const unsigned* norm2,
                               int sh_fixed, __nv_bfloat16* R, long long* fixed, int max_ld, cudaStream_t st);
// First square (operand shifts from norm2): F (upper tiles) to the complete FP64 Y = X_0^2 (in F's memory),
// with ||Y - I||_F^2 into res2.
cudaError_t launch_rns_square0(const WaveDev& w, NsStateDev ns, const unsigned* norm2, long long* F, int max_ld,
                               cudaStream_t st);
// Y = X^2: its residues (both triangles) and ||Y - I||_F^2 into res2.
cudaError_t launch_rns_square(const WaveDev& w, NsStateDev ns, const long long* F, __nv_bfloat16* R, int max_ld,
                              cudaStream_t st);
// X <- (3 X - X Y) / 2, X Y = 2^shift times F's product, in fixed point (upper tiles) with its residues;
// for a submatrix in its last iteration X becomes the complete FP64 result.
cudaError_t launch_rns_update(const WaveDev& w, NsStateDev ns, const long long* F, int shift, long long* X,
                              __nv_bfloat16* R, int max_ld, cudaStream_t st);

// Chebyshev recurrences (fermi.cu).  All matrices have spectral norm 1 or less
// and move as 2^-RNS_FRAC fixed point on their upper tiles.
constexpr int RNS_COMB = 8;
struct RnsCheb {
  const long long* F;          // product, null: none
  int twice;                   // 2 F instead of F
  const long long* sub;        // subtracted (may be C), null: none
  const long long* odd;        // RNS_COMB matrices, stride entries apart, null: none ...
  int64_t stride;
  long long coef[RNS_COMB];    // ... combined with these 2^-58 coefficients, and added
  long long* C;                // the result (upper tiles), null: not stored
  __nv_bfloat16* R;            // its residues (both triangles), null: none
  double* out;                 // out_scale times the result, complete FP64 (may be C's memory), null: none
  double out_scale;
};
cudaError_t launch_rns_cheb(const WaveDev& w, const RnsCheb& c, int max_ld, cudaStream_t st);
// T2 = 2 X^2 - I, complete FP64, from X^2's sums.
cudaError_t launch_rns_cheb2(const WaveDev& w, const long long* F, double* T2, int max_ld, cudaStream_t st);

}  // namespace submat
