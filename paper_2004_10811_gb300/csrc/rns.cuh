// FP64-accurate products on the tensor cores by residue numbers (rns.cu).
//
// A product C = A B of fixed-point matrices is an integer product, and an
// integer below P / 2 in magnitude is determined by its residues modulo pairwise
// coprime m_1 .. m_19 with product P = 2^147.93 (Chinese remainder theorem).  The
// residues of A and B lie in [-128, 128], exact in BF16, so each modulus costs
// one BF16 tensor-core product whose FP32 accumulator is exact (1024 terms of
// at most 2^14).  Operands with rows of norm 1 or less are multiples of 1 / S,
// S = 2^73, so that |C| S^2 < P / 2 (Cauchy-Schwarz), and C follows from
//     C S^2 / P = frac(sum_i r_i w_i),   w_i = ((P / m_i)^-1 mod m_i) / m_i,
// summed modulo 1 in integers of 82 bits.
//
// The error of an entry is absolute, about 2^-73 (the rounding of the iterates and
// of the weights), where a chain of FP64 multiply-adds keeps it relative to
// (|A| |B|)_ij: 20 bits finer than FP64 for entries of order one, and as fine for
// entries of 2^-20.  A matrix whose extracted columns couple more weakly than that
// is evaluated by the chains (rns_route).  (Fourteen moduli, 2^-54, gave the same
// largest error as the chains, but ten times theirs in entries of 1e-3 and 5e4
// times in entries of 1e-6: the decay of D with distance needs the finer grid.)
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace submat {

constexpr int RNS_MODS = 19;
constexpr int RNS_FRAC = 73;   // fraction bits of the iterates
constexpr int RNS_GUARD = 18;  // guard bits of a product's sums
constexpr int RNS_COEF = 58;   // fraction bits of the series' coefficients
constexpr int RNS_CHUNK = 16;  // k-blocks of 64 per exact FP32 accumulation (1024 terms)

// A fixed-point matrix: (2^16 hi + lo) 2^-RNS_FRAC, [ld][ld] at off.
struct RnsFix {
  long long* hi;
  unsigned short* lo;
};
// Sums of a product: frac(C / P) = f 2^-64 + g 2^-82.
struct RnsSum {
  long long* f;
  int* g;
};

// Residue sets are complete (parts 1) or, where the workspace is small, hold one half
// of the moduli at a time (parts 2): the sums of the halves add up to the same bits.
constexpr int rns_planes(int parts) { return (RNS_MODS + parts - 1) / parts; }
// Per size bucket [count][planes][ld][ld] BF16, so submatrix s starts at
// planes * off[s] and its i-th modulus at + i ld^2.
struct RnsGemmParams {
  const int4* items;         // (s, ti, tj, bucket | slot << 8), 128 x 128 tiles
  int nitems;
  const CUtensorMap* map_a;  // device, one per bucket: [count * planes][ld][ld], 128-row boxes
  const CUtensorMap* map_b;  // rows of B^T (B itself when symmetric)
  const int64_t* off;
  const int32_t* ld;
  const int* state;          // optional: submatrices with state == skip_state are skipped
  int skip_state;
  int planes;                // of a residue set ...
  int mod0, nmod;            // ... which holds the moduli mod0 .. mod0 + nmod - 1
  int add;                   // 1: to the sums of the other moduli
  int split;                 // parts a tile's moduli are spread over (> 1: F zeroed beforehand, added to)
  RnsSum F;                  // on the listed tiles, [ld][ld] at off
  int* flags;
  long long timeout_cycles;
};
// split for a launch of ntiles tiles of nmod moduli: enough CTAs for every SM
int rns_split(int ntiles, int nmod, int nsm);
cudaError_t launch_rns_gemm(RnsGemmParams p, int nsm, cudaStream_t st);

// A submatrix with less than this, but not 0, in (|X| |X|)_rc of an extracted entry, or
// in a row's squared norm, goes to the FP64 chains (an entry that is 0 there is exactly
// zero on either path).  An entry's error is about 2^-73 here and 2^-53 of that measure
// there, so the line is 2^-20 with a margin of four.  Water at a 9 A cutoff lies at
// 6e-4 and above.  One with a row of norm above 2 goes there too.
constexpr float RNS_LEAST_COUPLING = 0x1p-18f;
// the coupling pass holds a block's diagonal in FP32 in shared memory
bool rns_route_fits(int bs_max);
// route[s] = ST_DONE for submatrices of the chains, else ST_ACTIVE, and their number
// into chains.  With state, submatrices not active are left out and those of the
// chains are held (ST_DONE) until launch_rns_resume.  norm2: the largest row 2-norm
// squared of X per submatrix (bits of a float).
cudaError_t launch_rns_route(const PatternDev& g, const WaveDev& w, const double* X, int* state, unsigned* norm2,
                             unsigned* least, int* route, int* chains, int bs_max, int max_ld, cudaStream_t st);
cudaError_t launch_rns_resume(const WaveDev& w, const int* route, int* state, cudaStream_t st);

// Residues of X 2^-sh for a complete FP64 matrix; sh from norm2 (the smallest
// that brings the row norms to 1), or the constant sh_fixed when norm2 is null.
// fixed (optional, its hi may be X's own memory): X in fixed point.  R null: only that.
cudaError_t launch_rns_convert(const WaveDev& w, const double* X, const int* state, const unsigned* norm2,
                               int sh_fixed, __nv_bfloat16* R, RnsFix fixed, int max_ld, cudaStream_t st,
                               int parts = 1, int part = 0);
// Residues (parts 2) of a matrix in fixed point on its upper tiles.
cudaError_t launch_rns_spread(const WaveDev& w, const int* state, RnsFix X, __nv_bfloat16* R, int max_ld,
                              cudaStream_t st, int part);
// First square (operand shifts from norm2): F (upper tiles) to the complete FP64 Y = X_0^2 (may be F.f's memory),
// with ||Y - I||_F^2 into res2.
cudaError_t launch_rns_square0(const WaveDev& w, NsStateDev ns, const unsigned* norm2, RnsSum F, double* Y,
                               int max_ld, cudaStream_t st);
// Y = X^2, with ||Y - I||_F^2 into res2: its residues (both triangles, parts 1) or itself (upper tiles).
cudaError_t launch_rns_square(const WaveDev& w, NsStateDev ns, RnsSum F, RnsFix Y, __nv_bfloat16* R, int max_ld,
                              cudaStream_t st);
// X <- (3 X - X Y) / 2, X Y = 2^shift times F's product, in fixed point (upper tiles) with its residues (R null:
// without); for a submatrix in its last iteration X.hi becomes the complete FP64 result.
cudaError_t launch_rns_update(const WaveDev& w, NsStateDev ns, RnsSum F, int shift, RnsFix X, __nv_bfloat16* R,
                              int max_ld, cudaStream_t st);

// Chebyshev recurrences (fermi.cu).  All matrices have spectral norm 1 or less
// and move in fixed point on their upper tiles.
constexpr int RNS_COMB = 8;
struct RnsCheb {
  const int* state;            // submatrices with ST_DONE are skipped
  RnsSum F;                    // product, null: none
  int twice;                   // 2 F instead of F
  RnsFix sub;                  // subtracted (may be C), null: none
  RnsFix odd;                  // RNS_COMB matrices, stride entries apart, null: none ...
  int64_t stride;
  long long coef[RNS_COMB];    // ... combined with these 2^-RNS_COEF coefficients, and added
  RnsFix C;                    // the result (upper tiles), null: not stored
  __nv_bfloat16* R;            // its residues (both triangles), null: none
  double* out;                 // out_scale times the result, complete FP64 (may be C.hi's memory), null: none
  double out_scale;
};
cudaError_t launch_rns_cheb(const WaveDev& w, const RnsCheb& c, int max_ld, cudaStream_t st);
// T2 = 2 X^2 - I, complete FP64, from X^2's sums.
cudaError_t launch_rns_cheb2(const WaveDev& w, RnsSum F, double* T2, int max_ld, cudaStream_t st);

}  // namespace submat
