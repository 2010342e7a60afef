// Grouped FP64 / FP32 GEMM over the submatrix batch (the plain FP64 and FP32
// Newton-Schulz paths and the high-precision residual products of the
// refinement).
//
// One CTA computes one 64x64 tile (s, ti, tj) of C = alpha A B + beta C0 for
// submatrix s; A, B, C0, C are row-major n x n blocks with leading dimension
// ld (a multiple of 64) at the same wave offset in each buffer.  FP64 is
// issued with DFMA from registers (4x4 outputs per thread, 16-deep k slices
// staged in shared memory with a register prefetch of the next slice).
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace submat {

namespace {

constexpr int TM = 64;
constexpr int TK = 16;

__global__ void __launch_bounds__(256) k_gemm_f64(GemmF64Args a) {
  using T = double;
  using V2 = double2;
  __shared__ __align__(16) T As[TK][TM + 2];  // As[k][m]
  __shared__ __align__(16) T Bs[TK][TM];      // Bs[k][n]
  __shared__ double red[8];
  const int4 item = a.items[blockIdx.x];
  const int s = item.x, ti = item.y, tj = item.z;
  if (a.state != nullptr && a.state[s] == a.skip_state) return;
  const int ld = a.w.ld[s];
  const int64_t off = a.w.off[s];
  const T* __restrict__ Ab = a.A + off + int64_t(ti) * TM * ld;
  const T* __restrict__ Bb = a.B + off + int64_t(tj) * TM;
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  // loader mapping
  const int a_row = tid >> 2, a_k = (tid & 3) * 4;   // A: 64 rows x 16 k
  const int b_k = tid >> 4, b_n = (tid & 15) * 4;    // B: 16 k x 64 n
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);

  V2 ra0, ra1, rb0, rb1;
  {
    const T* pa = Ab + int64_t(a_row) * ld + a_k;
    ra0 = *reinterpret_cast<const V2*>(pa);
    ra1 = *reinterpret_cast<const V2*>(pa + 2);
    const T* pb = Bb + int64_t(b_k) * ld + b_n;
    rb0 = *reinterpret_cast<const V2*>(pb);
    rb1 = *reinterpret_cast<const V2*>(pb + 2);
  }
  const int nk = ld / TK;
  for (int kt = 0; kt < nk; ++kt) {
    As[a_k + 0][a_row] = ra0.x;
    As[a_k + 1][a_row] = ra0.y;
    As[a_k + 2][a_row] = ra1.x;
    As[a_k + 3][a_row] = ra1.y;
    *reinterpret_cast<V2*>(&Bs[b_k][b_n]) = rb0;
    *reinterpret_cast<V2*>(&Bs[b_k][b_n + 2]) = rb1;
    __syncthreads();
    if (kt + 1 < nk) {
      const int k0 = (kt + 1) * TK;
      const T* pa = Ab + int64_t(a_row) * ld + k0 + a_k;
      ra0 = *reinterpret_cast<const V2*>(pa);
      ra1 = *reinterpret_cast<const V2*>(pa + 2);
      const T* pb = Bb + int64_t(k0 + b_k) * ld + b_n;
      rb0 = *reinterpret_cast<const V2*>(pb);
      rb1 = *reinterpret_cast<const V2*>(pb + 2);
    }
#pragma unroll
    for (int k = 0; k < TK; ++k) {
      T av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = As[k][ty * 4 + i];
      const V2 b01 = *reinterpret_cast<const V2*>(&Bs[k][tx * 4]);
      const V2 b23 = *reinterpret_cast<const V2*>(&Bs[k][tx * 4 + 2]);
      bv[0] = b01.x; bv[1] = b01.y; bv[2] = b23.x; bv[3] = b23.y;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }

  // epilogue
  const int n = a.w.n[s];
  T* Cb = a.C + off;
  const T* C0b = a.C0 ? a.C0 + off : nullptr;
  double part = 0.0;
  const int r0 = ti * TM + ty * 4, c0 = tj * TM + tx * 4;
  T v[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + i;
    V2 z0, z1;
    z0.x = z0.y = z1.x = z1.y = T(0);
    if (C0b) {
      z0 = *reinterpret_cast<const V2*>(C0b + int64_t(r) * ld + c0);
      z1 = *reinterpret_cast<const V2*>(C0b + int64_t(r) * ld + c0 + 2);
    }
    const T zc[4] = {z0.x, z0.y, z1.x, z1.y};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      T x = T(a.alpha) * acc[i][j];
      if (C0b) x = fma(T(a.beta), zc[j], x);
      if (a.diag != 0.0 && r == c0 + j && r < n) x += T(a.diag);
      v[i][j] = x;
      if (a.res2) {
        const int c = c0 + j;
        const double e = double(x) - ((r == c && r < n) ? 1.0 : 0.0);
        part = fma(e, e, part);
      }
    }
    V2 w0, w1;
    w0.x = v[i][0]; w0.y = v[i][1]; w1.x = v[i][2]; w1.y = v[i][3];
    *reinterpret_cast<V2*>(Cb + int64_t(r) * ld + c0) = w0;
    *reinterpret_cast<V2*>(Cb + int64_t(r) * ld + c0 + 2) = w1;
  }
  if (a.sym && ti != tj) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      T* row = Cb + int64_t(c0 + j) * ld + r0;
      V2 w0, w1;
      w0.x = v[0][j]; w0.y = v[1][j]; w1.x = v[2][j]; w1.y = v[3][j];
      *reinterpret_cast<V2*>(row) = w0;
      *reinterpret_cast<V2*>(row + 2) = w1;
    }
  }
  if (a.res2) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0) red[tid >> 5] = part;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int q = 0; q < 8; ++q) t += red[q];
      if (a.sym && ti != tj) t *= 2.0;
      atomicAdd(&a.res2[s], t);
    }
  }
}

// The FP32 product on packed multiply-adds (fma.rn.f32x2).  Bound by the FP32
// pipe (128 multiply-adds per clock and SM), so 64 threads hold 8 x 8 outputs
// each: 4 shared-memory loads of 16 bytes feed 64 multiply-adds, against 16 for
// 6 loads with 4 x 4 outputs.  The rows and columns of a thread are two runs of
// four, 32 apart, which keeps those loads free of bank conflicts; the next k
// slice comes in by cp.async (B) and through registers (A, transposed).  64 x 64
// tiles keep the padding of ragged dims small: 128 x 64 tiles measured 50.8
// TFLOP/s against 58.0 at 448 dims.  Every output is one chain over ascending k.
// Newton-Schulz on 125 submatrices of ~1100 dims: 106.5 -> 68.7 ms a build.
constexpr int FP = 68;  // pitch of the A slice: rows 16-byte aligned

__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}

__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

__device__ __forceinline__ void cp_async16(void* s, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(s))),
               "l"(g)
               : "memory");
}

__global__ void __launch_bounds__(64, 6) k_gemm_f32(const __grid_constant__ GemmF32Args a) {
  __shared__ __align__(16) float As[2][TK][FP];  // As[.][k][m]
  __shared__ __align__(16) float Bs[2][TK][TM];  // Bs[.][k][n]
  __shared__ double red[2];
  const int4 item = a.items[blockIdx.x];
  const int s = item.x, ti = item.y, tj = item.z;
  if (a.state != nullptr && a.state[s] == a.skip_state) return;
  const int ld = a.w.ld[s];
  const int64_t off = a.w.off[s];
  const float* Ab = a.A + off + int64_t(ti) * TM * ld;
  const float* Bb = a.B + off + int64_t(tj) * TM;
  const int tid = threadIdx.x;
  const int tx = tid & 7, ty = tid >> 3;
  // loader: A 16 rows x 16 k a pass, B 4 k x 64 columns a pass, four passes
  const int a_row = tid >> 2, a_k = (tid & 3) * 4;
  const int b_k = tid >> 4, b_n = (tid & 15) * 4;
  float4 ra[4];
  unsigned long long acc[8][4];  // column pairs
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0;
  auto fetch = [&](int kt, int buf) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      cp_async16(&Bs[buf][b_k + 4 * q][b_n], Bb + int64_t(kt * TK + b_k + 4 * q) * ld + b_n);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      ra[q] = *reinterpret_cast<const float4*>(Ab + int64_t(a_row + 16 * q) * ld + kt * TK + a_k);
  };
  auto settle = [&](int buf) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      As[buf][a_k + 0][a_row + 16 * q] = ra[q].x;
      As[buf][a_k + 1][a_row + 16 * q] = ra[q].y;
      As[buf][a_k + 2][a_row + 16 * q] = ra[q].z;
      As[buf][a_k + 3][a_row + 16 * q] = ra[q].w;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  };
  const int nk = ld / TK;
  fetch(0, 0);
  settle(0);
  __syncthreads();
  for (int kt = 0; kt < nk; ++kt) {
    const int buf = kt & 1;
    if (kt + 1 < nk) fetch(kt + 1, buf ^ 1);
#pragma unroll
    for (int k = 0; k < TK; ++k) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][k][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][k][32 + ty * 4]);
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][k][tx * 4]);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][k][32 + tx * 4]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const unsigned long long aa = pack2(av[i], av[i]);
        fma2(acc[i][0], aa, b0.x);
        fma2(acc[i][1], aa, b0.y);
        fma2(acc[i][2], aa, b1.x);
        fma2(acc[i][3], aa, b1.y);
      }
    }
    if (kt + 1 < nk) settle(buf ^ 1);
    __syncthreads();
  }

  // epilogue
  const int n = a.w.n[s];
  float* Cb = a.C + off;
  const float* C0b = a.C0 ? a.C0 + off : nullptr;
  const float alpha = float(a.alpha), beta = float(a.beta), diag = float(a.diag);
  Sum3 rest;          // sum of squares off the diagonal
  double part = 0.0;  // and on it
  const int c0 = tj * TM + tx * 4;
  float v[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = ti * TM + (i >> 2) * 32 + ty * 4 + (i & 3);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (C0b) z = *reinterpret_cast<const float4*>(C0b + int64_t(r) * ld + c0 + 32 * h);
      const float zc[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const unsigned long long w = acc[i][2 * h + (q >> 1)];
        const int c = c0 + 32 * h + q;
        float x = alpha * __uint_as_float(uint32_t(q & 1 ? w >> 32 : w));
        if (C0b) x = fmaf(beta, zc[q], x);
        if (r == c && r < n) {
          if (a.diag != 0.0) x += diag;
          if (a.res2) {
            const double e = double(x) - 1.0;
            part = fma(e, e, part);
          }
        } else if (a.res2) {
          rest.add_square(x);
        }
        v[i][4 * h + q] = x;
      }
      *reinterpret_cast<float4*>(Cb + int64_t(r) * ld + c0 + 32 * h) =
          make_float4(v[i][4 * h], v[i][4 * h + 1], v[i][4 * h + 2], v[i][4 * h + 3]);
    }
  }
  if (a.sym && ti != tj) {
    const int r0 = ti * TM + ty * 4;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float* row = Cb + int64_t(c0 + 32 * (j >> 2) + (j & 3)) * ld + r0;
      *reinterpret_cast<float4*>(row) = make_float4(v[0][j], v[1][j], v[2][j], v[3][j]);
      *reinterpret_cast<float4*>(row + 32) = make_float4(v[4][j], v[5][j], v[6][j], v[7][j]);
    }
  }
  if (a.res2) {
    part += rest.value();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0) red[tid >> 5] = part;
    __syncthreads();
    if (tid == 0) atomicAdd(&a.res2[s], (red[0] + red[1]) * (a.sym && ti != tj ? 2.0 : 1.0));
  }
}

}  // namespace

cudaError_t launch_gemm_f64(const GemmF64Args& a, cudaStream_t st) {
  if (a.nitems <= 0) return cudaSuccess;
  k_gemm_f64<<<a.nitems, 256, 0, st>>>(a);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_gemm_f32(const GemmF32Args& a, cudaStream_t st) {
  if (a.nitems <= 0) return cudaSuccess;
  k_gemm_f32<<<a.nitems, 64, 0, st>>>(a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace submat
