// submat_dense_sign_noalloc: the dense one-block case of the sign evaluation
// that allocates no memory at all.
//
// Who needs it: callers that may not call cudaMalloc or cudaMallocHost --
// codes that reserve the whole device up front for their own memory pool (a
// molecular-dynamics engine that hands out slices of one arena), runtimes
// whose allocator forbids foreign allocations, and code paths where an
// allocation would implicitly synchronise the device in the middle of a
// time step.  They pass device buffers for K and D; all scratch (the
// Newton-Schulz iterates, X^2, the tile list and the convergence state) lives
// in one file-scope device array of fixed size that every GPU loading this
// library holds until the process exits.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>

#include "common.cuh"
#include "submat.h"

namespace submat {

int num_sms();

namespace {

constexpr int NA_MAX_N = SUBMAT_NOALLOC_MAX_N;  // largest accepted dimension
constexpr int NA_LD = NA_MAX_N;                 // buffers are sized for the maximum
constexpr size_t NA_ELEMS = size_t(NA_LD) * NA_LD;
constexpr int NA_MAX_CTAS = 1024;               // partial results a grid keeps

// small-state block at the end of the scratch array
struct NaSmall {
  unsigned arrived;  // grid barrier: arrivals since the launch
  int flags, iters, notconv;
  double part[2][NA_MAX_CTAS];  // per CTA: row abs-sum maximum, sum of squares (residual)
  int bad[NA_MAX_CTAS];         // per CTA: a NaN or Inf among its entries
};

constexpr size_t NA_SMALL_DOUBLES = (sizeof(NaSmall) + sizeof(double) - 1) / sizeof(double);

// X0 | X1 | Y | small state.  6 MiB for n <= 512.
__device__ __align__(256) double g_noalloc_scratch[3 * NA_ELEMS + NA_SMALL_DOUBLES];

// Device address of g_noalloc_scratch on the current device, looked up on
// every call: the lookup is on the host and allocates nothing, and a cached
// address would go stale if the caller reset the device (the module, and
// with it the array, is then loaded again elsewhere).
submat_status setup(double** out) {
  void* p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess || !p) {
    set_error("cudaGetSymbolAddress of the scratch array failed: %s", cudaGetErrorString(e));
    return SUBMAT_ERR_CUDA;
  }
  *out = static_cast<double*>(p);
  return SUBMAT_OK;
}

constexpr int NA_THREADS = 256;
constexpr int NA_KPARTS = 4;  // the sum over k is split over four 64-thread groups
constexpr unsigned long long NA_LIMIT_NS = 2000000000ull;  // longest wait at the grid barrier

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the CTA, in warp order; thread 0 has it.
__device__ __forceinline__ double cta_sum(double v, double* red) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int q = 0; q < NA_THREADS / 32; ++q) t += red[q];
  return t;
}

// Barrier over the grid (a cooperative launch: every CTA is resident).  The
// wait is bounded: false for the whole CTA when it ran out.
__device__ bool grid_barrier(NaSmall* sm, unsigned* epoch) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned target = ++*epoch * gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&sm->arrived) : "memory");
    const unsigned long long t0 = now_ns();
    unsigned v;
    int good = 1;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&sm->arrived) : "memory");
      if (v >= target) break;
      if (now_ns() - t0 > NA_LIMIT_NS) { good = 0; break; }
    }
    __threadfence();
    ok = good;
    if (!good) atomicOr(&sm->flags, FLAG_TIMEOUT);
  }
  __syncthreads();
  return ok != 0;
}

// Fixed-order sum (or maximum) of one partial result per CTA, in every thread.
// Other CTAs wrote them before the barrier: read past L1.  One warp does the
// work: each FP64 instruction of a warp holds its pipe for 64 clocks.
__device__ double all_ctas(const double* part, bool maximum, double* red) {
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = 0.0;
    for (int q = threadIdx.x; q < int(gridDim.x); q += 32) {
      const double x = __ldcg(part + q);
      v = maximum ? fmax(v, x) : v + x;
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double x = __shfl_xor_sync(0xffffffffu, v, o);
      v = maximum ? fmax(v, x) : v + x;
    }
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  return red[0];
}

// Rows a and b of A and B for one 8 x 8 block into shared memory, past L1
__device__ __forceinline__ void na_stage(const double* A, const double* B, int a, int b, int ld, double* dst) {
  const int half = ld / 2, pitch = ld + 2;
  for (int e = threadIdx.x; e < 16 * half; e += NA_THREADS) {
    const int row = e / half, c = (e - row * half) * 2;
    const double* src = row < 8 ? A + int64_t(a * 8 + row) * ld + c : B + int64_t(b * 8 + row - 8) * ld + c;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst + row * pitch + c))),
                 "l"(src)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void na_block(int it, int T, int* a, int* b) {
  int x = 0, rem = it;
  while (rem >= T - x) { rem -= T - x; ++x; }
  *a = x;
  *b = x + rem;
}

// C = alpha A B + beta C0 on the CTA's share of the 8 x 8 blocks on or above
// the diagonal, each written to its mirrored place too (all matrices are
// symmetric, so B is read by rows).  Returns, in thread 0, the share's part of
// ||C - I_n||_F^2.
__device__ double na_product(const double* A, const double* B, const double* C0, double* C, double alpha,
                             double beta, int n, int ld, double* rows, double (*sum)[NA_KPARTS][64], double* red) {
  const int T = ld / 8, items = T * (T + 1) / 2, pitch = ld + 2;
  const int g = threadIdx.x >> 6, e = threadIdx.x & 63, i = e >> 3, j = e & 7;
  double part = 0.0;
  int buf = 0, a = 0, b = 0;
  __syncthreads();
  if (int(blockIdx.x) < items) {
    na_block(blockIdx.x, T, &a, &b);
    na_stage(A, B, a, b, ld, rows);
  }
  for (int it = blockIdx.x; it < items; it += gridDim.x, buf ^= 1) {
    const int r = a * 8 + i, c = b * 8 + j;
    const bool diagonal = a == b;
    const double* pa = rows + (buf * 16 + i) * pitch;
    const double* pb = rows + (buf * 16 + 8 + j) * pitch;
    double c0 = 0.0;
    if (C0 && g == 0) c0 = __ldcg(C0 + int64_t(r) * ld + c);
    if (it + int(gridDim.x) < items) {  // the next block's rows meanwhile
      na_block(it + gridDim.x, T, &a, &b);
      na_stage(A, B, a, b, ld, rows + (buf ^ 1) * 16 * pitch);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    double acc0 = 0.0, acc1 = 0.0;
#pragma unroll 4
    for (int k = 2 * g; k < ld; k += 2 * NA_KPARTS) {
      const double2 x = *reinterpret_cast<const double2*>(pa + k);
      const double2 y = *reinterpret_cast<const double2*>(pb + k);
      acc0 = fma(x.x, y.x, acc0);
      acc1 = fma(x.y, y.y, acc1);
    }
    sum[buf][g][e] = acc0 + acc1;
    __syncthreads();  // also: these rows may be overwritten
    if (g == 0) {
      double v = alpha * ((sum[buf][0][e] + sum[buf][1][e]) + (sum[buf][2][e] + sum[buf][3][e]));
      if (C0) v = fma(beta, c0, v);
      C[int64_t(r) * ld + c] = v;
      if (!diagonal) C[int64_t(c) * ld + r] = v;
      const double d = v - (r == c && r < n ? 1.0 : 0.0);
      part = fma(diagonal ? d : 2.0 * d, d, part);
    }
  }
  return cta_sum(part, red);
}

// The whole evaluation in one cooperative launch, one CTA per SM.  Bound by the
// FP64 pipe (2 multiply-adds per clock and SM) and, at small n, by the two grid
// barriers of an iteration (~2 us each), so the work is cut into 8 x 8 blocks:
// at n = 191, 300 of them over 152 SMs where 64 x 64 tiles keep 6 SMs busy.
// Four groups of 64 threads share a block's sum to cover the pipe's latency.
// n = 191: 6.12 -> 0.38 ms a call (one launch per product before).
__global__ void __launch_bounds__(NA_THREADS, 1) k_na_sign(int n, int ld, const double* K, double mu, double* D,
                                                           double* X0, double* X1, double* Y, NaSmall* sm,
                                                           double tol, double floor_thr, int max_iter) {
  extern __shared__ __align__(16) double rows[];  // two sets of 8 + 8 rows
  __shared__ double sum[2][NA_KPARTS][64];
  __shared__ double red[NA_THREADS / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nwarps = gridDim.x * (NA_THREADS / 32);
  unsigned epoch = 0;
  // beta = min(max row abs-sum, ||K - mu I||_F)
  double mx = 0.0, fro = 0.0;
  bool bad = false;
  for (int r = blockIdx.x * (NA_THREADS / 32) + warp; r < n; r += nwarps) {
    double rs = 0.0;
    for (int c = lane; c < n; c += 32) {
      double v = K[int64_t(r) * n + c];
      if (r == c) v -= mu;
      if (!isfinite(v)) bad = true;
      rs += fabs(v);
      fro += v * v;
    }
    mx = fmax(mx, warp_sum(rs));
  }
  if (lane == 0) red[warp] = mx;
  const int any_bad = __syncthreads_or(bad);
  for (int q = 0; q < NA_THREADS / 32; ++q) mx = fmax(mx, red[q]);
  fro = cta_sum(fro, red);
  if (threadIdx.x == 0) {
    sm->part[0][blockIdx.x] = mx;
    sm->part[1][blockIdx.x] = fro;
    sm->bad[blockIdx.x] = any_bad;
  }
  if (!grid_barrier(sm, &epoch)) return;
  int rejected = 0;
  for (int q = threadIdx.x; q < int(gridDim.x); q += NA_THREADS) rejected |= __ldcg(&sm->bad[q]);
  if (__syncthreads_or(rejected)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) sm->flags = FLAG_NONFINITE;
    return;
  }
  double b = fmin(all_ctas(sm->part[0], true, red), sqrt(all_ctas(sm->part[1], false, red)));
  const bool iterate = b > 0.0 && isfinite(b);
  if (!iterate) b = 1.0;
  if (threadIdx.x < 32) b = 1.0 / b;
  if (threadIdx.x == 0) red[1] = b;
  __syncthreads();
  const double ib = red[1];
  for (int e = blockIdx.x * NA_THREADS + threadIdx.x; e < ld * ld; e += gridDim.x * NA_THREADS) {
    const int r = e / ld, c = e - r * ld;
    double v = 0.0;
    if (r < n && c < n) {
      v = K[int64_t(r) * n + c];
      if (r == c) v -= mu;
      v *= ib;
    }
    X0[e] = v;
  }
  if (!grid_barrier(sm, &epoch)) return;
  double *X = X0, *Xn = X1;
  double prev = 1e300;
  int iters = 0, notconv = 0, diverged = 0;
  for (bool last = !iterate; !last;) {
    const double res = na_product(X, X, nullptr, Y, 1.0, 0.0, n, ld, rows, sum, red);
    // two sets of partial sums: a CTA may still read the previous square's
    double* part = sm->part[iters & 1];
    if (threadIdx.x == 0) part[blockIdx.x] = res;
    if (!grid_barrier(sm, &epoch)) return;
    // every CTA takes the same decision from the same sums
    double r = all_ctas(part, false, red);
    if (threadIdx.x < 32) r = sqrt(r / double(n));
    if (threadIdx.x == 0) red[1] = r;
    __syncthreads();
    r = red[1];
    ++iters;
    if (!isfinite(r) || r > 1e6) {
      notconv = diverged = 1;
      break;
    }
    if (r <= tol || (r < floor_thr && r > 0.5 * prev)) {
      last = true;
    } else if (iters >= max_iter) {
      last = true;
      notconv = 1;
    }
    prev = r;
    na_product(X, Y, X, Xn, -0.5, 1.5, n, ld, rows, sum, red);
    if (!grid_barrier(sm, &epoch)) return;
    double* t = X;
    X = Xn;
    Xn = t;
  }
  for (int e = blockIdx.x * NA_THREADS + threadIdx.x; e < n * n; e += gridDim.x * NA_THREADS) {
    const int r = e / n, c = e - r * n;
    D[e] = (r == c ? 0.5 : 0.0) - 0.5 * __ldcg(X + int64_t(r) * ld + c);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    sm->iters = iters;
    sm->notconv = notconv;
    if (diverged) atomicOr(&sm->flags, FLAG_DIVERGED);
  }
}

}  // namespace

}  // namespace submat

extern "C" submat_status submat_dense_sign_noalloc(int n, const double* K_dev, double mu,
                                                   double* D_dev, int* iters_out, void* stream) {
  using namespace submat;
  clear_error();
  if (n < 1 || n > NA_MAX_N) {
    set_error("submat_dense_sign_noalloc: n = %d outside [1, %d] (the fixed scratch holds %d x %d)",
              n, NA_MAX_N, NA_MAX_N, NA_MAX_N);
    return SUBMAT_ERR_INVALID_ARG;
  }
  if (!K_dev || !D_dev || !std::isfinite(mu)) {
    set_error("submat_dense_sign_noalloc: null buffer or non-finite mu");
    return SUBMAT_ERR_INVALID_ARG;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  double* base = nullptr;
  submat_status s = setup(&base);
  if (s != SUBMAT_OK) return s;
  double* X0 = base;
  double* X1 = base + NA_ELEMS;
  double* Y = base + 2 * NA_ELEMS;
  NaSmall* sm = reinterpret_cast<NaSmall*>(base + 3 * NA_ELEMS);
  int ld = (n + 7) / 8 * 8;
  const int max_iter = 100;
  const int blocks = ld / 8 * (ld / 8 + 1) / 2;  // 8 x 8 blocks on or above the diagonal
  const int grid = std::min(std::min(blocks, num_sms()), NA_MAX_CTAS);
  double tol = 1e-14, floor_thr = 1e-9;
  const int smem = 2 * 16 * (ld + 2) * int(sizeof(double));
  SM_CUDA(cudaFuncSetAttribute(k_na_sign, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  SM_CUDA(cudaMemsetAsync(sm, 0, offsetof(NaSmall, part), st));
  int max_it = max_iter;
  void* args[] = {&n, &ld, &K_dev, &mu, &D_dev, &X0, &X1, &Y, &sm, &tol, &floor_thr, &max_it};
  SM_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_na_sign), dim3(unsigned(grid)),
                                      dim3(NA_THREADS), args, size_t(smem), st));
  SM_KCHECK();
  int tail[4] = {0, 0, 0, 0};  // arrived, flags, iters, notconv
  static_assert(offsetof(NaSmall, part) >= sizeof(tail), "the state precedes the partial sums");
  SM_CUDA(cudaMemcpyAsync(tail, sm, sizeof(tail), cudaMemcpyDeviceToHost, st));
  SM_CUDA(cudaStreamSynchronize(st));
  if (tail[1] & FLAG_NONFINITE) {
    set_error("K holds a NaN or Inf value");
    return SUBMAT_ERR_NONFINITE;
  }
  if (tail[1] & FLAG_TIMEOUT) {
    set_error("a bounded device wait timed out");
    return SUBMAT_ERR_TIMEOUT;
  }
  if (iters_out) *iters_out = tail[2];
  if (tail[3]) {
    set_error("Newton-Schulz reached %d iterations without converging (D written)", max_iter);
    return SUBMAT_ERR_NOT_CONVERGED;
  }
  return SUBMAT_OK;
}
