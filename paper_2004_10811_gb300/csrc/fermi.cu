// Finite temperature: D = f(K - mu I) with the Fermi function
// f(x) = 1 / (1 + exp(x / kT)) in place of (1 - signum(x)) / 2 (Section IV-F,
// last paragraph: the eigendecomposition route extends to finite temperature
// by replacing signum; the Conclusion names the generalisation).
//
// f(x) = (1 - tanh(x / (2 kT))) / 2, so every submatrix needs tanh of its
// scaled matrix X = a / sigma, whose spectrum lies in [-1, 1].  tanh(c x),
// c = sigma / (2 kT), is analytic in the strip |Im x| < pi / (2c), so its
// Chebyshev series on [-1, 1] converges geometrically; the series is cut at
// the odd degree m whose tail sum_{k > m} |c_k| (a bound on the truncation
// error, |T_k| <= 1 on [-1, 1]) is below the precision's tolerance.
//
// Evaluation, baby steps and giant steps (all polynomials in X commute and are
// symmetric, so every product is a symmetric one):
//   baby:  T_2 = 2 X^2 - I, T_{k+2} = 2 T_2 T_k - T_{k-2} for the odd
//          k = 1..15 (eight stored), Y = T_16 = 2 T_9 T_7 - T_2;
//   fold:  with k = 16 j + i, T_{16j+i} = 2 T_{16j} T_i - T_{16j-i}, so the
//          series becomes sum_j R_j T_{16j} with R_j a combination of the
//          stored odd T_i, and T_{16j}(X) = T_j(Y);
//   giant: Clenshaw in Y: b_j = R_j + 2 Y b_{j+1} - b_{j+2}, p = R_0 + Y b_1 - b_2.
// That is 9 + ceil((m + 1) / 16) - 1 products for degree m.
//
// The scale sigma is common to a wave (one polynomial per wave): each
// submatrix starts at X = a / beta_bound (beta_bound = min(max row abs-sum,
// ||a||_F)), the first square gives the rigorous bound
// rho(X)^2 <= ||X^2||_inf (rounding included), and sigma is the largest
// beta_bound * sqrt(||X^2||_inf) of the wave, which roughly halves the degree
// against beta_bound alone.
//
// dN/dmu = sum_j sum_{c in block j} [f'(a_j)]_cc with f' = f (1 - f) / kT as a
// matrix function (d/dmu f(a - mu I) = -f'(a - mu I)), i.e. the adjoint's
// L_f(a_j, I): from the extracted columns of F_j = f(a_j) as
// sum_c (F_cc - sum_k F_kc^2) / kT.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "plan.cuh"
#include "rns.cuh"

namespace submat {

// ---------------------------------------------------------------------------
// host: the Chebyshev series of tanh(c x) and its baby-step / giant-step form
// ---------------------------------------------------------------------------

// Coefficients c_k, k < ncoef, of tanh(c x) on [-1, 1] from its values at the
// N Chebyshev nodes x_n = cos(theta_n), theta_n = pi (2n + 1) / (2N) (the
// discrete cosine transform of the first kind; exact for degree < N).
// cos(k theta_n) = cos(pi j / (2N)) with j = k (2n + 1) mod 4N, read from a
// table, so no rounding accumulates with k.
static submat_status cheb_coefficients(double c, int N, int ncoef, std::vector<double>* out,
                                       const ChebTransform& transform) {
  const int64_t P = 4 * int64_t(N);
  std::vector<double> cosv(static_cast<size_t>(P)), g(static_cast<size_t>(N));
  for (int64_t j = 0; j < P; ++j) cosv[size_t(j)] = std::cos(M_PI * double(j) / (2.0 * N));
  for (int n = 0; n < N; ++n) g[n] = std::tanh(c * cosv[size_t(2 * n + 1)]);
  out->assign(ncoef, 0.0);
  if (transform) {
    SM_TRY(transform(g, cosv, ncoef, out->data()));
  } else {
    for (int k = 0; k < ncoef; ++k) {
      double acc = 0.0;
      int64_t j = k, step = 2 * int64_t(k) % P;  // j = k (2n + 1) mod 4N
      for (int n = 0; n < N; ++n) {
        acc += g[n] * cosv[size_t(j)];
        j += step;
        if (j >= P) j -= P;
      }
      (*out)[k] = acc;
    }
  }
  for (int k = 0; k < ncoef; ++k) (*out)[k] = (k == 0 ? 1.0 : 2.0) * (*out)[k] / N;
  return SUBMAT_OK;
}

submat_status fermi_poly(double c, double tol, int max_degree, FermiPoly* out, const ChebTransform& transform) {
  if (!(c > 0.0) || !std::isfinite(c)) {
    set_error("finite temperature: bad scale c = %g", c);
    return SUBMAT_ERR_INVALID_ARG;
  }
  FermiPoly& P = *out;
  P = FermiPoly{};
  std::vector<double> coef;
  int m = -1;
  double tail = 0.0;
  for (int N = 256;; N *= 2) {
    const int ncoef = N / 2;
    SM_TRY(cheb_coefficients(c, N, ncoef, &coef, transform));
    // coefficients below the rounding floor of the transform are noise, not
    // truncation: the series counts up to the last one above it
    double cmax = 0.0;
    for (double v : coef) cmax = std::max(cmax, std::fabs(v));
    const double floor = 64.0 * 0x1p-52 * cmax;
    int last = 0;
    for (int k = 0; k < ncoef; ++k)
      if (std::fabs(coef[k]) > floor) last = k;
    // the series must reach the floor inside the first half of the computed range
    if (last > ncoef / 2) {
      if (N / 4 > max_degree + 1) break;  // would need a degree beyond the cap
      continue;
    }
    // smallest odd m with sum_{m < k <= last} |c_k| <= tol
    std::vector<double> suffix(ncoef + 1, 0.0);
    for (int k = last; k >= 0; --k) suffix[k] = suffix[k + 1] + std::fabs(coef[k]);
    for (int k = 1; k < ncoef; k += 2)
      if (suffix[k + 1] <= tol) { m = k; tail = suffix[k + 1]; break; }
    break;
  }
  if (m < 0 || m > max_degree) {
    set_error("finite temperature: tanh(%g x) needs a Chebyshev degree above %d (kT too small for the "
              "spectral scale)", c, max_degree);
    return SUBMAT_ERR_UNSUPPORTED;
  }
  P.m = m;
  P.trunc = tail;
  constexpr int S = kFermiBaby;
  P.blocks = (m + 1 + S - 1) / S;
  std::vector<double> a(size_t(P.blocks) * S, 0.0);
  for (int k = 1; k <= m; k += 2) a[k] = coef[k];  // tanh is odd: even terms vanish
  P.r.assign(size_t(P.blocks) * (S / 2), 0.0);
  for (int j = P.blocks - 1; j >= 1; --j)
    for (int i = 1; i < S; i += 2) {
      const double ck = a[size_t(S) * j + i];
      P.r[size_t(j) * (S / 2) + i / 2] = 2.0 * ck;
      a[size_t(S) * (j - 1) + (S - i)] -= ck;
    }
  for (int i = 1; i < S; i += 2) P.r[i / 2] = a[i];
  return SUBMAT_OK;
}

int fermi_clenshaw_exponent(const FermiPoly& P) {
  // The terms are polynomials of degree m or less: their maximum on [-1, 1] is
  // at most 1 / cos(pi / 4) times that over 2 (m + 1) Chebyshev nodes (Ehlich
  // and Zeller 1964).  They are odd or even, so half of the nodes suffice.
  constexpr int H = kFermiBaby / 2;
  const int nodes = 2 * (P.m + 1);
  double mx = 0.0;
  for (int i = 0; 2 * i < nodes; ++i) {
    const double th = M_PI * (2 * i + 1) / (2.0 * nodes), y = std::cos(kFermiBaby * th);
    double t[H], b1 = 0.0, b2 = 0.0;
    for (int q = 0; q < H; ++q) t[q] = std::cos((2 * q + 1) * th);
    for (int j = P.blocks - 1; j >= 0; --j) {
      double R = 0.0;
      for (int q = 0; q < H; ++q) R += P.r[size_t(j) * H + q] * t[q];
      const double b = R + (j == 0 ? 1.0 : 2.0) * y * b1 - b2;  // at j = 0: p
      mx = std::max(mx, std::fabs(b));
      b2 = b1;
      b1 = b;
    }
  }
  return std::max(0, int(std::ceil(std::log2(std::max(1e-300, 1.4143 * mx)))));
}

namespace {

// sums[k] = sum_n g_n cos(k theta_n), one thread per k in ascending n, as the host
// does.  The N^2 / 2 terms took the host 10 ms an evaluation at degree ~400 (N =
// 2048), a third of it; here a chain of N multiply-adds per warp, spread over the
// SMs, takes ~0.1 ms: FP32 mu search 171.3 -> 120.4 ms, FP64 build
// of 240 submatrices 28.3 -> 26.4.
__global__ void __launch_bounds__(32) k_cheb_sums(int N, int ncoef, const double* __restrict__ g,
                                                  const double* __restrict__ cosv, double* __restrict__ sums) {
  const int k = blockIdx.x * 32 + threadIdx.x;
  if (k >= ncoef) return;
  const int P = 4 * N, step = 2 * k;  // j = k (2n + 1) mod 4N; 2k < 4N
  int j = k;
  double acc = 0.0;
#pragma unroll 8
  for (int n = 0; n < N; ++n) {
    acc = fma(g[n], cosv[j], acc);
    j += step;
    if (j >= P) j -= P;
  }
  sums[k] = acc;
}

// X <- r_s X and T2 <- r_s^2 (T2 + I) - I (the square rescaled), r_s = ratio[s]
template <typename T>
__global__ void k_fermi_rescale(WaveDev w, T* __restrict__ X, T* __restrict__ T2, const double* __restrict__ ratio) {
  const int s = blockIdx.y;
  const double r = ratio[s];
  if (r == 1.0) return;
  const int ld = w.ld[s], n = w.n[s];
  const int64_t total = int64_t(ld) * ld, base = w.off[s];
  const T rt = T(r), r2 = T(r * r), dshift = T(r * r - 1.0);
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
       e += int64_t(gridDim.x) * blockDim.x) {
    const int row = int(e / ld), col = int(e - int64_t(row) * ld);
    X[base + e] *= rt;
    if (!T2) continue;
    T v = r2 * T2[base + e];
    if (row == col && row < n) v += dshift;
    T2[base + e] = v;
  }
}

// M <- r_s^2 M (the derivative part of the rescaled square)
template <typename T>
__global__ void k_fermi_scale_sq(WaveDev w, T* __restrict__ M, const double* __restrict__ ratio) {
  const int s = blockIdx.y;
  const double r = ratio[s];
  if (r == 1.0) return;
  const int ld = w.ld[s];
  const int64_t total = int64_t(ld) * ld, base = w.off[s];
  const T r2 = T(r * r);
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
       e += int64_t(gridDim.x) * blockDim.x)
    M[base + e] *= r2;
}

// W = sum_i r_i T_{2i+1} - B (B may be null): the giant-step coefficient R_j
// less the Clenshaw term b_{j+2}.  W may be B (each entry is read, then
// written by the same thread).  With route, only the submatrices of the chains.
struct CombArgs {
  double r[kFermiBaby / 2];
};

template <typename T>
__global__ void __launch_bounds__(256) k_cheb_comb(WaveDev w, const T* __restrict__ odd, int64_t stride,
                                                   CombArgs ca, const T* B, T* W, const int* __restrict__ route) {
  const int s = blockIdx.y;
  if (route && route[s] == ST_ACTIVE) return;
  const int ld = w.ld[s];
  const int64_t total = int64_t(ld) * ld, base = w.off[s];
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
       e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t i = base + e;
    T acc = B ? -B[i] : T(0);
#pragma unroll
    for (int q = 0; q < kFermiBaby / 2; ++q) acc = fma(T(ca.r[q]), odd[int64_t(q) * stride + i], acc);
    W[i] = acc;
  }
}

// The same on the 64 x 64 upper tiles only, which is all that a symmetric product
// reads of its C0: bound by memory traffic, so this halves it.
// FP32 mu search on 216 submatrices of 420-480 dims: 186.6 -> 171.3 ms.
template <typename T>
__global__ void __launch_bounds__(256) k_cheb_comb_upper(WaveDev w, const int4* __restrict__ items,
                                                         const T* __restrict__ odd, int64_t stride, CombArgs ca,
                                                         const T* B, T* W, const int* __restrict__ route) {
  constexpr int V = 16 / sizeof(T);  // entries of a 16-byte access
  struct alignas(16) Vec { T v[V]; };
  const int4 item = items[blockIdx.x];
  if (route && route[item.x] == ST_ACTIVE) return;
  const int ld = w.ld[item.x];
  const int64_t base = w.off[item.x] + int64_t(item.y) * 64 * ld + item.z * 64;
  for (int e = threadIdx.x; e < 64 * 64 / V; e += 256) {
    const int64_t i = base + int64_t(e / (64 / V)) * ld + e % (64 / V) * V;
    Vec acc{};
    if (B) {
      const Vec b = *reinterpret_cast<const Vec*>(B + i);
#pragma unroll
      for (int k = 0; k < V; ++k) acc.v[k] = -b.v[k];
    }
#pragma unroll
    for (int q = 0; q < kFermiBaby / 2; ++q) {
      const Vec t = *reinterpret_cast<const Vec*>(odd + int64_t(q) * stride + i);
#pragma unroll
      for (int k = 0; k < V; ++k) acc.v[k] = fma(T(ca.r[q]), t.v[k], acc.v[k]);
    }
    *reinterpret_cast<Vec*>(W + i) = acc;
  }
}

dim3 fermi_grid(const Wave& wv) {
  int64_t bx = (wv.max_ld2 + 256 * 8 - 1) / (256 * 8);
  bx = std::max<int64_t>(1, std::min<int64_t>(bx, 512));
  return dim3(unsigned(bx), unsigned(wv.count));
}

template <typename T> struct FermiGemm;
template <> struct FermiGemm<double> {
  using Args = GemmF64Args;
  static cudaError_t run(const Args& a, cudaStream_t st) { return launch_gemm_f64(a, st); }
  static cudaError_t scale(const WaveDev& w, const double* A, double* X, const double* b, int64_t m2,
                           cudaStream_t st) { return launch_scale_f64(w, A, X, b, m2, st); }
};
template <> struct FermiGemm<float> {
  using Args = GemmF32Args;
  static cudaError_t run(const Args& a, cudaStream_t st) { return launch_gemm_f32(a, st); }
  static cudaError_t scale(const WaveDev& w, const double* A, float* X, const double* b, int64_t m2,
                           cudaStream_t st) { return launch_scale_f32(w, A, X, b, m2, st); }
};

}  // namespace

size_t fermi_bytes_per_elem(int prec) {
  // A (FP64) + the eight odd T_k, T_2 / Y, and two Clenshaw buffers
  return 8 + size_t(kFermiBuffers) * (prec == SUBMAT_FP64 ? 8 : 4);
}

// The adjoint runs the same buffers twice: values and derivative parts.
size_t fermi_dual_bytes_per_elem(int prec) {
  return 8 + size_t(2 * kFermiBuffers) * (prec == SUBMAT_FP64 ? 8 : 4);
}

submat_status Plan::cheb_transform(const std::vector<double>& g, const std::vector<double>& cosv, int ncoef,
                                   double* sums, cudaStream_t st) {
  const size_t N = g.size(), need = N + cosv.size() + size_t(ncoef);
  if (need > cheb_cap) {  // kept by the plan; a larger N than before is rare
    SM_TRY(alloc(&d_cheb, need, "Chebyshev transform"));
    cheb_cap = need;
  }
  double* dc = d_cheb + N;
  double* ds = dc + cosv.size();
  SM_CUDA(cudaMemcpyAsync(d_cheb, g.data(), 8 * N, cudaMemcpyHostToDevice, st));
  SM_CUDA(cudaMemcpyAsync(dc, cosv.data(), 8 * cosv.size(), cudaMemcpyHostToDevice, st));
  k_cheb_sums<<<(ncoef + 31) / 32, 32, 0, st>>>(int(N), ncoef, d_cheb, dc, ds);
  SM_KCHECK();
  SM_CUDA(cudaMemcpyAsync(sums, ds, 8 * size_t(ncoef), cudaMemcpyDeviceToHost, st));
  SM_CUDA(cudaStreamSynchronize(st));
  return SUBMAT_OK;
}

// One wave.  Forward: D = (I - p(X)) / 2 on the extracted columns, with the
// trace and sum-of-squares partials for dN/dmu.  With Dbar (the adjoint):
// every matrix M of the evaluation carries a derivative part M' (dual
// numbers), (A B)' = A' B + A B', seeded with X' = G_j / sigma, G_j holding
// Dbar's block column j in the columns of block j; then p' = L_p(X, X') and
// L_f(a_j, G_j) = -1/2 p' is added into every stored block of Kbar that a_j
// came from (L_f(a, .) is self-adjoint in the Frobenius product for
// symmetric a).  The value part is evaluated exactly as in the forward path.
template <typename T>
submat_status Plan::fermi_wave(Wave& wv, int wi, const double* K, double mu, double* D, const double* Dbar, double* Kbar,
                               void* w, int64_t E, cudaStream_t st) {
  using G = FermiGemm<T>;
  using Args = typename G::Args;
  constexpr int S = kFermiBaby;
  const bool dual = Dbar != nullptr;
  double* A = static_cast<double*>(w);
  T* base = reinterpret_cast<T*>(A + E);
  T* odd = base;                  // T_1 = X, T_3, ..., T_15 at odd + q E
  T* T2 = base + (S / 2) * E;     // T_2, later Y = T_16
  T* bb[2] = {T2 + E, T2 + 2 * E};    // Clenshaw b_{j+1}, b_{j+2}
  // derivative parts, the same layout kFermiBuffers buffers further on
  const int64_t dofs = int64_t(kFermiBuffers) * E;
  auto dp = [&](const T* v) -> T* { return v ? const_cast<T*>(v) + dofs : nullptr; };
  const bool f64 = sizeof(T) == 8;
  // truncation tolerance of the series: below the products' own rounding
  const double tol_poly = f64 ? 1e-13 : 1e-8;
  SM_CUDA(cudaEventRecord(ev[0], st));
  SM_TRY(gather_wave(wv, K, mu, A, st));
  SM_CUDA(G::scale(wv.dev, A, odd, ns.beta, wv.max_ld2, st));
  if (dual) SM_CUDA(launch_bwd_seed<T>(g, wv, Dbar, ns.beta, dp(odd), 0, st));  // X' = G / beta
  SM_CUDA(cudaEventRecord(ev[1], st));
  int products = 0;
  auto gemm1 = [&](const Args& a) -> submat_status {
    size_t tk;
    SM_TRY(timer.start(KC_SIMT, st, &tk));
    SM_CUDA(G::run(a, st));
    SM_TRY(timer.stop(tk, st));
    return SUBMAT_OK;
  };
  // submatrices of the FP64 chains on a wave of residue products (null: all)
  const int* route = nullptr;
  // C = alpha A B + beta C0 + diag I (symmetric: A, B commute), and with
  // dual numbers C' = alpha (A' B + A B') + beta C0' (full tiles)
  auto gemm = [&](const T* Aop, const T* Bop, const T* C0, T* C, double alpha, double beta,
                  double diag) -> submat_status {
    Args a{};
    a.w = wv.dev; a.items = wv.sym64; a.nitems = wv.n_sym64;
    a.A = Aop; a.B = Bop; a.C0 = C0; a.C = C;
    a.alpha = alpha; a.beta = beta; a.diag = diag; a.sym = 1;
    a.res2 = nullptr; a.state = route; a.skip_state = ST_ACTIVE;
    if (dual) {  // derivative first: it reads the values of A, B (and C0 may alias C)
      Args d = a;
      d.items = wv.full64; d.nitems = wv.n_full64; d.sym = 0; d.diag = 0.0;
      d.A = dp(Aop); d.B = Bop; d.C0 = dp(C0); d.C = dp(C);
      SM_TRY(gemm1(d));
      d.A = Aop; d.B = dp(Bop); d.C0 = dp(C); d.beta = 1.0;
      SM_TRY(gemm1(d));
    }
    SM_TRY(gemm1(a));
    ++products;
    return SUBMAT_OK;
  };
  // T_2 = 2 X^2 - I at X = a / beta_bound, and from it the tight scale
  const bool residues = wi >= 0;  // FP64 forward only
  if (residues) {
    const RnsSum F = fermi_rns_sum();  // in A's memory, which has served its purpose
    for (int part = 0; part < rns_parts; ++part) {
      SM_CUDA(launch_rns_convert(wv.dev, reinterpret_cast<double*>(odd), nullptr, nullptr, 0, rns_residues(1),
                                 RnsFix{}, max_ld(wv), st, rns_parts, part));
      SM_TRY(rns_product(size_t(wi), 1, 1, F, nullptr, st, part));
    }
    SM_CUDA(launch_rns_cheb2(wv.dev, F, reinterpret_cast<double*>(T2), max_ld(wv), st));
    ++products;
  } else {
    SM_TRY(gemm(odd, odd, nullptr, T2, 2.0, 0.0, -1.0));
  }
  const CertSquare sq{f64 ? 0 : 1, T2, nullptr, 2.0f, -1.0f};
  SM_CUDA(cudaMemsetAsync(ns.cert, 0, sizeof(unsigned long long) * wv.count, st));
  SM_CUDA(launch_cert_rowsum(wv.dev, ns, sq, max_ld(wv), st));
  std::vector<unsigned long long> cert(wv.count), gersh(wv.count);
  std::vector<double> fro2(wv.count), beta(wv.count), ratio(wv.count, 1.0);
  SM_CUDA(cudaMemcpyAsync(cert.data(), ns.cert, 8 * wv.count, cudaMemcpyDeviceToHost, st));
  SM_CUDA(cudaMemcpyAsync(gersh.data(), ns.gersh, 8 * wv.count, cudaMemcpyDeviceToHost, st));
  SM_CUDA(cudaMemcpyAsync(fro2.data(), ns.fro2, 8 * wv.count, cudaMemcpyDeviceToHost, st));
  SM_CUDA(cudaMemcpyAsync(beta.data(), ns.beta, 8 * wv.count, cudaMemcpyDeviceToHost, st));
  SM_CUDA(cudaStreamSynchronize(st));
  double sigma = 0.0;
  std::vector<double> bound(wv.count, 0.0);
  const double eps0 = f64 ? 0x1p-50 : 0x1p-22, eps_ld = f64 ? 0x1p-52 : 0x1p-23;
  for (int s = 0; s < wv.count; ++s) {
    double cv = 0.0, gv = 0.0;
    std::memcpy(&cv, &cert[s], 8);
    std::memcpy(&gv, &gersh[s], 8);
    const double bnd = std::min(gv, std::sqrt(fro2[s])) * (1.0 + 1e-4);
    if (!(bnd > 0.0)) continue;  // a zero submatrix: f(0) = 1/2 whatever the scale
    const int ld = wv.host_ld[s];
    const double gx = gv / bnd;
    const double Gs = cv * (1.0 + ld * 0x1p-24) + (eps0 + eps_ld * ld) * gx * gx;
    bound[s] = beta[s] * std::min(1.0, std::sqrt(Gs));
    sigma = std::max(sigma, bound[s]);
  }
  sigma *= 1.0 + 1e-6;
  if (!(sigma > 0.0)) sigma = 1.0;
  for (int s = 0; s < wv.count; ++s)
    if (bound[s] > 0.0) ratio[s] = beta[s] / sigma;
  SM_CUDA(cudaMemcpyAsync(ns.cscale, ratio.data(), 8 * wv.count, cudaMemcpyHostToDevice, st));
  k_fermi_rescale<T><<<fermi_grid(wv), 256, 0, st>>>(wv.dev, odd, T2, ns.cscale);
  SM_KCHECK();
  if (dual) {  // X' and T_2' = 2 (X' X + X X') follow the scale linearly / quadratically
    k_fermi_rescale<T><<<fermi_grid(wv), 256, 0, st>>>(wv.dev, dp(odd), nullptr, ns.cscale);
    SM_KCHECK();
    k_fermi_scale_sq<T><<<fermi_grid(wv), 256, 0, st>>>(wv.dev, dp(T2), ns.cscale);
    SM_KCHECK();
  }
  if (residues) SM_TRY(rns_route(size_t(wi), reinterpret_cast<const double*>(odd), nullptr, &route, st));
  FermiPoly P;  // its transform waits for the stream
  SM_TRY(fermi_poly(sigma / (2.0 * opt.kT), tol_poly, kFermiMaxDegree, &P,
                    [&](const std::vector<double>& g, const std::vector<double>& cosv, int ncoef, double* sums) {
                      return cheb_transform(g, cosv, ncoef, sums, st);
                    }));
  fermi_degree = std::max(fermi_degree, P.m);
  fermi_trunc = std::max(fermi_trunc, P.trunc);
  T* out = bb[0];
  const bool chains = residues && static_cast<const int*>(h_pinned)[1] > 0;
  if (residues) SM_TRY(fermi_rns(wi, P, route, &products, st));
  if (chains) SM_TRY(collect_route(wv, st));
  if (!residues || chains) {
    const int counted = products;
    if (chains) SM_TRY(gemm(odd, odd, nullptr, T2, 2.0, 0.0, -1.0));
    // baby steps: T_3 = 2 T_2 X - X, T_{k+2} = 2 T_2 T_k - T_{k-2}
    for (int q = 1; q < S / 2; ++q)
      SM_TRY(gemm(T2, odd + int64_t(q - 1) * E, q >= 2 ? odd + int64_t(q - 2) * E : odd, odd + int64_t(q) * E,
                  2.0, -1.0, 0.0));
    // Y = T_16 = 2 T_9 T_7 - T_2, in T_2's buffer
    SM_TRY(gemm(odd + 4 * E, odd + 3 * E, T2, T2, 2.0, -1.0, 0.0));
    const T* Y = T2;
    // giant steps: Clenshaw in Y with the coefficients R_j
    auto comb = [&](int j, const T* B, T* W, bool upper) -> submat_status {
      CombArgs ca;
      for (int q = 0; q < S / 2; ++q) ca.r[q] = P.r[size_t(j) * (S / 2) + q];
      if (upper) k_cheb_comb_upper<T><<<wv.n_sym64, 256, 0, st>>>(wv.dev, wv.sym64, odd, E, ca, B, W, route);
      else k_cheb_comb<T><<<fermi_grid(wv), 256, 0, st>>>(wv.dev, odd, E, ca, B, W, route);
      SM_KCHECK();
      if (dual) {
        k_cheb_comb<T><<<fermi_grid(wv), 256, 0, st>>>(wv.dev, dp(odd), E, ca, dp(B), dp(W), nullptr);
        SM_KCHECK();
      }
      return SUBMAT_OK;
    };
    // b_j in bb[j mod 2], over b_{j+2}
    SM_TRY(comb(P.blocks - 1, nullptr, bb[(P.blocks - 1) & 1], false));
    for (int j = P.blocks - 2; j >= 0; --j) {
      // W = R_j - b_{j+2} (in place), then W += c Y b_{j+1}
      T* W = bb[j & 1];
      SM_TRY(comb(j, j < P.blocks - 2 ? W : nullptr, W, true));  // W is the product's C0
      SM_TRY(gemm(Y, bb[(j + 1) & 1], W, W, j == 0 ? 1.0 : 2.0, 1.0, 0.0));
    }
    if (chains) products = counted;  // the same products, on the other submatrices
  }
  SM_CUDA(cudaEventRecord(ev[2], st));
  // D = (I - p(X)) / 2 on the extracted columns, Tr and sum of squares
  SM_TRY(scatter_timed(wv, f64 ? 16.0 : 12.0, [&] {
    return launch_scatter_sq<T>(g, wv.dev, ns, out, D, d_trpart, d_sqpart, geom(wv), st);
  }, st));
  if (dual) SM_CUDA(launch_bwd_scatter_add<T>(g, wv, nb_max, dp(out), Kbar, st));
  SM_CUDA(cudaEventRecord(ev[3], st));
  SM_TRY(collect_wave(wv, st));
  SM_TRY(add_phase_times());
  for (int s = 0; s < wv.count; ++s) {
    res_iters[wv.first + s] = products;  // products of the evaluation, for the statistics
    const double n = wv.host_n[s];
    fermi_flops += 2.0 * n * n * n * products * (dual ? 3.0 : 1.0);
  }
  return SUBMAT_OK;
}

RnsSum Plan::fermi_rns_sum() const {
  double* w = static_cast<double*>(ws);
  return RnsSum{reinterpret_cast<long long*>(w), reinterpret_cast<int*>(w + (1 + kFermiBuffers) * ws_elems)};
}

// The recurrences of fermi_wave on exact residue products (rns.cuh), from X
// and T_2 in FP64, to p(X) in FP64 in the first Clenshaw buffer; submatrices of the
// chains are left as they are.  Every T_k has norm 1 or less; the Clenshaw terms
// move as b_j 2^-e (fermi_clenshaw_exponent).  Residue set 0 holds the factor that
// stays (T_2, then Y), set 1 the one that each pass renews; with the moduli in two
// parts, each product takes both from the fixed-point matrices instead.
// 240 submatrices of 219-384 dims (blocks of 13, 5 and 5 functions, kT 0.05): a
// build takes 33.4 ms, 15.4 of them in the products, against 574 ms with the FP64
// SIMT GEMM.
submat_status Plan::fermi_rns(int wi, const FermiPoly& P, const int* route, int* products, cudaStream_t st) {
  constexpr int H = kFermiBaby / 2;
  static_assert(H == RNS_COMB, "one coefficient per stored odd T_k");
  const Wave& wv = waves[size_t(wi)];
  const int64_t E = ws_elems;
  const int mld = max_ld(wv), e = fermi_clenshaw_exponent(P);
  const RnsSum F = fermi_rns_sum();
  auto fix = [&](int k) {  // the k-th FP64 buffer of fermi_wave: the odd T_k, T_2 / Y, two Clenshaw terms
    return RnsFix{F.f + (1 + k) * E, reinterpret_cast<unsigned short*>(F.g + E) + k * E};
  };
  auto odd = [&](int q) { return fix(q); };
  const RnsFix T2 = fix(H);
  const bool whole = rns_parts == 1;
  __nv_bfloat16* R[2] = {rns_residues(0), rns_residues(1)};
  __nv_bfloat16* made[2] = {whole ? R[0] : nullptr, whole ? R[1] : nullptr};  // written by the passes
  auto product = [&](const RnsFix& a, const RnsFix& b) -> submat_status {  // F = (set 0) (set 1) = a b
    ++*products;
    for (int part = 0; part < rns_parts; ++part) {
      if (!whole) {
        SM_CUDA(launch_rns_spread(wv.dev, route, a, R[0], mld, st, part));
        SM_CUDA(launch_rns_spread(wv.dev, route, b, R[1], mld, st, part));
      }
      SM_TRY(rns_product(size_t(wi), 0, 1, F, route, st, part));
    }
    return SUBMAT_OK;
  };
  auto dbl = [](const RnsFix& x) { return reinterpret_cast<double*>(x.hi); };
  SM_CUDA(launch_rns_convert(wv.dev, dbl(odd(0)), route, nullptr, 0, made[1], odd(0), mld, st));
  SM_CUDA(launch_rns_convert(wv.dev, dbl(T2), route, nullptr, 0, made[0], T2, mld, st));
  RnsCheb c{};
  c.state = route;
  c.F = F;
  c.twice = 1;
  c.R = made[1];
  for (int q = 1; q < H; ++q) {  // T_{2q+1} = 2 T_2 T_{2q-1} - T_{2q-3}, T_{-1} = T_1
    SM_TRY(product(T2, odd(q - 1)));
    c.sub = odd(std::max(0, q - 2));
    c.C = odd(q);
    if (q == H - 1) c.R = nullptr;
    SM_CUDA(launch_rns_cheb(wv.dev, c, mld, st));
  }
  for (int i = 0; whole && i < 2; ++i) {  // residues of -T_9 and -T_7
    RnsCheb t{};
    t.state = route;
    t.sub = odd(H / 2 - i);
    t.R = R[i];
    SM_CUDA(launch_rns_cheb(wv.dev, t, mld, st));
  }
  SM_TRY(product(odd(H / 2), odd(H / 2 - 1)));  // Y = T_16 = 2 T_9 T_7 - T_2
  c.sub = T2;
  c.C = T2;
  c.R = made[0];
  SM_CUDA(launch_rns_cheb(wv.dev, c, mld, st));
  // giant steps: b_j = R_j + 2 Y b_{j+1} - b_{j+2}, p = R_0 + Y b_1 - b_2
  c = RnsCheb{};
  c.state = route;
  c.odd = odd(0);
  c.stride = E;
  c.R = made[1];
  for (int j = P.blocks - 1; j >= 0; --j) {
    const RnsFix W = fix(H + 1 + (j & 1));  // b_{j+2}'s place
    for (int q = 0; q < H; ++q) c.coef[q] = std::llrint(std::ldexp(P.r[size_t(j) * H + q], RNS_COEF - e));
    if (j < P.blocks - 1) {
      SM_TRY(product(T2, fix(H + 1 + ((j + 1) & 1))));
      c.F = F;
    }
    c.twice = j > 0;
    c.sub = j < P.blocks - 2 ? W : RnsFix{};
    c.C = W;
    if (j == 0) {
      c.C = RnsFix{};
      c.R = nullptr;
      c.out = dbl(W);
      c.out_scale = std::ldexp(1.0, e);
    }
    SM_CUDA(launch_rns_cheb(wv.dev, c, mld, st));
  }
  return SUBMAT_OK;
}

template <typename T>
submat_status Plan::sign_fermi(const double* K, double mu, double* D, cudaStream_t st) {
  if (use_rns && !rns) SM_TRY(rns_setup(st));
  for (size_t wi = 0; wi < waves.size(); ++wi)
    SM_TRY(fermi_wave<T>(waves[wi], use_rns ? int(wi) : -1, K, mu, D, nullptr, nullptr, ws, ws_elems, st));
  return SUBMAT_OK;
}

template submat_status Plan::sign_fermi<double>(const double*, double, double*, cudaStream_t);
template submat_status Plan::sign_fermi<float>(const double*, double, double*, cudaStream_t);

// dN/dmu of the last finite-temperature evaluation: sum over the evaluated
// block columns of (Tr_j - sum of squares_j) / kT, in fixed order.
submat_status Plan::fermi_dn_dmu(cudaStream_t st, double* out) {
  std::vector<double> tr(nblk), sq(nblk);
  SM_CUDA(cudaMemcpyAsync(tr.data(), d_trpart, 8 * size_t(nblk), cudaMemcpyDeviceToHost, st));
  SM_CUDA(cudaMemcpyAsync(sq.data(), d_sqpart, 8 * size_t(nblk), cudaMemcpyDeviceToHost, st));
  SM_CUDA(cudaStreamSynchronize(st));
  double acc = 0.0;
  // block columns evaluated: all of them for grouped plans (col_lo / col_hi
  // count submatrices there), else the column range
  const int j0 = grouped ? 0 : col_lo, j1 = grouped ? nblk : col_hi;
  for (int j = j0; j < j1; ++j) acc += tr[j] - sq[j];
  *out = acc / opt.kT;
  return SUBMAT_OK;
}

// The adjoint at finite temperature (vector-Jacobian product of K -> D):
// fermi_wave on dual numbers, on the adjoint's own waves and workspace.
// dN/dmu = sum_j sum_{c in block j} [f'(a_j)]_cc comes from the value part
// of the same pass (f' = f (1 - f) / kT is a function of a_j itself).
submat_status Plan::backward_fermi(const double* K, double mu, const double* Dbar, double* Kbar,
                                   double* dN_dmu, cudaStream_t st) {
  reset_stats();
  fermi_degree = 0;
  fermi_trunc = fermi_flops = 0.0;
  SM_CUDA(cudaMemsetAsync(d_flags, 0, 4 * sizeof(int), st));
  SM_CUDA(launch_check_finite(Dbar, nvals, d_flags, st));
  int fl = 0;
  SM_TRY(read_flags(st, &fl));
  if (fl & FLAG_NONFINITE) {
    set_error("Dbar holds a NaN or Inf value");
    return SUBMAT_ERR_NONFINITE;
  }
  const size_t bpe = fermi_dual_bytes_per_elem(opt.prec);
  if (bwaves.empty()) {
    size_t fre = 0, tot = 0;
    SM_CUDA(cudaMemGetInfo(&fre, &tot));
    size_t cap = opt.workspace_cap_bytes ? opt.workspace_cap_bytes : size_t(double(fre) * 0.8);
    SM_TRY(build_waves(bpe, cap, bwaves, st));
    int64_t mx = 0;
    for (auto& wv : bwaves) {
      mx = std::max(mx, wv.elems);
      max_bwave = std::max(max_bwave, wv.count);
    }
    SM_TRY(grow_ns_state(max_bwave));
    bws_elems = mx;
    SM_TRY(dev_alloc(&bws, size_t(mx) * bpe, "adjoint workspace"));
    owned.push_back(bws);
  }
  SM_CUDA(cudaMemsetAsync(Kbar, 0, sizeof(double) * size_t(nvals), st));
  for (auto& wv : bwaves) {
    if (opt.prec == SUBMAT_FP64) SM_TRY(fermi_wave<double>(wv, -1, K, mu, nullptr, Dbar, Kbar, bws, bws_elems, st));
    else SM_TRY(fermi_wave<float>(wv, -1, K, mu, nullptr, Dbar, Kbar, bws, bws_elems, st));
  }
  SM_CUDA(cudaStreamSynchronize(st));
  finish_stats(true);
  stats.flops_ns = fermi_flops;
  stats.poly_degree = fermi_degree;
  stats.poly_trunc = fermi_trunc;
  SM_TRY(fermi_dn_dmu(st, &stats.dn_dmu));
  if (dN_dmu) *dN_dmu = stats.dn_dmu;
  SM_TRY(read_flags(st, &fl));
  if (fl & FLAG_NONFINITE) {
    set_error("K holds a NaN or Inf value");
    return SUBMAT_ERR_NONFINITE;
  }
  return SUBMAT_OK;
}

}  // namespace submat
