// FP64-accurate products on the tensor cores by residue numbers (rns.cuh): the
// grouped product kernel and the passes that turn its sums into the next
// iterate and the iterate into residues.
#include "rns.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "tcgen05.cuh"

namespace submat {

namespace {

// ---------------------------------------------------------------------------
// moduli
// ---------------------------------------------------------------------------

typedef unsigned __int128 u128;

// The largest pairwise coprime numbers up to 256 (256 = 2^8, 255 = 3 5 17,
// 253 = 11 23, 247 = 13 19, 217 = 7 31, the others prime).
constexpr int kMods[RNS_MODS] = {256, 255, 253, 251, 247, 239, 233, 229, 227, 223, 217, 211, 199, 197};

constexpr int balanced(int r, int m) { return 2 * r >= m ? r - m : r; }  // in [-m/2, m/2)

struct RnsTable {
  float m[RNS_MODS], inv[RNS_MODS];
  unsigned long long w[RNS_MODS];  // round(2^64 ((P / m)^-1 mod m) / m)
  int pow_lo[RNS_MODS], pow_hi[RNS_MODS];  // 256^k mod m, k = 0..3 and 4..7, packed signed bytes
  int bias[RNS_MODS];                      // the magic float's bits less 2^63 mod m
  unsigned long long scale;                // S 2^7: entries at 2^-58 to multiples of 1 / (2 S)
  unsigned long long pn;                   // P / S^2 2^62: C = mulhi(F, pn) 2^-62
};

// 1.5 2^23: adding it to a float of magnitude below 2^22 leaves the rounded
// integer in the low bits
constexpr float kMagic = 12582912.0f;
constexpr unsigned kMagicBits = 0x4B400000u;

constexpr RnsTable make_table() {
  RnsTable t{};
  u128 P = 1;
  for (int i = 0; i < RNS_MODS; ++i) P *= u128(kMods[i]);
  // S = floor(sqrt(P / 2.02)), P / S^2 by long division
  unsigned long long S = 0;
  for (int b = 55; b >= 0; --b) {
    const unsigned long long c = S | (1ull << b);
    if (u128(c) * c <= P / 202 * 100) S = c;
  }
  const u128 S2 = u128(S) * S;
  u128 q2 = P / S2, rem = P % S2;
  for (int b = 0; b < 62; ++b) {
    rem <<= 1;
    q2 <<= 1;
    if (rem >= S2) { rem -= S2; q2 |= 1; }
  }
  t.scale = S << 7;
  t.pn = static_cast<unsigned long long>(q2);
  for (int i = 0; i < RNS_MODS; ++i) {
    const int m = kMods[i];
    t.m[i] = float(m);
    t.inv[i] = 1.0f / float(m);
    const int r = int((P / u128(m)) % u128(m));
    int q = 1;
    while (q * r % m != 1) ++q;
    t.w[i] = static_cast<unsigned long long>(((u128(q) << 64) + u128(m / 2)) / u128(m));
    unsigned lo = 0, hi = 0;
    int pw = 1;
    for (int k = 0; k < 8; ++k) {
      const unsigned byte = unsigned(balanced(pw, m)) & 0xFFu;
      if (k < 4) lo |= byte << (8 * k); else hi |= byte << (8 * (k - 4));
      if (k < 7) pw = pw * 256 % m;
    }
    t.pow_lo[i] = int(lo);
    t.pow_hi[i] = int(hi);
    // the entry enters as its offset-binary form a + 2^63: take 2^63 mod m off again
    t.bias[i] = int(kMagicBits) - balanced(pw * 128 % m, m);
  }
  return t;
}

__constant__ RnsTable kTab = make_table();

// ---------------------------------------------------------------------------
// the product kernel
// ---------------------------------------------------------------------------

constexpr int TM = 128, TK = 64;
constexpr int TILE = TM * TK * 2;          // one 128 x 64 BF16 operand tile
constexpr int STAGES = 6;                   // operand pipeline: A and B tile per stage
constexpr int NBUF = 4;                     // accumulators in TMEM, 128 columns each
// warpgroup 0: TMA warp, MMA warp, two idle; warpgroups 1 and 2: epilogue (168
// registers a thread, no spills)
constexpr int THREADS = 384, EPI_THREADS = 256;
constexpr int SMEM = 1024 + STAGES * 2 * TILE + (2 * STAGES + 2 * NBUF + 1) * 8 + 16;
// D F32, A and B BF16, both K-major, M = N = 128
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(TM >> 3) << 17) | (uint32_t(TM >> 4) << 24);

// f += r w modulo 2^64: one wide multiply-add and one for the upper half
__device__ __forceinline__ void add_weighted(unsigned long long& f, uint32_t r, uint32_t wlo, uint32_t whi) {
  asm("{\n\t.reg .u32 lo, hi;\n\t.reg .u64 t;\n\t"
      "mad.wide.u32 t, %1, %2, %0;\n\t"
      "mov.b64 {lo, hi}, t;\n\t"
      "mad.lo.u32 hi, %1, %3, hi;\n\t"
      "mov.b64 %0, {lo, hi};\n\t}"
      : "+l"(f)
      : "r"(r), "r"(wlo), "r"(whi));
}

// One item is a 128 x 128 tile (or, split, some of its moduli).  It runs one
// phase per modulus and per 1024 terms of the sum: the MMAs of a phase fill one
// of four TMEM accumulators while the epilogue warps reduce earlier ones.  The
// reduction keeps frac(C / P) as one 64-bit integer per entry in registers (64
// entries a thread, half the register file: what limits the tile to 128 x 128);
// nothing but the final sums goes to memory.  Bound by operand ingest, 32 KB per
// 256 cycles of MMA: ncu shows the tensor pipe 39 % busy at ~50 B/clk/SM.
// Measured on 216 submatrices of 420-480 dims: 0.56 ms a product, against
// 23.5 ms for the FP64 SIMT GEMM; a whole build 425.9 -> 19.8 ms.
__global__ void __launch_bounds__(THREADS, 1) k_rns_gemm(const __grid_constant__ RnsGemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles + STAGES * 2 * TILE);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + NBUF;
  uint64_t* drain = tempty + NBUF;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < NBUF; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], EPI_THREADS); }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(uint32_t(NBUF * TM)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const long long limit = p.timeout_cycles;
  const int total = p.nitems * p.split;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    int stage = 0;
    uint32_t phase = 0, issued = 0, issued_phase = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
      const int4 item = p.items[it / p.split];
      if (p.state && p.state[item.x] == p.skip_state) continue;
      const int part = it % p.split;
      const int nk = p.ld[item.x] / TK, nc = (nk + RNS_CHUNK - 1) / RNS_CHUNK;
      const int bucket = item.w & 0xFF, slot = item.w >> 8;
      const int ph1 = (part + 1) * RNS_MODS * nc / p.split;
      for (int ph = part * RNS_MODS * nc / p.split; ph < ph1 && ok; ++ph) {
        const int plane = slot * RNS_MODS + ph / nc;
        const int k0 = (ph % nc) * RNS_CHUNK, k1 = min(nk, k0 + RNS_CHUNK);
        for (int kb = k0; kb < k1; ++kb) {
          if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, limit)) { ok = false; break; }
          uint8_t* st = tiles + stage * 2 * TILE;
          mbar_expect_tx(&full[stage], 2 * TILE);
          tma_load_3d(st, p.map_a + bucket, &full[stage], kb * TK, item.y * TM, plane);
          tma_load_3d(st + TILE, p.map_b + bucket, &full[stage], kb * TK, item.z * TM, plane);
          issued |= 1u << stage;
          issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
    if (!ok) {
      atomicOr(p.flags, FLAG_TIMEOUT);
      *abort_flag = 1;
      // let this CTA's copies in flight land before shared memory is released
      for (int i = 0; i < STAGES; ++i)
        if (issued & (1u << i)) {
          const long long t0 = clock64();
          while (!mbar_try_wait(&full[i], (issued_phase >> i) & 1u) && clock64() - t0 < limit) {
          }
        }
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer ----------------
    int stage = 0, buf = 0;
    uint32_t phase = 0, bphase = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
      const int4 item = p.items[it / p.split];
      if (p.state && p.state[item.x] == p.skip_state) continue;
      const int part = it % p.split;
      const int nk = p.ld[item.x] / TK, nc = (nk + RNS_CHUNK - 1) / RNS_CHUNK;
      const int ph1 = (part + 1) * RNS_MODS * nc / p.split;
      for (int ph = part * RNS_MODS * nc / p.split; ph < ph1 && ok; ++ph) {
        const int k0 = (ph % nc) * RNS_CHUNK, k1 = min(nk, k0 + RNS_CHUNK);
        if (!mbar_wait(&tempty[buf], bphase ^ 1u, abort_flag, limit)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d = tmem_base + uint32_t(buf * TM);
        for (int kb = k0; kb < k1; ++kb) {
          if (!mbar_wait(&full[stage], phase, abort_flag, limit)) { ok = false; break; }
          tc_fence_after();
          const uint64_t ad = sdesc(smem_u32(tiles + stage * 2 * TILE));
          const uint64_t bd = sdesc(smem_u32(tiles + stage * 2 * TILE + TILE));
#pragma unroll
          for (int k = 0; k < TK / 16; ++k)
            umma_bf16(d, ad + uint64_t(2 * k), bd + uint64_t(2 * k), IDESC, (kb > k0 || k > 0) ? 1u : 0u);
          umma_commit(&empty[stage]);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        umma_commit(&tfull[buf]);
        if (++buf == NBUF) { buf = 0; bphase ^= 1u; }
      }
    }
    if (!ok) {
      atomicOr(p.flags, FLAG_TIMEOUT);
      *abort_flag = 1;
    }
    // every MMA issued by this thread has completed once this commit lands
    umma_commit(drain);
    const long long t0 = clock64();
    while (!mbar_try_wait(drain, 0) && clock64() - t0 < limit) {
    }
  } else if (warp >= 4) {
    // ---------------- epilogue ----------------
    const int quarter = warp & 3, half = (warp - 4) >> 2;  // TMEM lanes 32 quarter .., columns 64 half ..
    const uint32_t tlane = tmem_base + (uint32_t(quarter * 32) << 16) + uint32_t(half * 64);
    int buf = 0;
    uint32_t bphase = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
      const int4 item = p.items[it / p.split];
      const int s = item.x;
      if (p.state && p.state[s] == p.skip_state) continue;
      const int part = it % p.split;
      const int ld = p.ld[s];
      const int nk = ld / TK, nc = (nk + RNS_CHUNK - 1) / RNS_CHUNK;
      const int ph1 = (part + 1) * RNS_MODS * nc / p.split;
      const int rg = item.y * TM + quarter * 32 + lane, cg = item.z * TM + half * 64;
      // a warp whose rows or columns lie beyond ld has nothing to reduce
      const bool work = item.y * TM + quarter * 32 < ld && cg < ld;
      unsigned long long f[64], corr = 0;
#pragma unroll
      for (int q = 0; q < 64; ++q) f[q] = 0;
      for (int ph = part * RNS_MODS * nc / p.split; ph < ph1; ++ph) {
        const int i = ph / nc;
        const float m = kTab.m[i], inv = kTab.inv[i];
        const unsigned long long w = kTab.w[i];
        const uint32_t wlo = uint32_t(w), whi = uint32_t(w >> 32);
        // a warp leaves the loop together: every lane sees the same outcome
        ok = __all_sync(0xffffffffu, mbar_wait(&tfull[buf], bphase, abort_flag, limit));
        if (!ok) break;
        tc_fence_after();
        // r = d mod m, balanced, enters as the bits of r + magic; the magic's
        // own share is taken off once per tile (corr)
        corr += w * kMagicBits;
        if (work) {
          const uint32_t t0 = tlane + uint32_t(buf * TM);
          float d[2][16];
          tmem_ld16(t0, d[0]);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            tmem_wait16(d[c & 1]);
            if (c < 3) tmem_ld16(t0 + uint32_t(16 * (c + 1)), d[(c + 1) & 1]);
            if (c == 3) {
              tc_fence_before();
              mbar_arrive(&tempty[buf]);
            }
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              const float x = d[c & 1][q];
              const float t = fmaf(x, inv, kMagic) - kMagic;
              add_weighted(f[c * 16 + q], __float_as_uint(fmaf(-m, t, x) + kMagic), wlo, whi);
            }
          }
        } else {
          tc_fence_before();
          mbar_arrive(&tempty[buf]);
        }
        if (++buf == NBUF) { buf = 0; bphase ^= 1u; }
      }
      if (!ok) {
        if (lane == 0) atomicOr(p.flags, FLAG_TIMEOUT);
        *abort_flag = 1;
        break;
      }
      if (!work) continue;
      long long* out = p.F + p.off[s] + int64_t(rg) * ld + cg;
      if (p.split == 1) {
#pragma unroll
        for (int q = 0; q < 64; q += 4) {
          unsigned long long v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = f[q + e] - corr;
          asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(out + q), "l"(v[0]), "l"(v[1]), "l"(v[2]),
                       "l"(v[3])
                       : "memory");
        }
      } else {
#pragma unroll
        for (int q = 0; q < 64; ++q)
          atomicAdd(reinterpret_cast<unsigned long long*>(out + q), f[q] - corr);
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(uint32_t(NBUF * TM)));
  }
}

// ---------------------------------------------------------------------------
// fixed point, residues
// ---------------------------------------------------------------------------

// x = b mod m_i for eight entries, as BF16: the bytes of each entry (offset
// binary) against 256^k mod m, then one balanced reduction in FP32.
template <int I>
__device__ __forceinline__ uint4 residues8(const unsigned long long* u) {
  uint32_t o[4];
  float r[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    int acc = kTab.bias[I];
    asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(acc) : "r"(uint32_t(u[e])), "r"(kTab.pow_lo[I]));
    asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(acc) : "r"(uint32_t(u[e] >> 32)), "r"(kTab.pow_hi[I]));
    const float x = __int_as_float(acc) - kMagic;  // |x| < 2^19
    const float t = fmaf(x, kTab.inv[I], kMagic) - kMagic;
    r[e] = fmaf(-kTab.m[I], t, x);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(r[2 * e], r[2 * e + 1]);
    o[e] = *reinterpret_cast<const uint32_t*>(&b);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

template <int I = 0>
__device__ __forceinline__ void store_residues8(const unsigned long long* u, __nv_bfloat16* dst, int64_t plane) {
  if constexpr (I < RNS_MODS) {
    *reinterpret_cast<uint4*>(dst + int64_t(I) * plane) = residues8<I>(u);
    store_residues8<I + 1>(u, dst, plane);
  }
}

__device__ __forceinline__ unsigned long long offset_binary(long long a) {
  return static_cast<unsigned long long>(a) ^ 0x8000000000000000ull;
}

// rint(x 2^e) of a double, |x 2^e| < 2^62, with integer operations
__device__ __forceinline__ long long to_fixed(double x, int e) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int ex = int((b >> 52) & 0x7FF);
  if (ex == 0) return 0;
  const unsigned long long mant = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const int sh = ex - 1075 + e;
  long long v = 0;
  if (sh >= 0) v = sh < 11 ? static_cast<long long>(mant << sh) : 0;  // callers keep sh below 11
  else if (sh > -54) v = static_cast<long long>(((mant >> (-sh - 1)) + 1) >> 1);
  return (b >> 63) ? -v : v;
}

// frac 2^64 to the product at 2^-62
__device__ __forceinline__ long long product62(long long f) {
  const unsigned long long pn = kTab.pn;
  const unsigned long long u = static_cast<unsigned long long>(f);
  return static_cast<long long>(__umul64hi(u, pn) - (f < 0 ? pn : 0ull));
}

// an entry at 2^-58 as the rounded multiple of 1 / S
__device__ __forceinline__ long long operand(long long x) {
  const unsigned long long g = kTab.scale, u = static_cast<unsigned long long>(x);
  return (static_cast<long long>(__umul64hi(u, g) - (x < 0 ? g : 0ull)) + 1) >> 1;
}

// smallest sh with row norms 2^-sh sqrt(norm2) <= 1
__device__ __forceinline__ int norm_shift(unsigned bits) {
  const float f = __uint_as_float(bits);
  if (!(f > 0.0f)) return 0;
  const int e = int(bits >> 23) - 126;  // f < 2^e
  return e >= 0 ? (e + 1) / 2 : -(-e / 2);
}

__global__ void __launch_bounds__(256) k_rns_rownorm(WaveDev w, const double* __restrict__ X,
                                                     const int* __restrict__ state, unsigned* norm2) {
  const int s = blockIdx.y;
  if (state && state[s] == ST_DONE) return;
  const int ld = w.ld[s], n = w.n[s];
  const double* Xs = X + w.off[s];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float best = 0.0f;
  for (int r = blockIdx.x * 8 + warp; r < n; r += gridDim.x * 8) {
    float acc = 0.0f;
    for (int c = 2 * lane; c < ld; c += 64) {
      const double2 v = *reinterpret_cast<const double2*>(Xs + int64_t(r) * ld + c);
      const float a = d2f_trunc(v.x), b = d2f_trunc(v.y);
      acc = fmaf(a, a, acc);
      acc = fmaf(b, b, acc);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    best = fmaxf(best, acc);
  }
  // sums of truncated squares: the margin covers truncation and rounding (ld <= 32768)
  if (lane == 0 && best > 0.0f) atomicMax(&norm2[s], __float_as_uint(best * 1.01f));
}

__global__ void __launch_bounds__(256) k_rns_convert(WaveDev w, const double* X, const int* __restrict__ state,
                                                     const unsigned* __restrict__ norm2, int sh_fixed,
                                                     __nv_bfloat16* __restrict__ R, long long* fixed) {
  const int s = blockIdx.y;
  if (state && state[s] == ST_DONE) return;
  const int e = RNS_FRAC - (norm2 ? norm_shift(norm2[s]) : sh_fixed);
  const int ld = w.ld[s];
  const int64_t plane = int64_t(ld) * ld, base = w.off[s];
  for (int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) * 8; i < plane;
       i += int64_t(gridDim.x) * blockDim.x * 8) {
    double x[8];
    unsigned long long u[8];
#pragma unroll
    for (int k = 0; k < 8; k += 2)
      *reinterpret_cast<double2*>(x + k) = *reinterpret_cast<const double2*>(X + base + i + k);
#pragma unroll
    for (int k = 0; k < 8; ++k) u[k] = offset_binary(operand(to_fixed(x[k], e)));
    store_residues8(u, R + RNS_MODS * base + i, plane);
    if (fixed) {
#pragma unroll
      for (int k = 0; k < 8; ++k) fixed[base + i + k] = to_fixed(x[k], RNS_FRAC);
    }
  }
}

// ---------------------------------------------------------------------------
// 64 x 64 tile pairs (a, b), a <= b: values from the upper tile, results to both
// ---------------------------------------------------------------------------

constexpr int PITCH = 65;

__device__ __forceinline__ void pair_of(int pi, int T, int* a, int* b) {
  int x = 0;
  while (pi >= T - x) { pi -= T - x; ++x; }
  *a = x;
  *b = x + pi;
}

// entry (r, c) of the pair's upper tile; a diagonal tile from its upper triangle
__device__ __forceinline__ long long tile_get(const long long (*v)[PITCH], int r, int c, bool diag) {
  return diag && r > c ? v[c][r] : v[r][c];
}

// residues of the staged tile into tile (a, b) and, transposed, (b, a):
// 512 segments of eight entries a tile, two per thread
__device__ __forceinline__ void tile_residues(const long long (*v)[PITCH], int a, int b, int ld, __nv_bfloat16* R,
                                              int64_t plane) {
  for (int t = 0; t < (a == b ? 1 : 2); ++t)
#pragma unroll 1
    for (int g = threadIdx.x; g < 512; g += 256) {
      const int r = g >> 3, c0 = (g & 7) * 8;
      unsigned long long u[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        u[k] = offset_binary(operand(t ? v[c0 + k][r] : tile_get(v, r, c0 + k, a == b)));
      const int row = (t ? b : a) * 64 + r, col = (t ? a : b) * 64 + c0;
      store_residues8(u, R + int64_t(row) * ld + col, plane);
    }
}

// staged tile as FP64 (times 2^-frac) into both tiles of the pair
__device__ __forceinline__ void tile_doubles(const long long (*v)[PITCH], int a, int b, int ld, double scale,
                                             double* X) {
  const int c = (threadIdx.x & 31) * 2;
  for (int t = 0; t < (a == b ? 1 : 2); ++t)
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      double2 o;
      if (t) { o.x = double(v[c][r]) * scale; o.y = double(v[c + 1][r]) * scale; }
      else { o.x = double(tile_get(v, r, c, a == b)) * scale; o.y = double(tile_get(v, r, c + 1, a == b)) * scale; }
      *reinterpret_cast<double2*>(X + int64_t((t ? b : a) * 64 + r) * ld + (t ? a : b) * 64 + c) = o;
    }
}

// (v - [diagonal] one) as FP32
__device__ __forceinline__ float residual32(long long v, bool diag, long long one) {
  const long long e = v - (diag ? one : 0);
  return fmaf(float(int(e >> 32)), 4294967296.0f, float(unsigned(e)));
}

__device__ __forceinline__ void add_block_sum(float part, double scale, double* out) {
  __shared__ float red[8];
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < 8; ++q) t += double(red[q]);
    if (t != 0.0) atomicAdd(out, t * scale);
  }
}

__global__ void __launch_bounds__(256) k_rns_square0(WaveDev w, NsStateDev ns, const unsigned* __restrict__ norm2,
                                                     long long* F) {
  __shared__ long long v[64][PITCH];
  const int s = blockIdx.y;
  if (ns.state[s] == ST_DONE) return;
  const int ld = w.ld[s], n = w.n[s], T = ld / 64;
  long long* Fs = F + w.off[s];
  const double scale = ldexp(1.0, 2 * norm_shift(norm2[s]) - 62);
  const int c = (threadIdx.x & 31) * 2;
  float part = 0.0f;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    __syncthreads();
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const longlong2 f = *reinterpret_cast<const longlong2*>(Fs + int64_t(a * 64 + r) * ld + b * 64 + c);
      v[r][c] = product62(f.x);
      v[r][c + 1] = product62(f.y);
    }
    __syncthreads();
    tile_doubles(v, a, b, ld, scale, reinterpret_cast<double*>(Fs));
    for (int r = threadIdx.x >> 5; r < 64; r += 8)
      for (int k = 0; k < 2; ++k) {
        const bool dg = a == b && r == c + k && a * 64 + r < n;
        const float e = float(double(v[r][c + k]) * scale - (dg ? 1.0 : 0.0));
        part = fmaf(a == b ? e : 2.0f * e, e, part);
      }
  }
  add_block_sum(part, 1.0, &ns.res2[s]);
}

__global__ void __launch_bounds__(256) k_rns_square(WaveDev w, NsStateDev ns, const long long* __restrict__ F,
                                                    __nv_bfloat16* __restrict__ R) {
  __shared__ long long v[64][PITCH];
  const int s = blockIdx.y;
  if (ns.state[s] == ST_DONE) return;
  const int ld = w.ld[s], n = w.n[s], T = ld / 64;
  const int64_t base = w.off[s], plane = int64_t(ld) * ld;
  const long long* Fs = F + base;
  const int c = (threadIdx.x & 31) * 2;
  float part = 0.0f;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    const float wgt = a == b ? 1.0f : 2.0f;
    __syncthreads();
#pragma unroll 4
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const longlong2 f = *reinterpret_cast<const longlong2*>(Fs + int64_t(a * 64 + r) * ld + b * 64 + c);
      const long long y[2] = {(product62(f.x) + 8) >> 4, (product62(f.y) + 8) >> 4};  // 2^-58
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        v[r][c + k] = y[k];
        const float e = residual32(y[k], a == b && r == c + k && a * 64 + r < n, 1ll << RNS_FRAC) * 0x1p-58f;
        part = fmaf(wgt * e, e, part);
      }
    }
    __syncthreads();
    tile_residues(v, a, b, ld, R + RNS_MODS * base, plane);
  }
  add_block_sum(part, 1.0, &ns.res2[s]);
}

__global__ void __launch_bounds__(256) k_rns_update(WaveDev w, NsStateDev ns, const long long* __restrict__ F,
                                                    int shift, long long* X, __nv_bfloat16* __restrict__ R) {
  __shared__ long long v[64][PITCH];
  const int s = blockIdx.y;
  const int state = ns.state[s];
  if (state == ST_DONE) return;
  const bool last = state == ST_LAST;
  const int ld = w.ld[s], T = ld / 64;
  const int64_t base = w.off[s], plane = int64_t(ld) * ld;
  const long long* Fs = F + base;
  long long* Xs = X + base;
  const int c = (threadIdx.x & 31) * 2;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    __syncthreads();
#pragma unroll 4
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const int64_t i = int64_t(a * 64 + r) * ld + b * 64 + c;
      const longlong2 f = *reinterpret_cast<const longlong2*>(Fs + i);
      longlong2 x = *reinterpret_cast<const longlong2*>(Xs + i);
      // product at 2^-58 (2^shift times the unit-scale one)
      const int sh = 4 - shift;
      const long long half = (1ll << sh) >> 1;
      x.x = (3 * x.x - ((product62(f.x) + half) >> sh) + 1) >> 1;
      x.y = (3 * x.y - ((product62(f.y) + half) >> sh) + 1) >> 1;
      v[r][c] = x.x;
      v[r][c + 1] = x.y;
      if (!last) *reinterpret_cast<longlong2*>(Xs + i) = x;
    }
    __syncthreads();
    if (last) tile_doubles(v, a, b, ld, 0x1p-58, reinterpret_cast<double*>(Xs));
    else tile_residues(v, a, b, ld, R + RNS_MODS * base, plane);
  }
}

__global__ void __launch_bounds__(256) k_rns_cheb2(WaveDev w, const long long* __restrict__ F,
                                                   double* __restrict__ T2) {
  __shared__ long long v[64][PITCH];
  const int s = blockIdx.y;
  const int ld = w.ld[s], n = w.n[s], T = ld / 64;
  const int64_t base = w.off[s];
  const int c = (threadIdx.x & 31) * 2;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    __syncthreads();
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const longlong2 f = *reinterpret_cast<const longlong2*>(F + base + int64_t(a * 64 + r) * ld + b * 64 + c);
      const bool row = a == b && a * 64 + r < n;  // 2 X^2 - I at 2^-61
      v[r][c] = product62(f.x) - (row && r == c ? 1ll << 61 : 0);
      v[r][c + 1] = product62(f.y) - (row && r == c + 1 ? 1ll << 61 : 0);
    }
    __syncthreads();
    tile_doubles(v, a, b, ld, 0x1p-61, T2 + base);
  }
}

// t c = 2^64 h + 2^32 m to a few 2^32, summed over the terms, from balanced
// 32-bit halves: |t| <= 2^58 and |c| < 2^60 keep the sums of RNS_COMB terms in range
__device__ __forceinline__ void add_product(long long t, long long c, long long& h, long long& m) {
  const int tl = int(t), th = int(t >> 32) - (tl >> 31);
  const int cl = int(c), ch = int(c >> 32) - (cl >> 31);
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(h) : "r"(th), "r"(ch));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(m) : "r"(th), "r"(cl));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(m) : "r"(tl), "r"(ch));
  m += __mulhi(tl, cl);
}

// One step of the recurrences, as a pass over tile pairs: bound by memory
// traffic (the residues written, 28 bytes an entry, are the largest part), so
// the combination of the stored odd T_k is formed here instead of in a pass of
// its own, and only upper tiles are read.
template <bool COMB>
__global__ void __launch_bounds__(256) k_rns_cheb(WaveDev w, const __grid_constant__ RnsCheb p) {
  __shared__ long long v[64][PITCH];
  const int s = blockIdx.y;
  const int ld = w.ld[s], T = ld / 64;
  const int64_t base = w.off[s], plane = int64_t(ld) * ld;
  const int c = (threadIdx.x & 31) * 2;
  const int sh = p.twice ? 3 : 4;  // product62 to 2^-58
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    __syncthreads();
#pragma unroll 2
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const int64_t i = base + int64_t(a * 64 + r) * ld + b * 64 + c;
      longlong2 x = make_longlong2(0, 0);
      if (p.F) {
        const longlong2 f = *reinterpret_cast<const longlong2*>(p.F + i);
        const long long half = (1ll << sh) >> 1;
        x.x = (product62(f.x) + half) >> sh;
        x.y = (product62(f.y) + half) >> sh;
      }
      if (p.sub) {
        const longlong2 z = *reinterpret_cast<const longlong2*>(p.sub + i);
        x.x -= z.x;
        x.y -= z.y;
      }
      if constexpr (COMB) {
        long long hx = 0, mx = 0, hy = 0, my = 0;
#pragma unroll
        for (int q = 0; q < RNS_COMB; ++q) {
          const longlong2 t = *reinterpret_cast<const longlong2*>(p.odd + q * p.stride + i);
          add_product(t.x, p.coef[q], hx, mx);
          add_product(t.y, p.coef[q], hy, my);
        }
        x.x += (hx << 6) + ((mx + (1ll << 25)) >> 26);
        x.y += (hy << 6) + ((my + (1ll << 25)) >> 26);
      }
      v[r][c] = x.x;
      v[r][c + 1] = x.y;
      if (p.C) *reinterpret_cast<longlong2*>(p.C + i) = x;
    }
    __syncthreads();
    if (p.out) tile_doubles(v, a, b, ld, p.out_scale, p.out + base);
    if (p.R) tile_residues(v, a, b, ld, p.R + RNS_MODS * base, plane);
  }
}

// about four tile pairs a block
dim3 tile_grid(int max_ld, int nsub) {
  const int T = max_ld / 64;
  return dim3(unsigned(std::min((T * (T + 1) / 2 + 3) / 4, 512)), unsigned(nsub));
}

}  // namespace

int rns_split(int ntiles, int nsm) {
  // Tiles alone fill the chip from two per SM on.  Below that the moduli of a
  // tile go to several CTAs, which add their sums modulo 2^64 (exact in any
  // order), at most one modulus each.
  if (ntiles >= 2 * nsm) return 1;
  return std::max(1, std::min(RNS_MODS, (2 * nsm) / std::max(1, ntiles)));
}

cudaError_t launch_rns_gemm(RnsGemmParams p, int nsm, cudaStream_t st) {
  if (p.nitems <= 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_rns_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
  if (e != cudaSuccess) return e;
  k_rns_gemm<<<std::min(p.nitems * p.split, nsm), THREADS, SMEM, st>>>(p);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_rownorm(const WaveDev& w, const double* X, const int* state, unsigned* norm2, int max_ld,
                               cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(norm2, 0, sizeof(unsigned) * size_t(w.nsub), st);
  if (e != cudaSuccess) return e;
  k_rns_rownorm<<<dim3(unsigned(std::min((max_ld + 31) / 32, 64)), unsigned(w.nsub)), 256, 0, st>>>(w, X, state, norm2);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_convert(const WaveDev& w, const double* X, const int* state, const unsigned* norm2,
                               int sh_fixed, __nv_bfloat16* R, long long* fixed, int max_ld, cudaStream_t st) {
  const int64_t bx = (int64_t(max_ld) * max_ld + 256 * 32 - 1) / (256 * 32);
  k_rns_convert<<<dim3(unsigned(std::min<int64_t>(bx, 1024)), unsigned(w.nsub)), 256, 0, st>>>(w, X, state, norm2,
                                                                                              sh_fixed, R, fixed);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_square0(const WaveDev& w, NsStateDev ns, const unsigned* norm2, long long* F, int max_ld,
                               cudaStream_t st) {
  k_rns_square0<<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, ns, norm2, F);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_square(const WaveDev& w, NsStateDev ns, const long long* F, __nv_bfloat16* R, int max_ld,
                              cudaStream_t st) {
  k_rns_square<<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, ns, F, R);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_update(const WaveDev& w, NsStateDev ns, const long long* F, int shift, long long* X,
                              __nv_bfloat16* R, int max_ld, cudaStream_t st) {
  k_rns_update<<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, ns, F, shift, X, R);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_cheb2(const WaveDev& w, const long long* F, double* T2, int max_ld, cudaStream_t st) {
  k_rns_cheb2<<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, F, T2);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_cheb(const WaveDev& w, const RnsCheb& c, int max_ld, cudaStream_t st) {
  if (c.odd) k_rns_cheb<true><<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, c);
  else k_rns_cheb<false><<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, c);
  count_launch();
  return cudaGetLastError();
}

}  // namespace submat
