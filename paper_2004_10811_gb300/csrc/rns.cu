// FP64-accurate products on the tensor cores by residue numbers (rns.cuh): the
// grouped product kernel and the passes that turn its sums into the next
// iterate and the iterate into residues.
#include "rns.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "tcgen05.cuh"

namespace submat {

int num_sms();

namespace {

// ---------------------------------------------------------------------------
// moduli
// ---------------------------------------------------------------------------

typedef unsigned __int128 u128;

// Pairwise coprime: 256 = 2^8, 255 = 3 5 17, 253 = 11 23, 247 = 13 19, 217 = 7 31,
// the others are prime.
constexpr int kMods[RNS_MODS] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227,
                                 223, 217, 211, 199, 197, 193, 191, 181, 179};

constexpr int balanced(int r, int m) { return 2 * r >= m ? r - m : r; }  // in [-m/2, m/2)

struct RnsTable {
  float m[RNS_MODS], inv[RNS_MODS];
  // weight round(2^82 ((P / m)^-1 mod m) / m): its upper 64 bits and the lower RNS_GUARD
  unsigned long long w[RNS_MODS];
  unsigned wl[RNS_MODS];
  // 256^k mod m as packed signed bytes: k = 0, 1 (the low half-word), 2..5 and 6..9
  int pow_lo[RNS_MODS], pow_mid[RNS_MODS], pow_hi[RNS_MODS];
  int bias[RNS_MODS];     // the magic float's bits less 2^79 mod m
  int ph, pl;             // P / S^2 2^61 (below 2^63) in balanced halves
};

// 1.5 2^23: adding it to a float of magnitude below 2^22 leaves the rounded
// integer in the low bits
constexpr float kMagic = 12582912.0f;
constexpr unsigned kMagicBits = 0x4B400000u;

constexpr RnsTable make_table() {
  RnsTable t{};
  unsigned long long P[3] = {1, 0, 0};  // the product, 64-bit limbs
  for (int i = 0; i < RNS_MODS; ++i) {
    u128 carry = 0;
    for (int l = 0; l < 3; ++l) {
      carry += u128(P[l]) * u128(kMods[i]);
      P[l] = static_cast<unsigned long long>(carry);
      carry >>= 64;
    }
  }
  // P / 2^146 2^61 = P 2^-85: bits 85 and up of the limbs
  static_assert(2 * RNS_FRAC - 61 == 85, "the shift below");
  const unsigned long long pn = (P[1] >> 21) | (P[2] << 43);
  t.pl = static_cast<int>(static_cast<unsigned>(pn));
  t.ph = static_cast<int>(static_cast<unsigned>(pn >> 32)) + (t.pl < 0 ? 1 : 0);
  for (int i = 0; i < RNS_MODS; ++i) {
    const int m = kMods[i];
    t.m[i] = float(m);
    t.inv[i] = 1.0f / float(m);
    int r = 1;  // P / m mod m
    for (int k = 0; k < RNS_MODS; ++k)
      if (k != i) r = r * kMods[k] % m;
    int q = 1;
    while (q * r % m != 1) ++q;
    const u128 w = ((u128(q) << (64 + RNS_GUARD)) + u128(m / 2)) / u128(m);
    t.w[i] = static_cast<unsigned long long>(w >> RNS_GUARD);
    t.wl[i] = unsigned(w & ((1u << RNS_GUARD) - 1));
    unsigned part[3] = {0, 0, 0};
    int pw = 1;
    for (int k = 0; k < 10; ++k) {
      const unsigned byte = unsigned(balanced(pw, m)) & 0xFFu;
      if (k < 2) part[0] |= byte << (8 * k); else part[(k + 2) / 4] |= byte << (8 * ((k + 2) % 4));
      if (k < 9) pw = pw * 256 % m;
    }
    t.pow_lo[i] = int(part[0]);
    t.pow_mid[i] = int(part[1]);
    t.pow_hi[i] = int(part[2]);
    // the entry enters as its offset-binary form N + 2^79: take 2^79 mod m off again
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
constexpr int NBUF = 3;                     // accumulators in TMEM, 128 columns each, and the guard sums
// warpgroup 0: TMA warp, MMA warp, two idle; warpgroups 1 and 2: epilogue (168
// registers a thread, no spills)
constexpr int THREADS = 384, EPI_THREADS = 256;
constexpr int FOLD = 60;  // phases after which the guard sums are folded: 60 128 2^18 < 2^31
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

// moves the whole units of f out of a guard sum (corrl: the magic's share in it)
__device__ __forceinline__ void fold_guard(unsigned long long& f, uint32_t& g, uint32_t corrl) {
  const int v = int(g - corrl);
  f += static_cast<unsigned long long>(static_cast<long long>(v >> RNS_GUARD));
  g = uint32_t(v) & ((1u << RNS_GUARD) - 1);
}

// One item is a 128 x 128 tile (or, split, some of its moduli).  It runs one
// phase per modulus and per 1024 terms of the sum: the MMAs of a phase fill one
// of three TMEM accumulators while the epilogue warps reduce earlier ones.  The
// reduction keeps frac(C / P) as one 64-bit integer per entry in registers (64
// entries a thread, half the register file: what limits the tile to 128 x 128), and
// the sums of the bits below in the rest of TMEM, which the epilogue has time to load
// and store between; nothing but the final sums goes to memory.  Bound by operand
// ingest, 32 KB per 256 cycles of MMA, of which an SM takes in about 50 bytes a
// clock, and by a tenth by the guard sums' way through TMEM (16.4 against 14.9 ms
// for 18 products without it; loading a chunk ahead of the one in work: 16.1).
// Measured on 216 submatrices of 420-480 dims: 0.89 ms a product, against
// 23.5 ms for the FP64 SIMT GEMM; a whole build 28.6 against 425.9 ms.
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
                 "r"(uint32_t((NBUF + 1) * TM)));
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
      const int ph1 = (part + 1) * p.nmod * nc / p.split;
      for (int ph = part * p.nmod * nc / p.split; ph < ph1 && ok; ++ph) {
        const int plane = slot * p.planes + ph / nc;
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
      const int ph1 = (part + 1) * p.nmod * nc / p.split;
      for (int ph = part * p.nmod * nc / p.split; ph < ph1 && ok; ++ph) {
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
    const uint32_t tguard = tlane + uint32_t(NBUF * TM);
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
      const int ph1 = (part + 1) * p.nmod * nc / p.split;
      const int rg = item.y * TM + quarter * 32 + lane, cg = item.z * TM + half * 64;
      // a warp whose rows or columns lie beyond ld has nothing to reduce
      const bool work = item.y * TM + quarter * 32 < ld && cg < ld;
      unsigned long long f[64], corr = 0;
      uint32_t corrl = 0;
#pragma unroll
      for (int q = 0; q < 64; ++q) f[q] = 0;
      int since = 0;  // phases in the guard sums
      for (int ph = part * p.nmod * nc / p.split; ph < ph1; ++ph) {
        const int i = p.mod0 + ph / nc;
        const float m = kTab.m[i], inv = kTab.inv[i];
        const unsigned long long w = kTab.w[i];
        const uint32_t wlo = uint32_t(w), whi = uint32_t(w >> 32), wl = kTab.wl[i];
        const bool fresh = since == 0;
        // a warp leaves the loop together: every lane sees the same outcome
        ok = __all_sync(0xffffffffu, mbar_wait(&tfull[buf], bphase, abort_flag, limit));
        if (!ok) break;
        tc_fence_after();
        // r = d mod m, balanced, enters as the bits of r + magic; the magic's
        // own share is taken off once per tile (corr)
        corr += w * kMagicBits;
        if (work) {
          const uint32_t t0 = tlane + uint32_t(buf * TM);
          float d[8], gf[8], dn[8], gn[8];
          tmem_ld8(t0, dn);
          tmem_ld8(tguard, gn);
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            uint32_t g[8];
            tmem_wait8(dn);
            tmem_wait8(gn);
#pragma unroll
            for (int q = 0; q < 8; ++q) { d[q] = dn[q]; gf[q] = gn[q]; }
            if (c < 7) {
              tmem_ld8(t0 + uint32_t(8 * c + 8), dn);
              tmem_ld8(tguard + uint32_t(8 * c + 8), gn);
            }
            if (c == 7) {
              tc_fence_before();
              mbar_arrive(&tempty[buf]);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              g[q] = fresh ? 0u : __float_as_uint(gf[q]);
              const float x = d[q];
              const float t = fmaf(x, inv, kMagic) - kMagic;
              const uint32_t r = __float_as_uint(fmaf(-m, t, x) + kMagic);
              add_weighted(f[c * 8 + q], r, wlo, whi);
              g[q] += r * wl;
            }
            tmem_st8(tguard + uint32_t(8 * c), g);
          }
          tmem_wait_st();
        } else {
          tc_fence_before();
          mbar_arrive(&tempty[buf]);
        }
        corrl += wl * kMagicBits;
        if (++since == FOLD) {
          if (work) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              float gf[8];
              uint32_t g[8];
              tmem_ld8(tguard + uint32_t(8 * c), gf);
              tmem_wait8(gf);
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                g[q] = __float_as_uint(gf[q]);
                fold_guard(f[c * 8 + q], g[q], corrl);
              }
              tmem_st8(tguard + uint32_t(8 * c), g);
            }
            tmem_wait_st();
          }
          corrl = 0;
          since = 1;
        }
        if (++buf == NBUF) { buf = 0; bphase ^= 1u; }
      }
      if (!ok) {
        if (lane == 0) atomicOr(p.flags, FLAG_TIMEOUT);
        *abort_flag = 1;
        break;
      }
      if (!work) continue;
      const int64_t at = p.off[s] + int64_t(rg) * ld + cg;
      long long* out = p.F.f + at;
      int* outl = p.F.g + at;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        float gf[8];
        uint32_t g[8];
        tmem_ld8(tguard + uint32_t(8 * c), gf);
        tmem_wait8(gf);
#pragma unroll
        for (int q = 0; q < 8; ++q) g[q] = __float_as_uint(gf[q]);
        // parts of a sum: folded, so that their guard sums add up without overflow
        if (p.split > 1 || p.planes < RNS_MODS)
#pragma unroll
          for (int q = 0; q < 8; ++q) fold_guard(f[c * 8 + q], g[q], corrl);
        else
#pragma unroll
          for (int q = 0; q < 8; ++q) g[q] -= corrl;
        if (p.split == 1) {
#pragma unroll
          for (int q = 0; q < 8; q += 4) {
            unsigned long long v[4];
            int4 u = make_int4(int(g[q]), int(g[q + 1]), int(g[q + 2]), int(g[q + 3]));
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = f[c * 8 + q + e] - corr;
            if (p.add) {
#pragma unroll
              for (int e = 0; e < 4; ++e) v[e] += static_cast<unsigned long long>(out[c * 8 + q + e]);
              const int4 o = *reinterpret_cast<const int4*>(outl + c * 8 + q);
              u = make_int4(u.x + o.x, u.y + o.y, u.z + o.z, u.w + o.w);
            }
            asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(out + c * 8 + q), "l"(v[0]), "l"(v[1]),
                         "l"(v[2]), "l"(v[3])
                         : "memory");
            *reinterpret_cast<int4*>(outl + c * 8 + q) = u;
          }
        } else {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            atomicAdd(reinterpret_cast<unsigned long long*>(out + c * 8 + q), f[c * 8 + q] - corr);
            atomicAdd(outl + c * 8 + q, int(g[q]));
          }
        }
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(uint32_t((NBUF + 1) * TM)));
  }
}

// ---------------------------------------------------------------------------
// fixed point, residues
// ---------------------------------------------------------------------------

// A value is (2^16 hi + lo) 2^-73, stored with lo in [0, 2^16) and worked on as
// h 2^-57 + l 2^-73 with any l (64-bit integers).
struct Fix {
  long long h, l;
  __device__ __forceinline__ long long hi() const { return h + (l >> 16); }
  __device__ __forceinline__ unsigned short lo() const { return static_cast<unsigned short>(l); }
};
__device__ __forceinline__ Fix operator-(Fix a, Fix b) { return Fix{a.h - b.h, a.l - b.l}; }
// a - 1 where cond holds
__device__ __forceinline__ Fix less_one(Fix a, bool cond) { return Fix{a.h - (cond ? 1ll << (RNS_FRAC - 16) : 0), a.l}; }

__device__ __forceinline__ unsigned long long offset_binary(long long a) {
  return static_cast<unsigned long long>(a) ^ 0x8000000000000000ull;
}

// N mod m_i for eight entries, as BF16: the ten bytes of each entry (offset
// binary, u the upper eight) against 256^k mod m, then one balanced reduction in FP32.
template <int I>
__device__ __forceinline__ uint4 residues8(const unsigned long long* u, const unsigned* lo) {
  uint32_t o[4];
  float r[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    int acc = kTab.bias[I];
    asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(acc) : "r"(lo[e]), "r"(kTab.pow_lo[I]));
    asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(acc) : "r"(uint32_t(u[e])), "r"(kTab.pow_mid[I]));
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

// The moduli that a residue set holds at a time: all, or a half (PARTS 2).
template <int PARTS, int PART>
struct ModRange {
  static constexpr int planes = rns_planes(PARTS), first = PART * planes;
  static constexpr int last = first + planes < RNS_MODS ? first + planes : RNS_MODS;
};

template <class M, int I = M::first>
__device__ __forceinline__ void store_residues8(const unsigned long long* u, const unsigned* lo, __nv_bfloat16* dst,
                                                int64_t plane) {
  if constexpr (I < M::last) {
    *reinterpret_cast<uint4*>(dst + int64_t(I - M::first) * plane) = residues8<I>(u, lo);
    store_residues8<M, I + 1>(u, lo, dst, plane);
  }
}

// rint(x 2^e) of a double, |x 2^e| < 2^77, at 2^-73, with integer operations
__device__ __forceinline__ Fix to_fixed(double x, int e) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int ex = int((b >> 52) & 0x7FF);
  if (ex == 0) return Fix{0, 0};
  const unsigned long long mant = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const int sh = ex - 1075 + e;  // callers keep it below 25
  unsigned long long h = 0, l = 0;
  if (sh >= 16) {
    h = sh < 25 ? mant << (sh - 16) : 0;
  } else if (sh >= 0) {
    h = mant >> (16 - sh);
    l = (mant << sh) & 0xFFFF;
  } else if (sh > -54) {
    l = ((mant >> (-sh - 1)) + 1) >> 1;
  }
  const long long sg = (b >> 63) ? -1 : 1;
  return Fix{sg * static_cast<long long>(h), sg * static_cast<long long>(l)};
}

// a product's sums times 2^shift, shift 0 .. 3, rounded: (f 2^-64 + g 2^-82) P / S^2
// from balanced 32-bit halves, |f| < 2^62.1 and P / S^2 below 4 keeping them in range.
// Sums that came about in other parts give the same bits.
__device__ __forceinline__ Fix product(long long f, int g, int shift) {
  f += g >> RNS_GUARD;
  g &= (1 << RNS_GUARD) - 1;
  const int fl = int(f), fh = int(f >> 32) - (fl >> 31), pl = kTab.pl, ph = kTab.ph;
  const long long a = static_cast<long long>(fh) * ph;  // at 2^-61
  long long b = static_cast<long long>(fh) * pl;        // at 2^-93
  b += static_cast<long long>(fl) * ph;
  b += __mulhi(fl, pl) + ((static_cast<long long>(g) * ph) >> RNS_GUARD);
  return Fix{a >> (4 - shift), ((a & ((16 >> shift) - 1)) << (12 + shift)) + ((b + (1ll << (19 - shift))) >> (20 - shift))};
}

// smallest sh with row norms 2^-sh sqrt(norm2) <= 1
__device__ __forceinline__ int norm_shift(unsigned bits) {
  const float f = __uint_as_float(bits);
  if (!(f > 0.0f)) return 0;
  const int e = int(bits >> 23) - 126;  // f < 2^e
  return e >= 0 ? (e + 1) / 2 : -(-e / 2);
}

// |x| as FP32, nonzero where x is (a floor that keeps products of two in range)
__device__ __forceinline__ float weight(double x) {
  return x == 0.0 ? 0.0f : fmaxf(fabsf(d2f_trunc(x)), 0x1p-60f);
}

__device__ __forceinline__ float warp_sum(float a) {
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

// Squared row norms: the largest into norm2, the smallest nonzero one into least (a
// level of its own that the grid would lose).  least becomes 0 where a norm is above
// 2, which the operands' scales do not allow for (values beyond FP32's range, whose
// bounds saturate, and power estimates far below the spectral radius).
__global__ void __launch_bounds__(256) k_rns_rownorm(WaveDev w, const double* __restrict__ X,
                                                     const int* __restrict__ state, unsigned* norm2, unsigned* least) {
  const int s = blockIdx.y;
  if (state && state[s] == ST_DONE) return;
  const int ld = w.ld[s], n = w.n[s];
  const double* Xs = X + w.off[s];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float most = 0.0f, few = __uint_as_float(0x7F7FFFFFu);
  for (int r = blockIdx.x * 8 + warp; r < n; r += gridDim.x * 8) {
    float acc = 0.0f;
    for (int c = 2 * lane; c < ld; c += 64) {
      const double2 v = *reinterpret_cast<const double2*>(Xs + int64_t(r) * ld + c);
      const float a = weight(v.x), b = weight(v.y);
      acc = fmaf(a, a, acc);
      acc = fmaf(b, b, acc);
    }
    acc = warp_sum(acc);
    most = fmaxf(most, acc);
    if (acc > 0.0f) few = fminf(few, acc);
  }
  if (most > 4.0f) few = 0.0f;
  // sums of truncated squares: the margin covers truncation and rounding (ld <= 32768)
  if (lane == 0 && most > 0.0f) {
    atomicMax(&norm2[s], __float_as_uint(most * 1.01f));
    atomicMin(&least[s], __float_as_uint(few));
  }
}

// Coupling of a submatrix's extracted columns to its rows: whether some entry that
// the scatter reads has 0 < (|X| |X|)_rc < RNS_LEAST_COUPLING (into least).  A warp
// takes 32 entries of a row: the term |X_rc| |X_cc| alone, a lower bound, decides
// nearly all of them with one read of the extracted columns; where it does not, the
// sum is formed, from the columns' own rows on and only until it is large enough.
__global__ void __launch_bounds__(256) k_rns_coupling(PatternDev g, WaveDev w, const double* __restrict__ X,
                                                      const int* __restrict__ state, unsigned* least) {
  extern __shared__ float diag[];  // |X_cc| of the block's columns
  const int s = blockIdx.y;
  if (state && state[s] == ST_DONE) return;
  const int ld = w.ld[s], n = w.n[s], q = w.sub[s];
  const double* Xs = X + w.off[s];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const volatile unsigned* known = least;
  int64_t k0 = 0;
  int b = 0;
  auto row = [&](int r) {
    const double* xr = Xs + int64_t(r) * ld;
    for (int c0 = 0; c0 < b; c0 += 32) {
      if (__uint_as_float(__shfl_sync(0xffffffffu, known[s], 0)) < RNS_LEAST_COUPLING) return;  // decided
      const int c = c0 + lane;
      const bool mine = c < b;
      if (__all_sync(0xffffffffu, !mine || weight(xr[k0 + c]) * diag[c] >= RNS_LEAST_COUPLING)) continue;
      const int chunks = (n + 31) / 32, first = int(k0 + c0) / 32;
      float a = 0.0f;
      for (int t = 0; t < chunks; ++t) {
        const int k1 = (first + t) % chunks * 32;
        const float x = k1 + lane < n ? weight(xr[k1 + lane]) : 0.0f;
        unsigned some = __ballot_sync(0xffffffffu, x != 0.0f);
        if (some == 0) continue;
        for (; some; some &= some - 1) {
          const int k = __ffs(int(some)) - 1;
          const float xk = __shfl_sync(0xffffffffu, x, k);
          if (mine) a = fmaf(xk, weight(Xs[int64_t(k1 + k) * ld + k0 + c]), a);
        }
        if (__all_sync(0xffffffffu, !mine || a >= RNS_LEAST_COUPLING)) break;
      }
      if (mine && a > 0.0f && a < RNS_LEAST_COUPLING) atomicMin(&least[s], __float_as_uint(a));
    }
  };
  auto columns = [&](int j, int64_t at) {
    k0 = at;
    b = g.bs[j];
    __syncthreads();
    for (int c = threadIdx.x; c < b; c += 256) diag[c] = weight(Xs[(k0 + c) * ld + k0 + c]);
    __syncthreads();
  };
  if (!g.mp) {  // one block column: every row
    columns(q, g.koff[q]);
    for (int r = blockIdx.x * 8 + warp; r < n; r += gridDim.x * 8) row(r);
    return;
  }
  for (int mi = g.mp[q]; mi < g.mp[q + 1]; ++mi) {
    const int j = g.mcol[mi];
    columns(j, g.mkoff[mi]);
    for (int64_t p = g.row_ptr[j] + blockIdx.x; p < g.row_ptr[j + 1]; p += gridDim.x) {
      const int r0 = g.dloc[g.tpos[p]], nr = g.bs[g.col[p]];
      for (int t = warp; t < nr; t += 8) row(r0 + t);
    }
  }
}

// route[s]: ST_DONE for the chains, ST_ACTIVE for the residues.  With state, an
// active submatrix of the chains is held (ST_DONE) meanwhile.
__global__ void k_rns_route(int nsub, const unsigned* __restrict__ least, int* __restrict__ route, int* state,
                            int* chains) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nsub) return;
  bool chain = __uint_as_float(least[s]) < RNS_LEAST_COUPLING;
  if (chain && state) {
    chain = state[s] == ST_ACTIVE;
    if (chain) state[s] = ST_DONE;
  }
  route[s] = chain ? ST_DONE : ST_ACTIVE;
  if (chain) atomicAdd(chains, 1);
}

__global__ void k_rns_resume(int nsub, const int* __restrict__ route, int* __restrict__ state) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < nsub && route[s] == ST_DONE) state[s] = ST_ACTIVE;
}

template <class M>
__global__ void __launch_bounds__(256) k_rns_convert(WaveDev w, const double* X, const int* __restrict__ state,
                                                     const unsigned* __restrict__ norm2, int sh_fixed,
                                                     __nv_bfloat16* __restrict__ R, RnsFix fixed) {
  const int s = blockIdx.y;
  if (state && state[s] == ST_DONE) return;
  const int e = RNS_FRAC - (norm2 ? norm_shift(norm2[s]) : sh_fixed);
  const int ld = w.ld[s];
  const int64_t plane = int64_t(ld) * ld, base = w.off[s];
  for (int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) * 8; i < plane;
       i += int64_t(gridDim.x) * blockDim.x * 8) {
    double x[8];
    unsigned long long u[8];
    unsigned lo[8];
#pragma unroll
    for (int k = 0; k < 8; k += 2)
      *reinterpret_cast<double2*>(x + k) = *reinterpret_cast<const double2*>(X + base + i + k);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const Fix v = to_fixed(x[k], e);
      u[k] = offset_binary(v.hi());
      lo[k] = v.lo();
    }
    if (R) store_residues8<M>(u, lo, R + M::planes * base + i, plane);
    if (fixed.hi) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const Fix v = to_fixed(x[k], RNS_FRAC);
        fixed.hi[base + i + k] = v.hi();
        fixed.lo[base + i + k] = v.lo();
      }
    }
  }
}

// ---------------------------------------------------------------------------
// 64 x 64 tile pairs (a, b), a <= b: values from the upper tile, results to both
// ---------------------------------------------------------------------------

// The upper tile; pitches that keep both triangles' accesses off the same banks.
struct Tile {
  long long hi[64][65];
  unsigned short lo[64][66];
  __device__ __forceinline__ void put(int r, int c, Fix n) {
    hi[r][c] = n.hi();
    lo[r][c] = n.lo();
  }
};

__device__ __forceinline__ void pair_of(int pi, int T, int* a, int* b) {
  int x = 0;
  while (pi >= T - x) { pi -= T - x; ++x; }
  *a = x;
  *b = x + pi;
}

// place of entry (r, c) in the pair's upper tile: transposed for the lower tile
// (t), and in a diagonal tile (a == b), which is read from its upper triangle
__device__ __forceinline__ int2 place(int r, int c, bool t, bool diag) {
  return t || (diag && r > c) ? make_int2(c, r) : make_int2(r, c);
}

// residues of the staged tile into tile (a, b) and, transposed, (b, a):
// 512 segments of eight entries a tile, two per thread
template <class M = ModRange<1, 0>>
__device__ __forceinline__ void tile_residues(const Tile& v, int a, int b, int ld, __nv_bfloat16* R, int64_t plane) {
  for (int t = 0; t < (a == b ? 1 : 2); ++t)
#pragma unroll 1
    for (int g = threadIdx.x; g < 512; g += 256) {
      const int r = g >> 3, c0 = (g & 7) * 8;
      unsigned long long u[8];
      unsigned lo[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int2 at = place(r, c0 + k, t != 0, a == b);
        u[k] = offset_binary(v.hi[at.x][at.y]);
        lo[k] = v.lo[at.x][at.y];
      }
      const int row = (t ? b : a) * 64 + r, col = (t ? a : b) * 64 + c0;
      store_residues8<M>(u, lo, R + int64_t(row) * ld + col, plane);
    }
}

// staged tile as FP64 (times scale 2^-73) into both tiles of the pair
__device__ __forceinline__ void tile_doubles(const Tile& v, int a, int b, int ld, double scale, double* X) {
  const double sh = scale * 0x1p-57, sl = scale * 0x1p-73;
  const int c = (threadIdx.x & 31) * 2;
  for (int t = 0; t < (a == b ? 1 : 2); ++t)
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      double o[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int2 at = place(r, c + k, t != 0, a == b);
        o[k] = fma(double(v.hi[at.x][at.y]), sh, double(int(v.lo[at.x][at.y])) * sl);
      }
      *reinterpret_cast<double2*>(X + int64_t((t ? b : a) * 64 + r) * ld + (t ? a : b) * 64 + c) =
          make_double2(o[0], o[1]);
    }
}

// 2^23 + a 23-bit piece, as a float, less 2^23: the piece, without a conversion
__device__ __forceinline__ float piece23(unsigned v) { return __uint_as_float(0x4B000000u | (v & 0x7FFFFFu)) - 8388608.0f; }

// sum += weight n^2, n to 2^-57 as an FP32 pair
__device__ __forceinline__ void add_square(Sum3& sum, Fix n, float weight) {
  const long long h = n.hi();
  const float c2 = float(int(h >> 46)) * 0x1p-11f, c1 = piece23(unsigned(h >> 23)) * 0x1p-34f;
  const float c0 = piece23(unsigned(h)) * 0x1p-57f;
  float a, e1, e0;
  two_sum(c2, c1, a, e1);
  two_sum(a, c0, a, e0);
  sum.add_square(a, __fadd_rn(e1, e0), weight);
}

__global__ void __launch_bounds__(256) k_rns_square0(WaveDev w, NsStateDev ns, const unsigned* __restrict__ norm2,
                                                     RnsSum F, double* Y) {
  __shared__ Tile v;
  const int s = blockIdx.y;
  if (ns.state[s] == ST_DONE) return;
  const int ld = w.ld[s], n = w.n[s], T = ld / 64;
  const long long* Fs = F.f + w.off[s];
  const int* Gs = F.g + w.off[s];
  const int sh = 2 * norm_shift(norm2[s]);
  const int c = (threadIdx.x & 31) * 2;
  Sum3 part;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    const float wgt = a == b ? 1.0f : 2.0f;
    __syncthreads();
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const int64_t i = int64_t(a * 64 + r) * ld + b * 64 + c;
      const longlong2 f = *reinterpret_cast<const longlong2*>(Fs + i);
      const int2 g = *reinterpret_cast<const int2*>(Gs + i);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const Fix y = product(k ? f.y : f.x, k ? g.y : g.x, 0);
        v.put(r, c + k, y);
        const bool dg = a == b && r == c + k && a * 64 + r < n;
        const Fix z = sh >= 0 ? Fix{y.h << sh, y.l << sh} : Fix{y.hi() >> min(-sh, 63), 0};
        add_square(part, less_one(z, dg), wgt);
      }
    }
    __syncthreads();
    tile_doubles(v, a, b, ld, ldexp(1.0, sh), Y + w.off[s]);
  }
  add_block_sum<8>(part.value(), &ns.res2[s]);
}

__global__ void __launch_bounds__(256) k_rns_square(WaveDev w, NsStateDev ns, RnsSum F, RnsFix Y,
                                                    __nv_bfloat16* __restrict__ R) {
  __shared__ Tile v;
  const int s = blockIdx.y;
  if (ns.state[s] == ST_DONE) return;
  const int ld = w.ld[s], n = w.n[s], T = ld / 64;
  const int64_t base = w.off[s], plane = int64_t(ld) * ld;
  const int c = (threadIdx.x & 31) * 2;
  Sum3 part;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    const float wgt = a == b ? 1.0f : 2.0f;
    __syncthreads();
#pragma unroll 4
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const int64_t i = base + int64_t(a * 64 + r) * ld + b * 64 + c;
      const longlong2 f = *reinterpret_cast<const longlong2*>(F.f + i);
      const int2 g = *reinterpret_cast<const int2*>(F.g + i);
      const Fix y[2] = {product(f.x, g.x, 0), product(f.y, g.y, 0)};
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        v.put(r, c + k, y[k]);
        const bool dg = a == b && r == c + k && a * 64 + r < n;
        add_square(part, less_one(y[k], dg), wgt);
      }
      if (Y.hi) {
        *reinterpret_cast<longlong2*>(Y.hi + i) = make_longlong2(y[0].hi(), y[1].hi());
        *reinterpret_cast<ushort2*>(Y.lo + i) = make_ushort2(y[0].lo(), y[1].lo());
      }
    }
    __syncthreads();
    if (R) tile_residues(v, a, b, ld, R + RNS_MODS * base, plane);
  }
  add_block_sum<8>(part.value(), &ns.res2[s]);
}

// (3 x - z) / 2
__device__ __forceinline__ Fix update(Fix x, Fix z) {
  const long long h = 3 * x.h - z.h, l = 3 * x.l - z.l + 1;
  return Fix{h >> 1, (l + ((h & 1) << 16)) >> 1};
}

__global__ void __launch_bounds__(256) k_rns_update(WaveDev w, NsStateDev ns, RnsSum F, int shift, RnsFix X,
                                                    __nv_bfloat16* __restrict__ R) {
  __shared__ Tile v;
  const int s = blockIdx.y;
  const int state = ns.state[s];
  if (state == ST_DONE) return;
  const bool last = state == ST_LAST;
  const int ld = w.ld[s], T = ld / 64;
  const int64_t base = w.off[s], plane = int64_t(ld) * ld;
  const int c = (threadIdx.x & 31) * 2;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    __syncthreads();
#pragma unroll 4
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const int64_t i = base + int64_t(a * 64 + r) * ld + b * 64 + c;
      const longlong2 f = *reinterpret_cast<const longlong2*>(F.f + i);
      const int2 g = *reinterpret_cast<const int2*>(F.g + i);
      const longlong2 xh = *reinterpret_cast<const longlong2*>(X.hi + i);
      const ushort2 xl = *reinterpret_cast<const ushort2*>(X.lo + i);
      const Fix x0 = update(Fix{xh.x, xl.x}, product(f.x, g.x, shift));
      const Fix x1 = update(Fix{xh.y, xl.y}, product(f.y, g.y, shift));
      v.put(r, c, x0);
      v.put(r, c + 1, x1);
      if (!last) {
        *reinterpret_cast<longlong2*>(X.hi + i) = make_longlong2(x0.hi(), x1.hi());
        *reinterpret_cast<ushort2*>(X.lo + i) = make_ushort2(x0.lo(), x1.lo());
      }
    }
    __syncthreads();
    if (last) tile_doubles(v, a, b, ld, 1.0, reinterpret_cast<double*>(X.hi + base));
    else if (R) tile_residues(v, a, b, ld, R + RNS_MODS * base, plane);
  }
}

// Residues of a fixed-point matrix for a part of the moduli.
template <class M>
__global__ void __launch_bounds__(256) k_rns_spread(WaveDev w, const int* __restrict__ state, RnsFix X,
                                                    __nv_bfloat16* __restrict__ R) {
  __shared__ Tile v;
  const int s = blockIdx.y;
  if (state[s] == ST_DONE) return;
  const int ld = w.ld[s], T = ld / 64;
  const int64_t base = w.off[s], plane = int64_t(ld) * ld;
  const int c = (threadIdx.x & 31) * 2;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    __syncthreads();
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const int64_t i = base + int64_t(a * 64 + r) * ld + b * 64 + c;
      const longlong2 h = *reinterpret_cast<const longlong2*>(X.hi + i);
      const ushort2 l = *reinterpret_cast<const ushort2*>(X.lo + i);
      v.put(r, c, Fix{h.x, l.x});
      v.put(r, c + 1, Fix{h.y, l.y});
    }
    __syncthreads();
    tile_residues<M>(v, a, b, ld, R + M::planes * base, plane);
  }
}

__global__ void __launch_bounds__(256) k_rns_cheb2(WaveDev w, RnsSum F, double* __restrict__ T2) {
  __shared__ Tile v;
  const int s = blockIdx.y;
  const int ld = w.ld[s], n = w.n[s], T = ld / 64;
  const int64_t base = w.off[s];
  const int c = (threadIdx.x & 31) * 2;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    __syncthreads();
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const int64_t i = base + int64_t(a * 64 + r) * ld + b * 64 + c;
      const longlong2 f = *reinterpret_cast<const longlong2*>(F.f + i);
      const int2 g = *reinterpret_cast<const int2*>(F.g + i);
      const bool row = a == b && a * 64 + r < n;
      v.put(r, c, less_one(product(f.x, g.x, 1), row && r == c));
      v.put(r, c + 1, less_one(product(f.y, g.y, 1), row && r == c + 1));
    }
    __syncthreads();
    tile_doubles(v, a, b, ld, 1.0, T2 + base);
  }
}

// Sum of t c over RNS_COMB terms, t at 2^-73 and c at 2^-58, from balanced 32-bit
// halves at 2^-51, 2^-83 and 2^-99: |t| <= 1 and |c| <= 5.1 (a combination of norm 4
// has coefficients of 4 / pi times that) keep them in range.
struct Comb {
  long long h = 0, m = 0, l = 0;
  __device__ __forceinline__ void add(long long t, unsigned tlo, long long c) {
    const int tl = int(t), th = int(t >> 32) - (tl >> 31);
    const int cl = int(c), ch = int(c >> 32) - (cl >> 31);
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(h) : "r"(th), "r"(ch));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(m) : "r"(th), "r"(cl));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(m) : "r"(tl), "r"(ch));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(l) : "r"(int(tlo)), "r"(ch));
    m += __mulhi(tl, cl);
  }
  __device__ __forceinline__ Fix sum() const {
    return Fix{h << 6, (m + (l >> 16) + (1ll << 9)) >> 10};
  }
};

// One step of the recurrences, as a pass over tile pairs: bound by memory
// traffic (the residues written, 38 bytes an entry, are the largest part), so
// the combination of the stored odd T_k is formed here instead of in a pass of
// its own, and only upper tiles are read.
template <bool COMB>
__global__ void __launch_bounds__(256) k_rns_cheb(WaveDev w, const __grid_constant__ RnsCheb p) {
  __shared__ Tile v;
  const int s = blockIdx.y;
  if (p.state[s] == ST_DONE) return;
  const int ld = w.ld[s], T = ld / 64;
  const int64_t base = w.off[s], plane = int64_t(ld) * ld;
  const int c = (threadIdx.x & 31) * 2;
  for (int pi = blockIdx.x; pi < T * (T + 1) / 2; pi += gridDim.x) {
    int a, b;
    pair_of(pi, T, &a, &b);
    __syncthreads();
#pragma unroll 2
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {
      const int64_t i = base + int64_t(a * 64 + r) * ld + b * 64 + c;
      Fix x0{0, 0}, x1{0, 0};
      if (p.F.f) {
        const longlong2 f = *reinterpret_cast<const longlong2*>(p.F.f + i);
        const int2 g = *reinterpret_cast<const int2*>(p.F.g + i);
        x0 = product(f.x, g.x, p.twice);
        x1 = product(f.y, g.y, p.twice);
      }
      if (p.sub.hi) {
        const longlong2 z = *reinterpret_cast<const longlong2*>(p.sub.hi + i);
        const ushort2 zl = *reinterpret_cast<const ushort2*>(p.sub.lo + i);
        x0 = x0 - Fix{z.x, zl.x};
        x1 = x1 - Fix{z.y, zl.y};
      }
      if constexpr (COMB) {
        Comb c0, c1;
#pragma unroll
        for (int q = 0; q < RNS_COMB; ++q) {
          const longlong2 t = *reinterpret_cast<const longlong2*>(p.odd.hi + q * p.stride + i);
          const ushort2 tl = *reinterpret_cast<const ushort2*>(p.odd.lo + q * p.stride + i);
          c0.add(t.x, tl.x, p.coef[q]);
          c1.add(t.y, tl.y, p.coef[q]);
        }
        const Fix s0 = c0.sum(), s1 = c1.sum();
        x0 = Fix{x0.h + s0.h, x0.l + s0.l};
        x1 = Fix{x1.h + s1.h, x1.l + s1.l};
      }
      v.put(r, c, x0);
      v.put(r, c + 1, x1);
      if (p.C.hi) {
        *reinterpret_cast<longlong2*>(p.C.hi + i) = make_longlong2(x0.hi(), x1.hi());
        *reinterpret_cast<ushort2*>(p.C.lo + i) = make_ushort2(x0.lo(), x1.lo());
      }
    }
    __syncthreads();
    if (p.out) tile_doubles(v, a, b, ld, p.out_scale, p.out + base);
    if (p.R) tile_residues(v, a, b, ld, p.R + RNS_MODS * base, plane);
  }
}

// about four tile pairs a block, but fewer where the wave would give less than four
// blocks per SM
dim3 tile_grid(int max_ld, int nsub) {
  const int T = max_ld / 64, pairs = T * (T + 1) / 2;
  int per = 4;
  while (per > 1 && int64_t((pairs + per - 1) / per) * nsub < 4 * int64_t(num_sms())) per /= 2;
  return dim3(unsigned(std::min((pairs + per - 1) / per, 512)), unsigned(nsub));
}

}  // namespace

int rns_split(int ntiles, int nmod, int nsm) {
  // Tiles alone fill the chip from two per SM on.  Below that the moduli of a
  // tile go to several CTAs, which add their sums modulo 2^64 (exact in any
  // order), at most one modulus each.
  if (ntiles >= 2 * nsm) return 1;
  return std::max(1, std::min(nmod, (2 * nsm) / std::max(1, ntiles)));
}

cudaError_t launch_rns_gemm(RnsGemmParams p, int nsm, cudaStream_t st) {
  if (p.nitems <= 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_rns_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
  if (e != cudaSuccess) return e;
  k_rns_gemm<<<std::min(p.nitems * p.split, nsm), THREADS, SMEM, st>>>(p);
  count_launch();
  return cudaGetLastError();
}

constexpr int ROUTE_SMEM = 200 * 1024;
bool rns_route_fits(int bs_max) { return size_t(bs_max) * sizeof(float) <= ROUTE_SMEM; }

cudaError_t launch_rns_route(const PatternDev& g, const WaveDev& w, const double* X, int* state, unsigned* norm2,
                             unsigned* least, int* route, int* chains, int bs_max, int max_ld, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(norm2, 0, sizeof(unsigned) * size_t(w.nsub), st);
  if (e != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(least, 0x7F, sizeof(unsigned) * size_t(w.nsub), st)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(chains, 0, sizeof(int), st)) != cudaSuccess) return e;
  const dim3 grid(unsigned(std::min((max_ld + 31) / 32, 64)), unsigned(w.nsub));
  k_rns_rownorm<<<grid, 256, 0, st>>>(w, X, state, norm2, least);
  count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_rns_coupling, cudaFuncAttributeMaxDynamicSharedMemorySize, ROUTE_SMEM)) !=
      cudaSuccess)
    return e;
  k_rns_coupling<<<grid, 256, size_t(bs_max) * sizeof(float), st>>>(g, w, X, state, least);
  count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_rns_route<<<(w.nsub + 255) / 256, 256, 0, st>>>(w.nsub, least, route, state, chains);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_resume(const WaveDev& w, const int* route, int* state, cudaStream_t st) {
  k_rns_resume<<<(w.nsub + 255) / 256, 256, 0, st>>>(w.nsub, route, state);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_convert(const WaveDev& w, const double* X, const int* state, const unsigned* norm2,
                               int sh_fixed, __nv_bfloat16* R, RnsFix fixed, int max_ld, cudaStream_t st, int parts,
                               int part) {
  const int64_t bx = (int64_t(max_ld) * max_ld + 256 * 32 - 1) / (256 * 32);
  const auto kern = parts == 1  ? k_rns_convert<ModRange<1, 0>>
                    : part == 0 ? k_rns_convert<ModRange<2, 0>>
                                : k_rns_convert<ModRange<2, 1>>;
  kern<<<dim3(unsigned(std::min<int64_t>(bx, 1024)), unsigned(w.nsub)), 256, 0, st>>>(w, X, state, norm2, sh_fixed, R,
                                                                                     fixed);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_spread(const WaveDev& w, const int* state, RnsFix X, __nv_bfloat16* R, int max_ld,
                              cudaStream_t st, int part) {
  const auto kern = part == 0 ? k_rns_spread<ModRange<2, 0>> : k_rns_spread<ModRange<2, 1>>;
  kern<<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, state, X, R);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_square0(const WaveDev& w, NsStateDev ns, const unsigned* norm2, RnsSum F, double* Y,
                               int max_ld, cudaStream_t st) {
  k_rns_square0<<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, ns, norm2, F, Y);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_square(const WaveDev& w, NsStateDev ns, RnsSum F, RnsFix Y, __nv_bfloat16* R, int max_ld,
                              cudaStream_t st) {
  k_rns_square<<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, ns, F, Y, R);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_update(const WaveDev& w, NsStateDev ns, RnsSum F, int shift, RnsFix X, __nv_bfloat16* R,
                              int max_ld, cudaStream_t st) {
  k_rns_update<<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, ns, F, shift, X, R);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_cheb2(const WaveDev& w, RnsSum F, double* T2, int max_ld, cudaStream_t st) {
  k_rns_cheb2<<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, F, T2);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rns_cheb(const WaveDev& w, const RnsCheb& c, int max_ld, cudaStream_t st) {
  if (c.odd.hi) k_rns_cheb<true><<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, c);
  else k_rns_cheb<false><<<tile_grid(max_ld, w.nsub), 256, 0, st>>>(w, c);
  count_launch();
  return cudaGetLastError();
}

}  // namespace submat
