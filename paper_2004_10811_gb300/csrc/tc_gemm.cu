// Grouped BF16 tensor-core GEMM for sm_103a: tcgen05.mma with TMEM
// accumulators, operands staged by TMA (cp.async.bulk.tensor, 128B swizzle),
// an mbarrier pipeline, and one persistent CTA per SM.
//
// Every work item is one 128x128 output tile (s, ti, tj) of
//     C_s = alpha * sum_p A_{a(p)} B_{b(p)}^T + beta * C0_s
// over the submatrix batch.  Operands are row-major n x n BF16 arrays stored
// per size bucket as [count][ld][ld]; B is read as rows (B^T with K major),
// which equals B for the symmetric operands of Newton-Schulz.  A product table
// lets one launch sum several slice products into the FP32 accumulator, e.g.
// the three-term split hi*hi + hi*lo + lo*hi that carries about 16 bits
// through the tensor cores.
//
// Roles (192 or 320 threads): warp 0 issues TMA loads, warp 1 owns TMEM and one of
// its lanes issues the MMAs, warps 2-5 (or 2-9) drain the accumulator (one TMEM
// lane quarter each, or half of one) and write the tile -- and, for symmetric
// outputs, its mirror.  Every mbarrier wait is bounded; on
// timeout the kernel raises FLAG_TIMEOUT, drains its own copies and MMAs,
// frees TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "tc_gemm.cuh"
#include "tcgen05.cuh"

namespace submat {

namespace {

constexpr int BM = 128, BK = 64;
constexpr int TILE_BYTES = BM * BK * 2;  // one 128 x 64 BF16 operand tile (A side)
// integer outputs: one 16-column int64 row segment per thread, rows 144 bytes
// apart (16-byte aligned for the bulk copy, padded against bank conflicts)
constexpr int I64_SEG = 16, I64_PITCH = 144;
constexpr int STG_BYTES = BM * I64_PITCH;

// instruction descriptor: D F32, A and B BF16, both K-major, M = 128, N = cols
// (FP16 operands clear the two format fields, bits 7-9 and 10-12)
__device__ __forceinline__ constexpr uint32_t idesc(int cols) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(cols >> 3) << 17) | (uint32_t(BM >> 4) << 24);
}

// Columns of a tile that its MMAs form: those inside the matrix (ld is a
// multiple of 64), and of a 256-wide tile of a symmetric result whose left half
// lies below the diagonal the right half only.
struct TileCols {
  int lo, hi;
};
template <int BN>
__device__ __forceinline__ TileCols tile_cols(const int4& item, int ld, int sym) {
  return TileCols{BN == 256 && sym && item.z * 2 < item.y ? 128 : 0, min(BN, ld - item.z * BN)};
}

__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_split(float o) {
  const __nv_bfloat16 h = __float2bfloat16_rn(o);
  const __nv_bfloat16 l = __float2bfloat16_rn(o - __bfloat162float(h));
  return uint32_t(__bfloat16_as_ushort(h)) | (uint32_t(__bfloat16_as_ushort(l)) << 16);
}

// two values as (hi, lo) BF16 pairs: hi = rn(v), lo = rn(v - hi), two
// values per conversion instruction; bit-identical to pack_split
__device__ __forceinline__ void pack_split2(float a, float b, uint32_t* hw, uint32_t* lw) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const float2 hf = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
  *hw = *reinterpret_cast<const uint32_t*>(&h);
  *lw = *reinterpret_cast<const uint32_t*>(&l);
}

// the FP16 forms of the two above (operands in FP16: TcGemmParams::f16)
__device__ __forceinline__ uint32_t pack_split_h(float o) {
  const __half h = __float2half_rn(o);
  const __half l = __float2half_rn(o - __half2float(h));
  return uint32_t(__half_as_ushort(h)) | (uint32_t(__half_as_ushort(l)) << 16);
}

__device__ __forceinline__ void pack_split2_h(float a, float b, uint32_t* hw, uint32_t* lw) {
  const __half2 h = __floats2half2_rn(a, b);
  const float2 hf = __half22float2(h);
  const __half2 l = __floats2half2_rn(a - hf.x, b - hf.y);
  *hw = *reinterpret_cast<const uint32_t*>(&h);
  *lw = *reinterpret_cast<const uint32_t*>(&l);
}

// one 32-byte store (a full L2 sector); the address is 32-byte aligned
__device__ __forceinline__ void st_v8(void* d, const uint32_t* w) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(d), "r"(w[0]), "r"(w[1]),
               "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

// write 32 values (one row segment, 64-byte aligned) in the output format,
// in whole 32-byte sectors
template <bool F16>
__device__ __forceinline__ void store_row(const TcGemmParams& p, int64_t idx, const float* o) {
  if (p.out_f32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) st_v8(p.out_f32 + idx + 8 * q, reinterpret_cast<const uint32_t*>(o + 8 * q));
  } else {
    uint32_t hw[16], lw[16];
    if constexpr (F16) {
#pragma unroll
      for (int q = 0; q < 16; ++q) pack_split2_h(o[2 * q], o[2 * q + 1], &hw[q], &lw[q]);
    } else {
#pragma unroll
      for (int q = 0; q < 16; ++q) pack_split2(o[2 * q], o[2 * q + 1], &hw[q], &lw[q]);
    }
    st_v8(p.out_hi + idx, hw);
    st_v8(p.out_hi + idx + 16, hw + 8);
    if (p.out_lo) {
      st_v8(p.out_lo + idx, lw);
      st_v8(p.out_lo + idx + 16, lw + 8);
    }
  }
}

// store o[q] for q >= q_lo only (diagonal tiles of symmetric outputs): whole
// segments as vectors, element stores only where the diagonal crosses
template <bool F16>
__device__ __forceinline__ void store_range(const TcGemmParams& p, int64_t idx, const float* o, int q_lo) {
  if (q_lo >= 32) return;
  if (q_lo <= 0) {
    store_row<F16>(p, idx, o);
    return;
  }
#pragma unroll
  for (int q = 0; q < 32; ++q) {
    if (q < q_lo) continue;
    if (p.out_f32) {
      p.out_f32[idx + q] = o[q];
    } else {
      const uint32_t w = F16 ? pack_split_h(o[q]) : pack_split(o[q]);
      p.out_hi[idx + q] = __ushort_as_bfloat16(static_cast<unsigned short>(w & 0xFFFFu));
      if (p.out_lo) p.out_lo[idx + q] = __ushort_as_bfloat16(static_cast<unsigned short>(w >> 16));
    }
  }
}

template <bool F16>
__device__ __forceinline__ void load_c0(const TcGemmParams& p, int64_t idx, float* c) {
  if (p.c0_f32) {
    // whole 32-byte sectors per load
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t w[8];
      asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]),
                     "=r"(w[7])
                   : "l"(p.c0_f32 + idx + 8 * q));
#pragma unroll
      for (int e = 0; e < 8; ++e) c[8 * q + e] = __uint_as_float(w[e]);
    }
  } else {
    const uint4* sh = reinterpret_cast<const uint4*>(p.c0_hi + idx);
    const uint4* sl = p.c0_lo ? reinterpret_cast<const uint4*>(p.c0_lo + idx) : nullptr;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 h = sh[q];
      const uint4 l = sl ? sl[q] : make_uint4(0, 0, 0, 0);
      const uint32_t hh[4] = {h.x, h.y, h.z, h.w}, ll[4] = {l.x, l.y, l.z, l.w};
      if constexpr (F16) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 fh = __half22float2(*reinterpret_cast<const __half2*>(&hh[e]));
          const float2 fl = __half22float2(*reinterpret_cast<const __half2*>(&ll[e]));
          c[8 * q + 2 * e] = fh.x + fl.x;
          c[8 * q + 2 * e + 1] = fh.y + fl.y;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          c[8 * q + 2 * e] = __uint_as_float(hh[e] << 16) + __uint_as_float(ll[e] << 16);
          c[8 * q + 2 * e + 1] =
              __uint_as_float(hh[e] & 0xFFFF0000u) + __uint_as_float(ll[e] & 0xFFFF0000u);
        }
      }
    }
  }
}

// The epilogue a launch compiles in, both draining 32 columns at a time:
// EPI_FLOAT one accumulator, a 16-bit pair or FP32 output, double-buffered TMEM;
// EPI_INT integer sums of slice products.
// EPI_FLOAT has eight warps, two for each TMEM lane quarter, which take the
// chunks in turn (with four, a tile of few k-blocks took longer to convert and
// store than its MMAs: 1000 FP16 products of 192 dims 129 -> 111 us, and 83 us at
// a width of 256).  They write the mirror of a symmetric result too, so that no
// pass reads it back: 700 submatrices of 504-704 dims 51.4 -> 48.7 ms a build.
enum Epilogue { EPI_FLOAT, EPI_INT };
__host__ __device__ constexpr int epi_warps(int mode) { return mode == EPI_FLOAT ? 8 : 4; }

// A warp's 32 x 32 chunk (lane: row, o: columns) to its mirrored place, whose
// first row and column are row0 and col0; diagonal: only entries below the
// diagonal.  FP32 goes out column by column; of a 16-bit pair two lanes exchange
// halves, so that each stores two rows' entries of one column as a word.  (Not
// through shared memory, whose bandwidth bounds the MMAs: a staged transpose
// made Newton-Schulz products 30 % longer.)
template <bool F16>
__device__ __forceinline__ void store_mirror(const TcGemmParams& p, int64_t base, int ld, int row0, int col0,
                                             const float* o, int lane, bool diagonal) {
  if (p.out_f32) {
    float* d = p.out_f32 + base + int64_t(row0) * ld + col0 + lane;
#pragma unroll
    for (int q = 0; q < 32; ++q)
      if (!diagonal || q > lane) d[int64_t(q) * ld] = o[q];
    return;
  }
  const int odd = lane & 1, c = lane & ~1;
  const int64_t idx = base + int64_t(row0 + odd) * ld + col0 + c;
  auto put = [&](__nv_bfloat16* out, int64_t i, uint32_t v, int r) {
    if (!diagonal || r > c + 1) *reinterpret_cast<uint32_t*>(out + i) = v;
    else if (r == c + 1) out[i] = __ushort_as_bfloat16(static_cast<unsigned short>(v & 0xFFFFu));
  };
#pragma unroll
  for (int q = 0; q < 32; q += 2) {
    uint32_t hw, lw;
    if constexpr (F16) pack_split2_h(o[q], o[q + 1], &hw, &lw);
    else pack_split2(o[q], o[q + 1], &hw, &lw);
    const uint32_t ph = __shfl_xor_sync(0xffffffffu, hw, 1), pl = __shfl_xor_sync(0xffffffffu, lw, 1);
    const int64_t i = idx + int64_t(q) * ld;
    put(p.out_hi, i, odd ? __byte_perm(ph, hw, 0x7632) : __byte_perm(hw, ph, 0x5410), q + odd);
    if (p.out_lo) put(p.out_lo, i, odd ? __byte_perm(pl, lw, 0x7632) : __byte_perm(lw, pl, 0x5410), q + odd);
  }
}

// A lane's part of a tile's sum: two to four chunk sums, in a pair (exact for two,
// else to 2^-48 of the lane's part, less than FP64 loses over the tile).  The warp's
// sum goes through integers, 25, 23 and 24 bits at a time below the largest part's
// exponent, by redux instead of FP64 shuffles (a warp's FP64 instruction holds its
// pipe for 64 clocks).
struct TileSum {
  float h = 0.0f, l = 0.0f;
  __device__ __forceinline__ void add(float x) {
    float e;
    two_sum(h, x, h, e);
    l = __fadd_rn(l, e);
  }
  __device__ __forceinline__ double warp_sum() const {
    const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(h) & 0x7F800000u);
    if (top == 0x7F800000u) return double(__uint_as_float(0x7FC00000u));  // NaN or Inf among them
    const unsigned e = max(top, 24u << 23);
    const float up = __uint_as_float((278u << 23) - e), t = h * up, u = l * up;  // |t| < 2^25, |u| <= 3
    const int a = __float2int_rn(t);
    const float r = (t - float(a)) * 0x1p23f, s = u * 0x1p23f;
    const int b0 = __float2int_rn(r), b1 = __float2int_rn(s);
    const int c = __float2int_rn((r - float(b0)) * 0x1p24f) + __float2int_rn((s - float(b1)) * 0x1p24f);
    const long long A = __reduce_add_sync(0xffffffffu, a), B = __reduce_add_sync(0xffffffffu, b0 + b1);
    const long long C = __reduce_add_sync(0xffffffffu, c);
    // A + B 2^-23 + C 2^-47, at 2^-32, and 2^(e - 151) back
    const double v = double((A << 32) + (B << 9) + (C >> 15));
    return v * __longlong_as_double(static_cast<long long>(1023 - 32 - 151 + int(e >> 23)) << 52);
  }
};

template <int BN, int MODE, bool F16>
__global__ void __launch_bounds__(64 + 32 * epi_warps(MODE), 1) k_tc_gemm(const __grid_constant__ TcGemmParams p) {
  constexpr int TILE_B = BN * BK * 2;  // one BN x 64 BF16 operand tile (B side)
  constexpr int HALVES = BN / 128;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const int stage_bytes = p.na * TILE_BYTES + p.nb * TILE_B;
  uint8_t* tiles = smem;
  uint32_t* stg = reinterpret_cast<uint32_t*>(tiles + size_t(p.nstage) * stage_bytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(stg) + STG_BYTES);
  uint64_t* full = bars;
  uint64_t* empty = bars + p.nstage;
  uint64_t* tfull = empty + p.nstage;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* epi_ok = abort_flag + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < p.nstage; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 32 * epi_warps(MODE));
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(uint32_t(p.tmem_cols)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const long long limit = p.timeout_cycles;
  // accumulator sets in TMEM: two (MMA of the next tile overlaps the drain of
  // this one) when they fit, else one (freed as soon as the epilogue has read it)
  const int nbuf = p.tmem_cols >= 2 * p.nacc * BN ? 2 : 1;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    for (int m = 0; m < p.nmaps; ++m)
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&p.maps[m])) : "memory");
    int stage = 0;
    uint32_t phase = 0;
    uint32_t issued = 0, issued_phase = 0;  // per-stage bits
    bool ok = true;
    for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
      const int4 item = p.items[it];
      if (p.state && p.state[item.x] == p.skip_state) continue;
      const int bucket = item.w & 0xFF, slot = item.w >> 8;
      const int ld = p.ld[item.x], nk = ld / BK;
      const CUtensorMap* maps = p.maps + bucket;
      // 128-row boxes of the B tile that hold wanted columns
      const TileCols tc = tile_cols<BN>(item, ld, p.sym);
      const int box0 = tc.lo / 128, box1 = (tc.hi + 127) / 128;
      const uint32_t bytes = uint32_t(p.na + p.nb * (box1 - box0)) * TILE_BYTES;
      for (int kb = 0; kb < nk; ++kb) {
        if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, limit)) { ok = false; break; }
        uint8_t* st = tiles + size_t(stage) * stage_bytes;
        mbar_expect_tx(&full[stage], bytes);
        for (int a = 0; a < p.na; ++a)
          tma_load_3d(st + a * TILE_BYTES, maps + p.a_set[a] * p.nbucket, &full[stage], kb * BK,
                      item.y * BM, slot);
        for (int b = 0; b < p.nb; ++b)
          for (int x = box0; x < box1; ++x)
            tma_load_3d(st + p.na * TILE_BYTES + b * TILE_B + x * TILE_BYTES, maps + p.b_set[b] * p.nbucket,
                        &full[stage], kb * BK, item.z * BN + x * 128, slot);
        issued |= 1u << stage;
        issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
        if (++stage == p.nstage) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok) {
      atomicOr(p.flags, FLAG_TIMEOUT);
      *abort_flag = 1;
      // let this CTA's copies in flight land before shared memory is released
      for (int i = 0; i < p.nstage; ++i)
        if (issued & (1u << i)) {
          const long long t0 = clock64();
          while (!mbar_try_wait(&full[i], (issued_phase >> i) & 1u) && clock64() - t0 < limit) {
          }
        }
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer ----------------
    int stage = 0;
    uint32_t phase = 0;
    int tcount = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
      const int4 item = p.items[it];
      if (p.state && p.state[item.x] == p.skip_state) continue;
      const int ld = p.ld[item.x], nk = ld / BK;
      const int ab = nbuf == 2 ? (tcount & 1) : 0;
      const uint32_t tph = nbuf == 2 ? (uint32_t(tcount >> 1) & 1u) : (uint32_t(tcount) & 1u);
      if (!mbar_wait(&tempty[ab], tph ^ 1u, abort_flag, limit)) { ok = false; break; }
      tc_fence_after();
      const uint32_t dbase = tmem_base + uint32_t(ab * p.nacc * BN);
      const TileCols tc = tile_cols<BN>(item, ld, p.sym);
      // operand format: BF16 (A and B fields 1) or FP16 (both 0)
      const uint32_t id = idesc(tc.hi - tc.lo) & (F16 ? ~((7u << 7) | (7u << 10)) : ~0u);
      const uint32_t boff = uint32_t(tc.lo * BK * 2), doff = uint32_t(tc.lo);
      for (int kb = 0; kb < nk; ++kb) {
        if (!mbar_wait(&full[stage], phase, abort_flag, limit)) { ok = false; break; }
        tc_fence_after();
        const uint32_t sb = smem_u32(tiles + size_t(stage) * stage_bytes);
        for (int pr = 0; pr < p.nprod; ++pr) {
          const uint64_t ad = sdesc(sb + uint32_t(p.prod_a[pr] * TILE_BYTES));
          const uint64_t bd = sdesc(sb + uint32_t(p.na * TILE_BYTES + p.prod_b[pr] * TILE_B) + boff);
          const uint32_t d = dbase + uint32_t(p.prod_acc[pr] * BN) + doff;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            umma_bf16(d, ad + uint64_t(2 * k), bd + uint64_t(2 * k), id,
                      (kb > 0 || k > 0 || !p.prod_first[pr]) ? 1u : 0u);
        }
        umma_commit(&empty[stage]);
        if (++stage == p.nstage) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      umma_commit(&tfull[ab]);
      ++tcount;
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
  } else if (warp >= 2) {
    // ---------------- epilogue ----------------
    const int quarter = warp & 3;
    const int r = quarter * 32 + lane;  // tile row == TMEM lane
    int tcount = 0;
    for (int it = blockIdx.x; it < p.nitems; it += gridDim.x) {
      const int4 item = p.items[it];
      const int s = item.x;
      if (p.state && p.state[s] == p.skip_state) continue;
      const int ab = nbuf == 2 ? (tcount & 1) : 0;
      const uint32_t tph = nbuf == 2 ? (uint32_t(tcount >> 1) & 1u) : (uint32_t(tcount) & 1u);
      if constexpr (MODE == EPI_FLOAT) {
        // no shared memory to agree on: every warp waits by itself
        if (!__all_sync(0xffffffffu, mbar_wait(&tfull[ab], tph, abort_flag, limit))) {
          if (lane == 0) atomicOr(p.flags, FLAG_TIMEOUT);
          *abort_flag = 1;
          break;
        }
      } else {
        // one bounded wait, result shared, so the four warps leave together
        if (threadIdx.x == 64) {
          const bool got = mbar_wait(&tfull[ab], tph, abort_flag, limit);
          if (!got) {
            atomicOr(p.flags, FLAG_TIMEOUT);
            *abort_flag = 1;
          }
          *epi_ok = got ? 1 : 0;
        }
        epi_bar();
        if (!*epi_ok) break;
      }
      tc_fence_after();
      ++tcount;
      const int ld = p.ld[s];
      const int n = p.n[s];
      const int64_t base = p.off[s];
      const int rg = item.y * BM + r;
      const uint32_t tbase = tmem_base + (uint32_t(quarter * 32) << 16) + uint32_t(ab * p.nacc * BN);
      // 32 columns at a time, so only one chunk is live in registers, and the
      // diagonal handled only on diagonal sub-tiles.  TMEM is released after its
      // last read.
      {
        if constexpr (MODE == EPI_INT) {
          // exact integer sums of slice products (full tiles): per 32-column
          // chunk the sum over the accumulators of acc_k * 2^shift_k in 64-bit
          // integers (|acc_k| < 2^24, shift_k <= 36, at most four terms),
          // handed to the L2 bulk add in 16-column row segments
          const uint32_t tb = tbase;
#pragma unroll 1
          for (int c = 0; c < 4 * HALVES; ++c) {
            long long v[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = 0;
#pragma unroll 1
            for (int k = 0; k < p.nacc; ++k) {
              float a[32];
              tmem_ld32(tb + uint32_t(k * BN + c * 32), a);
              tmem_wait_ld();
              const int sh = p.i64_shifts[k];
#pragma unroll
              for (int q = 0; q < 32; ++q) v[q] += (long long)__float2int_rn(a[q]) << sh;
            }
            if (c == 4 * HALVES - 1) {
              tc_fence_before();
              if (!p.test_skip_arrive) mbar_arrive(&tempty[ab]);
            }
            const int cg0 = item.z * BN + c * 32;
            if (rg >= ld || cg0 >= ld) continue;
            uint8_t* srow = reinterpret_cast<uint8_t*>(stg) + r * I64_PITCH;
#pragma unroll
            for (int seg = 0; seg < 32 / I64_SEG; ++seg) {
              asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
#pragma unroll
              for (int q = 0; q < I64_SEG; ++q)
                *reinterpret_cast<long long*>(srow + 8 * q) = v[seg * I64_SEG + q];
              asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
              long long* d = p.out_i64 + base + int64_t(rg) * ld + cg0 + seg * I64_SEG;
              if (p.i64_accumulate)
                asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.u64 [%0], [%1], %2;" ::"l"(d),
                             "r"(smem_u32(srow)), "n"(I64_SEG * 8)
                             : "memory");
              else
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(d),
                             "r"(smem_u32(srow)), "n"(I64_SEG * 8)
                             : "memory");
              asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
          }
        } else {
          const int side = (warp - 2) >> 2;  // chunks side, side + 2, ...
          const bool has_c0 = (p.c0_f32 || p.c0_hi) && p.beta != 0.0f && !p.dot_c0;
          TileSum sum;  // for res2 or dot_c0
#pragma unroll 1
          for (int hc = side; hc < 4 * HALVES; hc += 2) {
            const int h = hc >> 2, c = hc & 3;
            const int sub_tj = item.z * HALVES + h;
            // below the diagonal or beyond the matrix: not formed, not written
            const bool skip = (p.sym && sub_tj < item.y) || sub_tj * 128 + c * 32 >= ld;
            float a[32];
            if (!skip) {
              tmem_ld32(tbase + uint32_t(hc * 32), a);
              tmem_wait_ld();
            }
            if (hc >= 4 * HALVES - 2) {
              tc_fence_before();
              if (!p.test_skip_arrive) mbar_arrive(&tempty[ab]);
            }
            if (skip) continue;
            const bool dtile = item.y == sub_tj;  // the diagonal crosses this sub-tile
            const bool diag_sym = p.sym && dtile;
            const int cg0 = sub_tj * 128 + c * 32;
            if (rg >= ld) continue;
            const int64_t idx = base + int64_t(rg) * ld + cg0;
            float c0[32];
            if (has_c0 || p.dot_c0) load_c0<F16>(p, idx, c0);
            float o[32];
            float pr = 0.0f, pd = 0.0f;
            if (!dtile) {
#pragma unroll
              for (int q = 0; q < 32; ++q) {
                float v = p.alpha * a[q];
                if (has_c0) v = fmaf(p.beta, c0[q], v);
                o[q] = v;
                pr = fmaf(a[q], a[q], pr);
                if (p.dot_c0) pd = fmaf(v, c0[q], pd);
              }
            } else {
              const int dq = (rg < n) ? rg - cg0 : -1;  // diagonal position in this segment
#pragma unroll
              for (int q = 0; q < 32; ++q) {
                float v = p.alpha * a[q];
                if (has_c0) v = fmaf(p.beta, c0[q], v);
                if (q == dq) v += p.diag;
                o[q] = v;
                const float e = a[q] - ((q == dq) ? 1.0f : 0.0f);
                pr = fmaf(e, e, pr);
                if (p.dot_c0) pd = fmaf(v, c0[q], pd);
              }
            }
            if (p.res2) sum.add(p.sym && !diag_sym ? 2.0f * pr : pr);
            if (p.dot_c0) sum.add(2.0f * pd);
            if (diag_sym) store_range<F16>(p, idx, o, r - c * 32);
            else store_row<F16>(p, idx, o);
            if (!p.sym || (diag_sym && c < quarter)) continue;
            store_mirror<F16>(p, base, ld, cg0, item.y * BM + quarter * 32, o, lane, diag_sym && c == quarter);
          }
          if (p.res2 || p.dot_c0) {
            const double t = sum.warp_sum();
            if (lane == 0 && t != 0.0) atomicAdd(p.res2 ? &p.res2[s] : &p.dot_c0[s], t);
          }
        }
      }
    }
    // bulk copies and adds issued by this thread are complete and visible
    if constexpr (MODE == EPI_INT) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(uint32_t(p.tmem_cols)));
  }
}

}  // namespace

int tc_smem_bytes(int na, int nb, int nstage, int bn) {
  return 1024 + nstage * (na * TILE_BYTES + nb * bn * BK * 2) + STG_BYTES + (2 * nstage + 5) * 8 +
         32;
}

int tc_pick_stages(int na, int nb, int bn) {
  const int budget = 227 * 1024;
  int st = 6;
  while (st > 2 && tc_smem_bytes(na, nb, st, bn) > budget) --st;
  return st;
}

cudaError_t launch_tc_gemm(const TcGemmParams& p, int grid, cudaStream_t st) {
  if (p.nitems <= 0) return cudaSuccess;
  const int bn = p.bn == 256 ? 256 : 128;
  if (bn == 256 && (p.tmem_cols != 512 || !(p.nacc == 1 || (p.nacc == 2 && p.out_i64))))
    return cudaErrorInvalidValue;
  if (p.nacc * bn > p.tmem_cols) return cudaErrorInvalidValue;
  if (p.out_i64) {
    // full tiles; up to four accumulators of weights 2^i64_shifts[k], combined in 64
    // bits (double-buffered where TMEM holds two sets, else freed once read)
    if (p.sym || p.f16 || p.nacc > 4) return cudaErrorInvalidValue;
    for (int k = 0; k < p.nacc; ++k)
      if (p.i64_shifts[k] < 0 || p.i64_shifts[k] > 36) return cudaErrorInvalidValue;
  } else if (p.nacc != 1 || p.tmem_cols < 2 * bn || !(p.out_f32 || p.out_hi)) {
    return cudaErrorInvalidValue;
  }
  const int smem = tc_smem_bytes(p.na, p.nb, p.nstage, bn);
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  auto run = [&](auto kern, int mode) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, 64 + 32 * epi_warps(mode), smem, st>>>(p);
    return cudaSuccess;
  };
  cudaError_t e;
  auto pick = [&](auto width) -> cudaError_t {
    constexpr int W = decltype(width)::value;
    if (p.out_i64) return run(k_tc_gemm<W, EPI_INT, false>, EPI_INT);
    return p.f16 ? run(k_tc_gemm<W, EPI_FLOAT, true>, EPI_FLOAT) : run(k_tc_gemm<W, EPI_FLOAT, false>, EPI_FLOAT);
  };
  e = bn == 256 ? pick(std::integral_constant<int, 256>()) : pick(std::integral_constant<int, 128>());
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// tensor maps
// ---------------------------------------------------------------------------

typedef CUresult (*PFN_encodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                    const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                    const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static PFN_encodeTiled get_encoder() {
  static PFN_encodeTiled fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_encodeTiled>(ptr);
  }
  return fn;
}

int make_bucket_map(CUtensorMap* out, const void* base, int ld, int count, int box_k) {
  PFN_encodeTiled enc = get_encoder();
  if (!enc) return -1;
  const cuuint64_t dims[3] = {cuuint64_t(ld), cuuint64_t(ld), cuuint64_t(count)};
  const cuuint64_t strides[2] = {cuuint64_t(ld) * 2, cuuint64_t(ld) * ld * 2};
  const cuuint32_t box[3] = {cuuint32_t(box_k), BM, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides,
                   box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   box_k == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : int(r);
}

}  // namespace submat
