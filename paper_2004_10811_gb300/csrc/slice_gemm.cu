// The exact sliced product of the mixed path's first correction (the splitting
// of Ozaki et al., see k_slice in mixed.cu), all kept slice pairs in one launch.
//
// Every level t = p + q has its own FP32 accumulator, exact because a chunk of
// the sum stays below 2^24: at most `pairs` products of 63^2 per term.  TMEM
// holds four accumulators of a 128 x 128 tile, so a chunk runs in two phases,
// levels 2 .. 5 and 6 .. 8, each loading every slice that it uses once per
// k-block for all its products (k-blocks of 32, so that three stages of nine
// slices fit).  The epilogue adds the levels up in 64-bit integers in registers,
// over all chunks, and the sum goes to memory once.  (Launches of at most eight
// products each loaded up to six slices for them, 136 bytes per clock at the full
// MMA rate where an SM takes in about 50, and read and wrote the sums again.)
//
// The levels are handed over one by one: with the last k-block of a phase each
// level is committed as its products are issued, so draining it overlaps the
// MMAs of the levels behind it and, behind its release, those of the next phase.
#include "slice_gemm.cuh"

#include <algorithm>
#include <cstring>

#include "tcgen05.cuh"

namespace submat {

namespace {

constexpr int TM = 128, TK = 32;
constexpr int TILE = TM * TK * 2;
constexpr int STAGES = 3;
constexpr int SLOTS = 4;           // accumulators in TMEM, 128 columns each
constexpr int PHASES = 2;
constexpr int THREADS = 64 + 256;  // TMA warp, MMA warp, eight epilogue warps
constexpr int EPI_THREADS = 256;
constexpr int BAR_BYTES = (2 * STAGES + 2 * SLOTS + 1) * 8 + 16;
// D F32, A and B BF16, both K-major, M = N = 128
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(TM >> 3) << 17) | (uint32_t(TM >> 4) << 24);

// K-major operand tile with 64-byte swizzle: rows of 64 bytes, 8-row groups 512
// bytes apart
__device__ __forceinline__ uint64_t sdesc64(uint32_t saddr) {
  uint64_t d = 0;
  d |= uint64_t((saddr & 0x3FFFFu) >> 4);
  d |= uint64_t(1) << 16;
  d |= uint64_t(512 >> 4) << 32;
  d |= uint64_t(1) << 46;
  d |= uint64_t(4) << 61;
  return d;
}

// slices p of X whose products with slice t - p of Y make up level t
__host__ __device__ constexpr int first_p(int t, int ny) { return t - ny > 1 ? t - ny : 1; }
__host__ __device__ constexpr int last_p(int t, int nx) { return t - 1 < nx ? t - 1 : nx; }

// a phase: its levels, and the slices of X and Y that they use
struct Phase {
  int t0, t1, p0, p1, q0, q1;
};
__host__ __device__ inline Phase phase_of(int f, int nx, int ny) {
  Phase h;
  h.t0 = 2 + SLOTS * f;
  h.t1 = f == 0 ? 1 + SLOTS : 1 + SG_LEVELS;
  h.p0 = first_p(h.t0, ny);
  h.p1 = last_p(h.t1, nx);
  h.q0 = first_p(h.t0, nx);
  h.q1 = last_p(h.t1, ny);
  return h;
}

// most products of one level, and from it the k-blocks of an exact sum
__host__ __device__ inline int chunk_blocks(int nx, int ny) {
  int pairs = 1;
  for (int t = 2; t < 2 + SG_LEVELS; ++t) {
    const int np = last_p(t, nx) - first_p(t, ny) + 1;
    if (np > pairs) pairs = np;
  }
  return ((1 << 24) - 1) / (63 * 63 * pairs * TK);
}

__host__ __device__ inline int stage_tiles(int nx, int ny) {
  int most = 0;
  for (int f = 0; f < PHASES; ++f) {
    const Phase h = phase_of(f, nx, ny);
    const int n = (h.p1 - h.p0 + 1) + (h.q1 - h.q0 + 1);
    if (n > most) most = n;
  }
  return most;
}
int smem_bytes(int nx, int ny) { return 1024 + STAGES * stage_tiles(nx, ny) * TILE + BAR_BYTES; }

// Bound by operand ingest and the MMAs alike (50 bytes per clock at the full
// rate).  Both residual products of 700 submatrices of 504-704 dims: 14.7 ->
// 9.4 ms; of 64 of ~1470 dims: 8.3 -> 7.2 ms.  128 x 64 tiles, which hold all
// seven levels at once, took 15.6 and 11.9 ms: an MMA of 64 columns takes as long
// as one of 128.
__global__ void __launch_bounds__(THREADS, 1) k_slice_gemm(const __grid_constant__ SliceGemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int sbytes = stage_tiles(p.nx, p.ny) * TILE;
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles + STAGES * sbytes);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + SLOTS;
  uint64_t* drain = tempty + SLOTS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < SLOTS; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], EPI_THREADS); }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(uint32_t(SLOTS * TM)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const long long limit = p.timeout_cycles;
  const int chunk = chunk_blocks(p.nx, p.ny);

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    int stage = 0;
    uint32_t phase = 0, issued = 0, issued_phase = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
      const int4 item = p.items[it];
      const int nk = p.ld[item.x] / TK;
      const int bucket = item.w & 0xFF, slot = item.w >> 8;
      for (int k0 = 0; k0 < nk && ok; k0 += chunk)
        for (int f = 0; f < PHASES && ok; ++f) {
          const Phase h = phase_of(f, p.nx, p.ny);
          const uint32_t bytes = uint32_t(((h.p1 - h.p0 + 1) + (h.q1 - h.q0 + 1)) * TILE);
          if (h.p1 < h.p0 || h.q1 < h.q0) continue;
          for (int kb = k0; kb < min(nk, k0 + chunk); ++kb) {
            if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, limit)) { ok = false; break; }
            uint8_t* st = tiles + stage * sbytes;
            mbar_expect_tx(&full[stage], bytes);
            for (int a = h.p0; a <= h.p1; ++a, st += TILE)
              tma_load_3d(st, p.maps + p.a_set[a - 1] * p.nbucket + bucket, &full[stage], kb * TK, item.y * TM, slot);
            for (int b = h.q0; b <= h.q1; ++b, st += TILE)
              tma_load_3d(st, p.maps + p.b_set[b - 1] * p.nbucket + bucket, &full[stage], kb * TK, item.z * TM, slot);
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
    int stage = 0;
    uint32_t phase = 0, tphase = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
      const int4 item = p.items[it];
      const int nk = p.ld[item.x] / TK;
      for (int k0 = 0; k0 < nk && ok; k0 += chunk)
        for (int f = 0; f < PHASES && ok; ++f) {
          const Phase h = phase_of(f, p.nx, p.ny);
          if (h.p1 < h.p0 || h.q1 < h.q0) continue;
          const int k1 = min(nk, k0 + chunk);
          for (int kb = k0; kb < k1 && ok; ++kb) {
            if (!mbar_wait(&full[stage], phase, abort_flag, limit)) { ok = false; break; }
            tc_fence_after();
            const uint32_t sa = smem_u32(tiles + stage * sbytes), sb = sa + uint32_t((h.p1 - h.p0 + 1) * TILE);
            for (int l = 0; l < SLOTS; ++l) {
              const int t = h.t0 + l;
              if (kb == k0) {  // the accumulator has been drained
                if (!mbar_wait(&tempty[l], tphase ^ 1u, abort_flag, limit)) { ok = false; break; }
                tc_fence_after();
              }
              const uint32_t d = tmem_base + uint32_t(l * TM);
              bool more = kb > k0;
              if (t <= h.t1)
                for (int q = first_p(t, p.ny); q <= last_p(t, p.nx); ++q) {
                  const uint64_t ad = sdesc64(sa + uint32_t((q - h.p0) * TILE));
                  const uint64_t bd = sdesc64(sb + uint32_t((t - q - h.q0) * TILE));
#pragma unroll
                  for (int k = 0; k < TK / 16; ++k)
                    umma_bf16(d, ad + uint64_t(2 * k), bd + uint64_t(2 * k), IDESC, (more || k > 0) ? 1u : 0u);
                  more = true;
                }
              if (kb == k1 - 1) umma_commit(&tfull[l]);
            }
            if (!ok) break;
            umma_commit(&empty[stage]);
            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
          }
          tphase ^= 1u;
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
  } else if (warp >= 2) {
    // ---------------- epilogue ----------------
    const int quarter = warp & 3, half = (warp - 2) >> 2;  // TMEM lanes 32 quarter .., columns 64 half ..
    const uint32_t tlane = tmem_base + (uint32_t(quarter * 32) << 16) + uint32_t(half * 64);
    uint32_t tphase = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
      const int4 item = p.items[it];
      const int s = item.x, ld = p.ld[s];
      const int nk = ld / TK;
      const int rg = item.y * TM + quarter * 32 + lane, cg = item.z * TM + half * 64;
      // a warp whose rows or columns lie beyond ld has nothing to add up
      const bool work = item.y * TM + quarter * 32 < ld && cg < ld;
      long long v[64];
#pragma unroll
      for (int q = 0; q < 64; ++q) v[q] = 0;
      for (int k0 = 0; k0 < nk && ok; k0 += chunk)
        for (int f = 0; f < PHASES && ok; ++f) {
          const Phase h = phase_of(f, p.nx, p.ny);
          if (h.p1 < h.p0 || h.q1 < h.q0) continue;
#pragma unroll 1
          for (int l = 0; l < SLOTS; ++l) {
            // a warp leaves the loop together: every lane sees the same outcome
            ok = __all_sync(0xffffffffu, mbar_wait(&tfull[l], tphase, abort_flag, limit));
            if (!ok) break;
            tc_fence_after();
            const int t = h.t0 + l;
            const bool any = work && t <= h.t1 && first_p(t, p.ny) <= last_p(t, p.nx);
            const int shift = 6 * (SG_LEVELS + 1 - t);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              float a[16];
              if (any) {
                tmem_ld16(tlane + uint32_t(l * TM + c * 16), a);
                tmem_wait16(a);
              }
              if (c == 3) {
                tc_fence_before();
                mbar_arrive(&tempty[l]);
              }
              if (any) {
#pragma unroll
                for (int q = 0; q < 16; ++q) v[c * 16 + q] += static_cast<long long>(__float2int_rn(a[q])) << shift;
              }
            }
          }
          tphase ^= 1u;
        }
      if (!ok) {
        if (lane == 0) atomicOr(p.flags, FLAG_TIMEOUT);
        *abort_flag = 1;
        break;
      }
      if (!work) continue;
      long long* out = p.Z + p.off[s] + int64_t(rg) * ld + cg;
#pragma unroll
      for (int q = 0; q < 64; q += 4)
        asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(out + q), "l"(v[q]), "l"(v[q + 1]),
                     "l"(v[q + 2]), "l"(v[q + 3])
                     : "memory");
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(uint32_t(SLOTS * TM)));
  }
}

}  // namespace

bool slice_gemm_fits(int nx, int ny) {
  return nx >= 1 && ny >= 1 && nx <= SG_SLICES && ny <= SG_SLICES && smem_bytes(nx, ny) <= 227 * 1024;
}

int slice_gemm_products(int nx, int ny) {
  int np = 0;
  for (int t = 2; t < 2 + SG_LEVELS; ++t) np += std::max(0, last_p(t, nx) - first_p(t, ny) + 1);
  return np;
}

cudaError_t launch_slice_gemm(const SliceGemmParams& p, int nsm, cudaStream_t st) {
  if (p.nitems <= 0) return cudaSuccess;
  if (!slice_gemm_fits(p.nx, p.ny)) return cudaErrorInvalidValue;
  const int smem = smem_bytes(p.nx, p.ny);
  cudaError_t e = cudaFuncSetAttribute(k_slice_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  k_slice_gemm<<<std::min(p.nitems, nsm), THREADS, smem, st>>>(p);
  count_launch();
  return cudaGetLastError();
}

}  // namespace submat
