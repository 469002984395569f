// Products of sweeps over few rows:  C[M,N] = A[M,K] * W[N,K]^T, bf16 operands (A optionally a two-term pair), fp32 accumulation, one
// 128 x BN tile (or K slice of one) per CTA.
//
// Why: with a few hundred rows a sweep is a chain of short kernels.  A product's length is what one SM can take in (about 100 GB/s
// through TMA) plus the fixed cost of a kernel (1.3 us from the last CTA's end to the next kernel's first load, 1 us for that load), so
//   * tiles are narrow (64 or 32 columns): a 64-wide k slab costs 24 or 20 KB instead of 32 KB, and more SMs share the weights;
//   * the first weight slabs are requested, and the others prefetched into L2 (they mostly come from memory), before the previous
//     kernel has ended; in a ring of 144 or 120 KB (96 KB leave room for the next kernel's CTAs, but two slabs of a pair in flight
//     do not cover the latency: two-term sweep of 256 rows, width 1024: 525 us with 2 slabs, 414 with 3, 418 with 4);
//   * a weight slab is fetched once for both terms of a pair;
//   * eight warps share the epilogue (bulk stores, as in epilogue.cuh).
// 256 rows, width 1024, eight layers (128 x 128 tiles of gemm_tc.cuh -> these): single-term sweep 387 -> 333 us, two-term 523 -> 413;
// 1053 rows, width 256, two layers: 144 -> 76 and 164 -> 84 us.
// A split of K over the CTAs of a cluster with an exchange through distributed shared memory was slower (429 and 555 us): two CTAs
// take 1.8 us for the exchange and save 1.2 us of loads, eight take 2.7 us.
// Every wait is bounded as in gemm_tc.cuh.
#pragma once
#include <type_traits>

#include "gemm_tc.cuh"

namespace few {

using namespace tc;

constexpr int THREADS = 256, BOX = 4096, STAGES = 6, STAGES_SPLIT = 3;

template <int BN>
struct Cfg {
  static constexpr int CH = BN / 2;  // columns of a warp (two warps per tensor-memory quadrant)
  static constexpr int A_BYTES = BM * BK * 2, W_BYTES = BN * BK * 2;
  static constexpr int BARS = BN * 4, NBARS = 2 * STAGES + 1;  // behind the ring and the biases
  static constexpr int MAX_RING = STAGES * (A_BYTES + W_BYTES);
  static constexpr int EXTRA = BARS + NBARS * 8 + 16 + 1024;
};

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 o = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&o);
}
template <int CH>
__device__ __forceinline__ void tmem_chunk(uint32_t taddr, float (&v)[CH]) {
  static_assert(CH == 16 || CH == 32, "columns of a warp");
  if constexpr (CH == 32) {
    tmem_ld_32x32b_x32(taddr, v);
  } else {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
  }
}

// ---- epilogues.  A lane owns row `row` and CH columns from col0 on.  load() requests what the result is combined with (once the
// previous kernel has completed, while the products run); finish() gets the sums without bias and the operand ring, which is free.
struct Warp {
  int quad, half, lane;  // rows 32 quad .., columns CH half .. of the tile
};

template <int ACT>
struct Store {  // bf16(act(x)), and the second term of the pair where map_lo is set; N % 64 == 0
  static constexpr int kOld = 1;
  const CUtensorMap *map, *map_lo;
  __device__ __forceinline__ void prefetch() const {
    prefetch_map(map);
    if (map_lo != nullptr) prefetch_map(map_lo);
  }
  template <int CH>
  __device__ __forceinline__ void load(int, int, bool, float (&)[kOld]) const {}
  template <int CH>
  __device__ __forceinline__ void finish(int row0, int col0, bool, float (&v)[CH], float (&)[kOld], const float* bias, uint8_t* ring, int, Warp w) const {
    static_assert(CH == 32, "two warps fill a box of 64 columns");
    uint8_t *hi = ring + w.quad * 2 * BOX, *lo = hi + BOX;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      uint32_t h[4], l[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int j = 8 * k + 2 * i;
        float2 x = fadd2(make_float2(v[j], v[j + 1]), *reinterpret_cast<const float2*>(bias + j));
        if (ACT == ACT_GELU) x = gelu_erf_fast2(x);
        h[i] = pack_bf16(x.x, x.y);
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h[i]));
        l[i] = pack_bf16(x.x - f.x, x.y - f.y);
      }
      const uint32_t at = swz128(w.lane, 4 * w.half + k);
      *reinterpret_cast<uint4*>(hi + at) = make_uint4(h[0], h[1], h[2], h[3]);
      if (map_lo != nullptr) *reinterpret_cast<uint4*>(lo + at) = make_uint4(l[0], l[1], l[2], l[3]);
    }
    fence_proxy_async_smem();
    named_bar_sync(1 + w.quad, 64);
    if (w.half == 0 && w.lane == 0) {
      tma_store_2d(map, col0, row0, smem_u32(hi));
      if (map_lo != nullptr) tma_store_2d(map_lo, col0, row0, smem_u32(lo));
      tma_store_commit();
    }
  }
};

struct StoreF32 {  // fp32 sums, without bias (a K slice's go part_rows rows further down per slice)
  static constexpr int kOld = 1;
  const CUtensorMap* map;
  __device__ __forceinline__ void prefetch() const { prefetch_map(map); }
  template <int CH>
  __device__ __forceinline__ void load(int, int, bool, float (&)[kOld]) const {}
  template <int CH>
  __device__ __forceinline__ void finish(int row0, int col0, bool, float (&v)[CH], float (&)[kOld], const float*, uint8_t* ring, int N, Warp w) const {
    static_assert(CH == 32, "a box is 32 columns");
    if (col0 >= N) return;
    uint8_t* box = ring + (w.quad * 2 + w.half) * BOX;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      *reinterpret_cast<float4*>(box + swz128(w.lane, k)) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    fence_proxy_async_smem();
    __syncwarp();
    if (w.lane == 0) {
      tma_store_2d(map, col0, row0, smem_u32(box));
      tma_store_commit();
    }
  }
};

// Algorithm 1's update line, as EpiHeadUpdate does it: columns (2c, 2c + 1) = (mu~_c, alpha~_c).  V values per access (4 or 2), D % V == 0.
template <int V>
struct HeadUpdate {
  using Vec = std::conditional_t<V == 4, float4, float2>;
  static constexpr int kOld = 16;  // eight values of the iterate, eight of the block's input
  const float* v;
  float *u, *maxdiff;
  const int* idx;
  int L, D, reversed;
  __device__ __forceinline__ void prefetch() const {}
  __device__ __forceinline__ int sample(int row) const { return idx ? idx[row / L] : row / L; }
  __device__ __forceinline__ size_t element(int row, int b, bool& upd) const {
    const int l = row % L;
    upd = l < L - 1;  // the last position's head output is unused: that row copies token 0
    return ((size_t)b * L + tok_index(upd ? l + 1 : 0, L, reversed)) * D;
  }
  template <int CH>
  __device__ __forceinline__ void load(int row, int col0, bool ok, float (&old)[kOld]) const {
    static_assert(CH == 16, "eight values per lane");
    if (!ok) return;
    bool upd;
    const size_t e = element(row, sample(row), upd);
#pragma unroll
    for (int j = 0; j < 8; j += V) {
      const int c = col0 / 2 + j;
      if (c < D) {
        const Vec x = __ldcg(reinterpret_cast<const Vec*>(u + e + c)), y = __ldcg(reinterpret_cast<const Vec*>(v + e + c));
#pragma unroll
        for (int i = 0; i < V; ++i) {
          old[j + i] = reinterpret_cast<const float*>(&x)[i];
          old[8 + j + i] = reinterpret_cast<const float*>(&y)[i];
        }
      }
    }
  }
  template <int CH>
  __device__ __forceinline__ void finish(int row0, int col0, bool ok, float (&x)[CH], float (&old)[kOld], const float* bias, uint8_t*, int, Warp w) const {
    float m = 0.f;
    int b = -1;
    if (ok) {
      bool upd;
      b = sample(row0 + w.lane);
      const size_t e = element(row0 + w.lane, b, upd);
#pragma unroll
      for (int j = 0; j < 8; j += V) {
        const int c = col0 / 2 + j;
        if (c < D) {
          Vec nw;
#pragma unroll
          for (int i = 0; i < V; ++i) {
            const int k = j + i;
            const float mu = x[2 * k] + bias[2 * k], al = x[2 * k + 1] + bias[2 * k + 1], vv = old[8 + k];
            const float now = upd ? fmaf(vv, expf(al), mu) : vv, df = fabsf(now - old[k]);
            reinterpret_cast<float*>(&nw)[i] = now;
            m = (df > m || df != df) ? df : m;
          }
          *reinterpret_cast<Vec*>(u + e + c) = nw;
        }
      }
    }
    // NaN-propagating maximum; one atomic per warp where all its rows belong to one sample
    const int b0 = __shfl_sync(0xffffffffu, b, 0);
    if (__all_sync(0xffffffffu, b == b0 || b < 0)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float other = __shfl_xor_sync(0xffffffffu, m, o);
        m = (other > m || other != other) ? other : m;
      }
      if (w.lane == 0 && b0 >= 0) atomic_max_nonneg(maxdiff + b0, m);
    } else if (b >= 0) {
      atomic_max_nonneg(maxdiff + b, m);
    }
  }
};

// grid: tiles * ksplit; map_w has a box of BN rows; `bias` may be null
template <int BN, class Epi>
__global__ void __launch_bounds__(THREADS, 2)
gemm_few_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_a_lo,
                const __grid_constant__ CUtensorMap map_w, int M, int N, int K, int split, Epi epi, const float* bias, int* err,
                int ksplit, int part_rows, int ring_bytes) {
  using C = Cfg<BN>;
  constexpr int CH = C::CH;
  extern __shared__ uint8_t smem_few[];
  uint8_t* smem = align1024(smem_few);
  const uint32_t sb = smem_u32(smem), bars = sb + ring_bytes + C::BARS, done = bars + 8u * (2 * STAGES);
  auto full = [&](int s) { return bars + 8u * s; };
  auto empty = [&](int s) { return bars + 8u * (STAGES + s); };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + ring_bytes + C::BARS + C::NBARS * 8);
  float* s_bias = reinterpret_cast<float*>(smem + ring_bytes);

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int slice = blockIdx.x % ksplit, tile = blockIdx.x / ksplit, tiles_n = (N + BN - 1) / BN;
  const int m0 = tile / tiles_n * BM, n0 = tile % tiles_n * BN;
  const int slabs = (K + BK - 1) / BK;
  const SlabRange sr = {slabs * slice / ksplit, slabs * (slice + 1) / ksplit};
  const int n = sr.end - sr.begin;
  const uint32_t w_off = split ? 2u * C::A_BYTES : (uint32_t)C::A_BYTES, stage_bytes = w_off + C::W_BYTES;
  const int nst = ring_bytes / (int)stage_bytes, pre = n < nst ? n : nst;

  if (tid == 0) {
    prefetch_map(&map_w);
    prefetch_map(&map_a);
    if (split) prefetch_map(&map_a_lo);
    for (int i = 0; i < C::NBARS; ++i) mbar_init(bars + 8u * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int s = 0; s < pre; ++s) {  // weights do not depend on the previous kernel
      mbar_arrive_expect_tx(full(s), stage_bytes);
      tma_load_2d(sb + s * stage_bytes + w_off, &map_w, (sr.begin + s) * BK, n0, full(s));
    }
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "n"(BN) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 96) {
    if (m0 == 0)
      for (int s = sr.begin + pre; s < sr.end; ++s) prefetch_tile(&map_w, s * BK, n0);
    epi.prefetch();
  }
  if (tid >= 128 && tid < 128 + BN) {
    const int col = n0 + tid - 128;
    s_bias[tid - 128] = bias != nullptr && col < N ? __ldg(bias + col) : 0.f;
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = *tmem_slot;
  // Only now: the next kernel's CTAs may become resident beside this one's and must not take the tensor memory it still needs.
  pdl_launch_dependents();
  pdl_wait();  // everything above overlaps the previous kernel

  if (warp == 0) {
    if (lane == 0) {
      for (int s = 0; s < pre; ++s) {
        tma_load_2d(sb + s * stage_bytes, &map_a, (sr.begin + s) * BK, m0, full(s));
        if (split) tma_load_2d(sb + s * stage_bytes + C::A_BYTES, &map_a_lo, (sr.begin + s) * BK, m0, full(s));
      }
      int s = 0;
      uint32_t phase = 0;
      for (int kb = pre; kb < n; ++kb) {
        if (!mbar_wait(empty(s), phase, err, TFERR_WAIT_EMPTY)) break;
        mbar_arrive_expect_tx(full(s), stage_bytes);
        tma_load_2d(sb + s * stage_bytes, &map_a, (sr.begin + kb) * BK, m0, full(s));
        if (split) tma_load_2d(sb + s * stage_bytes + C::A_BYTES, &map_a_lo, (sr.begin + kb) * BK, m0, full(s));
        tma_load_2d(sb + s * stage_bytes + w_off, &map_w, (sr.begin + kb) * BK, n0, full(s));
        if (++s == nst) { s = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && *reinterpret_cast<volatile int*>(err) == 0) {  // after an earlier failure no product is issued
      constexpr uint32_t idesc = make_idesc(BN);
      int s = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int kb = 0; kb < n && ok; ++kb) {
        if (!mbar_wait(full(s), phase, err, TFERR_WAIT_FULL)) { ok = false; break; }
        tcgen05_fence_after();
        const uint32_t sa = sb + s * stage_bytes;
        const uint64_t ad = make_smem_desc(sa), wd = make_smem_desc(sa + w_off);
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; ++k) umma_f16(tmem, ad + 2u * k, wd + 2u * k, idesc, (kb | k) != 0);
        if (split) {  // the low halves against the same weight slab
          const uint64_t ld = make_smem_desc(sa + C::A_BYTES);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) umma_f16(tmem, ld + 2u * k, wd + 2u * k, idesc, 1u);
        }
        umma_commit(empty(s));
        if (++s == nst) { s = 0; phase ^= 1u; }
      }
      if (ok) umma_commit(done);
    }
  }
  __syncwarp();
  const Warp w = {warp & 3, warp >> 2, lane};
  const int row0 = m0 + w.quad * 32, col0 = n0 + w.half * CH;
  const bool row_ok = row0 + lane < M;
  float old[Epi::kOld];
  epi.template load<CH>(row0 + lane, col0, row_ok, old);
  bool ok = mbar_wait(done, 0u, err, TFERR_WAIT_TMEM_FULL);
  ok = __syncthreads_and(ok);  // all or none: two warps share a box
  tcgen05_fence_after();
  if (ok && row0 < M) {
    float v[CH];
    tmem_chunk<CH>(tmem + ((uint32_t)(w.quad * 32) << 16) + (uint32_t)(w.half * CH), v);
    epi.template finish<CH>(row0 + slice * part_rows, col0, row_ok, v, old, s_bias + w.half * CH, smem, N, w);
    if (lane == 0) tma_store_wait_all();
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == 2) {
    if (*reinterpret_cast<volatile int*>(err) != 0) {  // a wait gave up: let copies and products in flight drain
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(BN) : "memory");
  }
}

}  // namespace few
