// fp32 engine: matrix product and causal attention of a sweep, and the sequentially decoded block of models whose
// weights fit the shared memory of one thread-block cluster.  All arithmetic is fp32 FMA (the engine's contract is
// fp32 operands, sums and results), so the tensor cores have no part in it; at the sizes this engine serves (a few
// hundred to a few thousand rows, widths of a few hundred) every kernel is bound by latency: how many SMs share the work
// and how many dependent round trips a kernel makes.
#pragma once
#include "common.cuh"
#include "gemm_tc.cuh"

namespace f32 {

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool pred) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
  const int n = pred ? 16 : 0;  // 0 source bytes: zero fill
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// ---------------------------------------------------------------------------------------------
// C[M,N] = A[M,K] W[N,K]^T, K % 4 == 0.  BM x BN tile per CTA of (BM / TM) (BN / 4) KS threads: KS groups of threads share
// a tile and take turns along K (their sums are added in group order at the end), a thread owns TM x 4 outputs and reads
// both operands four k at a time.  KS is the same for every tile, so that an output's order of summation does not depend on
// the number of rows (two groups for the widest tile: 4096 rows of width 128 forward 502 us instead of 512, 20 000 rows of an MLP
// flow of width 512 1.60 ms instead of 1.55; 64 x 32 and 32 x 64 tiles with four: 549 us).  32-wide k slabs arrive through a deep ring of cp.async stages (the first weight
// slabs are requested before the wait on the previous kernel), so that a short K is one memory latency, not one per slab.  Row n of W sits at slot (n % 4) (BN / 4) + n / 4 of a slab, so
// that the column quads of a quarter warp lie in different banks.
// Why: the 64 x 64 tile this replaces left 8 to 24 CTAs for 256 rows and two barriers per 16 k; 256 x 128 x 512 took
// 48 us.
// ---------------------------------------------------------------------------------------------
constexpr int GK = 32, GPITCH = GK + 4;
constexpr int KS = 4;
template <int BM, int BN, int TM>
struct GemmCfg {
  static constexpr int GSTAGES = BM + BN > 64 ? 4 : 8;
  static constexpr int GROUP = (BM / TM) * (BN / 4), THREADS = GROUP * KS;
  static constexpr int STAGE = (BM + BN) * GPITCH;
  static constexpr int SMEM = GSTAGES * STAGE * (int)sizeof(float);
  static_assert(GK / 4 % KS == 0, "a slab's k quads are dealt to the groups evenly");
  static_assert((KS - 1) * GROUP * TM * 4 <= GSTAGES * STAGE, "the groups' sums must fit the ring");
};

template <int BM, int BN, int TM, class Epi>
__global__ void __launch_bounds__(GemmCfg<BM, BN, TM>::THREADS)
gemm_kernel(const float* __restrict__ A, const float* __restrict__ W, int M, int N, int K, Epi epi) {
  using C = GemmCfg<BM, BN, TM>;
  constexpr int GSTAGES = C::GSTAGES;
  extern __shared__ __align__(16) float s_ring[];
  pdl_launch_dependents();
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN, slabs = (K + GK - 1) / GK;
  const int grp = threadIdx.x / C::GROUP, gt = threadIdx.x % C::GROUP, tx = gt % (BN / 4), ty = gt / (BN / 4);
  auto load_w = [&](int slab) {
    float* dst = s_ring + (slab % GSTAGES) * C::STAGE + BM * GPITCH;
    for (int i = threadIdx.x; i < BN * (GK / 4); i += C::THREADS) {
      const int n = i / (GK / 4), q = i % (GK / 4), k = slab * GK + 4 * q;
      const bool ok = n0 + n < N && k < K;
      cp_async16(dst + ((n & 3) * (BN / 4) + (n >> 2)) * GPITCH + 4 * q, ok ? W + (size_t)(n0 + n) * K + k : W, ok);
    }
  };
  auto load_a = [&](int slab) {
    float* dst = s_ring + (slab % GSTAGES) * C::STAGE;
    for (int i = threadIdx.x; i < BM * (GK / 4); i += C::THREADS) {
      const int r = i / (GK / 4), q = i % (GK / 4), k = slab * GK + 4 * q;
      const bool ok = m0 + r < M && k < K;
      cp_async16(dst + r * GPITCH + 4 * q, ok ? A + (size_t)(m0 + r) * K + k : A, ok);
    }
  };
#pragma unroll
  for (int s = 0; s < GSTAGES - 1; ++s)
    if (s < slabs) load_w(s);
  pdl_wait();
#pragma unroll
  for (int s = 0; s < GSTAGES - 1; ++s) {
    if (s < slabs) load_a(s);
    cp_async_commit();  // the first group also holds the weights requested above
  }
  float acc[TM][4];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  for (int s = 0; s < slabs; ++s) {
    cp_async_wait<GSTAGES - 2>();
    __syncthreads();  // slab s has arrived for every thread, and nobody reads the stage overwritten next any more
    if (s + GSTAGES - 1 < slabs) { load_w(s + GSTAGES - 1); load_a(s + GSTAGES - 1); }
    cp_async_commit();
    const float* sa = s_ring + (s % GSTAGES) * C::STAGE + ty * TM * GPITCH;
    const float* sb = s_ring + (s % GSTAGES) * C::STAGE + BM * GPITCH + tx * GPITCH;
#pragma unroll
    for (int q = 0; q < GK / 4 / KS; ++q) {
      const int k4 = (q * KS + grp) * 4;
      float4 a[TM], b[4];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const float4*>(sa + i * GPITCH + k4);
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(sb + j * (BN / 4) * GPITCH + k4);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
          acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
          acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
          acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
        }
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  if (grp > 0) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
      *reinterpret_cast<float4*>(s_ring + (((grp - 1) * TM + i) * C::GROUP + gt) * 4) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  }
  __syncthreads();
  if (grp > 0) return;
#pragma unroll
  for (int g = 1; g < KS; ++g)
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const float4 o = *reinterpret_cast<const float4*>(s_ring + (((g - 1) * TM + i) * C::GROUP + gt) * 4);
      acc[i][0] += o.x; acc[i][1] += o.y; acc[i][2] += o.z; acc[i][3] += o.w;
    }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int row = m0 + ty * TM + i, col0 = n0 + tx * 4;
    if (row < M && col0 < N) epi.template apply<4>(row, col0, acc[i], N - col0 < 4 ? N - col0 : 4);
  }
}

// ---------------------------------------------------------------------------------------------
// Causal attention of a sweep.  One CTA of 8 / QW warps per (slot, head, 8 queries); keys and values pass through shared
// memory in tiles of 64, a warp handles its QW queries against a tile: a lane scores two keys (q comes with broadcast
// reads), the running maximum and sum are warp shuffles, then a lane accumulates channels lane, lane + 32, ... with the
// probabilities read back from shared memory.  qkv rows are [q | k | v], 3d wide; HD % 4 == 0, HD <= 128.
// QW = 1 halves the chain of a CTA, QW = 2 has fewer idle warps per loaded tile (64 tokens of width 128: sweep of 4 samples 76.8 us with
// two queries per warp, 70.9 with one; of 64 samples 251 and 258).
// The warp-per-query kernel it replaces read every key row from global memory one float at a time (19 us at 4 x 64 tokens).
// ---------------------------------------------------------------------------------------------
constexpr int AT_KEYS = 64, AT_Q = 8;
__host__ __device__ constexpr int attention_smem_floats(int hd) { return 2 * AT_KEYS * (hd + 4) + AT_Q * hd + AT_Q * AT_KEYS; }

template <int AT_QW>
__global__ void __launch_bounds__(32 * AT_Q / AT_QW)
attention_kernel(const float* __restrict__ qkv, float* __restrict__ out, int L, int d, int hd, float scale) {
  constexpr int THREADS = 32 * AT_Q / AT_QW;
  extern __shared__ __align__(16) float s_at[];
  pdl_launch_dependents();
  pdl_wait();
  const int pitch = hd + 4, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* sk = s_at;
  float* sv = sk + AT_KEYS * pitch;
  float* sq = sv + AT_KEYS * pitch;
  float* sp = sq + AT_Q * hd;
  const int q0 = blockIdx.x * AT_Q, head = blockIdx.y, slot = blockIdx.z, hq = hd >> 2;
  const size_t ld = 3 * (size_t)d;
  const float* base = qkv + (size_t)slot * L * ld + (size_t)head * hd;
  const int last_q = q0 + AT_Q - 1 < L - 1 ? q0 + AT_Q - 1 : L - 1;
  for (int i = threadIdx.x; i < AT_Q * hq; i += THREADS) {
    const int r = i / hq, c = i % hq, pos = q0 + r < L ? q0 + r : L - 1;
    float4 x = __ldg(reinterpret_cast<const float4*>(base + (size_t)pos * ld) + c);
    x.x *= scale; x.y *= scale; x.z *= scale; x.w *= scale;
    *reinterpret_cast<float4*>(sq + r * hd + 4 * c) = x;
  }
  float m[AT_QW], l[AT_QW], o[AT_QW][4];
#pragma unroll
  for (int r = 0; r < AT_QW; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) o[r][c] = 0.f;
  }
  for (int j0 = 0; j0 <= last_q; j0 += AT_KEYS) {
    __syncthreads();  // the previous tile has been consumed
    for (int i = threadIdx.x; i < AT_KEYS * hq; i += THREADS) {
      const int r = i / hq, c = i % hq;
      const bool ok = j0 + r <= last_q;
      const float* row = base + (size_t)(ok ? j0 + r : 0) * ld + 4 * c;
      cp_async16(sk + r * pitch + 4 * c, row + d, ok);
      cp_async16(sv + r * pitch + 4 * c, row + 2 * d, ok);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
#pragma unroll
    for (int r = 0; r < AT_QW; ++r) {
      const int qr = w * AT_QW + r, pos = q0 + qr;
      if (j0 > pos) continue;  // uniform across the warp
      float s0 = 0.f, s1 = 0.f;
      for (int c = 0; c < hq; ++c) {
        const float4 qv = *reinterpret_cast<const float4*>(sq + qr * hd + 4 * c);
        const float4 k0 = *reinterpret_cast<const float4*>(sk + lane * pitch + 4 * c);
        const float4 k1 = *reinterpret_cast<const float4*>(sk + (lane + 32) * pitch + 4 * c);
        s0 = fmaf(qv.x, k0.x, s0); s0 = fmaf(qv.y, k0.y, s0); s0 = fmaf(qv.z, k0.z, s0); s0 = fmaf(qv.w, k0.w, s0);
        s1 = fmaf(qv.x, k1.x, s1); s1 = fmaf(qv.y, k1.y, s1); s1 = fmaf(qv.z, k1.z, s1); s1 = fmaf(qv.w, k1.w, s1);
      }
      if (j0 + lane > pos) s0 = -INFINITY;
      if (j0 + lane + 32 > pos) s1 = -INFINITY;
      const float mn = fmaxf(m[r], warp_max(fmaxf(s0, s1)));  // finite: key j0 is visible
      const float corr = expf(m[r] - mn), p0 = expf(s0 - mn), p1 = expf(s1 - mn);
      m[r] = mn;
      l[r] = l[r] * corr + warp_sum(p0 + p1);
      float* p = sp + qr * AT_KEYS;
      __syncwarp();
      p[lane] = p0;
      p[lane + 32] = p1;
      __syncwarp();
      const int nk = pos - j0 + 1 < AT_KEYS ? pos - j0 + 1 : AT_KEYS;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int ch = lane + 32 * c;
        if (ch < hd) {
          float a0 = o[r][c] * corr, a1 = 0.f, a2 = 0.f, a3 = 0.f;
          int j = 0;
          for (; j + 4 <= nk; j += 4) {
            const float4 pj = *reinterpret_cast<const float4*>(p + j);
            a0 = fmaf(pj.x, sv[j * pitch + ch], a0);
            a1 = fmaf(pj.y, sv[(j + 1) * pitch + ch], a1);
            a2 = fmaf(pj.z, sv[(j + 2) * pitch + ch], a2);
            a3 = fmaf(pj.w, sv[(j + 3) * pitch + ch], a3);
          }
          for (; j < nk; ++j) a0 = fmaf(p[j], sv[j * pitch + ch], a0);
          o[r][c] = (a0 + a1) + (a2 + a3);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < AT_QW; ++r) {
    const int pos = q0 + w * AT_QW + r;
    if (pos >= L) continue;
    const float inv = 1.f / l[r];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (lane + 32 * c < hd) out[((size_t)slot * L + pos) * d + (size_t)head * hd + lane + 32 * c] = o[r][c] * inv;
  }
}

// ---------------------------------------------------------------------------------------------
// Sequentially decoded block (Eq. 5) in one launch, for models whose block fits the shared memory of a cluster.
//
// A cluster of 8 CTAs decodes S samples, all L - 1 steps of them.  Its shared memory holds the block's weights once (cut
// by attention heads and by hidden units of the MLP, as evenly in bytes as whole heads allow), so a step reads no weight
// from L2.  CTA r computes q, k, v and the attention of its heads and the product of their output with its columns of
// W_o; then the MLP of its hidden units; both leave a partial sum of the whole residual row, which it writes into the
// shared memory of all eight CTAs.  Two exchanges per layer are all the communication of a step: every CTA adds the partial
// rows itself (in CTA order), and LayerNorms, head, update and embedding are done by every CTA for itself.  Rows travel as
// st.async writes that complete on the receiver's mbarrier: a cluster barrier would also wait for the stores of keys,
// values and tokens to global memory (2.0-2.7k cycles per exchange).  The rows of an MLP exchange may only be overwritten once
// their reader is done with them, so CTAs without heads, which send no attention rows, arrive on that barrier instead.
// Products: eight lanes share an output pair (16-byte reads along K, three shuffles), so an output is finished where it is
// computed and its consumer is one barrier away.  Keys and values of the earlier tokens are requested before q is computed.
// Bound: the dependent chain of a step (six barriers and two cluster exchanges per layer), not bytes or FLOPs.
// 64 tokens, width 128, two layers, batch 4: 12.5 ms as 1070 launches of generic kernels (12 us each).
//
// Image of a CTA (SeqPlan::off[r], floats; copied to shared memory once): per layer  W_qkv [nq][d] (rows q | k | v of each
// of its heads), b_qkv [nq], W_o [d][nown hd], W_1 [nu][d], b_1 [nu], W_2 [d][nu], ln1_g ln1_b b_o ln2_g ln2_b b_2 [d each];
// then lnf_g lnf_b [d each], b_in [d];  then the tail part  W_out [No][d], b_out [No], W_in [d][Dp]
// (No = 2 D rounded up to 4, Dp = D rounded up to 4; zero padded), which stays in global memory where it does not fit.
// ---------------------------------------------------------------------------------------------
constexpr int SC = 8, ST = 512, SW = ST / 32;  // CTAs per cluster, threads and warps per CTA
constexpr int AU = 8;                          // parts into which the attention of a CTA's heads is cut for one sample, at least
struct SeqPlan {
  int n_layers = 0, heads = 0, hd = 0, d = 0, D = 0, L = 0, owners = 0;  // owners = CTAs that hold heads
  int off[SC + 1] = {0}, nown[SC] = {0}, nu[SC] = {0};
  __host__ __device__ static int pad4(int x) { return (x + 3) & ~3; }
  __host__ __device__ int layer_floats(int r) const {
    const int nq = 3 * hd * nown[r];
    return d * nq + nq + nown[r] * hd * d + 2 * d * nu[r] + nu[r] + 6 * d;
  }
  __host__ __device__ int fixed_floats(int r) const { return n_layers * layer_floats(r) + 3 * d; }
  // of the tail part: nothing, head matrix and bias, all
  __host__ __device__ int tail_floats(int level) const {
    return (level > 0 ? d * pad4(2 * D) + pad4(2 * D) : 0) + (level > 1 ? pad4(D) * d : 0);
  }
  __host__ __device__ int recv_floats(int S) const { return (owners + SC) * S * d; }
  // shared memory besides the image, S samples: receive buffers, h, xn, q k v, attention output, hidden units, token,
  // attention partials of the warps, v and position embedding of the next token (two each)
  __host__ __device__ int work_floats(int S) const {
    int nq = 0, nx = 0, no = 0;
    for (int r = 0; r < SC; ++r) {
      if (3 * hd * nown[r] > nq) nq = 3 * hd * nown[r];
      if (nu[r] > nx) nx = nu[r];
      if (nown[r] > no) no = nown[r];
    }
    return recv_floats(S) + 2 * S * d + S * nq + S * no * hd + S * nx + S * pad4(D) + S * (no > AU ? no : AU) * (hd + 4) +
           2 * S * pad4(D) + 2 * d;
  }
};

// Outputs n of W [N][K] times x [S][ldx], N even, K % 4 == 0, two consecutive ones per group of eight lanes; emit(n, acc0, acc1,
// lane of the group) is called by all lanes of the group with the finished sums of outputs n and n + 1 (every sample).
template <int S, class Emit>
__device__ __forceinline__ void products(const float* __restrict__ W, int N, int K, const float* __restrict__ x, int ldx, Emit emit) {
  const int sub = threadIdx.x & 7, kq = K >> 2;
  for (int n0 = 0; n0 < N; n0 += ST / 4) {  // the same trip count for every lane
    const int n = n0 + 2 * (threadIdx.x >> 3);
    if (n0 + 8 * (int)(threadIdx.x >> 5) >= N) break;  // none of the warp's eight outputs exists
    float a0[S], a1[S];
#pragma unroll
    for (int s = 0; s < S; ++s) a0[s] = a1[s] = 0.f;
    if (n < N) {
      const float4* w0 = reinterpret_cast<const float4*>(W + n * K);
      const float4* w1 = w0 + kq;
#pragma unroll 4
      for (int q = sub; q < kq; q += 8) {
        const float4 u0 = w0[q], u1 = w1[q];
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const float4 xv = *reinterpret_cast<const float4*>(x + s * ldx + 4 * q);
          a0[s] = fmaf(u0.x, xv.x, fmaf(u0.y, xv.y, fmaf(u0.z, xv.z, fmaf(u0.w, xv.w, a0[s]))));
          a1[s] = fmaf(u1.x, xv.x, fmaf(u1.y, xv.y, fmaf(u1.z, xv.z, fmaf(u1.w, xv.w, a1[s]))));
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
      for (int s = 0; s < S; ++s) {
        a0[s] += __shfl_xor_sync(0xffffffffu, a0[s], o);
        a1[s] += __shfl_xor_sync(0xffffffffu, a1[s], o);
      }
    if (n < N) emit(n, a0, a1, sub);
    __syncwarp();
  }
}
// n / div for n < 2^16 by a multiplication (an integer division is a chain of about 100 cycles)
struct FastDiv {
  uint32_t m;
  __device__ __forceinline__ explicit FastDiv(int div) : m(div > 1 ? 0xffffffffu / (uint32_t)div + 1u : 0u) {}
  __device__ __forceinline__ int operator()(int n) const { return m ? (int)__umulhi((uint32_t)n, m) : n; }
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(const void* p, int peer) {
  uint32_t dst;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(tc::smem_u32(p)), "r"(peer));
  return dst;
}
// columns n, n + 1 of this CTA's partial row, into the same place of CTA `peer`, completing on that CTA's barrier
__device__ __forceinline__ void push2(float* place, uint64_t* bar, int peer, float x, float y) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(peer_addr(place, peer)),
               "f"(x), "f"(y), "r"(peer_addr(bar, peer))
               : "memory");
}
__device__ __forceinline__ void arrive_at(uint64_t* bar, int peer) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(peer_addr(bar, peer)) : "memory");
}
// one warp: h += bias + the np <= 8 rows of `parts` (stride ps), xn = LayerNorm(h) gamma + beta; lane owns column quads
__device__ __forceinline__ void add_ln_row(float* h, float* xn, const float* parts, int np, int ps, const float* bias,
                                           const float* gamma, const float* beta, int d, float inv_d, int lane) {
  float sum = 0.f;
  for (int c = lane; c < d / 4; c += 32) {
    float4 x = *reinterpret_cast<float4*>(h + 4 * c);
    if (np > 0) {
      float4 a[8];
#pragma unroll
      for (int p = 0; p < 8; ++p)
        if (p < np) a[p] = *reinterpret_cast<const float4*>(parts + p * ps + 4 * c);
      const float4 b = *reinterpret_cast<const float4*>(bias + 4 * c);
      x.x += b.x; x.y += b.y; x.z += b.z; x.w += b.w;
#pragma unroll
      for (int p = 0; p < 8; ++p)
        if (p < np) { x.x += a[p].x; x.y += a[p].y; x.z += a[p].z; x.w += a[p].w; }
      *reinterpret_cast<float4*>(h + 4 * c) = x;
    }
    sum += (x.x + x.y) + (x.z + x.w);
  }
  const float mean = warp_sum(sum) * inv_d;
  float sq = 0.f;
  for (int c = lane; c < d / 4; c += 32) {
    const float4 x = *reinterpret_cast<const float4*>(h + 4 * c);
    const float a0 = x.x - mean, a1 = x.y - mean, a2 = x.z - mean, a3 = x.w - mean;
    sq += (a0 * a0 + a1 * a1) + (a2 * a2 + a3 * a3);
  }
  const float rstd = rsqrtf(warp_sum(sq) * inv_d + 1e-5f);
  for (int c = lane; c < d / 4; c += 32) {
    const float4 x = *reinterpret_cast<const float4*>(h + 4 * c), g = *reinterpret_cast<const float4*>(gamma + 4 * c);
    const float4 b = *reinterpret_cast<const float4*>(beta + 4 * c);
    *reinterpret_cast<float4*>(xn + 4 * c) = make_float4((x.x - mean) * rstd * g.x + b.x, (x.y - mean) * rstd * g.y + b.y,
                                                         (x.z - mean) * rstd * g.z + b.z, (x.w - mean) * rstd * g.w + b.w);
  }
}

template <int S, int TAIL>  // TAIL: 0 = the tail part stays in global memory, 1 = the head matrix is resident, 2 = all of it
__global__ void __launch_bounds__(ST, 1)
seq_cluster_kernel(const __grid_constant__ SeqPlan P, const float* __restrict__ image, const float* __restrict__ v,
                   float* __restrict__ u, const int* __restrict__ labels, const float* __restrict__ pos,
                   const float* __restrict__ cls, float* kcache, float* vcache, int max_batch, int B, int reversed, int* err) {
  extern __shared__ __align__(16) float s_all[];
  __shared__ __align__(8) uint64_t bar_a, bar_m;
  __shared__ int s_failed;
  const int r = (int)cluster_rank(), b0 = (blockIdx.x / SC) * S;
  const int d = P.d, D = P.D, L = P.L, hd = P.hd, nown = P.nown[r], nu = P.nu[r], nq = 3 * hd * nown, No = P.pad4(2 * D), Dp = P.pad4(D);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, layer_floats = P.layer_floats(r), owners = P.owners;
  const float inv_d = 1.f / (float)d;
  const float* gimg = image + P.off[r];
  // the receive buffers come first: peers address them by their own offsets, so these must not depend on the rank
  float* recv_a = s_all;
  float* recv_m = recv_a + owners * S * d;
  float* s_mem = recv_m + SC * S * d;
  // resident image
  const int img = P.fixed_floats(r) + P.tail_floats(TAIL);
  for (int i = threadIdx.x; i < img / 4; i += ST) cp_async16(s_mem + 4 * i, gimg + 4 * i, true);
  cp_async_commit();
  float* w = s_mem + img;
  float* h = w; w += S * d;
  float* xn = w; w += S * d;
  float* qkv = w; w += S * nq;
  float* att = w; w += S * nown * hd;
  float* hid = w; w += S * nu;
  float* tok = w; w += S * Dp;
  float* part = w; w += S * (nown > AU ? nown : AU) * (hd + 4);
  float* vnext = w; w += 2 * S * Dp;
  float* pnext = w;
  const float* fixed = s_mem + P.n_layers * layer_floats;  // lnf_g lnf_b b_in
  const float* w_out = TAIL > 0 ? fixed + 3 * d : gimg + P.fixed_floats(r);
  const float* b_out = w_out + d * No;
  const float* w_in = (TAIL == 1 ? gimg + P.fixed_floats(r) + d * No : b_out) + No;
  auto sample = [&](int s) { return b0 + s < B ? b0 + s : B - 1; };  // samples past the batch repeat the last one, unstored
  auto fetch_next = [&](int l) {  // values of the block's input at token l, position embedding of token l
    for (int i = threadIdx.x; i < S * D; i += ST) {
      const int s = i / D, c = i - s * D;
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(vnext + (l & 1) * S * Dp + s * Dp + c);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(v + ((size_t)sample(s) * L + tok_index(l, L, reversed)) * D + c) : "memory");
    }
    for (int i = threadIdx.x; i < d / 4; i += ST) cp_async16(pnext + (l & 1) * d + 4 * i, pos + (size_t)l * d + 4 * i, true);
    cp_async_commit();
  };
  for (int i = threadIdx.x; i < S * Dp; i += ST) tok[i] = 0.f;
  fetch_next(0);
  cp_async_wait<0>();
  __syncthreads();
  for (int i = threadIdx.x; i < S * D; i += ST) {  // the first token is copied (Eq. 5, first row)
    const int s = i / D, c = i - s * D;
    const float x = vnext[s * Dp + c];
    tok[s * Dp + c] = x;
    if (r == 0 && b0 + s < B) u[((size_t)(b0 + s) * L + tok_index(0, L, reversed)) * D + c] = x;
  }
  const float scale = 1.0f / sqrtf((float)hd);
  // Attention: hd / 4 lanes share a key (a power of two); the keys of a (sample, own head) pair are dealt to wpp units of a
  // warp's work, whatever S, so that a sample's sums do not depend on how many samples share the cluster (as many as S leaves
  // warps for: 1-4 % shorter blocks; 16 units instead of 8: 5-15 % longer ones from two samples on).  Unit i of the S nown wpp units is part i % wpp of pair i / wpp, a warp takes every SW-th.
  const int lpk = hd >> 2, llog = 31 - __clz(lpk), klog = 5 - llog, kpw = 1 << klog;  // kpw keys per warp and round
  const int pairs = S * nown, wpp = nown >= AU || nown == 0 ? 1 : AU / nown, ng = wpp * kpw, sub = lane & (lpk - 1);
  const FastDiv by_nown(nown), by_3hd(3 * hd), by_hd(hd), by_wpp(wpp);
  const size_t layer_cache = (size_t)max_batch * P.heads * L * hd;
  auto cache_row = [&](int layer, int s, int hl) {
    return layer * layer_cache + ((size_t)(sample(s) * P.heads + r + SC * hl) * L) * hd;
  };
  if (threadIdx.x == 0) {
    tc::mbar_init(tc::smem_u32(&bar_a), 1 + SC - owners);
    tc::mbar_init(tc::smem_u32(&bar_m), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_failed = 0;
  }
  // one thread arms the barriers; the warps that read the rows wait (bounded), everybody else at the block barrier
  auto arm = [&](uint64_t* bar, int bytes) {
    if (threadIdx.x == 0) tc::mbar_arrive_expect_tx(tc::smem_u32(bar), (uint32_t)bytes);
  };
  auto arrived = [&](uint64_t* bar, uint32_t parity) {
    if (tc::mbar_wait<true>(tc::smem_u32(bar), parity, err, TFERR_WAIT_FULL)) return true;
    s_failed = 1;
    return false;
  };
  uint32_t parity = 0;
  cluster_sync();  // every CTA of the cluster has started and set up its barriers before anything is written there
  for (int t = 0; t + 1 < L && !s_failed; ++t) {
    // embedding of token t, first LayerNorm
    products<S>(w_in, d, Dp, tok, Dp, [&](int n, const float (&a0)[S], const float (&a1)[S], int g8) {
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (g8 == s) {
          const float2 bp = *reinterpret_cast<const float2*>(pnext + (t & 1) * d + n);
          float e0 = a0[s] + (fixed[2 * d + n] + bp.x), e1 = a1[s] + (fixed[2 * d + n + 1] + bp.y);
          if (cls != nullptr) {
            const float2 cl = __ldg(reinterpret_cast<const float2*>(cls + (size_t)labels[sample(s)] * d + n));
            e0 += cl.x;
            e1 += cl.y;
          }
          *reinterpret_cast<float2*>(h + s * d + n) = make_float2(e0, e1);
        }
    });
    __syncthreads();
    if (warp < S) {
      const float* lv = s_mem + layer_floats - 6 * d;
      add_ln_row(h + warp * d, xn + warp * d, nullptr, 0, 0, nullptr, lv, lv + d, d, inv_d, lane);
    }
    __syncthreads();
    fetch_next(t + 1);
    for (int layer = 0; layer < P.n_layers; ++layer, parity ^= 1u) {
      arm(&bar_a, owners * S * d * (int)sizeof(float));
      arm(&bar_m, SC * S * d * (int)sizeof(float));
      const float* wl = s_mem + layer * layer_floats;
      const float *w_qkv = wl, *b_qkv = w_qkv + d * nq, *w_o = b_qkv + nq, *w_1 = w_o + nown * hd * d, *b_1 = w_1 + d * nu,
                  *w_2 = b_1 + nu, *vec = w_2 + nu * d;
      if (nown > 0) {
        // this lane's first key and value row of the warp's first unit, unless it is the new token's
        float4 k0 = make_float4(0.f, 0.f, 0.f, 0.f), v0 = k0;
        const int pr0 = by_wpp(warp), grp = (warp - pr0 * wpp) * kpw + (lane >> llog);
        if (pr0 < pairs && grp < t) {
          const int s = by_nown(pr0);
          const size_t at = cache_row(layer, s, pr0 - s * nown) + (size_t)grp * hd + 4 * sub;
          k0 = *reinterpret_cast<const float4*>(kcache + at);
          v0 = *reinterpret_cast<const float4*>(vcache + at);
        }
        products<S>(w_qkv, nq, d, xn, d, [&](int n, const float (&a0)[S], const float (&a1)[S], int g8) {
          const int hl = by_3hd(n), e = n - hl * 3 * hd;
#pragma unroll
          for (int s = 0; s < S; ++s)
            if (g8 == s) {
              const float2 o = make_float2(a0[s] + b_qkv[n], a1[s] + b_qkv[n + 1]);
              *reinterpret_cast<float2*>(qkv + s * nq + n) = o;
              if (e >= hd && b0 + s < B) {
                float* dst = (e < 2 * hd ? kcache : vcache) + cache_row(layer, s, hl) + (size_t)t * hd + (e < 2 * hd ? e - hd : e - 2 * hd);
                *reinterpret_cast<float2*>(dst) = o;
              }
            }
        });
        __syncthreads();
        // online softmax of every unit that has a key, two units of a warp at a time, then the units of a pair are merged
        constexpr int G = S > 2 ? 2 : 1;
        for (int unit0 = warp; unit0 < pairs * wpp; unit0 += G * SW) {
          const float* mine[G];
          size_t row0[G];
          float4 qv[G], o[G];
          float m[G], l[G];
          int first[G], lead = t + 1;  // a unit's first key; the smaller of them
#pragma unroll
          for (int i = 0; i < G; ++i) {
            const int unit = unit0 + i * SW, pr = by_wpp(unit < pairs * wpp ? unit : unit0), s = by_nown(pr), hl = pr - s * nown;
            first[i] = unit < pairs * wpp ? (unit - pr * wpp) * kpw : t + 1;
            lead = first[i] < lead ? first[i] : lead;
            mine[i] = qkv + s * nq + hl * 3 * hd + 4 * sub;
            row0[i] = cache_row(layer, s, hl) + 4 * sub;
            qv[i] = *reinterpret_cast<const float4*>(mine[i]);
            m[i] = -INFINITY;
            l[i] = 0.f;
            o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          }
          for (int r0 = 0; lead + r0 <= t; r0 += ng) {
            float4 kv[G], vv[G];
            float x[G], mx[G];
#pragma unroll
            for (int i = 0; i < G; ++i) {
              const int j = first[i] + r0 + (lane >> llog);
              kv[i] = vv[i] = make_float4(0.f, 0.f, 0.f, 0.f);  // masked keys: what is in memory may be NaN, and so is 0 x NaN
              if (j == t) {
                kv[i] = *reinterpret_cast<const float4*>(mine[i] + hd);
                vv[i] = *reinterpret_cast<const float4*>(mine[i] + 2 * hd);
              } else if (j < t) {
                if (i == 0 && unit0 == warp && r0 == 0) {
                  kv[i] = k0;
                  vv[i] = v0;
                } else {
                  kv[i] = *reinterpret_cast<const float4*>(kcache + row0[i] + (size_t)j * hd);
                  vv[i] = *reinterpret_cast<const float4*>(vcache + row0[i] + (size_t)j * hd);
                }
              }
              x[i] = fmaf(qv[i].x, kv[i].x, fmaf(qv[i].y, kv[i].y, fmaf(qv[i].z, kv[i].z, qv[i].w * kv[i].w)));
            }
            for (int off = lpk >> 1; off > 0; off >>= 1)
#pragma unroll
              for (int i = 0; i < G; ++i) x[i] += __shfl_xor_sync(0xffffffffu, x[i], off);
#pragma unroll
            for (int i = 0; i < G; ++i) mx[i] = x[i] = first[i] + r0 + (lane >> llog) <= t ? x[i] * scale : -INFINITY;
            for (int off = lpk; off < 32; off <<= 1)
#pragma unroll
              for (int i = 0; i < G; ++i) mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], off));
#pragma unroll
            for (int i = 0; i < G; ++i) {
              if (G > 1 && first[i] + r0 > t) continue;  // this unit has no more keys
              const float mn = fmaxf(m[i], mx[i]);       // its first key is visible: finite
              const float corr = expf(m[i] - mn), p = expf(x[i] - mn);
              m[i] = mn;
              l[i] = fmaf(l[i], corr, p);
              o[i].x = fmaf(o[i].x, corr, p * vv[i].x); o[i].y = fmaf(o[i].y, corr, p * vv[i].y);
              o[i].z = fmaf(o[i].z, corr, p * vv[i].z); o[i].w = fmaf(o[i].w, corr, p * vv[i].w);
            }
          }
          for (int off = lpk; off < 32; off <<= 1)
#pragma unroll
            for (int i = 0; i < G; ++i) {
              l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);
              o[i].x += __shfl_xor_sync(0xffffffffu, o[i].x, off); o[i].y += __shfl_xor_sync(0xffffffffu, o[i].y, off);
              o[i].z += __shfl_xor_sync(0xffffffffu, o[i].z, off); o[i].w += __shfl_xor_sync(0xffffffffu, o[i].w, off);
            }
#pragma unroll
          for (int i = 0; i < G; ++i) {
            float* pt = part + (unit0 + i * SW) * (hd + 4);
            if (first[i] <= t && lane < lpk) *reinterpret_cast<float4*>(pt + 4 * lane) = o[i];
            if (first[i] <= t && lane == 0) { pt[hd] = m[i]; pt[hd + 1] = l[i]; }
          }
        }
        __syncthreads();
        const int aw = (t + kpw) >> klog < wpp ? (t + kpw) >> klog : wpp;  // units of a pair that have a key
        for (int i = threadIdx.x; i < pairs * hd; i += ST) {
          const int pr = by_hd(i), c = i - pr * hd;
          const float* pt = part + pr * wpp * (hd + 4);
          float mx = pt[hd];
#pragma unroll 4
          for (int k = 1; k < aw; ++k) mx = fmaxf(mx, pt[k * (hd + 4) + hd]);
          float num = 0.f, den = 0.f;
#pragma unroll 4
          for (int k = 0; k < aw; ++k) {
            const float e = expf(pt[k * (hd + 4) + hd] - mx);
            num = fmaf(e, pt[k * (hd + 4) + c], num);
            den = fmaf(e, pt[k * (hd + 4) + hd + 1], den);
          }
          att[i] = num / den;  // [s][own head][hd]
        }
        __syncthreads();
        products<S>(w_o, d, nown * hd, att, nown * hd, [&](int n, const float (&a0)[S], const float (&a1)[S], int g8) {
#pragma unroll
          for (int s = 0; s < S; ++s) push2(recv_a + (r * S + s) * d + n, &bar_a, g8, a0[s], a1[s]);
        });
      } else if (threadIdx.x < SC) {
        arrive_at(&bar_a, threadIdx.x);  // this CTA has read the rows of the previous MLP exchange
      }
      if (warp < S && arrived(&bar_a, parity))
        add_ln_row(h + warp * d, xn + warp * d, recv_a + warp * d, owners, S * d, vec + 2 * d, vec + 3 * d, vec + 4 * d, d, inv_d, lane);
      __syncthreads();
      products<S>(w_1, nu, d, xn, d, [&](int n, const float (&a0)[S], const float (&a1)[S], int g8) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
          if (g8 == 2 * s) hid[s * nu + n] = gelu_erf(a0[s] + b_1[n]);
          if (g8 == 2 * s + 1) hid[s * nu + n + 1] = gelu_erf(a1[s] + b_1[n + 1]);
        }
      });
      __syncthreads();
      products<S>(w_2, d, nu, hid, nu, [&](int n, const float (&a0)[S], const float (&a1)[S], int g8) {
#pragma unroll
        for (int s = 0; s < S; ++s) push2(recv_m + (r * S + s) * d + n, &bar_m, g8, a0[s], a1[s]);
      });
      const bool last = layer + 1 == P.n_layers;
      const float* nv = last ? fixed : s_mem + (layer + 2) * layer_floats - 6 * d;  // the next LayerNorm's gain and shift
      if (warp < S && arrived(&bar_m, parity))
        add_ln_row(h + warp * d, xn + warp * d, recv_m + warp * d, SC, S * d, vec + 5 * d, nv, nv + d, d, inv_d, lane);
      if (last) cp_async_wait<0>();  // v of the next token
      __syncthreads();
      if (s_failed) break;
    }
    // head and update (Eq. 5), by every CTA for itself: outputs n, n + 1 are mu~, alpha~ of value n / 2
    products<S>(w_out, No, d, xn, d, [&](int n, const float (&a0)[S], const float (&a1)[S], int g8) {
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (g8 == s && n < 2 * D) {
          const int c = n >> 1;
          const float x = fmaf(vnext[((t + 1) & 1) * S * Dp + s * Dp + c], expf(a1[s] + b_out[n + 1]), a0[s] + b_out[n]);
          tok[s * Dp + c] = x;
          if (r == 0 && b0 + s < B) u[((size_t)(b0 + s) * L + tok_index(t + 1, L, reversed)) * D + c] = x;
        }
    });
    __syncthreads();
  }
  cluster_sync();  // nobody leaves while its shared memory may still be written
}

}  // namespace f32
