// A sequentially decoded block (Eq. 5 with a key/value cache) as ONE kernel: every decoding step of every layer, for widths
// 128, 256, 512 and 1024 with an MLP ratio of 4 (bf16 engine).
//
// Why: a step pushes one token per sample through the block, so it is a chain of small dependent pieces; as 8 kernels per
// layer each piece cost 3.4 us, most of it kernel boundary.  Here the CTAs stay resident (cooperative launch) and hand
// results on with data that carries its own sequence number.
//
// Work is cut two ways.  A cluster of CS CTAs owns one attention head and 256 hidden units of the MLP; inside a cluster, CTA
// (rank) r owns the K range r of its input projections and the output columns r CW .. of the residual row (CW = width / CS).
//   * inside a cluster (distributed shared memory, copies that complete on the receiver's mbarrier): partial q, k, v and
//     hidden units are reduce-scattered, attention outputs and hidden units all-gathered, row statistics exchanged;
//   * between clusters only CTAs of the same rank talk (through L2): the partial residual rows of the heads / unit groups
//     go to the row's owner cluster, whose ranks add them in slice order, keep the residual stream in registers, normalise
//     and publish their columns of the next projection's input, which are exactly the columns rank r of every cluster needs.
//   A word of such an exchange is 8 bytes {32 bits of data, sequence number}, stored and loaded as one 64-bit access: the
//   consumer polls the data itself, so there is no fence, no flag and no second round trip.  Sequence numbers grow over all
//   launches of a model, so the buffers are never reset.  One buffer each suffices: a producer reaches its next write only
//   through data that depends on every read of the previous one.
// Per half layer:   gather rows -> tcgen05 (weights as the M operand) -> reduce-scatter -> attention | GELU -> all-gather ->
//                   tcgen05 -> partial rows -> owner: residual + LayerNorm -> publish
// Weights travel through a ring of TMA slots in the order in which they are used, ahead of the activations (a warp of its own
// refills what has been used), and so do, between a layer's first and second projection, the keys and values of earlier
// tokens: up to 160 KB per CTA are on their way, where loads of the attending warps kept 32 KB (width 1024, 64 samples:
// 36 of a block's 85 ms went to attention).  Where a block's weights exceed half of L2 they are prefetched into L2 a layer
// ahead.
// A step's head, update and embedding are done by the row's owner cluster on the CUDA cores.
// Clusters are of 4 CTAs (2 at width 128): with most of an SM's shared memory per CTA, 33 of those fit the GPU side by side,
// but only 15 of 8, and width 1024 has 16 heads.
// Control flow is uniform per warp and visibly so to the compiler (rank from blockIdx, warp index and flags through a
// shuffle): with shuffles in code that it takes for divergent every shuffle costs 200 to 300 cycles instead of 30.
// A sample's arithmetic depends neither on the batch nor on its place in it: split and order of every sum are fixed.
// Every wait is bounded (2 s): a wait that runs out records a code, all later waits then fail at once, the kernel
// leaves at the next step, meets its cluster a last time and frees its tensor memory.
#pragma once
#include "common.cuh"
#include "gemm_tc.cuh"

namespace seqp {

using namespace tc;

constexpr int NTHREADS = 256, NWARPS = 8, HD = 64, UNITS = 256;  // compute threads; one more warp moves the weights

// what a layer needs, in device memory; tensor maps have boxes of 64 rows x 64 k
struct __align__(128) Layer {
  CUtensorMap qkv, wo, w1, w2;
};
// A layer's vectors, one after the other, in units of the width.  They are addressed by arithmetic: the waits at cluster scope
// leave nothing in L1, so a table of pointers would cost a second trip to L2 before each of them.
enum Vec { V_LN1G = 0, V_LN1B = 1, V_BQKV = 2, V_BO = 5, V_LN2G = 6, V_LN2B = 7, V_B1 = 8, V_B2 = 12, V_COUNT = 13 };
struct Job {
  CUtensorMap kmap, vmap;           // the caches as rows of 64, in boxes of 32 rows
  const Layer* layers;
  const float* vecs;                // [n_layers][V_COUNT][width]
  const float *lnf_g, *lnf_b, *w_in_t, *b_in, *pos, *cls, *b_out, *v;
  const bf16* w_out;
  float* u;
  const int* labels;
  bf16 *kc, *vc;
  int layer_rows;                   // cache rows of 64 per layer
  unsigned long long *xpart, *xrow; // exchange buffers
  int n_layers, B, rows, L, Dt, reversed;  // rows: samples per group (a group = one set of clusters); Dt: token dimension
  uint32_t seq0;
  int prefetch_w;
  float scale_log2e;
  int* err;
};

template <int D, int RT>
struct Cfg {
  static constexpr int HEADS = D / 64, CS = D >= 256 ? 4 : 2, N1 = D / 64 / CS, CW = 64 * N1;
  static constexpr int UNIT = 8192 * N1;           // a weight slot: N1 tiles of 64 rows x 64 k; a layer is 12 of them
  static constexpr int UPC = UNITS / CS;           // hidden units a CTA finishes
  static constexpr int BL = RT / CS;               // samples a CTA attends for, at most
  static constexpr int RPC = RT / HEADS;           // residual rows a cluster owns, at most
  static constexpr int QN = CW / 4, SG = NTHREADS / QN / RPC, NSL = HEADS / SG;  // column quads, groups of slices, slices per group
  // a row's slices are summed as SGC interleaved groups whatever RT, so that a sample's result does not depend on the batch
  static constexpr int SGC = NTHREADS / QN / (RT == 16 ? RPC : RPC / 2), NA = SGC / SG;
  static constexpr int GW = QN * RPC / 32;         // warps of group 0: they hold the residual stream
  static constexpr int SPR = QN > 32 ? QN / 32 : 1, NE = CS * SPR, CE = CW / SPR;  // statistics of a row: NE entries of CE columns
  static constexpr int MT = N1 > 2 ? N1 / 2 : 1;   // 128-row output tiles of a CTA
  // at most 10 slots: the cache rows of a step are then requested when the previous layer's first MLP product has freed a slot,
  // and the wait for that layer's new rows (B_ROWS) costs nothing
  static constexpr int NSLOT_MAX = (RT == 16 ? 163840 : 131072) / UNIT, NSLOT = NSLOT_MAX < 10 ? NSLOT_MAX : 10;
  // cache rows of one sample travel in units of KPU keys, KVS slots each (their keys, then their values)
  static constexpr int KVS = N1 == 1 ? 2 : 1, KPU = KVS * UNIT / 256, WPU = KPU / 16;
  static constexpr int MAXDT = D == 1024 ? 256 : 128;
  static constexpr int RING = 0, ACT = NSLOT * UNIT;  // activation tiles; a 64-row weight tile read as 128 rows may run on into them
  static constexpr int STG = ACT + 4 * RT * 128;      // what is sent to the peers, then what comes from them
  static constexpr int RECV = STG + RT * 1024;
  static constexpr int MERGE = RECV;                  // [sample][warp]: output, maximum, sum; q, k, v have left the place by then
  static constexpr int QKV = RECV + (RT * 1024 > BL * NWARPS * 288 ? RT * 1024 : BL * NWARPS * 288);
  static constexpr int QROW = 512;                    // per sample: q fp32 [64], the new k, the new v bf16 [64]
  static constexpr int SUM = QKV + BL * QROW;
  static constexpr int XN = SUM + (SGC - 1) * RPC * QN * 16;
  static constexpr int TOK = XN + RPC * CW * 4;
  static constexpr int STAT = TOK + RPC * MAXDT * 4;
  static constexpr int BIAS = STAT + RPC * NE * 8;
  static constexpr int BARS = BIAS + 192 * 4;
  static constexpr int NBARS = 3 * NSLOT + 11;
  static constexpr int TOTAL = BARS + NBARS * 8 + 32 + 1024;
  static constexpr uint32_t TMEM = RT == 16 ? 64 : 128;
  static_assert(sizeof(Layer) % sizeof(CUtensorMap) == 0, "tables of layers are stepped in tensor maps");
  static_assert(QN * RPC * SG == NTHREADS && SG * NSL == HEADS && NSL % NA == 0 && SGC > 1 && QN * RPC % 32 == 0 && NSLOT >= 4,
                "thread layout of the residual rows");
  static_assert(TOTAL <= 227 * 1024, "shared memory of a CTA");
  static_assert(N1 > 1 || NSLOT % 2 == 0, "pairs of 64-row tiles must not be split by the ring's end");
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t peer) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(peer));
  return r;
}
__device__ __forceinline__ void st_async1(uint32_t dst, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst), "r"(__float_as_uint(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async2(uint32_t dst, uint32_t a, uint32_t b, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(dst), "r"(a), "r"(b), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async4(uint32_t dst, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst), "r"(a), "r"(b),
               "r"(c), "r"(d), "r"(bar)
               : "memory");
}
// shared memory of this CTA -> shared memory of a peer, completing on the peer's barrier
__device__ __forceinline__ void copy_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "r"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
// Bounded wait; the slow path is a call, because a layer's code is run through once and jumps over inlined slow paths miss in the
// instruction cache (about 85 cycles each).
template <bool CLUSTER>
__device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, int* err, int code) { return mbar_wait<CLUSTER>(bar, parity, err, code); }
template <bool CLUSTER = false>
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, int* err, int code) {
  return mbar_try_wait<CLUSTER>(bar, parity) || wait_slow<CLUSTER>(bar, parity, err, code);
}
// the same for a warp that waits while others work: it sleeps between polls
template <unsigned long long LIMIT_NS = WAIT_LIMIT_NS>
__device__ __noinline__ bool wait_idle(uint32_t bar, uint32_t parity, int* err, int code) {
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    if (ok) return true;
    __nanosleep(100);
    const unsigned long long dt = globaltimer_ns() - t0;
    if (dt > LIMIT_NS) {
      atomicCAS(err, 0, code);
      return false;
    }
    if (dt > 1000000ull && *reinterpret_cast<volatile int*>(err) != 0) return false;
  }
}

// ---- words of the exchanges between clusters
__device__ __forceinline__ unsigned long long tagged(uint32_t v, uint32_t seq) { return ((unsigned long long)seq << 32) | v; }
__device__ __forceinline__ void ll_store(unsigned long long* p, uint32_t v, uint32_t seq) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(tagged(v, seq)) : "memory");
}
__device__ __forceinline__ void ll_store2(unsigned long long* p, uint32_t a, uint32_t b, uint32_t seq) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(tagged(a, seq)), "l"(tagged(b, seq)) : "memory");
}
__device__ __forceinline__ void ll_load2(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ bool ll_here(unsigned long long a, unsigned long long b, uint32_t seq) {
  return (uint32_t)(a >> 32) == seq && (uint32_t)(b >> 32) == seq;
}
template <int CODE = TFERR_WAIT_FULL, unsigned long long LIMIT_NS = WAIT_LIMIT_NS>
struct SpinOf {  // bound of a polling loop
  unsigned n = 0;
  unsigned long long t0 = 0;
  __device__ __noinline__ bool check(int* err) {
    if (*reinterpret_cast<volatile int*>(err) != 0) return false;
    const unsigned long long now = globaltimer_ns();
    if (n == 256u) t0 = now;
    if (now - t0 <= LIMIT_NS) return true;
    atomicCAS(err, 0, CODE);
    return false;
  }
  __device__ __forceinline__ bool more(int* err) { return (++n & 255u) != 0 || check(err); }
};
using Spin = SpinOf<>;

// Self-test of the two other forms of bounded wait: one thread polls a word that nothing writes (which = 0) or waits between naps
// for an mbarrier that nothing arrives on (1).  The wait runs out after a millisecond, is recorded, and the kernel returns normally.
__global__ void wait_selftest_kernel(int* err, int which, const unsigned long long* word) {
  constexpr unsigned long long kLimit = 1000000ull;
  __shared__ __align__(8) unsigned long long idle;
  if (threadIdx.x != 0) return;
  if (which == 0) {
    unsigned long long a, b;
    SpinOf<TFERR_WAIT_SELFTEST, kLimit> spin;
    do ll_load2(word, a, b);
    while (!ll_here(a, b, 1u) && spin.more(err));
  } else {
    mbar_init(smem_u32(&idle), 1);
    wait_idle<kLimit>(smem_u32(&idle), 0u, err, TFERR_WAIT_SELFTEST);
  }
}

// eight accumulator columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_cols8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void prefetch_line(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p) : "memory"); }
__device__ __forceinline__ uint4 lds128(uint32_t at) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 o = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&o);
}

// The ring's filling side (one thread): requests one unit after the other in the order of use, each when its slot's last contents
// have been used: weights by the products that read them, cache rows by the WPU warps that share a unit's tiles.  Before a layer's
// cache rows it waits on rows_bar for the new rows of the layer walked before it (and so of all earlier ones, this layer's in the
// step before among them): their writers have fenced the async proxy, and the arrival orders the bulk copies after those stores.
template <int D, int RT>
__device__ __forceinline__ void feed(const Job& job, uint32_t ring, uint32_t bars, uint32_t rows_bar, int r, int c, bool prefetch_w, int mine, int cache_row0) {
  using C = Cfg<D, RT>;
  constexpr int N1 = C::N1, CW = C::CW;
  const int n_steps = job.L - 1;
  int slot = 0;
  uint32_t used = 0, rows_held = 0, phase_w = 0, phase_kv = 0;  // a bit per slot
  auto acquire = [&](bool rows) {
    const uint32_t bit = 1u << slot;
    bool ok = true;
    if (used & bit) {
      if (rows_held & bit) {
        ok = wait_idle(bars + 8u * (2 * C::NSLOT + slot), (phase_kv & bit) != 0, job.err, TFERR_WAIT_EMPTY);
        phase_kv ^= bit;
      } else {
        ok = wait_idle(bars + 8u * (C::NSLOT + slot), (phase_w & bit) != 0, job.err, TFERR_WAIT_EMPTY);
        phase_w ^= bit;
      }
    }
    used |= bit;
    rows_held = rows ? rows_held | bit : rows_held & ~bit;
    return ok;
  };
  auto next = [&]() { slot = slot + 1 == C::NSLOT ? 0 : slot + 1; };
#pragma unroll 1
  for (int t = 0; t < n_steps; ++t)
#pragma unroll 1
    for (int layer = 0; layer < job.n_layers; ++layer) {
      const Layer* ly = job.layers + layer;
      const int nx = layer + 1 < job.n_layers ? layer + 1 : 0;
      const bool more = prefetch_w && (nx > 0 || t + 1 < n_steps);
#pragma unroll 1
      for (int u = 0; u < 12; ++u) {
        if (u == 3 && mine > 0) {
          const int before = t * job.n_layers + layer - 1;  // every phase is waited for, in order
          if (before >= 0 && !wait_idle(rows_bar, (uint32_t)before & 1u, job.err, TFERR_WAIT_FULL)) return;
#pragma unroll 1
          for (int p = 0; p < mine; ++p)
#pragma unroll 1
            for (int j0 = 0; j0 < t; j0 += C::KPU) {
              const int row = layer * job.layer_rows + cache_row0 + p * C::HEADS * job.L + j0;
              const int boxes = ((t - j0 < C::KPU ? t - j0 : C::KPU) + 31) / 32;
              if (!acquire(true)) return;
              uint32_t at = ring + slot * C::UNIT, full = bars + 8u * slot;
              mbar_arrive_expect_tx(full, boxes * (8192u / C::KVS));
#pragma unroll 1
              for (int b = 0; b < boxes; ++b) tma_load_2d(at + b * 4096, &job.kmap, 0, row + 32 * b, full);
              next();
              if (C::KVS == 2) {
                if (!acquire(true)) return;
                at = ring + slot * C::UNIT;
                full = bars + 8u * slot;
                mbar_arrive_expect_tx(full, boxes * 4096u);
                next();
              } else {
                at += C::KPU * 128;
              }
#pragma unroll 1
              for (int b = 0; b < boxes; ++b) tma_load_2d(at + b * 4096, &job.vmap, 0, row + 32 * b, full);
            }
        }
        if (!acquire(false)) return;
        const uint32_t full = bars + 8u * slot;
        mbar_arrive_expect_tx(full, C::UNIT);
#pragma unroll 1
        for (int z = 0; z < N1; ++z) {  // the unit's 8 KB tiles
          const CUtensorMap* map;
          int x, y;
          if (u < 2) {  // per slab: q, k
            const int i = u * N1 + z;
            map = &ly->qkv;
            x = (r * N1 + (i >> 1)) * 64;
            y = (i & 1) * D + c * HD;
          } else if (u == 2) {  // v of every slab
            map = &ly->qkv;
            x = (r * N1 + z) * 64;
            y = 2 * D + c * HD;
          } else if (u == 3) {
            map = &ly->wo;
            x = c * HD;
            y = r * CW + z * 64;
          } else if (u < 8) {  // per slab: four blocks of 64 hidden units
            const int i = (u - 4) * N1 + z;
            map = &ly->w1;
            x = (r * N1 + (i >> 2)) * 64;
            y = c * UNITS + (i & 3) * 64;
          } else {  // per slab of hidden units: the CTA's output rows
            map = &ly->w2;
            x = c * UNITS + (u - 8) * 64;
            y = r * CW + z * 64;
          }
          tma_load_2d(ring + slot * C::UNIT + z * 8192, map, x, y, full);
          if (more) prefetch_tile(map + (nx - layer) * (int)(sizeof(Layer) / sizeof(CUtensorMap)), x, y);
        }
        next();
      }
    }
}

// grid: groups * HEADS clusters of CS CTAs (cooperative), 256 threads and a warp that moves the weights
template <int D, int RT>
__global__ void __launch_bounds__(NTHREADS + 32, 1)
seq_block_kernel(const __grid_constant__ Job job) {
  using C = Cfg<D, RT>;
  constexpr int HEADS = C::HEADS, CS = C::CS, N1 = C::N1, CW = C::CW, QN = C::QN, SG = C::SG, NSL = C::NSL, UPC = C::UPC, NE = C::NE, NA = C::NA;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  const uint32_t sb = smem_u32(smem), bars = sb + C::BARS;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int r = blockIdx.x % CS, cl = blockIdx.x / CS, c = cl % HEADS, group = cl / HEADS;  // r: rank in the cluster
  const int row0 = group * job.rows, nb = job.B - row0 < job.rows ? job.B - row0 : job.rows;  // this group's samples
  const int L = job.L, Dt = job.Dt, n_steps = L - 1, nl = job.n_layers;
  int* err = job.err;
  auto bar = [&](int i) { return bars + 8u * (3 * C::NSLOT + i); };
  enum { B_IN0, B_IN1, B_RECV0, B_RECV1, B_ALL0, B_ALL1, B_OUT0, B_OUT1, B_STAT, B_HEAD, B_ROWS };  // 0: attention half, 1: MLP half
  uint8_t* tail_mem = smem + C::BARS + C::NBARS * 8;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(tail_mem);
  volatile int* s_bad = reinterpret_cast<volatile int*>(tail_mem + 4);

  if (tid == 0) {
    for (int i = 0; i < C::NBARS; ++i) mbar_init(bars + 8u * i, i / C::NSLOT == 2 ? C::WPU : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *s_bad = 0;
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(C::TMEM)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tcgen05_fence_before();
  __syncthreads();
  cluster_sync();  // every CTA of the cluster has set up its barriers
  tcgen05_fence_after();
  const uint32_t tmem = *tmem_slot;

  // samples this CTA attends for: bl r .. bl r + mine - 1 of the group
  const int bl = (nb + CS - 1) / CS, mine = nb - r * bl < bl ? (nb - r * bl > 0 ? nb - r * bl : 0) : bl;
  auto rows_of = [&](int p) { return ((row0 + r * bl + p) * HEADS + c) * L; };  // cache rows of (sample, head)

  if (warp == NWARPS) {
    // ==================================================================== weights
    if (lane == 0) feed<D, RT>(job, sb + C::RING, bars, bar(B_ROWS), r, c, job.prefetch_w && group == 0, mine, rows_of(0));
  } else {
    constexpr uint32_t idesc = make_idesc(RT);
    // attention: a sample's keys are cut into tiles of 16, dealt out to eight sets whatever the batch; a set belongs to a warp,
    // eight lanes share a key (eight channels each), the warp's four groups of lanes take every fourth key
    const int sub = lane & 7, kgrp = lane >> 3;
    // hidden units this thread finishes: eight of them, samples fb, fb + FB, ...
    constexpr int FB = NTHREADS / (UPC / 8);
    const int u8 = (tid % (UPC / 8)) * 8, fb = tid / (UPC / 8);
    // rows of the residual stream: the cluster owns rows own0 .. own0 + own - 1 of the group, this CTA their columns r CW ..;
    // thread = (column quad q, row, group g of slices); the warps of g == 0 hold the residual stream itself in h
    const int rpc = (nb + HEADS - 1) / HEADS, own0 = c * rpc, own = nb - own0 < rpc ? (nb - own0 > 0 ? nb - own0 : 0) : rpc;
    const int q = tid % QN, lrow = (tid / QN) % C::RPC, g = tid / (QN * C::RPC), col = r * CW + 4 * q;
    const bool my_row = lrow < own, holder = warp < C::GW;
    const float* cls_row = job.cls != nullptr && my_row ? job.cls + (size_t)job.labels[row0 + own0 + lrow] * D : nullptr;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 h = zero4;
    float4* s_sum = reinterpret_cast<float4*>(smem + C::SUM);
    float* s_xn = reinterpret_cast<float*>(smem + C::XN);
    float* s_tok = reinterpret_cast<float*>(smem + C::TOK);
    float* s_bias = reinterpret_cast<float*>(smem + C::BIAS);
    float* s_merge = reinterpret_cast<float*>(smem + C::MERGE);
    unsigned long long* xrow = job.xrow + (size_t)group * RT * (D / 2);
    unsigned long long* xpart = job.xpart + (size_t)group * RT * HEADS * D;
    int slot = 0;  // position in the weight ring
    uint32_t ring_parity = 0, stat_parity = 0, seq = job.seq0;
    bool alive = true;  // no wait of this thread has failed: after a failure no barrier is armed any more

    auto cbar = [&]() { named_bar_sync(1, NTHREADS); };
    auto await = [&](int b, uint32_t parity, int code) {
      if (!wait_bar(bar(b), parity, err, code)) alive = false;
      __syncwarp();
    };
    auto await_peers = [&](int b, uint32_t parity) {
      if (!wait_bar<true>(bar(b), parity, err, TFERR_WAIT_FULL)) alive = false;
      __syncwarp();
    };
    // unit u of the phase has arrived: its address (warp 0); the products of unit u have been issued; next phase
    auto take = [&](int u) {
      const int s = slot + u, wrap = s >= C::NSLOT;
      if (!wait_bar(bars + 8u * (s - (wrap ? C::NSLOT : 0)), ring_parity ^ (uint32_t)wrap, err, TFERR_WAIT_FULL)) alive = false;
      __syncwarp();
      return sb + C::RING + (s - (wrap ? C::NSLOT : 0)) * C::UNIT;
    };
    auto release = [&](int u) {
      const int s = slot + u;
      umma_commit(bars + 8u * (C::NSLOT + (s >= C::NSLOT ? s - C::NSLOT : s)));
    };
    auto advance = [&](int n) {
      slot += n;
      if (slot >= C::NSLOT) { slot -= C::NSLOT; ring_parity ^= 1u; }
    };
    auto mma = [&](uint32_t d, uint32_t w, uint32_t x, bool add) {
      const uint64_t wd = make_smem_desc(w), xd = make_smem_desc(x);
#pragma unroll
      for (int k = 0; k < 4; ++k) umma_f16(d, wd + 2u * k, xd + 2u * k, idesc, k > 0 || add);
    };
    // one warp polls, everybody else waits at the compute warps' barrier
    auto meet = [&](int b, uint32_t parity) {
      if (warp == 0) await_peers(b, parity);
      cbar();
    };
    auto ld4 = [&](const float* p) { return __ldg(reinterpret_cast<const float4*>(p + col)); };
    auto token_at = [&](int row, int l) { return ((size_t)(row0 + own0 + row) * L + tok_index(l, L, job.reversed)) * Dt; };

#pragma unroll 1
    for (int row = 0; row < own; ++row) {  // the first token is copied (Eq. 5, first row)
      const size_t e = token_at(row, 0);
#pragma unroll 1
      for (int cc = tid; cc < Dt; cc += NTHREADS) {
        const float x = job.v[e + cc];
        s_tok[row * Dt + cc] = x;
        if (r == 0) job.u[e + cc] = x;
      }
    }

    for (int t = 0; t < n_steps; ++t) {
      cbar();
      if (__shfl_sync(0xffffffffu, *s_bad, 0) != 0) break;
#pragma unroll 1
      for (int half = 0; half <= 2 * nl; ++half) {
        const float* vec = job.vecs + (size_t)(half >> 1) * (V_COUNT * D);
        const int mlp = half & 1;                                   // which half of the layer follows
        const uint32_t lp = (uint32_t)(t * nl + (half >> 1)) & 1u;  // parity of its barriers
        // ================================================================== residual rows of this cluster
        if (own > 0) {
          float4 gg = zero4, bb = zero4, add = zero4, sum[NA];
#pragma unroll
          for (int i = 0; i < NA; ++i) sum[i] = zero4;
          if (holder && my_row) {
            gg = ld4(half == 2 * nl ? job.lnf_g : vec + (mlp ? V_LN2G : V_LN1G) * D);
            bb = ld4(half == 2 * nl ? job.lnf_b : vec + (mlp ? V_LN2B : V_LN1B) * D);
            add = ld4(half == 0 ? job.b_in : mlp ? vec + V_BO * D : vec - (V_COUNT - V_B2) * D);
          }
          if (half == 0) {  // embedding of token t
            if (my_row) {
              if (holder) {
                const float4 p = ld4(job.pos + (size_t)t * D);
                add.x += p.x; add.y += p.y; add.z += p.z; add.w += p.w;
                if (cls_row != nullptr) {
                  const float4 y = ld4(cls_row);
                  add.x += y.x; add.y += y.y; add.z += y.z; add.w += y.w;
                }
                h = zero4;
              }
#pragma unroll
              for (int i = 0; i < NA; ++i)
#pragma unroll 4
                for (int cc = g + i * SG; cc < Dt; cc += C::SGC) {
                  const float4 w = ld4(job.w_in_t + (size_t)cc * D);
                  const float tv = s_tok[lrow * Dt + cc];
                  sum[i].x = fmaf(tv, w.x, sum[i].x); sum[i].y = fmaf(tv, w.y, sum[i].y);
                  sum[i].z = fmaf(tv, w.z, sum[i].z); sum[i].w = fmaf(tv, w.w, sum[i].w);
                }
            }
          } else if (my_row) {  // the slices of this thread's groups, added in index order
            unsigned long long w[NSL][4];
            Spin spin;
            bool ok = true, all;
            const unsigned long long* at = xpart + ((size_t)(own0 + lrow) * HEADS + g) * D + col;
            do {  // one slice is polled; when it is there, so are, nearly always, the others
              ll_load2(at, w[0][0], w[0][1]);
              ll_load2(at + 2, w[0][2], w[0][3]);
            } while (!(ll_here(w[0][0], w[0][1], seq) && ll_here(w[0][2], w[0][3], seq)) && (ok = spin.more(err)));
            if (NSL > 1) do {
                all = true;
#pragma unroll
                for (int k = 1; k < NSL; ++k) {
                  ll_load2(at + (size_t)k * SG * D, w[k][0], w[k][1]);
                  ll_load2(at + (size_t)k * SG * D + 2, w[k][2], w[k][3]);
                }
#pragma unroll
                for (int k = 1; k < NSL; ++k) all = all && ll_here(w[k][0], w[k][1], seq) && ll_here(w[k][2], w[k][3], seq);
              } while (!all && ok && (ok = spin.more(err)));
            alive = alive && ok;
#pragma unroll
            for (int k = 0; k < NSL; ++k) {
              float4& a = sum[k % NA];
              a.x += __uint_as_float((uint32_t)w[k][0]); a.y += __uint_as_float((uint32_t)w[k][1]);
              a.z += __uint_as_float((uint32_t)w[k][2]); a.w += __uint_as_float((uint32_t)w[k][3]);
            }
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < NA; ++i)
            if (i > 0 || !holder) s_sum[((g + i * SG - 1) * C::RPC + lrow) * QN + q] = sum[i];
          cbar();
          if (holder) {
            if (tid == 0 && alive) mbar_arrive_expect_tx(bar(B_STAT), (uint32_t)(own * NE * 8));
            __syncwarp();
            h.x += add.x + sum[0].x; h.y += add.y + sum[0].y; h.z += add.z + sum[0].z; h.w += add.w + sum[0].w;
#pragma unroll
            for (int k = 0; k < C::SGC - 1; ++k) {
              const float4 y = s_sum[(k * C::RPC + lrow) * QN + q];
              h.x += y.x; h.y += y.y; h.z += y.z; h.w += y.w;
            }
            // LayerNorm: (mean, squared deviations) of CE columns by shuffles, exchanged over the cluster and combined
            // (Chan et al.), as accurate as two passes over the row
            float s = (h.x + h.y) + (h.z + h.w);
#pragma unroll
            for (int o = (QN > 32 ? 32 : QN) / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            const float wmean = s * (1.f / C::CE);
            float a0 = h.x - wmean, a1 = h.y - wmean, a2 = h.z - wmean, a3 = h.w - wmean;
            float m2 = (a0 * a0 + a1 * a1) + (a2 * a2 + a3 * a3);
#pragma unroll
            for (int o = (QN > 32 ? 32 : QN) / 2; o > 0; o >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
            const int ql = QN > 32 ? q & 31 : q;
            if (my_row && ql < CS)
              st_async2(peer_addr(sb + C::STAT + (lrow * NE + r * C::SPR + (QN > 32 ? q >> 5 : 0)) * 8, ql), __float_as_uint(wmean),
                        __float_as_uint(m2), peer_addr(bar(B_STAT), ql));
            __syncwarp();
            await_peers(B_STAT, stat_parity);
            const float2* st = reinterpret_cast<const float2*>(smem + C::STAT) + lrow * NE;
            float mean = 0.f;
#pragma unroll
            for (int k = 0; k < NE; ++k) mean += st[k].x;
            mean *= 1.f / NE;
            m2 = 0.f;
#pragma unroll
            for (int k = 0; k < NE; ++k) {
              const float2 e = st[k];
              m2 += fmaf((float)C::CE * (e.x - mean), e.x - mean, e.y);
            }
            const float rstd = rsqrtf(m2 * (1.f / D) + 1e-5f);
            const uint32_t lo = pack_bf16(fmaf((h.x - mean) * rstd, gg.x, bb.x), fmaf((h.y - mean) * rstd, gg.y, bb.y));
            const uint32_t hi = pack_bf16(fmaf((h.z - mean) * rstd, gg.z, bb.z), fmaf((h.w - mean) * rstd, gg.w, bb.w));
            if (my_row) {
              if (half < 2 * nl) {  // this thread's columns of the next projection's input
                ll_store2(xrow + ((size_t)(own0 + lrow) * CS + r) * (CW / 2) + 2 * q, lo, hi, seq + 1);
              } else {  // the head's input
                const float2 f0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&lo));
                const float2 f1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hi));
                *reinterpret_cast<float4*>(s_xn + lrow * CW + 4 * q) = make_float4(f0.x, f0.y, f1.x, f1.y);
              }
            }
          }
          stat_parity ^= 1u;
          cbar();  // the other warps have waited here instead of polling for the next rows
        }
        ++seq;
        if (half == 2 * nl) break;
        // ================================================================== half a layer
        if (tid == 0 && alive) {
          if (mlp) {
            mbar_arrive_expect_tx(bar(B_RECV1), (uint32_t)(CS * nb * UPC * 4));
            mbar_arrive_expect_tx(bar(B_ALL1), (uint32_t)(nb * UNITS * 2));
          } else {
            if (mine > 0) mbar_arrive_expect_tx(bar(B_RECV0), (uint32_t)(CS * mine * 192 * 4));
            mbar_arrive_expect_tx(bar(B_ALL0), (uint32_t)(nb * 128));
          }
        }
        __syncwarp();
        if (half == 1 && own > 0 && t + 1 < n_steps) {  // what the end of the step will read from memory: on its way to L2
          if (holder && my_row) prefetch_line(job.pos + (size_t)(t + 1) * D + col);
          const int per = (Dt + 31) / 32;
          if (tid < own * per) prefetch_line(job.v + token_at(tid / per, t + 1) + (tid % per) * 32);
        }
        // stored below, once the rows are here: the waits at cluster scope leave nothing in L1, so this is a trip to L2
        float bias_qkv = 0.f;
        if (!mlp && tid < 192) bias_qkv = __ldg(vec + V_BQKV * D + (tid >> 6) * D + c * HD + (tid & 63));
        {  // rows of the projection's input (this rank's columns) into swizzled [RT][64] operand tiles
          constexpr int IT = RT * QN / NTHREADS;
          unsigned long long w[IT][2];
          Spin spin;
          bool ok = true, all;
          const int first = tid / QN;
          const unsigned long long* at = xrow + ((size_t)first * CS + r) * (CW / 2) + 2 * q;
          if (first < nb) {
            do ll_load2(at, w[0][0], w[0][1]);
            while (!ll_here(w[0][0], w[0][1], seq) && (ok = spin.more(err)));
          }
          if (IT > 1) do {
              all = true;
#pragma unroll
              for (int k = 1; k < IT; ++k)
                if (first + k * (NTHREADS / QN) < nb) ll_load2(at + (size_t)k * (NTHREADS / QN) * (D / 2), w[k][0], w[k][1]);
#pragma unroll
              for (int k = 1; k < IT; ++k)
                if (first + k * (NTHREADS / QN) < nb) all = all && ll_here(w[k][0], w[k][1], seq);
            } while (!all && ok && (ok = spin.more(err)));
          alive = alive && ok;
#pragma unroll
          for (int k = 0; k < IT; ++k) {
            const int row = first + k * (NTHREADS / QN);
            if (row < nb)
              *reinterpret_cast<uint2*>(smem + C::ACT + (q >> 4) * (RT * 128) + swz128(row, (q & 15) >> 1) + (q & 1) * 8) =
                  make_uint2((uint32_t)w[k][0], (uint32_t)w[k][1]);
          }
          if (!mlp && tid < 192) s_bias[tid] = bias_qkv;
          fence_proxy_async_smem();
          __syncwarp();
        }
        cbar();
        if (warp == 0) {
#pragma unroll 1
          for (int u = 0; u < (mlp ? 4 : 3); ++u) {
            const uint32_t w = take(u);
            tcgen05_fence_after();
            if (elect_one()) {
              const uint32_t act = sb + C::ACT;
              if (mlp) {  // per slab the cluster's 256 units; with 64-row tiles a pair of units is one operand
                if (N1 == 4) {
                  mma(tmem, w, act + u * (RT * 128), u > 0);
                  mma(tmem + RT, w + 16384, act + u * (RT * 128), u > 0);
                } else if (N1 == 2) {
                  mma(tmem + (u & 1) * RT, w, act + (u >> 1) * (RT * 128), u > 1);
                } else if (u & 1) {
                  mma(tmem + (u >> 1) * RT, w - C::UNIT, act, false);
                }
              } else if (u < 2) {  // q | k per slab
                if (N1 == 1) {
                  if (u == 1) mma(tmem, w - C::UNIT, act, false);
                } else {
#pragma unroll 1
                  for (int z = 0; z < N1 / 2; ++z) mma(tmem, w + z * 16384, act + (u * (N1 / 2) + z) * (RT * 128), u + z > 0);
                }
              } else {  // v of every slab
#pragma unroll 1
                for (int z = 0; z < N1; ++z) mma(tmem + RT, w + z * 8192, act + z * (RT * 128), z > 0);
              }
              if (N1 == 1 && (mlp || u < 2)) {
                if (u & 1) { release(u - 1); release(u); }
              } else {
                release(u);
              }
              if (u == (mlp ? 3 : 2)) umma_commit(bar(B_IN0 + mlp));
            }
            __syncwarp();
          }
          await(B_IN0 + mlp, lp, TFERR_WAIT_TMEM_FULL);
          tcgen05_fence_before();
        }
        advance(mlp ? 4 : 3);
        cbar();
        tcgen05_fence_after();
        const uint32_t t_lane = tmem + (warp >> 2) * RT + ((uint32_t)((warp & 3) * 32) << 16);
        if (!mlp) {
          // ---------------------------------------------------------------- attention
          if (warp < 6) {  // reduce-scatter: warp w holds channels 32 w .. of q | k | v, one sample per column
            float* stg = reinterpret_cast<float*>(smem + C::STG) + warp * 32 + lane;
#pragma unroll 1
            for (int b0 = 0; b0 < nb; b0 += 8) {
              float v[8];
              tmem_cols8(t_lane + b0, v);
#pragma unroll
              for (int b = 0; b < 8; ++b)
                if (b0 + b < nb) stg[(b0 + b) * 192] = v[b];
            }
            tcgen05_fence_before();
          }
          fence_proxy_async_smem();
          cbar();
          if (tid < CS) {  // samples bl p .. go to CTA p
            const int n = nb - tid * bl < bl ? nb - tid * bl : bl;
            if (n > 0)
              copy_to_peer(peer_addr(sb + C::RECV + r * C::BL * 768, tid), sb + C::STG + tid * bl * 768, (uint32_t)n * 768,
                           peer_addr(bar(B_RECV0), tid));
          }
          __syncwarp();
          if (mine > 0) {
            meet(B_RECV0, lp);
            for (int i = tid; i < mine * 48; i += NTHREADS) {  // four channels of q, k or v of one sample
              const int p = i / 48, c4 = i - p * 48;
              float4 x = *reinterpret_cast<const float4*>(s_bias + 4 * c4);
              const float* src = reinterpret_cast<const float*>(smem + C::RECV) + p * 192 + 4 * c4;
#pragma unroll
              for (int k = 0; k < CS; ++k) {
                const float4 y = *reinterpret_cast<const float4*>(src + k * C::BL * 192);
                x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
              }
              uint8_t* mem = smem + C::QKV + p * C::QROW;
              if (c4 < 16) {  // scores in base-2 units: softmax via exp2
                *reinterpret_cast<float4*>(mem + 16 * c4) =
                    make_float4(x.x * job.scale_log2e, x.y * job.scale_log2e, x.z * job.scale_log2e, x.w * job.scale_log2e);
              } else {
                const uint2 w2 = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
                *reinterpret_cast<uint2*>(mem + 256 + (c4 - 16) * 8) = w2;
                const size_t row = (size_t)(half >> 1) * job.layer_rows + rows_of(p) + t;
                *reinterpret_cast<uint2*>((c4 < 32 ? job.kc : job.vc) + row * HD + (c4 & 15) * 4) = w2;
              }
            }
            cbar();
            const int units = (t + C::KPU - 1) / C::KPU, tiles = t / 16 + 1, sets = tiles < NWARPS ? tiles : NWARPS;
#pragma unroll 1
            for (int p = 0; p < mine; ++p) {
              const uint8_t* mem = smem + C::QKV + p * C::QROW;
              const int set = C::WPU == NWARPS ? warp : (warp + 4 * p) & 7;  // where a unit has four tiles the other warps begin the next sample
              float2 q2[4], o2[4];
#pragma unroll
              for (int i = 0; i < 4; i += 2) {
                const float4 q4 = *reinterpret_cast<const float4*>(mem + sub * 32 + i * 8);
                q2[i] = make_float2(q4.x, q4.y);
                q2[i + 1] = make_float2(q4.z, q4.w);
                o2[i] = o2[i + 1] = make_float2(0.f, 0.f);
              }
              float m_run = -INFINITY, l_run = 0.f;  // of this group of lanes
              const int tile_end = tiles > units * C::WPU ? tiles : units * C::WPU;
#pragma unroll 1
              for (int tile = set; tile < tile_end; tile += NWARPS) {
                const int unit = tile / C::WPU, pos = slot + (p * units + unit) * C::KVS, wrap = pos / C::NSLOT, at = pos - wrap * C::NSLOT;
                const int av = C::KVS == 1 ? at : at + 1 == C::NSLOT ? 0 : at + 1;  // the values' slot
                if (unit < units) {
                  const uint32_t parity = ring_parity ^ (uint32_t)(wrap & 1);
                  if (!wait_bar(bars + 8u * at, parity, err, TFERR_WAIT_FULL)) alive = false;
                  if (C::KVS == 2 && !wait_bar(bars + 8u * av, parity ^ (uint32_t)(av == 0), err, TFERR_WAIT_FULL)) alive = false;
                  __syncwarp();
                }
                if (tile < tiles) {
                  const uint32_t kbase = sb + C::RING + at * C::UNIT + (tile % C::WPU) * 2048, new_row = sb + C::QKV + p * C::QROW + 256 + sub * 16;
                  const uint32_t vbase = sb + C::RING + av * C::UNIT + (C::KVS == 1 ? C::KPU * 128 : 0) + (tile % C::WPU) * 2048;
                  uint4 kn[4], vn[4];
#pragma unroll
                  for (int k = 0; k < 4; ++k) {  // rows that are not in the ring (the first of them is the new token's) read the new row
                    const int row = 4 * k + kgrp;
                    const bool in = tile * 16 + row < t;
                    kn[k] = lds128(in ? kbase + swz128(row, sub) : new_row);
                    vn[k] = lds128(in ? vbase + swz128(row, sub) : new_row + 128);
                  }
                  float sc[4];
#pragma unroll
                  for (int k = 0; k < 4; ++k) {
                    const __nv_bfloat162* k2 = reinterpret_cast<const __nv_bfloat162*>(&kn[k]);
                    float2 s2 = fmul2(q2[0], __bfloat1622float2(k2[0]));
#pragma unroll
                    for (int i = 1; i < 4; ++i) s2 = ffma2(q2[i], __bfloat1622float2(k2[i]), s2);
                    sc[k] = s2.x + s2.y;
                  }
#pragma unroll
                  for (int off = 1; off < 8; off <<= 1)
#pragma unroll
                    for (int k = 0; k < 4; ++k) sc[k] += __shfl_xor_sync(0xffffffffu, sc[k], off);
#pragma unroll
                  for (int k = 0; k < 4; ++k)
                    if (tile * 16 + 4 * k + kgrp > t) sc[k] = -INFINITY;
                  const float m_new = fmaxf(fmaxf(m_run, fmaxf(sc[0], sc[1])), fmaxf(sc[2], sc[3]));
                  const float m_ref = m_new > -INFINITY ? m_new : 0.f;  // a group that has seen no key yet keeps its zeros
                  const float corr = ex2_approx(m_run - m_ref);         // 0 when m_run = -inf
                  l_run *= corr;
#pragma unroll
                  for (int i = 0; i < 4; ++i) o2[i] = fmul2(o2[i], make_float2(corr, corr));
#pragma unroll
                  for (int k = 0; k < 4; ++k) {
                    const float pj = ex2_approx(sc[k] - m_ref);  // 0 for a masked key
                    l_run += pj;
                    const __nv_bfloat162* v2 = reinterpret_cast<const __nv_bfloat162*>(&vn[k]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) o2[i] = ffma2(make_float2(pj, pj), __bfloat1622float2(v2[i]), o2[i]);
                  }
                  m_run = m_new;
                }
                if (unit < units) {
                  __syncwarp();
                  if (elect_one()) {
                    mbar_arrive(bars + 8u * (2 * C::NSLOT + at));
                    if (C::KVS == 2) mbar_arrive(bars + 8u * (2 * C::NSLOT + av));
                  }
                  __syncwarp();
                }
              }
              if (set < sets) {  // the warp's four groups; a lane keeps the half of the channels that its partner gives up
                const float mw = fmaxf(fmaxf(m_run, __shfl_xor_sync(0xffffffffu, m_run, 8)),
                                       fmaxf(__shfl_xor_sync(0xffffffffu, m_run, 16), __shfl_xor_sync(0xffffffffu, m_run, 24)));
                const float f = ex2_approx(m_run - mw);  // mw is finite: the set has a key; 0 for a group without one
                l_run *= f;
                l_run += __shfl_xor_sync(0xffffffffu, l_run, 8);
                l_run += __shfl_xor_sync(0xffffffffu, l_run, 16);
                float2 a[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {  // channels 0-3 stay with the groups 0 and 2, 4-7 with 1 and 3
                  const float2 x = fmul2(o2[i], make_float2(f, f)), y = fmul2(o2[i + 2], make_float2(f, f));
                  const float2 keep = kgrp & 1 ? y : x, send = kgrp & 1 ? x : y;
                  a[i] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, 8), keep.y + __shfl_xor_sync(0xffffffffu, send.y, 8));
                }
                const float2 keep = kgrp & 2 ? a[1] : a[0], send = kgrp & 2 ? a[0] : a[1];
                float* mg = s_merge + (p * NWARPS + set) * 72;
                *reinterpret_cast<float2*>(mg + 8 * sub + 4 * (kgrp & 1) + (kgrp & 2)) =
                    make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, 16), keep.y + __shfl_xor_sync(0xffffffffu, send.y, 16));
                if (lane == 0) { mg[64] = mw; mg[65] = l_run; }
              }
              __syncwarp();
            }
            {
              const int pos = slot + mine * units * C::KVS, wraps = pos / C::NSLOT;
              slot = pos - wraps * C::NSLOT;
              ring_parity ^= (uint32_t)(wraps & 1);
            }
            cbar();
#pragma unroll 1
            for (int i = warp; i < mine * 2; i += NWARPS) {  // the sets (eight lanes per eight channels of a sample), all-gather
              const int k = lane & 7, c8 = (i & 1) * 4 + (lane >> 3), p = i >> 1;
              const float* mg = s_merge + (p * NWARPS + k) * 72;
              const bool has = k < sets;
              const float m_set = has ? mg[64] : -INFINITY;
              float mx = m_set;
#pragma unroll
              for (int off = 1; off < 8; off <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
              float den = 0.f, num[8];
#pragma unroll
              for (int z = 0; z < 8; ++z) num[z] = 0.f;
              if (has) {
                const float e = ex2_approx(m_set - mx);
                den = e * mg[65];
                const float4 a = *reinterpret_cast<const float4*>(mg + 8 * c8), b = *reinterpret_cast<const float4*>(mg + 8 * c8 + 4);
                num[0] = e * a.x; num[1] = e * a.y; num[2] = e * a.z; num[3] = e * a.w;
                num[4] = e * b.x; num[5] = e * b.y; num[6] = e * b.z; num[7] = e * b.w;
              }
              __syncwarp();
#pragma unroll
              for (int off = 1; off < 8; off <<= 1) {
                den += __shfl_xor_sync(0xffffffffu, den, off);
#pragma unroll
                for (int z = 0; z < 8; ++z) num[z] += __shfl_xor_sync(0xffffffffu, num[z], off);
              }
              const float inv = 1.f / den;
              if (k < CS)
                st_async4(peer_addr(sb + C::ACT + swz128(r * bl + p, c8), k), pack_bf16(num[0] * inv, num[1] * inv),
                          pack_bf16(num[2] * inv, num[3] * inv), pack_bf16(num[4] * inv, num[5] * inv), pack_bf16(num[6] * inv, num[7] * inv),
                          peer_addr(bar(B_ALL0), k));
              __syncwarp();
            }
            fence_proxy_async_global();  // the new cache rows: bulk copies read them from the next step on
          }
        } else {
          // ---------------------------------------------------------------- bias + GELU
          {  // reduce-scatter: warp w holds units 32 w .. of the cluster's 256, one sample per column
            const int unit = warp * 32 + lane;
            float* stg = reinterpret_cast<float*>(smem + C::STG) + (unit / UPC) * nb * UPC + unit % UPC;
#pragma unroll 1
            for (int b0 = 0; b0 < nb; b0 += 8) {
              float v[8];
              tmem_cols8(t_lane + b0, v);
#pragma unroll
              for (int b = 0; b < 8; ++b)
                if (b0 + b < nb) stg[(b0 + b) * UPC] = v[b];
            }
            tcgen05_fence_before();
          }
          const float4 bias0 = __ldg(reinterpret_cast<const float4*>(vec + V_B1 * D + c * UNITS + r * UPC + u8));
          const float4 bias1 = __ldg(reinterpret_cast<const float4*>(vec + V_B1 * D + c * UNITS + r * UPC + u8 + 4));
          fence_proxy_async_smem();
          cbar();
          if (tid < CS)
            copy_to_peer(peer_addr(sb + C::RECV + r * RT * UPC * 4, tid), sb + C::STG + tid * nb * UPC * 4, (uint32_t)(nb * UPC * 4),
                         peer_addr(bar(B_RECV1), tid));
          __syncwarp();
          meet(B_RECV1, lp);
#pragma unroll 1
          for (int b = fb; b < nb; b += FB) {
            const float* src = reinterpret_cast<const float*>(smem + C::RECV) + b * UPC + u8;
            float4 x = bias0, y = bias1;
#pragma unroll
            for (int k = 0; k < CS; ++k) {
              const float4 e = *reinterpret_cast<const float4*>(src + k * RT * UPC), f = *reinterpret_cast<const float4*>(src + k * RT * UPC + 4);
              x.x += e.x; x.y += e.y; x.z += e.z; x.w += e.w;
              y.x += f.x; y.y += f.y; y.z += f.z; y.w += f.w;
            }
            const float2 g0 = gelu_erf_fast2(make_float2(x.x, x.y)), g1 = gelu_erf_fast2(make_float2(x.z, x.w));
            const float2 g2 = gelu_erf_fast2(make_float2(y.x, y.y)), g3 = gelu_erf_fast2(make_float2(y.z, y.w));
            const uint32_t w0 = pack_bf16(g0.x, g0.y), w1 = pack_bf16(g1.x, g1.y), w2 = pack_bf16(g2.x, g2.y), w3 = pack_bf16(g3.x, g3.y);
            const int unit = r * UPC + u8;  // operand tile unit / 64, 16-byte piece (unit % 64) / 8
            const uint32_t off = sb + C::ACT + (unit >> 6) * (RT * 128) + swz128(b, (unit & 63) >> 3);
#pragma unroll
            for (int k = 0; k < CS; ++k) st_async4(peer_addr(off, k), w0, w1, w2, w3, peer_addr(bar(B_ALL1), k));
          }
        }
        // ------------------------------------------------------------------ output projection and this cluster's partial rows
        __syncwarp();
        if (warp == 0) {
          await_peers(B_ALL0 + mlp, lp);
          fence_proxy_async_smem();  // the tiles were written through the generic proxy
#pragma unroll 1
          for (int u = 0; u < (mlp ? 4 : 1); ++u) {
            const uint32_t w = take(u);
            tcgen05_fence_after();
            if (elect_one()) {
#pragma unroll
              for (int z = 0; z < C::MT; ++z) mma(tmem + (2 + z) * RT, w + z * 16384, sb + C::ACT + u * (RT * 128), u > 0);
              release(u);
              if (u == (mlp ? 3 : 0)) umma_commit(bar(B_OUT0 + mlp));
            }
            __syncwarp();
          }
          await(B_OUT0 + mlp, lp, TFERR_WAIT_TMEM_FULL);
          tcgen05_fence_before();
        }
        advance(mlp ? 4 : 1);
        cbar();
        if (tid == 0 && !mlp && mine > 0) mbar_arrive(bar(B_ROWS));  // every thread has fenced its new cache rows
        __syncwarp();
        tcgen05_fence_after();
        if ((warp & 3) * 32 < CW) {  // accumulator lane = column, column = sample; warps 4-7: the second output tile or half of the samples
          constexpr int NB = C::MT == 2 ? RT : RT / 2;
          const int c0 = C::MT == 2 ? 0 : (warp >> 2) * NB, m = C::MT == 2 ? warp >> 2 : 0;
          unsigned long long* out = xpart + ((size_t)c0 * HEADS + c) * D + r * CW + m * 128 + (warp & 3) * 32 + lane;
#pragma unroll 1
          for (int b0 = 0; b0 < NB && c0 + b0 < nb; b0 += 8) {
            float v[8];
            tmem_cols8(tmem + (2 + m) * RT + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(c0 + b0), v);
#pragma unroll
            for (int b = 0; b < 8; ++b)
              if (c0 + b0 + b < nb) ll_store(out + (size_t)(b0 + b) * HEADS * D, __float_as_uint(v[b]), seq);
          }
          tcgen05_fence_before();
        }
        __syncwarp();
      }
      // ==================================================================== head and update of the own rows
      const int bad = *reinterpret_cast<volatile int*>(err);  // looked at when the next step begins
      if (own > 0) {
        constexpr int KO = N1 == 4 ? 2 : 4;
        const int n2 = 2 * Dt, hs = tid & 7, og = tid >> 3;
        if (tid == 0 && alive) mbar_arrive_expect_tx(bar(B_HEAD), (uint32_t)(CS * own * n2 * 4));
        __syncwarp();
        float v_first = 0.f;  // operands of this thread's value of the first row: requested before the head is done
        float2 b_first = make_float2(0.f, 0.f);
        if (tid < Dt) {
          v_first = job.v[token_at(0, t + 1) + tid];
          b_first = __ldg(reinterpret_cast<const float2*>(job.b_out + 2 * tid));
        }
#pragma unroll 1
        for (int n0 = 0; n0 < n2; n0 += 32 * KO) {  // eight lanes share an output, KO outputs per lane group
          uint4 w[KO][N1];
#pragma unroll
          for (int k = 0; k < KO; ++k)
#pragma unroll
            for (int z = 0; z < N1; ++z) {
              const int n = n0 + k * 32 + og;
              w[k][z] = make_uint4(0u, 0u, 0u, 0u);
              if (n < n2) w[k][z] = __ldg(reinterpret_cast<const uint4*>(job.w_out + (size_t)n * D + r * CW + z * 64 + hs * 8));
            }
#pragma unroll 1
          for (int row = 0; row < own; ++row) {
            float acc[KO];
#pragma unroll
            for (int k = 0; k < KO; ++k) acc[k] = 0.f;
#pragma unroll
            for (int z = 0; z < N1; ++z) {
              const float4 x0 = *reinterpret_cast<const float4*>(s_xn + row * CW + z * 64 + hs * 8);
              const float4 x1 = *reinterpret_cast<const float4*>(s_xn + row * CW + z * 64 + hs * 8 + 4);
#pragma unroll
              for (int k = 0; k < KO; ++k) {
                const __nv_bfloat162* w2 = reinterpret_cast<const __nv_bfloat162*>(&w[k][z]);
                const float2 c0 = __bfloat1622float2(w2[0]), c1 = __bfloat1622float2(w2[1]);
                const float2 c2 = __bfloat1622float2(w2[2]), c3 = __bfloat1622float2(w2[3]);
                acc[k] = fmaf(x0.x, c0.x, acc[k]); acc[k] = fmaf(x0.y, c0.y, acc[k]);
                acc[k] = fmaf(x0.z, c1.x, acc[k]); acc[k] = fmaf(x0.w, c1.y, acc[k]);
                acc[k] = fmaf(x1.x, c2.x, acc[k]); acc[k] = fmaf(x1.y, c2.y, acc[k]);
                acc[k] = fmaf(x1.z, c3.x, acc[k]); acc[k] = fmaf(x1.w, c3.y, acc[k]);
              }
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
#pragma unroll
              for (int k = 0; k < KO; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
            if (hs < CS) {
              const uint32_t dst = peer_addr(sb + C::RECV + ((r * C::RPC + row) * n2 + n0 + og) * 4, hs), pbar = peer_addr(bar(B_HEAD), hs);
#pragma unroll
              for (int k = 0; k < KO; ++k)
                if (n0 + k * 32 + og < n2) st_async1(dst + k * 128, acc[k], pbar);
            }
            __syncwarp();
          }
        }
        meet(B_HEAD, (uint32_t)(t & 1));
#pragma unroll 1
        for (int row = 0; row < own; ++row) {
          const size_t e = token_at(row, t + 1);
#pragma unroll 1
          for (int cc = tid; cc < Dt; cc += NTHREADS) {
            const bool pre = cc == tid;
            const float vv = pre && row == 0 ? v_first : job.v[e + cc];
            float2 o = pre ? b_first : __ldg(reinterpret_cast<const float2*>(job.b_out + 2 * cc));  // (mu~, alpha~) of value cc
#pragma unroll
            for (int k = 0; k < CS; ++k) {
              const float2 y = *reinterpret_cast<const float2*>(smem + C::RECV + ((k * C::RPC + row) * n2 + 2 * cc) * 4);
              o.x += y.x;
              o.y += y.y;
            }
            const float x = fmaf(vv, expf(o.y), o.x);  // Eq. 5
            s_tok[row * Dt + cc] = x;
            if (r == 0) job.u[e + cc] = x;
          }
        }
      }
      if (tid == 0) *s_bad = bad;
    }
  }

  // every copy into this CTA has been waited for; the cluster meets before anyone leaves
  tcgen05_fence_before();
  __syncthreads();
  if (warp == 1 && *reinterpret_cast<volatile int*>(err) != 0) {  // a wait gave up: let copies and MMAs in flight drain
    unsigned long long t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
  }
  cluster_sync();
  if (warp == 1) {
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM) : "memory");
  }
}

}  // namespace seqp
