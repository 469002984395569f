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
// refills what has been used); where a block's weights exceed L2 they (and the next layer's cache rows) are prefetched into
// L2 a layer ahead.  A step's head, update and embedding are done by the row's owner cluster on the CUDA cores.
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
  const float *ln1_g, *ln1_b, *b_qkv, *b_o, *ln2_g, *ln2_b, *b_1, *b_2;
};
struct Job {
  const Layer* layers;
  const float *lnf_g, *lnf_b, *w_in_t, *b_in, *pos, *cls, *b_out, *v;
  const bf16* w_out;
  float* u;
  const int* labels;
  bf16 *kc, *vc;
  size_t layer_stride;              // cache elements per layer
  unsigned long long *xpart, *xrow; // exchange buffers
  int n_layers, B, rows, L, Dt, reversed;  // rows: samples per group (a group = one set of clusters); Dt: token dimension
  uint32_t seq0;
  int prefetch_w, prefetch_kv;
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
  static constexpr int NSLOT_MAX = (RT == 16 ? 163840 : 131072) / UNIT, NSLOT = NSLOT_MAX < 12 ? NSLOT_MAX : 12;
  static constexpr int MAXDT = D == 1024 ? 256 : 128;
  static constexpr int RING = 0, ACT = NSLOT * UNIT;  // activation tiles; a 64-row weight tile read as 128 rows may run on into them
  static constexpr int STG = ACT + 4 * RT * 128;      // what is sent to the peers, then what comes from them
  static constexpr int RECV = STG + RT * 1024;
  static constexpr int MERGE = RECV;                  // [sample][warp]: output, maximum, sum; q, k, v have left the place by then
  static constexpr int QKV = RECV + (RT * 1024 > BL * NWARPS * 288 ? RT * 1024 : BL * NWARPS * 288);  // per sample: q fp32 [64], k, v bf16 [64]
  static constexpr int SUM = QKV + BL * 512;
  static constexpr int XN = SUM + (SGC - 1) * RPC * QN * 16;
  static constexpr int TOK = XN + RPC * CW * 4;
  static constexpr int STAT = TOK + RPC * MAXDT * 4;
  static constexpr int BIAS = STAT + RPC * NE * 8;
  static constexpr int BARS = BIAS + 192 * 4;
  static constexpr int NBARS = 2 * NSLOT + 10;
  static constexpr int TOTAL = BARS + NBARS * 8 + 32 + 1024;
  static constexpr uint32_t TMEM = RT == 16 ? 64 : 128;
  static_assert(sizeof(Layer) % sizeof(CUtensorMap) == 0, "tables of layers are stepped in tensor maps");
  static_assert(QN * RPC * SG == NTHREADS && SG * NSL == HEADS && NSL % NA == 0 && SGC > 1 && QN * RPC % 32 == 0 && NSLOT >= 4,
                "thread layout of the residual rows");
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
__device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, int* err, int code) { return mbar_wait(bar, parity, err, code); }
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, int* err, int code) {
  return mbar_try_wait(bar, parity) || wait_slow(bar, parity, err, code);
}
// the same for a warp that waits while others work: it sleeps between polls
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
    if (dt > WAIT_LIMIT_NS) {
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
struct Spin {  // bound of a polling loop
  unsigned n = 0;
  unsigned long long t0 = 0;
  __device__ __noinline__ bool check(int* err) {
    if (*reinterpret_cast<volatile int*>(err) != 0) return false;
    const unsigned long long now = globaltimer_ns();
    if (n == 256u) t0 = now;
    if (now - t0 <= WAIT_LIMIT_NS) return true;
    atomicCAS(err, 0, TFERR_WAIT_FULL);
    return false;
  }
  __device__ __forceinline__ bool more(int* err) { return (++n & 255u) != 0 || check(err); }
};

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
__device__ __forceinline__ void prefetch_tile(const CUtensorMap* map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(map), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void prefetch_bytes(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ void prefetch_line(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p) : "memory"); }
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 o = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&o);
}

// The weight ring's filling side (one thread): where it stands in the order of use.
struct Feed {
  int t = 0, layer = 0, unit = 0, slot = 0;
  uint32_t phase = 0;
};
// requests one unit after the other (a layer is 12 of them), each when the products that read its slot's last contents are done
template <int D, int RT>
__device__ __forceinline__ void feed(const Job& job, Feed& f, uint32_t ring, uint32_t bars, int r, int c, bool prefetch_w, int mine,
                                     size_t cache_row0) {
  using C = Cfg<D, RT>;
  constexpr int N1 = C::N1, CW = C::CW;
  const int n_steps = job.L - 1;
#pragma unroll 1
  while (f.t < n_steps) {
    if (!wait_idle(bars + 8u * (C::NSLOT + f.slot), f.phase ^ 1u, job.err, TFERR_WAIT_EMPTY)) return;
    const Layer* ly = job.layers + f.layer;
    const int nx = f.layer + 1 < job.n_layers ? f.layer + 1 : 0;
    const bool more = nx > 0 || f.t + 1 < n_steps;
    const uint32_t full = bars + 8u * f.slot;
    mbar_arrive_expect_tx(full, C::UNIT);
    const int u = f.unit;
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
      tma_load_2d(ring + f.slot * C::UNIT + z * 8192, map, x, y, full);
      if (prefetch_w && more) prefetch_tile(map + (nx - f.layer) * (int)(sizeof(Layer) / sizeof(CUtensorMap)), x, y);
    }
    if (u == 4 && job.prefetch_kv && more && f.t > 0)
      for (int p = 0; p < mine; ++p) {
        const size_t at = nx * job.layer_stride + cache_row0 + (size_t)p * C::HEADS * job.L * HD;
        prefetch_bytes(job.kc + at, (uint32_t)f.t * HD * 2);
        prefetch_bytes(job.vc + at, (uint32_t)f.t * HD * 2);
      }
    if (++f.slot == C::NSLOT) { f.slot = 0; f.phase ^= 1u; }
    if (++f.unit == 12) {
      f.unit = 0;
      f.layer = nx;
      if (nx == 0) ++f.t;
    }
  }
}
