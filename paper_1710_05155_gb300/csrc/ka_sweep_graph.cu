// ka_sweep_graph.cu -- edge-gather sweep kernel for one bond class.
//
// One thread per (bond of the class, word): the bond (u, v) gathers its word
// of u, v and of their other neighbours from the int32 neighbour list, counts
// the occupied neighbours of u other than v and of v other than u with
// bit-sliced adders (64 replicas per word), and applies the exchange rule of
// section 2.1 (rules (a)-(c)) under the replica's Philox gate bit.  Bonds of a
// class form a strong matching, so bonds never touch each other's sites.
//
// A plane holds V = 1, 2 or 4 words per site, so a site's words share one
// 32-byte sector: every gather is a random access, and the sector is the
// unit the memory system moves.  The V words of a bond are V neighbouring
// lanes, whose accesses to a site fall into its sector together; one thread
// with all V words needed 110 registers (22 % of the warps) and V separate
// atomics per site.  Blocks are small: what bounds the gathers is sectors in
// flight and their reuse in the L1, and fewer, larger blocks (or more warps by
// fewer registers) lose the reuse: 2^20 sites, 512 replicas 320 us a sweep with
// 128 threads, 341 with 256, 395 with 1024, 376 with 5 instead of 4 blocks of
// 256.  us a sweep, z = 4, m = 2, before and after: 2^20 sites 512 replicas 623,
// 320; 256 replicas 301, 165; 2^17 256 replicas 117, 41; one word 2^15 47, 32;
// 2^17 60, 45; 2^20 160, 135.
// The partner's word is not gathered twice, and p is never read: the bits of
// p that a swap clears are cleared by an atomic AND in the L2.
// A thread first loads what depends only on static tables (its bond, the
// two neighbour rows) and computes the gate word, then gathers the state.
// Single-instance class launches are chained with programmatic dependent
// launch, so that this prologue overlaps the previous class's tail (small
// graphs are bound by launch latency); batched launches are not, since a
// grid waiting on the SMs slows the one it waits for.
#include "ka_internal.cuh"

namespace ka {
namespace {

struct ClassArgs {
  uint64_t* n;
  uint64_t* p;
  const int32_t* nbr;
  const int32_t* bu;
  const int32_t* bv;
  const uint32_t* bid;
  size_t plane_elems;
  int64_t count;
  int z;
  int q0;  // first plane of the launch
  uint32_t t, cls;
  uint32_t pair_stride;  // cubic lattices: stride of the bond direction, 0 on graphs
  RoundKeys rk;
};

// (c2 c1 c0) += x, bit-sliced; the count stays below 8 (at most 7 inputs)
__device__ __forceinline__ void add3(uint64_t& c2, uint64_t& c1, uint64_t& c0, uint64_t x) {
  const uint64_t k0 = c0 & x;
  c0 ^= x;
  const uint64_t k1 = c1 & k0;
  c1 ^= k0;
  c2 |= k1;
}

template <int T>
__device__ __forceinline__ uint64_t le3(uint64_t b2, uint64_t b1, uint64_t b0) {
  if constexpr (T < 0) {
    return 0ull;
  } else if constexpr (T >= 7) {
    return ~0ull;
  } else {
    const uint64_t g0 = (T & 1) ? 0ull : b0;
    const uint64_t g1 = (T & 2) ? (b1 & g0) : (b1 | g0);
    const uint64_t g2 = (T & 4) ? (b2 & g1) : (b2 | g1);
    return ~g2;
  }
}

constexpr int kMaxZ = 8;
constexpr int kThreads = 128;

// neighbour row of x (z <= 8); z = 4 rows are one 16-byte load
__device__ __forceinline__ void load_row(const int32_t* nbr, int z, int32_t x,
                                         int32_t (&r)[kMaxZ]) {
  if (z == 4) {
    const int4 q = *reinterpret_cast<const int4*>(nbr + (int64_t)x * 4);
    r[0] = q.x;
    r[1] = q.y;
    r[2] = q.z;
    r[3] = q.w;
  } else {
#pragma unroll
    for (int k = 0; k < kMaxZ; ++k)
      if (k < z) r[k] = nbr[(int64_t)x * z + k];
  }
}

// Graph gate stream: word w of bond id takes half w mod 2 of the block
// (t, class, id, w / 2).
__device__ __forceinline__ uint64_t graph_gate(uint32_t t, uint32_t cls, uint32_t id, uint32_t w,
                                               const RoundKeys& rk) {
  const uint4 b = philox(make_uint4(t, cls, id, w >> 1), rk);
  return (w & 1u) ? hi64(b) : lo64(b);
}

// The exchange on bond (u, v) for one word of a plane (np and pp at that
// word): counts of the other neighbours of u and of v, the rule, the gated
// swap, and the persistence update.
template <int V, int M>
__device__ __forceinline__ void exchange(uint64_t* np, uint64_t* pp, int z, int32_t u, int32_t v,
                                         const int32_t (&ru)[kMaxZ], const int32_t (&rv)[kMaxZ],
                                         uint64_t g) {
  const uint64_t nu = np[(int64_t)u * V], nv = np[(int64_t)v * V];
  uint64_t xu[kMaxZ], xv[kMaxZ];
#pragma unroll
  for (int k = 0; k < kMaxZ; ++k) {
    if (k < z) {  // the partner is not one of the "other" neighbours
      xu[k] = ru[k] != v ? np[(int64_t)ru[k] * V] : 0ull;
      xv[k] = rv[k] != u ? np[(int64_t)rv[k] * V] : 0ull;
    }
  }
  uint64_t cu2 = 0, cu1 = 0, cu0 = 0, cv2 = 0, cv1 = 0, cv0 = 0;
#pragma unroll
  for (int k = 0; k < kMaxZ; ++k) {
    if (k < z) {
      add3(cu2, cu1, cu0, xu[k]);
      add3(cv2, cv1, cv0, xv[k]);
    }
  }
  const uint64_t sw = (nu ^ nv) & g & le3<M>(cu2, cu1, cu0) & le3<M>(cv2, cv1, cv0);
  if (sw) {
    np[(int64_t)u * V] = nu ^ sw;
    np[(int64_t)v * V] = nv ^ sw;
    // Persistence: an atomic AND performed in the L2 (no reply), not a load
    // of p after the swap is known and a store: random gathers are bound by
    // the misses an SM keeps in flight, and this removes two of them per bond
    // and a dependent round trip.
    atomicAnd(reinterpret_cast<unsigned long long*>(pp + (int64_t)u * V), (unsigned long long)~sw);
    atomicAnd(reinterpret_cast<unsigned long long*>(pp + (int64_t)v * V), (unsigned long long)~sw);
  }
}

template <int V, int M, int MINB>
__global__ void __launch_bounds__(kThreads, MINB) k_graph_class(const __grid_constant__ ClassArgs a) {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t e = i / V;
  const int h = (int)(i % V);
  if (e >= a.count) return;
  const int q = a.q0 + (int)blockIdx.y;
  const int32_t u = a.bu[e], v = a.bv[e];
  const uint32_t id = a.bid[e];
  int32_t ru[kMaxZ], rv[kMaxZ];
  load_row(a.nbr, a.z, u, ru);
  load_row(a.nbr, a.z, v, rv);
  // gate word.  Graphs: the graph stream.  Cubic lattices on this path:
  // bonds of classes 4g+2b and 4g+2b+1 that start at neighbouring pencil
  // positions share the block (t, 4g+2b, base site of the first, word),
  // half = class parity.
  const uint32_t w = (uint32_t)(q * V + h);
  uint64_t g;
  if (a.pair_stride != 0) {
    const uint32_t odd = a.cls & 1u;
    const uint4 b = philox(make_uint4(a.t, a.cls - odd, id - odd * a.pair_stride, w), a.rk);
    g = odd ? hi64(b) : lo64(b);
  } else {
    g = graph_gate(a.t, a.cls, id, w, a.rk);
  }
  asm volatile("griddepcontrol.wait;\n" ::: "memory");  // the previous class is complete
  exchange<V, M>(a.n + (size_t)q * a.plane_elems + h, a.p + (size_t)q * a.plane_elems + h, a.z, u, v,
                 ru, rv, g);
}

// Batched form: one launch runs class cls of every graph unit (one state plane
// of one job); block b takes the bonds that blocks[b] says, up to
// kGraphBlock / V of one unit.  Units whose sweep counter reached t_end skip.
template <int V, int M>
__global__ void __launch_bounds__(kGraphBlock) k_graph_class_batch(const GraphUnit* __restrict__ units,
                                                           const GraphBlock* __restrict__ blocks,
                                                           uint32_t cls, uint32_t sweep_offset) {
  __shared__ GraphUnit gu;
  const GraphBlock b = blocks[blockIdx.x];
  const uint32_t* src = reinterpret_cast<const uint32_t*>(units + b.unit);
  if (threadIdx.x < sizeof(GraphUnit) / 4) reinterpret_cast<uint32_t*>(&gu)[threadIdx.x] = src[threadIdx.x];
  const int e = (int)threadIdx.x / V, h = (int)threadIdx.x % V;
  __syncthreads();
  const uint32_t t = gu.t_base + sweep_offset;
  if (t >= gu.t_end || e >= b.count) return;
  const int64_t k = (int64_t)b.first + e;
  const int32_t u = gu.bu[k], v = gu.bv[k];
  const uint32_t id = gu.bid[k];
  int32_t ru[kMaxZ], rv[kMaxZ];
  load_row(gu.nbr, gu.z, u, ru);
  load_row(gu.nbr, gu.z, v, rv);
  const uint64_t g = graph_gate(t, cls, id, gu.word0 + (uint32_t)h, gu.rk);
  exchange<V, M>(gu.n + h, gu.p + h, gu.z, u, v, ru, rv, g);
}

// single-instance launch with programmatic stream serialisation
template <typename Kern>
cudaError_t launch_pdl(Kern kern, dim3 grid, cudaStream_t s, const ClassArgs& a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int V, int MINB>
cudaError_t launch_v(const ClassArgs& a, int m, dim3 grid, cudaStream_t s) {
  switch (m < 7 ? m : 7) {
#define KA_CASE(MM) \
  case MM:          \
    return launch_pdl(k_graph_class<V, MM, MINB>, grid, s, a);
    KA_CASE(0)
    KA_CASE(1)
    KA_CASE(2)
    KA_CASE(3)
    KA_CASE(4)
    KA_CASE(5)
    KA_CASE(6)
    KA_CASE(7)
#undef KA_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

template <int V>
cudaError_t launch_batch_v(const GraphUnit* units, const GraphBlock* blocks, unsigned nblocks, int m,
                           uint32_t cls, uint32_t off, cudaStream_t s) {
  switch (m < 7 ? m : 7) {
#define KA_CASE(MM)                                                               \
  case MM:                                                                        \
    k_graph_class_batch<V, MM><<<nblocks, kGraphBlock, 0, s>>>(units, blocks, cls, off); \
    return cudaGetLastError();
    KA_CASE(0)
    KA_CASE(1)
    KA_CASE(2)
    KA_CASE(3)
    KA_CASE(4)
    KA_CASE(5)
    KA_CASE(6)
    KA_CASE(7)
#undef KA_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_graph_class_batch(const GraphUnit* units_dev, const GraphBlock* blocks_dev,
                                     int64_t nblocks, int V, int m, uint32_t cls,
                                     uint32_t sweep_offset, cudaStream_t s) {
  if (nblocks <= 0) return cudaSuccess;
  if (V == 4) return launch_batch_v<4>(units_dev, blocks_dev, (unsigned)nblocks, m, cls, sweep_offset, s);
  if (V == 2) return launch_batch_v<2>(units_dev, blocks_dev, (unsigned)nblocks, m, cls, sweep_offset, s);
  if (V == 1) return launch_batch_v<1>(units_dev, blocks_dev, (unsigned)nblocks, m, cls, sweep_offset, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_graph_class(const Planes& pl, const GraphDev& g, int64_t off, int64_t count,
                               uint32_t cls, uint32_t t, const RoundKeys& rk, int q0, int nq,
                               cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  ClassArgs a;
  a.n = pl.n;
  a.p = pl.p;
  a.nbr = g.nbr;
  a.bu = g.bu + off;
  a.bv = g.bv + off;
  a.bid = g.bid + off;
  a.plane_elems = pl.plane_elems();
  a.count = count;
  a.z = g.z;
  a.t = t;
  a.cls = cls;
  a.pair_stride = 0;
  if (g.cubic_L > 0) {
    uint32_t s = 1;
    for (uint32_t k = 0; k < cls / 8; ++k) s *= (uint32_t)g.cubic_L;
    a.pair_stride = s;
  }
  a.rk = rk;
  a.q0 = q0;
  const dim3 grid((unsigned)((count * pl.V + kThreads - 1) / kThreads), (unsigned)nq);
  if (pl.V == 4) return launch_v<4, 1>(a, g.m, grid, s);
  if (pl.V == 2) return launch_v<2, 1>(a, g.m, grid, s);
  // one word: a full device wants more warps (48 registers) once the gathers
  // miss the L1 anyway.  us a sweep with 8 and 10 blocks per SM: 2^17 sites 45,
  // 47; 2^19 109, 113; 2^20 155, 135; 3 planes of 2^18 121, 125, of 2^19 203, 175.
  return (int64_t)pl.N * nq >= (1 << 20) ? launch_v<1, 10>(a, g.m, grid, s)
                                         : launch_v<1, 1>(a, g.m, grid, s);
}

}  // namespace ka
