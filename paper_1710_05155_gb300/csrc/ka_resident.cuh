// ka_resident.cuh -- sweeps of small lattices and graphs that stay on chip.
//
// A word (64 replicas) of a small topology fits in the shared memory of one
// SM, so one launch runs all the sweeps of a call on it: the n plane is read
// once, every bond class works on shared memory, and n is written back at the
// end.  Per-class launches of such sizes are bound by the launch itself
// (about 2 us each, 6 to 20 per sweep) and by the tens of CTAs they fill.
//
// A word is run by a thread-block cluster of C CTAs.  Every CTA keeps its own
// copy of n; the bonds of a class group are dealt out to the CTAs, which read
// their own copy and send the sites that they may change to all the others
// (st.async into distributed shared memory).  A CTA's group ends when its own
// warps have arrived at its mbarrier and the other CTAs' bytes, a fixed number
// per group, have come in; no cluster barrier and no fence is needed (a
// releasing cluster barrier alone took 400-600 cycles a group).  The sites a
// CTA sends in a group are read in that group by no other CTA (a cubic group
// reads its own pencils and the inactive ones; a graph class is a strong
// matching), and a CTA starts a group only when all others have finished
// reading for the one before (each sends at least a word in every group), so
// two mbarriers in turn are enough.  The Philox
// gate words depend on no state: those of the next group are computed between
// arriving at the barrier and waiting for it.
//
// p is not read: the bits that swaps clear are collected in shared memory
// (cubic: per site; graphs: per bond) and cleared in p by one atomic AND per
// word at the end; where a lattice leaves no room for that, at each swap.
// They are collected outside the group ends, while the others' words are
// awaited: a graph's by the bond's own thread, a lattice's by whichever thread
// has the site in the group, with a CTA barrier at the end of each sweep.
#pragma once

#include "ka_internal.cuh"

namespace ka {
namespace resident {

constexpr size_t kSmemMax = 227 * 1024;
constexpr int kMaxCluster = 8;  // the portable cluster size
constexpr int64_t kMaxSweeps = 4096;  // sweeps per launch (a bound on one kernel's run time)
#ifndef KA_WAIT_POLLS  // test builds: 0, so that every wait runs out
#define KA_WAIT_POLLS (1 << 20)
#endif

// One word of one job: its plane base (element i of word h is n[i * stride]),
// the sweeps to run (count of them from t_base), and for graphs the packed bonds.
struct Unit {
  uint64_t* n;
  uint64_t* p;
  const uint4* rec;      // graphs: per bond u, v and their other neighbours (16 bit each)
  const uint32_t* bid;   // graphs: canonical bond ids, class order
  const int32_t* coff;   // graphs: first bond of every class
  int* err;              // set if a wait ran out: device memory, or a batch's page-locked word
  int32_t N, nclass, stride;
  uint32_t t_base, count, word;
  RoundKeys rk;
};

struct Args {
  Unit one;            // single job: word 0's unit
  const Unit* units;   // batched: one entry per word of every job, else null
  size_t plane_elems;  // single job
  int words_per_plane;
  uint32_t from, most; // run at most `most` of a unit's sweeps, from this one on
  int L;               // cubic
  int fsmem;           // cubic: the swapped bits are collected in shared memory
  int fslots, entries; // graphs: the words of the swapped bits; entries of a buffer
};

// threads of a CTA that has one C-th of a cubic lattice's pencils: a thread per
// segment, in whole rows per warp for mu = 0.  A CTA takes an even number of
// pencils, so that lane pairs hold neighbouring pencils of one half-row.
KA_HD constexpr int share_of(int pencils, int C) { return (pencils + 2 * C - 1) / (2 * C) * 2; }
inline int cubic_threads(int64_t N, int L, int C) {
  const int pc = share_of((int)(N / L / 2), C), pw = 32 / (L / 4);
  const int rows = (pc + pw - 1) / pw * 32, pencils = (pc * (L / 4) + 31) / 32 * 32;
  return rows > pencils ? rows : pencils;
}

// CTAs per word for `words` words of a cubic lattice (d, L) in one launch, or
// 0 when the lattice does not run here.
int cubic_cluster(int d, int L, int64_t words, int sms);
// whether n sweeps of `planes` one-word planes take less time on chip (C CTAs per
// word) than with a launch per group
bool cubic_pays(int d, int L, int64_t planes, int C, int sms, int64_t n);
cudaError_t launch_cubic(const Args& a, int d, int L, int m, unsigned words, int C,
                         cudaStream_t st);
// whether a graph of N sites may run here, and its CTAs per word (0: it does not)
bool graph_fits(int64_t N);
int graph_cluster(int64_t N, int64_t nbonds, int64_t class_max);
bool graph_pays(int64_t N, int z, int64_t nclass, int64_t words, int C, int sms, int64_t n);
// the packed record of every bond, from tables in storage positions
int graph_record_bytes(int z);
void graph_records(int64_t N, int z, const int32_t* nbr, const int32_t* bu, const int32_t* bv,
                   int64_t nbonds, uint16_t* rec);
// Nmax, bonds_max, class_max: the most sites, bonds and bonds of a class of the launch's units
cudaError_t launch_graph(const Args& a, int64_t Nmax, int64_t bonds_max, int64_t class_max, int z,
                         int m, unsigned words, int C, cudaStream_t st);
constexpr int kMaxClasses = 128;  // a greedy strong edge colouring needs at most 2 z (z - 1) + 1

// ---------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------
#ifdef KA_RESIDENT_DEVICE
namespace {

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// The end of a group (above).  bars: two mbarriers of this CTA, one arrival per
// warp.  A wait that runs out marks the context's error word (the result is not
// valid) and the CTA goes on without waits to the end of the sweep, where it
// leaves: no further, since nothing then bounds the bytes that an mbarrier has
// yet to see (at most 2^20 - 1; a sweep's are 290 KB at most), and the others
// then run out of their waits too.
struct GroupEnd {
  uint32_t bars;
  uint32_t phase;  // groups done
  bool dead;
  __device__ __forceinline__ uint32_t bar() const { return bars + 8u * (phase & 1u); }
  __device__ __forceinline__ void arrive(uint32_t bytes) const {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
      if (threadIdx.x == 0)
        asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(bar()), "r"(bytes)
                     : "memory");
      else
        asm volatile("mbarrier.arrive.shared.b64 _, [%0];" ::"r"(bar()) : "memory");
    }
  }
  __device__ __forceinline__ void wait(int* err) {
    const uint32_t parity = (phase >> 1) & 1u;
    uint32_t done = 0;
    for (int i = 0; i < KA_WAIT_POLLS && !done && !dead; ++i)
      asm volatile(
          "{\n.reg .pred q;\n"
          "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 q, [%1], %2;\n"
          "selp.u32 %0, 1, 0, q;\n}"
          : "=r"(done)
          : "r"(bar()), "r"(parity)
          : "memory");
    if (!done && !dead) {
      dead = true;
      *reinterpret_cast<volatile int*>(err) = 1;
    }
    ++phase;
  }
};

// the other C - 1 CTAs' copies of this CTA's shared memory: what has address x
// here has address x + delta there; a store counts its bytes at the receiver's
// mbarrier of the same place
template <int C>
struct Peers {
  uint32_t delta[C > 1 ? C - 1 : 1];
  __device__ __forceinline__ Peers(uint32_t addr, uint32_t rank) {
#pragma unroll
    for (uint32_t c = 1; c < C; ++c) delta[c - 1] = peer_addr(addr, (rank + c) % C) - addr;
  }
  __device__ __forceinline__ void st(uint32_t addr, uint64_t v, uint32_t bar) const {
#pragma unroll
    for (int c = 0; c < C - 1; ++c)
      asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(
                       addr + delta[c]),
                   "l"(v), "r"(bar + delta[c])
                   : "memory");
  }
  __device__ __forceinline__ void st2(uint32_t addr, uint64_t v, uint64_t w, uint32_t bar) const {
#pragma unroll
    for (int c = 0; c < C - 1; ++c)
      asm volatile(
          "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(
              addr + delta[c]),
          "l"(v), "l"(w), "r"(bar + delta[c])
          : "memory");
  }
};

__device__ __forceinline__ void clear_bits(uint64_t* p, uint64_t sw) {
  if (sw) atomicAnd(reinterpret_cast<unsigned long long*>(p), (unsigned long long)~sw);
}

// this CTA's unit: the single job's word, or its table entry
template <bool B>
__device__ __forceinline__ void unit_of(const Args& a, uint32_t w, Unit& su) {
  if constexpr (B) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(a.units + w);
    for (uint32_t k = threadIdx.x; k < sizeof(Unit) / 4; k += blockDim.x)
      reinterpret_cast<uint32_t*>(&su)[k] = src[k];
  } else if (threadIdx.x == 0) {
    su = a.one;
    const uint32_t q = w / (uint32_t)a.words_per_plane, h = w % (uint32_t)a.words_per_plane;
    su.n += (size_t)q * a.plane_elems + h;
    su.p += (size_t)q * a.plane_elems + h;
    su.word = w;
  }
  __syncthreads();
}

template <bool B>
__device__ __forceinline__ const RoundKeys& unit_keys(const Args& a, const Unit& su) {
  if constexpr (B) return su.rk;
  else return a.one.rk;
}

// the plane into this CTA's copy (contiguous planes in 16-byte pieces)
__device__ __forceinline__ void load_plane(const Unit& su, uint64_t* n, int N) {
  if (su.stride == 1 && N % 2 == 0) {
    const ulonglong2* g = reinterpret_cast<const ulonglong2*>(su.n);
    ulonglong2* s = reinterpret_cast<ulonglong2*>(n);
#pragma unroll 4
    for (int i = threadIdx.x; i < N / 2; i += blockDim.x) s[i] = g[i];
  } else {
#pragma unroll 4
    for (int i = threadIdx.x; i < N; i += blockDim.x) n[i] = su.n[(size_t)i * su.stride];
  }
}

// write back: every CTA its share of n
__device__ __forceinline__ void store_plane(const Unit& su, const uint64_t* n, int N, uint32_t rank,
                                            uint32_t size) {
  for (int i = (int)(rank * blockDim.x + threadIdx.x); i < N; i += (int)(size * blockDim.x))
    su.n[(size_t)i * su.stride] = n[i];
}

// most: the largest smem of any launch of the kernel.  The attribute belongs to the
// kernel, not to the launch: always the same value, so that host threads whose
// launches want different amounts do not take it from each other.
template <typename Kern>
cudaError_t launch_cluster(Kern kern, const Args& a, unsigned words, int C, int threads, size_t smem,
                           size_t most, cudaStream_t st) {
  const cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(words * (unsigned)C);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

}  // namespace
#endif

}  // namespace resident
}  // namespace ka
