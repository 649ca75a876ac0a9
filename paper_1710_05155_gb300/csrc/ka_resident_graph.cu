// ka_resident_graph.cu -- on-chip sweeps of small graphs (ka_resident.cuh):
// one cluster per word, one launch for all sweeps of a call.
//
// A bond's packed record holds the 16-bit positions of u, v and of their
// other neighbours (missing ones point at a word that stays 0), so a class
// needs one coalesced 16- or 32-byte load and the bond id per bond.  A thread
// takes one bond of a class; its record is loaded two classes ahead and its
// gate word computed one class ahead, while the group end is waited for.  The
// gathers of a bond are shared-memory reads.
//
// The CTAs of a cluster send a bond's swap word as one entry of a buffer in
// class order, and the receiver applies it to its copy: sent to their scattered
// sites, the new words cost about two cycles each at the receiver (N = 2^14,
// four CTAs: 3.0 us a class).
#include <algorithm>

#define KA_RESIDENT_DEVICE
#include "ka_resident.cuh"

namespace ka {
namespace resident {
namespace {

// (c2 c1 c0) += x, bit-sliced; the count stays below 8 (at most 7 inputs)
__device__ __forceinline__ void add3(uint64_t& c2, uint64_t& c1, uint64_t& c0, uint64_t x) {
  const uint64_t k0 = c0 & x;
  c0 ^= x;
  const uint64_t k1 = c1 & k0;
  c1 ^= k0;
  c2 |= k1;
}

// [count <= M] of Z - 1 words at the given positions
template <int Z, int M>
__device__ __forceinline__ uint64_t at_most(const uint64_t* n, const uint32_t (&r)[Z], int from) {
  uint64_t c2 = 0, c1 = 0, c0 = 0;
#pragma unroll
  for (int k = 0; k < Z - 1; ++k) {
    const int e = from + k;
    add3(c2, c1, c0, n[(r[e >> 1] >> (16 * (e & 1))) & 0xFFFFu]);
  }
  if constexpr (M >= Z - 1) {
    return ~0ull;
  } else {
    const uint64_t g0 = (M & 1) ? 0ull : c0;
    const uint64_t g1 = (M & 2) ? (c1 & g0) : (c1 | g0);
    return ~((M & 4) ? (c2 & g1) : (c2 | g1));
  }
}

// Z = 4 (records of 16 bytes, z <= 4) or 8 (32 bytes)
template <int Z, int M, int C, bool B>
__global__ void __launch_bounds__(1024) k_resident_graph(const __grid_constant__ Args a) {
  constexpr int RW = Z / 4;  // 16-byte pieces of a record
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ Unit su;
  // class c: bonds [coff[c], coff[c + 1]), share[c] of them per CTA at most, idle[c]
  // CTAs without any; the swapped bits of this CTA's are kept from slot[c] on
  __shared__ int32_t coff[kMaxClasses + 1], share[kMaxClasses], slot[kMaxClasses], idle[kMaxClasses];
  __shared__ __align__(8) uint64_t bars[2];
  const uint32_t rank = cluster_rank();
  unit_of<B>(a, blockIdx.x / C, su);
  uint32_t t = su.t_base + a.from, left_to_run = su.count > a.from ? min(su.count - a.from, a.most) : 0u;
  if (left_to_run == 0) return;  // the whole cluster: one unit
  const int N = su.N, nclass = su.nclass, tid = threadIdx.x;
  // two entry buffers (C > 1), n, the swapped bits of this CTA's bonds
  uint64_t* buf = reinterpret_cast<uint64_t*>(dsm);
  uint64_t* n = buf + 2 * a.entries;
  uint64_t* f = n + N + 2;
  const Peers<C> peers(smem_addr(dsm), rank);
  GroupEnd ge{smem_addr(bars), 0u, false};
  if (tid < 2) bar_init(ge.bars + 8 * tid, blockDim.x / 32);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  for (int c = tid; c <= nclass; c += blockDim.x) {
    coff[c] = su.coff[c];
    if (c < nclass) {
      const int count = su.coff[c + 1] - su.coff[c];
      share[c] = (count + C - 1) / C;
      idle[c] = C - (count + share[c] - 1) / share[c];
    }
  }
  load_plane(su, n, N);
  if (tid == 0) n[N] = 0;  // the word of missing neighbours
  __syncthreads();
  if (tid == 0) {
    int at = 0;
    for (int c = 0; c < nclass; ++c) {
      slot[c] = at;
      at += share[c];
    }
  }
  for (int i = tid; i < a.fslots; i += blockDim.x) f[i] = 0;
  // how many bonds of class c CTA r has, and their first
  auto first = [&](int c, int r) { return coff[c] + r * share[c]; };
  auto mine = [&](int c, int r) {
    return max(0, min(share[c], coff[c + 1] - first(c, r)));
  };

  const uint32_t word = su.word;
  uint32_t r[Z], rn[Z], id = 0;  // the records of this class and the next, the next one's id
  uint32_t uv[C > 1 ? C - 1 : 1];  // the ends of the bonds whose entries this thread puts in place
  uint64_t g = 0;
  bool live = false, live_n = false;
  auto fetch = [&](int c) {  // the record and id of this thread's bond of class c
    live_n = tid < mine(c, (int)rank);
    if (live_n) {
      const int k = first(c, (int)rank) + tid;
      const uint4* src = su.rec + (size_t)RW * k;
#pragma unroll
      for (int h = 0; h < RW; ++h) {
        const uint4 x = __ldg(src + h);
        rn[4 * h] = x.x;
        rn[4 * h + 1] = x.y;
        rn[4 * h + 2] = x.z;
        rn[4 * h + 3] = x.w;
      }
      id = __ldg(su.bid + k);
    }
  };
  auto ends = [&](int c) {  // entry tid of every other CTA's share of class c
#pragma unroll
    for (int d = 0; d < C - 1; ++d) {
      const int o = (int)((rank + 1 + d) % C);
      if (tid < mine(c, o))
        uv[d] = __ldg(reinterpret_cast<const uint32_t*>(su.rec + (size_t)RW * (first(c, o) + tid)));
    }
  };
  // the fetched class c becomes the current one: its gate words; the next is fetched
  auto turn = [&](uint32_t tt, int c) {
    live = live_n;
#pragma unroll
    for (int h = 0; h < Z; ++h) r[h] = rn[h];
    const uint32_t e = id;
    fetch(c + 1 < nclass ? c + 1 : 0);
    const uint4 b = philox(make_uint4(tt, (uint32_t)c, e, word >> 1), unit_keys<B>(a, su));
    g = (word & 1u) ? hi64(b) : lo64(b);
  };
  cluster_arrive();
  fetch(0);
  turn(t, 0);
  ends(0);
  cluster_wait();
  for (; left_to_run; --left_to_run, ++t) {
#pragma unroll 1
    for (int c = 0; c < nclass; ++c) {
      uint64_t sw = 0;
      const int u = (int)(r[0] & 0xFFFFu), v = (int)(r[0] >> 16);
      uint64_t* in = buf + (ge.phase & 1u) * a.entries;
      const bool act = live;
      if (act) {
        const uint64_t nu = n[u], nv = n[v];
        sw = (nu ^ nv) & g & at_most<Z, M>(n, r, 2) & at_most<Z, M>(n, r, 2 + Z - 1);
        n[u] = nu ^ sw;
        n[v] = nv ^ sw;
        if constexpr (C > 1)
          peers.st(smem_addr(in + first(c, (int)rank) - coff[c] + tid), sw, ge.bar());
      }
      // a CTA without a bond in the class sends a word all the same: the
      // others must not run two classes ahead of it
      const int own = mine(c, (int)rank);
      if constexpr (C > 1) {
        if (own == 0 && tid == 0) peers.st(smem_addr(in + a.entries - C + (int)rank), 0ull, ge.bar());
      }
      ge.arrive((uint32_t)(coff[c + 1] - coff[c] - own + idle[c] - (own == 0)) * 8u);
      if (act) f[slot[c] + tid] |= sw;
      const int cn = c + 1 < nclass ? c + 1 : 0;
      turn(cn ? t : t + 1, cn);
      ge.wait(su.err);
      if constexpr (C > 1) {
#pragma unroll
        for (int d = 0; d < C - 1; ++d) {
          const int o = (int)((rank + 1 + d) % C);
          if (tid < mine(c, o)) {
            const uint64_t e = in[o * share[c] + tid];
            n[uv[d] & 0xFFFFu] ^= e;
            n[uv[d] >> 16] ^= e;
          }
        }
        ends(cn);
        __syncthreads();
      }
    }
    if (__syncthreads_or(ge.dead)) break;  // a wait ran out
  }
  store_plane(su, n, N, rank, C);
  for (int c = 0; c < nclass; ++c) {
    if (tid >= mine(c, (int)rank)) continue;
    const uint32_t e =
        *reinterpret_cast<const uint32_t*>(su.rec + (size_t)RW * (first(c, (int)rank) + tid));
    const uint64_t sw = f[slot[c] + tid];
    clear_bits(su.p + (size_t)(e & 0xFFFFu) * su.stride, sw);
    clear_bits(su.p + (size_t)(e >> 16) * su.stride, sw);
  }
  cluster_arrive();  // a CTA stays until the others have sent it all
  cluster_wait();
}

constexpr size_t kGraphSmem = kSmemMax - 2560;  // beside the unit and the class tables

template <int Z, int M>
cudaError_t launch_m(const Args& a, unsigned words, int C, int threads, size_t smem, cudaStream_t st) {
  const bool b = a.units != nullptr;
  switch (C) {
#define KA_C(CC)                                                                              \
  case CC:                                                                                    \
    return b ? launch_cluster(k_resident_graph<Z, M, CC, true>, a, words, CC, threads, smem,   \
                              kGraphSmem, st)                                                 \
             : launch_cluster(k_resident_graph<Z, M, CC, false>, a, words, CC, threads, smem,  \
                              kGraphSmem, st);
    KA_C(1)
    KA_C(4)
#undef KA_C
    default:
      return cudaErrorInvalidValue;
  }
}

template <int Z>
cudaError_t launch_z(const Args& a, int m, unsigned words, int C, int threads, size_t smem,
                     cudaStream_t st) {
  switch (m < Z - 1 ? m : Z - 1) {  // m >= z - 1: no constraint
#define KA_CASE(MM) \
  case MM:          \
    return launch_m<Z, (MM < Z ? MM : 0)>(a, words, C, threads, smem, st);
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

// shared memory: entry buffers, n of N sites, the swapped bits of a share of the bonds
int64_t fslots_for(int64_t nbonds, int C) { return (nbonds + C - 1) / C + kMaxClasses; }
// of a buffer: the largest class, and a place for each CTA without a bond (even:
// n stays 16-byte aligned)
int64_t entries_for(int64_t class_max, int C) { return C > 1 ? ((class_max + 1) & ~1LL) + C : 0; }
size_t smem_for(int64_t N, int64_t class_max, int64_t nbonds, int C) {
  return 2 * (size_t)entries_for(class_max, C) * 8 + (size_t)(N + 2) * 8 +
         (size_t)fslots_for(nbonds, C) * 8;
}

}  // namespace

// 16-bit positions, and the measured limit (graph_cluster)
bool graph_fits(int64_t N) { return N >= 2 && N <= 11000; }

int graph_record_bytes(int z) { return z <= 4 ? 16 : 32; }

void graph_records(int64_t N, int z, const int32_t* nbr, const int32_t* bu, const int32_t* bv,
                   int64_t nbonds, uint16_t* rec) {
  const int Z = z <= 4 ? 4 : 8;
  for (int64_t e = 0; e < nbonds; ++e) {
    uint16_t* o = rec + e * 2 * Z;
    const int32_t end[2] = {bu[e], bv[e]};
    o[0] = (uint16_t)end[0];
    o[1] = (uint16_t)end[1];
    for (int s = 0; s < 2; ++s) {
      uint16_t* q = o + 2 + s * (Z - 1);
      int at = 0;
      for (int k = 0; k < z; ++k) {
        const int32_t x = nbr[(int64_t)end[s] * z + k];
        if (x != end[s ^ 1]) q[at++] = (uint16_t)x;
      }
      while (at < Z - 1) q[at++] = (uint16_t)N;
    }
  }
}

int graph_cluster(int64_t N, int64_t nbonds, int64_t class_max) {
  // A thread per bond of a class and all tables in shared memory, on the fewest
  // CTAs that do.  us a sweep (z = 4, 1 to 8 words) with one CTA, with four, and
  // with one launch per class: N = 2^12 17, -, 26-28; 6000 -, 19, 28-31; 2^13
  // -, 21, 27-30; 10^4 -, 24, 27-30; 12 000 -, 28, 27-31; 2^14 -, 45 (no room for
  // the swapped bits; with eight CTAs 33), 27-33.
  if (!graph_fits(N)) return 0;
  for (int C : {1, 4})
    if (class_max <= 1024 * C && smem_for(N, class_max, nbonds, C) <= kGraphSmem) return C;
  return 0;
}

bool graph_pays(int64_t N, int z, int64_t nclass, int64_t words, int C, int sms, int64_t n) {
  // us, fitted.  A launch per class 1.75 (z = 1 to 4 1.65 to 1.85), then with the
  // site-words.  On chip, a class of b bonds: one CTA 0.5 (b = 16), 0.55 (200),
  // 1.0 (512); four CTAs 1.4 (1024), 1.6 (1300), 2.0 (2000); a quarter more with
  // 32-byte records; for as many words as run at once.  The launch, the planes and
  // the records: one CTA 7 (64 sites), 13 (1000), 32 (4096), four CTAs 12 to 20.
  // Calls of one sweep and of 20, launches / on chip: z = 1, 64 sites 4.1, 34 / 7.5,
  // 17; z = 2, 10 000 sites 10, 168 / 22, 210; z = 4, 4096 sites 29, 590 / 48, 360.
  const double b = 0.5 * (double)N * (double)z / (double)nclass;
  const bool one = C == 1;
  const double group = 1.75 * (double)nclass + 2.0e-5 * (double)N * (double)words;
  const double chip = (double)nclass * (one ? 0.45 + 1.1e-3 * b : 0.75 + 0.62e-3 * b) * (z > 4 ? 1.25 : 1.0);
  const double launch = one ? 7.0 + 6.0e-3 * (double)N : 10.0 + 1.0e-3 * (double)N;
  const double waves = (double)((words * C + sms - 1) / (sms > 0 ? sms : 1));
  return group * (double)n > (launch + chip * (double)n) * waves;
}

cudaError_t launch_graph(const Args& args, int64_t Nmax, int64_t bonds_max, int64_t class_max, int z,
                         int m, unsigned words, int C, cudaStream_t st) {
  if (m < 0 || z < 1 || z > 8 || !graph_fits(Nmax) || class_max > 1024 * C)
    return cudaErrorInvalidValue;
  Args a = args;
  a.fslots = (int)fslots_for(bonds_max, C);
  a.entries = (int)entries_for(class_max, C);
  const size_t smem = smem_for(Nmax, class_max, bonds_max, C);
  if (smem > kGraphSmem) return cudaErrorInvalidValue;
  const int threads = (int)std::max<int64_t>(64, ((class_max + C - 1) / C + 31) / 32 * 32);
  return z <= 4 ? launch_z<4>(a, m, words, C, threads, smem, st)
                : launch_z<8>(a, m, words, C, threads, smem, st);
}

}  // namespace resident
}  // namespace ka
