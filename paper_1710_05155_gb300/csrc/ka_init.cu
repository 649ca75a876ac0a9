// ka_init.cu -- initial state: exactly K particles per replica, uniform.
//
// Section 3.1 draws the initial configurations at fixed density at random.
// Replica r occupies the K sites with the smallest composite key
// (key_r(i), i), where key_r(i) is half (r mod 2) of the Philox block at
// counter (r / 2, 0xFFFFFFFF, i, 0): the first K entries of a uniformly
// random permutation, so every K-subset is equally likely.
//
// The Philox blocks bound this (32 per site and word), so every key is drawn
// once: the K-th smallest of N uniform keys lies within a few standard
// deviations of K / N, a window that is the same for every replica, known
// before any key is drawn.
//  * k_init_draw: one thread per site and word writes n = [key below the
//    window] and collects the sites whose key lies in it (6 deviations to
//    either side: 6 sqrt(N) of them at most on average) in a list per replica.
//  * the particles so far are counted per replica (ka_observe.cu).
//  * k_init_select: one block per replica finds the exact K-th smallest
//    composite key among the list and sets the bits of the list's sites up to
//    it.  A replica whose K-th key is not in the window, or whose list is
//    full (about one in 10^9), and every replica of a lattice of less than
//    kListSites sites, takes all sites as its list.
// L = 128, 256 replicas, one GB300: 3.24 ms for the radix select that was here
// before (three full passes of 0.85 to 1.11 ms, 20 small launches and a wait
// for the host in between), 0.86 ms now; 268 million blocks at the 4.9e11 a
// second that a bare loop of them reaches take 0.55 ms.
#include <algorithm>
#include <cmath>

#include "ka_internal.cuh"

namespace ka {
namespace {

constexpr int kThreads = 256;       // of a draw block
constexpr int kStage = 2048;        // candidates a draw block collects before the lists
constexpr int kSelect = 512;        // threads of a select block, and most keys it ranks directly
constexpr int kBuckets = 1024;
constexpr int64_t kListSites = 2048;

struct InitArgs {
  uint32_t* list_n;    // [R] sites in each replica's list
  uint32_t* list;      // [replicas of the launch][cap] their storage positions
  const unsigned long long* below;  // [R] keys below the window
  uint32_t cap;
  uint32_t lo, span;   // the window of a key's high word: lo .. lo + span
  int64_t K;
  int q0;              // first plane of the launch
  bool all;            // no lists: all sites
  RoundKeys rk;
};

// the half of replica r's block at site i
__device__ __forceinline__ uint64_t init_key(const RoundKeys& rk, uint32_t r, uint32_t i) {
  const uint4 b = philox(make_uint4(r >> 1, kTagInit, i, 0u), rk);
  return (r & 1u) ? hi64(b) : lo64(b);
}

// one thread per element of a plane (site position e / V, word e % V)
template <int V>
__global__ void __launch_bounds__(kThreads) k_init_draw(const __grid_constant__ InitArgs a,
                                                        const __grid_constant__ Planes pl) {
  __shared__ uint32_t staged;
  __shared__ uint16_t stage[kStage];  // thread << 6 | replica of the word
  if (threadIdx.x == 0) staged = 0;
  __syncthreads();
  const int q = a.q0 + (int)blockIdx.y;
  const int64_t e0 = (int64_t)blockIdx.x * kThreads;
  const int64_t e = e0 + threadIdx.x;
  // record bit j of thread t's word in the list of its replica
  auto append = [&](int t, uint32_t j) {
    const int64_t et = e0 + t;
    const uint32_t r = (uint32_t)(q * V + (int)(et % V)) * 64u + j;
    const uint32_t k = atomicAdd(&a.list_n[r], 1u);
    if (k < a.cap) a.list[(size_t)(r - (uint32_t)(a.q0 * V) * 64u) * a.cap + k] = (uint32_t)(et / V);
  };
  if (e < pl.N * V) {
    const uint32_t i = (uint32_t)canon_pos(pl.inv, pl.xs, e / V);  // canonical site held here
    const uint32_t w = (uint32_t)(q * V + (int)(e % V));           // replicas 64 w .. 64 w + 63
    uint32_t half[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t bits = 0;
#pragma unroll 4
      for (uint32_t j = 0; j < 16; ++j) {
        const uint4 b = philox(make_uint4(32u * w + 16u * (uint32_t)h + j, kTagInit, i, 0u), a.rk);
        // the high words of the two keys
        const bool in0 = b.y - a.lo <= a.span, in1 = b.w - a.lo <= a.span;
        bits |= (uint32_t)(b.y < a.lo) << (2 * j) | (uint32_t)(b.w < a.lo) << (2 * j + 1);
        if (in0 || in1) {
          const uint32_t at = 32u * (uint32_t)h + 2 * j;
          const uint32_t k = atomicAdd(&staged, (uint32_t)in0 + (uint32_t)in1);
          if (k + 2 <= (uint32_t)kStage) {
            if (in0) stage[k] = (uint16_t)(threadIdx.x << 6 | at);
            if (in1) stage[k + in0] = (uint16_t)(threadIdx.x << 6 | (at + 1));
          } else {
            if (k < (uint32_t)kStage) stage[k] = 0xFFFFu;  // no room: a void entry
            if (in0) append(threadIdx.x, at);
            if (in1) append(threadIdx.x, at + 1);
          }
        }
      }
      half[h] = bits;
    }
    const size_t off = (size_t)q * pl.plane_elems() + (size_t)e;
    pl.n[off] = (uint64_t)half[0] | (uint64_t)half[1] << 32;
    pl.p[off] = ~0ull;
  }
  __syncthreads();
  const uint32_t n = min(staged, (uint32_t)kStage);
  for (uint32_t k = threadIdx.x; k < n; k += kThreads)
    if (stage[k] != 0xFFFFu) append(stage[k] >> 6, stage[k] & 63u);
}

// one block per replica
__global__ void __launch_bounds__(kSelect) k_init_select(const __grid_constant__ InitArgs a,
                                                         const __grid_constant__ Planes pl) {
  __shared__ uint32_t hist[kBuckets];
  __shared__ uint64_t gkey[kSelect];
  __shared__ uint32_t gsite[kSelect];
  __shared__ uint32_t found, bucket, before, held, tsite;
  __shared__ uint64_t tkey;
  const uint32_t tid = threadIdx.x;
  const uint32_t rl = blockIdx.x, r = (uint32_t)(a.q0 * pl.V) * 64u + rl;
  int64_t need = a.K, m = pl.N;
  uint64_t lo = 0, hi = ~0ull;
  bool all = a.all;
  if (!all) {
    const int64_t left = a.K - (int64_t)a.below[r], in = (int64_t)a.list_n[r];
    all = left < 1 || left > in || in > (int64_t)a.cap;
    if (!all) {
      need = left;
      m = in;
      lo = (uint64_t)a.lo << 32;
      hi = (uint64_t)(a.lo + a.span) << 32 | 0xFFFFFFFFull;
    }
  }
  const uint32_t* list = a.list + (size_t)rl * a.cap;
  auto position = [&](int64_t k) -> int64_t { return all ? k : (int64_t)list[k]; };
  auto site_at = [&](int64_t pos) { return (uint32_t)canon_pos(pl.inv, pl.xs, pos); };

  // Narrow [lo, hi] to the bucket of the need-th smallest value until few
  // enough keys are left to rank directly: values are keys, then (should more
  // than kSelect keys be equal) the sites of the key `tied`.
  bool ties = false;
  uint64_t tied = 0;
  auto value_in = [&](uint64_t key, uint32_t site, uint64_t& v) {
    v = ties ? (uint64_t)site : key;
    return (!ties || key == tied) && v >= lo && v <= hi;
  };
  for (;;) {
    const int width = 64 - __clzll((long long)(hi - lo));  // bits of hi - lo
    const int shift = width > 10 ? width - 10 : 0;
    for (uint32_t k = tid; k < kBuckets; k += kSelect) hist[k] = 0;
    __syncthreads();
    for (int64_t k = tid; k < m; k += kSelect) {
      const uint32_t site = site_at(position(k));
      uint64_t v;
      if (value_in(init_key(a.rk, r, site), site, v)) atomicAdd(&hist[(v - lo) >> shift], 1u);
    }
    __syncthreads();
    if (tid < 32) {  // the bucket: lane l sums buckets 32 l .. 32 l + 31
      uint32_t mine = 0;
      for (int k = 0; k < kBuckets / 32; ++k) mine += hist[tid * (kBuckets / 32) + k];
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)tid >= o) incl += v;
      }
      uint32_t excl = incl - mine;
      if ((int64_t)excl < need && need <= (int64_t)incl) {
        uint32_t k = tid * (kBuckets / 32);
        while ((int64_t)(excl + hist[k]) < need) excl += hist[k++];
        bucket = k;
        before = excl;
        held = hist[k];
      }
    }
    __syncthreads();
    need -= (int64_t)before;
    lo += (uint64_t)bucket << shift;
    const uint64_t end = lo + ((1ull << shift) - 1);
    if (end < hi) hi = end;
    if (held <= (uint32_t)kSelect) break;
    if (shift == 0) {
      ties = true;
      tied = lo;
      lo = 0;
      hi = 0xFFFFFFFFull;
    }
    __syncthreads();
  }
  if (tid == 0) found = 0;
  __syncthreads();
  for (int64_t k = tid; k < m; k += kSelect) {
    const uint32_t site = site_at(position(k));
    const uint64_t key = init_key(a.rk, r, site);
    uint64_t v;
    if (value_in(key, site, v)) {
      const uint32_t at = atomicAdd(&found, 1u);
      gkey[at] = key;
      gsite[at] = site;
    }
  }
  __syncthreads();
  if (tid < found) {
    int64_t rank = 1;
    for (uint32_t k = 0; k < found; ++k)
      rank += gkey[k] < gkey[tid] || (gkey[k] == gkey[tid] && gsite[k] < gsite[tid]);
    if (rank == need) {
      tkey = gkey[tid];
      tsite = gsite[tid];
    }
  }
  __syncthreads();
  // the sites up to the threshold (of all sites: also none beyond it)
  const uint32_t w = r >> 6;
  unsigned long long* n = reinterpret_cast<unsigned long long*>(
      pl.n + (size_t)(w / (uint32_t)pl.V) * pl.plane_elems() + w % (uint32_t)pl.V);
  const unsigned long long bit = 1ull << (r & 63u);
  for (int64_t k = tid; k < m; k += kSelect) {
    const int64_t pos = position(k);
    const uint32_t site = site_at(pos);
    const uint64_t key = init_key(a.rk, r, site);
    if (key < tkey || (key == tkey && site <= tsite))
      atomicOr(n + pos * pl.V, bit);
    else if (all)
      atomicAnd(n + pos * pl.V, ~bit);
  }
}

// half the window in sites: 6 standard deviations of the number of keys below K / N
double window_sites(int64_t N, int64_t K) {
  const double f = (double)K / (double)N;
  return 6.0 * std::sqrt((double)K * (1.0 - f)) + 8.0;
}

}  // namespace

// entries of a replica's list: its mean at density 1/2 and 8 deviations
int64_t init_list_cap(int64_t N) {
  if (N < kListSites) return 0;
  const double mean = 2.0 * window_sites(N, N / 2);
  return (int64_t)(mean + 8.0 * std::sqrt(mean)) + 32;
}

cudaError_t launch_init(const Planes& pl, const InitScratch& s, int R, int64_t K,
                        const RoundKeys& rk, cudaStream_t st) {
  const size_t bytes = (size_t)pl.P * pl.plane_elems() * sizeof(uint64_t);
  cudaError_t err;
  if (K <= 0 || K >= pl.N) {
    const int fill = (K <= 0) ? 0x00 : 0xFF;
    if ((err = cudaMemsetAsync(pl.n, fill, bytes, st)) != cudaSuccess) return err;
    if ((err = cudaMemsetAsync(pl.n0, fill, bytes, st)) != cudaSuccess) return err;
    return cudaMemsetAsync(pl.p, 0xFF, bytes, st);
  }
  InitArgs a{};
  a.K = K;
  a.rk = rk;
  a.list_n = s.list_n;
  a.list = s.list;
  a.below = s.below;
  a.cap = (uint32_t)init_list_cap(pl.N);
  a.all = a.cap == 0;
  if (a.all) {
    if ((err = cudaMemsetAsync(pl.p, 0xFF, bytes, st))) return err;
    k_init_select<<<R, kSelect, 0, st>>>(a, pl);
    if ((err = cudaGetLastError())) return err;
  } else {
    const double h = window_sites(pl.N, K), unit = 4294967296.0 / (double)pl.N;
    const double lo = std::max(0.0, std::floor(((double)K - h) * unit));
    const double hi = std::min(4294967295.0, std::ceil(((double)K + h) * unit));
    a.lo = (uint32_t)lo;
    a.span = (uint32_t)hi - a.lo;
    if ((err = cudaMemsetAsync(s.list_n, 0, (size_t)R * sizeof(uint32_t), st))) return err;
    // as many planes at a time as there is room for their lists
    const size_t plane_list = (size_t)64 * pl.V * a.cap * sizeof(uint32_t);
    const int most = (int)std::max<size_t>(1, std::min<size_t>((size_t)pl.P, s.list_bytes / plane_list));
    for (int q = 0; q < pl.P; q += most) {
      const int nq = std::min(most, pl.P - q);
      a.q0 = q;
      const dim3 grid((unsigned)((pl.N * pl.V + kThreads - 1) / kThreads), (unsigned)nq);
      if (pl.V == 4)
        k_init_draw<4><<<grid, kThreads, 0, st>>>(a, pl);
      else if (pl.V == 2)
        k_init_draw<2><<<grid, kThreads, 0, st>>>(a, pl);
      else
        k_init_draw<1><<<grid, kThreads, 0, st>>>(a, pl);
      if ((err = cudaGetLastError())) return err;
      if ((err = launch_particles(pl, q, nq, s.below, st))) return err;
      k_init_select<<<nq * 64 * pl.V, kSelect, 0, st>>>(a, pl);
      if ((err = cudaGetLastError())) return err;
    }
  }
  return cudaMemcpyAsync(pl.n0, pl.n, bytes, cudaMemcpyDeviceToDevice, st);
}

}  // namespace ka
