// ka_four_point.cu -- four-point correlations on cubic lattices.
//
// Section 2.2 defines the space-dependent susceptibility g_4(r, t) from the
// overlaps q_i = n_i(t) n_i(0) of pairs of sites at distance r, and section
// 3.3 computes its numerator Phi(r, t) as popcounts of n_i(t) & n_i(0) &
// n_j(t) & n_j(0) summed over pairs.  Here every ordered pair (i, j) is
// counted once, at the representative of its displacement with every
// component in [-L/2, L/2), in the shell s = |delta|^2:
//   phi[r][s] = sum over pairs in shell s of q_i q_j          (replica r)
//   psi[s]    = sum over pairs in shell s of M_i M_j,  M_i = sum_r q_i^r
// (psi gives the <q_i><q_j> term of g_4).
//
// The sums for delta and -delta are equal, so one of the two is run with
// weight 2.  q (and M) are first written as words in site order with a margin
// of the largest component on every side, filled periodically: site i + delta
// is then a fixed offset from i for all sites, and neighbouring threads read
// neighbouring words.  A thread takes sixteen sites and, shell by shell, adds
// q_i & q_{i + delta} for all of them into bit-sliced counters, eight words at
// a time (ka_count.cuh); a block sums a shell's counters in shared memory and
// adds 64 integers to phi.  One launch covers all shells; small lattices
// split the vectors over more blocks.
//
// Bound by the ALUs: about 12 instructions per site-word and vector (the
// adders 5, the AND 2, the load and its address 2, the sums over lanes the
// rest).  L = 64, 256 replicas, smax = 25 (515 vectors), the whole call: 4.56 ms
// before, when each shell was a launch and a thread worked out periodic
// coordinates for each vector; 0.35 ms now.
#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "ka_count.cuh"
#include "ka_ctx.cuh"

namespace ka {
namespace {

constexpr int kDigits = 8;            // per-thread counters hold up to 255
constexpr int kSites = 16;            // sites per thread
constexpr int kPsiSites = 4;          // of the sum over counts: more blocks
constexpr int kSegment = 15;          // vectors per segment: 240 words per thread
constexpr int kThreads = 256;
constexpr int kMaxVectors = 1 << 16;  // displacement vectors per call
// Scratch when the context's staging plane does not hold one word's padded
// lattice: this much, or one word's, a slab of layers at a time; less where the
// device has not that much left.
constexpr size_t kArena = (size_t)256 << 20;

// Passes over the words in the staging plane before an allocation is made: one
// takes 150 us, a pass over a small lattice 15 (L = 8, 4096 replicas, smax = 6:
// 64 passes 1530 us, one 220).
constexpr int kMostPasses = 8;
constexpr size_t kSmallScratch = (size_t)8 << 20;
constexpr size_t kSmallResult = (size_t)64 << 10;  // bytes that are cheaper to copy twice on the host

constexpr int64_t kMostPadded = (int64_t)1 << 29;  // elements: 32-bit byte offsets

// Vectors of one shell and weight: offsets [first, first + count).
struct Segment {
  int shell, first, count, weight;
};

// A slab of the padded lattice: layers z0 .. z0 + zc - 1 of the last dimension
// with a margin of rad all round.
struct Slab {
  int d, L, rad, z0, zc;
  int64_t ps[4];     // strides of the padded lattice
  int64_t padded;    // its elements
  int64_t sites;     // sites of the slab
};

// Sites (below 2^31) and padded elements (below kMostPadded) in 32 bits: a thread
// divides for each of its sites (one block of k_phi took 17 us with 64).
// storage position of the site that padded element k shows
__device__ __forceinline__ uint32_t shown(const Slab& g, int xs, uint32_t k) {
  uint32_t site = 0, stride = 1;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (m < g.d) {
      const uint32_t extent = (uint32_t)(m == g.d - 1 ? g.zc + 2 * g.rad : g.L + 2 * g.rad);
      int64_t x = (int64_t)(k % extent) - g.rad + (m == g.d - 1 ? g.z0 : 0);
      k /= extent;
      x += x < 0 ? g.L : 0;
      x -= x >= g.L ? g.L : 0;
      site += (uint32_t)x * stride;
      stride *= (uint32_t)g.L;
    }
  }
  if (!xs) return site;
  const uint32_t x = site % (uint32_t)xs;  // dev_site
  return site - x + (x & 1u) * ((uint32_t)xs >> 1) + (x >> 1);
}

// padded element of the slab's site k
__device__ __forceinline__ uint32_t centre(const Slab& g, uint32_t k) {
  uint32_t e = 0;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (m < g.d) {
      const uint32_t q = m == g.d - 1 ? 0 : k / (uint32_t)g.L, x = k - q * (uint32_t)g.L;
      k = q;
      e += (x + (uint32_t)g.rad) * (uint32_t)g.ps[m];
    }
  }
  return e;
}

// q = n & n0 of words w0 .. w0 + gridDim.y - 1, padded
__global__ void __launch_bounds__(kThreads) k_pad(const __grid_constant__ Planes pl,
                                                  const __grid_constant__ Slab g, int w0,
                                                  uint64_t* __restrict__ out) {
  const int64_t k = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (k >= g.padded) return;
  const int w = w0 + (int)blockIdx.y;
  const size_t e = (size_t)(w / pl.V) * pl.plane_elems() + (size_t)shown(g, pl.xs, (uint32_t)k) * pl.V + w % pl.V;
  out[(size_t)blockIdx.y * g.padded + k] = pl.n[e] & pl.n0[e];
}

// M = number of replicas with q = 1, padded
__global__ void __launch_bounds__(kThreads) k_pad_counts(const __grid_constant__ Planes pl,
                                                         const __grid_constant__ Slab g,
                                                         uint32_t* __restrict__ M) {
  const int64_t k = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (k >= g.padded) return;
  const size_t at = (size_t)shown(g, pl.xs, (uint32_t)k) * pl.V;
  const int lv = pl.V == 4 ? 2 : pl.V == 2 ? 1 : 0;
  uint32_t m = 0;
#pragma unroll 8
  for (int w = 0; w < pl.W; ++w) {  // eight words' loads at once
    const size_t e = (size_t)(w >> lv) * pl.plane_elems() + at + (w & (pl.V - 1));
    m += (uint32_t)__popcll(__ldg(pl.n + e) & __ldg(pl.n0 + e));
  }
  M[k] = m;
}

// phi of words w0 + blockIdx.y over the segments of blockIdx.z
__global__ void __launch_bounds__(kThreads, 2) k_phi(const __grid_constant__ Slab g,
                                                  const uint64_t* __restrict__ padded,
                                                  const Segment* __restrict__ seg,
                                                  const int32_t* __restrict__ offset, int nseg,
                                                  int w0, int nshell, unsigned long long* phi) {
  __shared__ unsigned int acc[64];
  const uint64_t* q = padded + (size_t)blockIdx.y * g.padded;
  const int64_t s0 = (int64_t)blockIdx.x * (kThreads * kSites) + threadIdx.x;
  uint32_t at[kSites];  // byte offsets
  uint64_t own[kSites];
#pragma unroll
  for (int u = 0; u < kSites; ++u) {
    const int64_t s = s0 + u * kThreads;
    const bool in = s < g.sites;
    at[u] = 8u * centre(g, in ? (uint32_t)s : 0u);
    own[u] = in ? *reinterpret_cast<const uint64_t*>(reinterpret_cast<const char*>(q) + at[u]) : 0ull;
  }
  const int b0 = (int)((int64_t)nseg * blockIdx.z / gridDim.z);
  const int b1 = (int)((int64_t)nseg * (blockIdx.z + 1) / gridDim.z);
  if (threadIdx.x < 64) acc[threadIdx.x] = 0;
  __syncthreads();
  for (int b = b0; b < b1; ++b) {
    const Segment sg = seg[b];
    uint64_t c[kDigits];
#pragma unroll
    for (int s = 0; s < kDigits; ++s) c[s] = 0;
    for (int v = 0; v < sg.count; ++v) {
      const uint32_t off = 8u * (uint32_t)__ldg(offset + sg.first + v);
      uint64_t x[2][8];
#pragma unroll
      for (int u = 0; u < kSites; ++u)
        x[u / 8][u % 8] =
            __ldg(reinterpret_cast<const uint64_t*>(reinterpret_cast<const char*>(q) + (at[u] + off)));
#pragma unroll
      for (int u = 0; u < kSites; ++u) x[u / 8][u % 8] &= own[u];
      add8(c, x[0]);
      add8(c, x[1]);
    }
    reduce<1, kDigits>(c, acc, (unsigned)sg.weight);
    if (b + 1 == b1 || seg[b + 1].shell != sg.shell) {
      __syncthreads();
      if (threadIdx.x < 64) {
        const unsigned int v = acc[threadIdx.x];
        acc[threadIdx.x] = 0;
        if (v)
          atomicAdd(&phi[((size_t)(w0 + (int)blockIdx.y) * 64 + threadIdx.x) * nshell + sg.shell],
                    (unsigned long long)v);
      }
      __syncthreads();
    }
  }
}

// psi over the segments of blockIdx.z
__global__ void __launch_bounds__(kThreads) k_psi(const __grid_constant__ Slab g,
                                                  const uint32_t* __restrict__ M,
                                                  const Segment* __restrict__ seg,
                                                  const int32_t* __restrict__ offset, int nseg,
                                                  unsigned long long* psi) {
  const int64_t s0 = (int64_t)blockIdx.x * (kThreads * kPsiSites) + threadIdx.x;
  int32_t at[kPsiSites];
  uint32_t own[kPsiSites];
#pragma unroll
  for (int u = 0; u < kPsiSites; ++u) {
    const int64_t s = s0 + u * kThreads;
    const bool in = s < g.sites;
    at[u] = (int32_t)centre(g, in ? (uint32_t)s : 0u);
    own[u] = in ? M[at[u]] : 0u;
  }
  const int b0 = (int)((int64_t)nseg * blockIdx.z / gridDim.z);
  const int b1 = (int)((int64_t)nseg * (blockIdx.z + 1) / gridDim.z);
  unsigned long long sum = 0;
  for (int b = b0; b < b1; ++b) {
    const Segment sg = seg[b];
    unsigned long long part = 0;
    for (int v = 0; v < sg.count; ++v) {
      const int32_t off = __ldg(offset + sg.first + v);
#pragma unroll
      for (int u = 0; u < kPsiSites; ++u) part += (unsigned long long)own[u] * __ldg(M + (at[u] + off));
    }
    sum += part * (unsigned)sg.weight;
    if (b + 1 == b1 || seg[b + 1].shell != sg.shell) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if ((threadIdx.x & 31) == 0 && sum) atomicAdd(psi + sg.shell, sum);
      sum = 0;
    }
  }
}

struct Scope {
  int prev = -1;
  explicit Scope(int dev) {
    if (cudaGetDevice(&prev) == cudaSuccess && prev != dev)
      cudaSetDevice(dev);
    else
      prev = -1;
  }
  ~Scope() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

ka_status four_point_fail(ka_ctx* c, ka_status st, const std::string& msg) {
  c->err = msg;
  return st;
}

}  // namespace
}  // namespace ka

extern "C" ka_status ka_four_point(ka_ctx* c, int32_t smax, int64_t* phi, int64_t* psi) {
  ka::NvtxRange nvtx_range("ka_four_point");
  using namespace ka;
  if (!c) return KA_EINVAL;
  if (!phi || smax < 0) return four_point_fail(c, KA_EINVAL, "phi must be non-NULL, smax >= 0");
  if (c->topo != KA_CUBIC)
    return four_point_fail(c, KA_EINVAL, "four-point correlations need a cubic lattice");
  if (ka_status st = valid_state(c, "four-point")) return st;
  const int d = c->d, L = c->L, half = L / 2;
  if ((int64_t)smax > (int64_t)d * half * half)
    return four_point_fail(c, KA_EINVAL, "smax above d (L/2)^2, the largest shell");
  // representative displacement vectors (components in [-L/2, L/2))
  int rad = 0;
  while ((int64_t)(rad + 1) * (rad + 1) <= smax) ++rad;
  rad = std::min(rad, half);
  const int lo = -rad, hi = std::min(rad, half - 1);
  const int S = smax + 1;

  // The padded lattice, a slab of its last dimension at a time if one word of
  // the whole is too large, and where it is kept: the staging plane (idle
  // here) if that holds a word of it and the rest, else an allocation.
  Slab g{};
  g.d = d;
  g.L = L;
  g.rad = rad;
  g.ps[0] = 1;
  for (int k = 1; k < 4; ++k) g.ps[k] = g.ps[k - 1] * (L + 2 * rad);
  const int64_t layer = g.ps[d - 1];
  const int64_t layer_sites = c->N / L;
  const int64_t most = (int64_t)(kArena / sizeof(uint64_t));
  const size_t stage_bytes = c->stage ? (size_t)c->N * c->pl.W * sizeof(uint64_t) : 0;

  struct Vec {
    int32_t shell, offset, weight;
  };
  std::vector<Vec> vecs;
  int64_t nvec = 0;
  int x[4] = {lo, lo, lo, lo};
  for (int k = d; k < 4; ++k) x[k] = 0;
  for (;;) {
    int64_t s2 = 0, off = 0;
    int sign = 0;  // of the first component that is not its own negative
    for (int k = 0; k < d; ++k) {
      s2 += (int64_t)x[k] * x[k];
      off += x[k] * g.ps[k];
      if (!sign && x[k] != 0 && x[k] != -half) sign = x[k] > 0 ? 1 : -1;
    }
    if (s2 <= smax) {
      if (++nvec > kMaxVectors)
        return four_point_fail(c, KA_EINVAL, "more than 65536 displacement vectors: lower smax");
      if (sign >= 0) vecs.push_back({(int32_t)s2, (int32_t)off, sign ? 2 : 1});
    }
    int k = 0;
    while (k < d && x[k] == hi) x[k++] = lo;
    if (k == d) break;
    ++x[k];
  }
  std::stable_sort(vecs.begin(), vecs.end(), [](const Vec& a, const Vec& b) {
    return a.shell != b.shell ? a.shell < b.shell : a.weight < b.weight;
  });
  std::vector<int32_t> offsets;
  std::vector<Segment> segs;
  for (const Vec& v : vecs) {
    if (segs.empty() || segs.back().shell != v.shell || segs.back().weight != v.weight ||
        segs.back().count == kSegment)
      segs.push_back({v.shell, (int)offsets.size(), 0, v.weight});
    ++segs.back().count;
    offsets.push_back(v.offset);
  }
  const int nseg = (int)segs.size();

  Scope scope(c->device);
  const cudaStream_t st = c->stream;
  const int R = c->R, W = c->pl.W;
  const size_t phi_bytes = (size_t)R * S * sizeof(unsigned long long);
  const size_t psi_bytes = (size_t)S * sizeof(unsigned long long);
  const size_t seg_bytes = segs.size() * sizeof(Segment), off_bytes = offsets.size() * sizeof(int32_t);
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t fixed = up(phi_bytes) + up(psi_bytes) + up(seg_bytes) + up(off_bytes);
  auto m_bytes = [&](int64_t zc) { return psi ? up((size_t)(layer * (zc + 2 * rad)) * sizeof(uint32_t)) : 0; };
  auto q_bytes = [&](int64_t zc) { return up((size_t)(layer * (zc + 2 * rad)) * sizeof(uint64_t)); };
  int64_t zc = L;
  int words = 0;  // per pass
  char* own = nullptr;
  size_t own_bytes = 0;
  char* mem = nullptr;
  if (layer * (L + 2 * rad) < kMostPadded && stage_bytes >= fixed + m_bytes(L) + q_bytes(L))
    words = (int)std::min<size_t>((size_t)W, (stage_bytes - fixed - m_bytes(L)) / q_bytes(L));
  if (words && (W + words - 1) / words <= kMostPasses) {
    mem = (char*)c->stage;
  } else {
    if (layer * (zc + 2 * rad) > most) zc = std::max<int64_t>(1, most / layer - 2 * rad);
    if (layer * (zc + 2 * rad) >= kMostPadded)
      return four_point_fail(c, KA_ENOMEM, "scratch: a padded layer is too large");
    words = (int)std::max<size_t>(1, std::min<size_t>((size_t)W, kArena / q_bytes(zc)));
    auto take = [&]() {
      own_bytes = fixed + m_bytes(zc) + (size_t)words * q_bytes(zc);
      const cudaError_t ea = cudaMallocAsync((void**)&own, own_bytes, st);
      if (ea) {
        own = nullptr;
        cudaGetLastError();
      }
      return ea;
    };
    cudaError_t ea = take();
    if (ea) {
      // a full device: the thickest slab that the staging plane holds, else
      // ever thinner ones in less memory (down to (L + 2 rad)^(d - 1) (2 rad + 1)
      // words, 0.7 MB at L = 64, rad = 5)
      words = 1;
      int64_t in_stage = 0, above = std::min<int64_t>(L, zc) + 1;
      while (above - in_stage > 1) {
        const int64_t mid = (in_stage + above) / 2;
        (fixed + m_bytes(mid) + q_bytes(mid) <= stage_bytes ? in_stage : above) = mid;
      }
      if (in_stage) {
        zc = in_stage;
        mem = (char*)c->stage;
        ea = cudaSuccess;
      } else {
        for (ea = take(); ea && zc > 1; ea = take()) zc /= 2;
      }
    }
    if (ea) return four_point_fail(c, KA_ENOMEM, std::string("scratch: ") + cudaGetErrorString(ea));
    if (own) mem = own;
  }
  unsigned long long* phi_dev = (unsigned long long*)mem;
  unsigned long long* psi_dev = (unsigned long long*)(mem + up(phi_bytes));
  Segment* seg_dev = (Segment*)(mem + up(phi_bytes) + up(psi_bytes));
  int32_t* off_dev = (int32_t*)((char*)seg_dev + up(seg_bytes));
  uint32_t* M = (uint32_t*)(mem + fixed);
  uint64_t* q = (uint64_t*)(mem + fixed + m_bytes(zc));
  cudaError_t e = cudaMemsetAsync(mem, 0, up(phi_bytes) + up(psi_bytes), st);
  // both tables in one copy, and below both results: a copy takes about 8 us
  std::vector<char> tables(up(seg_bytes) + off_bytes);
  std::memcpy(tables.data(), segs.data(), seg_bytes);
  std::memcpy(tables.data() + up(seg_bytes), offsets.data(), off_bytes);
  if (!e) e = cudaMemcpyAsync(seg_dev, tables.data(), tables.size(), cudaMemcpyHostToDevice, st);
  const Planes& pl = c->pl;
  // blocks along z share out the segments until the grid has four blocks per SM
  auto split = [&](int64_t blocks) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(nseg, 4 * (int64_t)c->sms / blocks));
  };
  for (int64_t z0 = 0; z0 < L && !e; z0 += zc) {
    g.z0 = (int)z0;
    g.zc = (int)std::min<int64_t>(zc, L - z0);
    g.padded = layer * (g.zc + 2 * rad);
    g.sites = layer_sites * g.zc;
    const unsigned pads = (unsigned)((g.padded + kThreads - 1) / kThreads);
    const unsigned tiles = (unsigned)((g.sites + kThreads * kSites - 1) / (kThreads * kSites));
    if (psi) {
      k_pad_counts<<<pads, kThreads, 0, st>>>(pl, g, M);
      const unsigned psi_tiles = (unsigned)((g.sites + kThreads * kPsiSites - 1) / (kThreads * kPsiSites));
      k_psi<<<dim3(psi_tiles, 1, split(psi_tiles)), kThreads, 0, st>>>(g, M, seg_dev, off_dev, nseg, psi_dev);
      e = cudaGetLastError();
    }
    for (int w0 = 0; w0 < W && !e; w0 += words) {
      const unsigned nw = (unsigned)std::min(words, W - w0);
      k_pad<<<dim3(pads, nw), kThreads, 0, st>>>(pl, g, w0, q);
      k_phi<<<dim3(tiles, nw, split((int64_t)tiles * nw)), kThreads, 0, st>>>(g, q, seg_dev, off_dev, nseg,
                                                                            w0, S, phi_dev);
      e = cudaGetLastError();
    }
  }
  std::vector<char> both(psi && up(phi_bytes) + psi_bytes <= kSmallResult ? up(phi_bytes) + psi_bytes : 0);
  if (!both.empty()) {
    if (!e) e = cudaMemcpyAsync(both.data(), mem, both.size(), cudaMemcpyDeviceToHost, st);
  } else {
    if (!e) e = cudaMemcpyAsync(phi, phi_dev, phi_bytes, cudaMemcpyDeviceToHost, st);
    if (!e && psi) e = cudaMemcpyAsync(psi, psi_dev, psi_bytes, cudaMemcpyDeviceToHost, st);
  }
  // A free before the wait gives the memory back to the device in the wait,
  // which takes 130 us; a small block is freed after it, so that the pool keeps
  // it until the next wait and the next call finds it there.
  cudaError_t ef = own && own_bytes > kSmallScratch ? cudaFreeAsync(own, st) : cudaSuccess;
  const cudaError_t es = cudaStreamSynchronize(st);
  if (own && own_bytes <= kSmallScratch) ef = cudaFreeAsync(own, st);
  if (!e) e = es;
  if (!e) e = ef;
  if (e) return four_point_fail(c, KA_ECUDA, std::string("four-point: ") + cudaGetErrorString(e));
  if (!both.empty()) {
    std::memcpy(phi, both.data(), phi_bytes);
    std::memcpy(psi, both.data() + up(phi_bytes), psi_bytes);
  }
  return c->waits ? check_waits(c) : KA_OK;
}
