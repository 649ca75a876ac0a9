// ka_observe.cu -- per-replica observables by vertical popcounts.
//
// Section 3.3 computes overlaps as bitwise ANDs of multispin words and
// counts their ones.  Here the counts are needed per replica, i.e. per bit
// position, summed over sites: for every replica r
//   particles   = sum_i n_i
//   overlap     = sum_i n_i & n0_i        (the q_i(t) = n_i(t) n_i(0) of section 2.2)
//   persist_occ = sum_i n0_i & p_i
//   persist_all = sum_i p_i
//
// Each thread adds up to 120 words of one word position into bit-sliced
// counters (one uint64 per binary digit, so all 64 replicas count at once),
// eight words at a time through a tree of full adders: 7 adders of two
// operations a half-word for eight words, where a ripple adder per word takes
// 12 on six digits.  Lanes of the same word position are then summed in
// bit-sliced form (the first exchange splits the 64 replicas over two lanes),
// the warp total is turned into one integer per replica, and blocks
// accumulate in shared memory before one 64-bit atomic per counter goes to
// global memory.  That summing costs about 200 operations a thread and
// observable, so the grid is one wave, of threads with as many words as that
// gives.
//
// What bounds it: the read of n, n0 and p (24 bytes a site-word).  L = 128, 256
// replicas: 201 MB, 39 us (5.1 TB/s, 0.76 of the copy rate).  With ripple adders
// 106 us (ALUs 82 %); eight words loaded, then added, 49; the next four words in
// flight meanwhile 42.4 (a ring of cp.async in shared memory with twice as many in
// flight gave the same, so that is enough).  The rest was around the reads:
// counts cleared by a launch that this one starts beside (instead of a memset
// before), additions to the counts in the order of the result (a warp's used to
// touch 32 sectors, now 8), words a thread in fours for a fuller wave: 39.2, and
// 16.6 -> 8.4 us for 2^18 sites with 128 replicas.
#include <algorithm>
#include <mutex>

#include "ka_count.cuh"

namespace ka {
namespace {

// binary digits of a thread's counters: up to 120 words, or (small planes) 8
constexpr int kDigits = 7, kFewDigits = 4;
constexpr int kPerThread = 120, kFew = 8;
constexpr size_t kOneBlock = 2048;  // words of a plane that one block takes

// ALL: the four observables; else only the particles
template <int V, bool ALL, int S>
__global__ void __launch_bounds__(256, 2) k_observe(Planes pl, unsigned long long* counts,
                                                 int per_thread) {
  constexpr int O = ALL ? 4 : 1;
  __shared__ unsigned int acc[O][64 * V];
  const int q = blockIdx.y;
  for (int k = threadIdx.x; k < O * 64 * V; k += blockDim.x) (&acc[0][0])[k] = 0;
  __syncthreads();

  const size_t E = pl.plane_elems();
  const uint64_t* gn = pl.n + (size_t)q * E;
  const uint64_t* g0 = ALL ? pl.n0 + (size_t)q * E : nullptr;
  const uint64_t* gp = ALL ? pl.p + (size_t)q * E : nullptr;
  // element e of the plane holds word h = e % V of site e / V; the block size
  // is a multiple of V, so a thread always sees the same h
  const size_t e0 = (size_t)blockIdx.x * blockDim.x * per_thread + threadIdx.x;
  uint64_t c[O][S];
#pragma unroll
  for (int o = 0; o < O; ++o)
#pragma unroll
    for (int s = 0; s < S; ++s) c[o][s] = 0;
  // four words of each array at a time, the next four in flight meanwhile
  struct Four {
    uint64_t n[4], n0[ALL ? 4 : 1], p[ALL ? 4 : 1];
  };
  auto load = [&](int k, Four& x) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t e = e0 + (size_t)(k + u) * blockDim.x;
      const bool in = k < per_thread && e < E;
      x.n[u] = in ? gn[e] : 0ull;
      if constexpr (ALL) {
        x.n0[u] = in ? g0[e] : 0ull;
        x.p[u] = in ? gp[e] : 0ull;
      }
    }
  };
  // the first two digits take four words; their carries of weight four
  auto first = [&](Four& x, uint64_t (&f)[O]) {
    f[0] = add4(c[0], x.n);
    if constexpr (ALL) {
      f[3] = add4(c[3], x.p);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        x.n[u] &= x.n0[u];
        x.p[u] &= x.n0[u];
      }
      f[1] = add4(c[1], x.n);
      f[2] = add4(c[2], x.p);
    }
  };
  Four a, b;
  uint64_t f0[O], f1[O];
  load(0, a);
  for (int k = 0; k < per_thread; k += 8) {
    load(k + 4, b);
    first(a, f0);
    load(k + 8, a);
    first(b, f1);
#pragma unroll
    for (int o = 0; o < O; ++o) carry8(c[o], f0[o], f1[o]);
  }
#pragma unroll
  for (int o = 0; o < O; ++o) reduce<V, S>(c[o], acc[o]);
  __syncthreads();
  // the clearing launch is complete
  if (gridDim.x > 1) asm volatile("griddepcontrol.wait;" ::: "memory");
  // in the order of the result, so that a warp's additions share sectors
  unsigned long long* out = counts + (size_t)q * V * 64 * O;
  for (int k = threadIdx.x; k < O * 64 * V; k += blockDim.x) {
    const unsigned int v = acc[k % O][k / O];  // k / O = h * 64 + bit
    if (gridDim.x == 1) out[k] = v;  // the plane's only block
    else if (v) atomicAdd(&out[k], (unsigned long long)v);
  }
}

// Sets the counts to zero; the counting launch starts at once beside it.  This
// launch itself starts when all work before it on the stream is complete.
__global__ void k_clear(unsigned long long* counts, int n) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) counts[k] = 0;
}

template <bool ALL>
cudaError_t launch_counts(const Planes& pl, unsigned long long* counts_dev, cudaStream_t st) {
  // words per thread, in fours: one wave of two blocks per SM over all planes
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t E = pl.plane_elems();
  const size_t wave = (size_t)256 * 2 * (size_t)(sms > 0 ? sms : 148);
  size_t per_thread = (E * (size_t)pl.P + wave - 1) / wave;
  // a small plane is one block's, which stores its counts: no clearing launch
  // before (us of ka_observe, one block and several: 1728 words 19.4, -; 4096
  // 27.9, 22.5; 8000 28.2, 22.2)
  if (E <= kOneBlock) per_thread = std::max(per_thread, (E + 255) / 256);
  per_thread = std::min<size_t>((per_thread + 3) / 4 * 4, kPerThread);
  const size_t per_block = 256 * per_thread;
  const dim3 grid((unsigned)((E + per_block - 1) / per_block), (unsigned)pl.P);
  const bool many = grid.x > 1;
  if (many) {
    const int n = pl.P * pl.V * 64 * (ALL ? 4 : 1);
    k_clear<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(counts_dev, n);
    const cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
  }
  const bool few = per_thread <= kFew;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = many ? 1 : 0;
#define KA_LAUNCH(V, S) \
  return cudaLaunchKernelEx(&cfg, k_observe<V, ALL, S>, pl, counts_dev, (int)per_thread)
  if (pl.V == 4) {
    if (few) KA_LAUNCH(4, kFewDigits);
    KA_LAUNCH(4, kDigits);
  } else if (pl.V == 2) {
    if (few) KA_LAUNCH(2, kFewDigits);
    KA_LAUNCH(2, kDigits);
  }
  if (few) KA_LAUNCH(1, kFewDigits);
  KA_LAUNCH(1, kDigits);
#undef KA_LAUNCH
}

}  // namespace

cudaError_t launch_observe(const Planes& pl, unsigned long long* counts_dev, cudaStream_t st) {
  return launch_counts<true>(pl, counts_dev, st);
}

cudaError_t launch_particles(const Planes& pl, int q0, int nq, unsigned long long* counts_dev,
                             cudaStream_t st) {
  Planes part = pl;
  part.n += (size_t)q0 * pl.plane_elems();
  part.P = nq;
  return launch_counts<false>(part, counts_dev + (size_t)q0 * pl.V * 64, st);
}

// ---------------------------------------------------------------------------
// Allocation-free variant (ka_observe_static): the per-replica accumulators
// live in a file-scope device array instead of memory the caller or the
// library allocates.  Every GPU that loads the library holds this array
// until the process exits.
// ---------------------------------------------------------------------------

constexpr int kStaticMaxReplicas = 4096;  // 4096 x 4 x 8 bytes = 128 KiB per device
static __device__ __align__(256) unsigned long long g_static_counts[kStaticMaxReplicas * 4];

namespace {
constexpr int kMaxDevices = 64;

// The array's device address on one device, looked up once: std::call_once
// orders the lookup before every use from any host thread.
struct StaticSlot {
  std::once_flag once;
  cudaError_t err = cudaSuccess;
  unsigned long long* ptr = nullptr;
};
StaticSlot g_static_slot[kMaxDevices];
}  // namespace

// Device address of the array on the current device.  In host code the
// symbol itself is only a host-side stand-in, so its address is looked up
// (with that device current) by the first call on each device and cached;
// a failed lookup is returned to every later call on that device.
cudaError_t static_counts_ptr(unsigned long long** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  StaticSlot& s = g_static_slot[dev];
  std::call_once(s.once, [&s] {
    void* ptr = nullptr;
    s.err = cudaGetSymbolAddress(&ptr, g_static_counts);
    s.ptr = (unsigned long long*)ptr;
  });
  if (s.err != cudaSuccess) return s.err;
  *out = s.ptr;
  return cudaSuccess;
}

}  // namespace ka

extern "C" ka_status ka_observe_static(const uint64_t* n, const uint64_t* n0, const uint64_t* p,
                                       int64_t N, int32_t replicas, int64_t* counts,
                                       void* stream) {
  if (!n || !n0 || !p || !counts || N < 1 || replicas <= 0 || replicas % 64 ||
      replicas > ka::kStaticMaxReplicas)
    return KA_EINVAL;
  const cudaStream_t st = (cudaStream_t)stream;
  if (st) {
    // the array whose address is used is the current device's: the stream
    // must belong to that device
    int cur = 0, sdev = 0;
    if (cudaGetDevice(&cur) != cudaSuccess || cudaStreamGetDevice(st, &sdev) != cudaSuccess)
      return KA_ECUDA;
    if (sdev != cur) return KA_EINVAL;
  }
  unsigned long long* scratch = nullptr;
  cudaError_t e = ka::static_counts_ptr(&scratch);
  if (e != cudaSuccess) return KA_ECUDA;
  // the canonical layout [R/64][N] is the device layout with one word per plane
  ka::Planes pl{};
  pl.n = const_cast<uint64_t*>(n);
  pl.n0 = const_cast<uint64_t*>(n0);
  pl.p = const_cast<uint64_t*>(p);
  pl.N = N;
  pl.W = replicas / 64;
  pl.V = 1;
  pl.P = pl.W;
  e = ka::launch_observe(pl, scratch, st);  // clears the scratch, then accumulates
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(counts, scratch, (size_t)replicas * 4 * sizeof(int64_t),
                        cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? KA_OK : KA_ECUDA;
}
