// ka_sequential.cu -- the random-sequential schedule of section 3.2.
//
// The paper's own update: each step picks one bond at random, shared by all
// replicas packed in a word, and exchanges the two sites in every replica
// where the rule of section 2.1 allows it (no per-replica gate).  N attempts
// make a sweep (the time unit of section 2.1).  Attempt k of sweep t of word
// w draws r uniform in [0, N z) by Lemire's method on the low 64 bits of the
// Philox block at counter (t, 0xFFFFFFFC - draw, k, w), key = seed, and takes
// site i = r / z and its neighbour in slot r mod z (slots 2 mu and 2 mu + 1
// are the up and down neighbours along mu on a cubic lattice; on a graph the
// slots follow the neighbour row, kept in ascending order).
//
// The attempts of one word form a chain, run 32 at a time, one per lane of
// one warp, with the result of the chain in order.  An attempt reads n on its
// read set R = {i, j} and the neighbours of i and of j, and writes n and p on
// W = {i, j}.  Attempts k and l conflict when W_k meets R_l or W_l meets R_k.
// The neighbour relation is symmetric (cubic lattices by construction, graphs
// are checked when the context is made), so the two are the same condition: a
// site of W_k equals a site of W_l or neighbours one.  The warp applies the
// pending attempts in rounds: in each, every pending attempt that conflicts
// with no earlier pending attempt (a set that always holds the earliest)
// reads, decides and writes.  Such an attempt sees exactly the state the
// chain would give it: no earlier attempt still pending writes what it
// reads, and it writes nothing that an earlier pending attempt has yet to
// read; attempts applied in one round touch disjoint sites.
//
// The chain's rounds are one warp's latency; all that does not depend on the
// state -- the draws, the sites, who conflicts with whom -- is prepared by seven
// other warps of the CTA, a batch of 32 attempts each, while the chain's warp
// applies the seven batches before (in turn; one warp doing both took 4500
// cycles a batch, most of them for the preparation).  A maker finds the
// conflicts by stamps: every attempt sets its lane bit in a word of a table
// for both sites of W, then ORs the words over R.  Sites share words of a
// table, which can only add conflicts; two tables under different hashes are
// ANDed, so that few are added.  The word's n and p planes sit in shared memory
// when they fit, else in global memory.
#include <algorithm>
#include <string>

#include "ka_ctx.cuh"

namespace ka {
namespace {

constexpr uint32_t kTagSequential = 0xFFFFFFFCu;
constexpr int kSmemWords = 20480;  // n and p of up to 10240 sites in shared memory
constexpr size_t kSmemMost = (size_t)227 * 1024;  // shared memory of a CTA
constexpr int kMakers = 7;         // warps that prepare attempts, or
constexpr int kFewMakers = 3;      // with more words than run at once
constexpr uint32_t kMaxStamps = 2048;  // words of one of a maker's two stamp tables, at most
constexpr size_t kSmSmem = (size_t)228 * 1024;  // shared memory of an SM (1 KB of it per CTA)
constexpr int kSmThreads = 2048;

struct SeqArgs {
  uint64_t* n;
  uint64_t* p;
  const int32_t* nbr;  // [N][z], or null: periodic cubic lattice from coordinates
  int64_t N;
  int z, d, L, V;
  int xs;  // split-row order of the planes (0: index order)
  const int32_t* perm;  // graphs: storage position of every canonical site (nbr in positions)
  size_t plane_elems;
  uint32_t t0;
  int nsweeps;
  uint32_t hmask, hshift;  // stamp words - 1 (a power of two), 32 - their binary logarithm
  RoundKeys rk;
};

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

// the bond draw of attempt k: r uniform in [0, range)
__device__ __forceinline__ uint64_t draw_bond(const RoundKeys& rk, uint32_t t, uint32_t k,
                                              uint32_t w, uint64_t range) {
  uint32_t draw = 0;
  uint64_t x = lo64(philox(make_uint4(t, kTagSequential, k, w), rk));
  uint64_t low = x * range;
  if (low < range) {
    const uint64_t threshold = (0ull - range) % range;
    while (low < threshold) {
      ++draw;
      x = lo64(philox(make_uint4(t, kTagSequential - draw, k, w), rk));
      low = x * range;
    }
  }
  return __umul64hi(x, range);
}

// the 2d neighbours of site i of a periodic cubic lattice, slot 2 mu up and
// 2 mu + 1 down along mu (32-bit arithmetic: N z < 2^32)
__device__ __forceinline__ void cubic_neighbours(const SeqArgs& a, uint32_t i, uint32_t (&out)[8]) {
  uint32_t rest = i, stride = 1;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    if (mu >= a.d) break;
    const uint32_t L = (uint32_t)a.L, q = rest / L, x = rest - q * L;
    rest = q;
    out[2 * mu] = (x == L - 1) ? i - (L - 1) * stride : i + stride;
    out[2 * mu + 1] = (x == 0) ? i + (L - 1) * stride : i - stride;
    stride *= L;
  }
}

// the z neighbours of site i
__device__ __forceinline__ void neighbours(const SeqArgs& a, int z, uint32_t i, uint32_t (&out)[8]) {
  if (a.nbr) {
#pragma unroll
    for (int s = 0; s < 8; ++s)
      if (s < z) out[s] = (uint32_t)a.nbr[(int64_t)i * z + s];
  } else {
    cubic_neighbours(a, i, out);
  }
}

// One CTA per word; n and p of the word at stride `st` (V in global memory, 1
// in shared memory).  Warp 0 applies the attempts, the others make them.
//
// A batch in the ring: per lane the sites i, j and their z - 1 other
// neighbours each (two 16-bit indices to a word for planes in shared memory),
// then the mask of the lanes it conflicts with (its own bit: the attempt
// exists); fields lane by lane.  With the planes in shared memory warp 0 leaves
// the swaps it made and the makers clear them in p in the turn after, in any
// order.
//
// us a sweep, before (one warp doing all) and after, one GB300: L = 8, 64
// replicas 48.8, 11.4; L = 16, 256 replicas 276, 58.7; L = 20 512, 107; planes in
// global memory: L = 32 8480, 1147; L = 64 68900, 8200; random regular N = 2^14
// 1825, 493.  Bound by the latency of the chain's rounds (two to three a batch
// on 4096 sites).
// Z = z where it has an instance of its own, else 0.
template <int Z, int M, bool SMEM>
__global__ void __launch_bounds__(32 * (kMakers + 1)) k_sequential(const __grid_constant__ SeqArgs a) {
  extern __shared__ uint64_t sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t w = blockIdx.x;  // word index
  const int q = (int)(w / (uint32_t)a.V), h = (int)(w % (uint32_t)a.V);
  uint64_t* gn = a.n + (size_t)q * a.plane_elems + h;
  uint64_t* gp = a.p + (size_t)q * a.plane_elems + h;
  uint64_t* n = gn;
  uint64_t* p = gp;
  const int64_t st = SMEM ? 1 : a.V;
  if constexpr (SMEM) {
    // shared memory holds the word's planes in site index order
    // (graphs: storage order, the labels the neighbour table uses)
    for (int64_t i = threadIdx.x; i < a.N; i += blockDim.x) {
      const int64_t g = (a.perm ? i : dev_site(a.xs, i)) * a.V;
      sm[i] = gn[g];
      sm[a.N + i] = gp[g];
    }
    n = sm;
    p = sm + a.N;
  }
  const int z = Z ? Z : a.z, fields = SMEM ? z + 1 : 2 * z + 1;
  const uint32_t makers = blockDim.x / 32 - 1;
  uint32_t* ring = reinterpret_cast<uint32_t*>(sm + (SMEM ? 2 * a.N : 0));  // [3][makers][fields][32]
  uint64_t* swaps = reinterpret_cast<uint64_t*>(ring + 3 * makers * fields * 32);  // [2][makers][32]
  uint32_t* stamps = reinterpret_cast<uint32_t*>(swaps + 2 * makers * 32);  // [makers][2][hmask + 1]
  for (uint32_t b = threadIdx.x; b < 2 * makers * (a.hmask + 1); b += blockDim.x) stamps[b] = 0;
  const uint32_t per_sweep = (uint32_t)((a.N + 31) / 32), batches = per_sweep * (uint32_t)a.nsweeps;
  const uint64_t range = (uint64_t)a.N * (uint64_t)z;
  const uint32_t earlier = (1u << lane) - 1u;  // lanes of the earlier attempts
  // element of site i in n and p (a graph's labels and a shared plane's are positions)
  auto at = [&](uint32_t i) -> uint32_t {
    return SMEM || a.perm ? i : (uint32_t)dev_site(a.xs, i);
  };

  auto make = [&](uint32_t batch, uint32_t* out, uint32_t* s0) {
    const uint32_t s = batch / per_sweep;
    const int64_t k = (int64_t)(batch - s * per_sweep) * 32 + lane;
    const bool live = k < a.N;
    const uint32_t r = live ? (uint32_t)draw_bond(a.rk, a.t0 + s, (uint32_t)k, w, range) : 0u;
    // this lane's bond (i, j) and the neighbours of both: drawn by canonical
    // site and slot, then (graphs) followed in storage positions
    uint32_t i = r / (uint32_t)z;
    const int sel = (int)(r - i * (uint32_t)z);
    if (a.perm && live) i = (uint32_t)a.perm[i];
    uint32_t ni_[8], nj_[8];
    neighbours(a, z, i, ni_);
    uint32_t j = 0;
#pragma unroll
    for (int s2 = 0; s2 < 8; ++s2)
      if (s2 == sel) j = ni_[s2];
    neighbours(a, z, j, nj_);
    // bit o of a table's OR: attempt o writes a site this attempt reads (or
    // one that shares its word)
    uint32_t* s1 = s0 + a.hmask + 1;
    auto h0 = [&](uint32_t x) { return x & a.hmask; };
    auto h1 = [&](uint32_t x) { return (x * 0x9E3779B1u) >> a.hshift; };
    if (live) {
      atomicOr(&s0[h0(i)], 1u << lane);
      atomicOr(&s0[h0(j)], 1u << lane);
      atomicOr(&s1[h1(i)], 1u << lane);
      atomicOr(&s1[h1(j)], 1u << lane);
    }
    __syncwarp();
    // site by site: a site's writers are among both words'
    uint32_t conf = (s0[h0(i)] & s1[h1(i)]) | (s0[h0(j)] & s1[h1(j)]);
#pragma unroll
    for (int slot = 0; slot < 8; ++slot) {
      if (slot >= z) break;
      conf |= (s0[h0(ni_[slot])] & s1[h1(ni_[slot])]) | (s0[h0(nj_[slot])] & s1[h1(nj_[slot])]);
    }
    __syncwarp();
    if (live) {
      s0[h0(i)] = 0;
      s0[h0(j)] = 0;
      s1[h1(i)] = 0;
      s1[h1(j)] = 0;
    }
    // the other neighbours of i, then of j, without the partner
    uint32_t site[16];
    site[0] = at(i);
    site[1] = at(j);
    int fi = 2, fj = 1 + z;
#pragma unroll
    for (int slot = 0; slot < 8; ++slot) {
      if (slot >= z) break;
      const bool other_i = ni_[slot] != j, other_j = nj_[slot] != i;
      const uint32_t ei = at(ni_[slot]), ej = at(nj_[slot]);
      if constexpr (SMEM) {
        uint16_t* o = reinterpret_cast<uint16_t*>(out);
        if (other_i) o[((fi >> 1) * 32 + lane) * 2 + (fi & 1)] = (uint16_t)ei;
        if (other_j) o[((fj >> 1) * 32 + lane) * 2 + (fj & 1)] = (uint16_t)ej;
      } else {
        if (other_i) out[fi * 32 + lane] = ei;
        if (other_j) out[fj * 32 + lane] = ej;
      }
      fi += other_i;
      fj += other_j;
    }
    if constexpr (SMEM) {
      out[lane] = site[0] | site[1] << 16;
    } else {
      out[lane] = site[0];
      out[32 + lane] = site[1];
    }
    out[(fields - 1) * 32 + lane] = conf;
  };

  // warp 0's attempt of a batch: elements (i, j, the others of i, those of j) and conflicts
  uint32_t e[16], conf = 0;
  auto take = [&](const uint32_t* in) {
    conf = in[(fields - 1) * 32 + lane];
#pragma unroll
    for (int f = 0; f < 16; ++f) {
      if (f >= 2 * z) break;
      if constexpr (SMEM) e[f] = (in[(f >> 1) * 32 + lane] >> (16 * (f & 1))) & 0xFFFFu;
      else e[f] = in[f * 32 + lane];
    }
  };
  auto apply = [&](uint64_t* swap_out) {
    uint64_t sw = 0;
    uint32_t pending = __ballot_sync(0xffffffffu, (conf >> lane) & 1u);
    while (pending) {
      const bool ready = ((pending >> lane) & 1u) && !(conf & pending & earlier);
      if (ready) {
        const uint64_t vi = n[(int64_t)e[0] * st], vj = n[(int64_t)e[1] * st];
        uint64_t x[16];
#pragma unroll
        for (int f = 2; f < 16; ++f) {
          if (f >= 2 * z) break;
          x[f] = n[(int64_t)e[f] * st];
        }
        uint64_t ci2 = 0, ci1 = 0, ci0 = 0, cj2 = 0, cj1 = 0, cj0 = 0;
#pragma unroll
        for (int f = 2; f < 16; ++f) {
          if (f >= 2 * z) break;
          if (f < 1 + z) add3(ci2, ci1, ci0, x[f]);
          else add3(cj2, cj1, cj0, x[f]);
        }
        // at most m occupied among the other neighbours of i and of j
        sw = (vi ^ vj) & le3<M>(ci2, ci1, ci0) & le3<M>(cj2, cj1, cj0);
        if constexpr (SMEM) {
          n[e[0]] = vi ^ sw;
          n[e[1]] = vj ^ sw;
        } else if (sw) {
          n[(int64_t)e[0] * st] = vi ^ sw;
          n[(int64_t)e[1] * st] = vj ^ sw;
          atomicAnd(reinterpret_cast<unsigned long long*>(p + (int64_t)e[0] * st), (unsigned long long)~sw);
          atomicAnd(reinterpret_cast<unsigned long long*>(p + (int64_t)e[1] * st), (unsigned long long)~sw);
        }
      }
      pending &= ~__ballot_sync(0xffffffffu, ready);
      __syncwarp();
    }
    if constexpr (SMEM) swap_out[lane] = sw;
  };
  // the bits of p that a batch's swaps clear
  auto clear = [&](const uint32_t* in, const uint64_t* swap) {
    const uint64_t sw = swap[lane];
    if (!sw) return;
    // in halves: shared memory has 32-bit atomics
    uint32_t* pi = reinterpret_cast<uint32_t*>(p + (in[lane] & 0xFFFFu));
    uint32_t* pj = reinterpret_cast<uint32_t*>(p + (in[lane] >> 16));
    const uint32_t a0 = (uint32_t)sw, a1 = (uint32_t)(sw >> 32);
    if (a0) {
      atomicAnd(pi, ~a0);
      atomicAnd(pj, ~a0);
    }
    if (a1) {
      atomicAnd(pi + 1, ~a1);
      atomicAnd(pj + 1, ~a1);
    }
  };

  // turn t: the makers prepare batches t makers .., warp 0 applies those of
  // turn t - 1, the makers clear p for those of turn t - 2
  const uint32_t turns = (batches + makers - 1) / makers + 2;
  const int batch_words = fields * 32;
  __syncthreads();
  for (uint32_t t = 0; t < turns; ++t) {
    if (warp > 0) {
      const uint32_t m = (uint32_t)warp - 1, b = t * makers + m;
      uint32_t* slot = ring + ((t % 3) * makers + m) * batch_words;
      if (b < batches) make(b, slot, stamps + (size_t)m * 2 * (a.hmask + 1));
      if (SMEM && t >= 2 && b - 2 * makers < batches)
        clear(ring + (((t + 1) % 3) * makers + m) * batch_words, swaps + ((t & 1) * makers + m) * 32);
    } else if (t > 0) {
      const uint32_t b0 = (t - 1) * makers, count = b0 < batches ? min(batches - b0, makers) : 0u;
      const uint32_t* in = ring + ((t + 2) % 3) * makers * batch_words;
      uint64_t* swap_out = swaps + ((t + 1) & 1) * makers * 32;
      for (uint32_t m = 0; m < count; ++m) {
        take(in + m * batch_words);
        apply(swap_out + m * 32);
      }
    }
    __syncthreads();
  }
  if constexpr (SMEM) {
    for (int64_t i = threadIdx.x; i < a.N; i += blockDim.x) {
      const int64_t g = (a.perm ? i : dev_site(a.xs, i)) * a.V;
      gn[g] = sm[i];
      gp[g] = sm[a.N + i];
    }
  }
}

template <int Z, int M, bool SMEM>
cudaError_t launch_k(const SeqArgs& a, unsigned words, int makers, size_t smem, cudaStream_t st) {
  auto kern = k_sequential<Z, M, SMEM>;
  // the kernel's attribute, not the launch's: always the most, so that host
  // threads on lattices of different sizes do not take it from each other
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMost);
  if (e != cudaSuccess) return e;
  kern<<<words, 32 * (makers + 1), smem, st>>>(a);
  return cudaGetLastError();
}

template <int Z, bool SMEM>
cudaError_t launch_m(const SeqArgs& a, int m, unsigned words, int makers, size_t smem, cudaStream_t st) {
  switch (m < 7 ? m : 7) {
#define KA_CASE(MM) \
  case MM:          \
    return launch_k<Z, (Z == 0 || MM < Z ? MM : 0), SMEM>(a, words, makers, smem, st);
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

template <bool SMEM>
cudaError_t launch_z(const SeqArgs& a, int m, unsigned words, int makers, size_t smem, cudaStream_t st) {
  // instances of their own where the loop over the neighbours costs time; with
  // the planes in global memory they were slower (L = 32: 1.67 ms a sweep, all
  // loads at once, against 1.15)
  if constexpr (SMEM) {
    if (a.z == 4) return launch_m<4, SMEM>(a, m, words, makers, smem, st);
    if (a.z == 6) return launch_m<6, SMEM>(a, m, words, makers, smem, st);
  }
  return launch_m<0, SMEM>(a, m, words, makers, smem, st);
}

}  // namespace
}  // namespace ka

extern "C" ka_status ka_sweep_sequential(ka_ctx* c, int64_t nsweeps) {
  ka::NvtxRange nvtx_range("ka_sweep_sequential");
  using namespace ka;
  if (!c || nsweeps < 0) return KA_EINVAL;
  if (ka_status st = valid_state(c, "sequential sweep")) return st;
  if (c->sweep + nsweeps > ((int64_t)1 << 32)) {
    c->err = "sweep counter would pass 2^32";
    return KA_EINVAL;
  }
  if ((uint64_t)c->N * (uint64_t)c->z > 0xFFFFFFFFull) {
    c->err = "N z must stay below 2^32";
    return KA_EINVAL;
  }
  if (nsweeps == 0) return KA_OK;
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess || prev == c->device) prev = -1;
  if (prev >= 0) cudaSetDevice(c->device);
  SeqArgs a{};
  a.n = c->pl.n;
  a.p = c->pl.p;
  a.nbr = c->pencil ? nullptr : c->g.nbr;
  a.N = c->N;
  a.z = c->z;
  a.d = c->d;
  a.L = c->L;
  a.V = c->pl.V;
  a.xs = c->pl.xs;
  a.perm = c->g.perm;
  a.plane_elems = c->pl.plane_elems();
  a.rk = c->rk;
  const unsigned words = (unsigned)(c->R / 64);
  const bool smem = 2 * c->N <= kSmemWords;
  // stamp tables in what the planes (if in shared memory) and the ring leave
  const size_t planes = smem ? (size_t)2 * c->N * sizeof(uint64_t) : 0;
  auto smem_for = [&](int makers, uint32_t stamps) {
    const size_t ring = (size_t)32 * (3 * 4 * (smem ? c->z + 1 : 2 * c->z + 1) + 2 * 8);
    return planes + (size_t)makers * (ring + 2 * (size_t)stamps * 4);
  };
  int makers = kMakers;
  uint32_t H = kMaxStamps;
  // no more stamps than sites (a power of two), nor than there is room for
  if (smem)
    while (H > 32 && H >= 2 * (uint64_t)c->N) H >>= 1;
  while (H > 32 && smem_for(makers, H) > kSmemMost) H >>= 1;
  // Words beyond what runs at once take turns: of seven makers and three, and of the
  // stamps down to 128 to 512 by the sites an attempt reads (fewer, more false
  // conflicts), the most with the fewest turns; but three makers where three or
  // more CTAs would share an SM anyway, whose warps then wait for each other.
  // us a sweep with seven makers and 2048 stamps whatever the words, and so: 1024
  // words of L = 4 27, 6.0; of L = 8 78, 22; 800 of L = 12 166, 74; 1024 of d = 1,
  // L = 64 8.0, 4.7 (one warp a word, many to an SM: 17, 54, 142, 4.8).
  if (smem) {
    auto per_sm = [&](int mk, uint32_t stamps) {
      return std::min<size_t>(kSmThreads / (32 * (mk + 1)), kSmSmem / (smem_for(mk, stamps) + 1024));
    };
    auto turns = [&](int mk, uint32_t stamps) {
      const size_t at_once = std::max<size_t>(1, per_sm(mk, stamps) * (size_t)std::max(0, c->sms));
      return (words + at_once - 1) / at_once;
    };
    const uint32_t most = H, least = c->z <= 2 ? 128 : c->z <= 4 ? 256 : 512;
    for (int mk : {kMakers, kFewMakers})
      for (uint32_t h = most; h == most || h >= least; h /= 2) {
        const size_t t = turns(mk, h), best = turns(makers, H);
        const bool crowded = mk < makers && (int)words > 2 * c->sms && per_sm(makers, H) >= 3;
        if (t < best || (t == best && crowded)) {
          makers = mk;
          H = h;
        }
      }
  }
  uint32_t log2H = 0;
  while ((1u << log2H) < H) ++log2H;
  a.hmask = H - 1;
  a.hshift = 32 - log2H;
  const size_t smem_bytes = smem_for(makers, H);
  if (smem_bytes > kSmemMost) {
    if (prev >= 0) cudaSetDevice(prev);
    c->err = "sequential sweep: shared memory plan too large";
    return KA_EINVAL;
  }
  // launches of at most about 2^20 attempts each
  const int64_t chunk = std::max<int64_t>(1, ((int64_t)1 << 20) / c->N);
  cudaError_t e = cudaSuccess;
  for (int64_t done = 0; done < nsweeps && !e; done += chunk) {
    a.t0 = (uint32_t)(c->sweep + done);
    a.nsweeps = (int)std::min<int64_t>(chunk, nsweeps - done);
    e = smem ? launch_z<true>(a, c->m, words, makers, smem_bytes, c->stream)
             : launch_z<false>(a, c->m, words, makers, smem_bytes, c->stream);
  }
  if (prev >= 0) cudaSetDevice(prev);
  if (e) {
    c->err = std::string("sequential sweep: ") + cudaGetErrorString(e);
    return KA_ECUDA;
  }
  c->sweep += nsweeps;
  return KA_OK;
}
