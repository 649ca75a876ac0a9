// ka_resident_cubic.cuh -- on-chip sweeps of small cubic lattices, d = 2, 3, 4
// (ka_resident.cuh): one cluster per word, one launch for all sweeps of a call.
//
// The work of a group (mu, par) is that of ka_cubic_stream.cuh: masks of the
// perpendicular counts, two Philox blocks and the four classes on each
// four-site segment of the active pencils, one segment per thread, planes in
// split-row order.  For mu = 0 the segments of a row are consecutive lanes and
// trade by shuffles.  For mu > 0 lanes take consecutive pencils (so shared
// memory is read without bank conflicts) and the segments of a pencil lie in
// different warps: they trade through shared memory, first the segment's first
// site after classes 0 and 1 with its rule mask, then the swap of the class-3
// bond that crosses.
//
// What a group sends bounds it: a receiver takes about 1.5 cycles per element
// of st.async whatever its size (8-byte elements for mu > 0: L = 20, four CTAs,
// 12.7 us a sweep), so elements are 16 bytes: chunks of a row for mu = 0, two
// neighbouring pencils' words, brought together by lane pairs, for mu > 0.
// Instantiated per dimension in ka_resident_cubic_d*.cu.
#pragma once

#define KA_RESIDENT_DEVICE
#include "ka_resident.cuh"

namespace ka {
namespace resident {
namespace {

__device__ __forceinline__ uint64_t okmask(uint64_t x, uint64_t A, uint64_t B) {
  return (x & A) | (~x & B);
}

// A = [count <= M-1], B = [count <= M] of K words (K = 2, 4 or 6)
template <int K, int M>
__device__ __forceinline__ void masks(const uint64_t (&x)[K], uint64_t& A, uint64_t& B) {
  uint64_t b0, b1, b2;
  if constexpr (K == 2) {
    b0 = x[0] ^ x[1];
    b1 = x[0] & x[1];
    b2 = 0;
  } else {
    const uint64_t s1 = x[0] ^ x[1] ^ x[2], c1 = (x[0] & x[1]) | (x[2] & (x[0] | x[1]));
    if constexpr (K == 4) {
      const uint64_t k = s1 & x[3];
      b0 = s1 ^ x[3];
      b1 = c1 ^ k;
      b2 = c1 & k;
    } else {
      const uint64_t s2 = x[3] ^ x[4] ^ x[5], c2 = (x[3] & x[4]) | (x[5] & (x[3] | x[4]));
      const uint64_t k = s1 & s2;
      b0 = s1 ^ s2;
      b1 = c1 ^ c2 ^ k;
      b2 = (c1 & c2) | (k & (c1 | c2));
    }
  }
  // [count <= t], t a constant
  auto le = [&](int t) -> uint64_t {
    if (t < 0) return 0ull;
    if (t >= K) return ~0ull;
    const uint64_t g0 = (t & 1) ? 0ull : b0;
    const uint64_t g1 = (t & 2) ? (b1 & g0) : (b1 | g0);
    return ~((t & 4) ? (b2 & g1) : (b2 | g1));
  };
  A = le(M - 1);
  B = le(M);
}

template <int D, int M, int C, bool B>
__global__ void __launch_bounds__(1024) k_resident_cubic(const __grid_constant__ Args a) {
  constexpr int K = 2 * (D - 1);
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ Unit su;
  __shared__ __align__(8) uint64_t bars[2];
  const uint32_t rank = cluster_rank();
  unit_of<B>(a, blockIdx.x / C, su);
  uint32_t t = su.t_base + a.from, left_to_run = su.count > a.from ? min(su.count - a.from, a.most) : 0u;
  if (left_to_run == 0) return;  // the whole cluster: one unit
  const int L = a.L, Lh = L / 2, S = L / 4;
  const int st1 = L, st2 = D > 2 ? L * L : 0, st3 = D > 3 ? L * L * L : 0;  // strides of y, z, w
  const int N = (D == 2 ? L : D == 3 ? L * L : L * L * L) * L;
  const int NP = N / L / 2;            // active pencils of a group
  const int PC = share_of(NP, C);      // of which this CTA takes at most
  const int P0 = (int)rank * PC;
  const int own = min(PC, max(0, NP - P0));
  const int tid = threadIdx.x, it = tid;
  // x: a segment's first site after classes 0 and 1 and its mask; xs: the
  // crossing swap; f: the swapped bits of every site (if fsmem)
  uint64_t* n = reinterpret_cast<uint64_t*>(dsm);
  ulonglong2* x = reinterpret_cast<ulonglong2*>(n + N);
  uint64_t* xs = reinterpret_cast<uint64_t*>(x + blockDim.x);
  uint64_t* f = xs + blockDim.x;
  const bool fsmem = a.fsmem != 0;
  const Peers<C> peers(smem_addr(dsm), rank);
  const uint32_t naddr = smem_addr(n);
  GroupEnd ge{smem_addr(bars), 0u, false};
  if (tid < 2) bar_init(ge.bars + 8 * tid, blockDim.x / 32);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  const uint32_t bytes = (uint32_t)(NP - own) * (uint32_t)L * 8u;  // of a group, from the others
  load_plane(su, n, N);
  if (fsmem)
    for (int i = tid; i < N; i += blockDim.x) f[i] = 0;

  // This thread's segment.  Rows (mu = 0): segment rs of row P0 + rj, warps hold
  // whole rows.  Pencils (mu > 0): segment ps of pencil P0 + pj.  Row or
  // pencil index = i + (L / 2) (o1 + L o2): i halves the first perpendicular
  // coordinate (y for mu = 0, x for mu > 0), o1, o2 are the others.
  const int lane = tid & 31, PW = 32 / S, gj = lane / S, rs = lane - gj * S;
  const int rj = (tid >> 5) * PW + gj, ps = tid / PC, pj = tid - ps * PC;
  const bool rlive = gj < PW && rj < own, plive = ps < S && pj < own;
  const int prev = gj < PW ? (rs == 0 ? lane + S - 1 : lane - 1) : lane;
  const int next = gj < PW ? (rs == S - 1 ? lane - S + 1 : lane + 1) : lane;
  const int pnext = ps == S - 1 ? pj : tid + PC, pprev = ps == 0 ? (S - 1) * PC + pj : tid - PC;
  const bool odd = tid & 1;
  auto split = [&](int r, int& i, int& o1, int& o2) {
    i = r % Lh;
    r /= Lh;
    o1 = D > 2 ? r % L : 0;
    o2 = D > 3 ? r / L : 0;
  };
  int ri, ro1, ro2, pi, po1, po2;
  split(P0 + rj, ri, ro1, ro2);
  split(P0 + pj, pi, po1, po2);
  auto around = [&](int c, int stride, int& up, int& down) {
    up = c == L - 1 ? -(L - 1) * stride : stride;
    down = c == 0 ? (L - 1) * stride : -stride;
  };

  uint64_t g0, g1, g2, g3;  // the gate words of the four bonds
  auto gates = [&](uint32_t tt, int mu, int par) {
    uint32_t site, step;  // the canonical site of the segment's first position
    if (mu == 0) {
      const int y = 2 * ri + ((par ^ ro1 ^ ro2) & 1);
      site = (uint32_t)(4 * rs + y * st1 + ro1 * st2 + ro2 * st3);
      step = 1;
    } else {
      const int xx = 2 * pi + ((par ^ po1 ^ po2) & 1);
      const int s1 = mu == 1 ? st2 : st1, s2 = mu == 3 ? st2 : st3;
      step = (uint32_t)(mu == 1 ? st1 : mu == 2 ? st2 : st3);
      site = (uint32_t)(xx + po1 * s1 + po2 * s2) + 4u * (uint32_t)ps * step;
    }
    const uint32_t cls = (uint32_t)(4 * (2 * mu + par));
    const uint4 g01 = philox(make_uint4(tt, cls, site, su.word), unit_keys<B>(a, su));
    const uint4 g23 = philox(make_uint4(tt, cls + 2, site + 2 * step, su.word), unit_keys<B>(a, su));
    g0 = lo64(g01);
    g1 = hi64(g01);
    g2 = lo64(g23);
    g3 = hi64(g23);
  };
  // the swaps of four sites go to f, or straight to p
  auto mark = [&](int i0, int i1, int i2, int i3, uint64_t f0, uint64_t f1, uint64_t f2, uint64_t f3) {
    if (fsmem) {
      const uint64_t e0 = f[i0], e1 = f[i1], e2 = f[i2], e3 = f[i3];
#ifdef KA_SLOW_MARKS  // test builds: a delay here lets the other warps run ahead
      KA_SLOW_MARKS;
#endif
      f[i0] = e0 | f0;
      f[i1] = e1 | f1;
      f[i2] = e2 | f2;
      f[i3] = e3 | f3;
    } else {
      clear_bits(su.p + i0, f0);
      clear_bits(su.p + i1, f1);
      clear_bits(su.p + i2, f2);
      clear_bits(su.p + i3, f3);
    }
  };

  cluster_arrive();
  gates(t, 0, 0);
  cluster_wait();
  for (; left_to_run; --left_to_run, ++t) {
#pragma unroll 1
    for (int par = 0; par < 2; ++par) {  // mu = 0
      const int y = 2 * ri + ((par ^ ro1 ^ ro2) & 1);
      const int e0 = y * st1 + ro1 * st2 + ro2 * st3 + 2 * rs, d0 = e0 + Lh;  // even, odd sites
      uint64_t nn[4], mA[4], mB[4], f0, f1, f2, f3;
#pragma unroll
      for (int k = 0; k < 4; ++k) nn[k] = mA[k] = mB[k] = 0;
      if (rlive) {
        int nb[K];
        around(y, st1, nb[0], nb[1]);
        if constexpr (D > 2) around(ro1, st2, nb[2], nb[3]);
        if constexpr (D > 3) around(ro2, st3, nb[4], nb[5]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int b0 = h ? d0 : e0;
          const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(n + b0);
          nn[h] = c.x;
          nn[h + 2] = c.y;
          uint64_t q0[K], q1[K];
#pragma unroll
          for (int k = 0; k < K; ++k) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(n + b0 + nb[k]);
            q0[k] = v.x;
            q1[k] = v.y;
          }
          masks<K, M>(q0, mA[h], mB[h]);
          masks<K, M>(q1, mA[h + 2], mB[h + 2]);
        }
      }
      const uint64_t left = __shfl_sync(0xffffffffu, nn[3], prev);
      uint64_t sw = (nn[0] ^ nn[1]) & g0 & okmask(left, mA[0], mB[0]) & okmask(nn[2], mA[1], mB[1]);
      nn[0] ^= sw;
      nn[1] ^= sw;
      f0 = f1 = sw;
      sw = (nn[1] ^ nn[2]) & g1 & okmask(nn[0], mA[1], mB[1]) & okmask(nn[3], mA[2], mB[2]);
      nn[1] ^= sw;
      nn[2] ^= sw;
      f1 |= sw;
      f2 = sw;
      const uint64_t right = __shfl_sync(0xffffffffu, nn[0], next);
      const uint64_t okn = __shfl_sync(0xffffffffu, okmask(nn[1], mA[0], mB[0]), next);
      sw = (nn[2] ^ nn[3]) & g2 & okmask(nn[1], mA[2], mB[2]) & okmask(right, mA[3], mB[3]);
      nn[2] ^= sw;
      nn[3] ^= sw;
      f2 |= sw;
      f3 = sw;
      sw = (nn[3] ^ right) & g3 & okmask(nn[2], mA[3], mB[3]) & okn;
      nn[3] ^= sw;
      f3 |= sw;
      const uint64_t in = __shfl_sync(0xffffffffu, sw, prev);
      nn[0] ^= in;
      f0 |= in;
      if (rlive) {
        *reinterpret_cast<ulonglong2*>(n + e0) = make_ulonglong2(nn[0], nn[2]);
        *reinterpret_cast<ulonglong2*>(n + d0) = make_ulonglong2(nn[1], nn[3]);
        peers.st2(naddr + 8 * e0, nn[0], nn[2], ge.bar());
        peers.st2(naddr + 8 * d0, nn[1], nn[3], ge.bar());
      }
      ge.arrive(bytes);
      if (rlive) mark(e0, d0, e0 + 1, d0 + 1, f0, f1, f2, f3);
      gates(t, par, par ^ 1);
      ge.wait(su.err);
    }
#pragma unroll 1
    for (int g = 2; g < 2 * D; ++g) {
      const int mu = g >> 1, par = g & 1;
      const int TS = mu == 1 ? st1 : mu == 2 ? st2 : st3;
      const int s1 = mu == 1 ? st2 : st1, s2 = mu == 3 ? st2 : st3;
      const int act = (par ^ po1 ^ po2) & 1;
      const int b0 = act * Lh + pi + po1 * s1 + po2 * s2 + 4 * ps * TS;
      uint64_t nn[4], f0 = 0, f1 = 0, f2 = 0, f3 = 0, A2 = 0, B2 = 0, A3 = 0, B3 = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) nn[k] = 0;
      if (plive) {
        int nb[K];
        // the x neighbours lie in the other half of the row
        nb[0] = act == 0 ? Lh + (pi == 0 ? Lh - 1 : -1) : -Lh;
        nb[1] = act == 0 ? Lh : (pi == Lh - 1 ? -2 * Lh + 1 : 1 - Lh);
        if constexpr (D > 2) around(po1, s1, nb[2], nb[3]);
        if constexpr (D > 3) around(po2, s2, nb[4], nb[5]);
        const uint64_t left = n[ps == 0 ? b0 + (L - 1) * TS : b0 - TS];
        uint64_t mA[4], mB[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int i = b0 + k * TS;
          nn[k] = n[i];
          uint64_t q[K];
#pragma unroll
          for (int v = 0; v < K; ++v) q[v] = n[i + nb[v]];
          masks<K, M>(q, mA[k], mB[k]);
        }
        // class 0: bond (0, 1); 0's other along-neighbour is the previous
        // segment's last site at its group-start value, 1's is 2
        uint64_t sw = (nn[0] ^ nn[1]) & g0 & okmask(left, mA[0], mB[0]) & okmask(nn[2], mA[1], mB[1]);
        nn[0] ^= sw;
        nn[1] ^= sw;
        f0 = f1 = sw;
        // class 1: bond (1, 2); other along-neighbours 0 and 3
        sw = (nn[1] ^ nn[2]) & g1 & okmask(nn[0], mA[1], mB[1]) & okmask(nn[3], mA[2], mB[2]);
        nn[1] ^= sw;
        nn[2] ^= sw;
        f1 |= sw;
        f2 = sw;
        x[tid] = make_ulonglong2(nn[0], okmask(nn[1], mA[0], mB[0]));
        A2 = mA[2];
        B2 = mB[2];
        A3 = mA[3];
        B3 = mB[3];
      }
      __syncthreads();
      if (plive) {
        // class 2: bond (2, 3); 3's other along-neighbour is the next
        // segment's first site, which only class 0 has written so far
        const ulonglong2 nx = x[pnext];
        uint64_t sw = (nn[2] ^ nn[3]) & g2 & okmask(nn[1], A2, B2) & okmask(nx.x, A3, B3);
        nn[2] ^= sw;
        nn[3] ^= sw;
        f2 |= sw;
        f3 = sw;
        // class 3: bond (3, the next segment's 0), whose rule mask came with it
        sw = (nn[3] ^ nx.x) & g3 & okmask(nn[2], A3, B3) & nx.y;
        nn[3] ^= sw;
        f3 |= sw;
        xs[tid] = sw;
#pragma unroll
        for (int k = 1; k < 4; ++k) n[b0 + k * TS] = nn[k];
      }
      if constexpr (C > 1) {
        // pencils 2i, 2i + 1 (lane pairs, both live or neither): the even lane
        // sends the words of sites 1 and 2, the odd one those of 3 and 0
        const uint64_t p1 = __shfl_xor_sync(0xffffffffu, odd ? nn[1] : nn[3], 1);
        const uint64_t p2 = __shfl_xor_sync(0xffffffffu, nn[2], 1);
        if (plive) {
          const uint32_t at = naddr + 8u * (uint32_t)(odd ? b0 - 1 + 3 * TS : b0 + TS);
          peers.st2(at, odd ? p1 : nn[1], odd ? nn[3] : p1, ge.bar());
          if (!odd) peers.st2(at + 8u * (uint32_t)TS, nn[2], p2, ge.bar());
        }
      }
      __syncthreads();
      if (plive) {
        const uint64_t in = xs[pprev];
        nn[0] ^= in;
        f0 |= in;
        n[b0] = nn[0];
      }
      if constexpr (C > 1) {
        const uint64_t p0 = __shfl_xor_sync(0xffffffffu, nn[0], 1);
        if (plive && odd) peers.st2(naddr + 8u * (uint32_t)(b0 - 1), p0, nn[0], ge.bar());
      }
      ge.arrive(bytes);
      if (plive) mark(b0, b0 + TS, b0 + 2 * TS, b0 + 3 * TS, f0, f1, f2, f3);
      const int gn = g + 1 < 2 * D ? g + 1 : 0;
      gates(gn ? t : t + 1, gn >> 1, gn & 1);
      ge.wait(su.err);
    }
    // Marks are made after the arrival, so a wait says nothing about other
    // warps' marks.  Inside a sweep none meet without a barrier between: the
    // two groups of mu = 0 have different rows, those of mu > 0 barriers of
    // their own.  The last group's would meet the next sweep's first and the
    // final loop's reads, so the CTA meets here (us a sweep without and with:
    // L = 16 6.4, 6.4; L = 20 9.7, 9.8; d = 2, L = 128, 256 replicas 10.6, 10.9).
    if (__syncthreads_or(ge.dead)) break;  // a wait ran out
  }
  store_plane(su, n, N, rank, C);
  if (fsmem)
    for (int i = tid; i < N; i += blockDim.x) clear_bits(su.p + i, f[i]);
  cluster_arrive();  // a CTA stays until the others have sent it all
  cluster_wait();
}

int64_t sites(int d, int L) {
  int64_t N = 1;
  for (int k = 0; k < d; ++k) N *= L;
  return N;
}

size_t smem_for(int64_t N, int threads, bool f) {
  return (size_t)N * 8 * (f ? 2 : 1) + (size_t)threads * 24;
}

constexpr size_t kCubicSmem = kSmemMax - 512;  // beside the unit and the mbarriers

template <int D, int M, int C, bool B>
cudaError_t launch_c(const Args& a, unsigned words, int threads, size_t smem, cudaStream_t st) {
  return launch_cluster(k_resident_cubic<D, M, C, B>, a, words, C, threads, smem, kCubicSmem, st);
}

template <int D, int M>
cudaError_t launch_m(const Args& a, unsigned words, int C, int threads, size_t smem, cudaStream_t st) {
  const bool b = a.units != nullptr;
  switch (C) {
    case 1:
      return b ? launch_c<D, M, 1, true>(a, words, threads, smem, st)
               : launch_c<D, M, 1, false>(a, words, threads, smem, st);
    case 2:
      return b ? launch_c<D, M, 2, true>(a, words, threads, smem, st)
               : launch_c<D, M, 2, false>(a, words, threads, smem, st);
    case 4:
      return b ? launch_c<D, M, 4, true>(a, words, threads, smem, st)
               : launch_c<D, M, 4, false>(a, words, threads, smem, st);
    case 8:
      return b ? launch_c<D, M, 8, true>(a, words, threads, smem, st)
               : launch_c<D, M, 8, false>(a, words, threads, smem, st);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace

template <int D>
cudaError_t launch_cubic_d(const Args& args, int L, int m, unsigned words, int C, cudaStream_t st) {
  const int64_t N = sites(D, L);
  const int threads = cubic_threads(N, L, C);
  if (threads > 1024) return cudaErrorInvalidValue;
  Args a = args;
  a.L = L;
  a.fsmem = smem_for(N, threads, true) <= kCubicSmem;
  const size_t smem = smem_for(N, threads, a.fsmem != 0);
  switch (m) {
#define KA_CASE(MM) \
  case MM:          \
    return launch_m<D, (MM < 2 * D ? MM : 0)>(a, words, C, threads, smem, st);
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

}  // namespace resident
}  // namespace ka
