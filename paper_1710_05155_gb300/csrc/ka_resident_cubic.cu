// ka_resident_cubic.cu -- which cubic lattices run on chip, and their launch
// (ka_resident_cubic.cuh).
#include "ka_resident.cuh"

namespace ka {
namespace resident {

template <int D>
cudaError_t launch_cubic_d(const Args& args, int L, int m, unsigned words, int C, cudaStream_t st);
extern template cudaError_t launch_cubic_d<2>(const Args&, int, int, unsigned, int, cudaStream_t);
extern template cudaError_t launch_cubic_d<3>(const Args&, int, int, unsigned, int, cudaStream_t);
extern template cudaError_t launch_cubic_d<4>(const Args&, int, int, unsigned, int, cudaStream_t);

int cubic_cluster(int d, int L, int64_t words, int sms) {
  if (d < 2 || d > 4 || L % 4 || L < 4 || L > 128) return 0;
  int64_t N = 1;
  for (int k = 0; k < d; ++k) N *= L;
  // n and the exchange slots (24 bytes for each of at most 1024 threads) in shared memory
  if (N * 8 + 24 * 1024 > (int64_t)kSmemMax - 512) return 0;
  // CTAs per word: a segment's latency bounds small shares, what a group sends
  // large clusters.  us a sweep with 1, 2, 4, 8: L = 8 4.5, 4.9, 5.2, 5.5; L = 12
  // 6.0, 5.1, 5.3, 5.8; L = 16 9.2, 6.6, 6.4, 7.0; L = 20 -, 11.5, 9.7, 10.3; L = 24
  // -, 21.0, 17.1, 14.8; d = 2, L = 128 -, 12.4, 10.6, 11.5.
  int C = N <= 1024 ? 1 : N <= 2048 ? 2 : N <= 8192 || d == 2 ? 4 : 8;
  while (cubic_threads(N, L, C) > 1024) C *= 2;
  // fewer once the words fill the device (L = 16, 128 words: 9.2 with one, 19.8 with four)
  while (C > 1 && words * C > sms && cubic_threads(N, L, C / 2) <= 1024) C /= 2;
  // every CTA has pencils: each must send in every group
  return (C - 1) * share_of((int)(N / L / 2), C) < N / L / 2 ? C : 0;
}

bool cubic_pays(int d, int L, int64_t planes, int C, int sms, int64_t n) {
  // us of a sweep, measured and fitted.  On chip: d = 3, L = 8 to 28 4.5, 5.2,
  // 6.4, 9.7, 14.8, 22.3; d = 2, L = 16, 64, 128 2.5, 3.6, 10.6; d = 4, L = 8, 12 10.8, 34;
  // for as many words as run at once.  A launch per group: 10 (L <= 16; 12 for
  // two planes and more) to 15 for up to four planes of a three-dimensional
  // lattice; 12 and 18 to 22 for every plane of the others.  A launch on chip
  // (planes in and out, the cluster) costs 12 us more, small lattices 8 to 10:
  // calls of 1, 2 and 3 sweeps of L = 16, 3 planes 12.4, 25, 37 in groups, on chip
  // 18, -, 30; L = 12 13, 25, 37, on chip -, 19, 24.
  double N = 1.0;
  for (int k = 0; k < d; ++k) N *= L;
  const double group = d == 3 ? (L > 16 ? 14.0 : planes > 1 ? 12.2 : 10.2) * (double)((planes + 3) / 4)
                              : (d == 2 ? 12.0 : 18.0) * (double)planes;
  const double chip = d == 3 ? 3.0 + 8.8e-4 * N : d == 2 ? 2.5 + 5.0e-4 * N : 5.0 + 1.4e-3 * N;
  const double waves = (double)((planes * C + sms - 1) / (sms > 0 ? sms : 1));
  const double launch = d == 3 && N < 4000.0 ? 8.0 + 1.0e-3 * N : 12.0;
  return group * (double)n > (launch + chip * (double)n) * waves;
}

cudaError_t launch_cubic(const Args& a, int d, int L, int m, unsigned words, int C,
                         cudaStream_t st) {
  if (m < 0 || m >= 2 * d) return cudaErrorInvalidValue;
  switch (d) {
    case 2: return launch_cubic_d<2>(a, L, m, words, C, st);
    case 3: return launch_cubic_d<3>(a, L, m, words, C, st);
    case 4: return launch_cubic_d<4>(a, L, m, words, C, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace resident
}  // namespace ka
