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
  // us a sweep of one word on chip, against a launch per group: d = 3, L = 16
  // 6.4 / 9.9, L = 20 9.7 / 14.4, L = 24 14.8 / 14.6, L = 28 22.3 / 15.2; d = 2,
  // L = 128 10.6 / 12.  On chip up to 19 words run at once in that time, while
  // group launches grow with them: four words 6.4 / 11.6, 9.7 / 18.2, 14.8 / 16.9,
  // 22.4 / 24.5 (three: 22.3 / 22.6) and 10.6 / 48.
  if (d > 2 && words < (N > 16384 ? 4 : N > 8192 ? 2 : 1)) return 0;
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
