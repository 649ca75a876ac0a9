// ka_resident_cubic_d4.cu -- on-chip cubic sweeps of dimension 4.
#include "ka_resident_cubic.cuh"

namespace ka {
namespace resident {
template cudaError_t launch_cubic_d<4>(const Args&, int, int, unsigned, int, cudaStream_t);
}  // namespace resident
}  // namespace ka
