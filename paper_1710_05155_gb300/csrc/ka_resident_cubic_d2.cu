// ka_resident_cubic_d2.cu -- on-chip cubic sweeps of dimension 2.
#include "ka_resident_cubic.cuh"

namespace ka {
namespace resident {
template cudaError_t launch_cubic_d<2>(const Args&, int, int, unsigned, int, cudaStream_t);
}  // namespace resident
}  // namespace ka
