// ka_cubic_stream_l64.cu -- instances of the group kernels for L = 64
// (one translation unit per side, so that they compile in parallel).
#define KA_STREAM_INSTANCES
#include "ka_cubic_stream.cuh"

namespace ka {
namespace stream {
template cudaError_t launch_l<64>(const Args&, int, cudaStream_t);
}  // namespace stream
}  // namespace ka
