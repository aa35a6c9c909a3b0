// The tcgen05 engine on 128 x 64 tiles (tc_kernel.cuh).
#include "tc_kernel.cuh"

namespace zf {
template cudaError_t tc_launch_tile<64, 1>(const TcArgs&, const TcMaps&, int, cudaStream_t);
}  // namespace zf
