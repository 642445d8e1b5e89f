#include "ptebd_jacobi64.cuh"

namespace ptebd {
namespace jac {
template cudaError_t prepare64<16>();
template cudaError_t launch64<16>(const LayerArgs<double>&, cudaStream_t);
}  // namespace jac
}  // namespace ptebd
