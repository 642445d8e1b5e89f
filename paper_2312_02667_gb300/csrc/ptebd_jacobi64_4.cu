#include "ptebd_jacobi64.cuh"

namespace ptebd {
namespace jac {
template cudaError_t prepare64<2>();
template cudaError_t launch64<2>(const LayerArgs<double>&, cudaStream_t);
template cudaError_t prepare64<4>();
template cudaError_t launch64<4>(const LayerArgs<double>&, cudaStream_t);
}  // namespace jac
}  // namespace ptebd
