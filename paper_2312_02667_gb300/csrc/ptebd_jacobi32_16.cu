#include "ptebd_jacobi32.cuh"

namespace ptebd {
namespace jac {
template cudaError_t prepare32<16>();
template cudaError_t launch32<16>(const LayerArgs<float>&, cudaStream_t);
}  // namespace jac
}  // namespace ptebd
