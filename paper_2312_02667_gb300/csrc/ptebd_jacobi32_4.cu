#include "ptebd_jacobi32.cuh"

namespace ptebd {
namespace jac {
template cudaError_t prepare32<4>();
template cudaError_t launch32<4>(const LayerArgs<float>&, cudaStream_t);
}  // namespace jac
}  // namespace ptebd
