#include "ptebd_jacobi32.cuh"

namespace ptebd {
namespace jac {
template cudaError_t prepare32<8>();
template cudaError_t launch32<8>(const LayerArgs<float>&, cudaStream_t);
}  // namespace jac
}  // namespace ptebd
