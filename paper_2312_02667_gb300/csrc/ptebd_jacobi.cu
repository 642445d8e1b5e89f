// Launches of the Jacobi SVD: the class of kernels for a matrix height
// (ptebd_jacobi32.cuh, ptebd_jacobi64.cuh).
#include "ptebd_internal.h"

namespace ptebd {

namespace jac {
template <int MAXRPL> cudaError_t prepare32();
template <int MAXRPL> cudaError_t launch32(const LayerArgs<float>& a, cudaStream_t s);
template <int MAXRPL> cudaError_t prepare64();
template <int MAXRPL> cudaError_t launch64(const LayerArgs<double>& a, cudaStream_t s);
}  // namespace jac

int jacobi_block_width(int precision, int requested) {
    if (precision == PTEBD_FP64) return 8;
    return requested == 8 ? 8 : 16;
}

template <> cudaError_t jacobi_prepare<float>() {
    cudaError_t e = jac::prepare32<4>();
    if (e == cudaSuccess) e = jac::prepare32<8>();
    if (e == cudaSuccess) e = jac::prepare32<16>();
    if (e == cudaSuccess) e = jacobi_blocks_prepare();
    return e;
}

template <> cudaError_t launch_jacobi<float>(const LayerArgs<float>& a, cudaStream_t s) {
    return a.ldw > 256 ? jac::launch32<16>(a, s) : a.ldw > 128 ? jac::launch32<8>(a, s) : jac::launch32<4>(a, s);
}

template <> cudaError_t jacobi_prepare<double>() {
    cudaError_t e = jac::prepare64<2>();
    if (e == cudaSuccess) e = jac::prepare64<4>();
    if (e == cudaSuccess) e = jac::prepare64<8>();
    if (e == cudaSuccess) e = jac::prepare64<16>();
    return e;
}

template <> cudaError_t launch_jacobi<double>(const LayerArgs<double>& a, cudaStream_t s) {
    return a.ldw > 256   ? jac::launch64<16>(a, s)
           : a.ldw > 128 ? jac::launch64<8>(a, s)
           : a.ldw > 64  ? jac::launch64<4>(a, s)
                         : jac::launch64<2>(a, s);
}

}  // namespace ptebd
