// The Jacobi SVD kernels of complex64 matrices (ptebd_jacobi.cuh), and what both precisions share.
#include "ptebd_jacobi.cuh"

namespace ptebd {

namespace {

// MAXRPL: rows a lane holds of the tallest matrix of the launch (ldw / 32).
template <int MAXRPL, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) k_jacobi(LayerArgs<float> A, int area) {
    extern __shared__ __align__(128) unsigned char smem[];
    const jac::Start<float> s = jac::start<float>(A, area, smem);
    if (!s.go) return;
    if (s.rows <= 64) {
        jac::jacobi_body<float, 2, true>(A, s.W, s.rows, s.cols, blockIdx.x, area, s.T, s.cbuf);
    } else if (MAXRPL <= 4 || s.rows <= 128) {
        jac::run_body<float, 4>(A, s);
    } else if constexpr (MAXRPL >= 8) {
        if (MAXRPL == 8 || s.rows <= 256) {
            jac::run_body<float, 8>(A, s);
        } else if constexpr (MAXRPL >= 16) {
            jac::jacobi_body<float, 16, false>(A, s.W, s.rows, s.cols, blockIdx.x, area, s.T, s.cbuf);
        }
    }
}

template <int MAXRPL, int THREADS> cudaError_t set_smem() {
    return cudaFuncSetAttribute(k_jacobi<MAXRPL, THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, jac::kSmemMax);
}

}  // namespace

int jacobi_block_width(int precision, int requested) {
    if (precision == PTEBD_FP64) return 8;
    return requested == 8 ? 8 : 16;
}

template <> cudaError_t jacobi_prepare<float>() {
    cudaError_t e = set_smem<4, 384>();
    if (e == cudaSuccess) e = set_smem<8, 256>();
    if (e == cudaSuccess) e = set_smem<16, 256>();
    return e;
}

template <> cudaError_t launch_jacobi<float>(const LayerArgs<float>& a, cudaStream_t s) {
    const bool half = a.nw == 8;  // half the warps and half the shared memory of a CTA
    const int area = jac::column_area<float>(a.ldw, half);
    const size_t smem = jac::table_bytes<float>() + area;
    if (a.ldw > 256)
        k_jacobi<16, 256><<<a.count, half ? 128 : 256, smem, s>>>(a, area);
    else if (a.ldw > 128)
        k_jacobi<8, 256><<<a.count, half ? 128 : 256, smem, s>>>(a, area);
    else
        k_jacobi<4, 384><<<a.count, 32 * jac::warps_for(a.ldw, half, 12), smem, s>>>(a, area);
    return cudaGetLastError();
}

}  // namespace ptebd
