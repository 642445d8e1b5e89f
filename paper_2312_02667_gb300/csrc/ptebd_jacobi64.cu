// The Jacobi SVD kernels of complex128 matrices (ptebd_jacobi.cuh).
#include "ptebd_jacobi.cuh"

namespace ptebd {

namespace {

// MAXRPL: rows a lane holds of the tallest matrix of the launch (ldw / 32).
template <int MAXRPL>
__global__ void __launch_bounds__(256, 1) k_jacobi64(LayerArgs<double> A, int area) {
    extern __shared__ __align__(128) unsigned char smem[];
    const jac::Start<double> s = jac::start<double>(A, area, smem);
    if (!s.go) return;
    if (s.rows <= 32) {
        jac::jacobi_body<double, 1, true>(A, s.W, s.rows, s.cols, blockIdx.x, area, s.T, s.cbuf);
    } else if (MAXRPL <= 2 || s.rows <= 64) {
        jac::jacobi_body<double, 2, true>(A, s.W, s.rows, s.cols, blockIdx.x, area, s.T, s.cbuf);
    } else if constexpr (MAXRPL >= 4) {
        if (MAXRPL == 4 || s.rows <= 128) {
            jac::run_body<double, 4>(A, s);
        } else if constexpr (MAXRPL >= 8) {
            if (MAXRPL == 8 || s.rows <= 256) {
                jac::run_body<double, 8>(A, s);
            } else if constexpr (MAXRPL >= 16) {
                jac::jacobi_body<double, 16, false>(A, s.W, s.rows, s.cols, blockIdx.x, area, s.T, s.cbuf);
            }
        }
    }
}

template <int MAXRPL> cudaError_t set_smem() {
    return cudaFuncSetAttribute(k_jacobi64<MAXRPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, jac::kSmemMax);
}

}  // namespace

template <> cudaError_t jacobi_prepare<double>() {
    cudaError_t e = set_smem<2>();
    if (e == cudaSuccess) e = set_smem<4>();
    if (e == cudaSuccess) e = set_smem<8>();
    if (e == cudaSuccess) e = set_smem<16>();
    return e;
}

template <> cudaError_t launch_jacobi<double>(const LayerArgs<double>& a, cudaStream_t s) {
    const int area = jac::column_area<double>(a.ldw, false);
    const size_t smem = jac::table_bytes<double>() + area;
    const int threads = 32 * jac::warps_for(a.ldw, false, 8);
    if (a.ldw > 256)
        k_jacobi64<16><<<a.count, threads, smem, s>>>(a, area);
    else if (a.ldw > 128)
        k_jacobi64<8><<<a.count, threads, smem, s>>>(a, area);
    else if (a.ldw > 64)
        k_jacobi64<4><<<a.count, threads, smem, s>>>(a, area);
    else
        k_jacobi64<2><<<a.count, threads, smem, s>>>(a, area);
    return cudaGetLastError();
}

}  // namespace ptebd
