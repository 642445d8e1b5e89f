// The Jacobi SVD kernels of complex64 matrices (ptebd_jacobi.cuh), by class of matrix
// height: MAXRPL is ldw / 32, the rows a lane holds of the tallest matrix of a launch.
// Each class is compiled in a translation unit of its own.
#pragma once
#include "ptebd_jacobi.cuh"

namespace ptebd {
namespace jac {

// 12 warps of 168 registers where the tile leaves room: at 256 rows (128 registers of
// columns) 8 warps of up to 255 are faster (152 of 200 x 200: 5.5 against 6.5 ms), at
// 512 rows 12 (75.7 -> 71.1 ms for 152 of 512 x 512).
template <int MAXRPL> constexpr int kThreads32 = MAXRPL == 8 ? 256 : 384;

template <int MAXRPL>
__global__ void __launch_bounds__(kThreads32<MAXRPL>, 1) k_jacobi(LayerArgs<float> A, int area) {
    extern __shared__ __align__(128) unsigned char smem[];
    const Start<float> s = start<float>(A, area, smem, blockIdx.x);
    if (!s.go) return;
    if (s.rows <= 64) {
        run<float, 2, kResident>(A, s);
    } else if (MAXRPL <= 4 || s.rows <= 128) {
        run_alone<float, 4>(A, s);
    } else if constexpr (MAXRPL >= 8) {
        if (s.rows <= 192) {
            run_alone<float, 6>(A, s);
        } else if (MAXRPL == 8 || s.rows <= 256) {
            run_alone<float, 8>(A, s);
        } else if constexpr (MAXRPL >= 16) {
            if (s.rows <= 384) run<float, 12, kStream>(A, s);
            else run<float, 16, kStream>(A, s);
        }
    }
}

// One cluster per matrix.
template <int MAXRPL>
__global__ void __launch_bounds__(256, 1) k_jacobi_cluster(LayerArgs<float> A, int area) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int n = cluster_size();
    const Start<float> s = start<float>(A, area, smem, blockIdx.x / n);
    if (!s.go) return;
    if (s.rows <= 64) {
        if (cluster_rank() == 0) run<float, 2, kResident>(A, s);
    } else if (MAXRPL <= 4 || s.rows <= 128) {
        run_cluster<float, 4>(A, s);
    } else if constexpr (MAXRPL >= 8) {
        if (s.rows <= 192) {
            run_cluster<float, 6>(A, s);
        } else if (MAXRPL == 8 || s.rows <= 256) {
            run_cluster<float, 8>(A, s);
        } else if constexpr (MAXRPL >= 16) {
            if (s.rows <= 384) run_cluster<float, 12>(A, s);
            else run_cluster<float, 16>(A, s);
        }
    }
}

template <int MAXRPL> cudaError_t prepare32() {
    const cudaError_t e = prepare_clusters(k_jacobi_cluster<MAXRPL>);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_jacobi<MAXRPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
}

template <int MAXRPL> cudaError_t launch32(const LayerArgs<float>& a, cudaStream_t s) {
    const bool half = a.nw == 8;  // half the warps and half the shared memory of a CTA
    const int area = column_area<float>(a.ldw, half);
    const size_t smem = table_bytes<float>() + area;
    const int n = half || a.ldw <= 64 ? 1
                                      : cluster_for(a.share > a.count ? a.share : a.count,
                                                    most_clusters(k_jacobi_cluster<MAXRPL>).n);
    if (n > 1) return launch_cluster(k_jacobi_cluster<MAXRPL>, a, n, 256, smem, area, s);
    k_jacobi<MAXRPL><<<a.count, 32 * warps_for(a.ldw, half, kThreads32<MAXRPL> / 32), smem, s>>>(a, area);
    return cudaGetLastError();
}

}  // namespace jac
}  // namespace ptebd
