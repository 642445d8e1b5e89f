// The Jacobi SVD kernels of complex128 matrices (ptebd_jacobi.cuh), by class of matrix
// height: MAXRPL is ldw / 32, the rows a lane holds of the tallest matrix of a launch.
// Each class is compiled in a translation unit of its own.
#pragma once
#include "ptebd_jacobi.cuh"

namespace ptebd {
namespace jac {

// CLUSTER: one cluster per matrix, else one CTA.
template <int MAXRPL, bool CLUSTER>
__global__ void __launch_bounds__(256, 1) k_jacobi64(LayerArgs<double> A, int area) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int n = CLUSTER ? cluster_size() : 1;
    const Start<double> s = start<double>(A, area, smem, blockIdx.x / n);
    if (!s.go) return;
    auto go = [&](auto rpl) {
        constexpr int RPL = decltype(rpl)::value;
        if constexpr (CLUSTER) run_cluster<double, RPL>(A, s);
        else if constexpr (RPL <= 2) run<double, RPL, kResident>(A, s);
        else run_alone<double, RPL>(A, s);
    };
    if (s.rows <= 32) {
        if (!CLUSTER || cluster_rank() == 0) run<double, 1, kResident>(A, s);
    } else if (MAXRPL <= 2 || s.rows <= 64) {
        go(std::integral_constant<int, 2>{});
    } else if constexpr (MAXRPL >= 4) {
        if (s.rows <= 96) {
            go(std::integral_constant<int, 3>{});
        } else if (MAXRPL == 4 || s.rows <= 128) {
            go(std::integral_constant<int, 4>{});
        } else if constexpr (MAXRPL >= 8) {
            if (s.rows <= 192) {
                go(std::integral_constant<int, 6>{});
            } else if (MAXRPL == 8 || s.rows <= 256) {
                go(std::integral_constant<int, 8>{});
            } else if constexpr (MAXRPL >= 16) {
                if (!CLUSTER || cluster_rank() == 0) run<double, 16, kStream>(A, s);
            }
        }
    }
}

template <int MAXRPL> cudaError_t prepare64() {
    const cudaError_t e = prepare_clusters(k_jacobi64<MAXRPL, true>);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_jacobi64<MAXRPL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
}

template <int MAXRPL> cudaError_t launch64(const LayerArgs<double>& a, cudaStream_t s) {
    const int area = column_area<double>(a.ldw, false);
    const size_t smem = table_bytes<double>() + area;
    const int threads = 32 * warps_for(a.ldw, false, 8);
    // The FP64 resolution of a complex64 state (refine == 1) counts all bonds as well, though
    // the decided ones return at once: how many are undecided is known on the device alone, and
    // while bonds grow it is most of them.  Counted as an eighth, clusters of 8 queue: circuits
    // of N = 400, chi = 128 and N = 140, chi = 200 take 167 and 329 ms instead of 134 and 310,
    // a routed 14 x 14 lattice at chi = 32 74.5 instead of 61.9; as a third, 136, 298 and 59.4.
    const int bonds = a.share > a.count ? a.share : a.count;
    const int n = a.ldw > 32 ? cluster_for(bonds, most_clusters(k_jacobi64<MAXRPL, true>).n) : 1;
    if (n > 1) return launch_cluster(k_jacobi64<MAXRPL, true>, a, n, threads, smem, area, s);
    k_jacobi64<MAXRPL, false><<<a.count, threads, smem, s>>>(a, area);
    return cudaGetLastError();
}

}  // namespace jac
}  // namespace ptebd
