// The Jacobi SVD kernels of complex64 matrices (ptebd_jacobi.cuh), and what both precisions share.
#include "ptebd_jacobi.cuh"

namespace ptebd {

namespace {

// MAXRPL: rows a lane holds of the tallest matrix of the launch (ldw / 32).
template <int MAXRPL, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) k_jacobi(LayerArgs<float> A, int area) {
    extern __shared__ __align__(128) unsigned char smem[];
    const jac::Start<float> s = jac::start<float>(A, area, smem, blockIdx.x);
    if (!s.go) return;
    if (s.rows <= 64) {
        jac::run<float, 2, jac::kResident>(A, s);
    } else if (MAXRPL <= 4 || s.rows <= 128) {
        jac::run_alone<float, 4>(A, s);
    } else if constexpr (MAXRPL >= 8) {
        if (MAXRPL == 8 || s.rows <= 256) {
            jac::run_alone<float, 8>(A, s);
        } else if constexpr (MAXRPL >= 16) {
            jac::run<float, 16, jac::kStream>(A, s);
        }
    }
}

// One cluster per matrix.
template <int MAXRPL>
__global__ void __launch_bounds__(256, 1) k_jacobi_cluster(LayerArgs<float> A, int area) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int n = jac::cluster_size();
    const jac::Start<float> s = jac::start<float>(A, area, smem, blockIdx.x / n);
    if (!s.go) return;
    if (s.rows <= 64) {
        if (jac::cluster_rank() == 0) jac::run<float, 2, jac::kResident>(A, s);
    } else if (MAXRPL <= 4 || s.rows <= 128) {
        jac::run_cluster<float, 4>(A, s);
    } else if constexpr (MAXRPL >= 8) {
        if (MAXRPL == 8 || s.rows <= 256) {
            jac::run_cluster<float, 8>(A, s);
        } else if constexpr (MAXRPL >= 16) {
            jac::run_cluster<float, 16>(A, s);
        }
    }
}

template <int MAXRPL, int THREADS> cudaError_t set_smem() {
    return cudaFuncSetAttribute(k_jacobi<MAXRPL, THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, jac::kSmemMax);
}

struct Most { int n[jac::kMaxCluster + 1]; };
// Clusters of k_jacobi_cluster that run at once, found on first use (zeros where it cannot be launched).
template <int MAXRPL> const Most& most() {
    static const Most m = [] {
        Most r{};
        if (cudaFuncSetAttribute(k_jacobi_cluster<MAXRPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 jac::kSmemMax) != cudaSuccess ||
            jac::clusters_at_once(k_jacobi_cluster<MAXRPL>, 256, jac::kSmemMax, r.n) != cudaSuccess) {
            cudaGetLastError();
            r = Most{};
        }
        return r;
    }();
    return m;
}

template <int MAXRPL>
cudaError_t launch_clusters(const LayerArgs<float>& a, int n, size_t smem, int area, cudaStream_t s) {
    return jac::launch_cluster(k_jacobi_cluster<MAXRPL>, a, n, 256, smem, area, s);
}

}  // namespace

int jacobi_block_width(int precision, int requested) {
    if (precision == PTEBD_FP64) return 8;
    return requested == 8 ? 8 : 16;
}

template <> cudaError_t jacobi_prepare<float>() {
    cudaError_t e = set_smem<4, 384>();
    if (e == cudaSuccess) e = set_smem<8, 256>();
    if (e == cudaSuccess) e = set_smem<16, 384>();
    most<4>();
    most<8>();
    most<16>();
    return e;
}

template <> cudaError_t launch_jacobi<float>(const LayerArgs<float>& a, cudaStream_t s) {
    const bool half = a.nw == 8;  // half the warps and half the shared memory of a CTA
    const int area = jac::column_area<float>(a.ldw, half);
    const size_t smem = jac::table_bytes<float>() + area;
    const int bonds = a.share > a.count ? a.share : a.count;
    if (!half && a.ldw > 64) {
        const int n = jac::cluster_for(bonds, a.ldw > 256 ? most<16>().n : a.ldw > 128 ? most<8>().n : most<4>().n);
        if (n > 1)
            return a.ldw > 256   ? launch_clusters<16>(a, n, smem, area, s)
                   : a.ldw > 128 ? launch_clusters<8>(a, n, smem, area, s)
                                 : launch_clusters<4>(a, n, smem, area, s);
    }
    if (a.ldw > 256)
        k_jacobi<16, 384><<<a.count, half ? 128 : 384, smem, s>>>(a, area);
    else if (a.ldw > 128)
        k_jacobi<8, 256><<<a.count, half ? 128 : 256, smem, s>>>(a, area);
    else
        k_jacobi<4, 384><<<a.count, 32 * jac::warps_for(a.ldw, half, 12), smem, s>>>(a, area);
    return cudaGetLastError();
}

}  // namespace ptebd
