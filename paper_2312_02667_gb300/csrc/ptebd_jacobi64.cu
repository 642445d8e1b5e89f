// The Jacobi SVD kernels of complex128 matrices (ptebd_jacobi.cuh).
#include "ptebd_jacobi.cuh"

namespace ptebd {

namespace {

// MAXRPL: rows a lane holds of the tallest matrix of the launch (ldw / 32).
// CLUSTER: one cluster per matrix, else one CTA.
template <int MAXRPL, bool CLUSTER>
__global__ void __launch_bounds__(256, 1) k_jacobi64(LayerArgs<double> A, int area) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int n = CLUSTER ? jac::cluster_size() : 1;
    const jac::Start<double> s = jac::start<double>(A, area, smem, blockIdx.x / n);
    if (!s.go) return;
    auto go = [&](auto rpl) {
        if constexpr (CLUSTER) jac::run_cluster<double, decltype(rpl)::value>(A, s);
        else if constexpr (decltype(rpl)::value <= 2) jac::run<double, decltype(rpl)::value, jac::kResident>(A, s);
        else if constexpr (decltype(rpl)::value >= 16) jac::run<double, decltype(rpl)::value, jac::kStream>(A, s);
        else jac::run_alone<double, decltype(rpl)::value>(A, s);
    };
    if (s.rows <= 32) {
        if (!CLUSTER || jac::cluster_rank() == 0) jac::run<double, 1, jac::kResident>(A, s);
    } else if (MAXRPL <= 2 || s.rows <= 64) {
        go(std::integral_constant<int, 2>{});
    } else if constexpr (MAXRPL >= 4) {
        if (MAXRPL == 4 || s.rows <= 128) {
            go(std::integral_constant<int, 4>{});
        } else if constexpr (MAXRPL >= 8) {
            if (MAXRPL == 8 || s.rows <= 256) {
                go(std::integral_constant<int, 8>{});
            } else if constexpr (MAXRPL >= 16) {
                if (!CLUSTER || jac::cluster_rank() == 0) jac::run<double, 16, jac::kStream>(A, s);
            }
        }
    }
}

template <int MAXRPL> cudaError_t set_smem() {
    return cudaFuncSetAttribute(k_jacobi64<MAXRPL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, jac::kSmemMax);
}

struct Most { int n[jac::kMaxCluster + 1]; };
// Clusters that run at once, found on first use (zeros where they cannot be launched).
template <int MAXRPL> const Most& most() {
    static const Most m = [] {
        Most r{};
        if (cudaFuncSetAttribute(k_jacobi64<MAXRPL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 jac::kSmemMax) != cudaSuccess ||
            jac::clusters_at_once(k_jacobi64<MAXRPL, true>, 256, jac::kSmemMax, r.n) != cudaSuccess) {
            cudaGetLastError();
            r = Most{};
        }
        return r;
    }();
    return m;
}

template <int MAXRPL>
cudaError_t launch_class(const LayerArgs<double>& a, cudaStream_t s) {
    const int area = jac::column_area<double>(a.ldw, false);
    const size_t smem = jac::table_bytes<double>() + area;
    const int threads = 32 * jac::warps_for(a.ldw, false, 8);
    int bonds = a.share > a.count ? a.share : a.count;
    if (a.refine == 1) bonds = (bonds + 7) / 8;  // (few of them are undecided; the others return at once)
    const int n = MAXRPL > 1 ? jac::cluster_for(bonds, most<MAXRPL>().n) : 1;
    if (n > 1 && a.ldw > 32) return jac::launch_cluster(k_jacobi64<MAXRPL, true>, a, n, threads, smem, area, s);
    k_jacobi64<MAXRPL, false><<<a.count, threads, smem, s>>>(a, area);
    return cudaGetLastError();
}

}  // namespace

template <> cudaError_t jacobi_prepare<double>() {
    cudaError_t e = set_smem<2>();
    if (e == cudaSuccess) e = set_smem<4>();
    if (e == cudaSuccess) e = set_smem<8>();
    if (e == cudaSuccess) e = set_smem<16>();
    most<2>();
    most<4>();
    most<8>();
    most<16>();
    return e;
}

template <> cudaError_t launch_jacobi<double>(const LayerArgs<double>& a, cudaStream_t s) {
    return a.ldw > 256   ? launch_class<16>(a, s)
           : a.ldw > 128 ? launch_class<8>(a, s)
           : a.ldw > 64  ? launch_class<4>(a, s)
                         : launch_class<2>(a, s);
}

}  // namespace ptebd
