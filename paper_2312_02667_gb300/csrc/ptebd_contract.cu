// Full contractions of an MPS (norm, overlap, expectation values, left
// environments of the sampling) by transfer matrices, every product accumulated
// in FP64 (the MPS decomposition of Sec. II A-B of arXiv:2312.02667).
//
// A contraction runs from both ends of the chain at once: the left environment
// E' = sum_x Gamma_a[x]^dag E Gamma_b[x] and the right one
// F' = sum_x conj(Gamma_a[x]) F Gamma_b[x]^T, each with the Lambda of its outer
// bond on both sides, take a step in the same two launches (T_x = E Gamma_b[x],
// conj(Gamma_a[x]) F; then the sums over x).  They meet at the site of the operator
// (or in the middle), where the four or sixteen overlaps of Gamma_a[x] with
// E Gamma_b[y] F^T are taken: an expectation value is a sum of those with the
// operator's entries over their trace, so numerator and denominator share
// everything.
//
//   k_zmm     : a batch of up to eight complex products, k in one or two segments,
//               rows and columns scaled, with the largest modulus of the result
//               gathered so that the next step can take a power of two out;
//   k_overlaps: sums of conj(P) Q;
//   k_sample_pick.
//
// What bounds it: the FP64 pipe (2 fused multiply-adds per SM and cycle: a 64 x 64 x
// 64 complex product is 1.7 us of the whole chip) and, at small bond dimensions, the
// latency of a launch.  Hence 4 x 8 output tiles of 128 threads: chi = 64 gives 256
// tiles a side (32 x 32 tiles of 256 threads kept 4 of 152 SMs busy at 65 us a
// product; 64 threads leave two of an SM's four FP64 units idle), and two launches
// a step for both sides instead of five for one.
#include <cmath>

#include "ptebd_internal.h"

namespace ptebd {

namespace {

// entry `i` of a complex64 or complex128 matrix
__device__ __forceinline__ double2 entry(const void* p, size_t i, bool f32) {
    if (f32) {
        const float2 v = static_cast<const float2*>(p)[i];
        return make_double2(v.x, v.y);
    }
    return static_cast<const double2*>(p)[i];
}

// 2^-e of the largest modulus gathered in *bits (1 when there is none, or it is not finite)
__device__ __forceinline__ double unit_scale(const unsigned long long* bits) {
    if (!bits) return 1.0;
    const int e = (int)(*bits >> 52) & 0x7ff;
    if (e == 0 || e >= 2046) return 1.0;
    return __longlong_as_double((long long)(2046 - e) << 52);
}

constexpr int kTileM = 4, kTileN = 8, kChunk = 64, kThreads = 128;

// grid (ceil(max m / 4), ceil(max n / 8), problems), 128 threads: each warp takes a
// quarter of every chunk of k for the tile's 32 outputs, so that all four schedulers'
// FP64 units work.  The chunk after the one being multiplied is already on its way
// from memory.  A Hermitian result is worked out on and above its diagonal.  The
// launches of a chain are programmatic ones, without an explicit trigger: the next
// one is set up as this one ends (8.1 -> 6.9 ms of measurements at N = 128, chi = 64);
// triggered early, waiting blocks of the launches to come fill some of the SMs and
// the next one's work piles up on the others (13.8 ms).
__global__ void __launch_bounds__(kThreads) k_zmm(ZmmBatch batch) {
    const Zmm& q = batch.p[blockIdx.z];
    const int i0 = blockIdx.x * kTileM, j0 = blockIdx.y * kTileN;
    if (i0 >= q.m || j0 >= q.n || (q.hermitian && i0 >= j0 + kTileN)) return;
    __shared__ double2 as[kChunk][kTileM + 1], bs[kChunk][kTileN + 1];
    const int t = threadIdx.x, quarter = t >> 5, ti = t & 3, tj = (t >> 2) & 7;
    const int per = (q.k + kChunk - 1) / kChunk, chunks = per * q.segments;
    double2 ra[2], rb[4];
    // element e of a chunk: the index that is contiguous in memory runs fastest
    auto fetch = [&](int c) {
        const int seg = c >= per ? 1 : 0, k0 = (c - seg * per) * kChunk;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = t + u * kThreads;
            int kk, ii;
            if (q.op_a == ZMM_C) { kk = e & 63; ii = e >> 6; } else { ii = e & 3; kk = e >> 2; }
            const int k = k0 + kk, i = i0 + ii;
            double2 v = make_double2(0.0, 0.0);
            if (k < q.k && i < q.m) {
                const size_t at = q.op_a == ZMM_C ? (size_t)i * q.lda + k : (size_t)k * q.lda + i;
                v = entry(q.a[seg], at, q.a32);
                if (q.op_a != ZMM_N) v.y = -v.y;
                if (q.kscale) { v.x *= q.kscale[k]; v.y *= q.kscale[k]; }
            }
            ra[u] = v;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = t + u * kThreads;
            int kb, jj;
            if (q.op_b == ZMM_T) { jj = e & 7; kb = e >> 3; } else { kb = e & 63; jj = e >> 6; }
            const int k = k0 + kb, j = j0 + jj;
            double2 w = make_double2(0.0, 0.0);
            if (k < q.k && j < q.n) {
                const size_t at = q.op_b == ZMM_T ? (size_t)k * q.ldb + j : (size_t)j * q.ldb + k;
                w = entry(q.b[seg], at, q.b32);
            }
            rb[u] = w;
        }
    };
    auto put = [&]() {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = t + u * kThreads;
            if (q.op_a == ZMM_C) as[e & 63][e >> 6] = ra[u]; else as[e >> 2][e & 3] = ra[u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = t + u * kThreads;
            if (q.op_b == ZMM_T) bs[e >> 3][e & 7] = rb[u]; else bs[e & 63][e >> 6] = rb[u];
        }
    };
    double2 acc = make_double2(0.0, 0.0);
    asm volatile("griddepcontrol.wait;" ::: "memory");  // everything before this launch is complete and visible
    fetch(0);
    for (int c = 0; c < chunks; ++c) {
        put();
        __syncthreads();
        if (c + 1 < chunks) fetch(c + 1);
        // (a chunk is zero beyond the end of k; a short one is quartered evenly)
        const int seg = c >= per ? 1 : 0, depth = (min(kChunk, q.k - (c - seg * per) * kChunk) + 3) / 4;
        const double2 (*pa)[kTileM + 1] = as + quarter * depth, (*pb)[kTileN + 1] = bs + quarter * depth;
#pragma unroll 8
        for (int kk = 0; kk < depth; ++kk) {
            const double2 x = pa[kk][ti], y = pb[kk][tj];
            acc.x = fma(x.x, y.x, acc.x); acc.y = fma(x.x, y.y, acc.y);
            acc.x = fma(-x.y, y.y, acc.x); acc.y = fma(x.y, y.x, acc.y);
        }
        __syncthreads();
    }
    double2* other = &as[0][0];  // (3 x 32 of its 320 entries)
    if (quarter) other[t - 32] = acc;
    __syncthreads();
    if (quarter) return;
#pragma unroll
    for (int h = 0; h < 3; ++h) {
        acc.x += other[32 * h + t].x;
        acc.y += other[32 * h + t].y;
    }
    const int i = i0 + ti, j = j0 + tj;
    double big = 0.0;
    if (i < q.m && j < q.n) {
        double f = unit_scale(q.scale_a) * unit_scale(q.scale_b);
        if (q.rowscale) f *= q.rowscale[i];
        if (q.colscale) f *= q.colscale[j];
        acc.x *= f;
        acc.y *= f;
        if (!q.hermitian || i <= j) {
            if (q.hermitian && i == j) acc.y = 0.0;
            q.c[(size_t)j * q.ldc + i] = acc;
            if (q.hermitian && i < j) q.c[(size_t)i * q.ldc + j] = make_double2(acc.x, -acc.y);
        }
        big = fmax(fabs(acc.x), fabs(acc.y));
    }
    if (q.largest) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
        if (t == 0) atomicMax(q.largest, (unsigned long long)__double_as_longlong(big));
    }
}

// (1) as the environments of both ends, and the exponents gathered along the chain cleared
__global__ void __launch_bounds__(256) k_chain_start(double2* e, double2* f, unsigned long long* largest, int n) {
    for (int i = threadIdx.x; i < n; i += 256) largest[i] = 0ull;
    if (threadIdx.x == 0) {
        if (e) e[0] = make_double2(1.0, 0.0);
        if (f) f[0] = make_double2(1.0, 0.0);
    }
}

// out[blockIdx.x]: sum over the m x n entries of conj(p) q, block x = pair (x / nq, x mod nq)
// of the np matrices P (stride p_step entries) and the nq matrices Q; and, in one
// block, out_exp = the power of two taken out along the chain.
__global__ void __launch_bounds__(512) k_overlaps(const void* p, bool p32, size_t p_step, int ldp, const double2* q,
                                                  size_t q_step, int ldq, int nq, int m, int n, double2* out,
                                                  const unsigned long long* largest, int n_largest, double* out_exp) {
    __shared__ double sx[512], sy[512];
    const int t = threadIdx.x;
    const size_t po = (size_t)(blockIdx.x / nq) * p_step, qo = (size_t)(blockIdx.x % nq) * q_step;
    double x = 0.0, y = 0.0;
    for (int e = t; e < m * n; e += 512) {
        const int i = e % m, j = e / m;
        const double2 u = entry(p, po + (size_t)j * ldp + i, p32), v = q[qo + (size_t)j * ldq + i];
        x = fma(u.x, v.x, x); x = fma(u.y, v.y, x);
        y = fma(u.x, v.y, y); y = fma(-u.y, v.x, y);
    }
    sx[t] = x;
    sy[t] = y;
    __syncthreads();
    for (int s = 256; s > 0; s >>= 1) {
        if (t < s) { sx[t] += sx[t + s]; sy[t] += sy[t + s]; }
        __syncthreads();
    }
    if (t == 0) out[blockIdx.x] = make_double2(sx[0], sy[0]);
    if (blockIdx.x == 0) {
        __shared__ int se[512];
        int sum = 0;
        for (int i = t; i < n_largest; i += 512) {
            const int e = (int)(largest[i] >> 52) & 0x7ff;
            if (e != 0 && e < 2046) sum += e - 1023;
        }
        se[t] = sum;
        __syncthreads();
        for (int s = 256; s > 0; s >>= 1) {
            if (t < s) se[t] += se[t + s];
            __syncthreads();
        }
        if (t == 0) *out_exp = (double)se[0];
    }
}

// One sampling decision at `site` for every sample (a warp each): w_x = t_x^dag u_x
// with t_x = Gamma[x] Lambda v and u_x = L t_x, sigma = 0 when u < w_0 / (w_0 + w_1),
// v <- t_sigma / |t_sigma|.  t, u: two matrices of chil x samples (ld chip), `step` apart.
__global__ void __launch_bounds__(256) k_sample_pick(const double2* __restrict__ tm, const double2* __restrict__ um,
                                                     size_t step, int chil, int chip, double2* __restrict__ v,
                                                     const double* __restrict__ uniforms, int site, int n_sites,
                                                     int32_t* __restrict__ bits, int samples) {
    const int k = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (k >= samples) return;
    double w[2] = {0.0, 0.0}, nn[2] = {0.0, 0.0};
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const double2* tc = tm + x * step + (size_t)k * chip;
        const double2* uc = um + x * step + (size_t)k * chip;
        for (int a = lane; a < chil; a += 32) {
            const double2 tv = tc[a], uv = uc[a];
            w[x] += tv.x * uv.x + tv.y * uv.y;
            nn[x] += tv.x * tv.x + tv.y * tv.y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            w[x] += __shfl_xor_sync(0xffffffffu, w[x], o);
            nn[x] += __shfl_xor_sync(0xffffffffu, nn[x], o);
        }
    }
    const double p0 = w[0] / (w[0] + w[1]);
    const int x = uniforms[(size_t)k * n_sites + site] < p0 ? 0 : 1;
    if (lane == 0) bits[(size_t)k * n_sites + site] = x;
    const double n2 = x ? nn[1] : nn[0], inv = n2 > 0.0 ? 1.0 / sqrt(n2) : 0.0;
    const double2* tc = tm + x * step + (size_t)k * chip;
    for (int a = lane; a < chil; a += 32) {
        double2 y = tc[a];
        y.x *= inv; y.y *= inv;
        v[(size_t)k * chip + a] = y;
    }
}

// v_k = (1), the right boundary of every sample
__global__ void k_sample_start(double2* v, int chip, int samples) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < samples) v[(size_t)k * chip] = make_double2(1.0, 0.0);
}

}  // namespace

cudaError_t launch_zmm(const ZmmBatch& b, int n, cudaStream_t s) {
    int m = 0, c = 0;
    for (int i = 0; i < n; ++i) {
        m = b.p[i].m > m ? b.p[i].m : m;
        c = b.p[i].n > c ? b.p[i].n : c;
    }
    if (m <= 0 || c <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((m + kTileM - 1) / kTileM, (c + kTileN - 1) / kTileN, n);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_zmm, b);
}

cudaError_t launch_chain_start(double2* e, double2* f, unsigned long long* largest, int n, cudaStream_t s) {
    k_chain_start<<<1, 256, 0, s>>>(e, f, largest, n);
    return cudaGetLastError();
}

cudaError_t launch_overlaps(const void* p, bool p32, size_t p_step, int ldp, int np, const double2* q, size_t q_step,
                            int ldq, int nq, int m, int n, double2* out, const unsigned long long* largest,
                            int n_largest, double* out_exp, cudaStream_t s) {
    k_overlaps<<<np * nq, 512, 0, s>>>(p, p32, p_step, ldp, q, q_step, ldq, nq, m, n, out, largest, n_largest, out_exp);
    return cudaGetLastError();
}

cudaError_t launch_sample_start(double2* v, int chip, int samples, cudaStream_t s) {
    k_sample_start<<<(samples + 255) / 256, 256, 0, s>>>(v, chip, samples);
    return cudaGetLastError();
}

cudaError_t launch_sample_pick(const double2* t, const double2* u, size_t step, int chil, int chip, double2* v,
                               const double* uniforms, int site, int n_sites, int32_t* bits, int samples,
                               cudaStream_t s) {
    k_sample_pick<<<(samples + 7) / 8, 256, 0, s>>>(t, u, step, chil, chip, v, uniforms, site, n_sites, bits, samples);
    return cudaGetLastError();
}

}  // namespace ptebd
