// Batched one-sided (Hestenes) Jacobi SVD of the two-site tensors of a layer
// (the SVD step of the TEBD procedure, Sec. II C of arXiv:2312.02667).
//
// One CTA per bond.  The matrix w (rows x cols, column-major, rows >= cols) is
// taken in groups of B columns, by decreasing column norm (re-sorted at the
// start of every sweep).  A sweep visits the pairs of groups in row-cyclic
// order, as a pipeline of compute warps: warp v takes groups I = v, v + nwc,
// v + 2 nwc, ... into registers, and every later group J flows past the warps in
// the order of their I.  A counter per group (prog, release/acquire in shared
// memory) says how many I it has met, so a warp waits only for its one
// predecessor.  A visit (I, J) holds the 2 B columns in registers and goes
// through their B^2 pairs in B rounds of B disjoint pairs: the B dot products
// are reduced together, lanes p (32/B)..(p + 1)(32/B) - 1 work out the
// rotation of pair p (the B rotations of a round side by side in one warp
// instruction stream, so that the square roots and reciprocals are paid once a
// round and not once a pair), and the coefficients come back through shared
// memory.
//
// Where the columns are: when the matrix fits in shared memory (`RES`) it stays
// there for the whole SVD.  Otherwise the groups are streamed: the last warp
// fetches them by TMA bulk copies (cp.async.bulk, completion on an mbarrier)
// into a ring of about 24 slots; the last warp of a row of I groups writes a
// changed group back from its registers.
//
// Rotations are "fast": with the columns held as a = (1 + da) a~, a pair takes two
// shears in place, a~ -= conj(tau) b~ and then b~ += kappa a~ (8 FMA per row
// instead of 16 operations, no temporaries), and the factors cos of a and 1/cos
// of b go into da and db, which stay with their columns and are multiplied out
// only once they have moved by 2^-6.  da is kept as the difference from 1: cos - 1
// and 1/cos - 1 = t^2 / (1 + sqrt(1 + t^2)) accumulate without rounding to zero
// when t^2 is below the unit roundoff (cos itself would round to 1 while t does
// not, and every such rotation would scale the pair by sqrt(1 + t^2)); multiplied
// out at once they would round away just so, entry by entry, and the thousands of
// small rotations of an SVD add up to 1e-6 in the complex64 norms.
//
// A pair (a, b) with |a^H b| > tol ||a|| ||b|| is rotated; the sweeps stop when
// none was (or, on the complex64 path, when every rotation of a sweep was a
// small one: Eps).  Where one CTA can hold the columns, the first sweeps run in
// twos without a sort and a barrier between (jacobi_body).  The squared column norms are recomputed at the start of every
// sweep and tracked through the rotations in between; a norm that drops a lot
// is recomputed from the rotated column.  On exit the columns are U S
// (orthogonal, unsorted); their FP64 norms are the singular values.
//
// What bounds it: on complex64 the latency of a round's chain (dot products,
// shuffles, the rotation, coefficients through shared memory), two or three warps
// per scheduler; on complex128 the FP64 pipe.  Against one column per warp and a
// rotation worked out by every lane of every pair (the kernel before this one, which
// ptebd_jacobi_blocks.cu keeps): 152 Ginibre matrices, complex64 128 x 128 3.48 -> 1.89 ms,
// 256 x 256 16.8 -> 8.6, 512 x 512 89 -> 67; complex128 128 x 128 99 -> 40.  Why the groups go
// in row-cyclic order: a tournament over all groups would keep every warp busy
// but takes 13 to 16 sweeps where this order takes 10 or 11.
//
// With few matrices, each is spread over the CTAs of a cluster (kCluster): the
// columns lie in the shared memory of all of them, the warps of all of them make
// one row of I groups, and counters, norms and scales are read through distributed
// shared memory.  The arithmetic and its order are the same, so the result does
// not depend on how a matrix was spread.  10 complex128 256 x 256: 313 -> 68 ms
// (8 CTAs each), 64 of 128 x 128: 41 -> 27 (2 each); complex64 37 of 200 x 200
// 5.6 -> 3.6 (3 or 4 each).  Each launch takes the largest cluster at which all its
// matrices still run at once (cluster_for).
//
// Every wait is bounded by a clock budget; one that runs out raises the CTA's
// abort flag, drains the CTA's own copies, latches DERR_TIMEOUT and returns.
#pragma once
#include <cmath>
#include <type_traits>

#include "ptebd_device.h"
#include "ptebd_internal.h"
#include "ptebd_vote.h"

namespace ptebd {
namespace jac {

// ------------------------------------------------------------------ PTX --
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void counter_release(int* p, int v) {
    asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int counter_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// all but the last N bulk groups of this thread are complete
template <int N> __device__ __forceinline__ void bulk_wait() {
    asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// thread-block clusters
__device__ __forceinline__ int cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
__device__ __forceinline__ int cluster_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return (int)r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address of p (in this CTA's shared memory) in CTA `rank` of the cluster
template <typename T> __device__ __forceinline__ T* peer(T* p, int rank) {
    uint64_t r;
    asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<uint64_t>(p)), "r"(rank));
    return reinterpret_cast<T*>(r);
}
__device__ __forceinline__ void counter_release_cluster(int* p, int v) {
    asm volatile("st.release.cluster.u32 [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int counter_acquire_cluster(const int* p) {
    int v;
    asm volatile("ld.acquire.cluster.u32 %0, [%1];" : "=r"(v) : "l"(reinterpret_cast<uint64_t>(p)) : "memory");
    return v;
}

constexpr long long kWaitLimit = 1ll << 31;  // SM cycles, about a second

// Bounded spin until *p >= target (or the CTA has aborted).  The clock and the
// abort flag are looked at every 32 polls only.
template <bool CL = false>
__device__ __forceinline__ bool counter_wait(const int* p, int target, const volatile int* abort_flag,
                                             long long limit = kWaitLimit) {
    const long long start = clock64();
    for (unsigned it = 0;; ++it) {
        if ((CL ? counter_acquire_cluster(p) : counter_acquire(p)) >= target) return true;
        __nanosleep(20);
        if ((it & 31u) == 0u) {
            if (clock64() - start > limit) return false;
            if (*abort_flag) return false;
        }
    }
}
// Bounded wait for a phase of an mbarrier; abort_flag may be null.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, const volatile int* abort_flag) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long start = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - start > kWaitLimit) return false;
        if (abort_flag && *abort_flag) return false;
    }
    return true;
}

// ---------------------------------------------------------- arithmetic --
// Unit roundoff and the rotation threshold factor: a pair is rotated when
// |a^H b| > k sqrt(rows) u ||a|| ||b||.  Rounding alone leaves |a^H b| of about
// sqrt(rows) u ||a|| ||b|| after a rotation, so the factor must sit well above 1
// or rounding keeps re-triggering rotations (more sweeps, and every extra
// rotation adds rounding error to the columns).
// early: the sweeps also stop after a sweep in which every rotated pair had
// cos^2 = |a^H b|^2 / (|a|^2 |b|^2) below early * tol^2 (0 = only after a sweep
// without rotations).  On the complex64 path the sweep after such a sweep was
// measured never to meet a pair above 1.04 tol^2 (gated and tSU matrices of
// saturated layers, Ginibre and graded spectra: thousands of SVDs), and to
// spend itself on 0 to 2 rotations of pairs barely above tol, so it is skipped;
// the columns are left orthogonal to about tol instead of below tol.
// range_e: matrices whose largest entry is not in [2^-range_e, 2^range_e) are
// rescaled before the sweeps (see the range guard in jacobi_body).
// polish: the factor of the last sweeps' tighter threshold (A.polish), taken once
// few pairs rotate (kPolishShare) or the stopping rule has fired: they rotate every pair with
// |a^H b| > polish sqrt(rows) u |a| |b|, which leaves the columns orthogonal to
// near the rounding of their storage (the truncated state depends on it: at 2 an
// observable after a 12-layer chi = 64 circuit is 1.2e-6 off the FP64 one, at 1
// 0.6e-6, at 0.5 0.5e-6, geometric means of 14 circuits).
template <typename R> struct Eps;
template <> struct Eps<float> {
    static constexpr double u = 5.9604644775390625e-08;  // 2^-24
    static constexpr double k = 8.0;
    static constexpr int range_e = 24;
    static constexpr double early = 256.0;
    static constexpr double polish = 1.0;
};
template <> struct Eps<double> {
    static constexpr double u = 1.1102230246251565e-16;  // 2^-53
    static constexpr double k = 4.0;
    static constexpr int range_e = 240;
    static constexpr double early = 0.0;
    static constexpr double polish = 0.0;
};

template <typename R>
__device__ __forceinline__ R warp_sum(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <typename R>
__device__ __forceinline__ R warp_max(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// The binary exponent of a non-negative value, offset so that 0 (no entry) stays
// below every real exponent: a shared atomicMax over it gives the exponent of the
// largest entry of a matrix.
constexpr int kExpOffset = 2048;
template <typename R> __device__ __forceinline__ int exp_key(R v) {
    return v > (R)0 ? ilogb((double)v) + kExpOffset : 0;
}

// Packed FP32 pairs (fma.rn.f32x2 and friends, sm_100 and later): two lanes of
// FP32 arithmetic per instruction on a register pair (lo, hi).
__device__ __forceinline__ unsigned long long pk2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 upk2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Columns.  complex64 (always RPL >= 2, rows even): pair-split layout while the
// sweeps run, every two rows r, r + 1 (r even) stored as
// (Re r, Re r+1, Im r, Im r+1), so that one 16-byte access moves the pair and the
// packed FP32 instructions find the real parts and the imaginary parts of the
// pair in one 64-bit register each.  Lane `lane` holds the pairs
// r = 64 h + 2 lane, h = 0 .. RPL/2 - 1: entry 2 h is (Re r, Re r+1), entry
// 2 h + 1 is (Im r, Im r+1).  complex128: entry q is row 32 q + lane.
template <typename R> struct Entry { using T = unsigned long long; };
template <> struct Entry<double> { using T = double2; };
template <typename R> using entry_t = typename Entry<R>::T;

template <int RPL>  // from a column in shared memory
__device__ __forceinline__ void col_load(unsigned long long (&v)[RPL], const float2* col, int lane) {
#pragma unroll
    for (int h = 0; h < RPL / 2; ++h) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(col + 64 * h + 2 * lane);
        v[2 * h] = t.x;
        v[2 * h + 1] = t.y;
    }
}
template <int RPL>
__device__ __forceinline__ void col_load(double2 (&v)[RPL], const double2* col, int lane) {
#pragma unroll
    for (int q = 0; q < RPL; ++q) v[q] = col[32 * q + lane];
}
template <int RPL>
__device__ __forceinline__ void col_store(const unsigned long long (&v)[RPL], float2* col, int lane, int rows) {
#pragma unroll
    for (int h = 0; h < RPL / 2; ++h) {
        const int r = 64 * h + 2 * lane;
        if (r < rows) *reinterpret_cast<ulonglong2*>(col + r) = make_ulonglong2(v[2 * h], v[2 * h + 1]);
    }
}
template <int RPL>
__device__ __forceinline__ void col_store(const double2 (&v)[RPL], double2* col, int lane, int rows) {
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
        const int r = 32 * q + lane;
        if (r < rows) col[r] = v[q];
    }
}

// a^H b over this lane's rows
template <int RPL>
__device__ __forceinline__ void col_dot(const unsigned long long (&a)[RPL], const unsigned long long (&b)[RPL],
                                        float& gr, float& gi) {
    unsigned long long r2 = 0ull, p2 = 0ull, m2 = 0ull;  // (0.f, 0.f)
#pragma unroll
    for (int h = 0; h < RPL / 2; ++h) {
        r2 = fma2(a[2 * h], b[2 * h], r2);
        p2 = fma2(a[2 * h], b[2 * h + 1], p2);
        m2 = fma2(a[2 * h + 1], b[2 * h], m2);
        r2 = fma2(a[2 * h + 1], b[2 * h + 1], r2);
    }
    const float2 r = upk2(r2), p = upk2(p2), m = upk2(m2);
    gr = r.x + r.y;
    gi = (p.x - m.x) + (p.y - m.y);
}
template <int RPL>
__device__ __forceinline__ void col_dot(const double2 (&a)[RPL], const double2 (&b)[RPL], double& gr, double& gi) {
    double r = 0.0, i = 0.0;
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
        r = fma(a[q].x, b[q].x, r);
        i = fma(a[q].x, b[q].y, i);
        r = fma(a[q].y, b[q].y, r);
        i = fma(-a[q].y, b[q].x, i);
    }
    gr = r;
    gi = i;
}

// The coefficients of a rotation as the columns' instructions take them, handed
// from the lanes that work them out to the whole warp through shared memory.
template <typename R> struct Coef;
template <> struct __align__(16) Coef<float> {
    float4 a, b, c;  // (-tr, -tr, -ti, -ti), (ti, ti, kr, kr), (-ki, -ki, ki, ki)
    __device__ __forceinline__ void set(float tr, float ti, float kr, float ki) {
        a = make_float4(-tr, -tr, -ti, -ti);
        b = make_float4(ti, ti, kr, kr);
        c = make_float4(-ki, -ki, ki, ki);
    }
};
template <> struct __align__(16) Coef<double> {
    double2 t, k;
    __device__ __forceinline__ void set(double tr, double ti, double kr, double ki) {
        t = make_double2(tr, ti);
        k = make_double2(kr, ki);
    }
};

// a -= conj(tau) b, then b += kappa a (the new a)
template <int RPL>
__device__ __forceinline__ void col_rotate(unsigned long long (&a)[RPL], unsigned long long (&b)[RPL],
                                           const Coef<float>& k) {
    const ulonglong2 ka = *reinterpret_cast<const ulonglong2*>(&k.a), kb = *reinterpret_cast<const ulonglong2*>(&k.b),
                     kc = *reinterpret_cast<const ulonglong2*>(&k.c);
#pragma unroll
    for (int h = 0; h < RPL / 2; ++h) {
        a[2 * h] = fma2(ka.x, b[2 * h], fma2(ka.y, b[2 * h + 1], a[2 * h]));
        a[2 * h + 1] = fma2(ka.x, b[2 * h + 1], fma2(kb.x, b[2 * h], a[2 * h + 1]));
        b[2 * h] = fma2(kb.y, a[2 * h], fma2(kc.x, a[2 * h + 1], b[2 * h]));
        b[2 * h + 1] = fma2(kb.y, a[2 * h + 1], fma2(kc.y, a[2 * h], b[2 * h + 1]));
    }
}
template <int RPL>
__device__ __forceinline__ void col_rotate(double2 (&a)[RPL], double2 (&b)[RPL], const Coef<double>& k) {
    const double tr = k.t.x, ti = k.t.y, kr = k.k.x, ki = k.k.y;
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
        a[q].x = fma(-tr, b[q].x, fma(-ti, b[q].y, a[q].x));
        a[q].y = fma(-tr, b[q].y, fma(ti, b[q].x, a[q].y));
        b[q].x = fma(kr, a[q].x, fma(-ki, a[q].y, b[q].x));
        b[q].y = fma(kr, a[q].y, fma(ki, a[q].x, b[q].y));
    }
}
// a += d a
template <int RPL>
__device__ __forceinline__ void col_scale(unsigned long long (&a)[RPL], float d) {
    const unsigned long long dd = pk2(d, d);
#pragma unroll
    for (int q = 0; q < RPL; ++q) a[q] = fma2(dd, a[q], a[q]);
}
template <int RPL>
__device__ __forceinline__ void col_scale(double2 (&a)[RPL], double d) {
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
        a[q].x = fma(d, a[q].x, a[q].x);
        a[q].y = fma(d, a[q].y, a[q].y);
    }
}
// |a|^2 over the warp
template <int RPL>
__device__ __forceinline__ float col_norm2(const unsigned long long (&a)[RPL]) {
    unsigned long long s = 0ull;
#pragma unroll
    for (int q = 0; q < RPL; ++q) s = fma2(a[q], a[q], s);
    const float2 t = upk2(s);
    return warp_sum(t.x + t.y);
}
template <int RPL>
__device__ __forceinline__ double col_norm2(const double2 (&a)[RPL]) {
    double s0 = 0, s1 = 0;
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
        s0 = fma(a[q].x, a[q].x, s0);
        s1 = fma(a[q].y, a[q].y, s1);
    }
    return warp_sum(s0 + s1);
}

// The sums over the warp of B complex values a lane, the p-th to the lanes
// p (32/B) .. (p + 1)(32/B) - 1.
template <typename R, int B>
__device__ __forceinline__ void reduce_pairs(R (&vr)[B], R (&vi)[B], int lane, R& gr, R& gi) {
    constexpr unsigned kAll = 0xffffffffu;
    if constexpr (B == 4) {
        const bool hi = lane & 16;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const R sr = hi ? vr[i] : vr[i + 2], si = hi ? vi[i] : vi[i + 2];
            const R kr = hi ? vr[i + 2] : vr[i], ki = hi ? vi[i + 2] : vi[i];
            vr[i] = kr + __shfl_xor_sync(kAll, sr, 16);
            vi[i] = ki + __shfl_xor_sync(kAll, si, 16);
        }
    }
    if constexpr (B >= 2) {
        constexpr int o = B == 4 ? 8 : 16;
        const bool hi = lane & o;
        const R sr = hi ? vr[0] : vr[1], si = hi ? vi[0] : vi[1];
        const R kr = hi ? vr[1] : vr[0], ki = hi ? vi[1] : vi[0];
        vr[0] = kr + __shfl_xor_sync(kAll, sr, o);
        vi[0] = ki + __shfl_xor_sync(kAll, si, o);
    }
#pragma unroll
    for (int o = 16 / B; o > 0; o >>= 1) {
        vr[0] += __shfl_xor_sync(kAll, vr[0], o);
        vi[0] += __shfl_xor_sync(kAll, vi[0], o);
    }
    gr = vr[0];
    gi = vi[0];
}

// The rotation that diagonalises [[al, g], [conj(g), be]] (al = |a|^2, be = |b|^2,
// g = a^H b): (tr, ti) = tan(angle) e^{i arg g}, tg = tan(angle) |g| (the norms
// become al - tg and be + tg), c2 = cos^2, cm1 = cos - 1, sm1 = 1/cos - 1.  In full,
// a' = cos (a - conj(tau) b) and b' = cos (b + tau a) with tau = (tr, ti); since
// b + tau a = (1 + |tau|^2) (b + cos^2 tau (a - conj(tau) b)), the second shear has
// kappa = cos^2 tau and b takes the factor 1/cos.
// t = 2 |g| sign(d) / (|d| + sqrt(d^2 + 4 |g|^2)), d = be - al: the smaller root
// of t^2 + (d / |g|) t - 1 = 0, formed without a quotient by |g|.
template <typename R> struct Rot { R tr, ti, tg, c2, cm1, sm1; };

__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 1 / w for w of moderate size: the approximate reciprocal and Newton steps to
// working precision (a biased quotient in every rotation would add up in the norms)
__device__ __forceinline__ float rcp_newton(float w) {
    const float y = rcp_approx(w);
    return fmaf(y, fmaf(-w, y, 1.0f), y);
}
__device__ __forceinline__ double rcp_newton(double w) {
    double y;  // (20 bits)
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(w));
    const double e = fma(-w, y, 1.0);  // y (1 + e + e^2): third order
    return fma(y, fma(e, e, e), y);
}

__device__ __forceinline__ Rot<float> rotation(float al, float be, float gr, float gi, float g2) {
    const float d = be - al;
    const float h = fmaf(d, d, 4.0f * g2);
    const float root = h * rsqrtf(h);
    float f = __fdividef(2.0f, fabsf(d) + root);
    if (d < 0.0f) f = -f;
    Rot<float> p;
    p.tr = f * gr;
    p.ti = f * gi;
    p.tg = f * g2;
    const float t2 = f * p.tg;
    const float q = 1.0f + t2;
    p.c2 = rcp_newton(q);
    // One Newton step adds the correction to c, so that only the last rounding is left.  As a
    // factor 1.5 - q c^2 / 2 it would round on another grid below 1 than above: the norms of
    // 600 matrices of 200 x 200 grew by 2.4e-8 in the mean, against 4e-10.
    float c = rsqrt_approx(q);
    c = fmaf(0.5f * c, fmaf(-q * c, c, 1.0f), c);
    p.sm1 = t2 * rcp_newton(fmaf(q, c, 1.0f));  // 1/cos = q c
    p.cm1 = -p.sm1 * c;
    return p;
}
// complex128.  Every value is FP64.  The FP64 unit takes 64 cycles for one instruction of a
// warp and the parameters of a round are worked out by every lane, so magnitudes are handled
// on the bits (exponents, powers of two, comparisons with one), and roots and quotients take
// the 20 bits of the hardware's approximations and one third-order step.  (A test and a
// tangent in FP32 would take 79 instead of 83 ms of an N = 128, chi = 64 step, and 7.6 instead
// of 8.4 ms of 40 SVDs of 90 x 70, but leave a rotated pair at 1e-7 of its cosine.)
__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }  // biased
__device__ __forceinline__ double pow2(int k) { return __hiloint2double((k + 1023) << 20, 0); }  // -1022 <= k <= 1023
__device__ __forceinline__ double with_exponent(double x, int e) {  // x normal and positive, e biased
    return __hiloint2double((__double2hiint(x) & 0xfffff) | (e << 20), __double2loint(x));
}
// 1 / sqrt(x) to 20 bits
__device__ __forceinline__ double rsqrt_approx(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
// g = a^H b of a pair in units of about |a| |b| (2^h), whatever the range of the columns, and
// whether |g|^2 > tol2 al be (never for a zero, subnormal or non-finite norm)
struct Unit64 { double x, y, g2; int h; bool over; };
__device__ __forceinline__ Unit64 in_units(double al, double be, double gr, double gi, double tol2) {
    const int ea = exponent(al), eb = exponent(be), sum = ea + eb - 2046;
    Unit64 s;
    s.h = sum >> 1;
    const double f = pow2(-s.h);
    s.x = gr * f;
    s.y = gi * f;
    s.g2 = fma(s.x, s.x, s.y * s.y);
    const double a = with_exponent(al, 1023), b = with_exponent(be, 1023 + (sum & 1));
    s.over = (unsigned)(ea - 1) < 2046u && (unsigned)(eb - 1) < 2046u && s.g2 > (tol2 * a) * b;
    return s;
}
struct Rot64 { double tr, ti, tg, c, c2, sq, cm1, sm1; };  // sq = 1/cos
__device__ __forceinline__ Rot64 rotation64(double al, double be, const Unit64& s) {
    const double d = (be - al) * pow2(-s.h);
    const double h = fma(d, d, 4.0 * s.g2);
    // sqrt(h) = r (1 + e/2 + 3 e^2/8) with r = h y, y about 1 / sqrt(h) and e = 1 - h y^2 of about 1e-6
    const double y = rsqrt_approx(h), r = h * y, e1 = fma(-r, y, 1.0);
    double root = fma(r * e1, fma(0.375, e1, 0.5), r);
    if (exponent(d) > 1023 + 500) root = fabs(d);  // (d^2 may overflow; g^2 is nothing beside it)
    double f = rcp_newton(fabs(d) + root);
    f = __hiloint2double((__double2hiint(f) + (1 << 20)) ^ (__double2hiint(d) & 0x80000000), __double2loint(f));  // 2 f sign(d)
    Rot64 p;
    p.tr = f * s.x;
    p.ti = f * s.y;
    p.tg = (f * s.g2) * pow2(s.h);
    const double t2 = fma(p.tr, p.tr, p.ti * p.ti), q = 1.0 + t2;
    // cos = 1 / sqrt(q) in the same way
    const double c0 = rsqrt_approx(q);
    const double qc = q * c0, e2 = fma(-qc, c0, 1.0);
    p.c = fma(c0 * e2, fma(0.375, e2, 0.5), c0);
    p.c2 = p.c * p.c;
    p.sq = q * p.c;
    p.sm1 = t2 * rcp_newton(1.0 + p.sq);
    p.cm1 = -p.sm1 * p.c;
    return p;
}
// ------------------------------------------------------------ one warp --
// Columns of a group: the 2 B columns of a visit take 2 B RPL complex registers (128
// 32-bit registers at 512 rows complex64, and at 128, 256 and 512 rows complex128).
// Short complex128 columns go in pairs: a group's visit is bound by its one
// scheduler's FP64 unit, and smaller groups spread it over more warps (64 of 64 x 64:
// 7.3 -> 6.8 ms; at 128 rows 2 instead of 4 would cost 152 matrices 41 -> 50 ms).
template <typename R, int RPL> struct GroupCols {
    static constexpr int v = std::is_same<R, float>::value ? (RPL >= 12 ? 2 : 4) : (RPL >= 12 ? 1 : RPL >= 6 ? 2 : RPL == 4 ? 4 : 2);
};

// What a warp carries through a sweep.
template <typename R> struct Sweep {
    R tol2, big2;
    bool big = false;  // this lane's pair was rotated with cos^2 >= big2
    int rot = 0;       // rotations of this warp
    int before = 0;    // of those, in sweeps of a run before its last
};

// A column as the lanes of its lane group hold it: true squared norm, scale minus 1,
// the scale's reciprocal, and (complex128) whether it was rotated, bit 0 in the sweep
// before and bit 1 in this one.
template <typename R> struct Lane {
    R n, d, i;
    int f;
    __device__ __forceinline__ R w() const { return (R)1 + d; }
    __device__ __forceinline__ bool far() const {  // the scale has moved by 2^-6
        if constexpr (std::is_same<R, float>::value) return fabs(d) > (R)(1.0 / 64);
        return (__double2hiint(d) & 0x7fffffff) >= 0x3f900000;
    }
    __device__ __forceinline__ void move(int src) {  // to the column of lane src
        n = __shfl_sync(0xffffffffu, n, src);
        d = __shfl_sync(0xffffffffu, d, src);
        if constexpr (!std::is_same<R, float>::value) {
            i = __shfl_sync(0xffffffffu, i, src);
            f = __shfl_sync(0xffffffffu, f, src);
        }
    }
};

// One round of B disjoint pairs (a[i], y[(i + r) mod B]).  Lane group p holds
// column p of a as ca and column (p + r) mod B of y as cy.  complex128: pairs of two
// columns with no flag set met in the sweep before as the same two vectors and
// were orthogonal: their dot product is left out (late sweeps are mostly such
// checks).  Returns the mask of lanes whose pair rotated.
template <typename R, int RPL, int B, int r>
__device__ __forceinline__ unsigned round_pairs(entry_t<R> (&a)[B][RPL], entry_t<R> (&y)[B][RPL], Lane<R>& ca,
                                                Lane<R>& cy, Sweep<R>& sw, Coef<R>* tb, int lane) {
    constexpr bool k64 = std::is_same<R, double>::value;
    constexpr int L = 32 / B;
    const int p = lane / L;
    R vr[B], vi[B];
    unsigned need = 0xffffffffu;
    if constexpr (k64) {
        need = __ballot_sync(0xffffffffu, ca.f | cy.f);
        if (!need) return 0u;
    }
#pragma unroll
    for (int i = 0; i < B; ++i) {
        vr[i] = 0;
        vi[i] = 0;
        if (!k64 || ((need >> (i * L)) & 1u)) col_dot<RPL>(a[i], y[(i + r) % B], vr[i], vi[i]);
    }
    const R wa = ca.w(), wb = cy.w();
    if constexpr (!k64) {
        ca.i = rcp_newton(wa);
        cy.i = rcp_newton(wb);
    }
    R gr, gi;
    reduce_pairs<R, B>(vr, vi, lane, gr, gi);
    const R sc = wa * wb;
    gr *= sc;
    gi *= sc;
    // a.n, b.n >= 0 (a tracked norm that shrinks a lot is recomputed from its
    // column), so a zero column (g = 0) or a non-finite value fails this test and
    // is left alone
    const R al = ca.n, be = cy.n;
    R g2 = 0;
    bool rot;
    [[maybe_unused]] Unit64 unit;
    if constexpr (k64) {
        unit = in_units(al, be, gr, gi, sw.tol2);
        rot = unit.over;
    } else {
        g2 = gr * gr + gi * gi;
        rot = g2 > (sw.tol2 * al) * be;
    }
    const unsigned m = __ballot_sync(0xffffffffu, rot);
    if (!m) return 0u;
    // (no branch: the lanes of pairs that stay compute along and drop the result)
    R tr, ti, kr, ki, al2, be2;
    if constexpr (k64) {
        const Rot64 q = rotation64(al, be, unit);
        const double u = wb * ca.i, w = (wa * cy.i) * q.c2;
        tr = q.tr * u; ti = q.ti * u; kr = q.tr * w; ki = q.ti * w;
        al2 = al - q.tg;
        be2 = be + q.tg;
        const double da = ca.d + fma(ca.d, q.cm1, q.cm1), db = cy.d + fma(cy.d, q.sm1, q.sm1);
        const double ia = ca.i * q.sq, ib = cy.i * q.c;
        if (rot) { ca.d = da; ca.i = ia; cy.d = db; cy.i = ib; ca.f |= 2; cy.f |= 2; }
    } else {
        if constexpr (Eps<R>::early > 0.0) sw.big = sw.big || (rot && g2 > (sw.big2 * al) * be);
        const Rot<R> q = rotation(al, be, gr, gi, g2);
        const R u = wb * ca.i, w = wa * cy.i * q.c2;
        tr = q.tr * u; ti = q.ti * u; kr = q.tr * w; ki = q.ti * w;
        al2 = al - q.tg;
        be2 = be + q.tg;
        const R cm1 = rot ? q.cm1 : (R)0, sm1 = rot ? q.sm1 : (R)0;
        ca.d = ca.d + fma(ca.d, cm1, cm1);
        cy.d = cy.d + fma(cy.d, sm1, sm1);
    }
    __syncwarp();  // the warp is done with the coefficients of the round before
    // short columns: every pair of the round is sheared, a pair that stays by zero
    // (cheaper than a branch per pair); long ones: only the pairs that rotate
    constexpr bool kAll = RPL <= 4 && !k64;
    if ((kAll || rot) && (lane & (L - 1)) == 0)
        tb[p].set(rot ? tr : (R)0, rot ? ti : (R)0, rot ? kr : (R)0, rot ? ki : (R)0);
    // a norm that lost most of its size (cancellation in the update) is taken from its column
    bool sa, sb;
    if constexpr (k64) {  // by exponents: less than an eighth, or negative
        sa = __double2hiint(al2) < __double2hiint(al) - (3 << 20);
        sb = __double2hiint(be2) < __double2hiint(be) - (3 << 20);
    } else {
        sa = !(al2 > (R)0.125 * al);
        sb = !(be2 > (R)0.125 * be);
    }
    const bool shrunk = rot && (sa || sb);
    if (rot) { ca.n = al2; cy.n = be2; }
    __syncwarp();
    sw.rot += __popc(m) / L;
#pragma unroll
    for (int i = 0; i < B; ++i)
        if (kAll || ((m >> (i * L)) & 1u)) col_rotate<RPL>(a[i], y[(i + r) % B], tb[i]);
    if (__any_sync(0xffffffffu, shrunk)) {
        const unsigned ma = __ballot_sync(0xffffffffu, shrunk && sa), mb = __ballot_sync(0xffffffffu, shrunk && sb);
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if ((ma >> (i * L)) & 1u) {
                const R n2 = col_norm2<RPL>(a[i]);
                if (p == i) ca.n = n2 * ca.w() * ca.w();
            }
            if ((mb >> (i * L)) & 1u) {
                const R n2 = col_norm2<RPL>(y[(i + r) % B]);
                if (p == i) cy.n = n2 * cy.w() * cy.w();
            }
        }
    }
    return m;
}

template <typename R, int RPL, int B, int r>
__device__ __forceinline__ unsigned visit_rounds(entry_t<R> (&a)[B][RPL], entry_t<R> (&y)[B][RPL], Lane<R>& ca,
                                                 Lane<R>& cy, Sweep<R>& sw, Coef<R>* tb, int lane) {
    if constexpr (r == B) {
        return 0u;
    } else {
        unsigned m = round_pairs<R, RPL, B, r>(a, y, ca, cy, sw, tb, lane);
        if constexpr (B > 1) cy.move((lane + 32 / B) & 31);  // lane group p goes on to column (p + r + 1) mod B of y
        return m | visit_rounds<R, RPL, B, r + 1>(a, y, ca, cy, sw, tb, lane);
    }
}

// Multiply the scales out: column i of a by the scale of lane group i.
template <typename R, int RPL, int B>
__device__ __forceinline__ void apply_scales(entry_t<R> (&a)[B][RPL], Lane<R>& c) {
#pragma unroll
    for (int i = 0; i < B; ++i) col_scale<RPL>(a[i], __shfl_sync(0xffffffffu, c.d, i * (32 / B)));
    c.d = (R)0;
    c.i = 1;
}

// The pairs inside a group.
template <typename R, int RPL, int B>
__device__ __forceinline__ bool inner_pairs(entry_t<R> (&a)[B][RPL], Lane<R>& c, Sweep<R>& sw, Coef<R>* tb, int lane) {
    if constexpr (B == 1) {
        return false;
    } else {
        // (B = 2) one pair; (B = 4) three rounds of two pairs: (0,1)(2,3), (0,2)(1,3), (0,3)(1,2).
        // Taken through round_pairs with B/2 columns a side; lane groups of B/2 pairs.
        constexpr int H = B / 2, L = 32 / B, LH = 32 / H;
        const int ph = lane / LH;
        unsigned any = 0u;
        auto one = [&](auto rc) {
            constexpr int k = decltype(rc)::value;
            // columns x(q), z(q) of pair q
            constexpr int x0 = 0, x1 = k == 0 ? 2 : 1;
            constexpr int z0 = k + 1, z1 = k == 0 ? 3 : k == 1 ? 3 : 2;
            entry_t<R> x[H][RPL], z[H][RPL];
#pragma unroll
            for (int q = 0; q < RPL; ++q) {
                x[0][q] = a[x0][q];
                z[0][q] = a[z0][q];
                if constexpr (H == 2) {
                    x[1][q] = a[x1][q];
                    z[1][q] = a[z1][q];
                }
            }
            Lane<R> cx = c, cz = c;
            cx.move((ph == 0 ? x0 : x1) * L);
            cz.move((ph == 0 ? z0 : z1) * L);
            const unsigned m = round_pairs<R, RPL, H, 0>(x, z, cx, cz, sw, tb, lane);
            if (m) {
                any |= m;
#pragma unroll
                for (int q = 0; q < RPL; ++q) {
                    a[x0][q] = x[0][q];
                    a[z0][q] = z[0][q];
                    if constexpr (H == 2) {
                        a[x1][q] = x[1][q];
                        a[z1][q] = z[1][q];
                    }
                }
                // back to one lane group per column
                const int p = lane / L;
                const bool is_x = p == x0 || (H == 2 && p == x1);
                const int src = ((p == x0 || p == z0) ? 0 : 1) * LH;
                cx.move(src);
                cz.move(src);
                c = is_x ? cx : cz;
            }
        };
        one(std::integral_constant<int, 0>{});
        if constexpr (B == 4) {
            one(std::integral_constant<int, 1>{});
            one(std::integral_constant<int, 2>{});
        }
        return any != 0u;
    }
}

// ------------------------------------------------------------- one CTA --
constexpr int kMaxCols = 2 * PTEBD_CHI_LIMIT;  // 512
constexpr int kMaxSlots = 32;
constexpr int kMaxWarps = 16;
// Of cols (cols - 1): a sweep that rotates more lets the next two run into each other.  Flat
// around 0.3 of the pairs: at 0.15, 0.3, 0.5 and never, a step of N = 16, chi = 16 takes 1.150,
// 1.146, 1.153 and 1.206 ms, of N = 128, chi = 64 7.59, 7.56, 7.55 and 7.83 (in FP64 82.4, 82.5,
// 82.4 and 84.8), a 12-layer circuit of N = 50, chi = 64 13.4, 13.5, 13.6 and 14.7.
constexpr float kBusyShare = 0.3f / 2;
// Of cols (cols - 1): a sweep that rotates fewer pairs hands the next the polish threshold.
// At none, 0.05, 0.15 and 0.3 of the pairs the same steps take 1.163, 1.162, 1.146 and 1.148,
// and 7.72, 7.63, 7.56 and 7.51 ms, one of N = 75, chi = 100 8.69, 8.76, 8.66 and 8.70.
constexpr float kPolishShare = 0.15f / 2;
constexpr int kLag = 6;  // positions between a group's way back to W and the reuse of its slot

// Tables of a CTA, ahead of the columns in shared memory.
template <typename R> struct Tables {
    uint64_t full[kMaxSlots];      // TMA loads of the slots
    Coef<R> tb[kMaxWarps][4];      // rotation coefficients of a round, per warp
    R nrm[kMaxCols];               // squared column norms (by column)
    R pnrm[kMaxCols];              // the same in sweep order
    R scl[kMaxCols];               // scales minus 1 (by column)
    R pscl[kMaxCols];              // the same in sweep order
    uint32_t key[kMaxCols];        // sort keys
    int cperm[kMaxCols];           // sweep order -> column
    int prog[kMaxCols];            // I groups that have met group j (in this sweep); j + 1 once it is taken itself
    int aux[kMaxCols];             // streaming: group j was rotated since it was last fetched; cluster: where
                                   // the column at a position lies (CTA << 16 | its place there)
    unsigned char flag[kMaxCols];  // complex128, by column: rotated in the sweep before
    unsigned char pflag[kMaxCols]; // by position: bit 0 the sweep before, bit 1 this one
    unsigned long long total;      // rotations of the SVD
    int rotations, before, abort, max_exp, big;
    int fetch_e, fetch_k, fetch_g, fetch_slot;  // streaming: the next position to fetch, its row, group and slot
};

// The tables, rounded up to 128 bytes, so that the columns start aligned.
template <typename R> constexpr size_t table_bytes() { return (sizeof(Tables<R>) + 127) / 128 * 128; }

// Dynamic shared memory: the tables and `column_area` bytes of columns.
constexpr int kSmemMax = 227 * 1024;
template <typename R> int column_area(int ldw, bool half) {
    // (a column of zeros beside the matrix; at least 64 rows a column on complex64)
    const size_t all = (size_t)(ldw + 1) * (ldw < 64 ? 64 : ldw) * sizeof(cx_t<R>);
    const size_t most = (half ? kSmemMax / 2 - 1024 : kSmemMax) - table_bytes<R>();
    return (int)(all < most ? all : most);
}
// Compute warps: no more than groups of the widest matrix, at most `most`; `half`: half of
// them, so that two CTAs share an SM's registers.
inline int warps_for(int ldw, bool half, int most) {
    if (half) most /= 2;
    return ldw / 4 < most ? ldw / 4 : most;
}

// Where the columns are: streamed from W, in this CTA's shared memory, or spread
// over the shared memory of a cluster.
enum { kStream = 0, kResident = 1, kCluster = 2 };

template <typename R, int RPL, int MODE>
__device__ __noinline__ void jacobi_body(const LayerArgs<R>& A, cx_t<R>* W, int rows, int cols, int j_slot,
                                         int area, Tables<R>* T, cx_t<R>* cbuf) {
    const bool wait_test = A.wait_test != 0;
    const int chi_max = A.chi_max, max_sweeps = A.max_sweeps;
    using C = cx_t<R>;
    constexpr bool RES = MODE != kStream, CL = MODE == kCluster;
    constexpr int B = GroupCols<R, RPL>::v;
    constexpr int L = 32 / B;
    constexpr int mpad = 32 * RPL;  // rows per column in shared memory
    constexpr bool kSkip = std::is_same<R, double>::value;
    constexpr bool kSplit = std::is_same<R, float>::value;
    const int ldw = A.ldw;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ncta = CL ? cluster_size() : 1, crank = CL ? cluster_rank() : 0;
    const int nwc = blockDim.x >> 5;                             // warps of the CTA
    const int nw = nwc * ncta, gw = crank * nwc + warp;          // of all CTAs of the matrix; this one
    const int held = (cols + ncta - 1) / ncta;                   // columns a CTA holds (RES): c = crank, crank + ncta, ...
    const int G = (cols + B - 1) / B;
    const int S = RES ? G : min(kMaxSlots, (int)((area - mpad * sizeof(C)) / (B * mpad * sizeof(C))));  // slots
    C* const zeros = cbuf + (RES ? held : S * B) * mpad;
    const uint32_t col_bytes = (uint32_t)(rows * sizeof(C));
    volatile int* abort_flag = &T->abort;

    // columns in shared memory start as zeros (rows beyond `rows` stay zero)
    for (int e = tid; e < (RES ? held + 1 : S * B + 1) * mpad; e += blockDim.x) cbuf[e] = cmake<C>(0, 0);
    for (int c = tid; c < cols; c += blockDim.x) {
        T->scl[c] = (R)0;
        if constexpr (kSkip) T->flag[c] = 1;  // sweep 0 checks every pair
    }
    fence_async_smem();
    auto sync = [&]() {
        if constexpr (CL) cluster_sync(); else __syncthreads();
    };
    sync();
    // the tables of the CTA that keeps group g's counter, norms and scales
    auto home = [&](int g) -> Tables<R>* {
        if constexpr (CL) return peer(T, g % ncta);
        return T;
    };
    // f(tables) for every CTA of the matrix
    auto everywhere = [&](auto&& f) {
        if constexpr (CL) {
            for (int r = 0; r < ncta; ++r) f(peer(T, r));
        } else {
            f(T);
        }
    };

    // squared norms of the columns (exact); with `first`, the exponent of the
    // largest |entry| is gathered, and the columns are read from W (RES) and put
    // into the pair-split layout (complex64)
    auto column = [&](int c) -> C* { return RES ? cbuf + (c / ncta) * mpad : W + (size_t)c * ldw; };  // (one this CTA holds)
    auto norm_pass = [&](bool first) {
        R mx = 0;
        for (int c = crank + ncta * warp; c < cols; c += nw) {
            R s0 = 0, s1 = 0;
            const C* src = first ? W + (size_t)c * ldw : column(c);
            C* dst = column(c);
            if constexpr (kSplit) {
                for (int g = lane; g < rows / 2; g += 32) {
                    const float4 v = reinterpret_cast<const float4*>(src)[g];
                    s0 = fma(v.x, v.x, s0); s1 = fma(v.y, v.y, s1);
                    s0 = fma(v.z, v.z, s0); s1 = fma(v.w, v.w, s1);
                    if (first) {
                        mx = fmax(mx, fmax(fmax(fabs(v.x), fabs(v.y)), fmax(fabs(v.z), fabs(v.w))));
                        reinterpret_cast<float4*>(dst)[g] = make_float4(v.x, v.z, v.y, v.w);
                    }
                }
            } else {
                for (int r = lane; r < rows; r += 32) {
                    const C v = src[r];
                    s0 = fma(v.x, v.x, s0);
                    s1 = fma(v.y, v.y, s1);
                    if (first) {
                        mx = fmax(mx, fmax(fabs(v.x), fabs(v.y)));
                        if constexpr (RES) dst[r] = v;
                    }
                }
            }
            const R w = (R)1 + T->scl[c], s2 = warp_sum(s0 + s1) * w * w;
            if (lane == 0) everywhere([&](Tables<R>* t) { t->nrm[c] = s2; });
        }
        if (first) {
            mx = warp_max(mx);
            if (lane == 0) everywhere([&](Tables<R>* t) { atomicMax(&t->max_exp, exp_key<R>(mx)); });
            if (!RES) fence_async_global();  // the sweeps read W through TMA as well
        }
    };

    const R tol = (R)(Eps<R>::k * sqrt((double)rows) * Eps<R>::u);
    Sweep<R> sw;
    sw.tol2 = tol * tol;
    sw.big2 = (R)Eps<R>::early * sw.tol2;
    const bool polish = A.polish && Eps<R>::polish > 0.0;
    bool polishing = false;  // the last sweep, with the tighter threshold
    bool converged = false;
    int scale_e = 0;
    int streamed = 0;  // groups streamed in the sweeps before this one (the same on every warp)
    int sweep = 0;
    Coef<R>* tb = T->tb[warp];

    // (one CTA streams columns of 12 and 16 rows a lane, however few)
    const bool twos = RES && (!CL || (RPL < 12 && (cols + 1) * mpad * (int)sizeof(C) <= area));
    bool busy = true;        // a third of the pairs rotated in the last sweep
    bool last_tail = false;  // the polish sweep may leave pairs of dropped columns alone
    int run = 1;             // sweeps between two sorts
    for (sweep = 0; sweep < max_sweeps; sweep += run) {
        // Columns that one CTA holds: while a third of the pairs rotate, sweeps run into each
        // other in twos, the second starting behind the first without a barrier, in the same order
        // of columns.  The pipeline of groups fills and drains once (3 G visits instead of 4 G for
        // G groups and as many warps); later sweeps are sorted each, which saves more rotations
        // than it costs.  complex64 25 of 128 x 128 1.58 -> 1.47 ms.  By size and not by where the
        // columns are: what a cluster holds is streamed in a larger launch, and both have to give
        // the same bits.
        // (Not a polish sweep: with GI < G the groups beyond never finish a sweep of their own.)
        run = twos && !polishing && busy && sweep + 2 <= max_sweeps ? 2 : 1;
        norm_pass(sweep == 0);
        sync();
        if (sweep == 0) {
            // Range guard.  Squared norms and |a^H b|^2 are formed in R: with entries of
            // 2^range_e and more they can overflow (and with tiny entries underflow),
            // which turns a rotation into a plain scaling of the pair.  Such a matrix is
            // scaled by 2^-e, exactly, so that its largest entry lies in [1, 2), and
            // scaled back after the sweeps: a power-of-two scaling commutes with every
            // rounding of the sweeps, so the result equals that of an unbounded exponent
            // range.
            const int ex = T->max_exp - kExpOffset;  // 2^ex <= max |entry| < 2^(ex + 1)
            if (T->max_exp > 0 && (ex >= Eps<R>::range_e || ex < -Eps<R>::range_e)) {
                scale_e = ex;
                const R f = ldexp((R)1, -scale_e);
                for (int c = crank + ncta * warp; c < cols; c += nw) {
                    C* col = column(c);
                    for (int r = lane; r < rows; r += 32) {
                        C v = col[r];
                        v.x *= f; v.y *= f;
                        col[r] = v;
                    }
                }
                if (!RES) fence_async_global();
                sync();
                norm_pass(false);
                sync();
            }
        }
        // sweep order: columns by decreasing norm, ties by index (ranks counted from
        // integer keys, so that any values give a permutation)
        for (int c = tid; c < cols; c += blockDim.x)
            T->key[c] = __float_as_uint((float)T->nrm[c]) & 0x7fffffffu;
        for (int g = tid; g < G; g += blockDim.x) {
            T->prog[g] = 0;
            if constexpr (!CL) T->aux[g] = 0;
        }
        __syncthreads();
        for (int c = tid; c < cols; c += blockDim.x) {
            const uint32_t mine = T->key[c];
            int rank = 0;
            for (int q = 0; q < cols; ++q) {
                const uint32_t k = T->key[q];
                rank += (k > mine || (k == mine && q < c)) ? 1 : 0;
            }
            T->cperm[rank] = c;
            if constexpr (CL) T->aux[rank] = (c % ncta) << 16 | (c / ncta);
            T->pnrm[rank] = T->nrm[c];
            T->pscl[rank] = T->scl[c];
            if constexpr (kSkip) T->pflag[rank] = T->flag[c];
        }
        sync();

        // the polish sweep leaves pairs of two columns beyond chi_max (in the sweep
        // order, by decreasing norm) alone: they are dropped together, a rotation
        // between them changes no kept column and keeps their summed weight
        const int GI = last_tail && chi_max > 0 ? min(G, (chi_max + B - 1) / B) : G;
        {
            bool ok = true;
            const int p = lane / L;
            // Streaming: position in the sweep's stream of groups (rows of I groups one after
            // the other, each from its first group k0 to G - 1), its slot and the slot's phase.
            int rel = 0, slot = 0;
            uint32_t phase = 0;
            if constexpr (!RES) { slot = streamed % S; phase = (uint32_t)(streamed / S) & 1u; }
            auto advance = [&](int d) {
                if constexpr (!RES) {
                    rel += d;
                    slot += d;
                    while (slot >= S) { slot -= S; phase ^= 1u; }
                }
            };
            // The last warp fetches the groups in the order the warps meet them.  `done`: the
            // last position it has met; every position it meets has its bulk group (empty if
            // nothing was stored), so that "all but the last kLag groups complete" says that
            // the positions up to done - kLag are back in W and their slots free.
            auto pump = [&](int done, bool drain) {
                if (lane == 0) {
                    int e = T->fetch_e, k0 = T->fetch_k, g = T->fetch_g, sl = T->fetch_slot;
                    if (drain) bulk_wait<0>(); else bulk_wait<kLag>();
                    const int free_to = drain ? done : done - kLag;
                    fence_async_smem();
                    while (k0 < GI && e - S <= free_to && (k0 == 0 || e - (G - k0) <= free_to)) {
                        const int nc = min(B, cols - g * B);
                        mbar_expect_tx(&T->full[sl], (uint32_t)nc * col_bytes);
                        for (int i = 0; i < nc; ++i)
                            bulk_g2s(cbuf + ((size_t)sl * B + i) * mpad, W + (size_t)T->cperm[g * B + i] * ldw,
                                     col_bytes, &T->full[sl]);
                        ++e;
                        if (++sl == S) sl = 0;
                        if (++g == G) { k0 += nwc; g = k0; }
                    }
                    T->fetch_e = e; T->fetch_k = k0; T->fetch_g = g; T->fetch_slot = sl;
                }
                __syncwarp();
            };
            // What is left to fetch once the last warp has no I group of its own (the last row
            // of a polish sweep): as the groups before get through.
            auto pump_rest = [&]() -> bool {
                bool fine = true;
                while (fine && T->fetch_k < GI) {
                    const int k0 = T->fetch_k, e = T->fetch_e;
                    int tj = e - S, tk = 0;  // the group in the slot
                    while (tj >= G - tk) { tj -= G - tk; tk += nwc; }
                    tj += tk;
                    fine = (e < S || counter_wait(&T->prog[tj], min(tj + 1, min(tk + nwc, GI)), abort_flag)) &&
                           (k0 == 0 || counter_wait(&T->prog[T->fetch_g], k0, abort_flag));
                    fine = __all_sync(0xffffffffu, fine);
                    if (fine) pump(max(e - S, e - (G - k0)), true);
                }
                return fine;
            };
            const bool fetcher = !RES && warp == nwc - 1;
            // column p of group g, from its tables
            auto lane_of = [&](const Tables<R>* t, int g) {
                const int pos = g * B + p;
                Lane<R> c{(R)0, (R)0, (R)1, 0};
                if (pos < cols) {
                    c.n = t->pnrm[pos];
                    c.d = t->pscl[pos];
                    if constexpr (kSkip) {
                        c.f = t->pflag[pos];
                    }
                }
                return c;
            };
            if (fetcher) {
                if (lane == 0) { T->fetch_e = T->fetch_k = T->fetch_g = 0; T->fetch_slot = slot; }
                __syncwarp();
                pump(-1, true);
            }
            const int rows_all = RES ? run * GI : GI;  // rows of I groups, over the sweeps of the run
            for (int k0 = 0; k0 < rows_all && ok; k0 += nw) {
                const int row = k0 + gw;
                if (row >= rows_all) break;
                const bool second = RES && row >= GI;            // of the run's sweeps
                const int I = second ? row - GI : row;
                const int base = second ? G + 1 : 0;             // its counts start here
                const bool counts = !RES || second || run == 1;  // the run's last sweep
                const int rot0 = sw.rot;
                const bool big0 = sw.big;
                const bool last = !RES && I == min(k0 + nw, GI) - 1;  // the last warp of the row
                // Group g has met every I before this one (streaming, the first warp of a row: it
                // has been fetched), the same answer on every lane (warp_ready).
                auto vote = [](bool x) -> bool { return __all_sync(0xffffffffu, x); };
                auto ready = [&](int g, Tables<R>* tg) -> bool {
                    if (RES ? row == 0 : warp == 0) {
                        if constexpr (!RES)
                            return warp_ready(mbar_try_wait(&T->full[slot], phase), vote,
                                              [&] { return mbar_wait(&T->full[slot], phase, abort_flag); });
                        return true;
                    }
                    const bool test = wait_test && sweep == 0 && row == 1 && g == 1;
                    const int met = CL ? counter_acquire_cluster(&tg->prog[g]) : counter_acquire(&tg->prog[g]);
                    return warp_ready(met >= base + I && !test, vote, [&] {
                        return counter_wait<CL>(&tg->prog[g], test ? 0x7fffffff : base + I, abort_flag,
                                                test ? (1ll << 20) : kWaitLimit);
                    });
                };
                auto release = [&](int* c, int v) {
                    if constexpr (CL) counter_release_cluster(c, v); else counter_release(c, v);
                };
                // address of column i of group g in shared memory
                auto sm_col = [&](int g, int i) -> C* {
                    const int pos = g * B + i;  // (columns missing from the last group: a column of zeros)
                    if (pos >= cols) return zeros;
                    if constexpr (CL) return peer(cbuf, T->aux[pos] >> 16) + (T->aux[pos] & 0xffff) * mpad;
                    if constexpr (RES) return cbuf + T->cperm[pos] * mpad;
                    return cbuf + (slot * B + i) * mpad;
                };
                advance(warp);
                Tables<R>* const ti = home(I);
                if (!ready(I, ti)) { ok = false; break; }
                entry_t<R> a[B][RPL];
#pragma unroll
                for (int i = 0; i < B; ++i) col_load<RPL>(a[i], sm_col(I, i), lane);
                const bool ip = I * B + p < cols;
                Lane<R> ca = lane_of(ti, I);
                if constexpr (kSkip) ca.i = rcp_newton(ca.w());
                bool changed = !RES && T->aux[I] != 0;
                __syncwarp();
                if constexpr (!RES)
                    if (lane == 0) release(&ti->prog[I], I + 1);
                if (fetcher) {
                    if (lane == 0)
                        for (int q = 0; q < nwc; ++q) bulk_commit();
                }
                changed = inner_pairs<R, RPL, B>(a, ca, sw, tb, lane) || changed;
                for (int J = I + 1; J < G; ++J) {
                    advance(1);
                    Tables<R>* const tj = home(J);
                    if (!ready(J, tj)) { ok = false; break; }
                    const bool jp = J * B + p < cols;
                    Lane<R> cy = lane_of(tj, J);
                    bool store = last && T->aux[J] != 0;
                    if (!kSkip || __any_sync(0xffffffffu, ca.f | cy.f)) {
                        if constexpr (kSkip) {  // (the reciprocals, the I one's refreshed: it runs along)
                            cy.i = rcp_newton(cy.w());
                            ca.i = fma(ca.i, fma(-ca.w(), ca.i, 1.0), ca.i);
                        }
                        entry_t<R> y[B][RPL];
#pragma unroll
                        for (int i = 0; i < B; ++i) col_load<RPL>(y[i], sm_col(J, i), lane);
                        if (visit_rounds<R, RPL, B, 0>(a, y, ca, cy, sw, tb, lane)) {
                            changed = true;
                            store = last;
                            if (__any_sync(0xffffffffu, cy.far())) apply_scales<R, RPL, B>(y, cy);
                            if (__any_sync(0xffffffffu, ca.far())) apply_scales<R, RPL, B>(a, ca);
                            if (jp && (lane & (L - 1)) == 0) {
                                tj->pnrm[J * B + p] = cy.n;
                                tj->pscl[J * B + p] = cy.d;
                                if constexpr (kSkip) tj->pflag[J * B + p] = (unsigned char)cy.f;
                            }
#pragma unroll
                            for (int i = 0; i < B; ++i)
                                if (J * B + i < cols) col_store<RPL>(y[i], sm_col(J, i), lane, mpad);
                            if constexpr (!RES)
                                if (!last && lane == 0) T->aux[J] = 1;
                        }
                    }
                    __syncwarp();
                    if constexpr (!RES) {
                        if (last) {  // a changed group goes back to W
                            if (lane == 0) {
                                if (store) {
                                    T->aux[J] = 0;
                                    fence_async_smem();
                                    const int nc = min(B, cols - J * B);
                                    for (int i = 0; i < nc; ++i)
                                        bulk_s2g(W + (size_t)T->cperm[J * B + i] * ldw, sm_col(J, i), col_bytes);
                                }
                                bulk_commit();
                                if (!fetcher) bulk_wait<0>();  // another warp refills the slot
                            }
                            __syncwarp();
                        }
                    }
                    if (lane == 0) release(&tj->prog[J], base + I + 1);
                    __syncwarp();
                    if (fetcher) pump(rel, false);
                }
                if (!ok) break;
                if (RES && !counts) {  // (the next sweep of the run decides)
                    sw.before += sw.rot - rot0;
                    sw.rot = rot0;
                    sw.big = big0;
                }
                if (kSkip && RES && ip && (lane & (L - 1)) == 0)
                    ti->pflag[I * B + p] = (unsigned char)(counts ? ca.f : ca.f >> 1);
                if (changed) {
                    if (ip && (lane & (L - 1)) == 0) {
                        ti->pscl[I * B + p] = ca.d;
                        if constexpr (RES) ti->pnrm[I * B + p] = ca.n;
                    }
#pragma unroll
                    for (int i = 0; i < B; ++i)
                        if (I * B + i < cols) {
                            if constexpr (RES) col_store<RPL>(a[i], sm_col(I, i), lane, mpad);
                            else col_store<RPL>(a[i], W + (size_t)T->cperm[I * B + i] * ldw, lane, rows);
                        }
                    if constexpr (kSkip && !RES)
                        if (ip && (lane & (L - 1)) == 0) ti->pflag[I * B + p] = (unsigned char)ca.f;
                }
                if constexpr (RES) {
                    __syncwarp();
                    if (lane == 0) release(&ti->prog[I], base + G + 1);  // through with this sweep
                }
                if (fetcher) pump(rel, true);  // rows shorter than the ring wait for all that was stored
                advance(1);
            }
            if constexpr (!RES) {
                if (ok && fetcher) ok = pump_rest();
                bulk_wait<0>();
                fence_async_global();  // the next sweep reads W through TMA and through plain loads
            }
            if (!ok) everywhere([&](Tables<R>* t) { t->abort = 1; });
        }
        // groups streamed in this sweep
        const int streamed_before = streamed;
        if constexpr (!RES)
            for (int k0 = 0; k0 < GI; k0 += nwc) streamed += G - k0;
        if (lane == 0 && sw.rot) everywhere([&](Tables<R>* t) { atomicAdd(&t->rotations, sw.rot); });
        if (lane == 0 && sw.before) everywhere([&](Tables<R>* t) { atomicAdd(&t->before, sw.before); });
        if (__any_sync(0xffffffffu, sw.big) && lane == 0) everywhere([&](Tables<R>* t) { t->big = 1; });
        sw.rot = 0;
        sw.before = 0;
        sw.big = false;
        sync();
        if (T->abort) {
            // A wait ran out: wait (bounded) for the fetches still in flight and latch the
            // error.  If one still has not landed, the CTA has to return with it in flight
            // (nothing can cancel a bulk copy, and waiting on would hang the GPU):
            // DERR_DRAIN marks the state unusable until it is re-created.
            if (tid == 0 && crank == 0) {
                bool drained = true;
                if constexpr (!RES) {
                    const int n = streamed_before + T->fetch_e;  // groups fetched, over all sweeps
                    for (int e = max(0, n - S); e < n; ++e)
                        if (!mbar_wait(&T->full[e % S], (uint32_t)(e / S) & 1u, nullptr)) drained = false;
                }
                atomicOr(A.err, drained ? DERR_TIMEOUT : (DERR_TIMEOUT | DERR_DRAIN));
            }
            sync();
            return;
        }
        const int rot = T->rotations;
        const bool small = Eps<R>::early > 0.0 && T->big == 0;
        busy = rot > kBusyShare * cols * (cols - 1);
        if (tid == 0) T->total += (unsigned long long)(rot + T->before);
        for (int q = tid; q < cols; q += blockDim.x)
            if (!CL || (q / B) % ncta == crank) {  // (by column, in every CTA)
                const int c = T->cperm[q];
                const R d = T->pscl[q];
                const unsigned char f = T->pflag[q] >> 1;
                everywhere([&](Tables<R>* t) {
                    t->scl[c] = d;
                    if constexpr (kSkip) t->flag[c] = f;
                });
            }
        sync();
        if (tid == 0) { T->rotations = 0; T->before = 0; T->big = 0; }
        // The polish threshold is taken once few pairs rotate; the sweep that under it met no
        // pair above the plain threshold is the last.  When the stopping rule fired before
        // (last_tail), one polish sweep follows.
        if (last_tail || (polishing ? small : !polish && (rot == 0 || small))) {
            converged = true;
            sweep += run;
            break;
        }
        if (polish && !polishing && (rot == 0 || small || rot < kPolishShare * cols * (cols - 1))) {
            polishing = true;
            last_tail = rot == 0 || small;
            const R pt = (R)(Eps<R>::polish * sqrt((double)rows) * Eps<R>::u);
            sw.big2 = sw.tol2;
            sw.tol2 = pt * pt;
        }
    }
    __syncthreads();
    if (!converged && tid == 0 && crank == 0) atomicOr(A.err, DERR_NOT_CONVERGED);
    if (tid == 0 && crank == 0) {
        const unsigned long long visits = (unsigned long long)sweep * (unsigned long long)(cols * (cols - 1) / 2) *
                                          (unsigned long long)rows;
        A.slot_sweeps[j_slot] = sweep;
        if (A.refine) {  // the FP64 resolution of a complex64 state, counted apart
            atomicAdd(&A.work[8], 1ull);
            atomicAdd(&A.work[9], visits);
        } else {
            atomicAdd(&A.work[0], visits);
            atomicAdd(&A.work[2], T->total);
            atomicAdd(&A.work[3], (unsigned long long)sweep);
            atomicAdd(&A.work[4], 1ull);
            if (A.mode == 1) {  // tSU factors, counted apart as well
                atomicAdd(&A.work[5], visits);
                atomicAdd(&A.work[6], (unsigned long long)sweep);
                atomicAdd(&A.work[7], 1ull);
            }
        }
    }
    // FP64 column norms = singular values; the columns' scales are multiplied out, the
    // range guard's scaling is undone and the pair-split layout turned back into plain
    // complex columns
    double* nrm = A.norms + (size_t)j_slot * ldw;
    const R unscale = ldexp((R)1, scale_e);
    for (int c = crank + ncta * warp; c < cols; c += nw) {
        double acc = 0.0;
        const C* src = column(c);
        C* dst = W + (size_t)c * ldw;
        const double w = 1.0 + (double)T->scl[c];
        const R f = (R)w * unscale;
        if constexpr (kSplit) {
            for (int g = lane; g < rows / 2; g += 32) {
                float4 v = reinterpret_cast<const float4*>(src)[g];
                acc = fma((double)v.x, (double)v.x, acc);
                acc = fma((double)v.z, (double)v.z, acc);
                acc = fma((double)v.y, (double)v.y, acc);
                acc = fma((double)v.w, (double)v.w, acc);
                v.x *= f; v.y *= f; v.z *= f; v.w *= f;
                reinterpret_cast<float4*>(dst)[g] = make_float4(v.x, v.z, v.y, v.w);
            }
        } else {
            for (int r = lane; r < rows; r += 32) {
                C v = src[r];
                acc = fma((double)v.x, (double)v.x, acc);
                acc = fma((double)v.y, (double)v.y, acc);
                v.x *= f; v.y *= f;
                dst[r] = v;
            }
        }
        acc = warp_sum(acc);
        if (lane == 0) {
            const double s = ldexp(sqrt(acc) * w, scale_e);
            if (!isfinite(s)) atomicOr(A.err, DERR_NONFINITE);
            nrm[c] = s;
        }
    }
}

// Prologue of the kernels: which matrix, its size, the tables.
template <typename R> struct Start {
    int rows, cols, area, slot;
    cx_t<R>* W;
    Tables<R>* T;
    cx_t<R>* cbuf;
    bool go;
};
template <typename R>
__device__ __forceinline__ Start<R> start(const LayerArgs<R>& A, int area, unsigned char* smem, int slot) {
    Start<R> s;
    s.slot = slot;
    const int32_t* d = A.dims + slot * kDims;
    s.go = !(A.refine == 1 && d[D_REFINE] != 1);  // the FP64 resolution runs only undecided bonds
    if (!s.go) return s;
    s.rows = A.pass == 1 ? 2 * d[D_CL] : d[D_ROWS];
    s.cols = A.pass == 1 ? d[D_CM] : d[D_COLS];
    s.area = area;
    s.W = A.w + (size_t)slot * A.ldw * A.ldw;
    s.T = reinterpret_cast<Tables<R>*>(smem);
    s.cbuf = reinterpret_cast<cx_t<R>*>(smem + table_bytes<R>());
    if (threadIdx.x == 0) {
        for (int i = 0; i < kMaxSlots; ++i) mbar_init(&s.T->full[i], 1);
        mbar_init_fence();
        s.T->rotations = 0; s.T->before = 0; s.T->total = 0; s.T->abort = 0; s.T->max_exp = 0; s.T->big = 0; s.T->fetch_e = 0;
    }
    return s;
}

template <typename R, int RPL, int MODE>
__device__ __forceinline__ void run(const LayerArgs<R>& A, const Start<R>& s) {
    jacobi_body<R, RPL, MODE>(A, s.W, s.rows, s.cols, s.slot, s.area, s.T, s.cbuf);
}
// One CTA: columns that fit in the area stay there.
template <typename R, int RPL>
__device__ __forceinline__ void run_alone(const LayerArgs<R>& A, const Start<R>& s) {
    const size_t need = (size_t)(s.cols + 1) * 32 * RPL * sizeof(cx_t<R>);
    if (need <= (size_t)s.area) run<R, RPL, kResident>(A, s);
    else run<R, RPL, kStream>(A, s);
}
// A cluster: spread over it when there are enough groups for its warps and the columns
// fit; otherwise its first CTA works alone.
template <typename R, int RPL>
__device__ __forceinline__ void run_cluster(const LayerArgs<R>& A, const Start<R>& s) {
    const int n = cluster_size();
    const size_t need = (size_t)((s.cols + n - 1) / n + 1) * 32 * RPL * sizeof(cx_t<R>);
    if (need <= (size_t)s.area && s.cols >= 12 * GroupCols<R, RPL>::v) {
        run<R, RPL, kCluster>(A, s);
    } else if (cluster_rank() == 0) {
        if constexpr (RPL >= 12) run<R, RPL, kStream>(A, s);
        else run_alone<R, RPL>(A, s);
    }
}

// Launch of `kernel` on `count` matrices by clusters of n CTAs.
template <typename R, typename K>
cudaError_t launch_cluster(K kernel, const LayerArgs<R>& a, int n, int threads, size_t smem, int area, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(a.count * n);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = n;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a, area);
}

// How many clusters of n CTAs (n = 2 .. 8) of a kernel run at once.
constexpr int kMaxCluster = 8;
template <typename K> cudaError_t clusters_at_once(K kernel, int threads, size_t smem, int (&most)[kMaxCluster + 1]) {
    for (int n = 2; n <= kMaxCluster; ++n) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(n);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = n;
        at.val.clusterDim.y = 1;
        at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int c = 0;
        const cudaError_t e = cudaOccupancyMaxActiveClusters(&c, kernel, &cfg);
        if (e != cudaSuccess) return e;
        most[n] = c;
    }
    return cudaSuccess;
}
struct MostClusters { int n[kMaxCluster + 1]; };
// The same on the current device, found on first use there (zeros, and no clusters, where
// the query fails).
template <typename R> MostClusters most_clusters(void (*kernel)(LayerArgs<R>, int)) {
    static PerDevice<const void*, MostClusters> found;
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return MostClusters{};
    return found.get(device, reinterpret_cast<const void*>(kernel), [&](MostClusters* m) {
        const cudaError_t e = clusters_at_once(kernel, 256, kSmemMax, m->n);
        if (e != cudaSuccess) cudaGetLastError();
        return (int)e;
    });
}
// The dynamic shared memory of a kernel that runs in clusters, and their number.  The
// attribute belongs to the device's context: set on every call.
template <typename R> cudaError_t prepare_clusters(void (*kernel)(LayerArgs<R>, int)) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e == cudaSuccess) most_clusters(kernel);
    return e;
}
// CTAs for each of `bonds` matrices in flight together: as many as still run all at once.
inline int cluster_for(int bonds, const int (&most)[kMaxCluster + 1]) {
    for (int n = kMaxCluster; n > 1; --n)
        if (bonds <= most[n]) return n;
    return 1;
}

}  // namespace jac
}  // namespace ptebd
