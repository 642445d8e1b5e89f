// One-sided Jacobi SVD of complex64 matrices whose left vectors a caller asked for
// (ptebd_svd_batched with u).
//
// The sweeps stop with the columns orthogonal to 8 sqrt(rows) 2^-24, and what is left
// below that depends on the order in which the pairs met: the isometry U S^-1 (U^H A)
// of a 300 x 240 Ginibre matrix lies 1.2e-4 off the exact one, in another direction for
// every order.  Callers hold vectors of the order below, so these keep it, where the
// pipeline of column groups (ptebd_jacobi.cuh, which takes the layers and the calls for
// singular values alone) would move them by as much.
//
// One CTA of 16 warps a matrix; the columns stay in global memory / L2.  Blocks of 16
// columns, by decreasing column norm (re-sorted at the start of every sweep), meet in
// row-cyclic order:
//   * block I is held in registers, one column per warp, after its own pairs have been
//     rotated in shared memory (round-robin);
//   * every later block J is streamed through a double-buffered stage by TMA bulk
//     copies and meets I in 16 rounds: warp w takes column (w + r) mod 16 of J, handed
//     on from warp w + 1 through that column's round counter (release / acquire), and a
//     TMA bulk store writes the block back.
// The squared norms are recomputed at the start of every sweep and tracked through the
// rotations; one that loses most of its size is recomputed from its column.  A rotation
// is applied as a + (cos - 1) a - s b, so that it keeps the norms when the angle is below
// the unit roundoff.
//
// What bounds it: the latency of a pair's chain, one pair a warp.  152 matrices of
// 64 x 50, 128 x 128, 256 x 200 and 512 x 400: 0.82, 3.92, 10.4 and 55.2 ms.
//
// Every wait is bounded and voted on by its warp; one that runs out raises the abort
// flag, drains the CTA's own copies, latches DERR_TIMEOUT and returns.
#include "ptebd_jacobi.cuh"

namespace ptebd {
namespace jac {

namespace {

constexpr int kBlock = 16;  // columns of a block = warps

struct BlockTables {
    uint64_t bar[2];                // TMA loads of the J stages
    float jn2[2][kBlock];           // tracked |col|^2 of the stages' columns
    float in2[kBlock];              // of block I, among its own pairs
    int done[2][kBlock];            // rounds completed on each column of each stage
    int pending[2], pending_phase[2];  // a load not yet waited for by thread 0, and the phase it completes
    int rotations, abort, max_exp, big;
    int order[kMaxCols];            // sweep order -> column
    uint32_t key[kMaxCols];
    float nrm2[kMaxCols];           // squared column norms (by column)
};

__device__ __forceinline__ void counter_release_add(int* p) {
    asm volatile("red.release.cta.shared::cta.add.u32 [%0], 1;" ::"r"(smem_u32(p)) : "memory");
}
__device__ __forceinline__ void bulk_wait_read_all() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Columns of more than 32 rows are kept pair-split while the sweeps run (ptebd_jacobi.cuh):
// entry 2 h is (Re r, Re r + 1), entry 2 h + 1 (Im r, Im r + 1), r = 64 h + 2 lane.  With one
// entry a lane (RPL = 1) entry 0 is row `lane` as a complex number.
template <int RPL>
__device__ __forceinline__ void load_rows(float2 (&v)[RPL], const float2* col, int lane, int rows, bool valid) {
    if constexpr (RPL >= 2) {
#pragma unroll
        for (int h = 0; h < RPL / 2; ++h) {
            const int r = 64 * h + 2 * lane;  // (rows is even)
            float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
            if (valid && r < rows) t = *reinterpret_cast<const float4*>(col + r);
            v[2 * h] = make_float2(t.x, t.y);
            v[2 * h + 1] = make_float2(t.z, t.w);
        }
    } else {
        v[0] = valid && lane < rows ? col[lane] : make_float2(0.f, 0.f);
    }
}
template <int RPL>
__device__ __forceinline__ void store_rows(const float2 (&v)[RPL], float2* col, int lane, int rows) {
    if constexpr (RPL >= 2) {
#pragma unroll
        for (int h = 0; h < RPL / 2; ++h) {
            const int r = 64 * h + 2 * lane;
            if (r < rows)
                *reinterpret_cast<float4*>(col + r) = make_float4(v[2 * h].x, v[2 * h].y, v[2 * h + 1].x, v[2 * h + 1].y);
        }
    } else {
        if (lane < rows) col[lane] = v[0];
    }
}
template <int RPL>
__device__ __forceinline__ float rows_norm2(const float2 (&a)[RPL]) {
    float s0 = 0, s1 = 0;
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
        s0 = fma(a[q].x, a[q].x, s0);
        s1 = fma(a[q].y, a[q].y, s1);
    }
    return warp_sum(s0 + s1);
}
// a^H b over this lane's rows
template <int RPL>
__device__ __forceinline__ void rows_dot(const float2 (&a)[RPL], const float2 (&b)[RPL], float& gr, float& gi) {
    if constexpr (RPL >= 2) {  // one partial sum per row of the pair
        float gr0 = 0, gr1 = 0, gi0 = 0, gi1 = 0;
#pragma unroll
        for (int h = 0; h < RPL / 2; ++h) {
            const float2 ar = a[2 * h], ai = a[2 * h + 1], br = b[2 * h], bi = b[2 * h + 1];
            gr0 = fmaf(ar.x, br.x, gr0); gr0 = fmaf(ai.x, bi.x, gr0);
            gi0 = fmaf(ar.x, bi.x, gi0); gi0 = fmaf(-ai.x, br.x, gi0);
            gr1 = fmaf(ar.y, br.y, gr1); gr1 = fmaf(ai.y, bi.y, gr1);
            gi1 = fmaf(ar.y, bi.y, gi1); gi1 = fmaf(-ai.y, br.y, gi1);
        }
        gr = gr0 + gr1;
        gi = gi0 + gi1;
    } else {
        gr = fmaf(a[0].y, b[0].y, a[0].x * b[0].x);
        gi = fmaf(-a[0].y, b[0].x, a[0].x * b[0].y);
    }
}

// tan (t), cos - 1 and sin e^{i arg g} of the rotation that diagonalises
// [[al, g], [conj(g), be]], and tan |g|.  t is the smaller root of t^2 + (d / |g|) t - 1 = 0,
// formed without the quotient; cos is refined by one Newton step.  (Taken as a factor, whose
// rounding leaves the norms 5e-8 to 1.2e-7 too small in the mean; another form would move the
// results, as another order would.)
struct Turn { float cm1, sr, si, tg; };
__device__ __forceinline__ Turn turn_of(float al, float be, float gr, float gi, float g2) {
    const float ig = rsqrtf(g2);
    const float g = g2 * ig;
    const float d = be - al;
    const float h = fmaf(d, d, 4.0f * g2);
    const float root = h * rsqrtf(h);
    float t = __fdividef(2.0f * g, fabsf(d) + root);
    if (d < 0.0f) t = -t;
    const float q = fmaf(t, t, 1.0f);
    float c = rsqrtf(q);
    c = c * fmaf(-0.5f * q * c, c, 1.5f);
    Turn p;
    p.cm1 = __fdividef(-(t * t) * (c * c), 1.0f + c);
    const float s = t * c;
    p.sr = s * gr * ig;
    p.si = s * gi * ig;
    p.tg = t * g;
    return p;
}
// The rotation; b, and with BOTH a, go to their slots in shared memory as soon as their rows
// are formed, so that the stores are under way before the rotation ends and the next warp
// waits less for the column (10 of 300 x 300: 35.8 -> 31.7 ms).
template <int RPL, bool BOTH>
__device__ __forceinline__ void rows_rotate(float2 (&a)[RPL], float2 (&b)[RPL], const Turn& p, float2* slot_a,
                                            float2* slot_b) {
    const int lane = threadIdx.x & 31;
    if constexpr (RPL >= 2) {
        const unsigned long long cm = pk2(p.cm1, p.cm1);
        const unsigned long long sr = pk2(p.sr, p.sr), msr = pk2(-p.sr, -p.sr);
        const unsigned long long si = pk2(p.si, p.si), msi = pk2(-p.si, -p.si);
#pragma unroll
        for (int h = 0; h < RPL / 2; ++h) {
            const unsigned long long ax = pk2(a[2 * h].x, a[2 * h].y), ay = pk2(a[2 * h + 1].x, a[2 * h + 1].y);
            const unsigned long long bx = pk2(b[2 * h].x, b[2 * h].y), by = pk2(b[2 * h + 1].x, b[2 * h + 1].y);
            const unsigned long long t1 = fma2(msi, by, mul2(msr, bx));  // -(sr br + si bi)
            const unsigned long long t2 = fma2(si, bx, mul2(msr, by));   // -(sr bi - si br)
            const unsigned long long t3 = fma2(msi, ay, mul2(sr, ax));   // sr ar - si ai
            const unsigned long long t4 = fma2(si, ax, mul2(sr, ay));    // sr ai + si ar
            a[2 * h] = upk2(add2(ax, fma2(cm, ax, t1)));
            a[2 * h + 1] = upk2(add2(ay, fma2(cm, ay, t2)));
            b[2 * h] = upk2(add2(bx, fma2(cm, bx, t3)));
            b[2 * h + 1] = upk2(add2(by, fma2(cm, by, t4)));
            *reinterpret_cast<float4*>(slot_b + 64 * h + 2 * lane) =
                make_float4(b[2 * h].x, b[2 * h].y, b[2 * h + 1].x, b[2 * h + 1].y);
            if constexpr (BOTH)
                *reinterpret_cast<float4*>(slot_a + 64 * h + 2 * lane) =
                    make_float4(a[2 * h].x, a[2 * h].y, a[2 * h + 1].x, a[2 * h + 1].y);
        }
    } else {
        const float ar = a[0].x, ai = a[0].y, br = b[0].x, bi = b[0].y;
        a[0].x = ar + (p.cm1 * ar - (p.sr * br + p.si * bi));
        a[0].y = ai + (p.cm1 * ai - (p.sr * bi - p.si * br));
        b[0].x = br + (p.cm1 * br + (p.sr * ar - p.si * ai));
        b[0].y = bi + (p.cm1 * bi + (p.sr * ai + p.si * ar));
        slot_b[lane] = b[0];
        if constexpr (BOTH) slot_a[lane] = a[0];
    }
}

struct Thresholds { float tol2, big2; };

// Rotates the pair (a, b) of one warp, and stores it, unless it is orthogonal to the
// threshold; al and be are its tracked squared norms.  A zero column or a non-finite value fails the test.
template <int RPL, bool BOTH>
__device__ __forceinline__ bool pair_rotate(float2 (&a)[RPL], float2 (&b)[RPL], float& al, float& be,
                                            const Thresholds& th, bool& big, float2* slot_a, float2* slot_b) {
    float gr, gi;
    rows_dot<RPL>(a, b, gr, gi);
    gr = warp_sum(gr);
    gi = warp_sum(gi);
    const float g2 = gr * gr + gi * gi;
    if (!(g2 > (th.tol2 * al) * be)) return false;
    big = big || (g2 > (th.big2 * al) * be);
    const Turn p = turn_of(al, be, gr, gi, g2);
    rows_rotate<RPL, BOTH>(a, b, p, slot_a, slot_b);
    float al2 = al - p.tg, be2 = be + p.tg;
    if (!(al2 > 0.125f * al)) al2 = rows_norm2<RPL>(a);
    if (!(be2 > 0.125f * be)) be2 = rows_norm2<RPL>(b);
    al = al2;
    be = be2;
    return true;
}

template <int RPL>
__device__ void blocks_body(float2* W, int ldw, int rows, int cols, int max_sweeps, double* norms, uint32_t* err,
                            float2* stage, BlockTables* T) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int mpad = 32 * RPL;  // = ldw: the class of a height is its power of two
    float2* const buf_j[2] = {stage, stage + kBlock * ldw};
    float2* const buf_i = stage + 2 * kBlock * ldw;
    const float tol = (float)(Eps<float>::k * sqrt((double)rows) * Eps<float>::u);
    Thresholds th;
    th.tol2 = tol * tol;
    th.big2 = (float)Eps<float>::early * th.tol2;
    const int nb = (cols + kBlock - 1) / kBlock;
    const uint32_t col_bytes = (uint32_t)(rows * sizeof(float2));
    uint32_t phase[2] = {0u, 0u};
    int passed[2] = {0, 0};  // J blocks that have been through each stage
    int cur = 0, scale_e = 0;
    bool converged = false;

    auto vote = [](bool x) -> bool { return __all_sync(0xffffffffu, x); };
    auto load_block = [&](int J, int buf) {  // one thread
        const int c0 = J * kBlock, n = min(kBlock, cols - c0);
        // the tracked norms the columns enter the stage with (published by the barrier's arrival)
        for (int c = 0; c < n; ++c) T->jn2[buf][c] = T->nrm2[T->order[c0 + c]];
        mbar_expect_tx(&T->bar[buf], (uint32_t)n * col_bytes);
        for (int c = 0; c < n; ++c)
            bulk_g2s(buf_j[buf] + (size_t)c * ldw, W + (size_t)T->order[c0 + c] * ldw, col_bytes, &T->bar[buf]);
        T->pending[buf] = 1;
        T->pending_phase[buf] = (int)phase[buf];
    };
    // exact squared norms; `first`: the exponent of the largest |entry| is gathered and the
    // columns are put into the pair-split layout
    auto norm_pass = [&](bool first) {
        float mx = 0;
        for (int c = warp; c < cols; c += kBlock) {
            float s0 = 0, s1 = 0;
            if constexpr (RPL >= 2) {
                float4* col = reinterpret_cast<float4*>(W + (size_t)c * ldw);
                for (int g = lane; g < rows / 2; g += 32) {
                    const float4 v = col[g];
                    s0 = fma(v.x, v.x, s0); s1 = fma(v.y, v.y, s1);
                    s0 = fma(v.z, v.z, s0); s1 = fma(v.w, v.w, s1);
                    if (first) {
                        mx = fmax(mx, fmax(fmax(fabs(v.x), fabs(v.y)), fmax(fabs(v.z), fabs(v.w))));
                        col[g] = make_float4(v.x, v.z, v.y, v.w);
                    }
                }
            } else {
                for (int r = lane; r < rows; r += 32) {
                    const float2 v = W[(size_t)c * ldw + r];
                    s0 = fma(v.x, v.x, s0);
                    s1 = fma(v.y, v.y, s1);
                    if (first) mx = fmax(mx, fmax(fabs(v.x), fabs(v.y)));
                }
            }
            const float s2 = warp_sum(s0 + s1);
            if (lane == 0) T->nrm2[c] = s2;
        }
        if (first) {
            mx = warp_max(mx);
            if (lane == 0) atomicMax(&T->max_exp, exp_key<float>(mx));
            fence_async_global();  // the sweeps read W through TMA as well
        }
    };

    for (int sweep = 0; sweep < max_sweeps && !converged; ++sweep) {
        if (tid == 0) {
            T->rotations = 0;
            T->big = 0;
            bulk_wait<0>();
            fence_async_global();
        }
        __syncthreads();
        norm_pass(sweep == 0);
        __syncthreads();
        if (sweep == 0) {  // range guard, as in ptebd_jacobi.cuh
            const int ex = T->max_exp - kExpOffset;
            if (T->max_exp > 0 && (ex >= Eps<float>::range_e || ex < -Eps<float>::range_e)) {
                scale_e = ex;
                const float f = ldexp(1.0f, -scale_e);
                for (int c = warp; c < cols; c += kBlock)
                    for (int r = lane; r < rows; r += 32) {
                        float2 v = W[(size_t)c * ldw + r];
                        v.x *= f; v.y *= f;
                        W[(size_t)c * ldw + r] = v;
                    }
                fence_async_global();
                __syncwarp();
                norm_pass(false);
                __syncthreads();
            }
        }
        // sweep order: columns by decreasing norm, ties by index
        for (int c = tid; c < cols; c += blockDim.x) T->key[c] = __float_as_uint(T->nrm2[c]) & 0x7fffffffu;
        __syncthreads();
        for (int c = tid; c < cols; c += blockDim.x) {
            const uint32_t mine = T->key[c];
            int rank = 0;
            for (int q = 0; q < cols; ++q) {
                const uint32_t k = T->key[q];
                rank += (k > mine || (k == mine && q < c)) ? 1 : 0;
            }
            T->order[rank] = c;
        }
        __syncthreads();

        int rot = 0;       // rotations of this warp in the sweep
        bool big = false;  // one of them had cos^2 >= big2
        for (int I = 0; I < nb; ++I) {
            // all earlier bulk stores have landed before the plain loads of block I
            if (tid == 0) { bulk_wait<0>(); fence_async_global(); }
            __syncthreads();
            const bool mine = I * kBlock + warp < cols;
            const int my_col = mine ? T->order[I * kBlock + warp] : 0;
            float2 a[RPL];
            load_rows<RPL>(a, W + (size_t)my_col * ldw, lane, rows, mine);
            store_rows<RPL>(a, buf_i + (size_t)warp * ldw, lane, mpad);
            if (lane == 0) T->in2[warp] = mine ? T->nrm2[my_col] : 0.0f;
            __syncthreads();
            for (int r = 0; r < kBlock - 1; ++r) {
                if (warp < kBlock / 2) {
                    auto player = [&](int pos) { return pos == 0 ? 0 : 1 + ((pos - 1 + r) % (kBlock - 1)); };
                    const int p = player(warp), q = player(kBlock - 1 - warp);
                    if (I * kBlock + p < cols && I * kBlock + q < cols) {
                        float2 x[RPL], y[RPL];
                        float2 *slot_p = buf_i + p * mpad, *slot_q = buf_i + q * mpad;
                        load_rows<RPL>(x, slot_p, lane, mpad, true);
                        load_rows<RPL>(y, slot_q, lane, mpad, true);
                        float nx = T->in2[p], ny = T->in2[q];
                        if (pair_rotate<RPL, true>(x, y, nx, ny, th, big, slot_p, slot_q)) {
                            __syncwarp();
                            if (lane == 0) {
                                T->in2[p] = nx;
                                T->in2[q] = ny;
                            }
                            ++rot;
                        }
                    }
                }
                __syncthreads();
            }
            load_rows<RPL>(a, buf_i + (size_t)warp * ldw, lane, mpad, true);
            float al = T->in2[warp];

            if (I + 1 < nb && tid == 0) load_block(I + 1, cur);
            for (int J = I + 1; J < nb; ++J) {
                const int nxt = cur ^ 1;
                if (J + 1 < nb && tid == 0) {
                    bulk_wait_read_all();  // the store that last read that stage is done reading
                    load_block(J + 1, nxt);
                }
                bool ok = vote(mbar_wait(&T->bar[cur], phase[cur], &T->abort));
                if (tid == 0 && ok) T->pending[cur] = 0;
                // (the counters only grow: no older round can be mistaken for the one needed)
                const int base = passed[cur] * kBlock;
                float2* const stage_j = buf_j[cur];
                float* const jn2 = T->jn2[cur];
                int* const done = T->done[cur];
                for (int r = 0; r < kBlock && ok; ++r) {
                    const int jc = (warp + r) & (kBlock - 1), place = J * kBlock + jc;
                    if (r > 0)
                        ok = warp_ready(counter_acquire(&done[jc]) >= base + r, vote,
                                        [&] { return counter_wait(&done[jc], base + r, &T->abort); });
                    if (!ok) break;
                    if (place < cols) {
                        float be = jn2[jc];
                        if (mine) {
                            float2 y[RPL];
                            float2* slot = stage_j + jc * mpad;
                            load_rows<RPL>(y, slot, lane, mpad, true);
                            if (pair_rotate<RPL, false>(a, y, al, be, th, big, nullptr, slot)) {
                                jn2[jc] = be;  // (every lane: the same value)
                                ++rot;
                            }
                        }
                        if (r == kBlock - 1) T->nrm2[T->order[place]] = be;
                    }
                    __syncwarp();
                    if (lane == 0) counter_release_add(&done[jc]);
                }
                if (!ok && lane == 0) atomicOr(&T->abort, 1);
                phase[cur] ^= 1u;
                ++passed[cur];
                fence_async_smem();
                __syncthreads();
                if (T->abort) {
                    // Wait (bounded) for the loads still in flight; one that has not landed
                    // cannot be cancelled, and the CTA returns with it in flight.
                    if (tid == 0) {
                        bool drained = true;
                        for (int b = 0; b < 2; ++b)
                            if (T->pending[b] && !mbar_wait(&T->bar[b], (uint32_t)T->pending_phase[b], nullptr))
                                drained = false;
                        bulk_wait<0>();
                        atomicOr(err, drained ? DERR_TIMEOUT : (DERR_TIMEOUT | DERR_DRAIN));
                    }
                    __syncthreads();
                    return;
                }
                if (tid == 0) {  // block J goes back
                    const int c0 = J * kBlock, n = min(kBlock, cols - c0);
                    for (int c = 0; c < n; ++c)
                        bulk_s2g(W + (size_t)T->order[c0 + c] * ldw, buf_j[cur] + (size_t)c * ldw, col_bytes);
                    bulk_commit();
                }
                cur = nxt;
            }
            if (mine) {
                store_rows<RPL>(a, W + (size_t)my_col * ldw, lane, rows);
                if (lane == 0) T->nrm2[my_col] = al;
            }
            fence_async_global();
            __syncthreads();
        }
        if (lane == 0 && rot) atomicAdd(&T->rotations, rot);
        if (lane == 0 && big) T->big = 1;
        __syncthreads();
        converged = T->rotations == 0 || T->big == 0;
        __syncthreads();
    }
    if (tid == 0) { bulk_wait<0>(); fence_async_global(); }
    __syncthreads();
    if (!converged && tid == 0) atomicOr(err, DERR_NOT_CONVERGED);
    // FP64 column norms = singular values; plain complex columns again, unscaled
    const float unscale = ldexp(1.0f, scale_e);
    for (int c = warp; c < cols; c += kBlock) {
        double acc = 0.0;
        if constexpr (RPL >= 2) {
            float4* col = reinterpret_cast<float4*>(W + (size_t)c * ldw);
            for (int g = lane; g < rows / 2; g += 32) {
                float4 v = col[g];
                acc = fma((double)v.x, (double)v.x, acc);
                acc = fma((double)v.z, (double)v.z, acc);
                acc = fma((double)v.y, (double)v.y, acc);
                acc = fma((double)v.w, (double)v.w, acc);
                if (scale_e != 0) { v.x *= unscale; v.y *= unscale; v.z *= unscale; v.w *= unscale; }
                col[g] = make_float4(v.x, v.z, v.y, v.w);
            }
        } else {
            for (int r = lane; r < rows; r += 32) {
                float2 v = W[(size_t)c * ldw + r];
                acc = fma((double)v.x, (double)v.x, acc);
                acc = fma((double)v.y, (double)v.y, acc);
                if (scale_e != 0) {
                    v.x *= unscale; v.y *= unscale;
                    W[(size_t)c * ldw + r] = v;
                }
            }
        }
        acc = warp_sum(acc);
        if (lane == 0) {
            const double s = ldexp(sqrt(acc), scale_e);
            if (!isfinite(s)) atomicOr(err, DERR_NONFINITE);
            norms[c] = s;
        }
    }
}

// grid (matrices), 512 threads; three stages of 16 columns, then the tables.
__global__ void __launch_bounds__(32 * kBlock, 1) k_jacobi_blocks(float2* w, int ldw, int rows, int cols, int max_sweeps,
                                                                  double* norms, uint32_t* err) {
    extern __shared__ __align__(128) unsigned char smem[];
    float2* stage = reinterpret_cast<float2*>(smem);
    const int entries = 3 * kBlock * ldw;
    BlockTables* T = reinterpret_cast<BlockTables*>(stage + entries);
    for (int e = threadIdx.x; e < entries; e += blockDim.x) stage[e] = make_float2(0.f, 0.f);  // (rows beyond `rows`)
    if (threadIdx.x < 2 * kBlock) T->done[threadIdx.x / kBlock][threadIdx.x % kBlock] = 0;
    if (threadIdx.x == 0) {
        mbar_init(&T->bar[0], 1);
        mbar_init(&T->bar[1], 1);
        mbar_init_fence();
        T->pending[0] = T->pending[1] = 0;
        T->abort = 0;
        T->max_exp = 0;
    }
    fence_async_smem();
    __syncthreads();
    float2* W = w + (size_t)blockIdx.x * ldw * ldw;
    double* nrm = norms + (size_t)blockIdx.x * ldw;
    if (rows <= 32) blocks_body<1>(W, ldw, rows, cols, max_sweeps, nrm, err, stage, T);
    else if (rows <= 64) blocks_body<2>(W, ldw, rows, cols, max_sweeps, nrm, err, stage, T);
    else if (rows <= 128) blocks_body<4>(W, ldw, rows, cols, max_sweeps, nrm, err, stage, T);
    else if (rows <= 256) blocks_body<8>(W, ldw, rows, cols, max_sweeps, nrm, err, stage, T);
    else blocks_body<16>(W, ldw, rows, cols, max_sweeps, nrm, err, stage, T);
}

size_t blocks_smem(int ldw) { return (size_t)3 * kBlock * ldw * sizeof(float2) + sizeof(BlockTables); }

}  // namespace
}  // namespace jac

cudaError_t jacobi_blocks_prepare() {
    return cudaFuncSetAttribute(jac::k_jacobi_blocks, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)jac::blocks_smem(jac::kMaxCols));
}

cudaError_t launch_jacobi_blocks(const LayerArgs<float>& a, int rows, int cols, cudaStream_t s) {
    jac::k_jacobi_blocks<<<a.count, 32 * jac::kBlock, jac::blocks_smem(a.ldw), s>>>(a.w, a.ldw, rows, cols, a.max_sweeps,
                                                                                 a.norms, a.err);
    return cudaGetLastError();
}

}  // namespace ptebd
