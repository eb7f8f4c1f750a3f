// The middle and first axes of the pair transform from the tensor-core last axis, for any pair of
// axis lengths: one kernel per middle-axis length N1 (a pair's slabs to the sphere's (k1, k2) cells)
// and one per first-axis length N0 (cells to sphere points), the cells [pair][n0][K12] in global
// memory between them.  Bound by issue like pair_kernel_tf_from_f, which runs both phases of the cubic
// 40^3 and 48^3 grids in one kernel with the cells in L2: 0.248 us a pair on 48^3 (K2 = 15) where these
// two take 2 % more.  72^3 (K2 = 23): 1.18 us a pair, and 3.1 with the last axis and its slices, where the
// FFT pair kernel takes 5.1; 30 x 36 x 40: 0.15, and 0.41, where the runtime-shape kernel takes 1.26.
#pragma once
#include "pair_tf_ct.cuh"

namespace gw {

constexpr int kSplitThreads = 192;
// resident blocks the register budget is sized for: 4 (80 a thread) for radix 3 and 4 stages, 3 with
// radix 5 or 8, 2 where two slab pairs of columns fill half the shared memory
template <int N>
constexpr int split_min_blocks()
{
    return N > 60 ? 2 : (N % 5 == 0 || N % 24 == 0) && N != 48 ? 3 : 4;
}

// Slab pairs of one pair of bands: F of two slabs by one TMA load (lines past the grid read as zero),
// i1 transformed in lazy two-float stages, the pruned last stage straight into S[row][i0][cell].
template <int N>
__global__ void __launch_bounds__(kSplitThreads, split_min_blocks<N>())
    pair_split1_kernel(const __grid_constant__ CUtensorMap tmF, PairPlan pp, TfConsts kc, float4 *__restrict__ S)
{
    constexpr int CS = N + 1;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ uint64_t fbar; // a slab pair's F has landed
    const int K2 = pp.K2, K12 = pp.K12, n0 = pp.n[0];
    const int ncols = 2 * K2, BUF = from_f_buf(ncols, CS), k2p = (K2 + 1) / 2 * 2;
    float4 *X = (float4 *)(((uintptr_t)smraw + 127) & ~(uintptr_t)127), *Y = X + BUF;
    float4 *tw = X + 2 * BUF;
    int *cell = (int *)(tw + N);
    for (int i = threadIdx.x; i < N; i += kSplitThreads) tw[i] = pp.ax[1].twf[i];
    for (int i = threadIdx.x; i < K12; i += kSplitThreads) cell[i] = pp.cell[i];
    if (threadIdx.x == 0) {
        bar_init(&fbar, 1);
        bar_fence_init();
    }
    __syncthreads();
    const int64_t row = blockIdx.x;
    const uint64_t stream = l2_policy_evict_first();
    auto fetch = [&](int i0, float4 *C) {
        if (threadIdx.x == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bar_expect(&fbar, (unsigned)(2 * N * K2 * 16));
            tma2_hint(C, &tmF, &fbar, (int)(row * k2p * 4), i0 * N, stream);
        }
    };
    const LMap lm = lmap_lines(ncols);
    fetch(0, X);
    uint32_t nf = 0;
    for (int i0 = 0; i0 < n0; i0 += 2, ++nf) {
        const bool late = !bar_wait(&fbar, nf & 1);
        if (__syncthreads_or(late)) { // X complete (or the wait ran out, for every thread alike)
            pair_give_up(&fbar, nf & 1, pp.status);
            return;
        }
        tstage0_rows<N>(X, Y, K2, K2, ncols, CS, lm, kc);
        __syncthreads();
        float4 *y = tstages_ct<N, 1, make_prune_plan(N).r[0], true, true>(Y, X, ncols, CS, tw, kc, 1, -1, lm);
        float4 *other = y == X ? Y : X; // free: its readers have passed a barrier
        if (i0 + 2 < n0) fetch(i0 + 2, other);
        const int cells = i0 + 1 < n0 ? 2 * K12 : K12;
        for (int d = threadIdx.x; d < cells; d += kSplitThreads) {
            const int sl = d >= K12, dd = d - sl * K12, cl = cell[dd];
            if (!GW_IN(cl >> 8, K2, pp.status)) continue;
            const tcx c = tprune_ct<N>(y + (sl * K2 + (cl >> 8)) * CS, cl & 255, tw);
            S[((int64_t)row * n0 + i0 + sl) * K12 + dd] = make_float4(c.re.hi, c.re.lo, c.im.hi, c.im.lo);
        }
        __syncthreads(); // y read before the next step writes it
        X = other;
        Y = y;
    }
}

// Batches of 2 K2 cells of one pair: all N slabs of a batch by one TMA load (cells past K12 read as
// zero), i0 transformed, the pruned last stage straight into M.
template <int N>
__global__ void __launch_bounds__(kSplitThreads, split_min_blocks<N>())
    pair_split2_kernel(const __grid_constant__ CUtensorMap tmS, int cb, int64_t sv, int64_t sc, PairPlan pp, TfConsts kc,
                       tf inv_nr, double2 *__restrict__ M)
{
    constexpr int CS = N + 1;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ uint64_t fbar;
    const int K12 = pp.K12, NB = 2 * pp.K2, BUF = from_f_buf(NB, CS);
    float4 *X = (float4 *)(((uintptr_t)smraw + 127) & ~(uintptr_t)127), *Y = X + BUF;
    float4 *tw = X + 2 * BUF;
    for (int i = threadIdx.x; i < N; i += kSplitThreads) tw[i] = pp.ax[0].twf[i];
    if (threadIdx.x == 0) {
        bar_init(&fbar, 1);
        bar_fence_init();
    }
    __syncthreads();
    const int64_t row = blockIdx.x, vl = row / cb;
    const uint64_t stream = l2_policy_evict_first();
    auto fetch = [&](int d0, float4 *C) {
        if (threadIdx.x == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bar_expect(&fbar, (unsigned)(N * NB * 16));
            tma2_hint(C, &tmS, &fbar, d0 * 4, (int)(row * N), stream);
        }
    };
    double2 *out = M + (vl * sv + (row - vl * cb) * sc) * pp.ng;
    fetch(0, X);
    uint32_t nf = 0;
    for (int d0 = 0; d0 < K12; d0 += NB, ++nf) {
        const int nbat = K12 - d0 < NB ? K12 - d0 : NB;
        const bool late = !bar_wait(&fbar, nf & 1);
        if (__syncthreads_or(late)) {
            pair_give_up(&fbar, nf & 1, pp.status);
            return;
        }
        const LMap lm = lmap_lines(nbat);
        tstage0_rows<N>(X, Y, nbat, NB, nbat, CS, lm, kc);
        __syncthreads();
        float4 *y = tstages_ct<N, 1, make_prune_plan(N).r[0], true, true>(Y, X, nbat, CS, tw, kc, 1, -1, lm);
        float4 *other = y == X ? Y : X;
        if (d0 + NB < K12) fetch(d0 + NB, other);
        const int m1 = pp.cstart[d0 + nbat];
        for (int m = pp.cstart[d0] + threadIdx.x; m < m1; m += kSplitThreads) {
            const int2 pt = pp.cpts[m];
            if (!GW_IN(pt.x, pp.ng, pp.status) || !GW_IN((pt.y >> 8) - d0, nbat, pp.status)) continue;
            const tcx f = tprune_ct<N>(y + ((pt.y >> 8) - d0) * CS, pt.y & 255, tw);
            out[pt.x] = make_double2(tf_to_d(tf_mul(f.re, inv_nr)), tf_to_d(tf_mul(f.im, inv_nr)));
        }
        __syncthreads();
        X = other;
        Y = y;
    }
}

template <int N>
inline size_t pair_split_smem(const PairPlan &pp)
{
    return 128 + sizeof(float4) * (2 * (size_t)from_f_buf(2 * pp.K2, N + 1) + N) + sizeof(int) * (size_t)pp.K12;
}

template <int N>
inline cudaError_t pair_split1(const CUtensorMap &tmF, int64_t R, const PairPlan &pp, const TfConsts &kc, float4 *S,
                               cudaStream_t st)
{
    const size_t sm = pair_split_smem<N>(pp);
    cudaError_t e = cudaFuncSetAttribute(pair_split1_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    pair_split1_kernel<N><<<(unsigned)R, kSplitThreads, sm, st>>>(tmF, pp, kc, S);
    return cudaGetLastError();
}

template <int N>
inline cudaError_t pair_split2(const CUtensorMap &tmS, int64_t R, int cb, int64_t sv, int64_t sc, const PairPlan &pp,
                               const TfConsts &kc, tf inv_nr, double2 *M, cudaStream_t st)
{
    const size_t sm = pair_split_smem<N>(pp);
    cudaError_t e = cudaFuncSetAttribute(pair_split2_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    pair_split2_kernel<N><<<(unsigned)R, kSplitThreads, sm, st>>>(tmS, cb, sv, sc, pp, kc, inv_nr, M);
    return cudaGetLastError();
}

// one pair of launchers per length, instantiated in pair_split_*.cu
#define GW_PAIR_SPLIT_DECL(N)                                                                                      \
    cudaError_t pair_split1_n##N(const CUtensorMap &tmF, int64_t R, const PairPlan &pp, const TfConsts &kc,         \
                                 float4 *S, cudaStream_t st);                                                      \
    cudaError_t pair_split2_n##N(const CUtensorMap &tmS, int64_t R, int cb, int64_t sv, int64_t sc,                 \
                                 const PairPlan &pp, const TfConsts &kc, tf inv_nr, double2 *M, cudaStream_t st);
#define GW_PAIR_SPLIT_DEF(N)                                                                                       \
    cudaError_t pair_split1_n##N(const CUtensorMap &tmF, int64_t R, const PairPlan &pp, const TfConsts &kc,         \
                                 float4 *S, cudaStream_t st)                                                       \
    {                                                                                                              \
        return pair_split1<N>(tmF, R, pp, kc, S, st);                                                              \
    }                                                                                                              \
    cudaError_t pair_split2_n##N(const CUtensorMap &tmS, int64_t R, int cb, int64_t sv, int64_t sc,                 \
                                 const PairPlan &pp, const TfConsts &kc, tf inv_nr, double2 *M, cudaStream_t st)   \
    {                                                                                                              \
        return pair_split2<N>(tmS, R, cb, sv, sc, pp, kc, inv_nr, M, st);                                          \
    }
// the lengths, 2^a 3^b 5^c from 20 to 72 that plane-wave grids use
#define GW_PAIR_SPLIT_LENGTHS(X) \
    X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64) X(72)

GW_PAIR_SPLIT_LENGTHS(GW_PAIR_SPLIT_DECL)

} // namespace gw
