// The middle and first axes of the pair transform from the FP64 last axis (zdft64.cu), in FP64: the
// kernels of pair_split_ct.cuh on double2 columns.
//
// What bounds them: the FP64 pipe (two FMAs a clock and SM).  Hence the pruned last stages, and stages
// that skip the products with W^0: 1.18 us a pair on 48^3 (K2 = 15, N_G = 2000; 0.53 million FP64
// instructions, 0.9 us at the pipe's rate), 0.20 on 24^3.  With the last axis and the slices 1.83 and 0.40
// where the FFT pair kernel takes 6.7 and 1.09.
#pragma once
#include "pair_split_ct.cuh"
#include "fft.cuh"

namespace gw {

// lines fastest over the threads (LMap); stage 0 of make_prune_plan(N) from rows as a TMA box leaves them
template <int N>
__device__ __forceinline__ void dstage0_rows(const double2 *__restrict__ x, double2 *__restrict__ y, int half, int es,
                                             int nlines, int CS, LMap lm)
{
    constexpr int R = make_prune_plan(N).r[0], nb = N / R;
    int l = lm.l0, j = lm.j0;
    while (j < nb) {
        const int sl = l >= half ? 1 : 0;
        const double2 *xl = x + sl * N * es + (l - sl * half);
        double2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = xl[(j + r * nb) * es];
        dftR<R>(v);
        double2 *yl = y + l * CS + j * R;
#pragma unroll
        for (int r = 0; r < R; ++r) yl[r] = v[r];
        l += lm.dl;
        j += lm.dj;
        if (l >= nlines) {
            l -= nlines;
            ++j;
        }
    }
}

// stages S.. of make_prune_plan(N) but the pruned last, a barrier after each; returns the result buffer
template <int N, int S, int NS>
__device__ __forceinline__ double2 *dstages(double2 *x, double2 *y, int nlines, int CS, const double2 *tw, LMap lm)
{
    constexpr RadPlan P = make_prune_plan(N);
    if constexpr (S + 1 >= P.nst) {
        return x;
    } else {
        constexpr int R = P.r[S], nb = N / R, tstride = N / (NS * R);
        int l = lm.l0, j = lm.j0;
        while (j < nb) {
            const int kk = j % NS;
            const double2 *xl = x + l * CS;
            double2 v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = xl[j + r * nb];
            if (kk != 0) {
#pragma unroll
                for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[r * kk * tstride]);
            }
            dftR<R>(v);
            double2 *yl = y + l * CS + (j / NS) * (NS * R) + kk;
#pragma unroll
            for (int r = 0; r < R; ++r) yl[r * NS] = v[r];
            l += lm.dl;
            j += lm.dj;
            if (l >= nlines) {
                l -= nlines;
                ++j;
            }
        }
        __syncthreads();
        return dstages<N, S + 1, NS * R>(y, x, nlines, CS, tw, lm);
    }
}

// output k of the pruned last stage (tprune_ct)
template <int N>
__device__ __forceinline__ double2 dprune(const double2 *__restrict__ x, int k, const double2 *__restrict__ tw)
{
    constexpr int R = prune_radix(N), NS = N / R;
    const int j = k % NS;
    double2 acc = x[j];
    int e = 0;
#pragma unroll
    for (int r = 1; r < R; ++r) {
        e += k;
        if (e >= N) e -= N;
        cfma(acc, x[j + r * NS], tw[e]);
    }
    return acc;
}

template <int N>
__global__ void __launch_bounds__(kSplitThreads, split_min_blocks<N>())
    pair_split64_1_kernel(const __grid_constant__ CUtensorMap tmF, PairPlan pp, double2 *__restrict__ S)
{
    if (pp.guard && *pp.guard) return;
    constexpr int CS = N + 1;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ uint64_t fbar; // a slab pair's F has landed
    const int K2 = pp.K2, K12 = pp.K12, n0 = pp.n[0];
    const int ncols = 2 * K2, BUF = from_f_buf(ncols, CS), k2p = (K2 + 1) / 2 * 2;
    double2 *X = (double2 *)(((uintptr_t)smraw + 127) & ~(uintptr_t)127), *Y = X + BUF;
    double2 *tw = X + 2 * BUF;
    int *cell = (int *)(tw + N);
    for (int i = threadIdx.x; i < N; i += kSplitThreads) tw[i] = pp.ax[1].tw[i];
    for (int i = threadIdx.x; i < K12; i += kSplitThreads) cell[i] = pp.cell[i];
    if (threadIdx.x == 0) {
        bar_init(&fbar, 1);
        bar_fence_init();
    }
    __syncthreads();
    const int64_t row = blockIdx.x;
    const uint64_t stream = l2_policy_evict_first();
    auto fetch = [&](int i0, double2 *C) {
        if (threadIdx.x == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bar_expect(&fbar, (unsigned)(2 * N * K2 * 16));
            tma2_hint(C, &tmF, &fbar, (int)(row * k2p * 4), i0 * N, stream);
        }
    };
    const LMap lm = lmap_lines_fastest(ncols);
    fetch(0, X);
    uint32_t nf = 0;
    for (int i0 = 0; i0 < n0; i0 += 2, ++nf) {
        const bool late = !bar_wait(&fbar, nf & 1);
        if (__syncthreads_or(late)) { // X complete (or the wait ran out, for every thread alike)
            pair_give_up(&fbar, nf & 1, pp.status);
            return;
        }
        dstage0_rows<N>(X, Y, K2, K2, ncols, CS, lm);
        __syncthreads();
        double2 *y = dstages<N, 1, make_prune_plan(N).r[0]>(Y, X, ncols, CS, tw, lm);
        double2 *other = y == X ? Y : X; // free: its readers have passed a barrier
        if (i0 + 2 < n0) fetch(i0 + 2, other);
        const int cells = i0 + 1 < n0 ? 2 * K12 : K12;
        for (int d = threadIdx.x; d < cells; d += kSplitThreads) {
            const int sl = d >= K12, dd = d - sl * K12, cl = cell[dd];
            if (!GW_IN(cl >> 8, K2, pp.status)) continue;
            S[((int64_t)row * n0 + i0 + sl) * K12 + dd] = dprune<N>(y + (sl * K2 + (cl >> 8)) * CS, cl & 255, tw);
        }
        __syncthreads(); // y read before the next step writes it
        X = other;
        Y = y;
    }
}

template <int N>
__global__ void __launch_bounds__(kSplitThreads, split_min_blocks<N>())
    pair_split64_2_kernel(const __grid_constant__ CUtensorMap tmS, int cb, int64_t sv, int64_t sc, PairPlan pp,
                          double inv_nr, double2 *__restrict__ M)
{
    if (pp.guard && *pp.guard) return;
    constexpr int CS = N + 1;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ uint64_t fbar;
    const int K12 = pp.K12, NB = 2 * pp.K2, BUF = from_f_buf(NB, CS);
    double2 *X = (double2 *)(((uintptr_t)smraw + 127) & ~(uintptr_t)127), *Y = X + BUF;
    double2 *tw = X + 2 * BUF;
    for (int i = threadIdx.x; i < N; i += kSplitThreads) tw[i] = pp.ax[0].tw[i];
    if (threadIdx.x == 0) {
        bar_init(&fbar, 1);
        bar_fence_init();
    }
    __syncthreads();
    const int64_t row = blockIdx.x, vl = row / cb;
    const uint64_t stream = l2_policy_evict_first();
    auto fetch = [&](int d0, double2 *C) {
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
        const LMap lm = lmap_lines_fastest(nbat);
        dstage0_rows<N>(X, Y, nbat, NB, nbat, CS, lm);
        __syncthreads();
        double2 *y = dstages<N, 1, make_prune_plan(N).r[0]>(Y, X, nbat, CS, tw, lm);
        double2 *other = y == X ? Y : X;
        if (d0 + NB < K12) fetch(d0 + NB, other);
        const int m1 = pp.cstart[d0 + nbat];
        for (int m = pp.cstart[d0] + threadIdx.x; m < m1; m += kSplitThreads) {
            const int2 pt = pp.cpts[m];
            if (!GW_IN(pt.x, pp.ng, pp.status) || !GW_IN((pt.y >> 8) - d0, nbat, pp.status)) continue;
            const double2 f = dprune<N>(y + ((pt.y >> 8) - d0) * CS, pt.y & 255, tw);
            out[pt.x] = make_double2(f.x * inv_nr, f.y * inv_nr);
        }
        __syncthreads();
        X = other;
        Y = y;
    }
}

template <int N>
inline cudaError_t pair_split64_1(const CUtensorMap &tmF, int64_t R, const PairPlan &pp, double2 *S, cudaStream_t st)
{
    const size_t sm = pair_split_smem<N>(pp);
    cudaError_t e =
        cudaFuncSetAttribute(pair_split64_1_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    pair_split64_1_kernel<N><<<(unsigned)R, kSplitThreads, sm, st>>>(tmF, pp, S);
    return cudaGetLastError();
}

template <int N>
inline cudaError_t pair_split64_2(const CUtensorMap &tmS, int64_t R, int cb, int64_t sv, int64_t sc, const PairPlan &pp,
                                  double2 *M, cudaStream_t st)
{
    const size_t sm = pair_split_smem<N>(pp);
    cudaError_t e =
        cudaFuncSetAttribute(pair_split64_2_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const double inv = 1.0 / ((double)pp.n[0] * pp.n[1] * pp.n[2]);
    pair_split64_2_kernel<N><<<(unsigned)R, kSplitThreads, sm, st>>>(tmS, cb, sv, sc, pp, inv, M);
    return cudaGetLastError();
}

#define GW_PAIR_SPLIT64_DECL(N)                                                                                     \
    cudaError_t pair_split64_1_n##N(const CUtensorMap &tmF, int64_t R, const PairPlan &pp, double2 *S,               \
                                    cudaStream_t st);                                                              \
    cudaError_t pair_split64_2_n##N(const CUtensorMap &tmS, int64_t R, int cb, int64_t sv, int64_t sc,               \
                                    const PairPlan &pp, double2 *M, cudaStream_t st);
#define GW_PAIR_SPLIT64_DEF(N)                                                                                      \
    cudaError_t pair_split64_1_n##N(const CUtensorMap &tmF, int64_t R, const PairPlan &pp, double2 *S,               \
                                    cudaStream_t st)                                                               \
    {                                                                                                              \
        return pair_split64_1<N>(tmF, R, pp, S, st);                                                               \
    }                                                                                                              \
    cudaError_t pair_split64_2_n##N(const CUtensorMap &tmS, int64_t R, int cb, int64_t sv, int64_t sc,               \
                                    const PairPlan &pp, double2 *M, cudaStream_t st)                               \
    {                                                                                                              \
        return pair_split64_2<N>(tmS, R, cb, sv, sc, pp, M, st);                                                   \
    }

GW_PAIR_SPLIT_LENGTHS(GW_PAIR_SPLIT64_DECL)

} // namespace gw
