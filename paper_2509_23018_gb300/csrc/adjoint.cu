// Adjoint of L = Re Tr(W chi0) with respect to band energies and plane-wave coefficients.
//
// With m_p = M[p][:] (a row) and a Hermitian W, L = sum_p Delta_p q_p where
// q_p = sum_{G,G'} m_p(G) W[G][G'] conj(m_p(G')) (real).  Wirtinger calculus gives
//   dL/dDelta_p       = q_p = Re sum_G' Y_p(G') conj(m_p(G')),   Y = M W
//   dL/dconj(m_p(G')) = g_p(G') = Delta_p Y_p(G')
// and, through M_vc(G) = (1/N_r) sum_r conj(psi_v(r)) psi_c(r) e^{+iG.r},
//   dL/dconj(psi_c(r)) = psi_v(r) h_p(r),  dL/dconj(psi_v(r)) = psi_c(r) conj(h_p(r)),
//   h_p(r) = (1/N_r) sum_G g_p(G) e^{-iG.r},
// and through psi_n(r) = sum_K c_n(K) e^{+iK.r},
//   dL/dconj(c_n(K)) = sum_r psibar_n(r) e^{-iK.r}.
// Gradients are reported as dL/dRe + i dL/dIm = 2 dL/dconj.  Energies enter through
// x = E_v - E_c and dDelta/dx = 4 (w^2 - x^2) / (x^2 + w^2)^2.
// (GWPT's derivative of the self-energy, Eq. gwpt, is what motivates this sensitivity.)
#include "internal.h"
#include "fft.cuh"
#include "fft_tf.cuh"

#include <algorithm>

namespace gw {

// ------------------------------------------------------------------ Y = M W (FP64 DMMA)
// C[m][n] = sum_k A[m][k] B[k][n], complex row-major A [mr x kd], B [kd x nc], C [mr x nc].
constexpr int kGT = 64, kGK = 16;

__device__ __forceinline__ void dmma8(double &d0, double &d1, double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                 : "+d"(d0), "+d"(d1)
                 : "d"(a), "d"(b));
}

// CA: conj(A) in place of A.  TB: B given as its transpose, row-major [nc][kd].  ACC: C += A B.
template <bool CA, bool TB, bool ACC>
__global__ void __launch_bounds__(256) zgemm_kernel(const double2 *__restrict__ A, const double2 *__restrict__ B,
                                                    double2 *__restrict__ C, int64_t mr, int kd, int nc)
{
    __shared__ double2 sa[kGT][kGK + 1];   // [m][k]
    __shared__ double2 sb[kGK][kGT + 1];   // [k][n]
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int wm = wid & 1, wn = wid >> 1;
    const int64_t m0 = (int64_t)blockIdx.y * kGT;
    const int n0 = blockIdx.x * kGT;
    double cre[4][2][2] = {}, cim[4][2][2] = {};
    for (int k0 = 0; k0 < kd; k0 += kGK) {
        for (int e = tid; e < kGT * kGK; e += blockDim.x) {
            int r = e / kGK, k = e % kGK;
            int64_t gm = m0 + r;
            int gk = k0 + k;
            double2 x = (gm < mr && gk < kd) ? A[gm * kd + gk] : make_double2(0.0, 0.0);
            if (CA) x.y = -x.y;
            sa[r][k] = x;
        }
        for (int e = tid; e < kGK * kGT; e += blockDim.x) {
            if (TB) {
                int n = e / kGK, k = e % kGK;
                int gk = k0 + k, gn = n0 + n;
                sb[k][n] = (gk < kd && gn < nc) ? B[(int64_t)gn * kd + gk] : make_double2(0.0, 0.0);
            } else {
                int k = e / kGT, n = e % kGT;
                int gk = k0 + k, gn = n0 + n;
                sb[k][n] = (gk < kd && gn < nc) ? B[(int64_t)gk * nc + gn] : make_double2(0.0, 0.0);
            }
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kGK / 4; ++kk) {
            const int k = kk * 4 + (lane & 3);
            double ar[4], ai[4], nai[4], br[2], bi[2];
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                double2 x = sa[wm * 32 + mt * 8 + (lane >> 2)][k];
                ar[mt] = x.x;
                ai[mt] = x.y;
                nai[mt] = -x.y;
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                double2 x = sb[k][wn * 16 + nt * 8 + (lane >> 2)];
                br[nt] = x.x;
                bi[nt] = x.y;
            }
#pragma unroll
            for (int mt = 0; mt < 4; ++mt)
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    // (ar + i ai)(br + i bi) = (ar br - ai bi) + i (ar bi + ai br)
                    dmma8(cre[mt][nt][0], cre[mt][nt][1], ar[mt], br[nt]);
                    dmma8(cre[mt][nt][0], cre[mt][nt][1], nai[mt], bi[nt]);
                    dmma8(cim[mt][nt][0], cim[mt][nt][1], ar[mt], bi[nt]);
                    dmma8(cim[mt][nt][0], cim[mt][nt][1], ai[mt], br[nt]);
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int mt = 0; mt < 4; ++mt) {
        const int64_t gm = m0 + wm * 32 + mt * 8 + (lane >> 2);
        if (gm >= mr) continue;
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int gn = n0 + wn * 16 + nt * 8 + 2 * (lane & 3) + q;
                if (gn < nc) {
                    double2 v = make_double2(cre[mt][nt][q], cim[mt][nt][q]);
                    if (ACC) {
                        const double2 o = C[gm * nc + gn];
                        v.x += o.x;
                        v.y += o.y;
                    }
                    C[gm * nc + gn] = v;
                }
            }
    }
}

cudaError_t launch_zgemm(const double2 *A, const double2 *B, double2 *C, int64_t mr, int kd, int nc, cudaStream_t st)
{
    if (mr == 0 || nc == 0) return cudaSuccess;
    dim3 grid((nc + kGT - 1) / kGT, (unsigned)((mr + kGT - 1) / kGT));
    zgemm_kernel<false, false, false><<<grid, 256, 0, st>>>(A, B, C, mr, kd, nc);
    return cudaGetLastError();
}

cudaError_t launch_zgemm_ex(const double2 *A, const double2 *B, double2 *C, int64_t mr, int kd, int nc, bool conj_a,
                            bool trans_b, bool accumulate, cudaStream_t st)
{
    if (mr == 0 || nc == 0) return cudaSuccess;
    dim3 grid((nc + kGT - 1) / kGT, (unsigned)((mr + kGT - 1) / kGT));
    if (conj_a && !trans_b && !accumulate) zgemm_kernel<true, false, false><<<grid, 256, 0, st>>>(A, B, C, mr, kd, nc);
    else if (!conj_a && trans_b && accumulate) zgemm_kernel<false, true, true><<<grid, 256, 0, st>>>(A, B, C, mr, kd, nc);
    else if (!conj_a && !trans_b && !accumulate) zgemm_kernel<false, false, false><<<grid, 256, 0, st>>>(A, B, C, mr, kd, nc);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

// ------------------------------------------------------------------ per-pair reductions
// One warp per pair: q_p = Re sum_G Y conj(M); g_p = Delta_p Y_p written over Y;
// L, dE_v, dE_c accumulated with atomics.
__global__ void adj_rows_kernel(const double2 *__restrict__ M, double2 *__restrict__ Y, int64_t P, int ng, int nc,
                                int64_t p0, const double *__restrict__ ev, const double *__restrict__ ec, double w,
                                double *__restrict__ Lacc, double *__restrict__ dEv, double *__restrict__ dEc)
{
    const int lane = threadIdx.x & 31;
    const int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (p >= P) return;
    const double2 *m = M + p * ng;
    double2 *y = Y + p * ng;
    double q = 0.0;
    for (int g = lane; g < ng; g += 32) {
        double2 a = y[g], b = m[g];
        q = fma(a.x, b.x, fma(a.y, b.y, q));
    }
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    const int64_t pg = p0 + p;
    const int v = (int)(pg / nc), c = (int)(pg - (int64_t)v * nc);
    const double x = ev[v] - ec[c];
    const double den = fma(x, x, w * w);
    const double dl = 4.0 * x / den;
    const double dd = 4.0 * (w * w - x * x) / (den * den);
    for (int g = lane; g < ng; g += 32) {
        double2 a = y[g];
        y[g] = make_double2(dl * a.x, dl * a.y);
    }
    if (lane == 0) {
        atomicAdd(Lacc, dl * q);
        atomicAdd(dEv + v, q * dd);
        atomicAdd(dEc + c, -q * dd);
    }
}

cudaError_t launch_adj_rows(const double2 *M, double2 *Y, int64_t P, int ng, int nc, int64_t p0, const double *ev,
                            const double *ec, double w, double *L, double *dEv, double *dEc, cudaStream_t st)
{
    if (P == 0) return cudaSuccess;
    adj_rows_kernel<<<(unsigned)((P + 7) / 8), 256, 0, st>>>(M, Y, P, ng, nc, p0, ev, ec, w, L, dEv, dEc);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ back-projection of g_p onto the grid
// h_p(r) = (1/N_r) sum_G g_p(G) e^{-iG.r} = conj( (1/N_r) sum_G conj(g_p(G)) e^{+iG.r} ).
// One block per pair; per i0 slab: the sphere values of each kept (k1, k2) cell are summed
// with e^{+2 pi i k0 i0/n0} (conjugated input), zero-padded columns are transformed along
// i1, zero-padded lines along i2, and the conjugated slab is written to H.
template <bool TF>
__global__ void __launch_bounds__(256) adj_pair_kernel(const double2 *__restrict__ Gb, int64_t P, PairPlan pp,
                                                       const int *__restrict__ cell_start,
                                                       const int *__restrict__ cell_g, int ncell,
                                                       double2 *__restrict__ H)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int n0 = pp.n[0], n1 = pp.n[1], n2 = pp.n[2];
    const int ns = n1 * n2;
    double2 *a = (double2 *)smem, *b = a + ns;
    double2 *tw0 = b + ns, *tw1 = tw0 + n0, *tw2 = tw1 + n1;
    double2 *gs = tw2 + n2;                       // [ng] conj(g_p)
    int *kz = (int *)(gs + pp.ng);
    for (int i = threadIdx.x; i < n0; i += blockDim.x) tw0[i] = pp.ax[0].tw[i];
    for (int i = threadIdx.x; i < n1; i += blockDim.x) tw1[i] = pp.ax[1].tw[i];
    for (int i = threadIdx.x; i < n2; i += blockDim.x) tw2[i] = pp.ax[2].tw[i];
    for (int i = threadIdx.x; i < pp.K2; i += blockDim.x) kz[i] = pp.kz[i];
    const int64_t p = blockIdx.x;
    for (int g = threadIdx.x; g < pp.ng; g += blockDim.x) {
        double2 x = Gb[p * pp.ng + g];
        gs[g] = make_double2(x.x, -x.y);
    }
    __syncthreads();
    const double sc = 1.0 / ((double)n0 * ns);
    double2 *out = H + p * (int64_t)n0 * ns;
    for (int i0 = 0; i0 < n0; ++i0) {
        // kept columns k2' (K2 of them), each a zero-padded line of n1 values
        for (int i = threadIdx.x; i < pp.K2 * n1; i += blockDim.x) a[i] = make_double2(0.0, 0.0);
        __syncthreads();
        for (int cidx = threadIdx.x; cidx < ncell; cidx += blockDim.x) {
            double2 acc = make_double2(0.0, 0.0);
            int cell_pos = 0;
            for (int t = cell_start[cidx]; t < cell_start[cidx + 1]; ++t) {
                const int g = cell_g[t];
                const int pk = pp.gpack[g];
                const int k0 = pk & 255;
                cell_pos = (pk >> 16) * n1 + ((pk >> 8) & 255);
                cfma(acc, tw0[(k0 * i0) % n0], gs[g]);
            }
            a[cell_pos] = acc;
        }
        __syncthreads();
        double2 *r = fft_lines(a, b, pp.K2, n1, 1, pp.ax[1], tw1); // along i1, K2 lines
        double2 *o = (r == a) ? b : a;
        // scatter the K2 columns into full i2 lines: o[i1][i2]
        for (int i = threadIdx.x; i < ns; i += blockDim.x) o[i] = make_double2(0.0, 0.0);
        __syncthreads();
        for (int i = threadIdx.x; i < pp.K2 * n1; i += blockDim.x) {
            int q = i / n1, i1 = i - q * n1;
            o[i1 * n2 + kz[q]] = r[i];
        }
        __syncthreads();
        double2 *t = fft_lines(o, r, n1, n2, 1, pp.ax[2], tw2); // along i2
        for (int i = threadIdx.x; i < ns; i += blockDim.x) {
            double2 z = t[i];
            out[(int64_t)i0 * ns + i] = make_double2(z.x * sc, -z.y * sc);
        }
        __syncthreads();
    }
}

// The same back-projection in two-float arithmetic on the FP32 pipes (bands held in two-float
// form): conj(g_p) converted once per pair, in place over the block's own row of Gb (16 bytes
// an entry either way; Gb is not read again), the i0 sums per cell reading it from L2, both line
// transforms in hi + lo pairs; H is written in two-float form.  Keeping conj(g_p) out of shared
// memory lets four blocks run per SM on 40^3 instead of two.
// Any grid, runtime plans; the cubic grids below take adj_cells_tf_kernel and adj_slab_tf_kernel.
__global__ void __launch_bounds__(256) adj_pair_tf_kernel(double2 *__restrict__ Gb, PairPlan pp,
                                                          const int *__restrict__ cell_start,
                                                          const int *__restrict__ cell_g, int ncell, TfConsts kc,
                                                          tf sc, float4 *__restrict__ H)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int n0 = pp.n[0], n1 = pp.n[1], n2 = pp.n[2];
    const int ns = n1 * n2;
    float4 *a = (float4 *)smem, *b = a + ns;
    float4 *tw0 = b + ns, *tw1 = tw0 + n0, *tw2 = tw1 + n1;
    int *kz = (int *)(tw2 + n2);
    for (int i = threadIdx.x; i < n0; i += blockDim.x) tw0[i] = pp.ax[0].twf[i];
    for (int i = threadIdx.x; i < n1; i += blockDim.x) tw1[i] = pp.ax[1].twf[i];
    for (int i = threadIdx.x; i < n2; i += blockDim.x) tw2[i] = pp.ax[2].twf[i];
    for (int i = threadIdx.x; i < pp.K2; i += blockDim.x) kz[i] = pp.kz[i];
    const int64_t p = blockIdx.x;
    float4 *gs = (float4 *)(Gb + p * pp.ng); // [ng] conj(g_p), two-float, over the row
    for (int g = threadIdx.x; g < pp.ng; g += blockDim.x) {
        const double2 x = Gb[p * pp.ng + g];
        const tf re = tf_from(x.x), im = tf_from(-x.y);
        gs[g] = make_float4(re.hi, re.lo, im.hi, im.lo);
    }
    __syncthreads();
    float4 *out = H + p * (int64_t)n0 * ns;
    for (int i0 = 0; i0 < n0; ++i0) {
        for (int i = threadIdx.x; i < pp.K2 * n1; i += blockDim.x) a[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        for (int cidx = threadIdx.x; cidx < ncell; cidx += blockDim.x) {
            tcx acc{{0.f, 0.f}, {0.f, 0.f}};
            int cell_pos = 0;
            for (int t = cell_start[cidx]; t < cell_start[cidx + 1]; ++t) {
                const int g = cell_g[t];
                const int pk = pp.gpack[g];
                const int k0 = pk & 255;
                cell_pos = (pk >> 16) * n1 + ((pk >> 8) & 255);
                acc = tc_add(acc, tc_mul(tc_load(gs + g), tc_load(tw0 + (k0 * i0) % n0)));
            }
            tc_store(a + cell_pos, acc);
        }
        __syncthreads();
        float4 *r = tfft_lines(a, b, pp.K2, n1, 1, pp.ax[1], tw1, kc); // along i1, K2 lines
        float4 *o = (r == a) ? b : a;
        for (int i = threadIdx.x; i < ns; i += blockDim.x) o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        for (int i = threadIdx.x; i < pp.K2 * n1; i += blockDim.x) {
            const int q = i / n1, i1 = i - q * n1;
            o[i1 * n2 + kz[q]] = r[i];
        }
        __syncthreads();
        const float4 *t = tfft_lines(o, r, n1, n2, 1, pp.ax[2], tw2, kc); // along i2
        for (int i = threadIdx.x; i < ns; i += blockDim.x) {
            const tcx z = tc_load(t + i);
            tc_store(out + (int64_t)i0 * ns + i, tcx{tf_mul(z.re, sc), tf_neg(tf_mul(z.im, sc))});
        }
        __syncthreads();
    }
}

// The back-projection on a cubic N^3 grid in two kernels, the transforms of the pair elements from F
// (pair_split_ct.cuh) turned around: the sphere's points along i0, (k1, k2) cell by cell, then slab by
// slab the K2 columns along i1 and all N lines along i2.
//
// What bounds them: issue on the FP32 pipes, about 10 million two-float operations a pair on 40^3, most
// of them along i2.  The cells' i0 transform is an FFT (a direct sum over the sphere for every slab costs as
// much as the lines along i2), lines run fastest over the threads at an odd stride, and the first stage
// of i1 and of i2 reads its inputs where they are, zeros never stored.  The cells pass through the
// end of the pair's own H: S row i0 lies behind every slab up to i0 - 1.
// 40^3, N_G = 1500: 0.67 us a pair, 0.09 of it the cells, where the runtime-shape kernel's scheme with
// compile-time lines took 1.29.
constexpr int kAdjBatch = 32; // cells per batch
template <int N>
__global__ void __launch_bounds__(192, N <= 48 ? 4 : 2)
    adj_cells_tf_kernel(const double2 *__restrict__ Gb, PairPlan pp, TfConsts kc, tf sc, float4 *__restrict__ H)
{
    constexpr int CS = N + 1;
    extern __shared__ __align__(16) unsigned char smem[];
    float4 *X = (float4 *)smem, *Y = X + kAdjBatch * CS, *tw = Y + kAdjBatch * CS;
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = pp.ax[0].twf[i];
    const int64_t p = blockIdx.x, nr = (int64_t)N * N * N;
    const int K12 = pp.K12;
    float4 *S = H + (p + 1) * nr - (int64_t)N * K12;
    const double2 *g = Gb + p * pp.ng;
    for (int d0 = 0; d0 < K12; d0 += kAdjBatch) {
        const int nbat = min(kAdjBatch, K12 - d0);
        for (int i = threadIdx.x; i < nbat * CS; i += blockDim.x) X[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        const int m1 = pp.cstart[d0 + nbat];
        for (int m = pp.cstart[d0] + threadIdx.x; m < m1; m += blockDim.x) {
            const int2 pt = pp.cpts[m];
            if (!GW_IN(pt.x, pp.ng, pp.status) || !GW_IN((pt.y >> 8) - d0, nbat, pp.status)) continue;
            const double2 x = g[pt.x]; // conj(g_p) / N_r
            tc_store(X + ((pt.y >> 8) - d0) * CS + (pt.y & 255), tcx{tf_mul(tf_from(x.x), sc), tf_mul(tf_from(-x.y), sc)});
        }
        __syncthreads();
        const float4 *r = tfft_lines_ct<N, true>(X, Y, nbat, CS, tw, kc);
        for (int e = threadIdx.x; e < nbat * N; e += blockDim.x) {
            const int i0 = e / nbat, d = e - i0 * nbat;
            S[(int64_t)i0 * K12 + d0 + d] = r[d * CS + i0];
        }
        __syncthreads();
    }
}

// 5-point transform of inputs 0 and 4 alone (v[1..3] zero)
__device__ __forceinline__ void adj_dft5_ends(tcx *v, const TfConsts &k)
{
    const tcx a = v[0], b = v[4];
    const tcx t1 = tc_addl(a, tc_rmul(b, k.c1)), u1 = tc_muli(tc_rmul(b, k.s1));
    const tcx t2 = tc_addl(a, tc_rmul(b, k.c2)), u2 = tc_muli(tc_rmul(b, k.s2));
    v[0] = tc_norm(tc_addl(a, b));
    v[1] = tc_norm(tc_subl(t1, u1)); // W_5^{4 k} = conj(W_5^k)
    v[4] = tc_norm(tc_addl(t1, u1));
    v[2] = tc_norm(tc_subl(t2, u2));
    v[3] = tc_norm(tc_addl(t2, u2));
}

// First stage of make_rad_plan(N) with inputs ld(line, point, present); lines fastest over the threads.
// The kept frequencies lie around 0, so that a 5-point transform mostly has its first and last input.
template <int N, class LD>
__device__ __forceinline__ void adj_stage0(LD ld, float4 *__restrict__ y, int nlines, int CS, LMap lm, const TfConsts &kc)
{
    constexpr int R = make_rad_plan(N).r[0], nb = N / R;
    int l = lm.l0, j = lm.j0;
    while (j < nb) {
        tcx v[R];
        bool in[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = ld(l, j + r * nb, in[r]);
        bool inner = R != 5;
#pragma unroll
        for (int r = 1; r + 1 < R; ++r) inner = inner || in[r];
        if (inner) tdftR<R>(v, kc);
        else if constexpr (R == 5) adj_dft5_ends(v, kc);
        float4 *yl = y + l * CS + j * R;
#pragma unroll
        for (int r = 0; r < R; ++r) tc_store(yl + r, v[r]);
        l += lm.dl;
        j += lm.dj;
        if (l >= nlines) {
            l -= nlines;
            ++j;
        }
    }
}

template <int N>
constexpr int adj_slab_threads()
{
    return N <= 24 ? 128 : N <= 40 ? 256 : N <= 48 ? 320 : 512;
}
template <int N>
__global__ void __launch_bounds__(adj_slab_threads<N>(), N <= 40 ? 3 : N <= 48 ? 2 : 1)
    adj_slab_tf_kernel(PairPlan pp, TfConsts kc, float4 *__restrict__ H)
{
    constexpr int CS = N + 1, ns = N * N, R0 = make_rad_plan(N).r[0];
    extern __shared__ __align__(16) unsigned char smem[];
    const int K2 = pp.K2, K12 = pp.K12;
    float4 *Z1 = (float4 *)smem, *Z2 = Z1 + N * CS, *tw = Z2 + N * CS, *srow = tw + N; // [2][K12]
    short *cm = (short *)(srow + 2 * K12), *qinv = cm + K2 * N; // cell at (k1, q), column of i2 (or -1)
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        tw[i] = pp.ax[0].twf[i];
        qinv[i] = -1;
    }
    for (int i = threadIdx.x; i < K2 * N; i += blockDim.x) cm[i] = -1;
    __syncthreads();
    for (int q = threadIdx.x; q < K2; q += blockDim.x) qinv[pp.kz[q]] = (short)q;
    for (int d = threadIdx.x; d < K12; d += blockDim.x) {
        const int cl = pp.cell[d];
        if (GW_IN(cl >> 8, K2, pp.status)) cm[(cl & 255) * K2 + (cl >> 8)] = (short)d;
    }
    const int64_t p = blockIdx.x, nr = (int64_t)N * ns;
    float4 *out = H + p * nr;
    const float4 *S = out + nr - (int64_t)N * K12;
    auto fetch = [&](int i0) {
        for (int d = threadIdx.x; d < K12; d += blockDim.x)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(srow + (i0 & 1) * K12 + d)),
                         "l"(S + (int64_t)i0 * K12 + d)
                         : "memory");
    };
    fetch(0);
    const LMap lm1 = lmap_lines_fastest(K2), lm2 = lmap_lines_fastest(N);
    const tcx zero{{0.f, 0.f}, {0.f, 0.f}};
    for (int i0 = 0; i0 < N; ++i0) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads(); // row i0 is here, and the slab before is written
        if (i0 + 1 < N) fetch(i0 + 1);
        const float4 *sr = srow + (i0 & 1) * K12;
        float4 *Y1 = Z2, *Y2 = Z2 + K2 * CS; // the K2 columns, K2 <= N / 2
        adj_stage0<N>(
            [&](int q, int k1, bool &in) {
                const int d = cm[k1 * K2 + q];
                in = d >= 0;
                return in ? tc_load(sr + d) : zero;
            },
            Y1, K2, CS, lm1, kc);
        __syncthreads();
        const float4 *r = tstages_ct<N, 1, R0, false, true>(Y1, Y2, K2, CS, tw, kc, 1, -1, lm1);
        adj_stage0<N>(
            [&](int i1, int i2, bool &in) {
                const int q = qinv[i2];
                in = q >= 0;
                return in ? tc_load(r + q * CS + i1) : zero;
            },
            Z1, N, CS, lm2, kc);
        __syncthreads();
        const float4 *t = tstages_ct<N, 1, R0, false, true>(Z1, Z2, N, CS, tw, kc, 1, -1, lm2);
        for (int i = threadIdx.x; i < ns; i += blockDim.x) {
            const float4 z = t[i / N * CS + i % N];
            out[(int64_t)i0 * ns + i] = make_float4(z.x, z.y, -z.z, -z.w);
        }
    }
}

static size_t adj_slab_smem(const PairPlan &pp)
{
    const size_t n = pp.n[0];
    return sizeof(float4) * (2 * n * (n + 1) + n + 2 * (size_t)pp.K12) + sizeof(short) * (pp.K2 * n + n);
}

// The spheres that the two kernels take: the columns of i1 lie in one of the two buffers of i2, and two rows of
// cells beside them fit a block's shared memory (always on 24^3 to 48^3, up to about 1800 cells on 72^3).
static bool adj_cube_supported(const PairPlan &pp)
{
    const int n = pp.n[0];
    return n == pp.n[1] && n == pp.n[2] && (n == 24 || n == 40 || n == 48 || n == 72) && 2 * pp.K2 <= n &&
           adj_slab_smem(pp) <= (size_t)227 * 1024;
}

template <int N>
static cudaError_t launch_adj_cube(const double2 *Gb, int64_t P, const PairPlan &pp, tf sc, float4 *H, cudaStream_t st)
{
    const size_t sm1 = sizeof(float4) * (2 * (size_t)kAdjBatch * (N + 1) + N);
    const size_t sm2 = adj_slab_smem(pp);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(adj_cells_tf_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm1)) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(adj_slab_tf_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm2)) !=
            cudaSuccess)
        return e;
    adj_cells_tf_kernel<N><<<(unsigned)P, 192, sm1, st>>>(Gb, pp, tf_consts(), sc, H);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    adj_slab_tf_kernel<N><<<(unsigned)P, adj_slab_threads<N>(), sm2, st>>>(pp, tf_consts(), H);
    return cudaGetLastError();
}

cudaError_t launch_adj_pair(double2 *Gb, int64_t P, const PairPlan &pp, const int *cell_start,
                            const int *cell_g, int ncell, double2 *H, bool twofloat, cudaStream_t st)
{
    if (P == 0) return cudaSuccess;
    if (twofloat) {
        const size_t sm = sizeof(float4) * (2 * (size_t)pp.n[1] * pp.n[2] + pp.n[0] + pp.n[1] + pp.n[2]) +
                          sizeof(int) * pp.K2;
        const double inv = 1.0 / ((double)pp.n[0] * pp.n[1] * pp.n[2]);
        const float hi = (float)inv;
        const tf sc{hi, (float)(inv - (double)hi)};
        if (adj_cube_supported(pp)) {
            if (pp.n[0] == 24) return launch_adj_cube<24>(Gb, P, pp, sc, (float4 *)H, st);
            if (pp.n[0] == 40) return launch_adj_cube<40>(Gb, P, pp, sc, (float4 *)H, st);
            if (pp.n[0] == 48) return launch_adj_cube<48>(Gb, P, pp, sc, (float4 *)H, st);
            return launch_adj_cube<72>(Gb, P, pp, sc, (float4 *)H, st);
        }
        cudaError_t e =
            cudaFuncSetAttribute(adj_pair_tf_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        adj_pair_tf_kernel<<<(unsigned)P, 256, sm, st>>>(Gb, pp, cell_start, cell_g, ncell, tf_consts(), sc, (float4 *)H);
        return cudaGetLastError();
    }
    size_t sm = sizeof(double2) * (2 * (size_t)pp.n[1] * pp.n[2] + pp.n[0] + pp.n[1] + pp.n[2] + pp.ng) +
                sizeof(int) * pp.K2;
    cudaError_t e = cudaFuncSetAttribute(adj_pair_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    adj_pair_kernel<false><<<(unsigned)P, 256, sm, st>>>(Gb, P, pp, cell_start, cell_g, ncell, H);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ products into the band adjoints
__device__ __forceinline__ double2 psi_at(const void *psi, int64_t i, bool tf)
{
    if (!tf) return ((const double2 *)psi)[i];
    float4 v = ((const float4 *)psi)[i];
    return make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
}

// psibar_c[c](r) += sum_{v in [v0, v0+nvc)} psi_v(r) H[(v - v0) nc + c](r)
__global__ void adj_cond_kernel(const void *__restrict__ psiv, int v0, int nvc, const double2 *__restrict__ H, int nc,
                                int64_t nr, bool tf, double2 *__restrict__ pbc)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (i >= nr) return;
    double2 acc = pbc[(int64_t)c * nr + i];
    for (int v = 0; v < nvc; ++v) cfma(acc, psi_at(psiv, (int64_t)(v0 + v) * nr + i, tf), H[((int64_t)v * nc + c) * nr + i]);
    pbc[(int64_t)c * nr + i] = acc;
}

// psibar_v[v](r) += sum_c psi_c(r) conj(H[(v - v0) nc + c](r))
__global__ void adj_val_kernel(const void *__restrict__ psic, int v0, const double2 *__restrict__ H, int nc,
                               int64_t nr, bool tf, double2 *__restrict__ pbv)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int vl = blockIdx.y;
    if (i >= nr) return;
    double2 acc = pbv[(int64_t)(v0 + vl) * nr + i];
    for (int c = 0; c < nc; ++c) {
        double2 hh = H[((int64_t)vl * nc + c) * nr + i];
        cfma(acc, psi_at(psic, (int64_t)c * nr + i, tf), make_double2(hh.x, -hh.y));
    }
    pbv[(int64_t)(v0 + vl) * nr + i] = acc;
}

// Two-float forms of the two products (bands, H and the accumulators psibar in two-float form,
// 16 bytes a point as in FP64): everything on the FP32 pipes -- adding into FP64 accumulators
// took eight FP64 instructions a thread, which bounded the conduction product on this GPU.
__global__ void adj_cond_tf_kernel(const float4 *__restrict__ psiv, int v0, int nvc, const float4 *__restrict__ H,
                                   int nc, int64_t nr, float4 *__restrict__ pbc)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (i >= nr) return;
    tcx acc{{0.f, 0.f}, {0.f, 0.f}};
    for (int v = 0; v < nvc; ++v)
        acc = tc_add(acc, tc_mul(tc_load(psiv + (int64_t)(v0 + v) * nr + i), tc_load(H + ((int64_t)v * nc + c) * nr + i)));
    float4 *o = pbc + (int64_t)c * nr + i;
    tc_store(o, tc_add(tc_load(o), acc));
}

__global__ void adj_val_tf_kernel(const float4 *__restrict__ psic, int v0, const float4 *__restrict__ H, int nc,
                                  int64_t nr, float4 *__restrict__ pbv)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int vl = blockIdx.y;
    if (i >= nr) return;
    tcx acc{{0.f, 0.f}, {0.f, 0.f}};
    for (int c = 0; c < nc; ++c) // psi_c conj(H) = conj(conj(psi_c) H)
        acc = tc_add(acc, tc_mulc(tc_load(psic + (int64_t)c * nr + i), tc_load(H + ((int64_t)vl * nc + c) * nr + i)));
    float4 *o = pbv + (int64_t)(v0 + vl) * nr + i;
    tc_store(o, tc_add(tc_load(o), tcx{acc.re, tf_neg(acc.im)}));
}

// Both products of NV valence rows from one pass over H, a grid point per thread: psibar_c[c] +=
// sum_v psi_v H[v][c] as it goes, psibar_v[v] += psi_c conj(H[v][c]) = conj(conj(psi_c) H[v][c]) in
// registers over all c.  The sums are lazy two-float (tc_acc), renormalised every fourth term.  H is the
// traffic: 384 conduction bands and 48 valence bands in rows of five on 40^3 (18.9 GB) take 7.1 ms where the
// two kernels above, which read it twice, take 9.2.  Segments of c in blocks of their own take 9.6.
template <int NV>
__global__ void __launch_bounds__(64) adj_products_tf_kernel(const float4 *__restrict__ psiv,
                                                             const float4 *__restrict__ psic,
                                                             const float4 *__restrict__ H, int nc, int64_t nr,
                                                             float4 *__restrict__ pbv, float4 *__restrict__ pbc)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nr) return;
    tcx pv[NV], av[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        pv[v] = tc_load(psiv + v * nr + i);
        av[v] = tcx{{0.f, 0.f}, {0.f, 0.f}};
    }
#pragma unroll 2
    for (int c = 0; c < nc; ++c) {
        const tcx pc = tc_load(psic + c * nr + i), pcc{pc.re, tf_neg(pc.im)};
        const tcx old = tc_load(pbc + c * nr + i);
        tcx h[NV], ac{{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
        for (int v = 0; v < NV; ++v) h[v] = tc_load(H + ((int64_t)v * nc + c) * nr + i);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            tc_acc(ac, pv[v], h[v]);
            if (v == 3) ac = tc_norm(ac);
            tc_acc(av[v], pcc, h[v]);
            if ((c & 3) == 3) av[v] = tc_norm(av[v]);
        }
        tc_store(pbc + c * nr + i, tc_add(old, tc_norm(ac)));
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const tcx a = tc_norm(av[v]);
        float4 *o = pbv + v * nr + i;
        tc_store(o, tc_add(tc_load(o), tcx{a.re, tf_neg(a.im)}));
    }
}

// Two-float accumulators to FP64, in place (same 16 bytes per point).
__global__ void tf_to_f64_kernel(void *__restrict__ x, int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 v = ((const float4 *)x)[i];
        ((double2 *)x)[i] = make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
    }
}

cudaError_t launch_tf_to_f64(void *x, int64_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, 4096);
    tf_to_f64_kernel<<<(unsigned)blocks, 256, 0, st>>>(x, n);
    return cudaGetLastError();
}

cudaError_t launch_adj_products(const void *psiv, const void *psic, int v0, int nvc, int nc, const double2 *H,
                                int64_t nr, bool tf, double2 *pbv, double2 *pbc, cudaStream_t st)
{
    if (tf) {
        // One pass where the grid's points alone fill the GPU and the rows fit the registers.  Two kernels
        // against one pass, 300 conduction bands, ms: one row .338 / .375 at 64000 points, .414 / .422 at 91125,
        // .465 / .434 at 110592; two rows .399 / .352 at 64000; three .469 / .489 at 64000, .719 / .537 at 81000;
        // four, five and six .693 / .489, .758 / .564 and .811 / .593 at 64000, and less on every larger grid.
        // 27000 points: one pass slower for any number of rows.
        if (nvc <= 6 && nr >= (nvc == 1 ? 100000 : nvc == 3 ? 70000 : 60000)) {
            const float4 *pv = (const float4 *)psiv + v0 * nr;
            auto run = [&](auto kern) {
                kern<<<(unsigned)((nr + 63) / 64), 64, 0, st>>>(pv, (const float4 *)psic, (const float4 *)H, nc, nr,
                                                                (float4 *)pbv + v0 * nr, (float4 *)pbc);
                return cudaGetLastError();
            };
            switch (nvc) {
            case 1: return run(adj_products_tf_kernel<1>);
            case 2: return run(adj_products_tf_kernel<2>);
            case 3: return run(adj_products_tf_kernel<3>);
            case 4: return run(adj_products_tf_kernel<4>);
            case 5: return run(adj_products_tf_kernel<5>);
            default: return run(adj_products_tf_kernel<6>);
            }
        }
        dim3 gc((unsigned)((nr + 255) / 256), nc);
        adj_cond_tf_kernel<<<gc, 256, 0, st>>>((const float4 *)psiv, v0, nvc, (const float4 *)H, nc, nr,
                                               (float4 *)pbc);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        dim3 gv((unsigned)((nr + 255) / 256), nvc);
        adj_val_tf_kernel<<<gv, 256, 0, st>>>((const float4 *)psic, v0, (const float4 *)H, nc, nr, (float4 *)pbv);
        return cudaGetLastError();
    }
    dim3 gc((unsigned)((nr + 255) / 256), nc);
    adj_cond_kernel<<<gc, 256, 0, st>>>(psiv, v0, nvc, H, nc, nr, tf, pbc);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    dim3 gv((unsigned)((nr + 255) / 256), nvc);
    adj_val_kernel<<<gv, 256, 0, st>>>(psic, v0, H, nc, nr, tf, pbv);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ band adjoint
// Pruned to the plane waves' box |G_a| <= m_a: all lines along i2, along i1 those of the K2 kept
// frequencies, along i0 those of the K1 x K2 kept ones.  FP64-bound like the band setup's transform,
// which does three full axes on all lines: 432 bands of 4500 plane waves on 40^3 3.42 -> 2.30 ms, 136 bands on
// 48^3 1.91 -> 1.06, 130 of 8000 on 72^3 9.1 -> 4.5.
struct KeptLines {
    int n, m, k; // k = min(n, 2 m + 1) kept indices: 0 .. m and n - m .. n - 1
};
__device__ __forceinline__ int kept_index(KeptLines a, int c) { return c <= a.m || a.k == a.n ? c : c + a.n - a.k; }

// One (band, i0) slab: conj, FFT along i2, the kept columns along i1, stored in place.
__global__ void __launch_bounds__(256) adj_band_slab_kernel(double2 *__restrict__ psi, int n0, int n1, int n2,
                                                             FftAxis ax1, FftAxis ax2, KeptLines q2)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int ns = n1 * n2;
    double2 *a = (double2 *)smem, *b = a + ns, *tw1 = b + ns, *tw2 = tw1 + n1;
    for (int i = threadIdx.x; i < n1; i += blockDim.x) tw1[i] = ax1.tw[i];
    for (int i = threadIdx.x; i < n2; i += blockDim.x) tw2[i] = ax2.tw[i];
    double2 *g = psi + ((int64_t)blockIdx.y * n0 + blockIdx.x) * ns;
    for (int i = threadIdx.x; i < ns; i += blockDim.x) a[i] = make_double2(g[i].x, -g[i].y);
    __syncthreads();
    double2 *r = fft_lines(a, b, n1, n2, 1, ax2, tw2);
    double2 *o = (r == a) ? b : a;
    for (int e = threadIdx.x; e < n1 * q2.k; e += blockDim.x) {
        const int i1 = e / q2.k, c = e - i1 * q2.k;
        o[e] = r[i1 * n2 + kept_index(q2, c)];
    }
    __syncthreads();
    const double2 *t = fft_lines(o, r, q2.k, 1, q2.k, ax1, tw1);
    for (int e = threadIdx.x; e < n1 * q2.k; e += blockDim.x) {
        const int i1 = e / q2.k, c = e - i1 * q2.k;
        g[i1 * n2 + kept_index(q2, c)] = t[e];
    }
}

// One (band, kept i1) plane: the kept columns along i0.
__global__ void __launch_bounds__(256) adj_band_axis0_kernel(double2 *__restrict__ psi, int n0, int n1, int n2,
                                                              FftAxis ax0, KeptLines q1, KeptLines q2)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int np = n0 * q2.k;
    double2 *a = (double2 *)smem, *b = a + np, *tw0 = b + np;
    for (int i = threadIdx.x; i < n0; i += blockDim.x) tw0[i] = ax0.tw[i];
    double2 *g = psi + (int64_t)blockIdx.y * n0 * n1 * n2 + (int64_t)kept_index(q1, blockIdx.x) * n2;
    const int64_t rs = (int64_t)n1 * n2;
    for (int e = threadIdx.x; e < np; e += blockDim.x) {
        const int i0 = e / q2.k, c = e - i0 * q2.k;
        a[e] = g[i0 * rs + kept_index(q2, c)];
    }
    __syncthreads();
    const double2 *r = fft_lines(a, b, q2.k, 1, q2.k, ax0, tw0);
    for (int e = threadIdx.x; e < np; e += blockDim.x) {
        const int i0 = e / q2.k, c = e - i0 * q2.k;
        g[i0 * rs + kept_index(q2, c)] = r[e];
    }
}

// dcoeff[b][k] = 2 conj(F[b][gofs[k]]) where F = FFT_+(conj(psibar)) = conj(FFT_-(psibar))
__global__ void gather_grad_kernel(const double2 *__restrict__ F, const int32_t *__restrict__ gofs, int nb, int ngpsi,
                                   int64_t nr, double2 *__restrict__ dc)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)nb * ngpsi) return;
    int b = (int)(i / ngpsi), k = (int)(i - (int64_t)b * ngpsi);
    double2 z = F[(int64_t)b * nr + gofs[k]];
    dc[i] = make_double2(2.0 * z.x, -2.0 * z.y);
}

cudaError_t launch_band_adjoint(double2 *pb, int nb, const int n[3], const FftAxis ax[3], const int maxabs[3],
                                const int32_t *gofs, int ngpsi, double2 *dc, cudaStream_t st)
{
    const int64_t nr = (int64_t)n[0] * n[1] * n[2];
    const int64_t tot = (int64_t)nb * nr;
    if (tot == 0) return cudaSuccess;
    KeptLines q[3];
    for (int a = 0; a < 3; ++a) q[a] = {n[a], maxabs[a], std::min(n[a], 2 * maxabs[a] + 1)};
    const size_t sm1 = sizeof(double2) * (2 * (size_t)n[1] * n[2] + n[1] + n[2]);
    const size_t sm0 = sizeof(double2) * (2 * (size_t)n[0] * q[2].k + n[0]);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(adj_band_slab_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm1)) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(adj_band_axis0_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm0)) !=
            cudaSuccess)
        return e;
    adj_band_slab_kernel<<<dim3(n[0], nb), 256, sm1, st>>>(pb, n[0], n[1], n[2], ax[1], ax[2], q[2]);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    adj_band_axis0_kernel<<<dim3(q[1].k, nb), 256, sm0, st>>>(pb, n[0], n[1], n[2], ax[0], q[1], q[2]);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int64_t ng = (int64_t)nb * ngpsi;
    gather_grad_kernel<<<(unsigned)((ng + 255) / 256), 256, 0, st>>>(pb, gofs, nb, ngpsi, nr, dc);
    return cudaGetLastError();
}

} // namespace gw
