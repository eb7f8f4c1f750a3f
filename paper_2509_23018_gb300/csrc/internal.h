// Internal launch interface between the host API and the kernel translation units.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>
#include "common.cuh"

namespace gw {

constexpr int kMaxOmega = 64;
struct OmegaList {
    int nw;
    double w[kMaxOmega];
};

// ---- stage (a): band setup and pair elements (mtxel.cu)
cudaError_t launch_scatter(const double2 *coeff, const int32_t *gofs, int nb, int ngpsi, int64_t nr, double2 *psi,
                           cudaStream_t st);
cudaError_t launch_band_fft(double2 *psi, int nb, const int n[3], const FftAxis ax[3], cudaStream_t st);

struct PairPlan {
    int n[3];
    FftAxis ax[3];
    int K2;              // number of needed frequencies along the last axis
    const int *kz;       // device [K2]   needed last-axis frequencies (0..n2-1)
    int ng;
    const int32_t *gpack; // device [ng]   k0 | k1 << 8 | k2index << 16
    int K12;              // number of (k1, k2) cells that hold sphere points
    const int32_t *cell;  // device [K12]  k2index << 8 | k1, ordered by (k2index, k1)
    const int *cstart;    // device [K12 + 1] points of cell d: cpts[cstart[d] .. cstart[d + 1])
    const int2 *cpts;     // device [ng]   (point index, k0 | cell << 8), grouped by cell
    // scratch of the two-float grid-specialised kernel (pair_tf_scratch): nslots slots of
    // n0 * K12 two-float values, one flag per slot
    float4 *scr;
    int *slot_flags;
    int nslots;
    int *status;          // device status word (kStatusNoSlot)
    // the FP64 pair kernel runs only where *guard is set, pair_split64_* only where it is not (null: both run)
    const int *guard = nullptr;
};
// Scratch the two-float pair kernel needs for a plan: *nslots slots of *slot_elems float4
// (0 slots: the plan runs on the runtime-shape kernel, which needs none).
cudaError_t pair_tf_scratch(const PairPlan &pp, int *nslots, size_t *slot_elems);
// Shared memory per block of the grid-specialised two-float pair kernel for this plan (0 when it
// does not take the plan).
size_t pair_tf_ct_smem_bytes(const PairPlan &pp);
// M[p - p0][g] for p in [p0, p0 + count); pair p = v * nc + c.
cudaError_t launch_pair(const double2 *psiv, const double2 *psic, int nc, int64_t p0, int64_t count,
                        const PairPlan &pp, double2 *M, cudaStream_t st);
int pair_max_ng();
// the same in two-float arithmetic; psiv/psic hold two-float grids (launch_band_setup_tf)
cudaError_t launch_pair_tf(const void *psiv, const void *psic, int nc, int64_t p0, int64_t count,
                           const PairPlan &pp, double2 *M, cudaStream_t st);
// band setup in two-float arithmetic: scatter (with hi/lo split) + 3D FFT, psi in two-float form
// maxabs: largest |G_a| of the plane waves (input pruning of the grid-specialised transforms)
cudaError_t launch_band_setup_tf(const double2 *coeff, const int32_t *gofs, int nb, int ngpsi, void *psi,
                                 const int n[3], const FftAxis ax[3], const int maxabs[3], cudaStream_t st);


// ---- stage (a) last-axis transform on the tensor cores (zdft.cu) and the rest of the pair
// transform from its output (pair_tf_ct.cuh)
constexpr int kZdSlices = 6; // BF16 slices per operand (balanced base-256 digits)
// n: points of a line (the last axis), lines: n0 n1
// row slices of nr two-float band grids psi [nr][lines][n], zd_row_bytes(nr, n, lines) bytes: images of
// the product's shared-memory tiles, [lines][row tiles of 128][stages of 8 points][kZdSlices]
cudaError_t launch_zd_rows(const void *psi, int nr, int n, int lines, void *A, cudaStream_t st);
size_t zd_row_bytes(int nr, int n, int lines);
// column exponents E[nb][lines] of two-float band grids psi [nb][lines][n]
cudaError_t launch_zd_colexp(const void *psi, int nb, int n, int lines, int *E, cudaStream_t st);
bool zd_supported(int n, int K2);
int zd_valence_per_tile(int n, int K2);
int zd_row_entries(int K2); // entries of F per (line, row): K2 rounded up to even
// F[l][vl cb + cl][q] (two-float, zd_row_entries(K2) entries a row) = sum_i2
// conj(psi_v[l][i2]) W^{kz[q] i2} psi_c[l][i2] for the valence bands v = v0 + vl, vl < vb, and the cb
// conduction bands whose row slices A holds; tmV maps the valence grids as FP32 [nv][lines][4n], box
// {4n, 1, zd_valence_per_tile(n, K2)}, or with s = zd_line_split(n) as [nv][s lines][4n / s], box
// {4n / s, s, zd_valence_per_tile(n, K2)}
int zd_line_split(int n);
cudaError_t launch_zd_gemm(const CUtensorMap &tmV, const void *A, const int *E, const int *kz, const float4 *twf, int n,
                           int lines, int nv, int v0, int vb, int cb, int K2, float4 *F, int *status, cudaStream_t st);
// The middle and first axes from F for any n0, n1 of pair_split_supported, in two kernels with the
// cells S [R][n0][K12] (two-float) between them: pair_split1 (tmF as below), pair_split2 (tmS: S as
// [R n0 rows][K12] entries, FP32 elements, box {8 K2, n0}).
bool pair_split_supported(int n);
cudaError_t launch_pair_split1(const CUtensorMap &tmF, int64_t R, const PairPlan &pp, float4 *S, cudaStream_t st);
cudaError_t launch_pair_split2(const CUtensorMap &tmS, int64_t R, int cb, int64_t sv, int64_t sc, const PairPlan &pp,
                               double2 *M, cudaStream_t st);
// M[(vl sv + cl sc) ng + g] of the block's R pairs, row vl cb + cl, from F (middle and first axis of
// the pair transform)
// (tmF: F as [N^2 lines][R rows of zd_row_entries(K2)] two-float entries, FP32 elements, box {4 K2, 2 N}; tmS: the plan's
// scratch slots as [nslots N rows][K12] two-float entries, box {8 K2, N}; no swizzle)
cudaError_t launch_pair_tf_from_f(const CUtensorMap &tmF, const CUtensorMap &tmS, int64_t R, int cb, int64_t sv,
                                  int64_t sc, const PairPlan &pp, double2 *M, cudaStream_t st);

// ---- the same in FP64 (zdft64.cu, pair_split64_ct.cuh): seven nine-bit slices per operand, double2 grids, F
// and cells.  Lines of 24 to 56 points.  guard: set by the slicing kernels where an entry is not finite
// or a line is scaled by more than 2^+-390; the product returns at once where it is set.
size_t zd64_row_bytes(int nr, int n, int lines); // row slices and exponents
cudaError_t launch_zd64_rows(const void *psi, int nr, int n, int lines, void *A, int *guard, cudaStream_t st);
cudaError_t launch_zd64_colexp(const void *psi, int nb, int n, int lines, int *E, int *guard, cudaStream_t st);
bool zd64_supported(int n, int K2);
int zd64_valence_per_tile(int K2);
cudaError_t launch_zd64_gemm(const CUtensorMap &tmV, const void *A, const int *E, const int *kz, const double2 *tw, int n,
                             int lines, int nv, int v0, int vb, int cb, int K2, double2 *F, const int *guard,
                             int *status, cudaStream_t st);
cudaError_t launch_pair_split64_1(const CUtensorMap &tmF, int64_t R, const PairPlan &pp, double2 *S, cudaStream_t st);
cudaError_t launch_pair_split64_2(const CUtensorMap &tmS, int64_t R, int cb, int64_t sv, int64_t sc, const PairPlan &pp,
                                  double2 *M, cudaStream_t st);

// ---- energy factor, diagonal, symmetrisation (reduce.cu)
// delta[w][p - p0] = 4x/(x^2 + w^2), x = ev[v] - ec[c]
cudaError_t launch_delta(const double *ev, const double *ec, int nc, int64_t p0, int64_t count, const OmegaList &om,
                         double *delta, cudaStream_t st);
// real axis with broadening: delta[3w + k][p - p0], k = 0: min(Re D, 0), 1: -max(Re D, 0), 2: Im D
cudaError_t launch_delta_real(const double *ev, const double *ec, int nc, int64_t p0, int64_t count,
                              const OmegaList &om, double eta, double *delta, cudaStream_t st);
// out[w] = (T[3w] - T[3w+1]) + i T[3w+2]
cudaError_t launch_combine_real(const double2 *T, int64_t nn, int nw, double2 *out, cudaStream_t st);
// forward derivative of Delta along (dE_v, dE_c), split: out[2w] = min(dD, 0), out[2w+1] = -max(dD, 0)
cudaError_t launch_delta_jvp(const double *ev, const double *ec, const double *dev, const double *dec, int nc,
                             int64_t p0, int64_t count, const OmegaList &om, double *out, cudaStream_t st);
// d = X1 + X2; X1 = M + d; X2 = M - d
cudaError_t launch_jvp_mix(const double2 *M, double2 *X1, double2 *X2, int64_t n, cudaStream_t st);
// out[w] = (Tp[w] - Tm[w]) / 2 + Tw[2w] - Tw[2w+1]
cudaError_t launch_combine_jvp(const double2 *Tp, const double2 *Tm, const double2 *Tw, int64_t nn, int nw,
                               double2 *out, cudaStream_t st);
// diag[w][g] += sum_p delta[w][p] |M[p][g]|^2
cudaError_t launch_diag(const double2 *M, int64_t P, int ng, const double *delta, int64_t dstride, int nw,
                        double *diag, int64_t diag_wstride, cudaStream_t st);
// ---- dielectric matrix inverse (epsilon.cu)
cudaError_t launch_eps_sqrt(const double *v, int ng, double *sv, cudaStream_t st);
// A = I - s chi s and bmax = Gershgorin bound of A (bits of a double)
cudaError_t launch_eps_sym(const double2 *chi, const double *sv, int ng, double2 *A, unsigned long long *bmax,
                           cudaStream_t st);
cudaError_t launch_eps_init(double2 *X, int ng, const unsigned long long *bmax, cudaStream_t st);
// *r = ||I - T||_F^2
cudaError_t launch_eps_resid(const double2 *T, int ng, double *r, cudaStream_t st);
cudaError_t launch_eps_step(double2 *X, const double2 *P, int64_t n, cudaStream_t st);
cudaError_t launch_eps_unsym(const double2 *X, const double *sv, int ng, double2 *out, cudaStream_t st);

// out[g][b] = conj(V[b n + g]) (column-major n x neig -> row-major [n][neig], conjugated)
cudaError_t launch_conj_transpose(const double2 *V, int n, int neig, double2 *out, cudaStream_t st);
// a bounded wait that is never satisfied: sets kStatusTimeout in *status after iters tries
cudaError_t launch_watchdog(long long iters, int *status, cudaStream_t st);
// out = (W + W^H) / 2 for a row-major n x n complex matrix (out must not alias W)
cudaError_t launch_herm_part(const double2 *W, int n, double2 *out, cudaStream_t st);
// lower triangle <- conj(upper), Im diag <- 0, for nw consecutive ng x ng blocks
cudaError_t launch_symmetrize(double2 *chi, int ng, int nw, cudaStream_t st);

// ---- stage (b), FP64 tensor cores (contract_f64.cu)
// One job = one chi block: chi[G][G'] += sum_p conj(M[p][G]) delta[p] M[p][G'] on upper tiles.
struct __align__(128) F64Job {
    CUtensorMap tm;       // M as doubles [P][2 ng], box {2 BT, 16}
    const double *delta;  // [P]
    double *chi;          // [ng][ng] complex
    int64_t P;
    int ng, ntile, ksplit, item_start;
};
// guard (or null): runs only where *guard is set
cudaError_t launch_contract_f64_jobs(int bt, const F64Job *jobs, int njobs, int nitems, int grid, int *status, const int *guard,
                                     cudaStream_t st);
int contract_f64_bk();
size_t contract_f64_smem(int bt);

// ---- stage (b), split precision on BF16 tensor cores (ozaki.cu)
// sp[i] = sqrt(-delta[i])
cudaError_t launch_oz_sqrt(const double *delta, int64_t n, double *sp, cudaStream_t st);
// E[g] = column exponent of s_p M[p][g] (sp null: of M[p][g]) over the chunk; guard (or null): set to 1 where the FP64
// contraction by slices does not hold (entries not finite, columns scaled by more than 2^+-390)
cudaError_t launch_oz_colexp(const double2 *M, int64_t P, int ng, const double *sp, int *E, int *guard,
                             cudaStream_t st);
// A group of nw <= oz_group_w() frequencies at once (scales sp + w dstride): exponents E[w][ng],
// slices of frequency w at Z + w zstride (bf16 elements); M read once per pass for the group.
int oz_group_w();
cudaError_t launch_oz_split_multi(const double2 *M, int64_t P, int ng, const double *sp, int64_t dstride, int nw,
                                  int *E, int s, int64_t kpad, void *Z, int64_t zstride, cudaStream_t st);
// Z[i][j][p] bf16 slices, rows p in [P, kpad) zero
cudaError_t launch_oz_slice(const double2 *M, int64_t P, int ng, const double *sp, const int *E, int s,
                            int64_t kpad, void *Z, int *guard, cudaStream_t st);
int oz_f64_slices(); // slices of the FP64 contraction
// One job = the split contraction of one chunk into one chi block (upper tiles).
struct __align__(128) OzJob {
    CUtensorMap tmA, tmB; // slices [s][2 ng][kpad] bf16, boxes {64, 128}
    const int *E;         // [ng] column exponents
    double *chi;          // [ng][ng] complex
    int ng, nk, s;
    // general product (launch_oz_gemm_general): out[rows_a][cols_b] (complex, rows of ldo doubles)
    // += A B with the slices of A's rows (tmA, exponents E[rows_a]) and of B's columns (tmB,
    // exponents E2[cols_b])
    const int *E2;
    double *out;
    int64_t ldo;
    int rows_a, cols_b, add; // add = 0: out = A B
};
// One unit of work of a launch: a tile of a job (oz_box_rows() complex rows and columns) over the
// K-steps [kb0, kb0 + nk).  parts > 1: part `part` of the K range of tile `slot` of the launch's split
// tiles; the parts' sums meet in scratch and are added in their order by whichever comes last.
struct OzItem {
    int job, I, J, kb0, nk, part, parts, slot;
};
// Scratch of a launch with split tiles: oz_part_bytes() per (slot, part), oz_slot_flags() counters per
// slot, zero before the first launch and again after every launch.
struct OzScratch {
    double *sums;
    int *flags;
};
size_t oz_part_bytes();
int oz_slot_flags();
// clusters: pairs of CTAs; guard (or null): the FP64 contraction (oz_f64_slices() slices), which leaves
// the chunk alone where *guard is set
cudaError_t launch_oz_gemm_jobs(const OzJob *jobs, const OzItem *items, int nitems, int clusters, OzScratch scr,
                                int *status, const int *guard, cudaStream_t st);
int oz_slices(int nslices); // 9-bit slices for the accuracy of nslices six-bit ones
// Slices of the general split product Y = A B: the rows of A or the columns of B, `rows` of them
// with ka complex entries each, entry g of row p at A[p sr + g sk], into s nine-bit BF16 slices
// Z[i][2 p + {Re, Im}][kpad] with exponents E[p]; kpad = ka rounded up to a multiple of 64.
// conj: of the conjugate.
cudaError_t launch_oz_split(const double2 *A, int64_t rows, int ka, int64_t sr, int64_t sk, bool conj, int s,
                            int64_t kpad, void *Z, int *E, cudaStream_t st);
// Plasmon-pole prep. step straight into row slices of P^T (the layout of launch_oz_split with
// rows = ka = ng): P[g][c] = A[g][c] / (d - sgn wt[g][c]) in two-float arithmetic, At / Wt = A
// and wt transposed [c][g] as two-float (hi, lo) pairs (gpp_setup_tf), for cnt <= kGppMaxE
// energies d[0..cnt) (host) at once: slices of energy j at Z + j zstride (bf16 elements),
// exponents at E + j ng.
constexpr int kGppMaxE = 16;
struct GppEnergies {
    double d[kGppMaxE];
};
cudaError_t launch_gpp_prep_split(const float4 *At, const float4 *Wt, int ng, const double *d, int cnt, float sgn,
                                  int s, int64_t kpad, int64_t zstride, void *Z, int *E, cudaStream_t st);
cudaError_t launch_oz_gemm_general(const OzJob *jobs, const OzItem *items, int nitems, int clusters, int *status,
                                   cudaStream_t st);
int oz_box_rows();
int oz_box_k();

// ---- adjoint of L = Re Tr(W chi) (adjoint.cu)
cudaError_t launch_zgemm(const double2 *A, const double2 *B, double2 *C, int64_t mr, int kd, int nc, cudaStream_t st);
// C (+)= op(A) op(B): conj_a takes conj(A); trans_b reads B as its transpose, row-major [nc][kd];
// accumulate adds into C.  Built for (conj_a), (trans_b, accumulate) and the plain product.
cudaError_t launch_zgemm_ex(const double2 *A, const double2 *B, double2 *C, int64_t mr, int kd, int nc, bool conj_a,
                            bool trans_b, bool accumulate, cudaStream_t st);
// ---- plasmon-pole self-energy, prep. step (sigma.cu)
// A[g][c] = v[c] Omega2[g][c] / (2 wt[g][c]) in FP64, stored [g][c]
cudaError_t launch_gpp_setup(const double2 *omega2, const double2 *wtilde, const double *vcoul, int ng, double2 *A,
                             cudaStream_t st);
// the same A and wt, transposed [c][g], as two-float (hi, lo) pairs for the split path
cudaError_t launch_gpp_setup_tf(const double2 *omega2, const double2 *wtilde, const double *vcoul, int ng, float4 *At,
                                float4 *Wt, cudaStream_t st);
// sigma[e][l][m] = ST[m][e nsig + l] (ST accumulated transposed by the split path)
cudaError_t launch_gpp_untranspose(const double2 *ST, int ne, int nsig, double2 *sigma, cudaStream_t st);
// P[g][c] = A[g][c] / (d - sgn wt[g][c]) (FP64, stored)
cudaError_t launch_gpp_prep_f64(const double2 *A, const double2 *wtilde, int ng, double d, double sgn, double2 *P,
                                cudaStream_t st);
cudaError_t launch_adj_rows(const double2 *M, double2 *Y, int64_t P, int ng, int nc, int64_t p0, const double *ev,
                            const double *ec, double w, double *L, double *dEv, double *dEc, cudaStream_t st);
// twofloat: the back-projection in two-float arithmetic (band grids in two-float form), H then
// holds float4 (hi, lo) pairs and launch_adj_products reads it that way and accumulates pbv / pbc
// in that form too (launch_tf_to_f64 converts them before the band adjoint), and Gb's rows are
// overwritten with conj(g_p) in two-float form; else FP64, Gb read only
cudaError_t launch_adj_pair(double2 *Gb, int64_t P, const PairPlan &pp, const int *cell_start,
                            const int *cell_g, int ncell, double2 *H, bool twofloat, cudaStream_t st);
// two-float (float4 hi/lo pairs) to complex128, in place, n points
cudaError_t launch_tf_to_f64(void *x, int64_t n, cudaStream_t st);
cudaError_t launch_adj_products(const void *psiv, const void *psic, int v0, int nvc, int nc, const double2 *H,
                                int64_t nr, bool tf, double2 *pbv, double2 *pbc, cudaStream_t st);
cudaError_t launch_band_adjoint(double2 *pb, int nb, const int n[3], const FftAxis ax[3], const int maxabs[3],
                                const int32_t *gofs, int ngpsi, double2 *dc, cudaStream_t st);

} // namespace gw
