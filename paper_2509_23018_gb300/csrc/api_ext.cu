// Entry points beyond chi0 itself: the adjoint of L = Re Tr(W chi0), the static subspace,
// the inverse dielectric matrix, chi0 on the real axis and the forward derivative.
#include "api_internal.h"

using namespace gwapi;

// Bytes of the slices of a product's B operand (ka complex inner entries, nout columns)
static size_t oz_b_bytes(const gw_chi0 *h, int ka, int nout)
{
    return h->d.prec == GW_PREC_OZAKI_BF16 ? (size_t)gw::oz_slices(h->d.nslices) * 4 * nout * oz_kpad(ka) : 0;
}

static gw_status adjoint(gw_chi0 *h, int iq, double omega, const double *W, double *L, double *dE_v, double *dE_c,
                         double *dcoeff_v, double *dcoeff_c)
{
    gw_status s = check_slot(h, iq);
    if (s) return s;
    if (!W || !dE_v || !dE_c || !dcoeff_v || !dcoeff_c) return fail(h, GW_ERR_ARG, "null pointer");
    if (!(omega >= 0.0) || !std::isfinite(omega)) return fail(h, GW_ERR_ARG, "omega must be finite and >= 0");
    const BandSet &v = h->val[iq];
    const BandSet &c = h->cond;
    const Sphere &sp = h->sph[iq];
    const int nv = v.nb, nc = c.nb, ng = sp.ng;
    const int64_t nr = h->nr;
    const bool tf = h->d.mtxel_prec == GW_MTXEL_TWOFLOAT;
    // valence bands per chunk: bounded by the pair chunk and by 2 GiB of back-projected grids
    int64_t vch = std::max<int64_t>(1, h->d.pair_chunk / nc);
    vch = std::min<int64_t>(vch, std::max<int64_t>(1, (int64_t(2) << 30) / ((int64_t)nc * nr * 16)));
    vch = std::min<int64_t>(vch, nv);
    const int64_t cmax = vch * nc;
    // work buffers, held only for this call
    double2 *Mb = nullptr, *Yb = nullptr, *Hb = nullptr, *pbv = nullptr, *pbc = nullptr, *Wh = nullptr;
    double *Lacc = nullptr;
    int *cs = nullptr, *cg = nullptr;
    const int ncell = (int)sp.cstart.size() - 1;
    size_t szM = sizeof(double2) * cmax * ng, szH = sizeof(double2) * cmax * nr;
    size_t szV = sizeof(double2) * (size_t)nv * nr, szC = sizeof(double2) * (size_t)nc * nr;
    const size_t szW = sizeof(double2) * (size_t)ng * ng;
    auto cleanup = [&]() {
        cudaStreamSynchronize(h->st);
        dfree(h, Wh, szW);
        dfree(h, Mb, szM);
        dfree(h, Yb, szM);
        dfree(h, Hb, szH);
        dfree(h, pbv, szV);
        dfree(h, pbc, szC);
        dfree(h, Lacc, sizeof(double));
        dfree(h, cs, sizeof(int) * (ncell + 1));
        dfree(h, cg, sizeof(int) * ng);
    };
#define ACK(x, what)                       \
    do {                                   \
        cudaError_t e_ = (x);              \
        if (e_ != cudaSuccess) {           \
            gw_status r_ = cuda_fail(h, e_, what); \
            cleanup();                     \
            return r_;                     \
        }                                  \
    } while (0)
    if ((s = dalloc(h, (void **)&Mb, szM, "adjoint M")) || (s = dalloc(h, (void **)&Yb, szM, "adjoint Y")) ||
        (s = dalloc(h, (void **)&Hb, szH, "adjoint grids")) || (s = dalloc(h, (void **)&pbv, szV, "valence adjoint")) ||
        (s = dalloc(h, (void **)&pbc, szC, "conduction adjoint")) ||
        (s = dalloc(h, (void **)&Lacc, sizeof(double), "L")) ||
        (s = dalloc(h, (void **)&cs, sizeof(int) * (ncell + 1), "cells")) ||
        (s = dalloc(h, (void **)&cg, sizeof(int) * ng, "cells")) ||
        (s = dalloc(h, (void **)&Wh, szW, "Hermitian part of W"))) {
        cleanup();
        return s;
    }
    // L sees W only through its Hermitian part (chi is Hermitian)
    ACK(gw::launch_herm_part((const double2 *)W, ng, Wh, h->st), "Hermitian part of W");
    ACK(cudaMemcpyAsync(cs, sp.cstart.data(), sizeof(int) * (ncell + 1), cudaMemcpyHostToDevice, h->st), "cells");
    ACK(cudaMemcpyAsync(cg, sp.cg.data(), sizeof(int) * ng, cudaMemcpyHostToDevice, h->st), "cells");
    ACK(cudaMemsetAsync(Lacc, 0, sizeof(double), h->st), "zero");
    ACK(cudaMemsetAsync(dE_v, 0, sizeof(double) * nv, h->st), "zero");
    ACK(cudaMemsetAsync(dE_c, 0, sizeof(double) * nc, h->st), "zero");
    ACK(cudaMemsetAsync(pbv, 0, szV, h->st), "zero");
    ACK(cudaMemsetAsync(pbc, 0, szC, h->st), "zero");
    gw::PairPlan pp = pair_plan(h, sp);
    ZdPlan z;
    ZdUse use{h};
    if ((s = zd_plan(h, sp, nv, nc, true, false, 1, 1, oz_b_bytes(h, ng, ng), cmax, z)) ||
        (z.on && ((s = zd_valence(h, z, sp, v.psi, nv)) || (s = zd_conduction(h, z, c.psi, 0, nc))))) {
        cleanup();
        return s;
    }
    // split precision: Y = M W as a split product, W's slices once per call
    const bool split = h->d.prec == GW_PREC_OZAKI_BF16;
    if (split && (s = oz_prepare_b(h, Wh, ng, ng))) {
        cleanup();
        return s;
    }
    for (int v0 = 0; v0 < nv; v0 += (int)vch) {
        const int nvc = (int)std::min<int64_t>(vch, nv - v0);
        const int64_t p0 = (int64_t)v0 * nc, cnt = (int64_t)nvc * nc;
        if ((s = pair_rows(h, z, sp, pp, v.psi, c.psi, nc, p0, cnt, Mb))) {
            cleanup();
            return s;
        }
        {
            Scope sc(h, "adj_zgemm");
            if (split) {
                if ((s = oz_product(h, Mb, cnt, ng, ng, Yb))) {
                    cleanup();
                    return s;
                }
            } else {
                ACK(gw::launch_zgemm(Mb, Wh, Yb, cnt, ng, ng, h->st), "Y = M W");
            }
        }
        {
            Scope sc(h, "adj_rows");
            ACK(gw::launch_adj_rows(Mb, Yb, cnt, ng, nc, p0, v.energy, c.energy, omega, Lacc, dE_v, dE_c, h->st),
                "row reductions");
        }
        {
            Scope sc(h, "adj_pair");
            ACK(gw::launch_adj_pair(Yb, cnt, pp, cs, cg, ncell, Hb, tf, h->st), "back-projection");
        }
        {
            Scope sc(h, "adj_products");
            ACK(gw::launch_adj_products(v.psi, c.psi, v0, nvc, nc, Hb, nr, tf, pbv, pbc, h->st), "products");
        }
    }
    {
        Scope sc(h, "adj_band");
        if (tf) {
            ACK(gw::launch_tf_to_f64(pbv, (int64_t)nv * nr, h->st), "valence adjoint to FP64");
            ACK(gw::launch_tf_to_f64(pbc, (int64_t)nc * nr, h->st), "conduction adjoint to FP64");
        }
        ACK(gw::launch_band_adjoint(pbv, nv, h->d.n, h->ax, v.maxabs, v.gofs, v.ngpsi, (double2 *)dcoeff_v, h->st),
            "valence band adjoint");
        ACK(gw::launch_band_adjoint(pbc, nc, h->d.n, h->ax, c.maxabs, c.gofs, c.ngpsi, (double2 *)dcoeff_c, h->st),
            "conduction band adjoint");
    }
    if (L) ACK(cudaMemcpyAsync(L, Lacc, sizeof(double), cudaMemcpyDeviceToHost, h->st), "L");
#undef ACK
    cleanup(); // synchronises: L is valid on return
    return GW_OK;
}

gw_status gw_chi0_adjoint(gw_chi0 *h, int iq, double omega, const double *W, double *L, double *dE_v, double *dE_c,
                          double *dcoeff_v, double *dcoeff_c)
{
    if (!h) return GW_ERR_ARG;
    return zd_or_fft(h, [&] { return adjoint(h, iq, omega, W, L, dE_v, dE_c, dcoeff_v, dcoeff_c); });
}

// ------------------------------------------------------------------ static subspace
namespace {
gw_status load_solver(gw_chi0 *h)
{
    if (h->sol.hdl) return GW_OK;
    const char *names[] = {"libcusolver.so.12", "libcusolver.so.11", "libcusolver.so",
                           "/usr/local/cuda/lib64/libcusolver.so.12", "/usr/local/cuda/lib64/libcusolver.so"};
    for (const char *n : names)
        if ((h->sol.lib = dlopen(n, RTLD_NOW | RTLD_LOCAL))) break;
    if (!h->sol.lib) return fail(h, GW_ERR_UNSUPPORTED, "the dense eigensolver (libcusolver) was not found");
    h->sol.create = (decltype(h->sol.create))dlsym(h->sol.lib, "cusolverDnCreate");
    h->sol.destroy = (decltype(h->sol.destroy))dlsym(h->sol.lib, "cusolverDnDestroy");
    h->sol.set_stream = (decltype(h->sol.set_stream))dlsym(h->sol.lib, "cusolverDnSetStream");
    h->sol.buffer_size = (decltype(h->sol.buffer_size))dlsym(h->sol.lib, "cusolverDnZheevdx_bufferSize");
    h->sol.heevdx = (decltype(h->sol.heevdx))dlsym(h->sol.lib, "cusolverDnZheevdx");
    if (!h->sol.create || !h->sol.destroy || !h->sol.set_stream || !h->sol.buffer_size || !h->sol.heevdx)
        return fail(h, GW_ERR_UNSUPPORTED, "libcusolver lacks the Hermitian eigensolver entry points");
    if (h->sol.create(&h->sol.hdl) != CUSOLVER_STATUS_SUCCESS) {
        h->sol.hdl = nullptr;
        return fail(h, GW_ERR_CUDA, "cusolverDnCreate failed");
    }
    return GW_OK;
}
} // namespace

gw_status gw_chi0_subspace_basis(gw_chi0 *h, int ng, const double *chi0, int neig, double *basis, double *evals)
{
    if (!h) return GW_ERR_ARG;
    if (ng < 1 || neig < 1 || neig > ng) return fail(h, GW_ERR_ARG, "need 1 <= neig <= ng");
    if (!chi0 || !basis) return fail(h, GW_ERR_ARG, "null pointer");
    gw_status st = load_solver(h);
    if (st) return st;
    const size_t nn = (size_t)ng * ng;
    if ((st = grow(h, (void **)&h->eigA, &h->eigA_cap, sizeof(double2) * nn, "eigensolver matrix")) ||
        (st = grow(h, (void **)&h->eigW, &h->eigW_cap, sizeof(double) * (size_t)ng, "eigenvalues")) ||
        (st = grow(h, (void **)&h->eigInfo, &h->eigInfo_cap, sizeof(int), "eigensolver status")))
        return st;
    // The row-major Hermitian chi0 read column-major is its transpose, conj(chi0): the solver
    // returns the conjugated eigenvectors, which the transposing copy conjugates back.
    CK(h, cudaMemcpyAsync(h->eigA, chi0, sizeof(double2) * nn, cudaMemcpyDeviceToDevice, h->st), "copy chi0");
    if (h->sol.set_stream(h->sol.hdl, h->st) != CUSOLVER_STATUS_SUCCESS) return fail(h, GW_ERR_CUDA, "solver stream");
    int meig = 0, lwork = 0;
    if (h->sol.buffer_size(h->sol.hdl, CUSOLVER_EIG_MODE_VECTOR, CUSOLVER_EIG_RANGE_I, CUBLAS_FILL_MODE_LOWER, ng,
                           (const cuDoubleComplex *)h->eigA, ng, 0.0, 0.0, 1, neig, &meig, h->eigW,
                           &lwork) != CUSOLVER_STATUS_SUCCESS)
        return fail(h, GW_ERR_CUDA, "eigensolver workspace query failed");
    if ((st = grow(h, (void **)&h->eigWork, &h->eigWork_cap, sizeof(double2) * (size_t)std::max(lwork, 1),
                   "eigensolver workspace")))
        return st;
    {
        Scope sc(h, "subspace_eig");
        if (h->sol.heevdx(h->sol.hdl, CUSOLVER_EIG_MODE_VECTOR, CUSOLVER_EIG_RANGE_I, CUBLAS_FILL_MODE_LOWER, ng,
                          (cuDoubleComplex *)h->eigA, ng, 0.0, 0.0, 1, neig, &meig, h->eigW,
                          (cuDoubleComplex *)h->eigWork, lwork, h->eigInfo) != CUSOLVER_STATUS_SUCCESS)
            return fail(h, GW_ERR_CUDA, "eigensolver failed");
        CK(h, gw::launch_conj_transpose(h->eigA, ng, neig, (double2 *)basis, h->st), "basis");
    }
    if (evals)
        CK(h, cudaMemcpyAsync(evals, h->eigW, sizeof(double) * neig, cudaMemcpyDeviceToDevice, h->st), "eigenvalues");
    int info = 0;
    CK(h, cudaMemcpyAsync(&info, h->eigInfo, sizeof(int), cudaMemcpyDeviceToHost, h->st), "solver status");
    CK(h, cudaStreamSynchronize(h->st), "subspace basis sync");
    if (info != 0) return fail(h, GW_ERR_CUDA, "eigensolver reported %d", info);
    if (meig != neig) return fail(h, GW_ERR_CUDA, "eigensolver returned %d of %d vectors", meig, neig);
    return GW_OK;
}

static gw_status compute_subspace(gw_chi0 *h, int iq, int neig, const double *basis, int nw, const double *omega,
                                  double *chi_sub)
{
    if (nw < 1 || nw > gw::kMaxOmega || !omega || !basis || !chi_sub)
        return fail(h, GW_ERR_ARG, "bad arguments (1 <= nw <= %d, non-null pointers)", gw::kMaxOmega);
    gw::OmegaList om;
    om.nw = nw;
    for (int i = 0; i < nw; ++i) {
        if (!(omega[i] >= 0.0) || !std::isfinite(omega[i])) return fail(h, GW_ERR_ARG, "omega must be finite and >= 0");
        om.w[i] = omega[i];
    }
    gw_status s = check_slot(h, iq);
    if (s) return s;
    const Sphere &sp = h->sph[iq];
    const BandSet &v = h->val[iq];
    const int ng = sp.ng;
    if (neig < 1 || neig > ng) return fail(h, GW_ERR_ARG, "need 1 <= neig <= ng");
    const int64_t P = (int64_t)v.nb * h->cond.nb;
    const double2 *Mres = resident_for(h, iq); // kept by the last gw_chi0_compute of this slot
    ZdPlan z;
    ZdUse use{h};
    if (!Mres && ((s = zd_plan(h, sp, v.nb, h->cond.nb, true, false, 1, nw, oz_b_bytes(h, ng, neig),
                              std::min<int64_t>(h->d.pair_chunk, P), z)) ||
                  (z.on && ((s = zd_valence(h, z, sp, v.psi, v.nb)) || (s = zd_conduction(h, z, h->cond.psi, 0, h->cond.nb))))))
        return s;
    const int64_t chunk = z.on ? (int64_t)z.vb * z.cb : std::min<int64_t>(h->d.pair_chunk, P);
    CK(h, cudaMemsetAsync(chi_sub, 0, sizeof(double2) * (size_t)nw * neig * neig, h->st), "zero chi");
    if ((s = ensure_work(h, (size_t)chunk * ng, (size_t)chunk * nw)) ||
        (s = grow(h, (void **)&h->MBbuf, &h->MBcap, sizeof(double2) * (size_t)chunk * neig, "projected M")))
        return s;
    const bool split = h->d.prec == GW_PREC_OZAKI_BF16;
    if (split && (s = oz_prepare_b(h, (const double2 *)basis, ng, neig))) return s;
    gw::PairPlan pp = pair_plan(h, sp);
    for (int64_t p0 = 0; p0 < P; p0 += chunk) {
        const int64_t cnt = std::min(chunk, P - p0);
        const double2 *Mc = Mres ? Mres + p0 * ng : h->Mbuf;
        if (!Mres && (s = pair_rows(h, z, sp, pp, v.psi, h->cond.psi, h->cond.nb, p0, cnt, h->Mbuf))) return s;
        {
            Scope sc(h, "subspace_projection");
            if (split) {
                if ((s = oz_product(h, Mc, cnt, ng, neig, h->MBbuf))) return s;
            } else {
                CK(h, gw::launch_zgemm(Mc, (const double2 *)basis, h->MBbuf, cnt, ng, neig, h->st), "projection");
            }
        }
        {
            Scope sc(h, "delta");
            CK(h, gw::launch_delta(v.energy, h->cond.energy, h->cond.nb, p0, cnt, om, h->dbuf, h->st), "delta");
        }
        if ((s = contract_chunk(h, h->MBbuf, cnt, neig, h->dbuf, cnt, nw, (double2 *)chi_sub))) return s;
    }
    Scope sc(h, "symmetrize");
    CK(h, gw::launch_symmetrize((double2 *)chi_sub, neig, nw, h->st), "symmetrize");
    return GW_OK;
}

gw_status gw_chi0_compute_subspace(gw_chi0 *h, int iq, int neig, const double *basis, int nw, const double *omega,
                                   double *chi_sub)
{
    if (!h) return GW_ERR_ARG;
    return zd_or_fft(h, [&] { return compute_subspace(h, iq, neig, basis, nw, omega, chi_sub); });
}

// ------------------------------------------------------------------ dielectric matrix inverse
// Dense product C = A B of two [n][n] complex matrices in the handle's precision mode.
static gw_status square_product(gw_chi0 *h, const double2 *A, const double2 *B, int n, double2 *C, int nslices = 0)
{
    if (h->d.prec == GW_PREC_OZAKI_BF16) {
        gw_status st = oz_prepare_b(h, B, n, n, nslices);
        if (st) return st;
        return oz_product(h, A, n, n, n, C, nslices);
    }
    CK(h, gw::launch_zgemm(A, B, C, n, n, n, h->st), "product");
    return GW_OK;
}

// Slices of the split products of the last Newton-Schulz steps (the most the digit step takes), the
// residual ||I - A X||_F from which one more of them ends at rounding, and the residual from which the
// early steps count as lost.
constexpr int kEpsFinalSlices = 8;
constexpr double kEpsNear = 1e-4, kEpsLost = 0.5;

// Accuracy (the ABI's nslices) of a step that starts at ||I - A X|| <= rho, which it squares: the least
// whose products change the residual by no more than a quarter of that and a quarter of its distance to 1
// (the residual has to keep falling), or than 2e-5, which the last two steps bring to 1e-19.  With n 9-bit
// slices an entry of a product of two N x N matrices carries about N^(1/2) 2^(-9n) of its row's and
// column's largest entries, the matrix N^(1/2) times that, and the residual ||A|| <= b times it; the
// factor 8 covers the step's two products.  That is what digits without a pattern leave, not a bound:
// equal entries can add up their errors.  So the residual that the early steps did reach is measured
// (epsilon_split).
static int eps_step_slices(const gw_chi0 *h, int ng, double b, double *rho)
{
    const double next = *rho * *rho;
    for (int nslices : {4, 5}) { // three and four slices
        const double f = 8.0 * ng * b * std::ldexp(1.0, -9 * gw::oz_slices(nslices));
        if (nslices < h->d.nslices && f <= std::max(0.25 * std::min(next, 1.0 - next), 2e-5)) {
            *rho = next + f;
            return nslices;
        }
    }
    *rho = next;
    return 0;
}

// X <- 2 X - X A X (T, Pm: work), products with the accuracy of nslices (0: the handle's).
// resid: where to leave ||I - A X||_F^2 of the X before the step (device), or null.
static gw_status eps_newton(gw_chi0 *h, const double2 *A, double2 *X, double2 *T, double2 *Pm, int ng, int nslices,
                            double *resid)
{
    Scope sp(h, "eps_products"); // two N_G^3 products per step: the launch count gives the steps
    gw_status st;
    if ((st = square_product(h, A, X, ng, T, nslices))) return st;
    if (resid) CK(h, gw::launch_eps_resid(T, ng, resid, h->st), "residual");
    if ((st = square_product(h, X, T, ng, Pm, nslices))) return st;
    CK(h, gw::launch_eps_step(X, Pm, (int64_t)ng * ng, h->st), "Newton-Schulz step");
    return GW_OK;
}

// Split precision: steps - 2 steps with no more slices than their error asks for, then steps with the most,
// each from a measured residual, until one has started below kEpsNear, and a last one.  The error of the
// result is the rounding of the last two (earlier errors are squared away).  Where the early steps lost
// the iterate they are taken again, from X0, with the most slices.  N_G = 2000, b = 52, two frequencies: six of
// eleven steps with three slices (6 products each), three with four (10), two with six (21), where nine had
// five (15): 30.2 -> 23.4 ms (21.8 with the column slices and the stores of the products as they are now).
// b = 374: four of fourteen steps with three slices, seven with four, 16.2 ms a frequency.
static gw_status epsilon_split(gw_chi0 *h, int ng, double b, int steps, const double2 *A, double2 *X, double2 *T,
                               double2 *Pm, double *resid, const unsigned long long *bmax)
{
    gw_status st;
    double rho = (b - 1.0) / (b + 1.0);
    for (int k = 0; k < steps - 2; ++k)
        if ((st = eps_newton(h, A, X, T, Pm, ng, eps_step_slices(h, ng, b, &rho), nullptr))) return st;
    bool again = false;
    for (int k = 0; k < steps; ++k) {
        double e2 = 0.0;
        if ((st = eps_newton(h, A, X, T, Pm, ng, kEpsFinalSlices, resid))) return st;
        CK(h, cudaMemcpyAsync(&e2, resid, sizeof e2, cudaMemcpyDeviceToHost, h->st), "residual");
        CK(h, cudaStreamSynchronize(h->st), "residual");
        const double e = std::sqrt(e2);
        if (e <= kEpsNear || (again && !(e < kEpsLost))) break;
        if (!(e < kEpsLost)) {
            again = true;
            CK(h, gw::launch_eps_init(X, ng, bmax, h->st), "X0");
            for (int j = 0; j < steps - 2; ++j)
                if ((st = eps_newton(h, A, X, T, Pm, ng, kEpsFinalSlices, nullptr))) return st;
        }
    }
    return eps_newton(h, A, X, T, Pm, ng, kEpsFinalSlices, nullptr);
}

gw_status gw_chi0_epsilon_inverse(gw_chi0 *h, int ng, int nw, const double *chi, const double *vcoul,
                                  double *epsinv)
{
    if (!h) return GW_ERR_ARG;
    if (ng < 1 || nw < 1 || !chi || !vcoul || !epsinv) return fail(h, GW_ERR_ARG, "bad arguments");
    {
        std::vector<double> v(ng);
        CK(h, cudaMemcpyAsync(v.data(), vcoul, sizeof(double) * ng, cudaMemcpyDeviceToHost, h->st), "read v");
        CK(h, cudaStreamSynchronize(h->st), "read v");
        for (int i = 0; i < ng; ++i)
            if (!(v[i] > 0.0) || !std::isfinite(v[i])) return fail(h, GW_ERR_ARG, "v[%d] must be finite and > 0", i);
    }
    const size_t nn = (size_t)ng * ng;
    gw_status st = grow(h, &h->epsbuf, &h->epscap, sizeof(double2) * 4 * nn + sizeof(double) * ng + 64,
                        "dielectric work");
    if (st) return st;
    double2 *A = (double2 *)h->epsbuf, *X = A + nn, *T = X + nn, *Pm = T + nn;
    double *sv = (double *)(Pm + nn);
    unsigned long long *bmax = (unsigned long long *)(((uintptr_t)(sv + ng) + 15) & ~(uintptr_t)15);
    CK(h, gw::launch_eps_sqrt(vcoul, ng, sv, h->st), "sqrt v");
    for (int w = 0; w < nw; ++w) {
        Scope sc(h, "epsilon_inverse");
        CK(h, gw::launch_eps_sym((const double2 *)chi + (int64_t)w * nn, sv, ng, A, bmax, h->st), "I - s chi s");
        unsigned long long bits = 0;
        CK(h, cudaMemcpyAsync(&bits, bmax, sizeof bits, cudaMemcpyDeviceToHost, h->st), "bound");
        CK(h, cudaStreamSynchronize(h->st), "bound");
        double b;
        std::memcpy(&b, &bits, sizeof b);
        if (!(b >= 1.0) || !std::isfinite(b)) return fail(h, GW_ERR_ARG, "I - v chi is not positive (bound %g)", b);
        // steps for (b - 1)/(b + 1) squared repeatedly to reach 1e-17, plus one for rounding
        const double r = (b - 1.0) / (b + 1.0);
        int steps = 1;
        if (r > 0.0) steps = (int)std::ceil(std::log2(std::log(1e-17) / std::log(r))) + 1;
        steps = std::max(steps, 1);
        CK(h, gw::launch_eps_init(X, ng, bmax, h->st), "X0");
        if (h->d.prec == GW_PREC_OZAKI_BF16) {
            if ((st = epsilon_split(h, ng, b, steps, A, X, T, Pm, (double *)(bmax + 1), bmax))) return st;
        } else {
            for (int k = 0; k < steps; ++k)
                if ((st = eps_newton(h, A, X, T, Pm, ng, 0, nullptr))) return st;
        }
        CK(h, gw::launch_eps_unsym(X, sv, ng, (double2 *)epsinv + (int64_t)w * nn, h->st), "s X s^-1");
    }
    return GW_OK;
}

// ------------------------------------------------------------------ real frequencies
static gw_status compute_real(gw_chi0 *h, int iq, int nw, const double *omega, double eta, double *chi)
{
    if (nw < 1 || 3 * nw > gw::kMaxOmega || !omega || !chi)
        return fail(h, GW_ERR_ARG, "bad arguments (1 <= nw <= %d, non-null pointers)", gw::kMaxOmega / 3);
    if (!(eta > 0.0) || !std::isfinite(eta)) return fail(h, GW_ERR_ARG, "eta must be finite and > 0");
    gw::OmegaList om;
    om.nw = nw;
    for (int i = 0; i < nw; ++i) {
        if (!(omega[i] >= 0.0) || !std::isfinite(omega[i])) return fail(h, GW_ERR_ARG, "omega must be finite and >= 0");
        om.w[i] = omega[i];
    }
    gw_status s = check_slot(h, iq);
    if (s) return s;
    const Sphere &sp = h->sph[iq];
    const BandSet &v = h->val[iq];
    const int ng = sp.ng;
    const int64_t nn = (int64_t)ng * ng;
    const int64_t P = (int64_t)v.nb * h->cond.nb;
    const double2 *Mres = resident_for(h, iq); // kept by the last gw_chi0_compute of this slot
    ZdPlan z;
    ZdUse use{h};
    const size_t parts = sizeof(double2) * 3 * nw * nn, pending = parts > h->realcap ? parts - h->realcap : 0;
    if (!Mres && ((s = zd_plan(h, sp, v.nb, h->cond.nb, true, false, 1, 3 * nw, pending,
                              std::min<int64_t>(h->d.pair_chunk, P), z)) ||
                  (z.on && ((s = zd_valence(h, z, sp, v.psi, v.nb)) || (s = zd_conduction(h, z, h->cond.psi, 0, h->cond.nb))))))
        return s;
    const int64_t chunk = z.on ? (int64_t)z.vb * z.cb : std::min<int64_t>(h->d.pair_chunk, P);
    if ((s = grow(h, (void **)&h->realbuf, &h->realcap, parts, "real-axis parts")) ||
        (s = ensure_work(h, (size_t)chunk * ng, (size_t)chunk * 3 * nw)))
        return s;
    CK(h, cudaMemsetAsync(h->realbuf, 0, parts, h->st), "zero parts");
    gw::PairPlan pp = pair_plan(h, sp);
    for (int64_t p0 = 0; p0 < P; p0 += chunk) {
        const int64_t cnt = std::min(chunk, P - p0);
        const double2 *Mc = Mres ? Mres + p0 * ng : h->Mbuf;
        if (!Mres && (s = pair_rows(h, z, sp, pp, v.psi, h->cond.psi, h->cond.nb, p0, cnt, h->Mbuf))) return s;
        {
            Scope sc(h, "delta");
            CK(h, gw::launch_delta_real(v.energy, h->cond.energy, h->cond.nb, p0, cnt, om, eta, h->dbuf, h->st),
               "real-axis delta");
        }
        if ((s = contract_chunk(h, Mc, cnt, ng, h->dbuf, cnt, 3 * nw, h->realbuf))) return s;
    }
    Scope sc(h, "symmetrize");
    CK(h, gw::launch_symmetrize(h->realbuf, ng, 3 * nw, h->st), "symmetrize");
    CK(h, gw::launch_combine_real(h->realbuf, nn, nw, (double2 *)chi, h->st), "combine");
    return GW_OK;
}

gw_status gw_chi0_compute_real(gw_chi0 *h, int iq, int nw, const double *omega, double eta, double *chi)
{
    if (!h) return GW_ERR_ARG;
    return zd_or_fft(h, [&] { return compute_real(h, iq, nw, omega, eta, chi); });
}

// ------------------------------------------------------------------ forward derivative (JVP)
// Real-space grids of caller coefficients on a stored band set's plane waves (the band
// setup of gw_chi0_set_bands, into psi).
static gw_status band_grids(gw_chi0 *h, const BandSet &b, const double *coeff, void *psi)
{
    CK(h, cudaMemsetAsync(psi, 0, sizeof(double2) * (size_t)b.nb * h->nr, h->st), "zero grids");
    if (h->d.mtxel_prec == GW_MTXEL_TWOFLOAT) {
        Scope sc(h, "band_setup_tf");
        CK(h, gw::launch_band_setup_tf((const double2 *)coeff, b.gofs, b.nb, b.ngpsi, psi, h->d.n, h->ax, b.maxabs,
                                       h->st),
           "tangent band setup (two-float)");
    } else {
        CK(h, gw::launch_scatter((const double2 *)coeff, b.gofs, b.nb, b.ngpsi, h->nr, (double2 *)psi, h->st),
           "tangent scatter");
        CK(h, gw::launch_band_fft((double2 *)psi, b.nb, h->d.n, h->ax, h->st), "tangent band fft");
    }
    return GW_OK;
}

static gw_status jvp(gw_chi0 *h, int iq, int nw, const double *omega, const double *dcoeff_v,
                     const double *dcoeff_c, const double *dE_v, const double *dE_c, double *dchi)
{
    if (nw < 1 || 2 * nw > gw::kMaxOmega || !omega || !dcoeff_v || !dcoeff_c || !dE_v || !dE_c || !dchi)
        return fail(h, GW_ERR_ARG, "bad arguments (1 <= nw <= %d, non-null pointers)", gw::kMaxOmega / 2);
    gw::OmegaList om;
    om.nw = nw;
    for (int i = 0; i < nw; ++i) {
        if (!(omega[i] >= 0.0) || !std::isfinite(omega[i])) return fail(h, GW_ERR_ARG, "omega must be finite and >= 0");
        om.w[i] = omega[i];
    }
    gw_status s = check_slot(h, iq);
    if (s) return s;
    const BandSet &v = h->val[iq];
    const BandSet &c = h->cond;
    const Sphere &sp = h->sph[iq];
    const int ng = sp.ng, nc = c.nb;
    const int64_t nn = (int64_t)ng * ng;
    const int64_t P = (int64_t)v.nb * nc;
    // work held only for this call
    const size_t szv = sizeof(double2) * (size_t)v.nb * h->nr, szc = sizeof(double2) * (size_t)nc * h->nr;
    const size_t szt = sizeof(double2) * 4 * nw * nn;
    ZdPlan z; // side 0: the stored bands, side 1: the tangents
    ZdUse use{h};
    if ((s = zd_plan(h, sp, v.nb, nc, true, false, 2, 2 * nw, szv + szc + szt,
                     std::min<int64_t>(h->d.pair_chunk, P), z))) return s;
    const int64_t chunk = z.on ? (int64_t)z.vb * z.cb : std::min<int64_t>(h->d.pair_chunk, P);
    void *gv = nullptr, *gc = nullptr;
    double2 *X1 = nullptr, *X2 = nullptr, *T = nullptr;
    double *wb = nullptr;
    const size_t szx = sizeof(double2) * (size_t)chunk * ng;
    const size_t szw = sizeof(double) * 2 * nw * (size_t)chunk;
    auto cleanup = [&]() {
        cudaStreamSynchronize(h->st);
        dfree(h, gv, szv);
        dfree(h, gc, szc);
        dfree(h, X1, szx);
        dfree(h, X2, szx);
        dfree(h, T, szt);
        dfree(h, wb, szw);
    };
    if ((s = dalloc(h, &gv, szv, "tangent valence grids")) || (s = dalloc(h, &gc, szc, "tangent conduction grids")) ||
        (s = dalloc(h, (void **)&X1, szx, "tangent pairs")) || (s = dalloc(h, (void **)&X2, szx, "tangent pairs")) ||
        (s = dalloc(h, (void **)&T, szt, "tangent parts")) || (s = dalloc(h, (void **)&wb, szw, "tangent weights")) ||
        (s = ensure_work(h, (size_t)chunk * ng, (size_t)chunk * 2 * nw)) || (s = band_grids(h, v, dcoeff_v, gv)) ||
        (s = band_grids(h, c, dcoeff_c, gc)) ||
        (z.on && ((s = zd_valence(h, z, sp, v.psi, v.nb, 0)) || (s = zd_valence(h, z, sp, gv, v.nb, 1)) ||
                  (s = zd_conduction(h, z, c.psi, 0, nc, 0)) || (s = zd_conduction(h, z, gc, 0, nc, 1))))) {
        cleanup();
        return s;
    }
#define JCK(x, what)                            \
    do {                                        \
        cudaError_t e_ = (x);                   \
        if (e_ != cudaSuccess) {                \
            gw_status r_ = cuda_fail(h, e_, what); \
            cleanup();                          \
            return r_;                          \
        }                                       \
    } while (0)
    JCK(cudaMemsetAsync(T, 0, szt, h->st), "zero parts");
    double2 *Tp = T, *Tm = T + (int64_t)nw * nn, *Tw = T + 2 * (int64_t)nw * nn;
    gw::PairPlan pp = pair_plan(h, sp);
    const double2 *Mres = resident_for(h, iq); // kept by the last gw_chi0_compute of this slot
    for (int64_t p0 = 0; p0 < P; p0 += chunk) {
        const int64_t cnt = std::min(chunk, P - p0);
        const double2 *Mc = Mres ? Mres + p0 * ng : h->Mbuf;
        if ((!Mres && (s = pair_rows(h, z, sp, pp, v.psi, c.psi, nc, p0, cnt, h->Mbuf))) ||
            (s = pair_rows(h, z, sp, pp, gv, c.psi, nc, p0, cnt, X1, 1, 0)) ||
            (s = pair_rows(h, z, sp, pp, v.psi, gc, nc, p0, cnt, X2, 0, 1))) {
            cleanup();
            return s;
        }
        {
            Scope sc(h, "jvp_mix");
            JCK(gw::launch_jvp_mix(Mc, X1, X2, cnt * ng, h->st), "M +- dM");
        }
        {
            Scope sc(h, "delta");
            JCK(gw::launch_delta(v.energy, c.energy, nc, p0, cnt, om, h->dbuf, h->st), "delta");
            JCK(gw::launch_delta_jvp(v.energy, c.energy, dE_v, dE_c, nc, p0, cnt, om, wb, h->st), "delta derivative");
        }
        // d chi = [chi(M + dM) - chi(M - dM)] / 2 + sum_p conj(M) dDelta M
        if ((s = contract_chunk(h, X1, cnt, ng, h->dbuf, cnt, nw, Tp)) ||
            (s = contract_chunk(h, X2, cnt, ng, h->dbuf, cnt, nw, Tm)) ||
            (s = contract_chunk(h, Mc, cnt, ng, wb, cnt, 2 * nw, Tw))) {
            cleanup();
            return s;
        }
    }
    {
        Scope sc(h, "symmetrize");
        JCK(gw::launch_symmetrize(T, ng, 4 * nw, h->st), "symmetrize");
        JCK(gw::launch_combine_jvp(Tp, Tm, Tw, nn, nw, (double2 *)dchi, h->st), "combine");
    }
#undef JCK
    cleanup();
    return GW_OK;
}

gw_status gw_chi0_jvp(gw_chi0 *h, int iq, int nw, const double *omega, const double *dcoeff_v,
                      const double *dcoeff_c, const double *dE_v, const double *dE_c, double *dchi)
{
    if (!h) return GW_ERR_ARG;
    return zd_or_fft(h, [&] { return jvp(h, iq, nw, omega, dcoeff_v, dcoeff_c, dE_v, dE_c, dchi); });
}
