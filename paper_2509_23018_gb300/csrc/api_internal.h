// Host side of the C ABI declared in include/gw_chi0.h: the handle, its band sets and
// spheres, and the helpers shared by api.cu (handle, setup, streamed path, status and
// timing), api_batch.cu (the batched graph path) and api_ext.cu (adjoint, static subspace,
// dielectric inverse, real axis, forward derivative).  Not part of the public interface.
#pragma once
#include "../../include/gw_chi0.h"
#include "internal.h"
#include "sphere_plan.h"

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cusolverDn.h>
#include <dlfcn.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <array>
#include <map>
#include <string>
#include <vector>

using gw::FftAxis;

namespace gwapi {
using gw::FftAxis;
struct BandSet {
    int nb = 0, ngpsi = 0;
    double2 *psi = nullptr;     // [nb][N_r]
    double *energy = nullptr;   // [nb] device copy
    int32_t *gvec = nullptr;    // [ngpsi][3] device copy (adjoint)
    int32_t *gofs = nullptr;    // [ngpsi] grid offsets
    std::vector<int32_t> g;     // host copy
    std::vector<double> e;      // host copy
    int maxabs[3] = {0, 0, 0};
};

struct Sphere {
    int ng = 0;
    std::vector<int32_t> g;
    int maxabs[3] = {0, 0, 0};
    int K2 = 0;
    int *kz = nullptr;          // device [K2]
    int32_t *gpack = nullptr;   // device [ng]
    int32_t *gvec = nullptr;    // device [ng][3]
    std::vector<int> cstart, cg; // (k1, k2) cells of the sphere, CSR (adjoint back-projection)
    int K12 = 0;                // number of cells
    int32_t *cell = nullptr;    // device [K12]  k2index << 8 | k1
    int *cstart_d = nullptr;    // device [K12 + 1] (cstart)
    int2 *cpts = nullptr;       // device [ng]   (point, k0 | cell << 8) in cell order
    int nslots = 0;             // scratch slots the two-float pair kernel needs (0: none)
};

struct TimerRec {
    std::string name;
    cudaEvent_t a, b;
};
} // namespace gwapi

using gwapi::BandSet;
using gwapi::Sphere;
using gwapi::TimerRec;

struct gw_chi0 {
    gw_chi0_desc d{};
    cudaStream_t st = nullptr;
    std::string err;
    int64_t nr = 0;
    FftAxis ax[3]{};
    double2 *tw = nullptr;
    float4 *twf = nullptr;
    BandSet cond;
    std::vector<BandSet> val;
    std::vector<Sphere> sph;
    double2 *Mbuf = nullptr;
    size_t Mcap = 0; // elements
    double *dbuf = nullptr;
    size_t dcap = 0;
    // split-precision work buffers
    void *Zbuf = nullptr;      // bf16 slices [s][2 ng][kpad]
    int *f64guard = nullptr;   // set by the slicing kernels where the sliced FP64 contraction does not hold
    size_t f64guard_cap = 0;
    bool zbusy = false;        // Zbuf is in use by the call that allocates (see dalloc)
    size_t Zcap = 0;           // bytes
    double *spbuf = nullptr;   // sqrt(-Delta) [nw][chunk]
    size_t spcap = 0;
    int *Ebuf = nullptr;       // column exponents [ng]
    size_t Ecap = 0;
    double *ozpart = nullptr;  // sums of the parts of split tiles (contraction launches run one at a time)
    size_t ozpart_cap = 0;
    int *ozflags = nullptr;    // their counters
    size_t ozflags_cap = 0;
    void *jobbuf = nullptr;    // job tables of the batched contraction kernels
    size_t jobcap = 0;
    // contraction launch shapes (set by the autotuner; these are the defaults)
    int tuned_bt = 64, tuned_waves = 4;
    std::map<std::string, std::array<int, 2>> tune_cache; // signature -> (bt, waves)
    // batched path: every slot's M resident, one graph per call signature
    double2 *Mall = nullptr;
    size_t Mall_cap = 0;
    double *Dall = nullptr, *SPall = nullptr;
    size_t Dall_cap = 0, SPall_cap = 0;
    void *Zall = nullptr;
    size_t Zall_cap = 0;
    int *Eall = nullptr;
    size_t Eall_cap = 0;
    cudaStream_t cap_st = nullptr;
    // overlapped streamed path: contractions on a high-priority second stream, buffers by parity
    cudaStream_t ov_st = nullptr;
    cudaEvent_t ov_split[2] = {nullptr, nullptr}, ov_gemm[2] = {nullptr, nullptr};
    void *ovZ[2] = {nullptr, nullptr};
    size_t ovZcap[2] = {0, 0};
    int *ovE[2] = {nullptr, nullptr};
    size_t ovEcap[2] = {0, 0};
    void *ovJ[2] = {nullptr, nullptr};
    size_t ovJcap[2] = {0, 0};
    struct Graph {
        std::string key;
        cudaGraphExec_t exec = nullptr;
        void *jobs = nullptr;
        size_t jobs_bytes = 0;
    };
    std::vector<Graph> graphs;
    int *status = nullptr;
    // split-precision general products (subspace projection, adjoint Y = M W)
    int *EAbuf = nullptr, *EBbuf = nullptr;
    size_t EAcap = 0, EBcap = 0;
    void *ZBbuf = nullptr;      // B operand slices [s][2 nout][kpad]
    size_t ZBcap = 0;
    double2 *MBbuf = nullptr;   // projected pair elements of a chunk [chunk][neig]
    size_t MBcap = 0;
    void *epsbuf = nullptr;     // dielectric inverse: A, X, T, P [ng][ng], sqrt(v) [ng], bound
    size_t epscap = 0;
    double2 *realbuf = nullptr; // real-axis chi: the three Hermitian parts per frequency
    size_t realcap = 0;
    // dense eigensolver (cuSOLVER, loaded on first use) for the subspace basis
    struct {
        void *lib = nullptr;
        cusolverDnHandle_t hdl = nullptr;
        decltype(&cusolverDnCreate) create = nullptr;
        decltype(&cusolverDnDestroy) destroy = nullptr;
        decltype(&cusolverDnSetStream) set_stream = nullptr;
        decltype(&cusolverDnZheevdx_bufferSize) buffer_size = nullptr;
        decltype(&cusolverDnZheevdx) heevdx = nullptr;
    } sol;
    double2 *eigA = nullptr, *eigWork = nullptr;
    double *eigW = nullptr;
    int *eigInfo = nullptr;
    size_t eigA_cap = 0, eigWork_cap = 0, eigW_cap = 0, eigInfo_cap = 0;
    // pair elements of one slot kept resident between calls (gw_chi0_keep_pair_elements): written
    // by gw_chi0_compute, reused by gw_chi0_compute_subspace / gw_chi0_compute_real
    bool keep_m = false;
    double2 *Mres = nullptr;
    size_t Mres_cap = 0; // bytes
    int Mres_iq = -1;    // slot whose elements the buffer holds; -1: none
    // plasmon-pole self-energy work buffers (api_sigma.cu)
    struct Buf {
        void *p = nullptr;
        size_t cap = 0;
    } gpp[9];
    // stage (a) with the last-axis transform on the tensor cores (zdft.cu): row slices of a conduction
    // block and column exponents of the valence bands (two of each: the forward derivative has
    // tangent grids too), and the transform output F of a sub-block
    void *zdA[2] = {nullptr, nullptr};
    size_t zdAcap[2] = {0, 0}; // bytes
    int *zdE[2] = {nullptr, nullptr};
    size_t zdEcap[2] = {0, 0}; // bytes
    float4 *zdF = nullptr;
    size_t zdFcap = 0;         // bytes
    float4 *zdS = nullptr;     // cells between the middle- and first-axis kernels, where they are two
    size_t zdScap = 0;         // bytes
    bool zdbusy = false;       // a call has planned with these buffers (ZdUse)
    bool zdran = false;        // a plan of this call took the route, and
    bool zdoff = false;        // none may (zd_or_fft)
    int *zdguard = nullptr;    // FP64: set where the slices do not hold and the FFT kernel takes over
    size_t zdguard_cap = 0;
    // scratch slots of the two-float pair kernel (sized in set_gsphere, outside any capture)
    float4 *pscr = nullptr;
    size_t pscr_cap = 0; // bytes
    int *pflags = nullptr;
    size_t pflags_cap = 0; // bytes
    size_t bytes = 0;
    PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    // timing
    bool timing = false;
    std::vector<TimerRec> pending;
    std::vector<cudaEvent_t> pool;
    std::map<std::string, std::pair<double, int64_t>> acc;
};

namespace gwapi {

#define CK(h, x, what)                                   \
    do {                                                 \
        cudaError_t e_ = (x);                            \
        if (e_ != cudaSuccess) return cuda_fail(h, e_, what); \
    } while (0)

cudaEvent_t ev_get(gw_chi0 *h);

// Per-kernel timing: events around the enqueued work when the handle's timing is on.
struct Scope {
    gw_chi0 *h;
    const char *name;
    cudaStream_t s;
    cudaEvent_t a = nullptr;
    Scope(gw_chi0 *h_, const char *n, cudaStream_t s_ = nullptr) : h(h_), name(n), s(s_ ? s_ : h_->st)
    {
        if (h->timing) {
            a = ev_get(h);
            cudaEventRecord(a, s);
        }
    }
    ~Scope()
    {
        if (h->timing) {
            cudaEvent_t b = ev_get(h);
            cudaEventRecord(b, s);
            h->pending.push_back({name, a, b});
        }
    }
};

gw_status fail(gw_chi0 *h, gw_status s, const char *fmt, ...);
gw_status cuda_fail(gw_chi0 *h, cudaError_t e, const char *what);
gw_status dalloc(gw_chi0 *h, void **p, size_t n, const char *what);
void dfree(gw_chi0 *h, void *p, size_t n);
bool factor(int n, FftAxis &a);
int mod(int a, int n);
void drain_timing(gw_chi0 *h);
gw_status ensure_work(gw_chi0 *h, size_t m_elems, size_t d_elems);
gw_status make_tmap(gw_chi0 *h, CUtensorMap *map, const void *M, int64_t P, int ng, int bt);
int num_sms();
void drop_graphs(gw_chi0 *h);
gw_status grow(gw_chi0 *h, void **p, size_t *cap, size_t bytes, const char *what);
gw_status upload_jobs(gw_chi0 *h, const void *src, size_t bytes, const void **dev);
gw_status f64_jobs(gw_chi0 *h, std::vector<gw::F64Job> &jobs, const double2 *M, int64_t P, int ng,
                   const double *delta, int64_t dstride, int nw, double2 *chi, int bt);
int f64_schedule(std::vector<gw::F64Job> &jobs, int waves);
gw_status launch_f64_jobs(gw_chi0 *h, std::vector<gw::F64Job> &jobs, int bt, int waves, const int *guard = nullptr);
gw_status make_tmap_z(gw_chi0 *h, CUtensorMap *map, void *Z, int64_t kpad, int nrows, int s, int box_rows);
// nslices: 9-bit slices, 0 for the handle's
gw_status oz_job(gw_chi0 *h, gw::OzJob &j, void *Z, int64_t kpad, int ng, const int *E, double2 *chi, int nslices = 0);
int oz_clusters(size_t nitems);
gw_status oz_items(gw_chi0 *h, std::vector<gw::OzJob> &jobs, std::vector<gw::OzItem> &items);
inline gw::OzScratch oz_scratch(const gw_chi0 *h) { return {h->ozpart, h->ozflags}; }
gw_status launch_oz_general(gw_chi0 *h, const std::vector<gw::OzJob> &jobs);
gw_status launch_oz_jobs(gw_chi0 *h, std::vector<gw::OzJob> &jobs, const int *guard = nullptr);
gw_status contract_chunk_ozaki(gw_chi0 *h, const double2 *M, int64_t P, int ng, const double *delta, int64_t dstride,
                               int nw, double2 *chi);
// given: M comes from the caller of the API rather than from the bands
gw_status contract_chunk(gw_chi0 *h, const double2 *M, int64_t P, int ng, const double *delta, int64_t dstride,
                         int nw, double2 *chi, bool given = false);
int64_t oz_kpad(int ka);
cudaError_t launch_oz_columns(const double2 *B, int ka, int nout, int64_t ldb, int s, int64_t kpad, void *Z, int *E,
                              cudaStream_t st);
// nslices > 0 overrides the handle's slice count (both calls of one product must agree)
gw_status oz_prepare_b(gw_chi0 *h, const double2 *B, int ka, int nout, int nslices = 0);
gw_status oz_product(gw_chi0 *h, const double2 *A, int64_t rows, int ka, int nout, double2 *Y, int nslices = 0);
bool alias_free(const gw_chi0 *h, const BandSet &v, const BandSet &c, const Sphere &s, int *axis);
gw_status check_slot(gw_chi0 *h, int iq);
cudaError_t run_pair(gw_chi0 *h, const void *psiv, const void *psic, int nc, int64_t p0, int64_t cnt,
                     const gw::PairPlan &pp, double2 *M);
gw::PairPlan pair_plan(gw_chi0 *h, const Sphere &s);
void free_bands(gw_chi0 *h, BandSet &b);
void free_sphere(gw_chi0 *h, Sphere &s);

// resident pair elements: resident_begin makes room for slot iq's P x ng elements when keeping is
// on and they fit (*use), invalidating what the buffer held; resident_for(h, iq) is the buffer when
// it holds slot iq, else null
gw_status resident_begin(gw_chi0 *h, int64_t P, int ng, bool *use);
double2 *resident_for(gw_chi0 *h, int iq);
// overlapped split-precision streamed compute of one slot (api.cu); Mres: resident output or null
gw_status compute_overlap(gw_chi0 *h, int iq, const gw::OmegaList &om, double2 *cq, double *dq, double2 *Mres);
// Stage (a) on the tensor cores for one call.  zd_plan: blocks of vb x cb pairs (rows: cb = nc, whole
// valence rows in pair order) and the buffers for `sides` sets of bands; on = false when the route
// does not take the sphere, would be slower (unless forced) or lacks memory.  zd_valence /
// zd_conduction prepare a side's bands; zd_block forms M[(v - v0) sv + c sc] of a block.
struct ZdPlan {
    bool on = false;
    bool f64 = false;                                  // FP64 (zdft64.cu), two-float otherwise
    int vb = 0, cb = 0, vs = 0;                        // vs: valence bands per sub-block
    size_t abytes = 0, ebytes = 0, fper = 0, sper = 0; // row slices, exponents; F and cells of one valence band
    int nv[2] = {0, 0};
    CUtensorMap tmV[2];
    const void *psiv[2] = {nullptr, nullptr}, *psic[2] = {nullptr, nullptr}; // each side's bands, as last prepared
};
// The route's buffers stay until the call that planned with them returns; between calls they make room
// for what others need (dalloc).
struct ZdUse {
    gw_chi0 *h;
    ~ZdUse() { h->zdbusy = false; }
};
// pending: bytes that the call will still allocate beside its chunk's pair elements, weights and slices;
// launch: pairs that the FFT kernel would take at once
gw_status zd_plan(gw_chi0 *h, const Sphere &sp, int nv, int nc, bool rows, bool force, int sides, int nw,
                  size_t pending, int64_t launch, ZdPlan &z);
// A call that plans: one that runs out of memory beside the route's buffers is made again without them.
template <class F>
gw_status zd_or_fft(gw_chi0 *h, F body)
{
    h->zdran = false;
    gw_status s = body();
    if (s != GW_ERR_OOM || !h->zdran) return s;
    h->zdoff = true;
    s = body();
    h->zdoff = false;
    return s;
}
bool zd_holds(const gw_chi0 *h, const ZdPlan &z); // side 0 and F as planned (a later plan may have lost them)
gw_status zd_valence(gw_chi0 *h, ZdPlan &z, const Sphere &sp, const void *psiv, int nv, int side = 0);
gw_status zd_conduction(gw_chi0 *h, ZdPlan &z, const void *psic, int c0, int cb, int side = 0);
gw_status zd_block(gw_chi0 *h, const ZdPlan &z, const Sphere &sp, const gw::PairPlan &pp, int vside, int cside, int v0,
                   int vb, int cb, double2 *M, int64_t sv, int64_t sc);
gw_status pair_rows(gw_chi0 *h, const ZdPlan &z, const Sphere &sp, const gw::PairPlan &pp, const void *psiv,
                    const void *psic, int nc, int64_t p0, int64_t cnt, double2 *M, int vside = 0, int cside = 0);
bool overlap_enabled(gw_chi0 *h, const Sphere &sp, const gw::PairPlan &pp, bool keep);

// batched path (api_batch.cu)
gw_status compute_batch(gw_chi0 *h, int nq, const int *iq, int nw, const double *omega, const gw::OmegaList &om,
                        double *chi, double *diag);

} // namespace gwapi
