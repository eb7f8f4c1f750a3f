// Host side of the C ABI declared in include/gw_chi0.h: handle state, validation,
// library-owned device memory, per-chunk orchestration and optional per-kernel timing.
#include "api_internal.h"

namespace gwapi {
gw_status fail(gw_chi0 *h, gw_status s, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (h) h->err = buf;
    return s;
}

gw_status cuda_fail(gw_chi0 *h, cudaError_t e, const char *what)
{
    return fail(h, e == cudaErrorMemoryAllocation ? GW_ERR_OOM : GW_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}



gw_status dalloc(gw_chi0 *h, void **p, size_t n, const char *what)
{
    if (n == 0) n = 16;
    // the buffers of stage (a) on the tensor cores and FP64 mode's slices are an optimisation: between
    // the calls that use them they make room for what another needs
    auto reclaim = [&] {
        const size_t held = h->bytes;
        auto give = [&](auto *&b, size_t &cap) {
            if (!b) return;
            drop_graphs(h);
            dfree(h, b, cap);
            b = nullptr;
            cap = 0;
        };
        if (h->d.prec == GW_PREC_FP64 && !h->zbusy) give(h->Zbuf, h->Zcap);
        if (!h->zdbusy) {
            for (int i = 0; i < 2; ++i) {
                give(h->zdA[i], h->zdAcap[i]);
                give(h->zdE[i], h->zdEcap[i]);
            }
            give(h->zdF, h->zdFcap);
            give(h->zdS, h->zdScap);
        }
        return h->bytes < held;
    };
    if (h->d.mem_budget_bytes && h->bytes + n > h->d.mem_budget_bytes) reclaim();
    if (h->d.mem_budget_bytes && h->bytes + n > h->d.mem_budget_bytes)
        return fail(h, GW_ERR_OOM, "%s: %zu bytes would exceed the memory budget (%zu held, budget %zu)", what, n,
                    h->bytes, h->d.mem_budget_bytes);
    cudaError_t e = cudaMalloc(p, n);
    if (e != cudaSuccess && reclaim()) {
        cudaGetLastError();
        e = cudaMalloc(p, n);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(h, GW_ERR_OOM, "%s: cudaMalloc(%zu) failed: %s", what, n, cudaGetErrorString(e));
    }
    h->bytes += n;
    return GW_OK;
}

void dfree(gw_chi0 *h, void *p, size_t n)
{
    if (!p) return;
    cudaFree(p);
    h->bytes -= (n == 0 ? 16 : n);
}

// Radices for an n-point line transform: as many 4s as possible, 3s and 5s, a leftover 2
// merged with a 4 into an 8.  Odd radices run first: the first Stockham stage stores with
// a stride of R elements, and a stride of 3 or 5 16-byte elements is free of shared-memory
// bank conflicts where 4 and 8 are not.
bool factor(int n, FftAxis &a)
{
    a.n = n;
    a.nst = 0;
    int m = n, n4 = 0, n2 = 0, n3 = 0, n5 = 0;
    while (m % 4 == 0) { ++n4; m /= 4; }
    while (m % 2 == 0) { ++n2; m /= 2; }
    while (m % 3 == 0) { ++n3; m /= 3; }
    while (m % 5 == 0) { ++n5; m /= 5; }
    if (m != 1) return false;
    int n8 = 0;
    if (n2 && n4) { n2 = 0; --n4; n8 = 1; }
    if (n3 + n5 + n4 + n8 + n2 > gw::kMaxStages) return false;
    for (int i = 0; i < n3; ++i) a.rad[a.nst++] = 3;
    for (int i = 0; i < n5; ++i) a.rad[a.nst++] = 5;
    for (int i = 0; i < n4; ++i) a.rad[a.nst++] = 4;
    for (int i = 0; i < n8; ++i) a.rad[a.nst++] = 8;
    for (int i = 0; i < n2; ++i) a.rad[a.nst++] = 2;
    return true;
}

int mod(int a, int n) { return ((a % n) + n) % n; }

// Host-side fault injection for tests: GW_CHI0_FAULT_AT_CHUNK=k makes the streamed compute
// fail before enqueueing chunk k (nothing faults on the device).
int64_t fault_chunk()
{
    const char *e = std::getenv("GW_CHI0_FAULT_AT_CHUNK");
    return e ? std::atoll(e) : -1;
}

// ------------------------------------------------------------------ timing helpers
cudaEvent_t ev_get(gw_chi0 *h)
{
    if (!h->pool.empty()) {
        cudaEvent_t e = h->pool.back();
        h->pool.pop_back();
        return e;
    }
    cudaEvent_t e;
    cudaEventCreate(&e);
    return e;
}



void drain_timing(gw_chi0 *h)
{
    if (h->pending.empty()) return;
    cudaStreamSynchronize(h->st);
    for (auto &r : h->pending) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, r.a, r.b);
        auto &x = h->acc[r.name];
        x.first += ms;
        x.second += 1;
        h->pool.push_back(r.a);
        h->pool.push_back(r.b);
    }
    h->pending.clear();
}

// ------------------------------------------------------------------ buffers
gw_status ensure_work(gw_chi0 *h, size_t m_elems, size_t d_elems)
{
    if (m_elems > h->Mcap) {
        dfree(h, h->Mbuf, h->Mcap * sizeof(double2));
        h->Mbuf = nullptr;
        h->Mcap = 0;
        gw_status s = dalloc(h, (void **)&h->Mbuf, m_elems * sizeof(double2), "M chunk buffer");
        if (s) return s;
        h->Mcap = m_elems;
    }
    if (d_elems > h->dcap) {
        dfree(h, h->dbuf, h->dcap * sizeof(double));
        h->dbuf = nullptr;
        h->dcap = 0;
        gw_status s = dalloc(h, (void **)&h->dbuf, d_elems * sizeof(double), "Delta buffer");
        if (s) return s;
        h->dcap = d_elems;
    }
    return GW_OK;
}

gw_status make_tmap(gw_chi0 *h, CUtensorMap *map, const void *M, int64_t P, int ng, int bt)
{
    if (((uintptr_t)M & 15) != 0) return fail(h, GW_ERR_ARG, "M must be 16-byte aligned");
    cuuint64_t dims[2] = {(cuuint64_t)2 * ng, (cuuint64_t)P};
    cuuint64_t strides[1] = {(cuuint64_t)2 * ng * sizeof(double)};
    cuuint32_t box[2] = {(cuuint32_t)(2 * bt), (cuuint32_t)gw::contract_f64_bk()};
    cuuint32_t es[2] = {1, 1};
    CUresult r = h->encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<void *>(M), dims, strides, box, es,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(h, GW_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return GW_OK;
}

int num_sms()
{
    int sms = 152, dev;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// Captured graphs hold raw device pointers: drop them whenever a buffer they may use is
// reallocated or the bands or spheres change (they are recaptured on the next call).
void drop_graphs(gw_chi0 *h)
{
    if (h->graphs.empty()) return;
    cudaStreamSynchronize(h->st); // a replay may still be running
    for (auto &g : h->graphs) {
        if (g.exec) cudaGraphExecDestroy(g.exec);
        dfree(h, g.jobs, g.jobs_bytes);
    }
    h->graphs.clear();
}

gw_status grow(gw_chi0 *h, void **p, size_t *cap, size_t bytes, const char *what)
{
    if (bytes <= *cap) return GW_OK;
    if (*p) drop_graphs(h);
    dfree(h, *p, *cap);
    *p = nullptr;
    *cap = 0;
    gw_status s = dalloc(h, p, bytes, what);
    if (s) return s;
    *cap = bytes;
    return GW_OK;
}

// Copy a job table into the handle's job buffer, in stream order (the copy runs after every
// kernel already enqueued, so rewriting the buffer never races a kernel that reads it).
gw_status upload_jobs(gw_chi0 *h, const void *src, size_t bytes, const void **dev)
{
    gw_status s = grow(h, &h->jobbuf, &h->jobcap, bytes, "job table");
    if (s) return s;
    CK(h, cudaMemcpyAsync(h->jobbuf, src, bytes, cudaMemcpyHostToDevice, h->st), "job table upload");
    *dev = h->jobbuf;
    return GW_OK;
}

// FP64 jobs for one M block and nw frequencies; item_start and ksplit filled in by the caller.
gw_status f64_jobs(gw_chi0 *h, std::vector<gw::F64Job> &jobs, const double2 *M, int64_t P, int ng,
                   const double *delta, int64_t dstride, int nw, double2 *chi, int bt)
{
    CUtensorMap map;
    gw_status s = make_tmap(h, &map, M, P, ng, bt);
    if (s) return s;
    for (int w = 0; w < nw; ++w) {
        gw::F64Job j;
        std::memset(&j, 0, sizeof j);
        j.tm = map;
        j.delta = delta + (int64_t)w * dstride;
        j.chi = (double *)(chi + (int64_t)w * ng * ng);
        j.P = P;
        j.ng = ng;
        j.ntile = (ng + bt - 1) / bt;
        jobs.push_back(j);
    }
    return GW_OK;
}

// Order jobs largest first, pick a uniform pair split for `waves` block waves, set item ranges.
int f64_schedule(std::vector<gw::F64Job> &jobs, int waves)
{
    std::stable_sort(jobs.begin(), jobs.end(), [](const gw::F64Job &a, const gw::F64Job &b) {
        return (double)a.ng * a.ng * a.P > (double)b.ng * b.ng * b.P;
    });
    int64_t tiles = 0;
    for (auto &j : jobs) tiles += (int64_t)j.ntile * (j.ntile + 1) / 2;
    const int64_t want = (int64_t)waves * 2 * num_sms();
    int64_t ks = std::max<int64_t>(1, (want + tiles - 1) / std::max<int64_t>(tiles, 1));
    int items = 0;
    for (auto &j : jobs) {
        int64_t kj = std::min<int64_t>(ks, std::max<int64_t>(1, (j.P + 255) / 256)); // >= 256 pairs per item
        j.ksplit = (int)kj;
        j.item_start = items;
        items += (int)(kj * j.ntile * (j.ntile + 1) / 2);
    }
    return items;
}

gw_status launch_f64_jobs(gw_chi0 *h, std::vector<gw::F64Job> &jobs, int bt, int waves, const int *guard)
{
    const int nitems = f64_schedule(jobs, waves);
    const void *dj;
    gw_status s = upload_jobs(h, jobs.data(), sizeof(gw::F64Job) * jobs.size(), &dj);
    if (s) return s;
    const int grid = std::max(1, std::min(nitems, 2 * num_sms()));
    Scope sc(h, "contract_f64");
    CK(h, gw::launch_contract_f64_jobs(bt, (const gw::F64Job *)dj, (int)jobs.size(), nitems, grid, h->status, guard,
                                        h->st),
       "contract_f64");
    return GW_OK;
}

gw_status make_tmap_z(gw_chi0 *h, CUtensorMap *map, void *Z, int64_t kpad, int nrows, int s, int box_rows)
{
    cuuint64_t dims[3] = {(cuuint64_t)kpad, (cuuint64_t)nrows, (cuuint64_t)s};
    cuuint64_t strides[2] = {(cuuint64_t)kpad * 2, (cuuint64_t)kpad * 2 * nrows};
    cuuint32_t box[3] = {(cuuint32_t)gw::oz_box_k(), (cuuint32_t)box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = h->encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, Z, dims, strides, box, es,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(h, GW_ERR_CUDA, "cuTensorMapEncodeTiled (slices) failed (%d)", (int)r);
    return GW_OK;
}

gw_status oz_job(gw_chi0 *h, gw::OzJob &j, void *Z, int64_t kpad, int ng, const int *E, double2 *chi, int nslices)
{
    std::memset(&j, 0, sizeof j);
    const int s = nslices > 0 ? nslices : gw::oz_slices(h->d.nslices);
    gw_status st;
    if ((st = make_tmap_z(h, &j.tmA, Z, kpad, 2 * ng, s, gw::oz_box_rows()))) return st;
    j.tmB = j.tmA;
    j.E = E;
    j.chi = (double *)chi;
    j.ng = ng;
    j.nk = (int)(kpad / gw::oz_box_k());
    j.s = s;
    return GW_OK;
}

int oz_clusters(size_t nitems) { return (int)std::max<size_t>(1, std::min<size_t>(nitems, num_sms() / 2)); }

// Items of the Hermitian contraction: the upper tiles of every job, largest job first.  The tiles
// beyond the last full wave of CTA pairs split their K range in p parts, one part of every tile
// after the other (pairs that run together then read the same pairs' slices from L2): at
// N_G = 2000, 136 tiles on 76 pairs run as 76 and 60 x 5 parts, 1.8 waves instead of 2.  A part has
// at least 4 K-steps and costs about 2.5 K-steps more for its own epilogue, and a launch has at most
// four waves of parts.  The scratch where the parts meet is the handle's; without room for it in
// the memory budget the tiles stay whole.
gw_status oz_items(gw_chi0 *h, std::vector<gw::OzJob> &jobs, std::vector<gw::OzItem> &items)
{
    std::stable_sort(jobs.begin(), jobs.end(), [](const gw::OzJob &a, const gw::OzJob &b) {
        return (double)a.ng * a.ng * a.nk > (double)b.ng * b.ng * b.nk;
    });
    items.clear();
    for (size_t j = 0; j < jobs.size(); ++j)
        for (int J = 0; J * gw::oz_box_rows() < jobs[j].ng; ++J)
            for (int I = 0; I <= J; ++I) items.push_back({(int)j, I, J, 0, jobs[j].nk, 0, 1, 0});
    const size_t ncl = std::max(1, num_sms() / 2), full = items.size() / ncl * ncl, rest = items.size() - full;
    if (rest == 0) return GW_OK;
    int nk = items[full].nk;
    for (size_t i = full; i < items.size(); ++i) nk = std::min(nk, items[i].nk);
    int p = 1;
    double best = 1e300;
    for (int q = 1; q <= std::max(1, nk / 4) && q <= 16 && (q == 1 || rest * q <= 4 * ncl); ++q) {
        const double c = (double)((rest * q + ncl - 1) / ncl) * (1.0 / q + 2.5 / nk);
        if (c < best) {
            best = c;
            p = q;
        }
    }
    if (p == 1) return GW_OK;
    const size_t need = gw::oz_part_bytes() * rest * p, flags = sizeof(int) * gw::oz_slot_flags() * ncl;
    if (h->ozpart_cap < need || !h->ozflags) {
        if (h->d.mem_budget_bytes && h->bytes - h->ozpart_cap + need + flags > h->d.mem_budget_bytes) return GW_OK;
        const std::string err = h->err;
        gw_status st = grow(h, (void **)&h->ozpart, &h->ozpart_cap, need, "split tile sums");
        if (st == GW_ERR_OOM) {
            h->err = err; // not a failure: whole tiles need no scratch
            return GW_OK;
        }
        if (st) return st;
        if (!h->ozflags) {
            if ((st = grow(h, (void **)&h->ozflags, &h->ozflags_cap, flags, "split tile counters"))) return st;
            // on the handle's stream: the default stream is not ordered with the launches that count here
            CK(h, cudaMemsetAsync(h->ozflags, 0, flags, h->st), "split tile counters");
        }
    }
    const std::vector<gw::OzItem> tail(items.begin() + full, items.end());
    items.resize(full);
    for (int i = 0; i < p; ++i)
        for (size_t k = 0; k < tail.size(); ++k) {
            const gw::OzItem &t = tail[k];
            const int k0 = (int)((int64_t)t.nk * i / p), k1 = (int)((int64_t)t.nk * (i + 1) / p);
            items.push_back({t.job, t.I, t.J, k0, k1 - k0, i, p, (int)k});
        }
    return GW_OK;
}

// A launch's job table with its item list behind it, in one block.
size_t oz_table(const std::vector<gw::OzJob> &jobs, const std::vector<gw::OzItem> &items,
                std::vector<unsigned char> &blob)
{
    const size_t nj = sizeof(gw::OzJob) * jobs.size(), ni = sizeof(gw::OzItem) * items.size();
    blob.resize(nj + ni);
    std::memcpy(blob.data(), jobs.data(), nj);
    std::memcpy(blob.data() + nj, items.data(), ni);
    return nj;
}

gw_status launch_oz_jobs(gw_chi0 *h, std::vector<gw::OzJob> &jobs, const int *guard)
{
    std::vector<gw::OzItem> items;
    std::vector<unsigned char> blob;
    gw_status s = oz_items(h, jobs, items);
    if (s) return s;
    const size_t off = oz_table(jobs, items, blob);
    const void *dj;
    if ((s = upload_jobs(h, blob.data(), blob.size(), &dj))) return s;
    Scope sc(h, guard ? "contract_f64" : "ozaki_gemm");
    CK(h, gw::launch_oz_gemm_jobs((const gw::OzJob *)dj, (const gw::OzItem *)((const char *)dj + off),
                                  (int)items.size(), oz_clusters(items.size()), oz_scratch(h), h->status, guard, h->st),
       "oz gemm");
    return GW_OK;
}

// Every tile of the general products, the tiles of one block of rows one after the other (pairs of
// CTAs that run together share A rows).
gw_status launch_oz_general(gw_chi0 *h, const std::vector<gw::OzJob> &jobs)
{
    std::vector<gw::OzItem> items;
    std::vector<unsigned char> blob;
    const int64_t b = gw::oz_box_rows(); // complex rows and columns of a tile
    for (size_t j = 0; j < jobs.size(); ++j)
        for (int I = 0; I * b < jobs[j].rows_a; ++I)
            for (int J = 0; J * b < jobs[j].cols_b; ++J) items.push_back({(int)j, I, J, 0, jobs[j].nk});
    const size_t off = oz_table(jobs, items, blob);
    const void *dj;
    gw_status s = upload_jobs(h, blob.data(), blob.size(), &dj);
    if (s) return s;
    CK(h, gw::launch_oz_gemm_general((const gw::OzJob *)dj, (const gw::OzItem *)((const char *)dj + off),
                                     (int)items.size(), oz_clusters(items.size()), h->status, h->st),
       "oz general product");
    return GW_OK;
}

// Split-precision contraction of one chunk for each frequency (chi blocks [nw][ng][ng]).
gw_status contract_chunk_ozaki(gw_chi0 *h, const double2 *M, int64_t P, int ng, const double *delta, int64_t dstride,
                               int nw, double2 *chi)
{
    const int s = gw::oz_slices(h->d.nslices);
    const int64_t kpad = (P + 63) / 64 * 64;
    const size_t zper = (size_t)s * 2 * ng * kpad; // bf16 slices of one frequency
    // several frequencies: slice a group at once (M read once per pass for the group), the group's
    // slices within 4 GiB
    const int wg = nw == 1 ? 1 : std::max(1, std::min({nw, gw::oz_group_w(), (int)(4294967296.0 / (2.0 * zper))}));
    gw_status st;
    if ((st = grow(h, &h->Zbuf, &h->Zcap, zper * 2 * wg, "slice buffer")) ||
        (st = grow(h, (void **)&h->spbuf, &h->spcap, sizeof(double) * (size_t)nw * dstride, "scale buffer")) ||
        (st = grow(h, (void **)&h->Ebuf, &h->Ecap, sizeof(int) * (size_t)ng * wg, "exponent buffer")))
        return st;
    {
        Scope sc(h, "oz_split");
        CK(h, gw::launch_oz_sqrt(delta, (int64_t)nw * dstride, h->spbuf, h->st), "oz sqrt");
    }
    for (int w0 = 0; w0 < nw; w0 += wg) {
        const int cnt = std::min(wg, nw - w0);
        const double *sp = h->spbuf + (int64_t)w0 * dstride;
        {
            Scope sc(h, "oz_split");
            if (cnt == 1) {
                CK(h, gw::launch_oz_colexp(M, P, ng, sp, h->Ebuf, nullptr, h->st), "oz exponents");
                CK(h, gw::launch_oz_slice(M, P, ng, sp, h->Ebuf, s, kpad, h->Zbuf, nullptr, h->st), "oz slices");
            } else {
                CK(h, gw::launch_oz_split_multi(M, P, ng, sp, dstride, cnt, h->Ebuf, s, kpad, h->Zbuf, (int64_t)zper,
                                                h->st),
                   "oz slices (frequency group)");
            }
        }
        // one launch per frequency, or for as many as fill a wave of CTA pairs when one has fewer tiles
        const int64_t nt = (ng + gw::oz_box_rows() - 1) / gw::oz_box_rows(), tiles = nt * (nt + 1) / 2;
        std::vector<gw::OzJob> jobs;
        for (int j = 0; j < cnt; ++j) {
            jobs.emplace_back();
            if ((st = oz_job(h, jobs.back(), (uint16_t *)h->Zbuf + zper * j, kpad, ng, h->Ebuf + (size_t)ng * j,
                             chi + (int64_t)(w0 + j) * ng * ng)))
                return st;
            if (j + 1 < cnt && tiles * (int64_t)jobs.size() < num_sms() / 2) continue;
            if ((st = launch_oz_jobs(h, jobs))) return st;
            jobs.clear();
        }
    }
    return GW_OK;
}

// FP64 contraction by slices (oz_gemm_kernel, OzProd::F64) of P pairs for each frequency, in pieces of
// at most 16384 pairs, smaller ones only where a memory budget or the device has no room for their slices;
// *done = false where it has none for 1024.  (How much memory happens to be free has no part in it: the pieces
// decide where the FP64 sums are rounded.)  The launch of the DMMA kernel behind it returns at once unless the
// slicing kernels found entries that are not finite or column scales beyond 2^+-390.
static gw_status contract_f64_slices(gw_chi0 *h, const double2 *M, int64_t P, int ng, const double *delta,
                                     int64_t dstride, int nw, double2 *chi, bool *done)
{
    *done = false;
    const int s = gw::oz_f64_slices();
    const int64_t per = (int64_t)s * 2 * ng * 2; // bytes of a pair's slices
    int64_t piece = std::min<int64_t>((P + 63) / 64 * 64, 16384);
    auto halve = [&] { piece = (piece / 2 + 63) / 64 * 64; };
    if (h->d.mem_budget_bytes) {
        const size_t rest = h->bytes - h->Zcap + (64 << 20);
        const size_t room = rest < h->d.mem_budget_bytes ? h->d.mem_budget_bytes - rest : 0;
        while (piece > 1024 && (size_t)(piece * per) > room) halve();
        if ((size_t)(piece * per) > room) return GW_OK;
    }
    const std::string err = h->err;
    const int64_t nt = (ng + gw::oz_box_rows() - 1) / gw::oz_box_rows(), tiles = nt * (nt + 1) / 2;
    gw_status st;
    h->zbusy = true;
    while ((st = grow(h, &h->Zbuf, &h->Zcap, (size_t)(piece * per), "slice buffer")) == GW_ERR_OOM && piece > 1024)
        halve();
    if (st || (st = grow(h, (void **)&h->spbuf, &h->spcap, sizeof(double) * (size_t)nw * dstride, "scale buffer")) ||
        (st = grow(h, (void **)&h->Ebuf, &h->Ecap, sizeof(int) * (size_t)ng, "exponent buffer")) ||
        (st = grow(h, (void **)&h->f64guard, &h->f64guard_cap, sizeof(int), "slice check")) ||
        (st = grow(h, &h->jobbuf, &h->jobcap,
                   std::max(sizeof(gw::OzJob) + sizeof(gw::OzItem) * (size_t)(tiles + 8 * num_sms()), sizeof(gw::F64Job)),
                   "job table"))) {
        h->zbusy = false;
        if (st != GW_ERR_OOM) return st;
        h->err = err; // the DMMA kernel needs none of these
        return GW_OK;
    }
    auto run = [&]() -> gw_status {
        {
            Scope sc(h, "oz_split");
            CK(h, gw::launch_oz_sqrt(delta, (int64_t)nw * dstride, h->spbuf, h->st), "oz sqrt");
        }
        for (int64_t p0 = 0; p0 < P; p0 += piece) {
            const int64_t cnt = std::min(piece, P - p0), kpad = (cnt + 63) / 64 * 64;
            const double2 *Mp = M + p0 * ng;
            for (int w = 0; w < nw; ++w) {
                double2 *out = chi + (int64_t)w * ng * ng;
                {
                    Scope sc(h, "oz_split");
                    const double *sp = h->spbuf + (int64_t)w * dstride + p0;
                    CK(h, cudaMemsetAsync(h->f64guard, 0, sizeof(int), h->st), "slice check");
                    CK(h, gw::launch_oz_colexp(Mp, cnt, ng, sp, h->Ebuf, h->f64guard, h->st), "oz exponents");
                    CK(h, gw::launch_oz_slice(Mp, cnt, ng, sp, h->Ebuf, s, kpad, h->Zbuf, h->f64guard, h->st), "oz slices");
                }
                std::vector<gw::OzJob> oj(1);
                std::vector<gw::F64Job> fj;
                gw_status e;
                if ((e = oz_job(h, oj[0], h->Zbuf, kpad, ng, h->Ebuf, out, s)) || (e = launch_oz_jobs(h, oj, h->f64guard)) ||
                    (e = f64_jobs(h, fj, Mp, cnt, ng, delta + (int64_t)w * dstride + p0, dstride, 1, out, h->tuned_bt)) ||
                    (e = launch_f64_jobs(h, fj, h->tuned_bt, h->tuned_waves, h->f64guard)))
                    return e;
            }
        }
        return GW_OK;
    };
    st = run();
    h->zbusy = false;
    *done = st == GW_OK;
    return st;
}

// FP64: computed pair elements go by slices where that takes less time, from 32 pairs on (16 pairs: 72 to 86
// us against 82 to 85 of the DMMA kernel for N_G = 40 to 500; 32: 72 to 87 against 158; 1024: 130 to 149
// against 1200; 8192 pairs at N_G = 2000: 3.5 ms against 138).  The slices cost five launches a frequency, 72 us
// and .055 a pair up to 1024 (.0135 beyond) beside their products, where one DMMA launch serves them all: 4.8 us a
// pair of an item while each has an SM of its own, 8.6 with two to an SM.  (56 pairs, N_G = 40, 27 weights: 1.84 ms
// by slices, .37 on DMMA; 1677 pairs, N_G = 40, 9 weights: 1.35 against 1.12.)  Elements that the caller passes in
// stay on the DMMA kernel, whose error is relative to each term of a sum where the slices' is relative to the
// columns' norms.
static bool f64_slices_faster(const gw_chi0 *h, int64_t P, int ng, int nw)
{
    if (P < 32) return false;
    const int64_t nt = (ng + h->tuned_bt - 1) / h->tuned_bt, tiles = nt * (nt + 1) / 2 * nw;
    const int64_t want = (int64_t)h->tuned_waves * 2 * num_sms(); // f64_schedule's split
    const int64_t ks = std::min<int64_t>(std::max<int64_t>(1, (want + tiles - 1) / tiles), std::max<int64_t>(1, (P + 255) / 256));
    const double items = (double)tiles * ks / num_sms(), per = (double)P / ks; // items an SM
    const double dmma = per * (items <= 1.0 ? 4.8 : items <= 2.0 ? 4.8 + 3.8 * (items - 1.0) : 4.3 * items);
    const double slices = 72.0 + 0.055 * std::min<int64_t>(P, 1024) + 0.0135 * std::max<int64_t>(P - 1024, 0) +
                          1e-7 * ng * ng * P;
    return nw * slices < dmma;
}

gw_status contract_chunk(gw_chi0 *h, const double2 *M, int64_t P, int ng, const double *delta, int64_t dstride,
                         int nw, double2 *chi, bool given)
{
    if (h->d.prec == GW_PREC_OZAKI_BF16) return contract_chunk_ozaki(h, M, P, ng, delta, dstride, nw, chi);
    if (!given && f64_slices_faster(h, P, ng, nw)) {
        bool done;
        gw_status s = contract_f64_slices(h, M, P, ng, delta, dstride, nw, chi, &done);
        if (s || done) return s;
    }
    std::vector<gw::F64Job> jobs;
    gw_status s = f64_jobs(h, jobs, M, P, ng, delta, dstride, nw, chi, h->tuned_bt);
    if (s) return s;
    return launch_f64_jobs(h, jobs, h->tuned_bt, h->tuned_waves);
}

// K extent of a general product with ka complex inner entries, padded for the TMA boxes.
int64_t oz_kpad(int ka) { return ((int64_t)ka + 63) / 64 * 64; }

// Slices of the nout columns of B [ka][ldb] for a general product.  Rows without a gap are the layout of
// the contraction's slices, whose two kernels (exponents, digits) read coalesced over the columns, once
// each; a block per column reads 16 bytes of each row, and its second pass finds them in L1.  The two
// passes are faster while B stays in L2 between them (2000 x 2000, 64 MB: 1.7 ms less over the 40
// products of a dielectric inverse), the block per column beyond (6000 x 3072, 295 MB: 0.66 against 0.89 ms
// for three).
cudaError_t launch_oz_columns(const double2 *B, int ka, int nout, int64_t ldb, int s, int64_t kpad, void *Z, int *E,
                              cudaStream_t st)
{
    if (ldb != nout || (size_t)ka * nout * sizeof(double2) > ((size_t)96 << 20))
        return gw::launch_oz_split(B, nout, ka, 1, ldb, false, s, kpad, Z, E, st);
    cudaError_t e = gw::launch_oz_colexp(B, ka, nout, nullptr, E, nullptr, st);
    return e != cudaSuccess ? e : gw::launch_oz_slice(B, ka, nout, nullptr, E, s, kpad, Z, nullptr, st);
}

// B operand of a general split product: the columns of B [ka][nout] (complex, row-major)
// into the handle's ZB / EB buffers.
gw_status oz_prepare_b(gw_chi0 *h, const double2 *B, int ka, int nout, int nslices)
{
    const int s = gw::oz_slices(nslices > 0 ? nslices : h->d.nslices);
    const int64_t kpad = oz_kpad(ka);
    gw_status st;
    if ((st = grow(h, &h->ZBbuf, &h->ZBcap, (size_t)s * 2 * nout * kpad * 2, "product operand slices")) ||
        (st = grow(h, (void **)&h->EBbuf, &h->EBcap, sizeof(int) * (size_t)nout, "product operand exponents")))
        return st;
    CK(h, launch_oz_columns(B, ka, nout, nout, s, kpad, h->ZBbuf, h->EBbuf, h->st), "oz column slices");
    return GW_OK;
}

// Y[rows][nout] = A[rows][ka] B[ka][nout] (complex, row-major) in split precision, B prepared
// by oz_prepare_b.  A's slices reuse the contraction's slice buffer (stream order separates
// the two uses).
gw_status oz_product(gw_chi0 *h, const double2 *A, int64_t rows, int ka, int nout, double2 *Y, int nslices)
{
    const int s = gw::oz_slices(nslices > 0 ? nslices : h->d.nslices);
    const int64_t kpad = oz_kpad(ka);
    gw_status st;
    if ((st = grow(h, &h->Zbuf, &h->Zcap, (size_t)s * 2 * rows * kpad * 2, "slice buffer")) ||
        (st = grow(h, (void **)&h->EAbuf, &h->EAcap, sizeof(int) * (size_t)rows, "product row exponents")))
        return st;
    CK(h, gw::launch_oz_split(A, rows, ka, ka, 1, false, s, kpad, h->Zbuf, h->EAbuf, h->st), "oz row slices");
    gw::OzJob j;
    std::memset(&j, 0, sizeof j);
    if ((st = make_tmap_z(h, &j.tmA, h->Zbuf, kpad, (int)(2 * rows), s, gw::oz_box_rows())) ||
        (st = make_tmap_z(h, &j.tmB, h->ZBbuf, kpad, 2 * nout, s, gw::oz_box_rows())))
        return st;
    j.E = h->EAbuf;
    j.E2 = h->EBbuf;
    j.out = (double *)Y;
    j.ldo = 2 * (int64_t)nout;
    j.rows_a = (int)rows;
    j.cols_b = nout;
    j.nk = (int)(kpad / gw::oz_box_k());
    j.s = s;
    return launch_oz_general(h, {j});
}

bool alias_free(const gw_chi0 *h, const BandSet &v, const BandSet &c, const Sphere &s, int *axis)
{
    for (int a = 0; a < 3; ++a)
        if (v.maxabs[a] + c.maxabs[a] + s.maxabs[a] >= h->d.n[a]) {
            *axis = a;
            return false;
        }
    return true;
}

gw_status check_slot(gw_chi0 *h, int iq)
{
    if (iq < 0 || iq >= h->d.nq) return fail(h, GW_ERR_ARG, "q slot %d out of range [0, %d)", iq, h->d.nq);
    const BandSet &v = h->val[iq];
    const Sphere &s = h->sph[iq];
    if (v.nb == 0) return fail(h, GW_ERR_STATE, "valence bands of slot %d not set", iq);
    if (h->cond.nb == 0) return fail(h, GW_ERR_STATE, "conduction bands not set");
    if (s.ng == 0) return fail(h, GW_ERR_STATE, "G-sphere of slot %d not set", iq);
    int ax;
    if (!alias_free(h, v, h->cond, s, &ax))
        return fail(h, GW_ERR_ARG, "slot %d: max|K_v| + max|K_c| + max|G| >= n on axis %d (aliasing)", iq, ax);
    double vmax = *std::max_element(v.e.begin(), v.e.end());
    double cmin = *std::min_element(h->cond.e.begin(), h->cond.e.end());
    if (!(vmax < cmin)) return fail(h, GW_ERR_ARG, "slot %d: a valence energy is not below every conduction energy", iq);
    return GW_OK;
}

cudaError_t run_pair(gw_chi0 *h, const void *psiv, const void *psic, int nc, int64_t p0, int64_t cnt,
                     const gw::PairPlan &pp, double2 *M)
{
    if (h->d.mtxel_prec == GW_MTXEL_TWOFLOAT) return gw::launch_pair_tf(psiv, psic, nc, p0, cnt, pp, M, h->st);
    return gw::launch_pair((const double2 *)psiv, (const double2 *)psic, nc, p0, cnt, pp, M, h->st);
}

gw::PairPlan pair_plan(gw_chi0 *h, const Sphere &s)
{
    gw::PairPlan pp;
    for (int a = 0; a < 3; ++a) {
        pp.n[a] = h->d.n[a];
        pp.ax[a] = h->ax[a];
    }
    pp.K2 = s.K2;
    pp.kz = s.kz;
    pp.ng = s.ng;
    pp.gpack = s.gpack;
    pp.K12 = s.K12;
    pp.cell = s.cell;
    pp.cstart = s.cstart_d;
    pp.cpts = s.cpts;
    pp.scr = h->pscr;
    pp.slot_flags = h->pflags;
    pp.nslots = s.nslots;
    pp.status = h->status;
    return pp;
}

void free_bands(gw_chi0 *h, BandSet &b)
{
    dfree(h, b.psi, sizeof(double2) * (size_t)b.nb * h->nr);
    dfree(h, b.energy, sizeof(double) * b.nb);
    dfree(h, b.gvec, sizeof(int32_t) * 3 * b.ngpsi);
    dfree(h, b.gofs, sizeof(int32_t) * b.ngpsi);
    b = BandSet();
}

void free_sphere(gw_chi0 *h, Sphere &s)
{
    dfree(h, s.kz, sizeof(int) * s.K2);
    dfree(h, s.gpack, sizeof(int32_t) * s.ng);
    dfree(h, s.gvec, sizeof(int32_t) * 3 * s.ng);
    dfree(h, s.cell, sizeof(int32_t) * s.K12);
    dfree(h, s.cstart_d, sizeof(int) * (s.K12 + 1));
    dfree(h, s.cpts, sizeof(int2) * s.ng);
    s = Sphere();
}
// The high-priority second stream and the events of the overlapped paths (created on first use).
gw_status ensure_overlap_stream(gw_chi0 *h)
{
    if (h->ov_st) return GW_OK;
    int lo = 0, hi = 0;
    CK(h, cudaDeviceGetStreamPriorityRange(&lo, &hi), "stream priorities");
    CK(h, cudaStreamCreateWithPriority(&h->ov_st, cudaStreamNonBlocking, hi), "contraction stream");
    for (int b = 0; b < 2; ++b) {
        CK(h, cudaEventCreateWithFlags(&h->ov_split[b], cudaEventDisableTiming), "event");
        CK(h, cudaEventCreateWithFlags(&h->ov_gemm[b], cudaEventDisableTiming), "event");
    }
    return GW_OK;
}

// ------------------------------------------------------------------ stage (a) on the tensor cores
// The last-axis transform of the pair products as a split product per grid line (zdft.cu), the
// middle and first axes from its output, for two-float stage (a): on the 40^3 and 48^3 grids in one
// kernel, on others of the lengths of pair_split_supported with the cells in global memory between
// two.  A block is vb valence x cb conduction bands; the row slices of the conduction block are formed
// once, and the valence bands run over it in sub-blocks whose transform output F fits the work buffer.
// On one stream: the last-axis product and the split contraction each need whole SMs.
// GW_CHI0_STAGE_A=fft selects the FFT pair kernel instead.  FP64 stage (a) takes the same steps with
// zdft64.cu and FP64 middle- and first-axis kernels.

// grids whose middle and first axes run in one kernel, with the pair kernel's scratch slots
static bool zd_fused(const gw_chi0 *h)
{
    const int *n = h->d.n;
    return h->d.mtxel_prec == GW_MTXEL_TWOFLOAT && n[0] == n[1] && n[1] == n[2] && (n[0] == 40 || n[0] == 48);
}

static bool zd_grid(const gw_chi0 *h, const Sphere &sp)
{
    static const bool fft_only = [] {
        const char *e = getenv("GW_CHI0_STAGE_A");
        return e && strcmp(e, "fft") == 0;
    }();
    const int *n = h->d.n;
    if (fft_only) return false;
    if (h->d.mtxel_prec == GW_MTXEL_FP64)
        return gw::zd64_supported(n[2], sp.K2) && gw::pair_split_supported(n[0]) && gw::pair_split_supported(n[1]);
    if (!gw::zd_supported(n[2], sp.K2)) return false;
    if (zd_fused(h)) return sp.nslots > 0 && h->pscr;
    // 24^3 keeps its grid-specialised FFT kernel, which runs beside the contraction on a second stream
    const bool small_cube = n[0] == n[1] && n[1] == n[2] && n[0] <= 24;
    return !small_cube && gw::pair_split_supported(n[0]) && gw::pair_split_supported(n[1]);
}

// Whether a call of nv x nc pairs in blocks of z.vb x z.cb takes less time this way than with the FFT kernel in
// launches of `launch` pairs.  From microseconds measured on one GB300 for 1 x 1 to 64 x 32 and 16 x 128 bands on
// thirteen grids, two-float:
//  the FFT kernel 1.12 a pair on 48^3, 0.84 on 40^3, 5.2 on 72^3, about 28e-6 a grid point where it is not
//  grid-specialised, a launch for its pairs rounded up to one an SM (its time is a staircase), and no less
//  than for 280, 300, 215 and 210; less with few kept frequencies (two bands on 48^3: 216 us with 3, 246 with 7,
//  314 with 21; 72^3: 693, 736, 829);
//  here 11e-3 per line, stage of 8 points and tile of 128 conduction bands x CT valence bands, however few of its
//  rows and columns hold bands (8e-3 with four row tiles to a column tile), 8.2e-6 per line and kept frequency of a
//  pair for the other two axes, no less than for 300 pairs, and 20 + the row slices' bytes at 4.3 TB/s per
//  conduction block.
// FP64: the FFT kernel 64e-6 a grid point (57e-6 on 32^3 to 75e-6 on 45^3) and no less than for 176 pairs; here 19e-3, 36e-6
// for at least 230 pairs, and 2.9 TB/s.
// Few conduction bands and many valence bands are what loses: 40 x 2 bands on 48^3 take 1.53 ms here and 0.31 there,
// on 72^3 7.7 and 1.1, 64 x 32 3.0 and 2.3; 8 x 128 0.74 and 1.17, 3.3 and 5.6.  Over the measured cases the rule's
// choice is at most 6 % slower than the better one; over thin boxes of 3 to 29 kept frequencies 17 % (36^3, 8 x 1
// bands, 298 us for 255), FP64 60 % (36^3, 2 x 1 bands, 29 kept, the FFT kernel's 727 us for 455).
static bool zd_faster(const gw_chi0 *h, const Sphere &sp, int nv, int nc, int64_t launch, const ZdPlan &z)
{
    const int *n = h->d.n, ct = z.f64 ? gw::zd64_valence_per_tile(sp.K2) : gw::zd_valence_per_tile(n[2], sp.K2);
    const bool cube = n[0] == n[1] && n[1] == n[2];
    const double lines = (double)n[0] * n[1], blocks = (double)((nv + z.vb - 1) / z.vb) * ((nc + z.cb - 1) / z.cb);
    const double pairs = (double)z.vb * z.cb, stages = (n[2] + 7) / 8;
    const double tiles = (double)((z.cb + 127) / 128) * ((z.vb + ct - 1) / ct);
    const double row_us = 20.0 + (z.f64 ? gw::zd64_row_bytes(z.cb, n[2], (int)lines) / 2.9e6
                                        : gw::zd_row_bytes(z.cb, n[2], (int)lines) / 4.3e6);
    const double here = blocks * (tiles * lines * stages * (z.f64 ? 19e-3 : 11e-3) +
                                  lines * sp.K2 * (z.f64 ? 36e-6 * std::max(pairs, 230.0) : 8.2e-6 * std::max(pairs, 300.0))) +
                        ((nc + z.cb - 1) / z.cb) * row_us;
    double per = 28e-6 * lines * n[2], least = 210.0; // the FFT kernel: a pair, and pairs that a launch costs at least
    if (z.f64) {
        per = 64e-6 * lines * n[2];
        least = 176.0;
    } else if (cube && (n[0] == 40 || n[0] == 48 || n[0] == 72)) {
        per = n[0] == 40 ? 0.84 : n[0] == 48 ? 1.12 : 5.2;
        least = n[0] == 40 ? 300.0 : n[0] == 48 ? 280.0 : 215.0;
    }
    if (!z.f64) per *= std::min(1.0, 0.62 + 1.2 * sp.K2 / n[2]);
    const int64_t P = (int64_t)nv * nc, sms = num_sms();
    auto fft = [&](int64_t pairs) { return per * std::max((double)((pairs + sms - 1) / sms * sms), least); };
    const double there = P / launch * fft(launch) + (P % launch ? fft(P % launch) : 0.0);
    return here < there;
}

// Room for the route's buffers beside what the call will still take: with a memory budget, what the
// caller names (pending), the pair elements of a chunk, their slices (for a group of frequencies) and
// the split tiles' scratch come first; without one, growth by a quarter of the free memory.
static bool zd_room(const gw_chi0 *h, size_t grow_by, int64_t pairs, int ng, int nw, size_t pending)
{
    if (grow_by == 0) return true;
    if (h->d.mem_budget_bytes) {
        const double m = 16.0 * pairs * ng, z = 4.0 * gw::oz_slices(h->d.nslices) * ng * (pairs + 64.0);
        const double later = pending + 3.0 * m + z * std::min(nw, gw::oz_group_w()) + 16.0 * pairs * nw + 100e6;
        return (double)h->bytes + grow_by + later <= (double)h->d.mem_budget_bytes;
    }
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return grow_by <= free_b / 4;
}

// Blocks and sub-blocks of a call's plan; false where the route does not take the call or has no room.
static bool zd_choose(const gw_chi0 *h, const Sphere &sp, int nv, int nc, bool rows, bool force, int sides, int nw,
                      size_t pending, int64_t launch, ZdPlan &z)
{
    z = ZdPlan();
    if (h->zdoff || !zd_grid(h, sp)) return false;
    z.f64 = h->d.mtxel_prec == GW_MTXEL_FP64;
    const int *n = h->d.n, lines = n[0] * n[1];
    const int ct = z.f64 ? gw::zd64_valence_per_tile(sp.K2) : gw::zd_valence_per_tile(n[2], sp.K2);
    const bool chi48 = zd_fused(h) && n[0] == 48 && !rows;
    // The route's pair elements carry 2e-13 (its fourth accumulator rounds in FP32), the FFT kernel's
    // 8e-15.  At up to seven slices the contraction's own error is ten times that and more.  At eight,
    // and with the FP64 contraction, the route serves chi on 48^3 alone (8.7e-14 at eight slices); on
    // the other calls it would raise the error, by up to three times for the gradients.
    if (!z.f64 && (h->d.prec == GW_PREC_FP64 || h->d.nslices > 7) && !chi48) return false;
    if (rows) {
        z.cb = nc;
    } else { // conduction blocks of about 512: four row tiles share a valence tile's columns
        const int nblk = (nc + 511) / 512;
        z.cb = (nc + nblk - 1) / nblk;
        if (nblk > 1) z.cb = (z.cb + 127) / 128 * 128;
        z.cb = (int)std::min<int64_t>(z.cb, h->d.pair_chunk);
    }
    int64_t vb = std::min<int64_t>(nv, h->d.pair_chunk / z.cb);
    if (vb < 1) return false;
    if (vb >= ct && vb < nv) vb -= vb % ct;
    z.vb = (int)vb;
    if (!force && !zd_faster(h, sp, nv, nc, launch, z)) return false;
    z.abytes = z.f64 ? gw::zd64_row_bytes(z.cb, n[2], lines) : gw::zd_row_bytes(z.cb, n[2], lines);
    z.ebytes = sizeof(int) * (size_t)lines * nv;
    // per valence band: F, and the cells between the two kernels of the other axes
    z.fper = sizeof(float4) * (size_t)lines * z.cb * gw::zd_row_entries(sp.K2);
    z.sper = zd_fused(h) ? 0 : sizeof(float4) * (size_t)n[0] * z.cb * sp.K12;
    // F of as many valence bands as 5 GB hold (whole tiles), fewer where memory is short.  Without a budget
    // at least one tile's: the size of a sub-block has no part in the results, the route has (2e-13), so
    // the free memory decides the one and not the other
    int vs = (int)std::min<size_t>(z.vb, std::max<size_t>(1, (size_t)5000000000 / z.fper));
    for (;; vs = vs > ct ? std::max(ct, vs / 2) : vs / 2) {
        if (vs < 1) return false;
        if (vs > ct) vs -= vs % ct;
        if (!h->d.mem_budget_bytes && vs <= ct) break;
        size_t by = 0;
        for (int i = 0; i < sides; ++i)
            by += (z.abytes > h->zdAcap[i] ? z.abytes - h->zdAcap[i] : 0) + (z.ebytes > h->zdEcap[i] ? z.ebytes - h->zdEcap[i] : 0);
        by += z.fper * vs > h->zdFcap ? z.fper * vs - h->zdFcap : 0;
        by += z.sper * vs > h->zdScap ? z.sper * vs - h->zdScap : 0;
        if (force || zd_room(h, by, (int64_t)z.vb * z.cb, sp.ng, nw, pending)) break;
    }
    z.vs = vs;
    return true;
}

gw_status zd_plan(gw_chi0 *h, const Sphere &sp, int nv, int nc, bool rows, bool force, int sides, int nw,
                  size_t pending, int64_t launch, ZdPlan &z)
{
    if (!zd_choose(h, sp, nv, nc, rows, force, sides, nw, pending, launch, z)) return GW_OK;
    const std::string err = h->err;
    gw_status s = GW_OK;
    const bool before = h->zdbusy; // an earlier plan of this call
    h->zdbusy = true;
    for (int i = 0; i < sides && !s; ++i)
        if (!(s = grow(h, &h->zdA[i], &h->zdAcap[i], z.abytes, "conduction slices")))
            s = grow(h, (void **)&h->zdE[i], &h->zdEcap[i], z.ebytes, "column exponents");
    if (!s) s = grow(h, (void **)&h->zdF, &h->zdFcap, z.fper * z.vs, "last-axis transform");
    if (!s && z.sper) s = grow(h, (void **)&h->zdS, &h->zdScap, z.sper * z.vs, "transform cells");
    if (!s && z.f64 && !(s = grow(h, (void **)&h->zdguard, &h->zdguard_cap, sizeof(int), "slice check")))
        CK(h, cudaMemsetAsync(h->zdguard, 0, sizeof(int), h->st), "slice check");
    if (s == GW_ERR_OOM && !force) { // the FFT route needs none of these
        h->err = err;
        h->zdbusy = before;
        return GW_OK;
    }
    if (s) return s;
    z.on = true;
    h->zdran = true;
    return GW_OK;
}

bool zd_holds(const gw_chi0 *h, const ZdPlan &z)
{
    return h->zdAcap[0] >= z.abytes && h->zdEcap[0] >= z.ebytes && h->zdFcap >= z.fper * z.vs &&
           h->zdScap >= z.sper * z.vs;
}

// A tensor map of two-float entries as FP32: rows of `row` entries, boxes of `w` entries x `hgt` rows.
static gw_status zd_map(gw_chi0 *h, CUtensorMap *tm, void *p, uint64_t row, uint64_t rows, int w, int hgt, const char *what)
{
    cuuint64_t d[2] = {(cuuint64_t)row * 4, (cuuint64_t)rows};
    cuuint64_t st[1] = {(cuuint64_t)row * 16};
    cuuint32_t box[2] = {(cuuint32_t)(4 * w), (cuuint32_t)hgt};
    cuuint32_t es[2] = {1, 1};
    CUresult r = h->encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, p, d, st, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? GW_OK : fail(h, GW_ERR_CUDA, "cuTensorMapEncodeTiled (%s) failed (%d)", what, (int)r);
}

gw_status zd_valence(gw_chi0 *h, ZdPlan &z, const Sphere &sp, const void *psiv, int nv, int side)
{
    const int n = h->d.n[2];
    const int64_t lines = (int64_t)h->d.n[0] * h->d.n[1];
    {
        Scope sc(h, "zd_slices");
        if (z.f64)
            CK(h, gw::launch_zd64_colexp(psiv, nv, n, (int)lines, h->zdE[side], h->zdguard, h->st), "column exponents");
        else CK(h, gw::launch_zd_colexp(psiv, nv, n, (int)lines, h->zdE[side], h->st), "column exponents");
    }
    // the valence grids, line by line: box of one line of CT bands
    const int part = gw::zd_line_split(n);
    cuuint64_t d[3] = {(cuuint64_t)4 * n / part, (cuuint64_t)lines * part, (cuuint64_t)nv};
    cuuint64_t st[2] = {(cuuint64_t)16 * n / part, (cuuint64_t)16 * lines * n};
    const int ct = z.f64 ? gw::zd64_valence_per_tile(sp.K2) : gw::zd_valence_per_tile(n, sp.K2);
    cuuint32_t box[3] = {(cuuint32_t)(4 * n / part), (cuuint32_t)part, (cuuint32_t)ct};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = h->encode(&z.tmV[side], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void *>(psiv), d, st, box, es,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(h, GW_ERR_CUDA, "cuTensorMapEncodeTiled (valence grids) failed (%d)", (int)r);
    z.nv[side] = nv;
    z.psiv[side] = psiv;
    return GW_OK;
}

gw_status zd_conduction(gw_chi0 *h, ZdPlan &z, const void *psic, int c0, int cb, int side)
{
    Scope sc(h, "zd_slices");
    const int n = h->d.n[2], lines = h->d.n[0] * h->d.n[1];
    z.psic[side] = (const double2 *)psic + (int64_t)c0 * h->nr; // 16 bytes an entry in either form
    if (z.f64)
        CK(h, gw::launch_zd64_rows(z.psic[side], cb, n, lines, h->zdA[side], h->zdguard, h->st), "conduction slices");
    else CK(h, gw::launch_zd_rows(z.psic[side], cb, n, lines, h->zdA[side], h->st), "conduction slices");
    return GW_OK;
}

gw_status zd_block(gw_chi0 *h, const ZdPlan &z, const Sphere &sp, const gw::PairPlan &pp, int vside, int cside, int v0,
                   int vb, int cb, double2 *M, int64_t sv, int64_t sc)
{
    const int *n = h->d.n;
    const int lines = n[0] * n[1];
    gw_status s;
    for (int b0 = 0; b0 < vb; b0 += z.vs) {
        const int nb = std::min(z.vs, vb - b0);
        {
            Scope t(h, "zdft");
            if (z.f64)
                CK(h, gw::launch_zd64_gemm(z.tmV[vside], h->zdA[cside], h->zdE[vside], sp.kz, pp.ax[2].tw, n[2], lines,
                                           z.nv[vside], v0 + b0, nb, cb, sp.K2, (double2 *)h->zdF, h->zdguard,
                                           h->status, h->st),
                   "last-axis transform");
            else CK(h, gw::launch_zd_gemm(z.tmV[vside], h->zdA[cside], h->zdE[vside], sp.kz, pp.ax[2].twf, n[2], lines,
                                     z.nv[vside], v0 + b0, nb, cb, sp.K2, h->zdF, h->status, h->st),
               "last-axis transform");
        }
        // F as [lines][R rows of K2P entries]: the middle-axis kernel loads the 2 n1 lines of a slab pair
        // of one row (K2 entries each) with one TMA box
        const int64_t R = (int64_t)nb * cb;
        CUtensorMap tmF, tmS;
        if ((s = zd_map(h, &tmF, h->zdF, R * gw::zd_row_entries(sp.K2), lines, sp.K2, 2 * n[1], "last-axis output")))
            return s;
        double2 *Mb = M + (int64_t)b0 * sv * sp.ng;
        Scope t(h, "pair_from_f");
        if (z.sper == 0) {
            // the scratch slots as [nslots n rows][K12] entries: phase 2 loads batches of 2 K2 cells of
            // all n rows of its slot with one TMA box
            if ((s = zd_map(h, &tmS, pp.scr, pp.K12, (uint64_t)pp.nslots * n[0], 2 * sp.K2, n[0], "pair scratch"))) return s;
            CK(h, gw::launch_pair_tf_from_f(tmF, tmS, R, cb, sv, sc, pp, Mb, h->st), "pair elements from F");
        } else {
            if ((s = zd_map(h, &tmS, h->zdS, pp.K12, (uint64_t)R * n[0], 2 * sp.K2, n[0], "transform cells"))) return s;
            if (z.f64) { // and the FFT pair kernel, which returns at once unless the slices do not hold
                gw::PairPlan pg = pp;
                pg.guard = h->zdguard;
                CK(h, gw::launch_pair_split64_1(tmF, R, pg, (double2 *)h->zdS, h->st), "middle axis from F");
                CK(h, gw::launch_pair_split64_2(tmS, R, cb, sv, sc, pg, Mb, h->st), "pair elements from cells");
                CK(h, gw::launch_pair((const double2 *)z.psiv[vside] + (int64_t)(v0 + b0) * h->nr,
                                      (const double2 *)z.psic[cside], cb, 0, R, pg, Mb, h->st),
                   "pair kernel");
                continue;
            }
            CK(h, gw::launch_pair_split1(tmF, R, pp, h->zdS, h->st), "middle axis from F");
            CK(h, gw::launch_pair_split2(tmS, R, cb, sv, sc, pp, Mb, h->st), "pair elements from cells");
        }
    }
    return GW_OK;
}

// Pairs [p0, p0 + cnt) of slot pairs (psiv, psic), whole valence rows when the plan is on.
gw_status pair_rows(gw_chi0 *h, const ZdPlan &z, const Sphere &sp, const gw::PairPlan &pp, const void *psiv,
                    const void *psic, int nc, int64_t p0, int64_t cnt, double2 *M, int vside, int cside)
{
    if (z.on) return zd_block(h, z, sp, pp, vside, cside, (int)(p0 / nc), (int)(cnt / nc), nc, M, nc, 1);
    Scope sc(h, "pair_mtxel");
    CK(h, run_pair(h, psiv, psic, nc, p0, cnt, pp, M), "pair kernel");
    return GW_OK;
}

// Split-precision streamed compute with the contraction of job j (chunk, frequency) on a
// high-priority second stream while the user stream forms the pair elements and slices of the jobs
// after it.  A contraction block takes a whole SM, so the two kernels share the GPU only where one
// of them leaves SMs idle (a launch's ramp and its last wave): 8 % faster for chunks of 500 pairs
// on 40^3, 2 % for 4096 on 24^3, no difference for full chunks.  Slices, exponents and job tables
// alternate between two buffer sets; job j waits for the contraction of job j - 2.  Taken where
// the pair kernel's blocks use at most 64 KB of shared memory (24^3 to 48^3).
// 48^3 slots that the route can serve report one stream, and keep it for the calls that its plan leaves (few
// conduction bands).
bool overlap_enabled(gw_chi0 *h, const Sphere &sp, const gw::PairPlan &pp, bool keep)
{
    if (zd_fused(h) && h->d.n[0] == 48 && !keep && zd_grid(h, sp)) return false;
    if (h->d.prec != GW_PREC_OZAKI_BF16 || h->d.single_stream || h->d.mtxel_prec != GW_MTXEL_TWOFLOAT) return false;
    const size_t ps = gw::pair_tf_ct_smem_bytes(pp);
    return ps > 0 && ps <= 64 * 1024;
}

gw_status resident_begin(gw_chi0 *h, int64_t P, int ng, bool *use)
{
    *use = false;
    h->Mres_iq = -1;
    if (!h->keep_m) return GW_OK;
    const size_t need = sizeof(double2) * (size_t)P * ng;
    if (h->d.mem_budget_bytes && h->bytes - h->Mres_cap + need > h->d.mem_budget_bytes) return GW_OK;
    size_t free_b = 0, total_b = 0;
    if (need > h->Mres_cap && (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess || need - h->Mres_cap > free_b / 2)) {
        cudaGetLastError();
        return GW_OK; // keep at most half of what is free: the elements are an optimisation, not a need
    }
    gw_status s = grow(h, (void **)&h->Mres, &h->Mres_cap, need, "resident pair elements");
    if (s) return s;
    *use = true;
    return GW_OK;
}

double2 *resident_for(gw_chi0 *h, int iq) { return h->keep_m && h->Mres_iq == iq ? h->Mres : nullptr; }

// The overlapped path's buffers, given back.
static void drop_overlap(gw_chi0 *h)
{
    cudaStreamSynchronize(h->st);
    if (h->ov_st) cudaStreamSynchronize(h->ov_st);
    for (int b = 0; b < 2; ++b) {
        dfree(h, h->ovZ[b], h->ovZcap[b]);
        dfree(h, h->ovE[b], h->ovEcap[b]);
        dfree(h, h->ovJ[b], h->ovJcap[b]);
        h->ovZ[b] = h->ovJ[b] = nullptr;
        h->ovE[b] = nullptr;
        h->ovZcap[b] = h->ovEcap[b] = h->ovJcap[b] = 0;
    }
}

gw_status compute_overlap(gw_chi0 *h, int iq, const gw::OmegaList &om, double2 *cq, double *dq, double2 *Mres)
{
    const Sphere &sp = h->sph[iq];
    const BandSet &v = h->val[iq];
    const int ng = sp.ng, nw = om.nw, s = gw::oz_slices(h->d.nslices);
    const int64_t P = (int64_t)v.nb * h->cond.nb;
    const int64_t chunk = std::min<int64_t>(h->d.pair_chunk, P);
    const int64_t kpad_max = (chunk + 63) / 64 * 64;
    gw_status st = ensure_work(h, (size_t)chunk * ng, (size_t)chunk * nw);
    if (st) return st;
    if ((st = grow(h, (void **)&h->spbuf, &h->spcap, sizeof(double) * (size_t)nw * chunk, "scale buffer"))) return st;
    for (int b = 0; b < 2; ++b)
        if ((st = grow(h, &h->ovZ[b], &h->ovZcap[b], (size_t)s * 2 * ng * kpad_max * 2, "slice buffer")) ||
            (st = grow(h, (void **)&h->ovE[b], &h->ovEcap[b], sizeof(int) * (size_t)ng, "exponent buffer")))
            return st;
    if ((st = ensure_overlap_stream(h))) return st;
    gw::PairPlan pp = pair_plan(h, sp);
    bool used[2] = {false, false};
    int64_t j = 0;
    for (int64_t p0 = 0; p0 < P; p0 += chunk) {
        const int64_t cnt = std::min(chunk, P - p0);
        const int64_t kpad = (cnt + 63) / 64 * 64;
        double2 *Mc = Mres ? Mres + p0 * ng : h->Mbuf;
        {
            Scope sc(h, "pair_mtxel");
            CK(h, run_pair(h, v.psi, h->cond.psi, h->cond.nb, p0, cnt, pp, Mc), "pair kernel");
        }
        {
            Scope sc(h, "delta");
            CK(h, gw::launch_delta(v.energy, h->cond.energy, h->cond.nb, p0, cnt, om, h->dbuf, h->st), "delta");
        }
        {
            Scope sc(h, "oz_split");
            CK(h, gw::launch_oz_sqrt(h->dbuf, (int64_t)nw * cnt, h->spbuf, h->st), "oz sqrt");
        }
        if (dq) {
            Scope sc(h, "diag");
            CK(h, gw::launch_diag(Mc, cnt, ng, h->dbuf, cnt, nw, dq, ng, h->st), "diag");
        }
        for (int w = 0; w < nw; ++w, ++j) {
            const int b = (int)(j & 1);
            if (used[b]) CK(h, cudaStreamWaitEvent(h->st, h->ov_gemm[b], 0), "wait contraction");
            {
                Scope sc(h, "oz_split");
                const double *spw = h->spbuf + (int64_t)w * cnt;
                CK(h, gw::launch_oz_colexp(Mc, cnt, ng, spw, h->ovE[b], nullptr, h->st), "oz exponents");
                CK(h, gw::launch_oz_slice(Mc, cnt, ng, spw, h->ovE[b], s, kpad, h->ovZ[b], nullptr, h->st), "oz slices");
            }
            std::vector<gw::OzJob> jobs(1);
            if ((st = oz_job(h, jobs[0], h->ovZ[b], kpad, ng, h->ovE[b], cq + (int64_t)w * ng * ng))) return st;
            std::vector<gw::OzItem> items;
            std::vector<unsigned char> blob;
            if ((st = oz_items(h, jobs, items))) return st;
            const size_t off = oz_table(jobs, items, blob);
            if ((st = grow(h, &h->ovJ[b], &h->ovJcap[b], blob.size(), "job table"))) return st;
            CK(h, cudaMemcpyAsync(h->ovJ[b], blob.data(), blob.size(), cudaMemcpyHostToDevice, h->st), "job table");
            CK(h, cudaEventRecord(h->ov_split[b], h->st), "record");
            CK(h, cudaStreamWaitEvent(h->ov_st, h->ov_split[b], 0), "wait slices");
            {
                Scope sc(h, "ozaki_gemm", h->ov_st);
                CK(h, gw::launch_oz_gemm_jobs((const gw::OzJob *)h->ovJ[b],
                                              (const gw::OzItem *)((const char *)h->ovJ[b] + off), (int)items.size(),
                                              oz_clusters(items.size()), oz_scratch(h), h->status, nullptr,
                                              h->ov_st),
                   "oz gemm");
            }
            CK(h, cudaEventRecord(h->ov_gemm[b], h->ov_st), "record");
            used[b] = true;
        }
    }
    for (int b = 0; b < 2; ++b)
        if (used[b]) CK(h, cudaStreamWaitEvent(h->st, h->ov_gemm[b], 0), "join");
    return GW_OK;
}
} // namespace gwapi

using namespace gwapi;
// =================================================================== C ABI
extern "C" {

gw_status gw_chi0_create(gw_chi0 **out, const gw_chi0_desc *d, void *stream)
{
    if (!out || !d) return GW_ERR_ARG;
    *out = nullptr;
    gw_chi0 *h = new (std::nothrow) gw_chi0();
    if (!h) return GW_ERR_OOM;
    h->d = *d;
    h->st = (cudaStream_t)stream;
    if (h->d.pair_chunk <= 0) h->d.pair_chunk = 8192;
    if (h->d.nq < 1) { delete h; return GW_ERR_ARG; }
    if (h->d.prec != GW_PREC_FP64 && h->d.prec != GW_PREC_OZAKI_BF16) { delete h; return GW_ERR_ARG; }
    if (h->d.prec == GW_PREC_OZAKI_BF16 && (h->d.nslices < 3 || h->d.nslices > 8)) { delete h; return GW_ERR_ARG; }
    if (h->d.mtxel_prec != GW_MTXEL_FP64 && h->d.mtxel_prec != GW_MTXEL_TWOFLOAT) { delete h; return GW_ERR_ARG; }
    if (h->d.single_stream != 0 && h->d.single_stream != 1) { delete h; return GW_ERR_ARG; }
    for (int a = 0; a < 3; ++a) {
        int n = h->d.n[a];
        if (n < 4 || n > 128 || !factor(n, h->ax[a])) { delete h; return GW_ERR_ARG; }
    }
    if (cudaSetDevice(h->d.device) != cudaSuccess) { cudaGetLastError(); delete h; return GW_ERR_CUDA; }
    h->nr = (int64_t)h->d.n[0] * h->d.n[1] * h->d.n[2];
    h->val.resize(h->d.nq);
    h->sph.resize(h->d.nq);

    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        delete h;
        return GW_ERR_CUDA;
    }
    h->encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;

    // twiddle tables e^{+2 pi i t/n}, computed in extended precision on the host
    int ntot = h->d.n[0] + h->d.n[1] + h->d.n[2];
    std::vector<double2> tw(ntot);
    int off = 0;
    for (int a = 0; a < 3; ++a) {
        int n = h->d.n[a];
        for (int t = 0; t < n; ++t) {
            long double ang = 2.0L * 3.141592653589793238462643383279502884L * (long double)t / (long double)n;
            tw[off + t] = make_double2((double)cosl(ang), (double)sinl(ang));
        }
        off += n;
    }
    std::vector<float4> twf(ntot);
    for (int t = 0; t < ntot; ++t) {
        float rh = (float)tw[t].x, ih = (float)tw[t].y;
        twf[t] = make_float4(rh, (float)(tw[t].x - (double)rh), ih, (float)(tw[t].y - (double)ih));
    }
    if (dalloc(h, (void **)&h->tw, sizeof(double2) * ntot, "twiddles") ||
        dalloc(h, (void **)&h->twf, sizeof(float4) * ntot, "twiddles (two-float)") ||
        dalloc(h, (void **)&h->status, sizeof(int), "status word")) {
        gw_chi0_destroy(h);
        return GW_ERR_OOM;
    }
    // in place before the caller may go on, with whatever stream
    if (cudaMemcpyAsync(h->tw, tw.data(), sizeof(double2) * ntot, cudaMemcpyHostToDevice, h->st) != cudaSuccess ||
        cudaMemcpyAsync(h->twf, twf.data(), sizeof(float4) * ntot, cudaMemcpyHostToDevice, h->st) != cudaSuccess ||
        cudaMemsetAsync(h->status, 0, sizeof(int), h->st) != cudaSuccess ||
        cudaStreamSynchronize(h->st) != cudaSuccess) {
        cudaGetLastError();
        gw_chi0_destroy(h);
        return GW_ERR_CUDA;
    }
    off = 0;
    for (int a = 0; a < 3; ++a) {
        h->ax[a].tw = h->tw + off;
        h->ax[a].twf = h->twf + off;
        off += h->d.n[a];
    }
    *out = h;
    return GW_OK;
}

int gw_chi0_streams(gw_chi0 *h, int iq)
{
    if (!h) return -(int)GW_ERR_ARG;
    gw_status s = check_slot(h, iq);
    if (s) return -(int)s;
    ZdPlan z; // stage (a) on the tensor cores runs on one stream
    const int nv = h->val[iq].nb, nc = h->cond.nb;
    const int64_t chunk = std::min<int64_t>(h->d.pair_chunk, (int64_t)nv * nc);
    if (zd_choose(h, h->sph[iq], nv, nc, h->keep_m, false, 1, 1, 0, chunk, z)) return 1;
    return overlap_enabled(h, h->sph[iq], pair_plan(h, h->sph[iq]), h->keep_m) ? 2 : 1;
}

void gw_chi0_destroy(gw_chi0 *h)
{
    if (!h) return;
    cudaStreamSynchronize(h->st);
    free_bands(h, h->cond);
    for (auto &b : h->val) free_bands(h, b);
    for (auto &s : h->sph) free_sphere(h, s);
    dfree(h, h->Mbuf, h->Mcap * sizeof(double2));
    dfree(h, h->dbuf, h->dcap * sizeof(double));
    dfree(h, h->Zbuf, h->Zcap);
    dfree(h, h->spbuf, h->spcap);
    dfree(h, h->Ebuf, h->Ecap);
    dfree(h, h->jobbuf, h->jobcap);
    dfree(h, h->Mall, h->Mall_cap);
    dfree(h, h->pscr, h->pscr_cap);
    dfree(h, h->pflags, h->pflags_cap);
    dfree(h, h->EAbuf, h->EAcap);
    dfree(h, h->EBbuf, h->EBcap);
    dfree(h, h->ZBbuf, h->ZBcap);
    dfree(h, h->MBbuf, h->MBcap);
    for (int i = 0; i < 2; ++i) {
        dfree(h, h->zdA[i], h->zdAcap[i]);
        dfree(h, h->zdE[i], h->zdEcap[i]);
    }
    dfree(h, h->zdF, h->zdFcap);
    dfree(h, h->zdS, h->zdScap);
    dfree(h, h->zdguard, h->zdguard_cap);
    for (int b = 0; b < 2; ++b) {
        dfree(h, h->ovZ[b], h->ovZcap[b]);
        dfree(h, h->ovE[b], h->ovEcap[b]);
        dfree(h, h->ovJ[b], h->ovJcap[b]);
        if (h->ov_split[b]) cudaEventDestroy(h->ov_split[b]);
        if (h->ov_gemm[b]) cudaEventDestroy(h->ov_gemm[b]);
    }
    if (h->ov_st) cudaStreamDestroy(h->ov_st);
    dfree(h, h->f64guard, h->f64guard_cap);
    dfree(h, h->ozpart, h->ozpart_cap);
    dfree(h, h->ozflags, h->ozflags_cap);
    dfree(h, h->epsbuf, h->epscap);
    dfree(h, h->Mres, h->Mres_cap);
    for (auto &b : h->gpp) dfree(h, b.p, b.cap);
    dfree(h, h->realbuf, h->realcap);
    dfree(h, h->eigA, h->eigA_cap);
    dfree(h, h->eigWork, h->eigWork_cap);
    dfree(h, h->eigW, h->eigW_cap);
    dfree(h, h->eigInfo, h->eigInfo_cap);
    if (h->sol.hdl) h->sol.destroy(h->sol.hdl);
    if (h->sol.lib) dlclose(h->sol.lib);
    dfree(h, h->Dall, h->Dall_cap);
    dfree(h, h->SPall, h->SPall_cap);
    dfree(h, h->Zall, h->Zall_cap);
    dfree(h, h->Eall, h->Eall_cap);
    for (auto &g : h->graphs) {
        if (g.exec) cudaGraphExecDestroy(g.exec);
        dfree(h, g.jobs, g.jobs_bytes);
    }
    if (h->cap_st) cudaStreamDestroy(h->cap_st);
    {
        size_t ntw = (size_t)h->d.n[0] + h->d.n[1] + h->d.n[2];
        dfree(h, h->tw, sizeof(double2) * ntw);
        dfree(h, h->twf, sizeof(float4) * ntw);
    }
    dfree(h, h->status, sizeof(int));
    for (auto &r : h->pending) {
        cudaEventDestroy(r.a);
        cudaEventDestroy(r.b);
    }
    for (auto e : h->pool) cudaEventDestroy(e);
    cudaGetLastError();
    delete h;
}

const char *gw_chi0_last_error(const gw_chi0 *h) { return h ? h->err.c_str() : "null handle"; }

gw_status gw_chi0_set_stream(gw_chi0 *h, void *stream)
{
    if (!h) return GW_ERR_ARG;
    h->st = (cudaStream_t)stream;
    return GW_OK;
}

gw_status gw_chi0_set_bands(gw_chi0 *h, int iq, int kind, int nb, int ngpsi, const int32_t *gvec, const double *coeff,
                            const double *energy)
{
    if (!h) return GW_ERR_ARG;
    if (kind != 0 && kind != 1) return fail(h, GW_ERR_ARG, "kind must be 0 (valence) or 1 (conduction)");
    if (kind == 0 && (iq < 0 || iq >= h->d.nq)) return fail(h, GW_ERR_ARG, "q slot %d out of range", iq);
    if (nb < 1 || ngpsi < 1) return fail(h, GW_ERR_ARG, "nb and ngpsi must be >= 1");
    if (!gvec || !coeff || !energy) return fail(h, GW_ERR_ARG, "null pointer");
    drop_graphs(h);
    BandSet nbs;
    nbs.nb = nb;
    nbs.ngpsi = ngpsi;
    nbs.g.resize((size_t)3 * ngpsi);
    nbs.e.resize(nb);
    CK(h, cudaMemcpyAsync(nbs.g.data(), gvec, sizeof(int32_t) * 3 * ngpsi, cudaMemcpyDeviceToHost, h->st), "copy gvec");
    CK(h, cudaMemcpyAsync(nbs.e.data(), energy, sizeof(double) * nb, cudaMemcpyDeviceToHost, h->st), "copy energy");
    CK(h, cudaStreamSynchronize(h->st), "set_bands sync");
    std::vector<int32_t> gofs(ngpsi);
    for (int k = 0; k < ngpsi; ++k) {
        int idx[3];
        for (int a = 0; a < 3; ++a) {
            int g = nbs.g[3 * k + a];
            if (2 * std::abs(g) >= h->d.n[a])
                return fail(h, GW_ERR_ARG, "plane wave %d: component %d outside (-n/2, n/2)", k, g);
            nbs.maxabs[a] = std::max(nbs.maxabs[a], std::abs(g));
            idx[a] = mod(g, h->d.n[a]);
        }
        gofs[k] = (idx[0] * h->d.n[1] + idx[1]) * h->d.n[2] + idx[2];
    }
    for (double e : nbs.e)
        if (!std::isfinite(e)) return fail(h, GW_ERR_ARG, "non-finite band energy");
    // energy ordering against the other set, when present
    const BandSet *other = nullptr;
    if (kind == 0 && h->cond.nb) other = &h->cond;
    if (other) {
        double vmax = *std::max_element(nbs.e.begin(), nbs.e.end());
        double cmin = *std::min_element(other->e.begin(), other->e.end());
        if (!(vmax < cmin)) return fail(h, GW_ERR_ARG, "a valence energy is not below every conduction energy");
    }
    if (kind == 1) {
        double cmin = *std::min_element(nbs.e.begin(), nbs.e.end());
        for (auto &v : h->val)
            if (v.nb && !(*std::max_element(v.e.begin(), v.e.end()) < cmin))
                return fail(h, GW_ERR_ARG, "a valence energy is not below every conduction energy");
    }
    if (kind == 1 || iq == h->Mres_iq) h->Mres_iq = -1; // resident pair elements no longer match
    BandSet &dst = kind == 0 ? h->val[iq] : h->cond;
    if (dst.nb == nb && dst.ngpsi == ngpsi) {
        // same shape: reuse the device buffers (no allocation on repeated setup)
        nbs.psi = dst.psi;
        nbs.energy = dst.energy;
        nbs.gvec = dst.gvec;
        nbs.gofs = dst.gofs;
        dst.psi = nullptr;
        dst.energy = nullptr;
        dst.gvec = nullptr;
        dst.gofs = nullptr;
        dst = BandSet();
    } else {
        free_bands(h, dst);
        gw_status s;
        if ((s = dalloc(h, (void **)&nbs.psi, sizeof(double2) * (size_t)nb * h->nr, "psi grids")) ||
            (s = dalloc(h, (void **)&nbs.energy, sizeof(double) * nb, "energies")) ||
            (s = dalloc(h, (void **)&nbs.gvec, sizeof(int32_t) * 3 * ngpsi, "gvec")) ||
            (s = dalloc(h, (void **)&nbs.gofs, sizeof(int32_t) * ngpsi, "grid offsets"))) {
            free_bands(h, nbs);
            return s;
        }
    }
    CK(h, cudaMemcpyAsync(nbs.energy, energy, sizeof(double) * nb, cudaMemcpyDeviceToDevice, h->st), "energies");
    CK(h, cudaMemcpyAsync(nbs.gvec, gvec, sizeof(int32_t) * 3 * ngpsi, cudaMemcpyDeviceToDevice, h->st), "gvec");
    CK(h, cudaMemcpyAsync(nbs.gofs, gofs.data(), sizeof(int32_t) * ngpsi, cudaMemcpyHostToDevice, h->st), "gofs");
    CK(h, cudaMemsetAsync(nbs.psi, 0, sizeof(double2) * (size_t)nb * h->nr, h->st), "zero psi");
    if (h->d.mtxel_prec == GW_MTXEL_TWOFLOAT) {
        Scope sc(h, "band_setup_tf");
        CK(h, gw::launch_band_setup_tf((const double2 *)coeff, nbs.gofs, nb, ngpsi, nbs.psi, h->d.n, h->ax,
                                       nbs.maxabs, h->st),
           "band setup (two-float)"); // three kernels
    } else {
        {
            Scope sc(h, "band_scatter");
            CK(h, gw::launch_scatter((const double2 *)coeff, nbs.gofs, nb, ngpsi, h->nr, nbs.psi, h->st), "scatter");
        }
        Scope sc(h, "band_fft");
        CK(h, gw::launch_band_fft(nbs.psi, nb, h->d.n, h->ax, h->st), "band fft"); // two kernels
    }
    CK(h, cudaStreamSynchronize(h->st), "set_bands sync"); // gofs host vector goes out of scope
    dst = std::move(nbs);
    return GW_OK;
}

gw_status gw_chi0_set_gsphere(gw_chi0 *h, int iq, int ng, const int32_t *gvec)
{
    if (!h) return GW_ERR_ARG;
    if (iq < 0 || iq >= h->d.nq) return fail(h, GW_ERR_ARG, "q slot %d out of range", iq);
    if (ng < 1) return fail(h, GW_ERR_ARG, "ng must be >= 1");
    if (ng > gw::pair_max_ng()) return fail(h, GW_ERR_UNSUPPORTED, "ng = %d exceeds %d", ng, gw::pair_max_ng());
    if (!gvec) return fail(h, GW_ERR_ARG, "null pointer");
    drop_graphs(h);
    Sphere s;
    s.ng = ng;
    s.g.resize((size_t)3 * ng);
    CK(h, cudaMemcpyAsync(s.g.data(), gvec, sizeof(int32_t) * 3 * ng, cudaMemcpyDeviceToHost, h->st), "copy sphere");
    CK(h, cudaStreamSynchronize(h->st), "set_gsphere sync");
    for (int i = 0; i < ng; ++i)
        for (int a = 0; a < 3; ++a) {
            int g = s.g[3 * i + a];
            if (2 * std::abs(g) >= h->d.n[a]) return fail(h, GW_ERR_ARG, "G %d: component %d outside (-n/2, n/2)", i, g);
            s.maxabs[a] = std::max(s.maxabs[a], std::abs(g));
        }
    gw::SpherePlanHost plan;
    gw::build_sphere_plan(h->d.n, ng, s.g.data(), plan);
    // alias check against whatever bands are already stored
    int ax;
    if (h->val[iq].nb && h->cond.nb && !alias_free(h, h->val[iq], h->cond, s, &ax))
        return fail(h, GW_ERR_ARG, "max|K_v| + max|K_c| + max|G| >= n on axis %d (aliasing)", ax);
    s.K2 = plan.K2;
    s.K12 = plan.K12;
    s.cstart = plan.cstart;
    s.cg = plan.cg;
    const std::vector<int> &kz = plan.kz;
    const std::vector<int32_t> &pack = plan.pack, &cell = plan.cell;
    std::vector<int2> cpts(ng);
    for (int m = 0; m < ng; ++m) cpts[m] = make_int2(plan.cpts[m].first, plan.cpts[m].second);
    gw_status st;
    if (iq == h->Mres_iq) h->Mres_iq = -1; // resident pair elements no longer match
    Sphere &old = h->sph[iq];
    if (old.ng == ng && old.K2 == s.K2 && old.K12 == s.K12) {
        s.kz = old.kz;
        s.gpack = old.gpack;
        s.gvec = old.gvec;
        s.cell = old.cell;
        s.cstart_d = old.cstart_d;
        s.cpts = old.cpts;
        old.kz = nullptr;
        old.gpack = nullptr;
        old.gvec = nullptr;
        old.cell = nullptr;
        old.cstart_d = nullptr;
        old.cpts = nullptr;
        old = Sphere();
    } else if ((st = dalloc(h, (void **)&s.kz, sizeof(int) * s.K2, "sphere kz")) ||
        (st = dalloc(h, (void **)&s.gpack, sizeof(int32_t) * ng, "sphere pack")) ||
        (st = dalloc(h, (void **)&s.gvec, sizeof(int32_t) * 3 * ng, "sphere gvec")) ||
        (st = dalloc(h, (void **)&s.cell, sizeof(int32_t) * s.K12, "sphere cells")) ||
        (st = dalloc(h, (void **)&s.cstart_d, sizeof(int) * (s.K12 + 1), "sphere cell starts")) ||
        (st = dalloc(h, (void **)&s.cpts, sizeof(int2) * ng, "sphere points by cell"))) {
        free_sphere(h, s);
        return st;
    }
    CK(h, cudaMemcpyAsync(s.kz, kz.data(), sizeof(int) * s.K2, cudaMemcpyHostToDevice, h->st), "kz");
    CK(h, cudaMemcpyAsync(s.gpack, pack.data(), sizeof(int32_t) * ng, cudaMemcpyHostToDevice, h->st), "pack");
    CK(h, cudaMemcpyAsync(s.cell, cell.data(), sizeof(int32_t) * s.K12, cudaMemcpyHostToDevice, h->st), "cells");
    CK(h, cudaMemcpyAsync(s.cstart_d, s.cstart.data(), sizeof(int) * (s.K12 + 1), cudaMemcpyHostToDevice, h->st),
       "cell starts");
    CK(h, cudaMemcpyAsync(s.cpts, cpts.data(), sizeof(int2) * ng, cudaMemcpyHostToDevice, h->st), "cell points");
    CK(h, cudaMemcpyAsync(s.gvec, gvec, sizeof(int32_t) * 3 * ng, cudaMemcpyDeviceToDevice, h->st), "gvec");
    if (h->d.mtxel_prec == GW_MTXEL_TWOFLOAT) {
        // scratch slots of the grid-specialised two-float pair kernel for this sphere
        size_t elems = 0;
        CK(h, gw::pair_tf_scratch(pair_plan(h, s), &s.nslots, &elems), "pair scratch size");
        if (s.nslots > 0) {
            if ((st = grow(h, (void **)&h->pscr, &h->pscr_cap, sizeof(float4) * elems * s.nslots, "pair scratch")) ||
                (st = grow(h, (void **)&h->pflags, &h->pflags_cap, sizeof(int) * s.nslots, "pair scratch flags"))) {
                free_sphere(h, s);
                return st;
            }
        }
    }
    CK(h, cudaStreamSynchronize(h->st), "set_gsphere sync");
    free_sphere(h, h->sph[iq]);
    h->sph[iq] = std::move(s);
    return GW_OK;
}

gw_status gw_chi0_pair_elements_block(gw_chi0 *h, int iq, int c0, int cb, double *M)
{
    if (!h) return GW_ERR_ARG;
    gw_status s = check_slot(h, iq);
    if (s) return s;
    if (c0 < 0 || cb < 0 || c0 + cb > h->cond.nb)
        return fail(h, GW_ERR_ARG, "conduction block [%d, %d) outside [0, %d)", c0, c0 + cb, h->cond.nb);
    if (cb && !M) return fail(h, GW_ERR_ARG, "null M");
    const BandSet &v = h->val[iq];
    const Sphere &sp = h->sph[iq];
    const int nv = v.nb;
    if (!zd_fused(h) || h->d.n[0] != 48 || h->keep_m || h->d.pair_chunk < nv || !zd_grid(h, sp))
        return fail(h, GW_ERR_UNSUPPORTED, "slot %d does not take the tensor-core route", iq);
    if (cb == 0) return GW_OK;
    ZdPlan z;
    ZdUse use{h};
    if ((s = zd_plan(h, sp, nv, cb, false, true, 1, 1, 0, 1, z))) return s;
    const gw::PairPlan pp = pair_plan(h, sp);
    if ((s = zd_valence(h, z, sp, v.psi, nv))) return s;
    for (int b0 = 0; b0 < cb; b0 += z.cb) {
        const int n = std::min(z.cb, cb - b0);
        if ((s = zd_conduction(h, z, h->cond.psi, c0 + b0, n)) ||
            (s = zd_block(h, z, sp, pp, 0, 0, 0, nv, n, (double2 *)M + (int64_t)b0 * nv * sp.ng, 1, nv)))
            return s;
    }
    return GW_OK;
}

gw_status gw_chi0_pair_elements(gw_chi0 *h, int iq, int64_t pair_begin, int64_t pair_count, double *M)
{
    if (!h) return GW_ERR_ARG;
    gw_status s = check_slot(h, iq);
    if (s) return s;
    const BandSet &v = h->val[iq];
    int64_t P = (int64_t)v.nb * h->cond.nb;
    if (pair_begin < 0 || pair_count < 0 || pair_begin + pair_count > P)
        return fail(h, GW_ERR_ARG, "pair range [%lld, %lld) outside [0, %lld)", (long long)pair_begin,
                    (long long)(pair_begin + pair_count), (long long)P);
    if (pair_count && !M) return fail(h, GW_ERR_ARG, "null M");
    Scope sc(h, "pair_mtxel");
    CK(h, run_pair(h, v.psi, h->cond.psi, h->cond.nb, pair_begin, pair_count, pair_plan(h, h->sph[iq]),
                   (double2 *)M),
       "pair kernel");
    return GW_OK;
}

static gw_status compute(gw_chi0 *h, int nq, const int *iq, int nw, const double *omega, double *chi, double *diag)
{
    if (nq < 1 || !iq || nw < 1 || nw > gw::kMaxOmega || !omega || !chi)
        return fail(h, GW_ERR_ARG, "bad arguments (nq >= 1, 1 <= nw <= %d, non-null pointers)", gw::kMaxOmega);
    gw::OmegaList om;
    om.nw = nw;
    for (int i = 0; i < nw; ++i) {
        if (!(omega[i] >= 0.0) || !std::isfinite(omega[i])) return fail(h, GW_ERR_ARG, "omega must be finite and >= 0");
        om.w[i] = omega[i];
    }
    for (int i = 0; i < nq; ++i) {
        gw_status s = check_slot(h, iq[i]);
        if (s) return s;
    }
    size_t off = 0, doff = 0;
    for (int i = 0; i < nq; ++i) {
        const Sphere &sp = h->sph[iq[i]];
        const BandSet &v = h->val[iq[i]];
        const int ng = sp.ng;
        const int64_t P = (int64_t)v.nb * h->cond.nb;
        const int64_t chunk = std::min<int64_t>(h->d.pair_chunk, P);
        double2 *cq = (double2 *)chi + off;
        double *dq = diag ? diag + doff : nullptr;
        CK(h, cudaMemsetAsync(cq, 0, sizeof(double2) * (size_t)nw * ng * ng, h->st), "zero chi");
        if (dq) CK(h, cudaMemsetAsync(dq, 0, sizeof(double) * (size_t)nw * ng, h->st), "zero diag");
        gw::PairPlan pp = pair_plan(h, sp);
        bool keep = false;
        gw_status s = resident_begin(h, P, ng, &keep);
        if (s) return s;
        double2 *Mres = keep ? h->Mres : nullptr;
        ZdPlan z;
        ZdUse use{h};
        if (fault_chunk() < 0 && (s = zd_plan(h, sp, v.nb, h->cond.nb, keep, false, 1, nw, 0, chunk, z))) return s;
        if (z.on) {
            const int nc = h->cond.nb;
            if ((s = ensure_work(h, keep ? 0 : (size_t)z.vb * z.cb * ng, (size_t)z.vb * z.cb * nw)) ||
                (s = zd_valence(h, z, sp, v.psi, v.nb)))
                return s;
            for (int c0 = 0; c0 < nc; c0 += z.cb) {
                const int cb = std::min(z.cb, nc - c0);
                if ((s = zd_conduction(h, z, h->cond.psi, c0, cb))) return s;
                for (int v0 = 0; v0 < v.nb; v0 += z.vb) {
                    const int vb = std::min(z.vb, v.nb - v0);
                    const int64_t cnt = (int64_t)vb * cb; // rows vl cb + cl
                    double2 *Mc = keep ? Mres + (int64_t)v0 * nc * ng : h->Mbuf;
                    if ((s = zd_block(h, z, sp, pp, 0, 0, v0, vb, cb, Mc, cb, 1))) return s;
                    {
                        Scope sc(h, "delta");
                        CK(h, gw::launch_delta(v.energy + v0, h->cond.energy + c0, cb, 0, cnt, om, h->dbuf, h->st),
                           "delta");
                    }
                    if ((s = contract_chunk(h, Mc, cnt, ng, h->dbuf, cnt, nw, cq))) return s;
                    if (dq) {
                        Scope sc(h, "diag");
                        CK(h, gw::launch_diag(Mc, cnt, ng, h->dbuf, cnt, nw, dq, ng, h->st), "diag");
                    }
                }
            }
            Scope sc(h, "symmetrize");
            CK(h, gw::launch_symmetrize(cq, ng, nw, h->st), "symmetrize");
            off += (size_t)nw * ng * ng;
            doff += (size_t)nw * ng;
            if (keep) h->Mres_iq = iq[i];
            continue;
        }
        const int64_t fault_at = fault_chunk();
        // with several frequencies the contractions queue up behind the two slice buffers: one stream
        if (nw == 1 && overlap_enabled(h, sp, pp, keep) && fault_at < 0) {
            s = compute_overlap(h, iq[i], om, cq, dq, Mres);
            if (s && s != GW_ERR_OOM) return s;
            if (!s) {
                Scope sc(h, "symmetrize");
                CK(h, gw::launch_symmetrize(cq, ng, nw, h->st), "symmetrize");
                off += (size_t)nw * ng * ng;
                doff += (size_t)nw * ng;
                if (keep) h->Mres_iq = iq[i];
                continue;
            }
            // no room for a second slice buffer: one stream
            drop_overlap(h);
            CK(h, cudaMemsetAsync(cq, 0, sizeof(double2) * (size_t)nw * ng * ng, h->st), "zero chi");
            if (dq) CK(h, cudaMemsetAsync(dq, 0, sizeof(double) * (size_t)nw * ng, h->st), "zero diag");
        }
        s = ensure_work(h, (size_t)chunk * ng, (size_t)chunk * nw);
        if (s) return s;
        for (int64_t p0 = 0, k = 0; p0 < P; p0 += chunk, ++k) {
            int64_t cnt = std::min(chunk, P - p0);
            if (k == fault_at) return fail(h, GW_ERR_CUDA, "injected host-side fault before chunk %lld", (long long)k);
            double2 *Mc = Mres ? Mres + p0 * ng : h->Mbuf;
            {
                Scope sc(h, "pair_mtxel");
                CK(h, run_pair(h, v.psi, h->cond.psi, h->cond.nb, p0, cnt, pp, Mc), "pair kernel");
            }
            {
                Scope sc(h, "delta");
                CK(h, gw::launch_delta(v.energy, h->cond.energy, h->cond.nb, p0, cnt, om, h->dbuf, h->st), "delta");
            }
            s = contract_chunk(h, Mc, cnt, ng, h->dbuf, cnt, nw, cq);
            if (s) return s;
            if (dq) {
                Scope sc(h, "diag");
                CK(h, gw::launch_diag(Mc, cnt, ng, h->dbuf, cnt, nw, dq, ng, h->st), "diag");
            }
        }
        {
            Scope sc(h, "symmetrize");
            CK(h, gw::launch_symmetrize(cq, ng, nw, h->st), "symmetrize");
        }
        off += (size_t)nw * ng * ng;
        doff += (size_t)nw * ng;
        if (keep) h->Mres_iq = iq[i];
    }
    return GW_OK;
}

gw_status gw_chi0_compute(gw_chi0 *h, int nq, const int *iq, int nw, const double *omega, double *chi, double *diag)
{
    if (!h) return GW_ERR_ARG;
    return zd_or_fft(h, [&] { return compute(h, nq, iq, nw, omega, chi, diag); });
}

gw_status gw_chi0_keep_pair_elements(gw_chi0 *h, int enable)
{
    if (!h) return GW_ERR_ARG;
    if (enable != 0 && enable != 1) return fail(h, GW_ERR_ARG, "enable must be 0 or 1");
    h->keep_m = enable == 1;
    h->Mres_iq = -1;
    if (!h->keep_m && h->Mres) {
        CK(h, cudaStreamSynchronize(h->st), "release resident pair elements");
        dfree(h, h->Mres, h->Mres_cap);
        h->Mres = nullptr;
        h->Mres_cap = 0;
    }
    return GW_OK;
}

gw_status gw_chi0_compute_batch(gw_chi0 *h, int nq, const int *iq, int nw, const double *omega, double *chi,
                                double *diag)
{
    if (!h) return GW_ERR_ARG;
    if (nq < 1 || !iq || nw < 1 || nw > gw::kMaxOmega || !omega || !chi)
        return fail(h, GW_ERR_ARG, "bad arguments (nq >= 1, 1 <= nw <= %d, non-null pointers)", gw::kMaxOmega);
    gw::OmegaList om;
    om.nw = nw;
    for (int i = 0; i < nw; ++i) {
        if (!(omega[i] >= 0.0) || !std::isfinite(omega[i])) return fail(h, GW_ERR_ARG, "omega must be finite and >= 0");
        om.w[i] = omega[i];
    }
    for (int i = 0; i < nq; ++i) {
        gw_status s = check_slot(h, iq[i]);
        if (s) return s;
        for (int j = 0; j < i; ++j)
            if (iq[j] == iq[i]) return fail(h, GW_ERR_ARG, "slot %d requested twice", iq[i]);
    }
    return zd_or_fft(h, [&] { return compute_batch(h, nq, iq, nw, omega, om, chi, diag); });
}

int gw_chi0_tuning(const gw_chi0 *h, int *tile_f64, int *waves_f64, int *tile_split)
{
    if (!h) return 0;
    if (tile_f64) *tile_f64 = h->tuned_bt;
    if (waves_f64) *waves_f64 = h->tuned_waves;
    if (tile_split) *tile_split = 256;
    return (int)h->tune_cache.size();
}

gw_status gw_chi0_contract(gw_chi0 *h, int nv, int nc, const double *ev, const double *ec, int ng, const double *M,
                           int nw, const double *omega, double *chi)
{
    if (!h) return GW_ERR_ARG;
    if (nv < 1 || nc < 1 || ng < 1 || nw < 1 || nw > gw::kMaxOmega || !ev || !ec || !M || !omega || !chi)
        return fail(h, GW_ERR_ARG, "bad arguments");
    gw::OmegaList om;
    om.nw = nw;
    for (int i = 0; i < nw; ++i) {
        if (!(omega[i] >= 0.0) || !std::isfinite(omega[i])) return fail(h, GW_ERR_ARG, "omega must be finite and >= 0");
        om.w[i] = omega[i];
    }
    const int64_t P = (int64_t)nv * nc;
    {
        std::vector<double> hv(nv), hc(nc);
        CK(h, cudaMemcpyAsync(hv.data(), ev, sizeof(double) * nv, cudaMemcpyDeviceToHost, h->st), "copy ev");
        CK(h, cudaMemcpyAsync(hc.data(), ec, sizeof(double) * nc, cudaMemcpyDeviceToHost, h->st), "copy ec");
        CK(h, cudaStreamSynchronize(h->st), "contract sync");
        if (!(*std::max_element(hv.begin(), hv.end()) < *std::min_element(hc.begin(), hc.end())))
            return fail(h, GW_ERR_ARG, "a valence energy is not below every conduction energy");
    }
    const int64_t chunk = std::min<int64_t>(h->d.pair_chunk, P);
    gw_status s = ensure_work(h, 0, (size_t)chunk * nw);
    if (s) return s;
    CK(h, cudaMemsetAsync(chi, 0, sizeof(double2) * (size_t)nw * ng * ng, h->st), "zero chi");
    for (int64_t p0 = 0; p0 < P; p0 += chunk) {
        const int64_t cnt = std::min(chunk, P - p0);
        {
            Scope sc(h, "delta");
            CK(h, gw::launch_delta(ev, ec, nc, p0, cnt, om, h->dbuf, h->st), "delta");
        }
        s = contract_chunk(h, (const double2 *)M + p0 * ng, cnt, ng, h->dbuf, cnt, nw, (double2 *)chi, true);
        if (s) return s;
    }
    Scope sc(h, "symmetrize");
    CK(h, gw::launch_symmetrize((double2 *)chi, ng, nw, h->st), "symmetrize");
    return GW_OK;
}

gw_status gw_chi0_sync(gw_chi0 *h)
{
    if (!h) return GW_ERR_ARG;
    int st = 0;
    CK(h, cudaMemcpyAsync(&st, h->status, sizeof(int), cudaMemcpyDeviceToHost, h->st), "status");
    CK(h, cudaStreamSynchronize(h->st), "sync");
    if (st != 0) { // on the handle's stream, and done before the caller may go on with another one
        CK(h, cudaMemsetAsync(h->status, 0, sizeof(int), h->st), "status reset");
        if ((st & gw::kStatusTimeout) && h->ozflags) // parts that never met leave their counters behind
            CK(h, cudaMemsetAsync(h->ozflags, 0, h->ozflags_cap, h->st), "split tile counters");
        CK(h, cudaStreamSynchronize(h->st), "status reset");
    }
    if (st & gw::kStatusTimeout) return fail(h, GW_ERR_TIMEOUT, "a bounded device-side wait gave up");
    if (st & gw::kStatusNoSlot) return fail(h, GW_ERR_CUDA, "a pair block found no free scratch slot");
    if (st & gw::kStatusBounds) return fail(h, GW_ERR_CUDA, "an index outside its buffer (bounds-checked build)");
    return GW_OK;
}

gw_status gw_chi0_check_watchdog(gw_chi0 *h, long long iterations)
{
    if (!h) return GW_ERR_ARG;
    if (iterations < 1) return fail(h, GW_ERR_ARG, "iterations must be >= 1");
    CK(h, gw::launch_watchdog(iterations, h->status, h->st), "watchdog");
    return GW_OK;
}

gw_status gw_chi0_set_timing(gw_chi0 *h, int enable)
{
    if (!h) return GW_ERR_ARG;
    h->timing = enable != 0;
    return GW_OK;
}

int gw_chi0_timing(gw_chi0 *h, int n, char (*names)[32], double *ms, int64_t *launches, int reset)
{
    if (!h) return 0;
    drain_timing(h);
    int i = 0;
    for (auto &kv : h->acc) {
        if (i < n) {
            if (names) {
                std::strncpy(names[i], kv.first.c_str(), 31);
                names[i][31] = 0;
            }
            if (ms) ms[i] = kv.second.first;
            if (launches) launches[i] = kv.second.second;
        }
        ++i;
    }
    if (reset) h->acc.clear();
    return i;
}

size_t gw_chi0_device_bytes(const gw_chi0 *h) { return h ? h->bytes : 0; }

} // extern "C"

