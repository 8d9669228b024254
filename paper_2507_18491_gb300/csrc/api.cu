// The C ABI (include/lmfmm.h): context, validation, device setup (tree
// upload, M2L tabulation, translation matrices, near-field precomputation)
// and the matvec pipeline P2M -> M2M -> M2L -> L2L -> L2P (+ S2T).
#include <algorithm>
#include <chrono>
#include <map>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <type_traits>

#include "kernels.cuh"
#include "quad.cuh"

using namespace lmf;

namespace {

thread_local std::string g_err;

struct DevState {
    std::vector<void *> allocs;
    double *xyz = nullptr;           // sorted [N][3]
    int64_t *perm = nullptr;
    BoxDev *boxes = nullptr;
    int64_t *leaves = nullptr;
    int64_t nleaves = 0;
    int *pt_box = nullptr;           // leaf box of every sorted point (mixed form)
    LeafUnit *units = nullptr;       // P2M units: at most 128 points of one leaf, largest first
    int64_t nunits = 0;
    bool p2m_many = false;           // P2M by the kernel for units of many points
    bool leaf_fast = false;          // mixed form, p <= 15: P2M and L2P of k_leaf.cu
    cd *qh = nullptr, *ph = nullptr; // helical, sorted [N][3]
    void *me = nullptr, *le = nullptr; // [nbox][3][P], complex T (scaled)
    CompDev *comps = nullptr;
    GeomDev *geoms = nullptr;
    void *tab = nullptr;             // [ngeom][5][P][P], complex T (scaled)
    LayerScale lscale{};
    M2LPair *m2l = nullptr;
    M2LWork *m2lwork = nullptr;
    int64_t n_m2lwork = 0;
    void *tup = nullptr, *tdn = nullptr;   // [ngroup][P][P], complex T (scaled)
    void *tupT = nullptr, *tdnT = nullptr; // their transposes (SIMT forms: the transposed operator)
    float *yscr = nullptr;           // persistent kernel: per-CTA accumulator scratch
    int64_t *tchild = nullptr, *tparent = nullptr;
    GemmWork *gwork = nullptr;
    std::vector<int64_t> gwork_off;  // per child level: [off[l], off[l+1])
    void *tupi = nullptr, *tdni = nullptr;    // persistent kernel: tiled translation matrices (bf16 x 3)
    M2LWork *twork = nullptr;        // persistent kernel: translation items, per child level
    bool trans_tc = false;           // M2M / L2L on the persistent kernel (tensor_cores = 3)
    std::vector<int64_t> twork_off;
    NearPair *near = nullptr;
    cd *s2t = nullptr;               // near field: 8 combined coefficients per point pair
    S2TRow *s2twork = nullptr;       // near-field target rows
    int64_t n_s2twork = 0;
    S2TRowT *s2tworkT = nullptr;     // transposed near field: (near pair, source) rows
    int64_t n_s2tworkT = 0;
    // free-space near field: runs of sorted points near every leaf, as target / as source
    int *froff = nullptr, *froffT = nullptr, *fbox = nullptr;
    FreeRun *fruns = nullptr, *frunsT = nullptr;
    bool free_near = false;
    // position gradient (allocated by the first lmfmm_gradient call): checkpoints
    // of the forward pass's local expansions and helical charges, a field buffer,
    // and 20 derivative integrals per near point pair
    cd *le_ck = nullptr, *qh_ck = nullptr, *gfield = nullptr, *s2tg = nullptr;
    int *flag = nullptr;
    int *mvstatus = nullptr;         // matvec status word (bit 4: tensor-core wait gave up)
    int fail_m2l = 0;                // test hook: status bits the next forward M2L leaves
    int m2l_kernel = 0;              // 0 FP64 (oz: which), 1 FP32 SIMT, 2 tcgen05 streamed, 3 tcgen05 persistent
    cf *ephase = nullptr;            // sector kernel: phases G[d] per pair
    void *mepk = nullptr;            // ... and the packed multipole expansions it reads
    // FP64 form on the tensor cores (k_m2l_oz.cu): images of the sector blocks and their
    // transposes, packed inputs, per-CTA scratch
    bool oz = false;
    void *ozimg = nullptr, *ozimgT = nullptr, *ozpk = nullptr, *ozscr = nullptr;
    int nsm = 0;
    int ncta = 0;                    // CTAs that yscr and ozscr hold (none of their launches has more)
    cd *stage = nullptr;             // [2][N][3] for host-buffer matvec
    cudaEvent_t ev[9]{};
    bool ev_ok = false;
    bool mv_recorded = false;        // stage events hold a matvec
    double bytes = 0;
};

DevState *DS(lmfmm_ctx *c) { return (DevState *)c->dev; }

#define CK(call)                                                                           \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            ctx->err = std::string(#call) + ": " + cudaGetErrorString(e_);                 \
            return e_ == cudaErrorMemoryAllocation ? LMFMM_ERR_OOM : LMFMM_ERR_CUDA;       \
        }                                                                                  \
    } while (0)

void free_dev(lmfmm_ctx *ctx)
{
    DevState *d = DS(ctx);
    if (!d) return;
    cudaSetDevice(ctx->device);
    for (void *p : d->allocs) cudaFree(p);
    d->allocs.clear();
    if (d->ev_ok)
        for (auto &e : d->ev) cudaEventDestroy(e);
    delete d;
    ctx->dev = nullptr;
}

template <typename T>
lmfmm_status dalloc(lmfmm_ctx *ctx, T **p, size_t count)
{
    *p = nullptr;
    if (count == 0) count = 1;
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, count * sizeof(T));
    if (e != cudaSuccess) {
        ctx->err = "cudaMalloc of " + std::to_string(count * sizeof(T)) + " bytes: " +
                   cudaGetErrorString(e);
        return LMFMM_ERR_OOM;
    }
    DS(ctx)->allocs.push_back(q);
    DS(ctx)->bytes += (double)(count * sizeof(T));
    *p = (T *)q;
    return LMFMM_OK;
}

void dfree(lmfmm_ctx *ctx, void *p)
{
    auto &v = DS(ctx)->allocs;
    auto it = std::find(v.begin(), v.end(), p);
    if (it != v.end()) {
        cudaFree(p);
        v.erase(it);
    }
}

// Host to device on the stream of the kernels that read the copy, complete on return.  A plain
// cudaMemcpy from pageable memory runs on the legacy stream and may return before its last
// transfer has landed, and a non-blocking stream does not wait for that one.
cudaError_t copy_in(void *dst, const void *src, size_t bytes, cudaStream_t st)
{
    if (bytes == 0) return cudaSuccess;
    const cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
    return e != cudaSuccess ? e : cudaStreamSynchronize(st);
}

template <typename T>
lmfmm_status dupload(lmfmm_ctx *ctx, cudaStream_t st, T **p, const std::vector<T> &h)
{
    lmfmm_status s = dalloc(ctx, p, h.size());
    if (s) return s;
    CK(copy_in(*p, h.data(), h.size() * sizeof(T), st));
    return LMFMM_OK;
}

#define TRY(x)                        \
    do {                              \
        lmfmm_status s_ = (x);        \
        if (s_ != LMFMM_OK) return s_; \
    } while (0)

// k_rho quadrature plan of an M2L geometry: the Chebyshev integrands carry
// a polynomial of degree up to 2p+5 in k_rho.
QuadPlanDev geom_plan(double a, int p, double rho, double dz) { return make_plan(a, rho, dz, 2 * p + 5); }

lmfmm_status check_flag(lmfmm_ctx *ctx)
{
    int f = 0;
    CK(cudaMemcpy(&f, DS(ctx)->flag, sizeof(int), cudaMemcpyDeviceToHost));
    if (f) {
        ctx->err = "device quadrature hit its cap (flag " + std::to_string(f) + ")";
        return LMFMM_ERR_QUAD;
    }
    return LMFMM_OK;
}

// Status word of the matvec kernels, cleared by every call before its first
// kernel (a gradient is one call of two passes): a tensor-core wait that gave up
// leaves bit 4.  Reads it after the stream's work is done.
lmfmm_status check_mvstatus(lmfmm_ctx *ctx, cudaStream_t st)
{
    int f = 0;
    CK(cudaStreamSynchronize(st));
    CK(cudaMemcpy(&f, DS(ctx)->mvstatus, sizeof(int), cudaMemcpyDeviceToHost));
    if (f) {
        ctx->err = "matvec: a bounded tensor-core wait gave up (status " + std::to_string(f) +
                   "); the result is incomplete";
        return LMFMM_ERR_TIMEOUT;
    }
    return LMFMM_OK;
}

// M2L work items of a built context: per geometry and table, runs of pairs
// giving at most `bn` helical columns (one column per pair for the (s5, 0)
// table, two for the others); prob tags them for a batched launch.  Returns the
// column count.
int64_t m2l_work_items(const lmfmm_ctx *ctx, int bn, int prob, std::vector<M2LWork> &mw)
{
    int64_t ncols = 0;
    for (size_t gi = 0; gi < ctx->geoms.size(); ++gi) {
        const Geom &g = ctx->geoms[gi];
        const CompDev &cg = ctx->comps[g.comp];
        // image maps of the component: the sign of odd degrees flips when the
        // source (target) side is mirrored an odd number of times
        const int flags = (((cg.s < 0) != (cg.has_src_refl != 0)) ? 1 : 0) |
                          (((cg.s < 0) != (cg.has_tgt_refl != 0)) ? 2 : 0);
        for (int t = 0; t < NTAB; ++t) {
            const int per = (t == 1) ? bn : bn / 2;
            for (int64_t q = g.pair0; q < g.pair1; q += per) {
                M2LWork w{};
                w.geom = (int)gi;
                w.t = t;
                w.flags = flags;
                w.pair0 = q;
                w.npair = (int)std::min<int64_t>(per, g.pair1 - q);
                w.prob = prob;
                ncols += w.npair * (t == 1 ? 1 : 2);
                mw.push_back(w);
            }
        }
    }
    return ncols;
}

// Work items of the sector kernels: per geometry, runs of at most `pairs` pairs.
void sec_work_items(const lmfmm_ctx *ctx, int pairs, int prob, std::vector<M2LWork> &mw)
{
    for (size_t gi = 0; gi < ctx->geoms.size(); ++gi) {
        const Geom &g = ctx->geoms[gi];
        for (int64_t q = g.pair0; q < g.pair1; q += pairs) {
            M2LWork w{};
            w.geom = (int)gi;
            w.pair0 = q;
            w.npair = (int)std::min<int64_t>(pairs, g.pair1 - q);
            w.prob = prob;
            mw.push_back(w);
        }
    }
}

// Tabulate a list of geometries into `tab` (device), batching node factors
// and Chebyshev integrals through a scratch buffer.
lmfmm_status tabulate(lmfmm_ctx *ctx, std::vector<GeomDev> &hg, const CompDev *dcomps,
                      const cd *dG, const int *dcg, cd *tab, cudaStream_t st, float *ms = nullptr)
{
    const int p = ctx->prm.p;
    const int LM = p + 2, DJ = 2 * p + 3;
    const int64_t per_node = 5 + 4 + 4 + LM + DJ;
    const int64_t ibr = tab_integrals(p);
    const size_t scratch_bytes = (size_t)1 << 30;
    // batches
    std::vector<int> bstart;
    std::vector<int64_t> bstride;
    int ng = (int)hg.size();
    int g = 0;
    while (g < ng) {
        int64_t nodes = 0;
        int gb = g;
        while (gb < ng) {
            int64_t q = plan_nodes(hg[gb].plan);
            int64_t need = (nodes + q) * per_node + (int64_t)(gb - g + 1) * ibr;
            if ((size_t)need * sizeof(cd) > scratch_bytes && gb > g) break;
            hg[gb].node0 = nodes;
            nodes += q;
            ++gb;
            if (gb - g >= 2048) break;
        }
        for (int i = g; i < gb; ++i) hg[i].stride = nodes;
        bstart.push_back(g);
        bstride.push_back(nodes);
        g = gb;
    }
    bstart.push_back(ng);
    size_t need_max = 0;
    for (size_t b = 0; b + 1 < bstart.size(); ++b)
        need_max = std::max(need_max, (size_t)(bstride[b] * per_node +
                                               (int64_t)(bstart[b + 1] - bstart[b]) * ibr));
    GeomDev *dgeo = nullptr;
    cd *scr = nullptr;
    void *qg = nullptr, *qs = nullptr;
    CK(cudaMalloc(&qg, std::max<size_t>(1, hg.size()) * sizeof(GeomDev)));
    dgeo = (GeomDev *)qg;
    cudaError_t e = cudaMalloc(&qs, std::max<size_t>(1, need_max) * sizeof(cd));
    if (e != cudaSuccess) {
        cudaFree(qg);
        ctx->err = "tabulation scratch allocation failed";
        return LMFMM_ERR_OOM;
    }
    scr = (cd *)qs;
    lmfmm_status rc = LMFMM_OK;
    if (copy_in(dgeo, hg.data(), hg.size() * sizeof(GeomDev), st)) rc = LMFMM_ERR_CUDA;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    const bool timed = ms && cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess;
    if (timed) cudaEventRecord(e0, st);
    for (size_t b = 0; rc == LMFMM_OK && b + 1 < bstart.size(); ++b) {
        int g0 = bstart[b], nb = bstart[b + 1] - g0;
        int qmax = 0;
        for (int i = g0; i < g0 + nb; ++i) qmax = std::max(qmax, plan_nodes(hg[i].plan));
        launch_tab_batch(dgeo, g0, nb, qmax, ctx->med, dcomps, p, dG, dcg, scr, bstride[b], tab,
                         DS(ctx)->flag, st);
        if (cudaGetLastError() != cudaSuccess) rc = LMFMM_ERR_CUDA;
    }
    if (timed) cudaEventRecord(e1, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) rc = LMFMM_ERR_CUDA;
    if (timed) {
        if (cudaEventElapsedTime(ms, e0, e1) != cudaSuccess) *ms = 0.f;
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
    }
    cudaFree(qg);
    cudaFree(qs);
    if (rc) {
        ctx->err = "tabulation kernels failed";
        return rc;
    }
    return check_flag(ctx);
}

}  // namespace

namespace lmf {
// the M2L work items the matvec builds, for the host-side plan check (plan.cpp)
int64_t plan_work_items(const lmfmm_ctx *ctx, int bn, std::vector<M2LWork> &mw)
{
    return m2l_work_items(ctx, bn, 0, mw);
}

void plan_sector_items(const lmfmm_ctx *ctx, int pairs, std::vector<M2LWork> &mw) { sec_work_items(ctx, pairs, 0, mw); }

// read-only view of the device state for lmfmm_direct_noalloc (noalloc.cu)
bool noalloc_state(lmfmm_ctx *ctx, const int64_t **perm, const BoxDev **boxes, const double **xyz,
                   const CompDev **comps, cd **qh, cd **ph, int **flag)
{
    DevState *d = DS(ctx);
    if (!d || !d->perm || !d->boxes || !d->xyz || !d->comps || !d->qh || !d->ph || !d->flag)
        return false;
    *perm = d->perm;
    *boxes = d->boxes;
    *xyz = d->xyz;
    *comps = d->comps;
    *qh = d->qh;
    *ph = d->ph;
    *flag = d->flag;
    return true;
}
}  // namespace lmf

// --------------------------------------------------------------------- ABI
extern "C" {

lmfmm_status lmfmm_default_params(lmfmm_params *prm)
{
    if (!prm) return LMFMM_ERR_ARG;
    prm->p = 8;
    prm->depth = -1;
    prm->leaf_cap = 64;
    prm->theta = 0.55;
    prm->eta = 0.1;
    prm->quad_tol = 1e-15;
    prm->precision = LMFMM_FP64;
    prm->tensor_cores = 1;
    prm->quad_node_cap = 1 << 20;
    prm->components = LMFMM_REACTION;
    return LMFMM_OK;
}

lmfmm_status lmfmm_create(lmfmm_ctx **out, const lmfmm_params *prm, int device)
{
    if (!out || !prm) {
        g_err = "lmfmm_create: NULL argument";
        return LMFMM_ERR_ARG;
    }
    *out = nullptr;
    if (prm->p < 1 || prm->p > 16 || !(prm->theta > 0 && prm->theta < 1) || !(prm->eta >= 0) ||
        prm->depth > 20 || (prm->depth < 0 && prm->leaf_cap < 1)) {
        g_err = "lmfmm_create: parameter out of range (1 <= p <= 16, 0 < theta < 1, eta >= 0, "
                "depth <= 20)";
        return LMFMM_ERR_ARG;
    }
    if (prm->precision != LMFMM_FP64 && prm->precision != LMFMM_MIXED) {
        g_err = "lmfmm_create: precision must be LMFMM_FP64 or LMFMM_MIXED";
        return LMFMM_ERR_ARG;
    }
    if (prm->tensor_cores < 0 || prm->tensor_cores > 3) {
        g_err = "lmfmm_create: tensor_cores must be 0, 1, 2 or 3";
        return LMFMM_ERR_ARG;
    }
    if (prm->components < LMFMM_REACTION || prm->components > LMFMM_TOTAL) {
        g_err = "lmfmm_create: components must be LMFMM_REACTION, LMFMM_FREE or LMFMM_TOTAL";
        return LMFMM_ERR_ARG;
    }
    if (prm->quad_node_cap < 64) {
        g_err = "lmfmm_create: quad_node_cap must be at least 64";
        return LMFMM_ERR_ARG;
    }
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) {
        g_err = std::string("cudaSetDevice: ") + cudaGetErrorString(e);
        return LMFMM_ERR_CUDA;
    }
    if ((e = configure_fmm_kernels()) != cudaSuccess || (e = configure_tab_kernels()) != cudaSuccess ||
        (e = configure_leaf_fast()) != cudaSuccess) {
        g_err = std::string("kernel configuration: ") + cudaGetErrorString(e);
        return LMFMM_ERR_CUDA;
    }
    lmfmm_ctx *ctx = new lmfmm_ctx();
    ctx->device = device;
    ctx->prm = *prm;
    *out = ctx;
    return LMFMM_OK;
}

lmfmm_status lmfmm_set_layers(lmfmm_ctx *ctx, int L, const double *d, const lmfmm_c128 *k)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (L < 0 || L > LMF_MAXL || (L > 0 && !d) || !k) {
        ctx->err = "set_layers: need 0 <= L <= " + std::to_string(LMF_MAXL) + " and non-NULL arrays";
        return LMFMM_ERR_ARG;
    }
    for (int i = 0; i < L; ++i) {
        if (!std::isfinite(d[i]) || (i > 0 && !(d[i] < d[i - 1]))) {
            ctx->err = "set_layers: interfaces must be finite and strictly decreasing";
            return LMFMM_ERR_ARG;
        }
    }
    for (int i = 0; i <= L; ++i) {
        if (!std::isfinite(k[i].re) || !std::isfinite(k[i].im) || k[i].im < 0 ||
            (k[i].re == 0 && k[i].im == 0)) {
            ctx->err = "set_layers: wavenumber " + std::to_string(i) + " must be finite, nonzero, Im >= 0";
            return LMFMM_ERR_ARG;
        }
    }
    ctx->med = MediumDev{};
    ctx->med.L = L;
    for (int i = 0; i < L; ++i) ctx->med.d[i] = d[i];
    for (int i = 0; i <= L; ++i) ctx->med.k[i] = cd{k[i].re, k[i].im};
    ctx->layers_set = true;
    ctx->built = false;
    return LMFMM_OK;
}

lmfmm_status lmfmm_set_points(lmfmm_ctx *ctx, int64_t N, const double *xyz)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (!ctx->layers_set) {
        ctx->err = "set_points: call lmfmm_set_layers first";
        return LMFMM_ERR_STATE;
    }
    if (N < 1 || !xyz) {
        ctx->err = "set_points: need N >= 1 and a non-NULL array";
        return LMFMM_ERR_ARG;
    }
    ctx->N = N;
    ctx->xyz.assign(xyz, xyz + 3 * N);
    ctx->built = false;
    lmfmm_status s = classify_and_sort(ctx);
    ctx->points_set = (s == LMFMM_OK);
    return s;
}

lmfmm_status lmfmm_set_points_device(lmfmm_ctx *ctx, int64_t N, const double *xyz, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (N < 1 || !xyz) {
        ctx->err = "set_points_device: need N >= 1 and a non-NULL array";
        return LMFMM_ERR_ARG;
    }
    CK(cudaSetDevice(ctx->device));
    std::vector<double> h((size_t)N * 3);
    cudaStream_t st = (cudaStream_t)stream;
    CK(cudaMemcpyAsync(h.data(), xyz, h.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    return lmfmm_set_points(ctx, N, h.data());
}

lmfmm_status lmfmm_build(lmfmm_ctx *ctx, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (!ctx->points_set) {
        ctx->err = "build: call lmfmm_set_points first";
        return LMFMM_ERR_STATE;
    }
    auto t0 = std::chrono::steady_clock::now();
    CK(cudaSetDevice(ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    free_dev(ctx);
    ctx->dev = new DevState();
    DevState *d = DS(ctx);
    ctx->built = false;
    TRY(build_host_structures(ctx));
    chebyshev_tables(ctx);
    const int p = ctx->prm.p, P = (p + 1) * (p + 1);
    const int64_t N = ctx->N, nbox = (int64_t)ctx->boxes.size();
    // memory estimate (tables dominate)
    const bool img_path = ctx->prm.precision == LMFMM_MIXED &&
                          (ctx->prm.tensor_cores == 1 || ctx->prm.tensor_cores == 3) && m2l_sec_supported(p);
    double need = (double)ctx->geoms.size() * NTAB * P * P * 16.0 +
                  (img_path ? (double)m2l_sec_image_bytes(p, (int64_t)ctx->geoms.size()) +
                                  (double)ctx->m2l.size() * m2l_sec_phases(p) * 8.0
                            : 0.0) +
                  (double)nbox * 6 * P * 16.0 + (double)ctx->tgroups.size() * 2 * P * P * 16.0 +
                  (double)ctx->n_near_pp * 13 * 16.0 + (double)N * 200.0;
    size_t fr = 0, tot = 0;
    CK(cudaMemGetInfo(&fr, &tot));
    if (need > 0.85 * (double)fr) {
        ctx->err = "build: needs about " + std::to_string(need / 1e9) + " GB of device memory, " +
                   std::to_string(fr / 1e9) + " GB free (reduce p or raise theta/depth)";
        return LMFMM_ERR_OOM;
    }
    CK(cudaDeviceGetAttribute(&d->nsm, cudaDevAttrMultiProcessorCount, ctx->device));
    // FP64 form: the tensor-core M2L holds two images of 32 bytes per sector entry (eight digits of
    // a complex number; 4.33 MB each per geometry at p = 12, where the five tables of the SIMT kernels
    // take 2.28 MB).  The SIMT kernels run where both do not fit, or on request
    if (ctx->prm.precision == LMFMM_FP64 && ctx->prm.tensor_cores != 0 && m2l_oz_supported(p)) {
        const double oz_need = 2.0 * (double)m2l_oz_image_bytes(p, (int64_t)ctx->geoms.size()) +
                               (double)m2l_oz_packed_bytes(p, nbox) + (double)m2l_oz_scratch_bytes(p, d->nsm);
        d->oz = need + oz_need <= 0.85 * (double)fr;
    }
    CK(cudaMalloc((void **)&d->flag, sizeof(int)));
    d->allocs.push_back(d->flag);
    CK(cudaMemsetAsync(d->flag, 0, sizeof(int), st));
    CK(cudaMalloc((void **)&d->mvstatus, sizeof(int)));
    d->allocs.push_back(d->mvstatus);
    CK(cudaMemsetAsync(d->mvstatus, 0, sizeof(int), st));
    for (auto &e : d->ev) CK(cudaEventCreate(&e));
    d->ev_ok = true;
    // points and boxes
    TRY(dupload(ctx, st, &d->xyz, ctx->sxyz));
    TRY(dupload(ctx, st, &d->perm, ctx->perm));
    std::vector<BoxDev> hb(nbox);
    std::vector<int64_t> leaves;
    for (int64_t i = 0; i < nbox; ++i) {
        const Box &b = ctx->boxes[i];
        hb[i] = BoxDev{b.p0, b.p1, {b.c[0], b.c[1], b.c[2]}, b.layer, 0};
        if (b.level == ctx->depth) leaves.push_back(i);
    }
    TRY(dupload(ctx, st, &d->boxes, hb));
    TRY(dupload(ctx, st, &d->leaves, leaves));
    d->nleaves = (int64_t)leaves.size();
    if (ctx->prm.precision == LMFMM_MIXED && leaf_fast_supported(p)) {
        std::vector<int> ptb(N > 0 ? N : 1, 0);
        std::vector<LeafUnit> units;
        for (int64_t li : leaves) {
            const Box &b = ctx->boxes[li];
            for (int64_t q = b.p0; q < b.p1; ++q) ptb[q] = (int)li;
            for (int64_t c0 = b.p0; c0 < b.p1; c0 += 128)
                units.push_back(LeafUnit{c0, std::min<int64_t>(c0 + 128, b.p1), (int)li, b.p1 - b.p0 <= 128 ? 1 : 0});
        }
        // largest units first, so that the last wave is made of small ones
        std::stable_sort(units.begin(), units.end(),
                         [](const LeafUnit &a, const LeafUnit &b) { return a.i1 - a.i0 > b.i1 - b.i0; });
        TRY(dupload(ctx, st, &d->pt_box, ptb));
        TRY(dupload(ctx, st, &d->units, units));
        d->nunits = (int64_t)units.size();
        // k_p2m_ms takes a time per point, k_p2m_pt one per unit (two layers at depth 5, 7.5 / 30 / 60 /
        // 120 points per unit: p = 6 45 / 84 / 143 / 239 against 65 / 74 / 86 / 127 us, p = 8 53 / 98 /
        // 172 / 288 against 91 / 106 / 123 / 192, p = 12 73 / 139 / 242 / 415 against 204 / 210 / 236 / 339);
        // they meet near 5 p points.  Not both in one call: two launches in a row lose more
        d->p2m_many = N > 5 * p * d->nunits;
        d->leaf_fast = true;
    }
    TRY(dalloc(ctx, &d->qh, 3 * N));
    TRY(dalloc(ctx, &d->ph, 3 * N));
    const bool f32 = ctx->prm.precision == LMFMM_MIXED;
    d->m2l_kernel = !f32 ? 0
                    : ctx->prm.tensor_cores == 0 ? 1
                    : ((ctx->prm.tensor_cores == 1 || ctx->prm.tensor_cores == 3) && m2l_sec_supported(p)) ? 3
                    : m2l_tc_supported(p) ? 2 : 1;
    const size_t esz = f32 ? sizeof(cf) : sizeof(cd);
    {
        unsigned char *q1 = nullptr, *q2 = nullptr;
        TRY(dalloc(ctx, &q1, (size_t)nbox * 3 * P * esz));
        TRY(dalloc(ctx, &q2, (size_t)nbox * 3 * P * esz));
        d->me = q1;
        d->le = q2;
    }
    const double Sroot = 2.0 * ctx->root_h;
    auto lev_size = [&](int lev) { return Sroot / (double)(1u << lev); };
    auto kabs = [&](int layer) { return std::hypot(ctx->med.k[layer].x, ctx->med.k[layer].y); };
    for (int j = 0; j <= ctx->med.L; ++j) d->lscale.s[j] = kabs(j) * lev_size(ctx->depth);
    TRY(dupload(ctx, st, &d->comps, ctx->comps));
    cd *dG = nullptr;
    int *dcg = nullptr;
    TRY(dupload(ctx, st, &dG, ctx->Gten));
    TRY(dupload(ctx, st, &dcg, ctx->comp_gidx));
    // M2L geometries, tables and work items
    const double a = medium_a(ctx->med);
    std::vector<GeomDev> hg(ctx->geoms.size());
    int64_t qtot = 0;
    double tab_terms = 0;   // per node: (tau, tau', table) combinations formed (10 of 16 within a layer)
    float ms_tab = 0.f;
    for (size_t i = 0; i < ctx->geoms.size(); ++i) {
        const Geom &g = ctx->geoms[i];
        const CompDev &c = ctx->comps[g.comp];
        GeomDev gd{};
        gd.comp = g.comp;
        if (i >= ctx->n_react_geoms) {
            // free-space table: built on the host (addition theorem), not tabulated
            gd.rho = g.rho;
            gd.zs = g.zs;
            gd.zt = g.zt;
            gd.scale_s = gd.scale_t = kabs(c.l) * lev_size(g.level);
            gd.tab_index = (int64_t)i;
            hg[i] = gd;
            continue;
        }
        gd.src_primary = std::hypot(ctx->med.k[c.l].x, ctx->med.k[c.l].y) <=
                         std::hypot(ctx->med.k[c.lp].x, ctx->med.k[c.lp].y);
        gd.rho = g.rho;
        gd.zs = g.zs;
        gd.zt = g.zt;
        gd.plan = geom_plan(a, p, g.rho, c.s * (g.zs - g.zt));
        gd.scale_s = kabs(c.l) * lev_size(g.level);
        gd.scale_t = kabs(c.lp) * lev_size(g.level);
        if (plan_nodes(gd.plan) > ctx->prm.quad_node_cap) {
            ctx->err = "build: an M2L geometry needs " + std::to_string(plan_nodes(gd.plan)) +
                       " quadrature nodes, more than quad_node_cap = " + std::to_string(ctx->prm.quad_node_cap);
            return LMFMM_ERR_QUAD;
        }
        qtot += plan_nodes(gd.plan);
        tab_terms += (double)plan_nodes(gd.plan) * NTAB * (c.l == c.lp ? 10 : 16);
        gd.tab_index = (int64_t)i;
        hg[i] = gd;
    }
    {
        // FP64 Chebyshev tabulation, then level scaling (and cast for the mixed form)
        cd *tab64 = nullptr;
        TRY(dalloc(ctx, &tab64, ctx->geoms.size() * (size_t)NTAB * P * P));
        if (ctx->n_react_geoms > 0) {
            std::vector<GeomDev> hr(hg.begin(), hg.begin() + ctx->n_react_geoms);
            TRY(tabulate(ctx, hr, d->comps, dG, dcg, tab64, st, &ms_tab));
        }
        if (!ctx->free_tables.empty())
            CK(copy_in(tab64 + ctx->n_react_geoms * (size_t)NTAB * P * P, ctx->free_tables.data(),
                       ctx->free_tables.size() * sizeof(cd), st));
        TRY(dupload(ctx, st, &d->geoms, hg));
        if (d->m2l_kernel == 3) {
            unsigned char *img = nullptr;
            TRY(dalloc(ctx, &img, m2l_sec_image_bytes(p, (int64_t)hg.size())));
            launch_sec_image(p, (int64_t)hg.size(), d->geoms, d->comps, tab64, img, st);
            CK(cudaGetLastError());
            CK(cudaStreamSynchronize(st));
            dfree(ctx, tab64);
            d->tab = img;
        } else if (f32) {
            cf *t32 = nullptr;
            TRY(dalloc(ctx, &t32, ctx->geoms.size() * (size_t)NTAB * P * P));
            launch_scale_tables<float>(p, 0, (int64_t)hg.size(), d->geoms, tab64, t32, st);
            CK(cudaGetLastError());
            CK(cudaStreamSynchronize(st));
            dfree(ctx, tab64);
            d->tab = t32;
        } else if (d->oz) {
            const int64_t ng = (int64_t)hg.size();
            unsigned char *q[3] = {};
            TRY(dalloc(ctx, &q[0], m2l_oz_image_bytes(p, ng)));
            TRY(dalloc(ctx, &q[1], m2l_oz_image_bytes(p, ng)));
            TRY(dalloc(ctx, &q[2], m2l_oz_packed_bytes(p, nbox)));
            launch_oz_images(p, ng, d->geoms, d->comps, tab64, q[0], q[1], st);
            CK(cudaGetLastError());
            CK(cudaStreamSynchronize(st));
            dfree(ctx, tab64);
            d->ozimg = q[0];
            d->ozimgT = q[1];
            d->ozpk = q[2];
        } else {
            launch_scale_tables<double>(p, 0, (int64_t)hg.size(), d->geoms, tab64, tab64, st);
            CK(cudaGetLastError());
            d->tab = tab64;
        }
    }
    TRY(dupload(ctx, st, &d->m2l, ctx->m2l));
    std::vector<M2LWork> mw;
    const int64_t ncols = 9 * (int64_t)ctx->m2l.size();   // helical columns: nine table applications per pair
    if (d->m2l_kernel == 3) {
        TRY(dalloc(ctx, &d->ephase, ctx->m2l.size() * (size_t)m2l_sec_phases(p)));
        unsigned char *pk = nullptr;
        TRY(dalloc(ctx, &pk, m2l_sec_packed_bytes(p, nbox)));
        d->mepk = pk;
        launch_pair_phases(p, (int64_t)ctx->m2l.size(), d->m2l, d->ephase, st);
        CK(cudaGetLastError());
        sec_work_items(ctx, m2l_sec_pairs(), 0, mw);
    } else if (d->oz) {
        // an item's time hardly depends on its pairs (padded products, one pass of phases): halve
        // them while the items still make one round of CTAs
        int pairs = m2l_oz_pairs();
        sec_work_items(ctx, pairs, 0, mw);
        while (pairs > m2l_oz_pairs() / 4) {
            std::vector<M2LWork> half;
            sec_work_items(ctx, pairs / 2, 0, half);
            if ((int64_t)half.size() > d->nsm) break;
            mw = half;
            pairs /= 2;
        }
    } else {
        m2l_work_items(ctx, d->m2l_kernel == 2 ? m2l_tc_cols() : f32 ? gemm_cols<float>() : gemm_cols<double>(), 0, mw);
    }
    TRY(dupload(ctx, st, &d->m2lwork, mw));
    d->n_m2lwork = (int64_t)mw.size();
    int64_t most_items = std::max<int64_t>(1, d->n_m2lwork);   // of one launch with a scratch per CTA
    // translation matrices (exact addition theorem), on the device from the groups' factors
    {
        const int64_t ngr = (int64_t)ctx->tgroups.size();
        const int nfac = trans_factor_count(p);
        std::vector<dd> fac((size_t)ngr * nfac), gw, gP;
        for (int64_t i = 0; i < ngr; ++i) {
            // scaled expansions: M~ = M / s^n, L~ = L s^nu, s = |k| S_level
            const TransGroup &g = ctx->tgroups[i];
            trans_factors(p, zc(ctx->med.k[g.layer].x, ctx->med.k[g.layer].y), g.t, kabs(g.layer) * lev_size(g.level),
                          kabs(g.layer) * lev_size(g.level - 1), &fac[i * nfac]);
        }
        gaunt_nodes(p, gw, gP);
        dd *dw = nullptr, *dP = nullptr, *dfac = nullptr;
        double *dGt = nullptr;
        cd *up64 = nullptr, *dn64 = nullptr;
        TRY(dupload(ctx, st, &dw, gw));
        TRY(dupload(ctx, st, &dP, gP));
        TRY(dupload(ctx, st, &dfac, fac));
        TRY(dalloc(ctx, &dGt, (size_t)P * P * (p + 1)));
        TRY(dalloc(ctx, &up64, (size_t)ngr * P * P));
        TRY(dalloc(ctx, &dn64, (size_t)ngr * P * P));
        launch_trans_build(p, (int)gw.size(), dw, dP, dGt, ngr, dfac, up64, dn64, st);
        CK(cudaGetLastError());
        d->trans_tc = d->m2l_kernel == 3 && ctx->prm.tensor_cores == 3 && trans_tc2_supported(p);
        // the SIMT forms also keep the transposes (the transposed operator runs on them)
        const bool want_tr = d->m2l_kernel <= 1;
        if (!f32) {
            d->tup = up64;
            d->tdn = dn64;
            cd *a1 = nullptr;
            for (int q = 0; q < 2; ++q) {
                TRY(dalloc(ctx, &a1, (size_t)ngr * P * P));
                launch_trans_copy<double>(p, ngr, true, q ? dn64 : up64, a1, st);
                (q ? d->tdnT : d->tupT) = a1;
            }
        } else if (!d->trans_tc) {
            cf *a1 = nullptr;
            for (int q = 0; q < (want_tr ? 4 : 2); ++q) {
                TRY(dalloc(ctx, &a1, (size_t)ngr * P * P));
                launch_trans_copy<float>(p, ngr, q >= 2, (q & 1) ? dn64 : up64, a1, st);
                (q == 0 ? d->tup : q == 1 ? d->tdn : q == 2 ? d->tupT : d->tdnT) = a1;
            }
        }
        TRY(dupload(ctx, st, &d->tchild, ctx->tpair_child));
        TRY(dupload(ctx, st, &d->tparent, ctx->tpair_parent));
        if (d->trans_tc) {
            // M2M / L2L on the persistent tensor-core kernel: tiled bf16 three-piece
            // images of the scaled FP64 matrices, items of 21 pairs (63 helical columns)
            unsigned char *a1 = nullptr, *a2 = nullptr;
            TRY(dalloc(ctx, &a1, (size_t)ngr * tc2_matrix_bytes(p)));
            TRY(dalloc(ctx, &a2, (size_t)ngr * tc2_matrix_bytes(p)));
            launch_tile_matrices(p, ngr, up64, a1, st);
            launch_tile_matrices(p, ngr, dn64, a2, st);
            d->tupi = a1;
            d->tdni = a2;
            std::vector<M2LWork> tw;
            d->twork_off.assign(ctx->depth + 2, 0);
            const int per = m2l_tc_cols() / 3;
            for (int lev = 1; lev <= ctx->depth; ++lev) {
                d->twork_off[lev] = (int64_t)tw.size();
                for (int64_t gi = 0; gi < ngr; ++gi) {
                    const TransGroup &g = ctx->tgroups[gi];
                    if (g.level != lev) continue;
                    for (int64_t q = g.pair0; q < g.pair1; q += per) {
                        M2LWork w{};
                        w.geom = (int)gi;
                        w.npair = (int)std::min<int64_t>(per, g.pair1 - q);
                        w.pair0 = q;
                        tw.push_back(w);
                    }
                }
            }
            d->twork_off[ctx->depth + 1] = (int64_t)tw.size();
            for (int lev = 1; lev <= ctx->depth; ++lev)
                most_items = std::max(most_items, d->twork_off[lev + 1] - d->twork_off[lev]);
            TRY(dupload(ctx, st, &d->twork, tw));
        }
        // work items per child level
        std::vector<GemmWork> gwk;
        d->gwork_off.assign(ctx->depth + 2, 0);
        for (int lev = 1; lev <= ctx->depth; ++lev) {
            d->gwork_off[lev] = (int64_t)gwk.size();
            for (size_t gi = 0; gi < ctx->tgroups.size(); ++gi) {
                const TransGroup &g = ctx->tgroups[gi];
                if (g.level != lev) continue;
                int per = (f32 ? gemm_cols<float>() : gemm_cols<double>()) / 3;
                for (int64_t q = g.pair0; q < g.pair1; q += per)
                    gwk.push_back(GemmWork{(int)gi, (int)std::min<int64_t>(per, g.pair1 - q), q});
            }
        }
        d->gwork_off[ctx->depth + 1] = (int64_t)gwk.size();
        TRY(dupload(ctx, st, &d->gwork, gwk));
        CK(cudaStreamSynchronize(st));
        for (void *q : {(void *)dw, (void *)dP, (void *)dGt, (void *)dfac}) dfree(ctx, q);
        if (f32) {
            dfree(ctx, up64);
            dfree(ctx, dn64);
        }
    }
    // scratch of the CTAs that a launch can have: a small problem has fewer items than the chip has SMs
    d->ncta = (int)std::min<int64_t>(d->nsm, most_items);
    if (d->m2l_kernel == 3) {
        // one scratch for the M2L and the translations, which run one after the other
        TRY(dalloc(ctx, &d->yscr, std::max(m2l_sec_scratch_floats(p, d->ncta), trans_tc2_scratch_floats(p, d->ncta))));
    } else if (d->oz) {
        unsigned char *q = nullptr;
        TRY(dalloc(ctx, &q, m2l_oz_scratch_bytes(p, d->ncta)));
        d->ozscr = q;
    }
    // near field
    TRY(dupload(ctx, st, &d->near, ctx->near));
    {
        // five Sommerfeld integrals per point pair, then the 8 combined coefficients
        cd *s2t5 = nullptr;
        TRY(dalloc(ctx, &s2t5, (size_t)ctx->n_near_pp * 5));
        launch_s2t_pre((int64_t)ctx->near.size(), d->near, d->boxes, d->xyz, ctx->med, d->comps, a,
                       ctx->prm.quad_node_cap, s2t5, d->flag, st);
        CK(cudaGetLastError());
        TRY(dalloc(ctx, &d->s2t, (size_t)ctx->n_near_pp * 8));
        launch_s2t_combine((int64_t)ctx->near.size(), d->near, d->boxes, d->xyz, s2t5, d->s2t, st);
        CK(cudaGetLastError());
        CK(cudaStreamSynchronize(st));
        dfree(ctx, s2t5);
        std::vector<S2TRow> sw;
        for (size_t i = 0; i < ctx->near.size(); ++i) {
            const NearPair &q = ctx->near[i];
            const Box &bs = ctx->boxes[q.src], &bt = ctx->boxes[q.tgt];
            for (int64_t s0 = 0; s0 < bs.p1 - bs.p0; s0 += S2T_SRC)
                for (int64_t ii = 0; ii < bt.p1 - bt.p0; ++ii) sw.push_back(S2TRow{(int64_t)i, (int)ii, (int)s0});
        }
        TRY(dupload(ctx, st, &d->s2twork, sw));
        d->n_s2twork = (int64_t)sw.size();
        std::vector<S2TRowT> swT;
        for (size_t i = 0; i < ctx->near.size(); ++i) {
            const Box &bs = ctx->boxes[ctx->near[i].src];
            for (int64_t jj = 0; jj < bs.p1 - bs.p0; ++jj) swT.push_back(S2TRowT{(int64_t)i, (int)jj, 0});
        }
        TRY(dupload(ctx, st, &d->s2tworkT, swT));
        d->n_s2tworkT = (int64_t)swT.size();
        // free-space near field: the near leaves of a leaf, consecutive sorted points joined
        d->free_near = !ctx->free_near.empty();
        if (d->free_near) {
            std::vector<int> fb(N, 0);
            for (int64_t li : leaves)
                for (int64_t q = ctx->boxes[li].p0; q < ctx->boxes[li].p1; ++q) fb[q] = (int)li;
            TRY(dupload(ctx, st, &d->fbox, fb));
            for (int tr = 0; tr < 2; ++tr) {
                std::vector<std::pair<int64_t, int64_t>> pr(ctx->free_near.size());   // (row leaf, column leaf)
                for (size_t i = 0; i < pr.size(); ++i) {
                    pr[i] = ctx->free_near[i];
                    if (!tr) std::swap(pr[i].first, pr[i].second);
                }
                std::sort(pr.begin(), pr.end());
                std::vector<int> off(nbox + 1, 0);
                std::vector<FreeRun> runs;
                size_t i = 0;
                for (int64_t b = 0; b < nbox; ++b) {
                    const size_t r0 = runs.size();
                    for (; i < pr.size() && pr[i].first == b; ++i) {
                        const Box &c = ctx->boxes[pr[i].second];
                        if (runs.size() > r0 && runs.back().p0 + runs.back().n == c.p0) runs.back().n += (int)(c.p1 - c.p0);
                        else runs.push_back(FreeRun{c.p0, (int)(c.p1 - c.p0), 0});
                    }
                    off[b + 1] = (int)runs.size();
                }
                TRY(dupload(ctx, st, tr ? &d->froffT : &d->froff, off));
                TRY(dupload(ctx, st, tr ? &d->frunsT : &d->fruns, runs));
            }
        }
    }
    TRY(check_flag(ctx));
    ctx->built = true;
    auto t1 = std::chrono::steady_clock::now();
    lmfmm_stats &S = ctx->stats;
    S = lmfmm_stats{};
    S.n_points = N;
    S.n_layers = ctx->med.L + 1;
    S.n_components = ctx->n_react_comps;
    S.depth = ctx->depth;
    S.n_boxes = nbox;
    S.n_m2l_pairs = (int64_t)ctx->m2l.size();
    S.n_geometries = (int64_t)ctx->geoms.size();
    S.n_near_pairs = (int64_t)ctx->near.size();
    S.n_near_point_pairs = ctx->n_near_pp;
    S.n_quad_nodes = qtot;
    S.bytes_tables = d->m2l_kernel == 3 ? (double)m2l_sec_image_bytes(p, (int64_t)ctx->geoms.size())
                     : d->oz ? 2.0 * (double)m2l_oz_image_bytes(p, (int64_t)ctx->geoms.size())
                             : (double)ctx->geoms.size() * NTAB * P * P * (f32 ? 8.0 : 16.0);
    S.ms_setup = std::chrono::duration<double, std::milli>(t1 - t0).count();
    S.m2l_columns = ncols;
    S.m2l_kernel = d->m2l_kernel;
    for (size_t i = 0; i < ctx->n_react_geoms; ++i)
        if (ctx->comps[ctx->geoms[i].comp].l == ctx->comps[ctx->geoms[i].comp].lp) ++S.n_geometries_same_layer;
    S.n_free_geometries = (int64_t)(ctx->geoms.size() - ctx->n_react_geoms);
    S.n_free_near_point_pairs = ctx->n_free_pp;
    S.ms_tabulate = ms_tab;
    S.adjoint_transposed = d->m2l_kernel <= 1;
    S.m2l_digits = d->oz;
    S.tab_flops = 8.0 * tab_terms * (p + 2) * (p + 2) +
                  8.0 * (double)ctx->geoms.size() * NTAB * (double)P * P * (p + 2);
    return LMFMM_OK;
}

extern "C++" {
// P2M / L2P at the leaves: the mixed form's kernels of k_leaf.cu where they
// apply (P2M one warp per unit of a leaf, L2P one thread per point), else one
// CTA per leaf.  l2p_basis / p2m_basis: the transposes.
template <typename T>
static void leaf_p2m(lmfmm_ctx *ctx, const cd *in, cx<T> *out, bool l2p_basis, cudaStream_t st)
{
    DevState *d = DS(ctx);
    const int p = ctx->prm.p;
    if constexpr (std::is_same<T, float>::value) {
        if (d->leaf_fast) {
            launch_p2m_fast(p, d->nunits, d->p2m_many, d->units, d->boxes, d->xyz, in, ctx->med, d->lscale, out, !l2p_basis,
                            l2p_basis ? 1.0 : 4.0 * 3.14159265358979323846, st);
            return;
        }
    }
    launch_p2m<T>(p, d->nleaves, d->leaves, d->boxes, d->xyz, in, ctx->med, d->lscale, out, st, l2p_basis);
}

template <typename T>
static void leaf_l2p(lmfmm_ctx *ctx, const cx<T> *in, cd *out, bool p2m_basis, cudaStream_t st)
{
    DevState *d = DS(ctx);
    const int p = ctx->prm.p;
    if constexpr (std::is_same<T, float>::value) {
        if (d->leaf_fast) {
            launch_l2p_fast(p, ctx->N, d->pt_box, d->boxes, d->xyz, in, ctx->med, d->lscale, out, p2m_basis,
                            p2m_basis ? 4.0 * 3.14159265358979323846 : 1.0, false, st);
            return;
        }
    }
    launch_l2p<T>(p, d->nleaves, d->leaves, d->boxes, d->xyz, in, ctx->med, d->lscale, out, st, p2m_basis, false);
}

// Y += A X over the pairs of translation items (one level of M2M or L2L); the FP64 form reads
// the transposes AT
template <typename T>
static void translate(int p, int64_t nwork, const GemmWork *work, const cx<T> *A, const cx<T> *AT, const int64_t *src,
                      const int64_t *dst, cx<T> *x, cudaStream_t st)
{
    if constexpr (std::is_same<T, double>::value) launch_trans_fp64(p, nwork, work, AT, src, dst, x, x, st);
    else launch_group_gemm_t<T>(p, nwork, work, A, src, dst, x, x, true, st);
}

// stages of one matvec, for the batched launch: the upward pass (gather, P2M,
// M2M), the M2L (own_m2l = false: only the clearing of the local expansions,
// the M2L itself runs in the batch's merged launch), the downward pass
enum { MV_UP = 1, MV_M2L = 2, MV_DOWN = 4, MV_ALL = 7 };

template <typename T>
static lmfmm_status matvec_t(lmfmm_ctx *ctx, const void *J, int dtype, void *Phi,
                             cudaStream_t st, bool cj, int parts = MV_ALL, bool own_m2l = true)
{
    DevState *d = DS(ctx);
    const int p = ctx->prm.p, P = (p + 1) * (p + 1);
    const int64_t N = ctx->N, nbox = (int64_t)ctx->boxes.size();
    cx<T> *me = (cx<T> *)d->me, *le = (cx<T> *)d->le;
    const cx<T> *tup = (const cx<T> *)d->tup, *tdn = (const cx<T> *)d->tdn;
    const cx<T> *tupT = (const cx<T> *)d->tupT, *tdnT = (const cx<T> *)d->tdnT;
    int nl = 0;   // kernels launched (launchers skip empty work)
    if (parts & MV_UP) {
    CK(cudaEventRecord(d->ev[0], st));
    CK(cudaMemsetAsync(d->mvstatus, 0, sizeof(int), st));
    launch_gather_in(N, d->perm, J, dtype, d->qh, cj, st);
    nl += N > 0;
    nl += d->nleaves > 0;   // P2M
    CK(cudaMemsetAsync(me, 0, (size_t)nbox * 3 * P * sizeof(cx<T>), st));
    leaf_p2m<T>(ctx, d->qh, me, false, st);
    CK(cudaEventRecord(d->ev[1], st));
    for (int lev = ctx->depth; lev >= 1; --lev) {
        if constexpr (std::is_same<T, float>::value) {
            if (d->trans_tc) {
                int64_t w0 = d->twork_off[lev], w1 = d->twork_off[lev + 1];
                CK(launch_trans_tc2(p, w1 - w0, d->twork + w0, d->tchild, d->tparent, d->tupi, me, me,
                                    d->yscr, d->ncta, d->mvstatus, st));
                nl += w1 > w0;
                continue;
            }
        }
        int64_t w0 = d->gwork_off[lev], w1 = d->gwork_off[lev + 1];
        translate<T>(p, w1 - w0, d->gwork + w0, tup, tupT, d->tchild, d->tparent, me, st);
        nl += w1 > w0;
    }
    CK(cudaEventRecord(d->ev[2], st));
    }
    if (parts & MV_M2L) {
    nl += d->n_m2lwork > 0;   // M2L
    bool packed = d->oz;   // the tensor-core kernels clear le themselves
    if constexpr (std::is_same<T, float>::value) {
        if (d->m2l_kernel == 3) {
            launch_sec_pack(p, nbox, me, d->mepk, le, st);   // clears le too
            packed = true;
            ++nl;
        }
    }
    if (!packed) CK(cudaMemsetAsync(le, 0, (size_t)nbox * 3 * P * sizeof(cx<T>), st));
    if (!own_m2l) {
        // the batch's merged launch applies this problem's M2L
    } else if constexpr (std::is_same<T, float>::value) {
        if (d->m2l_kernel == 3) {
            CK(launch_m2l_sec(p, d->n_m2lwork, d->m2lwork, TcProb{d->m2l, d->ephase, d->tab, d->mepk, le}, nullptr, d->yscr,
                              d->ncta, d->mvstatus, st));
        }
        else if (d->m2l_kernel == 2)
            CK(launch_m2l_tc(p, d->n_m2lwork, d->m2lwork, d->geoms, d->comps, d->m2l,
                             (const cf *)d->tab, me, le, d->mvstatus, st));
        else
            launch_m2l_t<T>(p, d->n_m2lwork, d->m2lwork, d->geoms, d->comps, d->m2l,
                            (const cx<T> *)d->tab, me, le, st);
    } else if (d->oz) {
        CK(launch_m2l_oz(p, false, (int64_t)ctx->geoms.size(), d->n_m2lwork, d->m2lwork, d->m2l, d->ozimg, nbox, me, le,
                         d->ozpk, d->ozscr, d->ncta, d->mvstatus, st));
        ++nl;
    } else {
        launch_m2l_t<T>(p, d->n_m2lwork, d->m2lwork, d->geoms, d->comps, d->m2l,
                        (const cx<T> *)d->tab, me, le, st);
    }
    if (own_m2l && d->fail_m2l) {
        CK(cudaMemsetAsync(d->mvstatus, d->fail_m2l, 1, st));
        d->fail_m2l = 0;
    }
    CK(cudaEventRecord(d->ev[3], st));
    }
    if (parts & MV_DOWN) {
    for (int lev = 1; lev <= ctx->depth; ++lev) {
        if constexpr (std::is_same<T, float>::value) {
            if (d->trans_tc) {
                int64_t w0 = d->twork_off[lev], w1 = d->twork_off[lev + 1];
                CK(launch_trans_tc2(p, w1 - w0, d->twork + w0, d->tparent, d->tchild, d->tdni, le, le,
                                    d->yscr, d->ncta, d->mvstatus, st));
                nl += w1 > w0;
                continue;
            }
        }
        int64_t w0 = d->gwork_off[lev], w1 = d->gwork_off[lev + 1];
        translate<T>(p, w1 - w0, d->gwork + w0, tdn, tdnT, d->tparent, d->tchild, le, st);
        nl += w1 > w0;
    }
    CK(cudaEventRecord(d->ev[4], st));
    leaf_l2p<T>(ctx, le, d->ph, false, st);
    CK(cudaEventRecord(d->ev[5], st));
    launch_s2t_apply8(d->n_s2twork, d->s2twork, d->near, d->boxes, d->s2t, d->qh, d->ph, st);
    if (d->free_near) {
        launch_p2p_free(N, d->fbox, d->froff, d->fruns, d->boxes, d->xyz, ctx->med, d->qh, d->ph, false, st);
        ++nl;
    }
    CK(cudaEventRecord(d->ev[6], st));
    launch_scatter_out(N, d->perm, d->ph, Phi, dtype, cj, st);
    nl += (d->nleaves > 0) + (d->n_s2twork > 0) + (N > 0);   // L2P, near field, scatter
    CK(cudaEventRecord(d->ev[7], st));
    d->mv_recorded = true;
    }
    CK(cudaGetLastError());
    if (parts == MV_ALL) ctx->stats.launches = nl;
    return LMFMM_OK;
}

// The transposed operator A^T = G^T (P2M^T M2M^T M2L^T L2L^T L2P^T + S2T^T) S^T,
// every factor the exact transpose of the forward one (SIMT forms): L2P^T sums
// the point values against L2P's functions (P2M's kernel), L2L^T and M2M^T run
// the transposed matrices up and down the tree, M2L^T applies the transposed
// tables, P2M^T evaluates with P2M's functions (L2P's kernel).  With cj the
// input and output are conjugated: conj(A^T conj y) = A^H y.  first: the call's
// first pass, which clears the status word (a later one keeps what an earlier left).
template <typename T>
static lmfmm_status matvec_tr_t(lmfmm_ctx *ctx, const void *y, int dtype, void *out, cudaStream_t st, bool cj,
                                bool first = true)
{
    DevState *d = DS(ctx);
    const int p = ctx->prm.p, P = (p + 1) * (p + 1);
    const int64_t N = ctx->N, nbox = (int64_t)ctx->boxes.size();
    cx<T> *me = (cx<T> *)d->me, *le = (cx<T> *)d->le;
    const cx<T> *tupT = (const cx<T> *)d->tupT, *tdnT = (const cx<T> *)d->tdnT;
    int nl = 0;
    CK(cudaEventRecord(d->ev[0], st));
    if (first) CK(cudaMemsetAsync(d->mvstatus, 0, sizeof(int), st));
    launch_gather_tr(N, d->perm, y, dtype, d->ph, cj, st);   // ph <- S^T y
    CK(cudaMemsetAsync(le, 0, (size_t)nbox * 3 * P * sizeof(cx<T>), st));
    leaf_p2m<T>(ctx, d->ph, le, true, st);
    nl += (N > 0) + (d->nleaves > 0);
    CK(cudaEventRecord(d->ev[1], st));
    for (int lev = ctx->depth; lev >= 1; --lev) {   // L2L^T: children into parents
        int64_t w0 = d->gwork_off[lev], w1 = d->gwork_off[lev + 1];
        translate<T>(p, w1 - w0, d->gwork + w0, tdnT, (const cx<T> *)d->tdn, d->tchild, d->tparent, le, st);
        nl += w1 > w0;
    }
    CK(cudaEventRecord(d->ev[2], st));
    bool done = false;
    if constexpr (std::is_same<T, double>::value) {
        if (d->oz) {
            CK(launch_m2l_oz(p, true, (int64_t)ctx->geoms.size(), d->n_m2lwork, d->m2lwork, d->m2l, d->ozimgT, nbox, le, me,
                             d->ozpk, d->ozscr, d->ncta, d->mvstatus, st));
            done = true;
            ++nl;
        }
    }
    if (!done) {
        CK(cudaMemsetAsync(me, 0, (size_t)nbox * 3 * P * sizeof(cx<T>), st));
        launch_m2l_tr<T>(p, d->n_m2lwork, d->m2lwork, d->geoms, d->comps, d->m2l, (const cx<T> *)d->tab, le, me, st);
    }
    nl += d->n_m2lwork > 0;
    CK(cudaEventRecord(d->ev[3], st));
    for (int lev = 1; lev <= ctx->depth; ++lev) {   // M2M^T: parents into children
        int64_t w0 = d->gwork_off[lev], w1 = d->gwork_off[lev + 1];
        translate<T>(p, w1 - w0, d->gwork + w0, tupT, (const cx<T> *)d->tup, d->tparent, d->tchild, me, st);
        nl += w1 > w0;
    }
    CK(cudaEventRecord(d->ev[4], st));
    leaf_l2p<T>(ctx, me, d->qh, true, st);
    CK(cudaEventRecord(d->ev[5], st));
    launch_s2t_apply8_tr(d->n_s2tworkT, d->s2tworkT, d->near, d->boxes, d->s2t, d->ph, d->qh, st);
    if (d->free_near) {
        launch_p2p_free(N, d->fbox, d->froffT, d->frunsT, d->boxes, d->xyz, ctx->med, d->ph, d->qh, true, st);
        ++nl;
    }
    CK(cudaEventRecord(d->ev[6], st));
    launch_scatter_tr(N, d->perm, d->qh, out, dtype, cj, st);
    nl += (d->nleaves > 0) + (d->n_s2tworkT > 0) + (N > 0);
    CK(cudaEventRecord(d->ev[7], st));
    CK(cudaGetLastError());
    d->mv_recorded = true;
    ctx->stats.launches = nl;
    return LMFMM_OK;
}

static lmfmm_status matvec_tr_impl(lmfmm_ctx *ctx, const void *y, int dtype, void *out, cudaStream_t st, bool cj)
{
    if (DS(ctx)->m2l_kernel > 1) {
        ctx->err = "the transposed operator runs in the FP64 form and the mixed form with tensor_cores = 0 "
                   "(the tensor-core forms hold their tables only as the tiled image)";
        return LMFMM_ERR_UNSUPPORTED;
    }
    if (ctx->prm.precision == LMFMM_MIXED) return matvec_tr_t<float>(ctx, y, dtype, out, st, cj);
    return matvec_tr_t<double>(ctx, y, dtype, out, st, cj);
}

static lmfmm_status matvec_impl(lmfmm_ctx *ctx, const void *J, int dtype, void *Phi,
                                cudaStream_t st, bool cj)
{
    if (ctx->prm.precision == LMFMM_MIXED) return matvec_t<float>(ctx, J, dtype, Phi, st, cj);
    return matvec_t<double>(ctx, J, dtype, Phi, st, cj);
}
}  // extern "C++"

static lmfmm_status matvec_args(lmfmm_ctx *ctx, const char *who, const void *J, int dtype, const void *Phi)
{
    if (!ctx->built) {
        ctx->err = std::string(who) + ": call lmfmm_build first";
        return LMFMM_ERR_STATE;
    }
    if (!J || !Phi) {
        ctx->err = std::string(who) + ": NULL buffer";
        return LMFMM_ERR_ARG;
    }
    if (dtype != LMFMM_C128 && dtype != LMFMM_C64) {
        ctx->err = std::string(who) + ": dtype must be LMFMM_C128 or LMFMM_C64";
        return LMFMM_ERR_ARG;
    }
    return LMFMM_OK;
}

lmfmm_status lmfmm_matvec(lmfmm_ctx *ctx, const void *J, int dtype, void *Phi, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    TRY(matvec_args(ctx, "matvec", J, dtype, Phi));
    CK(cudaSetDevice(ctx->device));
    return matvec_impl(ctx, J, dtype, Phi, (cudaStream_t)stream, false);
}

lmfmm_status lmfmm_matvec_adjoint(lmfmm_ctx *ctx, const void *y, int dtype, void *Phi, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    TRY(matvec_args(ctx, "matvec_adjoint", y, dtype, Phi));
    CK(cudaSetDevice(ctx->device));
    if (DS(ctx)->m2l_kernel <= 1) return matvec_tr_impl(ctx, y, dtype, Phi, (cudaStream_t)stream, true);
    return matvec_impl(ctx, y, dtype, Phi, (cudaStream_t)stream, true);
}

lmfmm_status lmfmm_matvec_transpose(lmfmm_ctx *ctx, const void *y, int dtype, void *out, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    TRY(matvec_args(ctx, "matvec_transpose", y, dtype, out));
    CK(cudaSetDevice(ctx->device));
    return matvec_tr_impl(ctx, y, dtype, out, (cudaStream_t)stream, false);
}

lmfmm_status lmfmm_matvec_host(lmfmm_ctx *ctx, const void *J, int dtype, void *Phi, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    TRY(matvec_args(ctx, "matvec_host", J, dtype, Phi));
    CK(cudaSetDevice(ctx->device));
    DevState *d = DS(ctx);
    cudaStream_t st = (cudaStream_t)stream;
    const size_t bytes = (size_t)ctx->N * 3 * (dtype == LMFMM_C64 ? sizeof(cf) : sizeof(cd));
    // staging [2][N][3] complex128, used at the caller's element size
    if (!d->stage) TRY(dalloc(ctx, &d->stage, (size_t)ctx->N * 6));
    unsigned char *sin = (unsigned char *)d->stage, *sout = (unsigned char *)(d->stage + 3 * ctx->N);
    CK(cudaMemcpyAsync(sin, J, bytes, cudaMemcpyHostToDevice, st));
    TRY(matvec_impl(ctx, sin, dtype, sout, st, false));
    CK(cudaMemcpyAsync(Phi, sout, bytes, cudaMemcpyDeviceToHost, st));
    return check_mvstatus(ctx, st);
}

lmfmm_status lmfmm_gradient(lmfmm_ctx *ctx, const void *J, const void *g, int dtype, void *gJ, double *gxyz,
                            void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    TRY(matvec_args(ctx, "gradient", J, dtype, g));
    if (!gJ && !gxyz) {
        ctx->err = "gradient: nothing to compute (gJ and gxyz are NULL)";
        return LMFMM_ERR_ARG;
    }
    if (ctx->prm.precision != LMFMM_FP64 || ctx->prm.components != LMFMM_REACTION) {
        ctx->err = "gradient: the position gradient runs in the FP64 form of the reaction part";
        return LMFMM_ERR_UNSUPPORTED;
    }
    CK(cudaSetDevice(ctx->device));
    DevState *d = DS(ctx);
    cudaStream_t st = (cudaStream_t)stream;
    const int p = ctx->prm.p, P = (p + 1) * (p + 1);
    const int64_t N = ctx->N, nbox = (int64_t)ctx->boxes.size();
    if (!d->le_ck) {
        TRY(dalloc(ctx, &d->le_ck, (size_t)nbox * 3 * P));
        TRY(dalloc(ctx, &d->qh_ck, (size_t)N * 3));
        TRY(dalloc(ctx, &d->gfield, (size_t)N * 3));
        TRY(dalloc(ctx, &d->s2tg, (size_t)std::max<int64_t>(1, ctx->n_near_pp) * 20));
        launch_s2t_pre_grad((int64_t)ctx->near.size(), d->near, d->boxes, d->xyz, ctx->med, d->comps,
                            medium_a(ctx->med), ctx->prm.quad_node_cap, d->s2tg, st);
        CK(cudaGetLastError());
    }
    // forward pass (its result is not needed), then checkpoint what the
    // transposed pass overwrites: the local expansions and the helical charges
    TRY(matvec_t<double>(ctx, J, dtype, d->gfield, st, false));
    CK(cudaMemcpyAsync(d->le_ck, d->le, (size_t)nbox * 3 * P * sizeof(cd), cudaMemcpyDeviceToDevice, st));
    CK(cudaMemcpyAsync(d->qh_ck, d->qh, (size_t)N * 3 * sizeof(cd), cudaMemcpyDeviceToDevice, st));
    // transposed pass of conj(g): gJ = A^H g; leaves ph = S^T conj(g), me = its multipole expansions
    TRY(matvec_tr_t<double>(ctx, g, dtype, gJ ? gJ : (void *)d->gfield, st, true, false));
    if (gxyz) {
        CK(cudaMemsetAsync(gxyz, 0, (size_t)N * 3 * sizeof(double), st));
        launch_grad_leaf(p, N, d->nleaves, d->leaves, d->boxes, d->xyz, d->perm, d->le_ck, (const cd *)d->me,
                         d->qh_ck, d->ph, ctx->med, d->lscale, gxyz, st);
        launch_grad_near((int64_t)ctx->near.size(), d->near, d->boxes, d->xyz, d->perm, d->comps, d->s2tg,
                         d->qh_ck, d->ph, gxyz, st);
        CK(cudaGetLastError());
    }
    return LMFMM_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ batches
struct lmfmm_batch {
    std::vector<lmfmm_ctx *> ctxs;
    int device = 0, p = 0, mixed = 0;
    bool merged = false;          // every problem on the persistent tensor-core M2L: one merged launch
    TcProb *dprobs = nullptr;
    M2LWork *dwork = nullptr;
    int64_t nwork = 0;
    int *status = nullptr;
    float *yscr = nullptr;        // scratch of the merged launch: a context's, or own
    float *own_yscr = nullptr;
    int ncta = 0;
    int variant = 0;
    double ms_variant[4] = {0, 0, 0, 0};
    cudaStream_t cap = nullptr;   // capture stream of the graph
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::vector<const void *> gJ;
    std::vector<void *> gPhi;
    int gdtype = -1;
    std::string err;
};

namespace {

void batch_drop_graph(lmfmm_batch *b)
{
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
}

// merged work list of a batch: variant bit 0 interleaves the problems' items
// round robin (else one problem after the other), bit 1 cuts items to 32
// pairs (else 64)
lmfmm_status batch_work(lmfmm_batch *b, int variant, M2LWork **dst, int64_t *n)
{
    std::vector<std::vector<M2LWork>> per(b->ctxs.size());
    for (size_t i = 0; i < b->ctxs.size(); ++i)
        sec_work_items(b->ctxs[i], (variant & 2) ? m2l_sec_pairs() / 2 : m2l_sec_pairs(), (int)i, per[i]);
    std::vector<M2LWork> all;
    if (variant & 1) {
        for (size_t k = 0;; ++k) {
            bool any = false;
            for (auto &v : per)
                if (k < v.size()) {
                    all.push_back(v[k]);
                    any = true;
                }
            if (!any) break;
        }
    } else {
        for (auto &v : per) all.insert(all.end(), v.begin(), v.end());
    }
    void *q = nullptr;
    if (cudaMalloc(&q, std::max<size_t>(1, all.size()) * sizeof(M2LWork)) != cudaSuccess) return LMFMM_ERR_OOM;
    if (copy_in(q, all.data(), all.size() * sizeof(M2LWork), b->cap)) {
        cudaFree(q);
        return LMFMM_ERR_CUDA;
    }
    *dst = (M2LWork *)q;
    *n = (int64_t)all.size();
    return LMFMM_OK;
}

template <typename T>
lmfmm_status batch_record(lmfmm_batch *b, const void *const *J, void *const *Phi, int dtype, cudaStream_t st)
{
    const size_t n = b->ctxs.size();
    for (size_t i = 0; i < n; ++i) {
        lmfmm_status r = matvec_t<T>(b->ctxs[i], J[i], dtype, Phi[i], st, false, MV_UP | MV_M2L, !b->merged);
        if (r) return r;
    }
    if (b->merged) {
        if (cudaMemsetAsync(b->status, 0, sizeof(int), st) != cudaSuccess) return LMFMM_ERR_CUDA;
        if (launch_m2l_sec(b->p, b->nwork, b->dwork, TcProb{}, b->dprobs, b->yscr, b->ncta, b->status, st) !=
            cudaSuccess)
            return LMFMM_ERR_CUDA;
    }
    for (size_t i = 0; i < n; ++i) {
        lmfmm_status r = matvec_t<T>(b->ctxs[i], J[i], dtype, Phi[i], st, false, MV_DOWN);
        if (r) return r;
    }
    return LMFMM_OK;
}

}  // namespace

extern "C" {

lmfmm_status lmfmm_batch_create(lmfmm_batch **out, lmfmm_ctx *const *ctxs, int n)
{
    if (!out || !ctxs || n < 1) {
        g_err = "batch_create: need n >= 1 contexts";
        return LMFMM_ERR_ARG;
    }
    *out = nullptr;
    for (int i = 0; i < n; ++i)
        if (!ctxs[i] || !ctxs[i]->built || ctxs[i]->device != ctxs[0]->device || ctxs[i]->prm.p != ctxs[0]->prm.p ||
            ctxs[i]->prm.precision != ctxs[0]->prm.precision) {
            g_err = "batch_create: every context must be built, on one device, with one p and one precision";
            return LMFMM_ERR_ARG;
        }
    if (cudaSetDevice(ctxs[0]->device) != cudaSuccess) return LMFMM_ERR_CUDA;
    lmfmm_batch *b = new lmfmm_batch();
    b->ctxs.assign(ctxs, ctxs + n);
    b->device = ctxs[0]->device;
    b->p = ctxs[0]->prm.p;
    b->mixed = ctxs[0]->prm.precision == LMFMM_MIXED;
    b->merged = true;
    for (int i = 0; i < n; ++i) b->merged = b->merged && DS(ctxs[i])->m2l_kernel == 3;
    lmfmm_status rc = LMFMM_OK;
    if (cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking) != cudaSuccess ||
        cudaMalloc((void **)&b->status, sizeof(int)) != cudaSuccess ||
        cudaMemsetAsync(b->status, 0, sizeof(int), b->cap) != cudaSuccess || cudaStreamSynchronize(b->cap) != cudaSuccess)
        rc = LMFMM_ERR_CUDA;
    if (!rc && b->merged) {
        std::vector<TcProb> hp(n);
        for (int i = 0; i < n; ++i) {
            DevState *d = DS(ctxs[i]);
            hp[i] = TcProb{d->m2l, d->ephase, d->tab, d->mepk, (cf *)d->le};
        }
        if (cudaMalloc((void **)&b->dprobs, n * sizeof(TcProb)) != cudaSuccess ||
            copy_in(b->dprobs, hp.data(), n * sizeof(TcProb), b->cap) != cudaSuccess)
            rc = LMFMM_ERR_CUDA;
        if (!rc) rc = batch_work(b, 0, &b->dwork, &b->nwork);
        // the merged launch has the items of all problems (twice as many where they are halved): the
        // largest scratch of a context, which is idle then, or a larger one of the batch's own
        for (lmfmm_ctx *c : b->ctxs)
            if (DS(c)->ncta > b->ncta) {
                b->ncta = DS(c)->ncta;
                b->yscr = DS(c)->yscr;
            }
        const int want = (int)std::min<int64_t>(DS(ctxs[0])->nsm, 2 * b->nwork);
        if (!rc && b->ncta < want) {
            if (cudaMalloc((void **)&b->own_yscr, m2l_sec_scratch_floats(b->p, want) * sizeof(float)) != cudaSuccess)
                rc = LMFMM_ERR_OOM;
            b->yscr = b->own_yscr;
            b->ncta = want;
        }
    }
    if (rc) {
        g_err = "batch_create: device setup failed";
        lmfmm_batch_destroy(b);
        return rc;
    }
    *out = b;
    return LMFMM_OK;
}

lmfmm_status lmfmm_batch_matvec(lmfmm_batch *b, const void *const *J, void *const *Phi, int dtype, void *stream)
{
    if (!b) return LMFMM_ERR_ARG;
    const size_t n = b->ctxs.size();
    if (!J || !Phi || (dtype != LMFMM_C128 && dtype != LMFMM_C64)) {
        b->err = "batch_matvec: NULL pointer arrays or bad dtype";
        return LMFMM_ERR_ARG;
    }
    for (size_t i = 0; i < n; ++i)
        if (!J[i] || !Phi[i]) {
            b->err = "batch_matvec: NULL buffer";
            return LMFMM_ERR_ARG;
        }
    if (cudaSetDevice(b->device) != cudaSuccess) return LMFMM_ERR_CUDA;
    const bool same = b->exec && b->gdtype == dtype && std::equal(b->gJ.begin(), b->gJ.end(), J) &&
                      std::equal(b->gPhi.begin(), b->gPhi.end(), Phi);
    if (!same) {
        // record every launch of the batch once, on the capture stream
        batch_drop_graph(b);
        if (cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
            b->err = "batch_matvec: stream capture failed to start";
            return LMFMM_ERR_CUDA;
        }
        lmfmm_status rc = b->mixed ? batch_record<float>(b, J, Phi, dtype, b->cap)
                                   : batch_record<double>(b, J, Phi, dtype, b->cap);
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(b->cap, &g);
        if (rc || e != cudaSuccess || !g) {
            if (g) cudaGraphDestroy(g);
            b->err = "batch_matvec: capture of the batch failed";
            return rc ? rc : LMFMM_ERR_CUDA;
        }
        b->graph = g;
        if (cudaGraphInstantiate(&b->exec, b->graph, 0) != cudaSuccess) {
            batch_drop_graph(b);
            b->err = "batch_matvec: graph instantiation failed";
            return LMFMM_ERR_CUDA;
        }
        b->gJ.assign(J, J + n);
        b->gPhi.assign(Phi, Phi + n);
        b->gdtype = dtype;
    }
    if (cudaGraphLaunch(b->exec, (cudaStream_t)stream) != cudaSuccess) {
        b->err = "batch_matvec: graph launch failed";
        return LMFMM_ERR_CUDA;
    }
    return LMFMM_OK;
}

lmfmm_status lmfmm_batch_tune(lmfmm_batch *b, void *stream)
{
    if (!b) return LMFMM_ERR_ARG;
    if (!b->merged) {
        b->err = "batch_tune: the merged M2L needs every problem on the persistent tensor-core kernel";
        return LMFMM_ERR_UNSUPPORTED;
    }
    if (cudaSetDevice(b->device) != cudaSuccess) return LMFMM_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    // defined inputs for the timing runs
    for (lmfmm_ctx *c : b->ctxs)
        if (cudaMemsetAsync(DS(c)->mepk, 0, m2l_sec_packed_bytes(b->p, (int64_t)c->boxes.size()), st) != cudaSuccess)
            return LMFMM_ERR_CUDA;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return LMFMM_ERR_CUDA;
    int best = 0;
    for (int v = 0; v < 4; ++v) {
        M2LWork *w = nullptr;
        int64_t nw = 0;
        lmfmm_status rc = batch_work(b, v, &w, &nw);
        if (rc) return rc;
        float tmin = 1e30f;
        for (int rep = 0; rep < 4; ++rep) {
            cudaEventRecord(e0, st);
            launch_m2l_sec(b->p, nw, w, TcProb{}, b->dprobs, b->yscr, b->ncta, b->status, st);
            cudaEventRecord(e1, st);
            cudaEventSynchronize(e1);
            float ms = 0;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep > 0) tmin = std::min(tmin, ms);   // first run warms the caches
        }
        cudaFree(w);
        b->ms_variant[v] = tmin;
        if (tmin < b->ms_variant[best]) best = v;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (cudaGetLastError() != cudaSuccess) return LMFMM_ERR_CUDA;
    M2LWork *w = nullptr;
    int64_t nw = 0;
    TRY(batch_work(b, best, &w, &nw));
    cudaFree(b->dwork);
    b->dwork = w;
    b->nwork = nw;
    b->variant = best;
    batch_drop_graph(b);   // the next matvec captures the chosen list
    int f = 0;
    cudaMemcpy(&f, b->status, sizeof(int), cudaMemcpyDeviceToHost);
    if (cudaMemsetAsync(b->status, 0, sizeof(int), st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        return LMFMM_ERR_CUDA;
    if (f) {
        b->err = "batch_tune: a bounded tensor-core wait gave up during the timing runs";
        return LMFMM_ERR_TIMEOUT;
    }
    return LMFMM_OK;
}

lmfmm_status lmfmm_batch_check(lmfmm_batch *b, void *stream)
{
    if (!b) return LMFMM_ERR_ARG;
    if (cudaSetDevice(b->device) != cudaSuccess || cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess)
        return LMFMM_ERR_CUDA;
    int f = 0;
    if (cudaMemcpy(&f, b->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return LMFMM_ERR_CUDA;
    for (lmfmm_ctx *c : b->ctxs) {
        int g = 0;
        if (cudaMemcpy(&g, DS(c)->mvstatus, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
            return LMFMM_ERR_CUDA;
        f |= g;
    }
    if (f) {
        b->err = "batch: a bounded tensor-core wait gave up; the results are incomplete";
        return LMFMM_ERR_TIMEOUT;
    }
    return LMFMM_OK;
}

lmfmm_status lmfmm_batch_info(const lmfmm_batch *b, int *merged, int64_t *nwork, int *variant, double *ms_variant)
{
    if (!b) return LMFMM_ERR_ARG;
    if (merged) *merged = b->merged;
    if (nwork) *nwork = b->nwork;
    if (variant) *variant = b->variant;
    if (ms_variant)
        for (int i = 0; i < 4; ++i) ms_variant[i] = b->ms_variant[i];
    return LMFMM_OK;
}

const char *lmfmm_batch_last_error(const lmfmm_batch *b) { return b ? b->err.c_str() : g_err.c_str(); }

void lmfmm_batch_destroy(lmfmm_batch *b)
{
    if (!b) return;
    cudaSetDevice(b->device);
    batch_drop_graph(b);
    if (b->cap) cudaStreamDestroy(b->cap);
    cudaFree(b->dprobs);
    cudaFree(b->dwork);
    cudaFree(b->status);
    cudaFree(b->own_yscr);
    delete b;
}

lmfmm_status lmfmm_check(lmfmm_ctx *ctx, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (!ctx->built || !DS(ctx) || !DS(ctx)->mvstatus) {
        ctx->err = "check: call lmfmm_build first";
        return LMFMM_ERR_STATE;
    }
    CK(cudaSetDevice(ctx->device));
    return check_mvstatus(ctx, (cudaStream_t)stream);
}

lmfmm_status lmfmm_test_set_status(lmfmm_ctx *ctx, int bits)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (!ctx->built || !DS(ctx) || !DS(ctx)->mvstatus) {
        ctx->err = "test_set_status: call lmfmm_build first";
        return LMFMM_ERR_STATE;
    }
    CK(cudaSetDevice(ctx->device));
    int f = 0;
    CK(cudaDeviceSynchronize());
    CK(cudaMemcpy(&f, DS(ctx)->mvstatus, sizeof(int), cudaMemcpyDeviceToHost));
    f |= bits;
    CK(copy_in(DS(ctx)->mvstatus, &f, sizeof(int), cudaStreamLegacy));
    return LMFMM_OK;
}

lmfmm_status lmfmm_test_fail_m2l(lmfmm_ctx *ctx, int bits)
{
    if (!ctx || bits < 0 || bits > 255) return LMFMM_ERR_ARG;
    if (!ctx->built || !DS(ctx)) {
        ctx->err = "test_fail_m2l: call lmfmm_build first";
        return LMFMM_ERR_STATE;
    }
    DS(ctx)->fail_m2l = bits;
    return LMFMM_OK;
}

lmfmm_status lmfmm_direct(lmfmm_ctx *ctx, const lmfmm_c128 *J, lmfmm_c128 *Phi, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (!ctx->built) {
        ctx->err = "direct: call lmfmm_build first";
        return LMFMM_ERR_STATE;
    }
    if (!J || !Phi) {
        ctx->err = "direct: NULL buffer";
        return LMFMM_ERR_ARG;
    }
    CK(cudaSetDevice(ctx->device));
    DevState *d = DS(ctx);
    cudaStream_t st = (cudaStream_t)stream;
    // every (component, source leaf, target leaf) pair is treated as near
    int64_t npp = 0, cnt = 0;
    for (int ci = 0; ci < ctx->n_react_comps; ++ci)
        cnt += (ctx->lvl1[ctx->comps[ci].l][ctx->depth] - ctx->lvl0[ctx->comps[ci].l][ctx->depth]) *
               (ctx->lvl1[ctx->comps[ci].lp][ctx->depth] - ctx->lvl0[ctx->comps[ci].lp][ctx->depth]);
    std::vector<NearPair> all((size_t)cnt);
    all_leaf_pairs(ctx, all.data(), cnt, &npp);
    NearPair *dn = nullptr;
    cd *coef = nullptr;
    void *q1 = nullptr, *q2 = nullptr;
    CK(cudaMalloc(&q1, std::max<size_t>(1, all.size()) * sizeof(NearPair)));
    dn = (NearPair *)q1;
    if (cudaMalloc(&q2, std::max<int64_t>(1, npp) * 5 * sizeof(cd)) != cudaSuccess) {
        cudaFree(q1);
        ctx->err = "direct: coefficient allocation failed";
        return LMFMM_ERR_OOM;
    }
    coef = (cd *)q2;
    lmfmm_status rc = LMFMM_OK;
    if (copy_in(dn, all.data(), all.size() * sizeof(NearPair), st)) rc = LMFMM_ERR_CUDA;
    if (!rc) {
        double a = medium_a(ctx->med);
        cudaMemsetAsync(d->flag, 0, sizeof(int), st);
        launch_gather_in(ctx->N, d->perm, J, LMFMM_C128, d->qh, false, st);
        cudaMemsetAsync(d->ph, 0, (size_t)ctx->N * 3 * sizeof(cd), st);
        launch_s2t_pre((int64_t)all.size(), dn, d->boxes, d->xyz, ctx->med, d->comps, a,
                       ctx->prm.quad_node_cap, coef, d->flag, st);
        launch_s2t_apply((int64_t)all.size(), dn, d->boxes, d->xyz, coef, d->qh, d->ph, st);
        launch_scatter_out(ctx->N, d->perm, d->ph, Phi, LMFMM_C128, false, st);
        if (cudaStreamSynchronize(st) != cudaSuccess) rc = LMFMM_ERR_CUDA;
    }
    cudaFree(q1);
    cudaFree(q2);
    if (rc) {
        ctx->err = "direct: CUDA failure";
        return rc;
    }
    return check_flag(ctx);
}

lmfmm_status lmfmm_densities(lmfmm_ctx *ctx, int l, int lp, int64_t n, const lmfmm_c128 *krho,
                             lmfmm_c128 *out, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (!ctx->layers_set) {
        ctx->err = "densities: call lmfmm_set_layers first";
        return LMFMM_ERR_STATE;
    }
    if (l < 0 || lp < 0 || l > ctx->med.L || lp > ctx->med.L || n < 0 || (n > 0 && (!krho || !out))) {
        ctx->err = "densities: layer index out of range or NULL buffer";
        return LMFMM_ERR_ARG;
    }
    if (ctx->med.L == 0) {
        ctx->err = "densities: no interfaces";
        return LMFMM_ERR_ARG;
    }
    CK(cudaSetDevice(ctx->device));
    launch_densities(ctx->med, l, lp, n, (const cd *)krho, (cd *)out, (cudaStream_t)stream);
    CK(cudaGetLastError());
    return LMFMM_OK;
}

lmfmm_status lmfmm_m2l_table(lmfmm_ctx *ctx, int l, int lp, int tgt_up, int src_up, double rho,
                             double zs, double zt, lmfmm_c128 *out, void *stream)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (!ctx->layers_set) {
        ctx->err = "m2l_table: call lmfmm_set_layers first";
        return LMFMM_ERR_STATE;
    }
    const int L = ctx->med.L;
    if (L < 1 || l < 0 || lp < 0 || l > L || lp > L || !out || !(rho >= 0) ||
        (tgt_up && l > L - 1) || (!tgt_up && l < 1) || (src_up && lp < 1) || (!src_up && lp > L - 1)) {
        ctx->err = "m2l_table: no such reaction component or bad argument";
        return LMFMM_ERR_ARG;
    }
    CompDev c{};
    c.l = l;
    c.lp = lp;
    c.tu = tgt_up ? 1 : 0;
    c.su = src_up ? 1 : 0;
    c.s = comp_sign(l, lp, c.su);
    if (!(c.s * (zs - zt) > 0)) {
        ctx->err = "m2l_table: centres are not separated in the direction of the component";
        return LMFMM_ERR_ARG;
    }
    CK(cudaSetDevice(ctx->device));
    const int p = ctx->prm.p, T = (p + 1) * (p + 2) / 2;
    std::vector<double> B;
    int KM = (p + 1) / 2;
    bcoef_table(p, KM, B);
    std::vector<cd> G((size_t)T * T * (p + 2));
    gtensor(p, B, KM, zc(ctx->med.k[l].x, ctx->med.k[l].y), zc(ctx->med.k[lp].x, ctx->med.k[lp].y),
            G.data());
    if (!ctx->dev) ctx->dev = new DevState();
    DevState *d = DS(ctx);
    if (!d->flag) {
        CK(cudaMalloc((void **)&d->flag, sizeof(int)));
        d->allocs.push_back(d->flag);
        CK(cudaMemsetAsync(d->flag, 0, sizeof(int), (cudaStream_t)stream));
    }
    std::vector<GeomDev> hg(1);
    hg[0].comp = 0;
    hg[0].src_primary = std::hypot(ctx->med.k[l].x, ctx->med.k[l].y) <=
                        std::hypot(ctx->med.k[lp].x, ctx->med.k[lp].y);
    hg[0].rho = rho;
    hg[0].zs = zs;
    hg[0].zt = zt;
    hg[0].plan = geom_plan(medium_a(ctx->med), p, rho, c.s * (zs - zt));
    hg[0].tab_index = 0;
    void *qc = nullptr, *qG = nullptr, *qi = nullptr;
    CK(cudaMalloc(&qc, sizeof(CompDev)));
    CK(cudaMalloc(&qG, G.size() * sizeof(cd)));
    CK(cudaMalloc(&qi, sizeof(int)));
    int zero = 0;
    CK(copy_in(qc, &c, sizeof(CompDev), (cudaStream_t)stream));
    CK(copy_in(qG, G.data(), G.size() * sizeof(cd), (cudaStream_t)stream));
    CK(copy_in(qi, &zero, sizeof(int), (cudaStream_t)stream));
    lmfmm_status rc = tabulate(ctx, hg, (const CompDev *)qc, (const cd *)qG, (const int *)qi,
                               (cd *)out, (cudaStream_t)stream);
    cudaFree(qc);
    cudaFree(qG);
    cudaFree(qi);
    return rc;
}

lmfmm_status lmfmm_translation_matrix(int p, lmfmm_c128 k, const double *t, lmfmm_c128 *m2m,
                                      lmfmm_c128 *l2l)
{
    if (p < 1 || p > 16 || !t || !m2m || !l2l || !std::isfinite(t[0]) || !std::isfinite(t[1]) ||
        !std::isfinite(t[2])) {
        g_err = "translation_matrix: bad argument";
        return LMFMM_ERR_ARG;
    }
    std::vector<int64_t> goff;
    std::vector<int> gl;
    std::vector<double> gv;
    gaunt_table(p, goff, gl, gv);
    translation_matrix(p, zc(k.re, k.im), t, goff, gl, gv, (cd *)m2m, (cd *)l2l);
    return LMFMM_OK;
}

lmfmm_status lmfmm_built_translation(lmfmm_ctx *ctx, int64_t group, int *layer, double *t, double *scales, lmfmm_c128 *m2m,
                                     lmfmm_c128 *l2l)
{
    if (!ctx) return LMFMM_ERR_ARG;
    if (!ctx->built) {
        ctx->err = "built_translation: call lmfmm_build first";
        return LMFMM_ERR_STATE;
    }
    if (ctx->prm.precision != LMFMM_FP64) {
        ctx->err = "built_translation: the mixed form holds its matrices in other formats";
        return LMFMM_ERR_UNSUPPORTED;
    }
    if (group < 0 || group >= (int64_t)ctx->tgroups.size() || !layer || !t || !scales || !m2m || !l2l) {
        ctx->err = "built_translation: no such group or NULL buffer";
        return LMFMM_ERR_ARG;
    }
    CK(cudaSetDevice(ctx->device));
    const DevState *d = DS(ctx);
    const TransGroup &g = ctx->tgroups[group];
    const int P = (ctx->prm.p + 1) * (ctx->prm.p + 1);
    const double s1 = std::hypot(ctx->med.k[g.layer].x, ctx->med.k[g.layer].y) * 2.0 * ctx->root_h;
    *layer = g.layer;
    std::copy(g.t, g.t + 3, t);
    scales[0] = s1 / (double)(1u << g.level);
    scales[1] = s1 / (double)(1u << (g.level - 1));
    CK(cudaMemcpy(m2m, (const cd *)d->tup + group * P * P, (size_t)P * P * sizeof(cd), cudaMemcpyDeviceToHost));
    CK(cudaMemcpy(l2l, (const cd *)d->tdn + group * P * P, (size_t)P * P * sizeof(cd), cudaMemcpyDeviceToHost));
    return LMFMM_OK;
}

lmfmm_status lmfmm_free_m2l_table(int p, lmfmm_c128 k, double rho, double dz, lmfmm_c128 *tables,
                                   lmfmm_c128 *blocks)
{
    if (p < 1 || p > 16 || !tables || !(rho >= 0) || !std::isfinite(rho) || !std::isfinite(dz) ||
        !(rho > 0 || dz != 0)) {
        g_err = "free_m2l_table: bad argument";
        return LMFMM_ERR_ARG;
    }
    free_m2l_tables(p, zc(k.re, k.im), rho, dz, (cd *)tables, (cd *)blocks);
    return LMFMM_OK;
}

lmfmm_status lmfmm_get_stats(const lmfmm_ctx *ctx, lmfmm_stats *out)
{
    if (!ctx || !out) return LMFMM_ERR_ARG;
    lmfmm_ctx *c = (lmfmm_ctx *)ctx;
    *out = c->stats;
    DevState *d = DS(c);
    if (c->built && d && d->ev_ok && d->mv_recorded && cudaEventQuery(d->ev[7]) == cudaSuccess) {
        float ms;
        for (int i = 0; i < 6; ++i)
            if (cudaEventElapsedTime(&ms, d->ev[i], d->ev[i + 1]) == cudaSuccess) out->ms_stage[i] = ms;
        if (cudaEventElapsedTime(&ms, d->ev[6], d->ev[7]) == cudaSuccess) out->ms_stage[6] = ms;
        if (cudaEventElapsedTime(&ms, d->ev[0], d->ev[7]) == cudaSuccess) out->ms_stage[7] = ms;
    }
    return LMFMM_OK;
}

const char *lmfmm_last_error(const lmfmm_ctx *ctx)
{
    if (!ctx) return g_err.c_str();
    return ctx->err.c_str();
}

void lmfmm_destroy(lmfmm_ctx *ctx)
{
    if (!ctx) return;
    free_dev(ctx);
    delete ctx;
}

}  // extern "C"
