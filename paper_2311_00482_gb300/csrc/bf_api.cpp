// C ABI of the beamformer: handles, resident tables, scratch, batches and the
// asynchronous submit / poll path.  See include/bf.h for the contract.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <tuple>
#include <vector>

#include "../../include/bf.h"
#include "bf_choice.h"
#include "bf_engine.h"

namespace bfi {

// ------------------------------------------------------------------ errors --

static thread_local std::string g_err;

int fail(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

int cuda_fail(cudaError_t e, const char *what)
{
    return fail(e == cudaErrorMemoryAllocation ? BF_ENOMEM : BF_ECUDA, "%s: %s", what,
                cudaGetErrorString(e));
}

// ------------------------------------------------------------- device mem --

bool fault_injected(const char *kind)
{
    const char *e = std::getenv("BF_FAULT");
    if (!e || !*e)
        return false;
    const size_t n = std::strlen(kind);
    for (const char *p = e;;) {
        const char *q = std::strchr(p, ',');
        const size_t len = q ? (size_t)(q - p) : std::strlen(p);
        if (len == n && std::strncmp(p, kind, n) == 0)
            return true;
        if (!q)
            return false;
        p = q + 1;
    }
}

int DevMem::ensure(size_t n)
{
    if (n <= bytes && p)
        return BF_OK;
    release();
    if (n == 0)
        return BF_OK;
    if (fault_injected("alloc"))
        return fail(BF_ENOMEM, "injected allocation failure (BF_FAULT=alloc)");
    cudaError_t e = cudaMalloc(&p, n);
    if (e != cudaSuccess) {
        p = nullptr;
        cudaGetLastError();
        return cuda_fail(e, "cudaMalloc");
    }
    bytes = n;
    return BF_OK;
}

int DevMem::reserve(size_t n)
{
    if (n <= bytes && p)
        return BF_OK;
    return ensure(std::max<size_t>({n, bytes + bytes / 2, 4096}));
}

void DevMem::release()
{
    if (p)
        cudaFree(p);
    p = nullptr;
    bytes = 0;
}

int DevMem::upload(const void *src, size_t n)
{
    int rc = ensure(n);
    if (rc)
        return rc;
    if (n == 0)
        return BF_OK;
    cudaError_t e = cudaMemcpy(p, src, n, cudaMemcpyHostToDevice);
    return e == cudaSuccess ? BF_OK : cuda_fail(e, "cudaMemcpy (tables)");
}

// ------------------------------------------------------------- tensor map --

static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// Tensor map over a row-major table of `rows` rows of `cols` elements of `elem`
// bytes (4 or 8), read in boxes of box_cols x box_rows; planes > 0: `planes` such
// tables back to back, boxes box_planes deep.  Out-of-range elements read as zero.
static int encode_map(CUtensorMap *map, const void *base, int rows, int cols, int elem, int box_cols,
                      int box_rows, int planes = 0, int box_planes = 1)
{
    auto enc = tensor_map_encoder();
    if (!enc)
        return fail(BF_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
    const cuuint64_t pitch = (cuuint64_t)cols * (cuuint64_t)elem;
    cuuint64_t strides[2] = {pitch, pitch * (cuuint64_t)rows};
    cuuint32_t boxd[3] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows, (cuuint32_t)box_planes};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(map, elem == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_UINT32,
                     planes > 0 ? 3 : 2, const_cast<void *>(base), dims, strides, boxd, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return fail(BF_ECUDA, "cuTensorMapEncodeTiled failed (%d): %d x %d of %d bytes, box %d x %d",
                    (int)r, rows, cols, elem, box_cols, box_rows);
    return BF_OK;
}

// Pairs per frame of one tensor copy of an nf-frame job's interleaved window
// ([pair][frame], wmax pairs): the largest divisor of wmax whose copy spans at
// most kMaxBox tensor elements (IQ pairs: two each) and a multiple of 16 bytes
// (0: none).
static int interleaved_box(int wmax, int nf, int prec)
{
    const int pb = pair_bytes(prec);
    if ((wmax * nf * pb) % 16 != 0)
        return 0;
    for (int d = std::min(wmax, kMaxBox / (nf * pair_elems(prec))); d >= 1; --d)
        if (wmax % d == 0 && (d * nf * pb) % 16 == 0)
            return d;
    return 0;
}

// -------------------------------------------------------- envelope tables --

// Transform tables are shared by the handles of a device: the twiddles of the
// powers of two up to 8192 (n = 0: the level twiddles of bf_fft16.cuh), kept,
// and the envelope factors of the depths and bands used last (at most
// kEnvTablesKept; frames that use older ones hold them).
static std::mutex g_tables_mu;
static std::map<std::pair<int, int>, std::shared_ptr<FftTablesDev>> g_fft_tables;  // (device, n)

struct EnvTablesKey {
    int dev, nz, band, lo, hi;
    bool operator==(const EnvTablesKey &o) const
    {
        return dev == o.dev && nz == o.nz && band == o.band && lo == o.lo && hi == o.hi;
    }
};
constexpr size_t kEnvTablesKept = 256;
static std::vector<std::pair<EnvTablesKey, std::shared_ptr<EnvTablesDev>>> g_env_tables;  // oldest first

static int fft_tables(int n, std::shared_ptr<FftTablesDev> &out)
{
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(g_tables_mu);
    auto it = g_fft_tables.find({dev, n});
    if (it != g_fft_tables.end()) {
        out = it->second;
        return BF_OK;
    }
    std::vector<float> tw;
    if (n == 0)
        fft16_twiddles(tw);
    else
        fft_twiddles(n, tw);
    auto t = std::make_shared<FftTablesDev>();
    int rc = t->tw.upload(tw.data(), tw.size() * sizeof(float));
    if (rc)
        return rc;
    g_fft_tables[{dev, n}] = t;
    out = t;
    return BF_OK;
}

static int env_tables(int nz, bool band, int lo, int hi, std::shared_ptr<EnvTablesDev> &out)
{
    EnvTablesKey key{0, nz, band ? 1 : 0, band ? lo : 0, band ? hi : 0};
    cudaGetDevice(&key.dev);
    std::lock_guard<std::mutex> lk(g_tables_mu);
    for (size_t i = g_env_tables.size(); i-- > 0;)
        if (g_env_tables[i].first == key) {
            out = g_env_tables[i].second;
            std::rotate(g_env_tables.begin() + i, g_env_tables.begin() + i + 1, g_env_tables.end());
            return BF_OK;
        }
    EnvHost eh;
    envelope_tables(nz, band, lo, hi, eh);
    auto t = std::make_shared<EnvTablesDev>();
    t->lg = eh.lg;
    t->conv = eh.conv;
    int rc = t->gh.upload(eh.gh.data(), eh.gh.size() * sizeof(float));
    if (!rc && band)
        rc = t->gr.upload(eh.gr.data(), eh.gr.size() * sizeof(float));
    if (rc)
        return rc;
    if (g_env_tables.size() >= kEnvTablesKept)
        g_env_tables.erase(g_env_tables.begin());
    g_env_tables.emplace_back(key, t);
    out = t;
    return BF_OK;
}

// ------------------------------------------------------------------ plans --

// BF_TILE_ROWS=8 forces entry 3 of kTileConfigs, 4 entry 0, 2 entry 6 (16-row tiles
// of up to 22 channels per stage); -1: not set.
static int forced_cfg()
{
    const char *e = std::getenv("BF_TILE_ROWS");
    const int rows = e ? std::atoi(e) : 0;
    return rows == 8 ? 3 : rows == 4 ? 0 : rows == 2 ? 6 : -1;
}

// bf_autotune's choice for a workload, or -1.  lone: for RF frames that share their plan
// with no other; two-row tiles only for frames that can take them.
static int tuned_cfg(const bf_handle *h, PlanKey key, bool lone, bool narrow_ok)
{
    key.cfg = lone ? 1 : 0;
    auto it = h->tuned.find(key);
    if (it == h->tuned.end())
        return -1;
    const int c = it->second;
    return c < kNumTileConfigs && kTileConfigs[c].rows == 2 && !narrow_ok ? (lone ? -1 : 0) : c;
}

// Configuration of a workload (of kTileConfigs, or a solo one): BF_TILE_ROWS, else
// what bf_autotune measured fastest for it, else (by_rule) by the frames that share it
// (bf_choice.h).
static int choose_cfg(const bf_handle *h, const PlanKey &key, const PlanWish &w, bool narrow_ok,
                      bool *by_rule)
{
    *by_rule = false;
    const int forced = forced_cfg();
    if (forced >= 0)
        return forced;
    const int tuned = tuned_cfg(h, key, w.alone && key.prec != kPrecIQ, narrow_ok);
    if (tuned >= 0)
        return tuned;
    *by_rule = true;
    return rule_config(key.prec, key.ns, (int)key.angles.size(), image_tiles(h->g.nx, h->g.nz), h->sms,
                       w.alone, narrow_ok, w.peers);
}

// The angle tables of a plan key, shared by its tilings (the handle's lock is held).
static int angle_tables_dev(bf_handle *h, PlanKey key, std::shared_ptr<AngleTablesDev> &out)
{
    key.prec = key.cfg = 0;
    auto it = h->angle_tabs.find(key);
    if (it != h->angle_tabs.end()) {
        out = it->second;
        return BF_OK;
    }
    PlanHost<int16_t> ph;
    angle_tables(h->g, h->geo, key.ns, key.angles, ph);
    auto t = std::make_shared<AngleTablesDev>();
    int rc = t->colK.upload(ph.colK.data(), ph.colK.size() * sizeof(int));
    if (!rc) rc = t->colF.upload(ph.colF.data(), ph.colF.size() * sizeof(float));
    if (!rc) rc = t->rowK.upload(ph.rowK.data(), ph.rowK.size() * sizeof(int));
    if (!rc) rc = t->rowF.upload(ph.rowF.data(), ph.rowF.size() * sizeof(float));
    if (!rc) rc = t->valid.upload(ph.valid.data(), ph.valid.size() * sizeof(int16_t));
    if (rc)
        return rc;
    h->angle_tabs.emplace(std::move(key), t);
    out = t;
    return BF_OK;
}

int handle_plan(bf_handle *h, int ns, const double *angles, int na, uint32_t flags, Plan **out,
                const PlanWish &wish)
{
    const int prec = frame_prec(flags), cfg = wish.cfg;
    const bool narrow_ok = sharing_modes(flags);
    PlanKey key{ns, prec, std::vector<double>(angles, angles + na), 0};
    std::lock_guard<std::mutex> lk(h->mu);
    bool by_rule = false;
    key.cfg = (cfg >= 0 && cfg < kNumConfigs) ? cfg : choose_cfg(h, key, wish, narrow_ok, &by_rule);
    if (key.cfg < kSoloConfig && kTileConfigs[key.cfg].rows == 2 && !narrow_ok) {
        if (cfg >= 0)
            return fail(BF_EINVAL, "two-row tiles serve DAS / DMAS and IQ-DAS / BB-DMAS only");
        key.cfg = 0;
    }
    auto it = h->plans.find(key);
    if (it != h->plans.end()) {
        *out = it->second.get();
        return BF_OK;
    }
    int wmax = 0, box = 0, group = 0;
    auto fits = [&](const TileConfig &t) {
        tile_window(h->g, key.angles, prec, tile_rows(t.rows), 1, wmax, box);
        group = stage_channels(wmax, prec, t.rows, t.stage_bytes, h->g.ne);
        return beamform_smem_bytes(wmax, group, prec, 1, t.rows) <= (size_t)kMaxSmemPerCta;
    };
    // the default tiles' window bounds the pixel spacing, whichever tiles a rule chose; a
    // workload that was tuned to smaller tiles keeps them where the default does not fit
    if (by_rule && !fits(kTileConfigs[0])) {
        const int tuned = tuned_cfg(h, key, false, narrow_ok);
        if (tuned > 0) {
            key.cfg = tuned;
            by_rule = false;
            it = h->plans.find(key);
            if (it != h->plans.end()) {
                *out = it->second.get();
                return BF_OK;
            }
        }
    }
    const bool solo = key.cfg >= kSoloConfig;
    const TileConfig tc = kTileConfigs[solo ? 0 : key.cfg];
    if ((by_rule && !fits(kTileConfigs[0])) || !fits(tc))
        return fail(BF_EINVAL,
                    "pixel spacing too coarse for the sample rate: one tile needs %d samples per channel",
                    wmax);
    int rows = tc.rows, bands = kWarps, tr = tile_rows(tc.rows), split = 0, ang = 1, ngr = 1, run = 1;
    if (solo) {
        split = 1 << (key.cfg - kSoloConfig);
        rows = 2;
        bands = kWarps / split;
        tr = rows * bands;
        // Channels per window copy (four, two or one) and angles per stage (up to
        // four): the most whose windows for one copy's channels leave three CTAs per
        // SM their shared memory; failing that what fits one CTA.
        const int all = BF_DMAS | BF_CF | BF_PDAS, pb = pair_bytes(prec);
        auto per_channel = [&](int an) { return kTileCols * 4 * (1 + an) + an * wmax * pb; };
        run = h->g.ne >= 4 ? 4 : h->g.ne >= 2 ? 2 : 1;
        for (ang = std::min(kSoloAngles, na);;) {
            tile_window(h->g, key.angles, prec, tr, run, wmax, box);
            if (wmax == box && run * per_channel(ang) <= kSoloStageBytes)
                break;
            if (run > 1)
                run /= 2;
            else if (ang > 1 && (ang > 2 || solo_smem_bytes(wmax, 1, prec, ang, split, all) >
                                                (size_t)kMaxSmemPerCta))
                --ang;
            else
                break;
        }
        // angle groups and channel steps as even as possible
        ngr = (na + ang - 1) / ang;
        ang = (na + ngr - 1) / ngr;
        const int cap = std::min({kMaxGroup, 32 / ang * run, h->g.ne}) / run * run;
        group = std::min(cap, std::max(run, kSoloStageBytes / per_channel(ang) / run * run));
        const int steps = (h->g.ne + group - 1) / group;
        group = std::min(cap, ((h->g.ne + steps - 1) / steps + run - 1) / run * run);
    }
    auto p = std::make_unique<Plan>();
    int rc = angle_tables_dev(h, key, p->at);
    if (rc)
        return rc;
    p->ns = ns;
    p->na = na;
    p->prec = prec;
    p->wmax = wmax;
    p->box = box;
    p->run = run;
    p->group = group;
    p->nsp = (ns + kPadL + 7) / 8 * 8;
    p->rows = rows;
    p->split = split;
    p->ang = ang;
    p->ang_groups = ngr;
    p->tiles_x = (h->g.nx + kTileCols - 1) / kTileCols;
    p->tiles_z = (h->g.nz + tr - 1) / tr;
    const int nxp = pad_cols(h->g.nx), ne = h->g.ne;
    const size_t ntiles = (size_t)p->tiles_x * p->tiles_z;
    if (solo) {
        const size_t steps = (size_t)ngr * ((ne + group - 1) / group);
        if (!rc) rc = p->wtab.ensure(steps * ntiles * solo_record_words(ang, group / run) * sizeof(int));
    } else {
        if (!rc) rc = p->wtab.ensure(na * ntiles * ne * sizeof(int));
        if (!rc) rc = p->btab.ensure(na * ntiles * ne * sizeof(int));
    }
    if (rc)
        return rc;
    CUtensorMap maps[2];
    rc = encode_map(&maps[0], p->at->valid.p, solo ? ne : na * ne, nxp, 4, kTileCols, p->group,
                    solo ? na : 0, ang);
    if (!rc)
        rc = encode_map(&maps[1], h->dx2.p, ne, nxp, 4, kTileCols, p->group);
    if (!rc)
        rc = p->maps.upload(maps, sizeof maps);
    if (rc)
        return rc;
    // window starts of every (angle, tile, channel), once per plan
    PlanJob pj{};
    pj.colK = (const int *)p->at->colK.p;
    pj.colF = (const float *)p->at->colF.p;
    pj.rowK = (const int *)p->at->rowK.p;
    pj.rowF = (const float *)p->at->rowF.p;
    pj.rowZ = (const float *)h->rowZ.p;
    pj.valid = (const short2 *)p->at->valid.p;
    pj.dx2 = (const float *)h->dx2.p;
    pj.wtab = (int *)p->wtab.p;
    pj.btab = (int *)p->btab.p;
    pj.nx = h->g.nx;
    pj.nxp = nxp;
    pj.nz = h->g.nz;
    pj.na = na;
    pj.ne = ne;
    pj.rows = p->rows;
    pj.bands = bands;
    pj.tiles_x = p->tiles_x;
    pj.tiles_z = p->tiles_z;
    pj.wmax = p->wmax;
    pj.align = 16 / pair_bytes(prec);
    pj.ang_groups = ngr;
    pj.run = run;
    pj.group = group;
    DevMem errw;
    rc = errw.ensure(sizeof(int));
    if (rc)
        return rc;
    cudaStream_t st;
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaStreamCreate");
    int herr = 0;
    e = cudaMemsetAsync(errw.p, 0, sizeof(int), st);
    if (e == cudaSuccess)
        e = solo ? launch_solo_plan(pj, (int *)errw.p, st) : launch_plan(pj, (int *)errw.p, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&herr, errw.p, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    if (e != cudaSuccess)
        return cuda_fail(e, "window planner");
    if (herr)
        return fail(BF_ECUDA, "window planner: a tile's delays span more than %d samples", p->wmax);
    *out = p.get();
    h->plans.emplace(std::move(key), std::move(p));
    return BF_OK;
}

// ------------------------------------------------------- frame preparation --

static constexpr double kPi = 3.14159265358979323846;

static int popcount4(int m) { return (m & 1) + ((m >> 1) & 1) + ((m >> 2) & 1) + ((m >> 3) & 1); }

// Images one frame produces: one per selected RF or IQ combiner.
static int frame_images(uint32_t flags)
{
    return popcount4(flags & BF_MODE_MASK) + ((flags & BF_IQDAS) ? 1 : 0) +
           ((flags & BF_BBDMAS) ? 1 : 0);
}

int frame_prec(uint32_t flags)
{
    return (flags & BF_IQ_MASK) ? (int)kPrecIQ : (int)((flags & BF_PREC_MASK) >> 4);
}

int check_frame_args(bf_handle *h, int ns, const double *angles, int na, uint32_t flags)
{
    if (!h)
        return fail(BF_EINVAL, "null handle");
    if (ns < 2 || ns > (1 << 24))
        return fail(BF_EINVAL, "n_samples must be in [2, 2^24], got %d", ns);
    if (na < 1 || na > 256)
        return fail(BF_EINVAL, "n_angles must be in [1, 256], got %d", na);
    if (!angles)
        return fail(BF_EINVAL, "null angles");
    for (int a = 0; a < na; ++a)
        if (!std::isfinite(angles[a]) || std::fabs(angles[a]) >= 1.5707963267948966)
            return fail(BF_EINVAL, "angle %d (%g rad) outside (-pi/2, pi/2)", a, angles[a]);
    const int modes = flags & BF_MODE_MASK, iq = flags & BF_IQ_MASK;
    if (!modes && !iq)
        return fail(BF_EINVAL,
                    "no combiner selected (BF_DAS / BF_DMAS / BF_CF / BF_PDAS / BF_IQDAS / BF_BBDMAS)");
    if (flags & ~(uint32_t)(BF_MODE_MASK | BF_IQ_MASK | BF_PREC_MASK | BF_OUT_MASK))
        return fail(BF_EINVAL, "unknown bits in mode_and_flags 0x%x", flags);
    const int prec = (flags & BF_PREC_MASK) >> 4;
    if (prec > kPrecBF16)
        return fail(BF_EINVAL, "unknown precision bits");
    if (iq) {
        if (modes)
            return fail(BF_EINVAL, "IQ combiners cannot be combined with RF combiners in one call");
        if (prec != kPrecF32)
            return fail(BF_EINVAL, "IQ combiners use FP32 storage");
        if (ns < 4 || ns > 8192 || (ns & (ns - 1)) != 0)
            return fail(BF_EINVAL, "IQ combiners need a power-of-two n_samples in [4, 8192] (got %d)",
                        ns);
    }
    const int stage = flags & BF_OUT_MASK;
    if (stage != BF_OUT_RF && stage != BF_OUT_ENV && stage != BF_OUT_LOGDB)
        return fail(BF_EINVAL, "unknown output stage bits");
    if (stage != BF_OUT_RF && h->g.nz > 4096)
        return fail(BF_EINVAL, "envelope detection supports nz <= 4096 (got %d)", h->g.nz);
    if ((long long)na * h->g.ne > (1LL << 30))
        return fail(BF_EINVAL, "too many channel records");
    return BF_OK;
}

size_t frame_out_bytes(const bf_handle *h, uint32_t flags)
{
    return (size_t)frame_images(flags) * (size_t)h->g.nx * (size_t)h->g.nz * sizeof(float);
}

static int plan_frames_per_job(const Plan *p, int modes, int prec, int cap);

int prepare_frame(bf_handle *h, const int16_t *rf_dev, int ns, const double *angles, int na,
                  uint32_t flags, float *out_dev, FrameScratch &s, FramePrep &fp, int nf_cap,
                  PlanWish wish, bool late_solo)
{
    int rc = check_frame_args(h, ns, angles, na, flags);
    if (rc)
        return rc;
    const int prec = frame_prec(flags);
    const bool iq = prec == kPrecIQ;
    Plan *plan = nullptr;
    wish.alone = nf_cap == 1 || !sharing_modes(flags);
    Plan *solo = nullptr;
    rc = handle_plan(h, ns, angles, na, flags, &plan, wish);
    if (!rc && late_solo && !wish.alone) {
        wish.alone = true;
        rc = handle_plan(h, ns, angles, na, flags, &solo, wish);
    }
    if (rc)
        return rc;
    const int modes = flags & (BF_MODE_MASK | BF_IQ_MASK), nm = frame_images(flags);
    const int stage = flags & BF_OUT_MASK;
    const size_t img = (size_t)h->g.nx * h->g.nz;
    const int rows = na * h->g.ne;
    // room for the frames of a job this frame may lead (interleaved pairs)
    int cap = plan_frames_per_job(plan, modes, prec, nf_cap);
    cap = wish.room > 0 ? std::min(cap, wish.room) : pairs_room(cap, wish.index, wish.peers, true);
    rc = s.pairs.ensure((size_t)cap * rows * plan->nsp * pair_bytes(prec));
    if (!rc && stage != BF_OUT_RF && !iq)  // IQ images are magnitudes already
        rc = s.y.ensure(nm * img * sizeof(float));
    if (!rc && stage == BF_OUT_LOGDB)
        rc = s.env.ensure(nm * img * sizeof(float));
    if (!rc)
        rc = s.maxbits.ensure(4 * sizeof(unsigned));
    if (rc)
        return rc;
    fp = FramePrep{};
    fp.h = h;
    fp.plan = plan;
    fp.solo = solo;
    fp.rf = rf_dev;
    fp.ns = ns;
    fp.na = na;
    fp.modes = modes;
    fp.pdas_p = h->pdas_p;
    fp.stage = stage;
    fp.prec = prec;
    fp.out = out_dev;
    fp.pairs = s.pairs.p;
    if (iq) {  // the beamformer writes magnitudes: straight out, or into the log stage's input
        fp.y = stage == BF_OUT_LOGDB ? (float *)s.env.p : out_dev;
        fp.env = stage == BF_OUT_LOGDB ? (float *)s.env.p : nullptr;
    } else {
        fp.y = stage == BF_OUT_RF ? out_dev : (float *)s.y.p;
        fp.env = stage == BF_OUT_ENV ? out_dev : (stage == BF_OUT_LOGDB ? (float *)s.env.p : nullptr);
    }
    fp.maxbits = (unsigned *)s.maxbits.p;
    fp.nf_cap = cap;
    fp.scratch = &s;
    if (stage != BF_OUT_RF && !iq) {
        const bool warp = envelope_warp_ok(h->g.nz);
        rc = fft_tables(warp ? h->g.nz : 0, fp.ft);
        if (!rc && !warp && (modes & ~BF_DMAS))
            rc = env_tables(h->g.nz, false, 0, 0, fp.et[0]);
        if (!rc && !warp && (modes & BF_DMAS))
            rc = env_tables(h->g.nz, true, h->kb_lo, h->kb_hi, fp.et[1]);
        if (rc)
            return rc;
    }
    if (iq) {
        rc = fft_tables(ns < 32 ? ns : 0, fp.dt);
        if (rc)
            return rc;
    }
    return BF_OK;
}

// Host-side launch description of a set of frames (job arrays + prefixes).
// Frames can share one beamforming job (and every delay) when they use the
// same plan with the same combiners: DAS and / or DMAS of RF records, or
// IQ-DAS and / or BB-DMAS (which share the carrier phase as well), up to two
// frames on 32-row tiles and four on 16-row tiles.
static int plan_frames_per_job(const Plan *p, int modes, int prec, int cap)
{
    const int m = modes & (BF_MODE_MASK | BF_IQ_MASK);
    if (p->split || !sharing_modes((uint32_t)m))
        return 1;
    if (prec == kPrecIQ && p->ns > 4096)
        return 1;  // long records: every frame alone
    for (int nf = p->rows == 2 ? 4 : p->rows == 4 ? 2 : 1; nf > 1; nf /= 2)
        if (nf <= cap &&
            beamform_smem_bytes(p->wmax, p->group, prec, nf, p->rows) <= (size_t)kMaxSmemPerCta &&
            interleaved_box(p->wmax, nf, prec) > 0)
            return nf;
    return 1;
}

int job_frames_cap(const Plan *p, uint32_t flags, int cap)
{
    return plan_frames_per_job(p, (int)(flags & (BF_MODE_MASK | BF_IQ_MASK)), frame_prec(flags), cap);
}

// Tensor map over the pairs of a job that frame f leads (nf frames interleaved, box
// pairs per copy), encoded when the layout changed.
static int job_map(const FramePrep &f, int nf, int box, CUtensorMap &out)
{
    FrameScratch &S = *f.scratch;
    const Plan *p = f.plan;
    const int rows = f.na * f.h->g.ne, run = nf == 1 ? p->run : 1;
    const int key[7] = {rows, p->nsp, box, run, f.prec, nf, 1};
    if (S.map_base != f.pairs || !std::equal(key, key + 7, S.map_key)) {
        const int k = pair_elems(f.prec);  // IQ pairs: two 8-byte elements each
        S.map_key[6] = 0;
        int rc = encode_map(&S.map, f.pairs, rows, p->nsp * nf * k, pair_bytes(f.prec) / k,
                            box * nf * k, run);
        if (rc)
            return rc;
        S.map_base = f.pairs;
        std::copy(key, key + 7, S.map_key);
    }
    out = S.map;
    return BF_OK;
}

static bool shareable(const FramePrep &a, const FramePrep &b)
{
    const int m = a.modes & (BF_MODE_MASK | BF_IQ_MASK);
    return a.plan == b.plan && a.h == b.h && m == (b.modes & (BF_MODE_MASK | BF_IQ_MASK)) &&
           a.prec == b.prec && a.na == b.na && a.ns == b.ns;
}

void use_solo_plans(std::vector<FramePrep> &frames)
{
    for (size_t i = 0; i < frames.size(); ++i) {
        FramePrep &f = frames[i];
        if (!f.solo || !f.solo->split)
            continue;
        bool alone = true;
        for (size_t j = 0; j < frames.size() && alone; ++j)
            alone = j == i || !(frames[j].solo == f.solo && shareable(f, frames[j]));
        if (alone)
            f.plan = f.solo;
    }
}

// The job of frame fi, the first that none has taken: its lead (whose pairs buffer holds
// them all) and its partners.  Frames that can lead nothing are taken before those that
// can, which are kept for further jobs.
static std::vector<size_t> job_frames(const std::vector<FramePrep> &frames, const std::vector<char> &taken,
                                      size_t fi)
{
    const FramePrep &f = frames[fi];
    const size_t want = (size_t)plan_frames_per_job(f.plan, f.modes, f.prec, kMaxFramesPerJob);
    std::vector<size_t> rest, leads;  // after fi, in order
    for (size_t gi = fi + 1; gi < frames.size() && want > 1; ++gi) {
        const bool full = rest.size() + 1 >= want || leads.size() >= 2 * want;
        if (full && (f.nf_cap > 1 || !leads.empty()))
            break;  // enough partners, and a lead among them
        if (taken[gi] || !shareable(f, frames[gi]))
            continue;
        if (frames[gi].nf_cap > 1)
            leads.push_back(gi);
        else if (rest.size() + 1 < want)
            rest.push_back(gi);
    }
    std::vector<size_t> job{fi};
    if (f.nf_cap == 1) {
        if (leads.empty())
            return job;
        auto most = std::max_element(leads.begin(), leads.end(), [&](size_t a, size_t b) {
            return frames[a].nf_cap < frames[b].nf_cap;
        });
        job.insert(job.begin(), *most);
        leads.erase(most);
    }
    rest.insert(rest.end(), leads.begin(), leads.end());
    const size_t most = std::min({want, (size_t)frames[job[0]].nf_cap, job.size() + rest.size()});
    const size_t nf = most >= 4 ? 4 : most >= 2 ? 2 : 1;
    for (size_t q = 0; job.size() < nf; ++q)
        job.push_back(rest[q]);
    return job;
}

int build_launch(const std::vector<FramePrep> &frames, HostLaunch &hl)
{
    hl = HostLaunch{};
    std::map<int, std::vector<BfJob>> groups;
    std::map<int, size_t> group_smem;
    std::vector<char> taken(frames.size(), 0);
    // frames riding in another frame's job (the lead carries the job's ingest)
    std::vector<char> member(frames.size(), 0);
    std::vector<std::vector<size_t>> partners(frames.size());
    for (size_t fi = 0; fi < frames.size(); ++fi) {
        if (taken[fi])
            continue;
        // partner frames of the same plan, if any: all ride in one job (1, 2 or 4 frames)
        std::vector<size_t> job = job_frames(frames, taken, fi);
        int nf = (int)job.size();
        int box_nf = 0;
        CUtensorMap map;
        if (nf > 1) {
            const FramePrep &l = frames[job[0]];
            box_nf = interleaved_box(l.plan->wmax, nf, l.prec);
            if (job_map(l, nf, box_nf, map) != BF_OK) {  // no interleaved map: every frame alone
                job = {fi};
                nf = 1;
            }
        }
        const size_t lead = job[0];
        const FramePrep &f = frames[lead];
        if (nf == 1) {
            int rc = job_map(f, 1, f.plan->box, map);
            if (rc)
                return rc;
        }
        const FramePrep *more[kMaxFramesPerJob - 1] = {};
        taken[lead] = 1;
        for (int q = 0; q < nf - 1; ++q) {
            more[q] = &frames[job[q + 1]];
            taken[job[q + 1]] = 1;
            member[job[q + 1]] = 1;
            partners[lead].push_back(job[q + 1]);
        }
        const bf_handle *h = f.h;
        const Plan *p = f.plan;
        BfJob j{};
        j.colK = (const int *)p->at->colK.p;
        j.colF = (const float *)p->at->colF.p;
        j.rowK = (const int *)p->at->rowK.p;
        j.rowF = (const float *)p->at->rowF.p;
        j.rowZ = (const float *)h->rowZ.p;
        j.wtab = (const int *)p->wtab.p;
        j.btab = (const int *)p->btab.p;
        j.apcnt = (const uint16_t *)h->apcnt.p;
        j.rf_map = (const CUtensorMap *)hl.maps.size();
        hl.maps.push_back(map);
        j.valid_map = (const CUtensorMap *)p->maps.p;
        j.dx2_map = (const CUtensorMap *)p->maps.p + 1;
        j.y = f.y;
        j.nx = h->g.nx;
        j.nz = h->g.nz;
        j.na = f.na;
        j.ne = h->g.ne;
        j.wmax = p->wmax;
        j.box = p->box;
        j.group = p->group;
        j.ang_groups = p->ang_groups;
        j.run = p->run;
        j.rows = p->rows;
        // the IQ kernel reads its two combiners from the DAS / DMAS slots of the mode word
        j.modes = f.prec == kPrecIQ ? (((f.modes & BF_IQDAS) ? BF_DAS : 0) |
                                       ((f.modes & BF_BBDMAS) ? BF_DMAS : 0))
                                    : f.modes;
        j.tiles_x = p->tiles_x;
        j.tiles_z = p->tiles_z;
        j.out_scale = (f.prec == kPrecF32 || f.prec == kPrecIQ) ? 1.0f : 32768.0f;
        j.pdas_p = (float)f.pdas_p;
        j.pdas_inv_p = (float)(1.0 / f.pdas_p);
        const double r = h->g.f0 / h->g.fs;  // carrier cycles per sample
        j.iq_c1 = (float)(2.0 * kPi * r);
        j.iq_c2 = (float)(kPi * r);
        j.maxbits = (f.prec == kPrecIQ && f.stage == BF_OUT_LOGDB) ? f.maxbits : nullptr;
        for (int q = 0; q < kMaxFramesPerJob - 1; ++q) {
            j.y_more[q] = more[q] ? more[q]->y : nullptr;
            j.maxbits_more[q] = (more[q] && f.prec == kPrecIQ && more[q]->stage == BF_OUT_LOGDB)
                                    ? more[q]->maxbits
                                    : nullptr;
        }
        if (nf > 1)  // the frames' pairs interleaved in the lead's scratch
            j.box = box_nf;
        const int combiners = j.modes & (BF_DMAS | BF_CF | BF_PDAS);
        const int variant =
            ((((p->split * 2 + (p->ang > 1 ? 1 : 0)) * 8 + nf) * 16 + p->rows) * 4 + f.prec) * 16 +
            combiners;
        groups[variant].push_back(j);
        const size_t sm = p->split
                              ? solo_smem_bytes(p->wmax, p->group, f.prec, p->ang, p->split, combiners)
                              : beamform_smem_bytes(p->wmax, p->group, f.prec, nf, p->rows);
        group_smem[variant] = std::max(group_smem[variant], sm);
        hl.smem = std::max(hl.smem, sm);
    }
    for (auto &kv : groups) {
        HostLaunch::Group g;
        g.split = kv.first / (2 * 8 * 16 * 4 * 16);
        g.ang = kv.first / (8 * 16 * 4 * 16) % 2 ? kSoloAngles : 1;
        g.nf = (kv.first / (16 * 4 * 16)) % 8;
        g.rows = (kv.first / 64) % 16;
        g.prec = (kv.first / 16) % 4;
        g.variant = kv.first % 16;
        g.smem = group_smem[kv.first];
        g.first = (int)hl.jobs.size();
        g.count = (int)kv.second.size();
        g.prefix_first = (int)hl.tile_prefix.size();
        int acc = 0;
        for (const BfJob &j : kv.second) {
            hl.tile_prefix.push_back(acc);
            acc += j.tiles_x * j.tiles_z;
            hl.jobs.push_back(j);
        }
        g.tiles = acc;
        hl.groups.push_back(g);
    }
    // the largest launches first: the others fill in as their last CTAs leave
    std::stable_sort(hl.groups.begin(), hl.groups.end(),
                     [](const HostLaunch::Group &a, const HostLaunch::Group &b) { return a.tiles > b.tiles; });
    std::map<int, std::vector<IngestJob>> ig;
    // IQ frames: one demodulation job per frame, or per frame pair of a
    // multi-frame job (into the lead's interleaved array)
    for (size_t fi = 0; fi < frames.size(); ++fi) {
        const FramePrep &f = frames[fi];
        if (f.prec != kPrecIQ || member[fi])
            continue;
        std::vector<size_t> job{fi};
        job.insert(job.end(), partners[fi].begin(), partners[fi].end());
        const int nf = (int)job.size();
        const double r = f.h->g.f0 / f.h->g.fs;
        for (int q = 0; q < (nf == 1 ? 1 : nf / 2); ++q) {
            const FramePrep &a = frames[job[nf == 1 ? 0 : 2 * q]];
            DemodJob d{};
            d.rf = a.rf;
            d.pairs = (float4 *)f.pairs;
            d.nf = nf;
            d.fi = nf == 1 ? 0 : 2 * q;
            d.rows = f.na * f.h->g.ne;
            d.ns = f.ns;
            d.nsp = f.plan->nsp;
            d.lgn = 0;
            while ((1 << d.lgn) < f.ns)
                ++d.lgn;
            d.rot = make_float2((float)std::cos(2.0 * kPi * r), (float)-std::sin(2.0 * kPi * r));
            (f.ns < 32 ? d.tw : d.ptw) = (const float2 *)f.dt->tw.p;
            d.maxbits = a.stage != BF_OUT_RF ? a.maxbits : nullptr;
            if (nf > 1) {
                const FramePrep &b = frames[job[2 * q + 1]];
                d.rf2 = b.rf;
                d.maxbits2 = b.stage != BF_OUT_RF ? b.maxbits : nullptr;
            }
            const int kind = f.ns < 32 ? 2 : f.ns > 4096 ? 1 : 0;
            const int per = kind == 2 ? 1 : demod_units_per_block(d.lgn);
            const int units = kind == 2 || nf > 1 ? d.rows : (d.rows + 1) / 2;
            hl.demod_prefix[kind].push_back(hl.demod_blocks[kind]);
            hl.demod_blocks[kind] += (units + per - 1) / per;
            hl.demod[kind].push_back(d);
        }
    }
    for (size_t fi = 0; fi < frames.size(); ++fi) {
        const FramePrep &f = frames[fi];
        if (f.prec == kPrecIQ || member[fi])
            continue;  // IQ frames demodulate; members of a job come with its lead
        IngestJob ij{};
        ij.rf = f.rf;
        ij.pairs = f.pairs;
        ij.rows = f.na * f.h->g.ne;
        ij.ns = f.ns;
        ij.nsp = f.plan->nsp;
        ij.maxbits = f.stage != BF_OUT_RF ? f.maxbits : nullptr;
        ij.nf = 1 + (int)partners[fi].size();
        if (ij.nf > 1) {  // the whole job, interleaved into the lead's pairs
            for (size_t q = 0; q < partners[fi].size(); ++q) {
                const FramePrep &g = frames[partners[fi][q]];
                ij.rf_more[q] = g.rf;
                ij.maxbits_more[q] = g.stage != BF_OUT_RF ? g.maxbits : nullptr;
            }
        }
        // nsp is a multiple of 8: units of sixteen bytes, or of eight pairs of a frame pair
        const bool frames_f32 = f.prec == kPrecF32 && ij.nf > 1;
        ij.units = ij.nsp / 8 * (frames_f32 ? ij.nf / 2 : ij.nf * pair_bytes(f.prec) / 2);
        ij.per = 1;
        ig[f.prec].push_back(ij);
    }
    for (auto &kv : ig) {
        HostLaunch::IGroup g;
        g.prec = kv.first;
        g.first = (int)hl.ingest.size();
        g.count = (int)kv.second.size();
        g.prefix_first = (int)hl.ingest_prefix.size();
        long long single = 0;
        for (const IngestJob &j : kv.second)
            single += ingest_blocks(j);
        g.wide = single >= kIngestWide;
        int acc = 0;
        for (IngestJob &j : kv.second) {
            if (g.wide && (j.nf == 1 || g.prec != kPrecF32))
                j.per = ingest_units(j.nf);
            hl.ingest_prefix.push_back(acc);  // first CTA of the job
            acc += ingest_blocks(j);
            hl.ingest.push_back(j);
        }
        g.blocks = acc;
        hl.igroups.push_back(g);
    }
    long long blks = 0;
    for (const FramePrep &f : frames) {
        if (f.stage == BF_OUT_RF)
            continue;
        const bf_handle *h = f.h;
        const size_t img = (size_t)h->g.nx * h->g.nz;
        if (f.prec == kPrecIQ) {  // magnitude images: only the log stage follows
            if (f.stage != BF_OUT_LOGDB)
                continue;
            const int nimg = ((f.modes & BF_IQDAS) ? 1 : 0) + ((f.modes & BF_BBDMAS) ? 1 : 0);
            for (int slot = 0; slot < nimg; ++slot) {
                LogJob l{};
                l.env = f.env + slot * img;
                l.out = f.out + slot * img;
                l.maxbits = f.maxbits + slot;
                l.n = (int)img;
                l.vec4 = (img % 4 == 0 && ((uintptr_t)l.env & 15) == 0 && ((uintptr_t)l.out & 15) == 0)
                             ? 1
                             : 0;
                hl.blk_prefix.push_back((int)blks);
                blks += log_blocks((long long)img);
                hl.log.push_back(l);
            }
            continue;
        }
        int slot = 0;
        for (int bit = 1; bit <= BF_PDAS; bit <<= 1) {
            if (!(f.modes & bit))
                continue;
            EnvJob e{};
            e.y = f.y + slot * img;
            e.env = f.env + slot * img;
            e.maxbits = f.maxbits + slot;
            e.nx = h->g.nx;
            e.nz = h->g.nz;
            e.band = bit == BF_DMAS ? 1 : 0;
            e.kb_lo = h->kb_lo;
            e.kb_hi = h->kb_hi;
            if (envelope_warp_ok(e.nz)) {
                e.tw = (const float2 *)f.ft->tw.p;
                hl.envw_prefix.push_back(hl.envw_pairs);
                hl.envw_pairs += (h->g.nx + 1) / 2;
                hl.envw.push_back(e);
            } else {
                const EnvTablesDev &t = *f.et[e.band];
                e.lg = t.lg;
                e.conv = t.conv;
                e.ptw = (const float2 *)f.ft->tw.p;
                e.gr = (const float *)t.gr.p;
                e.gh = (const float *)t.gh.p;
                const int big = e.lg > 12 ? 1 : 0, per = 2 * envelope_pairs_per_block(e.lg);
                hl.env_prefix[big].push_back(hl.env_blocks[big]);
                hl.env_blocks[big] += (h->g.nx + per - 1) / per;
                hl.env[big].push_back(e);
            }
            if (f.stage == BF_OUT_LOGDB) {
                LogJob l{};
                l.env = e.env;
                l.out = f.out + slot * img;
                l.maxbits = e.maxbits;
                l.n = (int)img;
                l.vec4 = (img % 4 == 0 && ((uintptr_t)l.env & 15) == 0 && ((uintptr_t)l.out & 15) == 0)
                             ? 1
                             : 0;
                hl.blk_prefix.push_back((int)blks);
                blks += log_blocks((long long)img);
                hl.log.push_back(l);
            }
            ++slot;
        }
    }
    hl.log_blocks = (int)blks;
    return BF_OK;
}

int DeviceLaunch::upload(const HostLaunch &hl, cudaStream_t st, bool async)
{
    size_t total = 0;
    auto room = [&](size_t n) {  // tensor maps want 64-byte alignment
        const size_t at = total;
        total += (n + 127) & ~(size_t)127;
        return at;
    };
    std::vector<std::pair<const void *, std::pair<size_t, size_t>>> parts;  // source, (offset, bytes)
    auto add = [&](const auto &v) {
        const size_t n = v.size() * sizeof(v[0]), at = room(n);
        parts.push_back({v.data(), {at, n}});
        return at;
    };
    const size_t a_maps = add(hl.maps), a_jobs = add(hl.jobs), a_tp = add(hl.tile_prefix),
                 a_in = add(hl.ingest), a_ip = add(hl.ingest_prefix), a_e0 = add(hl.env[0]),
                 a_ep0 = add(hl.env_prefix[0]), a_e1 = add(hl.env[1]), a_ep1 = add(hl.env_prefix[1]),
                 a_ew = add(hl.envw), a_ewp = add(hl.envw_prefix), a_log = add(hl.log),
                 a_bp = add(hl.blk_prefix);
    size_t a_dm[3], a_dp[3];
    for (int k = 0; k < 3; ++k) {
        a_dm[k] = add(hl.demod[k]);
        a_dp[k] = add(hl.demod_prefix[k]);
    }
    int rc = pack.reserve(std::max<size_t>(total, 128));
    if (!rc)
        rc = err.ensure(sizeof(int));
    if (rc)
        return rc;
    char *d = (char *)pack.p;
    std::vector<char> host(total);
    for (const auto &q : parts)
        if (q.second.second)
            std::memcpy(host.data() + q.second.first, q.first, q.second.second);
    for (size_t k = 0; k < hl.jobs.size(); ++k) {  // map indices to addresses
        BfJob j = hl.jobs[k];
        j.rf_map = (const CUtensorMap *)(d + a_maps) + (size_t)j.rf_map;
        std::memcpy(host.data() + a_jobs + k * sizeof(BfJob), &j, sizeof j);
    }
    if (total) {
        cudaError_t e = async ? cudaMemcpyAsync(d, host.data(), total, cudaMemcpyHostToDevice, st)
                              : cudaMemcpy(d, host.data(), total, cudaMemcpyHostToDevice);
        if (e != cudaSuccess)
            return cuda_fail(e, "cudaMemcpy (job lists)");
    }
    jobs = (const BfJob *)(d + a_jobs);
    tile_prefix = (const int *)(d + a_tp);
    ingest = (const IngestJob *)(d + a_in);
    ingest_prefix = (const int *)(d + a_ip);
    env[0] = (const EnvJob *)(d + a_e0);
    env[1] = (const EnvJob *)(d + a_e1);
    env_prefix[0] = (const int *)(d + a_ep0);
    env_prefix[1] = (const int *)(d + a_ep1);
    envw = (const EnvJob *)(d + a_ew);
    envw_prefix = (const int *)(d + a_ewp);
    log = (const LogJob *)(d + a_log);
    blk_prefix = (const int *)(d + a_bp);
    for (int k = 0; k < 3; ++k) {
        demod[k] = (const DemodJob *)(d + a_dm[k]);
        demod_prefix[k] = (const int *)(d + a_dp[k]);
    }
    return BF_OK;
}

// The envelope launches of a set of frames: 512-row images, then the others.
static cudaError_t launch_envelopes(const HostLaunch &hl, DeviceLaunch &dl, cudaStream_t st)
{
    cudaError_t e = launch_envelope_warp(dl.envw, dl.envw_prefix,
                                         (int)hl.envw.size(), hl.envw_pairs, st);
    for (int b = 1; b >= 0 && e == cudaSuccess; --b)
        e = launch_envelope(dl.env[b], dl.env_prefix[b],
                            (int)hl.env[b].size(), hl.env_blocks[b], b == 1, st);
    return e;
}

// The device work of a set of frames, in stream order: ingest, reset of the
// frame maxima, beamforming (one launch per precision / combiner variant),
// envelope, log compression.
int enqueue(const std::vector<FramePrep> &frames, const HostLaunch &hl, DeviceLaunch &dl,
            cudaStream_t st, cudaEvent_t *marks, const MarkBranch *branch)
{
    cudaError_t e;
    // Inside a stream capture the marks must be external event records (they
    // become graph nodes that record at replay time); outside, plain records.
    // An event record between two kernels of a graph costs about 2 us and
    // keeps the next kernel from being launched ahead, so in a capture with a
    // branch the marks hang off a side stream instead.
    unsigned mark_flags = cudaEventRecordDefault;
    if (marks) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        e = cudaStreamIsCapturing(st, &cs);
        if (e != cudaSuccess)
            return cuda_fail(e, "cudaStreamIsCapturing");
        if (cs == cudaStreamCaptureStatusActive)
            mark_flags = cudaEventRecordExternal;
        else
            branch = nullptr;
    }
    auto mark = [&](int k) -> cudaError_t {
        if (!marks)
            return cudaSuccess;
        if (!branch)
            return cudaEventRecordWithFlags(marks[k], st, mark_flags);
        cudaError_t r = cudaEventRecord(branch->fork[k], st);
        if (r == cudaSuccess)
            r = cudaStreamWaitEvent(branch->side, branch->fork[k], 0);
        if (r == cudaSuccess)
            r = cudaEventRecordWithFlags(marks[k], branch->side, mark_flags);
        return r;
    };
    e = mark(0);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaEventRecord (mark)");
    for (const HostLaunch::IGroup &g : hl.igroups) {
        e = launch_ingest(dl.ingest + g.first, dl.ingest_prefix + g.prefix_first, g.count, g.blocks,
                          g.prec, g.wide, st);
        if (e != cudaSuccess)
            return cuda_fail(e, "ingest launch");
    }
    for (int k = 0; k < 3; ++k) {
        const int n = (int)hl.demod[k].size();
        e = k == 2 ? launch_demod(dl.demod[k], dl.demod_prefix[k], n, hl.demod_blocks[k], st)
                   : launch_demod16(dl.demod[k], dl.demod_prefix[k], n, hl.demod_blocks[k], k == 1, st);
        if (e != cudaSuccess)
            return cuda_fail(e, "demodulation launch");
    }
    // (the ingest / demodulation launches above zeroed each frame's image maxima)
    e = mark(1);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaEventRecord (mark)");
    // in a capture with a branch, launches after the first go to its work streams
    const int spread = branch ? std::min<int>((int)hl.groups.size() - 1, MarkBranch::kWork) : 0;
    if (spread > 0)
        e = cudaEventRecord(branch->work_fork, st);
    for (int w = 0; w < spread && e == cudaSuccess; ++w)
        e = cudaStreamWaitEvent(branch->work[w], branch->work_fork, 0);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaEventRecord (fork)");
    for (size_t k = 0; k < hl.groups.size(); ++k) {
        const HostLaunch::Group &g = hl.groups[k];
        const cudaStream_t to = spread > 0 && k > 0 ? branch->work[(k - 1) % spread] : st;
        const BfJob *jobs = dl.jobs + g.first;
        const int *prefix = dl.tile_prefix + g.prefix_first;
        e = g.split ? launch_solo(jobs, prefix, g.count, g.tiles, g.smem, g.prec, g.variant, g.split,
                                  g.ang, (int *)dl.err.p, to)
                    : launch_beamform(jobs, prefix, g.count, g.tiles, g.smem, g.prec, g.variant,
                                      g.rows, g.nf, (int *)dl.err.p, to);
        if (e != cudaSuccess)
            return cuda_fail(e, "beamform launch");
    }
    for (int w = 0; w < spread && e == cudaSuccess; ++w) {
        e = cudaEventRecord(branch->work_join[w], branch->work[w]);
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(st, branch->work_join[w], 0);
    }
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaStreamWaitEvent (join)");
    e = mark(2);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaEventRecord (mark)");
    e = launch_envelopes(hl, dl, st);
    if (e != cudaSuccess)
        return cuda_fail(e, "envelope launch");
    if (!hl.log.empty()) {
        e = launch_log(dl.log, dl.blk_prefix, (int)hl.log.size(),
                       hl.log_blocks, 70.0f, st);
        if (e != cudaSuccess)
            return cuda_fail(e, "log launch");
    }
    e = mark(3);
    if (e == cudaSuccess && marks && branch) {  // the side branch back into st
        e = cudaEventRecord(branch->join, branch->side);
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(st, branch->join, 0);
    }
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaEventRecord (mark)");
    return BF_OK;
}

int read_device_error(DeviceLaunch &dl, cudaStream_t st)
{
    int v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, dl.err.p, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(st);
    if (e != cudaSuccess)
        return cuda_fail(e, "reading the device status word");
    if (v) {
        cudaMemsetAsync(dl.err.p, 0, sizeof(int), st);
        if (v & kErrTimeout)
            return fail(BF_ETIMEDOUT, "a bounded device wait gave up (status 0x%x)", v);
        return fail(BF_ECUDA, "device-side check failed (status 0x%x)", v);
    }
    return BF_OK;
}

bool is_device_pointer(const void *p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace bfi

using namespace bfi;

// ===================================================================== ABI ==

extern "C" {

BF_API const char *bf_last_error(void) { return g_err.c_str(); }

BF_API int bf_version(void) { return 100; }

BF_API int bf_create(const bf_geometry *geom, const bf_grid *grid, double fs_hz, double f0_hz,
                     double c_mps, bf_handle **out)
{
    if (!geom || !grid || !out)
        return fail(BF_EINVAL, "null argument");
    *out = nullptr;
    const int ne = geom->n_elements;
    if (ne < 1 || ne > 4096)
        return fail(BF_EINVAL, "n_elements must be in [1, 4096], got %d", ne);
    if (!(geom->f_number > 0.0) || !std::isfinite(geom->f_number))
        return fail(BF_EINVAL, "f_number must be > 0");
    if (!geom->x_elem_m && !(geom->pitch_m > 0.0 && std::isfinite(geom->pitch_m)))
        return fail(BF_EINVAL, "pitch_m must be > 0 when x_elem_m is NULL");
    if (grid->nx < 1 || grid->nz < 1 || grid->nx > 32767 || grid->nz > 32767)
        return fail(BF_EINVAL, "grid dimensions must be in [1, 32767]");
    const double v[] = {grid->x0_m, grid->x1_m, grid->z0_m, grid->z1_m, fs_hz, f0_hz, c_mps};
    for (double d : v)
        if (!std::isfinite(d))
            return fail(BF_EINVAL, "non-finite grid or acquisition parameter");
    if (grid->x1_m < grid->x0_m || grid->z1_m < grid->z0_m || grid->z0_m < 0.0)
        return fail(BF_EINVAL, "grid must satisfy x1 >= x0 and z1 >= z0 >= 0");
    if (!(fs_hz > 0.0) || !(c_mps > 0.0) || !(f0_hz > 0.0))
        return fail(BF_EINVAL, "fs, f0 and c must be > 0");
    auto h = std::make_unique<bf_handle>();
    GeomHost &g = h->g;
    g.ne = ne;
    g.xe.resize(ne);
    for (int i = 0; i < ne; ++i)
        g.xe[i] = geom->x_elem_m ? geom->x_elem_m[i]
                                 : ((double)i - 0.5 * (double)(ne - 1)) * geom->pitch_m;
    for (int i = 0; i < ne; ++i) {
        if (!std::isfinite(g.xe[i]))
            return fail(BF_EINVAL, "non-finite element position");
        if (i && !(g.xe[i] > g.xe[i - 1]))
            return fail(BF_EINVAL, "element positions must be strictly increasing");
    }
    g.fnum = geom->f_number;
    g.nx = grid->nx;
    g.nz = grid->nz;
    g.x0 = grid->x0_m;
    g.x1 = grid->x1_m;
    g.z0 = grid->z0_m;
    g.z1 = grid->z1_m;
    g.fs = fs_hz;
    g.f0 = f0_hz;
    g.c = c_mps;
    cudaError_t e = cudaGetDevice(&h->device);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaGetDevice");
    e = cudaStreamCreateWithFlags(&h->own_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaStreamCreate");
    h->stream = h->own_stream;
    e = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, h->device);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaDeviceGetAttribute");
    geometry_tables(g, h->geo);
    int rc = h->rowZ.upload(h->geo.rowZ.data(), h->geo.rowZ.size() * sizeof(float));
    if (!rc) rc = h->dx2.upload(h->geo.dx2.data(), h->geo.dx2.size() * sizeof(float));
    if (!rc) rc = h->apcnt.upload(h->geo.apcnt.data(), h->geo.apcnt.size() * sizeof(uint16_t));
    if (rc)
        return rc;
    bandpass_bins(g.nz, g.z0, g.z1, g.c, g.f0, h->kb_lo, h->kb_hi);
    *out = h.release();
    return BF_OK;
}

BF_API int bf_destroy(bf_handle *h)
{
    if (!h)
        return fail(BF_EINVAL, "null handle");
    {
        std::lock_guard<std::mutex> lk(h->mu);
        if (!h->tickets.empty())
            return fail(BF_EINVAL, "handle has %zu pending tickets", h->tickets.size());
    }
    cudaSetDevice(h->device);
    cudaStreamSynchronize(h->stream);
    h->call.clear();
    engine_forget(h);
    if (h->own_stream)
        cudaStreamDestroy(h->own_stream);
    delete h;
    return BF_OK;
}

BF_API int bf_set_stream(bf_handle *h, void *stream)
{
    if (!h)
        return fail(BF_EINVAL, "null handle");
    h->stream = stream ? (cudaStream_t)stream : h->own_stream;
    return BF_OK;
}

BF_API int bf_set_pdas_order(bf_handle *h, double p)
{
    if (!h)
        return fail(BF_EINVAL, "null handle");
    if (!(p >= 1.0 && p <= 16.0))
        return fail(BF_EINVAL, "pDAS order must be in [1, 16], got %g", p);
    h->pdas_p = p;
    return BF_OK;
}

BF_API size_t bf_output_bytes(const bf_handle *h, uint32_t flags)
{
    return h ? frame_out_bytes(h, flags) : 0;
}

BF_API int bf_beamform(bf_handle *h, const int16_t *rf_dev, int32_t n_samples,
                       const double *angles_rad, int32_t n_angles, uint32_t flags, float *out_dev)
{
    if (!h)
        return fail(BF_EINVAL, "null handle");
    if (!rf_dev || !out_dev)
        return fail(BF_EINVAL, "null data pointer");
    cudaSetDevice(h->device);
    CallCache &cc = h->call;
    if (cc.valid) {  // the same call as last time: no checks, no preparation, no uploads
        if (flags == cc.flags && rf_dev == cc.rf && out_dev == cc.out && n_samples == cc.ns &&
            n_angles == (int)cc.angles.size() && angles_rad && h->pdas_p == cc.pdas_p &&
            h->stream == cc.stream && forced_cfg() == cc.forced &&
            std::equal(cc.angles.begin(), cc.angles.end(), angles_rad)) {
            int rc = BF_OK;
            if (!cc.exec && ++cc.hits >= 1) {  // a repeat: capture the launches once
                cudaStream_t cap;
                cudaError_t e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
                if (e == cudaSuccess) {
                    e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
                    if (e == cudaSuccess) {
                        rc = enqueue(cc.frames, cc.hl, h->launch, cap);
                        cudaGraph_t g = nullptr;
                        e = cudaStreamEndCapture(cap, &g);
                        if (!rc && e == cudaSuccess)
                            e = cudaGraphInstantiate(&cc.exec, g, 0);
                        if (g)
                            cudaGraphDestroy(g);
                        if (e != cudaSuccess || rc) {
                            cudaGetLastError();
                            cc.exec = nullptr;  // stay on the plain replay
                        }
                        rc = BF_OK;
                    }
                    cudaStreamDestroy(cap);
                }
                cudaGetLastError();
            }
            if (cc.exec) {
                cudaError_t e = cudaGraphLaunch(cc.exec, h->stream);
                return e == cudaSuccess ? BF_OK : cuda_fail(e, "cudaGraphLaunch");
            }
            return enqueue(cc.frames, cc.hl, h->launch, h->stream);
        }
    }
    cc.clear();
    if (!is_device_pointer(rf_dev) || !is_device_pointer(out_dev))
        return fail(BF_EINVAL, "bf_beamform needs device pointers (use bf_submit for host data)");
    std::vector<FramePrep> frames(1);
    int rc = prepare_frame(h, rf_dev, n_samples, angles_rad, n_angles, flags, out_dev, h->scratch,
                           frames[0]);
    if (rc)
        return rc;
    HostLaunch hl;
    rc = build_launch(frames, hl);
    if (!rc)
        rc = h->launch.upload(hl, h->stream, true);
    if (!rc && !h->err_cleared) {
        cudaMemsetAsync(h->launch.err.p, 0, sizeof(int), h->stream);
        h->err_cleared = true;
    }
    if (!rc)
        rc = enqueue(frames, hl, h->launch, h->stream);
    if (!rc) {
        cc.valid = true;
        cc.forced = forced_cfg();
        cc.flags = flags;
        cc.rf = rf_dev;
        cc.out = out_dev;
        cc.ns = n_samples;
        cc.angles.assign(angles_rad, angles_rad + n_angles);
        cc.pdas_p = h->pdas_p;
        cc.stream = h->stream;
        cc.frames = frames;
        cc.hl = std::move(hl);
    }
    return rc;
}

// Plane-wave f-k migration of one device-resident frame onto the native grid
// (one column per element, depth step c / (2 fs)).
BF_API int bf_fkmig(bf_handle *h, const int16_t *rf_dev, int32_t n_samples,
                    const double *angles_rad, int32_t n_angles, uint32_t flags, float *out_dev)
{
    if (!h)
        return fail(BF_EINVAL, "null handle");
    if (!rf_dev || !out_dev || !angles_rad)
        return fail(BF_EINVAL, "null argument");
    if (flags & ~((uint32_t)BF_OUT_MASK | (uint32_t)BF_FK_STOLT))
        return fail(BF_EINVAL, "bf_fkmig takes only an output stage and BF_FK_STOLT in its flags");
    const bool stolt = (flags & BF_FK_STOLT) != 0;
    const int stage = flags & BF_OUT_MASK;
    if (stage != BF_OUT_RF && stage != BF_OUT_ENV && stage != BF_OUT_LOGDB)
        return fail(BF_EINVAL, "unknown output stage bits");
    if (n_samples < 2 || n_samples > 4096)
        return fail(BF_EINVAL, "bf_fkmig handles 2 <= n_samples <= 4096 (got %d)", n_samples);
    if (n_angles < 1 || n_angles > 256)
        return fail(BF_EINVAL, "n_angles must be in [1, 256], got %d", n_angles);
    for (int a = 0; a < n_angles; ++a)
        if (!std::isfinite(angles_rad[a]) || std::fabs(angles_rad[a]) >= 1.5707963267948966)
            return fail(BF_EINVAL, "angle %d (%g rad) outside (-pi/2, pi/2)", a, angles_rad[a]);
    const int ne = h->g.ne;
    if (ne < 2 || ne > 2048)
        return fail(BF_EINVAL, "bf_fkmig needs 2 to 2048 elements (got %d)", ne);
    const double pitch = (h->g.xe[ne - 1] - h->g.xe[0]) / (double)(ne - 1);
    for (int i = 0; i < ne; ++i)
        if (std::fabs(h->g.xe[i] - (h->g.xe[0] + i * pitch)) > 1e-9 * std::fabs(pitch) * ne)
            return fail(BF_EINVAL, "bf_fkmig needs equally spaced elements");
    cudaSetDevice(h->device);
    if (!is_device_pointer(rf_dev) || !is_device_pointer(out_dev))
        return fail(BF_EINVAL, "bf_fkmig needs device pointers");
    int nt = 1, lgt = 0, nk = 1, lgk = 0;
    while (nt < 2 * n_samples) {
        nt <<= 1;
        ++lgt;
    }
    while (nk < 2 * ne) {
        nk <<= 1;
        ++lgk;
    }
    const double c = h->g.c, fs = h->g.fs, dz = c / (2.0 * fs);
    // The mapping tables (geometry only): rebuilt when the sample count, the
    // angles or the mapping change.
    const int half = nt / 2;
    const size_t npts = (size_t)half * nk;
    std::vector<double> key{(double)n_samples, stolt ? 1.0 : 0.0};
    key.insert(key.end(), angles_rad, angles_rad + n_angles);
    const bool rebuild = key != h->fk_key;
    const bool regs = nt >= 32 && nk >= 32;  // both axes by the register transforms
    std::shared_ptr<FftTablesDev> tt, tk;
    int rc = fft_tables(regs ? 0 : nt, tt);
    if (!rc && !regs)
        rc = fft_tables(nk, tk);
    const size_t nf = (size_t)nt / 2 + 1, img = (size_t)ne * n_samples;
    if (!rc)
        rc = h->fk_D.ensure((regs ? fk_angles(n_angles, nt, nk) * nf + (size_t)n_angles * fk_pitch(nt)
                                  : n_angles * nf) *
                            nk * sizeof(float2));
    if (!rc)
        rc = h->fk_spec.ensure((size_t)(nt / 2) * nk * sizeof(float2));
    if (!rc && stage == BF_OUT_LOGDB)
        rc = h->fk_img.ensure(img * sizeof(float));
    if (!rc)
        rc = h->fk_max.ensure(sizeof(unsigned));
    if (!rc && rebuild) {
        // the previous call's kernels may still read the tables that are replaced
        h->fk_key.clear();
        cudaError_t ce = cudaStreamSynchronize(h->stream);
        rc = ce == cudaSuccess ? BF_OK : cuda_fail(ce, "cudaStreamSynchronize");
    }
    if (!rc && rebuild)
        rc = h->fk_beta.ensure((size_t)n_angles * ne * (regs ? 2 : 1) * sizeof(float));
    if (!rc && rebuild)
        rc = h->fk_i0.ensure((size_t)n_angles * npts * sizeof(int));
    if (!rc && rebuild)
        rc = h->fk_aw.ensure((size_t)n_angles * npts * sizeof(float2));
    if (rc)
        return rc;
    if (rebuild) {
        std::vector<float> beta;
        std::vector<double> sc((size_t)2 * n_angles);
        for (int a = 0; a < n_angles; ++a) {
            sc[2 * a] = std::sin(angles_rad[a]);
            sc[2 * a + 1] = std::cos(angles_rad[a]);
            for (int i = 0; i < ne; ++i) {
                const double x = ((double)i - 0.5 * (double)(ne - 1)) * pitch;
                const double turns = x * sc[2 * a] / ((double)nt * dz);  // half turns per bin
                beta.push_back((float)(regs ? turns : kPi * turns));
                if (regs)
                    beta.push_back((float)(turns - (double)beta.back()));
            }
        }
        std::vector<int> i0;
        std::vector<float> aw;
        fk_mapping_tables(nt, nk, pitch, dz, sc, stolt, regs ? lgk : 0, i0, aw);
        cudaError_t ce = cudaMemcpy(h->fk_i0.p, i0.data(), i0.size() * sizeof(int),
                                    cudaMemcpyHostToDevice);
        if (ce == cudaSuccess)
            ce = cudaMemcpy(h->fk_aw.p, aw.data(), aw.size() * sizeof(float), cudaMemcpyHostToDevice);
        if (ce == cudaSuccess)
            ce = cudaMemcpy(h->fk_beta.p, beta.data(), beta.size() * sizeof(float),
                            cudaMemcpyHostToDevice);
        if (ce != cudaSuccess)
            return cuda_fail(ce, "bf_fkmig mapping tables");
        h->fk_key = key;
    }
    h->call.clear();  // the device tables above may have moved
    cudaStream_t st = h->stream;
    FkJob J{};
    J.rf = rf_dev;
    J.D = (float2 *)h->fk_D.p;
    J.spec = (float2 *)h->fk_spec.p;
    J.img = stage == BF_OUT_LOGDB ? (float *)h->fk_img.p : out_dev;
    J.maxbits = stage == BF_OUT_LOGDB ? (unsigned *)h->fk_max.p : nullptr;
    J.beta = (const float *)h->fk_beta.p;
    J.map_i0 = (const int *)h->fk_i0.p;
    J.map_aw = (const float2 *)h->fk_aw.p;
    if (regs) {
        J.ptw = (const float2 *)tt->tw.p;
        J.E = J.D + (size_t)fk_angles(n_angles, nt, nk) * nf * nk;
    } else {
        J.tw_t = (const float2 *)tt->tw.p;
        J.tw_k = (const float2 *)tk->tw.p;
    }
    J.na = n_angles;
    J.ne = ne;
    J.ns = n_samples;
    J.nt = nt;
    J.lgt = lgt;
    J.nk = nk;
    J.lgk = lgk;
    cudaError_t e = regs ? launch_fkmig16(J, st) : launch_fkmig(J, st);
    if (e != cudaSuccess)
        return cuda_fail(e, "f-k migration launch");
    if (stage == BF_OUT_LOGDB) {
        // the log stage of the beamformer, one job over the native image
        LogJob l{};
        l.env = J.img;
        l.out = out_dev;
        l.maxbits = J.maxbits;
        l.n = (int)img;
        l.vec4 = (img % 4 == 0 && ((uintptr_t)l.env & 15) == 0 && ((uintptr_t)l.out & 15) == 0) ? 1 : 0;
        e = launch_log_one(l, 70.0f, st);
        if (e != cudaSuccess)
            return cuda_fail(e, "log launch");
    }
    return BF_OK;
}

BF_API int bf_beamform_plain(bf_handle *h, const int16_t *rf_dev, int32_t n_samples,
                             const double *angles_rad, int32_t n_angles, uint32_t flags,
                             float *out_dev)
{
    if (!h)
        return fail(BF_EINVAL, "null handle");
    if (!rf_dev || !out_dev)
        return fail(BF_EINVAL, "null data pointer");
    if (flags & BF_PREC_MASK)
        return fail(BF_EINVAL, "the plain kernel computes from int16 records in FP32 only");
    if (flags & BF_IQ_MASK)
        return fail(BF_EINVAL, "the plain kernel computes the RF combiners only");
    cudaSetDevice(h->device);
    if (!is_device_pointer(rf_dev) || !is_device_pointer(out_dev))
        return fail(BF_EINVAL, "bf_beamform_plain needs device pointers");
    h->call.clear();  // the plain path reuses the handle's scratch
    std::vector<FramePrep> frames(1);
    int rc = prepare_frame(h, rf_dev, n_samples, angles_rad, n_angles, flags, out_dev, h->scratch,
                           frames[0]);
    if (rc)
        return rc;
    HostLaunch hl;
    rc = build_launch(frames, hl);
    if (rc)
        return rc;
    const BfJob &job = hl.jobs[0];
    cudaError_t e = launch_plain(job, rf_dev, (const short2 *)frames[0].plan->at->valid.p,
                                 (const float *)h->dx2.p, pad_cols(h->g.nx), n_samples, h->stream);
    if (e != cudaSuccess)
        return cuda_fail(e, "plain kernel launch");
    if (frames[0].stage == BF_OUT_RF)
        return BF_OK;
    // envelope / log stages as in bf_beamform
    hl.jobs.clear();
    hl.groups.clear();
    hl.igroups.clear();
    rc = h->launch.upload(hl, h->stream, true);
    if (!rc && !h->err_cleared) {
        cudaMemsetAsync(h->launch.err.p, 0, sizeof(int), h->stream);
        h->err_cleared = true;
    }
    if (!rc)
        rc = cudaMemsetAsync(frames[0].maxbits, 0, 4 * sizeof(unsigned), h->stream) == cudaSuccess
                 ? BF_OK
                 : fail(BF_ECUDA, "cudaMemsetAsync");
    if (!rc) {
        e = launch_envelopes(hl, h->launch, h->stream);
        if (e != cudaSuccess)
            rc = cuda_fail(e, "envelope launch");
    }
    if (!rc && !hl.log.empty()) {
        e = launch_log(h->launch.log, h->launch.blk_prefix,
                       (int)hl.log.size(), hl.log_blocks, 70.0f, h->stream);
        if (e != cudaSuccess)
            rc = cuda_fail(e, "log launch");
    }
    return rc;
}

BF_API int bf_sync(bf_handle *h)
{
    if (!h)
        return fail(BF_EINVAL, "null handle");
    cudaSetDevice(h->device);
    cudaError_t e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaStreamSynchronize");
    if (!h->launch.err.p)
        return BF_OK;
    return read_device_error(h->launch, h->stream);
}

// Host-only view of the decision tables (no CUDA involved): first / last
// counted row per (angle, column, channel) and aperture counts per pixel.
BF_API int bf_host_tables(const bf_geometry *geom, const bf_grid *grid, double fs_hz, double f0_hz,
                          double c_mps, int32_t n_samples, const double *angles_rad,
                          int32_t n_angles, int32_t *valid_rows, uint16_t *aperture_count)
{
    if (!geom || !grid || !angles_rad || n_angles < 1 || n_samples < 2)
        return fail(BF_EINVAL, "bad arguments");
    GeomHost g;
    g.ne = geom->n_elements;
    if (g.ne < 1 || grid->nx < 1 || grid->nz < 1 || !(geom->f_number > 0.0))
        return fail(BF_EINVAL, "bad geometry");
    g.xe.resize(g.ne);
    for (int i = 0; i < g.ne; ++i)
        g.xe[i] = geom->x_elem_m ? geom->x_elem_m[i]
                                 : ((double)i - 0.5 * (double)(g.ne - 1)) * geom->pitch_m;
    g.fnum = geom->f_number;
    g.nx = grid->nx;
    g.nz = grid->nz;
    g.x0 = grid->x0_m;
    g.x1 = grid->x1_m;
    g.z0 = grid->z0_m;
    g.z1 = grid->z1_m;
    g.fs = fs_hz;
    g.f0 = f0_hz;
    g.c = c_mps;
    GeometryHost geo;
    geometry_tables(g, geo);
    PlanHost<int> ph;
    angle_tables(g, geo, n_samples, std::vector<double>(angles_rad, angles_rad + n_angles),
                 ph);
    const int nxp = pad_cols(g.nx);
    if (valid_rows)  // [na][ne][nxp][2] -> [na][nx][ne][2]
        for (int a = 0; a < n_angles; ++a)
            for (int ix = 0; ix < g.nx; ++ix)
                for (int i = 0; i < g.ne; ++i)
                    for (int q = 0; q < 2; ++q)
                        valid_rows[(((size_t)a * g.nx + ix) * g.ne + i) * 2 + q] =
                            ph.valid[(((size_t)a * g.ne + i) * nxp + ix) * 2 + q];
    if (aperture_count)
        std::memcpy(aperture_count, geo.apcnt.data(), geo.apcnt.size() * sizeof(uint16_t));
    return BF_OK;
}

// Plan introspection: tile shape and window sizes of the plan a frame with
// these arguments uses (built if needed), and optionally its window table.
BF_API int bf_plan_info(bf_handle *h, int32_t n_samples, const double *angles_rad,
                        int32_t n_angles, uint32_t flags, int32_t *info8, int32_t *wtab,
                        size_t wtab_entries)
{
    int rc = check_frame_args(h, n_samples, angles_rad, n_angles, flags);
    if (rc)
        return rc;
    if (!info8)
        return fail(BF_EINVAL, "null info");
    cudaSetDevice(h->device);
    Plan *p = nullptr;
    rc = handle_plan(h, n_samples, angles_rad, n_angles, flags, &p);
    if (rc)
        return rc;
    const size_t n = (size_t)n_angles * p->tiles_x * p->tiles_z * h->g.ne;
    const int32_t v[8] = {p->wmax, p->box, p->group, p->rows, p->tiles_x, p->tiles_z, p->nsp,
                          (int32_t)n};
    std::memcpy(info8, v, sizeof v);
    if (wtab) {
        if (wtab_entries < n)
            return fail(BF_EINVAL, "window table needs %zu entries", n);
        cudaError_t e = cudaMemcpy(wtab, p->wtab.p, n * sizeof(int32_t), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess)
            return cuda_fail(e, "cudaMemcpy (window table)");
    }
    return BF_OK;
}

// Autotuner: times the beamforming launches of `frames` copies of this
// workload under every tile configuration (synthetic zero records: the work
// does not depend on the data) and keeps the fastest for the handle's later
// work on it.  A lone frame, and frames whose combiners share no job, are also
// timed on the solo tiles; what is fastest then serves the handle's lone frames.
BF_API int bf_autotune(bf_handle *h, int32_t n_samples, const double *angles_rad,
                       int32_t n_angles, uint32_t flags, int32_t frames, int32_t *rows_out,
                       int32_t *stage_bytes_out, float *candidate_us, int32_t n_candidates)
{
    int rc = check_frame_args(h, n_samples, angles_rad, n_angles, flags);
    if (rc)
        return rc;
    if (frames < 1 || frames > 256)
        return fail(BF_EINVAL, "frames must be in [1, 256], got %d", frames);
    cudaSetDevice(h->device);
    const uint32_t fl = flags & ~(uint32_t)BF_OUT_MASK;  // beamformed output only
    const size_t rf_bytes = (size_t)n_angles * h->g.ne * n_samples * sizeof(int16_t);
    const size_t out_bytes = frame_out_bytes(h, fl);
    DevMem rf, out;
    rc = rf.ensure(rf_bytes);
    if (!rc)
        rc = out.ensure(out_bytes * frames);
    if (rc)
        return rc;
    cudaStream_t st;
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaStreamCreate");
    cudaEvent_t marks[4] = {};
    for (auto &m : marks)
        if (e == cudaSuccess)
            e = cudaEventCreate(&m);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(rf.p, 0, rf_bytes, st);
    std::vector<FrameScratch> scratch(frames);
    const bool lone = frame_prec(flags) != kPrecIQ && (frames == 1 || !sharing_modes(flags));
    std::vector<float> best_us(kNumConfigs, -1.f);
    int best = -1, best_lone = -1;  // of the tile configurations; of these and the solo ones
    for (int c = 0; c < (lone ? kNumConfigs : kNumTileConfigs) && e == cudaSuccess && !rc; ++c) {
        std::vector<FramePrep> fr(frames);
        int prc = BF_OK;
        for (int i = 0; i < frames && !prc; ++i)
            prc = prepare_frame(h, (const int16_t *)rf.p, n_samples, angles_rad, n_angles, fl,
                                (float *)out.p + (size_t)i * (out_bytes / sizeof(float)),
                                scratch[i], fr[i], kMaxFramesPerJob, PlanWish{c});
        if (prc)
            continue;  // this configuration does not fit the workload
        HostLaunch hl;
        DeviceLaunch dl;
        rc = build_launch(fr, hl);
        if (!rc)
            rc = dl.upload(hl, st, false);
        if (!rc && cudaMemsetAsync(dl.err.p, 0, sizeof(int), st) != cudaSuccess)
            rc = fail(BF_ECUDA, "cudaMemsetAsync");
        std::vector<float> t;
        for (int rep = 0; rep < 4 && !rc; ++rep) {  // one warm-up, three timed
            rc = enqueue(fr, hl, dl, st, marks);
            if (!rc && cudaStreamSynchronize(st) != cudaSuccess)
                rc = fail(BF_ECUDA, "autotune replay");
            float ms = 0.f;
            if (!rc && cudaEventElapsedTime(&ms, marks[1], marks[2]) == cudaSuccess && rep > 0)
                t.push_back(ms * 1e3f);
        }
        if (!rc)
            rc = read_device_error(dl, st);
        if (rc || t.empty())
            break;
        std::sort(t.begin(), t.end());
        best_us[c] = t[t.size() / 2];
        if (c < kNumTileConfigs && (best < 0 || best_us[c] < best_us[best]))
            best = c;
        if (best_lone < 0 || best_us[c] < best_us[best_lone])
            best_lone = c;
    }
    for (auto &m : marks)
        if (m)
            cudaEventDestroy(m);
    cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    if (rc)
        return rc;
    if (e != cudaSuccess)
        return cuda_fail(e, "autotune setup");
    if (best < 0)
        return fail(BF_EINVAL, "no tile configuration fits this workload");
    {
        std::lock_guard<std::mutex> lk(h->mu);
        PlanKey key{n_samples, frame_prec(flags),
                    std::vector<double>(angles_rad, angles_rad + n_angles), 0};
        h->tuned[key] = best;
        key.cfg = 1;  // see tuned_cfg
        if (lone)
            h->tuned[key] = best_lone;
    }
    h->call.clear();  // bf_beamform's last call may have used another configuration
    if (rows_out)
        *rows_out = kTileConfigs[best].rows;
    if (stage_bytes_out)
        *stage_bytes_out = kTileConfigs[best].stage_bytes;
    if (candidate_us)
        for (int c = 0; c < std::min<int>(n_candidates, kNumTileConfigs); ++c)
            candidate_us[c] = best_us[c];
    return BF_OK;
}

// ------------------------------------------------------------------ batch --

// What frames of a batch have in common that can share a beamforming job (see shareable).
using JobKey = std::tuple<const bf_handle *, int, uint32_t, std::vector<double>>;
static JobKey job_key(const bf_frame &f)
{
    return JobKey(f.h, f.n_samples, f.mode_and_flags & (BF_MODE_MASK | BF_IQ_MASK | BF_PREC_MASK),
                  std::vector<double>(f.angles_rad, f.angles_rad + f.n_angles));
}

BF_API int bf_batch_create(const bf_frame *frames, int32_t n, bf_batch **out)
{
    if (!frames || !out || n < 1)
        return fail(BF_EINVAL, "bad batch arguments");
    *out = nullptr;
    auto b = std::make_unique<bf_batch>();
    b->scratch.resize(n);
    b->frames.resize(n);
    // frames of the batch with the same plan and combiners; every frame's arguments are
    // checked before its angles are read
    std::map<JobKey, std::pair<int, int>> peers;  // (frames, of these prepared)
    int dev = -1;
    for (int i = 0; i < n; ++i) {
        const bf_frame &f = frames[i];
        if (!f.h || !f.rf_dev || !f.out_dev)
            return fail(BF_EINVAL, "frame %d: null handle or data pointer", i);
        if (dev < 0)
            dev = f.h->device;
        else if (dev != f.h->device)
            return fail(BF_EINVAL, "frame %d: all frames of a batch must use one device", i);
        cudaSetDevice(dev);
        if (!is_device_pointer(f.rf_dev) || !is_device_pointer(f.out_dev))
            return fail(BF_EINVAL, "frame %d: batches need device pointers", i);
        int rc = check_frame_args(f.h, f.n_samples, f.angles_rad, f.n_angles, f.mode_and_flags);
        if (rc)
            return fail(rc, "frame %d: %s", i, g_err.c_str());
        peers[job_key(f)].first += 1;
    }
    for (int i = 0; i < n; ++i) {
        const bf_frame &f = frames[i];
        auto &p = peers[job_key(f)];
        const int same = p.first, index = p.second++;
        int rc = prepare_frame(f.h, f.rf_dev, f.n_samples, f.angles_rad, f.n_angles,
                               f.mode_and_flags, f.out_dev, b->scratch[i], b->frames[i],
                               same > 1 ? kMaxFramesPerJob : 1, PlanWish{-1, same, false, index});
        if (rc)
            return fail(rc, "frame %d: %s", i, g_err.c_str());
    }
    b->device = dev;
    int rc = build_launch(b->frames, b->hl);
    if (!rc)
        rc = b->dl.upload(b->hl, nullptr, false);
    if (rc)
        return rc;
    cudaMemset(b->dl.err.p, 0, sizeof(int));
    // Capture the batch's launches once; bf_batch_launch replays the graph.
    // The stage marks sit on a side branch of the graph (MarkBranch).
    cudaStream_t cap;
    cudaError_t e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaStreamCreate");
    MarkBranch br;
    e = cudaStreamCreateWithFlags(&br.side, cudaStreamNonBlocking);
    for (auto &f : br.fork)
        if (e == cudaSuccess)
            e = cudaEventCreateWithFlags(&f, cudaEventDisableTiming);
    if (e == cudaSuccess)
        e = cudaEventCreateWithFlags(&br.join, cudaEventDisableTiming);
    if (e == cudaSuccess)
        e = cudaEventCreateWithFlags(&br.work_fork, cudaEventDisableTiming);
    for (int w = 0; w < MarkBranch::kWork && e == cudaSuccess; ++w) {
        e = cudaStreamCreateWithFlags(&br.work[w], cudaStreamNonBlocking);
        if (e == cudaSuccess)
            e = cudaEventCreateWithFlags(&br.work_join[w], cudaEventDisableTiming);
    }
    for (auto &m : b->marks)
        if (e == cudaSuccess)
            e = cudaEventCreate(&m);
    b->launches = (int)b->hl.igroups.size() + (b->hl.demod[0].empty() ? 0 : 1) +
                  (b->hl.demod[1].empty() ? 0 : 1) + (b->hl.demod[2].empty() ? 0 : 1) +
                  (int)b->hl.groups.size() + (b->hl.env[0].empty() ? 0 : 1) +
                  (b->hl.env[1].empty() ? 0 : 1) + (b->hl.envw.empty() ? 0 : 1) +
                  (b->hl.log.empty() ? 0 : 1);
    if (e == cudaSuccess)
        e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        rc = enqueue(b->frames, b->hl, b->dl, cap, b->marks, &br);
        cudaGraph_t g = nullptr;
        cudaError_t e2 = cudaStreamEndCapture(cap, &g);
        if (!rc && e2 == cudaSuccess) {
            e2 = cudaGraphInstantiate(&b->exec, g, 0);
            if (e2 != cudaSuccess)
                rc = cuda_fail(e2, "cudaGraphInstantiate");
        } else if (!rc) {
            rc = cuda_fail(e2, "cudaStreamEndCapture");
        }
        if (g)
            cudaGraphDestroy(g);
    } else {
        rc = cuda_fail(e, "cudaStreamBeginCapture");
    }
    cudaStreamDestroy(cap);
    for (auto &f : br.fork)
        if (f)
            cudaEventDestroy(f);
    if (br.join)
        cudaEventDestroy(br.join);
    if (br.work_fork)
        cudaEventDestroy(br.work_fork);
    for (int w = 0; w < MarkBranch::kWork; ++w) {
        if (br.work_join[w])
            cudaEventDestroy(br.work_join[w]);
        if (br.work[w])
            cudaStreamDestroy(br.work[w]);
    }
    if (br.side)
        cudaStreamDestroy(br.side);
    if (rc)
        return rc;
    *out = b.release();
    return BF_OK;
}

BF_API int bf_batch_launch(bf_batch *b, void *stream)
{
    if (!b)
        return fail(BF_EINVAL, "null batch");
    cudaSetDevice(b->device);
    cudaError_t e = cudaGraphLaunch(b->exec, (cudaStream_t)stream);
    return e == cudaSuccess ? BF_OK : cuda_fail(e, "cudaGraphLaunch");
}

BF_API int bf_batch_status(bf_batch *b, void *stream)
{
    if (!b)
        return fail(BF_EINVAL, "null batch");
    cudaSetDevice(b->device);
    return read_device_error(b->dl, (cudaStream_t)stream);
}

BF_API int bf_batch_timing(bf_batch *b, float *ms3, int32_t *kernel_launches)
{
    if (!b || !ms3)
        return fail(BF_EINVAL, "null argument");
    cudaSetDevice(b->device);
    for (int k = 0; k < 3; ++k) {
        cudaError_t e = cudaEventElapsedTime(&ms3[k], b->marks[k], b->marks[k + 1]);
        if (e != cudaSuccess)
            return cuda_fail(e, "cudaEventElapsedTime");
    }
    if (kernel_launches)
        *kernel_launches = b->launches;
    return BF_OK;
}

BF_API int bf_batch_destroy(bf_batch *b)
{
    if (!b)
        return fail(BF_EINVAL, "null batch");
    cudaSetDevice(b->device);
    cudaDeviceSynchronize();
    if (b->exec)
        cudaGraphExecDestroy(b->exec);
    for (auto &m : b->marks)
        if (m)
            cudaEventDestroy(m);
    delete b;
    return BF_OK;
}

}  // extern "C"
