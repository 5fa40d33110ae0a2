// Host-side structures of the beamformer library (handles, plans, scratch,
// launch descriptions, serving engine).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <condition_variable>
#include <cstddef>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/bf.h"
#include "bf_internal.h"
#include "bf_tables.h"

namespace bfi {

int fail(int code, const char *fmt, ...);
int cuda_fail(cudaError_t e, const char *what);

// Owning device allocation (freed on destruction).
// Host-side fault injection for tests of the error paths: true when the
// environment variable BF_FAULT, a comma-separated list, names `kind`.
// Kinds: alloc (device allocations fail with BF_ENOMEM), submit (admission
// refuses every request with BF_EAGAIN), copy (a request's RF copy fails
// with BF_ECUDA).  Read on every use, so a test can switch it on and off.
bool fault_injected(const char *kind);

struct DevMem {
    void *p = nullptr;
    size_t bytes = 0;
    DevMem() = default;
    DevMem(const DevMem &) = delete;
    DevMem &operator=(const DevMem &) = delete;
    DevMem(DevMem &&o) noexcept : p(o.p), bytes(o.bytes)
    {
        o.p = nullptr;
        o.bytes = 0;
    }
    DevMem &operator=(DevMem &&o) noexcept
    {
        if (this != &o) {
            release();
            p = o.p;
            bytes = o.bytes;
            o.p = nullptr;
            o.bytes = 0;
        }
        return *this;
    }
    ~DevMem() { release(); }
    int ensure(size_t n);  // grow to at least n bytes (contents not kept)
    int reserve(size_t n); // as ensure, growing by half again at least (lists that vary in size)
    void release();
    int upload(const void *src, size_t n);  // synchronous host -> device
};

struct PlanKey {
    int ns, prec;
    std::vector<double> angles;
    int cfg = 0;  // index into kTileConfigs, or kSoloConfig + log2 of the split
    bool operator<(const PlanKey &o) const
    {
        if (ns != o.ns)
            return ns < o.ns;
        if (prec != o.prec)
            return prec < o.prec;
        if (cfg != o.cfg)
            return cfg < o.cfg;
        return angles < o.angles;
    }
};

// Device tables of one (handle, sample count, angle set), shared by its plans: the
// transmit tables and the counted-row intervals.
struct AngleTablesDev {
    DevMem colK, colF, rowK, rowF, valid;
};

// Tiling of one (handle, sample count, precision, angle set): the tables above, the
// per-tile window starts and the tensor maps through which the beamformer stages
// its per-tile tables.
struct Plan {
    std::shared_ptr<AngleTablesDev> at;
    int ns = 0, na = 0, prec = 0;
    int wmax = 0, box = 0, group = 1, nsp = 0, rows = 8, tiles_x = 0, tiles_z = 0;
    // solo plans (split > 0): warps per row pair, angles per stage, groups of them,
    // channels per window copy
    int split = 0, ang = 1, ang_groups = 1;
    int run = 1;
    DevMem wtab, btab;
    DevMem maps;  // CUtensorMap[2]: valid rows, dx^2
};

// Device copies of transform tables: exp(-2 pi i k / n), and the spectral
// factors of one depth (and band).
struct FftTablesDev {
    DevMem tw;
};
struct EnvTablesDev {
    int lg = 0, conv = 0;
    DevMem gr, gh;
};

// Device scratch of one in-flight frame: staged sample pairs, beamformed
// image, envelope and frame maxima.
struct FrameScratch {
    // as the lead of a multi-frame job: pairs holds the job's frames interleaved
    // ([row][pair][frame])
    DevMem pairs, y, env, maxbits;
    // the tensor map over the pairs encoded last, and what it was encoded for
    CUtensorMap map{};
    const void *map_base = nullptr;
    int map_key[7] = {};  // rows, nsp, box, run, prec, frames, set
};

struct FramePrep {
    bf_handle *h = nullptr;
    Plan *plan = nullptr;
    Plan *solo = nullptr;  // the plan to use if the launch has no partner for the frame, or null
    std::shared_ptr<EnvTablesDev> et[2];  // envelope tables: without band, the DMAS band
    std::shared_ptr<FftTablesDev> ft;     // level twiddles, or the warp kernel's 512-point table
    std::shared_ptr<FftTablesDev> dt;     // demodulation twiddles (IQ only)
    const int16_t *rf = nullptr;
    int ns = 0, na = 0, modes = 0, stage = 0, prec = 0;
    double pdas_p = 2.0;
    float *out = nullptr;
    void *pairs = nullptr;
    float *y = nullptr, *env = nullptr;
    unsigned *maxbits = nullptr;
    FrameScratch *scratch = nullptr;
    int nf_cap = 1;  // frames of a job this frame may lead: its pairs buffer holds that many
};

struct HostLaunch {
    struct Group {  // one beamforming launch (split > 0: solo jobs)
        int prec, variant, rows, nf, split, ang, first, count, prefix_first, tiles;
        size_t smem;
    };
    struct IGroup {  // one ingest launch
        int prec, first, count, prefix_first, blocks;
        bool wide;  // several units per thread
    };
    std::vector<BfJob> jobs;        // rf_map: index into maps until the upload
    std::vector<CUtensorMap> maps;  // over the jobs' sample pairs
    std::vector<int> tile_prefix;
    std::vector<Group> groups;
    size_t smem = 0;
    std::vector<IngestJob> ingest;
    std::vector<int> ingest_prefix;
    std::vector<IGroup> igroups;
    // envelopes of the other depths: [0] transforms of up to 4096 points, [1] of 8192
    std::vector<EnvJob> env[2];
    std::vector<int> env_prefix[2];
    int env_blocks[2] = {0, 0};
    // 512-row images: the warp-per-column-pair envelope kernel (column pairs)
    std::vector<EnvJob> envw;
    std::vector<int> envw_prefix;
    int envw_pairs = 0;
    std::vector<LogJob> log;
    std::vector<int> blk_prefix;
    int log_blocks = 0;
    // IQ frames, records to analytic-signal pairs: [0] 32 to 4096 samples, [1] 8192, [2]
    // fewer than 32
    std::vector<DemodJob> demod[3];
    std::vector<int> demod_prefix[3];
    int demod_blocks[3] = {0, 0, 0};
};

// Device copy of a launch description: every list in one allocation, sent in one
// transfer (each transfer costs the stream a few microseconds before its kernels).
struct DeviceLaunch {
    DevMem pack, err;
    const BfJob *jobs = nullptr;
    const IngestJob *ingest = nullptr;
    const EnvJob *env[2] = {nullptr, nullptr}, *envw = nullptr;
    const LogJob *log = nullptr;
    const DemodJob *demod[3] = {nullptr, nullptr, nullptr};
    const int *tile_prefix = nullptr, *ingest_prefix = nullptr, *env_prefix[2] = {nullptr, nullptr},
              *envw_prefix = nullptr, *blk_prefix = nullptr,
              *demod_prefix[3] = {nullptr, nullptr, nullptr};
    int upload(const HostLaunch &hl, cudaStream_t st, bool async);
};

struct Request;

// The last bf_beamform call of a handle, kept so that the same call again
// (same arguments, order p, stream and BF_TILE_ROWS) skips the host-side
// preparation and, from its second repetition on, replays one CUDA graph.
struct CallCache {
    bool valid = false;
    int forced = -1;  // BF_TILE_ROWS's configuration
    uint32_t flags = 0;
    const int16_t *rf = nullptr;
    float *out = nullptr;
    int ns = 0;
    std::vector<double> angles;
    double pdas_p = 0;
    cudaStream_t stream = nullptr;
    int hits = 0;
    std::vector<FramePrep> frames;
    HostLaunch hl;
    cudaGraphExec_t exec = nullptr;
    void clear()
    {
        if (exec)
            cudaGraphExecDestroy(exec);
        exec = nullptr;
        valid = false;
        hits = 0;
        frames.clear();
        hl = HostLaunch{};
    }
};

}  // namespace bfi

struct bf_handle {
    int device = 0, sms = 1;
    bfi::GeomHost g;
    bfi::GeometryHost geo;
    cudaStream_t stream = nullptr, own_stream = nullptr;
    bfi::DevMem rowZ, dx2, apcnt;
    int kb_lo = 1, kb_hi = 0;
    double pdas_p = 2.0;  // order of the pDAS combiner
    std::mutex mu;  // plans, tickets, slot pool
    std::map<bfi::PlanKey, std::unique_ptr<bfi::Plan>> plans;
    // their angle tables (key prec = cfg = 0)
    std::map<bfi::PlanKey, std::shared_ptr<bfi::AngleTablesDev>> angle_tabs;
    // configurations bf_autotune chose (key cfg = 0; for lone frames 1)
    std::map<bfi::PlanKey, int> tuned;
    bfi::FrameScratch scratch;     // bf_beamform
    bfi::DeviceLaunch launch;      // bf_beamform
    bfi::CallCache call;           // bf_beamform's last call
    bfi::DevMem fk_D, fk_spec, fk_img, fk_beta, fk_max;  // bf_fkmig scratch
    bfi::DevMem fk_i0, fk_aw;     // bf_fkmig mapping tables, for fk_key
    std::vector<double> fk_key;   // (n_samples, Stolt?, angles...) of the tables
    bool err_cleared = false;
    std::map<uint64_t, std::shared_ptr<bfi::Request>> tickets;
};

struct bf_batch {
    int device = 0;
    std::vector<bfi::FrameScratch> scratch;
    std::vector<bfi::FramePrep> frames;
    bfi::HostLaunch hl;
    bfi::DeviceLaunch dl;
    cudaGraphExec_t exec = nullptr;
    cudaEvent_t marks[4] = {nullptr, nullptr, nullptr, nullptr};
    int launches = 0;  // kernels one replay launches
};

namespace bfi {

// What is known about a frame's launch when its plan is chosen.
struct PlanWish {
    int cfg = -1;   // a configuration of kTileConfigs, or < 0: by the rules of choose_cfg
    int peers = 1;  // frames of this plan and combiners submitted together (see bf_choice.h)
    bool alone = false;  // the frame shares its plan with no other: RF frames take solo tiles
    int index = -1;  // the frame's place among its peers, in a launch of just these (or < 0)
    int room = 0;    // frames its pairs buffer holds at most (0: by pairs_room)
};
// Plan of a frame with these arguments (`flags`: its mode and precision bits).
// BF_TILE_ROWS and bf_autotune's choice for the workload come before the rules; a
// two-row configuration serves DAS / DMAS of RF records and IQ-DAS / BB-DMAS only
// (an explicit one is refused for other frames, a tuned one replaced by the default).
int handle_plan(bf_handle *h, int ns, const double *angles, int na, uint32_t flags, Plan **out,
                const PlanWish &wish = {});
// Whether frames with these combiners ever share a job.
inline bool sharing_modes(uint32_t flags)
{
    return (flags & BF_MODE_MASK & ~(uint32_t)(BF_DAS | BF_DMAS)) == 0;
}
int check_frame_args(bf_handle *h, int ns, const double *angles, int na, uint32_t flags);
size_t frame_out_bytes(const bf_handle *h, uint32_t flags);
// Storage code of a frame's staged records (kPrecIQ for the IQ combiners).
int frame_prec(uint32_t flags);
// nf_cap: frames of one plan a later build_launch may put in one job with
// this frame (1: alone, as a single bf_beamform call); the frame's scratch
// is sized for the multi-frame jobs its plan and combiners allow up to that, or for what
// its place among its peers asks for (PlanWish).
// With nf_cap 1, or combiners no job shares, the plan is a solo plan where one
// applies; late_solo: also find that plan for a frame that may turn out alone
// (use_solo_plans).
int prepare_frame(bf_handle *h, const int16_t *rf_dev, int ns, const double *angles, int na,
                  uint32_t flags, float *out_dev, FrameScratch &s, FramePrep &fp, int nf_cap = 1,
                  PlanWish wish = {}, bool late_solo = false);
// Frames of a launch that share no job with another one go over to their solo plans.
void use_solo_plans(std::vector<FramePrep> &frames);
// Frames (at most cap) of one plan that can share a beamforming job with a
// frame of these flags (1 unless the combiners are DAS / DMAS of RF records
// or IQ-DAS / BB-DMAS; IQ frames with records above 4096 samples alone).
int job_frames_cap(const Plan *p, uint32_t flags, int cap);
int build_launch(const std::vector<FramePrep> &frames, HostLaunch &hl);
// Stage marks of a captured graph on a side branch: mark k is recorded on the
// side stream after it joins the capture behind stage k (fork[k] recorded on
// the capture stream), so each mark node depends on the work it closes and no
// kernel depends on a mark: the kernels keep direct edges.  Mark 0 is a root
// beside the first launch.  join brings the side branch back into the
// capture's origin stream at the end.
struct MarkBranch {
    cudaStream_t side = nullptr;
    cudaEvent_t fork[4] = {nullptr, nullptr, nullptr, nullptr};
    cudaEvent_t join = nullptr;
    // further beamforming launches run beside the first (their CTAs fill the SMs as its
    // last ones leave): streams to capture them on, forked after the ingest
    static constexpr int kWork = 3;
    cudaStream_t work[kWork] = {nullptr, nullptr, nullptr};
    cudaEvent_t work_fork = nullptr, work_join[kWork] = {nullptr, nullptr, nullptr};
};
// marks (optional, 4 events): recorded before the ingest, before and after the
// beamforming launches, and after the last launch; in line on st, or (branch,
// inside a capture of st) on the branch's side stream.
int enqueue(const std::vector<FramePrep> &frames, const HostLaunch &hl, DeviceLaunch &dl,
            cudaStream_t st, cudaEvent_t *marks = nullptr, const MarkBranch *branch = nullptr);
int read_device_error(DeviceLaunch &dl, cudaStream_t st);
bool is_device_pointer(const void *p);
void engine_forget(bf_handle *h);

}  // namespace bfi
