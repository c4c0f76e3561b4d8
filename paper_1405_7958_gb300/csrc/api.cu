// C-ABI entry points of the segmentation library (declared in rt.h):
// argument validation, the context and its device workspace, and the
// launch sequence of every operation and of the segmentation chain.
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "ccl.cuh"
#include "common.cuh"
#include "contract.cuh"
#include "edt.cuh"
#include "features.cuh"
#include "mlp.cuh"
#include "objects.cuh"
#include "recon.cuh"
#include "runs.cuh"
#include "synth.cuh"

using namespace rtk;

struct PhaseRec {
    int phase;
    cudaEvent_t a, b;
};

struct rt_ctx {
    int device = 0;
    int num_sms = 0;
    void *ws = nullptr;       // device workspace
    size_t ws_bytes = 0;
    bool ws_captured = false;   // a captured call has used ws
    std::vector<void *> kept;   // earlier workspaces that captured calls have used
    uint32_t *visits_dev = nullptr;  // [visits, iterations] of the last reconstruction (workspace)
    int64_t launches = 0;     // kernels launched
    bool timing = false;
    const uint16_t *picker_wb = nullptr;   // attached picker (caller-owned device memory)
    const float *picker_norm = nullptr;
    int32_t *picks_host = nullptr;         // pinned, mapped: picker classes of the last learned chunk
    int32_t *picks_mapped = nullptr;       // the same memory as the device sees it
    cudaEvent_t picks_ev = nullptr;        // recorded after their copy (not under stream capture)
    bool picks_ev_valid = false;
    cudaStream_t side = nullptr;           // the picker's stream where its picks change no schedule
    cudaEvent_t fork = nullptr, join = nullptr;   // order it behind the call's start and before its end
    int n_last_picks = 0;
    PickTable classes{{0, 0, 0, 0}, {4, 12, 24, 12}};   // picker classes (rt_set_picker_classes); entry 3 per call
    int max_iters = 0;                     // limits of the single-operation entry points (rt_set_limits)
    uint64_t timeout_ns = 0;
    int64_t fq_cap = 0;                    // entries per global frontier queue (0: one per padded pixel)
    std::vector<PhaseRec> recs;
    std::vector<cudaEvent_t> pool;
};

namespace {

cudaEvent_t take_event(rt_ctx *ctx)
{
    if (!ctx->pool.empty()) {
        cudaEvent_t e = ctx->pool.back();
        ctx->pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}

// Brackets one phase with events on the stream when timing is enabled.
class Phase {
  public:
    Phase(rt_ctx *ctx, int phase, cudaStream_t s) : ctx_(ctx), s_(s)
    {
        if (!ctx->timing) return;
        rec_.phase = phase;
        rec_.a = take_event(ctx);
        rec_.b = take_event(ctx);
        cudaEventRecord(rec_.a, s);
    }
    ~Phase()
    {
        if (!ctx_->timing || !rec_.a) return;
        cudaEventRecord(rec_.b, s_);
        ctx_->recs.push_back(rec_);
    }

  private:
    rt_ctx *ctx_;
    cudaStream_t s_;
    PhaseRec rec_{0, nullptr, nullptr};
};

// Default bound on one propagation (20 s). The barriers of the other
// cooperative kernels wait this long too, whatever the caller's bound on a
// propagation: they have no partial result to stop at.
constexpr uint64_t kSweepTimeoutNs = 20000000000ull;

// Bump allocator over the context workspace (256-byte aligned pieces).
struct Carve {
    size_t off = 0;
    char *base = nullptr;
    template <class T>
    T *take(size_t count)
    {
        off = (size_t)round_up((int64_t)off, 256);
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += count * sizeof(T);
        return p;
    }
};

class DeviceGuard {
  public:
    explicit DeviceGuard(int dev)
    {
        cudaGetDevice(&prev_);
        if (prev_ != dev) cudaSetDevice(dev);
        dev_ = dev;
    }
    ~DeviceGuard()
    {
        if (prev_ != dev_) cudaSetDevice(prev_);
    }

  private:
    int prev_ = 0, dev_ = 0;
};

// Whether work on s is being captured into a graph.
bool capturing(cudaStream_t s)
{
    cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &c) != cudaSuccess) cudaGetLastError();
    return c == cudaStreamCaptureStatusActive;
}

// A workspace of at least `bytes` for a call on s. A block that a graph may
// hold (ws_captured) is not freed when the workspace grows but kept for the
// graph until the context goes; the next block is then twice as large if it
// can be, so that the kept ones are never more than the current one. Under
// capture the allocation itself stays outside the graph (relaxed capture
// mode): operations have come to need more than a context was reserved with
// for them, and a call that fitted must not end its capture.
rt_status ensure_ws(rt_ctx *ctx, size_t bytes, cudaStream_t s)
{
    const bool cap = capturing(s);
    if (bytes > ctx->ws_bytes) {
        size_t want = (size_t)round_up((int64_t)bytes, 1 << 20);
        const size_t exact = want;
        const bool keep = ctx->ws && (cap || ctx->ws_captured);
        if (keep) {
            try {
                ctx->kept.reserve(ctx->kept.size() + 1);
            } catch (const std::bad_alloc &) {
                return RT_ENOMEM;
            }
            if (want < 2 * ctx->ws_bytes) want = 2 * ctx->ws_bytes;
        } else if (ctx->ws) {
            cudaFree(ctx->ws);
            ctx->ws = nullptr;
            ctx->ws_bytes = 0;
        }
        ctx->visits_dev = nullptr;
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        if (cap) cudaThreadExchangeStreamCaptureMode(&mode);
        void *ws = nullptr;
        while (cudaMalloc(&ws, want) != cudaSuccess) {
            cudaGetLastError();
            ws = nullptr;
            if (want == exact) break;
            want = exact;
        }
        if (cap) cudaThreadExchangeStreamCaptureMode(&mode);
        if (!ws) return RT_ENOMEM;
        if (keep) ctx->kept.push_back(ctx->ws);
        ctx->ws = ws;
        ctx->ws_bytes = want;
        ctx->ws_captured = false;
    }
    ctx->ws_captured |= cap;
    return RT_OK;
}

bool bad_dims(int H, int W) { return H < 1 || W < 1 || H > kMaxSide || W > kMaxSide; }

bool overlaps(const void *a, size_t na, const void *b, size_t nb)
{
    const char *pa = (const char *)a, *pb = (const char *)b;
    return pa < pb + nb && pb < pa + na;
}

// Releases the context's events, side stream and pinned buffer.
void free_host_side(rt_ctx *c)
{
    if (c->side) cudaStreamDestroy(c->side);
    for (cudaEvent_t e : {c->picks_ev, c->fork, c->join})
        if (e) cudaEventDestroy(e);
    if (c->picks_host) cudaFreeHost(c->picks_host);
}

size_t span(int H, int64_t ld, size_t elem, int W) { return ((size_t)(H - 1) * ld + W) * elem; }

rt_status cuda_status(cudaError_t e)
{
    if (e == cudaSuccess) return RT_OK;
    cudaGetLastError();
    return RT_ECUDA;
}

// Zeroes n words of device memory. The chain clears its control words with
// this kernel rather than cudaMemsetAsync, so that nothing in it can wait
// behind the caller's copies on a copy engine.
__global__ void zero_words_kernel(uint32_t *p, int n)
{
    start_early();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = 0u;
}
cudaError_t zero_words(void *p, int n, cudaStream_t s)
{
    launch_early(zero_words_kernel, (n + 255) / 256 < 16 ? (n + 255) / 256 : 16, 256, 0, s, static_cast<uint32_t *>(p), n);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- recon
struct ReconWs {
    uint32_t *flags;   // per tile
    uint32_t *ctl;     // kCtlWords control words (recon.cuh)
    int32_t *err;
    int32_t *map;      // kGroups x ntiles tile lists when the variant is chosen per image
    uint32_t *fq[2];   // RT_FRONTIER: global frontier queues (fq_cap entries each), or null
    uint32_t *fctl;    //              their kFqCtlWords control words
    uint32_t fq_cap;
};

// Whether a call runs RT_FRONTIER somewhere: as its variant, or as one of
// the picker's classes under the learned policy (ctx NULL: the default
// classes, all RT_RASTER).
bool uses_frontier(const rt_ctx *ctx, int variant, bool learned)
{
    if (variant == RT_FRONTIER) return true;
    if (!learned || !ctx) return false;
    for (int c = 0; c < kPickClasses; ++c)
        if (ctx->classes.group[c] == RT_FRONTIER - RT_RASTER) return true;
    return false;
}

// Entries of each global frontier queue for batch b: the context's setting,
// else one per padded pixel of the batch.
uint32_t frontier_capacity(const rt_ctx *ctx, const ReconBatch &b)
{
    int64_t px = 0;
    for (int i = 0; i < b.n; ++i) px += (int64_t)b.img[i].Hp * b.img[i].Wp;
    const int64_t cap = ctx && ctx->fq_cap > 0 ? ctx->fq_cap : px;
    return (uint32_t)(cap < 0xffffffffLL ? cap : 0xffffffffLL);
}

// Reserve the sweep control block and per-image padded buffers (and the
// global frontier queues when fq_cap > 0).
void carve_recon(Carve &cv, ReconBatch &b, ReconWs &w, bool grouped = false, uint32_t fq_cap = 0)
{
    w.flags = cv.take<uint32_t>((size_t)b.ntiles);
    w.ctl = cv.take<uint32_t>(kCtlWords);
    w.err = cv.take<int32_t>(1);
    w.map = grouped ? cv.take<int32_t>((size_t)kGroups * b.ntiles) : nullptr;
    w.fq_cap = fq_cap;
    w.fq[0] = fq_cap ? cv.take<uint32_t>(fq_cap) : nullptr;
    w.fq[1] = fq_cap ? cv.take<uint32_t>(fq_cap) : nullptr;
    w.fctl = fq_cap ? cv.take<uint32_t>(kFqCtlWords) : nullptr;
    for (int i = 0; i < b.n; ++i) {
        ReconImage &d = b.img[i];
        d.Rw = cv.take<uint8_t>((size_t)d.Hp * d.Wp);
        d.Iw = cv.take<uint8_t>((size_t)d.Hp * d.Wp);
        d.Cw = cv.take<uint8_t>((size_t)d.tiles_x * d.tiles_y * kEdgeBytes);
    }
}

// Enqueue init + propagation for a batch whose buffers are carved. `err`
// receives the device status. With `pick` (device, one picker class per
// image) every image propagates with its own variant: one launch per variant
// group over the group's tile list, with no host round trip.
// Bounds of a propagation: max_iters > 0 allows max_iters tile visits per
// 32 x 64 tile on average; timeout_ns bounds its device time.
struct Limits {
    int max_iters;
    uint64_t timeout_ns;
    int strip = 0;   // tiles per warp strip of the raster propagation (0: the library's choice)
};

Limits ctx_limits(const rt_ctx *ctx) { return {ctx->max_iters, ctx->timeout_ns ? ctx->timeout_ns : kSweepTimeoutNs}; }

Limits seg_limits(const rt_ctx *ctx, const rt_seg_params &P)
{
    Limits lim = ctx ? ctx_limits(ctx) : Limits{0, kSweepTimeoutNs};
    if (P.max_iters > 0) lim.max_iters = P.max_iters;
    if (P.timeout_ms > 0) lim.timeout_ns = (uint64_t)P.timeout_ms * 1000000ull;
    lim.strip = P.strip_tiles;
    return lim;
}

int default_max_local(int variant) { return variant == RT_HYBRID || variant == RT_FRONTIER ? 64 : 12; }

// sweep budget of every raster tile in a launch shared by several tiles
int shared_raster_budget(int max_local) { return max_local > 0 ? max_local : default_max_local(RT_RASTER); }

// Whether every class of the picker propagates by RT_RASTER.
bool raster_classes(const rt_ctx *ctx)
{
    for (int c = 0; ctx && c < kPickClasses; ++c)
        if (ctx->classes.group[c] != 0) return false;
    return true;
}

// In a launch shared by several tiles every raster class runs at the plain
// budget, so when the plain schedule and every class of the picker are
// raster, no pick can change a tile's schedule and the picker is not run.
bool picks_matter(const rt_ctx *ctx, const rt_seg_params &P, int n_tiles)
{
    if (n_tiles == 1) return true;
    if (P.variant != RT_AUTO && P.variant != RT_RASTER) return true;
    return !raster_classes(ctx);
}

rt_status run_recon(rt_ctx *ctx, ReconBatch &b, ReconWs &w, int conn, int variant, int max_local, int32_t *err,
                    cudaStream_t s, Limits lim, const int32_t *pick = nullptr)
{
    if (variant == RT_AUTO) variant = RT_RASTER;
    // the learned policy's schedules: the picker's classes, then the call's
    // plain schedule as the fall-back entry
    PickTable table = ctx->classes;
    table.group[kPickClasses] = variant - RT_RASTER;
    table.max_local[kPickClasses] = max_local > 0 ? max_local : default_max_local(variant);
    // A frontier entry names its tile in 21 bits, and the queues need their
    // workspace: without either, frontier schedules run as RT_HYBRID (the
    // same dense first pass, then per-tile queues; same output).
    const bool fq_ok = w.fq_cap > 0 && b.ntiles < kFqMaxTiles;
    for (int e = 0; e < kPickEntries; ++e)
        if (table.group[e] == RT_FRONTIER - RT_RASTER && !fq_ok) table.group[e] = RT_HYBRID - RT_RASTER;
    if (variant == RT_FRONTIER && !fq_ok) variant = RT_HYBRID;
    // The picker learned its budgets on lone tiles, where a tile's latency
    // sets the time and short visits can win. Tiles that share a launch with
    // others are bound by its throughput instead: there a budget below the
    // plain one only adds visits, and one above it adds visits too once
    // revisits start at the moved side of the halo (measured on uneven and
    // 4K batches). Raster classes run at the plain budget in shared launches.
    if (pick && b.n > 1)
        for (int c = 0; c < kPickClasses; ++c)
            if (table.group[c] == 0) table.max_local[c] = shared_raster_budget(max_local);
    // RT_RASTER / RT_QUEUE: every tile starts flagged for a dense visit (the
    // queue visit then seeds every pixel); RT_HYBRID / RT_FRONTIER: nothing
    // flagged, the dense pass over all tiles flags what remains.
    const uint32_t flag0 = variant == RT_HYBRID || variant == RT_FRONTIER ? 0u : 2u;
    RT_CUDA_TRY(zero_words(w.ctl, kCtlWords, s));
    ctx->launches += 1;
    {
        Phase ph(ctx, RT_PHASE_RECON_INIT, s);
        RT_CUDA_TRY(launch_recon_init(b, w.flags, w.ctl, flag0, pick, table, w.map, err, s));
        ctx->launches += 1;
    }
    ctx->visits_dev = w.ctl + kCtlVisits;
    SweepParams p;
    p.b = b;
    p.ntiles = b.ntiles;
    p.flags = w.flags;
    p.pending = w.ctl + kCtlPending;
    p.err = err;
    p.visits = w.ctl + kCtlVisits;
    p.timeout_ns = lim.timeout_ns;
    p.seg_max = lim.strip;
    const int64_t bound = (int64_t)lim.max_iters * b.ntiles;
    p.max_visits = lim.max_iters > 0 ? (uint32_t)(bound < 0xffffffffLL ? bound : 0xffffffffLL) : 0u;
    p.spent = w.ctl + kCtlSpent;
    p.abort = w.ctl + kCtlAbort;
    p.map = nullptr;
    p.nvirt = nullptr;
    p.pick = pick;
    p.table = table;
    p.fq[0] = w.fq[0];
    p.fq[1] = w.fq[1];
    p.fq_cap = w.fq_cap;
    p.fctl = w.fctl;
    int grid = 0;
    Phase ph(ctx, RT_PHASE_RECON_SWEEP, s);
    bool used[kGroups] = {false, false, false, false};   // groups some schedule of the table propagates in
    for (int e = 0; e < kPickEntries; ++e)
        if (table.group[e] >= 0 && table.group[e] < kGroups) used[table.group[e]] = true;
    for (int g = 0; g < (pick ? kGroups : 1); ++g) {
        if (pick && !used[g]) continue;
        const int v = pick ? RT_RASTER + g : variant;
        if (pick) {
            p.map = w.map + (size_t)g * b.ntiles;
            p.nvirt = w.ctl + kCtlGroupCount + g;
            p.pending = w.ctl + kCtlGroupPending + g;
        }
        p.max_local = max_local > 0 ? max_local : default_max_local(v);
        if (v == RT_HYBRID || v == RT_FRONTIER) {
            RT_CUDA_TRY(launch_recon_dense(p, conn, s));
            ctx->launches += 1;
        }
        if (v == RT_FRONTIER) {
            // seed and drain the global frontier queues; the directional
            // sweeps that follow find nothing flagged unless a queue
            // overflowed
            RT_CUDA_TRY(zero_words(w.fctl, kFqCtlWords, s));
            ctx->launches += 1;
            RT_CUDA_TRY(launch_recon_seed(p, conn, s));
            RT_CUDA_TRY(launch_recon_frontier(p, conn, ctx->num_sms, s, &grid));
            ctx->launches += 2;
            p.max_local = max_local > 0 ? max_local : default_max_local(RT_RASTER);
        }
        ctx->launches += 1;
        RT_CUDA_TRY(launch_recon_persistent(p, conn, v == RT_RASTER || v == RT_FRONTIER ? 0 : 1, ctx->num_sms, s,
                                            &grid));
    }
    return RT_OK;
}

// ------------------------------------------------------------ contraction
// RT_AUTO with 8-connectivity runs the reconstruction by contraction, unless
// the call sets something that only the propagation has: a bound on its tile
// visits or its device time, a visit budget, a strip length.
bool use_contraction(int conn, int variant, int max_local, int strip, const Limits &lim)
{
    return conn == 8 && variant == RT_AUTO && max_local == 0 && strip == 0 && lim.max_iters == 0 &&
           lim.timeout_ns == kSweepTimeoutNs;
}

void carve_contract(Carve &cv, CtBatch &b)
{
    const size_t nt = (size_t)b.ntiles;
    b.ctl = cv.take<uint32_t>(kCtCtlWords);
    b.plane = cv.take<uint16_t>(nt * kCtPx);
    b.cnt = cv.take<uint32_t>(nt);
    b.S = cv.take<uint32_t>(nt * kCtNodes);
    b.link = cv.take<unsigned long long>(nt * kCtNodes);
    b.best = cv.take<unsigned long long>(nt * kCtNodes);
    b.act = cv.take<uint32_t>(nt * kCtNodes);
    b.edge = cv.take<unsigned long long>(nt * kCtUnits * kCtUnitEdges);
    b.ecnt = cv.take<uint8_t>(nt * kCtUnits);
    b.rim = cv.take<uint16_t>(nt * 4 * kCtSide);
}

// Enqueue the contraction of a carved batch; launch_contract_out writes R.
rt_status run_contract(rt_ctx *ctx, CtBatch &b, int32_t *err, cudaStream_t s, const Limits &lim)
{
    b.err = err;
    ctx->visits_dev = nullptr;   // no tile visits
    RT_CUDA_TRY(zero_words(b.ctl, kCtCtlWords, s));
    Phase ph(ctx, RT_PHASE_RECON_SWEEP, s);
    RT_CUDA_TRY(launch_contract(b, ctx->num_sms, lim.timeout_ns, s));
    ctx->launches += 4;
    return RT_OK;
}

// Enqueue what a call that does not return R needs of it.
rt_status run_reach(rt_ctx *ctx, const RunBatch &b, cudaStream_t s)
{
    ctx->visits_dev = nullptr;   // no tile visits
    Phase ph(ctx, RT_PHASE_RECON_SWEEP, s);
    ctx->launches += 3;
    RT_CUDA_TRY(launch_run_reach(b, s));
    return RT_OK;
}

// Workspace of the hole filling and labeling stages: the bits first, then
// what no stage before them uses (carve_runs_late).
void carve_bits(Carve &cv, RunBatch &b) { b.bits = cv.take<unsigned long long>((size_t)b.ntiles * kRunSide); }
void carve_runs_late(Carve &cv, RunBatch &b, bool fill, bool label)
{
    const size_t nt = (size_t)b.ntiles, nodes = 1 + nt * kRunSlots;
    b.sides = cv.take<uint8_t>(nt * kRunSides);
    b.cnt = cv.take<uint8_t>(nt);
    b.lcnt = cv.take<uint8_t>(nt);
    b.kept = nullptr;
    b.outside = fill ? cv.take<uint32_t>(nodes) : nullptr;
    b.U = label ? cv.take<uint32_t>(nodes) : nullptr;
    b.A = label ? cv.take<uint32_t>(nodes) : nullptr;
    b.M = label ? cv.take<uint32_t>(nodes) : nullptr;
    b.words = cv.take<uint32_t>(nt * kRunWords);
}

void add_image(ReconBatch &b, const uint8_t *marker, int64_t ld_marker, const uint8_t *mask, int64_t ld_mask,
               int H, int W, int h_offset)
{
    ReconImage &d = b.img[b.n];
    std::memset(&d, 0, sizeof(d));
    d.marker = marker;
    d.ld_marker = ld_marker;
    d.mask = mask;
    d.ld_mask = ld_mask;
    d.h_offset = h_offset;
    plan_recon_image(d, H, W);
    d.tile_base = b.ntiles;
    b.ntiles += d.tiles_x * d.tiles_y;
    const int64_t words = (int64_t)d.Hp * d.Wp / 4;
    if (words > b.max_words) b.max_words = words;
    b.n++;
}

// the tiles' status words: the device status of the chunk that carried them
struct StatusOut {
    int32_t *dst[kMaxImgs];
};
__global__ void copy_status_kernel(const int32_t *src, StatusOut o, int n)
{
    start_early();
    if ((int)threadIdx.x < n && o.dst[threadIdx.x]) *o.dst[threadIdx.x] = *src;
}

// the picker's classes of a chunk into the caller-visible pinned buffer
// src NULL: every tile ran the plain schedule (class kPickClasses)
__global__ void copy_picks_kernel(const int32_t *src, int32_t *dst, int n)
{
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src ? src[i] : kPickClasses;
    __threadfence_system();
}

bool bad_params(const rt_seg_params &P)
{
    if (P.conn_recon != 4 && P.conn_recon != 8) return true;
    if (P.conn_fill != 4 && P.conn_fill != 8) return true;
    if (P.h_offset < 0 || P.h_offset > 255 || P.threshold < 0 || P.threshold > 256) return true;
    if (P.variant < RT_AUTO || P.variant > RT_FRONTIER) return true;
    if (P.policy != RT_POLICY_PLAIN && P.policy != RT_POLICY_LEARNED) return true;
    if (P.max_local < 0 || P.max_iters < 0 || P.timeout_ms < 0) return true;
    if (P.strip_tiles < 0 || P.strip_tiles > 32) return true;
    if (P.pick_min_prob < 0 || P.pick_min_prob > 1000) return true;
    return false;
}

bool bad_tile(const rt_tile &t)
{
    if (!t.img || !t.labels || !t.d2 || bad_dims(t.H, t.W)) return true;
    if (t.ld_img < t.W || t.ld_labels < t.W || t.ld_d2 < t.W) return true;
    if (t.recon && t.ld_recon < t.W) return true;
    if (t.filled && t.ld_filled < t.W) return true;
    return false;
}

// Whether an output of the chain lies over its image.
bool in_place(const rt_tile &t)
{
    const size_t n = span(t.H, t.ld_img, 1, t.W);
    return (t.recon && overlaps(t.img, n, t.recon, span(t.H, t.ld_recon, 1, t.W))) ||
           (t.filled && overlaps(t.img, n, t.filled, span(t.H, t.ld_filled, 1, t.W))) ||
           overlaps(t.img, n, t.labels, span(t.H, t.ld_labels, 4, t.W)) ||
           overlaps(t.img, n, t.d2, span(t.H, t.ld_d2, 4, t.W));
}

// Starts an EDT batch: takes its control words with the status word before
// them (`words` in all, to be cleared), for images of `bands` bands of rows.
int32_t *take_edt_ctl(Carve &cv, EdtBitsBatch &b, size_t bands, int &words)
{
    b.n = b.ntiles = b.nbands = b.maxW = 0;
    words = (int)(6 + 2 * bands);
    uint32_t *w = cv.take<uint32_t>((size_t)words);
    b.err = reinterpret_cast<int32_t *>(w);
    b.far_any = w ? w + 1 : nullptr;
    b.has_bg = w ? w + 2 : nullptr;
    b.bar = w ? w + 4 : nullptr;
    b.far_rows = reinterpret_cast<unsigned long long *>(w ? w + 6 : nullptr);
    return b.err;
}

// Workspace of one chunk (up to kMaxImgs tiles) of rt_segment_batch. Every
// stage runs once for the whole chunk, so every tile has its own buffers:
// the reconstruction's, the foreground bits, the component slots, the
// kept-pixel bit plane and the distance transform's column masks.
constexpr size_t kWsBytesPerPx = 13;
struct Chunk {
    bool contract = false;   // reconstruction by contraction (cb), else by propagation (b, w)
    bool reach = false;      // with contract: no tile asks for R, so only where it is below the threshold is found
    CtBatch cb;
    ReconBatch b;
    ReconWs w;
    int32_t *err = nullptr;   // first of the ctl_words words that a call clears
    int ctl_words = 0;
    FeatBatch fb;
    float *feat = nullptr;
    int32_t *picks = nullptr;
    RunBatch rb;
    EdtBitsBatch eb;
};

// Lays chunk [c0, c0 + cn) out in cv. With cv.base == nullptr only the size
// is measured (cv.off); no pointer is formed.
void layout_chunk(Carve &cv, Chunk &c, const rt_tile *tiles, int c0, int cn, const rt_seg_params &P, bool learned,
                  const rt_ctx *ctx, const Limits &lim, bool may_contract = true)
{
    const bool real = cv.base != nullptr;
    size_t bands = 0;
    for (int i = 0; i < cn; ++i) bands += (size_t)ceil_div(tiles[c0 + i].H, kEdtSide);
    c.err = take_edt_ctl(cv, c.eb, bands, c.ctl_words);
    c.cb.n = c.cb.ntiles = 0;
    for (int i = 0; i < cn; ++i) {
        const rt_tile &t = tiles[c0 + i];
        ct_plan_image(c.cb, nullptr, 0, t.img, t.ld_img, t.H, t.W, P.h_offset);
    }
    c.contract = may_contract && use_contraction(P.conn_recon, P.variant, P.max_local, P.strip_tiles, lim) &&
                 c.cb.ntiles < kCtMaxTiles && (!learned || raster_classes(ctx));
    if (!c.contract) {
        std::memset(&c.b, 0, sizeof(c.b));
        for (int i = 0; i < cn; ++i) {
            const rt_tile &t = tiles[c0 + i];
            add_image(c.b, nullptr, 0, t.img, t.ld_img, t.H, t.W, P.h_offset);
        }
        carve_recon(cv, c.b, c.w, learned,
                    uses_frontier(ctx, P.variant, learned) ? frontier_capacity(ctx, c.b) : 0u);
    }
    if (learned) {
        c.fb.n = cn;
        for (int i = 0; i < cn; ++i) {
            const rt_tile &t = tiles[c0 + i];
            const size_t nb = (size_t)((t.H + 7) / 8) * ((t.W + 7) / 8);
            FeatImage &d = c.fb.img[i];
            d.img = t.img;
            d.ld = t.ld_img;
            d.H = t.H;
            d.W = t.W;
            d.hist = cv.take<uint32_t>(256);
            d.acc = cv.take<unsigned long long>(4);
            d.dark = cv.take<uint8_t>(nb);
            d.bmax = cv.take<uint8_t>(nb);
        }
        c.feat = cv.take<float>((size_t)cn * kNumFeatures);
        c.picks = cv.take<int32_t>((size_t)cn);
    }
    c.rb.n = c.rb.ntiles = 0;
    c.rb.amin = P.min_area;
    c.rb.amax = P.max_area;
    size_t px = 0;
    for (int i = 0; i < cn; ++i) {
        const rt_tile &t = tiles[c0 + i];
        RunImage &u = run_add(c.rb, t.H, t.W);
        u.filled = t.filled;
        u.ld_filled = t.ld_filled;
        u.labels = t.labels;
        u.ld_lab = t.ld_labels;
        u.n_kept = t.n_kept;
        px += (size_t)t.H * t.W;
        if (c.contract) {   // B = (R < threshold) goes straight to the bits
            c.cb.img[i].out = t.recon;
            c.cb.img[i].ld_out = t.ld_recon;
            u.in = t.img;
            u.ld_in = t.ld_img;
        } else {
            uint8_t *B = cv.take<uint8_t>((size_t)t.H * t.W);
            ReconImage &d = c.b.img[i];
            d.out = t.recon;
            d.ld_out = t.ld_recon;
            d.bin = B;
            d.ld_bin = t.W;
            u.in = B;
            u.ld_in = t.W;
        }
    }
    carve_bits(cv, c.rb);
    c.cb.bits = c.contract ? c.rb.bits : nullptr;
    // The contraction's arrays are dead once R and the bits are written; the
    // later stages reuse their memory.
    size_t contract_end = 0;
    if (c.contract) {
        const size_t off = cv.off;
        carve_contract(cv, c.cb);
        contract_end = cv.off;
        cv.off = off;
    }
    carve_runs_late(cv, c.rb, true, true);
    c.rb.kept = cv.take<unsigned long long>((size_t)c.rb.ntiles * kRunSide);
    c.eb.bits = c.rb.kept;
    // R(p) >= t exactly where a path from a pixel q with J(q) >= t leads to p through pixels with I >= t. The seeds lie
    // where the kept pixels will be.
    c.reach = c.contract && real;
    for (int i = 0; real && i < cn; ++i) c.reach = c.reach && !tiles[c0 + i].recon;
    c.rb.seeds = c.rb.kept;
    c.rb.lo = P.threshold;
    c.rb.hi = P.threshold > 0 ? P.threshold + P.h_offset : 0;
    for (int i = 0; i < cn; ++i) {
        const rt_tile &t = tiles[c0 + i];
        char *ews = cv.take<char>(edt_bits_workspace_bytes(t.H, t.W));
        if (real) edt_bits_add(c.eb, t.H, t.W, t.d2, t.ld_d2, ews);
    }
    if (cv.off < contract_end) cv.off = contract_end;
    // The figure callers size their budgets by has always been at least 13
    // bytes per pixel, with the frontier queues on top; it stays so.
    const size_t floor = kWsBytesPerPx * px + (c.contract || !c.w.fq_cap ? 0 : 8 * (size_t)c.w.fq_cap + 4 * kFqCtlWords);
    if (cv.off < floor) cv.off = floor;
}

// Workspace bytes rt_segment_batch needs for these tiles (the largest chunk).
size_t segment_ws_bytes(const rt_tile *tiles, int n, const rt_seg_params &P, bool learned, const rt_ctx *ctx)
{
    const Limits lim = seg_limits(ctx, P);
    size_t most = 0;
    for (int c0 = 0; c0 < n; c0 += kMaxImgs) {
        const int cn = n - c0 < kMaxImgs ? n - c0 : kMaxImgs;
        // A call that contracts fits where the same call with a bound on its
        // propagation fits: a reservation serves both.
        for (bool may_contract : {true, false}) {
            Carve cv;
            Chunk c;
            layout_chunk(cv, c, tiles, c0, cn, P, learned, ctx, lim, may_contract);
            most = cv.off > most ? cv.off : most;
            if (!c.contract) break;
        }
    }
    return most;
}

// The picker's features and network on a chunk, into its picks.
rt_status run_picker(rt_ctx *ctx, const Chunk &c, const rt_seg_params &P, cudaStream_t s)
{
    Phase ph(ctx, RT_PHASE_PICK, s);
    RT_CUDA_TRY(launch_features_pick(c.fb, c.feat, ctx->picker_wb, ctx->picker_norm, c.picks,
                                     (float)P.pick_min_prob / 1000.0f, kPickClasses, s));
    ctx->launches += 4;
    return RT_OK;
}

// The chunk's picks for rt_last_picks (NULL: every tile ran the plain
// schedule), written by a kernel into the mapped pinned buffer: a copy-engine
// transfer would queue behind the caller's read-backs on the same engine and
// hold up the rest of the chain.
rt_status report_picks(rt_ctx *ctx, const int32_t *picks, int cn, cudaStream_t s)
{
    copy_picks_kernel<<<1, 32, 0, s>>>(picks, ctx->picks_mapped, cn);
    RT_CUDA_TRY(cudaGetLastError());
    ctx->launches += 1;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusActive;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) cudaGetLastError();
    ctx->picks_ev_valid = cap == cudaStreamCaptureStatusNone;
    if (ctx->picks_ev_valid) RT_CUDA_TRY(cudaEventRecord(ctx->picks_ev, s));
    ctx->n_last_picks = cn;
    return RT_OK;
}

}  // namespace

// ================================================================= C ABI
extern "C" {

int rt_version(void) { return 201; }

const char *rt_status_str(int status)
{
    switch (status) {
    case RT_OK: return "RT_OK";
    case RT_EINVAL: return "RT_EINVAL: invalid argument";
    case RT_ENOMEM: return "RT_ENOMEM: device workspace allocation failed";
    case RT_ECUDA: return "RT_ECUDA: CUDA runtime error";
    case RT_ETIMEOUT: return "RT_ETIMEOUT: device iteration or wait bound reached";
    case RT_EMARKER: return "RT_EMARKER: marker above mask (clamped)";
    case RT_EQUEUE: return "RT_EQUEUE: frontier queue overflow";
    case RT_EUNAVAIL: return "RT_EUNAVAIL: variant or feature unavailable";
    case RT_ESIZE: return "RT_ESIZE: image larger than the fixed scratch of the allocation-free entry point";
    default: return "unknown rt_status";
    }
}

rt_status rt_create(rt_ctx **ctx, int device, size_t workspace_bytes)
{
    if (!ctx) return RT_EINVAL;
    *ctx = nullptr;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) {
        cudaGetLastError();
        return RT_ECUDA;
    }
    rt_ctx *c = new (std::nothrow) rt_ctx;
    if (!c) return RT_ENOMEM;
    c->device = device;
    DeviceGuard g(device);
    if (cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaHostAlloc((void **)&c->picks_host, kMaxImgs * sizeof(int32_t), cudaHostAllocMapped) != cudaSuccess ||
        cudaHostGetDevicePointer((void **)&c->picks_mapped, c->picks_host, 0) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->picks_ev, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        free_host_side(c);
        delete c;
        return RT_ECUDA;
    }
    if (workspace_bytes > 0) {
        const size_t want = (size_t)round_up((int64_t)workspace_bytes, 1 << 20);
        if (cudaMalloc(&c->ws, want) == cudaSuccess) c->ws_bytes = want;
    }
    if (c->ws_bytes < workspace_bytes) {
        cudaGetLastError();
        free_host_side(c);
        delete c;
        return RT_ENOMEM;
    }
    *ctx = c;
    return RT_OK;
}

rt_status rt_set_limits(rt_ctx *ctx, int max_iters, int timeout_ms)
{
    if (!ctx || max_iters < 0 || timeout_ms < 0) return RT_EINVAL;
    ctx->max_iters = max_iters;
    ctx->timeout_ns = (uint64_t)timeout_ms * 1000000ull;
    return RT_OK;
}

size_t rt_segment_workspace_bytes(const rt_ctx *ctx, const rt_tile *tiles, int n, const rt_seg_params *params)
{
    if ((!tiles && n > 0) || n < 0 || !params || bad_params(*params)) return 0;
    for (int i = 0; i < n; ++i)
        if (bad_tile(tiles[i])) return 0;
    return segment_ws_bytes(tiles, n, *params, params->policy == RT_POLICY_LEARNED, ctx);
}

rt_status rt_set_queue_capacity(rt_ctx *ctx, int64_t entries)
{
    if (!ctx || entries < 0 || entries > 0xffffffffLL) return RT_EINVAL;
    ctx->fq_cap = entries;
    return RT_OK;
}

void rt_destroy(rt_ctx *ctx)
{
    if (!ctx) return;
    DeviceGuard g(ctx->device);
    if (ctx->ws) {
        cudaDeviceSynchronize();
        for (void *p : ctx->kept) cudaFree(p);
        cudaFree(ctx->ws);
    }
    for (const PhaseRec &r : ctx->recs) {
        cudaEventDestroy(r.a);
        cudaEventDestroy(r.b);
    }
    for (cudaEvent_t e : ctx->pool) cudaEventDestroy(e);
    free_host_side(ctx);
    delete ctx;
}

size_t rt_workspace_bytes(const rt_ctx *ctx) { return ctx ? ctx->ws_bytes : 0; }

rt_status rt_timing_enable(rt_ctx *ctx, int enable)
{
    if (!ctx) return RT_EINVAL;
    ctx->timing = enable != 0;
    return RT_OK;
}

rt_status rt_timing_read(rt_ctx *ctx, double *ms, int64_t *count, int reset)
{
    if (!ctx) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    for (const PhaseRec &r : ctx->recs) {
        if (cudaEventSynchronize(r.b) != cudaSuccess) {
            cudaGetLastError();
            return RT_ECUDA;
        }
        float t = 0.f;
        if (cudaEventElapsedTime(&t, r.a, r.b) != cudaSuccess) {
            cudaGetLastError();
            return RT_ECUDA;
        }
        if (r.phase >= 0 && r.phase < RT_NPHASES) {
            if (ms) ms[r.phase] += t;
            if (count) count[r.phase] += 1;
        }
    }
    if (reset) {
        for (const PhaseRec &r : ctx->recs) {
            ctx->pool.push_back(r.a);
            ctx->pool.push_back(r.b);
        }
        ctx->recs.clear();
    }
    return RT_OK;
}

int64_t rt_kernel_launches(const rt_ctx *ctx) { return ctx ? ctx->launches : 0; }

rt_status rt_recon_stats(rt_ctx *ctx, int64_t *visits, int64_t *iterations, int64_t *pops)
{
    if (!ctx) return RT_EINVAL;
    uint32_t v[3] = {0, 0, 0};
    if (ctx->visits_dev) {
        DeviceGuard g(ctx->device);
        if (cudaMemcpy(v, ctx->visits_dev, sizeof(v), cudaMemcpyDeviceToHost) != cudaSuccess) {
            cudaGetLastError();
            return RT_ECUDA;
        }
    }
    if (visits) *visits = v[0];
    if (iterations) *iterations = v[1];
    if (pops) *pops = v[2];
    return RT_OK;
}

rt_status rt_marker(rt_ctx *ctx, const uint8_t *mask, int64_t ld_mask, uint8_t *marker, int64_t ld_marker, int H,
                    int W, int h_offset, void *stream)
{
    if (!ctx || !mask || !marker || bad_dims(H, W) || ld_mask < W || ld_marker < W || h_offset < 0 ||
        h_offset > 255)
        return RT_EINVAL;
    if (overlaps(mask, span(H, ld_mask, 1, W), marker, span(H, ld_marker, 1, W))) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    Phase ph(ctx, RT_PHASE_RECON_INIT, (cudaStream_t)stream);
    ctx->launches += 1;
    return cuda_status(launch_marker(mask, ld_mask, marker, ld_marker, H, W, h_offset, (cudaStream_t)stream));
}

rt_status rt_reconstruct(rt_ctx *ctx, const uint8_t *marker, int64_t ld_marker, const uint8_t *mask,
                         int64_t ld_mask, uint8_t *out, int64_t ld_out, int H, int W, int conn, int variant,
                         int h_offset, int32_t *dev_status, void *stream)
{
    if (!ctx || !mask || !out || bad_dims(H, W) || ld_mask < W || ld_out < W) return RT_EINVAL;
    if (conn != 4 && conn != 8) return RT_EINVAL;
    if (variant < RT_AUTO || variant > RT_FRONTIER) return RT_EINVAL;
    if (marker && ld_marker < W) return RT_EINVAL;
    if (!marker && (h_offset < 0 || h_offset > 255)) return RT_EINVAL;
    if (overlaps(out, span(H, ld_out, 1, W), mask, span(H, ld_mask, 1, W))) return RT_EINVAL;
    if (marker && marker != out && overlaps(out, span(H, ld_out, 1, W), marker, span(H, ld_marker, 1, W)))
        return RT_EINVAL;
    if (marker && marker == out && ld_marker != ld_out) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;

    const Limits lim = ctx_limits(ctx);
    if (use_contraction(conn, variant, 0, 0, lim)) {
        CtBatch cb;
        cb.n = cb.ntiles = 0;
        ct_plan_image(cb, marker, ld_marker, mask, ld_mask, H, W, h_offset);
        cb.img[0].out = out;
        cb.img[0].ld_out = ld_out;
        cb.bits = nullptr;
        int32_t *cerr = nullptr;
        rt_status cst = RT_OK;
        for (int pass = 0; pass < 2; ++pass) {   // size, then carve
            Carve cc;
            if (pass) cc.base = (char *)ctx->ws;
            cerr = cc.take<int32_t>(1);
            carve_contract(cc, cb);
            if (!pass && (cst = ensure_ws(ctx, cc.off, s)) != RT_OK) return cst;
        }
        if (dev_status) cerr = dev_status;
        RT_CUDA_TRY(cudaMemsetAsync(cerr, 0, sizeof(int32_t), s));
        cst = run_contract(ctx, cb, cerr, s, lim);
        if (cst != RT_OK) return cst;
        Phase ph(ctx, RT_PHASE_RECON_OUT, s);
        ctx->launches += 1;
        return cuda_status(launch_contract_out(cb, 0, s));
    }
    ReconBatch b;
    std::memset(&b, 0, sizeof(b));
    add_image(b, marker, ld_marker, mask, ld_mask, H, W, h_offset);
    const uint32_t fq_cap = variant == RT_FRONTIER ? frontier_capacity(ctx, b) : 0u;
    Carve cv;
    ReconWs w;
    carve_recon(cv, b, w, false, fq_cap);
    rt_status st = ensure_ws(ctx, cv.off, s);
    if (st != RT_OK) return st;
    cv = Carve();
    cv.base = (char *)ctx->ws;
    carve_recon(cv, b, w, false, fq_cap);

    int32_t *err = dev_status ? dev_status : w.err;
    RT_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int32_t), s));
    st = run_recon(ctx, b, w, conn, variant, 0, err, s, lim);
    if (st != RT_OK) return st;
    b.img[0].out = out;
    b.img[0].ld_out = ld_out;
    Phase ph(ctx, RT_PHASE_RECON_OUT, s);
    ctx->launches += 1;
    return cuda_status(launch_recon_out(b, 0, s));
}

rt_status rt_fill_holes(rt_ctx *ctx, const uint8_t *in, int64_t ld_in, uint8_t *out, int64_t ld_out, int H, int W,
                        int conn, int32_t *dev_status, void *stream)
{
    if (!ctx || !in || !out || bad_dims(H, W) || ld_in < W || ld_out < W) return RT_EINVAL;
    if (conn != 4 && conn != 8) return RT_EINVAL;
    if ((const void *)in != (const void *)out && overlaps(in, span(H, ld_in, 1, W), out, span(H, ld_out, 1, W)))
        return RT_EINVAL;
    if ((const void *)in == (const void *)out && ld_in != ld_out) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    RunBatch b;
    b.n = b.ntiles = 0;
    RunImage &u = run_add(b, H, W);
    u.in = in;
    u.ld_in = ld_in;
    u.filled = out;
    u.ld_filled = ld_out;
    for (bool real : {false, true}) {   // size, then carve
        Carve cv;
        if (real) cv.base = (char *)ctx->ws;
        carve_bits(cv, b);
        carve_runs_late(cv, b, true, false);
        rt_status st = RT_OK;
        if (!real && (st = ensure_ws(ctx, cv.off, s)) != RT_OK) return st;
    }
    if (dev_status) RT_CUDA_TRY(cudaMemsetAsync(dev_status, 0, sizeof(int32_t), s));
    Phase ph(ctx, RT_PHASE_FILL, s);
    ctx->launches += 4;
    RT_CUDA_TRY(launch_run_pack(b, s));
    return cuda_status(launch_run_fill(b, conn, 0, s));
}

rt_status rt_label_area(rt_ctx *ctx, const uint8_t *bin, int64_t ld_bin, int32_t *labels, int64_t ld_lab, int H,
                        int W, int conn, int32_t min_area, int32_t max_area, int32_t *dev_n_kept,
                        int32_t *dev_status, void *stream)
{
    if (!ctx || !bin || !labels || bad_dims(H, W) || ld_bin < W || ld_lab < W) return RT_EINVAL;
    if (conn != 4 && conn != 8) return RT_EINVAL;
    if (overlaps(bin, span(H, ld_bin, 1, W), labels, span(H, ld_lab, 4, W))) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    if ((int64_t)run_tiles(H, W) <= kUfMaxTiles) {
        rt_status st = ensure_ws(ctx, uf_workspace_bytes(H, W), s);
        if (st != RT_OK) return st;
        UfImage u;
        std::memset(&u, 0, sizeof(u));
        uf_carve(u, (char *)ctx->ws, H, W);
        u.in = bin;
        u.ld_in = ld_bin;
        u.labels = labels;
        u.ld_lab = ld_lab;
        u.n_kept = dev_n_kept;
        UfBatch b;
        b.n = 0;
        uf_add(b, u);
        b.amin = min_area;
        b.amax = max_area;
        if (dev_status) RT_CUDA_TRY(cudaMemsetAsync(dev_status, 0, sizeof(int32_t), s));
        Phase ph(ctx, RT_PHASE_LABEL, s);
        ctx->launches += 4;
        return cuda_status(launch_label_batch(b, conn, s));
    }
    RunBatch b;
    b.n = b.ntiles = 0;
    b.amin = min_area;
    b.amax = max_area;
    RunImage &u = run_add(b, H, W);
    u.in = bin;
    u.ld_in = ld_bin;
    u.labels = labels;
    u.ld_lab = ld_lab;
    u.n_kept = dev_n_kept;
    for (bool real : {false, true}) {   // size, then carve
        Carve cv;
        if (real) cv.base = (char *)ctx->ws;
        carve_bits(cv, b);
        carve_runs_late(cv, b, false, true);
        rt_status st = RT_OK;
        if (!real && (st = ensure_ws(ctx, cv.off, s)) != RT_OK) return st;
    }
    if (dev_status) RT_CUDA_TRY(cudaMemsetAsync(dev_status, 0, sizeof(int32_t), s));
    Phase ph(ctx, RT_PHASE_LABEL, s);
    ctx->launches += 5;
    RT_CUDA_TRY(launch_run_pack(b, s));
    RT_CUDA_TRY(launch_run_local(b, conn, s));
    return cuda_status(launch_run_label(b, conn, s));
}

rt_status rt_edt(rt_ctx *ctx, const uint8_t *fg, int64_t ld_fg, int32_t *d2, int64_t ld_d2, int H, int W,
                 int32_t *dev_status, void *stream)
{
    if (!ctx || !fg || !d2 || bad_dims(H, W) || ld_fg < W || ld_d2 < W) return RT_EINVAL;
    if (overlaps(fg, span(H, ld_fg, 1, W), d2, span(H, ld_d2, 4, W))) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    RunBatch r;
    r.n = r.ntiles = 0;
    RunImage &u = run_add(r, H, W);
    u.in = fg;
    u.ld_in = ld_fg;
    EdtBitsBatch b;
    int words = 0;
    for (bool real : {false, true}) {   // size, then carve
        Carve cv;
        if (real) cv.base = (char *)ctx->ws;
        take_edt_ctl(cv, b, (size_t)ceil_div(H, kEdtSide), words);
        carve_bits(cv, r);
        char *ews = cv.take<char>(edt_bits_workspace_bytes(H, W));
        rt_status st = RT_OK;
        if (!real && (st = ensure_ws(ctx, cv.off, s)) != RT_OK) return st;
        if (real) edt_bits_add(b, H, W, d2, ld_d2, ews);
    }
    b.bits = r.bits;
    RT_CUDA_TRY(cudaMemsetAsync(b.err, 0, (size_t)words * 4, s));
    if (dev_status) {
        RT_CUDA_TRY(cudaMemsetAsync(dev_status, 0, sizeof(int32_t), s));
        b.err = dev_status;
    }
    Phase ph(ctx, RT_PHASE_EDT, s);
    ctx->launches += 3;
    RT_CUDA_TRY(launch_run_pack(r, s));
    return cuda_status(launch_edt_bits_batch(b, ctx->num_sms, kSweepTimeoutNs, s));
}

rt_status rt_watershed(rt_ctx *ctx, const int32_t *labels, int64_t ld_lab, const int32_t *d2, int64_t ld_d2, int H,
                       int W, int h, int32_t *basins, int64_t ld_b, int32_t *dev_n_basins, int32_t *dev_status,
                       void *stream)
{
    if (!ctx || !labels || !d2 || !basins || bad_dims(H, W) || ld_lab < W || ld_d2 < W || ld_b < W || h < 0)
        return RT_EINVAL;
    const size_t nb = span(H, ld_b, 4, W);
    if (overlaps(basins, nb, labels, span(H, ld_lab, 4, W)) || overlaps(basins, nb, d2, span(H, ld_d2, 4, W)))
        return RT_EINVAL;
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    rt_status st = ensure_ws(ctx, obj_workspace_bytes(H, W, false, true, 0), s);
    if (st != RT_OK) return st;
    ObjArgs a;
    std::memset(&a, 0, sizeof(a));
    a.L = labels;
    a.ld_L = ld_lab;
    a.D = d2;
    a.ld_D = ld_d2;
    a.H = H;
    a.W = W;
    a.h = h;
    a.basins = basins;
    a.ld_B = ld_b;
    a.n_basins = dev_n_basins;
    obj_carve(a, (char *)ctx->ws, false, true);
    a.err = dev_status;
    if (dev_status) RT_CUDA_TRY(cudaMemsetAsync(dev_status, 0, sizeof(int32_t), s));
    Phase ph(ctx, RT_PHASE_WATERSHED, s);
    int n = 0;
    const cudaError_t e = launch_watershed(a, ctx->num_sms, s, &n);
    ctx->launches += n;
    return cuda_status(e);
}

rt_status rt_object_features(rt_ctx *ctx, const int32_t *labels, int64_t ld_lab, const uint8_t *img, int64_t ld_img,
                             int H, int W, int32_t *obj_labels, double *feat, int cap, int32_t *dev_n_obj,
                             int32_t *dev_status, void *stream)
{
    if (!ctx || !labels || !img || bad_dims(H, W) || ld_lab < W || ld_img < W || cap < 0) return RT_EINVAL;
    if (cap > 0 && (!obj_labels || !feat)) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    rt_status st = ensure_ws(ctx, obj_workspace_bytes(H, W, true, false, cap), s);
    if (st != RT_OK) return st;
    ObjArgs a;
    std::memset(&a, 0, sizeof(a));
    a.L = labels;
    a.ld_L = ld_lab;
    a.I = img;
    a.ld_I = ld_img;
    a.H = H;
    a.W = W;
    a.cap = cap;
    a.out_labels = obj_labels;
    a.feat = feat;
    a.n_obj = dev_n_obj;
    obj_carve(a, (char *)ctx->ws, true, false);
    a.err = dev_status;
    if (dev_status) RT_CUDA_TRY(cudaMemsetAsync(dev_status, 0, sizeof(int32_t), s));
    Phase ph(ctx, RT_PHASE_OBJECTS, s);
    int n = 0;
    const cudaError_t e = launch_object_features(a, ctx->num_sms, s, &n);
    ctx->launches += n;
    return cuda_status(e);
}

rt_status rt_synth_tile(rt_ctx *ctx, uint8_t *out, int64_t ld, int H, int W, uint64_t seed, int n_shapes, int kind,
                        int vlo, int vhi, int rmin, int rmax, int amin, int amax, int flat, int noise, void *stream)
{
    if (!ctx || !out || bad_dims(H, W) || ld < W || n_shapes < 0 || (kind != 0 && kind != 1)) return RT_EINVAL;
    if (vlo < 0 || vhi > 255 || vlo > vhi || rmin < 0 || rmax < rmin || amin < 0 || amax < amin) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    rt_status st = ensure_ws(ctx, synth_workspace_bytes(H, W), s);
    if (st != RT_OK) return st;
    SynthArgs a;
    a.H = H;
    a.W = W;
    a.k0 = (uint32_t)(seed & 0xffffffffu);
    a.k1 = (uint32_t)(seed >> 32);
    a.n_shapes = n_shapes;
    a.kind = kind;
    a.vlo = vlo;
    a.vhi = vhi;
    a.rmin = rmin;
    a.rmax = rmax;
    a.amin = amin;
    a.amax = amax;
    a.flat = flat != 0;
    a.noise = noise != 0;
    ctx->launches += 3;
    return cuda_status(launch_synth(a, ctx->ws, out, ld, s));
}

rt_status rt_tile_features(rt_ctx *ctx, const uint8_t *const *imgs, const int64_t *lds, const int *Hs, const int *Ws,
                           int n, float *out, void *stream)
{
    if (!ctx || !imgs || !lds || !Hs || !Ws || !out || n < 1 || n > kMaxFeatImgs) return RT_EINVAL;
    for (int i = 0; i < n; ++i)
        if (!imgs[i] || bad_dims(Hs[i], Ws[i]) || lds[i] < Ws[i]) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    auto layout = [&](Carve &cv, FeatBatch &fb) {
        fb.n = n;
        for (int i = 0; i < n; ++i) {
            const size_t nb = (size_t)((Hs[i] + 7) / 8) * ((Ws[i] + 7) / 8);
            FeatImage &d = fb.img[i];
            d.img = imgs[i];
            d.ld = lds[i];
            d.H = Hs[i];
            d.W = Ws[i];
            d.hist = cv.take<uint32_t>(256);
            d.acc = cv.take<unsigned long long>(4);
            d.dark = cv.take<uint8_t>(nb);
            d.bmax = cv.take<uint8_t>(nb);
        }
    };
    FeatBatch fb;
    Carve cv;
    layout(cv, fb);
    rt_status st = ensure_ws(ctx, cv.off, s);
    if (st != RT_OK) return st;
    cv = Carve();
    cv.base = (char *)ctx->ws;
    layout(cv, fb);
    ctx->launches += 4;
    return cuda_status(launch_features(fb, out, s));
}

rt_status rt_mlp_forward(rt_ctx *ctx, const uint16_t *wb, const float *norm, const float *x, int B, float *logits,
                         float *act, int32_t *pick, float min_prob, int fallback, void *stream)
{
    if (!ctx || !wb || !norm || !x || B < 1 || !(min_prob <= 1.0f) || fallback < 0) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    ctx->launches += 1;
    return cuda_status(launch_mlp_forward(wb, norm, x, B, logits, act, pick, min_prob, fallback, (cudaStream_t)stream));
}

rt_status rt_mlp_forward_tc(rt_ctx *ctx, const uint16_t *wb, const float *norm, const float *x, int B, float *logits,
                            float *act, int32_t *pick, float min_prob, int fallback, int32_t *dev_status, void *stream)
{
    if (!ctx || !wb || !norm || !x || B < 1 || !(min_prob <= 1.0f) || fallback < 0) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    ctx->launches += 1;
    return cuda_status(
        launch_mlp_forward_tc(wb, norm, x, B, logits, act, pick, min_prob, fallback, dev_status, (cudaStream_t)stream));
}

rt_status rt_set_picker_classes(rt_ctx *ctx, const int *variants, const int *max_locals)
{
    if (!ctx || !variants || !max_locals) return RT_EINVAL;
    PickTable t = ctx->classes;
    for (int c = 0; c < kPickClasses; ++c) {
        const int v = variants[c] == RT_AUTO ? RT_RASTER : variants[c];
        if (v < RT_RASTER || v > RT_FRONTIER || max_locals[c] < 0) return RT_EINVAL;
        t.group[c] = v - RT_RASTER;
        t.max_local[c] = max_locals[c] > 0 ? max_locals[c] : default_max_local(v);
    }
    ctx->classes = t;
    return RT_OK;
}

rt_status rt_mlp_backward(rt_ctx *ctx, const uint16_t *wb, const float *norm, const float *x, const float *act,
                          const float *logits, const int32_t *label, int B, float *grad, float *loss, void *stream)
{
    if (!ctx || !wb || !norm || !x || !act || !logits || !label || !grad || B < 1) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    rt_status st = ensure_ws(ctx, mlp_backward_workspace_bytes(B), (cudaStream_t)stream);
    if (st != RT_OK) return st;
    ctx->launches += 2;
    return cuda_status(launch_mlp_backward(wb, norm, x, act, logits, label, B, grad, loss, (float *)ctx->ws,
                                           (cudaStream_t)stream));
}

rt_status rt_mlp_backward_tc(rt_ctx *ctx, const uint16_t *wb, const float *norm, const float *x, const float *act,
                             const float *logits, const int32_t *label, int B, float *grad, float *loss,
                             int32_t *dev_status, void *stream)
{
    if (!ctx || !wb || !norm || !x || !act || !logits || !label || !grad || B < 1) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    rt_status st = ensure_ws(ctx, mlp_backward_tc_workspace_bytes(B), (cudaStream_t)stream);
    if (st != RT_OK) return st;
    ctx->launches += 2;
    return cuda_status(launch_mlp_backward_tc(wb, norm, x, act, logits, label, B, grad, loss, (float *)ctx->ws,
                                              dev_status, (cudaStream_t)stream));
}

rt_status rt_feature_norm(rt_ctx *ctx, const float *x, int B, float *norm, void *stream)
{
    if (!ctx || !x || !norm || B < 1) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    ctx->launches += 1;
    return cuda_status(launch_feature_norm(x, B, norm, (cudaStream_t)stream));
}

rt_status rt_mlp_adamw(rt_ctx *ctx, float *master, uint16_t *wb, const float *grad, float *m, float *v, int step,
                       float lr, float beta1, float beta2, float eps, float weight_decay, void *stream)
{
    if (!ctx || !master || !wb || !grad || !m || !v || step < 1) return RT_EINVAL;
    DeviceGuard g(ctx->device);
    ctx->launches += 1;
    return cuda_status(
        launch_mlp_adamw(master, wb, grad, m, v, step, lr, beta1, beta2, eps, weight_decay, (cudaStream_t)stream));
}

int rt_last_picks(const rt_ctx *ctx, int *classes, int cap)
{
    if (!ctx) return 0;
    if (ctx->picks_ev_valid) {
        DeviceGuard g(ctx->device);
        if (cudaEventSynchronize(ctx->picks_ev) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
    }
    const int n = ctx->n_last_picks < cap ? ctx->n_last_picks : cap;
    for (int i = 0; classes && i < n; ++i) {
        const int c = ctx->picks_host[i];
        classes[i] = (c >= 0 && c < kPickClasses) ? c : kPickClasses;
    }
    return ctx->n_last_picks;
}

rt_status rt_set_picker(rt_ctx *ctx, const uint16_t *wb, const float *norm)
{
    if (!ctx || (!wb) != (!norm)) return RT_EINVAL;
    if (wb && !ctx->side) {   // a learned call may run the picker beside the chain
        DeviceGuard g(ctx->device);
        if ((!ctx->fork && cudaEventCreateWithFlags(&ctx->fork, cudaEventDisableTiming) != cudaSuccess) ||
            (!ctx->join && cudaEventCreateWithFlags(&ctx->join, cudaEventDisableTiming) != cudaSuccess) ||
            cudaStreamCreateWithFlags(&ctx->side, cudaStreamNonBlocking) != cudaSuccess) {
            cudaGetLastError();
            return RT_ECUDA;
        }
    }
    ctx->picker_wb = wb;
    ctx->picker_norm = norm;
    return RT_OK;
}

void rt_seg_params_default(rt_seg_params *p)
{
    if (!p) return;
    p->h_offset = 30;
    p->threshold = 80;
    p->min_area = 20;
    p->max_area = 1000;
    p->conn_recon = 8;
    p->conn_fill = 4;
    p->variant = RT_AUTO;
    p->max_local = 0;
    p->policy = RT_POLICY_PLAIN;
    p->max_iters = 0;
    p->timeout_ms = 0;
    p->pick_min_prob = 0;
    p->strip_tiles = 0;
}

rt_status rt_segment_batch(rt_ctx *ctx, const rt_tile *tiles, int n, const rt_seg_params *params, void *stream)
{
    if (!ctx || (!tiles && n > 0) || n < 0 || !params) return RT_EINVAL;
    const rt_seg_params &P = *params;
    if (bad_params(P)) return RT_EINVAL;
    for (int i = 0; i < n; ++i)
        if (bad_tile(tiles[i])) return RT_EINVAL;
    if (n == 0) return RT_OK;
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    const bool learned = P.policy == RT_POLICY_LEARNED && ctx->picker_wb && ctx->picker_norm;
    const Limits lim = seg_limits(ctx, P);
    // one allocation for the largest chunk, before anything is enqueued
    rt_status st = ensure_ws(ctx, segment_ws_bytes(tiles, n, P, learned, ctx), s);
    if (st != RT_OK) return st;

    for (int c0 = 0; c0 < n; c0 += kMaxImgs) {
        const int cn = n - c0 < kMaxImgs ? n - c0 : kMaxImgs;
        Chunk c;
        Carve cv;
        cv.base = (char *)ctx->ws;
        layout_chunk(cv, c, tiles, c0, cn, P, learned, ctx, lim);
        RT_CUDA_TRY(zero_words(c.err, c.ctl_words, s));
        ctx->launches += 1;
        auto reconstruct = [&](const int32_t *pick) {
            return c.reach ? run_reach(ctx, c.rb, s) : c.contract ? run_contract(ctx, c.cb, c.err, s, lim)
                              : run_recon(ctx, c.b, c.w, P.conn_recon, P.variant, P.max_local, c.err, s, lim, pick);
        };
        bool aside = false;
        if (!learned) {
            st = reconstruct(nullptr);
            if (st != RT_OK) return st;
        } else {
            // the picker chooses a variant per tile on the device; the
            // propagation reads its choices directly (no host round trip).
            // With raster classes and a contracted reconstruction the picks
            // are reported but change no schedule: then the picker runs
            // beside the chain on the context's own stream, forked at the
            // call's start and joined at its end (by events, so a capture of
            // the call captures both).
            const bool pick = picks_matter(ctx, P, cn);
            // Not where the chain writes over the image that the picker reads.
            aside = pick && c.contract;
            for (int i = 0; i < cn; ++i) aside = aside && !in_place(tiles[c0 + i]);
            if (aside) {
                RT_CUDA_TRY(cudaEventRecord(ctx->fork, s));
            } else if (pick) {
                st = run_picker(ctx, c, P, s);
                if (st != RT_OK) return st;
            }
            st = reconstruct(pick ? c.picks : nullptr);
            if (st != RT_OK) return st;
            if (!aside) {
                st = report_picks(ctx, pick ? c.picks : nullptr, cn, s);
                if (st != RT_OK) return st;
            }
        }
        if (!c.reach) {
            Phase ph(ctx, RT_PHASE_RECON_OUT, s);
            ctx->launches += 1;
            RT_CUDA_TRY(c.contract ? launch_contract_out(c.cb, P.threshold, s) : launch_recon_out(c.b, P.threshold, s));
        }
        {
            Phase ph(ctx, RT_PHASE_FILL, s);
            if (!c.contract) RT_CUDA_TRY(launch_run_pack(c.rb, s));
            RT_CUDA_TRY(launch_run_fill(c.rb, P.conn_fill, 8, s, c.reach));
            ctx->launches += c.contract ? 3 : 4;
        }
        {
            Phase ph(ctx, RT_PHASE_LABEL, s);
            ctx->launches += 3;
            RT_CUDA_TRY(launch_run_label(c.rb, 8, s));
        }
        {
            Phase ph(ctx, RT_PHASE_EDT, s);
            ctx->launches += 2;
            RT_CUDA_TRY(launch_edt_bits_batch(c.eb, ctx->num_sms, kSweepTimeoutNs, s));
        }
        if (aside) {   // enqueued last: its launches delay none of the chain's
            RT_CUDA_TRY(cudaStreamWaitEvent(ctx->side, ctx->fork, 0));
            st = run_picker(ctx, c, P, ctx->side);
            if (st == RT_OK) st = report_picks(ctx, c.picks, cn, ctx->side);
            RT_CUDA_TRY(cudaEventRecord(ctx->join, ctx->side));
            RT_CUDA_TRY(cudaStreamWaitEvent(s, ctx->join, 0));
            if (st != RT_OK) return st;
        }
        StatusOut so;
        bool any_status = false;
        for (int i = 0; i < cn; ++i) {
            so.dst[i] = tiles[c0 + i].status;
            any_status |= so.dst[i] != nullptr;
        }
        if (any_status) {
            launch_early(copy_status_kernel, 1, 32, 0, s, c.err, so, cn);
            ctx->launches += 1;
            RT_CUDA_TRY(cudaGetLastError());
        }
    }
    return RT_OK;
}

}  // extern "C"
