// C-ABI of libasicp (declared in include/asicp.h): context, inputs, the
// iteration loop of Algorithm 1 and result read-back.  Host code only; every
// arithmetic step of the method runs in the kernels of k_match.cu,
// k_collision.cu and k_update.cu.
//
// A context holds n_objects objects (one grasp set each) that are optimised
// together: every kernel covers the particles of all objects, each particle
// matched against its own object's cloud.  Particles are numbered object by
// object, preshape by preshape (groups g = o * P + p of K_g particles).
#include "../../include/asicp.h"
#include "asicp_internal.cuh"

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <queue>
#include <string>
#include <utility>
#include <vector>

using namespace asicp;
static_assert(kFwdVariants == ASICP_FWD_SHAPES, "kernel shape count differs from the header");

namespace {

struct Err {
    asicp_status st;
    std::string msg;
};

[[noreturn]] void fail(asicp_status st, const std::string &msg) { throw Err{st, msg}; }

void ck(cudaError_t e, const char *what)
{
    if (e == cudaSuccess) return;
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        fail(ASICP_ERR_OOM, std::string(what) + ": " + cudaGetErrorString(e));
    }
    fail(ASICP_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// Device allocation owned by the context; grows on demand, never shrinks.
struct DevMem {
    void *p = nullptr;
    size_t bytes = 0;
    DevMem() = default;
    DevMem(const DevMem &) = delete;
    DevMem &operator=(const DevMem &) = delete;
    DevMem(DevMem &&o) noexcept : p(o.p), bytes(o.bytes) { o.p = nullptr; o.bytes = 0; }
    ~DevMem() { if (p) cudaFree(p); }
    void ensure(size_t want, const char *what)
    {
        if (want <= bytes && p) return;
        if (p) { cudaFree(p); p = nullptr; bytes = 0; }
        if (want == 0) want = 16;
        ck(cudaMalloc(&p, want), what);
        bytes = want;
    }
    void release()
    {
        if (p) cudaFree(p);
        p = nullptr;
        bytes = 0;
    }
    template <class T> T *as() const { return static_cast<T *>(p); }
};

// Page-locked host memory that inputs and results of at most kPinPiece bytes pass through; grows on
// demand up to kPinMost.  Larger pieces (or without memory) are copied straight between the caller's
// arrays and the device.
constexpr size_t kPinPiece = (size_t)256 << 10, kPinMost = (size_t)2 << 20;
struct PinMem {
    unsigned char *p = nullptr;
    size_t bytes = 0;
    PinMem() = default;
    PinMem(const PinMem &) = delete;
    PinMem &operator=(const PinMem &) = delete;
    ~PinMem() { if (p) cudaFreeHost(p); }
    bool ensure(size_t want)       // (contents are not kept; no copy may be in flight)
    {
        if (want <= bytes) return true;
        if (want > kPinMost) return false;
        if (p) cudaFreeHost(p);
        p = nullptr;
        bytes = 0;
        want = std::max(want, (size_t)64 << 10);
        void *q = nullptr;
        if (cudaHostAlloc(&q, want, cudaHostAllocDefault) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        p = static_cast<unsigned char *>(q);
        bytes = want;
        return true;
    }
};

// Ordinary host memory, which an asynchronous copy would have to stage.
bool pageable(const void *p)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeUnregistered;
}

struct ObjBufs {
    DevMem R, Rx, Rt, C;      // C stays empty when the collision cloud is R itself
    DevMem nodes, leaves;     // matching cells of R
    DevMem Csort, Cball;      // the collision cloud in spatial order
    int M = 0, Mpad = 0, Mc = 0;
    float4 frame{};           // centre and radius of R, as on the device
    bool set = false, cells_built = false, sorted = false;
};

// Matching through cells (k_cells.cu): for clouds of kCellMinM points and more up to kCellMaxM
// (the build's 32-bit counters cannot overflow below it), once the passes known of on the
// present objects (those of an asicp_run, or the asicp_step calls so far) would take longer
// through the screening than the build: screening and exact choice take 1 us per kCellRate
// pairs, the build 100 us + 1 us per kCellRatePts points (measured: 0.27 ms at 8192 points,
// 1.4 ms at 65536), the matching through the cells little beside either.  kCellMinM keeps the
// tables (9.7 MB for the smallest cloud) from batches of many small clouds; it is not where the
// cells stop paying: 1.6 M queries on 256 / 512 / 1000 points take 160 / 181 / 230 us through
// the screening and 29 / 30 / 32 through cells (on 128 points the screening stays the cheaper).
constexpr int kCellMinM = 1024, kCellMaxM = 1 << 18;
constexpr double kCellRate = 1.65e7, kCellRatePts = 50.0;
// Clouds whose lists do not shrink (points on a common sphere or plane, many copies of a point) are matched faster by
// the screening.  So the work of one pass is counted on a sample of the queries when cells have been built (see
// cells_cost_kernel): a pass takes 1 us per kCellRounds rounds, or, where few warps have long lists, kCellLatency us
// per round of the longest one.  Screening and exact choice take kScreenLeast us (two kernels) and at least
// kScreenPoint us per object point (one CTA's chain over the tiles: 6144 queries on 200000 points 363 us).
constexpr double kCellRounds = 7.5e4, kCellLatency = 0.15, kScreenLeast = 15.0, kScreenPoint = 1.8e-3;
constexpr double kCellDoubt = 1.0 / 32.0;            // after such clouds the next ones' build is held against this much
constexpr size_t kCellScratch = (size_t)256 << 20;   // scratch of one build launch (at least one object)

enum { kTimeMatch = 0, kTimeCollide = 1, kTimeCollideNN = 2, kTimeFinalize = 3, kTimeStein = 4, kTimeExact = 5,
       kTimeKinds = 6 };
static_assert(kTimeKinds == ASICP_KERNEL_KINDS, "kernel kinds");

}  // namespace

struct asicp_ctx {
    asicp_config cfg{};
    cudaStream_t st = nullptr;
    std::string err;
    int N = 0;
    int nobj = 1;
    std::vector<int> Kg;              // particles per group, [nobj * P]
    std::vector<ObjBufs> objs;
    bool theta_set = false, stepped = false, run_done = false;
    std::vector<char> pre_set;
    std::vector<SdfMeta> meta;
    std::vector<DevMem> grids;
    std::vector<DevMem> cells;         // corner-packed grids
    std::vector<DevMem> clear;         // their cells' clearances
    int k_next = 0;

    // mini-batches of the object cloud per iteration (Table I), one object only
    std::vector<int> mb_off;          // [iters + 1] on the host (sizes are fixed at capture)
    DevMem mb_idx, mb_R, mb_Rx;
    bool table_mb = false;            // the object table on the device points at a mini-batch

    int fwd_variant = 0;              // forward-matching kernel shape (autotuner's choice)
    bool tuned = false;
    bool cells_oom = false;           // no room for matching cells: the screening is used
    bool cells_on = false;            // the passes being launched match through the cells
    bool cells_slow = false;          // the present objects' cells are built, but the screening is the faster
    double cells_worth = 1.0;         // share of the screening's time that the next clouds' build is weighed against
    double cells_share = 0.0;         // sample of the cost count that has been enqueued (0: none)
    unsigned weight_seq = 0;          // number of that count
    double cells_owed = 0.0;          // microseconds of screening on the present objects so far
    bool pre_oom = false;             // no room for the gripper clouds' cells
    int fail_cells = -1;              // this many more allocations for cells succeed, the next fails (testing; < 0: off)
    bool pre_on = false;              // the passes being launched match the colliding points through them
    std::vector<float4> preframe_h;   // the gripper clouds' centres and radii, as on the device
    bool pre_built = false;           // the gripper clouds' cells are built (all preshapes together)
    double pre_owed = 0.0;            // microseconds of reverse matching without them so far
    bool recording = false;           // the caller's stream is being captured (see note_capture)
    bool expire_test = false;         // the float32 matching kernels' first copy waits expire (testing)

    // layout (rebuilt when objects, particle counts or N change)
    bool layout_dirty = true;
    int T = 0, G = 0, n_items = 0;
    long long colidx_total = 0, colmap_total = 0;
    std::vector<int> grp_off_h;
    std::vector<ObjMeta> objmeta_h;

    DevMem partgrp, grpoff, objmeta, items, ctaoff, com, frame, colitems, collist, stage, S, Ssort, preframe, prenodes, preleaves, cellwork, refscr, pconst, dmeta, theta,
        ncol, colidx, colsrt, colnn, colmap, cost, grad, prev, frozen, phi, h, order, errw, out7, outc, outi, nnidx, tccand, dbg_d2, dbg_sp;

    // profiling: events recorded around launches (kind, start, stop)
    struct Ev { int kind; cudaEvent_t a, b; };
    std::vector<Ev> events;
    std::vector<cudaEvent_t> pool;
    double acc_ms[kTimeKinds] = {};
    long long acc_n[kTimeKinds] = {};

    // results on their way to the caller (flushed by finish()) and the page-locked memory they and the
    // inputs pass through; pin_busy: a copy from it has been enqueued and not waited for
    struct Out { void *dst; const void *src; size_t bytes; };
    std::vector<Out> outs;
    PinMem pin, pin_in;
    PinMem weights;                   // the cells' cost count, written by the device
    bool pin_busy = false;
    size_t pin_used = 0;              // bytes of pin_in taken by copies in flight
    DevMem outp, outg;                // phi and gradient as they are returned

    // CUDA graph of asicp_run's iteration loop (captured once per buffer layout)
    std::vector<int> loop_mb;         // mini-batch offsets it was captured with, and the object's entry
    ObjMeta loop_meta{};
    cudaStream_t cap_st = nullptr;
    // the collision test's branch of a pass and the events that part and join the two
    cudaStream_t side_st = nullptr;
    cudaEvent_t parted = nullptr, joined = nullptr;
    cudaGraphExec_t loop_exec = nullptr;
    std::vector<const void *> loop_key;
    std::vector<Ev> graph_events;     // event pairs inside the graph (profile = 1)
    bool graph_pending = false;       // a replay's events have not been accumulated yet
    bool capturing = false;

    bool inputs_ready() const
    {
        if (N == 0) return false;
        for (const auto &o : objs) if (!o.set) return false;
        for (char c : pre_set) if (!c) return false;
        return true;
    }
    Layout layout() const
    {
        Layout L;
        L.P = cfg.P;
        L.N = N;
        L.G = G;
        L.nobj = nobj;
        L.T = T;
        L.part_grp = partgrp.as<int>();
        L.grp_off = grpoff.as<int>();
        L.obj = objmeta.as<ObjMeta>();
        L.com = com.as<double>();
        L.frame = frame.as<float4>();
        return L;
    }
    cudaEvent_t take_event()
    {
        if (!pool.empty()) { cudaEvent_t e = pool.back(); pool.pop_back(); return e; }
        cudaEvent_t e;
        ck(cudaEventCreate(&e), "cudaEventCreate");
        return e;
    }
    ~asicp_ctx()
    {
        for (auto &e : events) { cudaEventDestroy(e.a); cudaEventDestroy(e.b); }
        for (auto &e : graph_events) { cudaEventDestroy(e.a); cudaEventDestroy(e.b); }
        for (auto e : pool) cudaEventDestroy(e);
        if (loop_exec) cudaGraphExecDestroy(loop_exec);
        if (cap_st) cudaStreamDestroy(cap_st);
        if (parted) cudaEventDestroy(parted);
        if (joined) cudaEventDestroy(joined);
        if (side_st) cudaStreamDestroy(side_st);
    }
};

namespace {

template <class F>
asicp_status guarded(asicp_ctx *ctx, F &&f)
{
    if (!ctx) return ASICP_ERR_INVALID_ARG;
    try {
        f();
        ctx->err.clear();
        return ASICP_OK;
    } catch (const Err &e) {
        ctx->err = e.msg;
        return e.st;
    } catch (const std::bad_alloc &) {
        ctx->err = "host allocation failed";
        return ASICP_ERR_OOM;
    } catch (...) {
        ctx->err = "unexpected internal error";
        return ASICP_ERR_CUDA;
    }
}

// Results of a call, copied as 32-bit words into page-locked memory by one kernel: word 0 is the error
// word, the pieces follow.
constexpr int kPieces = 8;
struct OutPieces {
    const unsigned *src[kPieces];
    unsigned words[kPieces];
    int n;
};
__global__ void collect_kernel(const OutPieces o, const int *err, unsigned *dst)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    if (i == 0) dst[0] = (unsigned)*err;
    unsigned base = 4;                     // (16 bytes: the pieces stay aligned for any type)
    for (int k = 0; k < o.n; ++k) {
        for (unsigned w = i; w < o.words[k]; w += step) dst[base + w] = o.src[k][w];
        base += (o.words[k] + 3u) & ~3u;
    }
}

// Enqueue a result: it is in the caller's array when finish() returns.
void copy_out(asicp_ctx *c, void *dst, const void *src, size_t bytes)
{
    if (dst && bytes) c->outs.push_back({dst, src, bytes});
}

// Wait for the stream, once: with the results asked for and the error word in page-locked memory; then
// hand the results over, or report the error.
void finish(asicp_ctx *c, const char *what)
{
    OutPieces o{};
    std::vector<asicp_ctx::Out> staged;
    size_t total = 16;
    for (const auto &x : c->outs) {
        const size_t room = (x.bytes + 15) / 16 * 16;
        if (o.n < kPieces && x.bytes % 4 == 0 && x.bytes <= kPinPiece && total + room <= kPinMost && pageable(x.dst)) {
            o.src[o.n] = static_cast<const unsigned *>(x.src);
            o.words[o.n++] = (unsigned)(x.bytes / 4);
            total += room;
            staged.push_back(x);
        } else {
            const cudaError_t e = cudaMemcpyAsync(x.dst, x.src, x.bytes, cudaMemcpyDefault, c->st);
            if (e != cudaSuccess) c->outs.clear();
            ck(e, what);
        }
    }
    int err = 0;
    if (c->pin.ensure(total)) {
        const int blocks = (int)std::min<size_t>((total / 4 + 255) / 256, 128);
        collect_kernel<<<blocks, 256, 0, c->st>>>(o, c->errw.as<int>(), reinterpret_cast<unsigned *>(c->pin.p));
        c->outs.clear();
        ck(cudaGetLastError(), what);
        ck(cudaStreamSynchronize(c->st), what);
        err = *reinterpret_cast<const int *>(c->pin.p);
        size_t at = 16;
        for (const auto &x : staged) {
            if (err == kDevOk) std::memcpy(x.dst, c->pin.p + at, x.bytes);
            at += (x.bytes + 15) / 16 * 16;
        }
    } else {
        c->outs.clear();
        for (const auto &x : staged) ck(cudaMemcpyAsync(x.dst, x.src, x.bytes, cudaMemcpyDefault, c->st), what);
        ck(cudaMemcpyAsync(&err, c->errw.p, sizeof(int), cudaMemcpyDeviceToHost, c->st), what);
        ck(cudaStreamSynchronize(c->st), what);
    }
    c->pin_busy = false;
    if (err == kDevNonFinite) {
        ck(cudaMemsetAsync(c->errw.p, 0, sizeof(int), c->st), "clear error word");
        fail(ASICP_ERR_INVALID_ARG, std::string(what) + ": non-finite value in the input");
    }
    if (err == kDevTimeout) {
        ck(cudaMemsetAsync(c->errw.p, 0, sizeof(int), c->st), "clear error word");
        fail(ASICP_ERR_TIMEOUT, std::string(what) + ": a bounded device wait expired");
    }
}

// Enqueue the copy of an input; the source may be reused once the call has returned (pageable memory is
// copied here and now, other memory by the time of finish()).
void upload(asicp_ctx *c, void *dst, const void *src, size_t bytes, const char *what)
{
    if (bytes > 0 && bytes <= kPinPiece && pageable(src)) {
        if (!c->pin_busy) c->pin_used = 0;
        if (c->pin_busy && c->pin_used + bytes > c->pin_in.bytes) {
            ck(cudaStreamSynchronize(c->st), what);
            c->pin_busy = false;
            c->pin_used = 0;
        }
        if (c->pin_busy || c->pin_in.ensure(bytes)) {
            unsigned char *at = c->pin_in.p + c->pin_used;
            std::memcpy(at, src, bytes);
            c->pin_busy = true;
            c->pin_used += (bytes + 255) / 256 * 256;
            ck(cudaMemcpyAsync(dst, at, bytes, cudaMemcpyHostToDevice, c->st), what);
            return;
        }
    }
    ck(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, c->st), what);
}

double gamma_of(const asicp_config &c, int k)
{
    if (c.schedule == 1) {
        if (c.k_max <= 1) return c.g1;
        return c.g0 + (double)(c.g1 - c.g0) * k / (double)(c.k_max - 1);
    }
    const double period = (double)c.k_max / c.C_cycles;          // Eq. 11 with T = k_max
    return std::pow(std::fmod((double)k, period) / period, (double)c.p_exp);
}

// Offsets, work items and buffers for the current objects, particle counts and N.
// Work plan of the forward matching for kernel shape v.  Items are whole
// multiples of the shape's CTA size (at most threads x queries per thread) of one
// object, sized so that about kPlanRounds items of equal cost fall to each CTA
// of the persistent grid; they are dealt out longest first, each to the CTA
// with the least work so far (cost = queries x padded object points), and
// every CTA gets a contiguous range of the item table.
void plan_fwd_items(asicp_ctx *c, int v)
{
    constexpr int kPlanRounds = 3;
    const int grid = fwd_shape_grid(v), threads = fwd_shape_threads(v), qmax = fwd_shape_queries(v), N = c->N;
    const std::vector<ObjMeta> &om = c->objmeta_h;
    double W = 0.0;
    for (const ObjMeta &m : om) W += (double)m.np * N * m.Mpad;
    const double unit = W / ((double)grid * kPlanRounds);
    std::vector<FwdItem> items;
    for (int o = 0; o < (int)om.size(); ++o) {
        const ObjMeta &m = om[o];
        long long nq = (long long)std::ceil(unit / std::max(1, m.Mpad) / threads) * threads;
        nq = std::min<long long>(std::max<long long>(nq, threads), qmax);
        // few queries for the grid: the item size that gives the shortest schedule
        if (nq == threads && om.size() == 1 && v != kFwdVariants - 1) nq = fwd_item_queries(v, (long long)m.np * N);
        const long long q0 = (long long)m.pfirst * N, q1 = (long long)(m.pfirst + m.np) * N;
        for (long long q = q0; q < q1; q += nq) {
            FwdItem it;
            it.q0 = q;
            it.nq = (int)std::min<long long>(nq, q1 - q);
            it.obj = o;
            items.push_back(it);
        }
    }
    auto cost = [&](const FwdItem &x) { return (long long)x.nq * om[x.obj].Mpad; };
    std::stable_sort(items.begin(), items.end(), [&](const FwdItem &x, const FwdItem &y) { return cost(x) > cost(y); });
    // least-loaded CTA first (ties: lowest CTA index)
    using Slot = std::pair<long long, int>;
    std::priority_queue<Slot, std::vector<Slot>, std::greater<Slot>> heap;
    for (int b = 0; b < grid; ++b) heap.push({0, b});
    std::vector<int> owner(items.size());
    std::vector<int> count(grid + 1, 0);
    for (size_t i = 0; i < items.size(); ++i) {
        Slot s = heap.top();
        heap.pop();
        owner[i] = s.second;
        ++count[s.second + 1];
        heap.push({s.first + cost(items[i]), s.second});
    }
    std::vector<int> off(grid + 1, 0);
    for (int b = 0; b < grid; ++b) off[b + 1] = off[b] + count[b + 1];
    std::vector<FwdItem> placed(items.size());
    std::vector<int> fill(off.begin(), off.end() - 1);
    for (size_t i = 0; i < items.size(); ++i) placed[fill[owner[i]]++] = items[i];

    c->items.ensure(sizeof(FwdItem) * std::max<size_t>(1, placed.size()), "matching work items");
    c->ctaoff.ensure(sizeof(int) * (grid + 1), "matching work plan");
    if (!placed.empty())
        ck(cudaMemcpyAsync(c->items.p, placed.data(), sizeof(FwdItem) * placed.size(), cudaMemcpyHostToDevice, c->st),
           "work items");
    ck(cudaMemcpyAsync(c->ctaoff.p, off.data(), sizeof(int) * (grid + 1), cudaMemcpyHostToDevice, c->st),
       "work plan");
    ck(cudaStreamSynchronize(c->st), "work plan");
    c->n_items = (int)placed.size();
}

void build_layout(asicp_ctx *c)
{
    if (!c->layout_dirty) return;
    if (!c->inputs_ready()) fail(ASICP_ERR_STATE, "objects and every preshape must be set first");
    const int P = c->cfg.P, G = c->nobj * P, N = c->N;
    std::vector<int> off(G + 1, 0);
    for (int g = 0; g < G; ++g) off[g + 1] = off[g] + c->Kg[g];
    const int T = off[G];
    std::vector<int> part_grp(T);
    for (int g = 0; g < G; ++g)
        for (int i = off[g]; i < off[g + 1]; ++i) part_grp[i] = g;
    std::vector<ObjMeta> om(c->nobj);
    long long colidx_total = 0, colmap_total = 0;
    for (int o = 0; o < c->nobj; ++o) {
        const ObjBufs &b = c->objs[o];
        ObjMeta &m = om[o];
        m.R = b.R.as<float4>();
        m.Rx = b.Rx.as<ulonglong2>();
        m.Rt = b.Rt.as<float>();
        m.nodes = b.nodes.as<int2>();
        m.leaves = b.leaves.as<int>();
        m.Csort = b.Csort.as<float4>();
        m.Cball = b.Cball.as<float4>();
        m.C = b.C.p ? b.C.as<float4>() : b.R.as<float4>();
        m.M = b.M;
        m.Mpad = b.Mpad;
        m.Mc = b.Mc;
        m.pfirst = off[o * P];
        m.np = off[(o + 1) * P] - off[o * P];
        m.colidx_base = colidx_total;
        m.colmap_base = colmap_total;
        colidx_total += (long long)m.np * m.Mc;
        colmap_total += (long long)m.np * ((m.Mc + 31) / 32);
    }

    if (T != c->T) {
        c->theta_set = false;
        c->run_done = false;
    }
    c->T = T;
    c->G = G;
    c->colidx_total = colidx_total;
    c->colmap_total = colmap_total;
    c->grp_off_h = off;
    c->objmeta_h = om;

    c->partgrp.ensure(sizeof(int) * T, "particle groups");
    c->grpoff.ensure(sizeof(int) * (G + 1), "group offsets");
    c->objmeta.ensure(sizeof(ObjMeta) * c->nobj, "object table");
    c->theta.ensure(sizeof(float) * 8 * (size_t)T, "poses");
    c->colitems.ensure(sizeof(int) * 2, "collision work counters");
    c->collist.ensure(sizeof(int) * 2 * std::max<long long>(1, colmap_total), "collision work list");
    c->colmap.ensure(sizeof(int2) * std::max<long long>(1, colmap_total), "collision bit maps");
    c->nnidx.ensure(sizeof(int) * (size_t)T * N, "nn_idx");
    c->tccand.ensure(sizeof(int4) * (size_t)T * N, "tensor-core candidate chunks");
    c->ncol.ensure(sizeof(int) * T, "ncol");
    c->colidx.ensure(sizeof(int) * std::max<long long>(1, colidx_total), "colidx");
    c->colnn.ensure(sizeof(int) * std::max<long long>(1, colidx_total), "colnn");
    c->cost.ensure(sizeof(double) * T, "cost");
    c->grad.ensure(sizeof(double) * T * 8, "grad");
    c->prev.ensure(sizeof(double) * T, "prev_cost");
    c->frozen.ensure(sizeof(int) * T, "frozen");
    c->phi.ensure(sizeof(float) * T * 8, "phi");
    c->h.ensure(sizeof(float) * G, "h");
    c->order.ensure(sizeof(int) * T, "order");
    c->out7.ensure(sizeof(float) * T * 8, "out7");
    c->outc.ensure(sizeof(float) * T, "outc");
    c->outi.ensure(sizeof(int) * T, "outi");
    if (c->cfg.debug) {
        c->dbg_d2.ensure(sizeof(float) * (size_t)T * N, "dbg_d2");
        c->dbg_sp.ensure(sizeof(float) * (size_t)T * N * 3, "dbg_sp");
    }
    // device tables (pageable sources: the copies complete before returning)
    ck(cudaMemcpyAsync(c->partgrp.p, part_grp.data(), sizeof(int) * T, cudaMemcpyHostToDevice, c->st), "particle groups");
    ck(cudaMemcpyAsync(c->grpoff.p, off.data(), sizeof(int) * (G + 1), cudaMemcpyHostToDevice, c->st), "group offsets");
    ck(cudaMemcpyAsync(c->objmeta.p, om.data(), sizeof(ObjMeta) * c->nobj, cudaMemcpyHostToDevice, c->st),
       "object table");
    ck(cudaStreamSynchronize(c->st), "layout");
    c->layout_dirty = false;
    c->table_mb = false;
    plan_fwd_items(c, c->fwd_variant);
}

__global__ void reset_convergence_kernel(double *prev, int *frozen, float *phi, int T, int *col_items)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) { col_items[0] = 0; col_items[1] = 0; }
    if (i >= T) return;
    prev[i] = -1.0;     // no previous cost
    frozen[i] = 0;
    for (int a = 0; a < 8; ++a) phi[(size_t)i * 8 + a] = 0.f;
}

// Stream the iteration kernels go to: the capture stream while a graph is being
// recorded, else the caller's stream.
cudaStream_t work_stream(const asicp_ctx *c) { return c->capturing ? c->cap_st : c->st; }

void reset_convergence(asicp_ctx *c)
{
    reset_convergence_kernel<<<(c->T + 255) / 256, 256, 0, work_stream(c)>>>(
        c->prev.as<double>(), c->frozen.as<int>(), c->phi.as<float>(), c->T, c->colitems.as<int>());
    ck(cudaGetLastError(), "reset convergence state");
}

template <class L>
void timed(asicp_ctx *c, int kind, L &&launch, const char *what, cudaStream_t side = nullptr)
{
    cudaEvent_t a = nullptr, b = nullptr;
    cudaStream_t st = side ? side : work_stream(c);
    // inside a capture, an external record makes the event a graph node that every
    // replay records (a plain record would only express a capture dependency)
    const unsigned flags = c->capturing ? cudaEventRecordExternal : cudaEventRecordDefault;
    // profile 1: every kernel; 2: the forward-matching (screening) kernel only.  Each event
    // record is a node of the captured loop and costs a few microseconds of the replay.
    const bool on = c->cfg.profile == 1 || (c->cfg.profile == 2 && kind == kTimeMatch);
    if (on) {
        a = c->take_event();
        b = c->take_event();
        ck(cudaEventRecordWithFlags(a, st, flags), "cudaEventRecord");
    }
    ck(launch(st), what);
    if (on) {
        ck(cudaEventRecordWithFlags(b, st, flags), "cudaEventRecord");
        (c->capturing ? c->graph_events : c->events).push_back({kind, a, b});
    }
}

// Add the device times of the last graph replay (its events are re-recorded by
// every replay, so they are read before the next one).
void accumulate_graph_events(asicp_ctx *c)
{
    if (!c->graph_pending) return;
    for (auto &e : c->graph_events) {
        float t = 0.f;
        ck(cudaEventSynchronize(e.b), "cudaEventSynchronize");
        ck(cudaEventElapsedTime(&t, e.a, e.b), "cudaEventElapsedTime");
        c->acc_ms[e.kind] += t;
        c->acc_n[e.kind] += 1;
    }
    c->graph_pending = false;
}

// Object 0's table points at the mini-batch of iteration k (k < the number of
// mini-batches) or back at the whole cloud (otherwise), on the work stream.
void select_minibatch(asicp_ctx *c, int k)
{
    if (c->mb_off.empty()) return;
    cudaStream_t st = work_stream(c);
    ObjMeta m = c->objmeta_h[0];
    c->table_mb = k >= 0 && k + 1 < (int)c->mb_off.size();
    if (c->table_mb) {
        const int first = c->mb_off[k], cnt = c->mb_off[k + 1] - first;
        const int Mpad = (cnt + kRefTilePts - 1) / kRefTilePts * kRefTilePts;
        m.R = c->mb_R.as<float4>();
        m.Rx = c->mb_Rx.as<ulonglong2>();
        m.M = cnt;
        m.Mpad = Mpad;
        ck(launch_minibatch(c->objs[0].R.as<float4>(), c->mb_idx.as<int>() + first, cnt, Mpad, c->mb_R.as<float4>(),
                            c->mb_Rx.p, c->frame.as<float4>(), c->objmeta.as<ObjMeta>(), m, st),
           "mini-batch");
        return;
    }
    ck(launch_store_meta(c->objmeta.as<ObjMeta>(), m, st), "object table");
}

// No mini-batches from here on: a table that a step has left at one points at the whole cloud again.
void drop_minibatches(asicp_ctx *c)
{
    c->mb_off.clear();
    if (!c->table_mb) return;
    c->table_mb = false;                  // (a layout to be rebuilt writes the whole table)
    if (!c->layout_dirty) ck(launch_store_meta(c->objmeta.as<ObjMeta>(), c->objmeta_h[0], c->st), "object table");
}

// Build the cells of the given clouds (at most kCellBatch of them, or as many as the scratch
// holds, per launch).
size_t cell_scratch(const CellSizes &s) { return 2 * sizeof(int) * (size_t)s.list_cap + s.rec_bytes; }
constexpr size_t kCellCtrBytes = sizeof(int) * kCellCounters * kCellBatch;

size_t scratch_bytes(const std::vector<int> &sizes)
{
    size_t need = 0, sum = 0;
    for (size_t i = 0, first = 0; i < sizes.size(); ++i) {
        const size_t w = cell_scratch(cell_sizes(sizes[i]));
        if (i > first && (sum + w > kCellScratch || i - first == kCellBatch)) { sum = 0; first = i; }
        sum += w;
        need = std::max(need, sum);
    }
    return kCellCtrBytes + need;
}

void build_cells(asicp_ctx *c, const std::vector<CellBuild> &todo)
{
    for (size_t i = 0; i < todo.size();) {
        CellBuildBatch batch{};
        unsigned char *at = c->cellwork.as<unsigned char>() + kCellCtrBytes,
                      *end = c->cellwork.as<unsigned char>() + c->cellwork.bytes;
        int n = 0;
        for (; i < todo.size() && n < kCellBatch; ++i, ++n) {
            const CellSizes s = cell_sizes(todo[i].M);
            if (n > 0 && (size_t)(end - at) < cell_scratch(s)) break;
            CellBuild &b = batch.b[n];
            b = todo[i];
            b.recs = at;
            b.lists = reinterpret_cast<int *>(at + s.rec_bytes);
            b.ctr = c->cellwork.as<int>() + kCellCounters * n;
            b.leaf_cap = s.leaf_cap; b.list_cap = s.list_cap; b.cell_cap = s.cell_cap; b.node_cap = s.node_cap;
            at += cell_scratch(s);
        }
        ck(cudaMemsetAsync(c->cellwork.p, 0, kCellCtrBytes, c->st), "matching cells");
        ck(launch_cells_build(batch, n, c->st), "matching cells");
    }
}

// Memory for cells.  They only make passes faster, so they take at most an eighth of what is free on the device
// (their size is a bound for any cloud, 9.7 MB and 1.15 KB per point of an object, and a few MB of it are used);
// without room the kernels that need none run.
void need_room(const std::vector<std::pair<const DevMem *, size_t>> &wants)
{
    size_t more = 0, avail = 0, total = 0;
    for (const auto &w : wants) more += w.second > w.first->bytes ? w.second - w.first->bytes : 0;
    if (more == 0) return;
    ck(cudaMemGetInfo(&avail, &total), "free memory");
    if (more > avail / 8) fail(ASICP_ERR_OOM, "cells would take more than an eighth of the free memory");
}

void cell_memory(asicp_ctx *c, DevMem &m, size_t bytes, const char *what)
{
    if (c->fail_cells >= 0 && c->fail_cells-- == 0) fail(ASICP_ERR_OOM, what);
    m.ensure(bytes, what);
}

// Decide whether the next `passes` passes of kernel shape v match through the cells, and build
// those of every object whose points are new (outside any capture).  The objects of a
// launch share it, so many small clouds cost little more than one.
void ensure_cells(asicp_ctx *c, int v, int passes)
{
    c->cells_on = false;
    c->cells_share = 0.0;
    if (v != kFwdVariants - 1 || c->cells_oom || c->recording) return;
    std::vector<int> todo;
    int most = 0;
    double pairs = 0.0, points = 0.0;
    for (int o = 0; o < c->nobj; ++o) {
        most = std::max(most, c->objs[o].M);
        pairs += (double)c->objmeta_h[o].np * c->N * c->objs[o].M;
        if (c->objs[o].cells_built) continue;
        todo.push_back(o);
        points += c->objs[o].M;
    }
    if (most < kCellMinM || most > kCellMaxM) return;
    if (todo.empty()) {
        c->cells_on = !c->cells_slow;
        return;
    }
    c->cells_owed += passes * pairs / kCellRate * c->cells_worth;
    if (c->cells_owed <= 100.0 + points / kCellRatePts) return;
    c->cells_on = true;
    std::vector<CellBuild> builds;
    bool moved = false;
    try {
        std::vector<std::pair<const DevMem *, size_t>> wants;
        std::vector<int> sizes;
        for (int i : todo) {
            sizes.push_back(c->objs[i].M);
            const CellSizes s = cell_sizes(c->objs[i].M);
            wants.push_back({&c->objs[i].nodes, sizeof(int2) * (size_t)s.node_cap});
            wants.push_back({&c->objs[i].leaves, sizeof(int) * (size_t)s.leaf_cap});
        }
        wants.push_back({&c->cellwork, scratch_bytes(sizes)});
        need_room(wants);
        cell_memory(c, c->cellwork, scratch_bytes(sizes), "matching cells' scratch");
        for (int i : todo) {
            ObjBufs &o = c->objs[i];
            const CellSizes s = cell_sizes(o.M);
            const void *was[2] = {o.nodes.p, o.leaves.p};
            cell_memory(c, o.nodes, sizeof(int2) * (size_t)s.node_cap, "matching cells");
            cell_memory(c, o.leaves, sizeof(int) * (size_t)s.leaf_cap, "matching cells");
            moved = moved || o.nodes.p != was[0] || o.leaves.p != was[1];
            CellBuild b{};
            b.R = o.R.as<float4>();
            b.frame = c->frame.as<float4>() + i;
            b.nodes = o.nodes.as<int2>();
            b.leaves = o.leaves.as<int>();
            b.M = o.M;
            b.log_factor = kObjectCells;
            builds.push_back(b);
        }
    } catch (const Err &e) {
        if (e.st != ASICP_ERR_OOM) throw;
        // nothing is kept: the memory is the caller's again, and the table holds no pointer into it
        c->cells_oom = true;
        c->cells_on = false;
        c->cellwork.release();
        for (ObjBufs &o : c->objs) {
            o.nodes.release();
            o.leaves.release();
            o.cells_built = false;
        }
        moved = true;
    }
    if (moved) {
        for (int o = 0; o < c->nobj; ++o) {
            c->objmeta_h[o].nodes = c->objs[o].nodes.as<int2>();
            c->objmeta_h[o].leaves = c->objs[o].leaves.as<int>();
        }
        ck(cudaMemcpyAsync(c->objmeta.p, c->objmeta_h.data(), sizeof(ObjMeta) * c->nobj, cudaMemcpyHostToDevice, c->st),
           "object table");
        ck(cudaStreamSynchronize(c->st), "object table");
    }
    if (!c->cells_on) return;
    build_cells(c, builds);
    for (int o : todo) c->objs[o].cells_built = true;

    // whether they are the faster way for these clouds: weigh_cells() reads the count
    FwdArgs fa{};
    fa.L = c->layout();
    fa.theta = c->theta.as<float>();
    fa.Ssort = c->Ssort.as<float4>();
    if (!c->weights.p) {
        if (!c->weights.ensure(sizeof(CellCost))) return;      // (the cells are taken as they are)
        std::memset(c->weights.p, 0, sizeof(CellCost));
    }
    ck(launch_cells_cost(fa, reinterpret_cast<CellCost *>(c->cellwork.as<int>() + kCellCounters / 2),
                         reinterpret_cast<CellCost *>(c->weights.p), ++c->weight_seq, &c->cells_share, c->st),
       "matching cells");
}

// Read the count that ensure_cells() has enqueued and keep the faster way.  Called after the other preparations of the
// call, which run meanwhile.
void weigh_cells(asicp_ctx *c)
{
    if (c->cells_share == 0.0) return;
    const double share = c->cells_share;
    c->cells_share = 0.0;
    const volatile CellCost *v = reinterpret_cast<const CellCost *>(c->weights.p);
    for (int n = 1; v->seq != c->weight_seq; ++n)
        if (n % 1024 == 0) {               // (an error would leave it unwritten)
            const cudaError_t e = cudaStreamQuery(c->st);
            if (e == cudaErrorNotReady) continue;
            ck(e, "matching cells");
            if (v->seq != c->weight_seq) fail(ASICP_ERR_CUDA, "matching cells: no count");
        }
    std::atomic_thread_fence(std::memory_order_acquire);
    double pairs = 0.0, most = 0.0, us = 0.0;
    for (const ObjMeta &m : c->objmeta_h) {
        pairs += (double)m.np * c->N * m.M;
        most = std::max(most, (double)m.M);
    }
    for (int k = 0; k < 2; ++k)
        us = std::max({us, (double)v->sum[k] / share / kCellRounds, (double)v->most[k] * kCellLatency});
    c->cells_slow = us > kScreenLeast + std::max(pairs / kCellRate, most * kScreenPoint);
    c->cells_worth = c->cells_slow ? kCellDoubt : 1.0;
    c->cells_on = c->cells_on && !c->cells_slow;
}

// Whether the caller's own stream is being captured: the launches of this call run when its graph is replayed,
// each time on the clouds the context then holds.  Nothing they prepare may count as done, and nothing that was
// prepared from the present clouds may be recorded.
void note_capture(asicp_ctx *c)
{
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    // (the default stream cannot be captured)
    if (c->st != nullptr && c->st != cudaStreamLegacy && cudaStreamIsCapturing(c->st, &s) != cudaSuccess) {
        cudaGetLastError();
        s = cudaStreamCaptureStatusNone;
    }
    c->recording = s != cudaStreamCaptureStatusNone;
}

// Sort the collision clouds that are new (in a capture: all of them, at every replay) into their spatial
// order before the kernels run, those of all objects together.
void ensure_sorted(asicp_ctx *c)
{
    CloudBatch batch{};
    int n = 0;
    for (const ObjBufs &o : c->objs) {
        if (o.sorted && !c->recording) continue;
        const float4 *src = o.C.p ? o.C.as<float4>() : o.R.as<float4>();
        for (int seg = 0; seg < o.Mc; seg += kColSegment) {
            batch.b[n++] = {src + seg, o.Csort.as<float4>() + seg, o.Cball.as<float4>() + seg / 32,
                            std::min(kColSegment, o.Mc - seg)};
            if (n == kCloudBatch) {
                ck(launch_sort_clouds(batch, n, c->st), "collision cloud order");
                n = 0;
            }
        }
    }
    if (n > 0) ck(launch_sort_clouds(batch, n, c->st), "collision cloud order");
    if (!c->recording)
        for (ObjBufs &o : c->objs) o.sorted = true;
}

// Decide whether the reverse matching of the next `passes` passes goes through the cells of the
// gripper clouds, and build those (all preshapes together) once the passes so far and to
// come would take longer without them: a pass of collide_nn_kernel takes 5 us more than
// one through the cells, and 1 us per kPreRate pairs, a colliding point in 32 assumed.
constexpr int kPreMinN = 512;
constexpr double kPreRate = 5.7e6;

// Whether the cells hold for colliding points of every object: collide_cells_kernel compares the whole gripper cloud for
// a point whose position is less exact than they allow, which takes five times as long as collide_nn_kernel (4.3e5
// points, N 2048, an object 8 m away or more, gripper radius 7 cm: 1106 us against 217).  Its bound, for a pose at
// the farthest object's centre and any point of the distance field's grid.
bool pre_cells_hold(const asicp_ctx *c)
{
    auto sum = [](float x, float y, float z) { return std::fabs(x) + std::fabs(y) + std::fabs(z); };
    float far = 0.f;
    for (const ObjBufs &o : c->objs) far = std::max(far, sum(o.frame.x, o.frame.y, o.frame.z));
    for (int p = 0; p < c->cfg.P; ++p) {
        const float4 &f = c->preframe_h[p];
        const SdfMeta &m = c->meta[p];
        auto end = [&](float o, int n) { return std::max(std::fabs(o), std::fabs(o + m.voxel * (float)(n - 1))); };
        const float reach = sum(f.x, f.y, f.z) + f.w, x = end(m.ox, m.nx) + end(m.oy, m.ny) + end(m.oz, m.nz);
        if (!(1.2e-6f * (x + reach) + 4e-7f * far <= 0.4f * kGripperTol * f.w)) return false;
    }
    return true;
}

void ensure_pre_cells(asicp_ctx *c, int passes)
{
    c->pre_on = false;
    if (c->pre_oom || c->N < kPreMinN || c->recording || !pre_cells_hold(c)) return;
    const int P = c->cfg.P;
    const size_t list = sizeof(int) * (size_t)std::max<long long>(1, c->colidx_total);
    if (c->pre_built) {
        c->pre_on = list <= c->colsrt.bytes;
        if (c->pre_on) return;
    } else {
        double tests = 0.0;
        for (const ObjMeta &m : c->objmeta_h) tests += (double)m.np * m.Mc;
        c->pre_owed += passes * (5.0 + tests / 32.0 * c->N / kPreRate);
        if (c->pre_owed <= 150.0 + (double)P * c->N / kCellRatePts) return;
    }
    std::vector<CellBuild> builds;
    const CellSizes s = cell_sizes(c->N);
    const size_t nodes = sizeof(int2) * (size_t)s.node_cap * P, leaves = sizeof(int) * (size_t)s.leaf_cap * P;
    try {
        const size_t scratch = c->pre_built ? 0 : scratch_bytes(std::vector<int>(P, c->N));
        need_room({{&c->prenodes, nodes}, {&c->preleaves, leaves}, {&c->colsrt, list}, {&c->cellwork, scratch}});
        cell_memory(c, c->colsrt, list, "colliding points in spatial order");
        if (!c->pre_built) {
            cell_memory(c, c->cellwork, scratch, "gripper cells' scratch");
            cell_memory(c, c->prenodes, nodes, "gripper cells");
            cell_memory(c, c->preleaves, leaves, "gripper cells");
            for (int p = 0; p < P; ++p) {
                CellBuild b{};
                b.R = c->S.as<float4>() + (size_t)p * c->N;
                b.frame = c->preframe.as<float4>() + p;
                b.nodes = c->prenodes.as<int2>() + (size_t)p * s.node_cap;
                b.leaves = c->preleaves.as<int>() + (size_t)p * s.leaf_cap;
                b.M = c->N;
                b.log_factor = kGripperCells;
                b.tol = kGripperTol;
                builds.push_back(b);
            }
        }
    } catch (const Err &e) {
        if (e.st != ASICP_ERR_OOM) throw;
        c->pre_oom = true;
        c->pre_built = false;
        c->prenodes.release();
        c->preleaves.release();
        c->colsrt.release();
        c->cellwork.release();
        return;
    }
    if (!c->pre_built) build_cells(c, builds);
    c->pre_on = c->pre_built = true;
}

// The collision test and the reverse matching of a pass read the poses only, as the forward matching
// does, and write buffers of their own: they run on a second stream beside it, and both are joined
// before the finalize kernel.  With kernel timers the pass is one stream, so that each time is the
// kernel's own.  What is on the second stream is joined also when a launch of the first one fails.
//
// Parting and joining cost about 3 us of a captured pass and 5 us of a direct one.  A captured loop gains
// more where the matching leaves room beside it: the float32 kernels with few queries (32 particles of 256
// points on 512 points, whole search: 2033 -> 1788 us; mini-batch ramp of 32 particles 2594 -> 2150 us) and
// the cells with many (6.3 M queries 4845 -> 4613 us; 1.6 M: 9637 -> 9590 us; but 0.13 M: 1857 -> 1900 us).
// A direct pass gains with many queries only (12.6 M: 1328 -> 1277 us; 0.16 M: 106 -> 111 us).
constexpr long long kPartQueries = 1 << 20;

bool parts(const asicp_ctx *c)
{
    return c->cfg.profile == 0 && ((c->capturing && !c->cells_on) || (long long)c->T * c->N >= kPartQueries);
}

class Branch {
public:
    Branch(asicp_ctx *c, bool on) : c_(c), on_(on)
    {
        if (!on_) return;
        ck(cudaEventRecord(c->parted, work_stream(c)), "part the pass");
        ck(cudaStreamWaitEvent(c->side_st, c->parted, 0), "part the pass");
        open_ = true;
    }
    ~Branch()
    {
        if (open_) (void)close();
    }
    cudaStream_t stream() const { return on_ ? c_->side_st : nullptr; }
    void join()
    {
        if (on_) ck(close(), "join the pass");
    }

private:
    cudaError_t close()
    {
        open_ = false;
        const cudaError_t e = cudaEventRecord(c_->joined, c_->side_st);
        return e == cudaSuccess ? cudaStreamWaitEvent(work_stream(c_), c_->joined, 0) : e;
    }
    asicp_ctx *c_;
    bool on_, open_ = false;
};

// One pass of cost/gradient evaluation (+ update for mode 1/2).
void iterate(asicp_ctx *c, int mode, float gamma, int k)
{
    select_minibatch(c, k);
    const Layout L = c->layout();
    FwdArgs fa{};
    fa.L = L;
    fa.S = c->S.as<float4>();
    fa.theta = c->theta.as<float>();
    fa.items = c->items.as<FwdItem>();
    fa.cta_off = c->ctaoff.as<int>();
    fa.n_items = c->n_items;
    fa.err = c->errw.as<int>();
    fa.nn_idx = c->nnidx.as<int>();
    fa.cand = c->tccand.as<int4>();
    fa.variant = c->fwd_variant;
    fa.Ssort = c->Ssort.as<float4>();
    fa.cells = c->cells_on;
    fa.expire_test = c->expire_test ? 1 : 0;
    if (c->cfg.debug) {
        fa.dbg_d2 = c->dbg_d2.as<float>();
        fa.dbg_sp = c->dbg_sp.as<float>();
    }
    Branch side(c, parts(c));
    timed(c, kTimeMatch, [&](cudaStream_t st) { return launch_fwd_match(fa, st); }, "forward matching kernel");
    if (fwd_has_exact_kernel(fa))
        timed(c, kTimeExact, [&](cudaStream_t st) { return launch_fwd_exact(fa, st); }, "exact choice kernel");

    CollideArgs ca{};
    ca.L = L;
    ca.theta = c->theta.as<float>();
    ca.meta = c->dmeta.as<SdfMeta>();
    ca.S = c->S.as<float4>();
    ca.ncol = c->ncol.as<int>();
    ca.colidx = c->colidx.as<int>();
    ca.colnn = c->colnn.as<int>();
    ca.colmap = c->colmap.as<int2>();
    ca.col_items = c->colitems.as<int>();
    ca.col_list = c->collist.as<int>();
    for (const ObjMeta &m : c->objmeta_h) ca.most_points = std::max(ca.most_points, m.Mc);
    ca.cells = c->pre_on;
    ca.colsrt = ca.cells ? c->colsrt.as<int>() : ca.colnn;
    if (ca.cells) {
        const CellSizes s = cell_sizes(c->N);
        ca.pre_nodes = c->prenodes.as<int2>();
        ca.pre_leaves = c->preleaves.as<int>();
        ca.pre_frame = c->preframe.as<float4>();
        ca.pre_node_cap = s.node_cap;
        ca.pre_leaf_cap = s.leaf_cap;
        ca.most_items = (int)std::min<long long>(std::max<long long>(1, c->colmap_total), INT_MAX);
    }
    timed(c, kTimeCollide, [&](cudaStream_t st) { return launch_collide(ca, st); }, "collision kernel", side.stream());
    timed(c, kTimeCollideNN, [&](cudaStream_t st) { return launch_collide_nn(ca, st); }, "collision matching kernel",
          side.stream());
    side.join();

    UpdateArgs ua{};
    ua.L = L;
    ua.theta = c->theta.as<float>();
    ua.S = c->S.as<float4>();
    ua.nn_idx = c->nnidx.as<int>();
    ua.colidx = c->colidx.as<int>();
    ua.colnn = c->colnn.as<int>();
    ua.ncol = c->ncol.as<int>();
    ua.pconst = c->pconst.as<double>();
    ua.w_com = c->cfg.w_com;
    ua.mode = mode;
    ua.gamma = gamma;
    ua.eta_svgd = c->cfg.eta_svgd > 0.f ? c->cfg.eta_svgd : 1.f / (float)c->N;
    ua.eta_sgd = c->cfg.eta_sgd;
    ua.bandwidth_mode = c->cfg.bandwidth_mode;
    ua.h_fixed = c->cfg.h_fixed;
    ua.conv_tol = c->cfg.conv_tol;
    ua.cost = c->cost.as<double>();
    ua.grad = c->grad.as<double>();
    ua.prev_cost = c->prev.as<double>();
    ua.frozen = c->frozen.as<int>();
    ua.phi = c->phi.as<float>();
    ua.h = c->h.as<float>();
    ua.col_items = c->colitems.as<int>();
    ua.err = c->errw.as<int>();
    ua.prior_t_sigma = c->cfg.prior_t_sigma;
    ua.prior_q_kappa = c->cfg.prior_q_kappa;
    {
        const float *m = c->cfg.prior_q_mean;
        const double n =
            std::sqrt((double)m[0] * m[0] + (double)m[1] * m[1] + (double)m[2] * m[2] + (double)m[3] * m[3]);
        for (int a = 0; a < 4; ++a) ua.prior_q_mean[a] = n > 0.0 ? (float)(m[a] / n) : (a == 0 ? 1.f : 0.f);
    }
    timed(c, kTimeFinalize, [&](cudaStream_t st) { return launch_finalize(ua, st); }, "finalize kernel");
    if (mode == 1)
        timed(c, kTimeStein, [&](cudaStream_t st) { return launch_stein(ua, st); }, "Stein kernel");
}

void step_impl(asicp_ctx *c, int k)
{
    const int mode = k < c->cfg.k_stein ? 1 : 2;
    iterate(c, mode, (float)gamma_of(c->cfg, k), k);
    c->k_next = k + 1;
    c->stepped = true;
}

// Everything asicp_run does after the initial poses: convergence reset, k_max
// iterations, final evaluation and ranking.
void run_loop(asicp_ctx *c)
{
    reset_convergence(c);
    for (int k = 0; k < c->cfg.k_max; ++k) step_impl(c, k);
    iterate(c, 0, 0.f, -1);   // final evaluation at the last poses (whole object cloud)
    ck(launch_select(c->layout(), c->cost.as<double>(), c->ncol.as<int>(), c->order.as<int>(), work_stream(c)),
       "select");
}

// Buffers and sizes the captured graph depends on (the tables they hold are
// read at replay, so new objects of the same sizes reuse the graph).
std::vector<const void *> loop_key(const asicp_ctx *c)
{
    return {c->partgrp.p, c->grpoff.p, c->objmeta.p, c->items.p, c->ctaoff.p, c->com.p, c->frame.p, c->colitems.p, c->collist.p,
            c->S.p, c->pconst.p, c->dmeta.p, c->theta.p, c->ncol.p, c->colidx.p, c->colsrt.p, c->colnn.p, c->colmap.p, c->cost.p,
            c->grad.p, c->prev.p, c->frozen.p, c->phi.p, c->h.p, c->order.p, c->errw.p, c->nnidx.p, c->tccand.p, c->dbg_d2.p,
            c->dbg_sp.p, c->mb_idx.p, c->mb_R.p, c->mb_Rx.p,
            reinterpret_cast<const void *>((size_t)c->T),
            reinterpret_cast<const void *>((size_t)c->G), reinterpret_cast<const void *>((size_t)c->n_items),
            reinterpret_cast<const void *>((size_t)c->N), reinterpret_cast<const void *>((size_t)c->fwd_variant),
            reinterpret_cast<const void *>((size_t)c->expire_test), c->Ssort.p,
            reinterpret_cast<const void *>((size_t)c->cells_on), c->prenodes.p, c->preleaves.p, c->preframe.p,
            reinterpret_cast<const void *>((size_t)c->pre_on), reinterpret_cast<const void *>((size_t)c->colmap_total)};
}

// Replay the captured loop on the caller's stream, capturing it first when the
// buffers changed.  Kernel arguments (buffer pointers, per-iteration gamma) are
// fixed at capture; the buffers' contents are read at replay.
void run_loop_graph(asicp_ctx *c)
{
    std::vector<const void *> key = loop_key(c);
    // (mini-batches: their sizes and the object's entry are in the graph, the indices are read at replay)
    const bool same_mb = c->mb_off == c->loop_mb &&
                         (c->mb_off.empty() || std::memcmp(&c->loop_meta, &c->objmeta_h[0], sizeof(ObjMeta)) == 0);
    if (!c->loop_exec || key != c->loop_key || !same_mb) {
        if (c->loop_exec) {
            cudaGraphExecDestroy(c->loop_exec);
            c->loop_exec = nullptr;
        }
        for (auto &e : c->graph_events) { c->pool.push_back(e.a); c->pool.push_back(e.b); }
        c->graph_events.clear();
        c->graph_pending = false;
        if (!c->cap_st) ck(cudaStreamCreateWithFlags(&c->cap_st, cudaStreamNonBlocking), "capture stream");
        ck(cudaStreamBeginCapture(c->cap_st, cudaStreamCaptureModeThreadLocal), "begin capture");
        c->capturing = true;
        cudaGraph_t g = nullptr;
        try {
            run_loop(c);
        } catch (...) {
            c->capturing = false;
            cudaStreamEndCapture(c->cap_st, &g);
            if (g) cudaGraphDestroy(g);
            throw;
        }
        c->capturing = false;
        ck(cudaStreamEndCapture(c->cap_st, &g), "end capture");
        cudaError_t e = cudaGraphInstantiate(&c->loop_exec, g, 0);
        cudaGraphDestroy(g);
        ck(e, "instantiate graph");
        c->loop_key = key;
        c->loop_mb = c->mb_off;
        c->loop_meta = c->objmeta_h[0];
    }
    accumulate_graph_events(c);
    ck(cudaGraphLaunch(c->loop_exec, c->st), "graph launch");
    if (!c->mb_off.empty()) c->table_mb = false;     // (the loop ends on the whole cloud)
    c->graph_pending = c->cfg.profile != 0;
}

__global__ void repack_kernel(const float *src8, int n, float *dst7)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int a = 0; a < 7; ++a) dst7[(size_t)i * 7 + a] = src8[(size_t)i * 8 + a];
}

__global__ void repack_f64_kernel(const double *src8, int n, double *dst7)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int a = 0; a < 7; ++a) dst7[(size_t)i * 7 + a] = src8[(size_t)i * 8 + a];
}

__global__ void gather_best_kernel(const int *order, int first, int n, const int *part_grp, int P, const float *theta8,
                                   const double *cost, float *o7, float *oc, int *oi)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int i = order[first + r];
    for (int a = 0; a < 7; ++a) o7[(size_t)r * 7 + a] = theta8[(size_t)i * 8 + a];
    oc[r] = (float)cost[i];
    oi[r] = part_grp[i] % P;
}

// Time every forward-matching kernel shape on the context's current work (poses
// as they are) and keep the fastest.  ms[v] receives the mean launch time.
void autotune_impl(asicp_ctx *c, float *ms_out)
{
    const int reps = 3;
    cudaEvent_t e0 = c->take_event(), e1 = c->take_event();
    float best = 0.f;
    int best_v = 0;
    for (int v = 0; v < kFwdVariants; ++v) {
        if (v == 7 && !c->mb_off.empty()) {   // the tensor-core kernel has no mini-batch tiles
            if (ms_out) ms_out[v] = 0.f;
            continue;
        }
        plan_fwd_items(c, v);
        FwdArgs fa{};
        fa.L = c->layout();
        fa.S = c->S.as<float4>();
        fa.theta = c->theta.as<float>();
        fa.items = c->items.as<FwdItem>();
        fa.cta_off = c->ctaoff.as<int>();
        fa.n_items = c->n_items;
        fa.err = c->errw.as<int>();
        fa.nn_idx = c->nnidx.as<int>();
        fa.cand = c->tccand.as<int4>();
        fa.variant = v;
        ensure_cells(c, v, c->cfg.k_max + 1);
        weigh_cells(c);
        fa.Ssort = c->Ssort.as<float4>();
        fa.cells = c->cells_on;
        ck(launch_fwd_match(fa, c->st), "autotune warm-up");
        if (fwd_has_exact_kernel(fa)) ck(launch_fwd_exact(fa, c->st), "autotune warm-up");
        ck(cudaEventRecord(e0, c->st), "cudaEventRecord");
        for (int r = 0; r < reps; ++r) {
            ck(launch_fwd_match(fa, c->st), "autotune launch");
            if (fwd_has_exact_kernel(fa)) ck(launch_fwd_exact(fa, c->st), "autotune launch");
        }
        ck(cudaEventRecord(e1, c->st), "cudaEventRecord");
        ck(cudaEventSynchronize(e1), "cudaEventSynchronize");
        float t = 0.f;
        ck(cudaEventElapsedTime(&t, e0, e1), "cudaEventElapsedTime");
        t /= reps;
        if (ms_out) ms_out[v] = t;
        if (v == 0 || t < best) { best = t; best_v = v; }
    }
    c->pool.push_back(e0);
    c->pool.push_back(e1);
    finish(c, "autotune");
    c->fwd_variant = best_v;
    plan_fwd_items(c, best_v);
    c->tuned = true;
}

void set_object_impl(asicp_ctx *ctx, int o, const float *R_xyz, int M, const float *C_xyz, int Mc)
{
    if (o < 0 || o >= ctx->nobj) fail(ASICP_ERR_INVALID_ARG, "set_object: object index out of range");
    if (!R_xyz || M < 1) fail(ASICP_ERR_INVALID_ARG, "set_object: R must be non-NULL with M >= 1");
    if (C_xyz && Mc < 1) fail(ASICP_ERR_INVALID_ARG, "set_object: Mc must be >= 1 when C is given");
    ObjBufs &b = ctx->objs[o];
    const int mc = C_xyz ? Mc : M;
    drop_minibatches(ctx);        // they index the previous cloud
    // what the layout (object table, work plan) and the captured loop depend on
    const bool was_set = b.set;
    const void *was[6] = {b.R.p, b.Rx.p, b.Rt.p, b.C.p, b.Csort.p, b.Cball.p};
    const int was_M = b.M, was_Mc = b.Mc, was_Mpad = b.Mpad;
    b.set = false;
    b.cells_built = b.sorted = false;
    ctx->cells_owed = 0.0;
    ctx->run_done = false;
    ctx->stage.ensure(sizeof(float) * 3 * (size_t)(M > mc ? M : mc), "staging");
    b.R.ensure(sizeof(float4) * M, "object cloud");
    upload(ctx, ctx->stage.p, R_xyz, sizeof(float) * 3 * (size_t)M, "copy R");
    const int Mpad = (M + kRefTilePts - 1) / kRefTilePts * kRefTilePts;
    b.Rx.ensure(sizeof(float4) * (size_t)Mpad, "screening layout");
    ck(launch_ref_prep(ctx->stage.as<float>(), M, Mpad, b.R.as<float4>(), b.Rx.p, ctx->frame.as<float4>() + o,
                       ctx->com.as<double>() + 3 * o, ctx->refscr.as<RefScratch>(), ctx->errw.as<int>(), ctx->st),
       "ref prep");
    if (C_xyz) {
        b.C.ensure(sizeof(float4) * mc, "collision cloud");
        upload(ctx, ctx->stage.p, C_xyz, sizeof(float) * 3 * (size_t)mc, "copy C");
        ck(launch_pack_points(ctx->stage.as<float>(), mc, b.C.as<float4>(), ctx->errw.as<int>(), ctx->st), "pack C");
    } else {
        b.C.release();
    }
    b.Csort.ensure(sizeof(float4) * (size_t)mc, "collision cloud, sorted");
    b.Cball.ensure(sizeof(float4) * (((size_t)mc + 31) / 32), "collision cloud, balls");
    b.Rt.ensure(tc_ref_bytes(Mpad), "tensor-core object tiles");
    ck(launch_tc_ref_prep(b.R.as<float4>(), M, Mpad, ctx->frame.as<float4>() + o, b.Rt.p, ctx->st),
       "tensor-core ref prep");
    copy_out(ctx, &b.frame, ctx->frame.as<float4>() + o, sizeof(float4));
    finish(ctx, "set_object");
    b.M = M;
    b.Mpad = Mpad;
    b.Mc = mc;
    b.set = true;
    // a new object of the same sizes in the same buffers keeps the layout, the poses
    // and the captured loop (whose kernels read the object's data at replay)
    if (!was_set || M != was_M || mc != was_Mc || Mpad != was_Mpad || b.R.p != was[0] || b.Rx.p != was[1] ||
        b.Rt.p != was[2] || b.C.p != was[3] || b.Csort.p != was[4] || b.Cball.p != was[5])
        ctx->layout_dirty = true;
}

}  // namespace

// ---------------------------------------------------------------------- ABI
extern "C" {

void asicp_config_default(asicp_config *cfg)
{
    if (!cfg) return;
    std::memset(cfg, 0, sizeof(*cfg));
    cfg->P = 1;
    cfg->K = 32;
    cfg->k_max = 40;
    cfg->k_stein = 15;          // Table I: 15 SVGD + 25 SGD iterations
    cfg->schedule = 0;
    cfg->C_cycles = 5.f;        // Table I annealing factor (mod(k, k_max/5) / (k_max/5))^2
    cfg->p_exp = 2.f;
    cfg->g0 = 0.1f;
    cfg->g1 = 1.f;
    cfg->eta_sgd = 1.f;         // Table I learning rate
    cfg->eta_svgd = 0.f;        // 1/N
    cfg->w_com = 1.f;           // Table I cost weights
    cfg->bandwidth_mode = 0;
    cfg->h_fixed = 1.f;
    cfg->conv_tol = 2e-4f;      // Table I convergence criterion 0.02 %
    cfg->init_radius = 0.15f;
    cfg->debug = 0;
    cfg->profile = 0;
    cfg->cuda_stream = nullptr;
    cfg->n_objects = 1;
    cfg->autotune = 0;
    cfg->fwd_shape = 0;
}

asicp_status asicp_create(const asicp_config *cfg, asicp_ctx **out)
{
    if (!cfg || !out) return ASICP_ERR_INVALID_ARG;
    *out = nullptr;
    if (cfg->P < 1 || cfg->P > 64 || cfg->K < 1 || cfg->K > kMaxK || cfg->k_max < 0 || cfg->k_stein < 0 ||
        cfg->k_stein > cfg->k_max || (cfg->schedule != 0 && cfg->schedule != 1) ||
        (cfg->schedule == 0 && !(cfg->C_cycles > 0.f)) || !(cfg->eta_sgd >= 0.f) ||
        (cfg->bandwidth_mode == 1 && !(cfg->h_fixed > 0.f)) || !std::isfinite(cfg->w_com) ||
        !(cfg->init_radius >= 0.f) || cfg->n_objects < 1 || cfg->n_objects > 4096 ||
        cfg->fwd_shape < 0 || cfg->fwd_shape >= kFwdVariants || cfg->init_mode < 0 || cfg->init_mode > 1 ||
        !std::isfinite(cfg->prior_t_sigma) || !std::isfinite(cfg->prior_q_kappa) ||
        (cfg->prior_q_kappa > 0.f && !(std::fabs(cfg->prior_q_mean[0]) + std::fabs(cfg->prior_q_mean[1]) +
                                       std::fabs(cfg->prior_q_mean[2]) + std::fabs(cfg->prior_q_mean[3]) > 0.f)))
        return ASICP_ERR_INVALID_ARG;
    asicp_ctx *c = new (std::nothrow) asicp_ctx();
    if (!c) return ASICP_ERR_OOM;
    c->cfg = *cfg;
    c->st = static_cast<cudaStream_t>(cfg->cuda_stream);
    c->nobj = cfg->n_objects;
    c->fwd_variant = cfg->fwd_shape;
    c->pre_set.assign(cfg->P, 0);
    c->meta.assign(cfg->P, SdfMeta{});
    c->grids.resize(cfg->P);
    c->cells.resize(cfg->P);
    c->clear.resize(cfg->P);
    c->preframe_h.assign(cfg->P, float4{});
    c->objs.resize(c->nobj);
    c->Kg.assign((size_t)c->nobj * cfg->P, cfg->K);
    asicp_status s = guarded(c, [&] {
        // one-time kernel attributes, set outside any graph capture
        fwd_grid_size();
        ck(cudaStreamCreateWithFlags(&c->side_st, cudaStreamNonBlocking), "side stream");
        ck(cudaEventCreateWithFlags(&c->parted, cudaEventDisableTiming), "side stream event");
        ck(cudaEventCreateWithFlags(&c->joined, cudaEventDisableTiming), "side stream event");
        ck(init_collision_attributes(), "collision kernel attributes");
        ck(init_update_attributes(), "update kernel attributes");
        ck(init_cells_attributes(), "cell kernel attributes");
        c->com.ensure(sizeof(double) * 3 * c->nobj, "com");
        c->frame.ensure(sizeof(float4) * c->nobj, "screening frames");
        c->pconst.ensure(sizeof(double) * 12 * cfg->P, "pconst");
        c->dmeta.ensure(sizeof(SdfMeta) * cfg->P, "sdf meta");
        c->refscr.ensure(sizeof(RefScratch), "object preparation");
        ck(cudaMemsetAsync(c->refscr.p, 0, sizeof(RefScratch), c->st), "clear object preparation");
        c->errw.ensure(sizeof(int), "error word");
        ck(cudaMemsetAsync(c->errw.p, 0, sizeof(int), c->st), "clear error word");
        ck(cudaStreamSynchronize(c->st), "create");
    });
    if (s != ASICP_OK) {
        delete c;
        return s;
    }
    *out = c;
    return ASICP_OK;
}

asicp_status asicp_destroy(asicp_ctx *ctx)
{
    if (!ctx) return ASICP_OK;
    cudaStreamSynchronize(ctx->st);
    delete ctx;
    return ASICP_OK;
}

asicp_status asicp_set_object(asicp_ctx *ctx, const float *R_xyz, int M, const float *C_xyz, int Mc)
{
    return guarded(ctx, [&] { set_object_impl(ctx, 0, R_xyz, M, C_xyz, Mc); });
}

asicp_status asicp_set_object_at(asicp_ctx *ctx, int object, const float *R_xyz, int M, const float *C_xyz, int Mc)
{
    return guarded(ctx, [&] { set_object_impl(ctx, object, R_xyz, M, C_xyz, Mc); });
}

asicp_status asicp_set_particle_counts(asicp_ctx *ctx, const int *K, int n)
{
    return guarded(ctx, [&] {
        if (!K || n != ctx->nobj * ctx->cfg.P)
            fail(ASICP_ERR_INVALID_ARG, "set_particle_counts: need n_objects * P counts");
        std::vector<int> k(n);
        ck(cudaMemcpy(k.data(), K, sizeof(int) * n, cudaMemcpyDefault), "copy particle counts");
        for (int v : k)
            if (v < 1 || v > kMaxK) fail(ASICP_ERR_INVALID_ARG, "set_particle_counts: every count must be in [1, 1024]");
        ctx->Kg = k;
        ctx->layout_dirty = true;
        ctx->theta_set = false;
        ctx->run_done = false;
    });
}

asicp_status asicp_set_minibatch(asicp_ctx *ctx, const int *offsets, const int *indices, int iters)
{
    return guarded(ctx, [&] {
        if (!offsets) {
            drop_minibatches(ctx);
            return;
        }
        if (ctx->nobj != 1) fail(ASICP_ERR_INVALID_ARG, "set_minibatch: one object per context");
        if (!ctx->objs[0].set) fail(ASICP_ERR_STATE, "set_minibatch: set the object first");
        if (!indices || iters < 1) fail(ASICP_ERR_INVALID_ARG, "set_minibatch: NULL indices or iters < 1");
        if (ctx->fwd_variant == 7) fail(ASICP_ERR_INVALID_ARG, "set_minibatch: not with the tensor-core kernel shape");
        const int M = ctx->objs[0].M;
        std::vector<int> off(iters + 1);
        ck(cudaMemcpy(off.data(), offsets, sizeof(int) * (iters + 1), cudaMemcpyDefault), "copy mini-batch offsets");
        if (off[0] != 0) fail(ASICP_ERR_INVALID_ARG, "set_minibatch: offsets must start at 0");
        for (int k = 0; k < iters; ++k)
            if (off[k + 1] - off[k] < 1 || off[k + 1] - off[k] > M)
                fail(ASICP_ERR_INVALID_ARG, "set_minibatch: every mini-batch needs 1..M points");
        std::vector<int> idx(off[iters]);
        ck(cudaMemcpy(idx.data(), indices, sizeof(int) * idx.size(), cudaMemcpyDefault), "copy mini-batch indices");
        for (int k = 0; k < iters; ++k)
            for (int i = off[k]; i < off[k + 1]; ++i)
                if (idx[i] < 0 || idx[i] >= M || (i > off[k] && idx[i] <= idx[i - 1]))
                    fail(ASICP_ERR_INVALID_ARG, "set_minibatch: indices must be ascending within [0, M)");
        const int Mpad = (M + kRefTilePts - 1) / kRefTilePts * kRefTilePts;
        drop_minibatches(ctx);    // (growing the buffers may fail: the old ramp must not outlive them)
        ctx->mb_idx.ensure(sizeof(int) * idx.size(), "mini-batch indices");
        ctx->mb_R.ensure(sizeof(float4) * M, "mini-batch points");
        ctx->mb_Rx.ensure(sizeof(float4) * Mpad, "mini-batch screening layout");
        upload(ctx, ctx->mb_idx.p, idx.data(), sizeof(int) * idx.size(), "upload indices");
        ck(cudaStreamSynchronize(ctx->st), "upload indices");
        ctx->pin_busy = false;
        ctx->mb_off = off;
        ctx->run_done = false;
    });
}

asicp_status asicp_set_gripper_sdf(asicp_ctx *ctx, int preshape, const float *S_xyz, int N, const float *sdf,
                                   int nx, int ny, int nz, const float origin[3], float voxel)
{
    return guarded(ctx, [&] {
        if (preshape < 0 || preshape >= ctx->cfg.P) fail(ASICP_ERR_INVALID_ARG, "set_gripper_sdf: preshape out of range");
        if (!S_xyz || !sdf || !origin) fail(ASICP_ERR_INVALID_ARG, "set_gripper_sdf: NULL array");
        if (N < 1 || N > kMaxN) fail(ASICP_ERR_INVALID_ARG, "set_gripper_sdf: N must be in [1, 6144]");
        if (nx < 2 || ny < 2 || nz < 2) fail(ASICP_ERR_INVALID_ARG, "set_gripper_sdf: every grid dimension must be >= 2");
        if (!(voxel > 0.f) || !std::isfinite(voxel)) fail(ASICP_ERR_INVALID_ARG, "set_gripper_sdf: voxel must be > 0");
        float org[3];
        ck(cudaMemcpy(org, origin, sizeof(org), cudaMemcpyDefault), "copy origin");
        for (float o : org)
            if (!std::isfinite(o)) fail(ASICP_ERR_INVALID_ARG, "set_gripper_sdf: non-finite origin");
        bool any_set = false;
        for (char s : ctx->pre_set) any_set = any_set || s;
        if (any_set && N != ctx->N) fail(ASICP_ERR_INVALID_ARG, "set_gripper_sdf: every preshape must have the same N");
        if (N != ctx->N) {
            ctx->N = N;
            ctx->layout_dirty = true;
        }
        ctx->pre_set[preshape] = 0;
        ctx->run_done = false;
        ctx->S.ensure(sizeof(float4) * (size_t)ctx->cfg.P * N, "gripper clouds");
        // (room for the clearances' intermediate grids too: growing the buffer between them waits for the device)
        const size_t nc = sdf_cells_bytes(nx, ny, nz) / (2 * sizeof(float4));
        ctx->stage.ensure(std::max(sizeof(float) * 3 * (size_t)N, nc), "staging");
        ck(cudaMemcpyAsync(ctx->stage.p, S_xyz, sizeof(float) * 3 * (size_t)N, cudaMemcpyDefault, ctx->st), "copy S");
        float4 *Sp = ctx->S.as<float4>() + (size_t)preshape * N;
        ck(launch_pack_points(ctx->stage.as<float>(), N, Sp, ctx->errw.as<int>(), ctx->st), "pack S");
        ctx->Ssort.ensure(sizeof(float4) * (size_t)ctx->cfg.P * N, "gripper clouds, sorted");
        ctx->preframe.ensure(sizeof(float4) * ctx->cfg.P, "gripper frames");
        ck(launch_gripper_cloud(Sp, N, ctx->Ssort.as<float4>() + (size_t)preshape * N, ctx->preframe.as<float4>() + preshape,
                                ctx->pconst.as<double>() + 12 * preshape, ctx->st), "gripper cloud");
        ctx->pre_built = false;
        ctx->pre_owed = 0.0;
        const size_t nv = (size_t)nx * ny * nz;
        ctx->grids[preshape].ensure(sizeof(float) * nv, "sdf grid");
        ck(cudaMemcpyAsync(ctx->grids[preshape].p, sdf, sizeof(float) * nv, cudaMemcpyDefault, ctx->st), "copy sdf");
        ck(launch_check_finite(ctx->grids[preshape].as<float>(), (long long)nv, ctx->errw.as<int>(), ctx->st), "check sdf");
        ctx->cells[preshape].ensure(sdf_cells_bytes(nx, ny, nz), "corner-packed sdf grid");
        // (S has been packed: the staging buffer is free again)
        ck(launch_sdf_pack_cells(ctx->grids[preshape].as<float>(), nx, ny, nz, ctx->cells[preshape].as<float4>(),
                                 ctx->stage.as<unsigned char>(), ctx->st), "pack sdf cells");
        ctx->clear[preshape].ensure(nc, "sdf clearances");
        ck(launch_sdf_clear(nx, ny, nz, ctx->stage.as<unsigned char>(), ctx->clear[preshape].as<unsigned char>(), ctx->st),
           "sdf clearances");
        copy_out(ctx, &ctx->preframe_h[preshape], ctx->preframe.as<float4>() + preshape, sizeof(float4));
        finish(ctx, "set_gripper_sdf");
        SdfMeta m{};
        m.grid = ctx->grids[preshape].as<float>();
        m.cells = ctx->cells[preshape].as<float4>();
        m.clear = ctx->clear[preshape].as<unsigned char>();
        m.nx = nx; m.ny = ny; m.nz = nz;
        m.ox = org[0]; m.oy = org[1]; m.oz = org[2];
        m.voxel = voxel;
        ctx->meta[preshape] = m;
        ck(cudaMemcpyAsync(ctx->dmeta.as<SdfMeta>() + preshape, &ctx->meta[preshape], sizeof(SdfMeta),
                           cudaMemcpyHostToDevice, ctx->st), "copy sdf meta");
        ck(cudaStreamSynchronize(ctx->st), "set_gripper_sdf");
        ctx->pre_set[preshape] = 1;
    });
}

asicp_status asicp_set_state(asicp_ctx *ctx, const float *theta, int k)
{
    return guarded(ctx, [&] {
        if (!ctx->inputs_ready()) fail(ASICP_ERR_STATE, "set_state: objects and every preshape must be set first");
        if (!theta || k < 0 || k > ctx->cfg.k_max) fail(ASICP_ERR_INVALID_ARG, "set_state: bad theta or k");
        build_layout(ctx);
        const size_t T = ctx->T;
        ctx->stage.ensure(sizeof(float) * 7 * T, "staging");
        upload(ctx, ctx->stage.p, theta, sizeof(float) * 7 * T, "copy theta");
        ck(launch_set_theta(ctx->stage.as<float>(), (int)T, ctx->theta.as<float>(), ctx->errw.as<int>(), ctx->st),
           "set theta");
        reset_convergence(ctx);
        finish(ctx, "set_state");
        ctx->k_next = k;
        ctx->theta_set = true;
        ctx->stepped = false;
        ctx->run_done = false;
    });
}

asicp_status asicp_set_convergence(asicp_ctx *ctx, const double *prev_cost, const int *frozen)
{
    return guarded(ctx, [&] {
        if (!ctx->theta_set || ctx->layout_dirty) fail(ASICP_ERR_STATE, "set_convergence: set the poses first");
        const size_t T = ctx->T;
        if (prev_cost)
            ck(cudaMemcpyAsync(ctx->prev.p, prev_cost, sizeof(double) * T, cudaMemcpyDefault, ctx->st),
               "copy prev_cost");
        if (frozen)
            ck(cudaMemcpyAsync(ctx->frozen.p, frozen, sizeof(int) * T, cudaMemcpyDefault, ctx->st), "copy frozen");
        ck(cudaStreamSynchronize(ctx->st), "set_convergence");
    });
}

asicp_status asicp_step(asicp_ctx *ctx, int k)
{
    return guarded(ctx, [&] {
        if (!ctx->inputs_ready() || !ctx->theta_set) fail(ASICP_ERR_STATE, "step: inputs and poses must be set first");
        if (ctx->layout_dirty) fail(ASICP_ERR_STATE, "step: inputs changed since the poses were set");
        if (k < 0 || k >= ctx->cfg.k_max) fail(ASICP_ERR_INVALID_ARG, "step: k out of [0, k_max)");
        note_capture(ctx);
        ensure_cells(ctx, ctx->fwd_variant, 1);
        ensure_pre_cells(ctx, 1);
        ensure_sorted(ctx);
        weigh_cells(ctx);
        step_impl(ctx, k);
        ctx->run_done = false;
    });
}

asicp_status asicp_run(asicp_ctx *ctx, const float *theta0)
{
    return guarded(ctx, [&] {
        if (!ctx->inputs_ready()) fail(ASICP_ERR_STATE, "run: objects and every preshape must be set first");
        build_layout(ctx);
        const int T = ctx->T;
        if (theta0) {
            ctx->stage.ensure(sizeof(float) * 7 * T, "staging");
            upload(ctx, ctx->stage.p, theta0, sizeof(float) * 7 * (size_t)T, "copy theta0");
            ck(launch_set_theta(ctx->stage.as<float>(), T, ctx->theta.as<float>(), ctx->errw.as<int>(), ctx->st),
               "set theta0");
            finish(ctx, "run");
        } else {
            ck(launch_fibonacci(ctx->layout(), ctx->cfg.init_radius, ctx->cfg.init_mode, ctx->theta.as<float>(),
                                ctx->st),
               "initial poses");
        }
        ctx->theta_set = true;
        note_capture(ctx);
        if (ctx->cfg.autotune && !ctx->tuned) autotune_impl(ctx, nullptr);
        ensure_cells(ctx, ctx->fwd_variant, ctx->cfg.k_max + 1);
        ensure_pre_cells(ctx, ctx->cfg.k_max + 1);
        ensure_sorted(ctx);
        weigh_cells(ctx);
        run_loop_graph(ctx);
        ctx->k_next = ctx->cfg.k_max;
        ctx->stepped = true;
        ctx->run_done = true;
    });
}

asicp_status asicp_best_grasps_at(asicp_ctx *ctx, int object, int topk, float *theta, float *cost, int *preshape,
                                  int *n_out)
{
    return guarded(ctx, [&] {
        if (!ctx->run_done) fail(ASICP_ERR_STATE, "best_grasps: no completed run");
        if (topk < 0) fail(ASICP_ERR_INVALID_ARG, "best_grasps: topk < 0");
        if (object < 0 || object >= ctx->nobj) fail(ASICP_ERR_INVALID_ARG, "best_grasps: object index out of range");
        const ObjMeta &om = ctx->objmeta_h[object];
        const int n = topk < om.np ? topk : om.np;
        if (n > 0) {
            gather_best_kernel<<<(n + 127) / 128, 128, 0, ctx->st>>>(ctx->order.as<int>(), om.pfirst, n,
                                                                     ctx->partgrp.as<int>(), ctx->cfg.P,
                                                                     ctx->theta.as<float>(), ctx->cost.as<double>(),
                                                                     ctx->out7.as<float>(), ctx->outc.as<float>(),
                                                                     ctx->outi.as<int>());
            ck(cudaGetLastError(), "gather best");
            copy_out(ctx, theta, ctx->out7.p, sizeof(float) * 7 * n);
            copy_out(ctx, cost, ctx->outc.p, sizeof(float) * n);
            copy_out(ctx, preshape, ctx->outi.p, sizeof(int) * n);
        }
        finish(ctx, "best_grasps");
        if (n_out) *n_out = n;
    });
}

asicp_status asicp_best_grasps(asicp_ctx *ctx, int topk, float *theta, float *cost, int *preshape, int *n_out)
{
    return asicp_best_grasps_at(ctx, 0, topk, theta, cost, preshape, n_out);
}

asicp_status asicp_get_state(asicp_ctx *ctx, const asicp_state_view *v)
{
    return guarded(ctx, [&] {
        if (!v) fail(ASICP_ERR_INVALID_ARG, "get_state: NULL view");
        if (!ctx->theta_set) fail(ASICP_ERR_STATE, "get_state: no poses yet");
        const bool dbg = v->nn_idx || v->nn_d2 || v->s_prime || v->col_list || v->col_nn;
        if (dbg && !ctx->cfg.debug) fail(ASICP_ERR_STATE, "get_state: debug arrays need config.debug = 1");
        const int T = ctx->T;
        if (!(ctx->stepped || ctx->run_done) && (v->cost || v->ncol || v->h || dbg))
            fail(ASICP_ERR_STATE, "get_state: no step has run since the poses were set");
        if (v->theta) {
            repack_kernel<<<(T + 127) / 128, 128, 0, ctx->st>>>(ctx->theta.as<float>(), T, ctx->out7.as<float>());
            ck(cudaGetLastError(), "repack theta");
        }
        if (v->phi) {
            ctx->outp.ensure(sizeof(float) * 7 * T, "phi");
            repack_kernel<<<(T + 127) / 128, 128, 0, ctx->st>>>(ctx->phi.as<float>(), T, ctx->outp.as<float>());
            ck(cudaGetLastError(), "repack phi");
        }
        if (v->grad) {
            ctx->outg.ensure(sizeof(double) * 7 * T, "gradient");
            repack_f64_kernel<<<(T + 127) / 128, 128, 0, ctx->st>>>(ctx->grad.as<double>(), T, ctx->outg.as<double>());
            ck(cudaGetLastError(), "repack grad");
        }
        copy_out(ctx, v->theta, ctx->out7.p, sizeof(float) * 7 * T);
        copy_out(ctx, v->phi, ctx->outp.p, sizeof(float) * 7 * T);
        copy_out(ctx, v->grad, ctx->outg.p, sizeof(double) * 7 * T);
        copy_out(ctx, v->cost, ctx->cost.p, sizeof(double) * T);
        copy_out(ctx, v->ncol, ctx->ncol.p, sizeof(int) * T);
        copy_out(ctx, v->h, ctx->h.p, sizeof(float) * ctx->G);
        copy_out(ctx, v->frozen, ctx->frozen.p, sizeof(int) * T);
        copy_out(ctx, v->nn_idx, ctx->nnidx.p, sizeof(int) * (size_t)T * ctx->N);
        copy_out(ctx, v->nn_d2, ctx->dbg_d2.p, sizeof(float) * (size_t)T * ctx->N);
        copy_out(ctx, v->s_prime, ctx->dbg_sp.p, sizeof(float) * 3 * (size_t)T * ctx->N);
        copy_out(ctx, v->col_list, ctx->colidx.p, sizeof(int) * (size_t)ctx->colidx_total);
        copy_out(ctx, v->col_nn, ctx->colnn.p, sizeof(int) * (size_t)ctx->colidx_total);
        finish(ctx, "get_state");
    });
}

asicp_status asicp_autotune(asicp_ctx *ctx, int *chosen, float *ms)
{
    return guarded(ctx, [&] {
        if (!ctx->inputs_ready()) fail(ASICP_ERR_STATE, "autotune: objects and every preshape must be set first");
        build_layout(ctx);
        if (!ctx->theta_set) {
            ck(launch_fibonacci(ctx->layout(), ctx->cfg.init_radius, ctx->cfg.init_mode, ctx->theta.as<float>(),
                                ctx->st),
               "initial poses");
            ctx->theta_set = true;
            ctx->stepped = false;
        }
        note_capture(ctx);
        autotune_impl(ctx, ms);
        if (chosen) *chosen = ctx->fwd_variant;
    });
}

asicp_status asicp_test_expire_waits(asicp_ctx *ctx, int on)
{
    return guarded(ctx, [&] { ctx->expire_test = on != 0; });
}

asicp_status asicp_test_fail_cell_memory(asicp_ctx *ctx, int after)
{
    return guarded(ctx, [&] { ctx->fail_cells = after; });
}

asicp_status asicp_kernel_times(asicp_ctx *ctx, double ms[ASICP_KERNEL_KINDS], long long launches[ASICP_KERNEL_KINDS],
                                int reset)
{
    return guarded(ctx, [&] {
        if (!ctx->cfg.profile) fail(ASICP_ERR_STATE, "kernel_times: config.profile is 0");
        ck(cudaStreamSynchronize(ctx->st), "kernel_times");
        accumulate_graph_events(ctx);
        for (auto &e : ctx->events) {
            float t = 0.f;
            ck(cudaEventElapsedTime(&t, e.a, e.b), "cudaEventElapsedTime");
            ctx->acc_ms[e.kind] += t;
            ctx->acc_n[e.kind] += 1;
            ctx->pool.push_back(e.a);
            ctx->pool.push_back(e.b);
        }
        ctx->events.clear();
        for (int i = 0; i < kTimeKinds; ++i) {
            if (ms) ms[i] = ctx->acc_ms[i];
            if (launches) launches[i] = ctx->acc_n[i];
        }
        if (reset)
            for (int i = 0; i < kTimeKinds; ++i) { ctx->acc_ms[i] = 0; ctx->acc_n[i] = 0; }
    });
}

const char *asicp_last_error(const asicp_ctx *ctx)
{
    if (!ctx) return "NULL context";
    return ctx->err.c_str();
}

}  // extern "C"
