// Forward matching through cells: exact nearest neighbours without visiting every
// object point.
//
// The space around an object is divided into cells, and every cell keeps the list of
// the points that can be nearest to some point of the cell.  A query then finds its
// cell and compares the few points of that list with the same exact-form float32
// distance, ties to the lowest index, as the other kernels: the result is the
// lowest-index minimum over the whole cloud.
//
// Which points a cell needs: with p' any object point, the difference
//     |x - p|^2 - |x - p'|^2 = |m - p|^2 - |m - p'|^2 + 2 (x - m).(p' - p)
// is linear in x, so over a cell of centre m and half width h it is at least
//     |m - p|^2 - |m - p'|^2 - 2 h |p - p'|_1,
// and p can be dropped when that is positive: every x of the cell is nearer to p'.
// Distances to the cloud do not enter, so cells far from it stay small lists too.  p'
// runs over the points nearest to the cell's centre and to its eight corners (against
// the centre's alone the lists are 2.5 times as long).  Rounding, u = 2^-24, in
// coordinates relative to the frame centre, B = max |b|, d = |m - p|^2:
//   - float32 evaluation of d, d' and the 1-norm: <= 5 u (d + d') and a factor on h;
//   - the exact-form float32 distances compared later, at any x of the cell (|x - p|^2
//     <= 2 d + 6 h^2): <= 10 u (d + d') + 60 u h^2;
//   - b = fl(r - c), u B per point: <= 4 u B (sqrt d + sqrt d' + 4 h);
//   - a = fl(s' - c) and its conversion to cell coordinates: the cell is taken wider by
//     2^-20 J (far cells 2^-17 of their shell's cube), five times the largest such error.
// The margin is twice the sum, so a dropped point's float32 distance is strictly
// greater than that of a kept one, and comparisons are written so that a NaN keeps
// the point.  Cells (relative to the frame centre, J = 4 * 2^e > 4 B):
//   near   |a| < J:     an 8^3 grid, halved where a list is longer than kLeaf; the 32^3
//                       level is a table, so a query starts there, and below it nodes
//                       of eight children;
//   far    J <= |a| < 64 J: six shells, each the outer 56 cells of a 4^3 grid over twice
//                       the previous cube, halved the same way;
//   beyond, or where a budget ran out: the whole cloud, scanned by the warp together.
// A list that stays above 0.8 of its parent's is not halved further (points on a
// common sphere or plane, float32 resolution far out): its queries scan it as it is.
//
// Measured on GB300 (per pass, against screening and exact choice on the tensor cores): 3 x 256
// particles, N 2048, M 8192 34 us against 783; 3 x 1024, N 4096, M 65536 0.28 ms against 41.4;
// lists of at most 12 points (with one flat grid of queries, which divided each by N: 12 38 us,
// 16 44, 24 46, 32 52, 48 60; at 8 they stop shrinking and the budgets run out).  What bounds the
// matching is the latency of its dependent loads (table, two or three nodes, list, points), all from
// L2 and L1, at half of the issue slots; queries in the gripper
// cloud's own order take 68 us.  The build (ten rounds of few and uneven cells, latency again)
// takes 0.10 ms at 1024 points, 0.27 at 8192, 1.4 at 65536.
#include "cells.cuh"

namespace asicp {

namespace {

constexpr int kLeaf = 12;                  // a list of at most this many points is not halved
constexpr int kNearLevels = 9, kFarLevels = 5;   // halvings at most (near cells: h = J / 4096 at the end)
constexpr int kStartNear = 8;              // the near grid the lists start from
constexpr int kTable = kCellTable, kShells = kCellShells, kFarBase = kCellFarBase;
constexpr int kFixedNodes = kFarBase + kShells * 64;
constexpr int kStartCells = kStartNear * kStartNear * kStartNear + kShells * 64;
constexpr int kStaged = 512;               // parent lists up to this length are staged in shared memory
constexpr int kBatch = 4;                  // points per lane and round
constexpr int kMaskPts = 4096;             // points per warp whose verdicts are kept between the two passes
constexpr int kStartMask = 256;            // words of a warp's mask in the start kernel (65536 points)
constexpr int kIterBits = 10;              // see nearest9
static_assert(kNearLevels - 2 <= kCellSubBits && kFarLevels <= kCellSubBits, "cell coordinates");
constexpr int kInner = kCellInner, kWhole = kCellWhole;
constexpr int kRounds = kNearLevels + 1;   // rounds of the build: the start lists' second pass, then the halvings
// counters: leaf entries, nodes, and per round the cells with short lists (recorded from the
// front of the round's records), with long ones (from the back) and the list entries
enum { kCtrLeaf = 0, kCtrNode = 1, kCtrShort = 2, kCtrLong = kCtrShort + kRounds, kCtrList = kCtrLong + kRounds };
static_assert(kCtrList + kRounds <= kCellCounters, "counters");

__device__ __forceinline__ float sqrt_about(float x)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The rounding bound above, doubled and split into the part of the point and the part of the
// point it is held against: p is dropped when need(p) > 2 h |p - p'|_1 + have(p').  k is
// 5e-7 B, more where positions are less exact (CellBuild::tol).
__device__ __forceinline__ float need_of(float d, float k) { return d - 2e-6f * d - k * sqrt_about(d); }
__device__ __forceinline__ float have_of(float d, float h, float k)
{
    return d + 2e-6f * d + k * (sqrt_about(d) + 4.f * h) + 8e-6f * h * h;
}

// q = (p', have(p')): whether p cannot be nearest anywhere in the cell (h2: twice its widened
// half width) because of p'.
__device__ __forceinline__ bool dropped_by(float4 q, float px, float py, float pz, float need, float h2)
{
    return need > fmaf(h2, fabsf(px - q.x) + fabsf(py - q.y) + fabsf(pz - q.z), q.w);
}

// Record of a cell that the next round works on: centre and half width, its list, where its
// children's nodes go (the block of eight; for a start cell before its second pass its own
// node; for the two grid levels above the near table the cell's grid coordinates) and
// whether it is a near cell or in which shell.
static_assert(kStaged % (32 * kBatch) == 0 && kMaskPts % (32 * kBatch) == 0 && kStaged <= kMaskPts, "whole batches");

struct CellRef {
    float4 c;
    int base, len, at, shell;              // shell = -1: near
};

__device__ __forceinline__ float widened(float h, int shell, float J)
{
    return h * 1.001f + (shell < 0 ? J * 9.5367432e-7f : ldexpf(J, shell + 1) * 7.6293945e-6f);
}

// Write the node of cell (level t, near grid coordinates or slot `at`).  Near cells of the
// two levels above the table fill all their table entries; call with a whole warp.
__device__ __forceinline__ void put_node(const CellBuild &b, int t, int shell, int at, int2 nd)
{
    const int lane = threadIdx.x & 31;
    if (shell >= 0 || t >= 2) {
        if (lane == 0) b.nodes[at] = nd;
        return;
    }
    const int w = t == 0 ? 4 : 2;          // table cells per side
    const int x = (at & 31) * w, y = ((at >> 5) & 31) * w, z = (at >> 10) * w;
    for (int e = lane; e < w * w * w; e += 32)
        b.nodes[((z + e / (w * w)) * kTable + y + (e / w) % w) * kTable + x + e % w] = nd;
}

// Room for a list of n points in the leaf lists (rounded up to whole int4), or -1.
__device__ __forceinline__ int take_leaf(const CellBuild &b, int n)
{
    const int n4 = (n + 3) & ~3;
    const int at = atomicAdd(b.ctr + kCtrLeaf, n4);
    return at <= b.leaf_cap - n4 ? at : -1;
}

__device__ __forceinline__ CellRef *recs(const CellBuild &b, int round)
{
    return reinterpret_cast<CellRef *>(b.recs) + (size_t)(round & 1) * b.cell_cap;
}

__device__ __forceinline__ int *lists(const CellBuild &b, int round)
{
    return b.lists + (size_t)(round & 1) * b.list_cap;
}

// Room for a cell of level t (< 0: a start cell before its second pass) with n points that the
// next round works on: its list, its children's nodes and its record (r.base, r.at and *rec);
// false when a budget ran out (the cell becomes a leaf then).  The three counters are taken
// together, so that one wait covers them; a record taken in vain is left empty.
__device__ __forceinline__ bool take_inner(const CellBuild &b, int t, int n, bool nodes, CellRef &r, CellRef *&rec)
{
    const int round = t + 1;
    const bool is_long = n > kStaged || t < 0;
    const int base = atomicAdd(b.ctr + kCtrList + round, n);
    const int k = atomicAdd(b.ctr + (is_long ? kCtrLong : kCtrShort) + round, 1);
    const int block = nodes ? atomicAdd(b.ctr + kCtrNode, 1) : 0;
    const int at = kFixedNodes + 8 * block;
    // (short records from the front, long ones from the back, half the room each)
    const bool room = k < b.cell_cap / 2;
    rec = recs(b, round) + (is_long ? b.cell_cap - 1 - k : k);
    if (room && base <= b.list_cap - n && at <= b.node_cap - 8) {
        r.base = base;
        if (nodes) r.at = at;
        return true;
    }
    if (room) rec->len = 0;
    return false;
}

// A leaf list's tail up to a whole int4 repeats its first point.
__device__ __forceinline__ void pad_leaf(int *l, int n, int first)
{
    const int lane = threadIdx.x & 31;
    if (lane < ((n + 3) & ~3) - n) l[n + lane] = first;
}

}  // namespace

// Lists of the start cells (the near 8^3 grid and the far shells) from the whole cloud,
// against the point nearest to the centre alone.  One CTA per cell; every warp works
// on a contiguous eighth of the cloud, so that the lists come out in index order.
__global__ void __launch_bounds__(256) cells_start_kernel(const CellBuildBatch batch)
{
    const CellBuild &b = batch.b[blockIdx.y];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, M = b.M;
    __shared__ unsigned long long s_best[8];
    __shared__ int s_cnt[8], s_leaf, s_base;
    __shared__ unsigned s_mask[8][kStartMask];
    const float4 fr = *b.frame;
    const float J = cell_half(fr.w, b.log_factor), k = (5e-7f + b.tol) * fr.w;
    int cell = blockIdx.x;
    CellRef r;
    r.shell = -1;
    if (cell < kStartNear * kStartNear * kStartNear) {
        const int x = cell % kStartNear, y = cell / kStartNear % kStartNear, z = cell / (kStartNear * kStartNear);
        r.c.w = J / kStartNear;
        r.c.x = (2 * x + 1) * r.c.w - J; r.c.y = (2 * y + 1) * r.c.w - J; r.c.z = (2 * z + 1) * r.c.w - J;
        r.at = x | (y << 5) | (z << 10);
    } else {
        cell -= kStartNear * kStartNear * kStartNear;
        r.shell = cell >> 6;
        const int x = cell & 3, y = (cell >> 2) & 3, z = (cell >> 4) & 3;
        const float H = ldexpf(J, r.shell + 1);
        r.c.w = 0.25f * H;
        r.c.x = (2 * x + 1) * r.c.w - H; r.c.y = (2 * y + 1) * r.c.w - H; r.c.z = (2 * z + 1) * r.c.w - H;
        r.at = kFarBase + cell;
        // inside: the near grid or a smaller shell covers it
        if (x % 3 != 0 && y % 3 != 0 && z % 3 != 0) {
            if (threadIdx.x == 0) b.nodes[r.at] = make_int2(0, kWhole);
            return;
        }
    }
    const float4 c = r.c;
    const int lo = (int)((long long)M * warp / 8), hi = (int)((long long)M * (warp + 1) / 8);
    auto rel = [&](int i, float &x, float &y, float &z) {
        const float4 p = __ldg(b.R + i);
        x = __fsub_rn(p.x, fr.x); y = __fsub_rn(p.y, fr.y); z = __fsub_rn(p.z, fr.z);
        const float ex = x - c.x, ey = y - c.y, ez = z - c.z;
        return ex * ex + ey * ey + ez * ez;
    };
    float bd = __int_as_float(0x7f800000);
    int bi = min(lo, M - 1);
#pragma unroll 4
    for (int i = lo + lane; i < hi; i += 32) {
        float x, y, z;
        const float d = rel(i, x, y, z);
        if (d < bd) { bd = d; bi = i; }
    }
    unsigned long long best = ((unsigned long long)__float_as_uint(bd) << 32) | (unsigned)bi;
    for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (lane == 0) s_best[warp] = best;
    __syncthreads();
    for (int w = 0; w < 8; ++w) best = min(best, s_best[w]);
    float4 q;
    {
        const float d = rel((int)(unsigned)best, q.x, q.y, q.z);
        q.w = have_of(d, c.w, k);
    }
    const float h2 = 2.f * widened(c.w, r.shell, J);
    auto kept = [&](int i) {
        float x, y, z;
        const float d = rel(min(i, M - 1), x, y, z);
        return i < hi && !dropped_by(q, x, y, z, need_of(d, k), h2);
    };
    const bool masks = hi - lo <= 32 * kStartMask;
    int cnt = 0;
#pragma unroll 4
    for (int i0 = lo; i0 < hi; i0 += 32) {
        const unsigned m = __ballot_sync(0xffffffffu, kept(i0 + lane));
        if (masks && lane == 0) s_mask[warp][(i0 - lo) >> 5] = m;
        cnt += __popc(m);
    }
    if (lane == 0) s_cnt[warp] = cnt;
    __syncthreads();
    int n = 0, pos = 0;
    for (int w = 0; w < 8; ++w) {
        pos += w < warp ? s_cnt[w] : 0;
        n += s_cnt[w];
    }
    CellRef *rec = nullptr;
    if (threadIdx.x == 0) {
        s_leaf = n <= kLeaf || !take_inner(b, -1, n, false, r, rec);
        s_base = s_leaf ? take_leaf(b, n) : r.base;
    }
    __syncthreads();
    const int base = s_base;
    const bool leaf = s_leaf != 0;
    if (base < 0) {
        if (warp == 0) put_node(b, 0, r.shell, r.at, make_int2(0, kWhole));
        return;
    }
    int *out = (leaf ? b.leaves : lists(b, 0)) + base;
#pragma unroll 4
    for (int i0 = lo; i0 < hi; i0 += 32) {
        const unsigned m = masks ? s_mask[warp][(i0 - lo) >> 5] : __ballot_sync(0xffffffffu, kept(i0 + lane));
        if (m >> lane & 1) out[pos + __popc(m & ((1u << lane) - 1u))] = i0 + lane;
        pos += __popc(m);
    }
    if (leaf) {
        __syncthreads();
        if (warp == 0) {
            pad_leaf(out, n, out[0]);
            put_node(b, 0, r.shell, r.at, make_int2(base, (n + 3) & ~3));
        }
    } else if (threadIdx.x == 0) {
        r.len = n;
        *rec = r;
    }
}

// Near the centre (slot 8) and the corners (0 .. 7) of cell c, per lane: the smallest squared
// distance among the points [lo, hi) of a list, its low kIterBits replaced by the loop's
// round (any point will do to hold the others against, so the lost bits do not matter; at
// most 2^kIterBits rounds); point(i) is the list's i-th point.  kBatch points per lane are
// loaded together (the tail repeats the last one): the lists are short, the loads' latency
// is what costs.
template <class P>
__device__ __forceinline__ void nearest9(P point, int lo, int hi, float4 c, unsigned (&key)[9])
{
#pragma unroll
    for (int k = 0; k < 9; ++k) key[k] = 0x7f800000u;
    const float h2 = 2.f * c.w, hh = 3.f * c.w * c.w;
    constexpr unsigned kIter = (1u << kIterBits) - 1u;
    const int lane = threadIdx.x & 31;
    for (int i0 = lo; i0 < hi; i0 += 32 * kBatch) {
        float4 p[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) p[j] = point(min(i0 + 32 * j + lane, hi - 1));
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const unsigned it = (unsigned)(i0 - lo) / 32u + j;
            const float ex = p[j].x - c.x, ey = p[j].y - c.y, ez = p[j].z - c.z;
            const float d = ex * ex + ey * ey + ez * ez;
            auto take = [&](int k, float v) { key[k] = min(key[k], (__float_as_uint(fmaxf(v, 0.f)) & ~kIter) | it); };
            take(8, d);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                take(k, fmaf(k & 1 ? -h2 : h2, ex, fmaf(k & 2 ? -h2 : h2, ey, fmaf(k & 4 ? -h2 : h2, ez, d + hh))));
        }
    }
}

// Reduce every slot over the warp: lane (k + 1) % 9 returns slot k's key and list position
// (lane 0: the centre's).
__device__ __forceinline__ void reduce9(const unsigned (&keys)[9], int lo, int hi, unsigned &key, int &pos)
{
    const int lane = threadIdx.x & 31;
    key = ~0u;
    pos = lo;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const unsigned m = __reduce_min_sync(0xffffffffu, keys[k]);
        const int src = __ffs(__ballot_sync(0xffffffffu, keys[k] == m)) - 1;
        if (lane == (k + 1) % 9) {
            key = m;
            pos = min(lo + (int)(m & ((1u << kIterBits) - 1u)) * 32 + src, max(hi - 1, lo));
        }
    }
}

// The distinct points of the warp's lanes 0 .. 8 as the points to hold the others against, the
// centre's first; returns their number.
template <class P>
__device__ __forceinline__ int make_doms(P point, int pos, float4 c, float k, float4 *dom)
{
    const int lane = threadIdx.x & 31;
    const unsigned same = __match_any_sync(0xffffffffu, lane < 9 ? pos : -1 - lane);
    const bool first = lane < 9 && (__ffs(same) - 1) == lane;
    const unsigned firsts = __ballot_sync(0xffffffffu, first);
    if (first) {
        float4 p = point(pos);
        const float ex = p.x - c.x, ey = p.y - c.y, ez = p.z - c.z;
        p.w = have_of(ex * ex + ey * ey + ez * ez, c.w, k);
        dom[__popc(firsts & ((1u << lane) - 1u))] = p;
    }
    __syncwarp();
    return __popc(firsts);
}

// Which of the points [i0, i0 + 32 kBatch) below hi no point of dom drops: bit lane of m[j] for
// point i0 + 32 j + lane.
template <class P>
__device__ __forceinline__ void keeps(P point, int i0, int hi, float4 c, const float4 *dom, int nd, float h2, float k,
                                      unsigned (&m)[kBatch])
{
    const int lane = threadIdx.x & 31;
    float4 p[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) p[j] = point(min(i0 + 32 * j + lane, hi - 1));
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
        const float ex = p[j].x - c.x, ey = p[j].y - c.y, ez = p[j].z - c.z;
        p[j].w = need_of(ex * ex + ey * ey + ez * ez, k);
    }
    bool out[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) out[j] = i0 + 32 * j + lane >= hi;
    for (int e = 0; e < nd; ++e) {
        const float4 q = dom[e];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) out[j] = out[j] || dropped_by(q, p[j].x, p[j].y, p[j].z, p[j].w, h2);
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j) m[j] = __ballot_sync(0xffffffffu, !out[j]);
}

// Child o of cell r of level t (t < 0: the start cell itself): its centre and half width and
// where its node goes (near grid coordinates above the table's level).
__device__ __forceinline__ CellRef child_of(const CellRef &r, int t, int o)
{
    CellRef q = r;
    if (t < 0) return q;
    q.c.w = 0.5f * r.c.w;
    q.c.x = r.c.x + (o & 1 ? q.c.w : -q.c.w);
    q.c.y = r.c.y + (o & 2 ? q.c.w : -q.c.w);
    q.c.z = r.c.z + (o & 4 ? q.c.w : -q.c.w);
    if (r.shell >= 0 || t >= 2) {
        q.at = r.at + o;
    } else {
        const int x = 2 * (r.at & 31) + (o & 1), y = 2 * ((r.at >> 5) & 31) + ((o >> 1) & 1), z = 2 * (r.at >> 10) + (o >> 2);
        q.at = t == 1 ? (z * kTable + y) * kTable + x : x | (y << 5) | (z << 10);
    }
    return q;
}

// Make cell q of level t1 a leaf or (unless `stop`) a cell to be halved: room for the n points kept of its
// parent's `len` (returned: base, < 0 for none, and leaf), and for the latter its record and
// node.  One thread.
struct Place {
    int leaf, base;
};
__device__ __forceinline__ Place place_cell(const CellBuild &b, int t1, bool stop, CellRef q, int n, int len)
{
    const bool near = q.shell < 0, node = !near || t1 >= 2;   // (the levels above the near table have no nodes)
    const bool last = stop || t1 >= (near ? kNearLevels : kFarLevels) || (t1 >= (near ? 3 : 2) && n > 0.8f * len);
    CellRef *rec;
    const int at = q.at;
    Place p;
    p.leaf = n <= kLeaf || last || !take_inner(b, t1, n, node, q, rec);
    if (p.leaf) {
        p.base = take_leaf(b, n);
    } else {
        p.base = q.base;
        q.len = n;
        *rec = q;
        if (node) b.nodes[at] = make_int2(q.at, kInner);
    }
    return p;
}

// One round of the build.  t >= 0: halve the cells of level t; t < 0: hold the start cells' own
// lists against the points near their corners too (before the first halving copies them
// eight times).  A cell with at most kStaged points is one CTA's: its list is staged in
// shared memory and warp w makes child w.  A child of a longer one (and a start cell) is
// made by a whole CTA, every warp on a contiguous eighth of the list: the upper levels
// have few cells and long lists, where a warp alone would set the pace.
__global__ void __launch_bounds__(256) cells_level_kernel(const CellBuildBatch batch, int t)
{
    const CellBuild &b = batch.b[blockIdx.y];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t1 = t + 1;
    const int round = t + 1, cap = b.cell_cap / 2;
    const int n_short = min(b.ctr[kCtrShort + round], cap), n_long = min(b.ctr[kCtrLong + round], cap);
    const int children = t < 0 ? 1 : 8;
    // half the leaf budget gone (exact planes and spheres): the cells stay as they are, which takes
    // less room than halving them would
    const bool stop = b.ctr[kCtrLeaf] > b.leaf_cap / 2;
    __shared__ float4 s_pt[kStaged];
    __shared__ unsigned s_mask[8][kMaskPts / 32];
    __shared__ float4 s_dom[8][9];
    __shared__ unsigned s_key[8][9];
    __shared__ int s_pos[8][9], s_cnt[8];
    __shared__ Place s_place;
    const float4 fr = *b.frame;
    const float J = cell_half(fr.w, b.log_factor), k = (5e-7f + b.tol) * fr.w;
    for (int u = blockIdx.x; u < n_long * children; u += gridDim.x) {
        const CellRef r = recs(b, round)[b.cell_cap - 1 - u / children];
        if (r.len <= 0) continue;
        const int *list = lists(b, round) + r.base;
        auto load = [&](int i) {
            const int idx = __ldg(list + i);
            const float4 v = __ldg(b.R + idx);
            return make_float4(__fsub_rn(v.x, fr.x), __fsub_rn(v.y, fr.y), __fsub_rn(v.z, fr.z), __int_as_float(idx));
        };
        const CellRef q = child_of(r, t, u % children);
        const int lo = (int)((long long)r.len * warp / 8), hi = (int)((long long)r.len * (warp + 1) / 8);
        unsigned keys[9], key;
        int pos;
        nearest9(load, lo, hi, q.c, keys);
        reduce9(keys, lo, hi, key, pos);
        __syncthreads();                   // the previous unit's shared values are no longer read
        if (lane < 9) { s_key[warp][lane] = key; s_pos[warp][lane] = pos; }
        __syncthreads();
        for (int w = 0; w < 8; ++w)
            if (lane < 9 && s_key[w][lane] < key) { key = s_key[w][lane]; pos = s_pos[w][lane]; }
        const int nd = make_doms(load, min(pos, r.len - 1), q.c, k, s_dom[warp]);
        const float h2 = 2.f * widened(q.c.w, r.shell, J);
        const bool masks = hi - lo <= kMaskPts;
        int cnt = 0;
        for (int i0 = lo; i0 < hi; i0 += 32 * kBatch) {
            unsigned m[kBatch];
            keeps(load, i0, hi, q.c, s_dom[warp], nd, h2, k, m);
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                if (masks && lane == 0) s_mask[warp][((i0 - lo) >> 5) + j] = m[j];
                cnt += __popc(m[j]);
            }
        }
        if (lane == 0) s_cnt[warp] = cnt;
        __syncthreads();
        int n = 0, o = 0;
        for (int w = 0; w < 8; ++w) {
            o += w < warp ? s_cnt[w] : 0;
            n += s_cnt[w];
        }
        if (threadIdx.x == 0) s_place = place_cell(b, t1, stop, q, n, r.len);
        __syncthreads();
        const Place p = s_place;
        if (p.base < 0) {
            if (warp == 0) put_node(b, t1, r.shell, q.at, make_int2(0, kWhole));
            continue;
        }
        int *out = (p.leaf ? b.leaves : lists(b, round + 1)) + p.base;
        for (int i0 = lo; i0 < hi; i0 += 32 * kBatch) {
            unsigned m[kBatch];
            if (!masks) keeps(load, i0, hi, q.c, s_dom[warp], nd, h2, k, m);
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                if (masks) m[j] = s_mask[warp][((i0 - lo) >> 5) + j];
                if (m[j] >> lane & 1) out[o + __popc(m[j] & ((1u << lane) - 1u))] = __ldg(list + i0 + 32 * j + lane);
                o += __popc(m[j]);
            }
        }
        if (p.leaf) {
            __syncthreads();
            if (warp == 0) {
                pad_leaf(out, n, out[0]);
                put_node(b, t1, r.shell, q.at, make_int2(p.base, (n + 3) & ~3));
            }
        }
    }
    for (int u = blockIdx.x; u < n_short; u += gridDim.x) {
        const CellRef r = recs(b, round)[u];
        if (r.len <= 0) continue;
        const int *list = lists(b, round) + r.base;
        __syncthreads();                   // the previous cell's points are no longer read
        for (int i = threadIdx.x; i < r.len; i += blockDim.x) {
            const int idx = __ldg(list + i);
            const float4 v = __ldg(b.R + idx);
            s_pt[i] = make_float4(__fsub_rn(v.x, fr.x), __fsub_rn(v.y, fr.y), __fsub_rn(v.z, fr.z), __int_as_float(idx));
        }
        __syncthreads();
        auto point = [&](int i) { return s_pt[i]; };
        const CellRef q = child_of(r, t, warp);
        unsigned keys[9], key;
        int pos;
        nearest9(point, 0, r.len, q.c, keys);
        reduce9(keys, 0, r.len, key, pos);
        const int nd = make_doms(point, pos, q.c, k, s_dom[warp]);
        const float h2 = 2.f * widened(q.c.w, r.shell, J);
        int n = 0;
        for (int i0 = 0; i0 < r.len; i0 += 32 * kBatch) {
            unsigned m[kBatch];
            keeps(point, i0, r.len, q.c, s_dom[warp], nd, h2, k, m);
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                if (lane == 0) s_mask[warp][(i0 >> 5) + j] = m[j];
                n += __popc(m[j]);
            }
        }
        __syncwarp();
        Place p{0, 0};
        if (lane == 0) p = place_cell(b, t1, stop, q, n, r.len);
        p.leaf = __shfl_sync(0xffffffffu, p.leaf, 0);
        p.base = __shfl_sync(0xffffffffu, p.base, 0);
        if (p.base < 0) {
            put_node(b, t1, r.shell, q.at, make_int2(0, kWhole));
            continue;
        }
        int *out = (p.leaf ? b.leaves : lists(b, round + 1)) + p.base;
        int o = 0;
        for (int i0 = 0; i0 < r.len; i0 += 32) {
            const unsigned m = s_mask[warp][i0 >> 5];
            if (m >> lane & 1) out[o + __popc(m & ((1u << lane) - 1u))] = __float_as_int(s_pt[i0 + lane].w);
            o += __popc(m);
        }
        if (p.leaf) {
            __syncwarp();
            pad_leaf(out, n, out[0]);
            put_node(b, t1, r.shell, q.at, make_int2(p.base, (n + 3) & ~3));
        }
    }
}

// The matching itself: one thread per query, a particle's queries in CTAs of their own (its pose
// and object are the CTA's, and no query divides by N).  Queries are taken in the gripper cloud's
// spatial order (S sorted along a space-filling curve, w = the point's own index), so that
// the lanes of a warp meet in the same cells.
constexpr int kMatchThreads = 128;

__global__ void __launch_bounds__(kMatchThreads) cells_match_kernel(const FwdArgs a, int ctas)
{
    const int pk = blockIdx.x / ctas, k = (blockIdx.x - pk * ctas) * kMatchThreads + threadIdx.x;
    const int lane = threadIdx.x & 31, N = a.L.N;
    const bool valid = k < N;
    const int grp = a.L.part_grp[pk], obj = grp / a.L.P;
    const float4 s = a.Ssort[(size_t)(grp - obj * a.L.P) * N + min(k, N - 1)];
    const float *th = a.theta + (size_t)pk * 8;
    float Rm[9];
    quat_rot_f32(th[3], th[4], th[5], th[6], Rm);
    const float3 o = xform_f32(Rm, th[0], th[1], th[2], s.x, s.y, s.z);
    const ObjMeta &om = a.L.obj[obj];
    const float4 *__restrict__ R = om.R;
    const float4 fr = a.L.frame[obj];

    const float J = cell_half(fr.w, kObjectCells);
    const int2 nd = find_cell(om.nodes, J, __fsub_rn(o.x, fr.x), __fsub_rn(o.y, fr.y), __fsub_rn(o.z, fr.z));

    // its list, four points at a time
    float best = __int_as_float(0x7f800000);
    int bi = 0x7fffffff;
    if (nd.y <= kCellOwn) {
        const int4 *l = reinterpret_cast<const int4 *>(om.leaves + nd.x);
        for (int e = 0; e < nd.y; e += 4, ++l) {
            const int4 id = __ldg(l);
            const float4 p0 = __ldg(R + id.x), p1 = __ldg(R + id.y), p2 = __ldg(R + id.z), p3 = __ldg(R + id.w);
            const float d0 = dist2_f32(o.x, o.y, o.z, p0.x, p0.y, p0.z), d1 = dist2_f32(o.x, o.y, o.z, p1.x, p1.y, p1.z),
                        d2 = dist2_f32(o.x, o.y, o.z, p2.x, p2.y, p2.z), d3 = dist2_f32(o.x, o.y, o.z, p3.x, p3.y, p3.z);
            // (index order; the padding repeats an earlier point)
            if (d0 < best) { best = d0; bi = id.x; }
            if (d1 < best) { best = d1; bi = id.y; }
            if (d2 < best) { best = d2; bi = id.z; }
            if (d3 < best) { best = d3; bi = id.w; }
        }
    }
    unsigned pending = __ballot_sync(0xffffffffu, valid && (nd.y == kWhole || nd.y > kCellOwn));
    while (pending) {
        const int src = __ffs(pending) - 1;
        pending &= pending - 1;
        const float qx = __shfl_sync(0xffffffffu, o.x, src), qy = __shfl_sync(0xffffffffu, o.y, src),
                    qz = __shfl_sync(0xffffffffu, o.z, src);
        const int base = __shfl_sync(0xffffffffu, nd.x, src), len = __shfl_sync(0xffffffffu, nd.y, src);
        float wb = __int_as_float(0x7f800000);
        int wi = 0x7fffffff;
        if (len == kWhole) {
            warp_exact_all(R, om.M, qx, qy, qz, wb, wi);
        } else {
            for (int e = lane; e < len; e += 32) {       // (index order: a lane's ties keep the lower index)
                const int r = __ldg(om.leaves + base + e);
                const float4 p = __ldg(R + r);
                const float d = dist2_f32(qx, qy, qz, p.x, p.y, p.z);
                if (d < wb) { wb = d; wi = r; }
            }
        }
        for (int off = 16; off > 0; off >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, wb, off);
            const int oi = __shfl_xor_sync(0xffffffffu, wi, off);
            if (ob < wb || (ob == wb && oi < wi)) { wb = ob; wi = oi; }
        }
        if (lane == src) { best = wb; bi = wi; }
    }
    if (!valid) return;
    const long long q = (long long)pk * N + __float_as_int(s.w);
    a.nn_idx[q] = best < __int_as_float(0x7f800000) ? bi : 0;      // no finite distance: 0
    if (a.dbg_d2) a.dbg_d2[q] = best;
    if (a.dbg_sp) {
        a.dbg_sp[q * 3 + 0] = o.x;
        a.dbg_sp[q * 3 + 1] = o.y;
        a.dbg_sp[q * 3 + 2] = o.z;
    }
}

// What the matching through the cells costs, counted on a sample of its warps: for the present poses, and for poses
// that much nearer to the object's centre (kCellPull), which is where a run takes them.  The unit is a round of 32 points
// of the whole cloud that a warp compares together; kCellList for 32 points of a long list (gathered through indices),
// kCellStep for each four points that the lanes compare from lists of their own (kCellWait where one warp's latency
// counts), kCellBase for the look-ups.  Warp i of n looks at one of the i-th n-th of all warps.  Measured on GB300 (1.6 M
// queries, M 8192; us per pass counted at kCellRounds and timed): noisy objects 37 and 42; boxes without noise 49 to 67
// and 51 to 70; every point four times 166 and 163; an ellipsoid without noise 1158 and 1300.
constexpr int kCellBase = 30, kCellStep = 9, kCellList = 3, kCellWait = 3;
constexpr float kCellPull = 0.25f;

constexpr int kCostThreads = 256;

__global__ void __launch_bounds__(kCostThreads) cells_cost_kernel(const FwdArgs a, long long warps, int n, CellCost *cost,
                                                                  CellCost *host, unsigned seq)
{
    __shared__ unsigned s_sum[2][kCostThreads / 32], s_most[2][kCostThreads / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, N = a.L.N;
    const int at = blockIdx.x * (kCostThreads / 32) + warp, i = min(at, n - 1);
    const long long lo = warps * i / n, room = warps * (i + 1) / n - lo;
    const long long w = lo + (long long)((i * 2654435761u) >> 8) % room;
    const int per = (N + 31) / 32, pk = (int)(w / per), k = (int)(w % per) * 32 + lane;
    const int grp = a.L.part_grp[pk], obj = grp / a.L.P;
    const float4 s = a.Ssort[(size_t)(grp - obj * a.L.P) * N + min(k, N - 1)];
    const ObjMeta &om = a.L.obj[obj];
    const float4 fr = a.L.frame[obj];
    const float *th = a.theta + (size_t)pk * 8;
    float Rm[9];
    quat_rot_f32(th[3], th[4], th[5], th[6], Rm);
    for (int near = 0; near < 2; ++near) {
        const float f = near ? kCellPull : 1.f;
        const float3 o = xform_f32(Rm, fr.x + f * (th[0] - fr.x), fr.y + f * (th[1] - fr.y), fr.z + f * (th[2] - fr.z), s.x, s.y,
                                   s.z);
        const int2 nd = find_cell(om.nodes, cell_half(fr.w, kObjectCells), __fsub_rn(o.x, fr.x), __fsub_rn(o.y, fr.y),
                                  __fsub_rn(o.z, fr.z));
        const int len = nd.y == kWhole ? om.M : nd.y;
        const bool own = nd.y != kWhole && len <= kCellOwn;
        const unsigned steps = __reduce_max_sync(0xffffffffu, own ? (unsigned)len / 4u : 0u);
        const unsigned mine = own || k >= N ? 0u : (unsigned)(len + 31) / 32u;
        const unsigned whole = __reduce_add_sync(0xffffffffu, nd.y == kWhole ? mine : 0u);
        const unsigned lists = __reduce_add_sync(0xffffffffu, nd.y == kWhole ? 0u : mine);
        if (lane == 0) {
            s_sum[near][warp] = at == i ? kCellBase + kCellStep * steps + whole + kCellList * lists : 0u;
            s_most[near][warp] = kCellBase + kCellWait * steps + whole + lists;
        }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int k = 0; k < 2; ++k) {
        unsigned long long sum = 0;
        unsigned most = 0u;
        for (int w = 0; w < kCostThreads / 32; ++w) {
            sum += s_sum[k][w];
            most = max(most, s_most[k][w]);
        }
        atomicAdd(&cost->sum[k], sum);
        atomicMax(&cost->most[k], most);
    }
    // the last CTA hands the counts over
    __threadfence();
    if (atomicAdd(&cost->seq, 1u) == gridDim.x - 1) {
        __threadfence();
        volatile CellCost *h = host;
        for (int k = 0; k < 2; ++k) {
            h->sum[k] = atomicAdd(&cost->sum[k], 0ull);
            h->most[k] = atomicAdd(&cost->most[k], 0u);
        }
        __threadfence_system();
        h->seq = seq;
    }
}

// The sum over the sample and the most rounds of a warp, of any kind, for the present poses and those pulled in, go to *cost
// (cleared before) and from there to *host, page-locked memory, whose seq is written last; *share: how much of all warps
// the sample is.
cudaError_t launch_cells_cost(const FwdArgs &a, CellCost *cost, CellCost *host, unsigned seq, double *share, cudaStream_t st)
{
    const long long warps = (long long)a.L.T * ((a.L.N + 31) / 32);
    const int n = (int)(warps < kCellSample ? warps : kCellSample);
    *share = (double)n / (double)warps;
    constexpr int kWarps = kCostThreads / 32;
    cells_cost_kernel<<<(n + kWarps - 1) / kWarps, kCostThreads, 0, st>>>(a, warps, n, cost, host, seq);
    return cudaGetLastError();
}

CellSizes cell_sizes(int M)
{
    CellSizes s;
    s.leaf_cap = 256 * M + (1 << 21);
    s.list_cap = 64 * M + (1 << 19);
    s.cell_cap = 4 * M + (1 << 16);
    s.node_cap = kFixedNodes + 16 * M + (1 << 17);
    s.rec_bytes = 2 * sizeof(CellRef) * (size_t)s.cell_cap;
    return s;
}

cudaError_t launch_cells_build(const CellBuildBatch &batch, int n, cudaStream_t st)
{
    cells_start_kernel<<<dim3(kStartCells, n), 256, 0, st>>>(batch);
    for (int t = -1; t < kNearLevels; ++t) cells_level_kernel<<<dim3(1216, n), 256, 0, st>>>(batch, t);
    return cudaGetLastError();
}

cudaError_t launch_cells_match(const FwdArgs &a, cudaStream_t st)
{
    if (a.L.T == 0) return cudaSuccess;
    const int ctas = (a.L.N + kMatchThreads - 1) / kMatchThreads;
    cells_match_kernel<<<(unsigned)(a.L.T * ctas), kMatchThreads, 0, st>>>(a, ctas);
    return cudaGetLastError();
}

// sum s and sum s s^T (upper triangle) of a gripper cloud in float64, for one CTA: fixed thread striding and tree.
__device__ __forceinline__ void preshape_sums(const float4 *S, int N, double *out12)
{
    __shared__ double red[32][9];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double acc[9] = {};
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const float4 s = S[i];
        const double x = s.x, y = s.y, z = s.z;
        acc[0] += x; acc[1] += y; acc[2] += z;
        acc[3] = fma(x, x, acc[3]); acc[4] = fma(x, y, acc[4]); acc[5] = fma(x, z, acc[5]);
        acc[6] = fma(y, y, acc[6]); acc[7] = fma(y, z, acc[7]); acc[8] = fma(z, z, acc[8]);
    }
    warp_sum_f64(acc);
    if (lane == 0)
        for (int c = 0; c < 9; ++c) red[warp][c] = acc[c];
    __syncthreads();
    if (threadIdx.x < 12) {
        double s = 0.0;
        if (threadIdx.x < 9)
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w][threadIdx.x];
        out12[threadIdx.x] = s;
    }
}

// Preparation of a gripper cloud, two CTAs of 25 us each side by side.  CTA 1: its sums.  CTA 0: its spatial order, a
// bitonic sort of (Morton code, index) keys, then the points in that order with their own index in w.  *frame: the centre
// of the bounding box and the largest distance from it, rounded up.
__global__ void __launch_bounds__(1024) gripper_cloud_kernel(const float4 *S, int N, int Npow, float4 *out, float4 *frame,
                                                             double *out12)
{
    extern __shared__ unsigned long long s_key[];
    __shared__ float s_lo[3][32], s_hi[3][32];
    if (blockIdx.x == 1) {
        preshape_sums(S, N, out12);
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float lo[3], hi[3];
    for (int k = 0; k < 3; ++k) { lo[k] = __int_as_float(0x7f800000); hi[k] = -lo[k]; }
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const float4 p = S[i];
        lo[0] = fminf(lo[0], p.x); lo[1] = fminf(lo[1], p.y); lo[2] = fminf(lo[2], p.z);
        hi[0] = fmaxf(hi[0], p.x); hi[1] = fmaxf(hi[1], p.y); hi[2] = fmaxf(hi[2], p.z);
    }
    for (int k = 0; k < 3; ++k) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
        if (lane == 0) { s_lo[k][warp] = lo[k]; s_hi[k][warp] = hi[k]; }
    }
    __syncthreads();
    for (int k = 0; k < 3; ++k)
        for (int w = 0; w < 32; ++w) { lo[k] = fminf(lo[k], s_lo[k][w]); hi[k] = fmaxf(hi[k], s_hi[k][w]); }
    const float cx = 0.5f * lo[0] + 0.5f * hi[0], cy = 0.5f * lo[1] + 0.5f * hi[1], cz = 0.5f * lo[2] + 0.5f * hi[2];
    float far2 = 0.f;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const float4 p = S[i];
        const float x = p.x - cx, y = p.y - cy, z = p.z - cz;
        far2 = fmaxf(far2, x * x + y * y + z * z);
    }
    for (int o = 16; o > 0; o >>= 1) far2 = fmaxf(far2, __shfl_xor_sync(0xffffffffu, far2, o));
    __syncthreads();                       // s_lo has been read
    if (lane == 0) s_lo[0][warp] = far2;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 0; w < 32; ++w) far2 = fmaxf(far2, s_lo[0][w]);
        *frame = make_float4(cx, cy, cz, sqrtf(far2) * (1.f + 1e-5f) + 1e-30f);
    }
    const float ext = fmaxf(fmaxf(hi[0] - lo[0], hi[1] - lo[1]), fmaxf(hi[2] - lo[2], 1e-30f));
    auto spread = [](unsigned v) {         // ten bits, two zeros after each
        v = (v | (v << 16)) & 0x030000ffu;
        v = (v | (v << 8)) & 0x0300f00fu;
        v = (v | (v << 4)) & 0x030c30c3u;
        return (v | (v << 2)) & 0x09249249u;
    };
    for (int i = threadIdx.x; i < Npow; i += blockDim.x) {
        unsigned long long key = ~0ull;
        if (i < N) {
            const float4 p = S[i];
            const unsigned x = (unsigned)min(max((int)((p.x - lo[0]) / ext * 1023.f), 0), 1023),
                           y = (unsigned)min(max((int)((p.y - lo[1]) / ext * 1023.f), 0), 1023),
                           z = (unsigned)min(max((int)((p.z - lo[2]) / ext * 1023.f), 0), 1023);
            key = ((unsigned long long)(spread(x) | (spread(y) << 1) | (spread(z) << 2)) << 32) | (unsigned)i;
        }
        s_key[i] = key;
    }
    for (int k = 2; k <= Npow; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            __syncthreads();
            for (int e = threadIdx.x; e < Npow / 2; e += blockDim.x) {
                const int i = ((e & ~(j - 1)) << 1) | (e & (j - 1)), p = i | j;
                const unsigned long long a = s_key[i], b = s_key[p];
                if ((a > b) == ((i & k) == 0)) { s_key[i] = b; s_key[p] = a; }
            }
        }
    __syncthreads();
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const int src = (int)(unsigned)s_key[i];
        float4 p = S[src];
        p.w = __int_as_float(src);
        out[i] = p;
    }
}

cudaError_t init_cells_attributes()
{
    return cudaFuncSetAttribute(gripper_cloud_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                8192 * (int)sizeof(unsigned long long));
}

cudaError_t launch_gripper_cloud(const float4 *S, int N, float4 *out, float4 *frame, double *out12, cudaStream_t st)
{
    static_assert(kMaxN <= 8192, "shared-memory sort");
    int Npow = 2;
    while (Npow < N) Npow <<= 1;
    gripper_cloud_kernel<<<2, 1024, (size_t)Npow * sizeof(unsigned long long), st>>>(S, N, Npow, out, frame, out12);
    return cudaGetLastError();
}

}  // namespace asicp
