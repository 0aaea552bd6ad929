// Internal declarations shared by the kernels and the C-ABI of libasicp.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

namespace asicp {

constexpr int kDeviceSlots = 64;       // devices a process can use the library on

// A launch value that depends on the device (its SM count, an occupancy) and
// sets the kernel attributes it relies on: compute() runs once per device, with
// that device current, under a lock, so several devices and several host
// threads each get their own value.  Returns 0 (an invalid grid, which the
// launch then reports) if the current device cannot be read.
template <class F>
int per_device_value(int (&cache)[kDeviceSlots], std::mutex &mu, F compute)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDeviceSlots) return 0;
    std::lock_guard<std::mutex> lock(mu);
    if (cache[dev] == 0) cache[dev] = compute();
    return cache[dev];
}

constexpr int kRefTilePts = 2048;      // object points per shared-memory tile of the matching kernel
constexpr int kFwdSums = 13;           // per-particle matching sums (see finalize_kernel)
constexpr int kColSums = 22;           // per-particle collision sums (see finalize_kernel)
constexpr int kMaxK = 1024;            // particles per preshape (one update CTA per preshape)
constexpr int kMaxN = 6144;            // gripper points per preshape (reverse matching keeps 32 B per point in shared memory)

// error word written by device code (host reads it back after synchronising)
enum : int { kDevOk = 0, kDevNonFinite = 1, kDevTimeout = 2 };

struct SdfMeta {           // one preshape's grid
    const float *grid;     // nx*ny*nz values, x fastest, positive inside the gripper
    const float4 *cells;   // the same values corner-packed: per cell (x fastest over the
                           // (nx-1)(ny-1)(nz-1) cells) its 8 corners as two float4,
                           // {c000, c100, c010, c110} {c001, c101, c011, c111} (index x, y, z)
    int nx, ny, nz;
    float ox, oy, oz;      // position of node (0,0,0)
    float voxel;
    const unsigned char *clear;   // per cell (same order) its distance in cells to the nearest one
                                  // with a positive corner (largest coordinate, at most 255)
};

// Rotation of a (unit) quaternion in the homogeneous form
// R = (w^2 - |v|^2) I + 2 v v^T + 2 w [v]_x, evaluated with explicit
// round-to-nearest operations so every kernel gets bit-identical matrices.
__device__ __forceinline__ void quat_rot_f32(float w, float x, float y, float z, float R[9])
{
    float a = __fsub_rn(__fmul_rn(w, w), __fadd_rn(__fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y)), __fmul_rn(z, z)));
    float xx = __fmul_rn(x, x), yy = __fmul_rn(y, y), zz = __fmul_rn(z, z);
    float xy = __fmul_rn(x, y), xz = __fmul_rn(x, z), yz = __fmul_rn(y, z);
    float wx = __fmul_rn(w, x), wy = __fmul_rn(w, y), wz = __fmul_rn(w, z);
    R[0] = __fadd_rn(a, __fmul_rn(2.f, xx));
    R[1] = __fmul_rn(2.f, __fsub_rn(xy, wz));
    R[2] = __fmul_rn(2.f, __fadd_rn(xz, wy));
    R[3] = __fmul_rn(2.f, __fadd_rn(xy, wz));
    R[4] = __fadd_rn(a, __fmul_rn(2.f, yy));
    R[5] = __fmul_rn(2.f, __fsub_rn(yz, wx));
    R[6] = __fmul_rn(2.f, __fsub_rn(xz, wy));
    R[7] = __fmul_rn(2.f, __fadd_rn(yz, wx));
    R[8] = __fadd_rn(a, __fmul_rn(2.f, zz));
}

__device__ __forceinline__ void quat_rot_f64(double w, double x, double y, double z, double R[9])
{
    double a = w * w - (x * x + y * y + z * z);
    R[0] = a + 2 * x * x;         R[1] = 2 * (x * y - w * z); R[2] = 2 * (x * z + w * y);
    R[3] = 2 * (x * y + w * z);   R[4] = a + 2 * y * y;       R[5] = 2 * (y * z - w * x);
    R[6] = 2 * (x * z - w * y);   R[7] = 2 * (y * z + w * x); R[8] = a + 2 * z * z;
}

// s' = R s + t in float32, fixed operation order (shared by every kernel that
// needs transformed gripper points, so forward and reverse matching agree).
__device__ __forceinline__ float3 xform_f32(const float R[9], float tx, float ty, float tz, float sx, float sy, float sz)
{
    float3 o;
    o.x = __fmaf_rn(R[0], sx, __fmaf_rn(R[1], sy, __fmaf_rn(R[2], sz, tx)));
    o.y = __fmaf_rn(R[3], sx, __fmaf_rn(R[4], sy, __fmaf_rn(R[5], sz, ty)));
    o.z = __fmaf_rn(R[6], sx, __fmaf_rn(R[7], sy, __fmaf_rn(R[8], sz, tz)));
    return o;
}

// Total order of float32 values (no NaN) as unsigned keys, and back.
__device__ __forceinline__ unsigned order_key(float f)
{
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float key_float(unsigned k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Exact-form squared distance |a - b|^2 in float32, fixed order.
__device__ __forceinline__ float dist2_f32(float ax, float ay, float az, float bx, float by, float bz)
{
    float dx = __fsub_rn(ax, bx), dy = __fsub_rn(ay, by), dz = __fsub_rn(az, bz);
    return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// Exact-form nearest point of query (qx, qy, qz) among all M object points, found by
// the whole warp together (lane l takes points l, l + 32, ...; ties to the lower
// index); every lane receives the result.  Call with all 32 lanes.
__device__ __forceinline__ void warp_exact_all(const float4 *__restrict__ R, int M, float qx, float qy, float qz,
                                               float &best, int &bi)
{
    float wb = __int_as_float(0x7f800000);
    int wi = 0x7fffffff;
    for (int r = (int)(threadIdx.x & 31); r < M; r += 32) {
        const float4 v = __ldg(R + r);
        const float d = dist2_f32(qx, qy, qz, v.x, v.y, v.z);
        if (d < wb) { wb = d; wi = r; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, wb, off);
        const int oi = __shfl_xor_sync(0xffffffffu, wi, off);
        if (ob < wb || (ob == wb && oi < wi)) { wb = ob; wi = oi; }
    }
    best = wb;
    bi = wi < M ? wi : 0;    // no finite distance at all (not reached with finite inputs)
}

// Double-float accumulation (hi + lo, ~48-bit significand) from float32 error-free
// transformations: products are split exactly by an FMA, sums by two-sum.  Used
// for the per-particle sums, where float64 arithmetic would dominate the run time
// on GB300 (float64 rate 1/64 of float32).
struct dfloat {
    float hi, lo;
};

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

__device__ __forceinline__ void df_add(dfloat &x, float v)
{
    float s, e;
    two_sum(x.hi, v, s, e);
    x.hi = s;
    x.lo = __fadd_rn(x.lo, e);
}

__device__ __forceinline__ void df_add_prod(dfloat &x, float a, float b)
{
    const float p = __fmul_rn(a, b);
    const float pe = __fmaf_rn(a, b, -p);      // a * b = p + pe exactly
    float s, e;
    two_sum(x.hi, p, s, e);
    x.hi = s;
    x.lo = __fadd_rn(x.lo, __fadd_rn(e, pe));
}

__device__ __forceinline__ void df_merge(dfloat &x, const dfloat &y)
{
    float s, e;
    two_sum(x.hi, y.hi, s, e);
    x.hi = s;
    x.lo = __fadd_rn(x.lo, __fadd_rn(e, y.lo));
}

template <int N>
__device__ __forceinline__ void warp_sum_df(dfloat (&v)[N])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < N; ++c) {
            dfloat y;
            y.hi = __shfl_xor_sync(0xffffffffu, v[c].hi, o);
            y.lo = __shfl_xor_sync(0xffffffffu, v[c].lo, o);
            df_merge(v[c], y);
        }
}

template <int N>
__device__ __forceinline__ void warp_sum_f64(double (&v)[N])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < N; ++c) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
}

// ---------------------------------------------------------------- launchers
// Every launcher enqueues on `st` and returns the launch status.
// ---------------------------------------------------------------- layout
// Several objects can be optimised in one pass.  Particles are numbered object
// by object, preshape by preshape: group g = o * P + p holds the K_g particles
// grp_off[g] .. grp_off[g + 1] - 1 of preshape p on object o.
struct ObjMeta {
    const float4 *R;          // [M] object points
    const ulonglong2 *Rx;     // [Mpad] screening layout (pairs of (-2r, |r|^2)), Mpad = whole tiles
    const float *Rt;          // [Mpad / 128] augmented tiles of the tensor-core kernel (8 KB each)
    const int2 *nodes;        // matching cells (k_cells.cu): tables and nodes, and the
    const int *leaves;        // points that can be nearest per cell; null where not built
    const float4 *C;          // [Mc] collision points (may alias R)
    const float4 *Csort;      // [Mc] the same in spatial order per segment, w = index in the segment
    const float4 *Cball;      // [ceil(Mc / 32)] bounding balls of 32 points of Csort (w = radius)
    int M, Mpad, Mc;
    int pfirst, np;           // first particle and number of particles of this object
    long long colidx_base;    // this object's collision lists start here ([np][Mc] ints)
    long long colmap_base;    // and their bit maps ([np][ceil(Mc / 32)] words)
};

struct Layout {
    int P, N, G, nobj, T;     // preshapes, gripper points, groups, objects, particles
    const int *part_grp;      // [T] group of every particle
    const int *grp_off;       // [G + 1] first particle of every group
    const ObjMeta *obj;       // [nobj]
    const double *com;        // [nobj][3] object centroids (CoM)
    const float4 *frame;      // [nobj] screening frame: centre c (x, y, z; the bounding-box
                              // centre) and w = max |fl(r - c)| rounded up (see ref_prep_kernel)
};

// A unit of forward-matching work: queries [q0, q0 + nq) of the flattened
// (particle, gripper point) space, all on object `obj` (nq <= 1024).
struct FwdItem {
    long long q0;
    int nq, obj;
};

struct FwdArgs {
    Layout L;
    const float4 *S;         // [P][N] gripper points (gripper frame)
    const float4 *Ssort;     // [P][N] the same along a space-filling curve, w = own index (cells only)
    const float *theta;      // [T][8]
    const FwdItem *items;    // [n_items] work items (null: object 0, consecutive 1024-query items)
    const int *cta_off;      // [grid + 1]: CTA b runs items cta_off[b] .. cta_off[b+1]-1 (null: round-robin)
    int n_items;
    int item_queries;        // queries per item when items is null
    int check_err;           // float32 shapes: skip the work if the error word is set
    int *err;                // error word
    int *nn_idx;             // [T][N] nearest object point per query
    float *dbg_d2;           // [T][N] or null
    float *dbg_sp;           // [T][N][3] or null
    int4 *cand;              // [T][N] tensor-core shape only: candidate chunks per query
    int variant;             // kernel shape (0 .. kFwdVariants - 1), chosen by the autotuner
    int cells;               // tensor-core shape only: match through the objects' cells instead
    int expire_test;         // float32 shapes: the first copy wait of a CTA waits on an mbarrier
                             // that nothing arrives at, for kTestWaitCycles (tests the timeout path)
};
constexpr int kFwdItemQueries = 1024;  // queries per forward-matching work item
constexpr int kFwdVariants = 8;        // kernel shapes of the forward matching (7: tensor cores)
cudaError_t launch_fwd_match(const FwdArgs &a, cudaStream_t st);
// The tensor-core shape leaves the exact choice to a second kernel (launch it after
// launch_fwd_match on the same stream); the float32 shapes make it themselves.
inline bool fwd_has_exact_kernel(const FwdArgs &a) { return a.variant == kFwdVariants - 1 && !a.cells; }
cudaError_t launch_fwd_exact(const FwdArgs &a, cudaStream_t st);
int fwd_grid_size();                   // first call sets the kernels' attributes
int fwd_shape_grid(int v);             // CTAs of kernel shape v (a whole number per SM)
int fwd_shape_threads(int v);          // threads per CTA of kernel shape v
int fwd_shape_queries(int v);          // queries per work item (at most) of kernel shape v
const char *fwd_variant_name(int v);
cudaError_t init_collision_attributes();
cudaError_t init_update_attributes();
// Preparation of an object cloud (see k_match.cu); the scratch is cleared before its first use.
constexpr int kRefCtas = 32;
struct RefScratch {
    unsigned lo[3], hi[3];            // bounding box: largest ~key / key (order_key) so far
    unsigned done, pad;
    unsigned long long rad;           // bits of the largest |r - c|^2 (float64)
    double part[kRefCtas][3];         // the centroid's sums
};
cudaError_t launch_ref_prep(const float *xyz, int M, int Mpad, float4 *R, void *Rx, float4 *frame, double *com,
                            RefScratch *scr, int *err, cudaStream_t st);
cudaError_t launch_minibatch(const float4 *R, const int *idx, int n, int Mpad, float4 *out, void *Rx, const float4 *frame,
                             ObjMeta *dst, const ObjMeta &v, cudaStream_t st);
int fwd_item_queries(int v, long long queries);
cudaError_t launch_tc_ref_prep(const float4 *R, int M, int Mpad, const float4 *frame, void *Rt, cudaStream_t st);
size_t tc_ref_bytes(int Mpad);         // bytes of the tensor-core object tiles
cudaError_t launch_fwd_match_tc(const FwdArgs &a, cudaStream_t st);
cudaError_t launch_tc_exact(const FwdArgs &a, cudaStream_t st);
int fwd_tc_grid();
int fwd_tc_threads();

// Matching cells (k_cells.cu).  One object's build: its points and frame, the tables it
// leaves behind (nodes, leaves) and the scratch of the build (lists and records of two
// levels in turn, counters cleared by the caller).
constexpr int kCellCounters = 64;      // ints per object
constexpr int kCellBatch = 32;         // objects per launch
struct CellBuild {
    const float4 *R;
    const float4 *frame;
    int2 *nodes;
    int *leaves, *lists;
    void *recs;
    int *ctr;
    int M, leaf_cap, list_cap, cell_cap, node_cap;
    int log_factor;           // near cells reach 2^log_factor times the power of two above the radius
    float tol;                // positions looked up may be off by 0.4 tol times the radius
};
// Cells of objects, and of gripper clouds in the gripper frame (see collide_cells_kernel for the tolerance).  Colliding
// points lie in the gripper's body, which may reach far beyond a cloud that covers its fingertips only: with the near
// cells alone a cloud a fifth of the body's size took 1033 us per pass against 217 without cells.
constexpr int kObjectCells = 2, kGripperCells = 1;     // (log_factor)
constexpr float kGripperTol = 1.25e-4f;
struct CellBuildBatch {
    CellBuild b[kCellBatch];
};
struct CellSizes {
    int leaf_cap, list_cap, cell_cap, node_cap;   // ints, ints per level, records per level, nodes
    size_t rec_bytes;                             // records of both levels
};
CellSizes cell_sizes(int M);
cudaError_t launch_cells_build(const CellBuildBatch &batch, int n, cudaStream_t st);
cudaError_t launch_cells_match(const FwdArgs &a, cudaStream_t st);
constexpr int kCellSample = 1024;      // warps looked at by launch_cells_cost
struct CellCost {
    unsigned long long sum[2];
    unsigned most[2], seq, pad;
};
cudaError_t launch_cells_cost(const FwdArgs &a, CellCost *cost, CellCost *host, unsigned seq, double *share, cudaStream_t st);
cudaError_t launch_gripper_cloud(const float4 *S, int N, float4 *out, float4 *frame, double *out12, cudaStream_t st);
cudaError_t init_cells_attributes();

constexpr int kColChunk = 64;          // colliding points per partial sum, and per work item of collide_nn_kernel

// Spatial order of the collision clouds: segments of at most kColSegment points, several
// (of several objects) per launch.
constexpr int kColSegment = 65536;
struct CloudSort {
    const float4 *src;
    float4 *dst, *balls;
    int n;
};
constexpr int kCloudBatch = 64;
struct CloudBatch {
    CloudSort b[kCloudBatch];
};
cudaError_t launch_sort_clouds(const CloudBatch &batch, int n, cudaStream_t st);

struct CollideArgs {
    Layout L;
    const float *theta;       // [T][8]
    const SdfMeta *meta;      // [P]
    const float4 *S;          // [P][N]
    int *ncol;                // [T]
    int *colidx;              // colliding points, ascending (see ObjMeta::colidx_base)
    int *colsrt;              // the same points as positions in Csort, in no particular order (without cells colnn, which
                              // the reverse matching overwrites)
    int *colnn;               // like colidx: nearest gripper point of each
    int2 *colmap;             // bit map of the colliding points: words (bits, number of earlier bits),
                              // only those with bits written (see ObjMeta::colmap_base)
    int *col_items;           // (count, next) of the reverse-matching work list
    int *col_list;            // [2 * items] (particle, item) pairs
    int cells;                // reverse matching through the gripper clouds' cells
    const int2 *pre_nodes;    // [P][pre_node_cap]
    const int *pre_leaves;    // [P][pre_leaf_cap]
    const float4 *pre_frame;  // [P]
    int pre_node_cap, pre_leaf_cap;
    int most_items;           // work-list entries at most
    int most_points;          // points of the largest collision cloud
};
cudaError_t launch_collide(const CollideArgs &a, cudaStream_t st);
cudaError_t launch_collide_nn(const CollideArgs &a, cudaStream_t st);

struct UpdateArgs {
    Layout L;
    float *theta;             // [T][8] in/out
    const float4 *S;          // [P][N]
    const int *nn_idx;        // [T][N] forward correspondences
    const int *ncol;          // [T]
    const int *colidx, *colnn;    // colliding points and their gripper points (see CollideArgs)
    const double *pconst;     // [P][12]: sum s (3), sum s s^T (xx,xy,xz,yy,yz,zz), pad
    double w_com;
    int mode;                 // 0: evaluate only, 1: SVGD step, 2: SGD step
    float gamma, eta_svgd, eta_sgd;
    int bandwidth_mode;
    float h_fixed;
    float conv_tol;           // < 0 disables
    double *cost;             // [T]
    double *grad;             // [T][8]
    double *prev_cost;        // [T]
    int *frozen;              // [T]
    float *phi;               // [T][8]
    float *h;                 // [G]
    int *col_items;           // collision work-list counters (count, next), cleared for the next pass
    float prior_t_sigma;      // Gaussian prior on t around the object's CoM (<= 0: off)
    float prior_q_kappa;      // von Mises prior on q (<= 0: off)
    float prior_q_mean[4];    // its unit mean
    const int *err;           // error word: a kernel of the pass found an error, skip the work
};
cudaError_t launch_finalize(const UpdateArgs &a, cudaStream_t st);   // cost/gradient, convergence, SGD step
cudaError_t launch_stein(const UpdateArgs &a, cudaStream_t st);      // SVGD step (mode 1)

cudaError_t launch_pack_points(const float *xyz, int n, float4 *out, int *err, cudaStream_t st);
cudaError_t launch_check_finite(const float *v, long long n, int *err, cudaStream_t st);
cudaError_t launch_fibonacci(const Layout &L, float radius, int mode, float *theta, cudaStream_t st);
cudaError_t launch_store_meta(ObjMeta *dst, const ObjMeta &v, cudaStream_t st);
cudaError_t launch_set_theta(const float *theta7, int T, float *theta8, int *err, cudaStream_t st);
cudaError_t launch_sdf_clear(int nx, int ny, int nz, unsigned char *away, unsigned char *clear, cudaStream_t st);
cudaError_t launch_sdf_pack_cells(const float *grid, int nx, int ny, int nz, float4 *cells, unsigned char *away,
                                  cudaStream_t st);
size_t sdf_cells_bytes(int nx, int ny, int nz);
cudaError_t launch_select(const Layout &L, const double *cost, const int *ncol, int *order, cudaStream_t st);
cudaError_t launch_uniform_groups(int *part_grp, int *grp_off, int P, int K, cudaStream_t st);

}  // namespace asicp
