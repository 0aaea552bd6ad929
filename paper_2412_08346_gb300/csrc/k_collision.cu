// The collision term: SDF test of the collision cloud in every particle's gripper
// frame (Eq. 12, Section IV-C) and the reverse matching of the colliding points
// onto the transformed contact cloud (Eq. 18).
#include "cells.cuh"

#include <climits>

namespace asicp {

namespace {
constexpr int kColThreads = 256;       // reverse matching
constexpr int kSegWords = kColSegment / 32;      // words of a segment's bit map = most chunks of a segment
constexpr int kTestB = 4;         // chunks per warp whose loads overlap

// Whether point (x, y, z) of the gripper frame collides: inside the grid's node box (the grid covers
// the gripper, so a point outside is not in it) and trilinear value > 0 (Eq. 12).  Only a
// cell with a positive corner (clear 0) can interpolate to a positive value; its eight
// corners come from the corner-packed copy of the grid, two float4 from one 32-byte sector.
__device__ __forceinline__ bool sdf_hit(const SdfMeta &m, float x, float y, float z)
{
    const float ux = __fdiv_rn(__fsub_rn(x, m.ox), m.voxel);
    const float uy = __fdiv_rn(__fsub_rn(y, m.oy), m.voxel);
    const float uz = __fdiv_rn(__fsub_rn(z, m.oz), m.voxel);
    if (!(ux >= 0.f && ux <= (float)(m.nx - 1) && uy >= 0.f && uy <= (float)(m.ny - 1) &&
          uz >= 0.f && uz <= (float)(m.nz - 1)))
        return false;
    const int ix = min((int)floorf(ux), m.nx - 2);
    const int iy = min((int)floorf(uy), m.ny - 2);
    const int iz = min((int)floorf(uz), m.nz - 2);
    const size_t at = (size_t)ix + (size_t)(m.nx - 1) * ((size_t)iy + (size_t)(m.ny - 1) * iz);
    if (__ldg(m.clear + at) != 0) return false;
    const float fx = ux - (float)ix, fy = uy - (float)iy, fz = uz - (float)iz;
    const float4 *cell = m.cells + 2 * at;
    const float4 z0 = __ldg(cell), z1 = __ldg(cell + 1);
    const float c000 = z0.x, c100 = z0.y, c010 = z0.z, c110 = z0.w;
    const float c001 = z1.x, c101 = z1.y, c011 = z1.z, c111 = z1.w;
    const float gx = 1.f - fx, gy = 1.f - fy, gz = 1.f - fz;
    const float val = gx * gy * gz * c000 + fx * gy * gz * c100 + gx * fy * gz * c010 + fx * fy * gz * c110 +
                      gx * gy * fz * c001 + fx * gy * fz * c101 + gx * fy * fz * c011 + fx * fy * fz * c111;
    return val > 0.f;
}

// clear of the cell that holds point (x, y, z), found without divisions: it may be a neighbour of the
// cell sdf_hit finds (inv = 1 / voxel is rounded), so the point cannot collide when this is above
// 1.  Points outside the grid get the nearest cell's.
__device__ __forceinline__ int cell_clear(const SdfMeta &m, float inv, float x, float y, float z)
{
    const int ix = (int)fminf(fmaxf((x - m.ox) * inv, 0.f), (float)(m.nx - 2));
    const int iy = (int)fminf(fmaxf((y - m.oy) * inv, 0.f), (float)(m.ny - 2));
    const int iz = (int)fminf(fmaxf((z - m.oz) * inv, 0.f), (float)(m.nz - 2));
    return __ldg(m.clear + (size_t)ix + (size_t)(m.nx - 1) * ((size_t)iy + (size_t)(m.ny - 1) * iz));
}

// Whether a ball of radius rho around the gripper-frame point (x, y, z) can hold a colliding point:
// clear is the distance in cells (largest coordinate) from a cell to the nearest one with a
// positive corner, and rho voxels reach ceil(rho) cells.  A centre outside the grid is
// moved to the nearest cell, which only shortens the distance.  The slack covers the rounding
// of the centre's and the points' coordinates (1e-6 of them).
__device__ __forceinline__ bool ball_may_hit(const SdfMeta &m, float inv, float x, float y, float z, float rho)
{
    const float reach = (rho + 1e-5f * (fabsf(x) + fabsf(y) + fabsf(z) + fabsf(m.ox) + fabsf(m.oy) + fabsf(m.oz))) * inv;
    return !((float)cell_clear(m, inv, x, y, z) > ceilf(reach + 0.02f));
}

}  // namespace

// Items of the reverse matching: the points of a warp (through the cells), or kColChunk.
__host__ __device__ constexpr int col_item_points(bool cells) { return cells ? 32 : kColChunk; }

// One CTA per particle: every collision point c is mapped into the gripper frame,
// c' = R^T (c - t), and kept when the preshape's distance field is > 0 there (Eq. 12).  The
// collision cloud is held in spatial order (sort_cloud_kernel) in chunks of 32 points with their
// bounding balls: a chunk whose ball is clear of the gripper is skipped, a warp tests the
// points of another one.  Hits are noted as they come (neighbours stay together, which is how
// the reverse matching wants them) and set bits by the points' own indices, which are then
// listed in ascending order, so results depend neither on the order of the chunks nor on
// scheduling.  Clouds beyond kColSegment points are taken segment by segment.
// Measured on GB300 (per pass; before: every point tested, and the sums of the forward pairs in the
// same CTA): 3 x 256 particles, M 8192 20 us against 58; 3 x 1024, M 65536 0.27 ms against 1.19;
// 2 x 64, Mc 4501 13 us against 27.  A quarter of the chunks survive (balls of 10 mm at 8192
// points against voxels of 3.2 mm); at 0.27 ms it takes three quarters of the issue slots.
template <int kTestThreads>
__global__ void __launch_bounds__(kTestThreads, 1280 / kTestThreads) collide_kernel(const CollideArgs a)
{
    const int pk = blockIdx.x;
    const int grp = a.L.part_grp[pk], p = grp % a.L.P;
    const ObjMeta &om = a.L.obj[grp / a.L.P];
    __shared__ unsigned s_bits[kSegWords];
    __shared__ unsigned short s_chunk[kSegWords];
    __shared__ int s_n, s_hits, s_wsum[kTestThreads / 32], s_base;
    const float *th = a.theta + (size_t)pk * 8;
    const float tx = th[0], ty = th[1], tz = th[2];
    float Rm[9];
    quat_rot_f32(th[3], th[4], th[5], th[6], Rm);
    const SdfMeta m = a.meta[p];
    const float inv = 1.f / m.voxel;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, Mc = om.Mc;
    auto local = [&](float4 c, float &lx, float &ly, float &lz) {
        const float dx = __fsub_rn(c.x, tx), dy = __fsub_rn(c.y, ty), dz = __fsub_rn(c.z, tz);
        lx = __fmaf_rn(Rm[0], dx, __fmaf_rn(Rm[3], dy, __fmul_rn(Rm[6], dz)));
        ly = __fmaf_rn(Rm[1], dx, __fmaf_rn(Rm[4], dy, __fmul_rn(Rm[7], dz)));
        lz = __fmaf_rn(Rm[2], dx, __fmaf_rn(Rm[5], dy, __fmul_rn(Rm[8], dz)));
    };
    const long long first = om.colidx_base + (long long)(pk - om.pfirst) * Mc;
    int *colidx = a.colidx + first, *colsrt = a.colsrt + first;
    int2 *colmap = a.colmap + om.colmap_base + (long long)(pk - om.pfirst) * ((Mc + 31) / 32);
    int count = 0;
    if (threadIdx.x == 0) s_hits = 0;
    for (int seg = 0; seg < Mc; seg += kColSegment) {
        const int pts = min(kColSegment, Mc - seg), chunks = (pts + 31) / 32;
        const float4 *balls = om.Cball + seg / 32, *cloud = om.Csort + seg;
        for (int w = threadIdx.x; w < chunks; w += kTestThreads) s_bits[w] = 0u;
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        for (int c0 = 0; c0 < chunks; c0 += kTestThreads) {
            const int c = c0 + threadIdx.x;
            bool may = false;
            if (c < chunks) {
                const float4 b = __ldg(balls + c);
                float lx, ly, lz;
                local(b, lx, ly, lz);
                may = ball_may_hit(m, inv, lx, ly, lz, b.w);
            }
            const unsigned bal = __ballot_sync(0xffffffffu, may);
            int base = 0;
            if (lane == 0 && bal) base = atomicAdd(&s_n, __popc(bal));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (may) s_chunk[base + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)c;
        }
        __syncthreads();
        const int n = s_n;
        // kTestB chunks per warp at a time: their loads are in flight together
        for (int k0 = warp; k0 < n; k0 += kTestB * (kTestThreads / 32)) {
            float4 c[kTestB];
            int near[kTestB], at[kTestB];
#pragma unroll
            for (int u = 0; u < kTestB; ++u) {
                const int k = k0 + u * (kTestThreads / 32);
                at[u] = (k < n ? s_chunk[k] * 32 : kColSegment) + lane;
                c[u] = __ldg(cloud + min(at[u], pts - 1));
            }
#pragma unroll
            for (int u = 0; u < kTestB; ++u) {
                float lx, ly, lz;
                local(c[u], lx, ly, lz);
                near[u] = cell_clear(m, inv, lx, ly, lz);
                c[u].x = lx; c[u].y = ly; c[u].z = lz;
            }
#pragma unroll
            for (int u = 0; u < kTestB; ++u) {
                const bool hit = near[u] <= 1 && at[u] < pts && sdf_hit(m, c[u].x, c[u].y, c[u].z);
                const unsigned bal = __ballot_sync(0xffffffffu, hit);
                if (!bal) continue;
                int base = 0;
                if (lane == 0) base = atomicAdd(&s_hits, __popc(bal));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (hit) {
                    const int own = __float_as_int(c[u].w);
                    atomicOr(&s_bits[own >> 5], 1u << (own & 31));
                    colsrt[base + __popc(bal & ((1u << lane) - 1u))] = seg + at[u];
                }
            }
        }
        __syncthreads();
        // list the set bits in ascending order: kTestThreads words a round
        for (int w0 = 0; w0 < chunks; w0 += kTestThreads) {
            const int w = w0 + threadIdx.x;
            unsigned bits = w < chunks ? s_bits[w] : 0u;
            int inc = __popc(bits);
            const int mine = inc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) s_wsum[warp] = inc;
            __syncthreads();
            int before = inc - mine, tot = 0;
#pragma unroll
            for (int v = 0; v < kTestThreads / 32; ++v) {
                const int y = s_wsum[v];
                before += v < warp ? y : 0;
                tot += y;
            }
            int *out = colidx + count + before;
            if (bits) colmap[seg / 32 + w] = make_int2((int)bits, count + before);
            while (bits) {
                const int b = __ffs(bits) - 1;
                bits &= bits - 1;
                *out++ = seg + w * 32 + b;
            }
            count += tot;
            __syncthreads();
        }
    }
    // queue this particle's colliding points for the reverse matching
    const int item = col_item_points(a.cells), used = (count + item - 1) / item;
    if (threadIdx.x == 0) {
        a.ncol[pk] = count;
        s_base = used > 0 ? atomicAdd(&a.col_items[0], used) : 0;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < used; c += kTestThreads)
        reinterpret_cast<int2 *>(a.col_list)[s_base + c] = make_int2(pk, c);
}

// Spatial order of (a segment of) a collision cloud, one CTA each: points sorted into the 32^3
// bins of their bounding box, bins along a space-filling curve (the order within a bin does not
// matter), w = the point's index in the segment; and per 32 points in that order a bounding
// ball (w = its radius, rounded up).
__global__ void __launch_bounds__(1024) sort_cloud_kernel(const CloudBatch batch)
{
    const CloudSort &b = batch.b[blockIdx.x];
    extern __shared__ int s_bin[];
    __shared__ float s_lo[3][32], s_hi[3][32];
    __shared__ int s_sum[32];
    constexpr int kBins = 32 * 32 * 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = b.n;
    float lo[3], hi[3];
    for (int k = 0; k < 3; ++k) { lo[k] = __int_as_float(0x7f800000); hi[k] = -lo[k]; }
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float4 p = __ldg(b.src + i);
        lo[0] = fminf(lo[0], p.x); lo[1] = fminf(lo[1], p.y); lo[2] = fminf(lo[2], p.z);
        hi[0] = fmaxf(hi[0], p.x); hi[1] = fmaxf(hi[1], p.y); hi[2] = fmaxf(hi[2], p.z);
    }
    for (int i = threadIdx.x; i < kBins; i += blockDim.x) s_bin[i] = 0;
    for (int k = 0; k < 3; ++k) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
        if (lane == 0) { s_lo[k][warp] = lo[k]; s_hi[k][warp] = hi[k]; }
    }
    __syncthreads();
    float ext = 1e-30f;
    for (int k = 0; k < 3; ++k) {
        lo[k] = s_lo[k][lane];
        hi[k] = s_hi[k][lane];
        for (int o = 16; o > 0; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
        ext = fmaxf(ext, hi[k] - lo[k]);
    }
    const float scale = 32.f / ext;
    auto bin = [&](float4 p) {
        auto spread = [](unsigned v) { v = (v | (v << 8)) & 0x100fu; v = (v | (v << 4)) & 0x10c3u; return (v | (v << 2)) & 0x1249u; };
        const unsigned x = (unsigned)min(max((int)((p.x - lo[0]) * scale), 0), 31),
                       y = (unsigned)min(max((int)((p.y - lo[1]) * scale), 0), 31),
                       z = (unsigned)min(max((int)((p.z - lo[2]) * scale), 0), 31);
        return (int)(spread(x) | (spread(y) << 1) | (spread(z) << 2));
    };
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += blockDim.x) atomicAdd(&s_bin[bin(__ldg(b.src + i))], 1);
    __syncthreads();
    // exclusive scan over the bins: warp w's 1024, then the warps
    int *mine = s_bin + warp * (kBins / 32);
    int carry = 0;
    for (int k = 0; k < kBins / 32; k += 32) {
        const int v = mine[k + lane];
        int inc = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        mine[k + lane] = carry + inc - v;
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) s_sum[warp] = carry;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += s_sum[w];
    for (int k = lane; k < kBins / 32; k += 32) mine[k] += before;
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        float4 p = __ldg(b.src + i);
        const int at = atomicAdd(&s_bin[bin(p)], 1);
        p.w = __int_as_float(i);
        b.dst[at] = p;
    }
    __syncthreads();
    for (int c = warp; c * 32 < n; c += 32) {
        const bool in = c * 32 + lane < n;
        const float4 p = b.dst[min(c * 32 + lane, n - 1)];
        float l[3] = {p.x, p.y, p.z}, h[3] = {p.x, p.y, p.z};
        for (int k = 0; k < 3; ++k)
            for (int o = 16; o > 0; o >>= 1) {
                l[k] = fminf(l[k], __shfl_xor_sync(0xffffffffu, l[k], o));
                h[k] = fmaxf(h[k], __shfl_xor_sync(0xffffffffu, h[k], o));
            }
        float4 ball = make_float4(0.5f * l[0] + 0.5f * h[0], 0.5f * l[1] + 0.5f * h[1], 0.5f * l[2] + 0.5f * h[2], 0.f);
        const float x = p.x - ball.x, y = p.y - ball.y, z = p.z - ball.z;
        float d = in ? x * x + y * y + z * z : 0.f;
        for (int o = 16; o > 0; o >>= 1) d = fmaxf(d, __shfl_xor_sync(0xffffffffu, d, o));
        ball.w = sqrtf(d) * 1.00001f + 1e-30f;
        if (lane == 0) b.balls[c] = ball;
    }
}

cudaError_t launch_sort_clouds(const CloudBatch &batch, int n, cudaStream_t st)
{
    sort_cloud_kernel<<<n, 1024, 32 * 32 * 32 * sizeof(int), st>>>(batch);
    return cudaGetLastError();
}

namespace {
__device__ __forceinline__ unsigned long long pk2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void upk2(unsigned long long v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

__device__ __forceinline__ unsigned long long ffma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ float fmin3(float a, float b, float c)
{
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// (best, bi) <- the smaller of itself and the partner lane's, ties to the lower index.
__device__ __forceinline__ void argmin_xor(float &best, int &bi, int o)
{
    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob < best || (ob == best && oi < bi)) { best = ob; bi = oi; }
}

}  // namespace

// Persistent: CTAs take (particle, chunk of kColChunk colliding points) items
// from the list the collision kernel filled.  Per item the particle's
// transformed contact cloud S' is built in shared memory twice, both arranged
// by lane chunks (chunk l = points l + 32 k): in the screening layout
// (-2 s', |s'|^2), point pairs (l + 64 m, l + 32 + 64 m) at slot 32 m + l, and
// exact (float4), chunk l contiguous with a stride of KC + 1 (no bank
// conflicts).  Each warp matches kQW colliding points c:
//  1. screening, relative to the particle's translation t (so the error does not
//     grow with the distance from the origin): with b = fl(s' - t) and
//     a = fl(c - t), lane l evaluates d~ = |b|^2 - 2 a.b over chunk l (packed
//     f32x2 FMAs, 3-input min); warp min-reductions give the best chunk minimum
//     b1 (lane l1, the lowest on ties) and the best of the other chunks b2;
//  2. exact choice: with delta = u (9 B^2 + 10.1 A B) bounding the error of d~
//     against |c - s'|^2 + const (B = max |b|, A = |a|: the float32 evaluation
//     within u (7 B^2 + 6.1 A B), the rounding of a and b within u (2 B^2 + 4 A B)
//     beyond a term that does not depend on s'), the nearest point lies in chunk
//     l1 unless b2 <= b1 + 2 delta; four lanes per colliding point re-evaluate chunk l1 with the
//     exact-form distance, ties to the lowest index; in the rare other case the
//     warp scans the whole cloud that way.
// For gripper clouds without cells (few points, or cells not built yet).
__global__ void __launch_bounds__(kColThreads) collide_nn_kernel(const CollideArgs a)
{
    constexpr int kWarps = kColThreads / 32;
    constexpr int kQW = kColChunk / kWarps;                  // colliding points per warp
    static_assert(kQW == 8 && kColChunk == 64, "lane groups of four per colliding point");
    extern __shared__ __align__(16) unsigned char smem_nn[];
    const int N = a.L.N;
    const int Npad = (N + 63) / 64 * 64;
    const int KC = Npad / 32, KCs = KC + 1;                  // points per lane chunk, exact-layout stride
    ulonglong2 *sXA = reinterpret_cast<ulonglong2 *>(smem_nn);             // [Npad/2] {-2x pair}{-2y pair}
    ulonglong2 *sXB = sXA + Npad / 2;                                      // [Npad/2] {-2z pair}{w pair}
    float4 *sE = reinterpret_cast<float4 *>(sXB + Npad / 2);               // [32][KC + 1] exact S'
    __shared__ float4 sC[kColChunk];                          // colliding points of the item
    __shared__ int s_item;
    __shared__ float s_smax[kWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slots = Npad / 64;                 // point pairs per lane
    // Two barriers per item.  The first parts the writes of the transformed cloud, sC and
    // s_smax from their reads; thread 0 takes the next item right after it (every thread has
    // read s_item at the top of the loop by then).  After the second nothing of this item is
    // read any more, and s_item holds the next one.
    if (threadIdx.x == 0) s_item = atomicAdd(&a.col_items[1], 1);
    __syncthreads();
    for (;;) {
        const int item = s_item;
        if (item >= a.col_items[0]) break;
        const int pk = a.col_list[2 * item], chunk = a.col_list[2 * item + 1];
        const int grp = a.L.part_grp[pk], p = grp % a.L.P;
        const ObjMeta om = a.L.obj[grp / a.L.P];
        const int n = a.ncol[pk];
        const int *colidx = a.colidx + om.colidx_base + (long long)(pk - om.pfirst) * om.Mc;
        const int l0 = chunk * kColChunk;
        const float *th = a.theta + (size_t)pk * 8;
        const float tx = th[0], ty = th[1], tz = th[2];
        float Rm[9];
        quat_rot_f32(th[3], th[4], th[5], th[6], Rm);
        const float4 *S = a.S + (size_t)p * N;
        if (threadIdx.x < kColChunk) {
            const int j = threadIdx.x;
            float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
            if (l0 + j < n) c = om.C[colidx[l0 + j]];
            sC[j] = c;
        }
        float smax2 = 0.f;
        for (int q = threadIdx.x; q < Npad / 2; q += kColThreads) {
            const int l = q & 31, m = q >> 5;
            float ax[2], ay[2], az[2], w[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = l + 32 * h + 64 * m;
                float4 e = make_float4(__int_as_float(0x7f800000), __int_as_float(0x7f800000),
                                       __int_as_float(0x7f800000), 0.f);
                if (r < N) {
                    const float4 sv = S[r];
                    const float3 o = xform_f32(Rm, tx, ty, tz, sv.x, sv.y, sv.z);
                    e = make_float4(o.x, o.y, o.z, 0.f);
                    const float bx = __fsub_rn(o.x, tx), by = __fsub_rn(o.y, ty), bz = __fsub_rn(o.z, tz);
                    ax[h] = -2.f * bx; ay[h] = -2.f * by; az[h] = -2.f * bz;
                    w[h] = __fmaf_rn(bx, bx, __fmaf_rn(by, by, __fmul_rn(bz, bz)));
                    smax2 = fmaxf(smax2, w[h]);
                } else {
                    ax[h] = ay[h] = az[h] = 0.f;
                    w[h] = __int_as_float(0x7f800000);
                }
                sE[l * KCs + 2 * m + h] = e;
            }
            ulonglong2 A, B;
            A.x = pk2(ax[0], ax[1]); A.y = pk2(ay[0], ay[1]);
            B.x = pk2(az[0], az[1]); B.y = pk2(w[0], w[1]);
            sXA[q] = A;
            sXB[q] = B;
        }
        for (int o = 16; o > 0; o >>= 1) smax2 = fmaxf(smax2, __shfl_xor_sync(0xffffffffu, smax2, o));
        if (lane == 0) s_smax[warp] = smax2;
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(&a.col_items[1], 1);
        float sm2 = 0.f;
        for (int w8 = 0; w8 < kWarps; ++w8) sm2 = fmaxf(sm2, s_smax[w8]);
        const float smax = sqrtf(sm2) * 1.0001f;

        // colliding points of this warp (warp-uniform): a warp whose eight slots are all past the
        // particle's count (the padding of its last item) skips the matching
        const int g = lane >> 2, gs = lane & 3;       // lane group g works on colliding point g
        const float4 cq = sC[warp * kQW + g];
        float best = __int_as_float(0x7f800000);
        int bi = 0x7fffffff;
        if (l0 + warp * kQW < n) {
            // 1. screening of this warp's colliding points, lane l over chunk l
            unsigned long long qx[kQW], qy[kQW], qz[kQW];
            float cm[kQW];
#pragma unroll
            for (int q = 0; q < kQW; ++q) {
                const float4 c = sC[warp * kQW + q];
                const float ax = __fsub_rn(c.x, tx), ay = __fsub_rn(c.y, ty), az = __fsub_rn(c.z, tz);
                qx[q] = pk2(ax, ax); qy[q] = pk2(ay, ay); qz[q] = pk2(az, az);
                cm[q] = __int_as_float(0x7f800000);
            }
            for (int m = 0; m < slots; ++m) {
                const ulonglong2 A = sXA[m * 32 + lane];
                const ulonglong2 B = sXB[m * 32 + lane];
#pragma unroll
                for (int q = 0; q < kQW; ++q) {
                    const unsigned long long d = ffma2(qx[q], A.x, ffma2(qy[q], A.y, ffma2(qz[q], B.x, B.y)));
                    float d0, d1;
                    upk2(d, d0, d1);
                    cm[q] = fmin3(cm[q], d0, d1);
                }
            }
            // best chunk l1 (lowest lane on ties) and whether another chunk may hold the nearest point
            int my_l1 = 0;
            unsigned full_scan = 0u;
#pragma unroll
            for (int q = 0; q < kQW; ++q) {
                const unsigned key = order_key(cm[q]);
                const unsigned k1 = __reduce_min_sync(0xffffffffu, key);
                const int l1 = __ffs(__ballot_sync(0xffffffffu, key == k1)) - 1;
                const unsigned k2 = __reduce_min_sync(0xffffffffu, lane == l1 ? 0xffffffffu : key);
                const float4 c = sC[warp * kQW + q];
                const float ax = __fsub_rn(c.x, tx), ay = __fsub_rn(c.y, ty), az = __fsub_rn(c.z, tz);
                const float cn = sqrtf(ax * ax + ay * ay + az * az) * 1.001f;
                const float win = 2.02f * 5.9604645e-8f * (9.f * smax * smax + 10.1f * cn * smax);
                if (key_float(k2) <= key_float(k1) + win) full_scan |= 1u << q;
                if (g == q) my_l1 = l1;
            }
            // 2. exact choice: four lanes per colliding point over its chunk l1
            for (int k = gs; k < KC; k += 4) {
                const int r = my_l1 + 32 * k;
                if (r >= N) break;
                const float4 e = sE[my_l1 * KCs + k];
                const float d = dist2_f32(e.x, e.y, e.z, cq.x, cq.y, cq.z);
                if (d < best) { best = d; bi = r; }
            }
            argmin_xor(best, bi, 1);
            argmin_xor(best, bi, 2);
            if (bi >= N) bi = 0;     // no finite distance at all (not reached with finite inputs)
            // rare: the whole cloud, lane l over chunk l
            while (full_scan) {
                const int q = __ffs(full_scan) - 1;
                full_scan &= full_scan - 1;
                const float4 c = sC[warp * kQW + q];
                float fb = __int_as_float(0x7f800000);
                int fi = 0x7fffffff;
                for (int k = 0; k < KC; ++k) {
                    const int r = lane + 32 * k;
                    if (r >= N) break;
                    const float4 e = sE[lane * KCs + k];
                    const float d = dist2_f32(e.x, e.y, e.z, c.x, c.y, c.z);
                    if (d < fb) { fb = d; fi = r; }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) argmin_xor(fb, fi, o);
                if (g == q) { best = fb; bi = fi < N ? fi : 0; }
            }
        }
        if (gs == 0 && l0 + warp * kQW + g < n)
            a.colnn[om.colidx_base + (long long)(pk - om.pfirst) * om.Mc + l0 + warp * kQW + g] = bi;
        __syncthreads();
    }
}

// Reverse matching through the cells of the gripper clouds: the nearest gripper point of a
// colliding point c among the transformed cloud, by the same float32 distances |c - s'| in the
// object frame as collide_nn_kernel, but only of the points that can be nearest.  The
// cells belong to the gripper cloud in its own frame (built once per gripper), where c is
// at x = R^T (c - t).  What that mapping and the rounding of s' can change, u = 2^-24: x is off
// by at most 20 u |x| (a rounded c - t, three products and sums per coordinate, R
// orthonormal up to 8 u), s' by 6 u (|t|_1 + 2 max |s|) and by 8 u |s| for R again; distances
// all scale by |q|^2 alike.  The lists hold for positions off by kGripperTol / 2.5 of the
// cloud's radius; a colliding point beyond that bound (an object metres from its frame's origin)
// compares the whole cloud.  A warp takes 32 colliding points that lie together in the sorted
// collision cloud, so its lanes meet in the same cells (in ascending order they do not, and the
// scattered loads set the pace: 0.80 ms on 9.8e6 points); the bit map gives each point's
// place in the ascending list.
// Measured on GB300 (per pass, against collide_nn_kernel with its sums): 3 x 256 particles, N 2048
// 14.6 us against 71 (2.3e5 colliding points); 3 x 1024, N 4096 0.39 ms against 14.6 (9.8e6);
// 57 % of the issue slots, the rest waits for the scattered loads.
__global__ void __launch_bounds__(128, 10) collide_cells_kernel(const CollideArgs a)
{
    const int lane = threadIdx.x & 31, N = a.L.N;
    const int count = a.col_items[0];
    for (int item = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; item < count; item += (gridDim.x * blockDim.x) >> 5) {
        const int2 it = reinterpret_cast<const int2 *>(a.col_list)[item];
        const int pk = it.x, slot = it.y * 32 + lane;
        const int grp = a.L.part_grp[pk], p = grp % a.L.P;
        const ObjMeta &om = a.L.obj[grp / a.L.P];
        const bool valid = slot < a.ncol[pk];
        const long long first = om.colidx_base + (long long)(pk - om.pfirst) * om.Mc;
        const int at = valid ? a.colsrt[first + slot] : 0;
        const float4 c = __ldg(om.Csort + at);
        const float *th = a.theta + (size_t)pk * 8;
        const float tx = th[0], ty = th[1], tz = th[2];
        float Rm[9];
        quat_rot_f32(th[3], th[4], th[5], th[6], Rm);
        const float4 *__restrict__ S = a.S + (size_t)p * N;
        const int *__restrict__ leaves = a.pre_leaves + (size_t)p * a.pre_leaf_cap;
        const float4 fr = __ldg(a.pre_frame + p);
        auto dist = [&](int i, float cx, float cy, float cz) {
            const float4 s = __ldg(S + i);
            const float3 o = xform_f32(Rm, tx, ty, tz, s.x, s.y, s.z);
            return dist2_f32(o.x, o.y, o.z, cx, cy, cz);
        };

        int2 nd = make_int2(0, 0);
        int rank = 0;
        if (valid) {
            const int own = __float_as_int(c.w) + (at & ~(kColSegment - 1));
            const int2 word = __ldg(a.colmap + om.colmap_base + (long long)(pk - om.pfirst) * ((om.Mc + 31) / 32) + (own >> 5));
            rank = word.y + __popc((unsigned)word.x & ((1u << (own & 31)) - 1u));
            const float dx = __fsub_rn(c.x, tx), dy = __fsub_rn(c.y, ty), dz = __fsub_rn(c.z, tz);
            const float x = fmaf(Rm[0], dx, fmaf(Rm[3], dy, Rm[6] * dz)), y = fmaf(Rm[1], dx, fmaf(Rm[4], dy, Rm[7] * dz)),
                        z = fmaf(Rm[2], dx, fmaf(Rm[5], dy, Rm[8] * dz));
            const float reach = fabsf(fr.x) + fabsf(fr.y) + fabsf(fr.z) + fr.w;      // >= max |s|
            const float off = 1.2e-6f * (fabsf(x) + fabsf(y) + fabsf(z) + reach) + 4e-7f * (fabsf(tx) + fabsf(ty) + fabsf(tz));
            nd = off <= 0.4f * kGripperTol * fr.w
                     ? find_cell(a.pre_nodes + (size_t)p * a.pre_node_cap, cell_half(fr.w, kGripperCells), x - fr.x, y - fr.y,
                                 z - fr.z)
                     : make_int2(0, kCellWhole);
        }
        float best = __int_as_float(0x7f800000);
        int bi = 0x7fffffff;
        if (nd.y <= kCellOwn) {
            const int4 *l = reinterpret_cast<const int4 *>(leaves + nd.x);
            for (int e = 0; e < nd.y; e += 4, ++l) {
                const int4 id = __ldg(l);
                const float d0 = dist(id.x, c.x, c.y, c.z), d1 = dist(id.y, c.x, c.y, c.z), d2 = dist(id.z, c.x, c.y, c.z),
                            d3 = dist(id.w, c.x, c.y, c.z);
                if (d0 < best) { best = d0; bi = id.x; }
                if (d1 < best) { best = d1; bi = id.y; }
                if (d2 < best) { best = d2; bi = id.z; }
                if (d3 < best) { best = d3; bi = id.w; }
            }
        }
        unsigned pending = __ballot_sync(0xffffffffu, nd.y == kCellWhole || nd.y > kCellOwn);
        while (pending) {
            const int src = __ffs(pending) - 1;
            pending &= pending - 1;
            const float qx = __shfl_sync(0xffffffffu, c.x, src), qy = __shfl_sync(0xffffffffu, c.y, src),
                        qz = __shfl_sync(0xffffffffu, c.z, src);
            const int base = __shfl_sync(0xffffffffu, nd.x, src), len = __shfl_sync(0xffffffffu, nd.y, src);
            float wb = __int_as_float(0x7f800000);
            int wi = 0x7fffffff;
            for (int e = lane; e < (len == kCellWhole ? N : len); e += 32) {
                const int i = len == kCellWhole ? e : __ldg(leaves + base + e);
                const float d = dist(i, qx, qy, qz);
                if (d < wb || (d == wb && i < wi)) { wb = d; wi = i; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) argmin_xor(wb, wi, o);
            if (lane == src) { best = wb; bi = wi; }
        }
        if (valid) a.colnn[first + rank] = bi < N ? bi : 0;      // no finite distance at all: 0
    }
}

cudaError_t launch_collide(const CollideArgs &a, cudaStream_t st)
{
    // Many particles with small clouds keep the chip busy with small CTAs; few of them, or large clouds,
    // want more warps per particle (256 against 128 threads, us per pass: T 154, Mc 5003 16 against
    // 23; T 768, 8192 21 against 23; T 3072, 65536 286 against 300; but T 3072, 2048 47
    // against 39, T 7040, 1k to 32k 91 against 78).
    if (a.L.T <= 1024 || a.most_points >= 32768)
        collide_kernel<256><<<a.L.T, 256, 0, st>>>(a);
    else
        collide_kernel<128><<<a.L.T, 128, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_collide_nn(const CollideArgs &a, cudaStream_t st)
{
    static int grids[kDeviceSlots] = {};
    static std::mutex mu;
    const int grid = per_device_value(grids, mu, [] {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        return 4 * sms;
    });
    if (a.cells) {          // ten CTAs of four warps per SM, no more than the work list can fill
        const int ctas = (a.most_items + 3) / 4;
        collide_cells_kernel<<<ctas < 5 * grid / 2 ? ctas : 5 * grid / 2, 128, 0, st>>>(a);
        return cudaGetLastError();
    }
    const size_t smem = 2 * sizeof(float4) * (size_t)((a.L.N + 63) / 64 * 64) + 32 * sizeof(float4);
    collide_nn_kernel<<<grid, kColThreads, smem, st>>>(a);
    return cudaGetLastError();
}

constexpr int kClearSeg = 512, kClearHalo = 256, kClearMost = 255;     // (see sdf_clear_rows_kernel)

// Corner-packed copy of a grid: cell (ix, iy, iz), x fastest over the
// (nx-1)(ny-1)(nz-1) cells, gets its eight corner values as two float4.  away: 0 for a cell with a positive corner, 255
// for another one.
__global__ void sdf_pack_cells_kernel(const float *grid, int nx, int ny, int nz, float4 *cells, unsigned char *away)
{
    const long long nc = (long long)(nx - 1) * (ny - 1) * (nz - 1);
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < nc; c += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(c % (nx - 1)), iy = (int)((c / (nx - 1)) % (ny - 1)), iz = (int)(c / ((long long)(nx - 1) * (ny - 1)));
        const float *g = grid + (size_t)ix + (size_t)nx * ((size_t)iy + (size_t)ny * iz);
        const size_t sy = nx, sz = (size_t)nx * ny;
        const float4 u = make_float4(g[0], g[1], g[sy], g[sy + 1]), v = make_float4(g[sz], g[sz + 1], g[sz + sy], g[sz + sy + 1]);
        cells[2 * c] = u;
        cells[2 * c + 1] = v;
        away[c] = fmaxf(fmaxf(fmaxf(u.x, u.y), fmaxf(u.z, u.w)), fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w))) > 0.f ? 0 : kClearMost;
    }
}

size_t sdf_cells_bytes(int nx, int ny, int nz) { return 2 * sizeof(float4) * (size_t)(nx - 1) * (ny - 1) * (nz - 1); }

cudaError_t launch_sdf_pack_cells(const float *grid, int nx, int ny, int nz, float4 *cells, unsigned char *away,
                                  cudaStream_t st)
{
    const long long nc = (long long)(nx - 1) * (ny - 1) * (nz - 1);
    long long blocks = (nc + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) return cudaSuccess;
    sdf_pack_cells_kernel<<<(int)blocks, 256, 0, st>>>(grid, nx, ny, nz, cells, away);
    return cudaGetLastError();
}

// Clearance of every cell of a grid: the distance in cells (largest coordinate, at most 255) to
// the nearest cell with a positive corner, 0 for such a cell.  One axis at a time: along x the distance to the nearest
// positive cell of the row, along y and z min over steps r of max(r, the previous axis's distance r cells away).
//
// Rows: a warp takes up to 1024 cells as 32 words of bits, one per lane; the last set bit before and the first one
// after each word come from scans over the lanes.  Longer rows are taken in pieces of 512 cells that look 256 to either
// side (the distance ends at 255).
__global__ void __launch_bounds__(256) sdf_clear_rows_kernel(const unsigned char *away, long long rows, int cx, int segs,
                                                             unsigned char *out)
{
    const long long id = (long long)blockIdx.x * 8 + (threadIdx.x >> 5), row = id / segs;
    if (row >= rows) return;
    const int lane = threadIdx.x & 31, seg = (int)(id % segs);
    const int o0 = segs == 1 ? 0 : seg * kClearSeg, o1 = segs == 1 ? cx : min(cx, o0 + kClearSeg);
    const int b0 = segs == 1 ? 0 : o0 - kClearHalo, words = min(32, (cx - b0 + 31) / 32);
    const unsigned char *in = away + row * cx;
    unsigned mine = 0u;
#pragma unroll 4
    for (int j = 0; j < words; ++j) {
        const int i = b0 + 32 * j + lane;
        const unsigned w = __ballot_sync(0xffffffffu, i >= 0 && i < cx && in[i] == 0);
        if (lane == j) mine = w;
    }
    constexpr int kNone = 1 << 28;
    int last = mine ? b0 + 32 * lane + 31 - __clz(mine) : -kNone, first = mine ? b0 + 32 * lane + __ffs(mine) - 1 : 2 * kNone;
    for (int o = 1; o < 32; o <<= 1) {
        const int l = __shfl_up_sync(0xffffffffu, last, o), f = __shfl_down_sync(0xffffffffu, first, o);
        if (lane >= o) last = max(last, l);
        if (lane + o < 32) first = min(first, f);
    }
    int before = __shfl_up_sync(0xffffffffu, last, 1), after = __shfl_down_sync(0xffffffffu, first, 1);
    if (lane == 0) before = -kNone;
    if (lane == 31) after = 2 * kNone;
    for (int k = (o0 - b0) / 32; b0 + 32 * k < o1; ++k) {
        const unsigned w = __shfl_sync(0xffffffffu, mine, k);
        const int pb = __shfl_sync(0xffffffffu, before, k), pa = __shfl_sync(0xffffffffu, after, k), i = b0 + 32 * k + lane;
        const unsigned wl = w & (0xffffffffu >> (31 - lane)), wr = w >> lane;
        const int l = wl ? b0 + 32 * k + 31 - __clz(wl) : pb, r = wr ? i + __ffs(wr) - 1 : pa;
        if (i < o1) out[row * cx + i] = (unsigned char)min(kClearMost, min(i - l, r - i));
    }
}

// Lines: a CTA stages 32 neighbouring lines in shared memory (256 cells of them and 255 to either side) and the least
// values of 2, 4, .. 128 consecutive cells from each.  The distance is above v when no cell up to v away has a value of v or
// less, so v grows by 128, 64, .. 1 cells where the least value of the wider reach stays above it: sixteen loads
// a cell however far it lies from the gripper.
// Measured on GB300, the three launches at 64^3 / 128^3 / 256^3 nodes: 22 / 54 / 295 us (a search outwards from each cell
// in global memory, through the packed cells along x, 75 / 701 / 10100; in shared memory, four lines per thread,
// 30 / 118 / 728; a line per lane with a queue of the cells that can still decide 37 / 70 / 432).
constexpr int kLineSeg = 256, kLineThreads = 256, kLineLevels = 8;
constexpr int kLineRows = kLineSeg + 2 * kClearMost;       // staged at most
static_assert((1 << kLineLevels) - 1 == kClearMost && kLineRows * 32 * kLineLevels <= 227 * 1024, "levels");

__global__ void __launch_bounds__(kLineThreads) sdf_clear_lines_kernel(const unsigned char *in, unsigned char *out, int cx,
                                                                       int len, long long stride, long long outer_stride,
                                                                       int tiles, int segs)
{
    extern __shared__ __align__(16) unsigned char sm_lines[];      // [kLineLevels][rows][32]
    const int x0 = 32 * (int)(blockIdx.x % tiles), seg = (int)(blockIdx.x / tiles % segs);
    const long long first = (blockIdx.x / tiles / segs) * outer_stride;
    const int s0 = seg * kLineSeg, s1 = min(len, s0 + kLineSeg), lo = max(0, s0 - kClearMost), rows = min(len, s1 + kClearMost) - lo;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool valid = x0 + lane < cx;
#pragma unroll 8
    for (int i = warp; i < rows; i += kLineThreads / 32)
        sm_lines[i * 32 + lane] = valid ? in[first + (lo + i) * stride + x0 + lane] : (unsigned char)kClearMost;
    __syncthreads();
    unsigned *words = reinterpret_cast<unsigned *>(sm_lines);
    for (int k = 1; k < kLineLevels; ++k) {        // (past the line's end there is nothing)
        const unsigned *from = words + (k - 1) * rows * 8;
        const int half = 8 << (k - 1);
        for (int e = threadIdx.x; e < rows * 8; e += kLineThreads)
            words[k * rows * 8 + e] = e + half < rows * 8 ? __vminu4(from[e], from[e + half]) : from[e];
        __syncthreads();
    }
    for (int i = s0 - lo + warp; i < s1 - lo; i += kLineThreads / 32) {
        int best = sm_lines[i * 32 + lane], v = 0;
        const bool zero = best == 0;
#pragma unroll
        for (int k = kLineLevels - 1; k >= 0; --k) {
            const unsigned char *level = sm_lines + k * rows * 32 + lane;
            const int up = i + v + 1, down = i - v - (1 << k);
            int m = best;
            if (up < rows) m = min(m, (int)level[up * 32]);
            // (a start before the line's is moved to it: the cells past i - v - 1 lie in the reach too)
            if (i - v > 0) m = min(m, (int)level[max(down, 0) * 32]);
            if (m > v + (1 << k)) {
                v += 1 << k;
                best = m;
            }
        }
        if (valid) out[first + (lo + i) * stride + x0 + lane] = (unsigned char)(zero ? 0 : min(kClearMost, v + 1));
    }
}

size_t lines_smem(int len) { return (size_t)32 * kLineLevels * (len < kLineRows ? len : kLineRows); }

// clear and away: one byte per cell; away (see sdf_pack_cells_kernel) is overwritten.
cudaError_t launch_sdf_clear(int nx, int ny, int nz, unsigned char *away, unsigned char *clear, cudaStream_t st)
{
    const int cx = nx - 1, cy = ny - 1, cz = nz - 1;
    const long long rows = (long long)cy * cz;
    const int row_segs = cx <= 1024 ? 1 : (cx + kClearSeg - 1) / kClearSeg;
    sdf_clear_rows_kernel<<<(unsigned)((rows * row_segs + 7) / 8), 256, 0, st>>>(away, rows, cx, row_segs, clear);
    const int tiles = (cx + 31) / 32;
    auto lines = [&](const unsigned char *in, unsigned char *out, int len, long long stride, int outer, long long outer_stride) {
        const int segs = (len + kLineSeg - 1) / kLineSeg;
        sdf_clear_lines_kernel<<<(unsigned)((long long)tiles * segs * outer), kLineThreads, lines_smem(len), st>>>(
            in, out, cx, len, stride, outer_stride, tiles, segs);
    };
    lines(clear, away, cy, cx, cz, (long long)cx * cy);
    lines(away, clear, cz, (long long)cx * cy, cy, cx);
    return cudaGetLastError();
}

cudaError_t init_collision_attributes()
{
    const cudaError_t e = cudaFuncSetAttribute(sort_cloud_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               32 * 32 * 32 * (int)sizeof(int));
    if (e != cudaSuccess) return e;
    const cudaError_t l = cudaFuncSetAttribute(sdf_clear_lines_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)lines_smem(INT_MAX));
    if (l != cudaSuccess) return l;
    return cudaFuncSetAttribute(collide_nn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(2 * sizeof(float4) * kMaxN + 32 * sizeof(float4)));
}

}  // namespace asicp
