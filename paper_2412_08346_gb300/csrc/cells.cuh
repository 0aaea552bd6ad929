// Looking a point up in the cells of a cloud (built by k_cells.cu): shared by the forward
// matching (cells of the object) and the reverse matching (cells of the gripper cloud).
#pragma once
#include "asicp_internal.cuh"

namespace asicp {

constexpr int kCellTable = 32;             // near table: kCellTable^3 cells
constexpr int kCellShells = 6;
constexpr int kCellFarBase = kCellTable * kCellTable * kCellTable;
constexpr int kCellSubBits = 10;           // cell coordinates below a table or shell cell
constexpr int kCellOwn = 128;              // a thread scans lists up to this length itself, longer ones are the warp's
enum { kCellInner = -1, kCellWhole = -2 }; // node.y: children at node.x .. + 7 / the whole cloud; else list length

// J: half width of the near cells of a cloud of radius B (normal), 2^log_factor times the power of
// two above B.
__device__ __forceinline__ float cell_half(float B, int log_factor)
{
    return __uint_as_float(((__float_as_uint(fmaxf(B, 1e-30f)) >> 23) + 1u + log_factor) << 23);
}

// 1 / x of a power of two (as J, and 1 / J not below the normal range).
__device__ __forceinline__ float power_inv(float x) { return __uint_as_float((254u << 23) - __float_as_uint(x)); }

// The list of point a (relative to the frame centre): (first entry, length), or y = kCellWhole.
__device__ __forceinline__ int2 find_cell(const int2 *__restrict__ nodes, float J, float ax, float ay, float az)
{
    const float inv = power_inv(J), v = fmaxf(fabsf(ax), fmaxf(fabsf(ay), fabsf(az))) * inv;
    // (a NaN or infinite coordinate has no cell)
    if (!(fabsf(ax) + fabsf(ay) + fabsf(az) < __int_as_float(0x7f800000) && v < (float)(1 << kCellShells)))
        return make_int2(0, kCellWhole);
    int x, y, z, at;
    if (v < 1.f) {
        const float k = (float)(kCellTable << kCellSubBits) * 0.5f * inv;
        const int top = (kCellTable << kCellSubBits) - 1;
        x = min(max((int)((ax + J) * k), 0), top);
        y = min(max((int)((ay + J) * k), 0), top);
        z = min(max((int)((az + J) * k), 0), top);
        at = ((z >> kCellSubBits) * kCellTable + (y >> kCellSubBits)) * kCellTable + (x >> kCellSubBits);
    } else {
        const int shell = (int)(__float_as_uint(v) >> 23) - 127;
        const float k = 1.f / ldexpf(J, shell + 1), f = (float)(2 << kCellSubBits);
        const int top = (4 << kCellSubBits) - 1;
        x = min(max((int)((ax * k + 1.f) * f), 0), top);
        y = min(max((int)((ay * k + 1.f) * f), 0), top);
        z = min(max((int)((az * k + 1.f) * f), 0), top);
        at = kCellFarBase + 64 * shell + ((z >> kCellSubBits) * 4 + (y >> kCellSubBits)) * 4 + (x >> kCellSubBits);
    }
    int2 nd = __ldg(nodes + at);
    for (int bit = kCellSubBits - 1; nd.y == kCellInner && bit >= 0; --bit)
        nd = __ldg(nodes + nd.x + (((x >> bit) & 1) | (((y >> bit) & 1) << 1) | (((z >> bit) & 1) << 2)));
    return nd;
}

}  // namespace asicp
