// Per-particle cost and gradient, Stein direction and the particle update
// (Eqs. 3, 7-11, 13-18), plus the small set-up kernels (packing, centroids,
// Fibonacci initial poses, ranking).
#include "asicp_internal.cuh"

namespace asicp {

namespace {

__device__ __forceinline__ float pair_d2(float4 a, float4 b)
{
    return dist2_f32(a.x, a.y, a.z, b.x, b.y, b.z);
}

}  // namespace

// Two particles per CTA, kFinalizeThreads threads each.
//  1. The sums its cost and gradient are linear in, over pairs of a point x and a gripper point s (both
//     float32, so every product is exact in double-float): sum s, sum s s^T, sum x,
//     sum x s^T and sum |x|^2.  Of a particle without colliding points the forward pairs
//     (x the matched object point): 128 threads take every 128th pair, kPairB at a time so that
//     their loads overlap; sum s and sum s s^T are the preshape's.  Of another one the colliding
//     points and their gripper points: per kColChunk of them, in ascending order, eight lanes add
//     eight points each, merged in a fixed tree; the chunks are added in order.  A warp takes
//     four chunks and half of the sums, its records straight from memory, eight loads at a time.
//     The result depends on nothing but the pairs.
//  2. Half a warp each: cost and gradient (Eqs. 13-17, or Eq. 18 with Eqs. 4-5) in float64, quaternion
//     block projected onto the tangent space at q.  With E = sum_i e_i s_i^T, e_i = R s_i + t - x_i,
//     the quaternion gradient is g_k = sum_ab (dR_ab/dq_k) E_ab for the homogeneous form
//     R = (w^2 - |v|^2) I + 2 v v^T + 2 w [v]_x:
//       dR/dw   = 2 w I + 2 [v]_x
//       dR/dv_k = -2 v_k I + 2 (e_k v^T + v e_k^T) + 2 w [e_k]_x,
//     which equals sum_i J(s_i)^T e_i of Eqs. 5 and 17; R is |q|^2 times a rotation, so
//     R^T R = |q|^4 I and sum_i |R s_i|^2 = |q|^4 tr(sum s s^T).  Entries of a vector or matrix are
//     the lanes'; the float64 pipe takes 16 cycles per instruction whatever the number of lanes,
//     so the two particles share a warp.
//  3. Convergence bookkeeping (SGD phase) and, in mode 2, the SGD-ICP update of Eq. 3 (A = I);
//     modes 0 (evaluate only) and 1 (SVGD, done by stein_kernel) leave the poses alone.
//  CTA 0 also clears the collision work-list counters for the next pass.
// Measured on GB300, per pass: 3 x 256 particles, N 2048 26 us (28 us for part 2 alone with a thread
// per particle, the sums in the collision kernel and the reverse matching besides); 3 x 1024,
// 9.8e6 colliding points 0.27 ms (with 192 threads summing from shared memory 0.50). With few
// particles the float64 chain of part 2 bounds it, with many the sums' instructions (55 % of the
// issue slots).
constexpr int kFinalizeThreads = 128;      // four warps: eight chunks of colliding points a round
constexpr int kSumThreads = 128;           // threads that add forward pairs
constexpr int kPairB = 4;                  // forward pairs per thread whose loads overlap
constexpr int kRecB = 4;                   // colliding points per lane whose loads overlap
static_assert(kSumThreads == kFinalizeThreads && kColChunk == 64, "finalize_kernel");

namespace {
__constant__ unsigned char kSym[9] = {0, 1, 2, 1, 3, 4, 2, 4, 5};   // 3 x 3 entry -> upper-triangle entry

// sum r (3), sum r s^T (9), sum |r|^2 (1) of a particle's forward pairs, for kSumThreads threads; the
// warps' sums go to sred.
__device__ __forceinline__ void pair_sums(const float4 *__restrict__ S, const int *__restrict__ idx,
                                          const float4 *__restrict__ R, int N, int tid, double (*sred)[kFwdSums])
{
    dfloat acc[kFwdSums];
#pragma unroll
    for (int c = 0; c < kFwdSums; ++c) acc[c] = dfloat{0.f, 0.f};
    auto add_pair = [&](float4 r, float4 s) {
        const float rv[3] = {r.x, r.y, r.z}, sv[3] = {s.x, s.y, s.z};
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            df_add(acc[u], rv[u]);
#pragma unroll
            for (int v = 0; v < 3; ++v) df_add_prod(acc[3 + 3 * u + v], rv[u], sv[v]);
            df_add_prod(acc[12], rv[u], rv[u]);
        }
    };
    int i = tid;
    for (; i + (kPairB - 1) * kSumThreads < N; i += kPairB * kSumThreads) {
        int id[kPairB];
        float4 s[kPairB], r[kPairB];
#pragma unroll
        for (int u = 0; u < kPairB; ++u) { id[u] = idx[i + u * kSumThreads]; s[u] = S[i + u * kSumThreads]; }
#pragma unroll
        for (int u = 0; u < kPairB; ++u) r[u] = __ldg(R + id[u]);
#pragma unroll
        for (int u = 0; u < kPairB; ++u) add_pair(r[u], s[u]);
    }
    for (; i < N; i += kSumThreads) add_pair(__ldg(R + idx[i]), S[i]);
    warp_sum_df(acc);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int c = 0; c < kFwdSums; ++c) sred[tid >> 5][c] = (double)acc[c].hi + (double)acc[c].lo;
}
}  // namespace

namespace {
// Half of the sums of four chunks of a particle's colliding points, for a warp: lane = 8 * chunk +
// part, part adds points part + 8 u, u = 0 .. 7.  HALF 0: sum s (3), sum s s^T (6), sum c (3); 1:
// sum c s^T (9), sum |c|^2 (1), s the gripper point, c the colliding point.  Points past the end add zeros.
// The chunks' sums go to out[0 .. 3].
template <int HALF>
__device__ __forceinline__ void chunk_sums(const float4 *__restrict__ S, const float4 *__restrict__ C,
                                           const int *__restrict__ colidx, const int *__restrict__ colnn, int l0, int nc,
                                           dfloat (*out)[kColSums])
{
    constexpr int kN = HALF == 0 ? 12 : 10;
    const int lane = threadIdx.x & 31, base = l0 + (lane >> 3) * kColChunk + (lane & 7);
    dfloat acc[kN];
#pragma unroll
    for (int k = 0; k < kN; ++k) acc[k] = dfloat{0.f, 0.f};
#pragma unroll 1                           // (both halves unrolled whole overflow the instruction cache)
    for (int u0 = 0; u0 < 8; u0 += kRecB) {
        float4 s[kRecB], c[kRecB];
        int is[kRecB], ic[kRecB];
#pragma unroll
        for (int u = 0; u < kRecB; ++u) {
            const int l = min(base + 8 * (u0 + u), nc - 1);
            ic[u] = __ldg(colidx + l);
            is[u] = __ldg(colnn + l);
        }
#pragma unroll
        for (int u = 0; u < kRecB; ++u) { c[u] = __ldg(C + ic[u]); s[u] = __ldg(S + is[u]); }
#pragma unroll
        for (int u = 0; u < kRecB; ++u) {
            const bool in = base + 8 * (u0 + u) < nc;
            const float sv[3] = {in ? s[u].x : 0.f, in ? s[u].y : 0.f, in ? s[u].z : 0.f};
            const float cv[3] = {in ? c[u].x : 0.f, in ? c[u].y : 0.f, in ? c[u].z : 0.f};
            if (HALF == 0) {
                int k = 3;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    df_add(acc[i], sv[i]);
                    df_add(acc[9 + i], cv[i]);
#pragma unroll
                    for (int j = i; j < 3; ++j) df_add_prod(acc[k++], sv[i], sv[j]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 3; ++i) {
#pragma unroll
                    for (int j = 0; j < 3; ++j) df_add_prod(acc[3 * i + j], cv[i], sv[j]);
                    df_add_prod(acc[9], cv[i], cv[i]);
                }
            }
        }
    }
#pragma unroll 1
    for (int w = 1; w < 8; w <<= 1)
#pragma unroll
        for (int k = 0; k < kN; ++k) {
            dfloat y;
            y.hi = __shfl_xor_sync(0xffffffffu, acc[k].hi, w);
            y.lo = __shfl_xor_sync(0xffffffffu, acc[k].lo, w);
            df_merge(acc[k], y);
        }
    if ((lane & 7) == 0)
#pragma unroll
        for (int k = 0; k < kN; ++k) out[lane >> 3][(HALF == 0 ? 0 : 12) + k] = acc[k];
}
}  // namespace

// Barrier of the kFinalizeThreads threads of one particle.
__device__ __forceinline__ void half_sync(int half)
{
    asm volatile("bar.sync %0, %1;" ::"r"(half + 1), "n"(kFinalizeThreads) : "memory");
}

__global__ void __launch_bounds__(2 * kFinalizeThreads, 4) finalize_kernel(const UpdateArgs a)
{
    // (cleared also when the matching gave up: the collision test beside it may have run)
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.col_items) { a.col_items[0] = 0; a.col_items[1] = 0; }
    if (a.err && *a.err != kDevOk) return;    // an earlier kernel of the pass gave up: its results are not valid
    constexpr int kChunks = 2 * kFinalizeThreads / 32;     // chunks a round
    __shared__ dfloat sPart_[2][2][kChunks][kColSums];
    __shared__ double sred_[2][kSumThreads / 32][kFwdSums];
    // the sums {s (3), s s^T (6), x (3), x s^T (9), |x|^2} and the half warp's vectors and matrices
    __shared__ double sm_[2][kColSums], sR_[2][9], sE_[2][9], sRs_[2][3], sTcp_[2][3], sEc_[2][3], sG_[2][4];
    const int N = a.L.N;
    {
        const int half = threadIdx.x / kFinalizeThreads, tid = threadIdx.x % kFinalizeThreads;
        const int pk = 2 * blockIdx.x + half;
        double *sm = sm_[half];
        if (pk < a.L.T) {
            const int grp = a.L.part_grp[pk], p = grp % a.L.P;
            const ObjMeta &om = a.L.obj[grp / a.L.P];
            const float4 *__restrict__ S = a.S + (size_t)p * N;
            const int nc = a.ncol[pk];
            if (nc == 0) {
                double (*sred)[kFwdSums] = sred_[half];
                pair_sums(S, a.nn_idx + (size_t)pk * N, om.R, N, tid, sred);
                half_sync(half);
                if (tid < kFwdSums) {
                    double v = 0.0;
                    for (int w = 0; w < kSumThreads / 32; ++w) v += sred[w][tid];
                    sm[9 + tid] = v;
                } else if (tid >= 32 && tid < 41) {
                    sm[tid - 32] = a.pconst[(size_t)p * 12 + tid - 32];
                }
            } else {
                const long long first = om.colidx_base + (long long)(pk - om.pfirst) * om.Mc;
                double total = 0.0;
                int buf = 0;
                for (int l0 = 0; l0 < nc; l0 += kChunks * kColChunk, buf ^= 1) {
                    dfloat (*part)[kColSums] = sPart_[half][buf];
                    const int warp = tid >> 5, w0 = (warp >> 1) * 4, l = l0 + w0 * kColChunk;
                    if (l < nc) {
                        if (warp & 1)
                            chunk_sums<1>(S, om.C, a.colidx + first, a.colnn + first, l, nc, part + w0);
                        else
                            chunk_sums<0>(S, om.C, a.colidx + first, a.colnn + first, l, nc, part + w0);
                    }
                    // (one barrier a round: the next round writes the other buffer, the one after waits here)
                    half_sync(half);
                    if (tid < kColSums)
                        for (int k = 0; k < kChunks && l0 + k * kColChunk < nc; ++k)
                            total += (double)part[k][tid].hi + (double)part[k][tid].lo;
                }
                if (tid < kColSums) sm[tid] = total;
            }
        }
    }
    __syncthreads();
    const int half = threadIdx.x >> 4, lane = threadIdx.x & 15, pk = 2 * blockIdx.x + half;
    if (threadIdx.x >= 32 || pk >= a.L.T) return;
    const unsigned hmask = 0xffffu << (16 * half);
    const double *sm = sm_[half];
    double *sR = sR_[half], *sE = sE_[half], *sRs = sRs_[half], *sTcp = sTcp_[half], *sEc = sEc_[half], *sG = sG_[half];
    const int grp = a.L.part_grp[pk], o = grp / a.L.P;
    const double *pc = a.pconst + (size_t)(grp % a.L.P) * 12;
    const int nc = a.ncol[pk];

    const float *th = a.theta + (size_t)pk * 8;
    double t[3], q[4], R[9];
    for (int c = 0; c < 3; ++c) t[c] = th[c];
    for (int c = 0; c < 4; ++c) q[c] = th[3 + c];
    quat_rot_f64(q[0], q[1], q[2], q[3], R);
    if (lane == 0)
        for (int c = 0; c < 9; ++c) sR[c] = R[c];
    const double *ss = sm, *S6 = sm + 3, *xs = sm + 9, *XS = sm + 12;
    const double xx = sm[21], n = nc == 0 ? (double)N : (double)nc;
    const int r3 = lane % 3;               // this lane's entry of a 3-vector (lanes 0 .. 2)
    const int u9 = min(lane, 8), ra = u9 / 3, rb = u9 % 3;     // and of a 3 x 3 matrix (lanes 0 .. 8)
    const double tr3 = th[r3], tra = th[ra];
    __syncwarp(hmask);
    const double rs = sR[r3 * 3 + 0] * ss[0] + sR[r3 * 3 + 1] * ss[1] + sR[r3 * 3 + 2] * ss[2];
    if (lane < 3) sRs[lane] = rs;
    const double q4 = R[0] * R[0] + R[3] * R[3] + R[6] * R[6];
    const double quad = q4 * (S6[0] + S6[3] + S6[5]);
    double cross = 0.0;
    for (int c = 0; c < 9; ++c) cross += R[c] * XS[c];
    __syncwarp(hmask);
    const double tt = t[0] * t[0] + t[1] * t[1] + t[2] * t[2];
    const double tRs = t[0] * sRs[0] + t[1] * sRs[1] + t[2] * sRs[2];
    const double tx = t[0] * xs[0] + t[1] * xs[1] + t[2] * xs[2];
    double se2 = quad + n * tt + xx + 2 * tRs - 2 * tx - 2 * cross;
    double Se = rs + n * tr3 - xs[r3];
    double E = sR[ra * 3 + 0] * S6[kSym[rb]] + sR[ra * 3 + 1] * S6[kSym[3 + rb]] + sR[ra * 3 + 2] * S6[kSym[6 + rb]] +
               tra * ss[rb] - XS[u9];
    if (nc == 0) {
        // TCP-CoM term (Eq. 15) inside the 1/N, weight w_com (Eqs. 16-17)
        const double tcp = pc[r3] / N;
        if (lane < 3) sTcp[lane] = tcp;
        __syncwarp(hmask);
        const double ec = sR[r3 * 3 + 0] * sTcp[0] + sR[r3 * 3 + 1] * sTcp[1] + sR[r3 * 3 + 2] * sTcp[2] + tr3 -
                          a.L.com[3 * o + r3];
        if (lane < 3) sEc[lane] = ec;
        __syncwarp(hmask);
        se2 += a.w_com * (sEc[0] * sEc[0] + sEc[1] * sEc[1] + sEc[2] * sEc[2]);
        Se += a.w_com * ec;
        E += a.w_com * sEc[ra] * sTcp[rb];
    }
    if (lane < 9) sE[lane] = E;
    __syncwarp(hmask);
    const double inv = 1.0 / n;
    // quaternion gradient: lane 0 the scalar part, lanes 1 .. 3 the vector part
    const double tr = sE[0] + sE[4] + sE[8];
    const double kx = sE[7] - sE[5], ky = sE[2] - sE[6], kz = sE[3] - sE[1];   // <[e_k]_x, E>
    double gq;
    if (lane == 0) {
        gq = 2 * q[0] * tr + 2 * (q[1] * kx + q[2] * ky + q[3] * kz);
    } else {
        const int k = min(lane, 3) - 1;
        const double rowv = sE[k * 3 + 0] * q[1] + sE[k * 3 + 1] * q[2] + sE[k * 3 + 2] * q[3];
        const double colv = sE[0 * 3 + k] * q[1] + sE[1 * 3 + k] * q[2] + sE[2 * 3 + k] * q[3];
        const double ks = k == 0 ? kx : k == 1 ? ky : kz;
        gq = -2 * (double)th[4 + k] * tr + 2 * rowv + 2 * colv + 2 * q[0] * ks;
    }
    gq *= inv;
    if (lane < 4) sG[lane] = gq;
    __syncwarp(hmask);
    const double dq = sG[0] * q[0] + sG[1] * q[1] + sG[2] * q[2] + sG[3] * q[3];
    const double qo = th[3 + min(lane, 3)];
    const double gt = Se * inv, gr = gq - dq * qo;          // lanes 0 .. 2: translation; 0 .. 3: rotation
    const double cost = se2 * inv;
    if (lane < 3) a.grad[(size_t)pk * 8 + lane] = gt;
    if (lane < 4) a.grad[(size_t)pk * 8 + 3 + lane] = gr;
    int frozen = a.frozen[pk];
    if (a.mode == 2 && a.conv_tol >= 0.f) {
        const double prev = a.prev_cost[pk];
        if (nc > 0) frozen = 0;
        else if (prev >= 0.0 && fabs(cost - prev) <= (double)a.conv_tol * prev) frozen = 1;
    }
    __syncwarp(hmask);                          // (prev_cost and frozen have been read)
    if (lane == 0) {
        a.cost[pk] = cost;
        a.frozen[pk] = frozen;
        if (a.mode != 0) a.prev_cost[pk] = cost;
    }
    if (a.mode == 2) {
        float *tw = a.theta + (size_t)pk * 8;
        if (lane < 7) a.phi[(size_t)pk * 8 + lane] = 0.f;
        if (lane == 0 && pk < a.L.G) a.h[pk] = 0.f;
        if (!frozen) {
            const double nq = qo - (double)a.eta_sgd * gr;
            __syncwarp(hmask);                  // (sG and theta have been read)
            if (lane < 4) sG[lane] = nq;
            __syncwarp(hmask);
            const double nn = sqrt(sG[0] * sG[0] + sG[1] * sG[1] + sG[2] * sG[2] + sG[3] * sG[3]);
            if (lane < 3) tw[lane] = (float)(tr3 - (double)a.eta_sgd * gt);
            if (lane < 4) tw[3 + lane] = (float)(nq / nn);
        }
    }
}

// SVGD phase, kSteinSplit CTAs of kSteinThreads per preshape.  Every CTA of a
// preshape computes the bandwidth (the same deterministic selection), then the
// Stein direction of its share of ceil(K / kSteinSplit) particles; the poses are
// updated by stein_update_kernel afterwards, because every CTA reads all poses of
// its preshape.  For the bandwidth each particle i is served by T = kSteinThreads
// / K' threads (K' = K rounded up to a power of two); for the direction each
// particle of the share by T' = kSteinThreads / K'' threads (K'' = the share
// rounded up), at most a warp:
//  - bandwidth: exact lower median of |t_i - t_j|^2 (i < j): the value range is
//    narrowed by histograms over linear bins (usually one pass) until the bin
//    holding the median has at most kSelCand values, which are then ranked
//    exactly; every unordered pair is visited once per pass (thread (i, sub)
//    takes partners i + o (mod K), o = 1 + sub + T m <= K/2, the o = K/2 pairs
//    only from i < K/2 when K is even);
//  - Stein direction of Eq. 8 read as the mean of Eq. 6 with the kernels of
//    Eqs. 9-10 per block: thread (i, sub) sums over j = sub, sub + T', ..., the T'
//    partial sums of particle i (adjacent lanes) are added by shuffles, and
//    written to phi;
//  - the update of Eq. 7 (stein_update_kernel).
constexpr int kSteinThreads = 1024;
constexpr int kSteinSplit = 8;         // CTAs per preshape
constexpr int kSelBins = 1024;         // histogram bins per narrowing pass of the median selection
constexpr int kSelCand = 1024;         // values ranked exactly at the end

__global__ void __launch_bounds__(kSteinThreads) stein_kernel(const UpdateArgs a)
{
    if (a.err && *a.err != kDevOk) return;
    extern __shared__ float4 sm[];
    float4 *sT = sm;                  // [K] t (xyz)
    float4 *sQ = sm + kMaxK;          // [K] q (wxyz)
    float4 *sDt = sm + 2 * kMaxK;     // [K] -gamma N g_t
    float4 *sDq = sm + 3 * kMaxK;     // [K] -gamma N g_q
    __shared__ unsigned hist[kSelBins];
    __shared__ float cand[kSelCand];
    __shared__ unsigned s_wsum[kSteinThreads / 32];
    __shared__ unsigned s_lo, s_hi, s_rank, s_n, s_bin, s_before, s_fill;
    __shared__ float s_h;

    const int grp = blockIdx.x / kSteinSplit, part = blockIdx.x % kSteinSplit;
    const int base = a.L.grp_off[grp], K = a.L.grp_off[grp + 1] - base;
    const int share = (K + kSteinSplit - 1) / kSteinSplit, i0 = part * share;
    if (K <= 0 || i0 >= K) return;      // (whole CTAs; no CTA waits on another)
    int Kp = 1;
    while (Kp < K) Kp <<= 1;
    const int T = min(kSteinThreads / Kp, 32);        // threads per particle: a power of two <= a warp
    const int i = threadIdx.x / T, sub = threadIdx.x % T;
    const bool active = i < K;
    const float gN = -a.gamma * (float)a.L.N;
    const double *com = a.L.com + 3 * (grp / a.L.P);
    const float cx = (float)com[0], cy = (float)com[1], cz = (float)com[2];
    const float pt = a.prior_t_sigma > 0.f ? -a.gamma / (a.prior_t_sigma * a.prior_t_sigma) : 0.f;
    const float pq = a.prior_q_kappa > 0.f ? a.gamma * a.prior_q_kappa : 0.f;
    const float *mu = a.prior_q_mean;
    for (int j = threadIdx.x; j < K; j += blockDim.x) {
        const size_t pj = (size_t)base + j;
        const float *th = a.theta + pj * 8;
        const double *g = a.grad + pj * 8;
        sT[j] = make_float4(th[0], th[1], th[2], 0.f);
        sQ[j] = make_float4(th[3], th[4], th[5], th[6]);
        // drive gamma (-N g + grad log p): Gaussian prior on t, von Mises on q (both off at 0)
        const float m = mu[0] * th[3] + mu[1] * th[4] + mu[2] * th[5] + mu[3] * th[6];
        const float sq = m < 0.f ? -pq : pq;
        sDt[j] = make_float4(gN * (float)g[0] + pt * (th[0] - cx), gN * (float)g[1] + pt * (th[1] - cy),
                             gN * (float)g[2] + pt * (th[2] - cz), 0.f);
        sDq[j] = make_float4(gN * (float)g[3] + sq * mu[0], gN * (float)g[4] + sq * mu[1],
                             gN * (float)g[5] + sq * mu[2], gN * (float)g[6] + sq * mu[3]);
    }
    __syncthreads();

    float h;
    if (a.bandwidth_mode == 1) {
        h = a.h_fixed;
    } else if (K < 2) {
        h = 1.f;
    } else {
        const unsigned long long L = (unsigned long long)K * (K - 1) / 2;
        const int half = K / 2;
        const int trips = (half + T - 1) / T;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const float4 ti = sT[active ? i : 0];
        // squared distance of this thread's m-th pair, or -1 when it has none
        auto pair_at = [&](int m) -> float {
            const int o = 1 + sub + T * m;
            int jj = i + o;
            jj -= jj >= K ? K : 0;
            const bool valid = active && o <= half && !((K & 1) == 0 && o == half && i >= half);
            return valid ? pair_d2(ti, sT[jj]) : -1.f;
        };
        // range of all pair values (non-negative floats order like their bit patterns)
        unsigned vmin = 0xffffffffu, vmax = 0u;
        for (int m = 0; m < trips; ++m) {
            const float v = pair_at(m);
            if (v >= 0.f) { vmin = min(vmin, __float_as_uint(v)); vmax = max(vmax, __float_as_uint(v)); }
        }
        vmin = __reduce_min_sync(0xffffffffu, vmin);
        vmax = __reduce_max_sync(0xffffffffu, vmax);
        if (threadIdx.x == 0) { s_lo = 0xffffffffu; s_hi = 0u; s_rank = (unsigned)((L - 1) / 2); }
        __syncthreads();
        if (lane == 0) { atomicMin(&s_lo, vmin); atomicMax(&s_hi, vmax); }
        __syncthreads();
        // narrow [lo, hi] (it holds the answer, with s_rank values of the set below lo)
        // by histograms over kSelBins linear bins until the bin holding the answer has at
        // most kSelCand values, then rank those exactly; binning is monotone in the value,
        // so a bin holds a contiguous run of the sorted values
        float med = 0.f;
        for (int pass = 0;; ++pass) {
            const float lo = __uint_as_float(s_lo), hi = __uint_as_float(s_hi);
            if (!(lo < hi) || pass == 32) { med = lo; break; }   // (32: not reached with finite values)
            const float scale = (float)kSelBins / (hi - lo);
            auto bin_of = [&](float v) { return min(kSelBins - 1, (int)((v - lo) * scale)); };
            for (int b = threadIdx.x; b < kSelBins; b += blockDim.x) hist[b] = 0u;
            __syncthreads();
            for (int m = 0; m < trips; ++m) {
                const float v = pair_at(m);
                if (v >= lo && v <= hi) atomicAdd(&hist[bin_of(v)], 1u);
            }
            __syncthreads();
            // exclusive scan over the bins (one bin per thread), then the bin holding rank s_rank
            const int b = threadIdx.x;
            const unsigned cnt = b < kSelBins ? hist[b] : 0u;
            unsigned inc = cnt;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) s_wsum[warp] = inc;
            __syncthreads();
            unsigned before = inc - cnt;
            for (int w = 0; w < warp; ++w) before += s_wsum[w];
            const unsigned rank = s_rank;
            if (b < kSelBins && cnt > 0 && before <= rank && rank < before + cnt) {
                s_bin = (unsigned)b;
                s_before = before;
                s_n = cnt;
                s_fill = 0u;
                s_lo = 0xffffffffu;
                s_hi = 0u;
            }
            __syncthreads();
            const int bsel = (int)s_bin;
            const unsigned n = s_n;
            if (n <= (unsigned)kSelCand) {
                // gather the bin's values and rank them exactly
                for (int m = 0; m < trips; ++m) {
                    const float v = pair_at(m);
                    if (v >= lo && v <= hi && bin_of(v) == bsel) cand[atomicAdd(&s_fill, 1u)] = v;
                }
                __syncthreads();
                const unsigned r = s_rank - s_before;
                for (unsigned c = threadIdx.x; c < n; c += blockDim.x) {
                    const float v = cand[c];
                    unsigned less = 0u, equal = 0u;
                    for (unsigned e = 0; e < n; ++e) {
                        less += cand[e] < v;
                        equal += cand[e] == v;
                    }
                    if (less <= r && r < less + equal) s_lo = __float_as_uint(v);
                }
                __syncthreads();
                med = __uint_as_float(s_lo);
                break;
            }
            // too many: the bin's own value range becomes the new [lo, hi]
            unsigned bmin = 0xffffffffu, bmax = 0u;
            for (int m = 0; m < trips; ++m) {
                const float v = pair_at(m);
                if (v >= lo && v <= hi && bin_of(v) == bsel) {
                    bmin = min(bmin, __float_as_uint(v));
                    bmax = max(bmax, __float_as_uint(v));
                }
            }
            bmin = __reduce_min_sync(0xffffffffu, bmin);
            bmax = __reduce_max_sync(0xffffffffu, bmax);
            if (lane == 0) { atomicMin(&s_lo, bmin); atomicMax(&s_hi, bmax); }
            if (threadIdx.x == 0) s_rank -= s_before;
            __syncthreads();
        }
        if (threadIdx.x == 0) {     // float64 division and logarithm once, not per thread
            s_h = fmaxf((float)((double)med / log((double)K)), 1e-12f);
        }
        __syncthreads();
        h = s_h;
    }
    if (part == 0 && threadIdx.x == 0) a.h[grp] = h;

    // Stein direction of particles [i0, min(K, i0 + share)) of this preshape
    int Sp = 1;
    while (Sp < share) Sp <<= 1;
    const int T2 = min(kSteinThreads / Sp, 32);
    const int i2 = i0 + threadIdx.x / T2, sub2 = threadIdx.x % T2;
    const bool active2 = threadIdx.x / T2 < share && i2 < K;
    const float4 ti = sT[active2 ? i2 : 0], qi = sQ[active2 ? i2 : 0];
    const float inv_h = 1.f / h, two_h = 2.f / h;
    float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};     // t (3), q (4), sign count
    if (active2) {
        for (int jj = sub2; jj < K; jj += T2) {
            const float4 tj = sT[jj], qj = sQ[jj], dt = sDt[jj], dq = sDq[jj];
            const float ex = ti.x - tj.x, ey = ti.y - tj.y, ez = ti.z - tj.z;
            const float kt = expf(-(ex * ex + ey * ey + ez * ez) * inv_h);
            f[0] += kt * (dt.x + two_h * ex);
            f[1] += kt * (dt.y + two_h * ey);
            f[2] += kt * (dt.z + two_h * ez);
            const float c = qj.x * qi.x + qj.y * qi.y + qj.z * qi.z + qj.w * qi.w;
            f[3] += c * dq.x; f[4] += c * dq.y; f[5] += c * dq.z; f[6] += c * dq.w;
            f[7] += c < 0.f ? -1.f : 1.f;
        }
    }
    // the T2 threads of a particle are adjacent lanes of one warp (T2 is a power of two <= 32)
    for (int o = 1; o < T2; o <<= 1)
#pragma unroll
        for (int u = 0; u < 8; ++u) f[u] += __shfl_xor_sync(0xffffffffu, f[u], o);
    if (active2 && sub2 == 0) {
        const size_t pk = (size_t)base + i2;
        const float invK = 1.f / (float)K;
        float g[7] = {f[0] * invK, f[1] * invK, f[2] * invK,
                      (f[3] + f[7] * qi.x) * invK, (f[4] + f[7] * qi.y) * invK,
                      (f[5] + f[7] * qi.z) * invK, (f[6] + f[7] * qi.w) * invK};
        // tangent projection at q_i (removes the radial kernel-gradient term)
        const float d = g[3] * qi.x + g[4] * qi.y + g[5] * qi.z + g[6] * qi.w;
        g[3] -= d * qi.x; g[4] -= d * qi.y; g[5] -= d * qi.z; g[6] -= d * qi.w;
        for (int u = 0; u < 7; ++u) a.phi[pk * 8 + u] = g[u];
    }
}

// The SVGD update of Eq. 7 from the Stein direction: t += eta phi_t, q <-
// normalise(q + eta phi_q) (phi_q is tangent at q), one thread per particle.
__global__ void stein_update_kernel(const UpdateArgs a)
{
    if (a.err && *a.err != kDevOk) return;
    const int pk = blockIdx.x * blockDim.x + threadIdx.x;
    if (pk >= a.L.T) return;
    float *th = a.theta + (size_t)pk * 8;
    const float *g = a.phi + (size_t)pk * 8;
    const float tx = th[0], ty = th[1], tz = th[2], qw = th[3], qx = th[4], qy = th[5], qz = th[6];
    const double es = a.eta_svgd;
    double nq[4] = {qw + es * g[3], qx + es * g[4], qy + es * g[5], qz + es * g[6]};
    const double nn = sqrt(nq[0] * nq[0] + nq[1] * nq[1] + nq[2] * nq[2] + nq[3] * nq[3]);
    th[0] = (float)(tx + es * g[0]);
    th[1] = (float)(ty + es * g[1]);
    th[2] = (float)(tz + es * g[2]);
    for (int u = 0; u < 4; ++u) th[3 + u] = (float)(nq[u] / nn);
}

cudaError_t init_update_attributes()
{
    return cudaFuncSetAttribute(stein_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(sizeof(float4) * 4 * kMaxK));
}

cudaError_t launch_finalize(const UpdateArgs &a, cudaStream_t st)
{
    finalize_kernel<<<(a.L.T + 1) / 2, 2 * kFinalizeThreads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_stein(const UpdateArgs &a, cudaStream_t st)
{
    const size_t smem = sizeof(float4) * 4 * (size_t)kMaxK;
    stein_kernel<<<a.L.G * kSteinSplit, kSteinThreads, smem, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    stein_update_kernel<<<(a.L.T + 255) / 256, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ set-up kernels
__global__ void pack_points_kernel(const float *xyz, int n, float4 *out, int *err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float x = xyz[3 * (size_t)i], y = xyz[3 * (size_t)i + 1], z = xyz[3 * (size_t)i + 2];
    if (!isfinite(x) || !isfinite(y) || !isfinite(z)) atomicExch(err, kDevNonFinite);
    out[i] = make_float4(x, y, z, 0.f);
}

cudaError_t launch_pack_points(const float *xyz, int n, float4 *out, int *err, cudaStream_t st)
{
    pack_points_kernel<<<(n + 255) / 256, 256, 0, st>>>(xyz, n, out, err);
    return cudaGetLastError();
}

__global__ void check_finite_kernel(const float *v, long long n, int *err)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        if (!isfinite(v[i])) atomicExch(err, kDevNonFinite);
}

cudaError_t launch_check_finite(const float *v, long long n, int *err, cudaStream_t st)
{
    long long blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    check_finite_kernel<<<(int)blocks, 256, 0, st>>>(v, n, err);
    return cudaGetLastError();
}

// Fibonacci sphere of K directions around the CoM (Section V); the same set for
// every preshape.  u_j: z = 1 - (2j+1)/K, azimuth j * pi * (3 - sqrt 5);
// t_j = CoM + radius u_j; q_j the smallest rotation taking +z (the approach
// axis) to -u_j, pi about x when -u_j = -z.  mode 1: the quarter-sphere lattice
// facing +x (upper half) plus min(6, K) poses above the object (see asicp.h).
__global__ void fibonacci_kernel(const Layout L, float radius, int mode, float *theta)
{
    const int pk = blockIdx.x * blockDim.x + threadIdx.x;
    if (pk >= L.T) return;
    const int grp = L.part_grp[pk];
    const int j = pk - L.grp_off[grp], K = L.grp_off[grp + 1] - L.grp_off[grp];
    const double *com = L.com + 3 * (grp / L.P);
    const double ga = 3.14159265358979323846 * (3.0 - sqrt(5.0));
    float *th = theta + (size_t)pk * 8;
    th[7] = 0.f;
    double u[3];
    const int n_above = mode == 1 ? min(6, K) : 0, nq = K - n_above;
    if (j >= nq) {
        // above the object, approach axis -z (pi about x), yawed by (j - nq) * 60 degrees
        double sh, ch;
        sincos((j - nq) * (3.14159265358979323846 / 6.0), &sh, &ch);
        th[0] = (float)com[0];
        th[1] = (float)com[1];
        th[2] = (float)(com[2] + (double)radius);
        th[3] = 0.f; th[4] = (float)ch; th[5] = (float)sh; th[6] = 0.f;
        return;
    }
    if (mode == 1) {   // quarter sphere facing +x, upper half
        const double z = 1.0 - (j + 0.5) / nq;
        const double rho = sqrt(fmax(0.0, 1.0 - z * z));
        double sa, ca;
        sincos(fmod(j * ga, 3.14159265358979323846) - 0.5 * 3.14159265358979323846, &sa, &ca);
        u[0] = rho * ca; u[1] = rho * sa; u[2] = z;
    } else {
        const double z = 1.0 - (2.0 * j + 1.0) / K;
        const double rho = sqrt(fmax(0.0, 1.0 - z * z));
        double sa, ca;
        sincos(j * ga, &sa, &ca);
        u[0] = rho * ca; u[1] = rho * sa; u[2] = z;
    }
    for (int a = 0; a < 3; ++a) th[a] = (float)(com[a] + (double)radius * u[a]);
    const double w = 1.0 - u[2];
    if (w < 1e-12) {
        th[3] = 0.f; th[4] = 1.f; th[5] = 0.f; th[6] = 0.f;
    } else {
        const double qv[4] = {w, u[1], -u[0], 0.0};
        const double n = sqrt(qv[0] * qv[0] + qv[1] * qv[1] + qv[2] * qv[2]);
        for (int a = 0; a < 4; ++a) th[3 + a] = (float)(qv[a] / n);
    }
}

cudaError_t launch_fibonacci(const Layout &L, float radius, int mode, float *theta, cudaStream_t st)
{
    fibonacci_kernel<<<(L.T + 255) / 256, 256, 0, st>>>(L, radius, mode, theta);
    return cudaGetLastError();
}

__global__ void store_meta_kernel(ObjMeta *dst, const ObjMeta v) { *dst = v; }

cudaError_t launch_store_meta(ObjMeta *dst, const ObjMeta &v, cudaStream_t st)
{
    store_meta_kernel<<<1, 1, 0, st>>>(dst, v);
    return cudaGetLastError();
}

// Particle -> group map and group offsets for P groups of K particles (one object).
__global__ void uniform_groups_kernel(int *part_grp, int *grp_off, int P, int K)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < P * K) part_grp[i] = i / K;
    if (i <= P) grp_off[i] = i * K;
}

cudaError_t launch_uniform_groups(int *part_grp, int *grp_off, int P, int K, cudaStream_t st)
{
    const int n = P * K + 1;
    uniform_groups_kernel<<<(n + 255) / 256, 256, 0, st>>>(part_grp, grp_off, P, K);
    return cudaGetLastError();
}

__global__ void set_theta_kernel(const float *theta7, int PK, float *theta8, int *err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= PK) return;
    const float *s = theta7 + (size_t)i * 7;
    float *d = theta8 + (size_t)i * 8;
    bool ok = true;
    for (int a = 0; a < 7; ++a) ok = ok && isfinite(s[a]);
    const double n = sqrt((double)s[3] * s[3] + (double)s[4] * s[4] + (double)s[5] * s[5] + (double)s[6] * s[6]);
    if (!ok || !(n > 0.0)) {
        atomicExch(err, kDevNonFinite);
        return;
    }
    for (int a = 0; a < 3; ++a) d[a] = s[a];
    for (int a = 0; a < 4; ++a) d[3 + a] = (float)((double)s[3 + a] / n);
    d[7] = 0.f;
}

cudaError_t launch_set_theta(const float *theta7, int T, float *theta8, int *err, cudaStream_t st)
{
    set_theta_kernel<<<(T + 255) / 256, 256, 0, st>>>(theta7, T, theta8, err);
    return cudaGetLastError();
}

// Ranking for Algorithm 1's argmin: non-colliding first, ascending cost (NaN
// last), ties to the lower flat index.  Each particle counts the particles that
// precede it, which gives a dense, deterministic order.  The sort key packs the
// collision flag above the cost's order-preserving bit pattern (costs are >= 0).
constexpr int kSelectSmem = 8192;

__device__ __forceinline__ unsigned long long select_key(const double *cost, const int *ncol, int i)
{
    double v = cost[i];
    if (isnan(v) || v < 0.0) v = __longlong_as_double(0x7ff0000000000000LL);
    return ((unsigned long long)(ncol[i] > 0) << 63) | (unsigned long long)__double_as_longlong(v);
}

// One CTA per object: ranks the object's particles; order[pfirst + r] is the
// global index of the particle of rank r.
__global__ void select_kernel(const Layout L, const double *cost, const int *ncol, int *order)
{
    __shared__ unsigned long long keys[kSelectSmem];
    const ObjMeta &om = L.obj[blockIdx.x];
    const int total = om.np;
    const double *c = cost + om.pfirst;
    const int *nc = ncol + om.pfirst;
    const bool staged = total <= kSelectSmem;
    if (staged)
        for (int i = threadIdx.x; i < total; i += blockDim.x) keys[i] = select_key(c, nc, i);
    __syncthreads();
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const unsigned long long ki = staged ? keys[i] : select_key(c, nc, i);
        int rank = 0;
        for (int k = 0; k < total; ++k) {
            const unsigned long long kk = staged ? keys[k] : select_key(c, nc, k);
            rank += kk < ki || (kk == ki && k < i);
        }
        order[om.pfirst + rank] = om.pfirst + i;
    }
}

cudaError_t launch_select(const Layout &L, const double *cost, const int *ncol, int *order, cudaStream_t st)
{
    select_kernel<<<L.nobj, 1024, 0, st>>>(L, cost, ncol, order);
    return cudaGetLastError();
}

}  // namespace asicp
