// Learned initial-pose proposal (the data-driven initialisation the paper names
// as future work, after its Section VII ablation on mixture-of-Gaussian
// initialisations): PointNet-style encoder of the object cloud -> per-preshape
// mixture of SE(3) densities; forward, mixture loss, backward, Adam and
// sampling kernels.  Weights and stored activations are bfloat16 (round to
// nearest even), every product is accumulated in float32; master weights,
// gradients and the Adam state are float32.  The two per-point bfloat16
// contractions of the encoder (layers 2 and 3, every point of every cloud) run on
// the tensor cores (tcgen05, kind::f16), in one kernel with layer 1 and the
// max-pool; the head layers (one row per object) run on float32 FMAs.
//
// Network (x_i = r_i - centroid; W row-major [out][in]):
//   h1 = relu(W1 x + b1) 3->64, h2 = relu(W2 h1 + b2) 64->128,
//   h3 = relu(W3 h2 + b3) 128->256, g = max over points (ties: lowest point),
//   z = relu(W4 g + b4) 256->256, o = W5 z + b5 256->P*16*10.
// Mixture per preshape p, component c (raw o[0..9]): pi = softmax(o0),
// mu = 0.1 (o1, o2, o3), sigma = 0.1 exp(clip(o4, -4, 1)), nu = (o5..o8)/|.|,
// kappa = 4 exp(clip(o9, -2, 3)); log p(t, q) = LSE_c[log pi_c - |t' - mu_c|^2 /
// (2 sigma_c^2) - 3 log sigma_c + kappa_c (nu_c.q)^2 - log M(1/2, 2, kappa_c)]
// - 1.5 log 2 pi - log 2 pi^2: a Gaussian in translation times a Watson density on
// the quaternion sphere (q and -q score alike; M = Kummer's 1F1, summed as its
// series).  Loss of one object: -(1 / (P T)) sum over preshapes and targets.
//
// Backward: the max-pool passes a gradient to one point per channel, so at most 256
// points of a cloud have any; layers 3 to 1 work on those alone (a term left out is a
// product with zero).  What an object contributes to a parameter is added in object
// order, so a training step is deterministic.
#include "../../include/asicp_proposal.h"
#include "asicp_internal.cuh"
#include "tcgen05.cuh"

#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

namespace asicp {
namespace {

typedef __nv_bfloat16 bf16;
constexpr int kC = ASICP_PROP_COMPONENTS, kRaw = ASICP_PROP_RAW;
constexpr int kH1 = 64, kH2 = 128, kH3 = 256, kHead = 256;
constexpr int kMaxPre = 16, kMaxPoints = 65536, kMaxBatch = 256;

struct Layer {
    int out, in;
    size_t w, b;   // offsets of W and b in the flat parameters
};

void layers_for(int P, Layer L[5])
{
    const int dims[5][2] = {{kH1, 3}, {kH2, kH1}, {kH3, kH2}, {kHead, kH3}, {P * kC * kRaw, kHead}};
    size_t off = 0;
    for (int l = 0; l < 5; ++l) {
        L[l].out = dims[l][0];
        L[l].in = dims[l][1];
        L[l].w = off;
        off += (size_t)L[l].out * L[l].in;
        L[l].b = off;
        off += L[l].out;
    }
}

size_t params_for(int P)
{
    Layer L[5];
    layers_for(P, L);
    return L[4].b + L[4].out;
}

constexpr int kTile = 128;             // points per encoder CTA = MMA rows = tensor-memory lanes
constexpr unsigned kLbo = 128;         // K-adjacent core matrices (no-swizzle K-major layout); 8-row groups K * 16
constexpr unsigned kW2Bytes = kH2 * kH1 * 2u, kW3Bytes = kH3 * kH2 * 2u;

// ---------------------------------------------------------------- weights
// bfloat16 copies of the weights: flat as the parameters (wbf), W4 and W5 transposed
// (wt4 [in][out], wt5 [in][out]: the head reads neighbouring outputs together), and W2 and W3 in
// the MMA's shared-memory layout (wl: W2 then W3, one bulk copy each).
__global__ void refresh_weights_kernel(const float *w, size_t np, size_t w2, size_t w3, size_t w4, size_t w5, int no,
                                       bf16 *wbf, bf16 *wt4, bf16 *wt5, unsigned char *wl)
{
    const size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (j >= np) return;
    const bf16 v = __float2bfloat16_rn(w[j]);
    wbf[j] = v;
    if (j >= w2 && j < w2 + kH2 * kH1) {
        const int e = (int)(j - w2);
        *reinterpret_cast<bf16 *>(wl + kmajor_offset(e / kH1, e % kH1, kLbo, kH1 * 16)) = v;
    } else if (j >= w3 && j < w3 + kH3 * kH2) {
        const int e = (int)(j - w3);
        *reinterpret_cast<bf16 *>(wl + kW2Bytes + kmajor_offset(e / kH2, e % kH2, kLbo, kH2 * 16)) = v;
    } else if (j >= w4 && j < w4 + kHead * kH3) {
        const int e = (int)(j - w4);
        wt4[(e % kH3) * kHead + e / kH3] = v;
    } else if (j >= w5 && j < w5 + (size_t)no * kHead) {
        const int e = (int)(j - w5);
        wt5[(size_t)(e % kHead) * no + e / kHead] = v;
    }
}

// ---------------------------------------------------------------- encoder
// Centroid (float64) of every cloud; thread and warp order fixed.
__global__ void __launch_bounds__(256) centroid_kernel(const float *clouds, int npts, float *cen, double *mean)
{
    __shared__ double red[3][8];
    const int b = blockIdx.x;
    const float *r = clouds + (size_t)b * npts * 3;
    double s[3] = {0.0, 0.0, 0.0};
#pragma unroll 8
    for (int i = threadIdx.x; i < npts; i += 256)
        for (int c = 0; c < 3; ++c) s[c] += (double)r[(size_t)i * 3 + c];
    for (int c = 0; c < 3; ++c) {
        double v = s[c];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = v;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += red[threadIdx.x][w];
        mean[b * 3 + threadIdx.x] = v / npts;
        cen[b * 3 + threadIdx.x] = (float)(v / npts);
    }
}

// Layers 1 to 3 and the max-pool for kTile points of a cloud, one CTA, a point per thread:
//   x = bf16(r - mean); h1 = bf16(relu(W1 x + b1)) on the thread's FMAs, written as its row of the
//   first MMA's A operand; h2 = bf16(relu(h1 W2^T + b2)): four kind::f16 MMAs (K = 16), float32
//   accumulation in tensor memory; h2 becomes the second MMA's A operand, over the first one's
//   operands; h3 = bf16(relu(h2 W3^T + b3)): eight MMAs into the same columns; per channel the
//   largest value, ties to the lowest point, by warp reductions over the lanes (= points), then
//   over the cloud's tiles by an atomic maximum of (value, ~point).
// Weights arrive by two bulk copies in their shared-memory layout while the threads work on layer
// 1.  97 KB of shared memory and 256 tensor-memory columns: two CTAs per SM.  With store = 1 (training)
// h1 and h2 are kept.  Waits are bounded: on expiry the CTA sets *err and contributes nothing.
// Measured on GB300: 32 clouds of 2048 points 28 us, one cloud 9.6 us (separate kernels for centring,
// layer 1, layers 2 and 3, and a max-pool over stored h3: 177 and 136 us, of which the max-pool,
// one CTA per cloud, 91).  A tile is a chain (layer 1, MMA, epilogue, MMA, reduction) that the
// other CTA of the SM overlaps; the reductions take half of it.
constexpr size_t kEncSmem = kTile * kH2 * 2 + kW3Bytes;      // first region: h1 and W2, then h2
static_assert(kTile * kH1 * 2 + kW2Bytes == kTile * kH2 * 2, "h2 takes the place of h1 and W2");

__global__ void __launch_bounds__(kTile) encode_kernel(const float *clouds, int npts, const double *mean, const bf16 *W1,
                                                       const float *b1, const float *b2, const float *b3,
                                                       const unsigned char *wl, int store, bf16 *h1, bf16 *h2,
                                                       unsigned long long *pool, int *err, int expire)
{
    extern __shared__ __align__(1024) unsigned char sm_enc[];
    unsigned char *sA = sm_enc, *sW2 = sm_enc + kTile * kH1 * 2, *sW3 = sm_enc + kTile * kH2 * 2;
    __shared__ float s_w1[kH1 * 3], s_b1[kH1], s_b2[kH2], s_b3[kH3];
    __shared__ unsigned s_key[kTile / 32][kH3];
    __shared__ __align__(8) unsigned long long landed, done;
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, b = blockIdx.y;
    const int i = blockIdx.x * kTile + tid;
    const long long row = (long long)b * npts + i;
    if (tid == 0) {
        mbar_init(&landed, 1);
        mbar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_arrive_tx(&landed, kW2Bytes + kW3Bytes);
        bulk_load(sW2, wl, kW2Bytes, &landed);
        bulk_load(sW3, wl + kW2Bytes, kW3Bytes, &landed);
    }
    if (warp == 0) tc_alloc(&s_tmem, kH3);
    for (int e = tid; e < kH1 * 3; e += kTile) s_w1[e] = __bfloat162float(W1[e]);
    if (tid < kH1) s_b1[tid] = b1[tid];
    s_b2[tid] = b2[tid];
    s_b3[tid] = b3[tid];
    s_b3[tid + kTile] = b3[tid + kTile];
    float x[3] = {0.f, 0.f, 0.f};
    if (i < npts)
        for (int c = 0; c < 3; ++c)
            x[c] = __bfloat162float(__float2bfloat16_rn((float)((double)clouds[(size_t)row * 3 + c] - mean[b * 3 + c])));
    __syncthreads();
#pragma unroll 2
    for (int j = 0; j < kH1 / 8; ++j) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            uint32_t h[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int c = 8 * j + 2 * e + u;
                float v = s_b1[c];
                for (int k = 0; k < 3; ++k) v = fmaf(s_w1[c * 3 + k], x[k], v);
                h[u] = __bfloat16_as_ushort(__float2bfloat16_rn(fmaxf(v, 0.f)));
            }
            w[e] = h[0] | (h[1] << 16);
        }
        const uint4 q = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4 *>(sA + kmajor_offset(tid, 8 * j, kLbo, kH1 * 16)) = q;
        if (store && i < npts) *reinterpret_cast<uint4 *>(h1 + row * kH1 + 8 * j) = q;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem, mine = tmem + ((uint32_t)(warp * 32) << 16);
    // all threads learn whether the weights landed, so that they leave together
    bool ok = mbar_wait_warp(&landed, 0);
    if (expire) ok = mbar_wait(&done, 0, kTestWaitCycles);     // (nothing has been committed to it yet)
    ok = __syncthreads_and(ok);
    const bool first = ok;
    if (tid == 0 && ok) {
        const unsigned a0 = smem_u32(sA), w0 = smem_u32(sW2);
        for (int k = 0; k < kH1 / 16; ++k)
            tc_mma_f16(tmem, tc_smem_desc(a0 + k * 2 * kLbo, kLbo, kH1 * 16), tc_smem_desc(w0 + k * 2 * kLbo, kLbo, kH1 * 16),
                       tc_idesc_f16(true, kH2, kTile), (uint32_t)k);
        tc_commit(&done);
    }
    ok = ok && mbar_wait_warp(&done, 0);
    ok = __syncthreads_and(ok);
    tc_fence_after();
    if (ok) {
#pragma unroll 1
        for (int c0 = 0; c0 < kH2; c0 += 32) {
            float v[32];
            tc_ld32(mine + (uint32_t)c0, v);
            uint32_t w[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const bf16 l = __float2bfloat16_rn(fmaxf(v[2 * e] + s_b2[c0 + 2 * e], 0.f));
                const bf16 h = __float2bfloat16_rn(fmaxf(v[2 * e + 1] + s_b2[c0 + 2 * e + 1], 0.f));
                w[e] = (uint32_t)__bfloat16_as_ushort(l) | ((uint32_t)__bfloat16_as_ushort(h) << 16);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint4 u = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
                *reinterpret_cast<uint4 *>(sA + kmajor_offset(tid, c0 + 8 * q, kLbo, kH2 * 16)) = u;
                if (store && i < npts) *reinterpret_cast<uint4 *>(h2 + row * kH2 + c0 + 8 * q) = u;
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && ok) {
        const unsigned a0 = smem_u32(sA), w0 = smem_u32(sW3);
        for (int k = 0; k < kH2 / 16; ++k)
            tc_mma_f16(tmem, tc_smem_desc(a0 + k * 2 * kLbo, kLbo, kH2 * 16), tc_smem_desc(w0 + k * 2 * kLbo, kLbo, kH2 * 16),
                       tc_idesc_f16(true, kH3, kTile), (uint32_t)k);
        tc_commit(&done);
    }
    const bool second = ok;
    ok = ok && mbar_wait_warp(&done, 1);
    ok = __syncthreads_and(ok);
    tc_fence_after();
    if (ok) {
        // key: value (its bfloat16 bits order as integers, >= 0) over the lower point
#pragma unroll 1
        for (int c0 = 0; c0 < kH3; c0 += 32) {
            float v[32];
            tc_ld32(mine + (uint32_t)c0, v);
            unsigned best = 0u;
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                const unsigned h = __bfloat16_as_ushort(__float2bfloat16_rn(fmaxf(v[e] + s_b3[c0 + e], 0.f)));
                const unsigned m = __reduce_max_sync(0xffffffffu, i < npts ? (h << 8) | (unsigned)(kTile - 1 - tid) : 0u);
                if (lane == e) best = m;
            }
            s_key[warp][c0 + lane] = best;
        }
        __syncthreads();
        for (int c = tid; c < kH3; c += kTile) {
            unsigned m = s_key[0][c];
            for (int w = 1; w < kTile / 32; ++w) m = max(m, s_key[w][c]);
            const unsigned point = blockIdx.x * kTile + (kTile - 1 - (m & 255u));
            atomicMax(pool + (size_t)b * kH3 + c, ((unsigned long long)(m >> 8) << 32) | (0xffffffffu - point));
        }
    } else {
        if (tid == 0) atomicExch(err, kDevTimeout);
        // the MMAs and copies in flight must be done before the memory goes (bounded)
        if (second) mbar_wait_warp(&done, 1);
        else if (first) mbar_wait_warp(&done, 0);
        mbar_wait_warp(&landed, 0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tc_dealloc(tmem, kH3);
    }
}

// Pooled value of a channel and the point it came from.  A channel that no tile contributed to (its waits
// expired) keeps key 0: value 0 at point 0, a valid row.
__device__ __forceinline__ float pool_value(unsigned long long key)
{
    return __uint_as_float((unsigned)(key >> 32) << 16);
}
__device__ __forceinline__ int pool_point(unsigned long long key) { return key ? (int)(0xffffffffu - (unsigned)key) : 0; }

// ---------------------------------------------------------------- head
// out[m][n] = sum_k A[m][k] W[k][n], k ascending, one thread per output of a tile of kHeadRows x
// kHeadCols; W row-major bfloat16, N a multiple of 32.
//   kZ: A = pooled values, out = bf16(relu(. + bias));   kO: A = z (bf16), out = . + bias (float);
//   kDz: A = dO (float), out = z > 0 ? . : 0 (float);    kDg: A = dz (float), out = pooled > 0 ? . : 0.
// Latency bound (a few rows): kHeadK rows of the weights are staged in shared memory at a time,
// all their loads in flight together.  Measured on GB300 (K 256, N 256 and 480): 5.7 us for 1 to 32
// rows (64 x 64 tiles with 16-wide steps: 24 to 30; weights read where they are used: 30).
enum HeadMode { kZ, kO, kDz, kDg };
constexpr int kHeadCols = 64, kHeadRows = 4, kHeadK = 256;
constexpr int kHeadThreads = kHeadCols * kHeadRows;

template <HeadMode MODE>
__global__ void __launch_bounds__(kHeadThreads) head_kernel(const void *A, const bf16 *W, const float *bias,
                                                            const bf16 *z, const unsigned long long *pool, void *out, int M,
                                                            int N, int K)
{
    __shared__ __align__(16) bf16 sW[kHeadK][kHeadCols];
    __shared__ float sA[kHeadRows][kHeadK];
    const int tid = threadIdx.x, c = tid % kHeadCols, r = tid / kHeadCols;
    const int m = blockIdx.y * kHeadRows + r, n0 = blockIdx.x * kHeadCols, n = n0 + c;
    float acc = 0.f;
    for (int k0 = 0; k0 < K; k0 += kHeadK) {
        const int kn = min(kHeadK, K - k0);
        constexpr int kVec = kHeadK * kHeadCols / 8 / kHeadThreads;     // 16-byte pieces per thread
        uint4 w[kVec];
#pragma unroll
        for (int u = 0; u < kVec; ++u) {
            const int e = tid + u * kHeadThreads, k = e / (kHeadCols / 8), col = n0 + 8 * (e % (kHeadCols / 8));
            if (k < kn && col < N) w[u] = __ldg(reinterpret_cast<const uint4 *>(W + (size_t)(k0 + k) * N + col));
        }
#pragma unroll
        for (int u = 0; u < kHeadK / kHeadCols; ++u) {
            const int k = c + u * kHeadCols;
            const size_t at = (size_t)m * K + k0 + k;
            float v = 0.f;
            if (m < M && k < kn) {
                if (MODE == kZ) v = pool_value(static_cast<const unsigned long long *>(A)[at]);
                else if (MODE == kO) v = __bfloat162float(static_cast<const bf16 *>(A)[at]);
                else v = static_cast<const float *>(A)[at];
            }
            sA[r][k] = v;
        }
#pragma unroll
        for (int u = 0; u < kVec; ++u) {
            const int e = tid + u * kHeadThreads;
            *reinterpret_cast<uint4 *>(&sW[e / (kHeadCols / 8)][8 * (e % (kHeadCols / 8))]) = w[u];
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < kn; ++k) acc = fmaf(sA[r][k], __bfloat162float(sW[k][c]), acc);
        __syncthreads();
    }
    if (m >= M || n >= N) return;
    const size_t at = (size_t)m * N + n;
    float v = acc;
    if (MODE == kZ) {
        static_cast<bf16 *>(out)[at] = __float2bfloat16_rn(fmaxf(v + bias[n], 0.f));
    } else {
        if (MODE == kO) v += bias[n];
        if (MODE == kDz && !(__bfloat162float(z[at]) > 0.f)) v = 0.f;
        if (MODE == kDg && !(pool_value(pool[at]) > 0.f)) v = 0.f;
        static_cast<float *>(out)[at] = v;
    }
}

template <HeadMode MODE>
cudaError_t launch_head(const void *A, const bf16 *W, const float *bias, const bf16 *z, const unsigned long long *pool,
                        void *out, int M, int N, int K, cudaStream_t st)
{
    const dim3 grid((N + kHeadCols - 1) / kHeadCols, (M + kHeadRows - 1) / kHeadRows);
    head_kernel<MODE><<<grid, kHeadThreads, 0, st>>>(A, W, bias, z, pool, out, M, N, K);
    return cudaGetLastError();
}

struct Mix {
    float logpi[kC], mu[kC][3], sigma[kC], nu[kC][4], nv[kC], kappa[kC], logm[kC], dlogm[kC];
    int inside[kC], kin[kC];
};

// Kummer's 1F1(a; b; k) by its series (k <= 80 here: under 200 terms): term n + 1 is term n times
// k (a + n) / ((b + n) (n + 1)); the factors of k for the two functions used, (1/2; 2) and (3/2; 3),
// are tables, since a float64 division a term would set the kernel's pace.
constexpr int kTerms = 400;
struct KummerTables {
    double f[2][kTerms];
    constexpr KummerTables() : f()
    {
        for (int n = 0; n < kTerms; ++n) {
            f[0][n] = (0.5 + n) / ((2.0 + n) * (n + 1.0));
            f[1][n] = (1.5 + n) / ((3.0 + n) * (n + 1.0));
        }
    }
};
__device__ const KummerTables kKummer = KummerTables();

__device__ double kummer(int which, double k)
{
    double t = 1.0, s = 1.0;
    for (int n = 0; n < kTerms; ++n) {
        t *= kKummer.f[which][n] * k;
        s += t;
        if (t < 1e-17 * s) break;
    }
    return s;
}

// Mixture parameters of one preshape from its raw outputs; thread c < kC fills
// component c, thread kC + c helps with its series (call with whole warps, then synchronise).
__device__ void mixture_params(const float *o, Mix &m, int c)
{
    if (c >= 32) return;
    // the two series, 1F1(1/2; 2) and 1F1(3/2; 3), side by side
    const float kappa = 4.f * expf(fminf(fmaxf(o[(c % kC) * kRaw + 9], -2.f), 3.f));
    const double series = kummer(c < kC ? 0 : 1, kappa);
    const double m1 = __shfl_down_sync(0xffffffffu, series, kC), m0 = series;
    if (c >= kC) return;
    float amax = -INFINITY;
    for (int e = 0; e < kC; ++e) amax = fmaxf(amax, o[e * kRaw]);
    float se = 0.f;
    for (int e = 0; e < kC; ++e) se += expf(o[e * kRaw] - amax);
    const float *oc = o + c * kRaw;
    m.logpi[c] = oc[0] - (amax + logf(se));
    for (int k = 0; k < 3; ++k) m.mu[c][k] = 0.1f * oc[1 + k];
    m.inside[c] = oc[4] > -4.f && oc[4] < 1.f;
    m.sigma[c] = 0.1f * expf(fminf(fmaxf(oc[4], -4.f), 1.f));
    const float n = fmaxf(sqrtf(oc[5] * oc[5] + oc[6] * oc[6] + oc[7] * oc[7] + oc[8] * oc[8]), 1e-6f);
    m.nv[c] = n;
    for (int k = 0; k < 4; ++k) m.nu[c][k] = oc[5 + k] / n;
    m.kin[c] = oc[9] > -2.f && oc[9] < 3.f;
    m.kappa[c] = kappa;
    m.logm[c] = (float)log(m0);
    m.dlogm[c] = (float)(0.25 * m1 / m0);
}

// Loss of preshape p of object b and its gradient with respect to the raw outputs.
// One CTA per (p, b), thread j = target j; per component the contributions are
// summed by warp shuffles and then over warps in warp order (deterministic).
constexpr int kLossThreads = ASICP_PROP_MAX_TARGETS;

__global__ void __launch_bounds__(kLossThreads) loss_kernel(const float *out, const float *cen, const float *targets,
                                                            int P, int T, float *dO, float *lossp)
{
    __shared__ Mix mx;
    __shared__ float part[kLossThreads / 32][kC][kRaw];
    __shared__ float lpart[kLossThreads / 32];
    const int p = blockIdx.x, b = blockIdx.y, j = threadIdx.x, lane = j & 31, warp = j >> 5;
    const float *o = out + ((size_t)b * P + p) * kC * kRaw;
    mixture_params(o, mx, j);
    __syncthreads();
    const bool live = j < T;
    float t[3] = {0.f, 0.f, 0.f}, q[4] = {1.f, 0.f, 0.f, 0.f};
    if (live) {
        const float *tg = targets + (((size_t)b * P + p) * T + j) * 7;
        for (int k = 0; k < 3; ++k) t[k] = tg[k] - cen[b * 3 + k];
        for (int k = 0; k < 4; ++k) q[k] = tg[3 + k];
    }
    float ell[kC], dot[kC], d2[kC];
    float emax = -INFINITY;
    for (int c = 0; c < kC; ++c) {
        float dd = 0.f;
        for (int k = 0; k < 3; ++k) { const float e = t[k] - mx.mu[c][k]; dd = fmaf(e, e, dd); }
        float dq = 0.f;
        for (int k = 0; k < 4; ++k) dq = fmaf(q[k], mx.nu[c][k], dq);
        d2[c] = dd;
        dot[c] = dq;
        const float s = mx.sigma[c];
        ell[c] = mx.logpi[c] - dd / (2.f * s * s) - 3.f * logf(s) + mx.kappa[c] * dq * dq - mx.logm[c];
        emax = fmaxf(emax, ell[c]);
    }
    float se = 0.f;
    for (int c = 0; c < kC; ++c) se += expf(ell[c] - emax);
    const float lse = emax + logf(se);
    // constant: -1.5 log(2 pi) - log(2 pi^2)
    float nll = live ? -(lse - 2.75681559961402f - 2.98260695225875f) : 0.f;
    const float w = -1.f / (float)(P * T);
    for (int c = 0; c < kC; ++c) {
        const float r = live ? expf(ell[c] - lse) : 0.f;
        const float s = mx.sigma[c];
        float v[kRaw];
        v[0] = live ? w * (r - expf(mx.logpi[c])) : 0.f;
        for (int k = 0; k < 3; ++k) v[1 + k] = w * 0.1f * r * (t[k] - mx.mu[c][k]) / (s * s);
        v[4] = mx.inside[c] ? w * r * (d2[c] / (s * s * s) - 3.f / s) * s : 0.f;
        float dn[4], pr = 0.f;
        for (int k = 0; k < 4; ++k) { dn[k] = r * 2.f * mx.kappa[c] * dot[c] * q[k]; pr = fmaf(dn[k], mx.nu[c][k], pr); }
        for (int k = 0; k < 4; ++k) v[5 + k] = w * (dn[k] - pr * mx.nu[c][k]) / mx.nv[c];
        v[9] = mx.kin[c] ? w * r * (dot[c] * dot[c] - mx.dlogm[c]) * mx.kappa[c] : 0.f;
        for (int k = 0; k < kRaw; ++k) {
            float x = v[k];
            for (int o2 = 16; o2 > 0; o2 >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o2);
            if (lane == 0) part[warp][c][k] = x;
        }
    }
    for (int o2 = 16; o2 > 0; o2 >>= 1) nll += __shfl_xor_sync(0xffffffffu, nll, o2);
    if (lane == 0) lpart[warp] = nll;
    __syncthreads();
    for (int e = j; e < kC * kRaw; e += blockDim.x) {
        const int c = e / kRaw, k = e % kRaw;
        float s = 0.f;
        for (int wv = 0; wv < kLossThreads / 32; ++wv) s += part[wv][c][k];
        dO[((size_t)b * P + p) * kC * kRaw + e] = s;
    }
    if (j == 0) {
        float s = 0.f;
        for (int wv = 0; wv < kLossThreads / 32; ++wv) s += lpart[wv];
        lossp[b * P + p] = s;
    }
}

// ---------------------------------------------------------------- backward
// Layers 3 to 1 on the points of cloud b that a gradient reaches: the distinct pooled points, ascending
// (at most kH3; live[b] of them).  A CTA takes kBackRows of them:
//   dh2[r][j] = h2 > 0 ? sum over the channels pooled from r, ascending, of dg[ch] W3[ch][j] : 0,
//   dh1[r][k] = h1 > 0 ? sum_j dh2[r][j] W2[j][k] : 0
// into compact rows.  dg is already 0 where the pooled value is not positive.  (A cloud whose
// encoder CTAs gave up has point 0 for every channel: the call returns TIMEOUT, and looking at the error word here and
// in the next two kernels instead cost 3 us of a training step.)
// Measured on GB300 (32 clouds of 2048 points): this kernel, back_slices_kernel and grad_kernel 36 + 13
// + 12 us, against 1.4 ms for dense float32 products over all points, their bias sums and the
// slices of every parameter.
constexpr int kBackRows = 32;

__global__ void __launch_bounds__(256) back_rows_kernel(const unsigned long long *pool, const float *dg, const bf16 *W3,
                                                        const bf16 *W2, const bf16 *h2, const bf16 *h1, int npts, int *live,
                                                        int *rows, float *dh2, float *dh1)
{
    __shared__ unsigned s_key[kH3];        // (point, channel), sorted
    __shared__ int s_first[kH3 + 1], s_wsum[8];
    __shared__ float s_d2[kBackRows][kH2];
    __shared__ float s_dg[kH3];
    __shared__ __align__(16) bf16 s_w2[kH2 * kH1];
    const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint4 w2v[kH2 * kH1 / 8 / 256];        // W2, on its way while the points are sorted
#pragma unroll
    for (int q = 0; q < kH2 * kH1 / 8 / 256; ++q) w2v[q] = __ldg(reinterpret_cast<const uint4 *>(W2) + tid + 256 * q);
    s_key[tid] = ((unsigned)pool_point(pool[(size_t)b * kH3 + tid]) << 8) | (unsigned)tid;     // (points < 65536)
    s_dg[tid] = dg[(size_t)b * kH3 + tid];
    for (int k = 2; k <= kH3; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            __syncthreads();
            if (tid < kH3 / 2) {
                const int i = ((tid & ~(j - 1)) << 1) | (tid & (j - 1)), p = i | j;
                const unsigned u = s_key[i], v = s_key[p];
                if ((u > v) == ((i & k) == 0)) { s_key[i] = v; s_key[p] = u; }
            }
        }
    __syncthreads();
    // first channel of every distinct point
    const bool head = tid == 0 || (s_key[tid] >> 8) != (s_key[tid - 1] >> 8);
    const unsigned bal = __ballot_sync(0xffffffffu, head);
    if (lane == 0) s_wsum[warp] = __popc(bal);
    __syncthreads();
    int before = __popc(bal & ((1u << lane) - 1u)), u = 0;
    for (int w = 0; w < 8; ++w) {
        before += w < warp ? s_wsum[w] : 0;
        u += s_wsum[w];
    }
    if (head) s_first[before] = tid;
    if (tid == 0) s_first[u] = kH3;
    __syncthreads();
    if (blockIdx.x == 0) {
        if (tid == 0) live[b] = u;
        if (tid < u) rows[b * kH3 + tid] = (int)(s_key[s_first[tid]] >> 8);
    }
    const int r0 = blockIdx.x * kBackRows, nr = min(kBackRows, u - r0);
    if (nr <= 0) return;
#pragma unroll
    for (int q = 0; q < kH2 * kH1 / 8 / 256; ++q) reinterpret_cast<uint4 *>(s_w2)[tid + 256 * q] = w2v[q];
#pragma unroll 4
    for (int e = tid; e < nr * kH2; e += 256) {
        const int r = e / kH2, j = e % kH2;
        float v = 0.f;
        for (int q = s_first[r0 + r]; q < s_first[r0 + r + 1]; ++q) {
            const int ch = s_key[q] & 255u;
            v = fmaf(s_dg[ch], __bfloat162float(W3[ch * kH2 + j]), v);
        }
        const size_t row = (size_t)b * npts + (s_key[s_first[r0 + r]] >> 8);
        if (!(__bfloat162float(h2[row * kH2 + j]) > 0.f)) v = 0.f;
        s_d2[r][j] = v;
        dh2[((size_t)b * kH3 + r0 + r) * kH2 + j] = v;
    }
    __syncthreads();
    const int k = tid % kH1, rg = tid / kH1;       // four row groups of eight rows
    float acc[kBackRows / 4] = {};
#pragma unroll 8
    for (int j = 0; j < kH2; ++j) {
        const float w = __bfloat162float(s_w2[j * kH1 + k]);
#pragma unroll
        for (int q = 0; q < kBackRows / 4; ++q) acc[q] = fmaf(s_d2[rg + 4 * q][j], w, acc[q]);
    }
#pragma unroll
    for (int q = 0; q < kBackRows / 4; ++q) {
        const int r = rg + 4 * q;
        if (r >= nr) break;
        const size_t row = (size_t)b * npts + (s_key[s_first[r0 + r]] >> 8);
        dh1[((size_t)b * kH3 + r0 + r) * kH1 + k] = __bfloat162float(h1[row * kH1 + k]) > 0.f ? acc[q] : 0.f;
    }
}

// Object b's gradients of layers 2 and 1 from its compact rows, rows ascending: slice
// {dW2 [kH2][kH1], db2 [kH2], dW1 [kH1][3], db1 [kH1]}.  CTA x < 8 makes kH2 / 8 rows of dW2 (and db2), CTA
// 8 layer 1.
constexpr int kSlice = kH2 * kH1 + kH2 + kH1 * 3 + kH1;

__global__ void __launch_bounds__(256) back_slices_kernel(const float *clouds, const double *mean, const int *live,
                                                          const int *rows, const float *dh2, const float *dh1,
                                                          const bf16 *h1, int npts, float *slices)
{
    constexpr int kRowsTile = 128, kCols = kH2 / 8;     // rows staged together; rows of dW2 per CTA
    __shared__ __align__(16) unsigned char sm[kRowsTile * kH1 * 4];
    __shared__ float s_d2[kRowsTile][kCols];
    const int b = blockIdx.y, tid = threadIdx.x, u = live[b];
    float *out = slices + (size_t)b * kSlice;
    const float *d2 = dh2 + (size_t)b * kH3 * kH2, *d1 = dh1 + (size_t)b * kH3 * kH1;
    const int *row = rows + b * kH3;
    const int k = tid % kH1, g = tid / kH1;
    if (blockIdx.x < 8) {
        bf16 *s_h1 = reinterpret_cast<bf16 *>(sm);      // [kRowsTile][kH1]
        const int j0 = blockIdx.x * kCols;              // outputs (j0 + g + 4 q, k)
        float acc[kCols / 4] = {}, sum = 0.f;           // sum: db2, threads < kCols
        for (int r0 = 0; r0 < u; r0 += kRowsTile) {
            const int nr = min(kRowsTile, u - r0);
#pragma unroll 4
            for (int e = tid; e < nr * (kH1 / 8); e += 256)
                reinterpret_cast<uint4 *>(s_h1)[e] =
                    __ldg(reinterpret_cast<const uint4 *>(h1 + ((size_t)b * npts + row[r0 + e / (kH1 / 8)]) * kH1) + e % (kH1 / 8));
#pragma unroll 4
            for (int e = tid; e < nr * kCols; e += 256) s_d2[e / kCols][e % kCols] = d2[(r0 + e / kCols) * kH2 + j0 + e % kCols];
            __syncthreads();
#pragma unroll 4
            for (int r = 0; r < nr; ++r) {
                const float h = __bfloat162float(s_h1[r * kH1 + k]);
#pragma unroll
                for (int q = 0; q < kCols / 4; ++q) acc[q] = fmaf(s_d2[r][g + 4 * q], h, acc[q]);
            }
            if (tid < kCols)
                for (int r = 0; r < nr; ++r) sum += s_d2[r][tid];
            __syncthreads();
        }
#pragma unroll
        for (int q = 0; q < kCols / 4; ++q) out[(j0 + g + 4 * q) * kH1 + k] = acc[q];
        if (tid < kCols) out[kH2 * kH1 + j0 + tid] = sum;
    } else {
        float *s_d1 = reinterpret_cast<float *>(sm), *s_x = &s_d2[0][0];     // [kRowsTile][kH1], [kRowsTile][3]
        float acc = 0.f;                                                     // g = 3: the bias
        for (int r0 = 0; r0 < u; r0 += kRowsTile) {
            const int nr = min(kRowsTile, u - r0);
#pragma unroll 4
            for (int e = tid; e < nr * kH1; e += 256) s_d1[e] = d1[r0 * kH1 + e];
            for (int e = tid; e < nr * 3; e += 256) {
                const float v = (float)((double)clouds[((size_t)b * npts + row[r0 + e / 3]) * 3 + e % 3] - mean[b * 3 + e % 3]);
                s_x[e] = __bfloat162float(__float2bfloat16_rn(v));
            }
            __syncthreads();
            for (int r = 0; r < nr; ++r) {
                const float d = s_d1[r * kH1 + k];
                acc = g < 3 ? fmaf(d, s_x[r * 3 + g], acc) : acc + d;
            }
            __syncthreads();
        }
        out[kH2 * kH1 + kH2 + (g < 3 ? k * 3 + g : kH1 * 3 + k)] = acc;
    }
}

// grad[j] = (1/B) sum_b of object b's contribution, objects in order: layers 5, 4 and 3 are outer
// products (of dO and z, dz and the pooled values, dg and h2 at the pooled points), layers 2
// and 1 come from the slices.
__global__ void __launch_bounds__(256) grad_kernel(const float *dO, const bf16 *z, const float *dz,
                                                   const unsigned long long *pool, const float *dg, const bf16 *h2,
                                                   const float *slices, int npts, int B, int no, size_t w2, size_t w3,
                                                   size_t w4, size_t w5, size_t np, float *grad)
{
    const size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (j >= np) return;
    float s = 0.f;
    if (j >= w5) {
        const size_t e = j - w5;
        const bool bias = e >= (size_t)no * kHead;
        const int o = (int)(bias ? e - (size_t)no * kHead : e / kHead), k = (int)(e % kHead);
#pragma unroll 4
        for (int b = 0; b < B; ++b) {
            const float d = dO[(size_t)b * no + o];
            s = __fadd_rn(s, bias ? d : __fmul_rn(d, __bfloat162float(z[b * kHead + k])));
        }
    } else if (j >= w4) {
        const int e = (int)(j - w4);
        const bool bias = e >= kHead * kH3;
        const int n = bias ? e - kHead * kH3 : e / kH3, k = e % kH3;
#pragma unroll 4
        for (int b = 0; b < B; ++b) {
            const float d = dz[b * kHead + n];
            s = __fadd_rn(s, bias ? d : __fmul_rn(d, pool_value(pool[(size_t)b * kH3 + k])));
        }
    } else if (j >= w3) {
        const int e = (int)(j - w3);
        const bool bias = e >= kH3 * kH2;
        const int ch = bias ? e - kH3 * kH2 : e / kH2, k = e % kH2;
#pragma unroll 4
        for (int b = 0; b < B; ++b) {
            const float d = dg[b * kH3 + ch];
            const size_t row = (size_t)b * npts + pool_point(pool[(size_t)b * kH3 + ch]);
            s = __fadd_rn(s, bias ? d : __fmul_rn(d, __bfloat162float(h2[row * kH2 + k])));
        }
    } else {
        // parameters: W1, b1 (from 0), W2, b2 (from w2); slice: W2, b2, W1, b1
        const int e = j >= w2 ? (int)(j - w2) : (int)j + kH2 * kH1 + kH2;
#pragma unroll 4
        for (int b = 0; b < B; ++b) s = __fadd_rn(s, slices[(size_t)b * kSlice + e]);
    }
    grad[j] = s / (float)B;
}

__global__ void adam_kernel(float *w, float *m, float *v, const float *g, size_t n, float lr, float bc1, float bc2)
{
    const size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (j >= n) return;
    const float gj = g[j];
    const float mj = 0.9f * m[j] + 0.1f * gj;
    const float vj = 0.999f * v[j] + 0.001f * gj * gj;
    m[j] = mj;
    v[j] = vj;
    w[j] -= lr * (mj / bc1) / (sqrtf(vj / bc2) + 1e-8f);
}

// theta [B][P][K][7] from the mixtures and the caller's draws [B][P][K][8]
__global__ void sample_kernel(const float *out, const float *cen, const float *draws, int B, int P, int K,
                              float *theta)
{
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e >= (long long)B * P * K) return;
    const int b = (int)(e / ((long long)P * K)), p = (int)((e / K) % P);
    const float *o = out + ((size_t)b * P + p) * kC * kRaw;
    const float *d = draws + e * 8;
    float amax = -INFINITY;
    for (int c = 0; c < kC; ++c) amax = fmaxf(amax, o[c * kRaw]);
    float cdf[kC], tot = 0.f;
    for (int c = 0; c < kC; ++c) { tot += expf(o[c * kRaw] - amax); cdf[c] = tot; }
    const float u = d[0] * tot;
    int c = kC - 1;
    for (int k = kC - 1; k >= 0; --k)
        if (cdf[k] > u) c = k;
    const float *oc = o + c * kRaw;
    const float sigma = 0.1f * expf(fminf(fmaxf(oc[4], -4.f), 1.f));
    float *th = theta + e * 7;
    for (int k = 0; k < 3; ++k) th[k] = cen[b * 3 + k] + 0.1f * oc[1 + k] + sigma * d[1 + k];
    const float n = fmaxf(sqrtf(oc[5] * oc[5] + oc[6] * oc[6] + oc[7] * oc[7] + oc[8] * oc[8]), 1e-6f);
    const float kap = 4.f * expf(fminf(fmaxf(oc[9], -2.f), 3.f));
    const float spread = rsqrtf(2.f * kap);
    float qv[4], qq = 0.f;
    for (int k = 0; k < 4; ++k) { qv[k] = oc[5 + k] / n + d[4 + k] * spread; qq = fmaf(qv[k], qv[k], qq); }
    const float inv = 1.f / sqrtf(qq);
    for (int k = 0; k < 4; ++k) th[3 + k] = qv[k] * inv;
}

// ---------------------------------------------------------------- handle
struct Buf {
    void *p = nullptr;
    size_t bytes = 0;
    ~Buf() { if (p) cudaFree(p); }
    template <class T> T *as() const { return static_cast<T *>(p); }
};

struct PropErr {
    asicp_status st;
};

void pck(cudaError_t e)
{
    if (e != cudaSuccess) {
        cudaGetLastError();
        throw PropErr{e == cudaErrorMemoryAllocation ? ASICP_ERR_OOM : ASICP_ERR_CUDA};
    }
}

void alloc(Buf &b, size_t bytes)
{
    b.bytes = bytes < 16 ? 16 : bytes;
    pck(cudaMalloc(&b.p, b.bytes));
}

void grow(Buf &b, size_t bytes)
{
    if (bytes <= b.bytes) return;
    if (b.p) cudaFree(b.p);
    b.p = nullptr;
    b.bytes = 0;
    alloc(b, bytes);
}

}  // namespace
}  // namespace asicp

using namespace asicp;

struct asicp_prop {
    int P = 0, npts = 0, maxB = 0, nout = 0;
    size_t np = 0;
    Layer L[5];
    cudaStream_t st = nullptr;
    long long step = 0;
    int lastB = 0;
    int expire_test = 0;               // the encoder's first wait expires (testing)
    unsigned char *pin = nullptr;      // page-locked memory: inputs, then results; or null
    ~asicp_prop() { if (pin) cudaFreeHost(pin); }
    Buf w, m, v, grad, slices, wbf, wt4, wt5, wl, clouds, tg, cen, mean, h1, h2, pool, z, o, dO, lossp, dz, dg, live,
        rows, dh2, dh1, outb, sdraws, stheta, scen, errw;
};

namespace {

template <class F>
asicp_status prop_guard(F &&f)
{
    try {
        f();
        return ASICP_OK;
    } catch (const PropErr &e) {
        return e.st;
    } catch (const std::bad_alloc &) {
        return ASICP_ERR_OOM;
    }
}

// Small inputs and results in ordinary host memory pass through the handle's page-locked memory, with one
// wait per call.  Larger ones are copied straight: through page-locked memory a training step's 0.9 MB
// of gradients and parameters each took 60 us longer.
constexpr size_t kPinPiece = (size_t)64 << 10, kPinBytes = (size_t)256 << 10;

bool pageable(const void *p)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeUnregistered;
}

// One call's copies.  Inputs may be reused when the call returns, results are there.
struct Transfer {
    asicp_prop *pr;
    size_t in = 0, out = 0;
    struct Out { void *dst; size_t at, bytes; };
    std::vector<Out> outs;

    explicit Transfer(asicp_prop *p) : pr(p) {}
    ~Transfer() { if (in || out) cudaStreamSynchronize(pr->st); }      // (left by an error: nothing stays in flight)
    // device copy of an input that may be host memory
    const float *load(const float *src, size_t n, Buf &buf)
    {
        const size_t bytes = n * sizeof(float);
        if (pr->pin && bytes <= kPinPiece && in + bytes <= kPinBytes && pageable(src)) {
            unsigned char *at = pr->pin + in;
            std::memcpy(at, src, bytes);
            in += (bytes + 255) / 256 * 256;
            pck(cudaMemcpyAsync(buf.p, at, bytes, cudaMemcpyHostToDevice, pr->st));
        } else {
            pck(cudaMemcpyAsync(buf.p, src, bytes, cudaMemcpyDefault, pr->st));
        }
        return buf.as<float>();
    }
    void store(void *dst, const void *src, size_t bytes)
    {
        if (!dst || !bytes) return;
        if (pr->pin && bytes <= kPinPiece && out + bytes <= kPinBytes && pageable(dst)) {
            outs.push_back({dst, out, bytes});
            pck(cudaMemcpyAsync(pr->pin + kPinBytes + out, src, bytes, cudaMemcpyDeviceToHost, pr->st));
            out += (bytes + 255) / 256 * 256;
        } else {
            pck(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, pr->st));
        }
    }
    // A bounded device wait that expired (the tensor-core layers) is reported as TIMEOUT, once.
    void finish()
    {
        int e = 0;
        store(&e, pr->errw.p, sizeof(int));
        pck(cudaStreamSynchronize(pr->st));
        for (const Out &x : outs) std::memcpy(x.dst, pr->pin + kPinBytes + x.at, x.bytes);
        in = out = 0;
        if (e != kDevOk) {
            pck(cudaMemset(pr->errw.p, 0, sizeof(int)));
            throw PropErr{ASICP_ERR_TIMEOUT};
        }
    }
};

// The clouds' mixture outputs in pr->o, centroids in pr->cen; store: keep h1 and h2 for a backward pass.
void forward_impl(asicp_prop *pr, const float *clouds_dev, int B, bool store)
{
    cudaStream_t st = pr->st;
    const float *wf = pr->w.as<float>();
    unsigned long long *pool = pr->pool.as<unsigned long long>();
    pck(cudaMemsetAsync(pool, 0, sizeof(unsigned long long) * kH3 * B, st));
    centroid_kernel<<<B, 256, 0, st>>>(clouds_dev, pr->npts, pr->cen.as<float>(), pr->mean.as<double>());
    pck(cudaGetLastError());
    encode_kernel<<<dim3((pr->npts + kTile - 1) / kTile, B), kTile, kEncSmem, st>>>(
        clouds_dev, pr->npts, pr->mean.as<double>(), pr->wbf.as<bf16>() + pr->L[0].w, wf + pr->L[0].b, wf + pr->L[1].b,
        wf + pr->L[2].b, pr->wl.as<unsigned char>(), store, pr->h1.as<bf16>(), pr->h2.as<bf16>(), pool, pr->errw.as<int>(),
        pr->expire_test);
    pck(cudaGetLastError());
    pck(launch_head<kZ>(pool, pr->wt4.as<bf16>(), wf + pr->L[3].b, nullptr, nullptr, pr->z.p, B, kHead, kH3, st));
    pck(launch_head<kO>(pr->z.p, pr->wt5.as<bf16>(), wf + pr->L[4].b, nullptr, nullptr, pr->o.p, B, pr->nout, kHead, st));
}

void backward_impl(asicp_prop *pr, const float *clouds_dev, int B)
{
    cudaStream_t st = pr->st;
    const int n = pr->npts, no = pr->nout;
    const bf16 *W = pr->wbf.as<bf16>(), *z = pr->z.as<bf16>(), *h1 = pr->h1.as<bf16>(), *h2 = pr->h2.as<bf16>();
    const unsigned long long *pool = pr->pool.as<unsigned long long>();
    float *dz = pr->dz.as<float>(), *dg = pr->dg.as<float>(), *dh2 = pr->dh2.as<float>(), *dh1 = pr->dh1.as<float>();
    pck(launch_head<kDz>(pr->dO.p, W + pr->L[4].w, nullptr, z, nullptr, dz, B, kHead, no, st));
    pck(launch_head<kDg>(dz, W + pr->L[3].w, nullptr, nullptr, pool, dg, B, kH3, kHead, st));
    back_rows_kernel<<<dim3(kH3 / kBackRows, B), 256, 0, st>>>(pool, dg, W + pr->L[2].w, W + pr->L[1].w, h2, h1, n,
                                                              pr->live.as<int>(), pr->rows.as<int>(), dh2, dh1);
    pck(cudaGetLastError());
    back_slices_kernel<<<dim3(9, B), 256, 0, st>>>(clouds_dev, pr->mean.as<double>(), pr->live.as<int>(), pr->rows.as<int>(),
                                                   dh2, dh1, h1, n, pr->slices.as<float>());
    pck(cudaGetLastError());
    grad_kernel<<<(unsigned)((pr->np + 255) / 256), 256, 0, st>>>(pr->dO.as<float>(), z, dz, pool, dg, h2,
                                                                  pr->slices.as<float>(), n, B, no, pr->L[1].w, pr->L[2].w,
                                                                  pr->L[3].w, pr->L[4].w, pr->np, pr->grad.as<float>());
    pck(cudaGetLastError());
}

void refresh_bf16(asicp_prop *pr)
{
    refresh_weights_kernel<<<(unsigned)((pr->np + 255) / 256), 256, 0, pr->st>>>(
        pr->w.as<float>(), pr->np, pr->L[1].w, pr->L[2].w, pr->L[3].w, pr->L[4].w, pr->nout, pr->wbf.as<bf16>(),
        pr->wt4.as<bf16>(), pr->wt5.as<bf16>(), pr->wl.as<unsigned char>());
    pck(cudaGetLastError());
}

}  // namespace

extern "C" {

size_t asicp_prop_num_params(int P)
{
    if (P < 1 || P > kMaxPre) return 0;
    return params_for(P);
}

asicp_status asicp_prop_create(int P, int n_points, int max_batch, void *cuda_stream, asicp_prop **out)
{
    if (!out) return ASICP_ERR_INVALID_ARG;
    *out = nullptr;
    if (P < 1 || P > kMaxPre || n_points < 16 || n_points > kMaxPoints || max_batch < 1 || max_batch > kMaxBatch)
        return ASICP_ERR_INVALID_ARG;
    asicp_prop *pr = new (std::nothrow) asicp_prop();
    if (!pr) return ASICP_ERR_OOM;
    pr->P = P;
    pr->npts = n_points;
    pr->maxB = max_batch;
    pr->nout = P * kC * kRaw;
    layers_for(P, pr->L);
    pr->np = params_for(P);
    pr->st = static_cast<cudaStream_t>(cuda_stream);
    const size_t B = max_batch, rows = B * n_points, np = pr->np;
    asicp_status s = prop_guard([&] {
        pck(cudaFuncSetAttribute(encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEncSmem));
        alloc(pr->w, np * 4); alloc(pr->m, np * 4); alloc(pr->v, np * 4); alloc(pr->grad, np * 4);
        alloc(pr->slices, B * kSlice * 4); alloc(pr->wbf, np * 2);
        alloc(pr->wt4, (size_t)kHead * kH3 * 2); alloc(pr->wt5, (size_t)pr->nout * kHead * 2);
        alloc(pr->wl, kW2Bytes + kW3Bytes);
        alloc(pr->clouds, rows * 3 * 4); alloc(pr->tg, B * P * ASICP_PROP_MAX_TARGETS * 7 * 4);
        alloc(pr->cen, B * 3 * 4); alloc(pr->mean, B * 3 * 8);
        alloc(pr->h1, rows * kH1 * 2); alloc(pr->h2, rows * kH2 * 2);
        alloc(pr->pool, B * kH3 * 8); alloc(pr->z, B * kHead * 2);
        alloc(pr->o, B * pr->nout * 4); alloc(pr->dO, B * pr->nout * 4); alloc(pr->lossp, B * P * 4);
        alloc(pr->dz, B * kHead * 4); alloc(pr->dg, B * kH3 * 4);
        alloc(pr->live, B * 4); alloc(pr->rows, B * kH3 * 4);
        alloc(pr->dh2, B * kH3 * kH2 * 4); alloc(pr->dh1, B * kH3 * kH1 * 4);
        alloc(pr->outb, B * pr->nout * 4);
        alloc(pr->errw, sizeof(int));
        void *pin = nullptr;
        if (cudaHostAlloc(&pin, 2 * kPinBytes, cudaHostAllocDefault) == cudaSuccess) pr->pin = static_cast<unsigned char *>(pin);
        else cudaGetLastError();
        pck(cudaMemsetAsync(pr->errw.p, 0, sizeof(int), pr->st));
        pck(cudaMemsetAsync(pr->w.p, 0, np * 4, pr->st));
        pck(cudaMemsetAsync(pr->m.p, 0, np * 4, pr->st));
        pck(cudaMemsetAsync(pr->v.p, 0, np * 4, pr->st));
        pck(cudaMemsetAsync(pr->grad.p, 0, np * 4, pr->st));
        refresh_bf16(pr);
        pck(cudaStreamSynchronize(pr->st));
    });
    if (s != ASICP_OK) {
        delete pr;
        return s;
    }
    *out = pr;
    return ASICP_OK;
}

asicp_status asicp_prop_destroy(asicp_prop *pr)
{
    if (!pr) return ASICP_ERR_INVALID_ARG;
    cudaStreamSynchronize(pr->st);
    delete pr;
    return ASICP_OK;
}

asicp_status asicp_prop_set_params(asicp_prop *pr, const float *params)
{
    if (!pr || !params) return ASICP_ERR_INVALID_ARG;
    return prop_guard([&] {
        pck(cudaMemcpyAsync(pr->w.p, params, pr->np * 4, cudaMemcpyDefault, pr->st));
        pck(cudaMemsetAsync(pr->m.p, 0, pr->np * 4, pr->st));
        pck(cudaMemsetAsync(pr->v.p, 0, pr->np * 4, pr->st));
        pr->step = 0;
        refresh_bf16(pr);
        pck(cudaStreamSynchronize(pr->st));
    });
}

asicp_status asicp_prop_get_params(asicp_prop *pr, float *params)
{
    if (!pr || !params) return ASICP_ERR_INVALID_ARG;
    return prop_guard([&] {
        Transfer t(pr);
        t.store(params, pr->w.p, pr->np * 4);
        t.finish();
    });
}

asicp_status asicp_prop_forward(asicp_prop *pr, const float *clouds, int B, float *out, float *centroids)
{
    if (!pr || !clouds || !out || B < 1 || B > pr->maxB) return ASICP_ERR_INVALID_ARG;
    return prop_guard([&] {
        Transfer t(pr);
        const float *c = t.load(clouds, (size_t)B * pr->npts * 3, pr->clouds);
        forward_impl(pr, c, B, false);
        t.store(out, pr->o.p, (size_t)B * pr->nout * 4);
        t.store(centroids, pr->cen.p, (size_t)B * 3 * 4);
        t.finish();
    });
}

asicp_status asicp_prop_loss_grad(asicp_prop *pr, const float *clouds, const float *targets, int B, int T,
                                  float *loss, float *grad)
{
    if (!pr || !clouds || !targets || !loss || B < 1 || B > pr->maxB || T < 1 || T > ASICP_PROP_MAX_TARGETS)
        return ASICP_ERR_INVALID_ARG;
    return prop_guard([&] {
        Transfer io(pr);
        const float *c = io.load(clouds, (size_t)B * pr->npts * 3, pr->clouds);
        const float *t = io.load(targets, (size_t)B * pr->P * T * 7, pr->tg);
        forward_impl(pr, c, B, true);
        loss_kernel<<<dim3(pr->P, B), kLossThreads, 0, pr->st>>>(pr->o.as<float>(), pr->cen.as<float>(), t, pr->P, T,
                                                                 pr->dO.as<float>(), pr->lossp.as<float>());
        pck(cudaGetLastError());
        backward_impl(pr, c, B);
        std::vector<float> lp((size_t)B * pr->P);
        io.store(lp.data(), pr->lossp.p, lp.size() * 4);
        io.store(grad, pr->grad.p, pr->np * 4);
        io.finish();
        double s = 0.0;     // mean over objects of (1 / (P T)) sum over preshapes and targets
        for (float x : lp) s += x;
        *loss = (float)(s / ((double)pr->P * T * B));
        pr->lastB = B;
    });
}

asicp_status asicp_prop_adam_step(asicp_prop *pr, float lr)
{
    if (!pr || !(lr > 0.f) || pr->lastB == 0) return ASICP_ERR_INVALID_ARG;
    return prop_guard([&] {
        ++pr->step;
        const float bc1 = 1.f - powf(0.9f, (float)pr->step), bc2 = 1.f - powf(0.999f, (float)pr->step);
        adam_kernel<<<(unsigned)((pr->np + 255) / 256), 256, 0, pr->st>>>(pr->w.as<float>(), pr->m.as<float>(),
                                                                          pr->v.as<float>(), pr->grad.as<float>(),
                                                                          pr->np, lr, bc1, bc2);
        pck(cudaGetLastError());
        refresh_bf16(pr);
        pck(cudaStreamSynchronize(pr->st));
    });
}

asicp_status asicp_prop_sample(asicp_prop *pr, const float *out, const float *centroids, int B, int K,
                               const float *draws, float *theta)
{
    if (!pr || !out || !centroids || !draws || !theta || B < 1 || B > pr->maxB || K < 1 || K > 4096)
        return ASICP_ERR_INVALID_ARG;
    return prop_guard([&] {
        const size_t n = (size_t)B * pr->P * K;
        // room for the draws and the poses, kept (K is at most 4096)
        grow(pr->sdraws, n * 8 * 4);
        grow(pr->stheta, n * 7 * 4);
        grow(pr->scen, (size_t)B * 3 * 4);
        Transfer t(pr);
        t.load(out, (size_t)B * pr->nout, pr->outb);
        t.load(draws, n * 8, pr->sdraws);
        t.load(centroids, (size_t)B * 3, pr->scen);
        sample_kernel<<<(unsigned)((n + 255) / 256), 256, 0, pr->st>>>(pr->outb.as<float>(), pr->scen.as<float>(),
                                                                      pr->sdraws.as<float>(), B, pr->P, K,
                                                                      pr->stheta.as<float>());
        pck(cudaGetLastError());
        t.store(theta, pr->stheta.p, n * 7 * 4);
        t.finish();
    });
}

asicp_status asicp_test_expire_proposal_waits(asicp_prop *pr, int on)
{
    if (!pr) return ASICP_ERR_INVALID_ARG;
    pr->expire_test = on != 0;
    return ASICP_OK;
}

}  // extern "C"
