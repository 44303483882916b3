// The learned band form: quarter-resolution features, the band-proposal
// network's forward and training steps, the per-pixel bands and the
// band-restricted path (Eq. (6)-(10) over each pixel's band only).  The
// paper names a reduced search range as the way to avoid filtering the whole
// cost volume (Sec. V); see include/fbs_band.h for the definitions.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "fbs_band.h"
#include "fbs_band_net.cuh"
#include "fbs_context.cuh"

using namespace fbs_detail;

namespace fbs {
namespace {

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// BF16 tensor -> FP32 copy (fbs_band_net_trace)
__global__ void bf16_to_f32_kernel(const __nv_bfloat16* __restrict__ src, float* __restrict__ dst, size_t n)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        dst[i] = __bfloat162float(src[i]);
}

// ---- features (readings B1-B3) ---------------------------------------------------
// Quarter-resolution intensity of both images: integer sum of the channel
// sums over the 4x4 block, pixels clamped to the image; and, for the coarse
// costs, the sum of a pixel's 3x3 block of them (coordinates clamped to the
// quarter image) and nine times the sum of its squares less the squared sum, as
// a float (0 only for a constant block): 9 x 12240^2 < 2^31, the rest is exact
// in 64 bits.  A CTA sums its tile of 30 x 8 and the border once, one sum per
// thread, in shared memory.
constexpr int kQuarterX = 32;   // with the border
constexpr int kQuarterY = 10;

struct BlockStat {
    int sum;
    float var;
};

// Channel sum of the 4 x 4 pixels from column 4 X, row 4 Y on, clamped.
template <int C>
__device__ __forceinline__ int block_sum(const uint8_t* __restrict__ src, int X, int Y, int H, int W)
{
    int s = 0;
    if ((reinterpret_cast<uintptr_t>(src) & 3) == 0 && (W * C) % 4 == 0 && 4 * X + 3 < W) {
        uint32_t w[4][C];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int c = 0; c < C; ++c)
                w[j][c] = reinterpret_cast<const uint32_t*>(src + ((size_t)min(4 * Y + j, H - 1) * W + 4 * X) * C)[c];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int c = 0; c < C; ++c) s = (int)__dp4a(w[j][c], 0x01010101u, (uint32_t)s);
        return s;
    }
    for (int j = 0; j < 4; ++j)
        for (int i = 0; i < 4; ++i) {
            const uint8_t* p = src + ((size_t)min(4 * Y + j, H - 1) * W + min(4 * X + i, W - 1)) * C;
#pragma unroll
            for (int c = 0; c < C; ++c) s += p[c];
        }
    return s;
}

template <int C>
__global__ void __launch_bounds__(kQuarterX * kQuarterY)
band_quarter_kernel(const uint8_t* __restrict__ L, const uint8_t* __restrict__ R, int H, int W,
                    int32_t* __restrict__ gq, BlockStat* __restrict__ stat)
{
    __shared__ int g[kQuarterY][kQuarterX];
    asm volatile("griddepcontrol.launch_dependents;");
    const int Hq = (H + 3) / 4, Wq = (W + 3) / 4;
    const int tx = threadIdx.x % kQuarterX, ty = threadIdx.x / kQuarterX;
    const int X = blockIdx.x * (kQuarterX - 2) + tx - 1, Y = blockIdx.y * (kQuarterY - 2) + ty - 1;
    g[ty][tx] = block_sum<C>(blockIdx.z == 0 ? L : R, clampi(X, 0, Wq - 1), clampi(Y, 0, Hq - 1), H, W);
    __syncthreads();
    if (tx == 0 || tx == kQuarterX - 1 || ty == 0 || ty == kQuarterY - 1 || X >= Wq || Y >= Hq) return;
    int S = 0, Q = 0;
#pragma unroll
    for (int j = -1; j < 2; ++j)
#pragma unroll
        for (int i = -1; i < 2; ++i) {
            const int v = g[ty + j][tx + i];
            S += v;
            Q += v * v;
        }
    const size_t o = ((size_t)blockIdx.z * Hq + Y) * Wq + X;
    gq[o] = g[ty][tx];
    stat[o] = BlockStat{S, __ll2float_rn(9 * (long long)Q - (long long)S * S)};
}

// Row sums Kh [Hq][Wq][Dq] of the coarse cost volume over the clipped
// 5-column window (X' ascending; reading B3).  A thread takes one e and walks
// kRowX columns of a row (and two on either side, recomputed by the
// neighbours): the block product of a column is three new integer products and
// the two columns before it, the cost a handful of correctly rounded FP32
// operations more (every evaluation of the same (X, Y, e) gives the same bits),
// and the last five costs are in registers.  Lanes are consecutive e: the left
// pixels are broadcast from shared memory, the right ones adjacent there, and
// the sums stored 128 bytes at a time.  Bound by issue (the division and the
// square root are half of it).  The costs with nine products each, by way of a
// volume in memory and a kernel of row sums, took 30 + 22 us at 320 x 160
// quarter pixels, Dq = 64, now 15 (each alone, cold caches); the whole of
// fbs_band_features 120.4 us then, 31.1 now.
constexpr int kAggR = 2;
constexpr int kRowX = 16;
constexpr int kRowChunks = 4;                       // kRowX columns each, per CTA
constexpr int kRowSpan = kRowX * kRowChunks;
constexpr int kRowThreads = 256;

// One column of three rows, and the statistics of its middle pixel.
struct __align__(16) RowColumn {
    int g[3];
    int sum;
};

inline size_t row_sum_smem(int Dq) { return (size_t)(2 * (kRowSpan + 2 * kAggR + 2) + Dq) * (sizeof(RowColumn) + 4); }

__global__ void __launch_bounds__(kRowThreads)
band_row_sum_kernel(const int32_t* __restrict__ gq, const BlockStat* __restrict__ stat, int Hq, int Wq, int Dq,
                    float* __restrict__ Kh)
{
    extern __shared__ __align__(16) uint8_t row_smem[];
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // left columns xl0 .. , right columns xl0 - Dq ..: every column a window of
    // this CTA reads, coordinates clamped to the image
    constexpr int kLeft = kRowSpan + 2 * kAggR + 2;
    const int Y = blockIdx.y, xc = blockIdx.x * kRowSpan, xl0 = xc - kAggR - 1;
    const int nright = kLeft + Dq;
    RowColumn* lc = reinterpret_cast<RowColumn*>(row_smem);
    RowColumn* rc = lc + kLeft;
    float* lv = reinterpret_cast<float*>(rc + nright);
    float* rv = lv + kLeft;
    const size_t P = (size_t)Hq * Wq;
    for (int i = threadIdx.x; i < kLeft + nright; i += kRowThreads) {
        const bool right = i >= kLeft;
        const int x = clampi(right ? xl0 - Dq + i - kLeft : xl0 + i, 0, Wq - 1);
        const size_t o = right ? P : 0;
        RowColumn c;
#pragma unroll
        for (int j = 0; j < 3; ++j) c.g[j] = gq[o + (size_t)clampi(Y - 1 + j, 0, Hq - 1) * Wq + x];
        const BlockStat s = stat[o + (size_t)Y * Wq + x];
        c.sum = right ? s.sum : -s.sum;
        lc[i] = c;
        lv[i] = s.var;
    }
    __syncthreads();
    for (int item = threadIdx.x; item < kRowChunks * Dq; item += kRowThreads) {
        const int e = item % Dq, X0 = xc + item / Dq * kRowX;
        if (X0 >= Wq) break;
        // entry i: column X0 - kAggR - 1 + i, and that column less e
        const RowColumn *l = lc + (X0 - xc), *r = rc + (X0 - xc) + Dq - e;
        const float *vl = lv + (X0 - xc), *vr = rv + (X0 - xc) + Dq - e;
        auto product = [&](const RowColumn& a, const RowColumn& b) {
            return a.g[0] * b.g[0] + a.g[1] * b.g[1] + a.g[2] * b.g[2];
        };
        float* out = Kh + ((size_t)Y * Wq + X0) * Dq + e;
        float k[5] = {0.f, 0.f, 0.f, 0.f, 0.f};   // costs of the last five columns
        RowColumn a1 = l[1], b1 = r[1];
        int p0 = product(l[0], r[0]), p1 = product(a1, b1);
        const int nx = Wq - X0;
#pragma unroll
        for (int i = 0; i < kRowX + 2 * kAggR; ++i) {
            const int dx = i - kAggR;   // column X0 + dx
            const RowColumn a2 = l[i + 2], b2 = r[i + 2];
            const int p2 = product(a2, b2);
            float c = 0.f;              // outside the image: adds nothing
            if (X0 + dx >= 0 && dx < nx) {
                const float va = vl[i + 1], vb = vr[i + 1];
                const long long num = 9ll * (p0 + p1 + p2) + (long long)a1.sum * b1.sum;
                c = va != 0.f && vb != 0.f
                        ? __fsub_rn(1.f, __fdiv_rn(__ll2float_rn(num), __fsqrt_rn(__fmul_rn(va, vb)))) : 1.f;
                if (X0 + dx < e) c = 2.f;
            }
            k[i % 5] = c;
            if (i >= 2 * kAggR && dx - kAggR < nx) {
                out[(size_t)(i - 2 * kAggR) * Dq] =
                    __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(k[(i + 1) % 5], k[(i + 2) % 5]), k[(i + 3) % 5]),
                                        k[(i + 4) % 5]), c);
            }
            p0 = p1;
            p1 = p2;
            a1 = a2;
            b1 = b2;
        }
    }
}

// The minimum over a warp of finite floats.
__device__ __forceinline__ float warp_min(float v)
{
    // order-preserving: negative floats with their other bits inverted
    const int b = __float_as_int(v), k = b ^ ((b >> 31) & 0x7fffffff);
    const int m = __reduce_min_sync(0xffffffffu, k);
    return __int_as_float(m ^ ((m >> 31) & 0x7fffffff));
}

// The 5x5 means Kbar of a quarter pixel's coarse costs (sum of the row sums,
// Y' ascending, divided by the tap count), their winner (smallest e on ties),
// the best non-adjacent cost and the winner's neighbours give the six
// features; x0 receives them as BF16 [P][8] (two zero channels), feat
// (nullable) as FP32 [P][6], estar the winner.  A warp takes eight pixels of a
// column, lanes over e: the twelve row sums that their windows cover are read
// once each, and the eight pixels' features are finished together, one lane
// each.  Bound by issue.  The division by the tap count is a multiplication by
// its reciprocal and one residual step (Markstein's theorem; tested on the CPU for every
// significand and all tap counts to be the correctly rounded quotient).  A
// kernel that stored the means and one thread per pixel that read them twice
// took 23.5 + 35 us at 320 x 160, Dq = 64; now 14.6 (alone, cold caches).
constexpr int kFeatWarps = 4;
constexpr int kFeatRows = 8;

__global__ void __launch_bounds__(32 * kFeatWarps)
band_features_kernel(const int32_t* __restrict__ gq, const float* __restrict__ Kh, int H, int W, int C, int D,
                     __nv_bfloat16* __restrict__ x0, float* __restrict__ feat, int32_t* __restrict__ estar)
{
    extern __shared__ float means[];
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int Hq = (H + 3) / 4, Wq = (W + 3) / 4, Dq = (D + 3) / 4;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int X = blockIdx.x * kFeatWarps + warp, Y0 = blockIdx.y * kFeatRows;
    if (X >= Wq) return;
    float* mean = means + warp * kFeatRows * Dq;
    const int yl = Y0 + lane;   // lane q's pixel, q < kFeatRows
    const float taps_l = (float)((min(Hq - 1, yl + kAggR) - max(0, yl - kAggR) + 1) *
                                 (min(Wq - 1, X + kAggR) - max(0, X - kAggR) + 1));
    const float rtaps_l = __frcp_rn(taps_l);
    const size_t row = (size_t)Wq * Dq;
    const float* k = Kh + (ptrdiff_t)(Y0 - kAggR) * (ptrdiff_t)row + (size_t)X * Dq;
    float v1[kFeatRows];
    int b1[kFeatRows];
#pragma unroll
    for (int q = 0; q < kFeatRows; ++q) {
        v1[q] = __int_as_float(0x7f800000);
        b1[q] = 1 << 30;
    }
    for (int e0 = 0; e0 < Dq; e0 += 32) {
        const int e = e0 + lane;
        const bool ok = e < Dq;
        float t[kFeatRows + 2 * kAggR];   // rows outside the image add nothing
#pragma unroll
        for (int j = 0; j < kFeatRows + 2 * kAggR; ++j)
            t[j] = ok && (unsigned)(Y0 - kAggR + j) < (unsigned)Hq ? k[(ptrdiff_t)j * (ptrdiff_t)row + e] : 0.f;
#pragma unroll
        for (int q = 0; q < kFeatRows; ++q) {
            const float taps = __shfl_sync(0xffffffffu, taps_l, q), rtaps = __shfl_sync(0xffffffffu, rtaps_l, q);
            const float s = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(t[q], t[q + 1]), t[q + 2]), t[q + 3]), t[q + 4]);
            const float d = __fmul_rn(s, rtaps);
            const float v = __fmaf_rn(__fmaf_rn(-d, taps, s), rtaps, d);
            if (ok) {
                mean[q * Dq + e] = v;
                if (v < v1[q]) {
                    v1[q] = v;
                    b1[q] = e;
                }
            }
        }
    }
    __syncwarp();
    float k1 = 0.f, k2 = 0.f;
    int best = 0;
#pragma unroll
    for (int q = 0; q < kFeatRows; ++q) {
        const float m1 = warp_min(v1[q]);
        const int b = __reduce_min_sync(0xffffffffu, v1[q] == m1 ? b1[q] : 1 << 30);
        float m2 = 2.f;
        for (int e = lane; e < Dq; e += 32)
            if ((unsigned)(e - b + 1) > 2u) m2 = fminf(m2, mean[q * Dq + e]);
        m2 = warp_min(m2);
        if (lane == q) {
            k1 = m1;
            k2 = m2;
            best = b;
        }
    }
    if (lane >= kFeatRows || yl >= Hq) return;
    mean += lane * Dq;
    const size_t i = (size_t)yl * Wq + X;
    const float km = best > 0 ? mean[best - 1] : 2.f;
    const float kp = best < Dq - 1 ? mean[best + 1] : 2.f;
    float f[6];
    f[0] = __fsub_rn(__fdiv_rn((float)gq[i], (float)(16 * 255 * C)), 0.5f);
    f[1] = __fdiv_rn((float)best, (float)Dq);
    f[2] = k1;
    const float margin = __fsub_rn(k2, k1);
    f[3] = margin < 1.f ? margin : 1.f;
    f[4] = __fsub_rn(km, k1);
    f[5] = __fsub_rn(kp, k1);
    estar[i] = best;
    __nv_bfloat162 h[4];
    h[0] = __floats2bfloat162_rn(f[0], f[1]);
    h[1] = __floats2bfloat162_rn(f[2], f[3]);
    h[2] = __floats2bfloat162_rn(f[4], f[5]);
    h[3] = __floats2bfloat162_rn(0.f, 0.f);
    reinterpret_cast<uint4*>(x0)[i] = *reinterpret_cast<const uint4*>(h);
    if (feat) {
#pragma unroll
        for (int c = 0; c < 6; ++c) feat[i * 6 + c] = f[c];
    }
}

// ---- feature-point proposal (reading B7) -------------------------------------------
// Reliable feature points (margin f3 >= theta_m) of the 5x5 quarter window
// around a pixel's quarter pixel suggest its band: with at least 3 of them and
// a winner spread <= 2 the centre is 2 (max + min) and the confidence 1.
__global__ void band_feature_points_kernel(const float* __restrict__ feat, const int32_t* __restrict__ estar,
                                           int H, int W, float theta_m, float* __restrict__ centre,
                                           float* __restrict__ conf)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= W) return;
    const int Hq = (H + 3) / 4, Wq = (W + 3) / 4;
    const int Y = y >> 2, X = x >> 2;
    int n = 0, emin = 1 << 30, emax = -1;
    for (int j = max(0, Y - 2); j <= min(Hq - 1, Y + 2); ++j)
        for (int i = max(0, X - 2); i <= min(Wq - 1, X + 2); ++i) {
            const size_t q = (size_t)j * Wq + i;
            if (!(feat[q * 6 + 3] >= theta_m)) continue;
            ++n;
            emin = min(emin, estar[q]);
            emax = max(emax, estar[q]);
        }
    const size_t p = (size_t)y * W + x;
    const bool ok = n >= 3 && emax - emin <= 2;
    centre[p] = ok ? 2.f * (float)(emax + emin) : 0.f;
    conf[p] = ok ? 1.f : 0.f;
}

// ---- band rule (reading B4) and the per-tile ranges -----------------------------
__device__ __forceinline__ uint32_t band_of(float c, float k, int D, int h, float theta)
{
    if (!(k >= theta) || !isfinite(c)) return (uint32_t)(D - 1) << 16;
    float m = floorf(__fadd_rn(c, 0.5f));
    if (m < 0.f) m = 0.f;
    if (m > (float)(D - 1)) m = (float)(D - 1);
    const int mi = (int)m;
    const int lo = max(mi - h, 0), hi = min(mi + h, D - 1);
    return (uint32_t)lo | ((uint32_t)hi << 16);
}

__global__ void band_limits_kernel(const float* __restrict__ centre, const float* __restrict__ conf, int n, int D,
                                   int h, float theta, int32_t* __restrict__ lo, int32_t* __restrict__ hi)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t b = band_of(centre[i], conf[i], D, h, theta);
    lo[i] = (int32_t)(b & 0xffffu);
    hi[i] = (int32_t)(b >> 16);
}

// One CTA per aggregation tile (one thread per tile pixel).
__global__ void __launch_bounds__(kAggTileX * kAggTileY)
band_tiles_kernel(const float* __restrict__ centre, const float* __restrict__ conf, int H, int W, int D, int h,
                  float theta, uint32_t* __restrict__ band, int2* __restrict__ tile_range)
{
    __shared__ int lo_s, hi_s;
    if (threadIdx.x == 0) {
        lo_s = D;
        hi_s = 0;
    }
    __syncthreads();
    const int x = blockIdx.x * kAggTileX + threadIdx.x % kAggTileX;
    const int y = blockIdx.y * kAggTileY + threadIdx.x / kAggTileX;
    if (x < W && y < H) {
        const size_t p = (size_t)y * W + x;
        const uint32_t b = band_of(centre[p], conf[p], D, h, theta);
        band[p] = b;
        atomicMin(&lo_s, (int)(b & 0xffffu));
        atomicMax(&hi_s, (int)(b >> 16));
    }
    __syncthreads();
    if (threadIdx.x == 0) tile_range[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = make_int2(lo_s & ~3, hi_s + 1);
}

}  // namespace

cudaError_t launch_band_tiles(const float* centre, const float* conf, int H, int W, int D, int half_band,
                              float theta, uint32_t* band, int2* tile_range, cudaStream_t stream)
{
    dim3 grid((W + kAggTileX - 1) / kAggTileX, (H + kAggTileY - 1) / kAggTileY);
    fbs::note_launch();
    band_tiles_kernel<<<grid, kAggTileX * kAggTileY, 0, stream>>>(centre, conf, H, W, D, half_band, theta, band,
                                                                 tile_range);
    return cudaGetLastError();
}

}  // namespace fbs

// ---- state of the network in a context -------------------------------------------
using namespace fbs::bnet;

struct fbs_band_state {
    void* pmem = nullptr;            // parameters, optimiser state, packed images
    float* theta = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    float* grad = nullptr;
    float* loss = nullptr;
    __nv_bfloat16* images = nullptr;
    long long step = 0;
    bool ready = false;
    // shape of the last forward or training call, for fbs_band_net_trace
    int last_H = 0, last_W = 0, last_D = 0;
    bool last_training = false;
};

namespace {

size_t al256(size_t n) { return (n + 255) & ~(size_t)255; }

// Scratch of one quarter-resolution problem, carved from ctx->band_ws.
struct NetScratch {
    int32_t* gq;                 // [2][P]
    fbs::BlockStat* stat;        // [2][P]; lies in featf: read before the features are written
    float* kh;                   // row sums of the coarse costs [P][Dq]
    int32_t* estar;              // [P]
    float* featf;                // [P][6] FP32 features (feature-point proposal)
    __nv_bfloat16* x0;           // [P][8]
    __nv_bfloat16* y[5];         // [P][32]
    float* out;                  // [P][2]
    __nv_bfloat16* g[6];         // gradient w.r.t. the output of layer l: [P][32], g[5] = [P][8]
    float* partial;              // weight-gradient partials
    float* loss_partial;
    float* centre;               // [H][W] (learned entry point)
    float* conf;
    uint32_t* band;              // [H][W]
    int2* tile_range;
};

size_t net_scratch_bytes(int H, int W, int D, bool training, bool full_res)
{
    const size_t Hq = (H + 3) / 4, Wq = (W + 3) / 4, P = Hq * Wq, Dq = (D + 3) / 4;
    size_t n = al256(2 * P * 4) + al256(P * Dq * 4) + al256(P * 4) + al256(P * 24) + al256(P * 16) + 5 * al256(P * 64) + al256(P * 8);
    if (training)
        n += 5 * al256(P * 64) + al256(P * 16) + al256(wgrad_partial_floats((int)Hq, (int)Wq) * 4) +
             al256((size_t)loss_blocks((int)P) * 4);
    if (full_res) {
        const size_t px = (size_t)H * W;
        const size_t tiles = (size_t)((W + fbs::kAggTileX - 1) / fbs::kAggTileX) * ((H + fbs::kAggTileY - 1) / fbs::kAggTileY);
        n += 3 * al256(px * 4) + al256(tiles * 8);
    }
    return n;
}

NetScratch carve_net(void* base, int H, int W, int D, bool training, bool full_res)
{
    const size_t Hq = (H + 3) / 4, Wq = (W + 3) / 4, P = Hq * Wq, Dq = (D + 3) / 4;
    uint8_t* q = (uint8_t*)base;
    auto take = [&](size_t bytes) {
        void* r = q;
        q += al256(bytes);
        return r;
    };
    NetScratch s{};
    s.gq = (int32_t*)take(2 * P * 4);
    s.kh = (float*)take(P * Dq * 4);
    s.estar = (int32_t*)take(P * 4);
    s.featf = (float*)take(P * 24);
    s.x0 = (__nv_bfloat16*)take(P * 16);
    for (int l = 0; l < 5; ++l) s.y[l] = (__nv_bfloat16*)take(P * 64);
    s.stat = (fbs::BlockStat*)s.featf;
    static_assert(2 * sizeof(fbs::BlockStat) <= 24, "[2][P] statistics in [P][6] floats");
    s.out = (float*)take(P * 8);
    if (training) {
        for (int l = 0; l < 5; ++l) s.g[l] = (__nv_bfloat16*)take(P * 64);
        s.g[5] = (__nv_bfloat16*)take(P * 16);
        s.partial = (float*)take(wgrad_partial_floats((int)Hq, (int)Wq) * 4);
        s.loss_partial = (float*)take((size_t)loss_blocks((int)P) * 4);
    }
    if (full_res) {
        const size_t px = (size_t)H * W;
        const size_t tiles = (size_t)((W + fbs::kAggTileX - 1) / fbs::kAggTileX) * ((H + fbs::kAggTileY - 1) / fbs::kAggTileY);
        s.centre = (float*)take(px * 4);
        s.conf = (float*)take(px * 4);
        s.band = (uint32_t*)take(px * 4);
        s.tile_range = (int2*)take(tiles * 8);
    }
    return s;
}

fbs_status ensure_state(fbs_ctx* ctx)
{
    if (ctx->band) return FBS_OK;
    fbs_band_state* b = new (std::nothrow) fbs_band_state();
    if (!b) return fail(ctx, FBS_ERR_OOM, "band state");
    const size_t np = al256((size_t)kParams * 4);
    const size_t bytes = 4 * np + 256 + al256((size_t)kImageElems * 2);
    cudaError_t e = cudaMalloc(&b->pmem, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        delete b;
        return fail(ctx, FBS_ERR_OOM, "cudaMalloc(%zu) for the band network: %s", bytes, cudaGetErrorString(e));
    }
    uint8_t* q = (uint8_t*)b->pmem;
    b->theta = (float*)q;
    b->m = (float*)(q + np);
    b->v = (float*)(q + 2 * np);
    b->grad = (float*)(q + 3 * np);
    b->loss = (float*)(q + 4 * np);
    b->images = (__nv_bfloat16*)(q + 4 * np + 256);
    ctx->band = b;
    return FBS_OK;
}

fbs_status need_ready(fbs_ctx* ctx)
{
    if (!ctx->band || !ctx->band->ready)
        return fail(ctx, FBS_ERR_INVALID_ARG, "band network has no weights: call fbs_band_net_init or _load first");
    return FBS_OK;
}

// splitmix64 and a Box-Muller normal, for the initial weights
uint64_t splitmix64(uint64_t& s)
{
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
double uniform01(uint64_t& s) { return ((splitmix64(s) >> 11) + 0.5) * (1.0 / 9007199254740992.0); }

fbs_status upload_params(fbs_ctx* ctx, const float* host, cudaStream_t st)
{
    fbs_band_state* b = ctx->band;
    cudaError_t e = cudaMemcpyAsync(b->theta, host, (size_t)kParams * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->m, 0, (size_t)kParams * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->v, 0, (size_t)kParams * 4, st);
    if (e == cudaSuccess) {
        LaunchScope ls(ctx, FBS_KERNEL_NET, st);
        e = launch_pack_images(b->theta, b->images, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "band network upload");
    b->step = 0;
    b->ready = true;
    return FBS_OK;
}

fbs_status check_pair_shape(fbs_ctx* ctx, const uint8_t* left, const uint8_t* right, int H, int W, int C, int D)
{
    if (!left || !right) return fail(ctx, FBS_ERR_INVALID_ARG, "null image pointer");
    fbs_status s = check_shape(ctx, H, W, C, D);
    if (s != FBS_OK) return s;
    if (ctx->opt.cost != FBS_COST_NCC) return fail(ctx, FBS_ERR_UNSUPPORTED, "the band form uses the NCC cost only");
    return FBS_OK;
}

// Features into the scratch (and optionally the caller's buffers).
fbs_status run_features(fbs_ctx* ctx, const NetScratch& s, const uint8_t* L, const uint8_t* R, int H, int W, int C,
                        int D, float* feat, cudaStream_t st)
{
    const int Hq = (H + 3) / 4, Wq = (W + 3) / 4, Dq = (D + 3) / 4;
    cudaError_t e;
    {
        LaunchScope ls(ctx, FBS_KERNEL_NET, st);
        fbs::note_launch();
        const int tx = fbs::kQuarterX - 2, ty = fbs::kQuarterY - 2;
        const dim3 grid((Wq + tx - 1) / tx, (Hq + ty - 1) / ty, 2);
        auto kernel = C == 3 ? fbs::band_quarter_kernel<3> : fbs::band_quarter_kernel<1>;
        kernel<<<grid, fbs::kQuarterX * fbs::kQuarterY, 0, st>>>(L, R, H, W, s.gq, s.stat);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        LaunchScope ls(ctx, FBS_KERNEL_NET, st);
        const dim3 grid((Wq + fbs::kRowSpan - 1) / fbs::kRowSpan, Hq);
        e = fbs::launch_after(fbs::band_row_sum_kernel, grid, fbs::kRowThreads, fbs::row_sum_smem(Dq), st, s.gq, s.stat,
                              Hq, Wq, Dq, s.kh);
    }
    if (e == cudaSuccess) {
        LaunchScope ls(ctx, FBS_KERNEL_NET, st);
        const dim3 grid((Wq + fbs::kFeatWarps - 1) / fbs::kFeatWarps, (Hq + fbs::kFeatRows - 1) / fbs::kFeatRows);
        e = fbs::launch_after(fbs::band_features_kernel, grid, 32 * fbs::kFeatWarps,
                              fbs::kFeatWarps * fbs::kFeatRows * Dq * sizeof(float), st, s.gq, s.kh, H, W, C, D, s.x0, feat, s.estar);
    }
    return e == cudaSuccess ? FBS_OK : cuda_fail(ctx, e, "band feature launch");
}

// The six convolutions: x0 -> y[0..4] -> out (and the head's other outputs).
fbs_status run_forward(fbs_ctx* ctx, const NetScratch& s, int Hq, int Wq, const ConvHead& head, cudaStream_t st)
{
    fbs_band_state* b = ctx->band;
    const __nv_bfloat16* in = s.x0;
    for (int l = 0; l < kLayers; ++l) {
        const bool last = l == kLayers - 1;
        const float* bias = b->theta + param_offset(l) + 9 * cin(l) * cout(l);
        cudaError_t e;
        {
            LaunchScope ls(ctx, FBS_KERNEL_NET, st);
            e = launch_conv3x3(cin_pad(l), fwd_n(l), in, b->images + fwd_image_offset(l), bias, nullptr,
                               last ? (void*)s.out : (void*)s.y[l], last ? kOut : fwd_n(l), Hq, Wq, 0,
                               last ? kConvLinearF32 : kConvReluBf16, ctx->derr, ctx->wait_cycles, st, last ? head : ConvHead{});
        }
        if (e != cudaSuccess) return cuda_fail(ctx, e, "band network convolution launch");
        if (!last) in = s.y[l];
    }
    return FBS_OK;
}

ConvHead head_planes(const NetScratch& s, int H, int W, float* out_q, float* centre, float* conf)
{
    const bool aligned = (((uintptr_t)centre | (uintptr_t)conf) & 15) == 0;
    return ConvHead{s.estar, out_q, centre, conf, H, W, aligned && W % 4 == 0};
}

// Loss, backward pass into b->grad.
fbs_status run_backward(fbs_ctx* ctx, const NetScratch& s, int H, int W, int D, const int32_t* label_int,
                        const float* label_sub, int half_band, cudaStream_t st)
{
    fbs_band_state* b = ctx->band;
    const int Hq = (H + 3) / 4, Wq = (W + 3) / 4;
    cudaError_t e;
    {
        LaunchScope ls(ctx, FBS_KERNEL_NET, st);
        e = launch_loss(s.out, s.estar, label_int, label_sub, H, W, D, half_band, s.g[5], s.loss_partial, b->loss, st);
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "band loss launch");
    for (int l = kLayers - 1; l >= 0; --l) {
        const __nv_bfloat16* X = l == 0 ? s.x0 : s.y[l - 1];
        {
            LaunchScope ls(ctx, FBS_KERNEL_NET, st);
            e = launch_wgrad(l, X, s.g[l], Hq, Wq, s.partial, b->grad, ctx->derr, ctx->num_sms, st);
        }
        if (e != cudaSuccess) return cuda_fail(ctx, e, "band weight-gradient launch");
        if (l == 0) break;
        {
            // gradient w.r.t. Y_{l-1} through its ReLU
            LaunchScope ls(ctx, FBS_KERNEL_NET, st);
            e = launch_conv3x3(cout_pad(l), cin(l), s.g[l], b->images + dgrad_image_offset(l), nullptr, s.y[l - 1],
                               s.g[l - 1], cin(l), Hq, Wq, 1, kConvMaskBf16, ctx->derr, ctx->wait_cycles, st);
        }
        if (e != cudaSuccess) return cuda_fail(ctx, e, "band data-gradient launch");
    }
    return FBS_OK;
}

fbs_status run_banded(fbs_ctx* ctx, const fbs_pair* p, const float* centre, const float* conf, int h, float theta,
                      const NetScratch& s, cudaStream_t st)
{
    const int H = p->H, W = p->W, D = p->D;
    const int ld = fbs::padded_ld(D);
    const size_t stats = fbs::cost_scratch_bytes(H, W);
    const size_t need = stats + sizeof(float) * (size_t)H * W * ld;
    fbs_status r = ensure(ctx, &ctx->ws, &ctx->ws_bytes, need, "cost volume");
    if (r != FBS_OK) return r;
    const fbs::CostScratch sc = fbs::carve_cost_scratch(ctx->ws, H, W);
    float* cost = (float*)((uint8_t*)ctx->ws + stats);
    cudaError_t e;
    {
        LaunchScope ls(ctx, FBS_KERNEL_NET, st);
        e = fbs::launch_band_tiles(centre, conf, H, W, D, h, theta, s.band, s.tile_range, st);
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "band planning launch");
    {
        LaunchScope ls(ctx, FBS_KERNEL_COST, st);
        e = fbs::launch_cost_band(sc, p->left, p->right, H, W, p->C, D, ld, p->radius, s.tile_range, cost, ctx->num_sms,
                                  st);
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "band cost launch");
    {
        LaunchScope ls(ctx, FBS_KERNEL_AGG_F32, st);
        e = fbs::launch_aggregate_band(cost, ld, p->left, H, W, p->C, D, p->radius, p->sigma_s, p->sigma_r,
                                       s.tile_range, s.band, p->disp_int, p->disp_subpix, ctx->wait_cycles, ctx->derr, st);
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "band aggregation launch");
    return FBS_OK;
}

fbs_status check_band_args(fbs_ctx* ctx, const fbs_pair* p, int h, float theta)
{
    if (!p) return fail(ctx, FBS_ERR_INVALID_ARG, "null pair");
    fbs_status s = fbs::check_path_args(ctx, p->left, p->right, p->H, p->W, p->C, p->D, p->radius, p->sigma_s,
                                        p->sigma_r, p->tau, p->disp_int, p->disp_subpix);
    if (s != FBS_OK) return s;
    if (ctx->opt.cost != FBS_COST_NCC) return fail(ctx, FBS_ERR_UNSUPPORTED, "the band form uses the NCC cost only");
    if (h < 1 || h > 512) return fail(ctx, FBS_ERR_INVALID_ARG, "half_band=%d outside 1..512", h);
    if (std::isnan(theta)) return fail(ctx, FBS_ERR_INVALID_ARG, "conf_threshold is NaN");
    return FBS_OK;
}

}  // namespace

namespace fbs {
void band_free(fbs_ctx* ctx)
{
    if (ctx->band) {
        if (ctx->band->pmem) cudaFree(ctx->band->pmem);
        delete ctx->band;
        ctx->band = nullptr;
    }
    if (ctx->band_ws) cudaFree(ctx->band_ws);
    ctx->band_ws = nullptr;
    ctx->band_ws_bytes = 0;
}
}  // namespace fbs

extern "C" {

size_t fbs_band_net_param_count(void) { return (size_t)kParams; }

fbs_status fbs_band_net_init(fbs_ctx* ctx, uint64_t seed)
{
    if (!ctx) return FBS_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    fbs_status s = ensure_state(ctx);
    if (s != FBS_OK) return s;
    std::vector<float> h(kParams, 0.f);
    uint64_t st = seed ^ 0x6A09E667F3BCC909ull;
    for (int l = 0; l < kLayers; ++l) {
        const double sd = std::sqrt(2.0 / (9.0 * cin(l))) * (l == kLayers - 1 ? 0.1 : 1.0);
        float* W = h.data() + param_offset(l);
        for (int i = 0; i < 9 * cin(l) * cout(l); ++i) {
            const double u1 = uniform01(st), u2 = uniform01(st);
            W[i] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
        }
    }
    return upload_params(ctx, h.data(), ctx->stream);
}

fbs_status fbs_band_net_set_params(fbs_ctx* ctx, const float* params, size_t n)
{
    if (!ctx || !params) return fail(ctx, FBS_ERR_INVALID_ARG, "null context or parameters");
    if (n != (size_t)kParams) return fail(ctx, FBS_ERR_INVALID_ARG, "expected %d parameters, got %zu", kParams, n);
    for (size_t i = 0; i < n; ++i)
        if (!std::isfinite(params[i])) return fail(ctx, FBS_ERR_INVALID_ARG, "parameter %zu is not finite", i);
    DeviceGuard g(ctx->device);
    fbs_status s = ensure_state(ctx);
    if (s != FBS_OK) return s;
    return upload_params(ctx, params, ctx->stream);
}

fbs_status fbs_band_net_get_params(fbs_ctx* ctx, float* params, size_t n)
{
    if (!ctx || !params) return fail(ctx, FBS_ERR_INVALID_ARG, "null context or parameters");
    if (n != (size_t)kParams) return fail(ctx, FBS_ERR_INVALID_ARG, "expected %d parameters, got %zu", kParams, n);
    fbs_status s = need_ready(ctx);
    if (s != FBS_OK) return s;
    DeviceGuard g(ctx->device);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(params, ctx->band->theta, n * 4, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? FBS_OK : cuda_fail(ctx, e, "band parameters read-back");
}

fbs_status fbs_band_net_save(fbs_ctx* ctx, const char* path)
{
    if (!ctx || !path) return fail(ctx, FBS_ERR_INVALID_ARG, "null context or path");
    std::vector<float> h(kParams);
    fbs_status s = fbs_band_net_get_params(ctx, h.data(), h.size());
    if (s != FBS_OK) return s;
    FILE* f = std::fopen(path, "wb");
    if (!f) return fail(ctx, FBS_ERR_INVALID_ARG, "cannot open %s for writing", path);
    const uint32_t n = (uint32_t)kParams;
    bool ok = std::fwrite("FBSBAND1", 1, 8, f) == 8 && std::fwrite(&n, 4, 1, f) == 1 &&
              std::fwrite(h.data(), 4, h.size(), f) == h.size();
    ok = (std::fclose(f) == 0) && ok;
    return ok ? FBS_OK : fail(ctx, FBS_ERR_INVALID_ARG, "short write to %s", path);
}

fbs_status fbs_band_net_load(fbs_ctx* ctx, const char* path)
{
    if (!ctx || !path) return fail(ctx, FBS_ERR_INVALID_ARG, "null context or path");
    FILE* f = std::fopen(path, "rb");
    if (!f) return fail(ctx, FBS_ERR_INVALID_ARG, "cannot open %s", path);
    char tag[8];
    uint32_t n = 0;
    std::vector<float> h(kParams);
    bool ok = std::fread(tag, 1, 8, f) == 8 && std::memcmp(tag, "FBSBAND1", 8) == 0 && std::fread(&n, 4, 1, f) == 1 &&
              n == (uint32_t)kParams && std::fread(h.data(), 4, h.size(), f) == h.size();
    std::fclose(f);
    if (!ok) return fail(ctx, FBS_ERR_INVALID_ARG, "%s is not a band-network file of %d parameters", path, kParams);
    return fbs_band_net_set_params(ctx, h.data(), h.size());
}

fbs_status fbs_band_features(fbs_ctx* ctx, const uint8_t* left, const uint8_t* right, int H, int W, int C, int D,
                             float* feat, int32_t* estar, void* cuda_stream)
{
    if (!ctx) return FBS_ERR_INVALID_ARG;
    fbs_status s = check_pair_shape(ctx, left, right, H, W, C, D);
    if (s != FBS_OK) return s;
    if (!feat && !estar) return fail(ctx, FBS_ERR_INVALID_ARG, "both outputs are NULL");
    DeviceGuard g(ctx->device);
    cudaStream_t st = pick_stream(ctx, cuda_stream);
    s = ensure(ctx, &ctx->band_ws, &ctx->band_ws_bytes, net_scratch_bytes(H, W, D, false, false), "band scratch");
    if (s != FBS_OK) return s;
    const NetScratch sc = carve_net(ctx->band_ws, H, W, D, false, false);
    s = run_features(ctx, sc, left, right, H, W, C, D, feat, st);
    if (s != FBS_OK || !estar) return s;
    const size_t P = (size_t)((H + 3) / 4) * ((W + 3) / 4);
    cudaError_t e = cudaMemcpyAsync(estar, sc.estar, P * 4, cudaMemcpyDeviceToDevice, st);
    return e == cudaSuccess ? FBS_OK : cuda_fail(ctx, e, "coarse winner copy");
}

fbs_status fbs_band_net_forward(fbs_ctx* ctx, const uint8_t* left, const uint8_t* right, int H, int W, int C, int D,
                                float* out_q, float* centre, float* conf, void* cuda_stream)
{
    if (!ctx) return FBS_ERR_INVALID_ARG;
    fbs_status s = check_pair_shape(ctx, left, right, H, W, C, D);
    if (s != FBS_OK) return s;
    if (!out_q && !centre && !conf) return fail(ctx, FBS_ERR_INVALID_ARG, "all outputs are NULL");
    if ((s = need_ready(ctx)) != FBS_OK) return s;
    DeviceGuard g(ctx->device);
    cudaStream_t st = pick_stream(ctx, cuda_stream);
    s = ensure(ctx, &ctx->band_ws, &ctx->band_ws_bytes, net_scratch_bytes(H, W, D, false, false), "band scratch");
    if (s != FBS_OK) return s;
    const NetScratch sc = carve_net(ctx->band_ws, H, W, D, false, false);
    const int Hq = (H + 3) / 4, Wq = (W + 3) / 4;
    if ((s = run_features(ctx, sc, left, right, H, W, C, D, nullptr, st)) != FBS_OK) return s;
    const bool direct = ((uintptr_t)out_q & 3) == 0;   // a copy takes any address
    s = run_forward(ctx, sc, Hq, Wq, head_planes(sc, H, W, direct ? out_q : nullptr, centre, conf), st);
    if (s != FBS_OK) return s;
    ctx->band->last_H = H;
    ctx->band->last_W = W;
    ctx->band->last_D = D;
    ctx->band->last_training = false;
    if (direct) return FBS_OK;
    cudaError_t e = cudaMemcpyAsync(out_q, sc.out, (size_t)Hq * Wq * 8, cudaMemcpyDeviceToDevice, st);
    return e == cudaSuccess ? FBS_OK : cuda_fail(ctx, e, "band network output copy");
}

fbs_status fbs_band_net_train_step(fbs_ctx* ctx, const uint8_t* left, const uint8_t* right, int H, int W, int C,
                                   int D, const int32_t* label_int, const float* label_sub, int half_band, float lr,
                                   float* loss, float* grad, void* cuda_stream)
{
    if (!ctx) return FBS_ERR_INVALID_ARG;
    fbs_status s = check_pair_shape(ctx, left, right, H, W, C, D);
    if (s != FBS_OK) return s;
    if (!label_int || !label_sub) return fail(ctx, FBS_ERR_INVALID_ARG, "null label pointer");
    if (half_band < 1 || half_band > 512) return fail(ctx, FBS_ERR_INVALID_ARG, "half_band=%d outside 1..512", half_band);
    if (!(std::isfinite(lr) && lr >= 0.f)) return fail(ctx, FBS_ERR_INVALID_ARG, "lr must be finite and >= 0");
    if ((s = need_ready(ctx)) != FBS_OK) return s;
    DeviceGuard g(ctx->device);
    cudaStream_t st = pick_stream(ctx, cuda_stream);
    s = ensure(ctx, &ctx->band_ws, &ctx->band_ws_bytes, net_scratch_bytes(H, W, D, true, false), "band scratch");
    if (s != FBS_OK) return s;
    const NetScratch sc = carve_net(ctx->band_ws, H, W, D, true, false);
    const int Hq = (H + 3) / 4, Wq = (W + 3) / 4;
    fbs_band_state* b = ctx->band;
    if ((s = run_features(ctx, sc, left, right, H, W, C, D, nullptr, st)) != FBS_OK) return s;
    if ((s = run_forward(ctx, sc, Hq, Wq, ConvHead{}, st)) != FBS_OK) return s;
    if ((s = run_backward(ctx, sc, H, W, D, label_int, label_sub, half_band, st)) != FBS_OK) return s;
    b->last_H = H;
    b->last_W = W;
    b->last_D = D;
    b->last_training = true;
    cudaError_t e = cudaSuccess;
    if (grad) e = cudaMemcpyAsync(grad, b->grad, (size_t)kParams * 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, b->loss, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && lr > 0.f) {
        b->step += 1;
        const double c1 = 1.0 / (1.0 - std::pow(0.9, (double)b->step));
        const double c2 = 1.0 / (1.0 - std::pow(0.999, (double)b->step));
        {
            LaunchScope ls(ctx, FBS_KERNEL_NET, st);
            e = launch_adam(b->theta, b->m, b->v, b->grad, kParams, lr, (float)c1, (float)c2, st);
        }
        if (e == cudaSuccess) {
            LaunchScope ls(ctx, FBS_KERNEL_NET, st);
            e = launch_pack_images(b->theta, b->images, st);
        }
    }
    if (e == cudaSuccess && (grad || loss)) e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? FBS_OK : cuda_fail(ctx, e, "band training step");
}

fbs_status fbs_band_net_trace(fbs_ctx* ctx, float* acts, float* grads, void* cuda_stream)
{
    if (!ctx) return FBS_ERR_INVALID_ARG;
    if (!acts && !grads) return fail(ctx, FBS_ERR_INVALID_ARG, "both outputs are NULL");
    if (!ctx->band || ctx->band->last_H == 0)
        return fail(ctx, FBS_ERR_INVALID_ARG, "no band-network forward or training call to trace");
    fbs_band_state* b = ctx->band;
    if (grads && !b->last_training)
        return fail(ctx, FBS_ERR_INVALID_ARG, "gradients exist only after fbs_band_net_train_step");
    DeviceGuard g(ctx->device);
    cudaStream_t st = pick_stream(ctx, cuda_stream);
    const int H = b->last_H, W = b->last_W, D = b->last_D;
    const NetScratch sc = carve_net(ctx->band_ws, H, W, D, b->last_training, false);
    const size_t P = (size_t)((H + 3) / 4) * ((W + 3) / 4);
    cudaError_t e = cudaSuccess;
    LaunchScope ls(ctx, FBS_KERNEL_OTHER, st);
    auto convert = [&](const __nv_bfloat16* src, float* dst, size_t n) {
        if (e != cudaSuccess) return;
        fbs::note_launch();
        const int blocks = (int)std::min<size_t>((n + 255) / 256, 1024);
        fbs::bf16_to_f32_kernel<<<blocks, 256, 0, st>>>(src, dst, n);
        e = cudaGetLastError();
    };
    if (acts) {
        float* o = acts;
        convert(sc.x0, o, P * 8);
        o += P * 8;
        for (int l = 0; l < 5; ++l, o += P * 32) convert(sc.y[l], o, P * 32);
        if (e == cudaSuccess) e = cudaMemcpyAsync(o, sc.out, P * 8, cudaMemcpyDeviceToDevice, st);
    }
    if (grads) {
        float* o = grads;
        for (int l = 0; l < 5; ++l, o += P * 32) convert(sc.g[l], o, P * 32);
        convert(sc.g[5], o, P * 8);
    }
    return e == cudaSuccess ? FBS_OK : cuda_fail(ctx, e, "band network trace");
}

fbs_status fbs_band_feature_points(fbs_ctx* ctx, const uint8_t* left, const uint8_t* right, int H, int W, int C,
                                  int D, float margin_threshold, float* centre, float* conf, void* cuda_stream)
{
    if (!ctx) return FBS_ERR_INVALID_ARG;
    fbs_status s = check_pair_shape(ctx, left, right, H, W, C, D);
    if (s != FBS_OK) return s;
    if (!centre || !conf) return fail(ctx, FBS_ERR_INVALID_ARG, "null centre or confidence");
    if (std::isnan(margin_threshold)) return fail(ctx, FBS_ERR_INVALID_ARG, "margin_threshold is NaN");
    DeviceGuard g(ctx->device);
    cudaStream_t st = pick_stream(ctx, cuda_stream);
    s = ensure(ctx, &ctx->band_ws, &ctx->band_ws_bytes, net_scratch_bytes(H, W, D, false, false), "band scratch");
    if (s != FBS_OK) return s;
    const NetScratch sc = carve_net(ctx->band_ws, H, W, D, false, false);
    if ((s = run_features(ctx, sc, left, right, H, W, C, D, sc.featf, st)) != FBS_OK) return s;
    LaunchScope ls(ctx, FBS_KERNEL_NET, st);
    fbs::note_launch();
    fbs::band_feature_points_kernel<<<dim3((W + 255) / 256, H), 256, 0, st>>>(sc.featf, sc.estar, H, W,
                                                                           margin_threshold, centre, conf);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? FBS_OK : cuda_fail(ctx, e, "feature-point proposal launch");
}

fbs_status fbs_band_limits(fbs_ctx* ctx, const float* centre, const float* conf, int n, int D, int half_band,
                           float conf_threshold, int32_t* lo, int32_t* hi, void* cuda_stream)
{
    if (!ctx) return FBS_ERR_INVALID_ARG;
    if (!centre || !conf || !lo || !hi) return fail(ctx, FBS_ERR_INVALID_ARG, "null pointer");
    if (n < 1 || D < 1 || D > 1024) return fail(ctx, FBS_ERR_INVALID_ARG, "n=%d or D=%d out of range", n, D);
    if (half_band < 1 || half_band > 512) return fail(ctx, FBS_ERR_INVALID_ARG, "half_band=%d outside 1..512", half_band);
    if (std::isnan(conf_threshold)) return fail(ctx, FBS_ERR_INVALID_ARG, "conf_threshold is NaN");
    DeviceGuard g(ctx->device);
    cudaStream_t st = pick_stream(ctx, cuda_stream);
    LaunchScope ls(ctx, FBS_KERNEL_NET, st);
    fbs::note_launch();
    fbs::band_limits_kernel<<<(n + 255) / 256, 256, 0, st>>>(centre, conf, n, D, half_band, conf_threshold, lo, hi);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? FBS_OK : cuda_fail(ctx, e, "band limits launch");
}

fbs_status fbs_compute_disparity_banded(fbs_ctx* ctx, const fbs_pair* pair, const float* centre, const float* conf,
                                        int half_band, float conf_threshold, void* cuda_stream)
{
    if (!ctx) return FBS_ERR_INVALID_ARG;
    fbs_status s = check_band_args(ctx, pair, half_band, conf_threshold);
    if (s != FBS_OK) return s;
    if (!centre || !conf) return fail(ctx, FBS_ERR_INVALID_ARG, "null centre or confidence");
    DeviceGuard g(ctx->device);
    cudaStream_t st = pick_stream(ctx, cuda_stream);
    s = ensure(ctx, &ctx->band_ws, &ctx->band_ws_bytes, net_scratch_bytes(pair->H, pair->W, pair->D, false, true),
               "band scratch");
    if (s != FBS_OK) return s;
    const NetScratch sc = carve_net(ctx->band_ws, pair->H, pair->W, pair->D, false, true);
    return run_banded(ctx, pair, centre, conf, half_band, conf_threshold, sc, st);
}

fbs_status fbs_compute_disparity_learned(fbs_ctx* ctx, const fbs_pair* pair, int half_band, float conf_threshold,
                                         void* cuda_stream)
{
    if (!ctx) return FBS_ERR_INVALID_ARG;
    fbs_status s = check_band_args(ctx, pair, half_band, conf_threshold);
    if (s != FBS_OK) return s;
    if ((s = need_ready(ctx)) != FBS_OK) return s;
    DeviceGuard g(ctx->device);
    cudaStream_t st = pick_stream(ctx, cuda_stream);
    const int H = pair->H, W = pair->W;
    s = ensure(ctx, &ctx->band_ws, &ctx->band_ws_bytes, net_scratch_bytes(H, W, pair->D, false, true), "band scratch");
    if (s != FBS_OK) return s;
    const NetScratch sc = carve_net(ctx->band_ws, H, W, pair->D, false, true);
    const int Hq = (H + 3) / 4, Wq = (W + 3) / 4;
    if ((s = run_features(ctx, sc, pair->left, pair->right, H, W, pair->C, pair->D, nullptr, st)) != FBS_OK) return s;
    s = run_forward(ctx, sc, Hq, Wq, head_planes(sc, H, W, nullptr, sc.centre, sc.conf), st);
    if (s != FBS_OK) return s;
    return run_banded(ctx, pair, sc.centre, sc.conf, half_band, conf_threshold, sc, st);
}

}  // extern "C"
