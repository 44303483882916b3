// Step 1 of fast bilateral stereo: the matching-cost volume.
//
// NCC (Sec. II-A, Eq. (1)-(3), varrho = 1): with the intensity g taken as the
// channel sum, n = 9 and the block sums S = sum g, Q = sum g^2 and
// P = sum g_l g_r, Eq. (1) multiplied through by n^2 reads
//     c = (n P - S_l S_r) / sqrt((n Q_l - S_l^2) (n Q_r - S_r^2)).
// Every sum and both numerator terms are exact in int32 (g <= 765), so only the
// final normalisation is rounded.  Stored cost: C = 1 - c.  Boundary rules:
// blocks clamp to the image; u - d < 0 gives the maximum cost 2; a block of
// zero variance gives c = 0.
//
// As in the paper (Sec. II-A, Sec. III) the per-pixel block statistics are
// computed once per pixel, so the per-(p, d) work is the dot product P.  Two
// kernels write the two layouts:
//   * cost_kernel, [H][W][ld] float32 (D innermost; the FP32 aggregation),
//     padding d in [D, ld) written as 0.  A pre-pass (grey_stats_kernel: g, S,
//     1/sqrt(nQ - S^2)) fills statistics planes; a thread owns a run of 4
//     pixels and 8 consecutive disparities (left 3x6 grey window in
//     registers, right window sliding one column per disparity, three column
//     products per output column summed by a sliding 3-column window);
//     results are staged in shared memory as [d][x] and written out with D
//     innermost.
//   * cost_xb_ncc_kernel, 16-bit x-blocked [H][ceil(W/8)][Dp][8] (the tensor-core
//     aggregation): for a row y and a block of 8 columns, the Dp x 8 block is
//     contiguous, so the tensor-core kernel's TMA reads contiguous blocks that
//     land as K-major core matrices; columns x >= W of the last block are 0.
//     One launch computes the statistics of the rows it stages, the costs, the
//     pad rows D .. Dp-1 and the left image's packed guide (its comment says how);
//     cost_xb_tad_kernel does the same for TAD.
// Both round the normalisation the same way (ncc_cost), so the 16-bit volume
// equals the FP32 volume rounded to 16 bits.
//
// TAD (not in the paper): C = min(mean_c |I_l(u,v) - I_r(u-d,v)|, tau), tau
// when u - d < 0.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "fbs_internal.cuh"
#include "packed_f32.cuh"
#include "tc_aggregate.cuh"

namespace fbs {
namespace {

constexpr int kXS = 128;          // pixels per CTA along x
constexpr int kDC = 64;           // disparities per pass
constexpr int kThreads = 256;     // 32 runs of 4 pixels x 8 groups of 8 disparities
constexpr int kStage = kXS + 1;   // staged row pitch (odd: conflict-free transposed reads)
constexpr int kNRG = kXS + kDC + 2;        // right grey columns per pass
constexpr int kQR = (kNRG + 3) / 4;        // de-interleaved quarter length of a right row
constexpr int kQS = (kXS + kDC) / 4;       // same for the right block statistics

// Lanes of a warp own pixel runs 4*run .. 4*run+3 and read or write column
// 4*run + k together; storing column c at (c & 3) * quarter + (c >> 2) puts
// those 32 accesses in 32 different banks.
__device__ __forceinline__ int stage_pos(int x) { return (x & 3) * 32 + (x >> 2); }
__device__ __forceinline__ int rpos(int c) { return (c & 3) * kQR + (c >> 2); }
__device__ __forceinline__ int spos(int c) { return (c & 3) * kQS + (c >> 2); }

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// C = 1 - c with c = num * (rv_l * rv_r): one rounded product of the two
// normalisers, then one fused multiply-add (every cost kernel uses this, so the
// FP32 and the 16-bit volumes hold the same values before the 16-bit rounding).
__device__ __forceinline__ float ncc_cost(int num, float rv_l, float rv_r)
{
    return __fmaf_rn(-__int2float_rn(num), __fmul_rn(rv_l, rv_r), 1.f);
}

// Per-pixel statistics of one image: g = channel sum, S = 3x3 box sum of g
// (clamped), rv = 1/sqrt(9 Q - S^2) or 0 for a flat block.
__device__ __forceinline__ void stats_pixel(const uint8_t* __restrict__ src, int img, int H, int W, int C, int x,
                                            int y, int16_t* __restrict__ g_out, int* __restrict__ s_out,
                                            float* __restrict__ rv_out, uint2* __restrict__ rgbx)
{
    const size_t plane = (size_t)H * W;
    int s = 0, q = 0;
#pragma unroll
    for (int j = -1; j <= 1; ++j) {
        const int yy = clampi(y + j, 0, H - 1);
#pragma unroll
        for (int k = -1; k <= 1; ++k) {
            const uint8_t* p = src + ((size_t)yy * W + clampi(x + k, 0, W - 1)) * C;
            int g = p[0];
            if (C == 3) g += p[1] + p[2];
            s += g;
            q += g * g;
        }
    }
    const uint8_t* p = src + ((size_t)y * W + x) * C;
    int g = p[0];
    if (C == 3) g += p[1] + p[2];
    if (rgbx != nullptr && img == 0) {
        const uint32_t c = C == 3 ? (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) : (uint32_t)p[0];
        rgbx[(size_t)y * rgbx_pitch(W) + x] = make_uint2(c, (uint32_t)__dp4a(c, c, 0u));
    }
    const int v = 9 * q - s * s;
    const size_t o = img * plane + (size_t)y * W + x;
    g_out[o] = (int16_t)g;
    s_out[o] = s;
    rv_out[o] = v > 0 ? rsqrtf((float)v) : 0.f;
}

__global__ void __launch_bounds__(256)
grey_stats_kernel(const uint8_t* __restrict__ L, const uint8_t* __restrict__ R, int H, int W, int C,
                  int16_t* __restrict__ g_out, int* __restrict__ s_out, float* __restrict__ rv_out,
                  uint2* __restrict__ rgbx)
{
    const int img = blockIdx.z;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= W) return;
    stats_pixel(img == 0 ? L : R, img, H, W, C, x, blockIdx.y, g_out, s_out, rv_out, rgbx);
}

// Batched statistics: an item is one row of one pair (both images).
__global__ void __launch_bounds__(256)
grey_stats_batched_kernel(const BatchPair* __restrict__ pairs, int npairs, int nitems, int* __restrict__ counter)
{
    __shared__ int item_s;
    for (;;) {
        if (threadIdx.x == 0) item_s = atomicAdd(counter, 1);
        __syncthreads();
        const int item = item_s;
        __syncthreads();
        if (item >= nitems) break;
        const BatchPair& bp = pairs[find_pair(pairs, npairs, item, &BatchPair::stat_off)];
        const int y = item - bp.stat_off;
        if (bp.mode != 0) continue;   // TAD needs no statistics
        for (int x = threadIdx.x; x < bp.W; x += blockDim.x)
            for (int img = 0; img < 2; ++img)
                stats_pixel(img == 0 ? bp.left : bp.right, img, bp.H, bp.W, bp.C, x, y, bp.sc.g, bp.sc.s, bp.sc.rv,
                            bp.sc.rgbx);
    }
}

template <typename T>
__device__ __forceinline__ T to_out(float v);
template <>
__device__ __forceinline__ float to_out<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 to_out<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <>
__device__ __forceinline__ __half to_out<__half>(float v) { return __float2half_rn(v); }

template <typename T>
__device__ __forceinline__ uint4 pack8(const T (&v)[8])
{
    static_assert(sizeof(T) == 2, "16-bit values");
    uint32_t w[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
        w[c] = (uint32_t)*reinterpret_cast<const unsigned short*>(&v[2 * c]) |
               ((uint32_t)*reinterpret_cast<const unsigned short*>(&v[2 * c + 1]) << 16);
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// MODE 0: NCC from the statistics planes; MODE 1: TAD from the raw images.
// out is [H][W][ld] (T = float).
// One row y and 128 pixels from x0, disparities [d_begin, d_end) (all: 0, D);
// ends with a __syncthreads.  out_r (nullable, FP32 layout only): the right
// view's volume, which holds the same costs at (x - d, y, d) (Sec. II-A, Sec. III).
template <int MODE, typename T>
__device__ __forceinline__ void cost_tile(const int16_t* __restrict__ gplane, const int* __restrict__ splane,
                                          const float* __restrict__ rvplane, const uint8_t* __restrict__ L,
                                          const uint8_t* __restrict__ R, int H, int W, int C, int D, int ld, float tau,
                                          T* __restrict__ out, int x0, int y, int* smem_i, int d_begin, int d_end,
                                          float* __restrict__ out_r = nullptr)
{
    const int tid = threadIdx.x;
    const int nxs = min(kXS, W - x0);
    const size_t plane = (size_t)H * W;
    // layout: stage [kDC][kStage] float | left grey [3][kXS+2] | right grey [3][kXS+kDC+2] |
    //         S_l, rv_l [kXS] | S_r, rv_r [kXS+kDC]
    float* stage = (float*)smem_i;
    int* gl = (int*)(stage + kDC * kStage);
    int* gr = gl + 3 * (kXS + 2);      // [3][4 * kQR], column c at rpos(c)
    int* sl = gr + 3 * 4 * kQR;
    float* rl = (float*)(sl + kXS);
    int* sr = (int*)(rl + kXS);
    float* rr = (float*)(sr + kXS + kDC);
    uchar4* pl = (uchar4*)gl;          // TAD: raw left row [kXS]
    uchar4* pr = pl + kXS;             // TAD: raw right row [kXS + kDC]

    const int run = tid & 31;          // pixels 4*run .. 4*run+3 of the CTA
    const int dg = tid >> 5;           // disparities dc + 8*dg .. +7
    const int xl0 = 4 * run;

    if (MODE == 0) {
        // left grey window rows y-1..y+1, virtual columns x0-1 .. x0+kXS
        for (int i = tid; i < 3 * (kXS + 2); i += kThreads) {
            const int j = i / (kXS + 2), c = i - j * (kXS + 2);
            gl[i] = gplane[(size_t)clampi(y - 1 + j, 0, H - 1) * W + clampi(x0 - 1 + c, 0, W - 1)];
        }
        for (int i = tid; i < kXS; i += kThreads) {
            const int x = clampi(x0 + i, 0, W - 1);
            sl[i] = splane[(size_t)y * W + x];
            rl[i] = rvplane[(size_t)y * W + x];
        }
    } else {
        for (int i = tid; i < kXS; i += kThreads) {
            const uint8_t* p = L + ((size_t)y * W + clampi(x0 + i, 0, W - 1)) * C;
            pl[i] = C == 3 ? make_uchar4(p[0], p[1], p[2], 0) : make_uchar4(p[0], 0, 0, 0);
        }
    }

    for (int dc = d_begin; dc < d_end; dc += kDC) {
        // right columns for this pass: virtual columns rb .. rb + NRG - 1 with
        // rb = x0 - dc - kDC - 1; the right block of (x, d) spans x-d-1 .. x-d+1
        const int rb = x0 - dc - kDC - 1;
        if (MODE == 0) {
            for (int i = tid; i < 3 * kNRG; i += kThreads) {
                const int j = i / kNRG, c = i - j * kNRG;
                gr[j * 4 * kQR + rpos(c)] =
                    gplane[plane + (size_t)clampi(y - 1 + j, 0, H - 1) * W + clampi(rb + c, 0, W - 1)];
            }
            // right block centres rb+1 .. rb+kXS+kDC
            for (int i = tid; i < kXS + kDC; i += kThreads) {
                const int x = clampi(rb + 1 + i, 0, W - 1);
                sr[spos(i)] = splane[plane + (size_t)y * W + x];
                rr[spos(i)] = rvplane[plane + (size_t)y * W + x];
            }
        } else {
            for (int i = tid; i < kXS + kDC; i += kThreads) {
                const uint8_t* p = R + ((size_t)y * W + clampi(rb + 1 + i, 0, W - 1)) * C;
                pr[i] = C == 3 ? make_uchar4(p[0], p[1], p[2], 0) : make_uchar4(p[0], 0, 0, 0);
            }
        }
        __syncthreads();

        const int d_first = dc + 8 * dg;
        if (MODE == 0) {
            int glw[3][6];
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int c = 0; c < 6; ++c) glw[j][c] = gl[j * (kXS + 2) + xl0 + c];
            int sli[4];
            float rli[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                sli[i] = sl[xl0 + i];
                rli[i] = rl[xl0 + i];
            }
            // right window for d_first: virtual columns x0+xl0-d-1 .. +4, index (col - rb)
            int grw[3][6];
            int srw[4];
            float rrw[4];
            {
                const int base = x0 + xl0 - d_first - 1 - rb;
#pragma unroll
                for (int j = 0; j < 3; ++j)
#pragma unroll
                    for (int c = 0; c < 6; ++c) grw[j][c] = gr[j * 4 * kQR + rpos(base + c)];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    srw[i] = sr[spos(base + i)];
                    rrw[i] = rr[spos(base + i)];
                }
            }
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const int d = d_first + s;
                if (s > 0) {
                    // slide one column to the left: d grew by one
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
#pragma unroll
                        for (int c = 5; c > 0; --c) grw[j][c] = grw[j][c - 1];
                    }
                    const int base = x0 + xl0 - d - 1 - rb;
#pragma unroll
                    for (int j = 0; j < 3; ++j) grw[j][0] = gr[j * 4 * kQR + rpos(base)];
#pragma unroll
                    for (int i = 3; i > 0; --i) {
                        srw[i] = srw[i - 1];
                        rrw[i] = rrw[i - 1];
                    }
                    srw[0] = sr[spos(base)];
                    rrw[0] = rr[spos(base)];
                }
                int cp[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) cp[c] = glw[0][c] * grw[0][c] + glw[1][c] * grw[1][c] + glw[2][c] * grw[2][c];
                float* st = stage + (d - dc) * kStage + run;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int x = x0 + xl0 + i;
                    const int num = 9 * (cp[i] + cp[i + 1] + cp[i + 2]) - sli[i] * srw[i];
                    st[32 * i] = x - d < 0 ? 2.f : ncc_cost(num, rli[i], rrw[i]);
                }
            }
        } else {
            const float inv_c = 1.f / (float)C;
#pragma unroll 2
            for (int s = 0; s < 8; ++s) {
                const int d = d_first + s;
                float* st = stage + (d - dc) * kStage + run;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int x = x0 + xl0 + i;
                    float cst = tau;
                    if (x - d >= 0) {
                        const uchar4 a = pl[xl0 + i];
                        const uchar4 b = pr[x - d - (rb + 1)];
                        const int sad = abs((int)a.x - (int)b.x) + abs((int)a.y - (int)b.y) + abs((int)a.z - (int)b.z);
                        cst = fminf((float)sad * inv_c, tau);
                    }
                    st[32 * i] = cst;
                }
            }
        }
        __syncthreads();

        const int nd = min(kDC, d_end - dc);
        // out[(y*W + x)*ld + d]; padding d in [D, ld) of the last pass written as 0
        const int ndw = (dc + kDC >= d_end) ? (d_end == D ? ld - dc : d_end - dc) : kDC;
        const int warp = tid >> 5, lane = tid & 31;
        for (int x = warp; x < nxs; x += kThreads / 32) {
            T* o = out + ((size_t)y * W + x0 + x) * ld + dc;
            const int px = stage_pos(x);
            for (int dd = lane; dd < ndw; dd += 32) o[dd] = to_out<T>(dd < nd ? stage[dd * kStage + px] : 0.f);
        }
        if (out_r != nullptr) {
            // right pixel xr = x - d receives the contiguous disparities
            // max(dc, x0 - xr) .. min(dc + nd - 1, x0 + nxs - 1 - xr) of this pass
            const int xr_lo = max(0, x0 - dc - nd + 1), xr_hi = x0 + nxs - 1 - dc;
            for (int xr = xr_lo + warp; xr <= xr_hi; xr += kThreads / 32) {
                const int dlo = max(dc, x0 - xr), dhi = min(dc + nd - 1, x0 + nxs - 1 - xr);
                float* o = out_r + ((size_t)y * W + xr) * ld;
                for (int d = dlo + lane; d <= dhi; d += 32) o[d] = stage[(d - dc) * kStage + stage_pos(xr + d - x0)];
            }
        }
        __syncthreads();
    }
}

template <int MODE, typename T>
__global__ void __launch_bounds__(kThreads)
cost_kernel(const int16_t* __restrict__ gplane, const int* __restrict__ splane, const float* __restrict__ rvplane,
            const uint8_t* __restrict__ L, const uint8_t* __restrict__ R, int H, int W, int C, int D, int ld,
            float tau, T* __restrict__ out)
{
    extern __shared__ int smem_i[];
    cost_tile<MODE, T>(gplane, splane, rvplane, L, R, H, W, C, D, ld, tau, out, blockIdx.x * kXS, blockIdx.y,
                               smem_i, 0, D);
}

// Batched FP32 cost volumes [H][W][ld]: an item is (row, 128-pixel segment) of a pair.
__global__ void __launch_bounds__(kThreads)
cost_batched_kernel(const BatchPair* __restrict__ pairs, int npairs, int nitems, int* __restrict__ counter)
{
    extern __shared__ int smem_i[];
    __shared__ int item_s;
    for (;;) {
        if (threadIdx.x == 0) item_s = atomicAdd(counter, 1);
        __syncthreads();
        const int item = item_s;
        __syncthreads();
        if (item >= nitems) break;
        const BatchPair& bp = pairs[find_pair(pairs, npairs, item, &BatchPair::cost_off)];
        const int t = item - bp.cost_off;
        const int nseg = (bp.W + kXS - 1) / kXS;
        const int x0 = (t % nseg) * kXS, y = t / nseg;
        if (bp.mode == 0)
            cost_tile<0, float>(bp.sc.g, bp.sc.s, bp.sc.rv, bp.left, bp.right, bp.H, bp.W, bp.C, bp.D, bp.ld,
                                       bp.tau, bp.cost, x0, y, smem_i, 0, bp.D);
        else
            cost_tile<1, float>(bp.sc.g, bp.sc.s, bp.sc.rv, bp.left, bp.right, bp.H, bp.W, bp.C, bp.D, bp.ld,
                                       bp.tau, bp.cost, x0, y, smem_i, 0, bp.D);
    }
}

// Band form: NCC costs of row y, pixels x0 .. x0+127, for the disparities
// that some aggregation tile reading this segment needs: the hull of the
// ranges [d_begin, d_end) of every tile whose window halo (the tile grown by
// rho) overlaps the segment.  Entries outside that hull are not written.
__global__ void __launch_bounds__(kThreads)
cost_band_kernel(const int16_t* __restrict__ gplane, const int* __restrict__ splane,
                 const float* __restrict__ rvplane, int H, int W, int D, int ld, int rho,
                 const int2* __restrict__ tile_range, int ntx, int nty, float* __restrict__ out)
{
    extern __shared__ int smem_i[];
    __shared__ int lo_s, hi_s;
    const int x0 = blockIdx.x * kXS, y = blockIdx.y;
    if (threadIdx.x == 0) {
        lo_s = D;
        hi_s = 0;
    }
    __syncthreads();
    // tiles ty with 4ty - rho <= y <= 4ty + 3 + rho, tx with halo columns meeting [x0, x0 + 127]
    const int ty0 = max(0, (y - rho + kAggTileY * 64) / kAggTileY - 64);
    const int ty1 = min(nty - 1, (y + rho) / kAggTileY);
    const int tx0 = max(0, (x0 - rho + kAggTileX * 64) / kAggTileX - 64);
    const int tx1 = min(ntx - 1, (x0 + kXS - 1 + rho) / kAggTileX);
    const int nx = tx1 - tx0 + 1;
    int lo = D, hi = 0;
    for (int i = threadIdx.x; i < (ty1 - ty0 + 1) * nx; i += kThreads) {
        const int2 r = tile_range[(size_t)(ty0 + i / nx) * ntx + tx0 + i % nx];
        lo = min(lo, r.x);
        hi = max(hi, r.y);
    }
    if (ty0 <= ty1 && tx0 <= tx1) {
        atomicMin(&lo_s, lo);
        atomicMax(&hi_s, hi);
    }
    __syncthreads();
    const int d_begin = lo_s, d_end = hi_s;
    if (d_begin >= d_end) return;
    cost_tile<0, float>(gplane, splane, rvplane, nullptr, nullptr, H, W, 1, D, ld, 0.f, out, x0, y, smem_i,
                               d_begin, d_end);
}

// Both views at once (FP32 layouts): the left volume as cost_kernel writes it
// and the right volume from the same staged costs.
template <int MODE>
__global__ void __launch_bounds__(kThreads)
cost_lr_kernel(const int16_t* __restrict__ gplane, const int* __restrict__ splane, const float* __restrict__ rvplane,
               const uint8_t* __restrict__ L, const uint8_t* __restrict__ R, int H, int W, int C, int D, int ld,
               float tau, float* __restrict__ out, float* __restrict__ out_r)
{
    extern __shared__ int smem_i[];
    cost_tile<MODE, float>(gplane, splane, rvplane, L, R, H, W, C, D, ld, tau, out, blockIdx.x * kXS, blockIdx.y,
                                  smem_i, 0, D, out_r);
}

// Right volume entries with no left pixel (xr + d >= W): the maximum cost;
// d in [D, ld) padding: 0.
__global__ void right_edge_fill_kernel(int H, int W, int D, int ld, float maxc, float* __restrict__ out_r)
{
    const int y = blockIdx.x;
    const int x_first = max(0, W - D);
    const int n = (W - x_first) * ld;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int xr = x_first + i / ld, d = i % ld;
        if (d >= D) out_r[((size_t)y * W + xr) * ld + d] = 0.f;
        else if (xr + d >= W) out_r[((size_t)y * W + xr) * ld + d] = maxc;
    }
}

// ---- TAD, 16-bit x-blocked volume: one thread per (block of 8 columns, 8 disparities)
//
// The layout [H][ceil(W/8)][Dp][8] keeps the 8 columns of a block contiguous
// for each d, so a thread that owns one block and 8 consecutive disparities
// computes the 8 x 8 costs in registers, one 16-byte row per d.  Lanes own
// consecutive disparity groups of a block; the warp passes its 256 rows
// through a private shared-memory buffer so that each store instruction
// writes 32 consecutive rows (512 contiguous bytes within a block).  The left
// pixels stay in registers, the right ones slide one column per disparity.
// Staged rows use a skewed index c + c/8, so lanes reading columns 8 apart hit
// different banks.
constexpr int kXbThreads = 256;

__device__ __forceinline__ int skew(int c) { return c + (c >> 3); }
__host__ __device__ inline int skew_len(int n) { return n + (n - 1) / 8; }

// x-blocks per CTA: 16 up to 8 disparity groups, then 8 (measured best on
// GB300 for D = 64, 128 and 256; smaller CTAs interleave their staging and
// compute phases better, and 640 columns split evenly into 16-block CTAs)
__host__ __device__ inline int xb_blocks_per_cta(int D)
{
    const int ndg = (D + 7) / 8;
    const int b = ndg <= 8 ? 16 : 8;
    return b * ndg <= kXbThreads ? b : kXbThreads / ndg;
}

// Per-warp output buffer: 256 rows of 16 bytes, row r at r + r/8 (conflict-free
// both when lanes write their 8 rows and when the warp reads 32 consecutive rows).
constexpr int kXbWarpRows = 256 + 32;

// Output rows per CTA (1, 2 or 4, chosen at launch).
constexpr int kXbMaxRows = 4;

__host__ __device__ inline size_t cost_xb_stage_ints(int D, int rows)
{
    const int npx = 8 * xb_blocks_per_cta(D);
    const int Lr = skew_len(npx + D + 9), Lp = skew_len(npx);
    // per output row the packed pixels of both images
    return ((size_t)rows * (Lp + Lr) + 3) & ~(size_t)3;   // the output buffers that follow are 16-byte aligned
}

template <typename T>
__global__ void __launch_bounds__(kXbThreads, 2)
cost_xb_tad_kernel(const uint8_t* __restrict__ L, const uint8_t* __restrict__ R, int H, int W, int C, int D, float tau,
               T* __restrict__ out, uint2* __restrict__ rgbx, int rows)
{
    extern __shared__ int sm_xb[];
    // let a programmatically launched successor (the tensor-core aggregation)
    // start its set-up once every CTA of this grid has started; it waits for
    // this grid's completion before it reads anything this kernel writes
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int ndg = (D + 7) >> 3;
    const int xbc = xb_blocks_per_cta(D);
    const int nxb = (W + 7) >> 3;
    const int xb0 = blockIdx.x * xbc;
    const int y0 = blockIdx.y * rows;
    const int nrows = min(rows, H - y0);
    const int x0 = xb0 * 8;
    const int npx = xbc * 8;
    // right columns x0-D-8 .. x0+npx (origin rb): the 8 extra columns keep every
    // index of a thread's 8 disparities >= 0 also past D (those rows are not stored)
    const int nr = npx + D + 9;
    const int rb = x0 - D - 8;
    const int Lr = skew_len(nr), Lp = skew_len(npx);

    uint32_t* pl = (uint32_t*)sm_xb;             // left pixels [rows][Lp]
    uint32_t* pr = pl + rows * Lp;               // right pixels [rows][Lr], origin rb

    // staging: the pixels of the output rows at clamped columns, and the left
    // image's packed guide
    auto colour = [&](const uint8_t* img, int yy, int x) -> uint32_t {
        const uint8_t* q = img + ((size_t)yy * W + clampi(x, 0, W - 1)) * C;
        return C == 3 ? (uint32_t)q[0] | ((uint32_t)q[1] << 8) | ((uint32_t)q[2] << 16) : (uint32_t)q[0];
    };
    for (int e = tid; e < nrows * npx; e += nthr) {
        const int k = e / npx, c = e - k * npx;
        const uint32_t col = colour(L, y0 + k, x0 + c);
        pl[k * Lp + skew(c)] = col;
        if (x0 + c < W)
            rgbx[(size_t)(y0 + k) * rgbx_pitch(W) + x0 + c] = make_uint2(col, (uint32_t)__dp4a(col, col, 0u));
    }
    for (int e = tid; e < nrows * nr; e += nthr) {
        const int k = e / nr, c = e - k * nr;
        pr[k * Lr + skew(c)] = colour(R, y0 + k, rb + c);
    }
    __syncthreads();

    const int dg = tid % ndg, xbl = tid / ndg;
    const int xb = xb0 + xbl;
    // threads past xbc * ndg (the block is a whole number of warps) and blocks
    // beyond the image compute nothing and store nothing
    const bool active = xbl < xbc && xb < nxb;
    const int d0 = 8 * dg;
    const int xl = 8 * xbl;            // the block's first pixel, relative to x0
    const int xbase = x0 + xl;
    const int lane = tid & 31;
    uint4* wbuf = (uint4*)(sm_xb + cost_xb_stage_ints(D, rows)) + (size_t)(tid >> 5) * kXbWarpRows;
    uint4* mine = wbuf + 9 * lane;     // rows 8*lane + s at 9*lane + s

    for (int k = 0; k < nrows; ++k) {
        const int y = y0 + k;
        const uint32_t* plk = pl + k * Lp;
        const uint32_t* prk = pr + k * Lr;
        if (active) {
            const float inv_c = 1.f / (float)C;
            uint32_t pli[8], prw[8];
    #pragma unroll
            for (int i = 0; i < 8; ++i) pli[i] = plk[skew(xl + i)];
            // right pixel of (x, d): index (x - d) - rb
            int base = xl - d0 + D + 8;
    #pragma unroll
            for (int i = 0; i < 8; ++i) prw[i] = prk[skew(base + i)];
    #pragma unroll
            for (int s = 0; s < 8; ++s) {
                const int d = d0 + s;
                if (s > 0) {
                    --base;
    #pragma unroll
                    for (int i = 7; i > 0; --i) prw[i] = prw[i - 1];
                    prw[0] = prk[skew(base)];
                }
                T v[8];
    #pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int x = xbase + i;
                    const int sad = (int)__dp4a(__vabsdiffu4(pli[i], prw[i]), 0x01010101u, 0u);
                    const float cst = x - d < 0 ? tau : fminf((float)sad * inv_c, tau);
                    v[i] = to_out<T>(x < W ? cst : 0.f);
                }
                mine[s] = pack8(v);
            }
        }
        // write-out: entry e = 32k + lane is row s = e % 8 of lane e / 8 (its block
        // xbl and group dg come by shuffle); rows d >= D and inactive lanes are skipped
        __syncwarp();
        const int Dp = tc_block_rows(D);
        const int code = active ? (xbl << 8) | dg : -1;
    #pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int e = 32 * k + lane;
            const int src = __shfl_sync(0xffffffffu, code, e >> 3);
            const int s = e & 7;
            if (src >= 0 && 8 * (src & 255) + s < D) {
                const int xbs = xb0 + (src >> 8);
                const uint4 row = wbuf[e + (e >> 3)];
                *(uint4*)(out + (((size_t)y * nxb + xbs) * Dp + 8 * (src & 255) + s) * 8) = row;
            }
        }
        // rows D .. Dp-1 of the CTA's blocks: zero, except row round_up(D,16) all
        // ones when the normaliser rides with the volume
        const int extra = Dp - D;
        if (extra > 0) {
            const int n16 = (D + 15) / 16 * 16;
            const T one1[2] = {to_out<T>(1.f), to_out<T>(1.f)};
            const uint32_t ones = *reinterpret_cast<const uint32_t*>(one1);
            const int nb = min(xbc, nxb - xb0);
            for (int i = tid; i < nb * extra; i += nthr) {
                const int b = i / extra, d = D + (i - b * extra);
                const uint32_t v = (d == n16 && Dp > n16) ? ones : 0u;
                *(uint4*)(out + (((size_t)y * nxb + xb0 + b) * Dp + d) * 8) = make_uint4(v, v, v, v);
            }
        }
        __syncwarp();   // the warp's buffer is read out before the next row's sweep refills it
    }
}

// ---- NCC, 16-bit x-blocked volume ----------------------------------------------
// A CTA covers 64 pixels x 4 rows and every disparity.  All of Eq. (1) runs in
// FP32 on exact integers: with the grey values moved by a constant a
// (which changes neither 9 P - S_l S_r nor the variances) |g - a| <= 383, so
// every product, block sum, 9 P' and S_l' S_r' is an integer below 2^24, and
// 9 P' - S_l' S_r' comes out of one FMA rounded once -- the integer converted to
// float.  A thread computes two output rows y, y + 1 at once: with p_j the
// products of grey rows y-1 .. y+2, the column sums are p_0 + t and t + p_3,
// t = p_1 + p_2 (4 FMAs for two sums), and everything after them is packed, one
// row per half.
//   * Staging: per column and pair of output rows a float4 of the four grey rows
//     y-1 .. y+2, then per block centre a float4 (S(y), S(y+1), 1/sqrt V(y),
//     1/sqrt V(y+1)).  Index c + c/4: lanes 4 columns apart read 16 bytes each
//     without conflicts.
//   * A lane owns 4 pixels x 2 rows (lanes 0-15: the 64 pixels of rows y0, y0+1;
//     16-31: of the next two) and 16 disparities of its warp: the left window
//     (6 columns x 4 rows) stays in registers, the right one slides one column
//     (2 shared loads) per disparity.  Per pair of costs: 6 FMAs and 1.75 packed
//     additions for the block sum P', 3 packed operations for the normalisation.
//   * Lanes 2i, 2i + 1 hold the two halves of a block of 8 pixels: they exchange
//     a row each, so that a lane has 16 bytes (8 pixels) of its row per
//     disparity, and stage them in the warp's buffer; one TMA store per pair of
//     rows writes 8 blocks x 16 disparities.  (Direct stores of 32 bytes per
//     lane, each in a line of its own, kept the load/store pipe 76% busy:
//     123 us at 1280x960, D = 128.)
// Bound: instruction issue of the sweep (11.5 instructions per cost with the
// staging; the integer form it replaces took 30), then the volume's writes to HBM.
// CTAs of 4 warps (four per SM) overlap one another's staging best: 1920x1080,
// D = 256: 316 us against 334 us with 8 warps, 345 us with 8 warps and 8 rows
// (before the column sums went from packed to scalar FMAs).
// Measured on GB300 (CUDA events), BF16, before -> now: 640x480, D = 64: 35.5 ->
// 19.8 us; 1280x960, D = 128: 188 -> 89.5 us; 1920x1080, D = 256: 557 -> 274 us
// (1.13 GB written: 4.1 TB/s).
constexpr int kNccPx = 64;
constexpr int kNccWarps = 4;
constexpr int kNccRows = 4;      // two pairs

__host__ __device__ inline int skew4(int c) { return c + (c >> 2); }
__host__ __device__ inline int ncc_groups(int D) { return (D + 15) / 16; }          // of 16 disparities
__host__ __device__ inline int ncc_right_cols(int D) { return 16 * ncc_groups(D) + kNccPx + 1; }
// float4 entries of the four staged arrays, per pair of rows
__host__ __device__ inline int ncc_left_len() { return skew4(kNccPx + 2); }
__host__ __device__ inline int ncc_right_len(int D) { return skew4(ncc_right_cols(D)) + 1; }
// Store buffer of a warp: two pairs of rows, each [d / 8][block][row][8 d x 8
// pixels] (128-byte lines, TMA's 128-byte swizzle) of 16 disparities and 8 blocks.
constexpr int kNccPairBytes = 2 * 8 * 2 * 128, kNccWarpBytes = 2 * kNccPairBytes;
__host__ __device__ inline size_t ncc_smem_bytes(int D)
{
    return 1024 + (size_t)kNccWarps * kNccWarpBytes + (size_t)2 * 16 * 2 * (ncc_left_len() + ncc_right_len(D));
}

template <bool BF16>
__global__ void __launch_bounds__(32 * kNccWarps, 4)
cost_xb_ncc_kernel(const __grid_constant__ CUtensorMap out_map, const uint8_t* __restrict__ L,
                   const uint8_t* __restrict__ R, int H, int W, int C, int D, uint2* __restrict__ rgbx)
{
    extern __shared__ uint8_t sm_ncc[];
    // let a programmatically launched successor (the tensor-core aggregation)
    // start its set-up once every CTA of this grid has started; it waits for
    // this grid's completion before it reads anything this kernel writes
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int ROWS = kNccRows, PAIRS = ROWS / 2, nthr = 32 * kNccWarps;
    const int tid = threadIdx.x, lane = tid & 31;
    const int x0 = blockIdx.x * kNccPx, y0 = blockIdx.y * ROWS;
    const int ng = ncc_groups(D), nr = ncc_right_cols(D);
    const int rb = x0 - 16 * ng;             // image column of right column 0
    const int LL = ncc_left_len(), RL = ncc_right_len(D);
    uint8_t* const buffers = sm_ncc + ((1024u - (tc::smem_u32(sm_ncc) & 1023u)) & 1023u);
    float4* const gl = (float4*)(buffers + kNccWarps * kNccWarpBytes);   // [PAIRS][LL]: columns x0 - 1 ..
    float4* const sl = gl + PAIRS * LL;      // [PAIRS][LL]: centres x0 ..
    float4* const gr = sl + PAIRS * LL;      // [PAIRS][RL]: columns rb ..
    float4* const sr = gr + PAIRS * RL;      // [PAIRS][RL]: centres rb ..

    // ---- grey rows y0-1 .. y0+ROWS of both images at clamped columns, and the
    // left image's packed guide
    const int shift = C == 3 ? 382 : 128;
    for (int e = tid; e < kNccPx + 2 + nr; e += nthr) {
        const bool left = e < kNccPx + 2;
        const int c = left ? e : e - (kNccPx + 2);
        const int xs = left ? x0 - 1 + c : rb + c;
        const uint8_t* img = (left ? L : R) + (size_t)clampi(xs, 0, W - 1) * C;
        uint32_t col[ROWS + 2];
#pragma unroll
        for (int j = 0; j < ROWS + 2; ++j) {
            const uint8_t* q = img + (uint32_t)(clampi(y0 - 1 + j, 0, H - 1) * W) * (uint32_t)C;
            col[j] = C == 3 ? (uint32_t)q[0] | ((uint32_t)q[1] << 8) | ((uint32_t)q[2] << 16) : (uint32_t)q[0];
        }
        float4* dst = (left ? gl : gr) + skew4(c);
        float g[ROWS + 2];
#pragma unroll
        for (int j = 0; j < ROWS + 2; ++j) g[j] = (float)((int)__dp4a(col[j], 0x01010101u, 0u) - shift);
#pragma unroll
        for (int k = 0; k < PAIRS; ++k)
            dst[k * (left ? LL : RL)] = make_float4(g[2 * k], g[2 * k + 1], g[2 * k + 2], g[2 * k + 3]);
        if (left && c >= 1 && c <= kNccPx && xs < W) {
            uint2* o = rgbx + (size_t)y0 * rgbx_pitch(W) + xs;
#pragma unroll
            for (int j = 1; j <= ROWS; ++j)
                if (y0 + j - 1 < H)
                    o[(size_t)(j - 1) * rgbx_pitch(W)] = make_uint2(col[j], (uint32_t)__dp4a(col[j], col[j], 0u));
        }
    }
    __syncthreads();
    // ---- block statistics of every centre (all exact up to the reciprocal square root)
    const int ncl = kNccPx, ncr = nr - 2;    // right centres rb + 1 .. rb + nr - 2
    for (int q = tid; q < ncl + ncr; q += nthr) {
        const bool left = q < ncl;
        const int cc = left ? q + 1 : q - ncl + 1;   // the centre's column in the grey array
        const float4* g = (left ? gl : gr);
        const int i0 = skew4(cc - 1), i1 = skew4(cc), i2 = skew4(cc + 1), len = left ? LL : RL;
        float4* dst = left ? sl + skew4(q) : sr + i1;
#pragma unroll
        for (int k = 0; k < PAIRS; ++k, g += len, dst += len) {
            const float4 v3[3] = {g[i0], g[i1], g[i2]};
            float s0 = 0.f, s1 = 0.f, q0 = 0.f, q1 = 0.f;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float4 v = v3[j];
                const float m = v.y + v.z, mq = fmaf(v.y, v.y, v.z * v.z);
                s0 += m + v.x;
                s1 += m + v.w;
                q0 += fmaf(v.x, v.x, mq);
                q1 += fmaf(v.w, v.w, mq);
            }
            const float a0 = fmaf(9.f, q0, -(s0 * s0)), a1 = fmaf(9.f, q1, -(s1 * s1));
            *dst = make_float4(s0, s1, a0 > 0.f ? rsqrtf(a0) : 0.f, a1 > 0.f ? rsqrtf(a1) : 0.f);
        }
    }
    __syncthreads();

    const int p = lane & 15, odd = lane & 1;
    const int xl = 4 * p, xbase = x0 + xl;
    // the lane's line of its pair's buffer, (block, row) = (p / 2, odd): chunk s of
    // 8 disparities sits at chunk s ^ (line % 8)
    const int line = 2 * (p >> 1) + odd;
    const uint32_t buf = tc::smem_u32(buffers) + (tid >> 5) * kNccWarpBytes;
    const uint32_t chunk0 = buf + (lane >> 4) * kNccPairBytes + line * 128 + (line & 7) * 16;
    auto put = [&](int s, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"((chunk0 ^ ((s & 7) * 16)) + (s >> 3) * (8 * 2 * 128)),
                     "r"(a), "r"(b), "r"(c), "r"(d)
                     : "memory");
    };

    const int rp = lane >> 4;
    for (int grp = tid >> 5; grp <= ng; grp += kNccWarps) {
        // the warp's previous stores have read its buffer
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
        auto store = [&]() {
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (y0 + 2 * h < H)
                        asm volatile(
                            "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(
                                (uint64_t)&out_map),
                            "r"(0), "r"(y0 + 2 * h), "r"(x0 >> 3), "r"(2 * grp), "r"(buf + h * kNccPairBytes)
                            : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        };
        if (grp == ng) {
            // the 16 rows after the costs: one of ones (the normaliser), then zeros
            const uint32_t one = BF16 ? 0x3F803F80u : 0x3C003C00u;
#pragma unroll
            for (int s = 0; s < 16; ++s) put(s, s == 0 ? one : 0u, s == 0 ? one : 0u, s == 0 ? one : 0u, s == 0 ? one : 0u);
            store();
            continue;
        }

        // left window and statistics
        const float4* glw = gl + rp * LL + skew4(xl);
        const float4* slw = sl + rp * LL + skew4(xl);
        float4 lw[6];
        uint64_t sli[4], rli[4];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            // -9 g: the block sums come out as -9 P' (the products stay below 2^24 / 9)
            const float4 v = glw[j + (j >> 2)];
            lw[j] = make_float4(-9.f * v.x, -9.f * v.y, -9.f * v.z, -9.f * v.w);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 v = slw[i];
            sli[i] = f2_pack(v.x, v.y);
            rli[i] = f2_pack(v.z, v.w);
        }
        const uint64_t one2 = f2_pack(1.f, 1.f);

        const int d0 = 16 * grp;
        // right column of (x, d), window offset k: x - d + k - rb = base + (i + k - s)
        const int base = xl + 16 * ng - d0;
        const float4* grw = gr + rp * RL + skew4(base);
        const float4* srw = sr + rp * RL + skew4(base);
        auto at = [](int m) { return m + (m >> 2); };   // offset of column base + m (base is a multiple of 4)
        float4 rw[6];
        uint64_t sri[4], rri[4];
#pragma unroll
        for (int j = 0; j < 6; ++j) rw[j] = grw[at(j - 1)];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 v = srw[at(i)];
            sri[i] = f2_pack(v.x, v.y);
            rri[i] = f2_pack(v.z, v.w);
        }
        // lanes whose 4 pixels are inside the image and match inside it for all 16
        // disparities of the range skip the masks
        auto sweep = [&](auto masked) {
#pragma unroll
            for (int s = 0; s < 16; ++s) {
                const int d = d0 + s;
                if (s > 0) {
                    // d grew by one: the window slides one column to the left
#pragma unroll
                    for (int j = 5; j > 0; --j) rw[j] = rw[j - 1];
                    rw[0] = grw[at(-1 - s)];
#pragma unroll
                    for (int i = 3; i > 0; --i) {
                        sri[i] = sri[i - 1];
                        rri[i] = rri[i - 1];
                    }
                    const float4 v = srw[at(-s)];
                    sri[0] = f2_pack(v.x, v.y);
                    rri[0] = f2_pack(v.z, v.w);
                }
                uint64_t cs[6];
#pragma unroll
                for (int j = 0; j < 6; ++j) {
                    const float t = fmaf(lw[j].y, rw[j].y, lw[j].z * rw[j].z);
                    cs[j] = f2_pack(fmaf(lw[j].x, rw[j].x, t), fmaf(lw[j].w, rw[j].w, t));
                }
                const uint64_t a0 = f2_add(cs[0], cs[1]), a1 = f2_add(cs[2], cs[3]), a2 = f2_add(cs[4], cs[5]);
                const uint64_t P[4] = {f2_add(a0, cs[2]), f2_add(cs[1], a1), f2_add(a1, cs[4]), f2_add(cs[3], a2)};
                float c0[4], c1[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    // S_l' S_r' - 9 P' rounded once, times the rounded product of the normalisers, plus 1
                    const uint64_t nn = f2_fma(sli[i], sri[i], P[i]);
                    f2_unpack(f2_fma(nn, f2_mul(rli[i], rri[i]), one2), c0[i], c1[i]);
                    if (decltype(masked)::value) {
                        const int x = xbase + i;
                        if (x - d < 0) c0[i] = c1[i] = 2.f;
                        if (x >= W || d >= D) c0[i] = c1[i] = 0.f;
                    }
                }
                const uint32_t w0 = pack_16x2<BF16>(c0[0], c0[1]), w1 = pack_16x2<BF16>(c0[2], c0[3]);
                const uint32_t v0 = pack_16x2<BF16>(c1[0], c1[1]), v1 = pack_16x2<BF16>(c1[2], c1[3]);
                const uint32_t e0 = __shfl_xor_sync(0xffffffffu, odd ? w0 : v0, 1);
                const uint32_t e1 = __shfl_xor_sync(0xffffffffu, odd ? w1 : v1, 1);
                const uint32_t o0 = odd ? e0 : w0, o1 = odd ? e1 : w1, o2 = odd ? v0 : e0, o3 = odd ? v1 : e1;
                put(s, o0, o1, o2, o3);
            }
        };
        const bool inside = xbase + 3 < W && xbase >= d0 + 15 && d0 + 16 <= D;
        if (__all_sync(0xffffffffu, inside))
            sweep(std::integral_constant<bool, false>{});
        else
            sweep(std::integral_constant<bool, true>{});
        store();
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

template <bool BF16>
cudaError_t launch_cost_xb_ncc(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W, int C,
                               int D, void* out, cudaStream_t stream)
{
    // the volume as (8 disparities x 8 columns = 128 contiguous bytes, image row, block, d / 8)
    const tca::EncodeTiledFn enc = tca::encode_fn();
    if (!enc) return cudaErrorNotSupported;
    const int nxb = (W + 7) / 8, Dp = tc_block_rows(D);
    cuuint64_t dims[4] = {64, (cuuint64_t)H, (cuuint64_t)nxb, (cuuint64_t)(Dp / 8)};
    cuuint64_t strides[3] = {(cuuint64_t)nxb * Dp * 16, (cuuint64_t)Dp * 16, 128};
    cuuint32_t box[4] = {64, 2, kNccPx / 8, 2};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUtensorMap map;
    if (enc(&map, BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, out, dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    const size_t smem = ncc_smem_bytes(D);
    cudaError_t e = fbs::raise_smem_limit(cost_xb_ncc_kernel<BF16>, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((W + kNccPx - 1) / kNccPx, (H + kNccRows - 1) / kNccRows);
    fbs::note_launch();
    cost_xb_ncc_kernel<BF16><<<grid, 32 * kNccWarps, smem, stream>>>(map, left, right, H, W, C, D, sc.rgbx);
    return cudaGetLastError();
}

size_t cost_xb_tad_smem_bytes(int D, int rows)
{
    const int nwarps = (xb_blocks_per_cta(D) * ((D + 7) / 8) + 31) / 32;
    return sizeof(int) * cost_xb_stage_ints(D, rows) + (size_t)nwarps * kXbWarpRows * 16;
}

template <typename T>
cudaError_t launch_cost_xb_tad(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W, int C,
                           int D, float tau, T* out, cudaStream_t stream)
{
    const int ndg = (D + 7) / 8;
    const int xbc = xb_blocks_per_cta(D);
    const int nxb = (W + 7) / 8;
    const int gx = (nxb + xbc - 1) / xbc;
    // the most rows per CTA that still leave about four CTAs per SM (small
    // images need the CTAs more than the shared staging)
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    int rows = kXbMaxRows;
    while (rows > 1 && (long long)gx * ((H + rows - 1) / rows) < 4LL * sms) rows /= 2;
    const size_t smem = cost_xb_tad_smem_bytes(D, rows);
    e = fbs::raise_smem_limit(cost_xb_tad_kernel<T>, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid(gx, (H + rows - 1) / rows);
    fbs::note_launch();
    const int nthr = (xbc * ndg + 31) / 32 * 32;   // whole warps (the write-out shuffles need all lanes)
    cost_xb_tad_kernel<T><<<grid, nthr, smem, stream>>>(left, right, H, W, C, D, tau, out, sc.rgbx, rows);
    return cudaGetLastError();
}

size_t cost_smem_bytes()
{
    return sizeof(float) * (size_t)kDC * kStage +
           sizeof(int) * (size_t)(3 * (kXS + 2) + 3 * 4 * kQR + 2 * kXS + 2 * (kXS + kDC));
}

template <int MODE, typename T>
cudaError_t launch_cost_kernel(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W,
                               int C, int D, int ld, float tau, T* out, cudaStream_t stream)
{
    const size_t smem = cost_smem_bytes();
    cudaError_t e = fbs::raise_smem_limit(cost_kernel<MODE, T>, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((W + kXS - 1) / kXS, H);
    fbs::note_launch();
    cost_kernel<MODE, T><<<grid, kThreads, smem, stream>>>(sc.g, sc.s, sc.rv, left, right, H, W, C, D, ld,
                                                                   tau, out);
    return cudaGetLastError();
}

cudaError_t launch_stats(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W, int C,
                         cudaStream_t stream)
{
    dim3 grid((W + 255) / 256, H, 2);
    fbs::note_launch();
    grey_stats_kernel<<<grid, 256, 0, stream>>>(left, right, H, W, C, sc.g, sc.s, sc.rv, sc.rgbx);
    return cudaGetLastError();
}

}  // namespace

int stats_items(int H, int W) { return H; }
int cost_items(int H, int W) { return H * ((W + kXS - 1) / kXS); }
size_t cost_kernel_smem() { return cost_smem_bytes(); }

cudaError_t prepare_cost_batched()
{
    return fbs::raise_smem_limit(cost_batched_kernel, (int)cost_smem_bytes());
}

cudaError_t launch_stats_batched(const BatchPair* pairs, int npairs, int nitems, int* counter, int grid,
                                 cudaStream_t stream)
{
    fbs::note_launch();
    grey_stats_batched_kernel<<<grid, 256, 0, stream>>>(pairs, npairs, nitems, counter);
    return cudaGetLastError();
}

cudaError_t launch_cost_batched(const BatchPair* pairs, int npairs, int nitems, int* counter, int grid,
                                cudaStream_t stream)
{
    fbs::note_launch();
    cost_batched_kernel<<<grid, kThreads, cost_smem_bytes(), stream>>>(pairs, npairs, nitems, counter);
    return cudaGetLastError();
}

size_t cost_scratch_bytes(int H, int W)
{
    const size_t n = (size_t)2 * H * W;
    return ((n * sizeof(int16_t) + 255) & ~(size_t)255) + ((n * sizeof(int) + 255) & ~(size_t)255) +
           ((n * sizeof(float) + 255) & ~(size_t)255);
}

size_t rgbx_bytes(int H, int W) { return ((size_t)H * rgbx_pitch(W) * 8 + 255) & ~(size_t)255; }

__global__ void pack_rgbx_kernel(const uint8_t* __restrict__ img, int H, int W, int C, uint2* __restrict__ out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= W) return;
    const uint8_t* p = img + ((size_t)y * W + x) * C;
    const uint32_t c = C == 3 ? (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) : (uint32_t)p[0];
    out[(size_t)y * rgbx_pitch(W) + x] = make_uint2(c, (uint32_t)__dp4a(c, c, 0u));
}

cudaError_t launch_pack_rgbx(const uint8_t* img, int H, int W, int C, uint2* rgbx, cudaStream_t stream)
{
    dim3 grid((W + 255) / 256, H);
    fbs::note_launch();
    pack_rgbx_kernel<<<grid, 256, 0, stream>>>(img, H, W, C, rgbx);
    return cudaGetLastError();
}

CostScratch carve_cost_scratch(void* base, int H, int W)
{
    const size_t n = (size_t)2 * H * W;
    CostScratch sc;
    sc.rgbx = nullptr;
    uint8_t* p = (uint8_t*)base;
    sc.g = (int16_t*)p;
    p += (n * sizeof(int16_t) + 255) & ~(size_t)255;
    sc.s = (int*)p;
    p += (n * sizeof(int) + 255) & ~(size_t)255;
    sc.rv = (float*)p;
    return sc;
}

cudaError_t launch_cost_build(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W,
                              int C, int D, int ld, int mode, float tau, float* cost, cudaStream_t stream)
{
    if (mode == 0) {
        cudaError_t e = launch_stats(sc, left, right, H, W, C, stream);
        if (e != cudaSuccess) return e;
        return launch_cost_kernel<0, float>(sc, left, right, H, W, C, D, ld, tau, cost, stream);
    }
    return launch_cost_kernel<1, float>(sc, left, right, H, W, C, D, ld, tau, cost, stream);
}

cudaError_t launch_cost_band(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W,
                             int C, int D, int ld, int radius, const int2* tile_range, float* cost, cudaStream_t stream)
{
    cudaError_t e = launch_stats(sc, left, right, H, W, C, stream);
    if (e != cudaSuccess) return e;
    const size_t smem = cost_smem_bytes();
    e = fbs::raise_smem_limit(cost_band_kernel, (int)smem);
    if (e != cudaSuccess) return e;
    const int ntx = (W + kAggTileX - 1) / kAggTileX, nty = (H + kAggTileY - 1) / kAggTileY;
    dim3 grid((W + kXS - 1) / kXS, H);
    fbs::note_launch();
    cost_band_kernel<<<grid, kThreads, smem, stream>>>(sc.g, sc.s, sc.rv, H, W, D, ld, radius, tile_range, ntx, nty,
                                                       cost);
    return cudaGetLastError();
}

cudaError_t launch_cost_build_lr(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W,
                                 int C, int D, int ld, int mode, float tau, float* cost, float* cost_r,
                                 cudaStream_t stream)
{
    cudaError_t e = cudaSuccess;
    if (mode == 0) e = launch_stats(sc, left, right, H, W, C, stream);
    if (e != cudaSuccess) return e;
    const size_t smem = cost_smem_bytes();
    dim3 grid((W + kXS - 1) / kXS, H);
    if (mode == 0) {
        e = fbs::raise_smem_limit(cost_lr_kernel<0>, (int)smem);
        fbs::note_launch();
        if (e == cudaSuccess)
            cost_lr_kernel<0><<<grid, kThreads, smem, stream>>>(sc.g, sc.s, sc.rv, left, right, H, W, C, D, ld, tau,
                                                                cost, cost_r);
    } else {
        e = fbs::raise_smem_limit(cost_lr_kernel<1>, (int)smem);
        fbs::note_launch();
        if (e == cudaSuccess)
            cost_lr_kernel<1><<<grid, kThreads, smem, stream>>>(sc.g, sc.s, sc.rv, left, right, H, W, C, D, ld, tau,
                                                                cost, cost_r);
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    fbs::note_launch();
    right_edge_fill_kernel<<<H, 256, 0, stream>>>(H, W, D, ld, mode == 0 ? 2.f : tau, cost_r);
    return cudaGetLastError();
}

cudaError_t launch_cost_build_xblock16(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H,
                                       int W, int C, int D, int mode, float tau, bool bf16, void* cost,
                                       cudaStream_t stream)
{
    // one launch: statistics, costs, pad rows and the packed guide (sc.rgbx)
    if (D > 256 || !sc.rgbx) return cudaErrorInvalidValue;   // serves the tensor-core form only
    if (mode == 0)
        return bf16 ? launch_cost_xb_ncc<true>(sc, left, right, H, W, C, D, cost, stream)
                    : launch_cost_xb_ncc<false>(sc, left, right, H, W, C, D, cost, stream);
    return bf16 ? launch_cost_xb_tad(sc, left, right, H, W, C, D, tau, (__nv_bfloat16*)cost, stream)
                : launch_cost_xb_tad(sc, left, right, H, W, C, D, tau, (__half*)cost, stream);
}

}  // namespace fbs
