// Step 1 of fast bilateral stereo: the matching-cost volume.
//
// NCC (Sec. II-A, Eq. (1)-(3), varrho = 1): with the intensity g taken as the
// channel sum, n = 9 and the block sums S = sum g, Q = sum g^2 and
// P = sum g_l g_r, Eq. (1) multiplied through by n^2 reads
//     c = (n P - S_l S_r) / sqrt((n Q_l - S_l^2) (n Q_r - S_r^2)).
// Every sum and both numerator terms are exact integers (grey_shift), so only the
// final normalisation is rounded.  Stored cost: C = 1 - c.  Boundary rules:
// blocks clamp to the image; u - d < 0 gives the maximum cost 2; a block of
// zero variance gives c = 0.
//
// As in the paper (Sec. II-A, Sec. III) the per-pixel block statistics are
// computed once per pixel, so the per-(p, d) work is the dot product P.  Two
// kernels write the two layouts:
//   * cost_kernel, [H][W][ld] float32 (D innermost; the FP32 aggregation),
//     padding d in [D, ld) written as 0.  A pre-pass (grey_stats_kernel) fills
//     planes of the shifted grey value, its block sum and 1/sqrt(nQ - S^2).
//   * cost_xb_ncc_kernel, 16-bit x-blocked [H][ceil(W/8)][Dp][8] (the tensor-core
//     aggregation): for a row y and a block of 8 columns, the Dp x 8 block is
//     contiguous, so the tensor-core kernel's TMA reads contiguous blocks that
//     land as K-major core matrices; columns x >= W of the last block are 0.
//     One launch computes the statistics of the rows it stages, the costs, the
//     pad rows D .. Dp-1 and the left image's packed guide (its comment says how);
//     cost_xb_tad_kernel does the same for TAD.
// Both round the normalisation the same way (ncc_cost2), so the 16-bit volume
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

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// Grey values are moved by this constant: 9 P - S_l S_r and the variances do not
// change, and with |g - a| <= 383 every product, block sum, 9 P' and S_l' S_r'
// is an integer below 2^24, exact in FP32.
__host__ __device__ inline int grey_shift(int C) { return C == 3 ? 382 : 128; }

// ---- statistics pre-pass of the FP32 layout (Sec. II-A, Sec. III) ----------------
// Per pixel and image: g' = channel sum - shift, S' = 3x3 sum of g' (clamped),
// rv = 1 / sqrt(9 Q - S^2) or 0 for a flat block.  A CTA stages the grey values of
// 128 x 8 pixels and their border once; a thread owns a column and carries the
// row sums of three rows.
constexpr int kStatX = 128, kStatY = 8;

__device__ __forceinline__ void stats_tile(const uint8_t* __restrict__ src, int H, int W, int C, int x0, int y0,
                                           int16_t* __restrict__ g_out, float* __restrict__ s_out,
                                           float* __restrict__ rv_out, float (*g)[kStatX + 2])
{
    const int shift = grey_shift(C);
    for (int c = threadIdx.x; c < kStatX + 2; c += kStatX) {
        const uint8_t* p = src + (size_t)clampi(x0 - 1 + c, 0, W - 1) * C;
#pragma unroll
        for (int j = 0; j < kStatY + 2; ++j) {
            const uint8_t* q = p + (size_t)clampi(y0 - 1 + j, 0, H - 1) * W * C;
            g[j][c] = (float)((C == 3 ? (int)q[0] + (int)q[1] + (int)q[2] : (int)q[0]) - shift);
        }
    }
    __syncthreads();
    const int c = threadIdx.x, x = x0 + c;
    if (x < W) {
        float h0 = 0.f, h1 = 0.f, q0 = 0.f, q1 = 0.f;
#pragma unroll
        for (int j = 0; j < kStatY + 2; ++j) {
            const float a = g[j][c], b = g[j][c + 1], d = g[j][c + 2];
            const float h = a + b + d, q = fmaf(a, a, fmaf(b, b, d * d));
            const int y = y0 + j - 2;
            if (j >= 2 && y < H) {
                const float s = h0 + h1 + h, v = fmaf(9.f, q0 + q1 + q, -(s * s));
                const size_t o = (size_t)y * W + x;
                g_out[o] = (int16_t)g[j - 1][c + 1];
                s_out[o] = s;
                rv_out[o] = v > 0.f ? rsqrtf(v) : 0.f;
            }
            h0 = h1, h1 = h;
            q0 = q1, q1 = q;
        }
    }
}

__global__ void __launch_bounds__(kStatX)
grey_stats_kernel(const uint8_t* __restrict__ L, const uint8_t* __restrict__ R, int H, int W, int C, CostScratch sc)
{
    __shared__ float g[kStatY + 2][kStatX + 2];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t o = blockIdx.z * (size_t)H * W;
    stats_tile(blockIdx.z == 0 ? L : R, H, W, C, blockIdx.x * kStatX, blockIdx.y * kStatY, sc.g + o, sc.s + o, sc.rv + o, g);
}

// Batched statistics: an item is one 128 x 8 tile of one pair (both images).
__global__ void __launch_bounds__(kStatX)
grey_stats_batched_kernel(const BatchPair* __restrict__ pairs, int npairs, int nitems, int* __restrict__ counter)
{
    __shared__ float g[kStatY + 2][kStatX + 2];
    __shared__ int item_s;
    for (;;) {
        if (threadIdx.x == 0) item_s = atomicAdd(counter, 1);
        __syncthreads();
        const int item = item_s;
        __syncthreads();
        if (item >= nitems) break;
        const BatchPair& bp = pairs[find_pair(pairs, npairs, item, &BatchPair::stat_off)];
        if (bp.mode != 0) continue;   // TAD needs no statistics
        const int t = item - bp.stat_off, nx = (bp.W + kStatX - 1) / kStatX;
        for (int img = 0; img < 2; ++img) {
            const size_t o = img * (size_t)bp.H * bp.W;
            stats_tile(img == 0 ? bp.left : bp.right, bp.H, bp.W, bp.C, (t % nx) * kStatX, (t / nx) * kStatY, bp.sc.g + o,
                       bp.sc.s + o, bp.sc.rv + o, g);
            __syncthreads();
        }
    }
}

template <typename T>
__device__ __forceinline__ T to_out(float v);
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

// Index of column c in a staged row of 16-byte entries: lanes 4 columns apart
// read 16 bytes each without conflicts.
__host__ __device__ inline int skew4(int c) { return c + (c >> 2); }

// The block sums of two output rows y, y + 1 for 4 pixels: lw, rw are 6 columns of
// the two windows, each the grey rows y-1 .. y+2.  With p_j the products of a
// column's rows, its sums are p_0 + t and t + p_3, t = p_1 + p_2.
__device__ __forceinline__ void block_sums(const float4 (&lw)[6], const float4 (&rw)[6], uint64_t (&P)[4])
{
    uint64_t cs[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const float t = fmaf(lw[j].y, rw[j].y, lw[j].z * rw[j].z);
        cs[j] = f2_pack(fmaf(lw[j].x, rw[j].x, t), fmaf(lw[j].w, rw[j].w, t));
    }
    const uint64_t a0 = f2_add(cs[0], cs[1]), a1 = f2_add(cs[2], cs[3]), a2 = f2_add(cs[4], cs[5]);
    P[0] = f2_add(a0, cs[2]);
    P[1] = f2_add(cs[1], a1);
    P[2] = f2_add(a1, cs[4]);
    P[3] = f2_add(cs[3], a2);
}

// The costs C = 1 - c of two rows from -9 P' (minus9p), S' and rv of both blocks:
// S_l' S_r' - 9 P' rounded once, times the rounded product of the normalisers,
// plus 1 (every cost kernel uses this, so the FP32 and the 16-bit volumes hold
// the same values before the 16-bit rounding).
__device__ __forceinline__ uint64_t ncc_cost2(uint64_t minus9p, uint64_t sl, uint64_t sr, uint64_t rl, uint64_t rr,
                                              uint64_t one2)
{
    return f2_fma(f2_fma(sl, sr, minus9p), f2_mul(rl, rr), one2);
}

// ---- FP32 volume [H][W][ld], D innermost ------------------------------------------
// A CTA (4 warps) covers 64 pixels x 4 rows of one view and disparities
// [d_begin, d_end), up to 128 per staging of the other image and 32 per step; a
// warp takes 8 of them, a lane 4 pixels x 2 rows (lanes 0-15: rows y0, y0+1;
// 16-31: the next two).  The window of the view's own image (6 columns x 4 grey
// rows) stays in registers, the other image's slides one column (2 shared loads)
// per disparity; NCC as above, TAD from the packed pixels.  Costs are transposed
// through a buffer of the CTA ([row][pixel][32 d], entry XOR pixel / 4,
// conflict-free) and leave as runs of up to 128 bytes per pixel, a row per warp.
// MIRROR computes the right view: its own image is the right one, and the other
// window slides the other way (Sec. II-A, Sec. III); the two products and sums
// commute, so cost_r(x, y, d) = cost(x + d, y, d) bit for bit.
// VW: floats per store -- 4 (ld % 4 == 0, 16-byte aligned), 2 (ld even, 8-byte
// aligned) or 1.
// Bound: the load/store pipe.  A store instruction costs it a cycle per line of
// 128 bytes that it touches, so a warp that wrote its own 8 disparities of 16
// pixels (runs of 32 bytes) spent two thirds of its cycles there.  Measured on
// GB300 with the pre-pass, integer products, one row x 128 pixels per CTA and
// stores after a block-wide transposition -> runs of 32 bytes per warp -> now:
// 640x480, D = 64: 50 -> 33.5 -> 26.4 us; 1280x960, D = 128: 293 -> 177 -> 138 us;
// 1920x1080, D = 256: 906 -> 554 -> 414 us; 767x575, D = 93: 108 -> 61 -> 46 us;
// TAD 641x479, D = 71 (4-byte stores): 54 us in runs of 32 bytes, now 30.
constexpr int kCostPx = 64, kCostRows = 4, kCostWarps = 4, kCostThreads = 32 * kCostWarps;
constexpr int kCostPass = 128;                               // disparities per pass
constexpr int kCostLeft = 82;                                // >= skew4(66)
constexpr int kCostRight = (kCostPass + 68) * 5 / 4 + 2;     // >= skew4(16 ng + 68)
constexpr int kCostStep = 8 * kCostWarps;                    // disparities per step, 8 per warp
constexpr int kCostBuf = kCostRows * kCostPx * kCostStep * 4;   // bytes of the buffer
constexpr size_t kCostSmem = (size_t)kCostBuf + (size_t)4 * 16 * (kCostLeft + kCostRight);

struct CostArgs {
    CostScratch sc;                 // NCC: statistics of both images
    const uint8_t *left, *right;    // TAD
    int H, W, C, D, ld;
    float tau;
    float* out;
    bool early;                     // see agg_early
};

template <int MODE, bool MIRROR, int VW>
__device__ __forceinline__ void cost_tile(const CostArgs& a, int x0, int y0, int d_begin, int d_end, void* smem)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int H = a.H, W = a.W, D = a.D;
    uint8_t* const buf = (uint8_t*)smem;
    float4* const gl = (float4*)((uint8_t*)smem + kCostBuf);   // [2][kCostLeft]: columns x0 - 1 ..
    float4* const sl = gl + 2 * kCostLeft;    // [2][kCostLeft]: centres x0 ..
    float4* const gr = sl + 2 * kCostLeft;    // [2][kCostRight]: columns rb ..
    float4* const sr = gr + 2 * kCostRight;   // [2][kCostRight]: centres rb ..
    const size_t plane = (size_t)H * W;
    const size_t own = MIRROR ? plane : 0, other = MIRROR ? 0 : plane;
    const uint8_t* const own_img = MIRROR ? a.right : a.left;
    const uint8_t* const other_img = MIRROR ? a.left : a.right;

    // one column of an image: grey rows y0-1 .. y0+4 and the statistics of rows
    // y0 .. y0+3 (NCC), or the packed pixels of rows y0 .. y0+3 (TAD, in gl / gr)
    auto stage = [&](size_t img, const uint8_t* src, int x, float4* g0, float4* g1, float4* s0, float4* s1) {
        x = clampi(x, 0, W - 1);
        if (MODE == 0) {
            float g[6], s[4], v[4];
#pragma unroll
            for (int j = 0; j < 6; ++j) g[j] = (float)a.sc.g[img + (uint32_t)(clampi(y0 - 1 + j, 0, H - 1) * W + x)];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const size_t o = img + (uint32_t)(min(y0 + j, H - 1) * W + x);
                s[j] = a.sc.s[o];
                v[j] = a.sc.rv[o];
            }
            *g0 = make_float4(g[0], g[1], g[2], g[3]);
            *g1 = make_float4(g[2], g[3], g[4], g[5]);
            if (s0) {
                *s0 = make_float4(s[0], s[1], v[0], v[1]);
                *s1 = make_float4(s[2], s[3], v[2], v[3]);
            }
        } else {
            uint32_t c[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint8_t* q = src + ((size_t)min(y0 + j, H - 1) * W + x) * a.C;
                c[j] = a.C == 3 ? (uint32_t)q[0] | ((uint32_t)q[1] << 8) | ((uint32_t)q[2] << 16) : (uint32_t)q[0];
            }
            *g0 = make_float4(__uint_as_float(c[0]), __uint_as_float(c[1]), 0.f, 0.f);
            *g1 = make_float4(__uint_as_float(c[2]), __uint_as_float(c[3]), 0.f, 0.f);
        }
    };
    for (int c = tid; c < kCostPx + 2; c += kCostThreads) {
        // centre x0 + c - 1 sits at column c of gl and entry c - 1 of sl
        const bool centre = c >= 1 && c <= kCostPx;
        float4* s0 = sl + skew4(centre ? c - 1 : 0);
        stage(own, own_img, x0 - 1 + c, gl + skew4(c), gl + kCostLeft + skew4(c), centre ? s0 : nullptr, s0 + kCostLeft);
    }

    const int p = lane & 15, rp = lane >> 4;
    const int xl = 4 * p, xbase = x0 + xl;
    const float inv_c = 1.f / (float)a.C;
    const uint64_t one2 = f2_pack(1.f, 1.f);
    auto at = [](int m) { return m + (m >> 2); };   // offset of column base + m (base a multiple of 4)
    // buffer [row][pixel][step's disparities]; entry e of 8 bytes (disparities 2 e,
    // 2 e + 1) of pixel 4 p + i at 8 * (e ^ p)
    constexpr int PB = kCostStep * 4, RB = kCostPx * PB;   // bytes of a pixel, of a row
    static_assert(PB == 128, "16 entries per pixel, XORed with 16 pixel groups");
    const uint32_t put0 = tc::smem_u32(buf) + 2 * rp * RB + 4 * p * PB + 8 * (p ^ (4 * warp));

    for (int dp = d_begin; dp < d_end; dp += kCostPass) {
        const int ng = min(kCostPass / 16, (d_end - dp + 15) / 16);
        // other image's columns of this pass, from rb on; column x -+ d + k of
        // disparity dp + 16 g + s is base + m with base = xl + (MIRROR ? 4 + 16 g : 16 (ng - g)),
        // m = i + k -+ s
        const int rb = MIRROR ? x0 + dp - 4 : x0 - dp - 16 * ng;
        const int nr = 16 * ng + (MIRROR ? 68 : 65);
        for (int c = tid; c < nr; c += kCostThreads)
            stage(other, other_img, rb + c, gr + skew4(c), gr + kCostRight + skew4(c), sr + skew4(c),
                  sr + kCostRight + skew4(c));
        __syncthreads();
        for (int dq = dp; dq < min(dp + kCostPass, d_end); dq += kCostStep) {
            const int d0 = dq + 8 * warp;
            const int base = xl + (MIRROR ? 4 + d0 - dp : 16 * ng - (d0 - dp));
            const float4* glw = gl + rp * kCostLeft + skew4(xl);
            const float4* slw = sl + rp * kCostLeft + skew4(xl);
            const float4* grw = gr + rp * kCostRight + skew4(base);
            const float4* srw = sr + rp * kCostRight + skew4(base);
            constexpr int IN = MIRROR ? 5 : 0;      // where the new column comes in

            auto put = [&](int s, const float (&c)[4][2][2]) {   // c[pixel][row][s even, odd]
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"((put0 ^ (8 * (s >> 1))) + i * PB + h * RB),
                                     "f"(c[i][h][0]), "f"(c[i][h][1])
                                     : "memory");
            };
            // outside the image or no match there: the maximum; d >= D: 0
            auto mask = [&](float v, int i, int d, float most) {
                const int x = xbase + i;
                return d >= D ? 0.f : (MIRROR ? x + d >= W : x - d < 0) ? most : v;
            };

            if (d0 >= d_end) {
            } else if (MODE == 0) {
                float4 lw[6], rw[6];
                uint64_t sli[4], rli[4], sri[4], rri[4];
#pragma unroll
                for (int j = 0; j < 6; ++j) {
                    // -9 g': the block sums come out as -9 P' (exact: products below 2^24 / 9)
                    const float4 v = glw[at(j)];
                    lw[j] = make_float4(-9.f * v.x, -9.f * v.y, -9.f * v.z, -9.f * v.w);
                    rw[j] = grw[at(j - 1)];
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 v = slw[i], w = srw[at(i)];
                    sli[i] = f2_pack(v.x, v.y);
                    rli[i] = f2_pack(v.z, v.w);
                    sri[i] = f2_pack(w.x, w.y);
                    rri[i] = f2_pack(w.z, w.w);
                }
                auto sweep = [&](auto masked) {
                    float c[4][2][2];
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        if (s > 0) {
#pragma unroll
                            for (int j = 0; j < 5; ++j) {
                                if (MIRROR) rw[j] = rw[j + 1];
                                else rw[5 - j] = rw[4 - j];
                            }
                            rw[IN] = grw[at(MIRROR ? 4 + s : -1 - s)];
#pragma unroll
                            for (int i = 0; i < 3; ++i) {
                                if (MIRROR) sri[i] = sri[i + 1], rri[i] = rri[i + 1];
                                else sri[3 - i] = sri[2 - i], rri[3 - i] = rri[2 - i];
                            }
                            const float4 v = srw[at(MIRROR ? 3 + s : -s)];
                            sri[MIRROR ? 3 : 0] = f2_pack(v.x, v.y);
                            rri[MIRROR ? 3 : 0] = f2_pack(v.z, v.w);
                        }
                        uint64_t P[4];
                        block_sums(lw, rw, P);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float v0, v1;
                            f2_unpack(ncc_cost2(P[i], sli[i], sri[i], rli[i], rri[i], one2), v0, v1);
                            c[i][0][s & 1] = decltype(masked)::value ? mask(v0, i, d0 + s, 2.f) : v0;
                            c[i][1][s & 1] = decltype(masked)::value ? mask(v1, i, d0 + s, 2.f) : v1;
                        }
                        if (s & 1) put(s, c);
                    }
                };
                const bool inside = d0 + 8 <= D && (MIRROR ? xbase + 3 + d0 + 7 < W : xbase >= d0 + 7);
                if (__all_sync(0xffffffffu, inside)) sweep(std::integral_constant<bool, false>{});
                else sweep(std::integral_constant<bool, true>{});
            } else {
                uint32_t pl[4][2], pr[4][2];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 v = glw[at(i + 1)], w = grw[at(i)];
                    pl[i][0] = __float_as_uint(v.x), pl[i][1] = __float_as_uint(v.y);
                    pr[i][0] = __float_as_uint(w.x), pr[i][1] = __float_as_uint(w.y);
                }
                float c[4][2][2];
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    if (s > 0) {
#pragma unroll
                        for (int i = 0; i < 3; ++i)
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                if (MIRROR) pr[i][h] = pr[i + 1][h];
                                else pr[3 - i][h] = pr[2 - i][h];
                            }
                        const float4 w = grw[at(MIRROR ? 3 + s : -s)];
                        pr[MIRROR ? 3 : 0][0] = __float_as_uint(w.x);
                        pr[MIRROR ? 3 : 0][1] = __float_as_uint(w.y);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int sad = (int)__dp4a(__vabsdiffu4(pl[i][h], pr[i][h]), 0x01010101u, 0u);
                            c[i][h][s & 1] = mask(fminf((float)sad * inv_c, a.tau), i, d0 + s, a.tau);
                        }
                    if (s & 1) put(s, c);
                }
            }
            __syncthreads();
            // a warp writes one row: up to 128 contiguous bytes per pixel
            if (y0 + warp < H) {
                constexpr int L = kCostStep / VW, PXI = 32 / L;      // lanes per pixel, pixels per store
                const int e = lane % L, d = dq + VW * e;
                const bool din = VW == 4 ? d < a.ld && d < ((d_end + 3) & ~3) : d < min(D, d_end);
                const int npx = din ? min(kCostPx, W - x0) : 0;
                float* o = a.out + ((size_t)(y0 + warp) * W + x0 + lane / L) * a.ld + d;
                const uint8_t* q = buf + warp * RB + (lane / L) * PB;
#pragma unroll 4
                for (int px = lane / L; px < npx; px += PXI, o += (size_t)PXI * a.ld, q += PXI * PB) {
                    const int pp = px >> 2, c = e * VW / 2;
                    if (VW == 4) {
                        const float4 v = *(const float4*)(q + 8 * ((c ^ pp) & ~1));
                        *(float4*)o = pp & 1 ? make_float4(v.z, v.w, v.x, v.y) : v;
                    } else if (VW == 2) {
                        *(float2*)o = *(const float2*)(q + 8 * (c ^ pp));
                    } else {
                        *o = *(const float*)(q + 8 * (c ^ pp) + 4 * (e & 1));
                    }
                }
            }
            __syncthreads();   // the buffer, and after the last step the staged columns, may be overwritten
        }
    }
}

template <int MODE, bool MIRROR, int VW>
__global__ void __launch_bounds__(kCostThreads, 4) cost_kernel(const CostArgs a)
{
    extern __shared__ __align__(128) float4 sm_cost[];
    if (a.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the statistics must have been written
    cost_tile<MODE, MIRROR, VW>(a, blockIdx.x * kCostPx, blockIdx.y * kCostRows, 0, a.D, sm_cost);
    if (!a.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ CostArgs pair_args(const BatchPair& bp)
{
    return CostArgs{bp.sc, bp.left, bp.right, bp.H, bp.W, bp.C, bp.D, bp.ld, bp.tau, bp.cost, false};
}

// Batched FP32 cost volumes [H][W][ld]: an item is one 64 x 4 tile of a pair.
__global__ void __launch_bounds__(kCostThreads, 4)
cost_batched_kernel(const BatchPair* __restrict__ pairs, int npairs, int nitems, int* __restrict__ counter)
{
    extern __shared__ __align__(128) float4 sm_cost[];
    __shared__ int item_s;
    for (;;) {
        if (threadIdx.x == 0) item_s = atomicAdd(counter, 1);
        __syncthreads();
        const int item = item_s;
        __syncthreads();
        if (item >= nitems) break;
        const BatchPair& bp = pairs[find_pair(pairs, npairs, item, &BatchPair::cost_off)];
        const int t = item - bp.cost_off;
        const int nseg = (bp.W + kCostPx - 1) / kCostPx;
        const CostArgs a = pair_args(bp);
        const int x0 = (t % nseg) * kCostPx, y0 = (t / nseg) * kCostRows;
        if (bp.mode == 0) cost_tile<0, false, 4>(a, x0, y0, 0, bp.D, sm_cost);
        else cost_tile<1, false, 4>(a, x0, y0, 0, bp.D, sm_cost);
    }
}

// Band form: NCC costs of a 64 x 4 tile for the disparities that some aggregation
// tile reading it needs: the hull of the ranges [d_begin, d_end) of every
// aggregation tile whose window halo (the tile grown by rho) overlaps it.
// Entries outside that hull are not written (but for the rest of a run of 4).
__global__ void __launch_bounds__(kCostThreads, 4)
cost_band_kernel(const CostArgs a, int rho, const int2* __restrict__ tile_range, int ntx, int nty)
{
    extern __shared__ __align__(128) float4 sm_cost[];
    __shared__ int lo_s, hi_s;
    if (a.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int x0 = blockIdx.x * kCostPx, y0 = blockIdx.y * kCostRows;
    if (threadIdx.x == 0) {
        lo_s = a.D;
        hi_s = 0;
    }
    __syncthreads();
    // aggregation tiles ty with 4 ty - rho <= y0 + 3 and y0 <= 4 ty + 3 + rho, tx likewise
    const int ty0 = max(0, (y0 - rho + kAggTileY * 64) / kAggTileY - 64);
    const int ty1 = min(nty - 1, (y0 + kCostRows - 1 + rho) / kAggTileY);
    const int tx0 = max(0, (x0 - rho + kAggTileX * 64) / kAggTileX - 64);
    const int tx1 = min(ntx - 1, (x0 + kCostPx - 1 + rho) / kAggTileX);
    const int nx = tx1 - tx0 + 1;
    int lo = a.D, hi = 0;
    for (int i = threadIdx.x; i < (ty1 - ty0 + 1) * nx; i += kCostThreads) {
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
    cost_tile<0, false, 4>(a, x0, y0, d_begin, d_end, sm_cost);
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
// A CTA covers 64 pixels x 4 rows and every disparity (ncc_groups_per_cta: fewer on
// small frames).  All of Eq. (1) runs in
// FP32 on exact integers (grey_shift), and 9 P' - S_l' S_r' comes out of one FMA
// rounded once -- the integer converted to float.  A thread computes two output
// rows at once (block_sums: 4 FMAs for a column's two sums), and everything
// after them is packed, one row per half.
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

__host__ __device__ inline int ncc_groups(int D) { return (D + 15) / 16; }          // of 16 disparities
__host__ __device__ inline int ncc_right_cols(int groups) { return 16 * groups + kNccPx + 1; }
// float4 entries of the four staged arrays, per pair of rows
__host__ __device__ inline int ncc_left_len() { return skew4(kNccPx + 2); }
__host__ __device__ inline int ncc_right_len(int groups) { return skew4(ncc_right_cols(groups)) + 1; }
// Store buffer of a warp: two pairs of rows, each [d / 8][block][row][8 d x 8
// pixels] (128-byte lines, TMA's 128-byte swizzle) of 16 disparities and 8 blocks.
constexpr int kNccPairBytes = 2 * 8 * 2 * 128, kNccWarpBytes = 2 * kNccPairBytes;
__host__ __device__ inline size_t ncc_smem_bytes(int groups)
{
    return 1024 + (size_t)kNccWarps * kNccWarpBytes + (size_t)2 * 16 * 2 * (ncc_left_len() + ncc_right_len(groups));
}
// Groups per CTA, of the ng groups of costs and one more (the rows after them): all,
// or where the tiles leave SMs without a CTA, a share of them (whole rounds of the
// warps) such that no SM gets two, if that saves two rounds (each CTA stages the
// grey rows of its own range; one round saved was 300x60, D = 128, radius 0 14.7 ->
// 15.5 us).  On the smallest frames one CTA for all of D was slower than the
// integer form: BF16 path, integer form -> undivided -> now: 80x60, D = 208, radius
// 5 16.5 -> 20.6 -> 14.5 us; 40x24, D = 256, radius 0 14.5 -> 18.5 -> 12.3 us; 300x60,
// D = 256, radius 5 22.7 -> 24.7 -> 22.6 us.
inline int ncc_groups_per_cta(int D, int tiles, int num_sms)
{
    const int all = ncc_groups(D) + 1, rounds = (all + kNccWarps - 1) / kNccWarps;
    const int share = num_sms / tiles < 1 ? 1 : num_sms / tiles;
    const int own = (rounds + share - 1) / share;
    return (rounds - own < 2 ? rounds : own) * kNccWarps;
}

template <bool BF16>
__global__ void __launch_bounds__(32 * kNccWarps, 4)
cost_xb_ncc_kernel(const __grid_constant__ CUtensorMap out_map, const uint8_t* __restrict__ L,
                   const uint8_t* __restrict__ R, int H, int W, int C, int D, int per_cta, uint2* __restrict__ rgbx)
{
    extern __shared__ uint8_t sm_ncc[];
    // let a programmatically launched successor (the tensor-core aggregation)
    // start its set-up once every CTA of this grid has started; it waits for
    // this grid's completion before it reads anything this kernel writes
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int ROWS = kNccRows, PAIRS = ROWS / 2, nthr = 32 * kNccWarps;
    const int tid = threadIdx.x, lane = tid & 31;
    const int x0 = blockIdx.x * kNccPx, y0 = blockIdx.y * ROWS;
    const int ng = ncc_groups(D);
    // this CTA's groups g0 .. g1-1, of which those before gc have costs
    const int g0 = blockIdx.z * per_cta, g1 = min(g0 + per_cta, ng + 1), gc = min(g1, ng);
    const int nr = ncc_right_cols(gc - g0);
    const int rb = x0 - 16 * gc;             // image column of right column 0
    const int LL = ncc_left_len(), RL = ncc_right_len(gc - g0);
    uint8_t* const buffers = sm_ncc + ((1024u - (tc::smem_u32(sm_ncc) & 1023u)) & 1023u);
    float4* const gl = (float4*)(buffers + kNccWarps * kNccWarpBytes);   // [PAIRS][LL]: columns x0 - 1 ..
    float4* const sl = gl + PAIRS * LL;      // [PAIRS][LL]: centres x0 ..
    float4* const gr = sl + PAIRS * LL;      // [PAIRS][RL]: columns rb ..
    float4* const sr = gr + PAIRS * RL;      // [PAIRS][RL]: centres rb ..

    // ---- grey rows y0-1 .. y0+ROWS of both images at clamped columns, and the
    // left image's packed guide
    const int shift = grey_shift(C);
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
        if (left && c >= 1 && c <= kNccPx && xs < W && g0 == 0) {
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
    for (int grp = g0 + (tid >> 5); grp < g1; grp += kNccWarps) {
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
        const int base = xl + 16 * gc - d0;
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
                uint64_t P[4];
                block_sums(lw, rw, P);
                float c0[4], c1[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    f2_unpack(ncc_cost2(P[i], sli[i], sri[i], rli[i], rri[i], one2), c0[i], c1[i]);
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
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    dim3 grid((W + kNccPx - 1) / kNccPx, (H + kNccRows - 1) / kNccRows);
    const int ng = ncc_groups(D), per_cta = ncc_groups_per_cta(D, (int)(grid.x * grid.y), sms);
    grid.z = (ng + per_cta) / per_cta;   // ng + 1 groups
    const size_t smem = ncc_smem_bytes(per_cta < ng ? per_cta : ng);
    e = fbs::raise_smem_limit(cost_xb_ncc_kernel<BF16>, (int)smem);
    if (e != cudaSuccess) return e;
    fbs::note_launch();
    cost_xb_ncc_kernel<BF16><<<grid, 32 * kNccWarps, smem, stream>>>(map, left, right, H, W, C, D, per_cta, sc.rgbx);
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

template <int MODE, bool MIRROR, int VW>
cudaError_t launch_cost_vw(const CostArgs& a, cudaStream_t stream)
{
    cudaError_t e = fbs::raise_smem_limit(cost_kernel<MODE, MIRROR, VW>, (int)kCostSmem);
    if (e != cudaSuccess) return e;
    const dim3 grid((a.W + kCostPx - 1) / kCostPx, (a.H + kCostRows - 1) / kCostRows);
    if (MODE == 0 || MIRROR)   // behind the statistics or the other view
        return fbs::launch_after(cost_kernel<MODE, MIRROR, VW>, grid, kCostThreads, kCostSmem, stream, a);
    fbs::note_launch();
    cost_kernel<MODE, MIRROR, VW><<<grid, kCostThreads, kCostSmem, stream>>>(a);
    return cudaGetLastError();
}

// When may the aggregation's CTAs start: with the cost kernel's (they set up
// while it runs), or as its CTAs end?  An early CTA takes any place that is
// free, so where the aggregation does not fill the chip (four CTAs per SM) some
// SMs get several and others none.  Early for a grid that fills it, for one so
// small that every CTA of both kernels finds an SM of its own, and for tiles of so
// little work that the set-up is what counts (work: window rows x window columns
// of 8 pixels x disparities staged).  Measured, early and late, at 12 to 640 tiles,
// D = 8 .. 200, radius 0 .. 15, calls in a row: up to 45 tiles early is 0 - 16%
// faster, most of all at little work (40x24, D = 64, radius 3 20.6 and 22.6 us); at
// 150 to 350 tiles late wins from about 6400 on (160x120, D = 128, radius 15 by 40%;
// 160x120, D = 16, radius 4 takes 20.7 us early, 22.6 late); at 480 tiles late is
// 8% faster at most; from 600 on early is never more than 2% behind.  Over all of
// these the rule is 0.2% above the better of the two on average, always early 3.7%.
bool agg_early(int H, int W, int D, int radius, int num_sms)
{
    const long long tiles = (long long)((W + kAggTileX - 1) / kAggTileX) * ((H + kAggTileY - 1) / kAggTileY);
    const long long staged = D <= 16 ? 16 : (D + 31) / 32 * 32;
    return tiles >= 4LL * num_sms || 2 * tiles <= num_sms ||
           (kAggTileY + 2 * radius) * (8 + 2 * radius) * staged < 100 * 64;
}

// One view of the FP32 volume (mode 0: after the statistics).
cudaError_t launch_cost_view(const CostArgs& a, int mode, bool mirror, cudaStream_t stream)
{
    const uintptr_t o = reinterpret_cast<uintptr_t>(a.out);
    if (a.ld % 4 == 0 && (o & 15) == 0) {
        if (mirror) return mode == 0 ? launch_cost_vw<0, true, 4>(a, stream) : launch_cost_vw<1, true, 4>(a, stream);
        return mode == 0 ? launch_cost_vw<0, false, 4>(a, stream) : launch_cost_vw<1, false, 4>(a, stream);
    }
    if (mirror) return cudaErrorInvalidValue;   // the context's own volume
    if (a.ld % 2 == 0 && (o & 7) == 0)
        return mode == 0 ? launch_cost_vw<0, false, 2>(a, stream) : launch_cost_vw<1, false, 2>(a, stream);
    return mode == 0 ? launch_cost_vw<0, false, 1>(a, stream) : launch_cost_vw<1, false, 1>(a, stream);
}

cudaError_t launch_stats(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W, int C,
                         cudaStream_t stream)
{
    fbs::note_launch();
    grey_stats_kernel<<<dim3((W + kStatX - 1) / kStatX, (H + kStatY - 1) / kStatY, 2), kStatX, 0, stream>>>(left, right, H, W,
                                                                                                        C, sc);
    return cudaGetLastError();
}

}  // namespace

int stats_items(int H, int W) { return ((H + kStatY - 1) / kStatY) * ((W + kStatX - 1) / kStatX); }
int cost_items(int H, int W) { return ((H + kCostRows - 1) / kCostRows) * ((W + kCostPx - 1) / kCostPx); }

cudaError_t prepare_cost_batched() { return fbs::raise_smem_limit(cost_batched_kernel, (int)kCostSmem); }

cudaError_t launch_stats_batched(const BatchPair* pairs, int npairs, int nitems, int* counter, int grid,
                                 cudaStream_t stream)
{
    fbs::note_launch();
    grey_stats_batched_kernel<<<grid, kStatX, 0, stream>>>(pairs, npairs, nitems, counter);
    return cudaGetLastError();
}

cudaError_t launch_cost_batched(const BatchPair* pairs, int npairs, int nitems, int* counter, int grid,
                                cudaStream_t stream)
{
    fbs::note_launch();
    cost_batched_kernel<<<grid, kCostThreads, kCostSmem, stream>>>(pairs, npairs, nitems, counter);
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
    sc.s = (float*)p;
    p += (n * sizeof(int) + 255) & ~(size_t)255;
    sc.rv = (float*)p;
    return sc;
}

cudaError_t launch_cost_build(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W,
                              int C, int D, int ld, int mode, float tau, float* cost, int agg_radius, int num_sms,
                              cudaStream_t stream)
{
    cudaError_t e = mode == 0 ? launch_stats(sc, left, right, H, W, C, stream) : cudaSuccess;
    if (e != cudaSuccess) return e;
    return launch_cost_view(CostArgs{sc, left, right, H, W, C, D, ld, tau, cost, agg_early(H, W, D, agg_radius, num_sms)},
                            mode, false, stream);
}

cudaError_t launch_cost_band(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W,
                             int C, int D, int ld, int radius, const int2* tile_range, float* cost, int num_sms, cudaStream_t stream)
{
    cudaError_t e = launch_stats(sc, left, right, H, W, C, stream);
    if (e == cudaSuccess) e = fbs::raise_smem_limit(cost_band_kernel, (int)kCostSmem);
    if (e != cudaSuccess) return e;
    const int ntx = (W + kAggTileX - 1) / kAggTileX, nty = (H + kAggTileY - 1) / kAggTileY;
    return fbs::launch_after(cost_band_kernel, dim3((W + kCostPx - 1) / kCostPx, (H + kCostRows - 1) / kCostRows), kCostThreads,
                             kCostSmem, stream,
                             CostArgs{sc, left, right, H, W, C, D, ld, 0.f, cost, agg_early(H, W, D, radius, num_sms)}, radius,
                             tile_range, ntx, nty);
}

cudaError_t launch_cost_build_lr(const CostScratch& sc, const uint8_t* left, const uint8_t* right, int H, int W,
                                 int C, int D, int ld, int mode, float tau, float* cost, float* cost_r, int agg_radius,
                                 int num_sms, cudaStream_t stream)
{
    cudaError_t e = launch_cost_build(sc, left, right, H, W, C, D, ld, mode, tau, cost, agg_radius, num_sms, stream);
    if (e != cudaSuccess) return e;
    return launch_cost_view(CostArgs{sc, left, right, H, W, C, D, ld, tau, cost_r, agg_early(H, W, D, agg_radius, num_sms)},
                            mode, true, stream);
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
