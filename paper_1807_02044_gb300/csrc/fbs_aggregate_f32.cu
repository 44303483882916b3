// Steps 2-4 of fast bilateral stereo in FP32: bilateral aggregation of every
// disparity slice (Sec. II-B, Eq. (6)-(8)), winner-take-all (Sec. II-C) and
// the parabola refinement of Eq. (10) (Sec. II-D), in one kernel.
//
//   Agg(p, d) = sum_q w(p, q) C(q, d) / sum_q w(p, q),
//   w(p, q)   = exp(-|q - p|^2 / gamma_d^2) * exp(-|I(q) - I(p)|^2 / gamma_r^2),
// q over the (2 rho + 1)^2 window clipped to the image; I is the left image
// (for RGB the squared Euclidean colour distance).  The two exponentials are
// evaluated as one exp2 of the summed exponent.
//
// Work decomposition (one CTA = a 32 x 4 pixel tile, 4 warps, four CTAs per
// SM; the disparities in chunks of 64, 32 or 16):
//   * The tile's guide window is staged once.  Cost rows r = y0-rho .. y0+3+rho
//     are streamed through a ring of S rows, one TMA box per row (zeros outside
//     the image and past D).  The last of the four warps to finish a row issues
//     the row S later into its slot, so no warp waits for another one except
//     through a full ring, and warps run up to S - 1 rows apart.
//   * A warp owns 32 pixels (16 x 2, or 8 x 4 in the band form) and every
//     disparity of the chunk: it computes their weights for the row (lane =
//     pixel, once per (p, q) and chunk) into its own shared buffer and then
//     accumulates, so warps exchange nothing but the staged rows.
//   * A thread accumulates 8 pixels along x by 8 (4, 2) disparities.  It walks
//     the columns of the row: a column's costs are loaded once and used for
//     all of the 8 pixels whose window holds the column, each with its weight
//     (the 8 weights of a column are contiguous).  Per column: 4 shared loads
//     of 16 bytes for 32 packed FMAs (two disparities each).
//   * After the last row the sums are normalised, staged per warp and reduced
//     per pixel by one lane: WTA with the smallest d on ties, plus the values
//     at d*-1 and d*+1 carried across chunks for Eq. (10).
// Every sum runs over the rows and, in a row, over the columns in ascending
// order, whatever the tile or the chunk.
//
// Why this split.  The bound is the FP32 pipe.  A packed FMA takes half the
// issue slots of two scalar ones, and the freed slots hold the weights; with
// three fresh register pairs it runs at 94 multiply-adds per clock and SM, with
// one operand shared by consecutive FMAs at up to 118 (of 128).  An 8 x 8
// register tile needs (8 + 8) / 64 shared values per multiply-add.  A shared load
// of 16 bytes takes 2 cycles when no four adjacent lanes hold more than two
// distinct addresses and 4 cycles otherwise (measured, whatever the number of
// distinct addresses in the warp), so lane bit 1 never selects a cost address
// and lane bit 0 never a weight address.  The accumulation loop alone runs at
// 73% of 128 multiply-adds per clock and SM; with everything around it the
// kernel is at 45%.  Copying a row with one bulk copy per column instead of one
// box cost 22 cycles per column and SM and bound the kernel (322 against 244 us),
// and a __syncthreads per row 313 us.
//
// Measured on GB300 (CUDA events), before -> now; before: 4 pixels x 8 disparities
// per thread, scalar FMAs, 256-thread CTAs in step through a cp.async ring:
//   640x480,  D = 64,  rho = 7:    427 ->  232 us (38.1 TFLOP/s)
//   640x480,  D = 64,  rho = 2:    132 ->   62 us
//   767x575,  D = 96,  rho = 11:  2261 -> 1131 us
//   1280x960, D = 128, rho = 15: 10383 -> 6550 us (46.2 TFLOP/s)
// and where the wide windows leave fewer warps per SM (12 at rho = 13 .. 19, 8 at 20
// .. 24, 4 at 31, for 16, 16 and 8 before):
//   640x480,  D = 64,  rho = 20:  2173 -> 1572 us (42.1 TFLOP/s)
//   640x480,  D = 64,  rho = 24:  2983 -> 2178 us (43.4 TFLOP/s)
//   640x480,  D = 64,  rho = 31:  6079 -> 4860 us (32.1 TFLOP/s)
#include "fbs_internal.cuh"
#include "packed_f32.cuh"
#include "tc_aggregate.cuh"

namespace fbs {
namespace {

constexpr int kTX = kAggTileX;   // tile width (pixels)
constexpr int kTY = kAggTileY;   // tile height (rows)
constexpr int kPX = 8;           // pixels per thread along x
constexpr int kWarps = 4;
constexpr int kThreads = 32 * kWarps;
static_assert(kTX * kTY == 32 * kWarps, "a warp owns 32 pixels of the tile");
// 2^23 as an FP32 bit pattern: for 0 <= c < 2^23 the pattern kMagic + c is the
// float 2^23 + c exactly.
constexpr uint32_t kMagic = 0x4B000000u;

// Weights of a group of 8 pixels and one row: [column j][pixel i], j = dx + i
// (dx = 0 .. 2 rho), so 2 rho + 8 columns of 8 floats; == 8 (mod 32) floats, so
// that lanes writing pixels i of four groups, 9 i + 8 g, hit 32 banks.
__host__ __device__ inline int weight_stride(int rho) { return (((2 * rho + kPX) * kPX + 31) & ~31) + 8; }

// Disparities per staged column: 64, or what a short range needs.
__host__ __device__ inline int column_size(int D) { return D > 32 ? 64 : D > 16 ? 32 : 16; }

// How a cost row is copied to shared memory: one TMA box (volumes that are 16-byte
// aligned with ld % 4 == 0), or cp.async of so many bytes by every thread: 16
// (the same volumes, where no tensor map is at hand) or 4 (any volume: 640x480,
// D = 63, rho = 7: 328 us against 232 us at D = 64 by TMA; 474 us before).
enum Copy { kTma = 0, kAsync16 = 16, kAsync4 = 4 };

template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t smem, const void* gmem, int src_bytes)
{
    if (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem), "l"(gmem), "r"(src_bytes) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;\n" ::"r"(smem), "l"(gmem), "r"(src_bytes), "n"(BYTES)
                     : "memory");
}
// The mbarrier gets one arrival of this thread when its earlier cp.async have landed.
__device__ __forceinline__ void cp_async_arrive(uint32_t bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int d, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"((uint64_t)map), "r"(d), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
// Counts one more warp done with a slot (its reads before, the caller's writes after).
__device__ __forceinline__ uint32_t count_done(uint32_t word)
{
    uint32_t old;
    asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(word) : "memory");
    return old;
}

// Spatial terms of Eq. (7): row dy = 0 .. rho of 2 rho + 2 floats (dx = -rho ..
// rho and one more).
__host__ __device__ inline int spatial_floats(int rho) { return (rho + 1) * (2 * rho + 2); }
// Guide window of a tile: (kTY + 2 rho) rows of kTX + 2 rho words, and one more.
__host__ __device__ inline int guide_words(int rho) { return (kTY + 2 * rho) * (kTX + 2 * rho) + 1; }

// Shared memory of a CTA, in order: the barriers of the S slots, the
// spatial terms, the guide window, then the cost rows [S][NC][DC] and the warps'
// weights [4][4][WS]; the stage [4][32][DC + 4] of the epilogue lies over these.
constexpr int kMaxSlots = 4;
constexpr int kHeaderBytes = 88;   // RingState
__host__ __device__ inline size_t front_bytes(int rho)
{
    return (kHeaderBytes + 4 * (size_t)spatial_floats(rho) + 4 * (size_t)guide_words(rho) + 127) & ~(size_t)127;
}
__host__ __device__ inline size_t smem_bytes(int rho, int dc, int slots)
{
    const int NC = kTX + 2 * rho;
    const size_t rows = (size_t)slots * NC * dc + (size_t)kWarps * 4 * weight_stride(rho);
    const size_t stage = (size_t)kWarps * 32 * (dc + 4);
    return front_bytes(rho) + sizeof(float) * (rows > stage ? rows : stage);
}

// The ring of cost rows.  Every warp walks every row, so slot and parity (of
// the row it is at) are the same sequence in all of them.
//   kTma: done[slot] counts the warps that have finished the slot's row; the
//   last one issues the box of the row S later.  The word after the count is 0,
//   or 2 + the parity of the phase that the slot's last box completes.
//   cp.async: every warp loads a quarter of each row, once all of them have
//   arrived at the barrier done[slot]; a warp waits for that when it starts
//   the next row.
// Every wait is bounded.  When one runs out the error word is set, the warps walk
// the rows that are left without waiting or copying, and the CTA lets the copies
// in flight land (drain) and leaves its tile without storing anything.
struct RingState {
    uint64_t full[kMaxSlots], done[kMaxSlots];
    uint32_t abort;           // a wait ran out
    int* err;
    long long limit;          // SM clock cycles that a wait may take
};
static_assert(sizeof(RingState) == kHeaderBytes, "at the start of shared memory");

// A bounded wait for the phase of the given parity: by tries that sleep, or, for
// limits shorter than a sleep, by polling.  One block, because it is inlined at
// every wait and the small frames pay for the kernel's size.
template <bool POLLS>
__device__ __forceinline__ bool wait_within(uint32_t bar, uint32_t par, uint32_t limit_addr)
{
    uint32_t ok;
    if (POLLS)
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t.reg .b64 t, u, lim;\n\t"
            "ld.shared.b64 lim, [%3];\n\t"
            "mov.u64 t, %%clock64;\n"
            "POLL:\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "@p bra DONE;\n\t"
            "mov.u64 u, %%clock64;\n\t"
            "sub.s64 u, u, t;\n\t"
            "setp.le.s64 q, u, lim;\n\t"
            "@q bra POLL;\n"
            "DONE:\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(par), "r"(limit_addr)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t.reg .b64 t, u, lim;\n\t"
            "ld.shared.b64 lim, [%3];\n\t"
            "mov.u64 t, %%clock64;\n"
            "TRY:\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %4;\n\t"
            "@p bra DONE;\n\t"
            "mov.u64 u, %%clock64;\n\t"
            "sub.s64 u, u, t;\n\t"
            "setp.le.s64 q, u, lim;\n\t"
            "@q bra TRY;\n"
            "DONE:\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(par), "r"(limit_addr), "n"(tc::kSuspendNs)
            : "memory");
    return ok != 0;
}

template <bool POLLS>
struct Ring {
    RingState* st;
    uint32_t full, done;      // shared addresses, 8 bytes per slot
    int S, slot;
    uint32_t parity;
    // by every thread, before a barrier of the CTA
    __device__ __forceinline__ void set_limit(long long limit)
    {
        if (threadIdx.x == 0) st->limit = limit;
    }
    __device__ __forceinline__ void next()
    {
        if (++slot == S) {
            slot = 0;
            parity ^= 1u;
        }
    }
    __device__ __forceinline__ bool aborted() const { return *(volatile uint32_t*)&st->abort != 0; }
    // False when the phase is not complete and nothing is waited for any more.
    __device__ __forceinline__ bool wait(uint32_t bar, uint32_t par) const
    {
        if (!POLLS && tc::mbar_try_wait(bar, par)) return true;
        if (aborted()) return false;
        if (wait_within<POLLS>(bar, par, tc::smem_u32(&st->limit))) return true;
        *(volatile uint32_t*)&st->abort = 1u;
        atomicCAS(st->err, 0, 31);
        return false;
    }
    // After a wait ran out and a barrier of the CTA: the copies in flight (those of a
    // slot's last box; the ones before it were waited for) have landed, or had about
    // 2 s more.
    template <Copy COPY>
    __device__ __forceinline__ void drain() const
    {
        if constexpr (COPY == kTma) {
            if ((int)threadIdx.x < S) {
                uint32_t armed;
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(armed) : "r"(done + 8 * threadIdx.x + 4) : "memory");
                if (armed != 0) tc::mbar_wait(full + 8 * threadIdx.x, armed & 1u);
            }
        } else {
            asm volatile("cp.async.wait_all;" ::: "memory");
        }
        __syncthreads();
    }
};

// The cost volume of a tile's pair.
struct Volume {
    const float* cost;
    const CUtensorMap* map;   // kTma: dimensions (D, W, H), box (DC, kTX + 2 rho, 1)
    int ld, W, D;
};

// Load cost row r, columns xlo .. xlo+NC-1, disparities dc0 .. dc0+DC-1 into a
// slot; zeros outside the image and for disparities >= D.  kTma: one warp, which
// notes the phase (parity) that the box completes; otherwise all of them, a thread
// its share.
template <int DC, Copy COPY, bool POLLS>
__device__ __forceinline__ void load_cost_row(const Ring<POLLS>& ring, int slot, uint32_t parity, uint32_t rows_a, const Volume& v,
                                              int r, int xlo, int NC, int dc0)
{
    const uint32_t dst = rows_a + slot * (uint32_t)(NC * DC * 4), bar = ring.full + 8 * slot;
    if constexpr (COPY == kTma) {
        if ((threadIdx.x & 31) == 0) {
            tc::fence_proxy_async();   // the slot was read, and may hold staged sums, through the generic proxy
            tc::mbar_expect_tx(bar, 4u * DC * (uint32_t)NC);
            tma_load_3d(dst, v.map, dc0, xlo, r, bar);
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(ring.done + 8 * slot + 4), "r"(2u + parity) : "memory");
        }
    } else {
        constexpr int E = COPY / 4;                     // floats per copy
        constexpr int Q = DC / E, STEP = kThreads / Q;  // copies per column, columns per pass
        static_assert(STEP >= 1, "a pass covers whole columns");
        const int q = threadIdx.x % Q, c0 = threadIdx.x / Q, d = dc0 + E * q, bytes = d < v.D ? 4 * min(E, v.D - d) : 0;
        const float* src = v.cost + ((ptrdiff_t)r * v.W + xlo + c0) * v.ld + d;
        const ptrdiff_t step = (ptrdiff_t)STEP * v.ld;
        uint32_t to = dst + 4 * (c0 * DC + E * q);
        if (xlo >= 0 && xlo + NC <= v.W && dc0 + DC <= v.D) {
#pragma unroll 4
            for (int c = c0; c < NC; c += STEP, to += 4 * STEP * DC, src += step) cp_async<COPY>(to, src, COPY);
        } else {
#pragma unroll 2
            for (int c = c0; c < NC; c += STEP, to += 4 * STEP * DC, src += step) {
                const bool in = (unsigned)(xlo + c) < (unsigned)v.W && bytes > 0;
                cp_async<COPY>(to, in ? src : v.cost, in ? bytes : 0);
            }
        }
        cp_async_arrive(bar);
    }
}

// A guide pixel as R | G << 8 | B << 16; grey images use the first channel only.
__device__ __forceinline__ uint32_t packed_colour(const uint8_t* p, int C)
{
    return C == 3 ? (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) : (uint32_t)p[0];
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two consecutive taps dx, dx + 1 of one pixel and window row: Eq. (7)-(8) as
// one exp2, colour distance exact in integers (bytewise differences, their
// squares: one instruction less per weight than |q|^2 + |p|^2 - 2 q.p, 1203 ->
// 1136 us at 767x575, D = 93, rho = 11), then float(c) = (2^23 + c) - 2^23 exactly.  sp: the two spatial terms
// ((dx - rho)^2 + dy^2) times -log2(e) / sigma_s^2.  EDGE: a tap outside the
// image columns has weight 0.
struct Pixel {
    uint32_t col;             // its colour
    uint64_t magic2, nkr2;    // (-2^23, -2^23) and -log2(e) / sigma_r^2 twice
    int qx, W;                // image column of tap 0
};
template <bool EDGE>
__device__ __forceinline__ void weight_pair(const Pixel& p, uint32_t q0, uint32_t q1, uint64_t sp, int dx, float& w0,
                                            float& w1)
{
    const uint32_t d0 = __vabsdiffu4(q0, p.col), d1 = __vabsdiffu4(q1, p.col);
    const uint32_t e0 = __dp4a(d0, d0, kMagic), e1 = __dp4a(d1, d1, kMagic);
    f2_unpack(f2_fma(f2_add(u2_pack(e0, e1), p.magic2), p.nkr2, sp), w0, w1);
    w0 = ex2_approx(w0);
    w1 = ex2_approx(w1);
    if (EDGE) {
        w0 = (unsigned)(p.qx + dx) < (unsigned)p.W ? w0 : 0.f;
        w1 = (unsigned)(p.qx + dx + 1) < (unsigned)p.W ? w1 : 0.f;
    }
}

// All taps of one pixel and window row, in order: tap dx goes to w[8 dx] (w
// offset by the pixel's place in its group) and to den0 (dx <= rho) or den1.
// sp holds 2 rho + 2 spatial terms; g[2 rho + 1] is read and not used.
template <bool EDGE>
__device__ __forceinline__ void weight_row(const Pixel& p, const uint32_t* g, const uint64_t* sp, float* w, int rho,
                                           float& den0, float& den1)
{
    float a, b;
    int dx = 0;
    auto pair = [&]() {
        weight_pair<EDGE>(p, g[0], g[1], sp[0], dx, a, b);
        w[0] = a;
        w[kPX] = b;
        g += 2;
        sp += 1;
        w += 2 * kPX;
        dx += 2;
    };
    const int n0 = (rho + 1) >> 1;
#pragma unroll 4
    for (int j = 0; j < n0; ++j) {
        pair();
        den0 += a;
        den0 += b;
    }
    if (!(rho & 1) && rho > 0) {   // taps rho and rho + 1
        pair();
        den0 += a;
        den1 += b;
    }
#pragma unroll 4
    for (int j = (rho >> 1) + 1; j < rho; ++j) {
        pair();
        den1 += a;
        den1 += b;
    }
    weight_pair<EDGE>(p, g[0], g[1], sp[0], dx, a, b);   // tap 2 rho
    w[0] = a;
    if (rho == 0) den0 += a;
    else den1 += a;
}

// Two consecutive costs of a column as a packed pair, KD of them per thread:
// disparities 4 k .. 4 k + 3 (and 32 + the same) of the chunk, or 2 k, 2 k + 1.
template <int KD>
__device__ __forceinline__ void load_costs(uint32_t a, uint64_t (&c)[KD / 2])
{
    if (KD == 2) {
        asm volatile("ld.shared.b64 %0, [%1];" : "=l"(c[0]) : "r"(a) : "memory");
    } else {
#pragma unroll
        for (int q = 0; q < KD / 4; ++q)
            asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];"
                         : "=l"(c[2 * q]), "=l"(c[2 * q + 1])
                         : "r"(a + 128 * q)
                         : "memory");
    }
}

__device__ __forceinline__ void load_weights(uint32_t a, float (&w)[4])
{
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(w[0]), "=f"(w[1]), "=f"(w[2]), "=f"(w[3])
                 : "r"(a)
                 : "memory");
}

// One column: pixels LO .. HI-1 of the thread's 8 get their weight times the
// column's costs.  The cost pair is the operand that consecutive FMAs share
// (an FMA with three fresh register pairs issues every 2.7 cycles instead of 2).
template <int KD, int LO, int HI>
__device__ __forceinline__ void column(uint64_t (&acc)[kPX][KD / 2], uint32_t ca, uint32_t wa)
{
    uint64_t c[KD / 2], ww[kPX];
    load_costs<KD>(ca, c);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 0 ? LO >= 4 : HI <= 4) continue;
        float w[4];
        load_weights(wa + 16 * h, w);
#pragma unroll
        for (int i = 0; i < 4; ++i) ww[4 * h + i] = f2_pack(w[i], w[i]);
    }
#pragma unroll
    for (int k = 0; k < KD / 2; ++k)
#pragma unroll
        for (int i = LO; i < HI; ++i) acc[i][k] = f2_fma(c[k], ww[i], acc[i][k]);
}

// Columns J, J + 1, .. of a window of a fixed radius RHO < 4.
template <int KD, int DC, int RHO, int J>
__device__ __forceinline__ void narrow_columns(uint64_t (&acc)[kPX][KD / 2], uint32_t ca, uint32_t wa)
{
    if constexpr (J < 2 * RHO + kPX) {
        column<KD, (J > 2 * RHO ? J - 2 * RHO : 0), (J < kPX ? J + 1 : kPX)>(acc, ca + J * DC * 4, wa + J * kPX * 4);
        narrow_columns<KD, DC, RHO, J + 1>(acc, ca, wa);
    }
}

// One window row of a thread: columns j = 0 .. 2 rho + 7, pixel i takes part in
// columns i .. i + 2 rho.  ca, wa: shared addresses of column 0's costs and weights.
template <int KD, int DC>
__device__ __forceinline__ void accumulate_row(uint64_t (&acc)[kPX][KD / 2], uint32_t ca, uint32_t wa, int rho)
{
    constexpr uint32_t CS = DC * 4, WC = kPX * 4;   // bytes from a column to the next
    if (rho >= 4) {
        column<KD, 0, 1>(acc, ca, wa);
        column<KD, 0, 2>(acc, ca + CS, wa + WC);
        column<KD, 0, 3>(acc, ca + 2 * CS, wa + 2 * WC);
        column<KD, 0, 4>(acc, ca + 3 * CS, wa + 3 * WC);
        column<KD, 0, 5>(acc, ca + 4 * CS, wa + 4 * WC);
        column<KD, 0, 6>(acc, ca + 5 * CS, wa + 5 * WC);
        column<KD, 0, 7>(acc, ca + 6 * CS, wa + 6 * WC);
        ca += 7 * CS;
        wa += 7 * WC;
#pragma unroll 1
        for (int n = rho - 3; n > 0; --n) {     // 2 rho - 6 columns with all 8 pixels
            column<KD, 0, 8>(acc, ca, wa);
            column<KD, 0, 8>(acc, ca + CS, wa + WC);
            ca += 2 * CS;
            wa += 2 * WC;
        }
        column<KD, 1, 8>(acc, ca, wa);
        column<KD, 2, 8>(acc, ca + CS, wa + WC);
        column<KD, 3, 8>(acc, ca + 2 * CS, wa + 2 * WC);
        column<KD, 4, 8>(acc, ca + 3 * CS, wa + 3 * WC);
        column<KD, 5, 8>(acc, ca + 4 * CS, wa + 4 * WC);
        column<KD, 6, 8>(acc, ca + 5 * CS, wa + 5 * WC);
        column<KD, 7, 8>(acc, ca + 6 * CS, wa + 6 * WC);
    } else {
        // windows narrower than the thread's 8 pixels: no column belongs to all of them
        if (rho == 3) narrow_columns<KD, DC, 3, 0>(acc, ca, wa);
        else if (rho == 2) narrow_columns<KD, DC, 2, 0>(acc, ca, wa);
        else if (rho == 1) narrow_columns<KD, DC, 1, 0>(acc, ca, wa);
        else narrow_columns<KD, DC, 0, 0>(acc, ca, wa);
    }
}

// What a tile's chunks share: the arguments, the lane's own pixel (the one
// whose weights, WTA and Eq. (10) it does) and that pixel's WTA state.
struct Tile {
    Volume vol;
    int H, W, D, rho;
    float neg_kr;
    int x0, y0, r_lo, r_hi, d_end;
    const float* spatial;
    const uint32_t* guide;   // row r_lo, column x0 - rho
    float* rows;             // cost rows, weights, stage
    int wy;                  // the warp's first row
    int px, py;              // the lane's pixel
    uint32_t pcol;
    int blo, bhi;            // its band
    int wlo, whi;            // union of the bands of the warp's pixels
    float best, a_prev, a_next, last;
    int bidx;
    bool pending;
};

// WTA of one pixel over the staged values j0 .. j1-1 (disparities dc0 + j):
// the smallest value, the first of equal ones (a NaN never wins), and the
// neighbours of the winner for Eq. (10), which may lie in the chunks before and after.
__device__ __forceinline__ void wta_chunk(Tile& t, const float* st, int dc0, int j0, int j1)
{
    if (j0 >= j1) return;
    const float inf = __int_as_float(0x7f800000);
    auto read4 = [&](int j4, float (&v)[4]) {
        const float4 q = *(const float4*)(st + j4);
        v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
        if (j4 < j0 || j4 + 4 > j1) {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = j4 + e < j0 || j4 + e >= j1 ? inf : v[e];
        }
    };
    float m = inf, v[4];
#pragma unroll 4
    for (int j4 = j0 & ~3; j4 < j1; j4 += 4) {
        read4(j4, v);
        m = fminf(m, fminf(fminf(v[0], v[1]), fminf(v[2], v[3])));
    }
    if (t.pending) {
        t.a_next = st[j0];
        t.pending = false;
    }
    if (m < t.best) {
        int k = j1 - 1;
#pragma unroll 4
        for (int j4 = (j1 - 1) & ~3; j4 >= j0 - 3; j4 -= 4) {
            read4(j4, v);
#pragma unroll
            for (int e = 3; e >= 0; --e) k = v[e] == m ? j4 + e : k;
        }
        t.best = st[k];
        t.bidx = dc0 + k;
        t.a_prev = k > j0 ? st[k - 1] : t.last;
        t.pending = k + 1 == j1;
        if (k + 1 < j1) t.a_next = st[k + 1];
    }
    t.last = st[j1 - 1];
}

// Disparities dc0 .. dc0 + 8 KD - 1 of a tile (columns of DC staged disparities).
// Starts and ends with every warp at the same point (a __syncthreads).
template <int KD, int DC, Copy COPY, int ROWS, bool POLLS>
__device__ __forceinline__ void aggregate_chunk(Tile& t, Ring<POLLS>& ring, float* agg_out, int dc0)
{
    constexpr int NDC = 8 * KD;       // disparities of this chunk
    constexpr int PW = 32 / ROWS;     // pixels of a warp along x
    constexpr int SEGS = PW / kPX;    // groups of 8 pixels along x
    constexpr int SP = NDC + 4;       // stage pitch: 16-byte reads of 8 lanes hit 8 different bank groups
    static_assert(NDC <= DC, "a chunk lies in its columns");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rho = t.rho, NC = kTX + 2 * rho, WS = weight_stride(rho);
    const int xlo = t.x0 - rho;
    const uint32_t slot_bytes = (uint32_t)NC * DC * 4;
    float* const wbuf = t.rows + ring.S * NC * DC + warp * 4 * WS;
    const uint32_t rows_a = tc::smem_u32(t.rows);

    // rows some pixel of the warp needs (none when no pixel has its band in this chunk)
    const bool on = t.whi >= dc0 && t.wlo < dc0 + NDC;
    const int w_lo = on ? t.wy - rho : t.H, w_hi = min(t.H - 1, t.wy + ROWS - 1) + rho;
    // a chunk that no warp needs is passed over, and every one after a wait that ran out
    if (!__syncthreads_or(on && !ring.aborted())) return;
    auto load_row = [&](int r, int slot, uint32_t parity) {
        load_cost_row<DC, COPY>(ring, slot, parity, rows_a, t.vol, r, xlo, NC, dc0);
    };
    // the first S rows
    for (int i = COPY == kTma ? warp : 0; i < ring.S && t.r_lo + i <= t.r_hi; i += COPY == kTma ? kWarps : 1) {
        const int slot = ring.slot + i;
        const bool wraps = slot >= ring.S;
        load_row(t.r_lo + i, wraps ? slot - ring.S : slot, ring.parity ^ (wraps ? 1u : 0u));
    }

    // accumulating role: lane bits 0, 2, 3 = disparity group k, bits 1, 4 = pixel group
    const int k = (lane & 1) | ((lane >> 1) & 6);
    const int grow = ROWS == 2 ? (lane >> 1) & 1 : ((lane >> 1) & 1) | ((lane >> 3) & 2);
    const int gseg = ROWS == 2 ? lane >> 4 : 0;
    const int gy = t.wy + grow;
    const int wx = t.px - t.x0 - lane % PW;      // the warp's first column in the tile
    const uint32_t ca0 = rows_a + 4 * ((wx + kPX * gseg) * DC + (KD == 2 ? 2 : 4) * k);
    const uint32_t wa0 = tc::smem_u32(wbuf) + 4 * (grow * SEGS + gseg) * WS;
    // weight role: lane = pixel (lane / PW, lane % PW) of the warp
    float* const wout = wbuf + (lane / kPX) * WS + (lane % kPX) * (kPX + 1);
    const Pixel self{t.pcol, f2_pack(-8388608.f, -8388608.f),
                     f2_pack(t.neg_kr, t.neg_kr), t.px - rho, t.W};
    const bool edge = xlo < 0 || xlo + NC > t.W;

    uint64_t acc[kPX][KD / 2];
#pragma unroll
    for (int i = 0; i < kPX; ++i)
#pragma unroll
        for (int q = 0; q < KD / 2; ++q) acc[i][q] = 0ull;
    float den0 = 0.f, den1 = 0.f;

    const uint32_t* g = t.guide + (t.px - t.x0);
    for (int r = t.r_lo; r <= t.r_hi; ++r, g += NC) {
        if constexpr (COPY != kTma) {
            // refill the slot of the row before
            if (r > t.r_lo && r - 1 + ring.S <= t.r_hi) {
                const int slot = ring.slot == 0 ? ring.S - 1 : ring.slot - 1;
                const uint32_t parity = ring.slot == 0 ? ring.parity ^ 1u : ring.parity;
                if (ring.wait(ring.done + 8 * slot, parity)) load_row(r - 1 + ring.S, slot, parity ^ 1u);
            }
        }
        if (r >= w_lo && r <= w_hi) {
            const int dy = r - t.py;
            if (t.py < t.H && dy >= -rho && dy <= rho) {
                const uint64_t* sp = (const uint64_t*)(t.spatial + abs(dy) * (2 * rho + 2));
                if (edge) weight_row<true>(self, g, sp, wout, rho, den0, den1);
                else weight_row<false>(self, g, sp, wout, rho, den0, den1);
            }
            __syncwarp();
            ring.wait(ring.full + 8 * ring.slot, ring.parity);
            const int gdy = r - gy;
            if (gy < t.H && gdy >= -rho && gdy <= rho) accumulate_row<KD, DC>(acc, ca0 + ring.slot * slot_bytes, wa0, rho);
        } else {
            ring.wait(ring.full + 8 * ring.slot, ring.parity);   // a row not needed is waited for too: a warp must not count a slot's next row early
        }
        __syncwarp();
        if constexpr (COPY == kTma) {
            uint32_t done = 0;
            if (lane == 0) done = count_done(ring.done + 8 * ring.slot);
            done = __shfl_sync(0xffffffffu, done, 0);
            // the last warp to finish the row refills its slot
            if ((done & (kWarps - 1)) == kWarps - 1 && r + ring.S <= t.r_hi && !ring.aborted())
                load_row(r + ring.S, ring.slot, ring.parity ^ 1u);
        } else {
            if (lane == 0) tc::mbar_arrive(ring.done + 8 * ring.slot);
        }
        ring.next();
    }
    __syncthreads();   // every row consumed: the stage may overwrite the rows and weights
    // disparities to store and to search: none after a wait that ran out (no wait
    // follows the barrier, so every thread reads the same)
    const int nd = ring.aborted() ? 0 : min(NDC, t.d_end - dc0);

    // normalise and stage [pixel of the warp][d]
    float* const stage = t.rows + warp * 32 * SP;
    const float inv_own = 1.f / (den0 + den1);
#pragma unroll
    for (int i = 0; i < kPX; ++i) {
        const int pix = grow * PW + gseg * kPX + i;
        const float inv = __shfl_sync(0xffffffffu, inv_own, pix);
        float* st = stage + pix * SP + (KD == 2 ? 2 : 4) * k;
        float v[KD];
#pragma unroll
        for (int q = 0; q < KD / 2; ++q) {
            f2_unpack(acc[i][q], v[2 * q], v[2 * q + 1]);
            v[2 * q] *= inv;
            v[2 * q + 1] *= inv;
        }
        if (KD == 2) {
            *(float2*)st = make_float2(v[0], v[1]);
        } else {
#pragma unroll
            for (int q = 0; q < KD / 4; ++q)
                *(float4*)(st + 32 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
    }
    __syncwarp();
    if (agg_out != nullptr) {
        for (int row = 0; row < ROWS && t.wy + row < t.H; ++row) {
            const int npx = min(PW, t.W - t.x0 - wx);
            float* o = agg_out + ((size_t)(t.wy + row) * t.W + t.x0 + wx) * t.D + dc0 + lane;
            const float* st = stage + row * PW * SP + lane;
#pragma unroll 4
            for (int pix = 0; pix < npx; ++pix, o += t.D, st += SP) {
#pragma unroll
                for (int j = 0; j < NDC; j += 32)
                    if (lane + j < nd) o[j] = st[j];
            }
        }
    }
    wta_chunk(t, stage + lane * SP, dc0, max(0, t.blo - dc0), min(nd, t.bhi + 1 - dc0));
    tc::fence_proxy_async();   // the next chunk's bulk copies overwrite the stage
    __syncthreads();
}

// The ring's barriers and counters, set up once per CTA (ends with a __syncthreads).
template <Copy COPY, bool POLLS>
__device__ __forceinline__ Ring<POLLS> make_ring(void* smem, int slots, long long limit, int* err)
{
    Ring<POLLS> ring;
    ring.st = (RingState*)smem;
    ring.full = tc::smem_u32(ring.st->full);
    ring.done = tc::smem_u32(ring.st->done);
    ring.S = slots;
    ring.slot = 0;
    ring.parity = 0;
    ring.set_limit(limit);
    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxSlots; ++s) {
            tc::mbar_init(ring.full + 8 * s, COPY == kTma ? 1 : kThreads);
            if (COPY == kTma) ring.st->done[s] = 0;
            else tc::mbar_init(ring.done + 8 * s, kWarps);
        }
        ring.st->abort = 0;
        ring.st->err = err;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    return ring;
}

// One 32 x 4 tile with top-left pixel (x0, y0), disparities [d_begin, d_end)
// (the full range: 0, D); ends with a __syncthreads, so a CTA may call it for
// several tiles in a row.  band (nullable) restricts the WTA and Eq. (10) of
// each pixel to its own band [lo, hi], a sub-range of [d_begin, d_end);
// without it every pixel uses [0, D-1].  d_begin must be a multiple of 4.
// False (in every thread) when a wait ran out: nothing was stored.
template <Copy COPY, int ROWS, bool POLLS>
__device__ __forceinline__ bool aggregate_tile(const float* __restrict__ cost, const CUtensorMap* map, int ld,
                                               const uint8_t* __restrict__ guide, int H, int W, int C, int D,
                                               int rho, float neg_ks, float neg_kr, float* __restrict__ agg_out,
                                               int32_t* __restrict__ disp_int, float* __restrict__ disp_sub, int x0,
                                               int y0, void* smem, Ring<POLLS>& ring, int d_begin, int d_end,
                                               const uint32_t* __restrict__ band)
{
    constexpr int PW = 32 / ROWS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int NC = kTX + 2 * rho;
    float* const spatial = (float*)((uint8_t*)smem + kHeaderBytes);
    uint32_t* const gtile = (uint32_t*)(spatial + spatial_floats(rho));
    Tile t;
    t.vol = Volume{cost, map, ld, W, D};
    t.H = H;
    t.W = W;
    t.D = D;
    t.rho = rho;
    t.neg_kr = neg_kr;
    t.x0 = x0;
    t.y0 = y0;
    t.r_lo = max(0, y0 - rho);
    t.r_hi = min(H - 1, y0 + kTY - 1 + rho);
    t.d_end = d_end;
    t.spatial = spatial;
    t.guide = gtile;
    t.rows = (float*)((uint8_t*)smem + front_bytes(rho));
    t.wy = y0 + ROWS * (warp / (kTX / PW));
    t.px = x0 + PW * (warp % (kTX / PW)) + lane % PW;
    t.py = t.wy + lane / PW;

    for (int i = tid; i < spatial_floats(rho); i += kThreads) {
        const int dy = i / (2 * rho + 2), dx = i - dy * (2 * rho + 2) - rho;
        spatial[i] = __fmul_rn((float)(dx * dx + dy * dy), neg_ks);
    }
    // the guide window (columns outside the image: 0, their weights are 0)
    for (int c = tid & 63; c < NC; c += 64) {
        const int gx = x0 - rho + c;
        const bool in = (unsigned)gx < (unsigned)W;
        const uint8_t* src = guide + ((size_t)t.r_lo * W + (in ? gx : 0)) * C;
#pragma unroll 4
        for (int r = tid >> 6; r <= t.r_hi - t.r_lo; r += kThreads / 64)
            gtile[r * NC + c] = in ? packed_colour(src + (size_t)r * W * C, C) : 0u;
    }
    // what precedes needs only the caller's image; the cost volume is written by the
    // kernel before this one (a no-op for an ordinary launch)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    const bool valid = t.py < H && t.px < W;
    t.pcol = valid ? gtile[(t.py - t.r_lo) * NC + t.px - x0 + rho] : 0u;
    t.best = __int_as_float(0x7f800000);
    t.a_prev = t.a_next = t.last = 0.f;
    t.pending = false;
    t.blo = t.wlo = 0;
    t.bhi = t.whi = D - 1;
    if (band != nullptr) {
        // a warp skips the chunks that none of its pixels needs
        int lo = D, hi = -1;
        if (valid) {
            const uint32_t b = band[(size_t)t.py * W + t.px];
            t.blo = lo = (int)(b & 0xffffu);
            t.bhi = hi = (int)(b >> 16);
        }
        t.wlo = __reduce_min_sync(0xffffffffu, lo);
        t.whi = __reduce_max_sync(0xffffffffu, hi);
    }
    t.bidx = t.blo;

    for (int dc0 = d_begin; dc0 < d_end; dc0 += 64) {
        const int left = d_end - dc0;
        if (D > 32) {
            if (left > 32) aggregate_chunk<8, 64, COPY, ROWS>(t, ring, agg_out, dc0);
            else aggregate_chunk<4, 64, COPY, ROWS>(t, ring, agg_out, dc0);
        } else if (D > 16) {
            aggregate_chunk<4, 32, COPY, ROWS>(t, ring, agg_out, dc0);
        } else {
            aggregate_chunk<2, 16, COPY, ROWS>(t, ring, agg_out, dc0);
        }
    }
    if (ring.aborted()) {
        ring.template drain<COPY>();
        return false;
    }

    if (valid) {
        float ds = (float)t.bidx;
        if (t.bidx > t.blo && t.bidx < t.bhi) {
            const float den = 2.f * t.a_prev + 2.f * t.a_next - 4.f * t.best;
            if (den > 0.f) ds = (float)t.bidx + (t.a_prev - t.a_next) / den;
        }
        const size_t o = (size_t)t.py * W + t.px;
        if (disp_int) disp_int[o] = t.bidx;
        if (disp_sub) disp_sub[o] = ds;
    }
    __syncthreads();   // the guide window may be overwritten
    return true;
}

constexpr int kCtasPerSm = 4;

template <Copy COPY, bool POLLS>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
aggregate_f32_kernel(const __grid_constant__ CUtensorMap map, const float* __restrict__ cost, int ld,
                     const uint8_t* __restrict__ guide, int H, int W, int C, int D, int rho, float neg_ks, float neg_kr,
                     float* __restrict__ agg_out, int32_t* __restrict__ disp_int, float* __restrict__ disp_sub,
                     int slots, long long wait_cycles, int* __restrict__ err)
{
    extern __shared__ __align__(128) float4 smem_f4[];
    Ring<POLLS> ring = make_ring<COPY, POLLS>(smem_f4, slots, wait_cycles, err);
    aggregate_tile<COPY, 2>(cost, &map, ld, guide, H, W, C, D, rho, neg_ks, neg_kr, agg_out, disp_int, disp_sub,
                            blockIdx.x * kTX, blockIdx.y * kTY, smem_f4, ring, 0, D, nullptr);
}

// Band form: tile t aggregates its range tile_range[t] and each pixel takes
// its winner inside its own band.  A warp owns 8 x 4 pixels here (bands come in
// 4 x 4 blocks, and a warp computes the chunks that any of its pixels needs).
template <bool POLLS>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
aggregate_band_kernel(const __grid_constant__ CUtensorMap map, const float* __restrict__ cost, int ld,
                      const uint8_t* __restrict__ guide, int H, int W, int C, int D, int rho, float neg_ks, float neg_kr,
                      const int2* __restrict__ tile_range, const uint32_t* __restrict__ band,
                      int32_t* __restrict__ disp_int, float* __restrict__ disp_sub, int slots, long long wait_cycles,
                      int* __restrict__ err)
{
    extern __shared__ __align__(128) float4 smem_f4[];
    Ring<POLLS> ring = make_ring<kTma, POLLS>(smem_f4, slots, wait_cycles, err);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the ranges and bands come from earlier kernels
    const int2 r = tile_range[(size_t)blockIdx.y * gridDim.x + blockIdx.x];
    aggregate_tile<kTma, 4>(cost, &map, ld, guide, H, W, C, D, rho, neg_ks, neg_kr, nullptr, disp_int, disp_sub,
                            blockIdx.x * kTX, blockIdx.y * kTY, smem_f4, ring, r.x, r.y, band);
}

// Persistent form over a batch: CTAs claim (pair, tile) items from a counter;
// pairs[p].agg_off is the first item of pair p, items of a pair are its tiles
// in row-major order.  No CTA waits on another.
template <bool POLLS>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
aggregate_f32_batched_kernel(const BatchPair* __restrict__ pairs, int npairs, int nitems, int* __restrict__ counter,
                             int slots, int* __restrict__ err)
{
    extern __shared__ __align__(128) float4 smem_f4[];
    Ring<POLLS> ring = make_ring<kAsync16, POLLS>(smem_f4, slots, 0, err);
    __shared__ int item_s;
    for (;;) {
        if (threadIdx.x == 0) item_s = atomicAdd(counter, 1);
        __syncthreads();
        const int item = item_s;
        __syncthreads();
        if (item >= nitems) break;
        const int pi = find_pair(pairs, npairs, item, &BatchPair::agg_off);
        const BatchPair& bp = pairs[pi];
        const int t = item - bp.agg_off;
        const int ntx = (bp.W + kTX - 1) / kTX;
        ring.set_limit(bp.wait_cycles);
        if (!aggregate_tile<kAsync16, 2>(bp.cost, nullptr, bp.ld, bp.left, bp.H, bp.W, bp.C, bp.D, bp.radius, bp.neg_ks,
                                         bp.neg_kr, nullptr, bp.disp_int, bp.disp_sub, (t % ntx) * kTX, (t / ntx) * kTY,
                                         smem_f4, ring, 0, bp.D, nullptr))
            break;
    }
}

// Slots of the ring: as many as still leave the most CTAs per SM (at least 2).
int ring_slots(int rho, int dc)
{
    constexpr size_t kSmem = 227 * 1024, kReserved = 1024;
    auto ctas = [&](int slots) {
        const size_t n = kSmem / (smem_bytes(rho, dc, slots) + kReserved);
        return n < (size_t)kCtasPerSm ? n : (size_t)kCtasPerSm;
    };
    int slots = 2;
    while (slots < kMaxSlots && ctas(slots + 1) == ctas(2)) ++slots;
    return slots;
}

// The cost volume [H][W][ld] as a 3-D tensor (D, W, H); a box is one row of a
// tile's window.  False where the volume does not allow it.
bool encode_volume(CUtensorMap* map, const float* cost, int ld, int H, int W, int D, int rho)
{
    if (ld % 4 != 0 || (reinterpret_cast<uintptr_t>(cost) & 15) != 0) return false;
    const tca::EncodeTiledFn enc = tca::encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)W, (cuuint64_t)H};
    cuuint64_t strides[2] = {(cuuint64_t)ld * 4, (cuuint64_t)W * ld * 4};
    cuuint32_t box[3] = {(cuuint32_t)column_size(D), (cuuint32_t)(kTX + 2 * rho), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(cost), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <Copy COPY, bool POLLS>
cudaError_t launch_copy(const CUtensorMap& map, const float* cost, int ld, const uint8_t* guide, int H, int W, int C,
                        int D, int rho, float neg_ks, float neg_kr, float* agg_out, int32_t* disp_int, float* disp_sub,
                        long long wait_cycles, int* err, bool after_cost, cudaStream_t stream)
{
    const int slots = ring_slots(rho, column_size(D));
    const size_t smem = smem_bytes(rho, column_size(D), slots);
    cudaError_t e = fbs::raise_smem_limit(aggregate_f32_kernel<COPY, POLLS>, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((W + kTX - 1) / kTX, (H + kTY - 1) / kTY);
    if (after_cost)
        return fbs::launch_after(aggregate_f32_kernel<COPY, POLLS>, grid, kThreads, smem, stream, map, cost, ld, guide, H, W, C, D,
                                 rho, neg_ks, neg_kr, agg_out, disp_int, disp_sub, slots, wait_cycles, err);
    fbs::note_launch();
    aggregate_f32_kernel<COPY, POLLS><<<grid, kThreads, smem, stream>>>(
        map, cost, ld, guide, H, W, C, D, rho, neg_ks, neg_kr, agg_out, disp_int, disp_sub, slots, wait_cycles, err);
    return cudaGetLastError();
}

}  // namespace

long long wait_limit(long long wait_cycles) { return wait_cycles > 0 ? wait_cycles : tc::kWaitCycles; }
bool wait_polls(long long wait_cycles) { return wait_limit(wait_cycles) < tc::kShortWait; }

int agg_f32_tiles(int H, int W) { return ((W + kTX - 1) / kTX) * ((H + kTY - 1) / kTY); }

cudaError_t prepare_aggregate_f32_batched(int max_radius, bool polls, size_t* smem_out, int* slots_out)
{
    *slots_out = ring_slots(max_radius, 64);
    const size_t smem = smem_bytes(max_radius, 64, *slots_out);
    *smem_out = smem;
    return fbs::raise_smem_limit(polls ? aggregate_f32_batched_kernel<true> : aggregate_f32_batched_kernel<false>, (int)smem);
}

cudaError_t launch_aggregate_f32_batched(const BatchPair* pairs, int npairs, int nitems, int* counter, int grid,
                                         size_t smem, int slots, bool polls, int* err, cudaStream_t stream)
{
    fbs::note_launch();
    auto kernel = polls ? aggregate_f32_batched_kernel<true> : aggregate_f32_batched_kernel<false>;
    kernel<<<grid, kThreads, smem, stream>>>(pairs, npairs, nitems, counter, slots, err);
    return cudaGetLastError();
}

cudaError_t launch_aggregate_band(const float* cost, int ld, const uint8_t* guide, int H, int W, int C, int D,
                                  int radius, float sigma_s, float sigma_r, const int2* tile_range,
                                  const uint32_t* band, int32_t* disp_int, float* disp_sub, long long wait_cycles, int* err,
                                  cudaStream_t stream)
{
    const double log2e = 1.4426950408889634;
    const float neg_ks = (float)(-log2e / ((double)sigma_s * sigma_s));
    const float neg_kr = (float)(-log2e / ((double)sigma_r * sigma_r));
    const int slots = ring_slots(radius, column_size(D));
    const size_t smem = smem_bytes(radius, column_size(D), slots);
    CUtensorMap map;
    if (!encode_volume(&map, cost, ld, H, W, D, radius)) return cudaErrorInvalidValue;   // the context's own volume
    auto kernel = wait_polls(wait_cycles) ? aggregate_band_kernel<true> : aggregate_band_kernel<false>;
    cudaError_t e = fbs::raise_smem_limit(kernel, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((W + kTX - 1) / kTX, (H + kTY - 1) / kTY);
    return fbs::launch_after(kernel, grid, kThreads, smem, stream, map, cost, ld, guide, H, W, C, D, radius, neg_ks,
                             neg_kr, tile_range, band, disp_int, disp_sub, slots, wait_limit(wait_cycles), err);
}

cudaError_t launch_aggregate_f32(const float* cost, int ld, const uint8_t* guide, int H, int W, int C,
                                 int D, int radius, float sigma_s, float sigma_r, float* agg_out,
                                 int32_t* disp_int, float* disp_sub, long long wait_cycles, int* err, bool after_cost,
                                 cudaStream_t stream)
{
    // exp(-a/g^2) = exp2(-a * log2(e) / g^2)
    const double log2e = 1.4426950408889634;
    const float neg_ks = (float)(-log2e / ((double)sigma_s * sigma_s));
    const float neg_kr = (float)(-log2e / ((double)sigma_r * sigma_r));
    CUtensorMap map{};
    const bool tma = encode_volume(&map, cost, ld, H, W, D, radius), polls = wait_polls(wait_cycles);
    auto launch = tma ? (polls ? launch_copy<kTma, true> : launch_copy<kTma, false>)
                      : (polls ? launch_copy<kAsync4, true> : launch_copy<kAsync4, false>);
    return launch(map, cost, ld, guide, H, W, C, D, radius, neg_ks, neg_kr, agg_out, disp_int, disp_sub,
                  wait_limit(wait_cycles), err, after_cost, stream);
}

}  // namespace fbs
