// Weight-only low-bit GEMM for few rows (a serving step): Y = X v^T with X bf16
// [M][K] and v = 2 c + 1 or c from packed b-bit codes (paper Table 7's W-bit / 32
// rows, Algorithm 1 step 4 on the weights).
//
// With few rows the weights are read once and used once: expanding them to a bf16
// copy first (the path of the large problems) writes and reads 4 N K bytes to
// multiply N K b / 8 bytes of codes.  Here a warp takes the packed words straight
// from global memory to tensor-core operands in registers.  The row-fragment
// instruction (mma.sync m16n8k16) fits that: tcgen05 takes its operands from shared
// or tensor memory, one more pass over them, for a tile of 128 rows of which M are
// real; at these sizes the arithmetic is under a microsecond either way.
//
//   * K is cut into chunks of 128 codes; lane (n = lane / 4, j = lane & 3) of a warp
//     holds the 32 codes 32 j .. 32 j + 31 of weight row n: eight k16 steps of four
//     codes.  The order of K inside a chunk is free as long as both operands agree.
//   * A code becomes a bf16 by bit operations: the field n' = (code ^ half) placed in
//     the low mantissa bits of 128.0 is 128 + 2 n' + 1 (or 128 + n'), and one
//     subtraction leaves 2 c + 1 (or c) exactly: three instructions for two codes.
//     Fields come in pairs D apart (the low half-words' and the high half-words'), so
//     the operand of X pairs elements k and k + D.
//   * The warps of a block (16; 8 where a lane's sums take the registers) take the
//     chunks of the same 8 NT columns in turn and add their sums in shared memory in
//     a fixed order: the result does not depend on timing.  All of a chunk's loads
//     are issued before its arithmetic, the next chunk's weights with them.
//
// Bound: latency (one wave of blocks, four dependent round trips to memory).
// 16 x 4096 x 4096, 4-bit: 45.2 us in two passes, 5.9 here.
#include <cuda_bf16.h>

#include "dsq_gemm8_rule.h"
#include "dsq_launch.h"
#include "dsq_tc_host.h"

namespace {

template <int MT> struct Warps { static constexpr int N = MT <= 2 ? 16 : 8; };

struct WsParams {
    const uint8_t *X, *W;
    int M, N, K, pitch;           // pitch: bytes of a weight row
    int odd;                      // values 2 c + 1 (else c)
    const float *col_scale, *col_bias;
    float *Y;
};

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// G = 2 D consecutive codes (a 32-bit word of 4-, 2- or 1-bit codes, 24 bits of 3-bit
// codes) as fields: field i at bit BITS * i of the low half, field i + D of the high
template <int BITS> struct Fields {
    static constexpr int D = BITS == 3 ? 4 : 16 / BITS;
    static constexpr int GROUPS = 32 / (2 * D);       // of a lane's 32 codes
};

template <int BITS>
__device__ __forceinline__ uint32_t group_of(const uint32_t (&w)[BITS], int g)
{
    if (BITS != 3) return w[BITS == 3 ? 0 : g];
    const int bit = 24 * g, i = bit >> 5;
    const uint32_t x = __funnelshift_r(w[i], w[i + 1 < BITS ? i + 1 : i], bit & 31);
    return (x & 0xFFFu) | ((x & 0xFFF000u) << 4);
}

// fields i and i + D of a group -> bf16 pair
template <int BITS>
__device__ __forceinline__ uint32_t value_pair(uint32_t x, int i, uint32_t mask, uint32_t flip,
                                               uint32_t base, int odd)
{
    // (odd: the field goes one bit up; bit 0 of `flip` is the + 1)
    const int sh = BITS * i;
    const uint32_t y = odd ? (sh == 0 ? x << 1 : x >> (sh - 1)) : x >> sh;
    const uint32_t v = (y & mask) ^ flip;
    const __nv_bfloat162 r = __hsub2(*reinterpret_cast<const __nv_bfloat162 *>(&v),
                                     *reinterpret_cast<const __nv_bfloat162 *>(&base));
    return *reinterpret_cast<const uint32_t *>(&r);
}

template <int BITS, int MT, int NT, bool ODD>
__global__ void __launch_bounds__(Warps<MT>::N * 32)
wgemm_small_kernel(const WsParams p)
{
    constexpr int D = Fields<BITS>::D, GROUPS = Fields<BITS>::GROUPS, WARPS = Warps<MT>::N;
    constexpr bool ALL = MT <= 2;              // X of a whole chunk in registers
    constexpr int XG = ALL ? GROUPS : 1;
    constexpr int PARTS = MT * NT > 8 ? 4 : 8;
    __shared__ float part[PARTS][MT * NT][32][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = lane >> 2, j = lane & 3;
    const int n0 = blockIdx.x * 8 * NT, m0 = blockIdx.y * 16 * MT;
    constexpr uint32_t HALF = 1u << (BITS - 1), F = (1u << BITS) - 1u;
    constexpr uint32_t MASK = (ODD ? F << 1 : F) * 0x00010001u;
    constexpr uint32_t FLIP = (0x4300u ^ (ODD ? (HALF << 1) | 1u : HALF)) * 0x00010001u;
    // 128 + 2 HALF or 128 + HALF as bf16 (ulp 1 between 128 and 256)
    constexpr uint32_t BASE = (0x4300u + (ODD ? 2 * HALF : HALF)) * 0x00010001u;
    const int chunks = (p.K + 127) / 128;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    float acc[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[m][t][i] = 0.f;

    uint32_t wn[NT][BITS];
    auto load_w = [&](int c) {
        const int at = c * 16 * BITS + 4 * BITS * j;          // this lane's 4 * BITS bytes
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int row = n0 + 8 * t + n;
            const uint8_t *src = p.W + (int64_t)row * p.pitch + at;
            const bool in = row < p.N && c < chunks;
            if (BITS == 4) {
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (in && at < p.pitch) v = __ldg(reinterpret_cast<const uint4 *>(src));
                wn[t][0] = v.x; wn[t][1 % BITS] = v.y; wn[t][2 % BITS] = v.z; wn[t][3 % BITS] = v.w;
            } else {
#pragma unroll
                for (int i = 0; i < BITS; ++i) {
                    wn[t][i] = 0u;
                    if (in && at + 4 * i < p.pitch)
                        wn[t][i] = __ldg(reinterpret_cast<const uint32_t *>(src) + i);
                }
            }
        }
    };
    // X: 2 D elements of rows n and n + 8 of every 16-row tile (K is a multiple of 8:
    // elements past it are zero)
    uint32_t xa[XG][MT][2][D];
    auto load_x = [&](int k0, int g, int to) {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = m0 + 16 * m + 8 * h + n;
                const uint8_t *src = p.X + ((int64_t)row * p.K + k0 + 2 * D * g) * 2;
#pragma unroll
                for (int q = 0; q < D / 4; ++q) {
                    uint4 v = make_uint4(0u, 0u, 0u, 0u);
                    if (row < p.M && k0 + 2 * D * g + 8 * q < p.K)
                        v = __ldg(reinterpret_cast<const uint4 *>(src) + q);
                    xa[to][m][h][4 * q] = v.x; xa[to][m][h][4 * q + 1] = v.y;
                    xa[to][m][h][4 * q + 2] = v.z; xa[to][m][h][4 * q + 3] = v.w;
                }
            }
    };
    load_w(warp);
    // A thread's outputs lie in one column.  Its scale and bias come with the first loads where the
    // loop leaves registers for them (asked for behind the last barrier, in a graph: 48x1000x3000
    // 3-bit 9.0 us, so 7.9; 8x1024x1024 4-bit 2.3 / 2.1; 17 to 32 rows, blocks of
    // 32 columns and 16 rows at 3 bits are slower with them: 24x600x5000 2-bit 7.5 / 8.3, 8x1024x1024 3-bit
    // 2.55 / 2.68).
    constexpr bool FIRST = (MT == 4 && NT == 2) || (MT == 1 && NT == 2 && BITS != 3);
    float cs = 0.f, cb = 0.f;
    if (FIRST) {
        static_assert(WARPS * 32 % (8 * NT) == 0, "one column a thread");
        const int at = n0 + threadIdx.x % (8 * NT);
        if (at < p.N) {
            cs = __ldg(p.col_scale + at);
            if (p.col_bias) cb = __ldg(p.col_bias + at);
        }
    }
#pragma unroll 1
    for (int c = warp; c < chunks; c += WARPS) {
        uint32_t w[NT][BITS];
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int i = 0; i < BITS; ++i) w[t][i] = wn[t][i];
        const int k0 = c * 128 + 32 * j;                      // this lane's 32 elements
        if (ALL) {
#pragma unroll
            for (int g = 0; g < GROUPS; ++g) load_x(k0, g, g);
        }
        load_w(c + WARPS);
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) {
            uint32_t x[NT];
#pragma unroll
            for (int t = 0; t < NT; ++t) x[t] = group_of<BITS>(w[t], g);
            const int xg = ALL ? g : 0;
            if (!ALL) load_x(k0, g, 0);
#pragma unroll
            for (int i = 0; i < D; i += 2) {                  // one k16 step: pairs i and i + 1
                uint32_t a[MT][4];
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        // elements (i, i + D) and (i + 1, i + 1 + D)
                        a[m][h] = __byte_perm(xa[xg][m][h][i / 2], xa[xg][m][h][i / 2 + D / 2], 0x5410);
                        a[m][h + 2] = __byte_perm(xa[xg][m][h][i / 2], xa[xg][m][h][i / 2 + D / 2], 0x7632);
                    }
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    const uint32_t b0 = value_pair<BITS>(x[t], i, MASK, FLIP, BASE, ODD);
                    const uint32_t b1 = value_pair<BITS>(x[t], i + 1, MASK, FLIP, BASE, ODD);
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_bf16(acc[m][t], a[m], b0, b1);
                }
            }
        }
    }
    // the warps' sums, added in a fixed order: those from PARTS on into the ones before, those in turn
    auto put = [&](int at) {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int t = 0; t < NT; ++t)
                *reinterpret_cast<float4 *>(part[at][m * NT + t][lane]) =
                    make_float4(acc[m][t][0], acc[m][t][1], acc[m][t][2], acc[m][t][3]);
    };
    static_assert(WARPS <= 2 * PARTS, "two rounds of sums");
    if (WARPS > PARTS) {
        if (warp >= PARTS) put(warp - PARTS);
        __syncthreads();
        if (warp < PARTS)
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int t = 0; t < NT; ++t)
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[m][t][i] += part[warp][m * NT + t][lane][i];
    }
    if (warp < PARTS) put(warp);
    __syncthreads();
    for (int e = threadIdx.x; e < MT * NT * 128; e += WARPS * 32) {
        // element e of the tile in row-major order: row 16 MT, column 8 NT
        const int col = e % (8 * NT), row = e / (8 * NT);
        const int t = col >> 3, m = row >> 4;
        const int l = (row & 7) * 4 + ((col & 7) >> 1), i = 2 * ((row >> 3) & 1) + (col & 1);
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < PARTS; ++w) s += part[w][m * NT + t][l][i];
        if (m0 + row < p.M && n0 + col < p.N)
            p.Y[(int64_t)(m0 + row) * p.N + n0 + col] =
                FIRST ? __fmaf_rn(s, cs, cb)
                      : __fmaf_rn(s, __ldg(p.col_scale + n0 + col), p.col_bias ? __ldg(p.col_bias + n0 + col) : 0.f);
    }
}

template <int BITS, int MT, int NT>
int launch(const WsParams &p, cudaStream_t s)
{
    const dim3 grid((p.N + 8 * NT - 1) / (8 * NT), (p.M + 16 * MT - 1) / (16 * MT));
    return dsq_launch(p.odd ? wgemm_small_kernel<BITS, MT, NT, true> : wgemm_small_kernel<BITS, MT, NT, false>,
                      grid, dim3(Warps<MT>::N * 32), 0, s, dsq_launch_hooks().pdl, 0, p);
}

template <int BITS>
int pick(const WsParams &p, cudaStream_t s)
{
    // Columns per block: 16 while those blocks are one to an SM at most (one fits: its
    // registers), 32 beyond, where a second wave costs more than the wider block.  4-bit,
    // K = 4096, us with 16 / 32 columns: N = 2048 (128 blocks of 16) 1 row 3.6 / 5.2, 16 rows
    // 4.6 / 5.7, 32 rows 7.2 / 8.3; N = 2400 (150) 5.3 / 5.2, 7.0 / 5.9, 12.7 / 8.5; N = 4096
    // 5.5 / 5.2, 7.2 / 5.9, 13.2 / 8.5.
    const int sms = dsq_sm_count() > 0 ? dsq_sm_count() : 148;
    const bool wide = p.N > 16 * sms;
    if (p.M <= 16) return wide ? launch<BITS, 1, 4>(p, s) : launch<BITS, 1, 2>(p, s);
    if (p.M <= 32) return wide ? launch<BITS, 2, 4>(p, s) : launch<BITS, 2, 2>(p, s);
    return dsq_wgemm_small_columns(p.M, p.N, sms) == 32 ? launch<BITS, 4, 4>(p, s) : launch<BITS, 4, 2>(p, s);
}

}  // namespace

int dsq_wgemm_small(const void *X, const void *W, int64_t M, int64_t N, int64_t K, int bits, int odd,
                    const float *col_scale, const float *col_bias, float *Y, cudaStream_t stream)
{
    WsParams p;
    p.X = (const uint8_t *)X; p.W = (const uint8_t *)W;
    p.M = (int)M; p.N = (int)N; p.K = (int)K;
    p.pitch = (int)dsq_row_pitch(K, bits);
    p.odd = odd;
    p.col_scale = col_scale; p.col_bias = col_bias;
    p.Y = Y;
    switch (bits) {
    case 1: return pick<1>(p, stream);
    case 2: return pick<2>(p, stream);
    case 3: return pick<3>(p, stream);
    default: return pick<4>(p, stream);
    }
}
