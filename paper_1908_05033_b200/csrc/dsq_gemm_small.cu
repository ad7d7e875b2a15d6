// Low-bit GEMMs with little work (Algorithm 1 step 5 on codes): C = A B^T, A [M][K] signed codes,
// B [N][K] unsigned, laid out for latency as the little-work convolution is (dsq_conv_small.cu).
//
// A 512^3 problem is 0.13 G multiply-accumulates: a tenth of a microsecond at the tensor cores'
// rate, and 6 to 9 us in the tcgen05 kernels, which start 23 warps (or two launches), set up tensor
// memory and barriers, hand every K step through shared memory and drain one or a few large
// tiles.  Here
//   * a block of 4 or 8 warps makes 16 MT rows x 32 columns (MT = 1, 2), its warps splitting K and adding
//     their sums in shared memory in a fixed order;
//   * every lane takes its packed words straight from global memory to the fragments of mma.sync
//     m16n8k32 (s8 x u8) in registers, the next chunk's before this one's arithmetic.
// Microseconds in a graph, the faster of the others / this: 4-bit 256^3 3.3 / 1.6, 512^3 3.9 / 2.3,
// 200x200x4000 9.6 / 3.1; 2-bit 512^3 4.4 / 2.3; 3-bit 5.7 / 3.4, but 1024^3 7.6 / 15.4.
// Bound: two to four dependent round trips to memory, and beyond about 0.5 G
// multiply-accumulates the expansion of both operands once per tile, which is why larger
// problems go elsewhere (dsq_gemm8_rule.h).
#include "dsq_fragments.cuh"
#include "dsq_gemm8_rule.h"
#include "dsq_tc_host.h"

namespace {

constexpr int GS_NT = 4;                              // column tiles of 8
constexpr int GS_MAX_WARPS = 8;

struct GsParams {
    const uint8_t *A, *B;
    int M, N, pitch, units;                           // units: of a row
    int shift, wide;                                  // wide: column pairs are whole 8-byte words
    int32_t *C_i32;
    const float *row_scale;
    float *D_f32;
};

// signed rows times unsigned columns
__device__ __forceinline__ void mma_s8u8(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.u8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int BITS, int MT>
__global__ void __launch_bounds__(GS_MAX_WARPS * 32, 1) gemm_small_kernel(const GsParams p)
{
    constexpr int WORDS = Unit<BITS>::WORDS, UNIT_BYTES = 4 * WORDS, NT = GS_NT;
    extern __shared__ int4 part[];                    // [warp][MT * NT][lane]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int g = lane >> 2, j = lane & 3;
    const int n0 = blockIdx.x * 8 * NT, m0 = blockIdx.y * 16 * MT;
    int u = 4 * warp + j;                             // this lane's unit of the warp's chunk
    uint32_t an[MT][2][WORDS], bn[NT][WORDS];
    auto load = [&]() {
        const int at = u * UNIT_BYTES;
        const bool in = u < p.units;
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = m0 + 16 * m + 8 * h + g;
                load_unit<BITS>(p.A + (int64_t)row * p.pitch + at, in && row < p.M, p.pitch - at, an[m][h]);
            }
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int col = n0 + 8 * t + g;
            load_unit<BITS>(p.B + (int64_t)col * p.pitch + at, in && col < p.N, p.pitch - at, bn[t]);
        }
    };
    grid_dependency_wait();
    grid_launch_dependents();
    load();
    int acc[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[m][t][i] = 0;
#pragma unroll 1
    while (u - j < p.units) {
        uint32_t av[MT][2][WORDS], bv[NT][WORDS];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < WORDS; ++i) av[m][h][i] = an[m][h][i];
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int i = 0; i < WORDS; ++i) bv[t][i] = bn[t][i];
        u += 4 * warps;
        load();
#pragma unroll
        for (int q = 0; q < Unit<BITS>::BYTE_WORDS; q += 2) {
            uint32_t a[MT][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    a[m][h] = byte_word<BITS, true>(av[m][h], q, 0u);
                    a[m][h + 2] = byte_word<BITS, true>(av[m][h], q + 1, 0u);
                }
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const uint32_t b0 = byte_word<BITS, false>(bv[t], q, 0u);
                const uint32_t b1 = byte_word<BITS, false>(bv[t], q + 1, 0u);
#pragma unroll
                for (int m = 0; m < MT; ++m) mma_s8u8(acc[m][t], a[m], b0, b1);
            }
        }
    }
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int t = 0; t < NT; ++t)
            part[(warp * MT * NT + m * NT + t) * 32 + lane] =
                make_int4(acc[m][t][0], acc[m][t][1], acc[m][t][2], acc[m][t][3]);
    __syncthreads();
    // the warps' sums and the outputs, a thread one fragment of one lane: rows r and r + 8,
    // columns c and c + 1
    for (int i = threadIdx.x; i < MT * NT * 32; i += blockDim.x) {
        const int m = i / (NT * 32), t = (i >> 5) & (NT - 1);
        const int row = m0 + 16 * m + g, col = n0 + 8 * t + 2 * j;   // (i & 31 is the lane)
        int4 s = part[i];
#pragma unroll 4
        for (int k = 1; k < warps; ++k) {
            const int4 x = part[k * (MT * NT * 32) + i];
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
        const int v[2][2] = {{s.x >> p.shift, s.y >> p.shift}, {s.z >> p.shift, s.w >> p.shift}};
        if (col >= p.N) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = row + 8 * h;
            if (r >= p.M) continue;
            const int64_t at = (int64_t)r * p.N + col;
            if (p.C_i32) {
                if (p.wide) *reinterpret_cast<int2 *>(p.C_i32 + at) = make_int2(v[h][0], v[h][1]);
                else {
                    p.C_i32[at] = v[h][0];
                    if (col + 1 < p.N) p.C_i32[at + 1] = v[h][1];
                }
            }
            if (p.D_f32) {
                const float rs = __ldg(p.row_scale + r);
                const float y0 = __fmul_rn((float)v[h][0], rs), y1 = __fmul_rn((float)v[h][1], rs);
                if (p.wide) *reinterpret_cast<float2 *>(p.D_f32 + at) = make_float2(y0, y1);
                else {
                    p.D_f32[at] = y0;
                    if (col + 1 < p.N) p.D_f32[at + 1] = y1;
                }
            }
        }
    }
}

template <int BITS, int MT>
int launch(const GsParams &p, int warps, cudaStream_t s)
{
    const size_t smem = (size_t)warps * MT * GS_NT * 32 * 16;
    static std::atomic<unsigned long long> configured{0ull};
    const int st = dsq_allow_smem((const void *)gemm_small_kernel<BITS, MT>, GS_MAX_WARPS * MT * GS_NT * 512, &configured);
    if (st) return st;
    return dsq_launch(gemm_small_kernel<BITS, MT>,
                      dim3((p.N + 8 * GS_NT - 1) / (8 * GS_NT), (p.M + 16 * MT - 1) / (16 * MT)),
                      dim3(32 * warps), smem, s, dsq_launch_hooks().pdl, 0, p);
}

template <int BITS>
int pick(const GsParams &p, const DsqGemmSmallTile &t, cudaStream_t s)
{
    return t.mt == 2 ? launch<BITS, 2>(p, t.warps, s) : launch<BITS, 1>(p, t.warps, s);
}

}  // namespace

int dsq_gemm_small(const void *A_codes, const void *B_codes, int64_t M, int64_t N, int64_t K, int bits,
                   int32_t *C_i32, const float *row_scale, float *D_f32, cudaStream_t stream)
{
    GsParams p = {};
    p.A = (const uint8_t *)A_codes;
    p.B = (const uint8_t *)B_codes;
    p.M = (int)M; p.N = (int)N;
    p.pitch = (int)dsq_row_pitch(K, bits);
    p.units = bits == 3 ? (int)((K + 31) / 32) : p.pitch / 16;
    p.shift = 8 - bits;
    p.wide = N % 2 == 0;                               // (outputs are 16-byte aligned)
    p.C_i32 = C_i32; p.row_scale = row_scale; p.D_f32 = D_f32;
    const DsqGemmSmallTile t = dsq_gemm_small_tile(M, N, p.units, bits, (C_i32 ? 1 : 0) + (D_f32 ? 1 : 0),
                                                   dsq_sm_count() > 0 ? dsq_sm_count() : 148);
    switch (bits) {
    case 2: return pick<2>(p, t, stream);
    case 3: return pick<3>(p, t, stream);
    default: return pick<4>(p, t, stream);
    }
}
