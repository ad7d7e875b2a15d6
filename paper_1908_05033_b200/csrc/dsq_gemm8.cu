// Large low-bit GEMMs in two passes (paper Sec. 3.5: the quantised layer as a
// GEMM over codes; Algorithm 1 step 5 on codes).
//
// The fused kernel (dsq_tc.cu) expands the packed codes of BOTH operands to
// 8-bit lanes again for every output tile: a 4096^3 problem expands each A row
// 16 times and each B row 16 times, and that expansion (shared-memory
// bandwidth, cluster-scope hand-over of the expanded halves) is what bounds it.
// Here every row is expanded ONCE:
//   pass 1  expand_rows_kernel: packed codes -> int8 rows in a scratch area
//           the caller provides (M*Kp + N*Kp bytes, Kp = K rounded up to 16;
//           HBM / L2-bound, a few microseconds); codes of 1 to 3 bits -> 4-bit
//           floating point (expand_rows_f4_kernel), half of that;
//   pass 2  gemm8_kernel: a GEMM whose operands go from that scratch straight into
//           swizzled shared memory by TMA - no thread touches an operand byte.
//           CTA pairs on tiles of 256 rows and 64 to 256 columns (tcgen05.mma
//           cta_group::2, kind::i8 or kind::mxf4, both operands through
//           shared-memory descriptors), a ring of six or more stages per CTA,
//           and TWO accumulators in tensor memory, so the epilogue of a tile (eight
//           warps per CTA) overlaps the next tile's instructions.
// The scratch for 4096^3 is 33.5 MB and stays in the 126 MB L2 between the
// passes.
//
// Every mbarrier wait is bounded (see dsq_tc_common.cuh).
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>

#include "dsq_common.cuh"
#include "dsq_gemm8_rule.h"
#include "dsq_tc_common.cuh"
#include "dsq_tc_host.h"

namespace {

enum G8Kind { G8_I8, G8_BF16, G8_F4 };       // operands: int8, bf16, 4-bit floating point
constexpr int G8_ROWS = 128;                 // A rows per CTA and stage
constexpr int G8_BM = DSQ_G8_BM;             // tile height of a pair
constexpr int G8_KB = 128;                   // bytes of K per stage
constexpr int G8_OP_BYTES = G8_ROWS * G8_KB;             // A of a stage: 16 KB
constexpr int G8_MAX_STAGES = 12;
// tensor-memory columns of an accumulator, which are the widest tile; behind the two
// accumulators of 4-bit operands lie the block scales
template <int KIND> constexpr int g8_acc() { return KIND == G8_F4 ? 240 : 256; }
constexpr int G8_F4_SF = 480;
constexpr int G8_WARP_TMA = 0, G8_WARP_MMA = 1, G8_WARP_TMEM = 2, G8_WARP_E0 = 4;
constexpr int G8_E_WARPS = 8;                // per CTA: two per tensor-memory lane quarter
constexpr int G8_THREADS = 32 * (G8_WARP_E0 + G8_E_WARPS);
constexpr int G8_BARS = 2 * G8_MAX_STAGES + 4 + 1;
// A block of the next expansion has room beside a CTA: 1 KB of an SM's 228 is the system's for
// each, and the CTA leaves 64 registers a thread for it.  The expansions are bound to 32, eight blocks an
// SM, which is what they take; the one that also sums rows of 3-bit codes takes 39 and is left unbound: with 32 and with
// 48 some problems gain 3 to 6 % and others lose 2 to 4 (us with 32 / 39 / 48: 400x2000x4000 13.4 / 12.8 / 12.2,
// 3394x232x1376 9.0 / 8.9 / 9.2, 1500x1304x1033 9.5 / 9.2 / 9.0, 3001x2001x700 15.0 / 15.5 / 15.5).
constexpr int G8_SMEM = 226 * 1024, G8_REGS = 128;
constexpr int EX_THREADS = 256, EX_BLOCKS = 8, EX_REGS = 64;
static_assert(G8_THREADS * G8_REGS + EX_THREADS * EX_REGS <= 65536, "a CTA and a block of the next expansion on an SM");
constexpr int G8_TAIL = 8 * G8_BARS + 24;    // barriers, tensor-memory slot, abort flag
constexpr int G8_STAGING = G8_E_WARPS * 32 * 32 * 4;     // a 32 x 32 block per epilogue warp
constexpr int G8_EXCHANGE = 64 * 1024;       // sums of the other pair, at most
static_assert(G8_TAIL % 128 == 0, "the staging blocks are 128-byte aligned");

struct G8Params {
    int M, N;
    int m_tiles, n_tiles, kblocks;
    int BN;                  // tile width (both CTAs' B halves): a multiple of 32
    int stages, stage_bytes; // A (16 KB), then BN / 2 rows of B
    int vec;                 // N is a multiple of 8: 32-byte stores
    uint32_t idesc;          // instruction descriptor (operand types, M = 256, N = BN)
    // integer problems: C = acc, D = (float)acc * row_scale[m]
    int32_t *C_i32;
    const float *row_scale;
    float *D_f32;
    const int32_t *sums;     // nullable: [parts][M], C = acc + 4 x their sum (expand_rows_f4_kernel<3>)
    int parts;
    // floating-point problems: Y = fma(acc, col_scale[n], col_bias[n])
    const float *col_scale;
    const float *col_bias;   // nullable
    float *Y_f32;
    int *ws;
    unsigned long long wait_ns;
};

// ---------------------------------------------------------------------------
// pass 1: packed codes -> int8 or bf16
// ---------------------------------------------------------------------------
// bytes (each < 2^BITS) -> two's-complement int8 of the BITS-bit signed code
template <int BITS>
__device__ __forceinline__ uint32_t sign_extend_bytes(uint32_t x)
{
    constexpr uint32_t HALF = 0x01010101u * (1u << (BITS - 1));
    // per byte (x ^ half) - half without borrows between bytes
    return (((x ^ HALF) | 0x80808080u) - HALF) ^ 0x80808080u;
}

// Work item of every expansion: one 16-byte chunk of an output row (16 int8 or 8
// bf16 values).  A warp's lanes take consecutive chunks of a row, so that it writes
// 512 contiguous bytes (with 64 bytes a thread every store touched half sectors all
// over, and the L2 took each sector twice); a thread does the same chunk of four
// rows, their loads first.
//
// Launched dependently, as every kernel behind another of the library is: the first blocks
// are on the SMs, beside the kernel ahead, when that ends (2500x1111x1777, 3-bit, among other
// passes 14.35 -> 13.1 us, 2048x4096x4096 weight-only 69.2 -> 68.5; 4096^3 is bound by power).
constexpr int EX_ROWS = 4;

// `BITS`-bit codes at bit 0 of a word, ascending -> one code per byte, four a word
template <int BITS>
__device__ __forceinline__ void spread_bytes(const uint2 v, uint32_t (&o)[4])
{
    if (BITS == 4) {
        const uint32_t w[2] = {v.x, v.y};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t lo = w[h] & 0x0F0F0F0Fu, hi = (w[h] >> 4) & 0x0F0F0F0Fu;
            o[2 * h] = __byte_perm(lo, hi, 0x5140);       // codes 0..3 of the word
            o[2 * h + 1] = __byte_perm(lo, hi, 0x7362);   // codes 4..7
        }
    } else if (BITS == 3) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t x = __funnelshift_r(v.x, v.y, 12 * j) >> (j == 3 ? 4 : 0);
            const uint32_t y = j == 3 ? v.y >> 4 : x;     // bits 12 j .. 12 j + 11
            o[j] = (y & 7u) | ((y & 0x38u) << 5) | ((y & 0x1C0u) << 10) | ((y & 0xE00u) << 15);
        }
    } else if (BITS == 2) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t x = (v.x >> (8 * j)) & 0xFFu;  // four codes
            o[j] = (x | (x << 6) | (x << 12) | (x << 18)) & 0x03030303u;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            o[j] = (((v.x >> (4 * j)) & 0xFu) * 0x00204081u) & 0x01010101u;
    }
}

// the 2 BITS bytes of chunk c of a packed row (3-bit chunks start at any even byte:
// the two or three aligned words they lie in, as far as the row goes)
template <int BITS>
__device__ __forceinline__ uint2 load_chunk(const uint8_t *row, int c, int pitch)
{
    if (BITS == 4) return __ldg(reinterpret_cast<const uint2 *>(row) + c);
    if (BITS == 2) return make_uint2(__ldg(reinterpret_cast<const uint32_t *>(row) + c), 0u);
    if (BITS == 1) return make_uint2(__ldg(reinterpret_cast<const uint16_t *>(row) + c), 0u);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(row);
    const int i = (6 * c) >> 2, last = pitch / 4 - 1, sh = 8 * ((6 * c) & 3);
    const uint32_t a = __ldg(w + i), b = __ldg(w + min(i + 1, last));
    return make_uint2(__funnelshift_r(a, b, sh), b >> sh);
}

// Integer operands: rows of A then rows of B.  A's codes are signed, B's unsigned
// (BITS = 1: both -1 / +1, positions past K 0 so that a row's tail adds nothing;
// elsewhere the codes past K are spare bits of the packed row: zero).
template <int BITS>
__global__ void __launch_bounds__(EX_THREADS, EX_BLOCKS)
expand_rows_kernel(const uint8_t *__restrict__ A, const uint8_t *__restrict__ B, int M, int N, int K,
                   int pitch_in, int pitch_out, uint8_t *__restrict__ A8, uint8_t *__restrict__ B8)
{
    grid_dependency_wait();
    // lets the second pass (queued behind with programmatic dependent launch) set
    // itself up while this grid runs; it waits for this grid before its first copy
    grid_launch_dependents();
    const int c = blockIdx.x * EX_THREADS + threadIdx.x;
    if (16 * c >= pitch_out) return;
    for (int r0 = blockIdx.y * EX_ROWS; r0 < M + N; r0 += gridDim.y * EX_ROWS) {
        uint2 v[EX_ROWS];
#pragma unroll
        for (int i = 0; i < EX_ROWS; ++i) {
            const int r = min(r0 + i, M + N - 1);
            v[i] = load_chunk<BITS>(r < M ? A + (int64_t)r * pitch_in : B + (int64_t)(r - M) * pitch_in,
                                    c, pitch_in);
        }
#pragma unroll
        for (int i = 0; i < EX_ROWS; ++i) {
            const int r = r0 + i;
            if (r >= M + N) break;
            uint32_t o[4];
            spread_bytes<BITS>(v[i], o);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (BITS == 1) {
                    // 2 x - 1 per byte
                    o[j] = (((o[j] << 1) | 0x80808080u) - 0x01010101u) ^ 0x80808080u;
                    const int left = K - (16 * c + 4 * j);
                    if (left < 4) o[j] = left <= 0 ? 0u : (o[j] & (0xFFFFFFFFu >> (8 * (4 - left))));
                } else if (r < M) {
                    o[j] = sign_extend_bytes<BITS>(o[j]);
                }
            }
            uint8_t *dst = r < M ? A8 + (int64_t)r * pitch_out : B8 + (int64_t)(r - M) * pitch_out;
            *reinterpret_cast<uint4 *>(dst + 16 * c) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}

// Eight 3-bit codes (bits 0 .. 23) -> one in the low three bits of every four; the fourth is
// anything.
__device__ __forceinline__ uint32_t spread_nibbles(uint32_t x)
{
    const uint32_t y = (x & 0x0000FFFFu) | ((x << 4) & 0xFFFF0000u);
    const uint32_t z = (y & 0x00FF00FFu) | ((y << 2) & 0xFF00FF00u);
    return (z & 0x0F0F0F0Fu) | ((z << 1) & 0xF0F0F0F0u);
}
// sum of the eight four-bit fields
__device__ __forceinline__ int sum_nibbles(uint32_t x)
{
    return (int)__dp4a((x & 0x0F0F0F0Fu) + ((x >> 4) & 0x0F0F0F0Fu), 0x01010101u, 0u);
}

// Integer operands of 1 to 3 bits as 4-bit floating point (E2M1 in steps of 1/2, as
// expand_word_f4; block scales of 2 make the products whole numbers): a chunk of 16 output
// bytes is 32 values, in the order in which a shift and a mask find them (the same for
// both operands).  A 2-bit signed code -2 .. 1 is 1010, 1001, 0000, 0001, an unsigned one
// its own pattern; a bit is 0001 (+1) or 1001 (-1), past K 0.
// 3 bits: E2M1 has the whole numbers -4 .. 4, so A's codes -4 .. 3 are exact, and B's go less
// 4: a (q - 4) summed is the result less 4 sum a.  The sums of A's rows are kept for the
// second pass, one for every 1024 codes (`sums`: [part][M]).
template <int BITS>
__global__ void __launch_bounds__(EX_THREADS, BITS == 3 ? 0 : EX_BLOCKS)
expand_rows_f4_kernel(const uint8_t *__restrict__ A, const uint8_t *__restrict__ B, int M, int N, int K,
                      int pitch_in, int pitch_out, uint8_t *__restrict__ A4, uint8_t *__restrict__ B4,
                      int32_t *__restrict__ sums)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const int c = blockIdx.x * EX_THREADS + threadIdx.x;
    const bool inside = 16 * c < pitch_out;
    if (BITS == 3 ? 16 * (c & ~31) >= pitch_out : !inside) return;    // (3 bits: warps as a whole)
    constexpr int WORDS = BITS == 3 ? 3 : BITS == 2 ? 2 : 1;
    for (int r0 = blockIdx.y * EX_ROWS; r0 < M + N; r0 += gridDim.y * EX_ROWS) {
        uint32_t v[EX_ROWS][WORDS];
#pragma unroll
        for (int i = 0; i < EX_ROWS; ++i) {
            const int r = min(r0 + i, M + N - 1);
            const uint8_t *row = r < M ? A + (int64_t)r * pitch_in : B + (int64_t)(r - M) * pitch_in;
            if (BITS == 3) {
                // (a row may end inside its last chunk)
#pragma unroll
                for (int l = 0; l < WORDS; ++l)
                    v[i][l] = 4 * (3 * c + l) < pitch_in ? __ldg(reinterpret_cast<const uint32_t *>(row) + 3 * c + l)
                                                         : 0u;
            } else if (BITS == 2) {
                const uint2 t = __ldg(reinterpret_cast<const uint2 *>(row) + c);
                v[i][0] = t.x;
                v[i][WORDS - 1] = t.y;
            } else v[i][0] = __ldg(reinterpret_cast<const uint32_t *>(row) + c);
        }
#pragma unroll
        for (int i = 0; i < EX_ROWS; ++i) {
            const int r = r0 + i;
            if (r >= M + N) break;
            uint32_t o[4], low = 0u, neg = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (BITS == 3) {
                    const uint32_t lo = j == 0 ? 0u : v[i][j - 1], hi = j == 3 ? 0u : v[i][j];
                    const uint32_t f = spread_nibbles(j == 0 ? hi : __funnelshift_r(lo, hi, 32 - 8 * j)) ^
                                       (r < M ? 0u : 0x44444444u);
                    // -4 + l is 12 - l
                    const uint32_t l = f & 0x33333333u, s = f & 0x44444444u;
                    o[j] = (l ^ ((s >> 2) | (s >> 1))) + ((s >> 2) | (s << 1));
                    low += l;
                    neg += s >> 2;
                } else if (BITS == 2) {
                    const uint32_t x = ((j < 2 ? v[i][0] : v[i][WORDS - 1]) >> (2 * (j & 1))) & 0x33333333u;
                    const uint32_t hi = x & 0x22222222u, lo = x & 0x11111111u;
                    o[j] = r < M ? (hi << 2) | (hi & ~(lo << 1)) | lo : x;
                } else {
                    const int left = K - 32 * c;
                    const uint32_t in = left >= 32 ? 0xFFFFFFFFu : (1u << left) - 1u;
                    const uint32_t on = (in >> j) & 0x11111111u;
                    o[j] = ((on & ~(v[i][0] >> j)) << 3) | on;
                }
            }
            if (BITS == 3 && r < M) {
                const int sum = __reduce_add_sync(0xffffffffu, sum_nibbles(low) - 4 * sum_nibbles(neg));
                if ((threadIdx.x & 31) == 0) sums[(int64_t)(c >> 5) * M + r] = sum;
            }
            uint8_t *dst = r < M ? A4 + (int64_t)r * pitch_out : B4 + (int64_t)(r - M) * pitch_out;
            if (BITS != 3 || inside) *reinterpret_cast<uint4 *>(dst + 16 * c) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}

// Weight codes -> bf16: value 2 c + 1 (grid Delta (c + 1/2), `odd`) or c, c the
// signed BITS-bit code; K is a multiple of 8, a chunk of 8 values lies inside the
// row.  By bit operations: the field (code ^ half) in the low mantissa bits of
// 128.0 is 128 + field (128 + 2 field + 1), one subtraction leaves the value.
template <int BITS>
__global__ void __launch_bounds__(EX_THREADS, EX_BLOCKS)
expand_w_bf16_kernel(const uint8_t *__restrict__ W, int N, int K, int pitch_in, int pitch_out, int odd,
                     uint8_t *__restrict__ W16)
{
    grid_dependency_wait();
    grid_launch_dependents();
    constexpr uint32_t F = (1u << BITS) - 1u, HALF = 1u << (BITS - 1);
    const int c = blockIdx.x * EX_THREADS + threadIdx.x;
    if (8 * c >= K) return;
    const uint32_t flip = (0x4300u ^ (odd ? (HALF << 1) | 1u : HALF)) * 0x00010001u;
    const uint32_t base = (0x4300u + (odd ? 2 * HALF : HALF)) * 0x00010001u;
    const uint32_t mask = (odd ? F << 1 : F) * 0x00010001u;
    for (int r0 = blockIdx.y * EX_ROWS; r0 < N; r0 += gridDim.y * EX_ROWS) {
        uint32_t v[EX_ROWS];
#pragma unroll
        for (int i = 0; i < EX_ROWS; ++i) {
            const uint8_t *row = W + (int64_t)min(r0 + i, N - 1) * pitch_in;
            // eight codes: BITS bytes
            if (BITS == 4) v[i] = __ldg(reinterpret_cast<const uint32_t *>(row) + c);
            else if (BITS == 2) v[i] = __ldg(reinterpret_cast<const uint16_t *>(row) + c);
            else if (BITS == 1) v[i] = __ldg(row + c);
            else {
                const uint32_t *w = reinterpret_cast<const uint32_t *>(row);
                const int q = (3 * c) >> 2;
                v[i] = __funnelshift_r(__ldg(w + q), __ldg(w + min(q + 1, pitch_in / 4 - 1)),
                                       8 * ((3 * c) & 3));
            }
        }
#pragma unroll
        for (int i = 0; i < EX_ROWS; ++i) {
            if (r0 + i >= N) break;
            // codes 0..3 in the low half, 4..7 in the high half
            constexpr uint32_t LOW = BITS == 4 ? 0xFFFFu : (1u << (4 * BITS)) - 1u;
            const uint32_t x = (v[i] & LOW) | ((v[i] << (16 - 4 * BITS)) & ~0xFFFFu);
            uint32_t q[4];                                 // values (j, j + 4)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t y = odd ? (j == 0 ? x << 1 : x >> (BITS * j - 1)) : x >> (BITS * j);
                const uint32_t f = (y & mask) ^ flip;
                const __nv_bfloat162 t = __hsub2(*reinterpret_cast<const __nv_bfloat162 *>(&f),
                                                 *reinterpret_cast<const __nv_bfloat162 *>(&base));
                q[j] = *reinterpret_cast<const uint32_t *>(&t);
            }
            *reinterpret_cast<uint4 *>(W16 + (int64_t)(r0 + i) * pitch_out + 16 * c) =
                make_uint4(__byte_perm(q[0], q[1], 0x5410), __byte_perm(q[2], q[3], 0x5410),
                           __byte_perm(q[0], q[1], 0x7632), __byte_perm(q[2], q[3], 0x7632));
        }
    }
}

// grid of an expansion: about eight resident blocks per SM
inline dim3 expand_grid(int64_t chunks, int64_t rows)
{
    const int sms = dsq_sm_count() > 0 ? dsq_sm_count() : 148;
    const int64_t gx = (chunks + EX_THREADS - 1) / EX_THREADS;
    const int64_t gy = std::min<int64_t>((rows + EX_ROWS - 1) / EX_ROWS, std::max<int64_t>(8 * sms / gx, 1));
    return dim3((unsigned)gx, (unsigned)gy);
}

// ---------------------------------------------------------------------------
// pass 2: GEMM of the expanded rows, CTA pairs
// ---------------------------------------------------------------------------
// Integer and scaled outputs of an accumulator (f32 ones of 4-bit operands: `more` and the sum
// are whole numbers below 2^24).
template <int KIND>
__device__ __forceinline__ uint32_t g8_whole(uint32_t x, float more)
{
    return KIND == G8_I8 ? x : (uint32_t)__float2int_rn(__fadd_rn(__uint_as_float(x), more));
}
template <int KIND>
__device__ __forceinline__ uint32_t g8_scaled(uint32_t x, float more, float rs)
{
    return __float_as_uint(__fmul_rn(KIND == G8_I8 ? (float)(int)x : __fadd_rn(__uint_as_float(x), more), rs));
}

// Outputs of a 32 x 32 block of accumulators: r[j] is row m + lane, column n + j; columns
// from `limit` on belong to another tile or lie outside.
// Where rows are full 32-byte sectors (p.vec) a lane stores its row from its registers.
// Elsewhere, and for the last weight-only tile of a CTA (no operands arrive any more), the block
// is turned round in shared memory (`stage`: rows of 128 bytes, 16-byte units XOR-ed with the
// row: no bank conflicts either way), and a warp stores whole lines: there a lane's scales and
// biases are those of eight columns, not of all 32.
// An SM takes 27 bytes of stores a clock in whole lines, 16 in sectors of 32 lines; beside the
// next tile's instructions that does not show, and the integer kernels' last tile is no faster
// turned round (4096^3 4-bit 61.4 us against 60.5).  2500x1111x1777 3-bit with 16-byte
// stores to shared memory and the next block already on its way 12.7 -> 12.0 us, weight-only
// 2048x4096x4096 55.5 -> 54.1, 3000x1000x512 11.6 -> 10.6, in a graph.
template <int KIND>
__device__ __forceinline__ void g8_store_rows(const G8Params &p, int m, int n, int limit, int lane,
                                              const uint32_t (&r)[32], float more)
{
    const int row = m + lane;
    if (row >= p.M) return;
    const float rs = KIND != G8_BF16 && p.D_f32 ? __ldg(p.row_scale + row) : 0.0f;
    const int64_t at = (int64_t)row * p.N + n;
#pragma unroll
    for (int j = 0; j < 32; j += 8) {
        if (n + j >= limit) break;
        uint32_t f[8];
        if (KIND == G8_BF16) {
#pragma unroll
            for (int t = 0; t < 8; ++t)
                f[t] = __float_as_uint(
                    __fmaf_rn(__uint_as_float(r[j + t]), __ldg(p.col_scale + n + j + t),
                              p.col_bias ? __ldg(p.col_bias + n + j + t) : 0.0f));
            stg_256(p.Y_f32 + at + j, f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7]);
            continue;
        }
        if (p.C_i32) {
#pragma unroll
            for (int t = 0; t < 8; ++t) f[t] = g8_whole<KIND>(r[j + t], more);
            stg_256(p.C_i32 + at + j, f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7]);
        }
        if (p.D_f32) {
#pragma unroll
            for (int t = 0; t < 8; ++t) f[t] = g8_scaled<KIND>(r[j + t], more, rs);
            stg_256(p.D_f32 + at + j, f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7]);
        }
    }
}

// (`next` is called, on the one way through here, when r has been read for the last time.  One loop for
// each form of the values: with the choice at every word 2500x1111x1777 3-bit takes 0.3 us longer.  Both
// outputs are turned round one after the other: with the whole numbers scaled on their way out, 13.5 us
// became 15.0.)
template <int KIND, class F>
__device__ __forceinline__ void g8_store_turned(const G8Params &p, int m, int n, int limit, int lane,
                                                uint32_t stage, const uint32_t (&r)[32], float more, F next)
{
    const int rows = min(32, p.M - m);
    const bool whole = KIND != G8_BF16 && p.C_i32;
    const float rs = KIND != G8_BF16 && p.D_f32 && lane < rows ? __ldg(p.row_scale + m + lane) : 0.0f;
    const uint32_t mine = stage + 128u * (uint32_t)lane;
    __syncwarp();                                         // (the block before has been read)
    auto put = [&](auto value) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
            sts_128(mine + (uint32_t)((u ^ (lane & 7)) << 4), value(r[4 * u]), value(r[4 * u + 1]), value(r[4 * u + 2]),
                    value(r[4 * u + 3]));
    };
    const int col = n + lane;
    auto word = [&](int i) { return lds_32(stage + (uint32_t)(128 * i + ((lane * 4) ^ ((i & 7) << 4)))); };
    auto write = [&](uint32_t *out) {
        if (col >= limit) return;
        uint32_t *dst = out + (int64_t)m * p.N + col;
#pragma unroll 8
        for (int i = 0; i < rows; ++i, dst += p.N) *dst = word(i);
    };
    if (KIND == G8_BF16) put([](uint32_t x) { return x; });
    else if (whole) put([&](uint32_t x) { return g8_whole<KIND>(x, more); });
    if (whole && p.D_f32) {
        __syncwarp();
        write((uint32_t *)p.C_i32);
        __syncwarp();
    }
    if (KIND != G8_BF16 && p.D_f32) put([&](uint32_t x) { return g8_scaled<KIND>(x, more, rs); });
    next();
    __syncwarp();
    if (KIND != G8_BF16) {
        write(p.D_f32 ? (uint32_t *)p.D_f32 : (uint32_t *)p.C_i32);
        return;
    }
    if (p.vec) {
        const int u = 2 * (lane & 3), r0 = lane >> 2, col = n + 4 * u;
        if (col >= limit) return;
        float cs[8], cb[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            cs[t] = __ldg(p.col_scale + col + t);
            cb[t] = p.col_bias ? __ldg(p.col_bias + col + t) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = 8 * i + r0;
            const uint32_t at = stage + 128u * (uint32_t)row;
            const uint4 x = lds_128(at + (uint32_t)((u ^ (row & 7)) << 4));
            const uint4 y = lds_128(at + (uint32_t)(((u + 1) ^ (row & 7)) << 4));
            uint32_t f[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
            for (int t = 0; t < 8; ++t)
                f[t] = __float_as_uint(__fmaf_rn(__uint_as_float(f[t]), cs[t], cb[t]));
            if (row < rows)
                stg_256(p.Y_f32 + (int64_t)(m + row) * p.N + col, f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7]);
        }
        return;
    }
    if (col >= limit) return;
    const float cs = __ldg(p.col_scale + col), cb = p.col_bias ? __ldg(p.col_bias + col) : 0.0f;
    float *dst = p.Y_f32 + (int64_t)m * p.N + col;
#pragma unroll 8
    for (int i = 0; i < rows; ++i, dst += p.N) *dst = __fmaf_rn(__uint_as_float(word(i)), cs, cb);
}

// what is added to the accumulators of row m: 4-bit operands of 3-bit codes
template <int KIND>
__device__ __forceinline__ float g8_row_more(const G8Params &p, int m)
{
    int s = 0;
    if (KIND == G8_F4 && p.sums && m < p.M)
        for (int i = 0; i < p.parts; ++i) s += __ldg(p.sums + (int64_t)i * p.M + m);
    return (float)(4 * s);
}

// KIND: 8-bit integer operands with s32 accumulators (kind::i8), bf16 operands or 4-bit
// floating-point ones with f32 accumulators (kind::f16, kind::mxf4).  A stage row is 128
// bytes of K (128, 64 or 256 elements), four instructions per stage.
//
// S > 1: few tiles and a long K.  A cluster is S pairs on ONE tile, pair s taking the
// s-th part of K; when all are done, pair s gets the other pairs' partial sums of
// columns s * BN / S .. through distributed shared memory (into the stage ring,
// which nothing reads any more), adds them to its own in a fixed order and writes
// those columns.  One tile per cluster.
template <int KIND, int S>
__global__ void __maxnreg__(G8_REGS)
gemm8_kernel(const __grid_constant__ CUtensorMap tmap_a,
             const __grid_constant__ CUtensorMap tmap_b, const G8Params p)
{
    extern __shared__ uint8_t smem_raw[];
    constexpr int ACC = g8_acc<KIND>();
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023u) & ~(uintptr_t)1023u);
    uint8_t *tail = smem + p.stages * p.stage_bytes;
    const uint32_t bars = smem_u32(tail);
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(tail + 8 * G8_BARS);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tail + 8 * G8_BARS + 8);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // (of the last tile in the ring, which nothing reads any more, behind the exchanged sums; where
    // every tile needs it, behind the ring)
    const uint32_t staging = smem_u32(p.vec ? smem + (S > 1 ? G8_EXCHANGE : 0) : tail + G8_TAIL) +
                             (uint32_t)((warp - G8_WARP_E0) * 32 * 32 * 4);
    const uint32_t crank = cluster_ctarank();
    const uint32_t rank = crank & 1u, split = crank >> 1;       // in the pair; which part of K
    const uint32_t leader = crank & ~1u;
    const uint16_t pair_mask = (uint16_t)(3u << leader);
    Ctl ctl{abort_flag, p.ws, p.wait_ns};

    // full: operand bytes of BOTH CTAs' stage s have landed (counted on the
    //       leader's barrier only: the leader's producer expects both stages' bytes,
    //       both producers' copies complete on it);
    // empty: the pair's instructions on stage s are done (tcgen05.commit,
    //       signalled in both CTAs);
    // acc_full[b]: the tile in accumulator b is complete (both CTAs);
    // acc_empty[b]: (leader) all epilogue warps of both CTAs have read it.
    auto bar_full = [&](int s) { return bars + 8u * s; };
    auto bar_empty = [&](int s) { return bars + 8u * (G8_MAX_STAGES + s); };
    auto bar_acc_full = [&](int b) { return bars + 8u * (2 * G8_MAX_STAGES + b); };
    auto bar_acc_empty = [&](int b) { return bars + 8u * (2 * G8_MAX_STAGES + 2 + b); };
    const uint32_t bar_drain = bars + 8u * (2 * G8_MAX_STAGES + 4);

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(bar_full(s), 1);
            mbar_init(bar_empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_acc_full(b), 1);
            mbar_init(bar_acc_empty(b), 2 * G8_E_WARPS);
        }
        mbar_init(bar_drain, 1);
        *abort_flag = 0;
        mbar_init_fence();
    }
    if (warp == G8_WARP_TMEM) {
        tmem_alloc<2>(smem_u32((const void *)tmem_slot), 512);
        tmem_relinquish<2>();
    }
    if (warp == G8_WARP_TMA && lane == 0) {
        tma_prefetch_desc(&tmap_a);
        tma_prefetch_desc(&tmap_b);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    if (KIND == G8_F4 && warp >= G8_WARP_E0 && warp < G8_WARP_E0 + 4) {
        // every block scale is 2 (UE8M0 128), whatever place the tensor core reads it from
        uint32_t two[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) two[i] = 0x80808080u;
        tmem_st_32x32(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + G8_F4_SF, two);
        tmem_st_wait();
        tc_fence_before_sync();
    }
    __syncwarp();
    // the peer's barriers must be initialised (and its scales written) before anything
    // signals (reads) them
    cluster_sync_all();
    tc_fence_after_sync();

    const int pair = blockIdx.x / (2 * S), npairs = gridDim.x / (2 * S);
    const int kb0 = S == 1 ? 0 : (int)split * p.kblocks / S;
    const int kb1 = S == 1 ? p.kblocks : ((int)split + 1) * p.kblocks / S;
    const int total_tiles = p.m_tiles * p.n_tiles;
    grid_dependency_wait();
    grid_launch_dependents();

    if (warp == G8_WARP_TMA) {
        // ---------------- TMA producer (one thread per CTA) -----------------
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int tile = pair; ok && tile < total_tiles; tile += npairs) {
                const int m0 = (tile / p.n_tiles) * G8_BM + (int)rank * G8_ROWS;
                const int n0 = (tile % p.n_tiles) * p.BN + (int)rank * (p.BN / 2);
                for (int kb = kb0; kb < kb1; ++kb) {
                    if (!(ok = wait_bar(bar_empty(s), ph ^ 1u, ctl, 21))) break;
                    const uint32_t full0 = map_to_cta(bar_full(s), leader);
                    if (rank == 0) mbar_arrive_expect_tx(bar_full(s), 2 * (uint32_t)p.stage_bytes);
                    const uint32_t dst = smem_u32(smem + s * p.stage_bytes);
                    tma_load_2d_pair(dst, &tmap_a, kb * G8_KB, m0, full0);
                    tma_load_2d_pair(dst + G8_OP_BYTES, &tmap_b, kb * G8_KB, n0, full0);
                    if (++s == p.stages) { s = 0; ph ^= 1u; }
                }
            }
            if (!ok) {
                // copies in flight write this CTA's shared memory: give them time
                const uint64_t t0 = global_timer_ns();
                while (global_timer_ns() - t0 < 200000ull) { }
            }
        }
    } else if (warp == G8_WARP_MMA) {
        // ---------------- MMA issuer (leader CTA; whole warp, elected lane) ---
        if (rank == 0) {
            const uint32_t idesc = p.idesc;
            const uint64_t desc = smem_desc_sw128(smem_u32(smem));
            const uint32_t hi = (uint32_t)(desc >> 32);
            uint32_t it = 0, ph = 0;
            int s = 0;
            bool ok = true;
            // (a stage is asked for while the one before it is being issued)
            uint32_t ready = mbar_test_wait<true>(bar_full(0), 0u);
            for (int tile = pair; ok && tile < total_tiles; tile += npairs, ++it) {
                const int b = it & 1;
                if (!(ok = wait_bar_warp<true>(bar_acc_empty(b), ((it >> 1) & 1u) ^ 1u, ctl, 22)))
                    break;
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + b * ACC;
                for (int kb = kb0; kb < kb1; ++kb) {
                    if (!__all_sync(0xffffffffu, ready) &&
                        !(ok = wait_bar_warp<true>(bar_full(s), ph, ctl, 23)))
                        break;
                    tc_fence_after_sync();
                    const uint32_t bar_used = bar_empty(s);
                    // (a stage lies below 256 KB: the address field does not overflow)
                    const uint32_t ad = (uint32_t)desc + (uint32_t)s * (uint32_t)(p.stage_bytes >> 4);
                    const uint32_t bd = ad + (G8_OP_BYTES >> 4);
                    if (++s == p.stages) { s = 0; ph ^= 1u; }
                    ready = mbar_test_wait<true>(bar_full(s), ph);
                    if (KIND == G8_BF16)
                        mma_f16_ss_pair_x4_elect(d_tmem, ad, hi, bd, hi, idesc, (uint32_t)(kb - kb0));
                    else if (KIND == G8_F4)
                        mma_f4_ss_pair_x4_elect(d_tmem, ad, hi, bd, hi, idesc, tmem_base + G8_F4_SF,
                                                tmem_base + G8_F4_SF + 16, (uint32_t)(kb - kb0));
                    else
                        mma_i8_ss_pair_x4_elect(d_tmem, ad, hi, bd, hi, idesc, (uint32_t)(kb - kb0));
                    mma_commit_pair_elect(bar_used, pair_mask);
                }
                if (ok) mma_commit_pair_elect(bar_acc_full(b), pair_mask);
            }
            if (!ok) {
                // instructions already issued still read shared memory and write
                // the accumulators: they finish before either is given up
                mma_commit_elect(bar_drain);
                wait_bar_drain(bar_drain, 0u);
            }
        }
    } else if (S > 1 && warp >= G8_WARP_E0) {
        // (the exchange below starts when every pair's instructions are done)
        wait_bar_warp(bar_acc_full(0), 0u, ctl, 24);
    } else if (warp >= G8_WARP_E0) {
        // ---------------- epilogue: eight warps per CTA ----------------------
        const int quarter = warp & 3;                      // tensor-memory lane quarter
        const int half = (warp - G8_WARP_E0) >> 2;         // every other block of 32 columns
        const int blocks = p.BN / 32;
        uint32_t it = 0;
        bool ok = true;
        for (int tile = pair; ok && tile < total_tiles; tile += npairs, ++it) {
            const int b = it & 1;
            const int m = (tile / p.n_tiles) * G8_BM + (int)rank * G8_ROWS + quarter * 32;
            const int n0 = (tile % p.n_tiles) * p.BN, limit = min(p.N, n0 + p.BN);
            const float more = g8_row_more<KIND>(p, m + lane);
            if (!(ok = wait_bar_warp(bar_acc_full(b), (it >> 1) & 1u, ctl, 24))) break;
            tc_fence_after_sync();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + b * ACC;
            auto release = [&]() {
                // the accumulator is in registers: hand it back
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    if (rank != 0) mbar_arrive_cluster(map_to_cta(bar_acc_empty(b), leader));
                    else mbar_arrive(bar_acc_empty(b));
                }
            };
            if (p.vec && (KIND != G8_BF16 || tile + npairs < total_tiles)) {
#pragma unroll 1
                for (int c = half; c < blocks; c += 2) {
                    uint32_t r[32];
                    __syncwarp();
                    tmem_ld_32x32(taddr + 32 * c, r);
                    tmem_ld_wait();
                    if (c + 2 >= blocks) release();
                    if (n0 + 32 * c < limit) g8_store_rows<KIND>(p, m, n0 + 32 * c, limit, lane, r, more);
                }
                continue;
            }
            // (a block is on its way from tensor memory while the one before it is stored)
            const int end = m < p.M ? min(blocks, (limit - n0 + 31) / 32) : 0;
            if (half >= end) {
                release();
                continue;
            }
            uint32_t r[32];
            tmem_ld_32x32(taddr + 32 * half, r);
            tmem_ld_wait(r);
#pragma unroll 1
            for (int c = half;; c += 2) {
                const bool ahead = c + 2 < end;
                if (!ahead) release();
                g8_store_turned<KIND>(p, m, n0 + 32 * c, limit, lane, staging, r, more,
                                      [&]() { tmem_ld_32x32_if(ahead, taddr + 32 * (c + 2), r); });
                if (!ahead) break;
                __syncwarp();                              // (lanes without a column are back)
                tmem_ld_wait(r);
            }
        }
    }

    if (S > 1) {
        // ---------------- exchange of the partial sums --------------------------
        const int cols = p.BN / S;                         // columns a pair writes: a multiple of 32
        const uint32_t block = 128u * (uint32_t)cols * 4u; // one pair's sums of them, 128 rows
        // [row][cols] words, 16-byte units XOR-ed with the row: conflict-free for a
        // lane per row
        auto unit = [&](int row, int u) { return (uint32_t)(row * (cols * 4) + ((u ^ (row & 7)) << 4)); };
        const int quarter = warp & 3, k = (warp - G8_WARP_E0) >> 2;
        const uint32_t ring = smem_u32(smem);
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const int row = quarter * 32 + lane;
        tc_fence_after_sync();
        __syncwarp();
        cluster_sync_all();                                // every pair's instructions are done
        if (warp >= G8_WARP_E0) {
#pragma unroll 1
            for (int c0 = 32 * k; c0 < p.BN; c0 += 64) {
                const uint32_t d = (uint32_t)(c0 / cols);  // the pair these columns belong to
                if (d == split) continue;
                uint32_t r[32];
                tmem_ld_32x32(taddr + c0, r);
                tmem_ld_wait();
                const uint32_t dst = map_to_cta(ring, 2 * d + rank) + (split - (split > d)) * block;
#pragma unroll
                for (int v = 0; v < 8; ++v)
                    st_cluster_128(dst + unit(row, (c0 % cols) / 4 + v), r[4 * v], r[4 * v + 1],
                                   r[4 * v + 2], r[4 * v + 3]);
            }
        }
        __syncwarp();
        cluster_sync_all();
        if (warp >= G8_WARP_E0 && pair < total_tiles) {
            const int m = (pair / p.n_tiles) * G8_BM + (int)rank * G8_ROWS + quarter * 32;
            const int n0 = (pair % p.n_tiles) * p.BN + (int)split * cols, limit = min(p.N, n0 + cols);
            const float more = g8_row_more<KIND>(p, m + lane);
#pragma unroll 1
            for (int c0 = 32 * k; c0 < cols; c0 += 64) {
                uint32_t r[32];
                __syncwarp();
                tmem_ld_32x32(taddr + split * cols + c0, r);
                tmem_ld_wait();
#pragma unroll
                for (int o = 0; o < S - 1; ++o)
#pragma unroll
                    for (int v = 0; v < 8; ++v) {
                        const uint4 x = lds_128(ring + o * block + unit(row, c0 / 4 + v));
                        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                        for (int t = 0; t < 4; ++t)
                            r[4 * v + t] = KIND == G8_I8 ? r[4 * v + t] + w[t]
                                                         : __float_as_uint(__uint_as_float(r[4 * v + t]) +
                                                                           __uint_as_float(w[t]));
                    }
                if (m >= p.M || n0 + c0 >= limit) continue;
                if (p.vec && KIND != G8_BF16) g8_store_rows<KIND>(p, m, n0 + c0, limit, lane, r, more);
                else g8_store_turned<KIND>(p, m, n0 + c0, limit, lane, staging, r, more, [] {});
            }
        }
    }

    // ---------------- teardown ---------------------------------------------
    tc_fence_before_sync();
    __syncthreads();
    // a CTA stays until its peer has stopped signalling its barriers and reading
    // operands from its shared memory
    cluster_sync_all();
    if (warp == G8_WARP_TMEM) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc<2>(tmem_base, 512);
    }
}

int make_rows_tmap(CUtensorMap *map, const void *base, uint64_t k_bytes, uint64_t rows,
                   uint64_t pitch, int box_rows)
{
    DsqEncodeTiledFn fn = dsq_encode_tiled_fn();
    if (!fn) return DSQ_ERR_CUDA;
    cuuint64_t dims[2] = {k_bytes, rows};
    cuuint64_t strides[1] = {pitch};
    cuuint32_t box[2] = {G8_KB, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(base), dims, strides,
                    box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? DSQ_OK : DSQ_ERR_CUDA;
}

inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

template <int KIND, int S>
int launch_split(const CUtensorMap &ta, const CUtensorMap &tb, const G8Params &p, int clusters,
                 cudaStream_t stream)
{
    static std::atomic<unsigned long long> configured{0};
    const int st = dsq_allow_smem((const void *)gemm8_kernel<KIND, S>, G8_SMEM, &configured);
    if (st) return st;
    // (dependent launch: set-up overlaps the tail of pass 1; the kernel waits for it
    // itself before the first copy)
    return dsq_launch(gemm8_kernel<KIND, S>, dim3(2 * S * clusters), dim3(G8_THREADS), (size_t)G8_SMEM,
                      stream, dsq_launch_hooks().pdl, 2 * S, ta, tb, p);
}

// Clusters of S pairs that fit on the GPU at once (a cluster lives inside one group
// of SMs, so this is less than SMs / 2 S).
template <int KIND, int S>
int resident_clusters()
{
    static std::atomic<int> cached[DSQ_MAX_DEVICES];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= DSQ_MAX_DEVICES) return 0;
    int n = cached[dev].load(std::memory_order_relaxed);
    if (n) return n;
    if (cudaFuncSetAttribute(gemm8_kernel<KIND, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, G8_SMEM) !=
        cudaSuccess)
        return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * S);
    cfg.blockDim = dim3(G8_THREADS);
    cfg.dynamicSmemBytes = G8_SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2 * S;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, gemm8_kernel<KIND, S>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    cached[dev].store(n, std::memory_order_relaxed);
    return n;
}

template <int KIND>
DsqG8Tile pick_tile(int64_t M, int64_t N, int64_t kblocks)
{
    return dsq_g8_tile(M, N, kblocks, g8_acc<KIND>(), dsq_sm_count() > 0 ? dsq_sm_count() : 148,
                       [] { return resident_clusters<KIND, 2>(); });
}

// Pass 2 over operands that are rows of k_bytes bytes of K (byte maps: the
// kernel never looks at an element, only the tensor core does).
template <int KIND>
int launch_pass2(const void *A, size_t a_pitch, const void *B, size_t b_pitch, size_t k_bytes,
                 int64_t M, int64_t N, bool a_signed, bool b_signed, G8Params p, cudaStream_t stream)
{
    p.M = (int)M; p.N = (int)N;
    p.kblocks = (int)((k_bytes + G8_KB - 1) / G8_KB);
    const DsqG8Tile tile = pick_tile<KIND>(M, N, p.kblocks);
    p.BN = tile.bn;
    p.m_tiles = (int)((M + G8_BM - 1) / G8_BM);
    p.n_tiles = (int)((N + p.BN - 1) / p.BN);
    p.idesc = KIND == G8_F4     ? idesc_mxf4(p.BN, G8_BM)
              : KIND == G8_BF16 ? idesc_bf16(p.BN, G8_BM)
                                : idesc_i8(p.BN, a_signed, b_signed, G8_BM);
    p.vec = N % 8 == 0 && (!p.C_i32 || (reinterpret_cast<uintptr_t>(p.C_i32) & 31u) == 0) &&
            (!p.D_f32 || (reinterpret_cast<uintptr_t>(p.D_f32) & 31u) == 0) &&
            (!p.Y_f32 || (reinterpret_cast<uintptr_t>(p.Y_f32) & 31u) == 0);
    p.stage_bytes = G8_OP_BYTES + p.BN / 2 * G8_KB;
    p.stages = std::min(G8_MAX_STAGES,
                        (G8_SMEM - 1024 - G8_TAIL - (p.vec ? 0 : G8_STAGING)) / p.stage_bytes);
    p.wait_ns = dsq_launch_hooks().wait_ns;
    CUtensorMap ta, tb;
    int st = make_rows_tmap(&ta, A, k_bytes, (uint64_t)M, a_pitch, G8_ROWS);
    if (st) return st;
    st = make_rows_tmap(&tb, B, k_bytes, (uint64_t)N, b_pitch, p.BN / 2);
    if (st) return st;
    const int sms = dsq_sm_count() > 0 ? dsq_sm_count() : 148;
    const int tiles = p.m_tiles * p.n_tiles;
    if (tile.split == 2) return launch_split<KIND, 2>(ta, tb, p, tiles, stream);
    return launch_split<KIND, 1>(ta, tb, p, std::min(sms / 2, tiles), stream);
}

// first 1024-byte boundary behind the status words of a caller workspace
inline uint8_t *scratch_of(void *workspace)
{
    const uintptr_t w0 = reinterpret_cast<uintptr_t>(workspace);
    return reinterpret_cast<uint8_t *>((w0 + DSQ_WS_BYTES + 1023u) & ~(uintptr_t)1023u);
}

}  // namespace

// whether every partial sum of 4-bit operands stays below 2^23 (3 bits: products of -4 .. 4 by
// -4 .. 3, and the results below 2^24)
static bool f4_exact(int64_t K, int bits)
{
    return bits < 4 && K * (bits == 3 ? 16 : bits == 2 ? 6 : 1) < (1 << 23);
}
// bytes of a row, and the parts of a row whose sums are kept
static size_t f4_pitch(int64_t K) { return round_up((size_t)(K + 1) / 2, 16); }
static int64_t f4_parts(int64_t K) { return (K + 1023) / 1024; }

// clocks of the second pass
static double pass2_clocks(int64_t M, int64_t N, int64_t K, int bits)
{
    return f4_exact(K, bits) ? pick_tile<G8_F4>(M, N, (K + 255) / 256).clocks
                             : pick_tile<G8_I8>(M, N, (K + 127) / 128).clocks;
}

// Scratch the two-pass path needs behind the status words (0: the problem is
// one the fused kernel keeps).
size_t dsq_gemm8_scratch_bytes(int64_t M, int64_t N, int64_t K, int bits, int force)
{
    if (!force && (!dsq_gemm_may_take_two(M, N, K) ||
                   !dsq_g8_two_passes(M, N, K, bits, f4_exact(K, bits), pass2_clocks(M, N, K, bits))))
        return 0;
    const size_t kp = round_up((size_t)K, 16);             // (4-bit operands fill half of it)
    const size_t need = round_up((size_t)M * kp, 1024) + round_up((size_t)N * kp, 1024);
    if (bits != 3) return need;
    const size_t k4 = f4_pitch(K);                         // (more than that only below 128 of K)
    return std::max(need, round_up((size_t)M * k4, 1024) + round_up((size_t)N * k4, 1024) +
                              (size_t)(f4_parts(K) * M) * sizeof(int32_t));
}

DsqGemmForm dsq_gemm8_form(int64_t M, int64_t N, int64_t K, int bits, int outs, bool room, bool little)
{
    return dsq_gemm_form(M, N, K, bits, outs, f4_exact(K, bits),
                         room && dsq_gemm_may_take_two(M, N, K) ? pass2_clocks(M, N, K, bits) : 0.0, room, little,
                         dsq_sm_count() > 0 ? dsq_sm_count() : 148);
}

// 1- to 3-bit operands as 4-bit floating point where every sum stays below 2^23 (f32
// accumulators then hold it exactly whatever the order of the additions): twice the values
// per instruction and half of the expanded bytes of int8.
template <int BITS>
static int launch_f4(const void *A, const void *B, int64_t M, int64_t N, int64_t K, G8Params p,
                     void *scratch, cudaStream_t stream)
{
    const size_t kp = f4_pitch(K);
    uint8_t *A4 = (uint8_t *)scratch, *B4 = A4 + round_up((size_t)M * kp, 1024);
    int32_t *sums = nullptr;
    if (BITS == 3) {
        p.sums = sums = (int32_t *)(B4 + round_up((size_t)N * kp, 1024));
        p.parts = (int)f4_parts(K);
    }
    const int st = dsq_launch(expand_rows_f4_kernel<BITS>, expand_grid((int64_t)kp / 16, M + N),
                              dim3(EX_THREADS), 0, stream, dsq_launch_hooks().pdl, 0, (const uint8_t *)A, (const uint8_t *)B,
                              (int)M, (int)N, (int)K, (int)dsq_row_pitch(K, BITS), (int)kp, A4, B4, sums);
    if (st) return st;
    return launch_pass2<G8_F4>(A4, kp, B4, kp, kp, M, N, true, true, p, stream);
}
// Arguments as dsq_gemm after validation; `scratch` 1024-byte aligned.
int dsq_gemm8_launch(const void *A_codes, const void *B_codes, int64_t M, int64_t N, int64_t K,
                     int bits, int32_t *C_i32, const float *row_scale, float *D_f32,
                     void *workspace, void *scratch, cudaStream_t stream)
{
    G8Params p = {};
    p.C_i32 = C_i32; p.row_scale = row_scale; p.D_f32 = D_f32;
    p.ws = (int *)workspace;
    if (f4_exact(K, bits))
        return bits == 2 ? launch_f4<2>(A_codes, B_codes, M, N, K, p, scratch, stream)
                         : launch_f4<3>(A_codes, B_codes, M, N, K, p, scratch, stream);
    const size_t kp = round_up((size_t)K, 16);
    uint8_t *A8 = (uint8_t *)scratch;
    uint8_t *B8 = A8 + round_up((size_t)M * kp, 1024);
    const int pitch_in = (int)dsq_row_pitch(K, bits);
    const uint8_t *A = (const uint8_t *)A_codes, *B = (const uint8_t *)B_codes;
    const int st = dsq_launch(bits == 2   ? expand_rows_kernel<2>
                              : bits == 3 ? expand_rows_kernel<3>
                                          : expand_rows_kernel<4>,
                              expand_grid((int64_t)kp / 16, M + N), dim3(EX_THREADS), 0, stream, dsq_launch_hooks().pdl, 0,
                              A, B, (int)M, (int)N, (int)K, pitch_in, (int)kp, A8, B8);
    if (st) return st;
    return launch_pass2<G8_I8>(A8, kp, B8, kp, (size_t)K, M, N, true, false, p, stream);
}

// ---------------------------------------------------------------------------
// binary GEMM (both operands 1 bit, values -1 / +1)
// ---------------------------------------------------------------------------
size_t dsq_binary_gemm_workspace_bytes(int64_t M, int64_t N, int64_t K)
{
    if (M <= 0 || N <= 0 || K <= 0) return DSQ_WS_BYTES;
    const size_t kp = round_up((size_t)K, 16);
    return DSQ_WS_BYTES + 1024 + round_up((size_t)M * kp, 1024) + round_up((size_t)N * kp, 1024);
}

int dsq_binary_gemm(const void *A_bits, const void *B_bits, int64_t M, int64_t N, int64_t K,
                    int32_t *C_i32, const float *row_scale, float *D_f32, void *workspace,
                    size_t ws_bytes, void *stream)
{
    if (!A_bits || !B_bits || !workspace) return DSQ_ERR_NULL;
    if (!C_i32 && !D_f32) return DSQ_ERR_NULL;
    if (D_f32 && !row_scale) return DSQ_ERR_NULL;
    if (M <= 0 || N <= 0 || K <= 0 || M > (1 << 24) || N > (1 << 24) || K > (1 << 24))
        return DSQ_ERR_SHAPE;
    if (!dsq_aligned16(A_bits) || !dsq_aligned16(B_bits) || !dsq_aligned16(workspace) ||
        (C_i32 && !dsq_aligned16(C_i32)) || (D_f32 && !dsq_aligned16(D_f32)))
        return DSQ_ERR_ALIGN;
    uint8_t *scratch = scratch_of(workspace);
    const size_t kp = round_up((size_t)K, 16);
    const size_t need = round_up((size_t)M * kp, 1024) + round_up((size_t)N * kp, 1024);
    if (ws_bytes < (size_t)(scratch - (uint8_t *)workspace) + need) return DSQ_ERR_SIZE;
    G8Params p = {};
    p.C_i32 = C_i32; p.row_scale = row_scale; p.D_f32 = D_f32;
    p.ws = (int *)workspace;
    if (f4_exact(K, 1)) return launch_f4<1>(A_bits, B_bits, M, N, K, p, scratch, (cudaStream_t)stream);
    uint8_t *A8 = scratch, *B8 = scratch + round_up((size_t)M * kp, 1024);
    const int st = dsq_launch(expand_rows_kernel<1>, expand_grid((int64_t)kp / 16, M + N),
                              dim3(EX_THREADS), 0, (cudaStream_t)stream, dsq_launch_hooks().pdl, 0, (const uint8_t *)A_bits,
                              (const uint8_t *)B_bits, (int)M, (int)N, (int)K,
                              (int)dsq_row_pitch(K, 1), (int)kp, A8, B8);
    if (st) return st;
    return launch_pass2<G8_I8>(A8, kp, B8, kp, (size_t)K, M, N, true, true, p, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------
// weight-only low-bit GEMM: bf16 activations x b-bit weights
// ---------------------------------------------------------------------------
size_t dsq_wgemm_workspace_bytes(int64_t N, int64_t K)
{
    if (N <= 0 || K <= 0) return DSQ_WS_BYTES;
    return DSQ_WS_BYTES + 1024 + round_up((size_t)N * round_up((size_t)K, 8) * 2, 1024);
}

int dsq_wgemm_bf16(const void *X_bf16, const void *W_codes, int64_t M, int64_t N, int64_t K,
                   int bits, float w_offset, const float *col_scale, const float *col_bias,
                   float *Y_f32, void *workspace, size_t ws_bytes, void *stream)
{
    if (!X_bf16 || !W_codes || !col_scale || !Y_f32 || !workspace) return DSQ_ERR_NULL;
    if (bits < 1 || bits > 4) return DSQ_ERR_BITS;
    if (M <= 0 || N <= 0 || K <= 0 || M > (1 << 24) || N > (1 << 24) || K > (1 << 24))
        return DSQ_ERR_SHAPE;
    if (w_offset != 0.0f && w_offset != 0.5f) return DSQ_ERR_UNSUPPORTED;
    // rows of X are read by TMA: 16-byte pitch
    if ((K % 8) != 0 || !dsq_aligned16(X_bf16) || !dsq_aligned16(W_codes) ||
        !dsq_aligned16(Y_f32) || !dsq_aligned16(workspace))
        return DSQ_ERR_ALIGN;
    uint8_t *W16 = scratch_of(workspace);
    const size_t wp = round_up((size_t)K, 8) * 2;          // scratch row pitch in bytes
    if (ws_bytes < (size_t)(W16 - (uint8_t *)workspace) + round_up((size_t)N * wp, 1024))
        return DSQ_ERR_SIZE;
    const int sms = dsq_sm_count() > 0 ? dsq_sm_count() : 148;
    const double clocks = M <= 32 ? 0.0 : pick_tile<G8_BF16>(M, N, (K + 63) / 64).clocks;
    if (M <= 32 || dsq_wgemm_takes_small(M, N, K, sms, clocks) || dsq_wgemm_takes_wide(M, N, K, sms, clocks))
        return dsq_wgemm_small(X_bf16, W_codes, M, N, K, bits, w_offset == 0.5f, col_scale, col_bias,
                               Y_f32, (cudaStream_t)stream);
    const int pitch_in = (int)dsq_row_pitch(K, bits);
    const int odd = w_offset == 0.5f;
    const uint8_t *W = (const uint8_t *)W_codes;
    cudaStream_t s = (cudaStream_t)stream;
    const int st = dsq_launch(bits == 1   ? expand_w_bf16_kernel<1>
                              : bits == 2 ? expand_w_bf16_kernel<2>
                              : bits == 3 ? expand_w_bf16_kernel<3>
                                          : expand_w_bf16_kernel<4>,
                              expand_grid(K / 8, N), dim3(EX_THREADS), 0, s, dsq_launch_hooks().pdl, 0, W, (int)N,
                              (int)K, pitch_in, (int)wp, odd, W16);
    if (st) return st;
    G8Params p = {};
    p.col_scale = col_scale; p.col_bias = col_bias; p.Y_f32 = Y_f32;
    p.ws = (int *)workspace;
    return launch_pass2<G8_BF16>(X_bf16, (size_t)K * 2, W16, wp, (size_t)K * 2, M, N, true, true, p, s);
}
