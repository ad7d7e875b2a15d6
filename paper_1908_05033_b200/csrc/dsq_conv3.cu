// 3x3, pad 1 low-bit convolution (strides 1 and 2) on the tensor cores, with the A
// operand read from an expanded WINDOW of the input in shared memory
// (Algorithm 1 step 5 on codes, plus the fused epilogue of steps 4, 1, 3).
//
// An im2col formulation expands every input pixel nine times, once per filter
// tap.  Here every input pixel of a tile is expanded ONCE:
//
//   * Output positions are numbered in a zero-padded, stacked coordinate
//     g = (n * (H+1) + ho) * (W+1) + wo.  The input pixel under filter tap
//     (kh, kw) of output g then sits at padded position g + kh*(W+1) + kw,
//     whatever g is: one constant shift per tap.  (Positions with ho >= H or
//     wo >= W are padding of the numbering; their results are dropped.)
//   * A tile is 128 consecutive positions g0 .. g0+127.  The padded input
//     pixels g0 .. g0+129+2(W+1) are fetched by TMA im2col loads whose
//     bounding box is the image grown by one pixel at its left and top (the loads
//     traverse W, then H, then N and fill what lies outside the image with
//     zeros = code 0), into a packed staging buffer.
//   * Four warps expand the staged codes to int8 rows of 128 bytes (128
//     channels; wider inputs take several such "planes") in the K-major
//     128-byte-swizzled layout the tensor core reads.
//   * For tap (kh, kw) the A operand of tcgen05.mma is that SAME buffer, its
//     descriptor's start address moved by (kh*(W+1) + kw) rows.  Nine taps x
//     Cin/32 instructions of 128 x BN x 32 accumulate one tile in tensor
//     memory (two accumulator buffers: the epilogue of a tile overlaps the
//     next tile's instructions).
//   * B (weights): TMA brings packed rows of one K step (128 codes of one tap)
//     into a small ring, eight warps expand them to int8, as in the im2col
//     kernel; a weight matrix of few K steps stays resident.
//   * Sixteen epilogue warps (four per tensor-memory lane quarter) take
//     16-column units of a tile: tcgen05.ld, dequantise, residual, requantise,
//     pack, store.  The epilogue is a long chain of dependent arithmetic per
//     element, so it wants many warps in flight; the per-channel scale and bias
//     of the whole layer sit in shared memory, the residual words of a tile
//     are fetched before its accumulators are waited for.
//
// Measured: alone on an SM, instructions issued four at a time run for N / 2 clocks each
// (40 at least; both operands through shared-memory descriptors).  In this kernel a block of
// four takes 480 to 700: the issuing warp shares its scheduler with epilogue warps, and the
// operands' reads (12 KB an instruction of 256 columns) share the shared-memory port with the
// expansion.  So instructions should be wide and few.  (Two issuing warps on alternate tiles,
// single instructions in a tight loop: no faster, slower.  A variant that copied each K step
// of the window to tensor memory - ld.shared + tcgen05.st, A taken from there - was
// slower than this one at every layer size.)
//
// Wide images (W + 1 > 139) would need a window of more than 416 pixels; they
// are staged as three bands of 136 pixels, one per filter row, instead.
//
// Every wait on a barrier is bounded, as in the im2col kernel.
#include <algorithm>

#include "dsq_tc_common.cuh"
#include "dsq_conv_rule.h"
#include "dsq_tc_host.h"

// Cycle stamps of the roles of CTA 0 (profiling builds only: -DDSQ_W3_STAMPS).
#ifdef DSQ_W3_STAMPS
__device__ long long g_w3_stamps[16][64];
#define W3_STAMP(row, col)                                                          \
    do {                                                                            \
        if (blockIdx.x == 0 && (threadIdx.x & 31) == 0 && (col) < 64)               \
            g_w3_stamps[row][col] = clock64();                                      \
    } while (0)
extern "C" int dsq_w3_read_stamps(long long *out)
{
    if (cudaMemcpyFromSymbol(out, g_w3_stamps, sizeof(g_w3_stamps)) != cudaSuccess) return -9;
    void *dev = nullptr;
    if (cudaGetSymbolAddress(&dev, g_w3_stamps) != cudaSuccess) return -9;
    return cudaMemset(dev, 0, sizeof(g_w3_stamps)) == cudaSuccess ? 0 : -9;
}
#else
#define W3_STAMP(row, col) do { } while (0)
#endif

namespace {

constexpr int W3_WARP_TMA_B = 0, W3_WARP_MMA = 1, W3_WARP_TMA_A = 2, W3_WARP_A0 = 3,
              W3_NUM_A_WARPS = 4, W3_WARP_B0 = 7, W3_NUM_B_WARPS = 8, W3_WARP_E0 = 15,
              W3_NUM_E_WARPS = 16, W3_NUM_WARPS = 31;
constexpr int W3_B_GROUP_WARPS = W3_NUM_B_WARPS / 2;   // two B groups take alternate K steps
constexpr int W3_EPQ = W3_NUM_E_WARPS / 4;   // epilogue warps per tensor-memory lane quarter
constexpr int W3_THREADS = W3_NUM_WARPS * 32;
constexpr int W3_A_SLOTS = 2;          // expanded windows, at most
constexpr int W3_MAX_BP = 4;           // packed B ring slots
constexpr int W3_MAX_AS = 3;           // packed A staging slots
constexpr int W3_MAX_BST = 10;         // expanded B stages (resident: all K steps)
constexpr int W3_BAND_PX = 136;        // pixels of a band (three-band staging)
constexpr int W3_F4_BAND_PX = 248;
constexpr int W3_MAX_WINDOW_PX = 416;
// 4-bit floating-point operands (see F4 below)
constexpr uint32_t W3_F4_MARK = 0x34463271u;   // behind the blob's copy of the weights
constexpr int W3_F4_SF = 2 * W3_F4_TP; // tensor-memory columns of the block scales: 480 .. 511

// byte offsets of the kernel's shared-memory regions (w3_layout)
struct W3Smem {
    uint32_t a_slots, b_tiles, a_stage, b_packed, epi, lut, bars, tmem_slot, abort_flag, total;
};

struct W3Params {
    // geometry
    int N, H, W, Ho, Wo, Hp, Wp;       // input and output; Hp, Wp: positions of an image (see W3Pos)
    int stride;
    int sh, sw;                        // input rows and columns between two positions: 1 or 2
    int m_tiles, n_tiles, BN, Ncols;
    int E;                             // operand bytes per pixel: Cin (F4: Cin / 2)
    int npl, kpp, ksteps;              // planes of 128 (F4: 256) channels, K steps per plane, total
    int PB, cpp;                       // packed bytes per pixel and plane; 16-byte chunks of it
    int tps;                           // filter taps of a K step: 2 with 64-channel rows (3-bit: transposed
                                       // tiles only); F4: 4 with 64 channels, 2 with 128
    int pk;                            // packed bytes of a K step in a weight row
    int rb;                            // bytes of a window row: 128, or 64 (transposed tiles over 64
                                       // channels: half the shared memory, which is what leaves room
                                       // for resident weights beside the window of a wide image);
                                       // F4: 32, 64 or 128 for 64, 128 or more channels
    int xstep;                         // bytes between two K steps of a plane in a weight row
    int apx, a_slots;                  // pixels of an A slot, slots
    // A window is nbands bands of band_px positions, each fetched by a_nload loads of a_box;
    // band b starts band_pos[b] positions behind the tile's first and takes the input pixels
    // of filter tap band_tap[b] (column | row << 8) of a filter whose corner is at (-2, -2)
    int a_box, a_nload, nbands, band_px;
    int band_pos[4], band_tap[4];
    int as_slots, bp_slots, b_stages, b_res;
    int w8;                            // weight K steps come expanded, by TMA, into the operand ring
    int pair;                          // transposed tiles, <= 64 output channels: two image rows a position
    int cout_pad;                      // Cout rounded up to the N tiling
    int tr;                            // transposed tiles (kernel form TR)
    int tp;                            // positions of a tile: 128; TR: a multiple of 16 (w3_tile)
    int f4;                            // 4-bit floating-point operands (kernel form F4)
    int mstep;                         // M tiles between two tiles of a CTA
    int t_dn, t_dh, t_dw;              // the positions of mstep tiles as images, padded rows, columns
    int smem_bytes;
    uint32_t zero;                     // 0 (see w3_release_slot)
    int early;                         // dsq_early_constants
    unsigned long long wait_ns;
    int skip_b_round;
    // epilogue
    int shift, out_pitch;
    float r_hi;                        // fmaf(hi - lo, inv, 0.5f) of the requantiser
    DsqEpi e;
    uint32_t orv;
    const uint32_t *mark;              // F4: W3_F4_MARK, if the blob's copy is of that form
    const uint8_t *act;                // input codes and pixel pitch (general weight offset: S_a)
    int P;
    // window offsets (16-byte units) of the four instructions of every K step of a plane
    // (MMA_NONE: left out); in the parameters, so that the issuing warp keeps them, and what
    // it makes of them, in uniform registers
    uint4 x_off[12];
    W3Smem L;                          // shared-memory layout (host-made: w3_layout)
    int *ws;
};


__host__ __device__ inline W3Smem w3_layout(int apx, int a_slots, int rb, int BN, int pk, int PB, int as_slots,
                                            int b_stages, int bp_slots, int cout_pad)
{
    W3Smem L;
    uint32_t o = 0;
    L.a_slots = o;  o += a_slots * apx * rb;            // apx is a multiple of 8
    o = (o + 1023u) & ~1023u;
    L.b_tiles = o;  o += b_stages * BN * 128;              // BN is a multiple of 8
    L.a_stage = o;  o += as_slots * apx * PB;
    L.b_packed = o; o += bp_slots * BN * pk;
    L.epi = o;      o += 2 * cout_pad * 4;                  // scale[cout_pad], bias[cout_pad]
    L.lut = o;      o += 16 * 4;
    o = (o + 127u) & ~127u;
    // barriers: a_full/a_empty[2], as_full/as_empty[3], bp_full/bp_empty[4],
    // b_full/b_empty[W3_MAX_BST], acc_full/acc_empty[2], drain, scales
    L.bars = o;     o += 8 * (2 * W3_A_SLOTS + 2 * W3_MAX_AS + 2 * W3_MAX_BP + 2 * W3_MAX_BST + 4 + 2);
    L.tmem_slot = o; o += 8;
    L.abort_flag = o; o += 8;
    L.total = o;
    return L;
}

// 16 columns of one accumulator row -> BITS/2 words of codes, codes-only form
// with requantiser range [0, hi]: per element
//   v  = raw >> shift                       (the factor of the top-bit expansion)
//   vf = (float)v by the 1.5 * 2^23 trick   (|v| < 2^22, checked by the host)
//   y  = fma(vf, scale, bias) (+ lut[q_r])  (lut[q] = fma((float)q, Delta_r, l_r))
//   r  = min(fma(max(y, 0), inv, 0.5), r_hi)
// which is the pinned sequence: max(y, 0) - 0 = max(y, 0); clipping y at hi
// first or r at r_hi = fma(hi, inv, 0.5) afterwards gives the same r because
// fma is monotone; floor(r) <= qmax because floor(r_hi) = qmax (host-checked).
// floor and the packing use the 2^23 trick: the bits of r + 2^23 (rounded
// down) are 0x4B000000 + floor(r); the codes are summed into their fields and
// the constant is taken out once per word.
template <int BITS, bool RES>
__device__ __forceinline__ void w3_codes_unit(const uint32_t (&r)[16], const float *sc,
                                              const float *bi, const uint32_t (&resw)[BITS / 2],
                                              const float *lut, int shift, float inv,
                                              float r_hi, uint32_t (&cw)[BITS / 2])
{
    constexpr uint32_t MASK = (1u << BITS) - 1u;
#pragma unroll
    for (int w = 0; w < BITS / 2; ++w) cw[w] = 0u;
    const float4 *sc4 = reinterpret_cast<const float4 *>(sc);
    const float4 *bi4 = reinterpret_cast<const float4 *>(bi);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const float4 s4 = sc4[v], b4 = bi4[v];
        const float scs[4] = {s4.x, s4.y, s4.z, s4.w};
        const float bis[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = 4 * v + u;
            const float vf =
                __fsub_rn(__int_as_float(0x4B400000 + ((int)r[c] >> shift)), 12582912.0f);
            float y = __fmaf_rn(vf, scs[u], bis[u]);
            if (RES) {
                const uint32_t qr = (resw[(c * BITS) >> 5] >> ((c * BITS) & 31)) & MASK;
                y = __fadd_rn(y, lut[qr]);
            }
            const float rr = fminf(__fmaf_rn(fmaxf(y, 0.0f), inv, 0.5f), r_hi);
            const uint32_t rb = (uint32_t)__float_as_int(__fadd_rd(rr, 8388608.0f));
            cw[(c * BITS) >> 5] += rb << ((c * BITS) & 31);
        }
    }
    // 0x4B000000 summed over the fields of a word (mod 2^32)
    constexpr uint32_t FIELDS = BITS == 4 ? 0x11111111u : 0x55555555u;
#pragma unroll
    for (int w = 0; w < BITS / 2; ++w) cw[w] -= 0x4B000000u * FIELDS;
}

// Position in the padded, stacked numbering: image, padded row, padded column.  One
// column of zeros serves as the right edge of a row and the left edge of the next, one
// row of them as the bottom of an image and the top of the next: (H + 1)(W + 1)
// positions an image, tap (kh, kw) of position g reads position g + kh (W + 1) + kw.
// (With edges of their own, (H + 2)(W + 2), 28x28 512->512 at batch 32 was 113 tiles a
// channel tile, four passes of 37 CTAs, instead of 106, three: 49.1 -> 38.8 us.)
// Moving by a fixed number of positions is an addition of its (host-made)
// decomposition plus at most one carry per digit: no division in any loop.
struct W3Pos {
    int n, h, w;
};
__device__ __forceinline__ W3Pos w3_add(W3Pos a, int dn, int dh, int dw, int Hp, int Wp)
{
    a.w += dw;
    a.h += dh;
    a.n += dn;
    if (a.w >= Wp) { a.w -= Wp; ++a.h; }
    if (a.h >= Hp) { a.h -= Hp; ++a.n; }
    return a;
}

// Gives a packed slot back to the TMA producer when every lane of the warp HOLDS what it
// read from it: `seen` is made of a word of each of the lane's loads, and the arrival
// depends on a vote over it that only the kernel's parameter (zero) makes constant.
// Loads merely written before the arrival are not enough: a warp that had arrived could
// still read its rows after the slot had been filled again (seen on images more than 139
// columns wide, whose windows take longest to expand: the weights of tap t + 4 in place
// of tap t's, in one warp's rows of a CTA's second window).
__device__ __forceinline__ void w3_release_slot(uint32_t bar, uint32_t seen, uint32_t zero, int lane)
{
    const bool never = __any_sync(0xffffffffu, (seen & zero) != 0u);
    if (lane == 0 && !never) mbar_arrive(bar);
}

// word c of a packed word's operand words
template <int BITS, bool SIGNED, bool F4>
__device__ __forceinline__ uint32_t w3_operand(uint32_t w, int c, uint32_t orv)
{
    if constexpr (F4) return expand_word_f4<SIGNED>(w, c);
    else return expand_word<BITS, SIGNED>(w, c, orv);
}

// Transposed tiles (template parameter TR).  An instruction should carry as many columns
// as there are (see above).  With the roles swapped - A = 128 weight rows of the K
// step, B = 256 rows of the window - every instruction is 128 x 256 x 32 even
// for 64 or 128 output channels.  The accumulator then has output CHANNELS on
// the tensor-memory lanes and POSITIONS in the columns: an epilogue thread owns
// one channel, gathers its codes of 8 (16 at 2 bits) positions in a word and an
// 8 x 8 (16 x 16) transpose of bit fields across the lanes of a channel group
// (shuffles) turns that into the packed NHWC words of those positions.  3-bit codes
// take four-bit fields up to there; then a lane's eight channels are 24 bits and the
// four groups of a quarter put three words together.
//
// 3-bit, batch 64, plain tiles or the im2col kernel before -> transposed: 64->64 at 56x56
// 70.9 -> 18.6 us, 128->128 at 28x28 28.7 -> 15.7, 512->512 at 7x7 40 -> 21.
template <int BITS>
__device__ __forceinline__ uint32_t w3_transpose_fields(uint32_t x, int lane)
{
    constexpr int E = 32 / BITS;                 // fields per word = lanes per group
#pragma unroll
    for (int d = E / 2; d >= 1; d >>= 1) {
        const int block = BITS * d;
        const uint32_t M = block == 16 ? 0x0000FFFFu : block == 8 ? 0x00FF00FFu
                           : block == 4 ? 0x0F0F0F0Fu : 0x33333333u;
        const uint32_t px = __shfl_xor_sync(0xffffffffu, x, d);
        x = (lane & d) ? (((px >> block) & M) | (x & ~M)) : ((x & M) | ((px << block) & ~M));
    }
    return x;
}

//
// Pairs of image rows (p.pair).  With up to 64 output channels half of the 128 A rows
// would be idle.  The lower 64 rows then are the same channels of the NEXT image row: a
// position stands for two output rows, the four input rows under them lie in two bands of
// the window (rows -1, 1, .. and 0, 2, .., fetched by im2col loads that step over every other row), and of twelve
// taps (four rows) the upper 64 weight rows have the first nine, the lower ones the last
// nine, zeros elsewhere.  12 taps for two output rows instead of 18, and every input row
// is expanded 1.0 + 1/tile times instead of once per tile of its neighbours' too.
// 64->64, one row a position / pairs: 224x224 2-bit, batch 32 60 / 45 us, 56x56 4-bit, batch 64 15.3 / 12.2,
// 3-bit 18.3 / 17.3.
//
// Stride 2: positions are output pixels; the window is four bands (even and odd rows and
// columns of the image), and a tap is a band and a shift in it.  Batch 64, im2col kernel /
// this, us: 56x56 64->128 4-bit 12.7 / 10.5, 3-bit 36 / 13, 2-bit 12.2 / 8.2; 28x28 128->256
// 11.9 / 10.3, 21.8 / 12.7, 11.2 / 8.6; 14x14 256->512 10.8 / 12.2, 22 / 14.2, 10.1 / 10.0.
//
// F4: 2-bit codes (weight grid Delta (c + 1/2)) as 4-bit floating-point operands.  E2M1
// holds the codes 0 .. 3 and the weights 2 c + 1 exactly, and every partial sum is a whole
// number of at most 9 * 9 * 1024, so the f32 accumulators hold the int32 sums bit for bit
// (the adder is exact up to 2^23, large steps of both signs among least ones included:
// tests/test_gpu_gemm_exact_sums.py).  An instruction covers K = 64 in the clocks in which
// kind::i8 covers 32, from the same 32 bytes a row; the window and the weights take half of
// the shared memory.  The block scales (all 2, so that the accumulators come as 2 acc + S_a)
// need tensor memory beside the two accumulators, so a tile is 240 positions instead of 256.
//
// int8 -> F4, batch 32: 64->64 at 224x224 82 -> 60 us, 128->128 at 112x112 44.7 -> 26.3,
// 256->256 at 56x56 41.3 -> 25.6, 512->512 at 28x28 38.9 -> 27.6 (four passes of 240
// positions for three of 256), at 14x14 16.3 -> 11.0.  What bounds it now: shared-memory
// bandwidth (an instruction reads 11.5 KB in 120 clocks) and, with 64 channels, the epilogue.
//
// PAIR3: pairs of image rows at 3 bits, whose weights' expansion masks the taps outside the
// filter (in the common form the masks cost the wide layers 6 %: these instructions bound
// them).
template <int BITS, int EPI, bool TR, bool F4 = false, bool PAIR3 = false>
__global__ void __launch_bounds__(W3_THREADS, 1)
dsq_win3_kernel(const __grid_constant__ CUtensorMap tmap_b,
                const __grid_constant__ CUtensorMap tmap_a, const W3Params p)
{
    constexpr int CH = F4 ? 4 : Chunks<BITS>::CH;      // packed 16-byte chunks per 128 operand bytes
    constexpr int OUT = F4 ? 2 : Chunks<BITS>::OUT;    // operand chunks per packed chunk
    constexpr int ACC = F4 ? W3_F4_TP : 256;   // TR: tensor-memory columns of an accumulator
    const int TP = TR ? p.tp : W3_BM;          // positions of a tile
    static_assert(!F4 || (TR && BITS == 2), "F4: 2-bit codes, transposed tiles");
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    if ((threadIdx.x >> 5) == 1) W3_STAMP(13, 0);
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023u) & ~(uintptr_t)1023u);
    const int BN = p.BN;
    // (the layout comes ready-made: every warp's first instructions are on the
    // critical path of a launch)
    const W3Smem &L = p.L;
    if ((uint32_t)(smem - smem_raw) + L.total > (uint32_t)p.smem_bytes) {
        grid_dependency_wait();
        if (threadIdx.x == 0) atomicCAS(p.ws + DSQ_WS_STATUS, 0, (int)DSQ_ERR_UNSUPPORTED);
        return;
    }
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    // CTA c works on N tile c % n_tiles and on the M tiles m_first, m_first +
    // mstep, ... (the grid is a multiple of n_tiles)
    const int n_tile = p.n_tiles == 1 ? 0 : (int)blockIdx.x % p.n_tiles;
    const int m_first = p.n_tiles == 1 ? (int)blockIdx.x : (int)blockIdx.x / p.n_tiles;
    const int my_tiles = m_first < p.m_tiles ? (p.m_tiles - 1 - m_first) / p.mstep + 1 : 0;
    const uint32_t n_b_fills =
        my_tiles == 0 ? 0u : (p.b_res ? (uint32_t)p.ksteps : (uint32_t)my_tiles * p.ksteps);
    const uint32_t n_a_fills = (uint32_t)my_tiles * p.npl;
    const uint32_t a_slot_bytes = (uint32_t)(p.apx * p.rb);
    const uint32_t a_stage_bytes = (uint32_t)p.apx * p.PB;
    const uint32_t b_stage_bytes = (uint32_t)BN * 128u;
    const uint32_t b_packed_bytes = (uint32_t)BN * p.pk;
    const int img_positions = p.Hp * p.Wp;
    // F4: where the weights come expanded, their expansion warps work on the window, too (2-bit
    // 64->64 at 56x56 with residual 14.4 -> 13.7 us, 14x14 256->256 8.1 -> 7.9; the int8 form's epilogue
    // loses more to them than the first window gains: 15.9 -> 16.6)
    const int a_warps = F4 && p.w8 ? W3_NUM_A_WARPS + W3_NUM_B_WARPS : W3_NUM_A_WARPS;

    const uint32_t bars = smem_u32(smem + L.bars);
    auto bar_a_full = [&](int s) { return bars + 8u * s; };
    auto bar_a_empty = [&](int s) { return bars + 8u * (W3_A_SLOTS + s); };
    constexpr int O_AS = 2 * W3_A_SLOTS;
    auto bar_as_full = [&](int s) { return bars + 8u * (O_AS + s); };
    auto bar_as_empty = [&](int s) { return bars + 8u * (O_AS + W3_MAX_AS + s); };
    constexpr int O_BP = O_AS + 2 * W3_MAX_AS;
    auto bar_bp_full = [&](int s) { return bars + 8u * (O_BP + s); };
    auto bar_bp_empty = [&](int s) { return bars + 8u * (O_BP + W3_MAX_BP + s); };
    constexpr int O_B = O_BP + 2 * W3_MAX_BP;
    auto bar_b_full = [&](int s) { return bars + 8u * (O_B + s); };
    auto bar_b_empty = [&](int s) { return bars + 8u * (O_B + W3_MAX_BST + s); };
    constexpr int O_ACC = O_B + 2 * W3_MAX_BST;
    auto bar_acc_full = [&](int s) { return bars + 8u * (O_ACC + s); };
    auto bar_acc_empty = [&](int s) { return bars + 8u * (O_ACC + 2 + s); };
    const uint32_t bar_drain = bars + 8u * (O_ACC + 4);
    const uint32_t bar_scales = bars + 8u * (O_ACC + 5);
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + L.tmem_slot);
    Ctl ctl{reinterpret_cast<volatile int *>(smem + L.abort_flag), p.ws, p.wait_ns};

    if (warp == 0) W3_STAMP(13, 9);
    if (threadIdx.x == 0) {
        for (int s = 0; s < W3_A_SLOTS; ++s) {
            mbar_init(bar_a_full(s), a_warps);
            mbar_init(bar_a_empty(s), 1);            // tcgen05.commit
        }
        for (int s = 0; s < W3_MAX_AS; ++s) {
            mbar_init(bar_as_full(s), 1);            // TMA producer (+ bytes)
            mbar_init(bar_as_empty(s), a_warps);
        }
        for (int s = 0; s < W3_MAX_BP; ++s) {
            mbar_init(bar_bp_full(s), 1);            // TMA producer (+ bytes)
            mbar_init(bar_bp_empty(s), W3_B_GROUP_WARPS);
        }
        for (int s = 0; s < W3_MAX_BST; ++s) {
            mbar_init(bar_b_full(s), p.w8 ? 1 : W3_B_GROUP_WARPS);   // (w8: TMA producer + bytes)
            mbar_init(bar_b_empty(s), 1);            // tcgen05.commit
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_acc_full(s), 1);           // tcgen05.commit
            mbar_init(bar_acc_empty(s), W3_NUM_E_WARPS);
        }
        mbar_init(bar_drain, 1);
        if (F4) mbar_init(bar_scales, 4);
        *ctl.abort_flag = 0;
        W3_STAMP(13, 10);
        mbar_init_fence();
        W3_STAMP(13, 11);
    }
    if (warp == W3_WARP_MMA) {
        W3_STAMP(13, 5);
        tmem_alloc(smem_u32((const void *)tmem_slot), 512);
        tmem_relinquish();
        W3_STAMP(13, 6);
    }
    if (warp == W3_WARP_TMA_B && lane == 0) tma_prefetch_desc(&tmap_b);
    if (warp == W3_WARP_TMA_A && lane == 0) tma_prefetch_desc(&tmap_a);
    // residual table: the 2^BITS dequantised residual values
    if (EPI != DSQ_EPI_CODES && threadIdx.x >= 64 && threadIdx.x < 64 + (1 << BITS)) {
        const int q = threadIdx.x - 64;
        reinterpret_cast<float *>(smem + L.lut)[q] = __fmaf_rn((float)q, p.e.res_delta, p.e.res_lo);
    }
    // the window producer's first positions, a lane per load (two divisions), worked out
    // here, where the warp would otherwise only wait for the slower warps at the
    // barrier: it is on the critical path of a launch
    W3Pos ld_pos = {0, 0, 0};
    int ld_tap = 0;
    if (warp == W3_WARP_TMA_A && lane < p.nbands * p.a_nload) {
        const int band = lane / p.a_nload;
        const int g0 = m_first * TP + p.band_pos[band] + (lane - band * p.a_nload) * p.a_box;
        ld_tap = p.band_tap[band];
        ld_pos.n = g0 / img_positions;
        const int rem = g0 - ld_pos.n * img_positions;
        ld_pos.h = rem / p.Wp;
        ld_pos.w = rem - ld_pos.h * p.Wp;
    }
    if (warp == W3_WARP_MMA) W3_STAMP(13, 7);
    if (warp == W3_WARP_E0) W3_STAMP(13, 8);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    // everything above touched no global data; nothing below starts before the
    // kernels ahead of this one in the stream have completed
    W3_STAMP(13, 1);
    // (the window producer first works out its coordinates, then waits; the weights'
    // producer does not wait where its constants may be read early)
    if (warp != W3_WARP_TMA_A && !(warp == W3_WARP_TMA_B && p.early)) {
        grid_dependency_wait();
        grid_launch_dependents();
    }
    W3_STAMP(13, 2);

    if (warp == W3_WARP_TMA_B) {
        // ---------------- producer: packed B rows of one K step ------------------
        if (lane == 0 && p.w8) {
            // weights already expanded (blob's int8 copy): K step g of this CTA's
            // sequence goes straight into stage g % b_stages of the operand ring
            uint32_t issued = 0, ph = 0;
            const int BST = p.b_stages;
            const int y = n_tile * BN;
            int s = 0, x = 0, kk = 0, pl = 0;
            bool ok = true;
            // (a blob packed by a library that kept its copy in another form)
            if (F4 && n_b_fills > 0 && __ldg(p.mark) != W3_F4_MARK) {
                if (atomicCAS(p.ws + DSQ_WS_STATUS, 0, (int)DSQ_ERR_UNSUPPORTED) == 0)
                    p.ws[DSQ_WS_DETAIL] = 17;
                *ctl.abort_flag = 1;
                ok = false;
            }
#pragma unroll 1
            for (uint32_t g = 0; ok && g < n_b_fills; ++g) {
                if (!wait_bar(bar_b_empty(s), ph ^ 1u, ctl, 1)) break;
                if ((int)g == p.skip_b_round) break;
                mbar_arrive_expect_tx(bar_b_full(s), b_stage_bytes);
                const uint32_t dst = smem_u32(smem + L.b_tiles + s * b_stage_bytes);
                if (p.pair) {
                    // a K step's taps for the upper 64 rows, those a filter row before them for
                    // the lower ones; zeros before a plane's first and behind its last tap
                    tma_load_3d(dst, &tmap_b, 128 * kk, pl, 0, bar_b_full(s));
                    tma_load_3d(dst + 64 * 128, &tmap_b, 128 * kk - 3 * p.rb, pl, 0, bar_b_full(s));
                    if (++kk == p.kpp) {
                        kk = 0;
                        if (++pl == p.npl) pl = 0;
                    }
                } else {
                    tma_load_2d(dst, &tmap_b, x, y, bar_b_full(s));
                }
                ++issued;
                x += 128;
                if (x == p.ksteps * 128) x = 0;
                if (++s == BST) { s = 0; ph ^= 1u; }
            }
            for (uint32_t k = (issued > (uint32_t)BST ? issued - BST : 0); k < issued; ++k)
                wait_bar_drain(bar_b_full(k % BST), (k / BST) & 1u);
        } else if (lane == 0) {
            uint32_t issued = 0, ph = 0;
            const int BP = p.bp_slots;
            const int y = n_tile * BN;
            // byte offset of a K step in a weight row of 9 taps x Cin codes: tap kk,
            // plane pl (64-channel inputs: two taps per K step)
            const int xstep = p.xstep;
            int s = 0, kk = 0, xk = 0, xpl = 0;
#pragma unroll 1
            for (uint32_t g = 0; g < n_b_fills; ++g) {
                if (!wait_bar(bar_bp_empty(s), ph ^ 1u, ctl, 1)) break;
                if ((int)g == p.skip_b_round) break;
                mbar_arrive_expect_tx(bar_bp_full(s), b_packed_bytes);
                const uint32_t dst = smem_u32(smem + L.b_packed + s * b_packed_bytes);
                tma_load_2d(dst, &tmap_b, xk + xpl, y, bar_bp_full(s));
                if (p.pair)
                    tma_load_2d(dst + 64 * p.pk, &tmap_b, xk + xpl - 3 * p.P, y, bar_bp_full(s));
                ++issued;
                W3_STAMP(12, g);
                xk += xstep;
                if (++kk == p.kpp) {
                    kk = 0; xk = 0;
                    xpl += p.pk;
                    if (xpl == p.npl * p.pk) xpl = 0;
                }
                if (++s == BP) { s = 0; ph ^= 1u; }
            }
            for (uint32_t k = (issued > (uint32_t)BP ? issued - BP : 0); k < issued; ++k)
                wait_bar_drain(bar_bp_full(k % BP), (k / BP) & 1u);
        }
    } else if (warp == W3_WARP_TMA_A) {
        // ---------------- producer: packed window of a tile and plane ------------
        // Lane i issues load i of a fill.  Loads that start behind the last image are left
        // out (and not counted); the zeros below that image, if they begin there, are
        // written here.  An im2col load must start inside the map's bounding box
        // (0 <= h < Hp, 0 <= w < Wp, n >= 0, which the position arithmetic guarantees): a
        // position outside it is never issued - the roles then run into their wait limit
        // and the kernel reports the failure.
        uint32_t issued = 0, ph = 0;
        const int AS = p.as_slots;
        const bool mine = lane < p.nbands * p.a_nload;
        const uint32_t box_bytes = (uint32_t)(p.a_box * p.PB);
        int s = 0, pl = 0;
        grid_dependency_wait();
#pragma unroll 1
        for (uint32_t g = 0; g < n_a_fills; ++g) {
            if (!wait_bar_warp(bar_as_empty(s), ph ^ 1u, ctl, 11)) break;
            const W3Pos q = ld_pos;
            const bool live = mine && q.n < p.N;
            if (__any_sync(0xffffffffu, live && (q.n < 0 || q.h < 0 || q.h >= p.Hp || q.w < 0 || q.w >= p.Wp))) {
                if (lane == 0) {
                    if (atomicCAS(p.ws + DSQ_WS_STATUS, 0, (int)DSQ_ERR_SHAPE) == 0)
                        p.ws[DSQ_WS_DETAIL] = 16;
                    *ctl.abort_flag = 1;
                }
                break;
            }
            const uint32_t dst = smem_u32(smem + L.a_stage) + s * a_stage_bytes + lane * box_bytes;
            if (mine && !live) {
                // positions p.N * Hp * Wp .. + Wp of a load that is left out
                const int behind = (q.n - p.N) * img_positions + q.h * p.Wp + q.w;
                if (behind <= p.Wp) {
                    const int bytes = min(p.a_box, p.Wp + 1 - behind) * p.PB;
                    for (int k = 0; k < bytes; k += 16) sts_128(dst + k, 0u, 0u, 0u, 0u);
                    fence_proxy_async_smem();
                }
            }
            const uint32_t bytes = (uint32_t)__popc(__ballot_sync(0xffffffffu, live)) * box_bytes;
            if (lane == 0) mbar_arrive_expect_tx(bar_as_full(s), bytes);
            __syncwarp();
            if (live)
                tma_load_im2col_4d(dst, &tmap_a, pl * p.PB, q.w * p.sw - 2, q.h * p.sh - 2, q.n,
                                   (uint16_t)(ld_tap & 255), (uint16_t)(ld_tap >> 8), bar_as_full(s));
            ++issued;
            W3_STAMP(0, g);
            if (++pl == p.npl) {
                pl = 0;
                ld_pos = w3_add(ld_pos, p.t_dn, p.t_dh, p.t_dw, p.Hp, p.Wp);
            }
            if (++s == AS) { s = 0; ph ^= 1u; }
        }
        if (lane == 0)
            for (uint32_t k = (issued > (uint32_t)AS ? issued - AS : 0); k < issued; ++k)
                wait_bar_drain(bar_as_full(k % AS), (k / AS) & 1u);
        __syncwarp();
    } else if (warp == W3_WARP_MMA) {
        // ---------------- MMA issuer (whole warp, uniform; one lane issues) --------
        // (TR: A = 128 weight rows, signed; B = 256 window rows, unsigned)
        const uint32_t idesc = F4   ? idesc_mxf4(TP)
                               : TR ? idesc_i8(TP, true, false, 128)
                                    : idesc_i8(BN, false, true, W3_BM);
        const uint64_t desc0 = smem_desc_sw128(0u);
        const uint32_t desc_hi = (uint32_t)(desc0 >> 32), desc_lo = (uint32_t)desc0;
        const uint32_t win_hi = p.rb == 64         ? (uint32_t)(smem_desc_sw64(0u) >> 32)
                                : F4 && p.rb == 32 ? (uint32_t)(smem_desc_sw32(0u) >> 32)
                                                   : desc_hi;
        const uint32_t a_lo_base = desc_lo + (smem_u32(smem + L.a_slots) >> 4);
        const uint32_t b_lo_base = desc_lo + (smem_u32(smem + L.b_tiles) >> 4);
        const int BST = p.b_stages;
        int aslot = 0, st = 0;
        uint32_t aph = 0, bph = 0, ready = 0u;
        uint4 tn = p.x_off[0];
        bool ok = !F4 || wait_bar_warp(bar_scales, 0u, ctl, 14);
#pragma unroll 1
        for (int it = 0; ok && it < my_tiles; ++it) {
            const int as = it & 1;
            if (!(ok = wait_bar_warp(bar_acc_empty(as), ((it >> 1) & 1) ^ 1u, ctl, 3))) break;
            W3_STAMP(4, it);
            tc_fence_after_sync();
            const uint32_t d_tmem = tmem_base + as * (TR ? ACC : BN);
            uint32_t first = 0u;                    // 0: the tile's first instruction overwrites
#pragma unroll 1
            for (int pl = 0; ok && pl < p.npl; ++pl) {
                if (!(ok = wait_bar_warp(bar_a_full(aslot), aph, ctl, 4))) break;
                if (pl == 0) W3_STAMP(5, it);
                tc_fence_after_sync();
                const uint32_t x_lo = a_lo_base + aslot * (a_slot_bytes >> 4);
                // (slots and stages lie below 256 KB, so the sums stay inside the
                // 14-bit address field)
                auto issue = [&](uint4 t, int stage) {
                    const uint32_t w_lo = b_lo_base + stage * (b_stage_bytes >> 4);
                    const uint32_t x0 = x_lo + t.x, x1 = t.y == MMA_NONE ? t.y : x_lo + t.y,
                                   x2 = t.z == MMA_NONE ? t.z : x_lo + t.z,
                                   x3 = t.w == MMA_NONE ? t.w : x_lo + t.w;
                    if (F4)
                        mma_f4_ss_x4b_elect(d_tmem, w_lo, desc_hi, x0, x1, x2, x3, win_hi, idesc,
                                            tmem_base + W3_F4_SF, tmem_base + W3_F4_SF + 16, first);
                    else if (TR)
                        mma_i8_ss_x4b_elect(d_tmem, w_lo, desc_hi, x0, x1, x2, x3, win_hi, idesc, first);
                    else
                        mma_i8_ss_x4_elect(d_tmem, x0, x1, x2, x3, desc_hi, w_lo, desc_hi, idesc, first);
                    first = 1u;
                };
                if (p.b_res) {
                    st = pl * p.kpp;
#pragma unroll 1
                    for (int kk = 0; kk < p.kpp; ++kk, ++st) {
                        if (it == 0) {
                            if (!(ok = wait_bar_warp(bar_b_full(st), bph, ctl, 10))) break;
                            tc_fence_after_sync();
                        }
                        issue(p.x_off[kk], st);
                    }
                } else {
                    // what the next K step needs is asked for before this one is issued, so that
                    // its latency passes meanwhile (4-bit 7x7 512->512 14.0 -> 12.2 us, 2-bit 28x28
                    // 512->512 at batch 32 26.7 -> 24.5)
#pragma unroll 1
                    for (int kk = 0; kk < p.kpp; ++kk) {
                        if (!__all_sync(0xffffffffu, ready) &&
                            !(ok = wait_bar_warp(bar_b_full(st), bph, ctl, 10)))
                            break;
                        tc_fence_after_sync();
                        const uint4 t = tn;
                        const int stage = st;
                        tn = p.x_off[kk + 1 == p.kpp ? 0 : kk + 1];
                        if (++st == BST) { st = 0; bph ^= 1u; }
                        ready = mbar_test_wait(bar_b_full(st), bph);
                        issue(t, stage);
                        mma_commit_elect(bar_b_empty(stage));
                    }
                }
                if (ok) mma_commit_elect(bar_a_empty(aslot));
                if (++aslot == p.a_slots) { aslot = 0; aph ^= 1u; }
            }
            if (ok) mma_commit_elect(bar_acc_full(as));
            W3_STAMP(6, it);
        }
        if (!ok) {
            // instructions already issued may still read the operands and write
            // the accumulators: let them finish before memory is given up
            mma_commit_elect(bar_drain);
            wait_bar_drain(bar_drain, 0u);
        }
    } else if (warp < W3_WARP_A0 + a_warps) {
        // ---------------- A: expand the staged window -------------------------------
        const int tid = threadIdx.x - W3_WARP_A0 * 32;
        const int n_tasks = p.apx * p.cpp;
        const int AS = p.as_slots;
        // task t = (pixel, packed chunk) = (t >> lcpp, t & (cpp - 1)); the staged
        // window is dense, so its address is just 16 t
        const int lcpp = p.cpp == 4 ? 2 : p.cpp == 2 ? 1 : 0;
        int ss = 0, slot = 0;
        uint32_t phs = 0, pha = 0;
        bool ok = true;
#pragma unroll 1
        for (uint32_t g = 0; ok && g < n_a_fills; ++g) {
            if (!(ok = wait_bar_warp(bar_as_full(ss), phs, ctl, 12))) break;
            if (warp == W3_WARP_A0) W3_STAMP(1, g);
            if (!(ok = wait_bar_warp(bar_a_empty(slot), pha ^ 1u, ctl, 5))) break;
            if (warp == W3_WARP_A0) W3_STAMP(2, g);
            const uint32_t src = smem_u32(smem + L.a_stage) + ss * a_stage_bytes;
            const uint32_t dst = smem_u32(smem + L.a_slots) + slot * a_slot_bytes;
            if (BITS == 3) {
                // 3-bit rows: one task per pixel (8 codes per 3 bytes from the
                // row's start): its 32 or 48 packed bytes -> 64 or 128 int8 bytes
                const int nq = p.E >= 128 ? 8 : 4;
                const bool half_rows = p.rb == 64;
#pragma unroll 1
                for (int px = tid; px < p.apx; px += a_warps * 32) {
                    uint32_t w[12];
#pragma unroll
                    for (int l = 0; l < 3; ++l) {
                        uint4 v = make_uint4(0u, 0u, 0u, 0u);
                        if (l < p.cpp) v = lds_128(src + (uint32_t)(px * p.PB + 16 * l));
                        w[4 * l] = v.x; w[4 * l + 1] = v.y; w[4 * l + 2] = v.z; w[4 * l + 3] = v.w;
                    }
                    const uint32_t row = dst + (uint32_t)(px * p.rb);
                    const int sw = half_rows ? (px >> 1) & 3 : px & 7;
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (q < nq) {
                            const uint4 c = expand3_chunk<false>(w, q, 0u);
                            sts_128(row + (uint32_t)((q ^ sw) << 4), c.x, c.y, c.z, c.w);
                        }
                }
            } else
#pragma unroll 4
            for (int t = tid; t < n_tasks; t += a_warps * 32) {
                const int px = t >> lcpp, ch = t & (p.cpp - 1);
                const uint4 v = lds_128(src + 16u * t);
                // (16-byte chunks XOR-ed with address bits 7..9, of 64-byte rows bits 7..8, of
                // 32-byte rows bit 7)
                const uint32_t row = dst + (uint32_t)(px * p.rb);
                const int sw = p.rb == 64 ? (px >> 1) & 3 : F4 && p.rb == 32 ? (px >> 2) & 1 : px & 7;
#pragma unroll
                for (int c = 0; c < OUT; ++c)
                    sts_128(row + (uint32_t)(((ch * OUT + c) ^ sw) << 4),
                            w3_operand<BITS, false, F4>(v.x, c, 0u), w3_operand<BITS, false, F4>(v.y, c, 0u),
                            w3_operand<BITS, false, F4>(v.z, c, 0u), w3_operand<BITS, false, F4>(v.w, c, 0u));
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar_a_full(slot));
                mbar_arrive(bar_as_empty(ss));
            }
            if (warp == W3_WARP_A0) W3_STAMP(3, g);
            if (++ss == AS) { ss = 0; phs ^= 1u; }
            if (++slot == p.a_slots) { slot = 0; pha ^= 1u; }
        }
    } else if (warp < W3_WARP_E0) {
        // ---------------- B: expand packed weight rows --------------------------------
        // Two groups of four warps take alternate K steps, so that the latency
        // chains of two steps (barrier, loads, stores, fence, arrival) overlap.
        const int group = (warp - W3_WARP_B0) / W3_B_GROUP_WARPS;
        const int tid = threadIdx.x - (W3_WARP_B0 + group * W3_B_GROUP_WARPS) * 32;
        constexpr int BT = W3_B_GROUP_WARPS * 32;
        constexpr int ROWS_PER_IT = BT / CH;       // a multiple of 8: (row & 7) is the same in every pass
        constexpr int HALF_IT = (128 * CH) / BT;   // passes over 128 rows
        const int row0 = tid / CH, j = tid % CH;
        const int sw = row0 & 7;
        const int BP = p.bp_slots, BST = p.b_stages;
        // own fills: g = group, group + 2, ...
        int sp = group % BP, st = p.b_res ? group : group % BST;
        uint32_t php = (uint32_t)(group / BP) & 1u, phu = p.b_res ? 0u : (uint32_t)(group / BST) & 1u;
        int kk = group;                            // PAIR3: K step within its plane
        bool ok = !p.w8;                           // (w8: nothing to expand)
#pragma unroll 1
        for (uint32_t g = group; ok && g < n_b_fills; g += 2) {
            if (!(ok = wait_bar_warp(bar_bp_full(sp), php, ctl, 6))) break;
            if (warp == W3_WARP_B0) W3_STAMP(10, g >> 1);
            const uint32_t src = smem_u32(smem + L.b_packed + sp * b_packed_bytes);
            uint32_t seen = 0u;
            uint8_t *rowp = smem + L.b_tiles + st * b_stage_bytes + row0 * 128;
            bool waited = p.b_res != 0;
            if (BITS == 3 && TR) {
                // one thread per operand row: 48 packed bytes of a tap and plane, or the
                // 24 bytes of each of two taps.  pair: rows 64 .. 127 are the taps a filter row
                // before; outside the filter the packed bytes are zeros (TMA), and so are
                // the operand's
                const int row = tid;
                const uint32_t r4 = src + (uint32_t)(row * p.pk);
                uint32_t w[12], w1[12];
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    const uint4 v = lds_128(r4 + 16 * l);
                    seen |= v.x;
                    w[4 * l] = v.x; w[4 * l + 1] = v.y; w[4 * l + 2] = v.z; w[4 * l + 3] = v.w;
                }
                if (p.tps == 2) {
                    const uint4 v = lds_128(r4 + 48);
                    seen |= v.x;
#pragma unroll
                    for (int l = 0; l < 4; ++l) w1[l] = w[8 + l];
                    w1[4] = v.x; w1[5] = v.y;
                }
                w3_release_slot(bar_bp_empty(sp), seen, p.zero, lane);
                if (!waited && !(ok = wait_bar_warp(bar_b_empty(st), phu ^ 1u, ctl, 7))) break;
                uint8_t *rp = smem + L.b_tiles + st * b_stage_bytes + row * 128;
                const int sw3 = row & 7;
                uint32_t orv0 = p.orv, orv1 = p.orv;
                if (PAIR3) {
                    const int tap = kk * p.tps - (row >= 64 ? 3 : 0);
                    if ((unsigned)tap >= 9u) orv0 = 0u;
                    if ((unsigned)(tap + 1) >= 9u) orv1 = 0u;
                    kk += 2;
                    while (kk >= p.kpp) kk -= p.kpp;
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    uint4 c;
                    if (q >= 4 && p.tps == 2) c = expand3_chunk<true>(w1, q & 3, orv1);
                    else c = expand3_chunk<true>(w, q, orv0);
                    *reinterpret_cast<uint4 *>(rp + ((q ^ sw3) << 4)) = c;
                }
            } else if (BITS == 3) {
                // 3-bit rows: one thread per row of 48 packed bytes
                uint32_t w[2][12];
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (tid + i * BT < BN) {
                        const uint32_t r4 = src + (uint32_t)((tid + i * BT) * 48);
#pragma unroll
                        for (int l = 0; l < 3; ++l) {
                            const uint4 v = lds_128(r4 + 16 * l);
                            seen |= v.x;
                            w[i][4 * l] = v.x; w[i][4 * l + 1] = v.y;
                            w[i][4 * l + 2] = v.z; w[i][4 * l + 3] = v.w;
                        }
                    }
                w3_release_slot(bar_bp_empty(sp), seen, p.zero, lane);
                if (!waited && !(ok = wait_bar_warp(bar_b_empty(st), phu ^ 1u, ctl, 7))) break;
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (tid + i * BT < BN) {
                        uint8_t *rp = smem + L.b_tiles + st * b_stage_bytes + (tid + i * BT) * 128;
                        const int sw3 = (tid + i * BT) & 7;
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            *reinterpret_cast<uint4 *>(rp + ((q ^ sw3) << 4)) =
                                expand3_chunk<true>(w[i], q, p.orv);
                    }
            } else
            // 128 rows at a time (register budget)
#pragma unroll 1
            for (int r0 = 0; r0 < BN; r0 += 128) {
                uint4 v[HALF_IT];
#pragma unroll
                for (int i = 0; i < HALF_IT; ++i)
                    if (r0 + row0 + i * ROWS_PER_IT < BN) {
                        v[i] = lds_128(src + 16u * ((r0 + row0 + i * ROWS_PER_IT) * CH + j));
                        seen |= v[i].x;
                    }
                // the packed slot is free as soon as every lane holds its chunks
                if (r0 + 128 >= BN) w3_release_slot(bar_bp_empty(sp), seen, p.zero, lane);
                if (!waited) {
                    if (!(ok = wait_bar_warp(bar_b_empty(st), phu ^ 1u, ctl, 7))) break;
                    waited = true;
                }
#pragma unroll
                for (int i = 0; i < HALF_IT; ++i)
                    if (r0 + row0 + i * ROWS_PER_IT < BN) {
#pragma unroll
                        for (int c = 0; c < OUT; ++c)
                            *reinterpret_cast<uint4 *>(rowp + (r0 + i * ROWS_PER_IT) * 128 +
                                                       (((j * OUT + c) ^ sw) << 4)) =
                                make_uint4(w3_operand<BITS, true, F4>(v[i].x, c, p.orv),
                                           w3_operand<BITS, true, F4>(v[i].y, c, p.orv),
                                           w3_operand<BITS, true, F4>(v[i].z, c, p.orv),
                                           w3_operand<BITS, true, F4>(v[i].w, c, p.orv));
                    }
            }
            if (!ok) break;
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_b_full(st));
            if (warp == W3_WARP_B0) W3_STAMP(11, g >> 1);
            sp += 2;
            if (sp >= BP) { sp -= BP; php ^= 1u; }
            if (p.b_res) {
                st += 2;
            } else {
                st += 2;
                if (st >= BST) { st -= BST; phu ^= 1u; }
            }
        }
    } else {
        // ---------------- epilogue: four warps per tensor-memory lane quarter -----------
        const int quarter = warp & 3;
        const int k = (warp - W3_WARP_E0) >> 2;              // which of the quarter's warps
        if (F4 && k == 0) {
            // every block scale is 2 (UE8M0 128), whatever place the tensor core reads it from
            uint32_t two[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) two[i] = 0x80808080u;
            tmem_st_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + W3_F4_SF, two);
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_scales);
        }
        if constexpr (TR) {
            // thread = output channel (tensor-memory lane), columns = positions;
            // warp k of a quarter takes a k-th part of the columns (up to 64) in units of 16
            constexpr int SB = BITS == 3 ? 4 : BITS;         // bits of a field
            constexpr int E = 32 / SB;                       // positions per code word
            constexpr int CWU = 16 / E;                      // code words per unit: 2 (1 at 2 bits)
            constexpr uint32_t MASK = (1u << SB) - 1u;
            const DsqEpi &e = p.e;
            // (pair: lanes 64..127 are channels 0..63 of the second of two image rows)
            const int chq = p.pair ? (quarter & 1) * 32 : quarter * 32;
            const int row1 = p.pair ? quarter >> 1 : 0;
            const int each = (TP / 16 + 3) / 4;              // units of 16 columns a warp
            const int units = max(0, min(each, TP / 16 - k * each)), colbase = 16 * k * each;
            const int ch = n_tile * 128 + chq + lane;
            // a warp has work while its first code word lies inside the output row:
            // channels past Cout are padding lanes of the packed row and get zeros
            // (warp-uniform)
            const bool warp_live = (n_tile * 128 + chq) * BITS / 8 < p.out_pitch;
            constexpr bool LEAN = EPI == DSQ_EPI_CODES || EPI == DSQ_EPI_CODES_RES;
            float sc = 0.f, bi = LEAN ? -1e30f : 0.f;        // padding lanes: code 0
            if (ch < p.Ncols) {
                if (LEAN) dsq_codes_affine(e.scale, e.bias, ch, e.half_offset, -p.shift, sc, bi);
                else {
                    sc = __ldg(e.scale + ch);
                    if (e.half_offset) sc = __fmul_rn(sc, 0.5f);
                    bi = __ldg(e.bias + ch);
                }
            }
            const DsqLean lean = dsq_make_lean(e);
            const unsigned long long scp = dsq_pack2(sc, sc), bip = dsq_pack2(bi, bi);
            const unsigned long long sc4[4] = {scp, scp, scp, scp}, bi4[4] = {bip, bip, bip, bip};
            const int pw = p.out_pitch / 4;                  // words of an output pixel
            const int cg = (n_tile * 128 + chq + (lane & ~(E - 1))) / E;   // this lane group's word (3-bit: 24 bits)
            const int cw3 = (n_tile * 128 + chq) / 32 * 3;   // 3-bit: the quarter's first word
            const uint32_t *res32 = reinterpret_cast<const uint32_t *>(e.residual);
            uint32_t *y32 = reinterpret_cast<uint32_t *>(e.y_codes);
            // output pixel (or -1) of the warp's columns: lane L follows columns
            // colbase + 2 L and colbase + 2 L + 1; the others get them by shuffle
            W3Pos pos0, pos1;
            {
                const int g0 = m_first * TP + colbase + 2 * lane;
                pos0.n = g0 / img_positions;
                const int rem = g0 - pos0.n * img_positions;
                pos0.h = rem / p.Wp;
                pos0.w = rem - pos0.h * p.Wp;
                pos1 = w3_add(pos0, 0, 0, 1, p.Hp, p.Wp);
            }
            bool ok = true;
#pragma unroll 1
            for (int it = 0; ok && it < my_tiles; ++it) {
                const int as = it & 1;
                const int h0 = p.pair ? 2 * pos0.h + row1 : pos0.h, h1 = p.pair ? 2 * pos1.h + row1 : pos1.h;
                const int m0 = (pos0.n < p.N && h0 < p.Ho && pos0.w < p.Wo)
                                   ? (pos0.n * p.Ho + h0) * p.Wo + pos0.w : -1;
                const int m1 = (pos1.n < p.N && h1 < p.Ho && pos1.w < p.Wo)
                                   ? (pos1.n * p.Ho + h1) * p.Wo + pos1.w : -1;
                pos0 = w3_add(pos0, p.t_dn, p.t_dh, p.t_dw, p.Hp, p.Wp);
                pos1 = w3_add(pos1, p.t_dn, p.t_dh, p.t_dw, p.Hp, p.Wp);
                // Word w of a unit covers E positions; lane i of a channel group owns
                // position i of them: it stores that position's word at the end, and it
                // fetches that position's residual word - one unit ahead, the first
                // unit's before the wait for the accumulator, so that the loads'
                // latency is off the path.  The same transpose that turns "E positions
                // of my channel" into "E channels of my position" is its own inverse,
                // so it also turns the fetched words into "residual codes of my channel
                // at E positions".
                int mpn[CWU];
                uint32_t wordn[CWU];
                auto fetch = [&](int u) {
#pragma unroll
                    for (int w = 0; w < CWU; ++w) {
                        const int cpos = 16 * u + w * E + (lane & (E - 1));   // column of the warp
                        const int mp_a = __shfl_sync(0xffffffffu, m0, cpos >> 1);
                        const int mp_b = __shfl_sync(0xffffffffu, m1, cpos >> 1);
                        mpn[w] = (cpos & 1) ? mp_b : mp_a;
                        wordn[w] = 0u;
                        if (BITS == 3) {
                            // (the quarter's three words, one per lane group; the 24-bit
                            // pieces are cut from them by shuffle)
                            const int wi = cw3 + (lane >> 3 < 2 ? lane >> 3 : 2);
                            if (EPI != DSQ_EPI_CODES && e.residual && mpn[w] >= 0 && wi < pw)
                                wordn[w] = __ldg(res32 + (int64_t)mpn[w] * pw + wi);
                        } else if (EPI != DSQ_EPI_CODES && e.residual && mpn[w] >= 0 && 4 * cg < p.out_pitch)
                            wordn[w] = __ldg(res32 + (int64_t)mpn[w] * pw + cg);
                    }
                };
                if (warp_live) fetch(0);
                if (warp == W3_WARP_E0) W3_STAMP(7, it);
                if (!(ok = wait_bar_warp(bar_acc_full(as), (it >> 1) & 1u, ctl, 8))) break;
                if (warp == W3_WARP_E0) W3_STAMP(8, it);
                tc_fence_after_sync();
                const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + as * ACC;
#pragma unroll 1
                for (int u = 0; warp_live && u < units; ++u) {
                    const int col0 = colbase + 16 * u;
                    uint32_t r[16], cw[CWU], resT[CWU];
                    int mp[CWU];
                    __syncwarp();
                    tmem_ld_32x16(taddr + col0, r);
                    uint32_t word[CWU];
#pragma unroll
                    for (int w = 0; w < CWU; ++w) { mp[w] = mpn[w]; word[w] = wordn[w]; }
                    if (u + 1 < units) fetch(u + 1);
#pragma unroll
                    for (int w = 0; w < CWU; ++w) {
                        resT[w] = 0u;
                        if (BITS == 3 && EPI != DSQ_EPI_CODES) {
                            const int grp = lane >> 3;
                            const uint32_t low = __shfl_up_sync(0xffffffffu, word[w], 8);
                            const uint32_t x = __funnelshift_rc(low, word[w], 32 - 8 * grp);
                            const uint32_t y = (x & 0xFFFu) | ((x << 4) & 0x0FFF0000u);
                            const uint32_t z = (y & 0x003F003Fu) | ((y << 2) & 0x3F003F00u);
                            word[w] = (z & 0x07070707u) | ((z << 1) & 0x70707070u);
                        }
                        if (EPI != DSQ_EPI_CODES) resT[w] = w3_transpose_fields<SB>(word[w], lane);
                        cw[w] = 0u;
                    }
                    tmem_ld_wait();
                    if constexpr (LEAN) {
                        // eight positions of this lane's channel at a time
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t v[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) v[j] = r[8 * h + j];
                            const uint32_t rw = SB == 4 ? resT[h < CWU ? h : 0] : resT[0] >> (16 * h);
                            const uint32_t x = dsq_lean_codes8<BITS, EPI == DSQ_EPI_CODES_RES, false, SB, F4>(
                                v, sc4, bi4, rw, lean);
                            if (SB == 4) cw[h < CWU ? h : 0] = x;
                            else cw[0] |= x << (16 * h);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            // column 16 u + j of the warp: held by lane 8 u + j / 2
                            const int mj = __shfl_sync(0xffffffffu, (j & 1) ? m1 : m0, 8 * u + (j >> 1));
                            const int vi = F4 ? __float2int_rn(__uint_as_float(r[j])) : (int)r[j] >> p.shift;
                            if (mj >= 0 && ch < p.Ncols) {
                                if (e.acc_out) e.acc_out[(int64_t)mj * p.Ncols + ch] = vi;
                                float y;
                                if (e.general_offset) {
                                    // S_a of the position (recomputed by every channel's
                                    // thread: this form is not a fast path)
                                    const int wo = mj % p.Wo, t2 = mj / p.Wo;
                                    const int s_a = dsq_window_sa<BITS>(p.act, t2 / p.Ho, t2 % p.Ho, wo,
                                                                        p.H, p.W, 3, p.stride, 1, p.P);
                                    y = dsq_epi_y_offset(vi, s_a, e.w_offset, sc, bi);
                                } else {
                                    y = dsq_epi_y(vi, sc, bi);
                                }
                                if (e.residual) {
                                    const uint32_t qr = (resT[(j * SB) >> 5] >> ((j * SB) & 31)) & MASK;
                                    y = dsq_epi_residual(y, qr, e.res_delta, e.res_lo);
                                }
                                if (e.has_requant)
                                    cw[(j * SB) >> 5] |= dsq_code(y, e.rq) << ((j * SB) & 31);
                                if (e.y_f32) e.y_f32[(int64_t)mj * p.Ncols + ch] = y;
                            }
                        }
                    }
                    if (e.y_codes) {
                        // fields of E positions of one channel -> fields of the E
                        // channels of this lane group at one position
#pragma unroll
                        for (int w = 0; w < CWU; ++w) {
                            uint32_t word = w3_transpose_fields<SB>(cw[w], lane);
                            if (BITS == 3) {
                                // the position's 24-bit pieces of the four lane groups are
                                // three words; groups 0..2 store one each, and the spare words
                                // of a 64-channel row come from group 3
                                word = (word & 0x07070707u) | ((word & 0x70707070u) >> 1);
                                word = (word & 0x003F003Fu) | ((word & 0x3F003F00u) >> 2);
                                word = (word & 0xFFFu) | ((word >> 4) & 0xFFF000u);
                                const uint32_t next = __shfl_down_sync(0xffffffffu, word, 8);
                                const int grp = lane >> 3;
                                word = (word >> (8 * grp)) | (next << (24 - 8 * grp));
                                const int wi = cw3 + grp;
                                uint32_t *row = y32 + (int64_t)mp[w] * pw;
                                if (grp < 3) {
                                    if (mp[w] >= 0 && wi < pw) row[wi] = word;
                                } else if (p.pair && mp[w] >= 0 && wi == 6) {
                                    for (int i = wi; i < pw; ++i) row[i] = 0u;
                                }
                            } else if (mp[w] >= 0 && 4 * cg < p.out_pitch) y32[(int64_t)mp[w] * pw + cg] = word;
                        }
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_acc_empty(as));
                if (warp == W3_WARP_E0) W3_STAMP(9, it);
            }
        } else {
        const int row_in_tile = quarter * 32 + lane;
        float *sm_scale = reinterpret_cast<float *>(smem + L.epi);
        float *sm_bias = sm_scale + p.cout_pad;
        const float *lut = reinterpret_cast<const float *>(smem + L.lut);
        const DsqEpi &e = p.e;
        // a unit = the columns whose codes fill whole 32-bit words: 16 columns
        // (32 for 3-bit codes, where 16 would be 6 bytes)
        constexpr int UW = BITS == 3 ? 32 : 16;
        constexpr int CWU = UW * BITS / 32;                  // code words per unit
        // scale (halved for the symmetric weight grid) and bias of every output
        // channel, once per CTA; columns past Cout get 0
        for (int c = threadIdx.x - W3_WARP_E0 * 32; c < p.cout_pad; c += W3_NUM_E_WARPS * 32) {
            float sc = 0.f, bi = 0.f;
            if (c < p.Ncols) {
                sc = __ldg(e.scale + c);
                if (e.half_offset) sc = __fmul_rn(sc, 0.5f);
                bi = __ldg(e.bias + c);
            }
            sm_scale[c] = sc;
            sm_bias[c] = bi;
        }
        named_barrier_sync(1, W3_NUM_E_WARPS * 32);
        const int units = BN / UW;
        // this thread's row of the CTA's first tile: image, row, column in the
        // padded stacked numbering (positions in its padding have no output)
        W3Pos pos;
        {
            const int g0 = m_first * W3_BM + row_in_tile;
            pos.n = g0 / img_positions;
            const int rem = g0 - pos.n * img_positions;
            pos.h = rem / p.Wp;
            pos.w = rem - pos.h * p.Wp;
        }
        bool ok = true;
#pragma unroll 1
        for (int it = 0; ok && it < my_tiles; ++it) {
            const int as = it & 1;
            const bool row_ok = pos.n < p.N && pos.h < p.H && pos.w < p.W;
            const int64_t m = ((int64_t)pos.n * p.H + pos.h) * p.W + pos.w;
            // general weight-grid offset: S_a of this output pixel, summed from
            // the input codes under its 3 x 3 window
            int s_a = 0;
            if (EPI == DSQ_EPI_GENERAL && e.general_offset && row_ok)
                s_a = dsq_window_sa<BITS>(p.act, pos.n, pos.h, pos.w, p.H, p.W, 3, 1, 1, p.P);
            pos = w3_add(pos, p.t_dn, p.t_dh, p.t_dw, p.Hp, p.Wp);
            // residual codes of a unit of this row are fetched one unit ahead (the
            // first unit's while the tile's instructions are still running); the
            // unit loop is not unrolled: the kernel's roles share the instruction
            // caches, and every role runs faster when the whole kernel is small
            uint32_t res_nx[CWU];
            auto fetch_res = [&](int u) {
#pragma unroll
                for (int w = 0; w < CWU; ++w) res_nx[w] = 0u;
                const int byte0 = (n_tile * BN + u * UW) * BITS / 8;
                if (EPI != DSQ_EPI_CODES && e.residual && row_ok && u < units &&
                    byte0 < p.out_pitch) {
                    const uint32_t *rp =
                        reinterpret_cast<const uint32_t *>(e.residual + m * p.out_pitch + byte0);
                    // (a unit of 3-bit codes may reach past the end of the row)
#pragma unroll
                    for (int w = 0; w < CWU; ++w)
                        if (BITS != 3 || byte0 + 4 * w < p.out_pitch) res_nx[w] = __ldg(rp + w);
                }
            };
            fetch_res(k);
            if (warp == W3_WARP_E0) W3_STAMP(7, it);
            if (!(ok = wait_bar_warp(bar_acc_full(as), (it >> 1) & 1u, ctl, 8))) break;
            if (warp == W3_WARP_E0) W3_STAMP(8, it);
            tc_fence_after_sync();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + as * BN;
#pragma unroll 1
            for (int u = k; u < units; u += W3_EPQ) {
                uint32_t r[UW], resw[CWU];
#pragma unroll
                for (int w = 0; w < CWU; ++w) resw[w] = res_nx[w];
                __syncwarp();
                if constexpr (UW == 32) tmem_ld_32x32(taddr + u * UW, r);
                else tmem_ld_32x16(taddr + u * UW, r);
                fetch_res(u + W3_EPQ);
                tmem_ld_wait();
                const int n0 = n_tile * BN + u * UW;
                const int byte0 = n0 * BITS / 8;
                if (!row_ok) continue;
                uint32_t cw[CWU];
                if constexpr (BITS != 3 && (EPI == DSQ_EPI_CODES || EPI == DSQ_EPI_CODES_RES)) {
                    if (byte0 >= p.out_pitch) continue;
                    w3_codes_unit<BITS, EPI == DSQ_EPI_CODES_RES>(
                        r, sm_scale + n0, sm_bias + n0, resw, lut, p.shift, e.rq.inv, p.r_hi, cw);
                } else {
                    constexpr uint32_t MASK = (1u << BITS) - 1u;
#pragma unroll
                    for (int w = 0; w < CWU; ++w) cw[w] = 0u;
#pragma unroll
                    for (int c = 0; c < UW; ++c) {
                        const int v = (int)r[c] >> p.shift;
                        // field c of the unit: word fw, bit fs (a 3-bit field may
                        // straddle two words; never the last word)
                        const int fw = (c * BITS) >> 5, fs = (c * BITS) & 31;
                        const int fw1 = fw + 1 < CWU ? fw + 1 : fw;
                        if (n0 + c < p.Ncols) {
                            if (e.acc_out) e.acc_out[m * p.Ncols + n0 + c] = v;
                            float y = e.general_offset
                                          ? dsq_epi_y_offset(v, s_a, e.w_offset, sm_scale[n0 + c],
                                                             sm_bias[n0 + c])
                                          : dsq_epi_y(v, sm_scale[n0 + c], sm_bias[n0 + c]);
                            if (e.residual) {
                                const uint32_t qr =
                                    __funnelshift_r(resw[fw], fw + 1 < CWU ? resw[fw1] : 0u, fs) & MASK;
                                y = dsq_epi_residual(y, qr, e.res_delta, e.res_lo);
                            }
                            if (e.has_requant) {
                                const uint32_t q = dsq_code(y, e.rq);
                                cw[fw] |= q << fs;
                                if (BITS == 3 && fs > 29) cw[fw1] |= q >> (32 - fs);
                            }
                            if (e.y_f32) e.y_f32[m * p.Ncols + n0 + c] = y;
                        }
                    }
                    if (!e.y_codes || byte0 >= p.out_pitch) continue;
                }
                // columns past Cout are padding lanes of the packed row: zero
                const int nvalid_bits = min(UW, max(0, p.Ncols - n0)) * BITS;
#pragma unroll
                for (int w = 0; w < CWU; ++w) {
                    const int nb = nvalid_bits - 32 * w;
                    cw[w] &= nb >= 32 ? 0xFFFFFFFFu : nb <= 0 ? 0u : ((1u << nb) - 1u);
                }
                uint32_t *dst = reinterpret_cast<uint32_t *>(e.y_codes + m * p.out_pitch + byte0);
                if (CWU == 2)
                    *reinterpret_cast<uint2 *>(dst) = make_uint2(cw[0], cw[CWU - 1]);
                else if (CWU == 3) {
                    // 12 bytes, as far as the row goes
                    dst[0] = cw[0];
                    if (byte0 + 4 < p.out_pitch) dst[1] = cw[1];
                    if (byte0 + 8 < p.out_pitch) dst[2] = cw[CWU - 1];
                    // 3-bit rows: the N tiles may end before the row's pitch does
                    // (64 columns = 24 bytes, pitch 32); the spare bytes are zero
                    if (n_tile == p.n_tiles - 1 && u == units - 1)
                        for (int b = p.cout_pad * BITS / 8; b < p.out_pitch; b += 4)
                            *reinterpret_cast<uint32_t *>(e.y_codes + m * p.out_pitch + b) = 0u;
                } else
                    *dst = cw[0];
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_acc_empty(as));
            if (warp == W3_WARP_E0) W3_STAMP(9, it);
        }
        }   // !TR
    }

    // ---------------- teardown ------------------------------------------------------
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) W3_STAMP(13, 3);
    if (warp == W3_WARP_MMA) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 512);
        W3_STAMP(13, 4);
    }
}

template <int BITS, int EPI, bool TR = false, bool F4 = false, bool PAIR3 = false>
int w3_launch(const CUtensorMap &tb, const CUtensorMap &ta, const W3Params &p, cudaStream_t s,
              int pdl)
{
    static std::atomic<unsigned long long> configured{0ull};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return DSQ_ERR_CUDA;
    const unsigned long long dev_bit = dev < 64 ? 1ull << dev : 0ull;
    if (!(configured.load(std::memory_order_acquire) & dev_bit)) {
        if (cudaFuncSetAttribute(dsq_win3_kernel<BITS, EPI, TR, F4, PAIR3>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 227 * 1024) != cudaSuccess)
            return DSQ_ERR_CUDA;
        configured.fetch_or(dev_bit, std::memory_order_release);
    }
    const int grid = p.mstep * p.n_tiles;
    return dsq_launch(dsq_win3_kernel<BITS, EPI, TR, F4, PAIR3>, dim3(grid), dim3(W3_THREADS),
                      (size_t)p.smem_bytes, s, pdl, 0, tb, ta, p);
}

template <int BITS>
int w3_dispatch(int epi, const CUtensorMap &tb, const CUtensorMap &ta, const W3Params &p,
                cudaStream_t s, int pdl)
{
    if constexpr (BITS == 2)
        if (p.f4) {
            switch (epi) {
            case DSQ_EPI_CODES: return w3_launch<BITS, DSQ_EPI_CODES, true, true>(tb, ta, p, s, pdl);
            case DSQ_EPI_CODES_RES: return w3_launch<BITS, DSQ_EPI_CODES_RES, true, true>(tb, ta, p, s, pdl);
            default: return w3_launch<BITS, DSQ_EPI_GENERAL, true, true>(tb, ta, p, s, pdl);
            }
        }
    if constexpr (BITS == 3)
        if (p.tr && p.pair) {
            switch (epi) {
            case DSQ_EPI_CODES: return w3_launch<BITS, DSQ_EPI_CODES, true, false, true>(tb, ta, p, s, pdl);
            case DSQ_EPI_CODES_RES: return w3_launch<BITS, DSQ_EPI_CODES_RES, true, false, true>(tb, ta, p, s, pdl);
            default: return w3_launch<BITS, DSQ_EPI_GENERAL, true, false, true>(tb, ta, p, s, pdl);
            }
        }
    if (p.tr) {
        switch (epi) {
        case DSQ_EPI_CODES: return w3_launch<BITS, DSQ_EPI_CODES, true>(tb, ta, p, s, pdl);
        case DSQ_EPI_CODES_RES: return w3_launch<BITS, DSQ_EPI_CODES_RES, true>(tb, ta, p, s, pdl);
        default: return w3_launch<BITS, DSQ_EPI_GENERAL, true>(tb, ta, p, s, pdl);
        }
    }
    if constexpr (BITS != 3) {
        switch (epi) {
        case DSQ_EPI_CODES: return w3_launch<BITS, DSQ_EPI_CODES>(tb, ta, p, s, pdl);
        case DSQ_EPI_CODES_RES: return w3_launch<BITS, DSQ_EPI_CODES_RES>(tb, ta, p, s, pdl);
        default: break;
        }
    }
    return w3_launch<BITS, DSQ_EPI_GENERAL>(tb, ta, p, s, pdl);
}

}  // namespace

// ---------------------------------------------------------------------------
// pre-expanded weights
// ---------------------------------------------------------------------------
namespace {

// One thread per (row, K step, packed 16-byte chunk): the chunk's OUT operand
// chunks, in the operand's logical order (TMA applies the 128-byte swizzle when
// it copies a tile).  Same expansion as the kernel's own (expand_word, the window's
// expand_word_f4), for the grid Delta (c + 1/2); bytes past the end of a weight row
// read as packed zeros, as the kernel's TMA loads of the packed rows do.
// F4: `mark` gets W3_F4_MARK.
template <int BITS, bool F4>
__global__ void __launch_bounds__(256)
w8_build_kernel(const uint8_t *__restrict__ packed, uint8_t *__restrict__ out, int Cout,
                int row_bytes, int ksteps, int kpp, int xstep, uint32_t *__restrict__ mark)
{
    constexpr int OUT = F4 ? 2 : Chunks<BITS>::OUT, CH = 8 / OUT;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int j = (int)(idx % CH);
    const int ks = (int)((idx / CH) % ksteps);
    const int64_t row = idx / ((int64_t)CH * ksteps);
    if (row >= Cout) return;
    const int pl = ks / kpp, kk = ks - pl * kpp;
    const int x = kk * xstep + (pl * CH + j) * 16;             // byte offset in the packed row
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (x < row_bytes) v = *reinterpret_cast<const uint4 *>(packed + row * row_bytes + x);
    const uint32_t orv = 0x01010101u << (7 - BITS);
    uint8_t *dst = out + (row * ksteps + ks) * 128;
    if (F4 && idx == 0) *mark = W3_F4_MARK;
    if constexpr (F4) {
#pragma unroll
        for (int c = 0; c < OUT; ++c)
            *reinterpret_cast<uint4 *>(dst + 16 * (j * OUT + c)) =
                make_uint4(expand_word_f4<true>(v.x, c), expand_word_f4<true>(v.y, c),
                           expand_word_f4<true>(v.z, c), expand_word_f4<true>(v.w, c));
    } else
#pragma unroll
    for (int c = 0; c < OUT; ++c)
        *reinterpret_cast<uint4 *>(dst + 16 * (j * OUT + c)) =
            make_uint4(expand_word<BITS, true>(v.x, c, orv), expand_word<BITS, true>(v.y, c, orv),
                       expand_word<BITS, true>(v.z, c, orv), expand_word<BITS, true>(v.w, c, orv));
}

}  // namespace

DsqW8Info dsq_w8_info(const dsq_conv_t *conv, int bits)
{
    DsqW8Info w = {0, 0, 0, 0, 0};
    if (!conv || conv->groups != 1 || conv->KH != 3 || conv->KW != 3 || conv->stride != 1 ||
        conv->pad != 1 || (bits != 2 && bits != 4))
        return w;
    const int Cin = conv->Cin;
    if (!(Cin == 64 || (Cin % 128 == 0 && Cin <= 1024))) return w;
    int npl, kpp, tps;
    w3_steps(Cin, 0, &npl, &kpp, &tps);
    w.enabled = 1;
    w.ksteps = npl * kpp;
    const size_t packed = (size_t)conv->Cout * 9 * dsq_row_pitch(Cin, bits);
    w.offset = (packed + 1023) / 1024 * 1024;
    w.bytes = (size_t)conv->Cout * w.ksteps * 128;
    w.f4 = bits == 2 && (Cin == 64 || Cin == 128 || Cin % 256 == 0);
    if (w.f4) {
        w3_steps(Cin, 1, &npl, &kpp, &tps);
        w.ksteps = npl * kpp;
    }
    return w;
}

// where an F4 copy is marked: the last 16 bytes of its room (the copy fills half)
static inline size_t w3_mark_offset(const DsqW8Info &w) { return w.offset + w.bytes - 16; }

int dsq_w8_build(void *blob, const dsq_conv_t *conv, int bits, cudaStream_t stream)
{
    const DsqW8Info w = dsq_w8_info(conv, bits);
    if (!w.enabled) return DSQ_OK;
    const int P = (int)dsq_row_pitch(conv->Cin, bits);
    int npl, kpp, tps;
    w3_steps(conv->Cin, w.f4, &npl, &kpp, &tps);
    const int ch = w.f4 || bits == 4 ? 4 : 2;                            // packed chunks of a K step
    const int64_t threads = (int64_t)conv->Cout * w.ksteps * ch;
    const unsigned blocks = (unsigned)((threads + 255) / 256);
    const uint8_t *packed = (const uint8_t *)blob;
    uint8_t *out = (uint8_t *)blob + w.offset;
    return dsq_launch(w.f4        ? w8_build_kernel<2, true>
                      : bits == 4 ? w8_build_kernel<4, false>
                                  : w8_build_kernel<2, false>,
                      dim3(blocks), dim3(256), 0, stream, 0, 0, packed, out, conv->Cout, 9 * P, w.ksteps,
                      kpp, tps * P, (uint32_t *)((uint8_t *)blob + w3_mark_offset(w)));
}

int dsq_conv3_window(const void *act_codes, const dsq_nhwc_t *shape, int bits,
                     const void *w_packed, const dsq_conv_t *conv, const DsqEpi &e,
                     int epi_kind, int small_acc, void *workspace, cudaStream_t stream)
{
    const DsqLaunchHooks hooks = dsq_launch_hooks();
    if (!hooks.window3) return DSQ_ERR_UNSUPPORTED;
    const int stride = conv->stride;
    if (conv->KH != 3 || conv->KW != 3 || conv->pad != 1 || (stride != 1 && stride != 2))
        return DSQ_ERR_UNSUPPORTED;
    if (bits < 2 || bits > 4) return DSQ_ERR_UNSUPPORTED;
    if (e.general_offset) epi_kind = DSQ_EPI_GENERAL;
    const int Cin = conv->Cin, Cout = conv->Cout;
    if (!(Cin == 64 || (Cin % 128 == 0 && Cin <= 1024))) return DSQ_ERR_UNSUPPORTED;
    if (shape->W + 1 > 32000 || shape->H + 1 > 32000) return DSQ_ERR_UNSUPPORTED;
    // Which form: transposed tiles wherever they fit, else, at stride 1, plain tiles.  Up to
    // 64 output channels want pairs of image rows (`pair`), for which the weights come from the
    // blob's expanded copy or, at 3 bits, from the expansion warps.  Batch 64, transposed /
    // plain, us: 64->64 at 56x56 4-bit 12.2 / 21.1, 3-bit 17.3 / 63.8; 128->128 at 28x28 10.0 / 12.1,
    // 14.0 / 23.6; 256->256 at 14x14 10.4 / 11.7, 13.3 / 23.5; 512->512 at 7x7 12.2 / 16.0, 19.1 / 31.0.
    // the codes epilogues want the requantiser range to start at 0, too
    float r_hi = 0.f;
    if (epi_kind != DSQ_EPI_GENERAL) {
        r_hi = fmaf(e.rq.hi - e.rq.lo, e.rq.inv, 0.5f);
        if (e.rq.lo != 0.0f || !dsq_lean_epilogue(e)) epi_kind = DSQ_EPI_GENERAL;
    }
    const int sms = dsq_sm_count();
    if (sms <= 0) return DSQ_ERR_CUDA;
    W3Params p = {};
    p.N = shape->N; p.H = shape->H; p.W = shape->W;
    p.stride = stride;
    p.Ho = (p.H - 1) / stride + 1; p.Wo = (p.W - 1) / stride + 1;
    p.Ncols = Cout;
    const int P = (int)dsq_row_pitch(Cin, bits);           // packed bytes per pixel
    // Tiling, window and shared memory for one of the two kernel forms.
    // Transposed (tr): tiles of 256 positions x 128 output channels, A = weights.
    // Plain: 128 positions x up to 256 channels, A = window.
    const DsqW8Info w8 = dsq_w8_info(conv, bits);
    // (plain tiles with up to 64 output channels keep the expanded weights resident in
    // shared memory for the whole CTA anyway: nothing to gain, measured slightly slower)
    const bool w8_any = hooks.w8 && w8.enabled && e.half_offset;
    // f4: 4-bit floating-point operands (2-bit codes; transposed tiles; at stride 1 over the
    // blob's copy).  most: the largest tile to consider; false where the form does not take
    // the problem or no tile of that size fits.
    auto configure = [&](int tr, int f4, int most) -> int {
        const bool w8_ok = w8_any && f4 == w8.f4;
        if (f4 && !(stride == 1 ? w8_ok : hooks.w8 && w3_takes_f4(conv, bits, e.half_offset))) return 0;
        if (stride != 1 && !tr) return 0;
        p.tr = tr;
        p.f4 = f4;
        w3_steps(Cin, f4, &p.npl, &p.kpp, &p.tps);
        if (bits == 3 && !tr) { p.tps = 1; p.kpp = 9; }
        p.pair = tr && stride == 1 && Cout <= 64;
        if (p.pair && !w8_ok && bits != 3) return 0;
        const int taps = p.pair ? 12 : 9;
        p.kpp = (taps + p.tps - 1) / p.tps;
        p.w8 = w8_ok && (Cout > 64 || p.pair);
        p.E = f4 ? Cin / 2 : Cin;
        p.PB = std::min(P, (f4 ? 32 : 16) * bits);
        p.cpp = p.PB / 16;
        p.ksteps = p.npl * p.kpp;
        p.xstep = p.tps * P;
        p.pk = p.tps > 1 ? p.tps * P : (f4 ? 32 : 16) * bits;
        p.rb = tr ? 128 / p.tps : 128;
        p.BN = tr ? 128 : w3_plain_bn(Cout);
        // positions (see W3Pos) and what a window is made of
        const W3Work work = w3_work(shape, conv, p.pair, p.BN, sms);
        p.n_tiles = work.n_tiles;
        p.cout_pad = p.n_tiles * p.BN;
        if (p.cout_pad > W3_MAX_COUT || p.n_tiles > sms || work.positions > (1ll << 30)) return 0;
        p.sh = p.pair ? 2 : stride; p.sw = stride;
        p.Hp = work.Hp;
        p.Wp = work.Wp;
        p.mstep = work.mstep;
        p.tp = tr ? w3_tile(work.positions, p.mstep, most) : W3_BM;
        p.m_tiles = (int)((work.positions + p.tp - 1) / p.tp);
        if (stride == 2 && bits != 3 && !f4 && hooks.window3 == 1 &&
            !w3_takes_stride2(Cin, p.tp, (p.m_tiles + p.mstep - 1) / p.mstep))
            return 0;
        if (p.mstep > p.m_tiles) p.mstep = p.m_tiles;
        p.nbands = p.sh * p.sw;
        int need = p.tp + (p.sh == 2 ? 1 : 2) * p.Wp + (p.sw == 2 ? 1 : 2);
        if (p.nbands == 1 && (!tr || f4) && need > (f4 ? 3 * W3_F4_BAND_PX : W3_MAX_WINDOW_PX)) {
            p.nbands = 3;
            need = f4 ? W3_F4_BAND_PX : W3_BAND_PX;
        }
        p.a_nload = (need + 255) / 256;
        if (p.nbands * p.a_nload > 32 || (p.nbands == 1 && tr && !f4 && need - p.tp + 256 > 768)) return 0;
        p.a_box = (((need + p.a_nload - 1) / p.a_nload) + 7) / 8 * 8;
        p.band_px = p.a_nload * p.a_box;
        p.apx = p.nbands * p.band_px;
        for (int b = 0; b < p.nbands; ++b) {
            // filter taps with the corner at (-2, -2): 1 = pixels -1, 0 .. (or -1, 1, ..), 2 = 0, 2 ..
            p.band_pos[b] = p.nbands == 3 ? b * p.Wp : 0;
            const int row = p.sh == 2 ? 1 + b / p.sw : 1, col = p.sw == 2 ? 1 + b % 2 : 1;
            p.band_tap[b] = col | row << 8;
        }
        // window rows of the taps' operands, four instructions of 32 bytes a K step
        for (int i = 0; i < 4 * p.kpp; ++i) {
            const int tap = p.tps * (i >> 2) + ((i & 3) * p.tps >> 2), within = 32 * (i & (4 / p.tps - 1));
            const int kh = tap / 3, kw = tap % 3;
            int row;
            if (p.nbands == 3) row = kh * p.band_px + kw;
            else {
                const int b = (p.sh == 2 ? (kh & 1) * p.sw : 0) + (p.sw == 2 ? kw & 1 : 0);
                row = b * p.band_px + kh / p.sh * p.Wp + kw / p.sw;
            }
            (&p.x_off[i >> 2].x)[i & 3] =
                tap < taps && within < p.E ? (uint32_t)(row * (p.rb >> 4) + (within >> 4)) : MMA_NONE;
        }
        p.a_slots = W3_A_SLOTS;
        // shared memory: resident B where one N tile's K steps all fit, else rings
        p.b_res = 0;
        if (p.ksteps <= W3_MAX_BST) {
            for (int as = W3_MAX_AS; as >= 1; --as) {
                const int bp = p.w8 ? 0 : 2;
                const W3Smem L = w3_layout(p.apx, p.a_slots, p.rb, p.BN, p.pk, p.PB, as, p.ksteps, bp, p.cout_pad);
                if (L.total + 1024 <= 227u * 1024u) {
                    p.b_res = 1; p.b_stages = p.ksteps; p.as_slots = as; p.bp_slots = bp;
                    return 1;
                }
            }
        }
        // {A staging slots, expanded B stages, packed B slots}: the packed ring is
        // what hides the latency of the weight loads, so it goes first
        if (p.w8) {
            // no packed ring: the operand ring itself hides the latency of the loads
            // (one window slot: 256 channels as 4-bit operands in three bands)
            for (p.a_slots = W3_A_SLOTS; p.a_slots >= (f4 ? 1 : 2); --p.a_slots)
            for (int as = W3_MAX_AS; as >= 1; --as)
                for (int bst = 6; bst >= 2; --bst) {
                    const W3Smem L = w3_layout(p.apx, p.a_slots, p.rb, p.BN, p.pk, p.PB, as, bst, 0, p.cout_pad);
                    if (L.total + 1024 <= 227u * 1024u) {
                        p.as_slots = as; p.b_stages = bst; p.bp_slots = 0;
                        return 1;
                    }
                }
            return 0;
        }
        // (packed slots: a multiple of the two groups, so that a slot's rounds are one
        // group's - a parity cannot tell a round from the one two before it)
        const int tries[5][3] = {{3, 3, 4}, {2, 3, 4}, {2, 2, 4}, {2, 2, 2}, {1, 2, 2}};
        for (p.a_slots = W3_A_SLOTS; p.a_slots >= (stride == 2 ? 1 : 2); --p.a_slots)
        for (int t = 0; t < 5; ++t) {
            const W3Smem L = w3_layout(p.apx, p.a_slots, p.rb, p.BN, p.pk, p.PB, tries[t][0], tries[t][1],
                                       tries[t][2], p.cout_pad);
            if (L.total + 1024 <= 227u * 1024u) {
                p.as_slots = tries[t][0]; p.b_stages = tries[t][1]; p.bp_slots = tries[t][2];
                return 1;
            }
        }
        return 0;
    };
    int found = 0;
    const bool want_tr = hooks.window3 == 3 || hooks.window3 == 1;
    for (int f4 = 1; want_tr && !found && f4 >= 0; --f4)
        for (int most = f4 ? W3_F4_TP : 256; !found && most >= 112; most -= 16) found = configure(1, f4, most);
    if (!found) found = configure(0, 0, 0);
    if (!found) return DSQ_ERR_UNSUPPORTED;
    // (plain tiles convert accumulators by the 2^22 trick)
    if (!p.tr && (!small_acc || bits == 3)) epi_kind = DSQ_EPI_GENERAL;
    p.L = w3_layout(p.apx, p.a_slots, p.rb, p.BN, p.pk, p.PB, p.as_slots, p.b_stages, p.bp_slots, p.cout_pad);
    p.smem_bytes = (int)p.L.total + 1024;
    {
        // (grid: a multiple of n_tiles; CTA c takes N tile c % n_tiles and every mstep-th M tile)
        const int64_t d = (int64_t)p.mstep * p.tp, img = (int64_t)p.Hp * p.Wp;
        p.t_dn = (int)(d / img);
        p.t_dh = (int)((d % img) / p.Wp);
        p.t_dw = (int)((d % img) % p.Wp);
    }
    p.wait_ns = hooks.wait_ns;
    p.skip_b_round = hooks.skip_b_round;
    p.early = dsq_early_constants();
    p.e = e;
    p.r_hi = r_hi;
    p.out_pitch = (int)dsq_row_pitch(Cout, bits);
    if (p.f4 && p.w8) {
        p.mark = (const uint32_t *)((const uint8_t *)w_packed + w3_mark_offset(w8));
    }
    if (p.f4) {
        p.shift = 0;
    } else if (e.half_offset) {
        p.shift = 7 - bits;
        p.orv = 0x01010101u << (7 - bits);
    } else {
        p.shift = 8 - bits;
        p.orv = 0;
    }
    p.ws = (int *)workspace;
    p.act = (const uint8_t *)act_codes;
    p.P = P;

    // weights: Cout rows of 9 taps x P bytes; one box = BN rows x one K step
    DsqEncodeTiledFn enc = dsq_encode_tiled_fn();
    DsqEncodeIm2colFn enc_i2c = dsq_encode_im2col_fn();
    if (!enc || !enc_i2c) return DSQ_ERR_CUDA;
    CUtensorMap tb, ta;
    if (p.w8) {
        // the blob's expanded copy: Cout rows of ksteps x 128 bytes; one box = BN
        // rows x one K step, swizzled on the way in.  pair: 64 rows, and a plane's nine taps
        // are a dimension of their own, so that taps before and behind them are zeros
        const int steps = w8.ksteps / p.npl * 128;              // bytes of a row's plane
        cuuint64_t dims[3] = {(cuuint64_t)(p.pair ? 9 * p.rb : w8.ksteps * 128),
                              (cuuint64_t)(p.pair ? p.npl : Cout), (cuuint64_t)Cout};
        cuuint64_t strides[2] = {(cuuint64_t)(p.pair ? steps : w8.ksteps * 128), (cuuint64_t)w8.ksteps * 128};
        cuuint32_t box[3] = {128u, (cuuint32_t)(p.pair ? 1 : p.BN), 64u};
        cuuint32_t estr[3] = {1, 1, 1};
        if (enc(&tb, CU_TENSOR_MAP_DATA_TYPE_UINT8, p.pair ? 3 : 2,
                const_cast<uint8_t *>((const uint8_t *)w_packed + w8.offset), dims, strides, box,
                estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return DSQ_ERR_CUDA;
    } else {
        cuuint64_t dims[2] = {(cuuint64_t)9 * P, (cuuint64_t)Cout};
        cuuint64_t strides[1] = {(cuuint64_t)9 * P};
        cuuint32_t box[2] = {(cuuint32_t)p.pk, (cuuint32_t)(p.pair ? 64 : p.BN)};
        cuuint32_t estr[2] = {1, 1};
        if (enc(&tb, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(w_packed), dims, strides,
                box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return DSQ_ERR_CUDA;
    }
    {
        // im2col map over the NHWC codes: the bounding box of base positions is
        // [-2, W-2] x [-2, H-2] (lower corner -2, upper corner -1), taken in steps of
        // sw and sh; the loads' filter offsets make pixels -1, .. or 0, .. of them
        cuuint64_t dims[4] = {(cuuint64_t)P, (cuuint64_t)p.W, (cuuint64_t)p.H, (cuuint64_t)p.N};
        cuuint64_t strides[3] = {(cuuint64_t)P, (cuuint64_t)P * p.W, (cuuint64_t)P * p.W * p.H};
        int lower[2] = {-2, -2};
        int upper[2] = {-1, -1};
        cuuint32_t estr[4] = {1, (cuuint32_t)p.sw, (cuuint32_t)p.sh, 1};
        if (enc_i2c(&ta, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(act_codes), dims,
                    strides, lower, upper, (cuuint32_t)p.PB, (cuuint32_t)p.a_box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return DSQ_ERR_UNSUPPORTED;
    }
    if (bits == 4) return w3_dispatch<4>(epi_kind, tb, ta, p, stream, hooks.pdl);
    if (bits == 3) return w3_dispatch<3>(epi_kind, tb, ta, p, stream, hooks.pdl);
    return w3_dispatch<2>(epi_kind, tb, ta, p, stream, hooks.pdl);
}
