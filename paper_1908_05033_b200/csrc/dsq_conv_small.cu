// Dense convolutions with little work (one or a few images): Algorithm 1 step 5 on
// codes plus the fused epilogue, laid out for latency.
//
// At batch 1 a layer of the ResNet-18-shaped network is 0.1 G multiply-accumulates:
// well under a microsecond of arithmetic.  The tcgen05 kernels took 4 to 14 us for
// it: 1.5 us before their roles start (23 to 31 warps, tensor memory, barriers), a
// chain of hand-offs, and one to four CTAs that walk the whole of K alone.  Here
//   * a block of 4 to 16 warps makes 16 MT pixels x 8 NT channels, its warps splitting
//     K (so a layer is a few hundred blocks whose warps load a chunk or two each) and
//     adding their sums in shared memory;
//   * every lane takes its packed words straight from global memory to the fragments
//     of mma.sync m16n8k32 (u8 x s8) in registers - three instructions for eight
//     codes.  tcgen05 would need them in shared or tensor memory first; the fragment
//     instruction does 1,861 multiply-accumulates a clock and SM (measured), a
//     quarter of its rate, which is plenty here;
//   * a warp that walks several chunks asks for the next one's words, activations and
//     weights, before this one's arithmetic (AHEAD).  At one image the loads and the
//     arithmetic are 1.3 to 2.6 us of a layer's 3.4 to 4.5, half of it the latency of a chunk's
//     activations: 14x14 256->256 with residual 4.07 -> 3.21 us, 7x7 512->512 4.47 -> 3.86, two
//     images 5.60 -> 4.06.  In tiles of two pixel rows the registers for it cost the block
//     that could sit beside: only where a warp walks four chunks or more (7x7 512->512 at
//     batch 8 8.84 -> 8.32; 28x28 128->128 at batch 3, two to three chunks, 4.27 -> 4.57);
//   * the weights of the first chunk, the scales and the biases are fetched before the
//     wait for the previous kernel, and blocks are small enough to sit beside that
//     kernel's.
// Channels are dealt to the fragment columns so that a lane's columns of four column
// tiles are eight consecutive channels (column 8 t + 2 j + e <- channel 8 j + 2 t + e of
// 32): a lane then finishes a word of codes.
//
// K is a list of units: 16 bytes of one filter tap of a pixel row (32 codes of 4 bits,
// 64 of 2; 12 bytes = 32 codes at 3 bits), four units - lanes j = 0 .. 3 - a chunk.
// The order of K inside a unit is free as long as both operands agree.
#include "dsq_conv_rule.h"
#include "dsq_fragments.cuh"
#include "dsq_tc_host.h"

namespace {

constexpr int CS_MAX_WARPS = 16;

struct CsParams {
    const uint8_t *act, *w;
    int H, W, Ho, Wo, stride, pad, ksize;
    int M, Ncols, P, w_row;           // pixels, channels, bytes of a pixel row, of a weight row
    int upt, chunks;                  // units per tap; chunks of four units
    int units, d_tap, d_s;            // all units; a warp's step of 4 * warps units as taps, units
    int shift, out_pitch, lean;
    int early;                        // dsq_early_constants
    uint32_t orv;
    DsqEpi e;
};

// (NT is 4 wherever it is launched; as a constant of the file the same source compiles to
// a kernel that is slower for the ResNet-18-shaped network at batch 1, 67.0 -> 69.0 us)
template <int BITS, int MT, int NT, bool AHEAD>
__global__ void __launch_bounds__((MT == 1 ? CS_MAX_WARPS : 8) * 32, AHEAD && MT == 1 ? 1 : 0)
conv_small_kernel(const CsParams p)
{
    constexpr int WORDS = Unit<BITS>::WORDS, UNIT_BYTES = 4 * WORDS;
    extern __shared__ int4 part[];                    // [warp][MT * NT][lane]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int g = lane >> 2, j = lane & 3;
    const int n0 = blockIdx.x * 8 * NT, m0 = blockIdx.y * 16 * MT;

    // this lane's unit of the warp's first chunk, as filter tap and unit of the tap
    int c = warp;
    int tap = (4 * warp + j) / p.upt, s = (4 * warp + j) - tap * p.upt;
    uint32_t wv[NT][WORDS];
    auto load_w = [&]() {
        const int at = tap * p.P + s * UNIT_BYTES;
        const bool in = c < p.chunks && tap < p.ksize * p.ksize;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            // (column g of tile t)
            const int row = n0 + 32 * (t >> 2) + 8 * (g >> 1) + 2 * (t & 3) + (g & 1);
            load_unit<BITS>(p.w + (int64_t)row * p.w_row + at, in && row < p.Ncols, p.P - s * UNIT_BYTES, wv[t]);
        }
    };
    if (!p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    load_w();
    // this lane's pixels (rows g and g + 8 of every tile): corner of the filter window
    int hb[MT][2], wb[MT][2], at0[MT][2];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int px = m0 + 16 * m + 8 * h + g;
            const int t = px / p.Wo, n = t / p.Ho;
            hb[m][h] = px < p.M ? (t - n * p.Ho) * p.stride - p.pad : -(1 << 20);
            wb[m][h] = (px - t * p.Wo) * p.stride - p.pad;
            at0[m][h] = (n * p.H + hb[m][h]) * p.W + wb[m][h];       // pixel index (< 2^30)
        }
    int acc[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[m][t][i] = 0;
    // epilogue item of this thread: half eh (rows g + 8 eh) of pixel tile em, channels
    // 8 j .. of group et of 32 (a block has at least as many threads as items)
    const DsqEpi &e = p.e;
    const int ew = warp, eh = ew & 1, em = (ew >> 1) % MT, et = (ew >> 1) / MT;
    const int px = m0 + 16 * em + 8 * eh + g, ch = n0 + 32 * et + 8 * j, byte0 = ch * BITS / 8;
    const bool mine = et < NT / 4 && px < p.M && (ch < p.Ncols || byte0 < p.out_pitch);
    float sc8[8], bi8[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        sc8[k] = 0.f;
        bi8[k] = -1e30f;                              // padding lanes: code 0
        if (!mine || ch + k >= p.Ncols) continue;
        if (p.lean) dsq_codes_affine(e.scale, e.bias, ch + k, e.half_offset, -p.shift, sc8[k], bi8[k]);
        else {
            sc8[k] = __ldg(e.scale + ch + k);
            if (e.half_offset) sc8[k] = __fmul_rn(sc8[k], 0.5f);
            bi8[k] = __ldg(e.bias + ch + k);
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint32_t res = 0u;
    if (e.residual && mine && byte0 < p.out_pitch) {
        const uint8_t *rp = e.residual + (int64_t)px * p.out_pitch + byte0;
        if (BITS == 4) res = __ldg(reinterpret_cast<const uint32_t *>(rp));
        else if (BITS == 2) res = __ldg(reinterpret_cast<const uint16_t *>(rp));
        else
            for (int b = 0; b < 3; ++b)
                if (byte0 + b < p.out_pitch) res |= (uint32_t)__ldg(rp + b) << (8 * b);
    }

    uint32_t an[MT][2][WORDS];
    auto load_a = [&]() {
        const int kh = p.ksize == 1 ? 0 : (tap * 11) >> 5, kw = tap - kh * p.ksize;
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int hi = hb[m][h] + kh, wi = wb[m][h] + kw;
                const bool in = tap < p.ksize * p.ksize && hi >= 0 && hi < p.H && wi >= 0 && wi < p.W;
                load_unit<BITS>(p.act + (int64_t)(at0[m][h] + kh * p.W + kw) * p.P + s * UNIT_BYTES, in,
                                p.P - s * UNIT_BYTES, an[m][h]);
            }
    };
    if (AHEAD) load_a();
#pragma unroll 1
    while (c < p.chunks) {
        if (!AHEAD) load_a();
        uint32_t av[MT][2][WORDS];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < WORDS; ++i) av[m][h][i] = an[m][h][i];
        uint32_t w[NT][WORDS];
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int i = 0; i < WORDS; ++i) w[t][i] = wv[t][i];
        c += warps;
        tap += p.d_tap;
        s += p.d_s;
        if (s >= p.upt) { s -= p.upt; ++tap; }
        load_w();
        if (AHEAD) load_a();
#pragma unroll
        for (int q = 0; q < Unit<BITS>::BYTE_WORDS; q += 2) {
            uint32_t a[MT][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    a[m][h] = byte_word<BITS, false>(av[m][h], q, 0u);
                    a[m][h + 2] = byte_word<BITS, false>(av[m][h], q + 1, 0u);
                }
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const uint32_t b0 = byte_word<BITS, true>(w[t], q, p.orv);
                const uint32_t b1 = byte_word<BITS, true>(w[t], q + 1, p.orv);
#pragma unroll
                for (int m = 0; m < MT; ++m) mma_u8s8(acc[m][t], a[m], b0, b1);
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
    // the warps' sums, each thread one fragment word of one lane
    for (int i = threadIdx.x; i < MT * NT * 32; i += blockDim.x) {
        int4 sum = part[i];
        for (int k = 1; k < warps; ++k) {
            const int4 x = part[k * (MT * NT * 32) + i];
            sum.x += x.x; sum.y += x.y; sum.z += x.z; sum.w += x.w;
        }
        part[i] = sum;
    }
    __syncthreads();

    // epilogue: a thread takes eight channels of one pixel
    const DsqLean lean = dsq_make_lean(e);
    if (mine) {
        uint32_t v[8];
        const int2 *src = reinterpret_cast<const int2 *>(part) + (((em * NT + 4 * et) * 32 + lane) * 2 + eh);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int2 x = src[t * 64];
            v[2 * t] = (uint32_t)x.x;
            v[2 * t + 1] = (uint32_t)x.y;
        }
        uint32_t codes = 0u;
        if (p.lean) {
            unsigned long long sc[4], bi[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                sc[k] = dsq_pack2(sc8[2 * k], sc8[2 * k + 1]);
                bi[k] = dsq_pack2(bi8[2 * k], bi8[2 * k + 1]);
            }
            codes = e.residual ? dsq_lean_codes8<BITS, true, true>(v, sc, bi, res, lean)
                               : dsq_lean_codes8<BITS, false, true>(v, sc, bi, 0u, lean);
        } else {
            float y[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                y[k] = 0.f;
                if (ch + k >= p.Ncols) continue;
                const int a = (int)v[k] >> p.shift;
                v[k] = (uint32_t)a;
                y[k] = dsq_epi_y(a, sc8[k], bi8[k]);
                if (e.residual)
                    y[k] = dsq_epi_residual(y[k], (res >> (BITS * k)) & ((1u << BITS) - 1u), e.res_delta,
                                            e.res_lo);
                if (e.has_requant) codes |= dsq_code(y[k], e.rq) << (BITS * k);
            }
            const int64_t at = (int64_t)px * p.Ncols + ch;
            const bool full = (p.Ncols & 3) == 0 && ch + 8 <= p.Ncols;
            if (e.acc_out && full) {
                reinterpret_cast<int4 *>(e.acc_out + at)[0] = make_int4(v[0], v[1], v[2], v[3]);
                reinterpret_cast<int4 *>(e.acc_out + at)[1] = make_int4(v[4], v[5], v[6], v[7]);
            }
            if (e.y_f32 && full) {
                reinterpret_cast<float4 *>(e.y_f32 + at)[0] = make_float4(y[0], y[1], y[2], y[3]);
                reinterpret_cast<float4 *>(e.y_f32 + at)[1] = make_float4(y[4], y[5], y[6], y[7]);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (full || ch + k >= p.Ncols) continue;
                if (e.acc_out) e.acc_out[at + k] = (int)v[k];
                if (e.y_f32) e.y_f32[at + k] = y[k];
            }
        }
        if (!e.y_codes) return;
        uint8_t *dst = e.y_codes + (int64_t)px * p.out_pitch + byte0;
        if (BITS == 4) *reinterpret_cast<uint32_t *>(dst) = codes;
        else if (BITS == 2) *reinterpret_cast<uint16_t *>(dst) = (uint16_t)codes;
        else
            for (int b = 0; b < 3; ++b)
                if (byte0 + b < p.out_pitch) dst[b] = (uint8_t)(codes >> (8 * b));
        // (the tiles may end before the row's pitch does: spare bytes are zero)
        if (BITS != 4 && blockIdx.x == gridDim.x - 1 && et == NT / 4 - 1 && j == 3)
            for (int b = BITS; byte0 + b < p.out_pitch; ++b) dst[b] = 0;
    }
}

template <int BITS, int MT, int NT, bool AHEAD>
int launch(const CsParams &p, int warps, cudaStream_t s)
{
    const size_t smem = (size_t)warps * MT * NT * 32 * 16;
    static std::atomic<unsigned long long> configured{0ull};
    const int st = dsq_allow_smem((const void *)conv_small_kernel<BITS, MT, NT, AHEAD>,
                                  CS_MAX_WARPS * MT * NT * 512, &configured);
    if (st) return st;
    return dsq_launch(conv_small_kernel<BITS, MT, NT, AHEAD>,
                      dim3((p.Ncols + 8 * NT - 1) / (8 * NT), (p.M + 16 * MT - 1) / (16 * MT)),
                      dim3(32 * warps), smem, s, dsq_launch_hooks().pdl, 0, p);
}

template <int BITS>
int pick(CsParams &p, int mt, int warps, cudaStream_t s)
{
    p.d_tap = 4 * warps / p.upt;
    p.d_s = 4 * warps - p.d_tap * p.upt;
    if (mt == 1) return launch<BITS, 1, 4, true>(p, warps, s);
    return p.chunks > 3 * warps ? launch<BITS, 2, 4, true>(p, warps, s) : launch<BITS, 2, 4, false>(p, warps, s);
}

}  // namespace

int dsq_conv_small(const void *act_codes, const dsq_nhwc_t *shape, int bits, const void *w_packed,
                   const dsq_conv_t *conv, const DsqEpi &e, int lean, cudaStream_t stream)
{
    if (e.general_offset) return DSQ_ERR_UNSUPPORTED;
    CsParams p = {};
    p.act = (const uint8_t *)act_codes;
    p.w = (const uint8_t *)w_packed;
    p.H = shape->H; p.W = shape->W;
    p.stride = conv->stride; p.pad = conv->pad; p.ksize = conv->KH;
    p.Ho = (shape->H + 2 * conv->pad - conv->KH) / conv->stride + 1;
    p.Wo = (shape->W + 2 * conv->pad - conv->KW) / conv->stride + 1;
    p.M = shape->N * p.Ho * p.Wo;
    p.Ncols = conv->Cout;
    p.P = (int)dsq_row_pitch(conv->Cin, bits);
    const int taps = conv->KH * conv->KW;
    p.w_row = taps * p.P;
    p.upt = bits == 3 ? (conv->Cin + 31) / 32 : p.P / 16;
    p.units = taps * p.upt;
    p.chunks = (p.units + 3) / 4;
    p.out_pitch = (int)dsq_row_pitch(conv->Cout, bits);
    p.lean = lean;
    p.early = dsq_early_constants();
    p.shift = e.half_offset ? 7 - bits : 8 - bits;
    p.orv = e.half_offset ? 0x01010101u << (7 - bits) : 0u;
    p.e = e;
    if ((p.M + 15) / 16 > 65535 || (int64_t)shape->N * shape->H * shape->W >= (1ll << 30))
        return DSQ_ERR_UNSUPPORTED;
    const int sms = dsq_sm_count() > 0 ? dsq_sm_count() : 148;
    const DsqSmallTile best = dsq_small_tile(p.M, p.Ncols, p.chunks, bits, sms);
    if (best.us > dsq_small_other(shape, bits, conv, p.M, e.half_offset && dsq_launch_hooks().w8, lean, sms,
                                  e.residual != nullptr))
        return DSQ_ERR_UNSUPPORTED;
    switch (bits) {
    case 2: return pick<2>(p, best.mt, best.warps, stream);
    case 3: return pick<3>(p, best.mt, best.warps, stream);
    default: return pick<4>(p, best.mt, best.warps, stream);
    }
}
