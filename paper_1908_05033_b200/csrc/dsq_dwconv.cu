// Depthwise 3x3 convolution on packed codes, CUDA cores.  A depthwise
// convolution has no shared contraction dimension across channels, so it is
// not tensor-core work: each thread owns 8 channels (one 32-bit word at 4
// bits, one 16-bit half-word at 2 bits) of four adjacent output pixels, walks
// the 3x3 taps on packed words and applies the dequantise / requantise
// epilogue.  Inputs and outputs move as packed codes only: bits/8 bytes per
// element each way.
#include <cuda_fp16.h>

#include <algorithm>
#include <numeric>

#include "dsq_epilogue.cuh"
#include "dsq_launch.h"
#include "dsq_tc_host.h"

namespace {

// (left: bytes of the row from p on.  A 3-bit row may end inside its last unit, whose
// other codes are then not channels: 41 channels are 16 bytes, six units 18)
template <int BITS>
__device__ __forceinline__ uint32_t load_unit(const uint8_t *p, int left)
{
    if (BITS == 4) return __ldg(reinterpret_cast<const uint32_t *>(p));
    if (BITS == 3) {    // 8 codes = 3 bytes at an odd offset: byte loads
        uint32_t v = (uint32_t)__ldg(p);
        if (left > 1) v |= (uint32_t)__ldg(p + 1) << 8;
        if (left > 2) v |= (uint32_t)__ldg(p + 2) << 16;
        return v;
    }
    return __ldg(reinterpret_cast<const uint16_t *>(p));
}

// One thread: 8 channels (one unit) of OW = 4 horizontally adjacent output
// pixels.  The 3 x (OW-1)*stride+3 input window and the 9 weight units are
// loaded once as packed words; then channel by channel the fields are
// extracted (each activation field is used by up to three outputs) and the
// four 9-tap sums are formed.  With the symmetric weight grid the weights are
// taken as 2c+1, so the sum is 2*acc + S_a directly.  Per output element this
// is about 30 integer / fp32 instructions against 1 byte of HBM traffic.
template <int BITS, int STRIDE>
__global__ void __launch_bounds__(256)
dwconv3x3_kernel(const uint8_t *__restrict__ act, const uint8_t *__restrict__ wgt,
                 int N, int H, int W, int C, int Ho, int Wo, int pitch, DsqEpi e)
{
    // lets a tensor-core kernel queued behind this one (programmatic dependent
    // launch) set itself up while this grid runs; it still waits for this grid
    // to complete before touching global data
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int UB = BITS;                 // bytes per 8-channel unit
    constexpr uint32_t MASK = (1u << BITS) - 1u;
    constexpr int OW = 4;                    // outputs per thread along W
    constexpr int IW = (OW - 1) * STRIDE + 3;
    const int units = BITS == 3 ? (C + 7) / 8 : pitch / UB;
    const int strips = (Wo + OW - 1) / OW;
    const int64_t total = (int64_t)N * Ho * strips * units;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int u = (int)(i % units);
        int64_t t = i / units;
        const int sx = (int)(t % strips);
        t /= strips;
        const int ho = (int)(t % Ho);
        const int n = (int)(t / Ho);
        const int wo0 = sx * OW;
        const int hi0 = ho * STRIDE - 1, wi0 = wo0 * STRIDE - 1;
        const int left = pitch - u * UB;

        uint32_t a[3][IW], wv[9];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int hi = hi0 + r;
#pragma unroll
            for (int x = 0; x < IW; ++x) {
                const int wi = wi0 + x;
                a[r][x] = 0u;
                if (hi >= 0 && hi < H && wi >= 0 && wi < W)
                    a[r][x] = load_unit<BITS>(
                        act + (((int64_t)n * H + hi) * W + wi) * pitch + u * UB, left);
            }
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) wv[k] = load_unit<BITS>(wgt + k * pitch + u * UB, left);

        const int64_t pix0 = ((int64_t)n * Ho + ho) * Wo + wo0;
        uint32_t res[OW], cw[OW];
#pragma unroll
        for (int o = 0; o < OW; ++o) {
            cw[o] = 0u;
            res[o] = 0u;
            if (e.residual && wo0 + o < Wo)
                res[o] = load_unit<BITS>(e.residual + (pix0 + o) * pitch + u * UB, left);
        }
#pragma unroll
        for (int f = 0; f < 8; ++f) {
            const int ch = 8 * u + f;
            if (ch >= C) continue;
            int wq[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const int c = ((int)(wv[k] << (32 - BITS * (f + 1)))) >> (32 - BITS);
                wq[k] = e.half_offset ? 2 * c + 1 : c;
            }
            int acc[OW], sa[OW];
#pragma unroll
            for (int o = 0; o < OW; ++o) acc[o] = sa[o] = 0;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                int q[IW];
#pragma unroll
                for (int x = 0; x < IW; ++x) q[x] = (int)((a[r][x] >> (BITS * f)) & MASK);
#pragma unroll
                for (int o = 0; o < OW; ++o)
#pragma unroll
                    for (int kw = 0; kw < 3; ++kw) {
                        acc[o] += q[o * STRIDE + kw] * wq[r * 3 + kw];
                        sa[o] += q[o * STRIDE + kw];      // (dead unless the offset is general)
                    }
            }
            float sc = __ldg(e.scale + ch);
            if (e.half_offset) sc = __fmul_rn(sc, 0.5f);
            const float bi = __ldg(e.bias + ch);
#pragma unroll
            for (int o = 0; o < OW; ++o) {
                if (wo0 + o >= Wo) continue;
                // |acc| <= 9*15*17: the 1.5*2^23 bias trick converts exactly
                const float vf = __fsub_rn(__int_as_float(0x4B400000 + acc[o]), 12582912.0f);
                float y = __fmaf_rn(vf, sc, bi);
                // general weight-grid offset: per-channel S_a (taps outside the
                // image were loaded as code 0)
                if (e.general_offset) y = dsq_epi_y_offset(acc[o], sa[o], e.w_offset, sc, bi);
                if (e.residual) {
                    const uint32_t qr = (res[o] >> (BITS * f)) & MASK;
                    y = __fadd_rn(y, __fmaf_rn(__fsub_rn(__int_as_float(0x4B000000 | qr),
                                                         8388608.0f),
                                               e.res_delta, e.res_lo));
                }
                if (e.acc_out) e.acc_out[(pix0 + o) * C + ch] = acc[o];
                if (e.y_f32) e.y_f32[(pix0 + o) * C + ch] = y;
                if (e.has_requant) {
                    const float xc = fminf(fmaxf(y, e.rq.lo), e.rq.hi);
                    const float rr = __fmaf_rn(__fsub_rn(xc, e.rq.lo), e.rq.inv, 0.5f);
                    const uint32_t q = min(
                        (uint32_t)__float_as_int(__fadd_rd(rr, 8388608.0f)) - 0x4B000000u,
                        (uint32_t)e.rq.qmax);
                    cw[o] |= q << (BITS * f);
                }
            }
        }
        if (e.y_codes) {
#pragma unroll
            for (int o = 0; o < OW; ++o) {
                if (wo0 + o >= Wo) continue;
                uint8_t *dst = e.y_codes + (pix0 + o) * pitch + u * UB;
                if (BITS == 4) *reinterpret_cast<uint32_t *>(dst) = cw[o];
                else if (BITS == 3) {
                    dst[0] = (uint8_t)cw[o];
                    if (left > 1) dst[1] = (uint8_t)(cw[o] >> 8);
                    if (left > 2) dst[2] = (uint8_t)(cw[o] >> 16);
                    // the row's spare bytes behind the last unit are zero
                    if (u == units - 1)
                        for (int b = 3 * units; b < pitch; ++b) dst[b - u * UB] = 0;
                } else *reinterpret_cast<uint16_t *>(dst) = (uint16_t)cw[o];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Codes in, codes out (the form the stacks use), any bit width.
//
// The nine-tap sums run on packed half precision: a code q placed in the low
// bits of a 16-bit half IS the (denormal) number q * 2^-24, so two channels of a
// pixel become an operand with one shift and one AND, and one fma.f16x2 does two
// channels' tap.  Weights are small integers as halves; every partial sum is an
// integer times 2^-24 with magnitude at most 9 * 15 * 15 = 2025 < 2^11, so the
// half-precision sums are exact.  Widened to binary32 the sum is acc * 2^-24,
// and fma(acc 2^-24, scale 2^24, bias) is the pinned fma(acc, scale, bias): a
// power of two moved between the factors changes no bit (|scale| < 2^100).
//
// A thread owns eight channels (pairs j, j + 4 share a register) of a strip of
// four output columns and walks down the rows: every input row is loaded and
// split once and feeds the (up to) three output rows it lies under, whose sums
// stay in registers.
//
// Bound: instructions, 16 per element (14.4 M warp instructions for 28.9 M elements, counted;
// 4.5 of them fma.f16x2, at 62 lanes a clock and SM).  The dp4a form this replaces took 30
// (byte transposes, funnel shifts and an epilogue of 9) and only existed for 4-bit codes:
// C = 144, 56x56, batch 64, 4-bit 41.9 -> 22.9 us.
// Loaded words are kept as they came until a row's arithmetic is done (DwhRaw), and
// the padding behind 2- and 3-bit rows is no unit of work: 112x112, 32 channels, batch 64
// 2-bit 45.2 -> 22.6 us, 3-bit 42.4 -> 31.4 us (4-bit 19.8).
// ---------------------------------------------------------------------------
constexpr int DWH_THREADS = 128, DWH_BLOCKS_PER_SM = 3;

struct DwHalf {
    int N, H, W, C, Ho, Wo, pitch;
    int units;                // 8-channel units of a row (4-bit: padding lanes included)
    int spare;                // 2- and 3-bit: bytes of a row behind them
    int strips, rows, chunks; // strips of four columns; output rows of a work item
    int half_offset;
    int early;                // dsq_early_constants
    float inv;
};

// the words a unit's packed codes lie in (3-bit: 3 bytes at 3 u, one or two aligned
// words), as loaded: what is done to them waits for the load, so it is left to the place
// that uses them, a row of arithmetic later
template <int BITS> struct DwhRaw { uint32_t v[BITS == 3 ? 2 : 1]; };
template <int BITS>
__device__ __forceinline__ void dwh_load(const uint8_t *row, int u, int pitch, DwhRaw<BITS> &r)
{
    if (BITS == 4) r.v[0] = __ldg(reinterpret_cast<const uint32_t *>(row) + u);
    if (BITS == 2) r.v[0] = __ldg(reinterpret_cast<const uint16_t *>(row) + u);
    if (BITS == 3) {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(row);
        const int i = (3 * u) >> 2, last = pitch / 4 - 1;
        r.v[0] = __ldg(w + min(i, last));
        r.v[BITS == 3] = __ldg(w + min(i + 1, last));
    }
}
// 4 + 4 fields: field j at bit BITS * j, field j + 4 at bit 16 + BITS * j
template <int BITS>
__device__ __forceinline__ uint32_t dwh_split(const DwhRaw<BITS> &r, int u)
{
    if (BITS == 4) return r.v[0];
    if (BITS == 2) return __byte_perm(r.v[0], 0u, 0x4140);   // byte 1 -> byte 2
    const uint32_t x = __funnelshift_r(r.v[0], r.v[BITS == 3], 8 * ((3 * u) & 3));
    return (x & 0xFFFu) | ((x & 0xFFF000u) << 4);
}

template <int BITS>
__device__ __forceinline__ uint32_t dwh_field(uint32_t x, int j)
{
    constexpr uint32_t M = (1u << BITS) - 1u;
    return (x >> (BITS * j)) & (M | (M << 16));
}

// the 2^24-scaled sums of one output pixel's eight channels -> packed codes of the
// unit (8 * BITS bits)
template <int BITS>
__device__ __forceinline__ uint32_t dwh_codes(const uint32_t (&acc)[4],
                                              const unsigned long long (&sc)[4],
                                              const unsigned long long (&bi)[4],
                                              unsigned long long inv2)
{
    int q[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&acc[j]));
        const unsigned long long y = dsq_fma2(dsq_pack2(f.x, f.y), sc[j], bi[j]);
        dsq_requant2<BITS>(y, inv2, q[j], q[j + 4]);
    }
    return dsq_pack8<BITS>(q);
}

template <int BITS, int STRIDE>
__global__ void __launch_bounds__(DWH_THREADS, DWH_BLOCKS_PER_SM)
dwconv3x3_half_kernel(const uint8_t *__restrict__ act, const uint8_t *__restrict__ wgt,
                      const float *__restrict__ scale, const float *__restrict__ bias,
                      uint8_t *__restrict__ y_codes, const DwHalf p)
{
    constexpr int OW = 4, NP = (OW - 1) * STRIDE + 3;
    const uint32_t gtid = blockIdx.x * DWH_THREADS + threadIdx.x;
    const uint32_t lanes = gridDim.x * DWH_THREADS / (uint32_t)p.units;   // exact (host)
    const int u = (int)(gtid % (uint32_t)p.units);
    const uint32_t per_img = (uint32_t)p.strips * p.chunks;
    const uint32_t n_items = per_img * (uint32_t)p.N;
    uint32_t item = gtid / (uint32_t)p.units;
    if (!p.early) asm volatile("griddepcontrol.wait;" ::: "memory");

    // weights as halves: c = (n ^ half) - half of the stored field n, or 2 c + 1;
    // 0x6400 | m is the half 1024 + m
    __half2 w[9][4];
    {
        constexpr uint32_t HALF = 1u << (BITS - 1);
        const __half2 mul = __float2half2_rn(p.half_offset ? 2.0f : 1.0f);
        const __half2 add = __float2half2_rn(p.half_offset ? 1.0f : 0.0f);
        const __half2 base = __float2half2_rn(1024.0f + HALF);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            DwhRaw<BITS> raw;
            dwh_load<BITS>(wgt + k * p.pitch, u, p.pitch, raw);
            const uint32_t x = dwh_split<BITS>(raw, u);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t m = (dwh_field<BITS>(x, j) ^ (HALF | (HALF << 16))) | 0x64006400u;
                w[k][j] = __hfma2(__hsub2(*reinterpret_cast<const __half2 *>(&m), base), mul, add);
            }
        }
    }
    unsigned long long sc[4], bi[4];
    {
        float s[8], b[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            s[i] = b[i] = 0.f;                              // padding lanes: code 0
            if (8 * u + i < p.C) dsq_codes_affine(scale, bias, 8 * u + i, p.half_offset, 24, s[i], b[i]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            sc[j] = dsq_pack2(s[j], s[j + 4]);
            bi[j] = dsq_pack2(b[j], b[j + 4]);
        }
    }
    const unsigned long long inv2 = dsq_pack2(p.inv, p.inv);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    for (; item < n_items; item += lanes) {
        const uint32_t n = item / per_img, rem = item - n * per_img;
        const uint32_t chunk = rem / (uint32_t)p.strips;
        const int wo0 = (int)(rem - chunk * p.strips) * OW;
        const int ho0 = (int)chunk * p.rows;
        const int rows = min(p.rows, p.Ho - ho0);
        const int hi0 = ho0 * STRIDE - 1, wi0 = wo0 * STRIDE - 1;
        const uint8_t *base = act + ((int64_t)n * p.H * p.W + wi0) * p.pitch;
        const bool inner = wi0 >= 0 && wi0 + NP <= p.W;
        DwhRaw<BITS> next[NP];
        auto load_row = [&](int hi) {
            const bool in = hi >= 0 && hi < p.H;
            const uint8_t *row = base + (int64_t)hi * p.W * p.pitch;
#pragma unroll
            for (int x = 0; x < NP; ++x) {
                next[x] = DwhRaw<BITS>{};
                if (in && (inner || (wi0 + x >= 0 && wi0 + x < p.W)))
                    dwh_load<BITS>(row + x * p.pitch, u, p.pitch, next[x]);
            }
        };
        uint8_t *out = y_codes + (((int64_t)n * p.Ho + ho0) * p.Wo + wo0) * p.pitch;
        __half2 acc[STRIDE == 1 ? 3 : 2][OW][4];
        __half2 q[NP][4];
        auto taps = [&](__half2 (&a)[OW][4], int kh, bool first) {
#pragma unroll
            for (int kw = 0; kw < 3; ++kw)
#pragma unroll
                for (int o = 0; o < OW; ++o)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        a[o][j] = __hfma2(q[o * STRIDE + kw][j], w[3 * kh + kw][j],
                                          first && kw == 0 ? __half2half2(__ushort_as_half(0)) : a[o][j]);
        };
        auto finish = [&](__half2 (&a)[OW][4]) {
#pragma unroll
            for (int o = 0; o < OW; ++o) {
                uint32_t s[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) s[j] = *reinterpret_cast<const uint32_t *>(&a[o][j]);
                const uint32_t cw = dwh_codes<BITS>(s, sc, bi, inv2);
                uint8_t *dst = out + o * p.pitch;
                const bool live = wo0 + o < p.Wo;
                if (BITS == 4) {
                    if (live) reinterpret_cast<uint32_t *>(dst)[u] = cw;
                } else if (BITS == 2) {
                    if (live) reinterpret_cast<uint16_t *>(dst)[u] = (uint16_t)cw;
                } else if (live) {
                    // three bytes: the two at an even address together
                    const int odd = u & 1;
                    dst += 3 * u;
                    *reinterpret_cast<uint16_t *>(dst + odd) = (uint16_t)(cw >> (8 * odd));
                    dst[odd ? 0 : 2] = (uint8_t)(cw >> (odd ? 0 : 16));
                    // and the row's spare bytes (a pass over the pixels: 2 % slower)
                    dst += 3 * (p.units - u);
                    for (int at = u; at < p.spare; at += p.units) dst[at] = 0;
                }
            }
            out += (int64_t)p.Wo * p.pitch;
        };
        // input row s of the item: rows hi0 .. hi0 + (rows - 1) * STRIDE + 2
        const int n_in = (rows - 1) * STRIDE + 3;
        load_row(hi0);
        constexpr int UNROLL = STRIDE == 1 ? 3 : 4;
#pragma unroll 1
        for (int s0 = 0; s0 < n_in; s0 += UNROLL) {
#pragma unroll
            for (int t = 0; t < UNROLL; ++t) {
                const int s = s0 + t;
                if (s >= n_in) break;
#pragma unroll
                for (int x = 0; x < NP; ++x) {
                    const uint32_t codes = dwh_split<BITS>(next[x], u);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t f = dwh_field<BITS>(codes, j);
                        q[x][j] = *reinterpret_cast<const __half2 *>(&f);
                    }
                }
                if (s + 1 < n_in) load_row(hi0 + s + 1);
                if (STRIDE == 1) {
                    // output row s starts, s - 1 goes on, s - 2 is completed
                    if (s >= 2) {
                        taps(acc[(t + 1) % 3], 2, false);
                        finish(acc[(t + 1) % 3]);
                    }
                    if (s >= 1 && s <= rows) taps(acc[(t + 2) % 3], 1, false);
                    if (s < rows) taps(acc[t % 3], 0, true);
                } else if (t & 1) {
                    taps(acc[t >> 1], 1, false);
                } else {
                    if (s >= 2) {
                        taps(acc[((t >> 1) + 1) & 1], 2, false);
                        finish(acc[((t >> 1) + 1) & 1]);
                    }
                    if (s >> 1 < rows) taps(acc[(t >> 1) & 1], 0, true);
                }
            }
        }
    }
    // 2 bits: the rows' spare bytes are zeros, written in a pass of their own over output
    // pixels (as units of work they were half of the whole on 32-channel rows)
    if (BITS == 2 && p.spare) {
        const int64_t pixels = (int64_t)p.N * p.Ho * p.Wo;
        for (int64_t i = gtid; i < pixels; i += gridDim.x * DWH_THREADS) {
            uint16_t *dst = reinterpret_cast<uint16_t *>(y_codes + i * p.pitch) + p.units;
            for (int k = 0; k < p.spare; k += 2) dst[k / 2] = 0;
        }
    }
}

}  // namespace

extern "C" int dsq_dwconv2d(const void *act_codes, const dsq_nhwc_t *shape,
                            const dsq_quant_t *act_q, const void *w_packed,
                            const dsq_conv_t *conv, const dsq_epilogue_t *ep,
                            float *y_f32, void *y_codes, int32_t *acc_out,
                            void *stream)
{
    if (!act_codes || !shape || !act_q || !w_packed || !conv || !ep)
        return DSQ_ERR_NULL;
    int st = dsq_check_quant(act_q);
    if (st) return st;
    const int bits = act_q->bits;
    if (shape->N <= 0 || shape->H <= 0 || shape->W <= 0 || shape->C <= 0)
        return DSQ_ERR_SHAPE;
    if (conv->groups != shape->C || conv->Cin != shape->C || conv->Cout != shape->C)
        return DSQ_ERR_SHAPE;
    if (conv->KH != 3 || conv->KW != 3 || conv->pad != 1 ||
        (conv->stride != 1 && conv->stride != 2))
        return DSQ_ERR_UNSUPPORTED;
    if (act_q->lo != 0.0f) return DSQ_ERR_UNSUPPORTED;   // padding is code 0
    if (!dsq_aligned16(act_codes) || !dsq_aligned16(w_packed)) return DSQ_ERR_ALIGN;
    DsqEpi e;
    st = dsq_make_epi(ep, bits, y_f32, y_codes, acc_out, &e);
    if (st) return st;
    const int Ho = (shape->H + 2 - 3) / conv->stride + 1;
    const int Wo = (shape->W + 2 - 3) / conv->stride + 1;
    const int pitch = (int)dsq_row_pitch(shape->C, bits);
    cudaStream_t s = (cudaStream_t)stream;
    // codes to codes, a requantiser range the lean epilogue takes that starts at 0 (it does
    // not subtract lo), rows that do not end inside a unit (3-bit rows of 41 or 84 channels
    // do); images of at least 2^31 bytes a row keep the general kernel's
    // 64-bit indexing
    const int units = bits == 4 ? pitch / 4 : (shape->C + 7) / 8;
    const int strips = (Wo + 3) / 4;
    if (y_codes && !y_f32 && !acc_out && !e.residual && !e.general_offset && e.rq.lo == 0.0f &&
        dsq_lean_epilogue(e) && units * bits <= pitch && (int64_t)units * strips * Ho * shape->N < (1ll << 31)) {
        DwHalf p;
        p.N = shape->N; p.H = shape->H; p.W = shape->W; p.C = shape->C;
        p.Ho = Ho; p.Wo = Wo; p.pitch = pitch;
        p.units = units; p.strips = strips;
        p.spare = pitch - units * bits;
        p.half_offset = e.half_offset;
        p.inv = e.rq.inv;
        p.early = dsq_early_constants();
        const int sms = dsq_sm_count() > 0 ? dsq_sm_count() : 148;
        // blocks: all resident, and a thread keeps its unit (blocks * 128 is a
        // multiple of `units`)
        const int per = units / std::gcd(units, DWH_THREADS);
        const int resident = std::max(sms * DWH_BLOCKS_PER_SM / per, 1) * per;
        const int64_t lanes = (int64_t)resident * DWH_THREADS / units;
        // rows of a work item: a thread's passes over items, each rows + 2 input
        // rows (stride 1) and about one row's worth of set-up, are what a launch
        // lasts; the fewest win
        int64_t best = -1;
        for (int chunks = 1; chunks <= Ho; ++chunks) {
            const int rows = (Ho + chunks - 1) / chunks;
            if (chunks > 1 && rows == (Ho + chunks - 2) / (chunks - 1)) continue;
            const int used = (Ho + rows - 1) / rows;
            const int64_t passes = ((int64_t)p.N * strips * used + lanes - 1) / lanes;
            const int64_t cost = passes * (8 * rows + (conv->stride == 1 ? 12 : 8)) ;
            if (best < 0 || cost < best) { best = cost; p.rows = rows; p.chunks = used; }
        }
        const int64_t need = ((int64_t)units * p.N * strips * p.chunks + DWH_THREADS - 1) / DWH_THREADS;
        const int blocks = (int)std::min<int64_t>(resident, (need + per - 1) / per * per);
        typedef void (*Kernel)(const uint8_t *, const uint8_t *, const float *, const float *,
                               uint8_t *, const DwHalf);
        static const Kernel kernels[3][2] = {
            {dwconv3x3_half_kernel<2, 1>, dwconv3x3_half_kernel<2, 2>},
            {dwconv3x3_half_kernel<3, 1>, dwconv3x3_half_kernel<3, 2>},
            {dwconv3x3_half_kernel<4, 1>, dwconv3x3_half_kernel<4, 2>}};
        return dsq_launch(kernels[bits - 2][conv->stride - 1], dim3(blocks), dim3(DWH_THREADS), 0, s,
                          dsq_launch_hooks().pdl, 0, (const uint8_t *)act_codes,
                          (const uint8_t *)w_packed, e.scale, e.bias, e.y_codes, p);
    }
    const int64_t total = (int64_t)shape->N * Ho * ((Wo + 3) / 4) *
                          (bits == 3 ? (shape->C + 7) / 8 : pitch / bits);
    int64_t g = (total + 255) / 256;
    if (g > 148 * 32) g = 148 * 32;
    if (g < 1) g = 1;
    const uint8_t *a = (const uint8_t *)act_codes, *w = (const uint8_t *)w_packed;
    const auto kernel = bits == 4 ? (conv->stride == 1 ? dwconv3x3_kernel<4, 1> : dwconv3x3_kernel<4, 2>)
                        : bits == 3
                            ? (conv->stride == 1 ? dwconv3x3_kernel<3, 1> : dwconv3x3_kernel<3, 2>)
                            : (conv->stride == 1 ? dwconv3x3_kernel<2, 1> : dwconv3x3_kernel<2, 2>);
    return dsq_launch(kernel, dim3((unsigned)g), dim3(256), 0, s, 0, 0, a, w, shape->N, shape->H,
                      shape->W, shape->C, Ho, Wo, pitch, e);
}
