// Dequantise / requantise epilogue shared by the depthwise and tensor-core
// kernels (Algorithm 1 steps 4-5 folded onto the integer accumulator, then
// steps 1 and 3 of the next layer).  The binary32 operation order is fixed.
#pragma once

#include "dsq_common.cuh"

struct DsqEpi {
    const float *scale;       // [Cout]
    const float *bias;        // [Cout]
    int half_offset;          // 1: accumulator is 2*acc + S_a, scale halved
    // general weight-grid offset o_w = l_w/Delta_w + 2^(b-1) (an asymmetric
    // learnt clip): y = fma(fma(o_w, (float)S_a, (float)acc), scale, bias), S_a
    // summed by the epilogue thread from the input codes under the filter
    int general_offset;
    float w_offset;
    const uint8_t *residual;  // packed NHWC codes of the output shape, or null
    float res_lo, res_delta;  // l_r and Delta_r = (hi_r - lo_r)/(2^b - 1)
    int has_requant;
    DsqQ rq;
    float *y_f32;             // nullable
    uint8_t *y_codes;         // nullable
    int32_t *acc_out;         // nullable
};

static inline int dsq_make_epi(const dsq_epilogue_t *ep, int bits, float *y_f32,
                               void *y_codes, int32_t *acc_out, DsqEpi *out)
{
    if (!ep || !ep->scale || !ep->bias) return DSQ_ERR_NULL;
    if (!y_f32 && !y_codes && !acc_out) return DSQ_ERR_NULL;
    if (!dsq_finite(ep->w_offset)) return DSQ_ERR_RANGE;
    DsqEpi e;
    e.scale = ep->scale;
    e.bias = ep->bias;
    e.half_offset = ep->w_offset == 0.5f ? 1 : 0;
    e.general_offset = ep->w_offset != 0.0f && ep->w_offset != 0.5f;
    e.w_offset = ep->w_offset;
    e.residual = (const uint8_t *)ep->residual_codes;
    e.res_lo = 0.f;
    e.res_delta = 0.f;
    if (e.residual) {
        int st = dsq_check_quant(&ep->residual_q);
        if (st) return st;
        if (ep->residual_q.bits != bits) return DSQ_ERR_BITS;
        if (!dsq_aligned16(e.residual)) return DSQ_ERR_ALIGN;
        e.res_lo = ep->residual_q.lo;
        e.res_delta = (ep->residual_q.hi - ep->residual_q.lo) /
                      (float)((1 << bits) - 1);
    }
    e.has_requant = 0;
    e.rq = DsqQ{0.f, 1.f, 1.f, 1};
    if (y_codes) {
        int st = dsq_check_quant(&ep->requant);
        if (st) return st;
        if (ep->requant.bits != bits) return DSQ_ERR_BITS;
        if (!dsq_aligned16(y_codes)) return DSQ_ERR_ALIGN;
        e.has_requant = 1;
        e.rq = dsq_make_q(ep->requant);
    }
    if (y_f32 && !dsq_aligned16(y_f32)) return DSQ_ERR_ALIGN;
    if (acc_out && !dsq_aligned16(acc_out)) return DSQ_ERR_ALIGN;
    e.y_f32 = y_f32;
    e.y_codes = (uint8_t *)y_codes;
    e.acc_out = acc_out;
    *out = e;
    return DSQ_OK;
}

// Whether the lean codes epilogues (below) take a layer's requantiser and residual
// operand: no NaN may arise in them, and they move powers of two between the accumulator
// and the scale, which rounds scales below 2^-118.  The host cannot see scales, but results
// that small fill no range wider than 2^-80.
static inline bool dsq_lean_epilogue(const DsqEpi &e)
{
    return dsq_lean_range(e.rq) && e.rq.hi - e.rq.lo >= 0x1p-80f &&
           (!e.residual || dsq_finite(e.res_delta));
}

#ifdef __CUDACC__
// v is acc (half_offset = 0) or 2*acc + S_a (half_offset = 1, with `scale`
// already multiplied by 0.5f by the caller of this function).
__device__ __forceinline__ float dsq_epi_y(int v, float scale, float bias)
{
    return __fmaf_rn((float)v, scale, bias);
}

// general weight-grid offset: v = acc, s_a = sum of the activation codes
// under the in-image filter taps
__device__ __forceinline__ float dsq_epi_y_offset(int v, int s_a, float w_offset, float scale,
                                                  float bias)
{
    return __fmaf_rn(__fmaf_rn(w_offset, (float)s_a, (float)v), scale, bias);
}

// Sum of the `bits`-bit fields of `nwords` 32-bit words of a packed row that
// starts at `row` (16-byte aligned, nwords a multiple of 4; spare bits are 0).
template <int BITS>
__device__ __forceinline__ int dsq_codes_sum(const uint8_t *row, int nwords)
{
    int s = 0;
    const uint4 *r4 = reinterpret_cast<const uint4 *>(row);
    for (int i = 0; i < nwords / 4; ++i) {
        const uint4 v = __ldg(r4 + i);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (BITS == 4) {
                const uint32_t t = (w[j] & 0x0F0F0F0Fu) + ((w[j] >> 4) & 0x0F0F0F0Fu);
                s = (int)__dp4a(t, 0x01010101u, (unsigned)s);
            } else if (BITS == 2) {
                uint32_t t = (w[j] & 0x33333333u) + ((w[j] >> 2) & 0x33333333u);
                t = (t & 0x0F0F0F0Fu) + ((t >> 4) & 0x0F0F0F0Fu);
                s = (int)__dp4a(t, 0x01010101u, (unsigned)s);
            } else {
                // 3-bit fields run across word boundaries: bit k of every field
                // sits at the row's bit positions = k (mod 3); word index mod 3
                // gives the phase of that pattern inside the word
                const int ph = (4 * i + j) % 3;
                const uint32_t m0 = ph == 0 ? 0x49249249u : ph == 1 ? 0x92492492u : 0x24924924u;
                const uint32_t m1 = ph == 0 ? 0x92492492u : ph == 1 ? 0x24924924u : 0x49249249u;
                const uint32_t m2 = ph == 0 ? 0x24924924u : ph == 1 ? 0x49249249u : 0x92492492u;
                s += __popc(w[j] & m0) + 2 * __popc(w[j] & m1) + 4 * __popc(w[j] & m2);
            }
        }
    }
    return s;
}

// S_a of one output pixel of a dense convolution: the codes of all channels
// of every in-image pixel under the k x k window (Algorithm 1 step 5 with the
// weight grid l_w + Delta_w q_w needs it next to the integer accumulator).
template <int BITS>
__device__ __forceinline__ int dsq_window_sa(const uint8_t *act, int n, int ho, int wo, int H,
                                             int W, int ksize, int stride, int pad, int P)
{
    int s = 0;
    for (int kh = 0; kh < ksize; ++kh)
        for (int kw = 0; kw < ksize; ++kw) {
            const int hi = ho * stride - pad + kh, wi = wo * stride - pad + kw;
            if (hi < 0 || hi >= H || wi < 0 || wi >= W) continue;
            s += dsq_codes_sum<BITS>(act + (((int64_t)n * H + hi) * W + wi) * P, P / 4);
        }
    return s;
}

__device__ __forceinline__ float dsq_epi_residual(float y, uint32_t q_r,
                                                  float res_delta, float res_lo)
{
    return __fadd_rn(y, __fmaf_rn((float)q_r, res_delta, res_lo));
}
// ---------------------------------------------------------------------------
// Lean codes epilogue: accumulator -> codes in about 3 instructions per element.
//
// Per element the pinned sequence is y = fma(v, scale, bias) (+ residual),
// r = fma(clip(y) - lo, inv, 0.5), q = min(floor(r), qmax).  Here
//   * arithmetic is on pairs (f32x2: one issue slot for two elements), each
//     operation rounding as the scalar one does;
//   * nothing is clipped before the rounding step: below the range r < 0.5 (codes
//     of negative numbers saturate to 0), above it r > qmax + 0.5;
//   * floor and clip are one multiply and half a pack.  r * 2^(-141 - BITS),
//     rounded down, is a denormal number whose bit pattern is the integer
//     floor(r * 2^(8 - BITS)); cvt.pack.sat.u8 clips two of those to 0 .. 255 and
//     packs them, and the top BITS bits of each byte are the code.
// Measured per SM and clock (lanes): f32x2 62, I2F 62, cvt.pack 62 - against an
// IADD, two FMNMX, a shift and a shift-add per element in the scalar form (all of
// them on the 62-lane pipe).
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long dsq_pack2(float a, float b)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ unsigned long long dsq_fma2(unsigned long long a, unsigned long long b,
                                                       unsigned long long c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long dsq_add2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// two values y - lo -> two integers whose saturated low byte holds the code in
// its top BITS bits (inv2: the requantiser's inv, twice)
template <int BITS>
__device__ __forceinline__ void dsq_requant2(unsigned long long y, unsigned long long inv2, int &q0,
                                             int &q1)
{
    constexpr unsigned long long DEN = 1ull << (8 - BITS);       // 2^(8 - BITS) * 2^-149
    const unsigned long long r = dsq_fma2(y, inv2, 0x3F0000003F000000ull);
    unsigned long long u;
    asm("mul.rm.f32x2 %0, %1, %2;" : "=l"(u) : "l"(r), "l"(DEN | (DEN << 32)));
    asm("mov.b64 {%0, %1}, %2;" : "=r"(q0), "=r"(q1) : "l"(u));
}

// bytes [sat(q0), sat(q1), sat(q2), sat(q3)]
__device__ __forceinline__ uint32_t dsq_sat_bytes(int q0, int q1, int q2, int q3)
{
    uint32_t t, r;
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, 0;" : "=r"(t) : "r"(q3), "r"(q2));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(q1), "r"(q0), "r"(t));
    return r;
}

// eight such integers of consecutive elements -> their codes, packed (8 * BITS bits;
// SLOT = 4: a 3-bit code in every four bits)
template <int BITS, int SLOT = BITS>
__device__ __forceinline__ uint32_t dsq_pack8(const int (&q)[8])
{
    if (BITS == 3 && SLOT == 4) {
        const uint32_t e = dsq_sat_bytes(q[0], q[2], q[4], q[6]);
        const uint32_t o = dsq_sat_bytes(q[1], q[3], q[5], q[7]);
        return ((e >> 5) & 0x07070707u) | ((o >> 1) & 0x70707070u);
    }
    if (BITS == 4) {
        const uint32_t e = dsq_sat_bytes(q[0], q[2], q[4], q[6]);
        const uint32_t o = dsq_sat_bytes(q[1], q[3], q[5], q[7]);
        return ((e >> 4) & 0x0F0F0F0Fu) | (o & 0xF0F0F0F0u);
    }
    if (BITS == 3) {
        const uint32_t e = dsq_sat_bytes(q[0], q[2], q[4], q[6]);
        const uint32_t o = dsq_sat_bytes(q[1], q[3], q[5], q[7]);
        const uint32_t t = ((e >> 5) & 0x07070707u) | ((o >> 2) & 0x38383838u);
        const uint32_t x = (t & 0x003F003Fu) | ((t & 0x3F003F00u) >> 2);
        return (x & 0xFFFu) | ((x >> 4) & 0xFFF000u);
    }
    const uint32_t x = dsq_sat_bytes(q[0], q[4], q[2], q[6]);
    const uint32_t y = dsq_sat_bytes(q[1], q[5], q[3], q[7]);
    const uint32_t z = ((x >> 6) & 0x03030303u) | ((y >> 4) & 0x0C0C0C0Cu);
    return (z & 0xFFFFu) | ((z >> 12) & 0xF0F0u);
}

// Scale (halved for the symmetric weight grid, times 2^e: the accumulator comes
// scaled by 2^-e) and bias of channel ch for the lean epilogue.  It does not clip
// before rounding, so a NaN y (non-finite scale or bias; code 0 in the pinned
// sequence) must not arise: such channels get finite numbers that give the
// same codes for every accumulator.
__device__ __forceinline__ void dsq_codes_affine(const float *scale, const float *bias, int ch,
                                                 int half_offset, int e, float &s, float &b)
{
    s = __ldg(scale + ch);
    b = __ldg(bias + ch);
    const bool odd = !(fabsf(s) <= 3.4e38f) || b != b;
    s = __fmul_rn(s, __int_as_float((127 + e - (half_offset ? 1 : 0)) << 23));
    if (odd) {
        s = (s != s || b != b || b == -__int_as_float(0x7F800000)) ? 0.0f : s;
        b = -1e30f;
    }
    s = fminf(fmaxf(s, -3.4e38f), 3.4e38f);
}

// Requantiser and residual operands of the lean epilogue, in the form it reads.
struct DsqLean {
    unsigned long long inv2;              // inv, twice
    unsigned long long neg_lo2;           // -lo, twice
    unsigned long long res_delta2, res_lo2;
};
__device__ __forceinline__ DsqLean dsq_make_lean(const DsqEpi &e)
{
    DsqLean l;
    l.inv2 = dsq_pack2(e.rq.inv, e.rq.inv);
    l.neg_lo2 = dsq_pack2(-e.rq.lo, -e.rq.lo);
    l.res_delta2 = dsq_pack2(e.res_delta, e.res_delta);
    l.res_lo2 = dsq_pack2(e.res_lo, e.res_lo);
    return l;
}

// Residual codes 2 j and 2 j + 1 of eight packed codes as binary32.  The code goes into the
// low byte of 2^23 (one byte permutation or one shift and one LOP3), which is taken off again
// for two codes at a time: extracted and converted (I2F) they were 30 instructions of eight
// elements' 58, most of them on the pipe that bounds the epilogue; now 26 (64->64 at 56x56
// with residual, 4-bit, batch 64 16.5 -> 15.9 us).
template <int BITS>
__device__ __forceinline__ unsigned long long dsq_code_pair(uint32_t x, int j)
{
    constexpr uint32_t MAGIC = 0x4B000000u;
    uint32_t a, b;
    if (BITS == 4) {
        a = __byte_perm(x & 0x0F0F0F0Fu, MAGIC, 0x7440 | j);
        b = __byte_perm((x >> 4) & 0x0F0F0F0Fu, MAGIC, 0x7440 | j);
    } else {
        constexpr uint32_t M = (1u << BITS) - 1u;
        a = ((x >> (2 * BITS * j)) & M) | MAGIC;
        b = ((x >> (2 * BITS * j + BITS)) & M) | MAGIC;
    }
    return dsq_add2(dsq_pack2(__uint_as_float(a), __uint_as_float(b)), 0xCB000000CB000000ull);
}

// Raw accumulators of eight consecutive output channels of one position -> their
// packed codes; sc, bi: the channels' dsq_codes_affine in pairs, res: the
// position's residual codes of those channels (both in fields of SLOT bits).  FACC: the
// accumulators are whole numbers in binary32.
template <int BITS, bool RES, bool LO, int SLOT = BITS, bool FACC = false>
__device__ __forceinline__ uint32_t dsq_lean_codes8(const uint32_t (&v)[8],
                                                    const unsigned long long (&sc)[4],
                                                    const unsigned long long (&bi)[4],
                                                    uint32_t res, const DsqLean &l)
{
    int q[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        unsigned long long y = dsq_fma2(
            FACC ? dsq_pack2(__uint_as_float(v[2 * c]), __uint_as_float(v[2 * c + 1]))
                 : dsq_pack2(__int2float_rn((int)v[2 * c]), __int2float_rn((int)v[2 * c + 1])),
            sc[c], bi[c]);
        if (RES) y = dsq_add2(y, dsq_fma2(dsq_code_pair<SLOT>(res, c), l.res_delta2, l.res_lo2));
        if (LO) y = dsq_add2(y, l.neg_lo2);
        dsq_requant2<BITS>(y, l.inv2, q[2 * c], q[2 * c + 1]);
    }
    return dsq_pack8<BITS, SLOT>(q);
}

// Which accumulator column holds output channel ch of a group of 32.  The epilogue
// reads tensor memory in the 16x256b shape, where a lane gets two columns of every
// block of eight; with the channels laid out like this (the weight rows are put in
// this order when they are expanded) those are eight CONSECUTIVE channels: one
// scale and bias set per lane for all its positions - they stay in registers - and
// a whole word of codes, with no exchange between lanes.
__host__ __device__ inline int dsq_column_of(int ch)
{
    return (ch & ~31) | (((ch >> 1) & 3) << 3) | (((ch >> 3) & 3) << 1) | (ch & 1);
}
#endif
