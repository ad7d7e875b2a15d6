// Packed codes straight from global memory to the operands of mma.sync m16n8k32: what the
// kernels for little work share (dsq_conv_small.cu, dsq_gemm_small.cu).
//
// K is a list of units: 16 bytes of a packed row (32 codes of 4 bits, 64 of 2; 12 bytes = 32 codes at
// 3 bits), a lane's.  The order of K inside a unit is free as long as both operands agree.
#pragma once

#include "dsq_tc_common.cuh"

namespace {

__device__ __forceinline__ void mma_u8s8(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// words of a unit, and the four-code byte words it expands to
template <int BITS> struct Unit {
    static constexpr int WORDS = BITS == 3 ? 3 : 4;
    static constexpr int BYTE_WORDS = BITS == 2 ? 16 : 8;
};

template <int BITS>
__device__ __forceinline__ void load_unit(const uint8_t *src, bool in, int left, uint32_t (&v)[Unit<BITS>::WORDS])
{
    if (BITS == 3) {
        // (the row may end inside the unit: `left` bytes of it remain)
#pragma unroll
        for (int i = 0; i < Unit<BITS>::WORDS; ++i) {
            v[i] = 0u;
            if (in && 4 * i < left) v[i] = __ldg(reinterpret_cast<const uint32_t *>(src) + i);
        }
    } else {
        uint4 t = make_uint4(0u, 0u, 0u, 0u);
        if (in) t = __ldg(reinterpret_cast<const uint4 *>(src));
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[Unit<BITS>::WORDS - 1] = BITS == 3 ? v[2] : t.w;
    }
}

// byte word q of a unit (the same order for both operands)
template <int BITS, bool SIGNED>
__device__ __forceinline__ uint32_t byte_word(const uint32_t (&v)[Unit<BITS>::WORDS], int q, uint32_t orv)
{
    if (BITS == 4) return expand_word<4, SIGNED>(v[q >> 1], q & 1, orv);
    if (BITS == 2) return expand_word<2, SIGNED>(v[q >> 2], q & 3, orv);
    const int bit = 12 * q, i = bit >> 5;
    const uint32_t x = __funnelshift_r(v[i], v[i + 1 < Unit<BITS>::WORDS ? i + 1 : i], bit & 31);
    uint32_t b = (x & 7u) | ((x & 0x38u) << 5) | ((x & 0x1C0u) << 10) | ((x & 0xE00u) << 15);
    if (SIGNED) b = (b << 5) | orv;
    return b;
}

}  // namespace
