// Host-side pieces that the kernels' translation units share.  Internal to the library.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "dsq_epilogue.cuh"
#include "dsq_gemm8_rule.h"
#include "dsq_launch.h"

typedef CUresult (*DsqEncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                     const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                     const cuuint32_t *, CUtensorMapInterleave,
                                     CUtensorMapSwizzle, CUtensorMapL2promotion,
                                     CUtensorMapFloatOOBfill);
typedef CUresult (*DsqEncodeIm2colFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                      const cuuint64_t *, const cuuint64_t *, const int *,
                                      const int *, cuuint32_t, cuuint32_t, const cuuint32_t *,
                                      CUtensorMapInterleave, CUtensorMapSwizzle,
                                      CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
// driver entry points (looked up once; nullptr when the driver lacks them)
DSQ_HIDDEN DsqEncodeTiledFn dsq_encode_tiled_fn();
DSQ_HIDDEN DsqEncodeIm2colFn dsq_encode_im2col_fn();

// epilogue variants of the convolution kernels: codes only, without / with a
// residual operand; any outputs
enum { DSQ_EPI_CODES = 1, DSQ_EPI_CODES_RES = 2, DSQ_EPI_GENERAL = 3 };

// 3x3, pad 1 convolution (strides 1 and 2) on an expanded shared-memory window
// (dsq_conv3.cu).  Arguments are those of dsq_conv2d after validation.
// Returns DSQ_ERR_UNSUPPORTED without launching anything when the geometry is
// not one it handles; the caller then takes the im2col kernel.
DSQ_HIDDEN int dsq_conv3_window(const void *act_codes, const dsq_nhwc_t *shape, int bits,
                                const void *w_packed, const dsq_conv_t *conv, const DsqEpi &e,
                                int epi_kind, int small_acc, void *workspace,
                                cudaStream_t stream);

// 1x1 convolution from codes to codes (dsq_pw.cu).  Arguments are those of
// dsq_conv2d after validation, `e` writing codes only.  Returns
// DSQ_ERR_UNSUPPORTED without launching anything where it does not apply.
DSQ_HIDDEN int dsq_pointwise(const void *act_codes, const dsq_nhwc_t *shape, int bits,
                             const void *w_packed, const dsq_conv_t *conv, const DsqEpi &e,
                             void *workspace, cudaStream_t stream);

// Dense convolution with little work (dsq_conv_small.cu).  Arguments as dsq_pointwise,
// any outputs; lean: codes only, with a requantiser the lean epilogue takes.
DSQ_HIDDEN int dsq_conv_small(const void *act_codes, const dsq_nhwc_t *shape, int bits,
                              const void *w_packed, const dsq_conv_t *conv, const DsqEpi &e,
                              int lean, cudaStream_t stream);

// Opt-in to large dynamic shared memory, once per kernel and device (an attribute
// of the function on a device): one bit per device ordinal in *configured.
static inline int dsq_allow_smem(const void *func, int bytes, std::atomic<unsigned long long> *configured)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return DSQ_ERR_CUDA;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (configured->load(std::memory_order_acquire) & bit) return DSQ_OK;
    if (cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess)
        return DSQ_ERR_CUDA;
    configured->fetch_or(bit, std::memory_order_release);
    return DSQ_OK;
}

// Two-pass GEMM (dsq_gemm8.cu): every packed row is expanded once, to int8 or 4-bit
// floating point, into caller-provided scratch, then a GEMM reads it by TMA.
// dsq_gemm8_scratch_bytes: scratch the path needs (0: not a problem it takes;
// force: whatever the size).
// dsq_gemm8_launch: arguments as dsq_gemm after validation, `scratch`
// 1024-byte aligned and at least that large.
// dsq_gemm8_form: the kernel that dsq_gemm takes (dsq_gemm8_rule.h), outs: arrays written.
DSQ_HIDDEN DsqGemmForm dsq_gemm8_form(int64_t M, int64_t N, int64_t K, int bits, int outs, bool room, bool little);
DSQ_HIDDEN size_t dsq_gemm8_scratch_bytes(int64_t M, int64_t N, int64_t K, int bits, int force);
DSQ_HIDDEN int dsq_gemm8_launch(const void *A_codes, const void *B_codes, int64_t M, int64_t N,
                                int64_t K, int bits, int32_t *C_i32, const float *row_scale,
                                float *D_f32, void *workspace, void *scratch,
                                cudaStream_t stream);

// GEMM with little work (dsq_gemm_small.cu): arguments as dsq_gemm after validation, of problems that
// dsq_gemm8_form gives it; no workspace.
DSQ_HIDDEN int dsq_gemm_small(const void *A_codes, const void *B_codes, int64_t M, int64_t N, int64_t K,
                              int bits, int32_t *C_i32, const float *row_scale, float *D_f32,
                              cudaStream_t stream);

// Weight-only GEMM for few rows (dsq_wgemm_small.cu): arguments as dsq_wgemm_bf16
// after validation; no workspace.
DSQ_HIDDEN int dsq_wgemm_small(const void *X, const void *W, int64_t M, int64_t N, int64_t K,
                               int bits, int odd, const float *col_scale, const float *col_bias,
                               float *Y, cudaStream_t stream);

// Weights of 3x3 stride-1 pad-1 dense convolutions (2- and 4-bit, 64 or a
// multiple of 128 input channels) are stored twice in the blob
// dsq_pack_weights writes: the packed rows, and behind them (1024-byte
// aligned) the same rows already expanded to the int8 bytes the tensor core
// multiplies for the grid Delta (c + 1/2), laid out K step by K step in the
// order the window kernel consumes them (Cout rows of ksteps x 128 bytes).
// The kernel then copies weight tiles by TMA straight into the swizzled operand
// ring, with no expansion warps.  enabled = 0: this geometry has no such copy.
// f4: 2-bit rows of 64, 128 or k * 256 channels are kept as 4-bit floating-point
// operands (expand_word_f4) instead, 256 codes to a K step of 128 bytes; they fill half
// of the room.
struct DsqW8Info { int enabled; size_t offset; int ksteps; size_t bytes; int f4; };
DSQ_HIDDEN DsqW8Info dsq_w8_info(const dsq_conv_t *conv, int bits);
// builds the expanded copy from the packed rows at the start of `blob`
DSQ_HIDDEN int dsq_w8_build(void *blob, const dsq_conv_t *conv, int bits, cudaStream_t stream);
