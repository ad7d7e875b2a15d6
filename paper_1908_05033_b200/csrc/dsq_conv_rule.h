// How the window kernel tiles a 3x3 convolution, and which kernel a dense convolution with little
// work takes.  Host code without CUDA, so that it can be compared with measured times
// anywhere (tests/test_conv_rule.py).  Internal to the library.
#pragma once

#include <algorithm>
#include <cstdint>

#include "../../include/dsq.h"

// ---------------------------------------------------------------------------
// the window kernel (dsq_conv3.cu)
// ---------------------------------------------------------------------------
constexpr int W3_BM = 128;             // positions of a plain tile
constexpr int W3_F4_TP = 240;          // of a transposed one on 4-bit floating-point operands, at most
constexpr int W3_MAX_COUT = 1024;      // scale / bias of the layer stay in shared memory

// planes of a pixel's channels, K steps of a plane and taps of a K step, the latter two of
// rows that are not 128 bytes long
inline void w3_steps(int Cin, int f4, int *npl, int *kpp, int *tps)
{
    const int full = f4 ? 256 : 128;               // channels of a 128-byte row
    *npl = Cin < full ? 1 : Cin / full;
    *tps = Cin < full ? full / Cin : 1;
    *kpp = (9 + *tps - 1) / *tps;
}

// Positions of a transposed tile, at most `most`: what fills as many passes of the `mstep`
// CTAs of an N tile as the largest tile would take, so that the last pass is no emptier than
// the others.  (4-bit, batch 64, largest / this: 28x28 128->128 11.6 / 10.8 us, 14x14 256->256
// 11.3 / 10.5, 7x7 512->512 15.6 / 14.2 (12.2 since); 2-bit 28x28 512->512 at batch 32 27.9 / 26.9.)  No
// fewer than 112: the instructions get shorter, the weights' K steps do not (28x28 128->128 at
// batch 16: 96 to 144 positions alike).  With more than four passes the last one weighs little, and
// larger tiles have less overhead each (64->64 at 56x56, six passes: 256 positions 15.4, 240
// 15.8).
inline int w3_tile(int64_t positions, int mstep, int most)
{
    const int64_t passes = (positions + (int64_t)most * mstep - 1) / ((int64_t)most * mstep);
    if (passes > 4) return most;
    const int64_t each = (positions + passes * mstep - 1) / (passes * mstep);
    return (int)std::min<int64_t>(most, std::max<int64_t>(112, (each + 15) / 16 * 16));
}

// Positions of the numbering up to the last pixel, channel tiles, CTAs a channel tile.
struct W3Work {
    int64_t positions;
    int Hp, Wp, n_tiles, mstep;
};
inline W3Work w3_work(const dsq_nhwc_t *shape, const dsq_conv_t *conv, int pair, int bn, int sms)
{
    W3Work w;
    const int Ho = (shape->H - 1) / conv->stride + 1, Wo = (shape->W - 1) / conv->stride + 1;
    const bool two = pair || conv->stride == 2;
    w.Hp = two ? shape->H / 2 + 1 : shape->H + 1;
    w.Wp = conv->stride == 2 ? shape->W / 2 + 1 : shape->W + 1;
    w.positions = ((int64_t)shape->N - 1) * w.Hp * w.Wp + (int64_t)((Ho - 1) / (pair ? 2 : 1)) * w.Wp + Wo;
    w.n_tiles = (conv->Cout + bn - 1) / bn;
    w.mstep = std::max(sms / w.n_tiles, 1);
    return w;
}

// channels of a plain tile
inline int w3_plain_bn(int Cout) { return Cout >= 256 ? 256 : (Cout + 63) / 64 * 64; }

inline bool w3_takes_f4(const dsq_conv_t *conv, int bits, int expanded)
{
    return bits == 2 && expanded && (conv->Cin <= 128 || conv->Cin % 256 == 0);
}

// 4-bit operands at stride 2, where the blob has no expanded weights: the im2col kernel is
// the faster one unless a CTA expands its weights once - they stay resident, or one pass
// of large tiles does (28x28 128->256 at batch 64 10.3 us against 11.9, at batch 16, tiles of 112, 7.7
// against 7.5; 112x112 128->128 18.8 against 17.3; 14x14 256->512 12.2 against 10.8).
inline bool w3_takes_stride2(int Cin, int tile, int64_t passes)
{
    return Cin == 64 || (Cin == 128 && passes == 1 && tile >= 160);
}

// Microseconds of the window kernel's plain tiles: `steps` K steps over all passes of a CTA.
// Fitted to 190 layers of up to 64 outputs at 2 and 4 bits without the expanded copy (5 % off, 14 % at
// most) and to 250 on images of 255 to 700 columns, whose windows come in three bands.
inline double dsq_conv3_plain_estimate(int bits, int bn, double steps, bool bands)
{
    if (!bands) return 3.7 + 0.29 * steps;
    if (bits == 3) return bn == 64 ? 0.1 + 1.25 * steps : bn < 256 ? 0.1 + 1.4 * steps : 15.0 + 0.6 * steps;
    return bn == 64 ? 3.7 + 0.41 * steps : bn < 256 ? 3.6 + 0.6 * steps : 7.2 + 0.5 * steps;
}

// Microseconds the window kernel takes for a layer of few tiles, or a negative number
// where it does not take it: start-up and the last epilogue, and for every pass of the
// CTAs its K steps.  expanded: the grid is Delta (c + 1/2), so that the weights come from the
// blob's expanded copy and 2-bit layers take 4-bit operands.  Fitted to 666 layers of 64 to 512
// channels at batches of 1 to 32 (5 % off in the mean, 17 % at most) and to 130 whose weights the kernel
// expands itself (4 %, 15 %).  Plain tiles: up to 64 outputs without the copy, which pairs of
// image rows want, and 8-bit windows that are too long for one piece.
inline double dsq_conv3_estimate(const dsq_nhwc_t *shape, int bits, const dsq_conv_t *conv, int expanded, int sms)
{
    const int Cin = conv->Cin;
    if (conv->KH != 3 || conv->pad != 1 || !(Cin == 64 || (Cin % 128 == 0 && Cin <= 1024)) ||
        conv->Cout > W3_MAX_COUT)
        return -1.0;
    const int f4 = w3_takes_f4(conv, bits, expanded), small = conv->stride == 1 && conv->Cout <= 64;
    int npl, kpp, tps;
    w3_steps(Cin, f4, &npl, &kpp, &tps);
    const bool bands = shape->W > 254;                    // of a plain tile's window
    if (conv->stride == 1 && !f4 && (small ? shape->W > 509 || (!expanded && bits != 3) : bands)) {
        const int bn = w3_plain_bn(conv->Cout);
        const W3Work w = w3_work(shape, conv, 0, bn, sms);
        const int64_t per_pass = (int64_t)W3_BM * w.mstep;
        return dsq_conv3_plain_estimate(
            bits, bn, (double)((w.positions + per_pass - 1) / per_pass * npl * (bits == 3 ? 9 : kpp)), bands);
    }
    if (small) kpp = (12 + tps - 1) / tps;               // (pairs of image rows: twelve taps)
    const W3Work w = w3_work(shape, conv, small, 128, sms);
    const int tile = w3_tile(w.positions, w.mstep, f4 ? W3_F4_TP : 256);
    const int64_t passes = (w.positions + (int64_t)tile * w.mstep - 1) / ((int64_t)tile * w.mstep);
    const double steps = (double)passes * npl * kpp, t = tile / 256.0;
    if (conv->stride == 1)
        return f4          ? 3.7 + steps * (1.41 * t - 0.36)
               : bits == 3 ? 4.5 + steps * (t - 0.07)
               : expanded  ? 3.8 + steps * (0.754 * t - 0.076)
                           : 3.7 + steps * (0.66 * t + 0.07);
    if (bits != 3 && !f4 && !w3_takes_stride2(Cin, tile, passes)) return -1.0;
    return f4 ? 3.4 + steps * (2.24 * t - 0.49) : bits == 3 ? 4.8 + steps * (1.59 * t - 0.27) : 3.6 + steps * (1.39 * t - 0.215);
}

// ---------------------------------------------------------------------------
// the little-work kernel (dsq_conv_small.cu)
// ---------------------------------------------------------------------------
// 16 mt pixels x 32 channels a block of `warps` warps, and the microseconds it is expected to take
struct DsqSmallTile {
    int mt, warps;
    double us;
};

// Fitted to the layers of the ResNet-18- and MobileNetV2-shaped networks at batches of 1, 2 and 4:
// the longer of a block's chain (0.55 us for every chunk a warp walks, 0.33 where it asks for the next one's
// activations ahead) and what the blocks of an SM take together (most of it per warp, whatever it
// has to do).  Of 159 layers of those networks, images of half to 1.2 times their sides, batches of 1 to
// 12: 1.1 % slower than the fastest of the five forms on average (2.0 % with 0.55 for both).
inline DsqSmallTile dsq_small_tile(int M, int Ncols, int chunks, int bits, int sms)
{
    DsqSmallTile best = {0, 0, 0.0};
    for (int mt = 1; mt <= 2; ++mt)
        for (int warps = 4; warps <= (mt == 1 ? 16 : 8); warps *= 2) {
            const double blocks = (double)((M + 16 * mt - 1) / (16 * mt)) * ((Ncols + 31) / 32);
            // (a 2-bit unit is twice the arithmetic, 3-bit fields take twice the instructions)
            const double f = bits == 4 ? 1.0 : 2.0;
            const double fixed = mt == 1 ? (warps == 4 ? 0.44 : warps == 8 ? 1.1 : 2.5) : (warps == 4 ? 0.7 : 1.35);
            const double per_block = fixed + f * (mt == 1 ? 0.06 : 0.09) * chunks;
            const double chain = 1.5 + 0.05 * warps + (mt == 1 ? 0.33 : 0.55) * (bits == 4 ? 1.0 : 1.3) * ((chunks + warps - 1) / warps);
            const double us = std::max(chain, 1.2 + blocks / sms * per_block);
            if (best.mt == 0 || us < best.us) best = DsqSmallTile{mt, warps, us};
        }
    return best;
}

// And what the other kernel for a layer of M output pixels takes: the window kernel as it says
// itself; the 1x1 kernel a launch, its outputs and its planes (464 layers of 16 to 1024 outputs, batches
// of 1 to 16, 6 % off in the mean; more than 3 % slower than the faster kernel 8 of them, 0.3 % on average, where
// 2.9 + M Cout / 3.7e6 left 73 and 3.0 %); the im2col kernel a floor that grows with K (the few CTAs such a layer has walk it
// alone) plus its work at full rate, and twice that at 3 bits, where a round is one K step.
// Measured: 1758 3x3 layers of 64 to 512 channels in and 32 to 1280 out (strides 1 and 2, 2 to
// 4 bits, both weight grids, batches of 1 to 32): the slower kernel for 23 of them, 0.2 % of time on average;
// 2970 others (1x1 to binary32, 16 to 320 channels): for 123, 1.1 %; 708 on images of 255 to 700 columns and
// 3 to 30 rows: for 32, 1.1 %.  (Without the limit on the outputs, the plain tiles and the factor for
// 3 bits: 53, 0.6 %; 205, 2.8 %; 72 and 3.4 % without the plain tiles.)
inline double dsq_small_other(const dsq_nhwc_t *shape, int bits, const dsq_conv_t *conv, int M, int expanded, int lean,
                              int sms, int residual = 0)
{
    const int ksize = conv->KH;
    if (ksize == 1 && lean)
        return 2.9 + 0.9e-6 * (double)M * conv->Cout + 0.41 * conv->Cin / 128.0 + (conv->stride == 2 ? 0.24 : 0.0) +
               (residual ? 0.73 : 0.0) + (bits == 3 ? 0.72 : 0.0);
    const double window = dsq_conv3_estimate(shape, bits, conv, expanded, sms);
    if (window > 0.0) return window;
    return (bits == 3 ? 2.05 : 1.0) *
           (4.3 + 0.23 * ksize * ksize * conv->Cin / 128.0 + (double)M * conv->Cout * ksize * ksize * conv->Cin / 4.5e8);
}
