// Which tiles the second pass of the two-pass GEMMs takes, and which problems take the two
// passes at all.  Host code without CUDA, so that it can be compared with measured times
// anywhere (tests/test_gemm_rule.py).  Internal to the library.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

constexpr int DSQ_G8_BM = 256;       // tile height of a CTA pair

// Tile width, whether K is split over the two pairs of a cluster, and the clocks (at 1.9 GHz)
// that the second pass is expected to take.
struct DsqG8Tile {
    int bn, split;
    double clocks;
};

// For a problem of kblocks K blocks of 128 bytes; widest: tensor-memory columns of an
// accumulator; resident(): clusters of two pairs that fit on the GPU at once.
//
// A pair reads 256 + BN rows of 128 bytes for a K block of a tile, and that is what a block's
// time goes with, for 8-bit, bf16 and 4-bit operands alike (about 15 TB/s over all pairs, from
// the L2): 1.2 clocks a row; a tile costs 1500 more.  The CTA pairs take their tiles in waves,
// and the width with the cheapest waves is taken.  Split: only with all the clusters resident
// at once and twelve K blocks a part; the exchange of the partial sums grows with the width.
// (Four pairs a cluster gained nothing more: 15 such clusters are resident and the exchange
// doubles.)
//
// Measured: all widths, whole and split K, of 591 problems of 64 to 6144 a side, 1 to 4
// bits, back to back in a graph and one at a time after an L2 flush, and of 233 more that it was
// not fitted to: of those the width taken is 0.22 % slower than the fastest one on average, more
// than 3 % in 11 of 466 timings.  (A rule from the tensor cores' rate, 2.5 BN clocks a block,
// 330 + 0.72 BN at least: 0.64 %, 33 of them.)
template <class Resident>
inline DsqG8Tile dsq_g8_tile(int64_t M, int64_t N, int64_t kblocks, int widest, int sms, Resident resident)
{
    const int64_t pairs = std::max(sms / 2, 1), m_tiles = (M + DSQ_G8_BM - 1) / DSQ_G8_BM;
    DsqG8Tile best = {0, 0, 0.0};
    for (int split = 1; split <= 2; ++split)
        for (int bn = widest / 32 * 32; bn >= 64; bn -= 32) {      // (pairs take N in steps of 32)
            if (split == 2 && (bn % 64 != 0 || kblocks < 24)) continue;
            const int64_t tiles = m_tiles * ((N + bn - 1) / bn);
            if (split == 2 && tiles > resident()) continue;
            const int64_t waves = split == 2 ? 1 : (tiles + pairs - 1) / pairs;
            const double block = 1.2 * (DSQ_G8_BM + bn);
            const double clocks = (double)waves * ((double)((kblocks + split - 1) / split) * block + 1500.0) +
                                  (split == 2 ? 1000 + 30 * bn : 20 * bn);
            if (best.bn == 0 || clocks < best.clocks) best = DsqG8Tile{bn, split, clocks};
        }
    return best;
}

// Whether dsq_gemm does better in two passes than in the fused kernel that expands both operands
// for every tile; clocks: of the second pass.  Microseconds of both, fitted to 522
// problems of 2 to 4 bits and 128 to 6144 a side with one or both outputs.  Two passes: their launches,
// the tiles of the second, the bytes of the first, the outputs (turned round in shared memory
// where rows are not whole sectors).  The fused kernel: its rounds of K, the expansion of each row
// once per tile (3-bit rows one K step a round), the outputs (one word at a time where rows
// are no multiple of 16 bytes).  The slower path is taken for 32 of them, 0.7 % of time on average
// (fitted to 292 of them, for 14 of the other 230, 0.7 %).  The expansion launched
// dependently costs less than the fits' 6.0 us: with 5.3 (4-bit floating point) and 5.7 the slower
// path is taken for 29 of 400 other problems, 0.7 % of time on average; with 6.0 for 34, 1.0 %.  Fused / two passes, us: 4-bit 1024^3
// 6.7 / 8.8, 2048^3 16.0 / 15.6 (either), 3072x3072x1024 20.6 / 18.1, 2500x1111x1777 29 / 12.5; 3-bit
// 1024^3 10.1 / 7.8, 2048^3 22 / 14.6; 2-bit 2048^3 16.1 / 13.9.
struct DsqGemmTimes { double fused, two; };
inline DsqGemmTimes dsq_gemm_times(int64_t M, int64_t N, int64_t K, int bits, bool f4, double clocks)
{
    struct Fused { double fixed, k, nk, out, words, word; };
    static const Fused fused[3] = {{4.3, 1.76, 0.483, 1.11, 2.5, 4.6},
                                   {4.7, 4.52, 1.015, 0.965, 0.8, 5.5},
                                   {4.3, 1.85, 0.506, 1.21, 0.5, 5.9}};
    const double out = (double)M * (double)N * 1e-6, k = (double)K * 1e-3;
    const Fused &f = fused[bits - 2];
    const double two = (f4 ? 5.3 : 5.7) + clocks / 2310.0 + (N % 8 ? 1.02 : 0.65) * out +
                       0.157e-6 * (double)(M + N) * (double)K * (bits / 8.0 + (f4 ? 0.5 : 1.0));
    return {f.fixed + f.k * k + f.nk * out * k + f.out * out + (N % 4 ? f.words + f.word * out : 0.0), two};
}
inline bool dsq_g8_two_passes(int64_t M, int64_t N, int64_t K, int bits, bool f4, double clocks)
{
    // beyond the range of the fits (4096^3: 75 / 52)
    if ((double)M * (double)N * (double)K >= 1.5e10) return true;
    const DsqGemmTimes t = dsq_gemm_times(M, N, K, bits, f4, clocks);
    return t.two < t.fused;
}

// The GEMM with little work (dsq_gemm_small.cu): 16 mt rows x 32 columns a block of `warps` warps, and the
// microseconds it is expected to take.  units: of a packed row; outs: arrays written.
// An SM holds as many blocks as their registers allow, and each round of them takes a block's chain
// (its launch, its chunks of K a warp) and what they do beside each other; the outputs come on top.
// 32 rows a block expand B's rows half as often, at more registers, us with 16 / 32 rows: 3-bit 2177x35x2843
// 7.4 / 5.3, 4-bit 150x2024x1052 4.9 / 3.9, 4-bit 512^3, one round of either, 2.3 / 2.9.  They count a tenth
// more than they are expected to take: where it is close, 16 rows are as good or better.
// Fitted to 1079 problems of 16 to 6144 a side and up to 1.5e9 multiply-accumulates, one or both outputs
// (8 % off in the mean).  Of 541 others what is taken, among these and the other kernels, is 1.2 %
// slower than the fastest on average (2.7 % with blocks of 16 rows alone and none above 1e9).
struct DsqGemmSmallTile { int mt, warps; double us; };
inline DsqGemmSmallTile dsq_gemm_small_tile(int64_t M, int64_t N, int64_t units, int bits, int outs, int sms)
{
    // blocks of four warps that an SM holds; a warp's time for a chunk; an SM's for a block and for a
    // chunk of one: [mt - 1][bits - 2] and with four and eight warps
    static const int held[2][3] = {{4, 3, 4}, {3, 2, 3}};
    static const double walk[2][3] = {{0.103, 0.153, 0.075}, {0.445, 0.338, 0.249}};
    static const double block[2][3][2] = {{{0.0, 0.128}, {0.023, 0.273}, {0.0, 0.088}},
                                          {{0.107, 0.129}, {0.347, 0.314}, {0.149, 0.102}}};
    static const double chunk[2][3][2] = {{{0.066, 0.061}, {0.080, 0.086}, {0.035, 0.035}},
                                          {{0.076, 0.075}, {0.090, 0.107}, {0.037, 0.040}}};
    const int64_t chunks = (units + 3) / 4;
    DsqGemmSmallTile best = {0, 0, 0.0};
    for (int mt = 1; mt <= 2; ++mt)
        for (int eight = 0; eight < 2; ++eight) {
            const int warps = 4 + 4 * eight, a = mt - 1, b = bits - 2;
            const int64_t blocks = (M + 16 * mt - 1) / (16 * mt) * ((N + 31) / 32);
            const int64_t most = held[a][b] / (1 + eight), rounds = blocks / (most * sms);
            const int64_t rest = (blocks - rounds * most * sms + sms - 1) / sms;
            const double chain = 0.731 + walk[a][b] * (double)((chunks + warps - 1) / warps);
            const double beside = block[a][b][eight] + chunk[a][b][eight] * (double)chunks;
            const double us = 0.867 + (double)rounds * (chain + (double)most * beside) +
                              (rest ? chain + (double)rest * beside : 0.0) +
                              (N % 2 ? 1.248e-6 : 1.079e-6) * (double)M * (double)N * outs;
            const double counted = mt == 2 ? 1.1 * us : us;
            if (best.mt == 0 || counted < best.us) best = DsqGemmSmallTile{mt, warps, counted};
        }
    return best;
}

// Which kernel dsq_gemm takes.  `room`: the caller's workspace holds the expanded operands; without
// it the little-work kernel has only the fused one to be faster than (3-bit 439x592x1602: fused 13.4 us,
// little work 7.9, two passes 8.6).  `little`: that kernel may be taken at all.
enum DsqGemmForm { DSQ_GEMM_FUSED, DSQ_GEMM_TWO_PASSES, DSQ_GEMM_SMALL };
inline bool dsq_gemm_may_take_two(int64_t M, int64_t N, int64_t K) { return M >= 128 && N >= 128 && K >= 128; }
inline DsqGemmForm dsq_gemm_form(int64_t M, int64_t N, int64_t K, int bits, int outs, bool f4, double clocks, bool room,
                                 bool little, int sms)
{
    const bool two = room && dsq_gemm_may_take_two(M, N, K) && dsq_g8_two_passes(M, N, K, bits, f4, clocks);
    // (up to what its estimate was fitted to, and the rows of a grid)
    if (little && (double)M * (double)N * (double)K < 1.5e9 && (M + 15) / 16 <= 65535) {
        const int64_t units = bits == 2 ? (K + 63) / 64 : (K + 31) / 32;
        const DsqGemmTimes t = dsq_gemm_times(M, N, K, bits, f4, clocks);
        if (dsq_gemm_small_tile(M, N, units, bits, outs, sms).us <= (two ? t.two : t.fused)) return DSQ_GEMM_SMALL;
    }
    return two ? DSQ_GEMM_TWO_PASSES : DSQ_GEMM_FUSED;
}

// The weight-only GEMM of few rows (dsq_wgemm_small.cu) for more than 32 rows: waves of blocks of 64 rows x 16
// or 32 columns, 2.6 us for every 1024 of K, three quarters of that at 33 rows; 32 columns take up to 1.5
// times as long, which pays where it saves a wave.  16 / 32 columns, us, 4-bit: 64x4096x4096
// 23.1 / 15.9, 150x1500x1000 8.1 / 6.3, 332x659x1136 9.4 / 7.8, 128x1024x1024 (one wave of either) 4.6 / 6.3.
inline double dsq_wgemm_small_waves(int64_t M, int64_t N, int sms, int columns)
{
    return std::ceil((double)((N + columns - 1) / columns) * (double)((M + 63) / 64) / sms) * (columns == 32 ? 1.5 : 1.0);
}
inline int dsq_wgemm_small_columns(int64_t M, int64_t N, int sms)
{
    return dsq_wgemm_small_waves(M, N, sms, 32) < dsq_wgemm_small_waves(M, N, sms, 16) ? 32 : 16;
}
inline double dsq_wgemm_small_us(int64_t M, int64_t N, int64_t K, int sms, int columns)
{
    const double rows = M < 64 ? 0.75 + 0.25 / 31.0 * (double)(M - 33) : 1.0;
    return 2.2 + dsq_wgemm_small_waves(M, N, sms, columns) * (double)((K + 1023) / 1024) * 2.6 * rows;
}
// And two passes, of `clocks` in the second.
inline double dsq_wgemm_two_us(int64_t N, int64_t K, double clocks)
{
    return 5.5 + 3.2e-7 * (double)N * (double)K + 5.22e-4 * clocks;
}

// Whether it does better than two passes, for more than 32 rows (up to those it always does:
// 4096x4096 4-bit 9.2 us): in blocks of 16 columns, or where those of 32 are the better ones and
// only they beat the two passes.  Of 360 problems of 33 to 1200 rows, 1 to 4 bits, what is taken is 1.0 % slower
// than the fastest of the three on average, 23 of them by more than 5 %.  (With 5.0 us of launches in
// place of 5.5 the same, and 22; but where it is close the kernel of few rows is the better one: its sums are closer to
// those in 64 bits, 5e-8 of the result against 5e-8 to 1e-7 in two passes at K = 2000, 1e-7 / 3e-7 at
// 5848.)  64 rows, 16 columns / 32 / two passes, us, 4-bit:
// 4096x4096 23.1 / 15.9 / 19.8, 6144x6144 47.8 / 41.8 / 34.8, 6144x1024 12.0 / 11.8 / 11.2, 1500x2000 7.0 / 9.0 / 11.5.
inline bool dsq_wgemm_takes_small(int64_t M, int64_t N, int64_t K, int sms, double clocks)
{
    return dsq_wgemm_small_us(M, N, K, sms, 16) < dsq_wgemm_two_us(N, K, clocks);
}
inline bool dsq_wgemm_takes_wide(int64_t M, int64_t N, int64_t K, int sms, double clocks)
{
    return dsq_wgemm_small_columns(M, N, sms) == 32 &&
           dsq_wgemm_small_us(M, N, K, sms, 32) < dsq_wgemm_two_us(N, K, clocks);
}
