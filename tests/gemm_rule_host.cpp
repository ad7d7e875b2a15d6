// The rules of csrc/dsq_gemm8_rule.h for a GPU of 148 SMs.  Built and driven by test_gemm_rule.py.
#include "../paper_1908_05033_b200/csrc/dsq_gemm8_rule.h"

extern "C" {
double tile(int64_t M, int64_t N, int64_t kblocks, int widest, int *bn, int *split)
{
    const DsqG8Tile t = dsq_g8_tile(M, N, kblocks, widest, 148, [] { return 33; });
    *bn = t.bn;
    *split = t.split;
    return t.clocks;
}
int two_passes(int64_t M, int64_t N, int64_t K, int bits, int f4, double clocks)
{
    return dsq_g8_two_passes(M, N, K, bits, f4 != 0, clocks);
}
int takes_small(int64_t M, int64_t N, int64_t K, double clocks)
{
    return dsq_wgemm_takes_small(M, N, K, 148, clocks);
}
}
