// More of the rules of csrc/dsq_gemm8_rule.h for a GPU of 148 SMs.  Built and driven by gemm_rules.py.
#include "gemm_rule_host.cpp"

extern "C" {
// 0 the fused kernel, 1 two passes, 2 the little-work kernel
int gemm_form(int64_t M, int64_t N, int64_t K, int bits, int outs, double clocks, int room)
{
    return dsq_gemm_form(M, N, K, bits, outs, bits != 4, clocks, room != 0, true, 148);
}
// rows and warps of a block of the little-work kernel
void gemm_small(int64_t M, int64_t N, int64_t K, int bits, int outs, int *rows, int *warps)
{
    const DsqGemmSmallTile t = dsq_gemm_small_tile(M, N, bits == 2 ? (K + 63) / 64 : (K + 31) / 32, bits, outs, 148);
    *rows = 16 * t.mt;
    *warps = t.warps;
}
// columns of a block of the weight-only kernel of few rows, 0: two passes
int wgemm_form(int64_t M, int64_t N, int64_t K, double clocks)
{
    if (!dsq_wgemm_takes_small(M, N, K, 148, clocks) && !dsq_wgemm_takes_wide(M, N, K, 148, clocks)) return 0;
    return dsq_wgemm_small_columns(M, N, 148);
}
}
