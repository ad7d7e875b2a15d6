// More of the rules of csrc/dsq_gemm8_rule.h for a GPU of 148 SMs.  Built and driven by gemm_rules.py.
#include "gemm_rule_host.cpp"

extern "C" {
// 0 the fused kernel, 1 two passes, 2 the little-work kernel
int gemm_form(int64_t M, int64_t N, int64_t K, int bits, int outs, double clocks, int room)
{
    return dsq_gemm_form(M, N, K, bits, outs, bits != 4, clocks, room != 0, true, 148);
}
}
