// The rules of csrc/dsq_conv_rule.h for a GPU of 148 SMs.  Built and driven by test_conv_rule.py.
#include "../paper_1908_05033_b200/csrc/dsq_conv_rule.h"

extern "C" {
double window_us(const dsq_nhwc_t *shape, const dsq_conv_t *conv, int bits, int expanded)
{
    return dsq_conv3_estimate(shape, bits, conv, expanded, 148);
}
int takes_small(const dsq_nhwc_t *shape, const dsq_conv_t *conv, int bits, int expanded, int lean, int M, int chunks)
{
    return dsq_small_tile(M, conv->Cout, chunks, bits, 148).us <=
           dsq_small_other(shape, bits, conv, M, expanded, lean, 148);
}
}
