// The rule for 1x1 layers from codes to codes on a GPU of 148 SMs.  Built and driven by test_conv_pointwise_rule.py.
#include "../paper_1908_05033_b200/csrc/dsq_conv_rule.h"

extern "C" int takes_small(const dsq_nhwc_t *shape, const dsq_conv_t *conv, int bits, int M, int chunks, int residual)
{
    return dsq_small_tile(M, conv->Cout, chunks, bits, 148).us <=
           dsq_small_other(shape, bits, conv, M, 1, 1, 148, residual);
}
