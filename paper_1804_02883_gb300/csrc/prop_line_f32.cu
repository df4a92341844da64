// prop_line_f32.cu -- the FP32 instantiations of the streaming propagator
// passes of prop_line.cuh.
#include "prop_line.cuh"

namespace epdlb {

cudaError_t line_col(const PropK<float> &k, cudaStream_t s) { return line_col_t<float>(k, s); }
cudaError_t line_row(const PropK<float> &k, int m, bool diff, int *blocks, cudaStream_t s)
{
    return diff ? line_row_t<float, true>(k, m, blocks, s) : line_row_t<float, false>(k, m, blocks, s);
}

} // namespace epdlb
