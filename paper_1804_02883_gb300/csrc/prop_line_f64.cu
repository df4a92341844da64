// prop_line_f64.cu -- the FP64 instantiations of the streaming propagator
// passes of prop_line.cuh (the differential solve is FP32 only).
#include "prop_line.cuh"

namespace epdlb {

cudaError_t line_col(const PropK<double> &k, cudaStream_t s) { return line_col_t<double>(k, s); }
cudaError_t line_row(const PropK<double> &k, int m, bool, int *blocks, cudaStream_t s) { return line_row_t<double, false>(k, m, blocks, s); }

} // namespace epdlb
