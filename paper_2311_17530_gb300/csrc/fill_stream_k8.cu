// Streamed line fill for k = 8: the whole-column form (fill_lines_wide.cuh).
#include "fill_lines_stream.cuh"
#include "fill_lines_wide.cuh"

namespace msadp {

cudaError_t launch_fill_stream_k8(const LaunchDesc &L, int grid, cudaStream_t s, int rho_s) { return launch_wide<8>(L, grid, s, rho_s); }
int fill_stream_ctas_k8() { return wide_ctas<8>(); }

}  // namespace msadp
