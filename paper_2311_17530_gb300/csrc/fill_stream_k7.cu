// Streamed line fill for k = 7: the whole-column form (fill_lines_wide.cuh).
#include "fill_lines_stream.cuh"
#include "fill_lines_wide.cuh"

namespace msadp {

cudaError_t launch_fill_stream_k7(const LaunchDesc &L, int grid, cudaStream_t s, int rho_s) { return launch_wide<7>(L, grid, s, rho_s); }
int fill_stream_ctas_k7() { return wide_ctas<7>(); }

}  // namespace msadp
