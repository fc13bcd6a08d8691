// pp_hlines_64.cu -- block-scaled FP64-class line kernels of 64 complex points.
#include "pp_hlines.cuh"

namespace pp {
cudaError_t hlines_64(const LineArgs& a, int oy, cudaStream_t st) { return dispatch_hlines<64>(a, oy, st); }
void hlines_shape_64(int oy, int* lpc, int* threads) { hlines_shape<64>(oy, lpc, threads); }
}  // namespace pp
