// pp_hlines_1024.cu -- block-scaled FP64-class line kernels of 1024 complex points.
#include "pp_hlines.cuh"

namespace pp {
cudaError_t hlines_1024(const LineArgs& a, int oy, cudaStream_t st) { return dispatch_hlines<1024>(a, oy, st); }
void hlines_shape_1024(int oy, int* lpc, int* threads) { hlines_shape<1024>(oy, lpc, threads); }
}  // namespace pp
