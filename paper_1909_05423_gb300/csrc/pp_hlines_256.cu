// pp_hlines_256.cu -- block-scaled FP64-class line kernels of 256 complex points.
#include "pp_hlines.cuh"

namespace pp {
cudaError_t hlines_256(const LineArgs& a, int oy, cudaStream_t st) { return dispatch_hlines<256>(a, oy, st); }
void hlines_shape_256(int oy, int* lpc, int* threads) { hlines_shape<256>(oy, lpc, threads); }
}  // namespace pp
