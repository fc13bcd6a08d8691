// pp_hlines_512.cu -- block-scaled FP64-class line kernels of 512 complex points.
#include "pp_hlines.cuh"

namespace pp {
cudaError_t hlines_512(const LineArgs& a, int oy, cudaStream_t st) { return dispatch_hlines<512>(a, oy, st); }
void hlines_shape_512(int oy, int* lpc, int* threads) { hlines_shape<512>(oy, lpc, threads); }
}  // namespace pp
