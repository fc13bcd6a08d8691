// pp_hlines_128.cu -- block-scaled FP64-class line kernels of 128 complex points.
#include "pp_hlines.cuh"

namespace pp {
cudaError_t hlines_128(const LineArgs& a, int oy, cudaStream_t st) { return dispatch_hlines<128>(a, oy, st); }
void hlines_shape_128(int oy, int* lpc, int* threads) { hlines_shape<128>(oy, lpc, threads); }
}  // namespace pp
