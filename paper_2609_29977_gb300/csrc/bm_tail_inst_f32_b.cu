// Explicit instantiations of the FP32 tail kernels (nb in [12, 16]).
#include "bm_tail_rows.cuh"

namespace bm {
template void rows::launch_tail_rows<float, 12>(const TailView<float> &, cudaStream_t);
template cudaError_t rows::prepare_rows<float, 12>();
template void rows::launch_tail_rows<float, 16>(const TailView<float> &, cudaStream_t);
template cudaError_t rows::prepare_rows<float, 16>();
}  // namespace bm
