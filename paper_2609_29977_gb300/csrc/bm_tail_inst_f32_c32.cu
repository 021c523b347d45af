// Explicit instantiations of the FP32 tail kernels (nb = 32).
#include "bm_tail_rows.cuh"

namespace bm {
template void rows::launch_tail_rows<float, 32>(const TailView<float> &, cudaStream_t);
template cudaError_t rows::prepare_rows<float, 32>();
}  // namespace bm
