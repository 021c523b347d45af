// Explicit instantiations of the FP32 tail kernels (nb in [48]).
#include "bm_tail_wide.cuh"

namespace bm {
template void rows::launch_tail_w<48>(const TailView<float> &, cudaStream_t);
template cudaError_t rows::prepare_w<48>();
}  // namespace bm
