// Explicit instantiations of the tail factorization kernels (float, nb in [48]).
#include "bm_tail_factor.cuh"
#include "bm_tail_wide.cuh"

namespace bm {
namespace tail {
template void launch_tail_nb<float, 48>(const TailView<float> &, cudaStream_t, const TailSched *, cudaEvent_t *);
template cudaError_t prepare_nb<float, 48>();
}  // namespace tail
template void rows::launch_tail_w<48>(const TailView<float> &, cudaStream_t);
template cudaError_t rows::prepare_w<48>();
}  // namespace bm
