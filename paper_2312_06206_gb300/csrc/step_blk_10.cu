// step_blk_10.cu -- explicit instantiation of the block-FFT step kernels (FFT length 2^10).
#include "step_blk.cuh"

namespace sadi {
namespace blk {
template cudaError_t launch_blk_conv<10>(const RegBatch&, cudaStream_t);
template cudaError_t launch_blk_impl<10>(const RegBatch&, int, cudaStream_t, cudaEvent_t*, bool);
}  // namespace blk
}  // namespace sadi
