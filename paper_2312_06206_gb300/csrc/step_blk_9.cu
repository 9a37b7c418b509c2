// step_blk_9.cu -- explicit instantiation of the block-FFT step kernels (FFT length 2^9).
#include "step_blk.cuh"

namespace sadi {
namespace blk {
template cudaError_t launch_blk_impl<9>(const RegBatch&, int, cudaStream_t, cudaEvent_t*, bool);
}  // namespace blk
}  // namespace sadi
