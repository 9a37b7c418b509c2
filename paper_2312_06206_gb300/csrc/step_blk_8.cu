// step_blk_8.cu -- explicit instantiation of the block-FFT step kernels (FFT length 2^8).
#include "step_blk.cuh"

namespace sadi {
namespace blk {
template cudaError_t launch_blk_impl<8>(const RegBatch&, int, cudaStream_t, cudaEvent_t*, bool);
}  // namespace blk
}  // namespace sadi
