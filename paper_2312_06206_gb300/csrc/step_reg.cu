// step_reg.cu -- dispatch of the register-FFT step paths by FFT length.
#include "../../include/sadi.h"
#include "sadi_internal.h"

namespace sadi {
namespace regk {
template <int LOGL>
cudaError_t launch_reg_impl(const RegBatch& b, int max_n, cudaStream_t st, cudaEvent_t* ev, bool dense);
}  // namespace regk
namespace blk {
template <int LOGL>
cudaError_t launch_blk_impl(const RegBatch& b, int max_n, cudaStream_t st, cudaEvent_t* ev, bool dense);
}  // namespace blk

// both FP32 forms at every FFT length
bool reg_path_supported(int logNp, int prec) {
  return (prec == SADI_PREC_FP32 || prec == SADI_PREC_FP32_DENSE) && logNp >= 3 && logNp <= 13;
}

// block: on step_blk.cuh (blk_path), else step_reg.cuh
cudaError_t launch_step_reg(const RegBatch& b, int logNp, bool block, int max_n, cudaStream_t st, cudaEvent_t* ev,
                            bool dense) {
  if (b.count < 1 || b.count > kMaxBatch) return cudaErrorInvalidValue;
  switch (block ? 16 + logNp : logNp) {
    case 3: return regk::launch_reg_impl<3>(b, max_n, st, ev, dense);
    case 4: return regk::launch_reg_impl<4>(b, max_n, st, ev, dense);
    case 5: return regk::launch_reg_impl<5>(b, max_n, st, ev, dense);
    case 6: return regk::launch_reg_impl<6>(b, max_n, st, ev, dense);
    case 7: return regk::launch_reg_impl<7>(b, max_n, st, ev, dense);
    case 10: return regk::launch_reg_impl<10>(b, max_n, st, ev, dense);
    case 16 + 8: return blk::launch_blk_impl<8>(b, max_n, st, ev, dense);
    case 16 + 9: return blk::launch_blk_impl<9>(b, max_n, st, ev, dense);
    case 16 + 10: return blk::launch_blk_impl<10>(b, max_n, st, ev, dense);
    case 16 + 11: return blk::launch_blk_impl<11>(b, max_n, st, ev, dense);
    case 16 + 12: return blk::launch_blk_impl<12>(b, max_n, st, ev, dense);
    case 16 + 13: return blk::launch_blk_impl<13>(b, max_n, st, ev, dense);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sadi
