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

// GS form up to N' = 1024, dense form up to 2048.  Above, the block-wide FFT
// was faster (N = 4095 GS step 0.91 ms against 1.56) but less exact: after 1000
// steps the GS form was 1.06e-6 from FP64 at N = 2047 against 4.7e-7 on the
// shared-memory engine, 5.9e-7 against 3.1e-7 at N = 4095; the dense form 3.4e-7
// against 1.9e-7 at N = 4095.  At the lengths kept it is the more exact one (N =
// 1023 GS 9.9e-7 against 1.4e-6, N = 2047 dense 3.1e-7 against 4.8e-7).
bool reg_path_supported(int logNp, int prec) {
  if (prec == SADI_PREC_FP32) return logNp >= 3 && logNp <= 10;
  return prec == SADI_PREC_FP32_DENSE && logNp >= 3 && logNp <= 11;
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
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sadi
