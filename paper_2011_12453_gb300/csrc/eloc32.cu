// FP32 kernels of the incremental local energy on warp tiles (eloc_impl.cuh): tanh, and ReLU +
// layer norm (the paper's f).
#include "eloc_impl.cuh"

namespace gna {

const void* el_kernel_f32(int np, int F, int mode) {
  if (mode == EL_F32_LN) return np == 2 ? el_kernel_np<2, EL_F32_LN>(F) : el_kernel_np<0, EL_F32_LN>(F);
  return np == 2 ? el_kernel_np<2, EL_F32>(F) : el_kernel_np<0, EL_F32>(F);
}

}  // namespace gna
