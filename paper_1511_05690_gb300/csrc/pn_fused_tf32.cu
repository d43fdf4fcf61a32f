// TF32 / 3xTF32 operand instantiations of the one-launch small product.
#include "pn_fused_kernel.cuh"

namespace pn {

int fused_launch_tf32(const Common& cm, const FusedArgs& fa, void* stream) {
  if (cm.mode == MODE_TF32)
    return cm.BN == 64 ? gemm::launch_fused_t<MODE_TF32, 64>(cm, fa, stream)
                       : gemm::launch_fused_t<MODE_TF32, 128>(cm, fa, stream);
  return cm.BN == 64 ? gemm::launch_fused_t<MODE_3XTF32, 64>(cm, fa, stream)
                     : gemm::launch_fused_t<MODE_3XTF32, 128>(cm, fa, stream);
}

}  // namespace pn
