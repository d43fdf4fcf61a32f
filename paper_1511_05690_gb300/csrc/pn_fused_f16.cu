// BF16 / FP16 operand instantiations of the one-launch small product.
#include "pn_fused_kernel.cuh"

namespace pn {

int fused_launch_f16(const Common& cm, const FusedArgs& fa, void* stream) {
  if (cm.mode == MODE_BF16)
    return cm.BN == 64 ? gemm::launch_fused_t<MODE_BF16, 64>(cm, fa, stream)
                       : gemm::launch_fused_t<MODE_BF16, 128>(cm, fa, stream);
  return cm.BN == 64 ? gemm::launch_fused_t<MODE_F16, 64>(cm, fa, stream)
                     : gemm::launch_fused_t<MODE_F16, 128>(cm, fa, stream);
}

}  // namespace pn
