// E4M3 operand instantiations of the one-launch small product, and the
// dispatch by format.
#include "pn_fused_kernel.cuh"

namespace pn {

int fused_launch_f16(const Common& cm, const FusedArgs& fa, void* stream);
int fused_launch_tf32(const Common& cm, const FusedArgs& fa, void* stream);

int launch_fused(const Common& cm, const FusedArgs& fa, void* stream) {
  if (cm.total_tiles < 1) return 0;
  switch (cm.mode) {
    case MODE_BF16:
    case MODE_F16: return fused_launch_f16(cm, fa, stream);
    case MODE_TF32:
    case MODE_3XTF32: return fused_launch_tf32(cm, fa, stream);
    case MODE_E4M3:
      return cm.BN == 64 ? gemm::launch_fused_t<MODE_E4M3, 64>(cm, fa, stream)
                         : gemm::launch_fused_t<MODE_E4M3, 128>(cm, fa, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pn
