// glynn_fwd_reg_b.cu -- register-resident forward kernels of classes 12, 14, 16.
#include "glynn_fwd.cuh"

namespace pqi {

const void* fwd_reg_kernel_b(int nl)
{
    switch (nl) {
    case 12: return (const void*)glynn_fwd_reg_kernel<12>;
    case 14: return (const void*)glynn_fwd_reg_kernel<14>;
    case 16: return (const void*)glynn_fwd_reg_kernel<16>;
    default: return nullptr;
    }
}

}  // namespace pqi
