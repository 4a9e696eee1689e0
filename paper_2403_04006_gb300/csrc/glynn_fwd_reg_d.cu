// glynn_fwd_reg_d.cu -- register-resident forward kernels of classes 24, 26, 28.
#include "glynn_fwd.cuh"

namespace pqi {

const void* fwd_reg_kernel_d(int nl)
{
    switch (nl) {
    case 24: return (const void*)glynn_fwd_reg_kernel<24>;
    case 26: return (const void*)glynn_fwd_reg_kernel<26>;
    case 28: return (const void*)glynn_fwd_reg_kernel<28>;
    default: return nullptr;
    }
}

}  // namespace pqi
