// glynn_fwd_reg_c.cu -- register-resident forward kernels of classes 18, 20, 22.
#include "glynn_fwd.cuh"

namespace pqi {

const void* fwd_reg_kernel_c(int nl)
{
    switch (nl) {
    case 18: return (const void*)glynn_fwd_reg_kernel<18>;
    case 20: return (const void*)glynn_fwd_reg_kernel<20>;
    case 22: return (const void*)glynn_fwd_reg_kernel<22>;
    default: return nullptr;
    }
}

}  // namespace pqi
