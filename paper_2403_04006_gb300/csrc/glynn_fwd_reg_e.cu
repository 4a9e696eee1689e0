// glynn_fwd_reg_e.cu -- register-resident forward kernels of classes 30, 32.
#include "glynn_fwd.cuh"

namespace pqi {

const void* fwd_reg_kernel_e(int nl)
{
    switch (nl) {
    case 30: return (const void*)glynn_fwd_reg_kernel<30>;
    case 32: return (const void*)glynn_fwd_reg_kernel<32>;
    default: return nullptr;
    }
}

}  // namespace pqi
