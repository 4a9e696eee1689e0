// glynn_fwd_reg_a.cu -- register-resident forward kernels of classes 4, 6, 8, 10.
#include "glynn_fwd.cuh"

namespace pqi {

const void* fwd_reg_kernel_a(int nl)
{
    switch (nl) {
    case 4: return (const void*)glynn_fwd_reg_kernel<4>;
    case 6: return (const void*)glynn_fwd_reg_kernel<6>;
    case 8: return (const void*)glynn_fwd_reg_kernel<8>;
    case 10: return (const void*)glynn_fwd_reg_kernel<10>;
    default: return nullptr;
    }
}

}  // namespace pqi
