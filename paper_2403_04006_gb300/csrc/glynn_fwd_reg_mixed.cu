// glynn_fwd_reg_mixed.cu -- register-resident forward kernel for batches of
// several column classes.
#include "glynn_fwd.cuh"

namespace pqi {

// All column classes in one persistent launch: each task runs the
// instantiation of its own class.
__global__ void __launch_bounds__(256, 2) glynn_fwd_reg_mixed_kernel(const __grid_constant__ ExecArgs a,
                                                                     int64_t t_begin,
                                                                     int64_t t_end, int kmax,
                                                                     int ld, int queue)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* raw = smem_raw + warp * reg_warp_smem_bytes(kmax, ld);
    Staged st;
    auto run = [&](int64_t ti) {
        const Task t = a.tasks[ti];
        const int32_t bad =
            task_guard(t, a.desc, a.nperm, a.nmeta, a.nslots, kmax, ld, kMaxLowDigits,
                       a.ngroups);
        if (bad) {
            if (lane == 0)
                record_error(a.err, bad, ti);
            return;
        }
        const int l = a.desc[t.perm].l;
        const int nl = l <= 4 ? 4 : l + (l & 1);
        if (nl > ld) {  // the class's rows do not fit the launch's layout
            if (lane == 0)
                record_error(a.err, kErrDescLayout, ti);
            return;
        }
        switch (nl) {
#define PQ_REG_CASE(N)                                   \
    case N: {                                            \
        WarpSmem sm(raw, kmax, N, false);                \
        process_task<N>(a, t, sm, st, lane);             \
        break;                                           \
    }
            PQ_REG_CASE(4)
            PQ_REG_CASE(6)
            PQ_REG_CASE(8)
            PQ_REG_CASE(10)
            PQ_REG_CASE(12)
            PQ_REG_CASE(14)
            PQ_REG_CASE(16)
            PQ_REG_CASE(18)
            PQ_REG_CASE(20)
#undef PQ_REG_CASE
        default:
            break;
        }
    };
    if (!queue) {
        const int64_t ti = t_begin + (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
        if (ti < t_end)
            run(ti);
        return;
    }
    for (;;) {
        int q = 0;
        if (lane == 0)
            q = atomicAdd(a.counters, 1);
        q = __shfl_sync(0xffffffffu, q, 0);
        const int64_t ti = t_begin + q;
        if (ti >= t_end)
            break;
        run(ti);
    }
}

const void* fwd_reg_kernel_mixed() { return (const void*)glynn_fwd_reg_mixed_kernel; }

}  // namespace pqi
