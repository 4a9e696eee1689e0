// glynn_fwd.cu -- the forward kernel with column sums in shared memory, and the
// launches of all forward kernels.  The walk is in glynn_fwd.cuh; the register
// kernels are instantiated in files of their own (glynn_fwd_reg_*.cu), which
// compile side by side.
#include "glynn_fwd.cuh"

namespace pqi {

// Tasks [t_begin, t_end) of the list.  queue != 0: every warp pulls tasks from
// the global counter until the range is exhausted (persistent launch of a
// whole batch); queue == 0: warp w of block b takes task t_begin + b * wpb + w
// (one launch per permanent, the plain method).
__global__ void __launch_bounds__(256, 2) glynn_fwd_kernel(const __grid_constant__ ExecArgs a, int64_t t_begin,
                                                         int64_t t_end, int kmax, int ld,
                                                         int queue)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    WarpSmem sm(smem_raw + warp * warp_smem_bytes(kmax, ld), kmax, ld, true);
    Staged st;
    if (!queue) {
        const int64_t ti = t_begin + (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
        if (ti < t_end)
            run_task<0>(a, ti, sm, kmax, ld, st, lane);
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
        run_task<0>(a, ti, sm, kmax, ld, st, lane);
    }
}

// ---------------------------------------------------------------- host side
int fwd_smem_per_warp(int kmax, int ld) { return warp_smem_bytes(kmax, ld); }

int fwd_regs_per_thread()
{
    cudaFuncAttributes at{};
    return cudaFuncGetAttributes(&at, glynn_fwd_kernel) == cudaSuccess ? at.numRegs : 255;
}

// Raise (never lower) the kernel's dynamic shared-memory limit: plans made
// earlier with larger workspaces must keep launching.
cudaError_t fwd_prepare(int smem_bytes)
{
    cudaFuncAttributes at{};
    cudaError_t e = cudaFuncGetAttributes(&at, glynn_fwd_kernel);
    if (e != cudaSuccess)
        return e;
    if (at.maxDynamicSharedSizeBytes >= smem_bytes)
        return cudaSuccess;
    return cudaFuncSetAttribute(glynn_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                smem_bytes);
}

cudaError_t fwd_launch_persistent(int ld, const ExecArgs& a, int kmax, int blocks, int wpb,
                                  cudaStream_t st)
{
    const int smem = wpb * warp_smem_bytes(kmax, ld);
    glynn_fwd_kernel<<<blocks, 32 * wpb, smem, st>>>(a, 0, a.ntasks, kmax, ld, 1);
    return cudaGetLastError();
}

cudaError_t fwd_launch_plain(int ld, const ExecArgs& a, int64_t t_begin, int64_t t_end, int kmax,
                             int wpb, cudaStream_t st)
{
    const int smem = wpb * warp_smem_bytes(kmax, ld);
    const int64_t nt = t_end - t_begin;
    const unsigned grid = (unsigned)((nt + wpb - 1) / wpb);
    glynn_fwd_kernel<<<grid, 32 * wpb, smem, st>>>(a, t_begin, t_end, kmax, ld, 0);
    return cudaGetLastError();
}

// ---- column sums in registers
int fwd_reg_class_of(int l) { return l <= 4 ? 4 : l + (l & 1); }

int fwd_reg_smem_per_warp(int kmax, int ld) { return reg_warp_smem_bytes(kmax, ld); }

// The kernel of class nl (0: the one for several classes).
static const void* fwd_reg_kernel_for(int nl)
{
    if (nl == 0)
        return fwd_reg_kernel_mixed();
    const void* f = fwd_reg_kernel_a(nl);
    f = f ? f : fwd_reg_kernel_b(nl);
    f = f ? f : fwd_reg_kernel_c(nl);
    f = f ? f : fwd_reg_kernel_d(nl);
    return f ? f : fwd_reg_kernel_e(nl);
}

int fwd_reg_regs_per_thread(int nl)
{
    cudaFuncAttributes at{};
    const void* f = fwd_reg_kernel_for(nl);
    return (f && cudaFuncGetAttributes(&at, f) == cudaSuccess) ? at.numRegs : 255;
}

int fwd_reg_max_warps(int nl)
{
    cudaFuncAttributes at{};
    const void* f = fwd_reg_kernel_for(nl);
    return (f && cudaFuncGetAttributes(&at, f) == cudaSuccess) ? at.maxThreadsPerBlock / 32 : 4;
}

cudaError_t fwd_reg_prepare(int nl, int smem_bytes)
{
    const void* f = fwd_reg_kernel_for(nl);
    if (!f)
        return cudaErrorInvalidValue;
    cudaFuncAttributes at{};
    cudaError_t e = cudaFuncGetAttributes(&at, f);
    if (e != cudaSuccess)
        return e;
    if (at.maxDynamicSharedSizeBytes >= smem_bytes)
        return cudaSuccess;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
}

cudaError_t fwd_reg_launch(int nl, const ExecArgs& a, int64_t t_begin, int64_t t_end, int kmax,
                           int ld, unsigned grid, int wpb, int queue, cudaStream_t st)
{
    const void* f = fwd_reg_kernel_for(nl);
    if (!f)
        return cudaErrorInvalidValue;
    void* args[] = {(void*)&a, &t_begin, &t_end, &kmax, &ld, &queue};
    return cudaLaunchKernel(f, dim3(grid), dim3(32 * wpb), args,
                            (size_t)wpb * reg_warp_smem_bytes(kmax, ld), st);
}

}  // namespace pqi
