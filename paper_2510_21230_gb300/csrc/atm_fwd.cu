// atm_fwd.cu -- launch of the forward-list kernel (atm_fwd.cuh).
#include <mutex>

#include "atm_fwd.cuh"

namespace atm3 {

using FwdKernel = void (*)(const FwdArgs);

static FwdKernel fwd_kernel(int lj, int det)
{
    // (a deterministic evaluation keeps no LJ apart)
    static const FwdKernel k[2][3] = {{k_atm_fwd<0, false>, k_atm_fwd<1, false>, k_atm_fwd<2, false>},
                                      {k_atm_fwd<0, true>, k_atm_fwd<1, true>, nullptr}};
    return lj >= 0 && lj <= 2 ? k[det ? 1 : 0][lj] : nullptr;
}

// raises the kernel's dynamic shared-memory limit on the current device (a
// process-wide attribute: never lowered)
static cudaError_t fwd_attr(int lj, int det, size_t smem)
{
    static std::mutex mu;
    static size_t done[ATM_MAX_DEVICES][2][3] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= ATM_MAX_DEVICES) return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lock(mu);
    if (smem <= done[dev][det][lj]) return cudaSuccess;
    e = cudaFuncSetAttribute(fwd_kernel(lj, det), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) done[dev][det][lj] = smem;
    return e;
}

cudaError_t launch_atm_fwd(const FwdArgs& a, int det, int nwarps, cudaStream_t s)
{
    if (a.b.ncell == 0) return cudaSuccess;
    det = det ? 1 : 0;
    const size_t smem = fwd_smem_plan(a.mcap, a.run, nwarps).total;
    const FwdKernel k = fwd_kernel(a.lj, det);
    if (!k) return cudaErrorInvalidValue;
    cudaError_t e = fwd_attr(a.lj, det, smem);
    if (e != cudaSuccess) return e;
    launch_after(k, (a.run > 1 ? a.nruns : a.b.ncell) * a.split, 32 * nwarps, smem, s, a);
    return cudaGetLastError();
}

}  // namespace atm3
