// atm_fwd.cu -- launch of the forward-list kernel (atm_fwd.cuh).
#include <mutex>

#include "atm_fwd.cuh"

namespace atm3 {

using FwdKernel = void (*)(const FwdArgs);

// form: 0 as the traversals of pair scalars, 1 deterministic, 2 3c01
static FwdKernel fwd_kernel(int lj, int form)
{
    // (a deterministic evaluation keeps no LJ apart, 3c01 always)
    static const FwdKernel k[3][3] = {
        {k_atm_fwd<0, false, false>, k_atm_fwd<1, false, false>, k_atm_fwd<2, false, false>},
        {k_atm_fwd<0, true, false>, k_atm_fwd<1, true, false>, nullptr},
        {nullptr, nullptr, k_atm_fwd<2, false, true>}};
    return lj >= 0 && lj <= 2 ? k[form][lj] : nullptr;
}

// raises the kernel's dynamic shared-memory limit on the current device (a
// process-wide attribute: never lowered)
static cudaError_t fwd_attr(int lj, int form, size_t smem)
{
    static std::mutex mu;
    static size_t done[ATM_MAX_DEVICES][3][3] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= ATM_MAX_DEVICES) return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lock(mu);
    if (smem <= done[dev][form][lj]) return cudaSuccess;
    e = cudaFuncSetAttribute(fwd_kernel(lj, form), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) done[dev][form][lj] = smem;
    return e;
}

cudaError_t launch_atm_fwd(const FwdArgs& a, int det, int nwarps, cudaStream_t s)
{
    if (a.b.ncell == 0) return cudaSuccess;
    const int form = a.trav == 0 ? 2 : (det ? 1 : 0);
    const size_t smem = fwd_smem_plan(a.mcap, a.run, nwarps).total;
    const FwdKernel k = fwd_kernel(a.lj, form);
    if (!k) return cudaErrorInvalidValue;
    cudaError_t e = fwd_attr(a.lj, form, smem);
    if (e != cudaSuccess) return e;
    launch_after(k, (a.run > 1 ? a.nruns : a.b.ncell) * a.split, 32 * nwarps, smem, s, a);
    return cudaGetLastError();
}

}  // namespace atm3
