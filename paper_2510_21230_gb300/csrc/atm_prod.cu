// atm_prod.cu -- launch of the product-rule kernels (atm_prod.cuh).
#include <mutex>

#include "atm_prod.cuh"

namespace atm3 {

template <typename R>
static void (*prod_kernel(int trav))(const AtmArgs<R>)
{
    switch (trav) {
    case 0: return k_atm_prod<0, R>;
    case 1: return k_atm_prod<1, R>;
    case 2: return k_atm_prod<2, R>;
    case 4: return k_atm_prod<4, R>;
    }
    return nullptr;
}

// raises the kernel's dynamic shared-memory limit on the current device (a
// process-wide attribute: never lowered)
template <typename R>
static cudaError_t prod_attr(int trav, size_t smem)
{
    static std::mutex mu;
    static size_t done[ATM_MAX_DEVICES][ATM_NTRAV] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= ATM_MAX_DEVICES) return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lock(mu);
    if (smem <= done[dev][trav]) return cudaSuccess;
    e = cudaFuncSetAttribute(prod_kernel<R>(trav), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) done[dev][trav] = smem;
    return e;
}

template <typename R>
cudaError_t launch_atm_prod(int trav, const AtmArgs<R>& a, int nwarps, cudaStream_t s)
{
    if (a.b.ncell == 0) return cudaSuccess;
    if (!prod_kernel<R>(trav)) return cudaErrorInvalidValue;
    cudaError_t e = prod_attr<R>(trav, (size_t)a.gcap);
    if (e != cudaSuccess) return e;
    launch_after(prod_kernel<R>(trav), a.b.ncell, 32 * nwarps, (size_t)a.gcap, s, a);
    return cudaGetLastError();
}

template cudaError_t launch_atm_prod<float>(int, const AtmArgs<float>&, int, cudaStream_t);
template cudaError_t launch_atm_prod<double>(int, const AtmArgs<double>&, int, cudaStream_t);

}  // namespace atm3
