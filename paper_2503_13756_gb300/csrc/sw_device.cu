// sw_device.cu -- what the launch rules (sw_forms.h) ask of a device.
#include <map>
#include <mutex>

#include "sw_forms.h"
#include "sw_internal.cuh"

namespace swk {
namespace {

// Never launched: stands for a kernel whose CTAs its shared memory limits.
__global__ void __launch_bounds__(256) k_resident(int *p)
{
    extern __shared__ int s[];
    p[threadIdx.x] = s[threadIdx.x];
}

// Clusters of w CTAs of `smem` bytes that the current device holds at once.
int resident_clusters(int w, int smem)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)w);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = (size_t)smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)w;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(k_resident, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k_resident, &cfg) != cudaSuccess) {
        cudaGetLastError();  // no clusters of this width
        return 0;
    }
    return n;
}

}  // namespace

cudaError_t device_form(const DeviceForm **out)
{
    static std::mutex mu;
    static std::map<int, DeviceForm> forms;  // an entry per device, never moved
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> g(mu);
    auto it = forms.find(dev);
    if (it == forms.end()) {
        DeviceForm f{};
        e = cudaDeviceGetAttribute(&f.sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        for (int w = 1; w <= 8; ++w) {
            f.clusters[0][w] = resident_clusters(w, 200 * 1024);
            f.clusters[1][w] = resident_clusters(w, 100 * 1024);
        }
        it = forms.emplace(dev, f).first;
    }
    *out = &it->second;
    return cudaSuccess;
}

}  // namespace swk
