// The cluster-reduced split-K GEMMs (splitk_cluster.cuh): their launcher.
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

#define COLA_DEFINE_CLUSTER_KERNEL
#include "splitk_cluster.cuh"

namespace cola {

namespace {

template <bool A_MN, bool B_MN, int OP, int SIG>
cudaError_t launch_one(const CredBatch& b, bool pdl, cudaStream_t stream)
{
    if (b.S < (OP == CRED_DZ ? 2 : 1) || b.S > MAX_CLUSTER || b.tiles < 1) return cudaErrorInvalidValue;
    constexpr int smem = CredCfg::SMEM_BYTES;
    auto kern = splitk_cluster_kernel<A_MN, B_MN, OP, SIG>;
    static std::atomic<unsigned long long> configured{0};   // bit d: attribute set on device d
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !((configured.load(std::memory_order_acquire) >> dev) & 1ull)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured.fetch_or(1ull << dev, std::memory_order_acq_rel);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(b.tiles * b.S));
    cfg.blockDim = dim3(CRED_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(b.S);
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, b);
}

}  // namespace

// Clusters of S CTAs that the current device runs at once, asked once per device.
const int* reduce_cluster_capacity(int sms)
{
    struct Caps {
        std::once_flag once;
        int n[MAX_CLUSTER + 1];
    };
    static Caps caps[65];   // [64]: no device, or one beyond the table
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 64;
    Caps& c = caps[dev];
    std::call_once(c.once, [&] {
        const auto kern = splitk_cluster_kernel<true, true, CRED_STORE, SIG_IDENTITY>;
        const bool set = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CredCfg::SMEM_BYTES) == cudaSuccess;
        for (int s = 0; s <= MAX_CLUSTER; ++s) {
            c.n[s] = s > 0 && sms >= s ? sms / s : 1;
            if (s < 2 || !set) continue;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(static_cast<unsigned>(s));
            cfg.blockDim = dim3(CRED_THREADS);
            cfg.dynamicSmemBytes = CredCfg::SMEM_BYTES;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = static_cast<unsigned>(s);
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) c.n[s] = n;
        }
    });
    return c.n;
}

cudaError_t launch_splitk_cluster(const CredBatch& b, int op, int sigma, bool pdl, cudaStream_t stream)
{
    if (op == CRED_STORE) return launch_one<true, true, CRED_STORE, SIG_IDENTITY>(b, pdl, stream);
    if (op == CRED_ACC) return launch_one<true, true, CRED_ACC, SIG_IDENTITY>(b, pdl, stream);
    const bool zh = op == CRED_ZH;
    if (!zh && op != CRED_DZ) return cudaErrorInvalidValue;
    switch (sigma) {
    case SIG_SILU:
        return zh ? launch_one<false, false, CRED_ZH, SIG_SILU>(b, pdl, stream)
                  : launch_one<false, true, CRED_DZ, SIG_SILU>(b, pdl, stream);
    case SIG_GELU:
        return zh ? launch_one<false, false, CRED_ZH, SIG_GELU>(b, pdl, stream)
                  : launch_one<false, true, CRED_DZ, SIG_GELU>(b, pdl, stream);
    case SIG_IDENTITY:
        return zh ? launch_one<false, false, CRED_ZH, SIG_IDENTITY>(b, pdl, stream)
                  : launch_one<false, true, CRED_DZ, SIG_IDENTITY>(b, pdl, stream);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace cola
