// The forward GEMMs of a handful of tokens (thin.cuh) and their launcher.
#include <cuda_runtime.h>

#include <atomic>

#define COLA_DEFINE_THIN_KERNEL
#include "thin.cuh"

namespace cola {

namespace {

template <int KIND, int SIG>
cudaError_t launch_one(const ThinBatch& b, cudaStream_t stream)
{
    const int smem = thin_smem_bytes(b.stages, b.NT, b.S, b.TB, KIND == THIN_GLU);
    if (smem > GemmCfg<128, 1>::SMEM_LIMIT) return cudaErrorInvalidValue;
    auto kern = thin_kernel<KIND, SIG>;
    static std::atomic<unsigned long long> configured{0};   // bit d: attribute set on device d
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !((configured.load(std::memory_order_acquire) >> dev) & 1ull)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, GemmCfg<128, 1>::SMEM_LIMIT);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured.fetch_or(1ull << dev, std::memory_order_acq_rel);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(b.tiles * b.S));
    cfg.blockDim = dim3(THIN_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(b.S);
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, b);
}

}  // namespace

cudaError_t launch_thin(const ThinBatch& b, int kind, int sigma, cudaStream_t stream)
{
    if (b.S < 1 || b.S > THIN_MAX_CLUSTER || b.tiles < 1 || b.n < 1 || b.n > THIN_MAX_TOKENS || b.stages < 1 ||
        b.stages > THIN_MAX_STAGES)
        return cudaErrorInvalidValue;
    if (kind == THIN_STORE) return launch_one<THIN_STORE, SIG_IDENTITY>(b, stream);
    if (kind == THIN_GLU) return launch_one<THIN_GLU, SIG_IDENTITY>(b, stream);
    switch (sigma) {
    case SIG_SILU: return launch_one<THIN_ZH, SIG_SILU>(b, stream);
    case SIG_GELU: return launch_one<THIN_ZH, SIG_GELU>(b, stream);
    case SIG_IDENTITY: return launch_one<THIN_ZH, SIG_IDENTITY>(b, stream);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace cola
