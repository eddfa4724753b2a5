// Host-side helpers of the TMA kernels: the driver's tensor-map encoder, looked up once.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

namespace nova {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled through the runtime's driver entry-point query (the library does not
// link libcuda).  The function-local static is initialised exactly once, also when several host
// threads make their first call at the same time; null if the driver lacks the entry point.
inline EncodeTiledFn tensor_map_encoder() {
  static const EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return (EncodeTiledFn)p;
    return (EncodeTiledFn) nullptr;
  }();
  return fn;
}

// Opt a kernel in to BYTES of dynamic shared memory, the most that any of its launches takes.  The attribute
// belongs to the (function, device) pair, so it is set on every launch path rather than remembered per process:
// the call is a few hundred nanoseconds of host time.  It is the same number every time, hence a template argument:
// another thread that launches the same kernel with less must not lower the limit between this call and its launch.
template <int BYTES, typename Kernel>
inline cudaError_t allow_dynamic_smem(Kernel kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BYTES);
}

// Launch a kernel that may be scheduled while the preceding kernel of the stream is still
// draining (programmatic dependent launch): its CTAs run their set-up - barrier initialisation,
// TMEM allocation, constant tables - early and call sm100::pdl_wait() before they touch anything
// the preceding kernels wrote or still read.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_overlapped(void (*kernel)(KArgs...), int grid, int threads, size_t smem, cudaStream_t s,
                                     Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace nova
