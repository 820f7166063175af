// rt_trace_closest_noalloc: closest-hit tracing that never allocates device
// memory.
//
// Some callers cannot let a library allocate device memory: a serving runtime
// that owns every byte of it through its own pool and budgets it per tenant,
// or a latency-critical loop where an allocation (which may synchronise the
// whole device) would stall other streams.  A trace needs no device memory of
// its own; this entry point promises it, for batches of up to
// RT_NOALLOC_MAX_RAYS rays.
#include <cuda_runtime.h>

#include "rt_internal.cuh"

extern "C" int rt_trace_closest_noalloc(rt_scene scene, const rt_ray* rays_dev, int64_t n, rt_hit* hits_dev,
                                        const rt_trace_params* params, void* stream) {
  return rt::abi_guard([&]() -> int {
    if (!scene) return rt::set_error(RT_EINVAL, "scene is NULL");
    if (n < 0) return rt::set_error(RT_EINVAL, "n out of range");
    if (n > RT_NOALLOC_MAX_RAYS)
      return rt::set_error(RT_EINVAL,
                           "rt_trace_closest_noalloc: n exceeds RT_NOALLOC_MAX_RAYS (262144); split the batch");
    if (n > 0 && (!rays_dev || !hits_dev)) return rt::set_error(RT_EINVAL, "NULL buffer");
    if (((uintptr_t)rays_dev & 15) || ((uintptr_t)hits_dev & 15))
      return rt::set_error(RT_EINVAL, "rays/hits must be 16-byte aligned");
    if (params && params->block != 0 && params->block != 64 && params->block != 128 && params->block != 256)
      return rt::set_error(RT_EINVAL, "block must be 0, 64, 128 or 256");
    if (params && ((params->stack != 0 && params->stack != 16 && params->stack != 32 && params->stack != 64)))
      return rt::set_error(RT_EINVAL, "stack must be 0, 16, 32 or 64");
    if (params && (params->flags & RT_QUANTIZED_NODES) && !scene->q_built)
      return rt::set_error(RT_EINVAL, "RT_QUANTIZED_NODES needs a build with quantize = 1");
    if (!scene->built) return rt::set_error(RT_ENOTBUILT, "BVH not built");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return rt::set_error(RT_ECUDA, "cudaGetDevice failed");
    // the kernel runs on the current device against the scene's tree: the scene must live here
    if (dev != scene->device)
      return rt::set_error(RT_EINVAL, "the scene was uploaded on another device; make that device current");
    cudaError_t e = rt::launch_trace(scene, rays_dev, n, hits_dev, nullptr, params, (cudaStream_t)stream);
    if (e != cudaSuccess) return rt::set_error(RT_ECUDA, cudaGetErrorString(e));
    return RT_OK;
  });
}
