// Launches with programmatic stream serialisation: the next kernel of a stream becomes resident while the one before it
// still runs and waits for it on the device.  Every kernel calls tad_wait_previous() before it touches global memory and
// only then lets its own successor start, so at most two kernels of a stream are resident and no kernel reads or
// writes anything before its predecessor has finished.  Steps of a dozen short kernels are bound by the gaps between
// them: see the figures at each change of the launch count.
#pragma once
#include <cuda_runtime.h>

#include <utility>

#ifdef __CUDACC__
__device__ __forceinline__ void tad_wait_previous()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif

// set while a kernel is launched beside a pass on the plan's second stream (runtime.cu): an early start would take the SMs
// before the pass that was issued first (8192-row gradient of the intro expression 149 instead of 130 us)
extern thread_local bool tad_launch_plain;

template <typename... Params, typename... Args>
inline cudaError_t tad_launch_cluster(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, int cluster, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute attr[2] = {};
    cfg.attrs = attr;
    // (a stream that is being captured gets plain edges: its graph may join this kernel with other streams)
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (!tad_launch_plain && cudaStreamIsCapturing(stream, &capturing) == cudaSuccess && capturing == cudaStreamCaptureStatusNone) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = (unsigned)cluster;
        attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

template <typename... Params, typename... Args>
inline cudaError_t tad_launch(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args &&...args)
{
    return tad_launch_cluster(kernel, grid, block, smem, stream, 1, std::forward<Args>(args)...);
}
