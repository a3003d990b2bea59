// Launches of the quantize kernels and what becomes of a refused one.  Host code alone.
#pragma once
#include "../../include/abs_b200.h"

#include <cuda_runtime.h>

namespace {

// Launch with programmatic stream serialization: the kernel may be scheduled while the previous
// kernel of the stream drains; every kernel here calls pdl_wait() before its first global access.
// together: the blocks wait for one another, so all of them have to be resident: as a cluster (one_cluster_alpha; the grid is at most kMaxCluster blocks) or by a
// cooperative launch (one_pass_alpha).  A single block needs neither; the latter costs half a microsecond more on the host (2.45 us instead of
// 1.93) and lets nothing overlap: such kernels start 4.1 us apart on a stream.
enum Together { kApart, kCooperative, kCluster };
// A grid whose blocks do not all fit what the stream may use (a green context, an MPS share: fewer SMs than the device has) is refused with
// cudaErrorCooperativeLaunchTooLarge, cooperative or cluster.  The runtime has that code for the former.  For a cluster, out of resources means no room (the
// kernels need no more than any block may have); after any other failure the runtime is asked whether there is room for one, and where there is, the
// launch failed for a reason that two kernels would only hide.
template <typename... KArgs, typename... Args>
cudaError_t launch_any(Together together, void (*kernel)(KArgs...), int grid, int block, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    if (together == kCluster) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)grid;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    } else {
        attr[1].id = cudaLaunchAttributeCooperative;
        attr[1].val.cooperative = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = together != kApart && grid > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    if (e == cudaSuccess || together != kCluster) return e;
    int clusters = -1;
    const bool no_room = e == cudaErrorLaunchOutOfResources || (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters == 0);
    return no_room ? cudaErrorCooperativeLaunchTooLarge : e;
}
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), int grid, int block, cudaStream_t s, Args... args) {
    return launch_any(kApart, kernel, grid, block, s, args...);
}

// Internal status: such a grid was refused.  Nothing was enqueued; the call takes the two kernels.
constexpr abs_status_t kNotResident = (abs_status_t)-1;

// Optional CUDA events recorded around the group-quantize kernel (abs_profile_events).
cudaEvent_t g_ev_quant_begin = nullptr, g_ev_quant_end = nullptr;

// Status of the launch of a quantize kernel on s; also ends the interval of abs_profile_events.
abs_status_t quantize_launched(cudaError_t e, cudaStream_t s, bool profile = true) {
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();                  // the refusal is answered here: it is not left for the caller's own error checks
        return kNotResident;
    }
    if (e != cudaSuccess) return ABS_ERR_CUDA;
    if (profile && g_ev_quant_end) cudaEventRecord(g_ev_quant_end, s);
    return cudaGetLastError() == cudaSuccess ? ABS_OK : ABS_ERR_CUDA;
}

}  // namespace
