// Launches that may begin before the stream's previous kernel has ended.
//
// Most calls are chains of kernels of a few microseconds, so what passes
// between the end of one and the start of the next counts. A kernel launched
// here is scheduled once every block of the stream's previous kernel has
// started, and begins with dep_entry(), which lets its own successor be
// scheduled and then waits until the previous kernel has ended and its writes
// are visible: nothing is read or written before that, and a kernel ends only
// after its predecessor has, so the order of a stream's kernels is as before.
// Behind anything but a kernel that calls dep_entry() it is an ordinary launch.
// Force calls: 192 atoms (20 kernels) 133 -> 98 us, 80 atoms (8 kernels) 53 ->
// 46 us, 23,558 atoms (the NC model) 161 -> 142 us.
//
// Where it does not help:
//  - a persistent kernel, or one of many waves, lets its successor in only at
//    its end (early = false): waiting blocks would hold shared memory and with
//    it L1 for as long as it runs;
//  - the layer kernels that live on L1 (k_mp_fwd, k_mp_bwd, k_mp_fwd_tc) are
//    launched in the ordinary way once they are more than a wave: started
//    beside a contraction they keep its shared-memory carve-out (100,000 atoms:
//    10.4 ms against 9.9);
//  - while a graph is captured: its replays were slower with such edges (an
//    outer step of 192 atoms 226 us against 214).
#pragma once
#include <algorithm>
#include <utility>

#include "common.cuh"
#include "per_device.h"

namespace dmts {

__device__ __forceinline__ void dep_entry(bool early = true) {
    if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

inline int current_device() {
    int dev = 0;
    cudaGetDevice(&dev);
    return dev;
}

// SMs of the current device.
inline int sm_count() {
    static PerDevice sms;
    const int dev = current_device();
    return sms.get(dev, [dev] {
        int n = 1;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return std::max(n, 1);
    });
}

template <typename... P, typename... A>
inline void launch_dep_if(bool dep, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                          A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (dep) cudaStreamIsCapturing(st, &cap);
    cfg.attrs = at;
    cfg.numAttrs = dep && cap == cudaStreamCaptureStatusNone ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}
template <typename... P, typename... A>
inline void launch_dep(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
    launch_dep_if(true, kernel, grid, block, smem, st, std::forward<A>(args)...);
}

}  // namespace dmts
