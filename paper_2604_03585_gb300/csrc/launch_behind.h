// Launching a kernel programmatically behind the last one on its stream.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sar {

// Up to this many threads in all, the time from one kernel's end to the next
// one's first instruction counts: it is then launched while its predecessor still
// runs and waits for it in the kernel (sar_common.cuh: grid_wait_predecessor).
// Every kernel launched here waits before it touches the caller's data or anything
// that a kernel of the library writes.  Before it, the kernels for few short lines
// read the plan's twiddles and filter: whoever hands tables to a launch has
// waited on the host until they were complete.
// The limit is in threads: two waves of the GB300's 152 SMs of kernels that fill
// them, and up to eight of the three-pass engines, which hold 512 threads per SM.
// It saves two to five us a scene: 1024 x 1024 18.6 -> 15.3, 2048 x 4096 84.5 ->
// 80.0, 4096 x 4096 158.0 -> 153.3.  Larger passes would save as much, below 2 %
// of theirs (8192 x 4096: 320 -> 316), and are launched ordinarily: blocks that
// wait hold slots that another stream's kernels could use.  (On four streams and in
// serving neither side of the limit showed a difference: 8.4 us a scene of 1024
// x 1024 either way, 8.9 without.)
constexpr int64_t kBehindThreads = 2 * 152 * 2048;
// Clusters are not where they take part of the GPU's slots: placed while the
// predecessor's last blocks still hold some, they crowd on the others (256
// lines of 4096, folded: 12.1 us against 10.3; 64 lines 7.5 against 7.6, 608
// lines 17.9 against 18.4).
inline bool launched_behind(int64_t blocks, int threads, int cluster) {
    if (blocks * threads > kBehindThreads) return false;
    return cluster == 1 || blocks <= 152 || blocks * threads >= 152 * 512;
}

// cluster: blocks per thread-block cluster (1: none).
template <class... Params, class... Args>
cudaError_t launch_behind(void (*kernel)(Params...), int64_t blocks, int threads, int smem, int cluster,
                          cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks, 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    if (launched_behind(blocks, threads, cluster)) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned)n;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace sar
