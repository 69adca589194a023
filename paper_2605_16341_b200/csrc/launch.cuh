// Kernel launches of the step.  Within a call the kernels of one stream form a chain; with
// programmatic dependent launch the next kernel's CTAs are set up (barriers, tensor memory, tensor-map
// fetches) while the current one still runs, and wait for its end and its memory before they touch
// global memory.  Every kernel of the library therefore starts with grid_dependency_wait() in front of its first global access, and
// lets its successor in right away.  One exception: the products with B prefetch M and G to L2 before they wait.  That is safe whatever
// is still at work, and only because it is a prefetch: L2 is where all kernels of the device meet, and no value gets into a register or
// shared memory before the wait.  A load in its place would need all writers of M and G to be done, which nothing promises: the packing kernel
// in front of a step's first product does wait before it lets that in (so that the prefetch finds what will be read), but the
// phases of a column-sharded step begin with other kernels too.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "profile.cuh"

namespace od {

__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// both at once, for kernels without a prologue of their own
__device__ __forceinline__ void grid_dependency() { grid_dependency_launch(); grid_dependency_wait(); }

// First error met while preparing launches of the current step call (0 = none, 1 and 2: tensor maps); one per host
// thread, so that concurrent step calls do not see each other's.
constexpr int LAUNCH_FAILED = 3;       // the runtime's last error says why
inline int& engine_error() { static thread_local int e = 0; return e; }

// Whether the launches of the current call overlap as described above (one flag per host thread).
inline bool& overlap_launches() { static thread_local bool on = false; return on; }

template <class... KArgs, class... Args>
inline void launch(void (*kernel)(KArgs...), dim3 grid, int block, size_t smem, int cluster, int stage, cudaStream_t st,
                   const Args&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)cluster; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (overlap_launches()) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned)n;
    prof::Scope scope(stage, st);
    if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess && !engine_error()) engine_error() = LAUNCH_FAILED;
}

// f(table) with the smaller table where it holds the matrices; table_t<decltype(table)>: its type.
template <class T>
using table_t = std::decay_t<T>;
template <class F>
inline void with_table(const Batch& b, F f) {
    if (b.count > MAXB_SMALL) { f(b); return; }
    SmallBatch s;
    s.count = b.count; s.pad = 0; s.scratch_stride = b.scratch_stride;
    std::copy(b.w, b.w + b.count, s.w);
    f(s);
}

}  // namespace od
