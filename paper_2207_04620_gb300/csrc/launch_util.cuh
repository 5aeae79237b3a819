// Launch helpers shared by the kernel files: grid sizing for the elementwise
// kernels, the per-class CUDA-event profiler hook and the launch check.
#pragma once
#include <string>
#include <utility>

#include "internal.h"

namespace hx {
namespace {

inline int ew_blocks(int n, int per_thread) { return (n / per_thread + 255) / 256; }

// records a start/stop event pair around the launches in its scope when profiling
struct Timed {
    const LaunchCtx &c;
    Profiler::Rec r;
    Timed(const LaunchCtx &cc, int cls, double bytes) : c(cc)
    {
        if (!c.prof) return;
        r.cls = cls;
        r.bytes = bytes;
        r.a = c.prof->get();
        r.b = c.prof->get();
        cudaEventRecord(r.a, c.stream);
    }
    ~Timed()
    {
        if (!c.prof) return;
        cudaEventRecord(r.b, c.stream);
        c.prof->recs.push_back(r);
    }
};

// Kernels launched by launch(): first of all they wait until the stream's previous kernel has
// finished and its writes are visible, and then let the next one be scheduled (in this order, so that
// one kernel at most waits on the SMs).  Such a kernel exists while its predecessor still writes, so what
// a kernel may have written -- every residue and every double -- is read through plain pointers:
// `const ... * __restrict__` allows the read-only path, which is defined only for data that nobody
// writes as long as the kernel exists.  Context tables and job lists (written by copies) keep it.
__device__ __forceinline__ void after_previous_kernel()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A launch of a kernel that begins with after_previous_kernel(): its blocks are scheduled as the
// previous kernel's last ones leave room, which takes the launch latency out of a chain of small
// kernels and fills the tails of larger ones.  One rotation of N = 2^12 53 -> 29 us, one 16x16 product
// 0.71 -> 0.50 ms, a small dense layer 10.4 -> 8.9 ms, 1600 transforms of N = 2^14 199 -> 194 us.
template <class... P, class... Args>
inline void launch(cudaStream_t s, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, Args &&...args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t launched = cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
    if (launched != cudaSuccess) cudaGetLastError();  // reported here, not by the next call as well
    HX_CUDA(launched);
}

inline void post(const LaunchCtx &c, int k = 1)
{
    if (c.launches) *c.launches += k;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw Error{HX_ECUDA, std::string("kernel launch: ") + cudaGetErrorString(e)};
}

} // namespace
} // namespace hx
