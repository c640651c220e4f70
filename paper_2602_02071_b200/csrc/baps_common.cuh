// Shared host/device plumbing of the BAPS CUDA library: status word, launch counter, checks.
#pragma once
#include <atomic>
#include <cstdint>
#include <cstdio>
#include <mutex>
#include <cuda_runtime.h>
#include "../../include/baps.h"

namespace baps {

// Device-side status word: 0 = fine; non-zero = a bounded wait expired (the value encodes
// which role gave up).  Read and cleared by baps_poll_async_error().
__device__ int g_async_status = 0;

// Host-side count of kernel launches issued by this library.
static std::atomic<int64_t> g_launches{0};

// Serialises the one-time, per-device set-up steps (table builds, symbol look-ups) when several
// host threads make their first call at the same time.
static std::mutex g_setup_mutex;

constexpr float kLog2e = 1.4426950408889634074f;

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline bool aligned4(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }

inline baps_status launch_status()
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return BAPS_ERR_CUDA;
    ++g_launches;
    return BAPS_OK;
}

// Programmatic dependent launch.  Every kernel of the library is launched with the attribute that lets it start
// before the kernel ahead of it in the stream has ended, does what needs no caller memory (tables, barriers,
// tensor memory), and waits for that kernel -- its completion, whatever it is -- before it touches any.  The wait
// hands the pointer through, so that no load from it, not even one the compiler takes for invariant, can
// move ahead of the wait.  The allow call is made by every CTA when it starts (attention_d64_kernel: when it has its
// tensor memory): the next kernel then comes in as this one's last CTAs drain.
__device__ __forceinline__ void allow_next_kernel() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void await_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename T>
__device__ __forceinline__ T *await_previous_kernel(T *p)
{
    asm volatile("griddepcontrol.wait;" : "+l"(p) :: "memory");
    return p;
}

template <typename... P, typename... A>
inline baps_status launch_kernel(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, A... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...) != cudaSuccess) {
        (void)cudaGetLastError();
        return BAPS_ERR_CUDA;
    }
    return launch_status();
}

inline bool have_device()
{
    int dev = -1;
    return cudaGetDevice(&dev) == cudaSuccess && dev >= 0;
}

inline cudaStream_t as_stream(baps_stream s) { return reinterpret_cast<cudaStream_t>(s); }

} // namespace baps
