// Launches that overlap the kernel before them in their stream (programmatic
// dependent launch), for every kernel that runs once per call.
//
// A stream starts a kernel once the one before it has ended and flushed; between
// two short kernels that gap is longer than the kernels (4.1 us per call for 4 KiB, of
// which the kernel itself takes 2.2, and 6.15 us for 1 MiB).  A kernel launched here
// may start while its predecessor still runs or drains: it fills its shared-memory
// tables, which depend on no earlier work, and then waits (pdl_wait) for everything
// before it in the stream to have ended and its writes to be visible.  Measured on a
// stream of such calls, before and after: 4 KiB 4.10 -> 1.9 us (host bound), 1 MiB 6.15 ->
// 2.4, 9 MiB 15.8 -> 11.8, 64 MiB 79.9 -> 74.6.  Filling the tables before the wait
// instead of after it is 0.7 us of that.  Where there is no predecessor to wait for,
// the fill would only keep the first blocks' loads waiting (4 KiB in a captured graph
// 2.32 us with the loads first, 2.46 with the fill first; up to 300 KiB 0.12-0.2 us):
// the single-call kernels take their loads first in a plain launch (EcbArgs::loads_first).
//
// Every kernel launched here calls pdl_wait in every thread before it touches
// global memory other than constants of the library, and pdl_trigger once.  A
// predecessor that never triggers (another library's kernel) ends first, as without
// the attribute; so does any kernel that follows with a plain launch.
#pragma once

#include <cuda_runtime.h>

namespace gbaes {

#ifdef __CUDACC__
// Waits until every earlier operation of the stream has ended and its writes are visible.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next kernel of the stream start (once every CTA has called this or ended).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Whether the next kernel of the stream may overlap its predecessor: not while the
// stream is being captured, so that a captured graph has ordinary edges.
inline bool may_overlap(cudaStream_t stream) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &cap) != cudaSuccess) {
        cudaGetLastError();  // (the legacy stream beside a capture: the launch reports it)
        return false;
    }
    return cap == cudaStreamCaptureStatusNone;
}

// fn<<<grid, threads, smem, stream>>>(a), overlapping its predecessor or (overlap
// false) a plain launch, in which pdl_wait returns at once.
template <class Args>
cudaError_t launch_overlapped(void (*fn)(Args), unsigned grid, unsigned threads, size_t smem, cudaStream_t stream,
                              const Args& a, bool overlap) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    if (overlap) {
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    return cudaLaunchKernelEx(&cfg, fn, a);
}

template <class Args>
cudaError_t launch_overlapped(void (*fn)(Args), unsigned grid, unsigned threads, size_t smem, cudaStream_t stream,
                              const Args& a) {
    return launch_overlapped(fn, grid, threads, smem, stream, a, may_overlap(stream));
}
#endif

}  // namespace gbaes
