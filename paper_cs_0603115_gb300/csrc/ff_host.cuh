// ff_host.cuh -- host-side helpers shared by the library's translation units:
// argument checks, CUDA error capture, device properties and launch sizing.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/ff.h"

namespace ffh {

// Remember a CUDA error for ff_last_cuda_error() (thread-local).
void set_cuda_error(cudaError_t e);

// FF_OK if no launch error is pending, else FF_ERR_CUDA (error recorded).
inline ff_status check_launch()
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_cuda_error(e);
        return FF_ERR_CUDA;
    }
    return FF_OK;
}

inline ff_status cuda_status(cudaError_t e)
{
    if (e != cudaSuccess) {
        set_cuda_error(e);
        return FF_ERR_CUDA;
    }
    return FF_OK;
}

// Launches `kernel` so that it may be scheduled while the kernel before it in
// the stream ends; every kernel launched here waits for that one's end itself,
// before its first access to memory (ffk::prior_kernel_done).  Measured on
// this GPU, a kernel launched the plain way behind another one completes on a
// raster of 2.05 us and starts about 1.3 us late: 304 blocks that do nothing
// take 4.10 us each, 1.43 launched this way; of 8.2 us, 5.2; of 53 us, 2 to 3 less.
// A stream under capture records plain launches, so graphs hold plain edges.
template <class... P, class... A>
ff_status launch_kernel(void (*kernel)(P...), dim3 grid, unsigned block, cudaStream_t s, A... args)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(s, &capture);
    if (e != cudaSuccess) (void)cudaGetLastError();   // the launch reports it
    cudaLaunchAttribute overlap;
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(block);
    c.stream = s;
    c.attrs = &overlap;
    c.numAttrs = e == cudaSuccess && capture == cudaStreamCaptureStatusNone ? 1 : 0;
    (void)cudaLaunchKernelEx(&c, kernel, P(args)...);
    return check_launch();
}

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// A device array argument: non-NULL when it holds elements, 8-byte aligned.
inline bool ok_ptr(const void* p, size_t n) { return n == 0 || (p != nullptr && aligned(p, 8)); }

struct DeviceInfo {
    int device;
    int sm_count;
    int max_threads_per_sm;
};

// Properties of the current device (cached per device).
ff_status device_info(DeviceInfo* out);

// Blocks per SM for `kernel` launched with `block` threads (cached by the
// caller in a function-local static keyed by device when needed).
int occupancy(const void* kernel, int block, size_t smem = 0);

// Grid for a grid-stride kernel: enough blocks to cover `work` items of
// `per_block` each, capped at SMs x resident blocks per SM.
inline unsigned grid_for(size_t work, size_t per_block, int sm_count, int blocks_per_sm)
{
    size_t want = (work + per_block - 1) / per_block;
    size_t cap = static_cast<size_t>(sm_count) * static_cast<size_t>(blocks_per_sm > 0 ? blocks_per_sm : 1);
    if (want < 1) want = 1;
    return static_cast<unsigned>(want < cap ? want : cap);
}

}  // namespace ffh
