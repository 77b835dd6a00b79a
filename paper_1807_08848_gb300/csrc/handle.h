// Giving a handle back: its buffers return to the pool of its own device once that device
// has no work left.  Host code only, of the CUDA runtime's device calls and nothing else.
#pragma once
#include <cuda_runtime_api.h>

namespace msp {

// A device made current for a scope.
struct DeviceScope {
    int before = -1;
    cudaError_t status;
    explicit DeviceScope(int device) {
        status = cudaGetDevice(&before);
        if (status != cudaSuccess) before = -1;
        else if (before != device) status = cudaSetDevice(device);
    }
    ~DeviceScope() {
        if (before >= 0) cudaSetDevice(before);
    }
    DeviceScope(const DeviceScope&) = delete;
    DeviceScope& operator=(const DeviceScope&) = delete;
};

// Waits for every kernel of `device`.  cudaFree of a stream-ordered allocation takes its
// accesses to be complete and waits for nothing, while a call that only enqueues (a solve
// without iteration counts, a snapshot copy) may still be running.  An error is returned and
// cleared.
inline cudaError_t wait_for_device(int device) {
    DeviceScope on(device);
    const cudaError_t e = on.status == cudaSuccess ? cudaDeviceSynchronize() : on.status;
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
}

// Deletes a handle of `device`, whichever device is current.  When the wait fails (the context
// is lost, a capture forbids it) the handle stays: memory that kernels may be using is not
// given back.
template <class Handle>
cudaError_t release_handle(Handle* h, int device) {
    DeviceScope on(device);
    const cudaError_t e = wait_for_device(device);
    if (e == cudaSuccess) delete h;
    return e;
}

}  // namespace msp
