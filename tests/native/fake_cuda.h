// A stand-in for the CUDA runtime on a machine without a GPU, for tests of the
// library's host code (fake_cuda.cpp): device memory is zeroed host memory,
// streams run at once, kernels do nothing (their launches are counted by
// name), and any allocation can be made to fail as a full device's would, with
// the error kept as the runtime's last error.  Linked with the library's
// objects in place of the CUDA runtime (nvcc -cudart none).
#pragma once

#include <cstddef>
#include <functional>

namespace fake {

// the next `skip` device allocations succeed, the `count` after them fail
void fail_after(long skip, long count);
void fail_none();
// device memory in use
size_t live_bytes();
// launches so far of the kernels whose name contains `part`
long launches(const char* part);
// whether the runtime holds an error for cudaGetLastError
bool last_error();
// calls so far that wait for the whole device: cudaMalloc and cudaFree
long device_waits();

// calls so far of cudaMemset and cudaMemsetAsync
long memsets();
// called after each copy from the device, with its destination and bytes (set
// it while no other thread copies)
extern std::function<void(void*, size_t)> on_read;

}  // namespace fake
