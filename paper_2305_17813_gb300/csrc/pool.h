// Device memory of the library (pool.cu).
#pragma once

#include <cuda_runtime_api.h>

#include <cstddef>
#include <cstdint>

namespace mk {

// Memory from the library's pool of the current device: usable in `s` from
// this point, anywhere once `s` has reached it.  pool_alloc is for workspaces
// freed in the same call; pool_alloc_kept for what outlives it (refused in a
// capture), which is given back with its size.  Freeing null does nothing.
cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s);
cudaError_t pool_free(void *p, cudaStream_t s);
cudaError_t pool_alloc_kept(void **p, size_t bytes, cudaStream_t s);
cudaError_t pool_free_kept(void *p, size_t bytes, cudaStream_t s);

// After an object's kept memory has been freed in the null stream (`bytes` of
// it with pool_free): what the pool holds beyond its bound goes back to the
// device before this returns.
cudaError_t pool_settle(uint64_t bytes);

// Makes `device` the thread's current device for a scope: an object may be
// destroyed while another device is current.
class DeviceScope {
  public:
    explicit DeviceScope(int device)
    {
        if (cudaGetDevice(&old_) != cudaSuccess || old_ == device || cudaSetDevice(device) != cudaSuccess)
            old_ = -1;
    }
    ~DeviceScope()
    {
        if (old_ >= 0)
            cudaSetDevice(old_);
    }
    DeviceScope(const DeviceScope &) = delete;
    DeviceScope &operator=(const DeviceScope &) = delete;

  private:
    int old_ = -1; // the device to go back to, -1 for none
};

} // namespace mk
