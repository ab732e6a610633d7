// device_launch.h -- launch facts of a kernel instance, kept per device
// (internal to libdtb.so).
#pragma once
#include <cuda_runtime.h>

#include <mutex>

namespace dtb {
namespace {

// Launch facts of one kernel instance on one device: its SM count, its
// resident CTAs per SM, and (once set) its dynamic shared-memory limit.  The
// function attribute and the occupancy are per device, so a process that
// drives several GPUs sets and queries them once on each.
constexpr int kMaxDevices = 64;
struct DeviceLaunch {
  int sms = 0, per_sm = 0;
};
template <typename Fn>
cudaError_t device_launch(DeviceLaunch (&cache)[kMaxDevices], std::mutex& mu, Fn&& setup, DeviceLaunch* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if (cache[dev].sms == 0) {
    DeviceLaunch d;
    e = cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = setup(d);
    if (e != cudaSuccess) return e;
    cache[dev] = d;
  }
  *out = cache[dev];
  return cudaSuccess;
}

// Kernels that run beside the neuron update ask for the same division of an
// SM's memory as it does (all of it shared): an SM that is divided otherwise
// must finish what it runs before it can be divided anew, so a kernel with
// another preference waits for the update instead of running beside it.
template <typename... K>
cudaError_t share_sm_division(K... kernel) {
  cudaError_t e = cudaSuccess;
  ((e = e != cudaSuccess ? e
                         : cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                                cudaSharedmemCarveoutMaxShared)),
   ...);
  return e;
}

}  // namespace
}  // namespace dtb
