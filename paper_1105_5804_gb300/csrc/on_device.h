// on_device.h -- a scope in which a given device is the calling thread's
// current one.  Kernels are launched only while their stream's device is current
// (graphs, which sweeps were before, know their own), so calls that enqueue
// sweeps make the handle's device current and put the caller's back.
#pragma once
#include <cuda_runtime.h>

namespace swccl {

class OnDevice {
 public:
  explicit OnDevice(int device) {
    error_ = cudaGetDevice(&before_);
    if (error_ == cudaSuccess && before_ != device) {
      error_ = cudaSetDevice(device);
      changed_ = error_ == cudaSuccess;
    }
  }
  ~OnDevice() {
    if (changed_) cudaSetDevice(before_);
  }
  OnDevice(const OnDevice&) = delete;
  OnDevice& operator=(const OnDevice&) = delete;
  cudaError_t error() const { return error_; }

 private:
  int before_ = 0;
  bool changed_ = false;
  cudaError_t error_;
};

}  // namespace swccl
