// dot_hostcopy.cuh -- device fields to the C ABI's packed FP64 host arrays.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <vector>

namespace dot {

// FP32, two-float, FP64 device elements; one lane of a pair of two-floats stored as
// (high 0, high 1, low 0, low 1)
enum HostElem { HOST_F32, HOST_FF, HOST_F64, HOST_LANE0, HOST_LANE1 };

// `rows` rows of `width` elements, `pitch` elements apart on the device, to packed
// doubles: (value * s1) * s2.
struct HostRead {
  const void* src;
  double* dst;
  size_t width, pitch, rows;
  HostElem elem;
  double s1, s2;
};

// Runs every read after the work queued on s; returns when the host arrays are filled.
cudaError_t read_to_host(const std::vector<HostRead>& parts, cudaStream_t s);

}  // namespace dot
