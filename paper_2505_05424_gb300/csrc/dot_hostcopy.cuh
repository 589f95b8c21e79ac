// dot_hostcopy.cuh -- device fields to the C ABI's packed FP64 host arrays.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <vector>

namespace dot {

// FP32, two-float and FP64 device elements; pairs of two-floats stored as (high 0, high 1,
// low 0, low 1), a row for each pair of cone components (dot_mixed.cuh: pair_of)
enum HostElem { HOST_F32, HOST_FF, HOST_F64, HOST_PAIRS };

// `rows` rows of `width` elements, `pitch` elements apart on the device, to packed
// doubles: (value * s1) * s2.  HOST_PAIRS: two host rows for each, in the components' order.
struct HostRead {
  const void* src;
  double* dst;
  size_t width, pitch, rows;
  HostElem elem;
  double s1, s2;
};

// The pinned buffer that the reads of one owner (a context, a batch) go through: allocated
// with the owner's other memory and given back with it (allocating it for each read took
// 0.3 ms of the read and, as page-locked allocation waits for the device, held up whatever
// else ran there).
class HostStage {
 public:
  HostStage() = default;
  HostStage(const HostStage&) = delete;
  HostStage& operator=(const HostStage&) = delete;
  ~HostStage();
  // for reads of about `bytes` device bytes; where they are few, or where it fails, reads
  // stay on the calling thread
  void reserve(size_t bytes, HostElem elem);
  char* get() const { return p_; }

 private:
  char* p_ = nullptr;
};

// Runs every read after the work queued on s; returns when the host arrays are filled.
cudaError_t read_to_host(const std::vector<HostRead>& parts, const HostStage& stage, cudaStream_t s);

}  // namespace dot
