// dot_hostcopy.cu -- device fields to packed FP64 host arrays (dot_get).
//
// Converting a field on one host thread after one copy into pageable memory ran at
// about 4 GB/s, page faults of the caller's fresh arrays included, and took as long as
// 60 iterations on 256^2 x 64.  The fields are cut into chunks that a few threads
// take in turn: copy the chunk into the thread's pinned buffer, convert it into the
// caller's array.  Smaller reads stay on the calling thread, as starting the others takes
// about what they save: two-floats, which have to be converted, below 4 MB (dot_get of
// 60^2 x 32, 3.7 MB, 0.53 ms; of 64^2 x 32, 4.3 MB, 0.60 with threads), and FP64, which the
// driver copies into the caller's array, below 12 MB (80^2 x 32, 6.8 MB, 0.60 ms so and 0.80
// with threads; 128^2 x 32, 17 MB, 1.39 and 1.22).
#include <algorithm>
#include <atomic>
#include <exception>
#include <thread>

#include "dot_hostcopy.cuh"
#include "dot_mixed.cuh"

namespace dot {
namespace {

constexpr size_t kChunk = 512 * 1024;            // bytes of one copy
constexpr size_t threaded_bytes(HostElem e) { return e == HOST_F64 ? 12 << 20 : 4 << 20; }
constexpr int kWorkers = 8;

struct Task {
  const HostRead* part;
  size_t r0, nr, c0, nc;   // nr rows from r0, columns [c0, c0 + nc)
};

size_t elem_bytes(HostElem e) { return e == HOST_F32 ? 4 : e == HOST_FF || e == HOST_F64 ? 8 : 16; }

cudaError_t run_task(const Task& t, void* buf, cudaStream_t s) {
  const HostRead& p = *t.part;
  const size_t eb = elem_bytes(p.elem);
  const char* src = static_cast<const char*>(p.src) + (t.r0 * p.pitch + t.c0) * eb;
  cudaError_t e;
  if (t.nr == 1 || (t.nc == p.pitch)) e = cudaMemcpyAsync(buf, src, t.nr * t.nc * eb, cudaMemcpyDeviceToHost, s);
  else e = cudaMemcpy2DAsync(buf, t.nc * eb, src, p.pitch * eb, t.nc * eb, t.nr, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  const double s1 = p.s1, s2 = p.s2;
  if (p.elem == HOST_PAIRS) {
    const float4* v = static_cast<const float4*>(buf);
    for (size_t r = 0; r < t.nr; ++r, v += t.nc) {
      int j0, j1;
      pair_members(2 * (int)p.rows, (int)(t.r0 + r), &j0, &j1);
      double *d0 = p.dst + j0 * p.width + t.c0, *d1 = p.dst + j1 * p.width + t.c0;
      for (size_t i = 0; i < t.nc; ++i) {
        d0[i] = s1 * ((double)v[i].x + (double)v[i].z) * s2;
        d1[i] = s1 * ((double)v[i].y + (double)v[i].w) * s2;
      }
    }
    return cudaSuccess;
  }
  double* d = p.dst + t.r0 * p.width + t.c0;
  const size_t n = t.nr * t.nc;
  if (p.elem == HOST_F32) {
    const float* v = static_cast<const float*>(buf);
    for (size_t i = 0; i < n; ++i) d[i] = (double)v[i] * s1 * s2;
  } else if (p.elem == HOST_FF) {
    const float2* v = static_cast<const float2*>(buf);
    for (size_t i = 0; i < n; ++i) d[i] = s1 * ((double)v[i].x + (double)v[i].y) * s2;
  } else {
    const double* v = static_cast<const double*>(buf);
    for (size_t i = 0; i < n; ++i) d[i] = v[i] * s1 * s2;
  }
  return cudaSuccess;
}

// FP64 fields copied into the caller's arrays and scaled there.
cudaError_t read_f64(const std::vector<HostRead>& parts, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  for (const HostRead& p : parts)
    if (e == cudaSuccess && p.width && p.rows)
      e = cudaMemcpy2DAsync(p.dst, p.width * 8, p.src, p.pitch * 8, p.width * 8, p.rows, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  for (const HostRead& p : parts) {
    double* d = p.dst;
    const double s1 = p.s1, s2 = p.s2;
    if (s1 == 1.0 && s2 == 1.0) continue;
    for (size_t i = 0, n = p.width * p.rows; i < n; ++i) d[i] = d[i] * s1 * s2;
  }
  return cudaSuccess;
}

}  // namespace

HostStage::~HostStage() {
  if (p_) cudaFreeHost(p_);
}

void HostStage::reserve(size_t bytes, HostElem elem) {
  if (p_ || bytes < threaded_bytes(elem)) return;
  if (cudaMallocHost(&p_, kWorkers * kChunk) != cudaSuccess) {
    cudaGetLastError();
    p_ = nullptr;
  }
}

cudaError_t read_to_host(const std::vector<HostRead>& parts, const HostStage& stage, cudaStream_t s) {
  size_t bytes = 0, most = 0;
  for (const HostRead& p : parts) {
    bytes += p.width * p.rows * elem_bytes(p.elem);
    most = std::max(most, threaded_bytes(p.elem));
  }
  const bool threaded = bytes >= most && stage.get();
  if (!threaded && most == threaded_bytes(HOST_F64)) return read_f64(parts, s);
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  std::vector<Task> tasks;
  for (const HostRead& p : parts) {
    const size_t cap = kChunk / elem_bytes(p.elem);
    if (p.width == 0 || p.rows == 0) continue;
    if (p.width >= cap) {
      for (size_t r = 0; r < p.rows; ++r)
        for (size_t c = 0; c < p.width; c += cap) tasks.push_back({&p, r, 1, c, std::min(cap, p.width - c)});
    } else {
      const size_t nr = cap / p.width;
      for (size_t r = 0; r < p.rows; r += nr) tasks.push_back({&p, r, std::min(nr, p.rows - r), 0, p.width});
    }
  }
  const int hw = (int)std::thread::hardware_concurrency();
  int workers = threaded ? std::min(kWorkers, std::max(1, hw)) : 1;
  workers = std::min<int>(workers, std::max<size_t>(1, tasks.size()));
  char* pinned = stage.get();
  std::vector<char> pageable(pinned ? 0 : std::min(bytes, kChunk));
  int dev = 0;
  cudaGetDevice(&dev);
  std::atomic<size_t> next{0};
  std::atomic<int> err{cudaSuccess};
  auto work = [&](char* buf) {
    for (size_t k; (k = next.fetch_add(1)) < tasks.size() && err.load() == cudaSuccess;) {
      const cudaError_t r = run_task(tasks[k], buf, s);
      if (r != cudaSuccess) err.store(r);
    }
  };
  std::vector<std::thread> th;
  th.reserve(workers);
  for (int w = 1; w < workers; ++w) {
    try {
      th.emplace_back([&, w] {
        if (cudaSetDevice(dev) == cudaSuccess) work(pinned + w * kChunk);
      });
    } catch (const std::exception&) {
      break;                                     // the threads that did start share the tasks
    }
  }
  work(pinned ? pinned : pageable.data());
  for (std::thread& t : th) t.join();
  return (cudaError_t)err.load();
}

}  // namespace dot
