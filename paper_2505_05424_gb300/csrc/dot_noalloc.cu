// dot_noalloc.cu -- the mixed-precision refined Poisson solve for callers that
// cannot allocate device memory.
//
// Some callers cannot call cudaMalloc or any allocating runtime: plugins of hosts
// that forbid allocation on their worker threads, processes whose device memory
// is already fully reserved by another allocator, and loops with a fixed memory
// budget that must not risk an allocation failing part way through a run.
// dot_poisson_f32_noalloc serves
// them: the caller passes the right-hand side and the output buffer, and every
// scratch buffer the solve needs (six node-sized FP32 fields, the FP64 partial sums of
// the zero mode, the transform tables) lives in one file-scope __device__ array of
// fixed size, which every GPU that loads this library holds until the process exits.
//
// Both solves of the refinement run the fast transforms (k_fft.cu), whose tables are
// O(N) per axis and go up in one copy with the eigenvalues: dense tables (O(N^2)
// cosines on the host and sixteen copies per call) took 0.25 ms of a call on
// 64 x 48 x 16 and 2.1 ms on 256^2 x 15.
//
// The array is shared by every call: a call overwrites what the previous one
// left there, and two calls whose work overlaps on the GPU (different streams, or
// different host threads on one device) race on it.  Serialise them.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "../../include/dot.h"
#include "dot_mixed.cuh"
#include "dot_paths.cuh"

namespace dot {
namespace {

constexpr long long kMaxNodes = 1LL << 20;  // (T+1) * N_1 * ... * N_D
constexpr int kMaxAxis = 256;               // largest node count along one spatial axis
constexpr int kMaxTimeNodes = 160;          // as DOT_MIXED contexts

// What a call uploads: per axis the transform tables and the eigenvalues, one active slot.
struct Upload {
  float tab[kMaxD][6 * kMaxAxis];
  float lam[kMaxD][kMaxAxis];
  SlotParam sp;
};

// Layout of the scratch array (256-byte aligned pieces, sizes in bytes).
constexpr size_t kField = (size_t)kMaxNodes * sizeof(float);
constexpr size_t kOffB = 0;
constexpr size_t kOffBlo = kOffB + kField;
constexpr size_t kOffPhi1 = kOffBlo + kField;
constexpr size_t kOffR = kOffPhi1 + kField;
constexpr size_t kOffW1 = kOffR + kField;
constexpr size_t kOffW2 = kOffW1 + kField;   // (on small grids with an odd N_y w1 runs up to (T+1) N_x floats into w2)
constexpr size_t kOffUp = kOffW2 + kField;
constexpr size_t kOffSum = kOffUp + (sizeof(Upload) + 255) / 256 * 256;   // partial sums of b, then mean(b)
constexpr size_t kScratchBytes = kOffSum + kBsumStride * sizeof(double);

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

// The host-side name g_scratch is a stand-in, not a device address: the address
// is fetched per device with cudaGetSymbolAddress.
std::mutex g_mu;
void* g_dev_ptr[64] = {nullptr};

Upload g_up;   // host staging (static: this path allocates nothing)

// error text in a fixed buffer (formatting it allocates nothing)
thread_local char g_err[256];

int fail(int code, const char* m, const char* detail = "") {
  std::snprintf(g_err, sizeof(g_err), "%s%s", m, detail);
  return code;
}

}  // namespace
}  // namespace dot

extern "C" const char* dot_noalloc_last_error(void) { return dot::g_err; }

extern "C" int dot_poisson_f32_noalloc(const dot_grid* grid, const float* b, float* phi, void* stream) {
  using namespace dot;
  if (!grid || !b || !phi) return fail(DOT_EINVAL, "grid, b and phi are required");
  if (grid->D != 2 && grid->D != 3) return fail(DOT_EINVAL, "D must be 2 or 3");
  if (grid->T < 1 || grid->T + 1 > kMaxTimeNodes) return fail(DOT_EINVAL, "T + 1 must lie in [2, 160]");
  long long nn = grid->T + 1;
  for (int d = 0; d < grid->D; ++d) {
    if (grid->N[d] < 2 || grid->N[d] > kMaxAxis) return fail(DOT_EINVAL, "every N[d] must lie in [2, 256]");
    nn *= grid->N[d];
  }
  if (nn > kMaxNodes) {
    std::snprintf(g_err, sizeof(g_err),
                  "grid has %lld nodes; this entry point handles at most %lld ((T+1) * N_1 * ... * N_D)", nn,
                  kMaxNodes);
    return DOT_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(DOT_ECUDA, "cudaGetDevice: ", cudaGetErrorString(e));
  if (dev < 0 || dev >= 64) return fail(DOT_EINVAL, "device ordinal out of range");
  std::lock_guard<std::mutex> lock(g_mu);
  // set-up once per device, with that device current (the first call on a device;
  // make it before any stream capture)
  if (!g_dev_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess || !p) return fail(DOT_ECUDA, "cudaGetSymbolAddress: ", cudaGetErrorString(e));
    g_dev_ptr[dev] = p;
  }
  unsigned char* base = (unsigned char*)g_dev_ptr[dev];
  dot_grid gr = *grid;
  Geo g = make_geo(gr);

  MxFields f;
  std::memset(&f, 0, sizeof(f));
  f.b = (float*)(base + kOffB);
  f.blo = (float*)(base + kOffBlo);
  f.phi1 = (float*)(base + kOffPhi1);
  f.r = (float*)(base + kOffR);
  f.bsum = (double*)(base + kOffSum);
  MxPoisson ps;
  std::memset(&ps, 0, sizeof(ps));
  Upload* up = (Upload*)(base + kOffUp);
  f.sp = &up->sp;
  ps.fast.w1 = (float*)(base + kOffW1);
  ps.fast.w2 = (float*)(base + kOffW2);
  ps.use_fast = true;
  for (int d = 0; d < g.D; ++d) {
    const int M = g.N[d];
    const double pi = 3.14159265358979323846;
    fft_tables_fill(M, g_up.tab[d]);
    for (int k = 0; k < M; ++k) {
      const double sv = std::sin(pi * k / (2.0 * M));
      g_up.lam[d][k] = (float)(4.0 * M * M * sv * sv);
    }
    ps.fast.tab[d] = (const float2*)up->tab[d];
    ps.fast.lam[d] = up->lam[d];
  }
  std::memset(&g_up.sp, 0, sizeof(g_up.sp));
  g_up.sp.rescale = make_float2(1.f, 0.f);
  g_up.sp.active = 1;
  // the right-hand side is copied in (the solve overwrites it with the correction); its low
  // part starts at zero
  e = cudaMemcpyAsync(up, &g_up, sizeof(g_up), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(f.b, b, (size_t)nn * sizeof(float), cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(f.blo, 0, (size_t)nn * sizeof(float), s);
  if (e != cudaSuccess) return fail(DOT_ECUDA, "scratch set-up: ", cudaGetErrorString(e));
  long launches = 0;
  LaunchCounter lc{&launches};
  static_assert(kBsumParts + 2 <= kBsumStride, "the partial sums and the mean fit one slot's stride");
  launch_poisson_refined_mx(g, 1, f, ps, reinterpret_cast<float2*>(phi), s, lc);
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail(DOT_ECUDA, "launch: ", cudaGetErrorString(e));
  e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return fail(DOT_ECUDA, "poisson: ", cudaGetErrorString(e));
  return DOT_OK;
}
