// dot_fft.cuh -- fast Poisson solve A^*A phi = b of the node grid (k_fft.cu): fast
// cosine transforms along the spatial axes and a tridiagonal solve along time, in FP32
// (the mixed path's iterations) or FP64 (the reference path).
#pragma once
#include <cuda_runtime.h>

#include <vector>

#include "dot_internal.cuh"

namespace dot {

struct SlotParam;

template <class R> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };

// Tables of one axis of N points, 3 N pairs: exp(-2 pi i j / N); the forward output
// factors and the inverse input factors (cos, sin)(pi k / 2N) with the orthonormal
// scaling folded in.
std::vector<double> fft_tables_host(int N);
void fft_tables_fill(int N, float* out);   // the same into 6 N floats
inline size_t fft_table_pairs(int N) { return (size_t)3 * N; }

template <class R>
struct FastPoisson {
  const typename Vec2<R>::type* tab[kMaxD];   // per spatial axis
  const R* lam[kMaxD];                        // 1D Neumann eigenvalues per spatial axis
  R* w1;                                      // scratch, one field per solve
  R* w2;
  const SlotParam* sp;                        // mixed path: slots whose `active` is 0 are skipped (nullptr: none)
};

// Whether the fast solve takes this grid (axis and time lengths that fit shared memory).
bool fast_poisson_supported(const Geo& g, size_t word);

// dst = (A^*A)^dagger src for G solves stored one after the other; src is preserved
// unless it is w1 or w2.  accum (FP32 only, two-float): the result is added into it
// instead of written to dst.
void launch_fast_poisson(const Geo& g, int G, const FastPoisson<float>& fp, const float* src, float* dst,
                         float2* accum, cudaStream_t s, LaunchCounter lc);
void launch_fast_poisson(const Geo& g, int G, const FastPoisson<double>& fp, const double* src, double* dst,
                         cudaStream_t s, LaunchCounter lc);

}  // namespace dot
