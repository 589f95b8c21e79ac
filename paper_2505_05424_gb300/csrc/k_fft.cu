// k_fft.cu -- fast Poisson solve of the node grid (Sec. 4, phi-subproblem of
// Algorithm 2): A^*A is the Neumann Laplacian, diagonalised along space by the
// orthonormal DCT-II of each axis and solved along time, for each pair of spatial
// frequencies, as the tridiagonal system (lambda I + L_t) x = b.
//
// Spatial transforms.  A DCT-II of N points is a DFT of the reordered sequence
// v = (x_0, x_2, ..., x_3, x_1) and one rotation per output (Makhoul, "A fast cosine
// transform in one and two dimensions", IEEE Trans. ASSP 28(1), 1980); the DCT-III runs
// it backwards.  Two real sequences travel as the real and imaginary part of one
// complex DFT, which any N allows.  The DFT is a Stockham autosort in shared memory:
// radices 8, 4, 2, 3, 5 in registers, any other prime p by sums over conjugate pairs
// (p - 1 multiply-adds per output).  Fields keep their natural layout: a CTA takes NP
// pairs of sequences, neighbouring columns of a strided axis (or pairs of rows of the
// innermost one), stored with the pair index fastest, so that every stage reads and
// writes shared memory without bank conflicts.
//
// Time solve.  Eliminated downwards without subtraction: with a = 1/h_0^2 and pivots
// d_i = a + s_i, s_i = lambda + a s_{i-1} / d_{i-1}, every s_i is a sum of positive terms,
// accurate to a few ulps for the smallest lambda.  The column lambda = 0 is singular:
// its mean is removed from b and from x (the zero mode of the DCT), in FP64.
//
// FP64: GB300 issues two FP64 lanes per SM and clock, so the count of operations is the
// time: 17 per element and axis here against 256 multiply-adds of a dense 256-point
// transform.  256^2 x 64, per iteration: four axis passes of 141 us and the time solve
// of 115 us (a dense transform: six passes of 1,789 us and 84 us of scaling);
// 37 x 21 x 50 x 20: 54 and 28 us (159 and 23).
#include <cmath>
#include <cstring>
#include <type_traits>

#include "dot_fft.cuh"
#include "dot_mixed.cuh"
#include "ffloat.cuh"

namespace dot {

std::vector<double> fft_tables_host(int N) {
  const double pi = 3.14159265358979323846;
  std::vector<double> t((size_t)6 * N);
  for (int j = 0; j < N; ++j) {
    const double w = 2.0 * pi * j / N, h = pi * j / (2.0 * N);
    const double fo = (j == 0 ? std::sqrt(1.0 / N) : std::sqrt(2.0 / N)) / 2.0;
    const double in = j == 0 ? std::sqrt(1.0 / N) : std::sqrt(1.0 / (2.0 * N));
    t[2 * j] = std::cos(w);
    t[2 * j + 1] = -std::sin(w);
    t[2 * (N + j)] = fo * std::cos(h);
    t[2 * (N + j) + 1] = fo * std::sin(h);
    t[2 * (2 * N + j)] = in * std::cos(h);
    t[2 * (2 * N + j) + 1] = in * std::sin(h);
  }
  return t;
}

namespace {

constexpr int kThreads = 256;
constexpr int kMaxStages = 16;

struct FftPlan {
  int N, nst;
  int rad[kMaxStages];
  FastDiv fs[kMaxStages];   // division by the stage's stride (product of the radices before it)
  FastDiv fr[kMaxStages];   // division by N / radix (other primes only)
  FastDiv fN;
};

FftPlan make_plan(int N) {
  FftPlan p;
  std::memset(&p, 0, sizeof(p));
  p.N = N;
  p.fN = make_fastdiv((unsigned)N);
  int n = N, e = 0, s = 1;
  while (n % 2 == 0) { n /= 2; ++e; }
  auto add = [&](int r) {
    p.rad[p.nst] = r;
    p.fs[p.nst] = make_fastdiv((unsigned)s);
    p.fr[p.nst] = make_fastdiv((unsigned)(N / r));
    ++p.nst;
    s *= r;
  };
  while (e >= 5 || e == 3) { add(8); e -= 3; }
  while (e >= 2) { add(4); e -= 2; }
  if (e) add(2);
  for (int r = 3; n > 1; r += 2)
    while (n % r == 0) { add(r); n /= r; }
  return p;
}

template <class R>
struct FftArgs {
  using R2 = typename Vec2<R>::type;
  const R* src;
  R* dst;
  float2* accum;
  const R2* tab;
  int inner;              // elements between neighbours along the axis; 1: contiguous rows
  long long npair;        // pairs of sequences
  FastDiv fpi;            // division by the pairs per outer index (inner > 1)
  int pin;                // pairs per outer index
  long long nseq;         // sequences (inner == 1)
  const SlotParam* sp;
  long long slot_pairs;   // pairs per slot (sp != nullptr)
  FftPlan plan;
};

template <class V, class R>
__device__ __forceinline__ V mk(R x, R y) { V v; v.x = x; v.y = y; return v; }
template <class V>
__device__ __forceinline__ V cadd(V a, V b) { return mk<V>(a.x + b.x, a.y + b.y); }
template <class V>
__device__ __forceinline__ V csub(V a, V b) { return mk<V>(a.x - b.x, a.y - b.y); }
// a * w, w conjugated for the inverse transform
template <bool INV, class V>
__device__ __forceinline__ V cmulw(V a, V w) {
  return INV ? mk<V>(a.x * w.x + a.y * w.y, a.y * w.x - a.x * w.y) : mk<V>(a.x * w.x - a.y * w.y, a.y * w.x + a.x * w.y);
}
// a * (-i) (forward), a * i (inverse)
template <bool INV, class V>
__device__ __forceinline__ V rot(V a) { return INV ? mk<V>(-a.y, a.x) : mk<V>(a.y, -a.x); }

template <bool INV, class V>
__device__ __forceinline__ void dft4(V& a, V& b, V& c, V& d) {
  const V s0 = cadd(a, c), d0 = csub(a, c), s1 = cadd(b, d), d1 = rot<INV>(csub(b, d));
  a = cadd(s0, s1);
  b = cadd(d0, d1);
  c = csub(s0, s1);
  d = csub(d0, d1);
}

template <int RAD, bool INV, class V>
__device__ __forceinline__ void dft(V* x) {
  using R = decltype(x[0].x);
  if constexpr (RAD == 2) {
    const V a = x[0];
    x[0] = cadd(a, x[1]);
    x[1] = csub(a, x[1]);
  } else if constexpr (RAD == 3) {
    const V s = cadd(x[1], x[2]), d = rot<INV>(csub(x[1], x[2]));
    const auto h = (std::remove_reference_t<R>)0.86602540378443864676;
    const V m = mk<V>(x[0].x - (std::remove_reference_t<R>)0.5 * s.x, x[0].y - (std::remove_reference_t<R>)0.5 * s.y);
    x[0] = cadd(x[0], s);
    x[1] = mk<V>(m.x + h * d.x, m.y + h * d.y);
    x[2] = mk<V>(m.x - h * d.x, m.y - h * d.y);
  } else if constexpr (RAD == 4) {
    dft4<INV>(x[0], x[1], x[2], x[3]);
  } else if constexpr (RAD == 5) {
    using S = std::remove_reference_t<R>;
    const S c1 = (S)0.30901699437494742410, c2 = (S)-0.80901699437494742410;
    const S s1 = (S)0.95105651629515357212, s2 = (S)0.58778525229247312917;
    const V a = cadd(x[1], x[4]), b = cadd(x[2], x[3]);
    const V c = rot<INV>(csub(x[1], x[4])), d = rot<INV>(csub(x[2], x[3]));
    const V m1 = mk<V>(x[0].x + c1 * a.x + c2 * b.x, x[0].y + c1 * a.y + c2 * b.y);
    const V m2 = mk<V>(x[0].x + c2 * a.x + c1 * b.x, x[0].y + c2 * a.y + c1 * b.y);
    const V n1 = mk<V>(s1 * c.x + s2 * d.x, s1 * c.y + s2 * d.y);
    const V n2 = mk<V>(s2 * c.x - s1 * d.x, s2 * c.y - s1 * d.y);
    x[0] = mk<V>(x[0].x + a.x + b.x, x[0].y + a.y + b.y);
    x[1] = cadd(m1, n1);
    x[4] = csub(m1, n1);
    x[2] = cadd(m2, n2);
    x[3] = csub(m2, n2);
  } else if constexpr (RAD == 8) {
    using S = std::remove_reference_t<R>;
    const S h = (S)0.70710678118654752440;
    dft4<INV>(x[0], x[2], x[4], x[6]);   // even inputs: outputs 0..3 in x[0], x[2], x[4], x[6]
    dft4<INV>(x[1], x[3], x[5], x[7]);
    const V e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    const V o0 = x[1], o2 = rot<INV>(x[5]);
    // x[3] w_8, x[7] w_8^3 with w_8 = (1 -+ i) / sqrt 2
    const V r1 = rot<INV>(x[3]), r3 = rot<INV>(x[7]);
    const V o1 = mk<V>(h * (x[3].x + r1.x), h * (x[3].y + r1.y));
    const V o3 = mk<V>(h * (r3.x - x[7].x), h * (r3.y - x[7].y));
    x[0] = cadd(e0, o0);
    x[4] = csub(e0, o0);
    x[1] = cadd(e1, o1);
    x[5] = csub(e1, o1);
    x[2] = cadd(e2, o2);
    x[6] = csub(e2, o2);
    x[3] = cadd(e3, o3);
    x[7] = csub(e3, o3);
  }
}

// One Stockham stage of radix RAD with stride s: butterfly b = p s + q reads elements
// b + (N / RAD) j and writes q + s (RAD p + k), times exp(-2 pi i s p k / N).
template <int RAD, int NP, bool INV, class V>
__device__ __forceinline__ void stage(const V* src, V* dst, const V* tw, int N, int s, FastDiv fs) {
  constexpr int kPitch = NP + 1;
  const int nb = N / RAD;
  for (int e = threadIdx.x; e < nb * NP; e += kThreads) {
    const int pr = e % NP, b = e / NP;
    const int p = (int)fdiv((unsigned)b, fs), q = b - p * s;
    V x[RAD];
#pragma unroll
    for (int j = 0; j < RAD; ++j) x[j] = src[(b + nb * j) * kPitch + pr];
    dft<RAD, INV>(x);
    V* o = dst + (q + s * RAD * p) * kPitch + pr;
    o[0] = x[0];
    if (nb > s) {   // not the last stage
#pragma unroll
      for (int k = 1; k < RAD; ++k) x[k] = cmulw<INV>(x[k], tw[s * p * k]);
    }
#pragma unroll
    for (int k = 1; k < RAD; ++k) o[s * k * kPitch] = x[k];
  }
}

// A stage of any odd radix r: outputs k and r - k share their sums over the conjugate
// input pairs, sum_j (x_j + x_{r-j}) cos and (x_j - x_{r-j}) sin.
template <int NP, bool INV, class V>
__device__ __forceinline__ void stage_any(const V* src, V* dst, const V* tw, int N, int r, int s, FastDiv fs,
                                          FastDiv fr) {
  constexpr int kPitch = NP + 1;
  const int nb = N / r, hk = (r + 1) / 2;
  for (int e = threadIdx.x; e < nb * hk * NP; e += kThreads) {
    const int pr = e % NP, bk = e / NP;
    const int k = (int)fdiv((unsigned)bk, fr), b = bk - k * nb;
    const int p = (int)fdiv((unsigned)b, fs), q = b - p * s;
    const V* x = src + b * kPitch + pr;
    V* o = dst + (q + s * r * p) * kPitch + pr;
    V re = x[0], im = mk<V>(re.x - re.x, re.y - re.y);
    int m = 0;   // j k mod r
    for (int j = 1; j < hk; ++j) {
      m += k;
      if (m >= r) m -= r;
      const V w = tw[m * nb];
      const V a = x[nb * j * kPitch], c = x[nb * (r - j) * kPitch];
      const V sm = cadd(a, c), df = csub(a, c);
      re = mk<V>(re.x + sm.x * w.x, re.y + sm.y * w.x);
      // i w.y df, w.y = -sin (forward)
      im = INV ? mk<V>(im.x + df.y * w.y, im.y - df.x * w.y) : mk<V>(im.x - df.y * w.y, im.y + df.x * w.y);
    }
    V y = cadd(re, im);
    if (k && nb > s) y = cmulw<INV>(y, tw[s * p * k]);
    o[s * k * kPitch] = y;
    if (k) {
      V z = csub(re, im);
      if (nb > s) z = cmulw<INV>(z, tw[s * p * (r - k)]);
      o[s * (r - k) * kPitch] = z;
    }
  }
}

// All stages; returns the buffer that holds the result.
template <int NP, bool INV, class V>
__device__ __forceinline__ V* transform(V* a, V* b, const V* tw, const FftPlan& pl) {
  int s = 1;
  for (int i = 0; i < pl.nst; ++i) {
    const int r = pl.rad[i];
    switch (r) {
      case 8: stage<8, NP, INV>(a, b, tw, pl.N, s, pl.fs[i]); break;
      case 4: stage<4, NP, INV>(a, b, tw, pl.N, s, pl.fs[i]); break;
      case 2: stage<2, NP, INV>(a, b, tw, pl.N, s, pl.fs[i]); break;
      case 3: stage<3, NP, INV>(a, b, tw, pl.N, s, pl.fs[i]); break;
      case 5: stage<5, NP, INV>(a, b, tw, pl.N, s, pl.fs[i]); break;
      default: stage_any<NP, INV>(a, b, tw, pl.N, r, s, pl.fs[i], pl.fr[i]); break;
    }
    __syncthreads();
    V* t = a;
    a = b;
    b = t;
    s *= r;
  }
  return a;
}

__device__ __forceinline__ void put(float* dst, float2* accum, long long i, float v) {
  if (accum) accum[i] = ff_add_f(accum[i], v);
  else dst[i] = v;
}
__device__ __forceinline__ void put(double* dst, float2*, long long i, double v) { dst[i] = v; }

// The DCT-II (INV false) or DCT-III of NP pairs of sequences.
template <class R, int NP, bool INV>
__global__ void __launch_bounds__(kThreads) k_dct_fft(const __grid_constant__ FftArgs<R> a) {
  using V = typename Vec2<R>::type;
  constexpr int kPitch = NP + 1;
  extern __shared__ __align__(16) unsigned char fsm[];
  const int N = a.plan.N;
  V* A = reinterpret_cast<V*>(fsm);
  V* B = A + N * kPitch;
  V* tw = B + N * kPitch;
  const long long p0 = (long long)blockIdx.x * NP;
  if (a.sp) {   // nothing to do where every slot of the CTA's pairs is empty
    const long long last = min(p0 + NP, a.npair) - 1;
    bool on = false;
    for (long long b = p0 / a.slot_pairs; b <= last / a.slot_pairs; ++b) on = on || a.sp[b].active;
    if (!on) return;
  }
  const V* rotf = a.tab + (INV ? 2 : 1) * N;
  for (int j = threadIdx.x; j < N; j += kThreads) tw[j] = a.tab[j];
  const R zero = (R)0;
  if (a.inner > 1) {
    // a thread keeps its pair of columns
    const int pr = threadIdx.x % NP, j0 = threadIdx.x / NP;
    const long long pg = p0 + pr;
    const bool ok = pg < a.npair;
    const long long o = ok ? (long long)fdiv((unsigned)pg, a.fpi) : 0;
    const int ci = ok ? 2 * (int)(pg - o * a.pin) : 0;
    const bool two = ok && ci + 1 < a.inner;
    const long long base = o * N * a.inner + ci;
    constexpr int kStep = kThreads / NP;
    if (!INV) {
      for (int j = j0; j < N; j += kStep) {
        const R* s = a.src + base + (long long)j * a.inner;
        const int pos = (j & 1) ? N - 1 - (j >> 1) : j >> 1;
        A[pos * kPitch + pr] = mk<V>(ok ? s[0] : zero, two ? s[1] : zero);
      }
    } else {
      for (int k = j0; k <= N / 2; k += kStep) {
        const int m = k ? N - k : 0;
        const R* sk = a.src + base + (long long)k * a.inner;
        const R* sm = a.src + base + (long long)m * a.inner;
        const R ak = ok ? sk[0] : zero, bk = two ? sk[1] : zero;
        const R am = ok && k ? sm[0] : zero, bm = two && k ? sm[1] : zero;
        const V w = rotf[k];
        // V_a = (c ak + s am) + i (s ak - c am), Z = V_a + i V_b
        A[k * kPitch + pr] = mk<V>((w.x * ak + w.y * am) - (w.y * bk - w.x * bm),
                                   (w.y * ak - w.x * am) + (w.x * bk + w.y * bm));
        if (k && m != k) {
          const V u = rotf[m];
          A[m * kPitch + pr] = mk<V>((u.x * am + u.y * ak) - (u.y * bm - u.x * bk),
                                     (u.y * am - u.x * ak) + (u.x * bm + u.y * bk));
        }
      }
    }
    __syncthreads();
    const V* Z = transform<NP, INV>(A, B, tw, a.plan);
    if (!ok) return;
    if (!INV) {
      for (int k = j0; k <= N / 2; k += kStep) {
        const int m = k ? N - k : 0;
        const V z = Z[k * kPitch + pr], y = Z[m * kPitch + pr];
        const V w = rotf[k];
        const V sp = cadd(z, y), sd = csub(z, y);
        // X_a = c (zr + mr) + s (zi - mi), X_b = c (zi + mi) + s (mr - zr)
        const long long ik = base + (long long)k * a.inner;
        put(a.dst, a.accum, ik, w.x * sp.x + w.y * sd.y);
        if (two) put(a.dst, a.accum, ik + 1, w.x * sp.y - w.y * sd.x);
        if (k && m != k) {
          const V u = rotf[m];
          const long long im = base + (long long)m * a.inner;
          put(a.dst, a.accum, im, u.x * sp.x - u.y * sd.y);
          if (two) put(a.dst, a.accum, im + 1, u.x * sp.y + u.y * sd.x);
        }
      }
    } else {
      for (int j = j0; j < N; j += kStep) {
        const int pos = (j & 1) ? N - 1 - (j >> 1) : j >> 1;
        const V z = Z[pos * kPitch + pr];
        const long long ij = base + (long long)j * a.inner;
        put(a.dst, a.accum, ij, z.x);
        if (two) put(a.dst, a.accum, ij + 1, z.y);
      }
    }
  } else {
    // pairs of contiguous rows: neighbouring threads take neighbouring elements
    const int np = (int)min((long long)NP, a.npair - p0);
    if (!INV) {
      for (int e = threadIdx.x; e < NP * N; e += kThreads) {
        const int pr = (int)fdiv((unsigned)e, a.plan.fN), j = e - pr * N;
        const long long row = 2 * (p0 + pr);
        const R* s = a.src + row * N + j;
        const int pos = (j & 1) ? N - 1 - (j >> 1) : j >> 1;
        A[pos * kPitch + pr] = mk<V>(row < a.nseq ? s[0] : zero, row + 1 < a.nseq ? s[N] : zero);
      }
    } else {
      for (int e = threadIdx.x; e < NP * N; e += kThreads) {
        const int pr = (int)fdiv((unsigned)e, a.plan.fN), k = e - pr * N;
        const long long row = 2 * (p0 + pr);
        const bool ok = row < a.nseq, two = row + 1 < a.nseq;
        const R* s = a.src + row * N;
        const int m = N - k;
        const R ak = ok ? s[k] : zero, bk = two ? s[N + k] : zero;
        const R am = ok && k ? s[m] : zero, bm = two && k ? s[N + m] : zero;
        const V w = rotf[k];
        A[k * kPitch + pr] = mk<V>((w.x * ak + w.y * am) - (w.y * bk - w.x * bm),
                                   (w.y * ak - w.x * am) + (w.x * bk + w.y * bm));
      }
    }
    __syncthreads();
    const V* Z = transform<NP, INV>(A, B, tw, a.plan);
    for (int e = threadIdx.x; e < np * N; e += kThreads) {
      const int pr = (int)fdiv((unsigned)e, a.plan.fN), k = e - pr * N;
      const long long row = 2 * (p0 + pr);
      R xa, xb;
      if (!INV) {
        const V z = Z[k * kPitch + pr], y = Z[(k ? N - k : 0) * kPitch + pr];
        const V w = rotf[k];
        xa = w.x * (z.x + y.x) + w.y * (z.y - y.y);
        xb = w.x * (z.y + y.y) - w.y * (z.x - y.x);
      } else {
        const V z = Z[((k & 1) ? N - 1 - (k >> 1) : k >> 1) * kPitch + pr];
        xa = z.x;
        xb = z.y;
      }
      put(a.dst, a.accum, row * N + k, xa);
      if (row + 1 < a.nseq) put(a.dst, a.accum, (row + 1) * N + k, xb);
    }
  }
}

// 1 / x, x > 0 and normal, to about an ulp
__device__ __forceinline__ float recip(float x) {
  const float r = rcp_approx(x);
  return fmaf(r, fmaf(-x, r, 1.f), r);
}
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }

template <class R>
struct TimeArgs {
  const R* src;
  R* dst;
  const R* lam[kMaxD];
  R a;                 // 1 / h_0^2
  long long ncol;      // columns over all slots
  const SlotParam* sp;
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// sum of v over the lanes before this one
__device__ __forceinline__ double warp_before(double v) {
  const int lane = threadIdx.x & 31;
  double s = v;
  for (int o = 1; o < 32; o *= 2) {
    const double u = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += u;
  }
  return s - v;
}

// The column lambda = 0 by one warp, in FP64: L_t x = b - mean(b) with mean(x) = 0, that is
// x_t = x_0 - sum_{i < t} S_i / a with S_i = sum_{j <= i} (b_j - mean(b)).  A lane holds a
// run of time nodes.
template <class R>
__device__ void zero_column(const R* b, R* x, int M, long long P, double a) {
  const int lane = threadIdx.x & 31, C = (M + 31) / 32;
  const int t0 = min(M, lane * C), t1 = min(M, t0 + C);
  double v = 0.0;
  for (int t = t0; t < t1; ++t) v += (double)b[t * P];
  const double mean = warp_sum(v) / M;
  const double S0 = warp_before(v - mean * (t1 - t0));   // S before this lane's first node
  double S = S0, run = 0.0;
  for (int t = t0; t < t1; ++t) {
    S += (double)b[t * P] - mean;
    run += S;
  }
  const double U0 = warp_before(run);                      // sum of S before this lane
  double u = U0, xs = 0.0;
  S = S0;
  for (int t = t0; t < t1; ++t) {
    xs -= u / a;
    S += (double)b[t * P] - mean;
    u += S;
  }
  const double shift = warp_sum(xs) / M;
  u = U0;
  S = S0;
  for (int t = t0; t < t1; ++t) {
    const double bt = (double)b[t * P];
    x[t * P] = (R)(-u / a - shift);
    S += bt - mean;
    u += S;
  }
}

// (lambda I + L_t) x = b along time, one thread per column of spatial frequencies; the
// eliminated right-hand sides and the pivots' reciprocals wait in shared memory.
template <class R, int THREADS>
__global__ void __launch_bounds__(THREADS) k_time_solve(const __grid_constant__ Geo g,
                                                        const __grid_constant__ TimeArgs<R> ta) {
  extern __shared__ __align__(16) unsigned char fsm[];
  const long long col = (long long)blockIdx.x * THREADS + threadIdx.x;
  const long long P = g.P;
  // the singular columns (p = 0 of a slot), by the first warp of the block they fall in
  {
    const long long c0 = (long long)blockIdx.x * THREADS;
    const long long z0 = (c0 + P - 1) / P;   // first slot whose column 0 is not before c0
    if (threadIdx.x < 32)
      for (long long z = z0; z * P < min(c0 + THREADS, ta.ncol); ++z)
        if (!ta.sp || ta.sp[z].active)
          zero_column(ta.src + z * (g.T + 1) * P, ta.dst + z * (g.T + 1) * P, g.T + 1, P, (double)ta.a);
  }
  if (col >= ta.ncol) return;
  const int slot = (int)fdiv((unsigned)col, g.fP), p = (int)(col - slot * P);
  if (p == 0) return;
  if (ta.sp && !ta.sp[slot].active) return;
  const int M = g.T + 1;
  const R* b = ta.src + slot * M * P + p;
  R* x = ta.dst + slot * M * P + p;
  R* y = reinterpret_cast<R*>(fsm) + threadIdx.x;        // y[t THREADS]
  R* rr = y + (size_t)M * THREADS;                       // 1 / d_t
  R lam = (R)0;
  for (int d = 0; d < g.D; ++d) lam += ta.lam[d][coord(g, p, d)];
  const R a = ta.a;
  R s = lam, yp = b[0];
  R r = recip(a + s);
  y[0] = yp;
  rr[0] = r;
#pragma unroll 8
  for (int t = 1; t < M; ++t) {
    const R ar = a * r;
    s = lam + ar * s;
    yp = b[t * P] + ar * yp;
    r = recip(t < M - 1 ? a + s : s);
    y[t * THREADS] = yp;
    rr[t * THREADS] = r;
  }
  R xp = yp * r;
  x[(M - 1) * P] = xp;
#pragma unroll 8
  for (int t = M - 2; t >= 0; --t) {
    xp = (y[t * THREADS] + a * xp) * rr[t * THREADS];
    x[t * P] = xp;
  }
}

constexpr int kMaxSmem = 220 * 1024;
template <class R> constexpr int time_threads() { return sizeof(R) == 4 ? 128 : 64; }

template <class R>
size_t fft_smem(int N, int NP) { return (size_t)(2 * N * (NP + 1) + N) * 2 * sizeof(R); }

template <class R, int NP, bool INV>
void launch_np(const FftArgs<R>& a, cudaStream_t s) {
  static std::atomic<unsigned long long> done{0};
  smem_optin((const void*)k_dct_fft<R, NP, INV>, kMaxSmem, &done);
  k_dct_fft<R, NP, INV><<<(unsigned)((a.npair + NP - 1) / NP), kThreads, fft_smem<R>(a.plan.N, NP), s>>>(a);
}

// One axis of G solves.  Pairs per CTA: 16 (8 in FP64: 128-byte segments of a strided
// axis), fewer while that leaves SMs without a CTA or does not fit shared memory.
template <class R, bool INV>
void fft_axis(const Geo& g, int G, int axis, const FastPoisson<R>& fp, const R* src, R* dst, float2* accum,
              cudaStream_t s, LaunchCounter lc) {
  FftArgs<R> a;
  std::memset(&a, 0, sizeof(a));
  const int N = g.N[axis];
  const long long total = (long long)G * (g.T + 1) * g.P;
  a.src = src;
  a.dst = dst;
  a.accum = accum;
  a.tab = fp.tab[axis];
  a.inner = (int)g.sst[axis];
  a.nseq = total / N;
  a.pin = (a.inner + 1) / 2;
  a.npair = a.inner > 1 ? total / ((long long)N * a.inner) * a.pin : (a.nseq + 1) / 2;
  a.fpi = make_fastdiv((unsigned)a.pin);
  a.plan = make_plan(N);
  a.sp = G > 1 ? fp.sp : nullptr;
  a.slot_pairs = G > 1 ? a.npair / G : a.npair;
  int np = sizeof(R) == 4 ? 16 : 8;
  while (np > 2 && (fft_smem<R>(N, np) > (size_t)kMaxSmem / 2 || (a.npair + np - 1) / np < 2 * 152)) np /= 2;
  while (np > 1 && fft_smem<R>(N, np) > (size_t)kMaxSmem) np /= 2;
  switch (np) {
    case 16: launch_np<R, 16, INV>(a, s); break;
    case 8: launch_np<R, 8, INV>(a, s); break;
    case 4: launch_np<R, 4, INV>(a, s); break;
    case 2: launch_np<R, 2, INV>(a, s); break;
    default: launch_np<R, 1, INV>(a, s); break;
  }
  lc.launched(KID_DCT_AXIS);
}

template <class R>
void fast_poisson(const Geo& g, int G, const FastPoisson<R>& fp, const R* src, R* dst, float2* accum, cudaStream_t s,
                  LaunchCounter lc) {
  R* w[2] = {fp.w1, fp.w2};
  const R* cur = src;
  int nx = 0;
  for (int d = g.D - 1; d >= 0; --d) {
    fft_axis<R, false>(g, G, d, fp, cur, w[nx], nullptr, s, lc);
    cur = w[nx];
    nx ^= 1;
  }
  constexpr int kT = time_threads<R>();
  TimeArgs<R> ta;
  std::memset(&ta, 0, sizeof(ta));
  ta.src = cur;
  ta.dst = w[nx];
  for (int d = 0; d < g.D; ++d) ta.lam[d] = fp.lam[d];
  ta.a = (R)(g.invh[0] * g.invh[0]);
  ta.ncol = (long long)G * g.P;
  ta.sp = G > 1 ? fp.sp : nullptr;
  static std::atomic<unsigned long long> done{0};
  smem_optin((const void*)k_time_solve<R, kT>, kMaxSmem, &done);
  k_time_solve<R, kT><<<(unsigned)((ta.ncol + kT - 1) / kT), kT, (size_t)2 * (g.T + 1) * kT * sizeof(R), s>>>(g, ta);
  lc.launched(KID_SCALE);
  cur = w[nx];
  nx ^= 1;
  for (int d = 0; d < g.D; ++d) {
    const bool last = d == g.D - 1;
    fft_axis<R, true>(g, G, d, fp, cur, last ? dst : w[nx], last ? accum : nullptr, s, lc);
    cur = w[nx];
    nx ^= 1;
  }
}

}  // namespace

bool fast_poisson_supported(const Geo& g, size_t word) {
  const int threads = word == 4 ? time_threads<float>() : time_threads<double>();
  if ((size_t)2 * (g.T + 1) * threads * word > (size_t)kMaxSmem) return false;
  for (int d = 0; d < g.D; ++d)
    if ((word == 4 ? fft_smem<float>(g.N[d], 1) : fft_smem<double>(g.N[d], 1)) > (size_t)kMaxSmem) return false;
  return true;
}

void launch_fast_poisson(const Geo& g, int G, const FastPoisson<float>& fp, const float* src, float* dst,
                         float2* accum, cudaStream_t s, LaunchCounter lc) {
  fast_poisson<float>(g, G, fp, src, dst, accum, s, lc);
}
void launch_fast_poisson(const Geo& g, int G, const FastPoisson<double>& fp, const double* src, double* dst,
                         cudaStream_t s, LaunchCounter lc) {
  fast_poisson<double>(g, G, fp, src, dst, nullptr, s, lc);
}

}  // namespace dot
