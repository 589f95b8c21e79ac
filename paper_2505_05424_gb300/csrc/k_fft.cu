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
// (p - 1 multiply-adds per output; 508 = 4 x 127 points 107 us per pass of 508^2 x 32, the
// dense tensor-core passes 76 and their two time passes 46 each).  Fields keep their natural layout: a CTA takes NP
// pairs of sequences, neighbouring columns of a strided axis (or pairs of rows of the
// innermost one), stored with the pair index fastest, so that every stage reads and
// writes shared memory without bank conflicts.
//
// Time solve.  Eliminated downwards without subtraction: with a = 1/h_0^2 and pivots
// d_i = a + s_i, s_i = lambda + a s_{i-1} / d_{i-1}, every s_i is a sum of positive terms,
// accurate to a few ulps for the smallest lambda.  The column lambda = 0 is singular:
// its mean is removed from b and from x (the zero mode of the DCT), in FP64.
//
// FP32 (every iteration of the mixed path): each pass reads and writes the field once,
// from L2 up to about 4 M nodes; a dense transform on the tensor cores in 3xTF32 needs
// 256 multiply-adds per element in three passes and a table stream per CTA, and two
// passes along time.  256^2 x 64, per iteration: 4 x 16.3 + 18.5 us (tensor cores
// 4 x 25.4 + 2 x 23.6); 1024^2 x 32: 4 x 115 + 62 (4 x 396 + 2 x 162); 64^3 x 32:
// 6 x 20.2 + 20.7 (6 x 30 + 2 x 54); 150 x 117 x 37, where the dense transform ran on
// the FP32 units: 2 x 14.8 + 20.7 (k_xtx; 4 x 22 + 19).  A cold solve's error is 2 to 5 times
// smaller than the 3xTF32 one's.
//
// FP64: GB300 issues two FP64 lanes per SM and clock, so the count of operations is the
// time: 17 per element and axis here against 256 multiply-adds of a dense 256-point
// transform.  256^2 x 64, per iteration: four axis passes of 141 us and the time solve
// of 115 us (a dense transform: six passes of 1,789 us and 84 us of scaling);
// 37 x 21 x 50 x 20: 45 and 25 us (159 and 23).
#include <cmath>
#include <cstring>
#include <type_traits>

#include "dot_fft.cuh"
#include "dot_mixed.cuh"
#include "ffloat.cuh"

namespace dot {

namespace {

template <class R>
void fill_tables(int N, R* t) {
  const double pi = 3.14159265358979323846;
  for (int j = 0; j < N; ++j) {
    const double w = 2.0 * pi * j / N, h = pi * j / (2.0 * N), ch = std::cos(h), sh = std::sin(h);
    const double fo = (j == 0 ? std::sqrt(1.0 / N) : std::sqrt(2.0 / N)) / 2.0;
    const double in = j == 0 ? std::sqrt(1.0 / N) : std::sqrt(1.0 / (2.0 * N));
    t[2 * j] = (R)std::cos(w);
    t[2 * j + 1] = (R)-std::sin(w);
    t[2 * (N + j)] = (R)(fo * ch);
    t[2 * (N + j) + 1] = (R)(fo * sh);
    t[2 * (2 * N + j)] = (R)(in * ch);
    t[2 * (2 * N + j) + 1] = (R)(in * sh);
  }
}

}  // namespace

std::vector<double> fft_tables_host(int N) {
  std::vector<double> t((size_t)6 * N);
  fill_tables(N, t.data());
  return t;
}
void fft_tables_fill(int N, float* out) { fill_tables(N, out); }

namespace {

constexpr int kThreads = 256;
constexpr int kMaxStages = 16;
constexpr int kMaxSmem = 220 * 1024;

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
  // inner == 1: the frequency side is not the field's layout but W[slot][k / 2][row][k % 2],
  // the layout of k_xtx (forward: of dst, inverse: of src); rows of a slot
  int rot, slot_rows;
  FastDiv fslot;          // division by the pairs of a slot
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

// The pairs of sequences a CTA holds, stored pair by pair at each position with an odd
// pitch: a number known at compile time, or any.
template <int NP>
struct FixedPairs {
  static constexpr int kThreads = 256;
  __device__ __forceinline__ int count() const { return NP; }
  __device__ __forceinline__ int pitch() const { return NP + 1; }
  __device__ __forceinline__ int split(int e, int* pr) const {   // e = rest * count + pair
    *pr = e % NP;
    return e / NP;
  }
};
struct AnyPairs {
  static constexpr int kThreads = 512;
  int n;
  FastDiv f;
  __device__ __forceinline__ int count() const { return n; }
  __device__ __forceinline__ int pitch() const { return n | 1; }
  __device__ __forceinline__ int split(int e, int* pr) const {
    const int b = (int)fdiv((unsigned)e, f);
    *pr = e - b * n;
    return b;
  }
};

// One Stockham stage of radix RAD with stride s: butterfly b = p s + q reads elements
// b + (N / RAD) j and writes q + s (RAD p + k), times exp(-2 pi i s p k / N).
template <int RAD, bool INV, class Q, class V>
__device__ __forceinline__ void stage(const Q& np, const V* src, V* dst, const V* tw, int N, int s, FastDiv fs) {
  const int kPitch = np.pitch();
  const int nb = N / RAD;
  for (int e = threadIdx.x; e < nb * np.count(); e += Q::kThreads) {
    int pr;
    const int b = np.split(e, &pr);
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
// input pairs, sum_j (x_j + x_{r-j}) cos and (x_j - x_{r-j}) sin.  KB > 1: the pairs are
// formed in their places first, and a thread runs over them for KB values of k, so that a
// pair is read once for KB outputs and their conjugates.  KB = 1: a thread forms them
// itself, for axes too short to give every thread more than one output.
template <int KB, bool INV, class Q, class V>
__device__ __forceinline__ void stage_any(const Q& np, V* src, V* dst, const V* tw, int N, int r, int s, FastDiv fs,
                                          FastDiv fr) {
  const int kPitch = np.pitch();
  const int nb = N / r, hk = (r + 1) / 2, step = nb * kPitch;
  // x_j + x_{r-j}, and i (x_j - x_{r-j}) (forward), which times sin adds to the sum
  auto pair = [](V* a, V* c) {
    const V x = *a, y = *c;
    *a = cadd(x, y);
    *c = rot<!INV>(csub(x, y));
  };
  if constexpr (KB > 1) {
    for (int e = threadIdx.x; e < nb * (hk - 1) * np.count(); e += Q::kThreads) {
      int pr;
      const int bj = np.split(e, &pr);
      const int j = (int)fdiv((unsigned)bj, fr), b = bj - j * nb;
      pair(src + (b + nb * (j + 1)) * kPitch + pr, src + (b + nb * (r - 1 - j)) * kPitch + pr);
    }
    __syncthreads();
  }
  const int nk = (hk + KB - 1) / KB;
  for (int e = threadIdx.x; e < nb * nk * np.count(); e += Q::kThreads) {
    int pr;
    const int bk = np.split(e, &pr);
    const int kb = (int)fdiv((unsigned)bk, fr), b = bk - kb * nb;
    const int p = (int)fdiv((unsigned)b, fs), q = b - p * s;
    const V* x = src + b * kPitch + pr;
    const V *xs = x, *xd = x + r * step;
    V re[KB], im[KB];
    int m[KB], dm[KB];                     // j k mod r, in units of N / r
    re[0] = x[0];
    im[0] = mk<V>(re[0].x - re[0].x, re[0].y - re[0].y);
#pragma unroll
    for (int i = 0; i < KB; ++i) {
      re[i] = re[0];
      im[i] = im[0];
      m[i] = 0;
      dm[i] = min(kb * KB + i, hk - 1) * nb;
    }
#pragma unroll 4
    for (int j = 1; j < hk; ++j) {
      xs += step;
      xd -= step;
      V sm = *xs, df = *xd;
      if constexpr (KB == 1) pair(&sm, &df);
#pragma unroll
      for (int i = 0; i < KB; ++i) {
        m[i] += dm[i];
        if (m[i] >= N) m[i] -= N;
        const V w = tw[m[i]];
        re[i] = mk<V>(re[i].x + sm.x * w.x, re[i].y + sm.y * w.x);
        im[i] = mk<V>(im[i].x + df.x * w.y, im[i].y + df.y * w.y);   // w.y = -sin (forward)
      }
    }
    V* o = dst + (q + s * r * p) * kPitch + pr;
#pragma unroll
    for (int i = 0; i < KB; ++i) {
      const int k = kb * KB + i;
      if (k >= hk) break;
      V y = cadd(re[i], im[i]);
      if (k && nb > s) y = cmulw<INV>(y, tw[s * p * k]);
      o[s * k * kPitch] = y;
      if (k) {
        V z = csub(re[i], im[i]);
        if (nb > s) z = cmulw<INV>(z, tw[s * p * (r - k)]);
        o[s * (r - k) * kPitch] = z;
      }
    }
  }
}

// All stages; returns the buffer that holds the result.
template <bool INV, int KB, class Q, class V>
__device__ __forceinline__ V* transform(const Q& np, V* a, V* b, const V* tw, const FftPlan& pl) {
  int s = 1;
  for (int i = 0; i < pl.nst; ++i) {
    const int r = pl.rad[i];
    switch (r) {
      case 8: stage<8, INV>(np, a, b, tw, pl.N, s, pl.fs[i]); break;
      case 4: stage<4, INV>(np, a, b, tw, pl.N, s, pl.fs[i]); break;
      case 2: stage<2, INV>(np, a, b, tw, pl.N, s, pl.fs[i]); break;
      case 3: stage<3, INV>(np, a, b, tw, pl.N, s, pl.fs[i]); break;
      case 5: stage<5, INV>(np, a, b, tw, pl.N, s, pl.fs[i]); break;
      default: stage_any<KB, INV>(np, a, b, tw, pl.N, r, s, pl.fs[i], pl.fr[i]); break;
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

// Four neighbouring values (16-byte aligned rows), read-only for the kernel's lifetime.
__device__ __forceinline__ void load4(const float* p, float* v) {
  const float4 t = __ldg(reinterpret_cast<const float4*>(p));
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load4(const double* p, double* v) {
  const double2 t = __ldg(reinterpret_cast<const double2*>(p)), u = __ldg(reinterpret_cast<const double2*>(p) + 1);
  v[0] = t.x; v[1] = t.y; v[2] = u.x; v[3] = u.y;
}
__device__ __forceinline__ void store4(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(double* p, const double* v) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}
// accum[i .. i + 3] += v, the old values in old (loaded ahead)
__device__ __forceinline__ void load_old(const float2* accum, long long i, float4* old) {
  old[0] = reinterpret_cast<const float4*>(accum + i)[0];
  old[1] = reinterpret_cast<const float4*>(accum + i)[1];
}
__device__ __forceinline__ void add4(float2* accum, long long i, const float4* old, const float* v) {
  const float2 a = ff_add_f(make_float2(old[0].x, old[0].y), v[0]), b = ff_add_f(make_float2(old[0].z, old[0].w), v[1]);
  const float2 c = ff_add_f(make_float2(old[1].x, old[1].y), v[2]), d = ff_add_f(make_float2(old[1].z, old[1].w), v[3]);
  reinterpret_cast<float4*>(accum + i)[0] = make_float4(a.x, a.y, b.x, b.y);
  reinterpret_cast<float4*>(accum + i)[1] = make_float4(c.x, c.y, d.x, d.y);
}

// Z[k] = V_a[k] + i V_b[k] of the inverse transform from X[k], X[N - k] of both sequences:
// V_a = (c ak + s am) + i (s ak - c am)
template <class V>
__device__ __forceinline__ V zk(V w, V xk, V xm) {
  return mk<V>((w.x * xk.x + w.y * xm.x) - (w.y * xk.y - w.x * xm.y),
               (w.y * xk.x - w.x * xm.x) + (w.x * xk.y + w.y * xm.y));
}
// (X_a[k], X_b[k]) from Z[k], Z[N - k]: X_a = c (zr + mr) + s (zi - mi),
// X_b = c (zi + mi) + s (mr - zr)
template <class V>
__device__ __forceinline__ V xk_of(V w, V z, V y) {
  return mk<V>(w.x * (z.x + y.x) + w.y * (z.y - y.y), w.x * (z.y + y.y) - w.y * (z.x - y.x));
}

// Element (pair kp of frequencies) of the first row of row pair pg in W.
template <class R>
__device__ __forceinline__ long long rot_at(const FftArgs<R>& a, long long pg, int kp) {
  const int z = (int)fdiv((unsigned)pg, a.fslot);
  const long long row = 2 * (pg - (long long)z * a.fslot.d);
  return ((long long)z * ((a.plan.N + 1) / 2) + kp) * a.slot_rows + row;
}

// Frequencies 2 kp, 2 kp + 1 of row pair pg: out of Z (forward) into W, or from W (inverse)
// into the raw spectrum B.
template <class R, class V>
__device__ __forceinline__ void rot_store(const FftArgs<R>& a, long long pg, int kp, const V* rotf, const V* Z, int pitch,
                                          int pr) {
  const int N = a.plan.N, k = 2 * kp;
  const V x = xk_of(rotf[k], Z[k * pitch + pr], Z[(k ? N - k : 0) * pitch + pr]);
  V y = mk<V>((R)0, (R)0);
  if (k + 1 < N) y = xk_of(rotf[k + 1], Z[(k + 1) * pitch + pr], Z[(N - k - 1) * pitch + pr]);
  if (2 * pg >= a.nseq) return;
  V* w = reinterpret_cast<V*>(a.dst) + rot_at(a, pg, kp);
  w[0] = mk<V>(x.x, y.x);
  if (2 * pg + 1 < a.nseq) w[1] = mk<V>(x.y, y.y);
}
template <class R, class V>
__device__ __forceinline__ void rot_load(const FftArgs<R>& a, long long pg, int kp, V* va, V* vb) {
  *va = *vb = mk<V>((R)0, (R)0);
  if (2 * pg >= a.nseq) return;
  const V* w = reinterpret_cast<const V*>(a.src) + rot_at(a, pg, kp);
  *va = __ldg(w);
  if (2 * pg + 1 < a.nseq) *vb = __ldg(w + 1);
}

// Whether any slot of the pairs [p0, p0 + np) holds a solve.
template <class R>
__device__ __forceinline__ bool any_active(const FftArgs<R>& a, long long p0, int np) {
  if (!a.sp) return true;
  const long long last = min(p0 + np, a.npair) - 1;
  bool on = false;
  for (long long b = p0 / a.slot_pairs; b <= last / a.slot_pairs; ++b) on = on || a.sp[b].active;
  return on;
}

// A pair of neighbouring columns of a strided axis, in 8-byte (FP64: 16) accesses where
// the rows are even.
template <class R>
struct Columns {
  using V = typename Vec2<R>::type;
  const FftArgs<R>& a;
  bool ok, two, vec;
  long long base;
  __device__ __forceinline__ Columns(const FftArgs<R>& args, long long pg) : a(args) {
    ok = pg < a.npair;
    const long long o = ok ? (long long)fdiv((unsigned)pg, a.fpi) : 0;
    const int ci = ok ? 2 * (int)(pg - o * a.pin) : 0;
    two = ok && ci + 1 < a.inner;
    vec = a.inner % 2 == 0;
    base = o * a.plan.N * a.inner + ci;
  }
  __device__ __forceinline__ V get(int j) const {
    if (!ok) return mk<V>((R)0, (R)0);
    const R* s = a.src + base + (long long)j * a.inner;
    if (vec) return __ldg(reinterpret_cast<const V*>(s));
    return mk<V>(__ldg(s), two ? __ldg(s + 1) : (R)0);
  }
  __device__ __forceinline__ void set(int j, V v) const {
    const long long i = base + (long long)j * a.inner;
    if (vec && !a.accum) {
      *reinterpret_cast<V*>(a.dst + i) = v;
    } else {
      put(a.dst, a.accum, i, v.x);
      if (two) put(a.dst, a.accum, i + 1, v.y);
    }
  }
};

// The DCT-II (INV false) or DCT-III of NP pairs of sequences of any length; KB as in
// stage_any.
template <class R, int NP, bool INV, int KB>
__global__ void __launch_bounds__(kThreads) k_dct_any(const __grid_constant__ FftArgs<R> a) {
  using V = typename Vec2<R>::type;
  constexpr int kPitch = NP + 1;
  extern __shared__ __align__(16) unsigned char fsm[];
  const int N = a.plan.N;
  V* A = reinterpret_cast<V*>(fsm);
  V* B = A + N * kPitch;
  V* tw = B + N * kPitch;
  const long long p0 = (long long)blockIdx.x * NP;
  if (!any_active(a, p0, NP)) return;
  const V* rotf = a.tab + (INV ? 2 : 1) * N;
  for (int j = threadIdx.x; j < N; j += kThreads) tw[j] = a.tab[j];
  const V zero = mk<V>((R)0, (R)0);
  if (a.inner > 1) {
    // a thread keeps its pair of columns
    constexpr int kStep = kThreads / NP;
    const int pr = threadIdx.x % NP, j0 = threadIdx.x / NP;
    const Columns<R> c(a, p0 + pr);
    if (!INV) {
#pragma unroll 4
      for (int j = j0; j < N; j += kStep) A[((j & 1) ? N - 1 - (j >> 1) : j >> 1) * kPitch + pr] = c.get(j);
    } else {
#pragma unroll 2
      for (int k = j0; k <= N / 2; k += kStep) {
        const int m = N - k;
        const V xk = c.get(k), xm = k ? c.get(m) : zero;
        A[k * kPitch + pr] = zk(rotf[k], xk, xm);
        if (k && m != k) A[m * kPitch + pr] = zk(rotf[m], xm, xk);
      }
    }
    __syncthreads();
    const V* Z = transform<INV, KB>(FixedPairs<NP>(), A, B, tw, a.plan);
    if (!c.ok) return;
    if (!INV) {
#pragma unroll 2
      for (int k = j0; k <= N / 2; k += kStep) {
        const int m = k ? N - k : 0;
        const V z = Z[k * kPitch + pr], y = Z[m * kPitch + pr];
        c.set(k, xk_of(rotf[k], z, y));
        if (k && m != k) c.set(m, xk_of(rotf[m], y, z));
      }
    } else {
#pragma unroll 4
      for (int j = j0; j < N; j += kStep) c.set(j, Z[((j & 1) ? N - 1 - (j >> 1) : j >> 1) * kPitch + pr]);
    }
  } else {
    // pairs of contiguous rows: neighbouring threads take neighbouring elements
    const int nk = (N + 1) / 2;
    if (INV && a.rot) {
#pragma unroll 4
      for (int e = threadIdx.x; e < NP * nk; e += kThreads) {
        const int pr = e % NP, kp = e / NP;
        V va, vb;
        rot_load(a, p0 + pr, kp, &va, &vb);
        B[2 * kp * kPitch + pr] = mk<V>(va.x, vb.x);
        if (2 * kp + 1 < N) B[(2 * kp + 1) * kPitch + pr] = mk<V>(va.y, vb.y);
      }
    } else {
#pragma unroll 4
      for (int e = threadIdx.x; e < NP * N; e += kThreads) {
        const int pr = (int)fdiv((unsigned)e, a.plan.fN), j = e - pr * N;
        const long long row = 2 * (p0 + pr);
        const R* s = a.src + row * N + j;
        const V v = mk<V>(row < a.nseq ? __ldg(s) : (R)0, row + 1 < a.nseq ? __ldg(s + N) : (R)0);
        if (INV) B[j * kPitch + pr] = v;
        else A[((j & 1) ? N - 1 - (j >> 1) : j >> 1) * kPitch + pr] = v;
      }
    }
    __syncthreads();
    if (INV) {
      for (int e = threadIdx.x; e < NP * (N / 2 + 1); e += kThreads) {
        const int pr = e % NP, k = e / NP, m = N - k;
        const V xk = B[k * kPitch + pr], xm = k ? B[m * kPitch + pr] : zero;
        A[k * kPitch + pr] = zk(rotf[k], xk, xm);
        if (k && m != k) A[m * kPitch + pr] = zk(rotf[m], xm, xk);
      }
      __syncthreads();
    }
    const V* Z = transform<INV, KB>(FixedPairs<NP>(), A, B, tw, a.plan);
    if (!INV && a.rot) {
      for (int e = threadIdx.x; e < NP * nk; e += kThreads) rot_store(a, p0 + e % NP, e / NP, rotf, Z, kPitch, e % NP);
      return;
    }
    const int np = (int)min((long long)NP, a.npair - p0);
#pragma unroll 4
    for (int e = threadIdx.x; e < np * N; e += kThreads) {
      const int pr = (int)fdiv((unsigned)e, a.plan.fN), k = e - pr * N;
      const long long row = 2 * (p0 + pr);
      const V x = INV ? Z[((k & 1) ? N - 1 - (k >> 1) : k >> 1) * kPitch + pr]
                      : xk_of(rotf[k], Z[k * kPitch + pr], Z[(k ? N - k : 0) * kPitch + pr]);
      put(a.dst, a.accum, row * N + k, x.x);
      if (row + 1 < a.nseq) put(a.dst, a.accum, (row + 1) * N + k, x.y);
    }
  }
}

// ---- power-of-two axes ------------------------------------------------------------
//
// The same transform with the length known at compile time: a thread holds sixteen
// complex elements in registers and runs a radix-16 butterfly (then radix 2 .. 16 ones on
// the rest), in place in shared memory; the columns of a strided axis enter the first
// butterfly (forward) and leave the last one (inverse) without passing through it.

// w_16^m, m = 1, 2, 3, 4, 6, 9 (conjugated for the inverse)
template <bool INV, int M, class V>
__device__ __forceinline__ V mul16(V a) {
  using S = std::remove_reference_t<decltype(a.x)>;
  const S c = (S)0.92387953251128675613, s = (S)0.38268343236508977173, h = (S)0.70710678118654752440;
  if constexpr (M == 1) return cmulw<INV>(a, mk<V>(c, -s));
  else if constexpr (M == 2) { const V r = rot<INV>(a); return mk<V>(h * (a.x + r.x), h * (a.y + r.y)); }
  else if constexpr (M == 3) return cmulw<INV>(a, mk<V>(s, -c));
  else if constexpr (M == 4) return rot<INV>(a);
  else if constexpr (M == 6) { const V r = rot<INV>(a); return mk<V>(h * (r.x - a.x), h * (r.y - a.y)); }
  else return cmulw<INV>(a, mk<V>(-c, s));
}
// Output k + 4 l of the 16-point DFT ends in x[4 k + l].
template <bool INV, class V>
__device__ __forceinline__ void dft16(V* x) {
#pragma unroll
  for (int j = 0; j < 4; ++j) dft4<INV>(x[j], x[j + 4], x[j + 8], x[j + 12]);
  x[5] = mul16<INV, 1>(x[5]);
  x[6] = mul16<INV, 2>(x[6]);
  x[7] = mul16<INV, 3>(x[7]);
  x[9] = mul16<INV, 2>(x[9]);
  x[10] = mul16<INV, 4>(x[10]);
  x[11] = mul16<INV, 6>(x[11]);
  x[13] = mul16<INV, 3>(x[13]);
  x[14] = mul16<INV, 6>(x[14]);
  x[15] = mul16<INV, 9>(x[15]);
#pragma unroll
  for (int k = 0; k < 4; ++k) dft4<INV>(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
}
// register of output k of a RAD-point DFT
template <int RAD>
__device__ __forceinline__ constexpr int reg_of(int k) { return RAD == 16 ? 4 * (k % 4) + k / 4 : k; }

template <int N, int NP>
struct Pow2 {
  static constexpr int kThreads = N / 16 * NP;   // a radix-16 butterfly each
  // radix of the stage that starts at stride S
  static constexpr int radix(int S) {
    const int rest = N / S;
    return S == 1 ? 16 : rest <= 16 ? rest : 8;
  }
};

// The stage at stride S on the thread's registers x: 16 / RAD butterflies, bb = b + i kNb.
template <int N, int NP, int S, bool INV, class V>
__device__ __forceinline__ void p2_compute(V* x, int b, const V* tw) {
  constexpr int RAD = Pow2<N, NP>::radix(S), kNb = N / 16;
#pragma unroll
  for (int i = 0; i < 16 / RAD; ++i) {
    V* y = x + i * RAD;
    if constexpr (RAD == 16) dft16<INV>(y);
    else dft<RAD, INV>(y);
    if constexpr (S * RAD < N) {
      const int p = (b + i * kNb) / S;
#pragma unroll
      for (int k = 1; k < RAD; ++k) y[reg_of<RAD>(k)] = cmulw<INV>(y[reg_of<RAD>(k)], tw[S * p * k]);
    }
  }
}
template <int N, int NP, int S, class V>
__device__ __forceinline__ void p2_read(V* x, const V* A, int b, int pr) {
  constexpr int RAD = Pow2<N, NP>::radix(S), kNb = N / 16, kPitch = NP + 1;
#pragma unroll
  for (int i = 0; i < 16 / RAD; ++i)
#pragma unroll
    for (int j = 0; j < RAD; ++j) x[i * RAD + j] = A[(b + i * kNb + (N / RAD) * j) * kPitch + pr];
}
// position of output k of butterfly bb
template <int S, int RAD>
__device__ __forceinline__ int p2_pos(int bb, int k) { return bb % S + S * (RAD * (bb / S) + k); }
template <int N, int NP, int S, class V>
__device__ __forceinline__ void p2_write(const V* x, V* A, int b, int pr) {
  constexpr int RAD = Pow2<N, NP>::radix(S), kNb = N / 16, kPitch = NP + 1;
#pragma unroll
  for (int i = 0; i < 16 / RAD; ++i)
#pragma unroll
    for (int k = 0; k < RAD; ++k) A[p2_pos<S, RAD>(b + i * kNb, k) * kPitch + pr] = x[i * RAD + reg_of<RAD>(k)];
}
// Stages from stride S to the end; the last one leaves its results in x when KEEP.
template <int N, int NP, int S, bool INV, bool KEEP, class V>
__device__ __forceinline__ void p2_stages(V* x, V* A, const V* tw, int b, int pr) {
  constexpr int RAD = Pow2<N, NP>::radix(S);
  p2_read<N, NP, S>(x, A, b, pr);
  p2_compute<N, NP, S, INV>(x, b, tw);
  if constexpr (S * RAD < N) {
    __syncthreads();
    p2_write<N, NP, S>(x, A, b, pr);
    __syncthreads();
    p2_stages<N, NP, S * RAD, INV, KEEP>(x, A, tw, b, pr);
  } else if constexpr (!KEEP) {
    __syncthreads();
    p2_write<N, NP, S>(x, A, b, pr);
    __syncthreads();
  }
}
template <int N, int NP>
__host__ __device__ constexpr int p2_last() {   // stride of the last stage
  int S = 1;
  while (S * Pow2<N, NP>::radix(S) < N) S *= Pow2<N, NP>::radix(S);
  return S;
}

template <class R, int N, int NP, bool INV, bool ROWS>
__global__ void __launch_bounds__(Pow2<N, NP>::kThreads) k_dct_pow2(const __grid_constant__ FftArgs<R> a) {
  using V = typename Vec2<R>::type;
  constexpr int kPitch = NP + 1, kNb = N / 16, kT = Pow2<N, NP>::kThreads;
  extern __shared__ __align__(16) unsigned char fsm[];
  V* A = reinterpret_cast<V*>(fsm);
  V* tw = A + N * kPitch;
  const long long p0 = (long long)blockIdx.x * NP;
  if (!any_active(a, p0, NP)) return;
  const V* rotf = a.tab + (INV ? 2 : 1) * N;
  const int tid = threadIdx.x, pr = tid % NP, b = tid / NP;
  for (int j = tid; j < N; j += kT) tw[j] = __ldg(a.tab + j);
  V x[16];
  const V zero = mk<V>((R)0, (R)0);
  if constexpr (!ROWS) {
    const Columns<R> c(a, p0 + pr);
    if constexpr (!INV) {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int n = b + kNb * j;
        x[j] = c.get(j < 8 ? 2 * n : 2 * (N - n) - 1);
      }
      __syncthreads();   // tw
      p2_compute<N, NP, 1, INV>(x, b, tw);
      p2_write<N, NP, 1>(x, A, b, pr);
      __syncthreads();
      if constexpr (N > 16) p2_stages<N, NP, 16, INV, false>(x, A, tw, b, pr);
      if (!c.ok) return;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k = b + kNb * i, m = k ? N - k : N / 2;
        const V z = A[k * kPitch + pr], y = A[m * kPitch + pr];
        c.set(k, xk_of(__ldg(rotf + k), z, k ? y : z));
        c.set(m, xk_of(__ldg(rotf + m), y, k ? z : y));
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k = b + kNb * i, m = k ? N - k : N / 2;
        x[2 * i] = c.get(k);
        x[2 * i + 1] = c.get(m);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k = b + kNb * i, m = k ? N - k : N / 2;
        A[k * kPitch + pr] = zk(__ldg(rotf + k), x[2 * i], k ? x[2 * i + 1] : zero);
        A[m * kPitch + pr] = zk(__ldg(rotf + m), x[2 * i + 1], k ? x[2 * i] : x[2 * i + 1]);
      }
      __syncthreads();
      p2_stages<N, NP, 1, INV, true>(x, A, tw, b, pr);
      if (!c.ok) return;
      constexpr int S = p2_last<N, NP>(), RAD = N / S;
#pragma unroll
      for (int i = 0; i < 16 / RAD; ++i)
#pragma unroll
        for (int k = 0; k < RAD; ++k) {
          const int n = p2_pos<S, RAD>(b + i * kNb, k);
          c.set(n < N / 2 ? 2 * n : 2 * (N - n) - 1, x[i * RAD + reg_of<RAD>(k)]);
        }
    }
  } else {
    // pairs of contiguous rows, four neighbouring elements of both per thread and step
    constexpr int kQ = N / 4, kIt = 4;                 // kT kIt chunks in all
    static_assert(kT * kIt == NP * kQ, "four chunks per thread");
    if (INV && a.rot) {
      V wa[8], wb[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) rot_load(a, p0 + pr, b + u * kNb, &wa[u], &wb[u]);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = 2 * (b + u * kNb);
        A[k * kPitch + pr] = mk<V>(wa[u].x, wb[u].x);
        A[(k + 1) * kPitch + pr] = mk<V>(wa[u].y, wb[u].y);
      }
    } else {
    R va[kIt][4], vb[kIt][4];
#pragma unroll
    for (int u = 0; u < kIt; ++u) {
      const int e = tid + u * kT, j = 4 * (e % kQ);
      const long long row = 2 * (p0 + e / kQ);
#pragma unroll
      for (int q = 0; q < 4; ++q) va[u][q] = vb[u][q] = (R)0;
      if (row < a.nseq) load4(a.src + row * N + j, va[u]);
      if (row + 1 < a.nseq) load4(a.src + (row + 1) * N + j, vb[u]);
    }
#pragma unroll
    for (int u = 0; u < kIt; ++u) {
      const int e = tid + u * kT, j = 4 * (e % kQ), r = e / kQ;
      if (!INV) {   // the reordered sequence
        V* lo = A + (j / 2) * kPitch + r;
        V* hi = A + (N - 1 - j / 2) * kPitch + r;
        lo[0] = mk<V>(va[u][0], vb[u][0]);
        hi[0] = mk<V>(va[u][1], vb[u][1]);
        lo[kPitch] = mk<V>(va[u][2], vb[u][2]);
        hi[-kPitch] = mk<V>(va[u][3], vb[u][3]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) A[(j + q) * kPitch + r] = mk<V>(va[u][q], vb[u][q]);
      }
    }
    }
    __syncthreads();
    if constexpr (INV) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {   // in place: a thread owns its pairs k, N - k
        const int k = b + kNb * i, m = k ? N - k : N / 2;
        const V xk = A[k * kPitch + pr], xm = A[m * kPitch + pr];
        A[k * kPitch + pr] = zk(__ldg(rotf + k), xk, k ? xm : zero);
        A[m * kPitch + pr] = zk(__ldg(rotf + m), xm, k ? xk : xm);
      }
      __syncthreads();
    }
    p2_stages<N, NP, 1, INV, false>(x, A, tw, b, pr);
    if (!INV && a.rot) {
#pragma unroll
      for (int u = 0; u < 8; ++u) rot_store(a, p0 + pr, b + u * kNb, rotf, A, kPitch, pr);
      return;
    }
    if constexpr (INV && sizeof(R) == 4) {
      if (a.accum) {
#pragma unroll
        for (int u = 0; u < kIt; u += 2) {
          float4 oa[2][2], ob[2][2];
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            const int e = tid + (u + v) * kT, j = 4 * (e % kQ);
            const long long row = 2 * (p0 + e / kQ);
            if (row < a.nseq) load_old(a.accum, row * N + j, oa[v]);
            if (row + 1 < a.nseq) load_old(a.accum, (row + 1) * N + j, ob[v]);
          }
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            const int e = tid + (u + v) * kT, j = 4 * (e % kQ), r = e / kQ;
            const long long row = 2 * (p0 + r);
            const V* lo = A + (j / 2) * kPitch + r;
            const V* hi = A + (N - 1 - j / 2) * kPitch + r;
            const V z[4] = {lo[0], hi[0], lo[kPitch], hi[-kPitch]};
            const float xa[4] = {z[0].x, z[1].x, z[2].x, z[3].x};
            const float xb[4] = {z[0].y, z[1].y, z[2].y, z[3].y};
            if (row < a.nseq) add4(a.accum, row * N + j, oa[v], xa);
            if (row + 1 < a.nseq) add4(a.accum, (row + 1) * N + j, ob[v], xb);
          }
        }
        return;
      }
    }
#pragma unroll
    for (int u = 0; u < kIt; ++u) {
      const int e = tid + u * kT, j = 4 * (e % kQ), r = e / kQ;
      const long long row = 2 * (p0 + r);
      R xa[4], xb[4];
      if constexpr (!INV) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int k = j + q;
          const V v = xk_of(__ldg(rotf + k), A[k * kPitch + r], A[(k ? N - k : 0) * kPitch + r]);
          xa[q] = v.x;
          xb[q] = v.y;
        }
      } else {
        const V* lo = A + (j / 2) * kPitch + r;
        const V* hi = A + (N - 1 - j / 2) * kPitch + r;
        const V v[4] = {lo[0], hi[0], lo[kPitch], hi[-kPitch]};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          xa[q] = v[q].x;
          xb[q] = v[q].y;
        }
      }
      if (row < a.nseq) store4(a.dst + row * N + j, xa);
      if (row + 1 < a.nseq) store4(a.dst + (row + 1) * N + j, xb);
    }
  }
}

// 1 / x, x > 0 and normal, to about an ulp
__device__ __forceinline__ float recip(float x) {
  const float r = rcp_approx(x);
  return fmaf(r, fmaf(-x, r, 1.f), r);
}
__device__ __forceinline__ double recip(double x) {
  double r;
  // the instruction reads and returns the upper words alone (PTX ISA): about 2^-20, which
  // two Newton steps bring to 2^-40 and to rounding
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

template <class R>
struct TimeArgs {
  const R* src;
  R* dst;
  const R* lam[kMaxD];
  R a;                 // 1 / h_0^2
  long long ncol;      // columns over all slots
  int slots;
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
__device__ void zero_column(const R* b, R* x, int M, long long P, double ia) {
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
    xs -= u * ia;
    S += (double)b[t * P] - mean;
    u += S;
  }
  const double shift = warp_sum(xs) / M;
  u = U0;
  S = S0;
  for (int t = t0; t < t1; ++t) {
    const double bt = (double)b[t * P];
    x[t * P] = (R)(-u * ia - shift);
    S += bt - mean;
    u += S;
  }
}

__device__ __forceinline__ void copy_async(uint32_t dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async(uint32_t dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// (lambda I + L_t) x = b along time, one thread per column of spatial frequencies.  The
// whole column is copied to shared memory at once while the pivots, which do not need
// it, are formed; the eliminated right-hand sides and the pivots' reciprocals stay
// there.  The first `slots` blocks take the singular columns, a warp each.
template <class R, int THREADS>
__global__ void __launch_bounds__(THREADS) k_time_solve(const __grid_constant__ Geo g,
                                                        const __grid_constant__ TimeArgs<R> ta) {
  extern __shared__ __align__(16) unsigned char fsm[];
  const long long P = g.P;
  const int M = g.T + 1;
  if ((int)blockIdx.x < ta.slots) {
    const int z = blockIdx.x;
    if (threadIdx.x < 32 && (!ta.sp || ta.sp[z].active))
      zero_column(ta.src + z * M * P, ta.dst + z * M * P, M, P, 1.0 / (double)ta.a);
    return;
  }
  const long long col = (long long)(blockIdx.x - ta.slots) * THREADS + threadIdx.x;
  if (col >= ta.ncol) return;
  const int slot = (int)fdiv((unsigned)col, g.fP), p = (int)(col - slot * P);
  if (p == 0 || (ta.sp && !ta.sp[slot].active)) return;
  const R* b = ta.src + slot * M * P + p;
  R* x = ta.dst + slot * M * P + p;
  R* y = reinterpret_cast<R*>(fsm) + threadIdx.x;        // y[t THREADS]
  R* rr = y + (size_t)M * THREADS;                       // 1 / d_t
  const uint32_t ys = (uint32_t)__cvta_generic_to_shared(y);
#pragma unroll 8
  for (int t = 0; t < M; ++t) copy_async(ys + t * THREADS * sizeof(R), b + t * P);
  asm volatile("cp.async.commit_group;" ::: "memory");
  R lam = (R)0;
  for (int d = 0; d < g.D; ++d) lam += ta.lam[d][coord(g, p, d)];
  const R a = ta.a;
  R s = lam, r = recip(a + s);
  rr[0] = r;
  for (int t = 1; t < M - 1; ++t) {
    s = lam + a * r * s;
    r = recip(a + s);
    rr[t * THREADS] = r;
  }
  s = lam + a * r * s;
  rr[(M - 1) * THREADS] = recip(s);
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  R yp = y[0];
#pragma unroll 8
  for (int t = 1; t < M; ++t) {
    yp = y[t * THREADS] + a * rr[(t - 1) * THREADS] * yp;
    y[t * THREADS] = yp;
  }
  R xp = yp * rr[(M - 1) * THREADS];
  x[(M - 1) * P] = xp;
#pragma unroll 8
  for (int t = M - 2; t >= 0; --t) {
    xp = (y[t * THREADS] + a * xp) * rr[t * THREADS];
    x[t * P] = xp;
  }
}

// ---- small grids (D = 2): the x transforms and the time solve in one block ------------
//
// On small grids a pass is a launch and one trip to memory and back for a few microseconds
// of work.  For a pair of y frequencies everything along x and time is independent of
// the others, so a block takes W[slot][kp] = (T + 1) x N_x pairs -- which the y pass wrote
// side by side -- and runs the x transform, the time solve of its 2 N_x columns and the
// x transform back in shared memory: three launches per solve instead of five.  Bound by
// launch, barriers and the serial time recurrence (128^2 x 32: 17 us).
struct XtxArgs {
  float2* w;              // in place
  const float2* tab;      // axis x
  const float* lam[2];    // eigenvalues along x and y
  float a;                // 1 / h_0^2
  int M, N1, rows;        // time nodes, points along y, rows of a slot
  FastDiv fN0;
  AnyPairs np;            // M pairs
  FftPlan plan;           // axis x
  const SlotParam* sp;
};

template <int KB>
__global__ void __launch_bounds__(AnyPairs::kThreads) k_xtx(const __grid_constant__ XtxArgs a) {
  using V = float2;
  constexpr int kT = AnyPairs::kThreads;
  extern __shared__ __align__(16) unsigned char fsm[];
  const int slot = blockIdx.y, kp = blockIdx.x;
  if (a.sp && !a.sp[slot].active) return;
  const int M = a.M, N = a.plan.N, pitch = a.np.pitch();
  V* A = reinterpret_cast<V*>(fsm);
  V* B = A + N * pitch;
  V* tw = B + N * pitch;
  V* W = a.w + ((long long)slot * gridDim.x + kp) * a.rows;
  for (int j = threadIdx.x; j < N; j += kT) tw[j] = __ldg(a.tab + j);
#pragma unroll 4
  for (int e = threadIdx.x; e < M * N; e += kT) {
    const int t = (int)fdiv((unsigned)e, a.fN0), x = e - t * N;
    A[((x & 1) ? N - 1 - (x >> 1) : x >> 1) * pitch + t] = W[e];
  }
  __syncthreads();
  V* Z = transform<false, KB>(a.np, A, B, tw, a.plan);
  V* Y = Z == A ? B : A;   // the free buffer
  const V* rf = a.tab + N;
  const int half = (N / 2 + 1) * M;
  for (int e = threadIdx.x; e < half; e += kT) {   // in place: a thread owns its k, N - k
    int t;
    const int k = a.np.split(e, &t), m = k ? N - k : 0;
    const V z = Z[k * pitch + t], y = Z[m * pitch + t];
    Z[k * pitch + t] = xk_of(__ldg(rf + k), z, y);
    if (k && m != k) Z[m * pitch + t] = xk_of(__ldg(rf + m), y, z);
  }
  __syncthreads();
  // the columns (k_x, lane): pivots' reciprocals in the free buffer, at the column's places
  const float c = a.a;
  if (kp == 0 && threadIdx.x >= kT - 32) {
    float* z = reinterpret_cast<float*>(Z);
    zero_column(z, reinterpret_cast<float*>(Y), M, 2LL, 1.0 / (double)c);
    __syncwarp();
    for (int t = threadIdx.x & 31; t < M; t += 32) z[2 * t] = reinterpret_cast<float*>(Y)[2 * t];
  }
  for (int e = threadIdx.x; e < 2 * N; e += kT) {
    const int k = e >> 1, l = e & 1, ky = 2 * kp + l;
    if (ky >= a.N1 || (k == 0 && ky == 0)) continue;
    const float lam = __ldg(a.lam[0] + k) + __ldg(a.lam[1] + ky);
    float* y = reinterpret_cast<float*>(Z + k * pitch) + l;
    float* rr = reinterpret_cast<float*>(Y + k * pitch) + l;
    float s = lam, r = recip(c + s), yp = y[0];
    rr[0] = r;
    for (int t = 1; t < M; ++t) {
      const float ar = c * r;
      s = lam + ar * s;
      r = recip(t < M - 1 ? c + s : s);
      yp = y[2 * t] + ar * yp;
      y[2 * t] = yp;
      rr[2 * t] = r;
    }
    float xp = yp * r;
    y[2 * (M - 1)] = xp;
#pragma unroll 4
    for (int t = M - 2; t >= 0; --t) {
      xp = (y[2 * t] + c * xp) * rr[2 * t];
      y[2 * t] = xp;
    }
  }
  __syncthreads();
  const V* ri = a.tab + 2 * N;
  for (int e = threadIdx.x; e < half; e += kT) {
    int t;
    const int k = a.np.split(e, &t), m = N - k;
    const V xk = Z[k * pitch + t], xm = k ? Z[m * pitch + t] : make_float2(0.f, 0.f);
    Z[k * pitch + t] = zk(__ldg(ri + k), xk, xm);
    if (k && m != k) Z[m * pitch + t] = zk(__ldg(ri + m), xm, xk);
  }
  __syncthreads();
  const V* X = transform<true, KB>(a.np, Z, Y, tw, a.plan);
#pragma unroll 4
  for (int e = threadIdx.x; e < M * N; e += kT) {
    const int t = (int)fdiv((unsigned)e, a.fN0), x = e - t * N;
    W[e] = X[((x & 1) ? N - 1 - (x >> 1) : x >> 1) * pitch + t];
  }
}

size_t xtx_smem(const Geo& g) { return ((size_t)2 * g.N[0] * ((g.T + 1) | 1) + g.N[0]) * sizeof(float2); }
// Small grids by their own size (not the batch's, whose members' results may not depend
// on it), up to the size where the passes of their own are as fast.  An iteration,
// with and without: 32^2 x 16 23.8 and 26.5 us, 64^2 x 32 37.9 and 41.5, 128^2 x 32 84.5 and
// 87.2, 150 x 117 x 37 103.0 and 105.4, 256^2 x 9 92.6 and 98.9, 512^2 x 8 243.6 and 250.7,
// 256^2 x 32 (8,448 pairs per block) 200.6 and 202.6.
bool use_xtx(const Geo& g) {
  return g.D == 2 && (long long)(g.T + 1) * g.N[0] <= 8704 && xtx_smem(g) <= (size_t)kMaxSmem;
}

template <int KB>
void launch_xtx(const XtxArgs& x, dim3 blocks, size_t smem, cudaStream_t s) {
  static std::atomic<unsigned long long> done{0};
  smem_optin((const void*)k_xtx<KB>, kMaxSmem, &done);
  k_xtx<KB><<<blocks, AnyPairs::kThreads, smem, s>>>(x);
}
// Two outputs per thread of a large odd radix where the block's rounds of such items take
// less than its rounds of single ones.
bool xtx_two(const XtxArgs& x) {
  const int r = x.plan.rad[x.plan.nst - 1], hk = (r + 1) / 2, n = x.plan.N / r * x.M, t = AnyPairs::kThreads;
  return r >= 7 && 3 * ((n * ((hk + 1) / 2) + t - 1) / t) < 2 * ((n * hk + t - 1) / t);
}

template <class R> constexpr int time_threads() { return sizeof(R) == 4 ? 128 : 64; }

template <class R>
size_t fft_smem(int N, int NP) { return (size_t)(2 * N * (NP + 1) + N) * 2 * sizeof(R); }

template <class R, int NP, bool INV, int KB>
void launch_np_kb(const FftArgs<R>& a, cudaStream_t s) {
  static std::atomic<unsigned long long> done{0};
  smem_optin((const void*)k_dct_any<R, NP, INV, KB>, kMaxSmem, &done);
  k_dct_any<R, NP, INV, KB><<<(unsigned)((a.npair + NP - 1) / NP), kThreads, fft_smem<R>(a.plan.N, NP), s>>>(a);
}
// Outputs per thread of a stage with an odd radix r (their number changes no value), each in a
// kernel of its own, as more take registers that cost other axes CTAs: two where the items of work then still
// fill half the block (FP64, which waits for its few lanes and not for the loads: a warp),
// four in FP32 from r = 64 where they fill it all, else one.  An iteration with one (every
// pair formed anew for each output), two and four: 508^2 x 32 1,398, 1,156 and 1,052 us;
// 1004^2 x 32 7,290, 5,473 and 4,802 (dense passes on the tensor cores, with the fused pass
// of then: 1,174 and 5,112); 61^3 x 16 758, 719 and 760; 127^2 x 32 120, 109 and 120;
// 61^2 x 32 44, 47 and 50; FP64 2801 x 2 x 2 8,493, 3,956 and 4,490; 37^3 x 16 944, 821 and
// 938; 19 x 23 x 20 90, 94 and -.
template <class R, int NP, bool INV>
void launch_np(const FftArgs<R>& a, cudaStream_t s) {
  const int r = a.plan.rad[a.plan.nst - 1];   // the largest odd prime factor, if there is one
  auto items = [&](int kb) { return a.plan.N / r * (((r + 1) / 2 + kb - 1) / kb) * NP; };
  if constexpr (sizeof(R) == 4) {
    if (r >= 64 && items(4) >= kThreads) return launch_np_kb<R, NP, INV, 4>(a, s);
  }
  if (r < 7 || items(2) < (sizeof(R) == 4 ? kThreads / 2 : 32)) launch_np_kb<R, NP, INV, 1>(a, s);
  else launch_np_kb<R, NP, INV, 2>(a, s);
}

template <class R, int N, int NP, bool INV, bool ROWS>
void launch_pow2(const FftArgs<R>& a, cudaStream_t s) {
  const size_t sm = (size_t)(N * (NP + 1) + N) * 2 * sizeof(R);
  static std::atomic<unsigned long long> done{0};
  smem_optin((const void*)k_dct_pow2<R, N, NP, INV, ROWS>, (int)sm, &done);
  k_dct_pow2<R, N, NP, INV, ROWS><<<(unsigned)((a.npair + NP - 1) / NP), Pow2<N, NP>::kThreads, sm, s>>>(a);
}
template <class R, int N, int NP, int NPS, bool INV>
bool try_pow2_np(const FftArgs<R>& a, cudaStream_t s) {
  const bool rows = a.inner == 1;
  if (a.npair >= (long long)NP * 152) {
    if (rows) launch_pow2<R, N, NP, INV, true>(a, s);
    else launch_pow2<R, N, NP, INV, false>(a, s);
    return true;
  }
  if constexpr (sizeof(R) == 4) {
    if (rows) launch_pow2<R, N, NPS, INV, true>(a, s);
    else launch_pow2<R, N, NPS, INV, false>(a, s);
    return true;
  }
  return false;
}
// Axes of 32 to 1024 points take the compile-time form: with many sequences 4,096
// elements per CTA, with few ones 1,024 to 2,048 for more CTAs (FP64: the general form).
// In FP32 the form may not depend on the number of solves in a batch, whose results are
// the same bit for bit whatever they are served with; the pairs per CTA change no value.
template <class R, bool INV>
bool try_pow2(const FftArgs<R>& a, cudaStream_t s) {
  constexpr bool f = sizeof(R) == 4;
  switch (a.plan.N) {
    case 32: return f && try_pow2_np<float, 32, 64, 32, INV>(reinterpret_cast<const FftArgs<float>&>(a), s);
    case 64: return try_pow2_np<R, 64, 32, 16, INV>(a, s);
    case 128: return try_pow2_np<R, 128, 16, 8, INV>(a, s);
    case 256: return try_pow2_np<R, 256, f ? 16 : 8, 8, INV>(a, s);
    case 512: return try_pow2_np<R, 512, 8, 4, INV>(a, s);
    case 1024: return try_pow2_np<R, 1024, f ? 8 : 4, 2, INV>(a, s);
    default: return false;
  }
}

// One axis of G solves.  Pairs per CTA: 16 (8 in FP64: 128-byte segments of a strided
// axis), fewer while that leaves SMs without a CTA or does not fit shared memory.
template <class R, bool INV>
void fft_axis(const Geo& g, int G, int axis, const FastPoisson<R>& fp, const R* src, R* dst, float2* accum, bool rot,
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
  a.rot = rot;
  a.slot_rows = (int)(a.nseq / G);
  a.fslot = make_fastdiv((unsigned)((a.slot_rows + 1) / 2));
  a.sp = G > 1 ? fp.sp : nullptr;
  a.slot_pairs = G > 1 ? a.npair / G : a.npair;
  if (try_pow2<R, INV>(a, s)) {
    lc.launched(KID_DCT_AXIS);
    return;
  }
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
  if constexpr (sizeof(R) == 4) {
    if (use_xtx(g)) {
      fft_axis<R, false>(g, G, 1, fp, src, fp.w1, nullptr, true, s, lc);
      XtxArgs x;
      std::memset(&x, 0, sizeof(x));
      x.w = reinterpret_cast<float2*>(fp.w1);
      x.tab = fp.tab[0];
      x.lam[0] = fp.lam[0];
      x.lam[1] = fp.lam[1];
      x.a = (float)(g.invh[0] * g.invh[0]);
      x.M = g.T + 1;
      x.N1 = g.N[1];
      x.rows = x.M * g.N[0];
      x.fN0 = make_fastdiv((unsigned)g.N[0]);
      x.np.n = x.M;
      x.np.f = make_fastdiv((unsigned)x.M);
      x.plan = make_plan(g.N[0]);
      x.sp = G > 1 ? fp.sp : nullptr;
      const dim3 blocks((g.N[1] + 1) / 2, G);
      if (xtx_two(x)) launch_xtx<2>(x, blocks, xtx_smem(g), s);
      else launch_xtx<1>(x, blocks, xtx_smem(g), s);
      lc.launched(KID_SCALE);
      fft_axis<R, true>(g, G, 1, fp, fp.w1, dst, accum, true, s, lc);
      return;
    }
  }
  R* w[2] = {fp.w1, fp.w2};
  const R* cur = src;
  int nx = 0;
  for (int d = g.D - 1; d >= 0; --d) {
    fft_axis<R, false>(g, G, d, fp, cur, w[nx], nullptr, false, s, lc);
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
  ta.slots = G;
  ta.sp = G > 1 ? fp.sp : nullptr;
  static std::atomic<unsigned long long> done{0};
  smem_optin((const void*)k_time_solve<R, kT>, kMaxSmem, &done);
  k_time_solve<R, kT><<<(unsigned)(G + (ta.ncol + kT - 1) / kT), kT, (size_t)2 * (g.T + 1) * kT * sizeof(R), s>>>(g, ta);
  lc.launched(KID_SCALE);
  cur = w[nx];
  nx ^= 1;
  for (int d = 0; d < g.D; ++d) {
    const bool last = d == g.D - 1;
    fft_axis<R, true>(g, G, d, fp, cur, last ? dst : w[nx], last ? accum : nullptr, false, s, lc);
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
