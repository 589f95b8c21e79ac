// ffloat.cuh -- two-float ("float-float") arithmetic: a value is hi + lo with
// |lo| <= ulp(hi)/2, about 48 significant bits, computed with FP32 instructions
// only.  Used for the ALM multipliers and the potential of the mixed path, whose
// per-element updates would otherwise need FP64 instructions (GB300 issues FP64
// FMA at about 1/70 of the FP32 rate).
//
// Error-free transformations: TwoSum (Knuth) and TwoProd via FMA.  No
// reassociation or contraction can change them: they contain no a*b+c patterns
// except the explicit fmaf.
#pragma once
#include <cuda_runtime.h>

namespace dot {

__device__ __forceinline__ float2 two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  const float e = (a - (s - bb)) + (b - bb);
  return make_float2(s, e);
}

// (hi, lo) renormalised so that hi = fl(hi + lo).
__device__ __forceinline__ float2 quick_two_sum(float a, float b) {
  const float s = a + b;
  const float e = b - (s - a);
  return make_float2(s, e);
}

// ff + float
__device__ __forceinline__ float2 ff_add_f(float2 a, float b) {
  float2 s = two_sum(a.x, b);
  s.y += a.y;
  return quick_two_sum(s.x, s.y);
}

// ff + ff
__device__ __forceinline__ float2 ff_add(float2 a, float2 b) {
  float2 s = two_sum(a.x, b.x);
  s.y += a.y + b.y;
  return quick_two_sum(s.x, s.y);
}

__device__ __forceinline__ float2 ff_neg(float2 a) { return make_float2(-a.x, -a.y); }

// ff * float
__device__ __forceinline__ float2 ff_mul_f(float2 a, float b) {
  const float p = a.x * b;
  float e = fmaf(a.x, b, -p);
  e = fmaf(a.y, b, e);
  return quick_two_sum(p, e);
}

// exact difference of two floats as an ff
__device__ __forceinline__ float2 ff_sub_exact(float a, float b) { return two_sum(a, -b); }

__device__ __forceinline__ double ff_to_double(float2 a) { return (double)a.x + (double)a.y; }

// exact product of two floats as an ff (TwoProd via FMA)
__device__ __forceinline__ float2 two_prod(float a, float b) {
  const float p = a * b;
  return make_float2(p, fmaf(a, b, -p));
}

// ff * ff
__device__ __forceinline__ float2 ff_mul(float2 a, float2 b) {
  const float p = a.x * b.x;
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  return quick_two_sum(p, e);
}

// a <= b for ff values
__device__ __forceinline__ bool ff_le(float2 a, float2 b) {
  return a.x < b.x || (a.x == b.x && a.y <= b.y);
}

__device__ __forceinline__ float ff_round(float2 a) { return a.x + a.y; }

// ---- packed pairs ---------------------------------------------------------
// sm_100-class GPUs execute add/sub/mul/fma on two FP32 lanes in one instruction
// (.f32x2), each lane an ordinary IEEE round-to-nearest operation.  A float2 here
// is such a lane pair; ff2 holds two two-float numbers, (h.x + l.x) and
// (h.y + l.y).  Every ff2 operation computes, lane by lane, exactly what the
// scalar operation of the same name above computes.

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 ra, rb, rc;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rc, ra, rb;\n\tmov.b64 {%0, %1}, rc;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 ra, rb, rc;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "sub.rn.f32x2 rc, ra, rb;\n\tmov.b64 {%0, %1}, rc;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 ra, rb, rc;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mul.rn.f32x2 rc, ra, rb;\n\tmov.b64 {%0, %1}, rc;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
// a * b + c, one rounding per lane
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mov.b64 rc, {%6, %7};\n\tfma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}

struct ff2 {
  float2 h, l;
};

__device__ __forceinline__ ff2 two_sum2(float2 a, float2 b) {
  const float2 s = add2(a, b);
  const float2 bb = sub2(s, a);
  const float2 e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
  return ff2{s, e};
}
__device__ __forceinline__ ff2 quick_two_sum2(float2 a, float2 b) {
  const float2 s = add2(a, b);
  return ff2{s, sub2(b, sub2(s, a))};
}
// lane-wise ff_add
__device__ __forceinline__ ff2 ff2_add(ff2 a, ff2 b) {
  ff2 s = two_sum2(a.h, b.h);
  s.l = add2(s.l, add2(a.l, b.l));
  return quick_two_sum2(s.h, s.l);
}
// lane-wise a - b: two_sum2(a, -b) without forming -b
__device__ __forceinline__ ff2 two_diff2(float2 a, float2 b) {
  const float2 s = sub2(a, b);
  const float2 bb = sub2(s, a);
  return ff2{s, sub2(sub2(a, sub2(s, bb)), add2(b, bb))};
}
// lane-wise ff_add of a and -b
__device__ __forceinline__ ff2 ff2_sub(ff2 a, ff2 b) {
  ff2 s = two_diff2(a.h, b.h);
  s.l = add2(s.l, sub2(a.l, b.l));
  return quick_two_sum2(s.h, s.l);
}
// lane-wise ff_add_f
__device__ __forceinline__ ff2 ff2_add_f(ff2 a, float2 b) {
  ff2 s = two_sum2(a.h, b);
  s.l = add2(s.l, a.l);
  return quick_two_sum2(s.h, s.l);
}
// lane-wise two_prod: the rounding error of each product by one FMA
__device__ __forceinline__ ff2 two_prod2(float2 a, float2 b) {
  const float2 p = mul2(a, b);
  return ff2{p, make_float2(fmaf(a.x, b.x, -p.x), fmaf(a.y, b.y, -p.y))};
}
// the two lanes of an ff2 as scalar two-floats, and back
__device__ __forceinline__ float2 ff2_lane0(ff2 a) { return make_float2(a.h.x, a.l.x); }
__device__ __forceinline__ float2 ff2_lane1(ff2 a) { return make_float2(a.h.y, a.l.y); }
__device__ __forceinline__ ff2 ff2_pack(float2 a, float2 b) {
  return ff2{make_float2(a.x, b.x), make_float2(a.y, b.y)};
}

// ---- cheaper forms used by the fused cone kernel ----------------------------

// ff / float given r ~ 1/b (a few ulps suffice): FP32 quotient a.x * r plus one
// correction from the exact remainder.
__device__ __forceinline__ float2 ff_div_f_r(float2 a, float b, float r) {
  const float q1 = a.x * r;
  const float2 p = two_prod(q1, b);
  const float rem = ((a.x - p.x) - p.y) + a.y;
  return quick_two_sum(q1, rem * r);
}

// sqrt of a non-negative ff from the FP32 reciprocal square root: s = a r with
// r ~ 1/sqrt(a), then one Newton correction (a - s^2) r / 2 from the exact square,
// accurate to ~2^-44 relative.  *rinv receives r (~1/sqrt(a) to a few ulps).
__device__ __forceinline__ float2 ff_sqrt_r(float2 a, float* rinv) {
  if (!(a.x > 0.f)) {
    *rinv = 0.f;
    return make_float2(0.f, 0.f);
  }
  const float r = rsqrtf(a.x);
  const float s = a.x * r;
  const float2 s2 = two_prod(s, s);
  const float rem = ((a.x - s2.x) - s2.y) + a.y;
  *rinv = r;
  return quick_two_sum(s, rem * (0.5f * r));
}

// 1/x to about one ulp (normal x)
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Running sum of two-float terms with one normalisation at the end: the high parts
// are added by TwoSum (each rounding error kept exactly), the low parts and those
// errors in one FP32 correction.  Same accuracy class as a chain of ff_add.
struct ff_acc {
  float h, c;
};
__device__ __forceinline__ ff_acc acc_init(float2 a) { return ff_acc{a.x, a.y}; }
__device__ __forceinline__ void acc_add(ff_acc& s, float2 b) {
  const float2 t = two_sum(s.h, b.x);
  s.h = t.x;
  s.c += t.y + b.y;
}
__device__ __forceinline__ void acc_add_f(ff_acc& s, float b) {
  const float2 t = two_sum(s.h, b);
  s.h = t.x;
  s.c += t.y;
}
// + b * x for a two-float b and an FP32 x: the exact product of the high part by
// TwoProd, the low part's product into the correction
__device__ __forceinline__ void acc_add_mul(ff_acc& s, float2 b, float x) {
  const float p = b.x * x;
  const float e = fmaf(b.y, x, fmaf(b.x, x, -p));
  const float2 t = two_sum(s.h, p);
  s.h = t.x;
  s.c += t.y + e;
}
__device__ __forceinline__ float2 acc_get(const ff_acc& s) { return quick_two_sum(s.h, s.c); }

// (b - a) invh for two two-float values, as an unevaluated pair: the difference of
// the high parts by TwoSum
__device__ __forceinline__ float2 ff_grad(float2 a, float2 b, float invh) {
  const float2 dh = two_sum(b.x, -a.x);
  const float dl = (b.y - a.y) + dh.y;
  return make_float2(dh.x * invh, dl * invh);
}
// ff_acc in two lanes
struct ff2_acc {
  float2 h, c;
};
__device__ __forceinline__ void acc2_add(ff2_acc& s, ff2 b) {
  const ff2 t = two_sum2(s.h, b.h);
  s.h = t.h;
  s.c = add2(s.c, add2(t.l, b.l));
}
__device__ __forceinline__ void acc2_add_f(ff2_acc& s, float2 b) {
  const ff2 t = two_sum2(s.h, b);
  s.h = t.h;
  s.c = add2(s.c, t.l);
}
// + (b.h + b.c) * x for an unnormalised sum b: the exact product of its high part by
// TwoProd, its correction's product into the correction
__device__ __forceinline__ void acc2_add_mul(ff2_acc& s, ff2_acc b, float2 x) {
  const ff2 p = two_prod2(b.h, x);
  const ff2 t = two_sum2(s.h, p.h);
  s.h = t.h;
  s.c = add2(s.c, add2(t.l, fma2(b.c, x, p.l)));
}

// Projection onto {y_0 >= |ybar|} (eq. (app-proj)) of a cone of K = 2 NP components held
// as lane pairs: P[0] = (y_0, y_{K-1}), P[1 .. NP - 1] = the others paired in any order.
// The input of the ALM projection is dominated by -beta/sigma, often 10^2 - 10^3 times
// the O(1) point it projects to, so the tests and the boundary value (y_0 + |ybar|)/2
// cancel: |ybar| and that sum are formed in two-float arithmetic (~2^-44 relative).  The
// boundary direction ybar/|ybar| only scales the O(1) result, so it is taken in FP32:
// every output component is then within a few FP32 ulps of its own (O(1)) value, the
// precision it is stored in.  Case order: y if |ybar| <= y_0; 0 if |ybar| <= -y_0; else
// the boundary formula.  |ybar|^2 is summed in two lanes, the square root comes from
// rsqrt and the boundary scale from its reciprocal r, two ulps at most off; CORRECT adds one
// correction from the remainder.  The scale's error is common to a cone's components: on
// 37 x 21 x 50 x 20 phi's error against 64 bits is 2.2e-7 without the correction and 2.1e-7
// with it (the 3D pass takes it).  In 2D, over 60 instances solved to 1e-6, it lowers the
// errors at a fixed iteration by some 7% but raises the mean count of iterations by 0.5% on
// 256^2 x 64, 0.8% on 128^2 x 32 and 2.6% on 64^2 x 32 with obstacles (the 2D pass does not).
// The three cases are one scale each for the high and low parts, without branches: zr = the
// result rounded to FP32, pairs as P; *z0 and the returned z_{K-1} are those two components
// as two-floats.
template <int NP, bool CORRECT>
__device__ __forceinline__ float2 ff2_project(const ff2* P, float2* zr, float2* z0) {
  float2 sh = make_float2(0.f, 0.f), sc = make_float2(0.f, 0.f);
#pragma unroll
  for (int k = 1; k < NP; ++k) {
    const float2 h = P[k].h;
    const float2 p = mul2(h, h);
    const float2 e0 = make_float2(fmaf(h.x, h.x, -p.x), fmaf(h.y, h.y, -p.y));
    const float2 e = fma2(add2(h, h), P[k].l, e0);
    if (k == 1) {
      sh = p;
      sc = e;
    } else {
      const ff2 t = two_sum2(sh, p);
      sh = t.h;
      sc = add2(sc, add2(t.l, e));
    }
  }
  // y_{K-1} and the two lanes
  const float h9 = P[0].h.y;
  const float p9 = h9 * h9;
  const float e9 = fmaf(2.f * h9, P[0].l.y, fmaf(h9, h9, -p9));
  const float2 t1 = two_sum(sh.x, sh.y);
  const float2 t2 = two_sum(t1.x, p9);
  const float corr = ((sc.x + sc.y) + (t1.y + t2.y)) + e9;
  float r;
  const float2 nb = ff_sqrt_r(quick_two_sum(t2.x, corr), &r);
  const float2 y0 = ff2_lane0(P[0]);
  const bool inside = ff_le(nb, y0), below = ff_le(nb, ff_neg(y0));
  const float2 sum = ff_add(y0, nb);
  const float2 a = make_float2(0.5f * sum.x, 0.5f * sum.y);
  // inside: h + l; below: 0; else the boundary point along ybar / |ybar|
  const float m = inside ? 1.f : 0.f;
  const float as = a.x + a.y, sr = as * r;
  const float edge = CORRECT ? fmaf(fmaf(-sr, nb.x, as), r, sr) : sr;
  const float scale = inside ? 1.f : below ? 0.f : edge;
  *z0 = inside ? y0 : below ? make_float2(0.f, 0.f) : a;
  const float2 m2 = make_float2(m, m), s2 = make_float2(scale, scale);
#pragma unroll
  for (int k = 1; k < NP; ++k) zr[k] = fma2(m2, P[k].l, mul2(s2, P[k].h));
  const float2 z9 = make_float2(scale * h9, m * P[0].l.y);
  zr[0] = make_float2(z0->x + z0->y, z9.x + z9.y);
  return z9;
}

}  // namespace dot
