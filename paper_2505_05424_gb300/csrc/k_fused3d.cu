// k_fused3d.cu -- lines 3-6 of Algorithm 2 for D = 3 in two passes over the
// mixed-path state, and the next iteration's lines 1-2 residual.
//
// The D = 2 pass (k_fused2d.cu) recomputes a one-cone halo around each tile so
// that z never reaches memory.  In three dimensions that halo would cost about two
// projections per cone, so z (FP32, K components) is stored once and read back:
//   k_cone3 : per cone, z = Pi_K(B F q^k + d - beta^k/sigma) and the q_0, alpha_0
//             update (diagonal 3, Proposition 3.2) into the k+1 set;
//   k_face3 : everything that meets at one time node t.  The space faces of node t
//             collect components 1, 2 (5, 6; 9, 10) of the cones of time t and 3, 4 (7, 8;
//             11, 12) of the cones of t - 1, and those same components of beta are the ones
//             whose update (line 6) reads q^{k+1} on node t: so a block that takes a 4 x 4 x 32
//             tile of cells at node t reads and writes each entry of beta once, and no two
//             nodes share one.  A thread owns one cell and the three faces above it:
//   1. it sums S = s (z + beta/sigma) over the two cone times for the face below it along
//      each axis, which it publishes, and O for its own faces; the cells above the tile
//      publish their S;
//   2. it updates q_d, alpha_d of its three faces (lines 4-5) from S of the cell above and
//      its own O; the faces below the tile, which the neighbouring tiles write, are
//      computed for their values;
//   3. it updates beta of its cell's node-t components from the six faces around it, and
//      writes the residual r = A^*(q - alpha/sigma - A phi) - c/sigma at the node, which the
//      next iteration's Poisson solve reads (the warm start of lines 1-2).
// beta of the tile is copied to shared memory (a slot per thread) while the halo work and
// the previous node's last step run.  q, alpha and beta are double-buffered (iteration k
// read, k+1 written).  Per element: two-float y, projection, face right-hand sides and
// multiplier updates (ffloat.cuh), FP32 q and z, as in the D = 2 pass; the two axes x and y
// and the two components of z are lane pairs, as beta is stored (dot_mixed.cuh).
//
// Bound by HBM (0.8 of a copy's rate on the pair's 4.95 GB) and, in k_face3, by the latency
// of a node's two barriers with two blocks of sixteen warps per SM.  64^3 x 32: k_face3 585 us
// per launch, k_cone3 308; 37 x 21 x 50 x 20: 84 and 32.  Before, the face pass marched along
// time over whole cones, reading each entry of beta and z for the faces of one node and
// again, from HBM, for the update after the next: 953 us (457 M warp instructions, 4.1 GB
// for 3.2), and 217 us on 37 x 21 x 50 x 20.
#include <cmath>

#include "dot_internal.cuh"
#include "dot_mixed.cuh"
#include "ffloat.cuh"

namespace dot {
namespace {

constexpr int NP3 = 7;                     // pairs of the K = 14 cone components
constexpr int FX = 4, FY = 4, FZ = 32;     // tile: cells along axes 1, 2, 3 (axis 3 contiguous)
constexpr int kCells3 = FX * FY * FZ;      // 512: a thread each
constexpr int kThreads3 = kCells3;
// slots along each axis: cells 0 .. F (S), faces -1 .. F - 1 (q, w)
constexpr int NSX = (FX + 1) * FY * FZ, NSY = FX * (FY + 1) * FZ, NSZ = FX * FY * (FZ + 1);
constexpr int NS3 = NSX + NSY + NSZ;
constexpr int kHalo = FY * FZ + FX * FZ + FX * FY;   // cells beyond one end of each axis: 272
static_assert(kHalo <= kThreads3 && FZ == 32 && FX == 4 && FY == 4, "cell and halo numbering below");
// shared memory (bytes): beta slots, S, w, q
constexpr int kOffS = NP3 * kThreads3 * 16;
constexpr int kOffW = kOffS + NS3 * 8;
constexpr int kOffQ = kOffW + NS3 * 8;
constexpr int kSmem3 = kOffQ + NS3 * 4;
constexpr int kConeThreads = 256;
constexpr float kSdef = 0.70710678118654752f;   // sqrt(omega/2) for omega = 1

struct Fused3Args {
  // iteration k (read)
  const float* q[4];
  const float2* al[4];
  const float4* beta;
  // iteration k+1 (written)
  float* qn[4];
  float2* aln[4];
  float4* betan;
  float2* z;             // pairs as beta, written by k_cone3, read by k_face3
  const float2* phi;     // phi^{k+1}
  const float* somega;   // sqrt(omega/2) per cell, or nullptr
  const SlotParam* sp;
  float* r;              // residual of the next iteration's lines 1-2
  const float2* c0;
  const float2* c1;
  float ih[4];           // 1/h per axis (0 = time)
  int tchunk;            // time nodes per block
  int nty, ntz;          // tiles along axes 2, 3
};

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ ff2 ff2_of(float4 b) { return ff2{make_float2(b.x, b.y), make_float2(b.z, b.w)}; }
__device__ __forceinline__ float4 f4_of(ff2 b) { return make_float4(b.h.x, b.h.y, b.l.x, b.l.y); }
__device__ __forceinline__ void copy16(uint32_t dst, const float4* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Line 3 and lines 4-5 on the time faces.  One thread per cone (t, x): the projection
// input y = B F q^k + d - beta^k/sigma in two-float arithmetic, z stored rounded to FP32,
// then q_0, alpha_0 of the cone from rhs = A_0 phi + alpha_0/sigma + u_{K-1} - u_0 with
// u = z + beta/sigma (F^*B^* of components 0 and K-1), diagonal 3.
__global__ void __launch_bounds__(kConeThreads) k_cone3(const __grid_constant__ Geo g,
                                                        const __grid_constant__ Fused3Args a) {
  if (!a.sp[0].active) return;
  const float ts = a.sp[0].tau;
  const int P = (int)g.P, n0 = g.T * P, N1 = g.N[1], N2 = g.N[2], sx = N1 * N2;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n0; i += gridDim.x * blockDim.x) {
    const int t = (int)fdiv((unsigned)i, g.fP), p = i - t * P;
    const int x = coord(g, p, 0), y = coord(g, p, 1), zc = coord(g, p, 2);
    const bool xl = x >= 1, xh = x <= g.N[0] - 2, yl = y >= 1, yh = y <= N1 - 2, zl = zc >= 1, zh = zc <= N2 - 2;
    // F q^k as lane pairs: per axis the faces below / above the cell on time nodes t and
    // t + 1 (zero where F has no source face)
    const float *q1 = a.q[1] + i, *q2 = a.q[2] + i, *q3 = a.q[3] + i;
    const float q0 = a.q[0][i];
    float2 x_[NP3];
    x_[1] = f2(xl ? q1[-sx] : 0.f, yl ? q2[-N2] : 0.f);
    x_[2] = f2(xh ? q1[0] : 0.f, yh ? q2[0] : 0.f);
    x_[3] = f2(xl ? q1[P - sx] : 0.f, yl ? q2[P - N2] : 0.f);
    x_[4] = f2(xh ? q1[P] : 0.f, yh ? q2[P] : 0.f);
    x_[5] = f2(zl ? q3[-1] : 0.f, zh ? q3[0] : 0.f);
    x_[6] = f2(zl ? q3[P - 1] : 0.f, zh ? q3[P] : 0.f);
    const float s = a.somega ? a.somega[p] : kSdef;
    const float2 s2 = f2(s, s);
    ff2 Y[NP3];
    const ff2 b0 = ff2_of(a.beta[i]);
    Y[0] = ff2_sub(two_sum2(f2(-q0, q0), f2(1.f, 1.f)), b0);
#pragma unroll
    for (int k = 1; k < NP3; ++k) Y[k] = ff2_sub(two_prod2(s2, x_[k]), ff2_of(a.beta[k * n0 + i]));
    float2 zr[NP3], z0;
    ff2_project<NP3, true>(Y, zr, &z0);
#pragma unroll
    for (int k = 0; k < NP3; ++k) a.z[k * n0 + i] = zr[k];
    const float2 gp = ff_grad(a.phi[i], a.phi[i + P], a.ih[0]);
    const float2 al = a.al[0][i];
    ff_acc acc = acc_init(gp);
    acc_add(acc, al);
    acc_add(acc, ff2_lane1(b0));
    acc_add(acc, ff_neg(ff2_lane0(b0)));
    acc_add_f(acc, zr[0].y - zr[0].x);
    const float qn = ff_round(ff_div_f_r(acc_get(acc), 3.f, 1.f / 3.f));
    a.qn[0][i] = qn;
    a.aln[0][i] = ff_add_f(al, ts * ((gp.x - qn) + gp.y));
  }
}

// w = q - alpha/sigma - A_0 phi of the time face of cone ic, negated, from the k+1 values
// k_cone3 wrote.
__device__ __forceinline__ float2 w_time(const Fused3Args& a, int ic, int P) {
  const float2 gp = ff_grad(a.phi[ic], a.phi[ic + P], a.ih[0]);
  const float gm = (gp.x - a.qn[0][ic]) + gp.y;
  const float2 al = a.aln[0][ic], e = two_sum(al.x, gm);
  return f2(e.x, e.y + al.y);
}

// s (z + beta/sigma) of one component over the two cone times (now: t, prev: t - 1), as an
// unnormalised two-float; b, z: the component's entries, or zero where there is no cone.
__device__ __forceinline__ float2 side_sum(float2 bn, float2 bp, float zn, float zp, float s) {
  ff_acc v = acc_init(bn);
  acc_add(v, bp);
  ff_acc o{0.f, 0.f};
  const float p = v.h * s;
  o.h = p;
  o.c = fmaf(v.c, s, fmaf(v.h, s, -p));
  acc_add_f(o, s * (zn + zp));
  return f2(o.h, o.c);
}
// the same in two lanes
__device__ __forceinline__ ff2_acc side_sum2(ff2 bn, ff2 bp, float2 zn, float2 zp, float2 s) {
  ff2_acc v{bn.h, bn.l};
  acc2_add(v, bp);
  const ff2 p = two_prod2(v.h, s);
  ff2_acc o{p.h, fma2(v.c, s, p.l)};
  acc2_add_f(o, mul2(s, add2(zn, zp)));
  return o;
}

// One face: rhs = A_d phi + alpha/sigma + S + O, q = rhs / den, alpha/sigma += tau (A_d phi - q);
// *w = alpha/sigma + A_d phi - q (unnormalised).
__device__ __forceinline__ float face_step(float2 gp, float2 al, float2 S, float2 O, float den, float ts, float2* aln,
                                           float2* w) {
  ff_acc acc = acc_init(gp);
  acc_add(acc, al);
  acc_add(acc, S);
  acc_add(acc, O);
  const float r = rcp_approx(den);
  const float q1 = acc.h * r;
  const float2 pr = two_prod(q1, den);
  const float q = fmaf(((acc.h - pr.x) - pr.y) + acc.c, r, q1);
  const float gm = (gp.x - q) + gp.y;
  *aln = ff_add_f(al, ts * gm);
  const float2 e = two_sum(aln->x, gm);
  *w = f2(e.x, e.y + aln->y);
  return q;
}

// Slots: S of cell (cx, cy, cz) along axis d (cx, cy or cz may be one beyond the tile), and
// q, w of the face above cell (cx, cy, cz) (whose coordinate along d may be -1).
__device__ __forceinline__ int slot_x(int cx, int cy, int cz) { return (cx * FY + cy) * FZ + cz; }
__device__ __forceinline__ int slot_y(int cx, int cy, int cz) { return NSX + (cx * (FY + 1) + cy) * FZ + cz; }
__device__ __forceinline__ int slot_z(int cx, int cy, int cz) { return NSX + NSY + (cx * FY + cy) * (FZ + 1) + cz; }

template <bool MASKED>
__global__ void __launch_bounds__(kThreads3, 2) k_face3(const __grid_constant__ Geo g,
                                                        const __grid_constant__ Fused3Args a) {
  if (!a.sp[0].active) return;
  extern __shared__ __align__(16) unsigned char sm[];
  float2* sS = reinterpret_cast<float2*>(sm + kOffS);
  float2* sw = reinterpret_cast<float2*>(sm + kOffW);
  float* sq = reinterpret_cast<float*>(sm + kOffQ);
  const int tid = threadIdx.x, cz = tid & 31, cy = (tid >> 5) & 3, cx = tid >> 7;
  float4* bslot = reinterpret_cast<float4*>(sm) + tid;
  const uint32_t bsm = (uint32_t)__cvta_generic_to_shared(bslot);
  const int tz = blockIdx.x % a.ntz, tyx = blockIdx.x / a.ntz, ty = tyx % a.nty, tx = tyx / a.nty;
  const int x0 = tx * FX, y0 = ty * FY, z0 = tz * FZ;
  const int T = g.T, P = (int)g.P, n0 = T * P, N0 = g.N[0], N1 = g.N[1], N2 = g.N[2], sx = N1 * N2;
  const int ta = blockIdx.y * a.tchunk, tb = min(T + 1, ta + a.tchunk);   // time nodes [ta, tb)
  const float ts = a.sp[0].tau;
  const int X = x0 + cx, Y = y0 + cy, Z = z0 + cz, p = (X * N1 + Y) * N2 + Z;
  const bool ok = X < N0 && Y < N1 && Z < N2;
  const bool fx = ok && X <= N0 - 2, fy = ok && Y <= N1 - 2, fz = ok && Z <= N2 - 2;
  float s = kSdef;
  float3 sn = make_float3(kSdef, kSdef, kSdef);
  if (MASKED && ok) {
    s = a.somega[p];
    if (fx) sn.x = a.somega[p + sx];
    if (fy) sn.y = a.somega[p + N2];
    if (fz) sn.z = a.somega[p + 1];
  }
  // halo cell of this thread (tid < kHalo above the tile; kThreads3 - 1 - tid < kHalo below)
  auto halo = [&](int h, bool up, int* d, int* hx, int* hy, int* hz) {
    if (h < FY * FZ) {
      *d = 0; *hx = up ? FX : -1; *hy = h >> 5; *hz = h & 31;
    } else if (h < FY * FZ + FX * FZ) {
      h -= FY * FZ;
      *d = 1; *hx = h >> 5; *hy = up ? FY : -1; *hz = h & 31;
    } else {
      h -= FY * FZ + FX * FZ;
      *d = 2; *hx = h >> 2; *hy = h & 3; *hz = up ? FZ : -1;
    }
  };
  // the node's components of beta: pairs 0, 1, 2, 5 of cone t and 3, 4, 6 of cone t - 1
  auto fetch = [&](int t) {
    if (ok) {
#pragma unroll
      for (int k = 0; k < NP3; ++k) {
        const bool now = k <= 2 || k == 5;
        if (now ? t < T : t >= 1) copy16(bsm + k * kThreads3 * 16, a.beta + k * n0 + (now ? t : t - 1) * P + p);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(ta);
  const float2 z2 = f2(0.f, 0.f);
  const ff2 zf{z2, z2};
  float2 w0p = ok && ta >= 1 ? w_time(a, (ta - 1) * P + p, P) : z2;

  for (int t = ta; t < tb; ++t) {
    const bool now = t < T, prev = t >= 1;
    const int i = t * P + p, im = i - P;
    // ---------------- 1: S and O ----------------
    if (tid < kHalo) {   // S of the cells above the tile
      int d, hx, hy, hz;
      halo(tid, true, &d, &hx, &hy, &hz);
      const int gx = x0 + hx, gy = y0 + hy, gz = z0 + hz;
      float2 S = z2;
      if (gx < N0 && gy < N1 && gz < N2) {
        const int hp = (gx * N1 + gy) * N2 + gz, lane = d == 1 ? 1 : 0;
        const int kn = d == 2 ? 5 : 1, kp = d == 2 ? 6 : 3;
        const float hs = MASKED ? a.somega[hp] : kSdef;
        float2 bn = z2, bp = z2;
        float zn = 0.f, zp = 0.f;
        if (now) {
          const int o = kn * n0 + t * P + hp;
          const float* b = reinterpret_cast<const float*>(a.beta + o) + lane;
          bn = f2(b[0], b[2]);
          zn = reinterpret_cast<const float*>(a.z + o)[lane];
        }
        if (prev) {
          const int o = kp * n0 + (t - 1) * P + hp;
          const float* b = reinterpret_cast<const float*>(a.beta + o) + lane;
          bp = f2(b[0], b[2]);
          zp = reinterpret_cast<const float*>(a.z + o)[lane];
        }
        S = side_sum(bn, bp, zn, zp, hs);
      }
      sS[d == 0 ? slot_x(hx, hy, hz) : d == 1 ? slot_y(hx, hy, hz) : slot_z(hx, hy, hz)] = S;
    }
    // this thread's potential and multipliers, in flight over step 1
    float2 ph = z2, px = z2, py = z2, pz = z2, a1 = z2, a2 = z2, a3 = z2;
    if (ok) ph = a.phi[i];
    if (fx) { px = a.phi[i + sx]; a1 = a.al[1][i]; }
    if (fy) { py = a.phi[i + N2]; a2 = a.al[2][i]; }
    if (fz) { pz = a.phi[i + 1]; a3 = a.al[3][i]; }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    ff2_acc Oxy{z2, z2}, Z56{z2, z2};
    if (ok) {
      const float2 s2 = f2(s, s);
      const float2 zz = z2;
      const ff2 b1 = now ? ff2_of(bslot[1 * kThreads3]) : zf, b3 = prev ? ff2_of(bslot[3 * kThreads3]) : zf;
      const ff2_acc S = side_sum2(b1, b3, now ? a.z[n0 + i] : zz, prev ? a.z[3 * n0 + im] : zz, s2);
      const ff2 b2 = now ? ff2_of(bslot[2 * kThreads3]) : zf, b4 = prev ? ff2_of(bslot[4 * kThreads3]) : zf;
      Oxy = side_sum2(b2, b4, now ? a.z[2 * n0 + i] : zz, prev ? a.z[4 * n0 + im] : zz, s2);
      const ff2 b5 = now ? ff2_of(bslot[5 * kThreads3]) : zf, b6 = prev ? ff2_of(bslot[6 * kThreads3]) : zf;
      Z56 = side_sum2(b5, b6, now ? a.z[5 * n0 + i] : zz, prev ? a.z[6 * n0 + im] : zz, s2);
      sS[slot_x(cx, cy, cz)] = f2(S.h.x, S.c.x);
      sS[slot_y(cx, cy, cz)] = f2(S.h.y, S.c.y);
      sS[slot_z(cx, cy, cz)] = f2(Z56.h.x, Z56.c.x);
    }
    __syncthreads();
    // ---------------- 2: the faces of node t ----------------
    const float nt = now && prev ? 2.f : 1.f;   // cone times that read the faces
    float3 qo = make_float3(0.f, 0.f, 0.f);
    float2 wx = z2, wy = z2, wz = z2;
    if (fx) {
      float2 aln;
      qo.x = face_step(ff_grad(ph, px, a.ih[1]), a1, sS[slot_x(cx + 1, cy, cz)], f2(Oxy.h.x, Oxy.c.x),
                       fmaf(nt, fmaf(sn.x, sn.x, s * s), 1.f), ts, &aln, &wx);
      a.qn[1][i] = qo.x;
      a.aln[1][i] = aln;
    }
    if (fy) {
      float2 aln;
      qo.y = face_step(ff_grad(ph, py, a.ih[2]), a2, sS[slot_y(cx, cy + 1, cz)], f2(Oxy.h.y, Oxy.c.y),
                       fmaf(nt, fmaf(sn.y, sn.y, s * s), 1.f), ts, &aln, &wy);
      a.qn[2][i] = qo.y;
      a.aln[2][i] = aln;
    }
    if (fz) {
      float2 aln;
      qo.z = face_step(ff_grad(ph, pz, a.ih[3]), a3, sS[slot_z(cx, cy, cz + 1)], f2(Z56.h.y, Z56.c.y),
                       fmaf(nt, fmaf(sn.z, sn.z, s * s), 1.f), ts, &aln, &wz);
      a.qn[3][i] = qo.z;
      a.aln[3][i] = aln;
    }
    sq[slot_x(cx + 1, cy, cz)] = qo.x;
    sq[slot_y(cx, cy + 1, cz)] = qo.y;
    sq[slot_z(cx, cy, cz + 1)] = qo.z;
    sw[slot_x(cx + 1, cy, cz)] = wx;
    sw[slot_y(cx, cy + 1, cz)] = wy;
    sw[slot_z(cx, cy, cz + 1)] = wz;
    if (kThreads3 - 1 - tid < kHalo) {   // the faces below the tile
      int d, hx, hy, hz;
      halo(kThreads3 - 1 - tid, false, &d, &hx, &hy, &hz);
      const int gx = x0 + hx, gy = y0 + hy, gz = z0 + hz;
      const int st = d == 0 ? sx : d == 1 ? N2 : 1;
      const int sl = d == 0 ? slot_x(0, hy, hz) : d == 1 ? slot_y(hx, 0, hz) : slot_z(hx, hy, 0);
      float q = 0.f;
      float2 w = z2;
      // the face exists where the cells on both its sides do
      if (gx >= 0 && gy >= 0 && gz >= 0 && gx + (d == 0) < N0 && gy + (d == 1) < N1 && gz + (d == 2) < N2) {
        const int hp = (gx * N1 + gy) * N2 + gz, lane = d == 0 ? 0 : 1;
        const int kn = d == 2 ? 5 : 2, kp = d == 2 ? 6 : 4;
        const float hs = MASKED ? a.somega[hp] : kSdef, hn = MASKED ? a.somega[hp + st] : kSdef;
        float2 bn = z2, bp = z2;
        float zn = 0.f, zp = 0.f;
        if (now) {
          const int o = kn * n0 + t * P + hp;
          const float* b = reinterpret_cast<const float*>(a.beta + o) + lane;
          bn = f2(b[0], b[2]);
          zn = reinterpret_cast<const float*>(a.z + o)[lane];
        }
        if (prev) {
          const int o = kp * n0 + (t - 1) * P + hp;
          const float* b = reinterpret_cast<const float*>(a.beta + o) + lane;
          bp = f2(b[0], b[2]);
          zp = reinterpret_cast<const float*>(a.z + o)[lane];
        }
        const int j = t * P + hp;
        const float2* ad = d == 0 ? a.al[1] : d == 1 ? a.al[2] : a.al[3];
        const float ihd = d == 0 ? a.ih[1] : d == 1 ? a.ih[2] : a.ih[3];
        float2 aln;
        q = face_step(ff_grad(a.phi[j], a.phi[j + st], ihd), ad[j], sS[sl], side_sum(bn, bp, zn, zp, hs),
                      fmaf(nt, fmaf(hn, hn, hs * hs), 1.f), ts, &aln, &w);
      }
      sq[sl] = q;
      sw[sl] = w;
    }
    __syncthreads();
    // ---------------- 3: beta and the residual ----------------
    if (ok) {
      const int lx = slot_x(cx, cy, cz), ly = slot_y(cx, cy, cz), lz = slot_z(cx, cy, cz);
      const float2 ql = f2(sq[lx], sq[ly]), qz = f2(sq[lz], qo.z), qxy = f2(qo.x, qo.y);
      const float2 ns2 = f2(-s, -s), ts2 = f2(ts, ts);
      auto upd = [&](int k, int o, float2 inc) {
        a.betan[k * n0 + o] = f4_of(ff2_add_f(ff2_of(bslot[k * kThreads3]), mul2(ts2, inc)));
      };
      float2 d0 = z2;
      if (now) {
        const float q0 = a.qn[0][i];
        upd(0, i, add2(sub2(a.z[i], f2(1.f, 1.f)), f2(q0, -q0)));
        upd(1, i, fma2(ns2, ql, a.z[n0 + i]));
        upd(2, i, fma2(ns2, qxy, a.z[2 * n0 + i]));
        upd(5, i, fma2(ns2, qz, a.z[5 * n0 + i]));
        d0 = w_time(a, i, P);
      }
      if (prev) {
        upd(3, im, fma2(ns2, ql, a.z[3 * n0 + im]));
        upd(4, im, fma2(ns2, qxy, a.z[4 * n0 + im]));
        upd(6, im, fma2(ns2, qz, a.z[6 * n0 + im]));
      }
      // A^* w - c/sigma with w of the node's faces (negated, zero at the walls)
      const float2 w0c = d0;
      {
        const float2 e = two_sum(d0.x, -w0p.x);
        d0 = f2(e.x, e.y + (d0.y - w0p.y));
      }
      ff_acc acc{0.f, 0.f};
      acc_add_mul(acc, d0, a.ih[0]);
      auto side = [&](float2 own, float2 low, float ih) {
        const float2 e = two_sum(own.x, -low.x);
        acc_add_mul(acc, f2(e.x, e.y + (own.y - low.y)), ih);
      };
      side(wx, sw[lx], a.ih[1]);
      side(wy, sw[ly], a.ih[2]);
      side(wz, sw[lz], a.ih[3]);
      if (t == 0) acc_add(acc, ff_neg(ff_mul(a.c0[p], a.sp[0].isg)));
      if (t == T) acc_add(acc, ff_mul(a.c1[p], a.sp[0].isg));
      a.r[i] = acc.h + acc.c;
      w0p = w0c;
    }
    if (t + 1 < tb) fetch(t + 1);   // the slots are this thread's own
    // no barrier here: step 1 of t + 1 writes S, last read in step 2 of t before the second
    // barrier; step 2 of t + 1, which writes q and w, follows the barrier after step 1
  }
}

}  // namespace

bool fused3d_supported(const Geo& g) { return g.D == 3; }

void launch_fused3d(const Geo& g, const MxFields& f, const MxFields& fn, cudaStream_t s, LaunchCounter lc) {
  Fused3Args a;
  for (int d = 0; d < 4; ++d) {
    a.q[d] = f.q[d];
    a.al[d] = f.al[d];
    a.qn[d] = fn.q[d];
    a.aln[d] = fn.al[d];
    a.ih[d] = g.ih[d];
  }
  a.beta = reinterpret_cast<const float4*>(f.beta);
  a.betan = reinterpret_cast<float4*>(fn.beta);
  a.z = reinterpret_cast<float2*>(f.z);
  a.phi = f.phi;
  a.somega = f.somega;
  a.sp = f.sp;
  a.r = f.r;
  a.c0 = f.c0;
  a.c1 = f.c1;
  const int ntx = (g.N[0] + FX - 1) / FX;
  a.nty = (g.N[1] + FY - 1) / FY;
  a.ntz = (g.N[2] + FZ - 1) / FZ;
  const int tiles = ntx * a.nty * a.ntz;
  // time nodes per block: eight, fewer while that leaves under eight blocks per SM slot
  int c = 8;
  while (c > 1 && (long long)tiles * ((g.T + c) / c) < 8LL * 2 * 152) c /= 2;
  a.tchunk = c;
  const long long n0 = (long long)g.T * g.P;
  long long nb = (n0 + kConeThreads - 1) / kConeThreads;
  if (nb > 152LL * 16) nb = 152LL * 16;
  k_cone3<<<(unsigned)nb, kConeThreads, 0, s>>>(g, a);
  lc.launched(KID_PROJECT);
  const dim3 grid((unsigned)tiles, (unsigned)((g.T + c) / c));
  static std::atomic<unsigned long long> done[2];
  if (f.somega) {
    smem_optin((const void*)k_face3<true>, kSmem3, &done[1]);
    k_face3<true><<<grid, kThreads3, kSmem3, s>>>(g, a);
  } else {
    smem_optin((const void*)k_face3<false>, kSmem3, &done[0]);
    k_face3<false><<<grid, kThreads3, kSmem3, s>>>(g, a);
  }
  lc.launched(KID_FACE3);
}

}  // namespace dot
