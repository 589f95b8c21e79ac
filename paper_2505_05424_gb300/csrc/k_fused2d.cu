// k_fused2d.cu -- lines 3-6 of Algorithm 2 (cone projection, q and alpha updates,
// beta update) fused into one pass over the mixed-path state, for D = 2, and the
// next iteration's lines 1-2 residual.
//
// A CTA works on a TX x 32 (x, y) tile of cells at a time and marches along time.  One
// thread owns one cone column: the cone (t, x, y) and the two space faces above it,
// (x + 1/2, y) and (x, y + 1/2).  Three more warps take the one-cone halo: the row
// x0 - 1 (with the x-faces the tile reads from below), the row x0 + TX, and the columns
// y0 - 1 (with its y-faces) and y0 + 32.  At time t a thread
//   A. projects z(t) = Pi_K(B F q^k + d - beta^k/sigma) and publishes the components
//      that the faces below it read (1 and 3 for the x-face, 5 and 7 for the y-face);
//      owners update q_0, alpha_0 (diagonal 3, Proposition 3.2);
//   B. updates q_d, alpha_d of its two faces on time node t, as the two lanes of packed
//      two-float arithmetic, from its own z and beta and its two neighbours', and
//      publishes q and w = q - alpha/sigma - A phi of them;
//   C. (owners) updates the components of beta whose update reads q^{k+1} on the faces of
//      node t -- 1, 2, 5, 6 of the cone at t and 3, 4, 7, 8 of the cone at t - 1, the ones
//      those faces collected (0 and 9 follow q_0 in step A) -- and writes the next
//      iteration's residual at node t from the faces' w.
// A thread copies its column's beta one cone time ahead into its own shared-memory
// slots (cp.async, any N_y), where step A, the faces below it and step C read it.  z
// never reaches HBM.  q, alpha and beta are double-buffered: every read is of iteration
// k and every write of k+1, so CTAs may run in any order.
// Per element: y and the projection tests in two-float arithmetic, FP32 z and q,
// two-float face right-hand sides and multiplier updates (ffloat.cuh).
//
// Bound by instruction issue and by the latency of a time step (two barriers, a
// dependent chain of some 100 FP operations): on 256^2 x 64 136 M warp
// instructions, 48% issue, 0.64 of the HBM bandwidth on its 1,026 MB, 236 us per launch;
// 128^2 x 32 40.8 us, 32^2 x 16 10.0 us (251, 47.5 and 10.4 with the sums of squared
// increments in FP64 and one CTA-wide sum per work unit).  The form before it (a thread per
// halo cone, faces dealt out in rounds, beta by TMA in component planes, 80 registers at two
// CTAs per SM, fixed 16-time chunks): 245 M instructions, 357, 62 and 19.6 us; and for odd
// N_y, where it could not use TMA, 262 us on 150 x 117 x 37 against 51 now.  Measured on the
// way: this mapping at two CTAs of 8 rows and 80 registers 429 us (spills), one CTA of 12
// rows and 128 registers 293; equal shares of work for every SM and beta in lane pairs
// 267; a segment owning whole cones, whose last update needs one projection and one face
// step beyond it, 257 (128^2 x 32: 53.5).
#include <cmath>

#include "dot_internal.cuh"
#include "dot_mixed.cuh"
#include "ffloat.cuh"

namespace dot {
namespace {

constexpr int K2 = 10;                    // 4D + 2 for D = 2
constexpr int TY = 32;                    // tile columns: one warp per row
constexpr int kStages = 3;                // beta of cone times t - 1, t, t + 1
constexpr int kSMs = 152;
constexpr float kSdef = 0.70710678118654752f;            // sqrt(omega / 2) for omega = 1

// Threads and shared memory of a CTA with TX tile rows.
template <int TX>
struct Tile {
  static constexpr int kWarps = TX + 3;   // owners, rows x0 - 1 and x0 + TX, columns y0 - 1 and y0 + 32
  static constexpr int kThreads = 32 * kWarps;
  static_assert(2 * TX <= 32, "one warp holds both halo columns");
  // bytes: beta slots, then one slot per thread of what its neighbours read
  static constexpr int kOffZ1 = kStages * (K2 / 2) * kThreads * 16;   // z_(1, 5) of cone time t
  static constexpr int kOffZ3 = kOffZ1 + kThreads * 8;                // z_(3, 7), two cone times
  static constexpr int kOffPh = kOffZ3 + 2 * kThreads * 8;            // phi on node t
  static constexpr int kOffQ = kOffPh + kThreads * 8;                 // q^{k+1} of the (x, y) faces
  static constexpr int kOffW = kOffQ + kThreads * 8;                  // alpha/sigma + A phi - q of the faces
  static constexpr int kSmem = kOffW + kThreads * 16;
};

// The multipliers are stored as alpha/sigma and beta/sigma (k_mixed.cu), so the
// projection input is BFq + d - (stored beta) and the updates add tau (...).
struct FusedArgs {
  // iteration k (read)
  const float* q[3];
  const float2* al[3];
  const float4* beta;
  // iteration k+1 (write)
  float* qn[3];
  float2* aln[3];
  float4* betan;
  const float2* phi;   // phi^{k+1}
  const float* somega;
  int G;               // slots
  int ntx, nty;        // tiles along x and y
  int unit, nunit;     // time nodes per work unit, units per tile
  int run;             // time nodes per partial sum (divides unit)
  const SlotParam* sp;
  float2* socp_part;   // [slot][run][y tile][x]: sums of |z - B F q^{k+1} - d|^2 over 32 cells of a row
  // the next iteration's lines 1-2 residual
  // r = A^*(q^{k+1} - alpha^{k+1}/sigma) - c/sigma - A^*A phi^{k+1} at every node
  float* r;
  const float2* c0;
  const float2* c1;
  float ih0, ih1, ih2; // 1/h of time and of the two axes
};

// 16-byte asynchronous copy into this thread's shared-memory slot
__device__ __forceinline__ void copy16(uint32_t dst, const float4* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// beta as stored for D = 2: component pairs (0, 9), (1, 5), (2, 6), (3, 7), (4, 8),
// high parts then low parts
__device__ __forceinline__ ff2 ff2_of(float4 b) { return ff2{make_float2(b.x, b.y), make_float2(b.z, b.w)}; }
__device__ __forceinline__ float4 f4_of(ff2 b) { return make_float4(b.h.x, b.h.y, b.l.x, b.l.y); }

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// Sum of a two-float over the warp, unnormalised.  (A 32-lane FP64 addition occupies an SM
// for 16 cycles; with FP64 shuffles here 300 iterations on 128^2 x 32 take 28.7 ms, not 26.4,
// and 32 served 64^2 x 32 solves 114 ms, not 107.)
__device__ __forceinline__ float2 warp_sum_ff(float2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float2 u = f2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
    const float2 e = two_sum(v.x, u.x);
    v = f2(e.x, e.y + (v.y + u.y));
  }
  return v;
}

// One segment: time nodes [ta, tb) of one tile of one slot.  socp_tile: the slot's partial
// sums of the tile's rows over the first run of time nodes.  Element indices stay below
// 2^31 over all slots of a batch (dot_server.cu bounds the batch).
template <int TX, bool MASKED>
__device__ __forceinline__ void segment(const Geo& g, const FusedArgs& a, unsigned char* sm, int slot, int x0, int y0,
                                        int ta, int tb, float2* socp_tile) {
  using L = Tile<TX>;
  constexpr int kThreads = L::kThreads;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int T = g.T, P = (int)g.P, n0 = T * P, N0 = g.N[0], N1 = g.N[1];
  const float ts = a.sp[slot].tau;
  const float ih0 = a.ih0, ih1 = a.ih1, ih2 = a.ih2;

  // this thread's cone column, as tile coordinates (xr, yc), and the threads of the
  // columns above (x + 1, y), (x, y + 1) and below (x - 1, y), (x, y - 1)
  const bool owner = warp < TX;
  int xr = warp, yc = lane;
  int hx = xr == TX - 1 ? tid + 64 : tid + 32, hy = lane == 31 ? (TX + 2) * 32 + TX + xr : tid + 1;
  const int lx = xr == 0 ? TX * 32 + lane : tid - 32, ly = lane == 0 ? (TX + 2) * 32 + xr : tid - 1;
  if (!owner) {
    hx = hy = tid;
    if (warp == TX) {
      xr = -1;
      hx = lane;
    } else if (warp == TX + 1) {
      xr = TX;
    } else if (lane < TX) {
      xr = lane;
      yc = -1;
      hy = lane * 32;
    } else {
      xr = lane - TX;
      yc = TY;
    }
  }
  const int x = x0 + xr, y = y0 + yc;
  const bool cone_ok = x >= 0 && y >= 0 && x < N0 && y < N1 && (warp < TX + 2 || lane < 2 * TX);
  // the column's own faces (x + 1/2, y), (x, y + 1/2), where the tile needs them
  const bool fx = cone_ok && warp <= TX && x <= N0 - 2;
  const bool fy = cone_ok && (owner || (warp == TX + 2 && lane < TX)) && y <= N1 - 2;
  const bool own_ok = owner && cone_ok;
  const bool xl = cone_ok && x >= 1, xh = cone_ok && x <= N0 - 2, yl = cone_ok && y >= 1, yh = cone_ok && y <= N1 - 2;

  // sqrt(omega / 2) of the cone and of the cones across its faces
  float s = kSdef;
  float2 sn = f2(kSdef, kSdef);
  if (MASKED && cone_ok) {
    const float* w = a.somega + slot * P + x * N1 + y;
    s = w[0];
    if (fx) sn.x = w[N1];
    if (fy) sn.y = w[1];
  }

  const int tstart = ta > 0 ? ta - 1 : 0;
  const int tlast = min(tb - 1, T - 1);     // last cone time this segment projects
  // element of the column on time plane t: of node fields; cone fields and beta's pair 0
  // at a fixed distance
  int i = slot * (n0 + P) + tstart * P + x * N1 + y;
  const int ocone = -slot * P, obeta = slot * (n0 * (K2 / 2 - 1) - P);

  // shared memory: this thread's beta slots (pair k of stage j at (j K/2 + k) kThreads)
  // and what it publishes
  float4* bslot = reinterpret_cast<float4*>(sm) + tid;
  const float* bx = reinterpret_cast<const float*>(reinterpret_cast<float4*>(sm) + hx);
  const float* by = reinterpret_cast<const float*>(reinterpret_cast<float4*>(sm) + hy) + 1;
  float2* sz1 = reinterpret_cast<float2*>(sm + L::kOffZ1);
  float2* sz3 = reinterpret_cast<float2*>(sm + L::kOffZ3);
  float2* sph = reinterpret_cast<float2*>(sm + L::kOffPh);
  float2* sq = reinterpret_cast<float2*>(sm + L::kOffQ);
  float4* sw = reinterpret_cast<float4*>(sm + L::kOffW);
  const uint32_t bsm = (uint32_t)__cvta_generic_to_shared(bslot);
  auto fetch = [&](int stage, int ii) {
    if (cone_ok) {
      const float4* src = a.beta + ii;
#pragma unroll
      for (int k = 0; k < K2 / 2; ++k) copy16(bsm + (stage * (K2 / 2) + k) * kThreads * 16, src + (long long)k * n0);
    }
  };
  int st_c = 0, st_n = 1, st_p = 2;         // stages of cone times t, t + 1, t - 1
  if (tstart <= tlast) fetch(st_c, i + obeta);
  asm volatile("cp.async.commit_group;" ::: "memory");

  // F q^k of the column: x-lane and y-lane faces below / above on node t (qa, qb), and
  // the next cone time's node (qc, qd) with q_0, one cone time ahead; the potential,
  // alpha_0 of the cone and alpha of the own faces one time ahead too
  const float2 z2 = f2(0.f, 0.f);
  float2 qa = z2, qb = z2, qc = z2, qd = z2;
  float qz = 0.f;
  float2 ph_t = z2, ph_n = z2, al0 = z2, a1 = z2, a2 = z2;
  if (cone_ok) {
    if (xl) qa.x = a.q[1][i - N1];
    if (yl) qa.y = a.q[2][i - 1];
    if (xh) qb.x = a.q[1][i];
    if (yh) qb.y = a.q[2][i];
    if (tstart <= tlast) {
      qz = a.q[0][i + ocone];
      if (xl) qc.x = a.q[1][i + P - N1];
      if (yl) qc.y = a.q[2][i + P - 1];
      if (xh) qd.x = a.q[1][i + P];
      if (yh) qd.y = a.q[2][i + P];
    }
    ph_t = a.phi[i];
    if (tstart < T) ph_n = a.phi[i + P];
    if (owner && tstart <= tlast) al0 = a.al[0][i + ocone];
    if (tstart >= ta) {
      if (fx) a1 = a.al[1][i];
      if (fy) a2 = a.al[2][i];
    }
  }

  float2 zc[5];                             // FP32 z of the cone at t: (0, 9), (1, 5), ..., (4, 8)
#pragma unroll
  for (int k = 0; k < 5; ++k) zc[k] = z2;
  float2 zp3 = z2, zp4 = z2;                // (3, 7) and (4, 8) of the cone at t - 1
  float2 w0c = z2, w0p = z2;                // alpha_0/sigma + A_0 phi - q_0 of cones t and t - 1 (unnormalised)
  float2 socp = z2;
  const float2 ts2 = f2(ts, ts);
  int left = a.run;                         // time nodes to the end of the partial sum
  float2* entry = socp_tile + (long long)(ta / a.run) * a.nty * N0 + warp;

  for (int t = tstart; t < tb; ++t, i += P) {
    const int lev = (t & 1) * kThreads;
    if (t + 1 <= tlast) fetch(st_n, i + obeta + P);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    // ---------------- A: cones at time t ----------------
    if (t <= T - 1 && cone_ok) {
      const float4* bt = bslot + st_c * (K2 / 2) * kThreads;
      const float2 s2 = f2(s, s);
      ff2 z[5];
      // y = B F q + d - beta/sigma as lane pairs (0, 9), (1, 5), (2, 6), (3, 7), (4, 8)
      z[0] = ff2_sub(two_sum2(f2(-qz, qz), f2(1.f, 1.f)), ff2_of(bt[0]));
      z[1] = ff2_sub(two_prod2(s2, qa), ff2_of(bt[1 * kThreads]));
      z[2] = ff2_sub(two_prod2(s2, qb), ff2_of(bt[2 * kThreads]));
      z[3] = ff2_sub(two_prod2(s2, qc), ff2_of(bt[3 * kThreads]));
      z[4] = ff2_sub(two_prod2(s2, qd), ff2_of(bt[4 * kThreads]));
      // the next cone time's q^k: node t + 1 moves down, the rest is loaded now
      qa = qc;
      qb = qd;
      if (t + 1 <= tlast) {
        qz = a.q[0][i + ocone + P];
        if (xl) qc.x = a.q[1][i + 2 * P - N1];
        if (yl) qc.y = a.q[2][i + 2 * P - 1];
        if (xh) qd.x = a.q[1][i + 2 * P];
        if (yh) qd.y = a.q[2][i + 2 * P];
      }
      float2 z0;
      const float2 z9 = ff2_project<5, false>(z, zc, &z0);
      sz1[tid] = zc[1];
      sz3[lev + tid] = zc[3];
      // q_0 (diagonal 3): rhs = A_0 phi + alpha_0/sigma + u_9 - u_0 with u = z + beta/sigma;
      // the cone before the segment (t = ta - 1) is updated for the residual only
      if (owner) {
        const float2 gp = ff_grad(ph_t, ph_n, ih0);
        const ff2 u = ff2_add(ff2_pack(z0, z9), ff2_of(bt[0]));
        ff_acc acc = acc_init(gp);
        acc_add(acc, al0);
        acc_add(acc, ff2_lane1(u));
        acc_add(acc, ff_neg(ff2_lane0(u)));
        const float qn = ff_round(ff_div_f_r(acc_get(acc), 3.f, 1.f / 3.f));
        const float gm = (gp.x - qn) + gp.y;
        const float2 aln = ff_add_f(al0, ts * gm);
        if (t >= ta) {
          a.qn[0][i + ocone] = qn;
          a.aln[0][i + ocone] = aln;
          const float2 inc = add2(sub2(zc[0], f2(1.f, 1.f)), f2(qn, -qn));
          socp = fma2(inc, inc, socp);
          a.betan[i + obeta] = f4_of(ff2_add_f(ff2_of(bt[0]), mul2(ts2, inc)));
        }
        const float2 e = two_sum(aln.x, gm);
        w0c = f2(e.x, e.y + aln.y);
        if (t + 1 <= tlast) al0 = a.al[0][i + ocone + P];
      }
    }
    sph[tid] = ph_t;
    __syncthreads();
    float2 qo = z2;
    ff2 wo{z2, z2};
    // ---------------- B: the column's faces on time node t ----------------
    if (t >= ta && (fx || fy)) {
      // A_d phi as an unevaluated pair, both lanes
      const float2 pa = sph[hx], pb = sph[hy];
      const ff2 dp = two_diff2(f2(pa.x, pb.x), f2(ph_t.x, ph_t.x));
      const float2 ih = f2(ih1, ih2);
      const float2 gh = mul2(dp.h, ih);
      const float2 gl = mul2(add2(sub2(f2(pa.y, pb.y), f2(ph_t.y, ph_t.y)), dp.l), ih);
      const ff2 al = ff2_pack(a1, a2);
      // sum over the cones reading the face of s (z + beta/sigma): the cone above it on
      // node times t (components 1, 5) and t - 1 (3, 7), the thread's own (2, 6), (4, 8)
      ff2_acc an{z2, z2}, ao{z2, z2};       // beta/sigma of the cone above, of the own cone
      float2 zn = z2, zo = z2;              // their z
      if (t <= T - 1) {
        const int o = (st_c * (K2 / 2) + 1) * kThreads * 4;
        an = ff2_acc{f2(bx[o], by[o]), f2(bx[o + 2], by[o + 2])};
        const ff2 b2 = ff2_of(bslot[(st_c * (K2 / 2) + 2) * kThreads]);
        ao = ff2_acc{b2.h, b2.l};
        zn = f2(sz1[hx].x, sz1[hy].y);
        zo = zc[2];
      }
      if (t >= 1) {
        const int o = (st_p * (K2 / 2) + 3) * kThreads * 4;
        acc2_add(an, ff2{f2(bx[o], by[o]), f2(bx[o + 2], by[o + 2])});
        acc2_add(ao, ff2_of(bslot[(st_p * (K2 / 2) + 4) * kThreads]));
        const int lp = kThreads - lev;
        zn = add2(zn, f2(sz3[lp + hx].x, sz3[lp + hy].y));
        zo = add2(zo, zp4);
      }
      // (the same operations with and without a mask: a solve served among masked ones
      // takes the masked kernel, with every weight 1)
      const float2 so = f2(s, s);
      ff2_acc acc{gh, gl};
      acc2_add(acc, al);
      acc2_add_mul(acc, an, sn);
      acc2_add_mul(acc, ao, so);
      acc2_add_f(acc, fma2(sn, zn, mul2(so, zo)));
      float2 dg = fma2(sn, sn, mul2(so, so));
      if (t >= 1 && t <= T - 1) dg = add2(dg, dg);
      const float2 den = add2(dg, f2(1.f, 1.f));
      const float2 rd = f2(rcp_approx(den.x), rcp_approx(den.y));
      // q = rhs / (1 + sum s^2)
      const float2 q1 = mul2(acc.h, rd);
      const ff2 pr = two_prod2(q1, den);
      qo = fma2(add2(sub2(sub2(acc.h, pr.h), pr.l), acc.c), rd, q1);
      const float2 gm = add2(sub2(gh, qo), gl);
      const ff2 aln = ff2_add_f(al, mul2(ts2, gm));
      wo = two_sum2(aln.h, gm);             // alpha/sigma + A phi - q (unnormalised)
      wo.l = add2(wo.l, aln.l);
      if (!fx) { qo.x = 0.f; wo.h.x = 0.f; wo.l.x = 0.f; }
      if (!fy) { qo.y = 0.f; wo.h.y = 0.f; wo.l.y = 0.f; }
      if (owner) {
        if (fx) {
          a.qn[1][i] = qo.x;
          a.aln[1][i] = ff2_lane0(aln);
        }
        if (fy) {
          a.qn[2][i] = qo.y;
          a.aln[2][i] = ff2_lane1(aln);
        }
      }
    }
    sq[tid] = qo;
    sw[tid] = f4_of(wo);
    // the next time's potential and alpha / sigma of the faces
    ph_t = ph_n;
    if (t + 1 < tb) {
      if (cone_ok && t + 2 <= T) ph_n = a.phi[i + 2 * P];
      if (fx) a1 = a.al[1][i + P];
      if (fy) a2 = a.al[2][i + P];
    }
    __syncthreads();
    if (own_ok && t >= ta) {
      // ---------------- C: beta and the residual at node t ----------------
      const float2 ql = f2(sq[lx].x, sq[ly].y);   // faces below
      const float2 ns2 = f2(-s, -s);
      auto upd = [&](const float4* bt, float4* bn, int k, float2 q, float2 z) {
        const float2 inc = fma2(ns2, q, z);
        socp = fma2(inc, inc, socp);
        bn[(long long)k * n0] = f4_of(ff2_add_f(ff2_of(bt[k * kThreads]), mul2(ts2, inc)));
      };
      if (t < T) {
        const float4* bt = bslot + st_c * (K2 / 2) * kThreads;
        upd(bt, a.betan + (i + obeta), 1, ql, zc[1]);
        upd(bt, a.betan + (i + obeta), 2, qo, zc[2]);
      }
      if (t >= 1) {
        const float4* bt = bslot + st_p * (K2 / 2) * kThreads;
        upd(bt, a.betan + (i + obeta - P), 3, ql, zp3);
        upd(bt, a.betan + (i + obeta - P), 4, qo, zp4);
      }
      // the next iteration's residual at node t: A^* w - c/sigma with w = q - alpha/sigma -
      // A phi of the node's faces (sw and w0 hold -w, zero at the walls)
      {
        const float* wx = reinterpret_cast<const float*>(sw + lx);
        const float* wy = reinterpret_cast<const float*>(sw + ly) + 1;
        const ff2 dw = two_diff2(wo.h, f2(wx[0], wy[0]));
        const float2 dl = add2(dw.l, sub2(wo.l, f2(wx[2], wy[2])));
        const float2 ih = f2(ih1, ih2);
        const ff2 pr = two_prod2(dw.h, ih);
        const float2 pl = fma2(dl, ih, pr.l);
        const float2 sxy = two_sum(pr.h.x, pr.h.y);
        ff_acc acc{sxy.x, sxy.y + (pl.x + pl.y)};
        float2 d0 = z2;
        if (t < T) d0 = w0c;
        if (t >= 1) {
          const float2 e = two_sum(d0.x, -w0p.x);
          d0 = f2(e.x, e.y + (d0.y - w0p.y));
        }
        acc_add_mul(acc, d0, ih0);
        if (t == 0) acc_add(acc, ff_neg(ff_mul(a.c0[slot * P + x * N1 + y], a.sp[slot].isg)));
        if (t == T) acc_add(acc, ff_mul(a.c1[slot * P + x * N1 + y], a.sp[slot].isg));
        a.r[i] = acc.h + acc.c;
      }
    }
    // the squared beta increments of a row's 32 cells over a run that ends with node t
    if (t >= ta && (--left == 0 || t == T)) {
      if (owner) {
        const float2 v = warp_sum_ff(two_sum(socp.x, socp.y));
        if (lane == 0 && x < N0) *entry = v;
        socp = z2;
      }
      entry += (long long)a.nty * N0;
      left = a.run;
    }
    w0p = w0c;
    zp3 = zc[3];
    zp4 = zc[4];
    const int s0 = st_p;
    st_p = st_c;
    st_c = st_n;
    st_n = s0;
    // no barrier here: step A of t + 1 writes z_1, z_3 (of the other level) and phi, last
    // read in step B of t; step B of t + 1, which overwrites the face values read above,
    // follows the barrier after A.  The neighbours read beta of stages t and t - 1 in
    // step B of t; the copies into stage t - 1's place start after the second barrier.
  }
}

// Work units -- a slot's tile and a run of `unit` time nodes -- in the order (active
// slot, tile, time), cut into one contiguous run per CTA: every SM gets the same
// number of nodes whatever the grid, and a CTA crosses from one tile to the next at most
// once more than its share needs.  Each segment projects one cone time more than it owns.
template <int TX, bool MASKED>
__global__ void __launch_bounds__(Tile<TX>::kThreads, 1) k_fused2d(const __grid_constant__ Geo g,
                                                                  const __grid_constant__ FusedArgs a) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ short act[256];
  __shared__ int nact_s;
  const int tid = threadIdx.x;
  if (tid < 32) {   // the active slots, in order
    int n = 0;
    for (int b0 = 0; b0 < a.G; b0 += 32) {
      const int b = b0 + tid;
      const unsigned m = __ballot_sync(0xffffffffu, b < a.G && a.sp[b].active);
      if (m >> tid & 1) act[n + __popc(m & ((1u << tid) - 1))] = (short)b;
      n += __popc(m);
    }
    if (tid == 0) nact_s = n;
  }
  __syncthreads();
  const int ntile = a.ntx * a.nty, nunit = a.nunit, nrun = (g.T + a.run) / a.run;
  const long long total = (long long)nact_s * ntile * nunit;
  long long k = total * blockIdx.x / gridDim.x;
  const long long kend = total * (blockIdx.x + 1) / gridDim.x;
  while (k < kend) {
    const int tl = (int)(k / nunit), u0 = (int)(k - (long long)tl * nunit);
    const int u1 = (int)min((long long)nunit, u0 + (kend - k));
    const int s = tl / ntile, tile = tl - s * ntile;
    const int ty = tile / a.ntx, tx = tile - ty * a.ntx;
    const int slot = act[s];
    segment<TX, MASKED>(g, a, sm, slot, tx * TX, ty * TY, u0 * a.unit, min(g.T + 1, u1 * a.unit),
                        a.socp_part + ((long long)slot * nrun * a.nty + ty) * g.N[0] + tx * TX);
    k += u1 - u0;
  }
}

int ntiles(const Geo& g, int tx) { return ((g.N[0] + tx - 1) / tx) * ((g.N[1] + TY - 1) / TY); }

// Tile rows.  13 is the most (16 warps at 128 registers fill an SM) and has the
// smallest halo; smaller tiles give small grids more CTAs and shorter time steps.
// A CTA's pass takes its share of the time nodes plus the cone time before each segment,
// at a time per step that grows with the rows, so the choice is the least of that product
// (with 1 + 0.2 rows for the step, the fit of these, taken with the sums still in FP64:
// 32^2 x 16 10.3 us with 4 rows, 11.8 with 8, 13.3 with 13; 64^2 x 32 22.5, 20.3, 22.6;
// 96^2 x 16 24.7, 22.0, 22.8; 128^2 x 32 64.0, 47.6, 47.4; 150 x 117 x 37 77.6, 59.4, 59.9).
int rows_of(const Geo& g, int G) {
  const int rows[3] = {13, 8, 4};
  int best = 13;
  double t = 1e300;
  for (int r : rows) {
    const long long w = (long long)G * ntiles(g, r) * (g.T + 1);
    const double e = (double)((w + kSMs - 1) / kSMs + 1) * (1.0 + 0.2 * r);
    if (e < t) { t = e; best = r; }
  }
  return best;
}

// Time nodes to hand out at once: about sixteen units per SM, at most eight.
int share_of(const Geo& g, int G) {
  const long long u = (long long)G * ntiles(g, rows_of(g, G)) * (g.T + 1) / (kSMs * 16);
  return (int)(u < 1 ? 1 : u > 8 ? 8 : u);
}

// Time nodes per partial sum of the squared beta increments: FP32 over a run of one
// cell's nodes, two-float over a row's 32 cells, FP64 from there.  Of the grid alone, as the order of these sums may not
// depend on the batch: they enter the penalty rule, and a served solve takes the steps of
// a solve alone.
int run_of(const Geo& g) { return share_of(g, 1); }
int runs(const Geo& g) { return (g.T + run_of(g)) / run_of(g); }

// Time nodes per work unit: whole runs.
int unit_of(const Geo& g, int G) {
  const int r = run_of(g), u = share_of(g, G) / r * r;
  return u > r ? u : r;
}

template <int TX, bool MASKED>
void launch(const Geo& g, const FusedArgs& a, int nb, cudaStream_t s) {
  static std::atomic<unsigned long long> done{0};
  smem_optin((const void*)k_fused2d<TX, MASKED>, Tile<TX>::kSmem, &done);
  k_fused2d<TX, MASKED><<<nb, Tile<TX>::kThreads, Tile<TX>::kSmem, s>>>(g, a);
}

}  // namespace

bool fused2d_supported(const Geo& g) { return g.D == 2; }

long long fused2d_partials(const Geo& g) { return (long long)runs(g) * ((g.N[1] + TY - 1) / TY) * g.N[0]; }

void launch_fused2d(const Geo& g, int G, const MxFields& f, const MxFields& fn, float2* socp_part, cudaStream_t s,
                    LaunchCounter lc) {
  FusedArgs a;
  for (int d = 0; d < 3; ++d) {
    a.q[d] = f.q[d];
    a.al[d] = f.al[d];
    a.qn[d] = fn.q[d];
    a.aln[d] = fn.al[d];
  }
  a.beta = reinterpret_cast<const float4*>(f.beta);
  a.betan = reinterpret_cast<float4*>(fn.beta);
  a.phi = f.phi;
  a.somega = f.somega;
  a.G = G;
  const int tx = rows_of(g, G);
  a.ntx = (g.N[0] + tx - 1) / tx;
  a.nty = (g.N[1] + TY - 1) / TY;
  a.unit = unit_of(g, G);
  a.nunit = (g.T + a.unit) / a.unit;
  a.run = run_of(g);
  a.sp = f.sp;
  a.socp_part = socp_part;
  a.r = f.r;
  a.c0 = f.c0;
  a.c1 = f.c1;
  a.ih0 = (float)g.invh[0];
  a.ih1 = (float)g.invh[1];
  a.ih2 = (float)g.invh[2];
  const long long units = (long long)G * a.ntx * a.nty * a.nunit;
  const int nb = (int)(units < kSMs ? units : kSMs);
  const bool m = f.somega != nullptr;
  if (tx == 13) m ? launch<13, true>(g, a, nb, s) : launch<13, false>(g, a, nb, s);
  else if (tx == 8) m ? launch<8, true>(g, a, nb, s) : launch<8, false>(g, a, nb, s);
  else m ? launch<4, true>(g, a, nb, s) : launch<4, false>(g, a, nb, s);
  lc.launched(KID_FUSED);
}

}  // namespace dot
