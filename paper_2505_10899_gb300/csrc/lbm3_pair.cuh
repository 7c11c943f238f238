// Per-node arithmetic of the 3-D step for two nodes adjacent in x at a time,
// in packed FP32 instructions (two values in a 64-bit register pair, one
// issue slot).  The strip kernel (lbm3_strip.cuh) is bound by instruction
// issue in FP16 storage, so it costs what its instructions count.
//
// The same equations as node3, in fewer operations:
//   - a pair (c, -c) of f: f*_{+-} = f + (s - w_f S/2) +- (v - w_f D/2), with
//       S, D the pair's sum and difference,
//       s = w w_f base + (c.u) [4.5 w w_f rho (c.u) + 3 w h_f (c.grad rho)],
//       v = c.[3 w (w_f rho u + h_f F)],
//     the bracketed vectors formed once per weight;
//   - the stencil's column sums and differences serve both nodes, phi and psi
//     packed.
// What a node conserves must not be scaled by a constant that is off by a
// rounding: every step would scale it again (rho u by 3e-8 w_f a step with the
// FP32 1/6, 1e-5 after 200 steps).  So base and w_f rho u + h_f F, which differ
// from node to node and so round either way, are divided by 18 and 6 with the
// constants' low parts; and f takes the small change of a collision, with one
// rounding at its own size and w_f unrounded at any relaxation time (a complement
// 1 - w_f loses a bit of it per doubling of tau_f above 2).
// Error against 64 bits, mean of 24 boxes of 64 x 40 x 40, FP32, register kernel /
// complement and rounded constants / this form:
//   column, tau_f 0.6: phi 4.96e-8 / 4.91e-8 / 4.87e-8, u 4.0e-6 / 7.5e-6 / 9.3e-7,
//                      p 1.9e-6 / 2.9e-6 / 3.4e-7
//   ball, tau_f 1:     phi 3.4e-7 / 2.9e-7 / 6.4e-8, u 2.7e-6 / 2.6e-6 / 3.5e-7,
//                      p 8.1e-6 / 1.0e-5 / 6.7e-6
//   ball, tau_f 9.3:   phi 6.4e-8 / 6.3e-8 / 4.9e-8, u 3.0e-7 / 2.5e-7 / 7.0e-8,
//                      p 6.3e-6 / 5.7e-6 / 5.0e-6
// It costs 1.8% in FP16 storage and 0.4% in FP32 (lbm3_strip.cuh).
//
// Multiplications and additions are fused where written, not by the compiler.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "lbm3_kernels.cuh"

namespace lbmk3 {

__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {  // one rounding, as a - b
  return __fadd2_rn(a, make_float2(-b.x, -b.y));
}

// Values at p - CX and p + 1 - CX (p even: without a shift one aligned load).
template <int CX>
__device__ __forceinline__ float2 ld2(const float* p) {
  if constexpr (CX == 0) return *reinterpret_cast<const float2*>(p);
  return make_float2(p[-CX], p[1 - CX]);
}
template <int CX>
__device__ __forceinline__ float2 ld2(const __half* p) {
  if constexpr (CX == 0) return __half22float2(*reinterpret_cast<const __half2*>(p));
  return make_float2(__half2float(p[-CX]), __half2float(p[1 - CX]));
}
__device__ __forceinline__ void st2(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
__device__ __forceinline__ void st2(__half* p, float2 v) {
  *reinterpret_cast<__half2*>(p) = __float22half2_rn(v);
}
template <typename S>
__device__ __forceinline__ float2 round2(float2 v) {
  if constexpr (sizeof(S) == 2) return __half22float2(__float22half2_rn(v));
  return v;
}

// Four consecutive (phi, psi) cells, 16-byte aligned.
__device__ __forceinline__ void row4(const float2* p, float2 (&v)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 2);
  v[0] = make_float2(a.x, a.y);
  v[1] = make_float2(a.z, a.w);
  v[2] = make_float2(b.x, b.y);
  v[3] = make_float2(b.z, b.w);
}

// phi, 12 grad(phi), lap(phi) and 12 grad(psi) of the two nodes.
struct Pair2 {
  float2 phi, gx, gy, gz, lap, qx, qy, qz;
};

// Stencils of the nodes in columns 1 and 2 of C: rows north (N) and south
// (S) of the same plane, the same row of the planes above (U) and below (D),
// and the rows beside those (columns 1 and 2).
__device__ __forceinline__ void stencils2(const float2 (&C)[4], const float2 (&N)[4],
                                          const float2 (&S)[4], const float2 (&U)[4],
                                          const float2 (&D)[4], const float2 (&un)[2],
                                          const float2 (&us)[2], const float2 (&dn)[2],
                                          const float2 (&ds)[2], Pair2& o) {
  float2 ns[4], ud[4], Y[4], dy[4], dz[4], g[3][2];
  float lap[2];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    ns[c] = add2(N[c], S[c]);
    ud[c] = add2(U[c], D[c]);
    Y[c] = add2(ns[c], ud[c]);
    dy[c] = sub2(N[c], S[c]);
    dz[c] = sub2(U[c], D[c]);
  }
  const float2 two = both(2.0f);
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    const int w = n, c = n + 1, e = n + 2;
    g[0][n] = fma2(two, sub2(C[e], C[w]), sub2(Y[e], Y[w]));
    g[1][n] = fma2(two, dy[c],
                   add2(add2(dy[w], dy[e]), add2(sub2(un[n], us[n]), sub2(dn[n], ds[n]))));
    g[2][n] = fma2(two, dz[c],
                   add2(add2(dz[w], dz[e]), add2(sub2(un[n], dn[n]), sub2(us[n], ds[n]))));
    // lap = (1/3) sum_axis (chi_n - chi) + (1/6) sum_diag (chi_n - chi)
    const float ax = ((C[e].x + C[w].x) + ns[c].x) + ud[c].x;
    const float di = (Y[w].x + Y[e].x) + ((un[n].x + us[n].x) + (dn[n].x + ds[n].x));
    lap[n] = 1.0f / 3.0f * fmaf(-6.0f, C[c].x, ax) + 1.0f / 6.0f * fmaf(-12.0f, C[c].x, di);
  }
  o.phi = make_float2(C[1].x, C[2].x);
  o.gx = make_float2(g[0][0].x, g[0][1].x);
  o.gy = make_float2(g[1][0].x, g[1][1].x);
  o.gz = make_float2(g[2][0].x, g[2][1].x);
  o.qx = make_float2(g[0][0].y, g[0][1].y);
  o.qy = make_float2(g[1][0].y, g[1][1].y);
  o.qz = make_float2(g[2][0].y, g[2][1].y);
  o.lap = make_float2(lap[0], lap[1]);
}

// x / 18 and x / 6 without the rounding of the constants.
__device__ __forceinline__ float2 over18(float2 x) {
  constexpr float c = 1.0f / 18.0f;
  return fma2(x, both(c), mul2(x, both((float)(1.0 / 18.0 - (double)c))));
}
__device__ __forceinline__ float2 over6(float2 x) {
  constexpr float c = 1.0f / 6.0f;
  return fma2(x, both(c), mul2(x, both((float)(1.0 / 6.0 - (double)c))));
}

// One population pair (c, -c): f*_{+-} = f + (s - w_f S/2) +- (v - w_f D/2), S
// and D the pair's sum and difference (see above; wh = -w_f/2).
__device__ __forceinline__ void pair_f2(float2& fp, float2& fm, float2 cu, float2 cR, float2 v,
                                        float2 k, float2 A, float2 wh) {
  const float2 S = add2(fp, fm), D = sub2(fp, fm);
  const float2 e = fma2(wh, S, fma2(cu, fma2(k, cu, cR), A)), o = fma2(wh, D, v);
  fp = add2(fp, add2(e, o));
  fm = add2(fm, sub2(e, o));
}

// Both collisions at two nodes (node3, kModeStep).  Returns a value that is
// finite where phi and u are; J = phi u.
template <typename S>
__device__ __forceinline__ float2 node3_pair(const Args3<float, S>& a, float2 (&F)[19],
                                             float2 (&G)[7], float2& Glo, const float2 (&jp)[3],
                                             const Pair2& N, float2 (&J)[3]) {
  const float2 phi = N.phi, half = both(0.5f), one = both(1.0f);
  const float2 k12 = both(1.0f / 12.0f);
  const float2 gpx = mul2(N.gx, k12), gpy = mul2(N.gy, k12), gpz = mul2(N.gz, k12);
  // chemical potential (Eq. 2) and surface force F = hbar grad(phi)
  const float2 mu =
      fma2(both(-a.kappa), N.lap,
           mul2(mul2(mul2(both(a.beta4), phi), add2(phi, both(-1.0f))), add2(phi, both(-0.5f))));
  const float2 Fx = mul2(mu, gpx), Fy = mul2(mu, gpy), Fz = mul2(mu, gpz);
  const float2 rho = fma2(phi, both(a.drho), both(a.rho_g));
  const float2 irho = make_float2(N3<float>::rcp(rho.x), N3<float>::rcp(rho.y));

  float2 d[9], s[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    d[k] = sub2(F[2 * k + 1], F[2 * k + 2]);
    s[k] = add2(F[2 * k + 1], F[2 * k + 2]);
  }
  const float2 jx = add2(add2(d[0], d[3]), add2(d[4], add2(d[5], d[6])));
  const float2 jy = add2(add2(d[1], d[3]), sub2(add2(d[7], d[8]), d[4]));
  const float2 jz = add2(add2(d[2], d[5]), sub2(sub2(d[7], d[6]), d[8]));
  const float2 snz = add2(add2(add2(add2(s[0], s[1]), add2(s[2], s[3])),
                               add2(add2(s[4], s[5]), add2(s[6], s[7]))),
                          s[8]);
  const float2 ux = mul2(fma2(half, Fx, jx), irho);  // Eq. 28
  const float2 uy = mul2(fma2(half, Fy, jy), irho);
  const float2 uz = mul2(fma2(half, Fz, jz), irho);
  const float2 dr = both(a.drho);  // grad(rho)
  const float2 Rx = mul2(dr, gpx), Ry = mul2(dr, gpy), Rz = mul2(dr, gpz);
  const float2 uR = fma2(uz, Rz, fma2(uy, Ry, mul2(ux, Rx)));
  const float2 ru2 = mul2(rho, fma2(uz, uz, fma2(uy, uy, mul2(ux, ux))));
  // Eq. 29 on D3Q19: c_s^2/(1-w0) = 1/2, rho s_0(u) = -rho |u|^2/2
  const float2 p = mul2(half, fma2(both(-0.5f), ru2, fma2(half, uR, snz)));

  float2 wf = both(a.wf), hf = both(a.hf);
  if (a.var_tau) {
    const float2 m = mul2(both(3.0f), fma2(phi, both(a.dmu), both(a.mu_g)));
    const float2 tau = fma2(m, irho, half);  // Eq. 27
    wf = make_float2(N3<float>::rcp(tau.x), N3<float>::rcp(tau.y));
    hf = fma2(both(-0.5f), wf, one);
  }
  // rest population: f_eq,0 = (w0 - 1) p / c_s^2 + rho s_0 = -2p - rho u^2/2; F_0 = 0
  F[0] = fma2(wf, sub2(fma2(both(-2.0f), p, mul2(both(-0.5f), ru2)), F[0]), F[0]);
  const float2 wh = mul2(both(-0.5f), wf);
  // the pairs' sums and differences are formed again below: kept, their 36
  // registers spill at three CTAs per SM
#pragma unroll
  for (int i = 1; i < 19; ++i) asm volatile("" : "+f"(F[i].x), "+f"(F[i].y));
  const float2 base = fma2(both(3.0f), p, mul2(both(-1.5f), ru2));
  const float2 h6 = mul2(both(1.0f / 6.0f), hf);  // 3 w h_f, w = 1/18
  float2 A = mul2(wf, over18(base));
  float2 k = mul2(both(0.25f), mul2(wf, rho));  // 4.5 w w_f rho
  float2 rx = mul2(h6, Rx), ry = mul2(h6, Ry), rz = mul2(h6, Rz);
  float2 vx = over6(fma2(wf, mul2(rho, ux), mul2(hf, Fx))),
         vy = over6(fma2(wf, mul2(rho, uy), mul2(hf, Fy))),
         vz = over6(fma2(wf, mul2(rho, uz), mul2(hf, Fz)));
  pair_f2(F[1], F[2], ux, rx, vx, k, A, wh);
  pair_f2(F[3], F[4], uy, ry, vy, k, A, wh);
  pair_f2(F[5], F[6], uz, rz, vz, k, A, wh);
  A = mul2(half, A), k = mul2(half, k);  // w = 1/36
  rx = mul2(half, rx), ry = mul2(half, ry), rz = mul2(half, rz);
  vx = mul2(half, vx), vy = mul2(half, vy), vz = mul2(half, vz);
  pair_f2(F[7], F[8], add2(ux, uy), add2(rx, ry), add2(vx, vy), k, A, wh);
  pair_f2(F[9], F[10], sub2(ux, uy), sub2(rx, ry), sub2(vx, vy), k, A, wh);
  pair_f2(F[11], F[12], add2(ux, uz), add2(rx, rz), add2(vx, vz), k, A, wh);
  pair_f2(F[13], F[14], sub2(ux, uz), sub2(rx, rz), sub2(vx, vz), k, A, wh);
  pair_f2(F[15], F[16], add2(uy, uz), add2(ry, rz), add2(vy, vz), k, A, wh);
  pair_f2(F[17], F[18], sub2(uy, uz), sub2(ry, rz), sub2(vy, vz), k, A, wh);

  // ---- phase field: SRT limit of Eq. 33 on D3Q7 (c_s^2 = 1/4) ----
  J[0] = mul2(phi, ux), J[1] = mul2(phi, uy), J[2] = mul2(phi, uz);
  const float2 pc = make_float2(N3<float>::clamp01(phi.x), N3<float>::clamp01(phi.y));
  const float2 ta = add2(pc, both(a.xi)), tb = add2(sub2(one, pc), both(a.xi));
  const float2 q2 = fma2(N.qz, N.qz, fma2(N.qy, N.qy, mul2(N.qx, N.qx)));
  // n := 0 on ridges of psi
  const float2 iq = make_float2(q2.x >= a.qmin2 ? N3<float>::rsq(q2.x) : 0.0f,
                                q2.y >= a.qmin2 ? N3<float>::rsq(q2.y) : 0.0f);
  // (1/4) (lambda/W)[1 - tanh^2(2 psi/W)] / |grad psi|, 1 - tanh^2 = 4ab/(a+b)^2
  const float2 sh = mul2(mul2(mul2(both(0.25f * (a.lamW * a.tfac)), ta), tb), iq);
  const float2 Vx = fma2(sh, N.qx, sub2(J[0], jp[0]));
  const float2 Vy = fma2(sh, N.qy, sub2(J[1], jp[1]));
  const float2 Vz = fma2(sh, N.qz, sub2(J[2], jp[2]));
  // movers: g + w_g (w_i (hbar + lambda phi) +- (1/2) c.J - g) +- h_g (1/2) c.V, the
  // small differences first: one rounding at the size of g (the phase field
  // keeps what it rounds; with a complement 1 - w_g phi's error after 200 steps of
  // a 256^3 column is 5.3e-8, so 5.0e-8)
  const float2 L8 = mul2(both(0.125f), fma2(both(a.lambda), phi, mu));
  float2 H[7];
  auto movers = [&](float2 gp, float2 gm, float2 Jc, float2 V, float2& hp, float2& hm) {
    const float2 w = both(a.wg), mhalf = both(-0.5f);
    const float2 tp = fma2(half, Jc, sub2(L8, gp)), tm = fma2(mhalf, Jc, sub2(L8, gm));
    hp = round2<S>(add2(gp, fma2(w, tp, mul2(both(0.5f * a.hg), V))));
    hm = round2<S>(add2(gm, fma2(w, tm, mul2(both(-0.5f * a.hg), V))));
  };
  movers(G[1], G[2], J[0], Vx, H[1], H[2]);
  movers(G[3], G[4], J[1], Vy, H[3], H[4]);
  movers(G[5], G[6], J[2], Vz, H[5], H[6]);
  // rest population from the conserved zeroth moment (node3): the stored
  // changes of the movers, added to the pair (g_0, lo) with a TwoSum
  const float2 dg = add2(add2(sub2(G[1], H[1]), sub2(G[2], H[2])),
                         add2(add2(sub2(G[3], H[3]), sub2(G[4], H[4])),
                              add2(sub2(G[5], H[5]), sub2(G[6], H[6]))));
  const float2 b = add2(Glo, dg), hi = add2(G[0], b), bb = sub2(hi, G[0]);
  Glo = add2(sub2(G[0], sub2(hi, bb)), sub2(b, bb));
  G[0] = hi;
#pragma unroll
  for (int i = 1; i < 7; ++i) G[i] = H[i];
  return add2(phi, add2(add2(ux, uy), uz));
}

}  // namespace lbmk3
