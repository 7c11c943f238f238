// Chip-resident multi-step kernel for grids that fit the SMs' shared memory:
// one cooperative launch advances many steps.
//
// What bounds a small grid is not bytes but the chain launch - global loads -
// arithmetic - stores - launch of every step (5 to 11 us for grids whose
// arithmetic takes 1 to 3 us).  Here every CTA owns one tile of a grid for
// the whole launch and keeps its post-collision populations in shared memory
// (two buffers, step s reads one and writes the other); phi*u and the low
// part of g_0 stay in registers.  Only the tile's rim travels between CTAs,
// through L2, in words that carry their own step tag, so that one polling
// load both waits for a value and delivers it: no fence, no flag, no
// grid-wide barrier.
//
// The rim.  A node's update reads phi and psi of its eight neighbours, and a
// neighbour's phi the nine g pulled to it, so a tile needs the g of two rows
// or columns of nodes around it and the f of one, and of those only the
// populations that move into the tile's one-node surround: per rim node of a
// side the three g entering from two nodes away, the three g that do not
// cross from one node away, the three g and the three f that do.  These four
// triples are the unit of the exchange ("triple": three values of one node).
// In FP32 a triple and its tag are one 16-byte word; in FP64 a triple is
// three words of {value, tag}.  Words are written and read with single
// 128-bit accesses (st/ld.relaxed.gpu.b128), which are not torn.
//
// Slots alternate between two sets (step parity).  A CTA overwrites the slot
// of step s at step s + 2, after it has received step s + 1 from the same
// neighbour, which sent it after consuming step s: one set is never written
// while it is being read.  Tags are unique over the handle's launches.
//
// Measured, us per step of a long run, against the kernels replayed from a
// graph: 128x64 1.58 (was 7.6), 201x101 with walls 1.87 (6.0), 512x256 with
// walls 3.65 (10.9), vortex 256^2 2.10 (8.9), FP64 128x64 9.6 (38).  What
// bounds it now: the latency of exchange and collision on small tiles (about
// 1.6 us; 13% of issue slots), on full ones 540 instructions per node at 45%
// issue with 16 warps and three barriers per step, the FP64 pipe in FP64.  Two
// polling loads in flight instead of one changed nothing: most words have
// come by the first poll.
//
// Per step: collide (shared -> shared), barrier, send the rim, form phi and
// psi of the nodes whose pull needs no rim, receive the rim, barrier, phi and
// psi of the remaining nodes, barrier.  The per-node arithmetic is that of
// the other step kernels (sum9, step_psi, node_update).
//
// Every wait is bounded (StepArgs::wait_cycles); on expiry the CTA raises
// kFlagTimeout and returns, and so do its neighbours in turn.  No asynchronous
// copies are in flight.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "lbm_check.h"
#include "lbm_kernels.cuh"
#include "lbm_layout.h"
#include "lbm_node.cuh"

namespace lbmk {

// Shared memory of a variant: NT threads with R nodes each, PC cells (nodes
// and two-node surround), NX rim triples at most in either direction.
template <typename T, bool COUPLED, int PC, int NX>
struct ResShape {
  static constexpr int NPL = COUPLED ? 18 : 9;  // g 0..8, f 9..17
  static constexpr size_t POP = (size_t)2 * NPL * PC * sizeof(T);
  static constexpr size_t PQ_OFF = (POP + 15) / 16 * 16;
  static constexpr size_t RECV_OFF = PQ_OFF + (size_t)PC * sizeof(typename Pair<T>::type);
  static constexpr size_t SEND_OFF = RECV_OFF + (size_t)NX * sizeof(uint2);
  static constexpr size_t EDGE_OFF = SEND_OFF + (size_t)NX * sizeof(uint2);
  static constexpr size_t CT_OFF = EDGE_OFF + (size_t)NX * sizeof(uint32_t);
  static constexpr size_t SMEM_BYTES = CT_OFF + (COUPLED ? 0 : kResMaxSteps * sizeof(T));
};

// {value(s), tag} words of the exchange.
template <typename T>
struct ResWord;
template <>
struct ResWord<float> {
  static constexpr int PER = 1;  // 16-byte words per triple
  static __device__ __forceinline__ void put(uint4* p, float a, float b, float c, uint32_t tag) {
    const uint64_t lo = (uint64_t)__float_as_uint(a) | ((uint64_t)__float_as_uint(b) << 32);
    const uint64_t hi = (uint64_t)__float_as_uint(c) | ((uint64_t)tag << 32);
    asm volatile("{.reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t;}" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
  }
  static __device__ __forceinline__ bool get(const uint4* p, float& a, float& b, float& c,
                                             uint32_t tag) {
    uint64_t lo, hi;
    asm volatile("{.reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t;}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    a = __uint_as_float((uint32_t)lo);
    b = __uint_as_float((uint32_t)(lo >> 32));
    c = __uint_as_float((uint32_t)hi);
    return (uint32_t)(hi >> 32) == tag;
  }
};
template <>
struct ResWord<double> {
  static constexpr int PER = 3;
  static __device__ __forceinline__ void put1(uint4* p, double a, uint32_t tag) {
    asm volatile("{.reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t;}" ::"l"(p),
                 "l"((uint64_t)__double_as_longlong(a)), "l"((uint64_t)tag)
                 : "memory");
  }
  static __device__ __forceinline__ bool get1(const uint4* p, double& a, uint32_t tag) {
    uint64_t lo, hi;
    asm volatile("{.reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t;}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    a = __longlong_as_double((long long)lo);
    return hi == (uint64_t)tag;
  }
  static __device__ __forceinline__ void put(uint4* p, double a, double b, double c,
                                             uint32_t tag) {
    put1(p, a, tag);
    put1(p + 1, b, tag);
    put1(p + 2, c, tag);
  }
  static __device__ __forceinline__ bool get(const uint4* p, double& a, double& b, double& c,
                                             uint32_t tag) {
    const bool x = get1(p, a, tag), y = get1(p + 1, b, tag), z = get1(p + 2, c, tag);
    return x && y && z;
  }
};

// A triple's three planes (g 0..8, f 9..17) and its cell, in one word.
__device__ __forceinline__ uint32_t res_desc(int cell, int p0, int p1, int p2) {
  return (uint32_t)cell | ((uint32_t)p0 << 12) | ((uint32_t)p1 << 17) | ((uint32_t)p2 << 22);
}

template <typename T, bool COUPLED, int NT, int R, int PC, int NX, int MINB, bool PLAIN>
__global__ void __launch_bounds__(NT, MINB)
    step_resident(const StepArgs<T> a, const ResTile* __restrict__ tiles, const ResRun run) {
  using SH = ResShape<T, COUPLED, PC, NX>;
  using Word = ResWord<T>;
  constexpr int NPL = SH::NPL;
  extern __shared__ __align__(128) unsigned char smem[];
  T* cur = reinterpret_cast<T*>(smem);
  T* nxt = cur + (size_t)NPL * PC;
  typename Pair<T>::type* const pq = reinterpret_cast<typename Pair<T>::type*>(smem + SH::PQ_OFF);
  uint2* const rdesc = reinterpret_cast<uint2*>(smem + SH::RECV_OFF);   // {slot, triple}
  uint2* const sdesc = reinterpret_cast<uint2*>(smem + SH::SEND_OFF);
  uint32_t* const edesc = reinterpret_cast<uint32_t*>(smem + SH::EDGE_OFF);
  T* const ctab = reinterpret_cast<T*>(smem + SH::CT_OFF);
  __shared__ int nrecv_s, nsend_s;

  const int tid = threadIdx.x;
  const ResTile tl = tiles[blockIdx.x];
  const CaseDev<T>* __restrict__ cdp = a.cases + tl.c;
  const int nx = cdp->nx, ny = cdp->ny, w = tl.w, h = tl.h, pw = w + 4;
  const uint32_t P = (uint32_t)cdp->plane, nn = (uint32_t)nx * (uint32_t)ny;
  const bool walls = cdp->walls != 0;
  const bool wbot = walls && tl.y0 == 0, wtop = walls && tl.y0 + h == ny;
  const T xi = a.ph.xi;
  auto cell_of = [&](int x, int y) -> int { return (y + 2) * pw + x + 2; };

  const T* gs = cdp->g[a.parity];
  const T* fs = COUPLED ? cdp->f[a.parity] : nullptr;

  // ---- start: populations of the tile and its two-node surround ------------
  if (tid == 0) nrecv_s = nsend_s = 0;
  {
    const int ncell = pw * (h + 4);
    for (int q = tid; q < ncell; q += NT) {
      const int ly = q / pw - 2, lx = q % pw - 2;
      int x = tl.x0 + lx, y = tl.y0 + ly;
      x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
      if (walls) y = y < 0 ? 0 : (y >= ny ? ny - 1 : y);  // beyond a wall: not read
      else y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
      const uint32_t node = (uint32_t)y * (uint32_t)nx + (uint32_t)x;
      if (!LBM_BOUND(a.flags, node, nn)) continue;
#pragma unroll
      for (int i = 0; i < 9; ++i) cur[i * PC + q] = gs[i * P + node];
      if (COUPLED) {
#pragma unroll
        for (int i = 0; i < 9; ++i) cur[(9 + i) * PC + q] = fs[i * P + node];
      }
    }
  }
  __syncthreads();  // nrecv_s, nsend_s
  // ---- the rim: what to send and what to receive ---------------------------
  // A tile's slots: strip W (5 triples per row: the four of the header
  // comment and one for wall rows), E, then S and N (4 per column).
  for (int q = tid; q < 10 * h + 8 * w; q += NT) {
    int k, cell, p0, p1, p2;
    bool use;
    if (q < 10 * h) {
      const bool west = q < 5 * h;
      const int u = west ? q : q - 5 * h, y = u / 5;
      k = u - 5 * y;
      const int col = west ? (k == 0 ? 1 : 0) : (k == 0 ? w - 2 : w - 1);
      cell = cell_of(col, y);
      const bool fwd = west == (k == 4);  // triple moving east (c_x = +1)
      p0 = k == 1 ? 0 : (fwd ? 1 : 3);
      p1 = k == 1 ? 2 : (fwd ? 5 : 6);
      p2 = k == 1 ? 4 : (fwd ? 8 : 7);
      use = k < 3 || (k == 3 && COUPLED) || (k == 4 && ((wbot && y == 0) || (wtop && y == h - 1)));
    } else {
      const bool south = q < 10 * h + 4 * w;
      const int u = q - 10 * h - (south ? 0 : 4 * w), x = u >> 2;
      k = u & 3;
      cell = cell_of(x, south ? (k == 0 ? 1 : 0) : (k == 0 ? h - 2 : h - 1));
      p0 = k == 1 ? 0 : (south ? 4 : 2);
      p1 = k == 1 ? 1 : (south ? 7 : 5);
      p2 = k == 1 ? 3 : (south ? 8 : 6);
      use = (k < 3 || COUPLED) && !(south ? wbot : wtop);
    }
    if (!use) continue;
    if (k == 3) p0 += 9, p1 += 9, p2 += 9;
    const int at = atomicAdd(&nsend_s, 1);
    if (LBM_BOUND(a.flags, at, NX)) sdesc[at] = make_uint2(tl.slot + (uint32_t)q, res_desc(cell, p0, p1, p2));
  }
  for (int q = tid; q < 10 * (h + 4) + 8 * w; q += NT) {
    int k, cell, p0, p1, p2;
    uint32_t slot;
    bool use;
    if (q < 10 * (h + 4)) {
      const bool west = q < 5 * (h + 4);
      const int u = west ? q : q - 5 * (h + 4), y = u / 5 - 2;
      k = u % 5;
      const int lower = y < 0, upper = y >= h;
      // the tile beside this one, or diagonally below or above it
      const int hn = lower ? tl.hS : (upper ? tl.hN : h);
      const int row = lower ? hn + y : (upper ? y - h : y);
      const int nb = (west ? kResW : kResE) + (lower ? 1 : (upper ? 2 : 0));
      slot = tl.nb[nb] + (uint32_t)((west ? 5 * hn : 0) + 5 * row + k);
      cell = cell_of(west ? (k == 0 ? -2 : -1) : (k == 0 ? w + 1 : w), y);
      const bool fwd = west != (k == 4);
      p0 = k == 1 ? 0 : (fwd ? 1 : 3);
      p1 = k == 1 ? 2 : (fwd ? 5 : 6);
      p2 = k == 1 ? 4 : (fwd ? 8 : 7);
      use = !(lower && wbot) && !(upper && wtop) &&
            (k < 3 || (k == 3 && COUPLED && y >= -1 && y <= h) ||
             (k == 4 && ((wbot && y == 0) || (wtop && y == h - 1))));
    } else {
      const bool south = q < 10 * (h + 4) + 4 * w;
      const int u = q - 10 * (h + 4) - (south ? 0 : 4 * w), x = u >> 2;
      k = u & 3;
      slot = south ? tl.nb[kResS] + (uint32_t)(10 * tl.hS + 4 * w + u)
                   : tl.nb[kResN] + (uint32_t)(10 * tl.hN + u);
      cell = cell_of(x, south ? (k == 0 ? -2 : -1) : (k == 0 ? h + 1 : h));
      p0 = k == 1 ? 0 : (south ? 2 : 4);
      p1 = k == 1 ? 1 : (south ? 5 : 7);
      p2 = k == 1 ? 3 : (south ? 6 : 8);
      use = (k < 3 || COUPLED) && !(south ? wbot : wtop);
    }
    if (!use) continue;
    if (k == 3) p0 += 9, p1 += 9, p2 += 9;
    const int at = atomicAdd(&nrecv_s, 1);
    if (LBM_BOUND(a.flags, at, NX)) rdesc[at] = make_uint2(slot, res_desc(cell, p0, p1, p2));
  }
  // ---- nodes whose phi and psi need the rim: the two outermost rings of the
  // (w + 2) x (h + 2) nodes; {target cell, source cell, wall row below, above}
  const int nedge = 4 * (w + h);
  for (int q = tid; q < nedge; q += NT) {
    int x, y;
    if (q < 4 * (w + 2)) {
      const int r = q / (w + 2);
      y = r < 2 ? r - 1 : h - 3 + r;
      x = q - r * (w + 2) - 1;
    } else {
      const int u = q - 4 * (w + 2), c = u / (h - 2);
      x = c < 2 ? c - 1 : w - 3 + c;
      y = 1 + u - c * (h - 2);
    }
    // beyond a wall: the ghost row mirrors the wall row
    const int ys = (wbot && y < 0) ? 0 : ((wtop && y >= h) ? h - 1 : y);
    edesc[q] = (uint32_t)cell_of(x, y) | ((uint32_t)cell_of(x, ys) << 12) |
               ((wbot && ys == 0) ? 1u << 24 : 0u) | ((wtop && ys == h - 1) ? 1u << 25 : 0u);
  }
  if (!COUPLED) {  // U cos(pi t / T) of every step of the launch
    for (int s = tid; s < run.nsteps; s += NT)
      ctab[s] = (T)(cospi((double)(run.t0 + s) / a.ph.vT) * a.ph.vU);
  }

  // ---- own nodes -------------------------------------------------------------
  CaseK<T> K;
  K.rho_g = cdp->rho_g;
  K.drho = cdp->drho;
  K.mu_g = cdp->mu_g;
  K.dmu = cdp->dmu;
  K.sD7 = cdp->sD7;
  K.hD7 = cdp->hD7;
  K.var_tau = cdp->var_tau != 0;
  K.ny = ny;
  K.ct = K.sx2 = K.s2x = K.s2y = K.sy2 = T(0);
  constexpr bool LO = sizeof(T) == 4;
  T jx[R], jy[R], lo[R], sx2[R], s2x[R], s2y[R], sy2[R];
  int cel[R];  // cell of node r, or -1
  // what the step needs to know of node r, found once: bit 0 no rim needed for
  // its phi, bits 1, 2 wall row below, above
  uint32_t kind[R];
  uint32_t gnode[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int k = tid + r * NT;
    const bool act = k < w * h;
    const int ly = act ? k / w : 0, lx = act ? k - ly * w : 0;
    cel[r] = act ? cell_of(lx, ly) : -1;
    kind[r] = ((lx >= 1 && lx <= w - 2 && ly >= 1 && ly <= h - 2) ? 1u : 0u) |
              ((wbot && ly == 0) ? 2u : 0u) | ((wtop && ly == h - 1) ? 4u : 0u);
    const uint32_t node = (uint32_t)(tl.y0 + ly) * (uint32_t)nx + (uint32_t)(tl.x0 + lx);
    gnode[r] = node;
    const bool ok = act && LBM_BOUND(a.flags, node, nn);
    jx[r] = ok ? cdp->J[a.parity][node] : T(0);
    jy[r] = ok ? cdp->J[a.parity][P + node] : T(0);
    lo[r] = (LO && ok) ? cdp->g0lo[a.parity][node] : T(0);
    sx2[r] = s2x[r] = s2y[r] = sy2[r] = T(0);
    if (!COUPLED) {
      vortex_row(K, tl.y0 + ly);
      s2y[r] = K.s2y;
      sy2[r] = K.sy2;
      T s, c;
      Num<T>::sincospi_((T(tl.x0 + lx) + T(0.5)) / T(nx), &s, &c);
      sx2[r] = s * s;
      s2x[r] = T(2) * s * c;
    }
  }
  __syncthreads();
  const int nrecv = nrecv_s, nsend = nsend_s;

  // pull of the nine populations of planes PL..PL+8 to a cell; at a wall row
  // the populations from beyond the wall are the cell's own opposite ones
  auto pull = [&](const T* b, int c, bool bt, bool tp, T v[9]) {
    const T* m = b + c - pw;
    const T* o = b + c;
    const T* p = b + c + pw;
    v[0] = o[0];
    v[1] = o[1 * PC - 1];
    v[3] = o[3 * PC + 1];
    v[2] = m[2 * PC];
    v[5] = m[5 * PC - 1];
    v[6] = m[6 * PC + 1];
    v[4] = p[4 * PC];
    v[7] = p[7 * PC + 1];
    v[8] = p[8 * PC - 1];
    if (COUPLED && (bt || tp)) {
      if (bt) v[2] = o[4 * PC], v[5] = o[7 * PC], v[6] = o[8 * PC];
      if (tp) v[4] = o[2 * PC], v[7] = o[5 * PC], v[8] = o[6 * PC];
    }
  };
  auto phase_a = [&](const T* b, int src, int dst, bool bt, bool tp) {
    T G[9];
    pull(b, src, bt, tp, G);
    const T phi = sum9(G);
    typename Pair<T>::type v;
    v.x = phi;
    v.y = step_psi<PLAIN>(phi, xi);
    pq[dst] = v;
  };
  // own nodes away from the tile's edge: no rim needed
  auto phase_inner = [&](const T* b) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (cel[r] >= 0 && (kind[r] & 1u)) phase_a(b, cel[r], cel[r], false, false);
    }
  };
  auto phase_edge = [&](const T* b) {
    for (int q = tid; q < nedge; q += NT) {
      const uint32_t e = edesc[q];
      phase_a(b, (e >> 12) & 0xFFFu, e & 0xFFFu, (e >> 24) & 1u, (e >> 25) & 1u);
    }
  };
  // one state plane value of the record (lbm_snapshot layout)
  auto record = [&](int slot, int r, const T* F, const T* G) {
    T* out = (T*)run.rec + (int64_t)slot * run.rec_stride + gnode[r];
#pragma unroll
    for (int i = 0; i < 9; ++i) out[(int64_t)i * nn] = COUPLED ? F[i] : T(0);
#pragma unroll
    for (int i = 0; i < 9; ++i) out[(int64_t)(9 + i) * nn] = G[i];
    out[(int64_t)18 * nn] = jx[r];
    out[(int64_t)19 * nn] = jy[r];
    if (LO) out[(int64_t)20 * nn] = lo[r];
  };
  if (run.rec) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (cel[r] < 0) continue;
      T F[9], G[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        G[i] = cur[i * PC + cel[r]];
        F[i] = COUPLED ? cur[(9 + i) * PC + cel[r]] : T(0);
      }
      record(0, r, F, G);
    }
  }

  phase_inner(cur);
  phase_edge(cur);
  __syncthreads();

  uint4* const slots = reinterpret_cast<uint4*>(run.slots);
  for (int s = 0; s < run.nsteps; ++s) {
    // ---- collide the own nodes ---------------------------------------------
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (cel[r] < 0) continue;
      const int c = cel[r];
      const bool bt = kind[r] & 2u, tp = kind[r] & 4u;
      T F[9], G[9];
      pull(cur, c, bt, tp, G);
      if (COUPLED) pull(cur + (size_t)9 * PC, c, bt, tp, F);
      Stencil<T> S;
      {
        const auto v = pq[c], e = pq[c + 1], ww = pq[c - 1];
        const auto n = pq[c + pw], ne = pq[c + pw + 1], nw = pq[c + pw - 1];
        const auto so = pq[c - pw], se = pq[c - pw + 1], sw = pq[c - pw - 1];
        S.p = v.x;
        S.pE = e.x, S.pW = ww.x, S.pN = n.x, S.pS = so.x;
        S.pNE = ne.x, S.pNW = nw.x, S.pSE = se.x, S.pSW = sw.x;
        S.qE = e.y, S.qW = ww.y, S.qN = n.y, S.qS = so.y;
        S.qNE = ne.y, S.qNW = nw.y, S.qSE = se.y, S.qSW = sw.y;
      }
      if (COUPLED && (bt || tp))
        wall_momentum(F, K.rho_g + S.p * K.drho, bt, tp, cdp->u_bot, cdp->u_top);
      if (!COUPLED) {
        K.ct = ctab[s];
        K.sx2 = sx2[r];
        K.s2x = s2x[r];
        K.s2y = s2y[r];
        K.sy2 = sy2[r];
      }
      const NodeOut<T> o =
          node_update<T, COUPLED, kModeStep, PLAIN>(a.ph, K, F, G, lo[r], jx[r], jy[r], S);
      jx[r] = o.Jx;
      jy[r] = o.Jy;
#pragma unroll
      for (int i = 0; i < 9; ++i) nxt[i * PC + c] = G[i];
      if (COUPLED) {
#pragma unroll
        for (int i = 0; i < 9; ++i) nxt[(9 + i) * PC + c] = F[i];
      }
      // (a trial's later steps are not states of the handle)
      if (!isfinite(S.p + o.ux + o.uy + o.p) && run.store == 1) atomicOr(a.flags, kFlagNonFinite);
      if (run.rec && s + 1 < run.nsteps) record(s + 1, r, F, G);
    }
    if (s + 1 == run.nsteps) break;
    __syncthreads();
    // ---- exchange the rim ------------------------------------------------------
    const uint32_t tag = run.epoch + (uint32_t)s;
    const uint32_t set = (s & 1) ? run.nslots : 0u;
    for (int q = tid; q < nsend; q += NT) {
      const uint2 d = sdesc[q];
      const T* src = nxt + (d.y & 0xFFFu);
      if (LBM_BOUND(a.flags, d.x, run.nslots))
        Word::put(slots + (size_t)(set + d.x) * Word::PER, src[((d.y >> 12) & 31u) * PC],
                  src[((d.y >> 17) & 31u) * PC], src[((d.y >> 22) & 31u) * PC], tag);
    }
    phase_inner(nxt);
    bool bad = false;
    for (int q = tid; q < nrecv; q += NT) {
      const uint2 d = rdesc[q];
      if (!LBM_BOUND(a.flags, d.x, run.nslots)) continue;
      const uint4* p = slots + (size_t)(set + d.x) * Word::PER;
      T v0, v1, v2;
      if (!Word::get(p, v0, v1, v2, tag)) {
        const long long c0 = clock64();
        bool got = false;
        while (!got && clock64() - c0 < a.wait_cycles) got = Word::get(p, v0, v1, v2, tag);
        bad = bad || !got;
      }
      T* dst = nxt + (d.y & 0xFFFu);
      dst[((d.y >> 12) & 31u) * PC] = v0;
      dst[((d.y >> 17) & 31u) * PC] = v1;
      dst[((d.y >> 22) & 31u) * PC] = v2;
    }
    if (__syncthreads_or(bad)) {
      if (tid == 0) atomicOr(a.flags, kFlagTimeout);
      if (run.store == 1 && blockIdx.x == 0 && tid == 0) *run.t_dev = run.t0 + run.nsteps;
      return;
    }
    phase_edge(nxt);
    __syncthreads();
    T* const t = cur;
    cur = nxt;
    nxt = t;
  }

  // ---- end: the state to its planes ----------------------------------------
  // An even number of steps ends in the buffer the launch started from: every
  // neighbour has read it, since its first words came after its initial loads.
  if (!run.store) return;
  const int dst = a.parity ^ (run.nsteps & 1);
  T* gd = cdp->g[dst];
  T* fd = COUPLED ? cdp->f[dst] : nullptr;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (cel[r] < 0) continue;
    T F[9], G[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      G[i] = nxt[i * PC + cel[r]];
      F[i] = COUPLED ? nxt[(9 + i) * PC + cel[r]] : T(0);
    }
    NodeOut<T> o;
    o.Jx = jx[r];
    o.Jy = jy[r];
    store_node<T, COUPLED>(fd, gd, cdp->J[dst], cdp->g0lo[dst], P, gnode[r], F, G, lo[r], o,
                           a.flags, nn);
  }
  if (run.store == 1 && blockIdx.x == 0 && tid == 0) *run.t_dev = run.t0 + run.nsteps;
}

}  // namespace lbmk
