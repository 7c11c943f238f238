// Chip-resident reverse sweep (FP32, coupled flow) for grids that fit the
// SMs' shared memory: one cooperative launch runs many adjoint steps over
// recorded states, as the forward kernel of lbm_resident.cuh runs many steps.
//
// Two launches per adjoint step (ad_node, ad_gather) spend their time on
// latency: 50 planes through L2 per node and step, a tail of 1.1 waves, the
// launches themselves.  Here a CTA keeps the adjoint state of its tile in
// shared memory; the recorded states are read from global memory, where every
// CTA reads its own halo; only adjoint values cross between tiles, in the
// tagged words of lbm_resident.cuh.
//
// Per step, for the state S_t: phi and psi of the tile and its one-node
// surround; the reverse arithmetic at the own nodes (ad_node_math), which
// leaves per node the adjoints of its 18 pulled populations and of its
// stencil differences (grad phi, lap phi, grad psi: five values) and of its
// phi; the exchange; per node the total adjoint of phi from the stencil
// adjoints of its neighbours (the sums of gather_uses, in its order).  The
// adjoint of the population that position p holds is then that of the node
// p + c_i that pulls it plus that node's phi total, formed where the next
// step reads it.  A tile needs the stencil adjoints of two rows or columns
// around it, and of one the phi adjoint and the populations that move into
// it: six triples per rim node (k = 0..5 below).
//
// Parameter terms: the sums of a warp's 32 nodes in R, as in ad_node, one per
// step and node of a thread; they accumulate in FP64, lanes 4q .. 4q+3 of a warp
// holding parameter q, and enter the CTA's slots in warp order at the end.  They
// count only if no wait of the sweep gave up (ad_commit).
//
// Measured, us per adjoint step (two launches per step -> here): 512 x 256 with
// walls 23.9 -> 11.6, 384 x 192 21.8 -> 7.8, 201 x 101 with walls 22.6 -> 4.9,
// 128 x 64 21.3 -> 4.5.  What bounds it: instruction issue and the latency of
// the recorded state's loads (27 a node) on full tiles, the exchange and four
// barriers on small ones.
#pragma once

// Threads, nodes per thread, cells with a two-node surround, rim triples; and
// the cells with a one-node surround: (w + 4)(h + 4) <= 1224 makes w + h >= 62
// or the tile smaller, so (w + 2)(h + 2) <= 1088.
constexpr int kAdNT = lbmk::kResAdjoint.nt, kAdR = lbmk::kResAdjoint.r;
constexpr int kAdV = lbmk::kResAdjoint.pc, kAdNX = lbmk::kResAdjoint.nx, kAdL = 1088;

struct AdShape {
  static constexpr size_t V_OFF = (size_t)2 * 18 * kAdL * sizeof(float);
  static constexpr size_t PQ_OFF = V_OFF + (size_t)6 * kAdV * sizeof(float);
  static constexpr size_t TOT_OFF = PQ_OFF + (size_t)kAdL * sizeof(float2);
  static constexpr size_t XY_OFF = TOT_OFF + (size_t)kAdL * sizeof(float);
  static constexpr size_t RECV_OFF = XY_OFF + (size_t)kAdL * sizeof(uint32_t);
  static constexpr size_t SEND_OFF = RECV_OFF + (size_t)kAdNX * sizeof(uint2);
  static constexpr size_t SMEM_BYTES = SEND_OFF + (size_t)kAdNX * sizeof(uint2);
};
static_assert(AdShape::SMEM_BYTES + 1024 <= 227 * 1024, "shared memory of one CTA");

struct AdRun {
  const float* states;   // recorded states, S_{t0 + j} at states + j * stride
  int64_t stride;        // elements
  int count;             // adjoint steps
  uint32_t epoch, nslots;
  uint4* slots;
  int prefetch;          // the launch's states exceed what L2 keeps
  float* adj;            // adjoint of S_{t0 + count} in, of S_{t0} out
  double* pend;          // [CTAs][kNParam] parameter sums, added to by launches
  int first;             // of one sweep after the first
  long long wait_cycles;
  int32_t* flags;
};

// Rim triple k of a strip: first value's plane.  Planes 0..8 lG, 9..17 lF,
// 18..22 the stencil adjoints, 23 the phi adjoint.
__device__ __forceinline__ void ad_triple(int k, int d0, int d1, int d2, int& p0, int& p1, int& p2) {
  if (k < 4) {  // k = 0, 2: first three stencil adjoints; 1, 3: the others and phi
    p0 = (k & 1) ? 21 : 18;
    p1 = (k & 1) ? 22 : 19;
    p2 = (k & 1) ? 23 : 20;
  } else {
    const int f = k == 4 ? 9 : 0;
    p0 = f + d0, p1 = f + d1, p2 = f + d2;
  }
}

__global__ void __launch_bounds__(kAdNT, 1)
    ad_resident(const AdArgs<float> a, const lbmk::ResTile* __restrict__ tiles, const AdRun run) {
  using R = float;
  using Word = lbmk::ResWord<float>;
  extern __shared__ __align__(128) unsigned char smem[];
  R* cur = reinterpret_cast<R*>(smem);  // [18][kAdL] adjoints of the pulled populations
  R* nxt = cur + 18 * kAdL;
  R* const V = reinterpret_cast<R*>(smem + AdShape::V_OFF);  // [6][kAdV]
  float2* const pq = reinterpret_cast<float2*>(smem + AdShape::PQ_OFF);
  R* const tot = reinterpret_cast<R*>(smem + AdShape::TOT_OFF);
  uint32_t* const gxy = reinterpret_cast<uint32_t*>(smem + AdShape::XY_OFF);
  uint2* const rdesc = reinterpret_cast<uint2*>(smem + AdShape::RECV_OFF);
  uint2* const sdesc = reinterpret_cast<uint2*>(smem + AdShape::SEND_OFF);
  __shared__ int nrecv_s, nsend_s;
  __shared__ double red[kAdNT / 32][kNParam];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const lbmk::ResTile tl = tiles[blockIdx.x];
  const int nx = a.nx, ny = a.ny, w = tl.w, h = tl.h, pl = w + 2, pv = w + 4;
  const int n = nx * ny;
  const bool walls = a.walls != 0;
  const bool wbot = walls && tl.y0 == 0, wtop = walls && tl.y0 + h == ny;
  auto lcell = [&](int x, int y) -> int { return (y + 1) * pl + x + 1; };
  auto vcell = [&](int x, int y) -> int { return (y + 2) * pv + x + 2; };
  const int ncell = pl * (h + 2);

  if (tid == 0) nrecv_s = nsend_s = 0;
  // global node of every cell of the one-node surround (beyond a wall: 0xFFFF
  // in y, not used)
  for (int q = tid; q < ncell; q += kAdNT) {
    int x = tl.x0 + q % pl - 1, y = tl.y0 + q / pl - 1;
    x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
    if (walls && (y < 0 || y >= ny)) y = 0xFFFF;
    else y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
    gxy[q] = (uint32_t)x | ((uint32_t)y << 16);
  }
  __syncthreads();
  // rim tables: {slot, x + 2 | y + 2 << 10 | k << 20 | side << 23}; side 0..3:
  // west, east, south, north (of the strip that is sent, of the halo received)
  for (int q = tid; q < 12 * (h + w); q += kAdNT) {
    int x, y, k, side;
    if (q < 12 * h) {
      side = q < 6 * h ? 0 : 1;
      const int u = q - side * 6 * h;
      y = u / 6, k = u - 6 * y;
      const int far = k == 2 || k == 3;
      x = side == 0 ? far : w - 1 - far;
    } else {
      side = q < 12 * h + 6 * w ? 2 : 3;
      const int u = q - 12 * h - (side - 2) * 6 * w;
      x = u / 6, k = u - 6 * x;
      const int far = k == 2 || k == 3;
      y = side == 2 ? far : h - 1 - far;
      if (side == 2 ? wbot : wtop) continue;
    }
    const int at = atomicAdd(&nsend_s, 1);
    if (at < kAdNX)
      sdesc[at] = make_uint2(tl.slot + (uint32_t)q, (uint32_t)(x + 2) | ((uint32_t)(y + 2) << 10) |
                                                        ((uint32_t)k << 20) | ((uint32_t)side << 23));
    else
      atomicOr(run.flags, lbmk::kFlagBounds);  // no plan gives such a tile
  }
  for (int q = tid; q < 12 * (h + 4) + 12 * w; q += kAdNT) {
    int x, y, k, side;
    uint32_t slot;
    if (q < 12 * (h + 4)) {
      side = q < 6 * (h + 4) ? 0 : 1;
      const int u = q - side * 6 * (h + 4);
      y = u / 6 - 2, k = u % 6;
      const int lower = y < 0, upper = y >= h;
      if ((lower && wbot) || (upper && wtop)) continue;
      const int hn = lower ? tl.hS : (upper ? tl.hN : h);
      const int row = lower ? hn + y : (upper ? y - h : y);
      const int nb = (side == 0 ? lbmk::kResW : lbmk::kResE) + (lower ? 1 : (upper ? 2 : 0));
      // from the neighbour's strip on the side that faces this tile
      slot = tl.nb[nb] + (uint32_t)((side == 0 ? 6 * hn : 0) + 6 * row + k);
      const int far = k == 2 || k == 3;
      x = side == 0 ? -1 - far : w + far;
      if (k >= 4 && (y < -1 || y > h)) continue;  // populations: one row beyond
    } else {
      side = q < 12 * (h + 4) + 6 * w ? 2 : 3;
      const int u = q - 12 * (h + 4) - (side - 2) * 6 * w;
      x = u / 6, k = u - 6 * x;
      if (side == 2 ? wbot : wtop) continue;
      slot = side == 2 ? tl.nb[lbmk::kResS] + (uint32_t)(12 * tl.hS + 6 * w + u)
                       : tl.nb[lbmk::kResN] + (uint32_t)(12 * tl.hN + u);
      const int far = k == 2 || k == 3;
      y = side == 2 ? -1 - far : h + far;
    }
    const int at = atomicAdd(&nrecv_s, 1);
    if (at < kAdNX)
      rdesc[at] = make_uint2(slot, (uint32_t)(x + 2) | ((uint32_t)(y + 2) << 10) |
                                       ((uint32_t)k << 20) | ((uint32_t)side << 23));
    else
      atomicOr(run.flags, lbmk::kFlagBounds);
  }
  __syncthreads();
  const int nrecv = min(nrecv_s, kAdNX), nsend = min(nsend_s, kAdNX);

  // own nodes
  int lx[kAdR], ly[kAdR];
  R aJx[kAdR], aJy[kAdR];
  bool act[kAdR];
#pragma unroll
  for (int r = 0; r < kAdR; ++r) {
    const int k = tid + r * kAdNT;
    act[r] = k < w * h;
    ly[r] = act[r] ? k / w : 0;
    lx[r] = act[r] ? k - ly[r] * w : 0;
    const int node = (tl.y0 + ly[r]) * nx + tl.x0 + lx[r];
    const bool ok = LBM_BOUND(run.flags, node, n);
    aJx[r] = ok ? run.adj[18 * n + node] : R(0);
    aJy[r] = ok ? run.adj[19 * n + node] : R(0);
  }
  static_assert(kNParam <= 8, "a warp's parameter sums");
  double pacc = 0.0;  // lanes 4q .. 4q+3: parameter q of this warp

  // adjoint of the population in plane i (0..8 g, 9..17 f) at own position (x, y)
  auto pulled = [&](const R* L, int i, int f, int x, int y, bool bt, bool tp) -> R {
    const bool back = (bt && kAY(i) == -1) || (tp && kAY(i) == 1);  // bounced: own opposite
    const int c = back ? lcell(x, y) : lcell(x + kAX(i), y + kAY(i));
    const R v = L[((f ? 9 : 0) + (back ? kAOPP(i) : i)) * kAdL + c];
    return f ? v : v + tot[c];
  };

  for (int j = run.count - 1; j >= 0; --j) {
    const R* __restrict__ st = run.states + (int64_t)j * run.stride;
    const R* __restrict__ fA = st;
    const R* __restrict__ gA = st + 9 * (int64_t)n;
    const R* __restrict__ JA = st + 18 * (int64_t)n;
    const bool first = j == run.count - 1;
    // ---- phi and psi of S_t on the tile and its surround --------------------
    for (int q = tid; q < ncell; q += kAdNT) {
      const uint32_t xy = gxy[q];
      const int x = xy & 0xFFFFu, y = xy >> 16;
      if (y == 0xFFFF) continue;
      R G[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        int p;
        const int pos = ad_src(i, x, y, nx, ny, a.walls, &p);
        G[i] = LBM_BOUND(run.flags, pos, n) ? __ldg(gA + p * n + pos) : R(0);
      }
      const R phi = lbmk::sum9(G);
      pq[q] = make_float2(phi, lbmk::psi_of(phi, a.ph.xi));
    }
    __syncthreads();
    // ---- the reverse arithmetic at the own nodes ------------------------------
#pragma unroll
    for (int r = 0; r < kAdR; ++r) {
      R gacc[kNParam] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
      if (act[r]) {
        const int x = tl.x0 + lx[r], y = tl.y0 + ly[r], c = lcell(lx[r], ly[r]);
        const int node = y * nx + x;
        const bool bt = walls && y == 0, tp = walls && y == ny - 1;
        R F[9], G[9], Pv[9], Qv[9], aF[9], aG[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          int p;
          const int pos = ad_src(i, x, y, nx, ny, a.walls, &p);
          const bool ok = LBM_BOUND(run.flags, pos, n);
          G[i] = ok ? __ldg(gA + p * n + pos) : R(0);
          F[i] = ok ? __ldg(fA + p * n + pos) : R(0);
        }
        const bool okn = LBM_BOUND(run.flags, node, n);
        const R jpx = okn ? __ldg(JA + node) : R(0), jpy = okn ? __ldg(JA + n + node) : R(0);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          // beyond a wall the ghost row mirrors the wall row
          const int dy = (bt && kAY(i) == -1) || (tp && kAY(i) == 1) ? 0 : kAY(i);
          const float2 v = pq[c + dy * pl + kAX(i)];
          Pv[i] = v.x;
          Qv[i] = v.y;
        }
        if (bt || tp) {
          const R rw = a.rho_g + Pv[0] * a.drho;
          if (bt) {
            const R d = rw * a.u_bot * R(1.0 / 6.0);
            F[5] += d;
            F[6] -= d;
          }
          if (tp) {
            const R d = rw * a.u_top * R(1.0 / 6.0);
            F[7] -= d;
            F[8] += d;
          }
        }
        if (first) {
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            aF[i] = okn ? run.adj[i * n + node] : R(0);
            aG[i] = okn ? run.adj[(9 + i) * n + node] : R(0);
          }
        } else {
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            aF[i] = pulled(cur, i, 1, lx[r], ly[r], bt, tp);
            aG[i] = pulled(cur, i, 0, lx[r], ly[r], bt, tp);
          }
        }
        const AdOut<R> o =
            ad_node_math(a, x, y, F, G, jpx, jpy, Pv, Qv, aF, aG, aJx[r], aJy[r], bt, tp, gacc);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          nxt[i * kAdL + c] = o.lG[i];
          nxt[(9 + i) * kAdL + c] = o.lF[i];
        }
        const int v = vcell(lx[r], ly[r]);
        V[v] = o.lgpx;
        V[kAdV + v] = o.lgpy;
        V[2 * kAdV + v] = o.llap;
        V[3 * kAdV + v] = o.lqx;
        V[4 * kAdV + v] = o.lqy;
        V[5 * kAdV + v] = R(-10.0 / 3.0) * o.llap + o.lphi;
        aJx[r] = o.ljpx;
        aJy[r] = o.ljpy;
      }
      // parameter terms: 32 nodes' sums in R, accumulated in FP64.  Every
      // exchange halves the values a lane holds, so lanes 4q .. 4q+3 end with
      // parameter q: 9 shuffles for a warp's 8 sums.
      R sum[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) sum[q] = q < kNParam ? gacc[q < kNParam ? q : 0] : R(0);
#pragma unroll
      for (int o = 16, m = 4; m > 0; o >>= 1, m >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int q = 0; q < m; ++q) {
          const R send = up ? sum[q] : sum[q + m], keep = up ? sum[q + m] : sum[q];
          sum[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], 2);
      sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], 1);
      pacc += (double)sum[0];
    }
    __syncthreads();
    // ---- exchange ---------------------------------------------------------------
    const uint32_t tag = run.epoch + (uint32_t)j;
    const uint32_t set = (j & 1) ? run.nslots : 0u;
    for (int q = tid; q < nsend; q += kAdNT) {
      const uint2 d = sdesc[q];
      if (!LBM_BOUND(run.flags, d.x, run.nslots)) continue;
      const int x = (int)(d.y & 1023u) - 2, y = (int)((d.y >> 10) & 1023u) - 2;
      const int k = (d.y >> 20) & 7u, side = (d.y >> 23) & 3u;
      int p0, p1, p2;
      // the populations that the neighbour's positions wait for: those whose
      // position p = q - c_i lies beyond this side
      if (side == 0) ad_triple(k, 1, 5, 8, p0, p1, p2);
      else if (side == 1) ad_triple(k, 3, 6, 7, p0, p1, p2);
      else if (side == 2) ad_triple(k, 2, 5, 6, p0, p1, p2);
      else ad_triple(k, 4, 7, 8, p0, p1, p2);
      if (k < 4) {
        const R* s = V + vcell(x, y);
        Word::put(run.slots + set + d.x, s[(p0 - 18) * kAdV], s[(p1 - 18) * kAdV],
                  s[(p2 - 18) * kAdV], tag);
      } else {
        const R* s = nxt + lcell(x, y);
        Word::put(run.slots + set + d.x, s[p0 * kAdL], s[p1 * kAdL], s[p2 * kAdL], tag);
      }
    }
    // The next state's tile on its way from HBM to L2, while the rim travels.
    // Only for sweeps over more states than L2 keeps: there it hides the HBM
    // latency (512 x 256: 13.0 -> 11.6 us per step), else it only adds
    // instructions (128 x 64: 4.3 -> 4.6).
    if (j > 0 && run.prefetch) {
      const int lines = (w + 31) / 32 + 1;
      for (int q = tid; q < 20 * h * lines; q += kAdNT) {
        const int row = q / lines, pl_ = row / h;
        const int64_t at = (int64_t)pl_ * n + (tl.y0 + row - pl_ * h) * nx + tl.x0 +
                           min((q - row * lines) * 32, w - 1);
        if (LBM_BOUND(run.flags, at, 20 * (int64_t)n))
          asm volatile("prefetch.global.L2 [%0];" ::"l"(st - run.stride + at));
      }
    }
    bool bad = false;
    auto place = [&](uint32_t d, const R (&v)[3]) {
      const int x = (int)(d & 1023u) - 2, y = (int)((d >> 10) & 1023u) - 2;
      const int k = (d >> 20) & 7u, side = (d >> 23) & 3u;
      int p0, p1, p2;
      if (side == 0) ad_triple(k, 3, 6, 7, p0, p1, p2);
      else if (side == 1) ad_triple(k, 1, 5, 8, p0, p1, p2);
      else if (side == 2) ad_triple(k, 4, 7, 8, p0, p1, p2);
      else ad_triple(k, 2, 5, 6, p0, p1, p2);
      R* s = k < 4 ? V + vcell(x, y) : nxt + lcell(x, y);
      const int st = k < 4 ? kAdV : kAdL, off = k < 4 ? 18 : 0;
      s[(p0 - off) * st] = v[0];
      s[(p1 - off) * st] = v[1];
      s[(p2 - off) * st] = v[2];
    };
    for (int q = tid; q < nrecv; q += 2 * kAdNT) {
      const bool two = q + kAdNT < nrecv;
      const uint2 d = rdesc[q], e = two ? rdesc[q + kAdNT] : d;
      if (!LBM_BOUND(run.flags, d.x, run.nslots) || !LBM_BOUND(run.flags, e.x, run.nslots)) continue;
      R v[3], u[3];
      const uint4 *p = run.slots + set + d.x, *p2 = run.slots + set + e.x;
      bool dv = Word::get(p, v[0], v[1], v[2], tag);
      bool du = !two || Word::get(p2, u[0], u[1], u[2], tag);
      const long long c0 = clock64();
      while (!(dv && du) && clock64() - c0 < run.wait_cycles) {
        if (!dv) dv = Word::get(p, v[0], v[1], v[2], tag);
        if (!du) du = Word::get(p2, u[0], u[1], u[2], tag);
      }
      bad = bad || !(dv && du);
      place(d.y, v);
      if (two) place(e.y, u);
    }
    if (__syncthreads_or(bad)) {
      if (tid == 0) atomicOr(run.flags, lbmk::kFlagTimeout);
      return;
    }
    // ---- phi totals of the tile and its surround (the order of gather_uses) ---
    for (int q = tid; q < ncell; q += kAdNT) {
      const int yg = gxy[q] >> 16;
      if (yg == 0xFFFF) continue;
      const int x = q % pl - 1, y = q / pl - 1, c = vcell(x, y);
      R sp = V[5 * kAdV + c], sq = R(0);
      auto use = [&](int i, int s) {
        const R lgpx = V[s], lgpy = V[kAdV + s], llap = V[2 * kAdV + s];
        const R lqx = V[3 * kAdV + s], lqy = V[4 * kAdV + s];
        const R gx3 = lgpx * R(1.0 / 3.0), gy3 = lgpy * R(1.0 / 3.0);
        const R gx12 = lgpx * R(1.0 / 12.0), gy12 = lgpy * R(1.0 / 12.0);
        const R la = R(2.0 / 3.0) * llap, ld6 = llap * R(1.0 / 6.0);
        const R P = i == 1   ? gx3 + la
                    : i == 3 ? -gx3 + la
                    : i == 2 ? gy3 + la
                    : i == 4 ? -gy3 + la
                    : i == 5 ? gx12 + gy12 + ld6
                    : i == 6 ? -gx12 + gy12 + ld6
                    : i == 7 ? -gx12 - gy12 + ld6
                             : gx12 - gy12 + ld6;
        const R Q = i == 1   ? R(4) * lqx
                    : i == 3 ? R(-4) * lqx
                    : i == 2 ? R(4) * lqy
                    : i == 4 ? R(-4) * lqy
                    : i == 5 ? lqx + lqy
                    : i == 6 ? -lqx + lqy
                    : i == 7 ? -lqx - lqy
                             : lqx - lqy;
        sp += P;
        sq += Q;
      };
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        const bool low = walls && yg - kAY(i) < 0, high = walls && yg - kAY(i) >= ny;
        if (!low && !high) use(i, c - kAY(i) * pv - kAX(i));
        // a wall row reads its own row through the ghost row beyond the wall
        if (walls && ((yg == 0 && kAY(i) == -1) || (yg == ny - 1 && kAY(i) == 1)))
          use(i, c - kAX(i));
      }
      const R p = pq[q].x;
      const R dpsi = (p > R(0) && p < R(1)) ? dpsi_dphi(p, a.ph.xi) : R(0);
      tot[q] = sp + dpsi * sq;
    }
    __syncthreads();
    R* const t = cur;
    cur = nxt;
    nxt = t;
  }

  // ---- end: the adjoint of S_t0, and the CTA's parameter sums ----------------
#pragma unroll
  for (int r = 0; r < kAdR; ++r) {
    if (!act[r]) continue;
    const int y = tl.y0 + ly[r], node = y * nx + tl.x0 + lx[r];
    const bool bt = walls && y == 0, tp = walls && y == ny - 1;
    if (!LBM_BOUND(run.flags, node, n)) continue;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      run.adj[i * n + node] = pulled(cur, i, 1, lx[r], ly[r], bt, tp);
      run.adj[(9 + i) * n + node] = pulled(cur, i, 0, lx[r], ly[r], bt, tp);
    }
    run.adj[18 * n + node] = aJx[r];
    run.adj[19 * n + node] = aJy[r];
  }
  if ((lane & 3) == 0 && (lane >> 2) < kNParam) red[warp][lane >> 2] = pacc;
  __syncthreads();
  if (tid < kNParam) {
    double v = 0.0;
    for (int q = 0; q < kAdNT / 32; ++q) v += red[q][tid];
    double* const s = run.pend + (int64_t)blockIdx.x * kNParam + tid;
    *s = run.first ? v : *s + v;
  }
}
