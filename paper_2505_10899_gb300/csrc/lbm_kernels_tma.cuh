// Staged step kernel (grids whose width nx is a multiple of 16 bytes of the
// working type and at least 4).
//
// Work decomposition is that of step_kernel (a CTA owns a strip of BX
// columns and marches down `nrows` rows), but the populations reach shared
// memory by asynchronous 16-byte copies instead of registers: for every row
// the CTA needs, its threads copy the pulled source rows (r - c_iy) of every
// population plane over columns [x0, x0+wact), the chunks beside them that the
// pull reads (periodic in x), and phi*u of the previous step.  Completion is
// counted on one mbarrier per stage.  S stages form a ring; rows are fetched
// S-1 ahead of the collision, so the consumer threads seldom wait on DRAM
// latency.  The halo columns of the phi/psi ring come from the same staged
// rows, without extra global loads.
//
// Why threads copy and not the bulk engine: a bulk copy takes its operands
// from uniform registers, so the 20 and more rows of a stage (512 bytes each)
// were issued lane after lane by one warp, for which the others waited.  A
// thread's 5 or 6 chunk copies are spread over the CTA.  FP32, 512 uneven cases
// with per-step volumes, 32 steps 41.6 -> 38.5 ms; 8192 x 4096 grid, 32 steps
// 31.7 -> 30.0 ms.  FP64 is bound by its pipe (18.4 ms either way for 64 uneven
// cases).  What bounds it now: HBM (0.87 of the measured copy rate on the
// large grid, the state's read-out included).
//
// Every wait of the consumers is bounded (StepArgs::wait_cycles); on expiry
// the CTA raises kFlagTimeout, waits for its own copies still in flight
// (bounded by kWaitCycles, whatever wait_cycles is, so that no CTA leaves
// while a copy into its shared memory is pending) and returns.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "lbm_layout.h"
#include "lbm_node.cuh"
#include "lbm_tma.cuh"

namespace lbmk {


// D2Q9 velocity components (Eq. 19) as compile-time functions of i.
__host__ __device__ constexpr int cx_of(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
}
__host__ __device__ constexpr int cy_of(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
}

template <typename T, int BX, bool COUPLED, int MODE, int S>
struct TmaShape {
  static constexpr int SEG = BX + 8;                 // staged columns per plane
  static constexpr int NPL = COUPLED ? 18 : 9;        // population planes
  static constexpr int NJ = (MODE == kModeStep) ? 2 : 0;  // phi*u planes
  static constexpr int STAGE = NPL * SEG + NJ * BX;   // elements per stage
  static constexpr int NPAD_G = 12, NPAD = COUPLED ? 18 : 12;  // chunks beside the strip: g, all
  static constexpr size_t STAGE_BYTES = (size_t)STAGE * sizeof(T);
  static constexpr size_t BAR_OFF = S * STAGE_BYTES;
  static constexpr size_t RING_OFF = (BAR_OFF + S * 8 + 127) / 128 * 128;
  static constexpr size_t VRED_OFF = RING_OFF + sizeof(Ring<T, BX>);
  static constexpr size_t SMEM_BYTES = VRED_OFF + (BX / 32) * sizeof(double);
  static_assert(STAGE_BYTES % 16 == 0, "stage must keep 16-byte alignment");
  static_assert((SEG * sizeof(T)) % 16 == 0, "plane segment must keep 16-byte alignment");
};

// The kernel body, for strips that hold a whole row (FROW: x0 = 0 and
// nx <= BX) or not; the kernel picks one per CTA, so that the strips of wide
// rows keep compile-time staged positions.
template <typename T, int BX, bool COUPLED, int MODE, int S, bool FROW, bool PLAIN>
__device__ __forceinline__ void tma_body(const StepArgs<T>& a, uint4* const rows) {
  using SH = TmaShape<T, BX, COUPLED, MODE, S>;
  constexpr int SEG = SH::SEG, NPL = SH::NPL, NJ = SH::NJ, STAGE = SH::STAGE;
  extern __shared__ __align__(128) unsigned char smem[];
  T* const stages = reinterpret_cast<T*>(smem);
  uint64_t* const bars = reinterpret_cast<uint64_t*>(smem + SH::BAR_OFF);
  Ring<T, BX>& ring = *reinterpret_cast<Ring<T, BX>*>(smem + SH::RING_OFF);
  double* const vred = reinterpret_cast<double*>(smem + SH::VRED_OFF);

  const Item it = a.items[blockIdx.x];
  const CaseDev<T>* __restrict__ cdp = a.cases + it.c;
  const int nx = cdp->nx, ny = cdp->ny;
  const uint32_t P = (uint32_t)cdp->plane;
  const int x0 = it.x0, y0 = it.y0, nrows = it.nrows;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wact = min(BX, nx - x0);
  const bool act = tid < wact;
  const int xc = act ? x0 + tid : x0;

  const T* __restrict__ gs = cdp->g[a.parity];
  T* __restrict__ gd = cdp->g[a.parity ^ 1];
  const T* __restrict__ fs = COUPLED ? cdp->f[a.parity] : nullptr;
  T* __restrict__ fd = COUPLED ? cdp->f[a.parity ^ 1] : nullptr;
  const T* __restrict__ Js = cdp->J[a.parity];
  T* __restrict__ Jd = cdp->J[a.parity ^ 1];
  // FP32: low part of g_0, read at the own node only (not staged: the ring's
  // phi is the plain sum of the nine staged values; the exact rest
  // population in node_update uses it)
  const T* __restrict__ los = cdp->g0lo[a.parity];
  T* __restrict__ lod = cdp->g0lo[a.parity ^ 1];

  // halo columns of the phi/psi ring: local column -1 (thread 0) and wact
  // (thread BX-1), both inside the staged segments
  const bool hthr = (tid == 0) || (tid == BX - 1);
  const int hcol = (tid == 0) ? -1 : wact;
  const int hslot = (tid == 0) ? 0 : wact + 1;
  // A strip that holds the whole row (x0 = 0, nx <= BX) stages the row once,
  // columns 0..nx-1 at positions 4..nx+3, and reads the periodic neighbours
  // of its edge columns from the other end of the same copy; other strips
  // stage global column x0 - 4 + j at position j.  Staged position of local
  // column c + d, d = -1, 0, +1 (the pull sources of c_x = +1, 0, -1):
  constexpr bool frow = FROW;
  auto spos = [&](int c, int d) -> int {
    int j = c + d;
    if (frow) j = j < 0 ? j + nx : (j >= nx ? j - nx : j);
    return j + 4;
  };
  const int om = spos(tid, -1), o0 = spos(tid, 0), op = spos(tid, 1);
  const int hm = spos(hcol, -1), h0 = spos(hcol, 0), hp = spos(hcol, 1);

  const T xi = a.ph.xi;
  const bool do_vol = (MODE == kModeStep) && (a.vol_part != nullptr);
  double vacc = 0.0;
  CaseK<T> K = case_consts<T, COUPLED>(a, cdp, xc);

  auto wrap = [&](int r) -> int { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
  auto slot_of = [](int k) -> int { return (k + 1) % S; };
  auto parity_of = [](int k) -> uint32_t { return (uint32_t)(((k + 1) / S) & 1); };
  auto stage_of = [&](int k) -> T* { return stages + slot_of(k) * STAGE; };

  // What a row copies, described once per CTA: the planes' own columns (g 0-8,
  // f 9-17, phi*u), and the chunks left and right of them that the pull reads
  // (wrapped at x = 0 and x = nx): left the g planes with c_x >= 0 (the halo
  // column -1 pulls from -1 - c_x) and the f planes with c_x = +1 (column 0
  // pulls from -1), right the mirror image.  {plane address, element offset in
  // a stage, column and which of rows r, r-1, r+1}.
  constexpr int E = 16 / (int)sizeof(T);  // elements of a chunk
  constexpr int CC = BX / E;              // chunks of a strip's columns
  constexpr int NPAD_G = SH::NPAD_G, NPAD = SH::NPAD;
  auto desc = [&](const T* plane, int at, int x, int cy) {
    const uint64_t p = reinterpret_cast<uint64_t>(plane);
    return make_uint4((uint32_t)p, (uint32_t)(p >> 32), (uint32_t)at,
                      ((uint32_t)x << 2) | (cy == 0 ? 0u : (cy == 1 ? 1u : 2u)));
  };
  if (tid < NPL + NJ) {
    const int i = tid < 9 ? tid : tid - 9;
    rows[tid] = tid < NPL ? desc((tid < 9 ? gs : fs) + (size_t)i * P, tid * SEG + 4, x0, cy_of(i))
                          : desc(Js + (size_t)(tid - NPL) * P, NPL * SEG + (tid - NPL) * BX, x0, 0);
  }
  for (int q = tid; q < NPAD; q += BX) {
    // planes, four bits each: g left 0 1 2 4 5 8, right 0 2 3 4 6 7; f left 1 5 8, right 3 6 7
    const bool g = q < NPAD_G, left = g ? q < 6 : q < NPAD_G + 3;
    const int u = g ? (left ? q : q - 6) : (left ? q - NPAD_G : q - NPAD_G - 3);
    const int i = (int)(((g ? (left ? 0x854210u : 0x764320u) : (left ? 0x851u : 0x763u)) >> (4 * u)) & 15u);
    const int x = left ? (x0 == 0 ? nx : x0) - E : (x0 + wact >= nx ? 0 : x0 + wact);
    rows[NPL + NJ + q] = desc((g ? gs : fs) + (size_t)i * P,
                              (g ? i : 9 + i) * SEG + (left ? 4 - E : 4 + wact), x, cy_of(i));
  }
  if (tid == 0) {
    for (int s = 0; s < S; ++s) mbar_init(&bars[s], BX);
    fence_mbar_init();
  }
  __syncthreads();

  // Issue the copies of local row k (k in [-1, nrows]): 16-byte chunks, one
  // per thread and pass, a thread keeping its chunk of the strip.  Rows -1 and
  // nrows (the halo rows of the item) need the g planes only.  Every thread
  // arrives once on the stage's barrier, when its own copies have landed.
  auto issue = [&](int k) {
    const bool full = (k >= 0 && k < nrows);
    T* const st = stage_of(k);
    const uint32_t st32 = smem_u32(st);
    const int r = wrap(y0 + k);
    [[maybe_unused]] const uint32_t nn = (uint32_t)nx * (uint32_t)ny;
    const uint32_t r0 = (uint32_t)r * (uint32_t)nx, rm = (uint32_t)wrap(r - 1) * (uint32_t)nx,
                   rp = (uint32_t)wrap(r + 1) * (uint32_t)nx;  // pull: source row r - c_iy
    // (checked build: the source must lie in the plane's nodes and the target
    // in this stage; otherwise the copy is redirected, see lbm_check.h)
    auto copy = [&](const uint4 d, uint32_t c) {
      const uint32_t code = d.w & 3u;
      const uint32_t first = (code == 0 ? r0 : (code == 1 ? rm : rp)) + (d.w >> 2) + c;
      const uint64_t plane = ((uint64_t)d.y << 32) | d.x;
      const bool ok = LBM_BOUND(a.flags, first + (E - 1), nn) &&
                      LBM_BOUND(a.flags, d.z + c + (E - 1), STAGE);
      copy16_g2s(st32 + (ok ? (d.z + c) * (uint32_t)sizeof(T) : 0u),
                 ok ? plane + (uint64_t)first * sizeof(T) : plane);
    };
    const int np = full ? NPL + NJ : 9;
    const uint32_t c = (uint32_t)(tid % CC) * E;
    if ((int)c < wact) {
#pragma unroll
      for (int it = 0; it < (NPL + NJ + E - 1) / E; ++it) {
        const int p = tid / CC + it * E;
        if (p < np) copy(rows[p], c);
      }
    }
    if (!frow) {  // a whole row has its neighbours in its own copy
      for (int q = tid; q < (full ? NPAD : NPAD_G); q += BX) copy(rows[NPL + NJ + q], 0u);
    }
    mbar_arrive_on_copies(&bars[slot_of(k)]);
  };

  // g of a local column from a staged row, given the staged positions of
  // its left, own and right neighbour columns
  auto staged_g = [&](const T* st, int pm, int p0, int pp, T G[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i)
      G[i] = st[i * SEG + (cx_of(i) == 1 ? pm : (cx_of(i) == -1 ? pp : p0))];
  };

  // phi and psi of local row k into the ring (row k must have landed)
  auto put_row = [&](int k) {
    const T* st = stage_of(k);
    const int s = (k + 4) & 3;
    T G[9];
    if (act) {
      staged_g(st, om, o0, op, G);
      const T phi = sum9(G);
      ring.put(s, tid + 1, phi, step_psi<PLAIN>(phi, xi));
    }
    if (hthr) {
      staged_g(st, hm, h0, hp, G);
      const T phi = sum9(G);
      ring.put(s, hslot, phi, step_psi<PLAIN>(phi, xi));
    }
  };

  // ---- prologue: rows -1 .. S-2 in flight; phi of rows -1 and 0 ----------
  const long long lim = a.wait_cycles;
  bool early = false;  // a bound of 0 is tested before the later rows' issue covers the flight
  for (int k = -1; k <= min(S - 2, nrows); ++k) {
    issue(k);
    if (k == -1) early = lim <= 0 && !mbar_test_wait(&bars[slot_of(-1)], parity_of(-1));
  }
  // rows up to `landed` have been seen complete by this thread
  int landed = -2;
  bool bad = early || !mbar_wait_bounded(&bars[slot_of(-1)], parity_of(-1), lim);
  if (!bad) {
    landed = -1;
    put_row(-1);
  }
  bad = bad || !mbar_wait_bounded(&bars[slot_of(0)], parity_of(0), lim);
  if (!bad) {
    landed = 0;
    put_row(0);
  }

  int issued_last = min(S - 2, nrows);  // highest row issued so far
  // FP32: low part of g_0 of the own node, loaded one row ahead
  auto lo_of = [&](int k) -> T {
    if (sizeof(T) != 4 || !act || k >= nrows) return T(0);
    const uint32_t at = (uint32_t)wrap(y0 + k) * (uint32_t)nx + (uint32_t)xc;
    return LBM_BOUND(a.flags, at, (uint32_t)nx * (uint32_t)ny) ? __ldg(los + at) : T(0);
  };
  T lo_next = lo_of(0);
  for (int k = 0; k < nrows; ++k) {
    T glo = lo_next;
    lo_next = lo_of(k + 1);
    // row k+1 (own row or the halo row below the item) into the ring
    bad = bad || !mbar_wait_bounded(&bars[slot_of(k + 1)], parity_of(k + 1), lim);
    if (!bad) {
      landed = k + 1;
      put_row(k + 1);
    }
    if (__syncthreads_or(bad)) {
      // a wait gave up: report, wait for every row issued but not yet seen
      // complete (its copies write into this CTA's shared memory), leave
      if (tid == 0) atomicOr(a.flags, kFlagTimeout);
      for (int m = landed + 1; m <= issued_last; ++m)
        mbar_wait_bounded(&bars[slot_of(m)], parity_of(m), kWaitCycles);
      return;
    }
    // the stage of row k-1 is free: refill it with row k-1+S
    const int nxt = k - 1 + S;
    if (nxt <= nrows) {
      issue(nxt);
      issued_last = nxt;
    }
    if (act) {
      const T* st = stage_of(k);
      T F[9], G[9];
      staged_g(st, om, o0, op, G);
      if (COUPLED) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
          F[i] = st[(9 + i) * SEG + (cx_of(i) == 1 ? om : (cx_of(i) == -1 ? op : o0))];
      }
      T jpx = T(0), jpy = T(0);
      if (MODE == kModeStep) {
        jpx = st[NPL * SEG + tid];
        jpy = st[NPL * SEG + BX + tid];
      }
      const int y = wrap(y0 + k);
      const uint32_t node = (uint32_t)y * (uint32_t)nx + (uint32_t)xc;
      const Stencil<T> Sn = read_stencil(ring, k, tid + 1);
      // fused volume: the plain phi (the low part of g_0, below 2^-24 g_0 per
      // node, is left out here; lbm_volume counts it)
      if (do_vol) vacc += (double)Sn.p;
      if (!COUPLED) vortex_row(K, y);
      const NodeOut<T> o = node_update<T, COUPLED, MODE, PLAIN>(a.ph, K, F, G, glo, jpx, jpy, Sn);
      if (MODE == kModeStep) {
        store_node<T, COUPLED>(fd, gd, Jd, lod, P, node, F, G, glo, o, a.flags,
                               (uint32_t)nx * (uint32_t)ny);
        if (!isfinite(Sn.p + o.ux + o.uy + o.p)) atomicOr(a.flags, kFlagNonFinite);
      } else if (LBM_BOUND(a.flags, node, (uint32_t)nx * (uint32_t)ny)) {
        a.out_phi[node] = (double)Sn.p;
        a.out_ux[node] = (double)o.ux;
        a.out_uy[node] = (double)o.uy;
        a.out_p[node] = (double)o.p;
      }
    }
  }

  if (do_vol) {
    for (int o = 16; o > 0; o >>= 1) vacc += __shfl_down_sync(0xffffffffu, vacc, o);
    if (lane == 0) vred[warp] = vacc;
    __syncthreads();
    if (tid == 0) {
      double v = 0.0;
      for (int w = 0; w < BX / 32; ++w) v += vred[w];
      a.vol_part[(int64_t)blockIdx.x * kMaxRegions] = v;
    }
  }
}

// CTAs per SM the FP32 kernel is register-capped for (its shared memory
// allows about as many): about 80 registers a thread in every width.
template <typename T, int BX>
constexpr int tma_min_blocks() {
  return sizeof(T) != 4 ? 1
         : BX == 128    ? 6
         : BX == 96     ? 6
         : BX == 192    ? 4
         : BX == 256    ? 3
                        : 1;
}

template <typename T, int BX, bool COUPLED, int MODE, int S, bool PLAIN>
__global__ void __launch_bounds__(BX, (tma_min_blocks<T, BX>()))
    step_kernel_tma(const StepArgs<T> a) {
  using SH = TmaShape<T, BX, COUPLED, MODE, S>;
  __shared__ uint4 rows[SH::NPL + SH::NJ + SH::NPAD];
  const Item it = a.items[blockIdx.x];
  if (it.x0 == 0 && a.cases[it.c].nx <= BX)
    tma_body<T, BX, COUPLED, MODE, S, true, PLAIN>(a, rows);
  else
    tma_body<T, BX, COUPLED, MODE, S, false, PLAIN>(a, rows);
}

}  // namespace lbmk
