// Strip-tiled staged variant of the three-dimensional step kernel (FP32
// arithmetic, FP32 or FP16 population storage) for boxes whose nx is a
// multiple of the strip width BX and at least 2 BX.  The equations of
// step3_kernel; the difference is how the pulled values reach the threads, and
// that a thread updates two nodes adjacent in x at a time (lbm3_pair.cuh).
//
// A CTA owns a BX x BY column tile (x0 .. x0+BX-1, y0 .. y0+BY-1) and marches
// along z over `zc` planes, like step3_kernel, so several CTAs share an SM.
// Every value it reads for plane z arrives in shared memory by asynchronous
// 16-byte copies, NST-1 planes ahead, counted on one mbarrier per stage:
//   - f_i: row (y - c_iy, z - c_iz) of plane i for each of the BY rows, over
//     columns x0 .. x0+BX-1 shifted by -c_ix;
//   - phi*u: rows (y, z), columns x0 .. x0+BX-1;
//   - the 7 g (and the low part of g_0) pulled to the BY + 2 rows y0-1 ..
//     y0+BY of plane z+1 over the BX + 2 columns x0-1 .. x0+BX, for phase A
//     (phi = sum g, Eq. 35; psi, Eq. 37) into a 4-plane ring of (phi, psi)
//     from which the D3Q19 stencils of Sec. 3.2 are read.
// A staged row starts one 16-byte chunk (ES stored values, or ET values of
// the arithmetic type for the g_0 rows) left of x0 and ends one chunk right
// of x0+BX-1, so that the pull's one-column shift and the halo columns are
// index offsets inside it; of the two outer chunks only those its population
// reads are copied, from the other end of the row at x = 0 and x = nx (nx is
// a multiple of the chunk, so every copy stays 16-byte aligned).  The pulled g
// of a thread's own nodes stay in registers from phase A (plane z+1) to the
// update of plane z+1.
//
// Why threads copy and not the bulk engine: a row is 128 to 288 bytes, and a
// plane's 136 to 198 row segments were as many bulk-copy instructions, which
// take their operands from uniform registers, so a warp issues them lane after
// lane (the profiler counted 198 of them and 23.7 active threads per
// instruction).  A thread's 11 (FP16) or 18 (FP32) chunk copies are 128-thread
// wide.  Per node 703 -> 557 instructions in FP16 storage, 642 -> 532 in FP32.
// Measured, 256 x 256 x 512, MLUPS, bulk copies -> chunk copies: FP16 64 x 4 x
// 32 with three CTAs per SM 31,300 -> 38,470, 64 x 2 x 64 25,270 -> 34,450, with
// three stages and two CTAs 24,930 -> 34,530; FP32 64 x 4 x 64 22,060 -> 24,290.
// One node per thread, not packed, with bulk copies: FP16 28,300, FP32 22,200.
// Now, with the collision in difference form (lbm3_pair.cuh; 573 and 544
// instructions per node): FP16 37,900 (0.72 of measured HBM), 34,730 and 33,760,
// FP32 24,270 (0.83).  What bounds it: HBM in FP32; in FP16 issue (51%) and the
// latency of shared loads at 12 warps per SM.
//
// Every wait is bounded (wait_cycles); on expiry the CTA raises
// kFlagTimeout3, waits (bounded by lbmk::kWaitCycles) for its own copies in
// flight and returns.
#pragma once
#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "lbm3_bulk.cuh"
#include "lbm3_kernels.cuh"
#include "lbm3_pair.cuh"
#include "lbm_tma.cuh"

namespace lbmk3 {

template <typename T, typename S, int BX, int BY, int NST>
struct StripShape {
  static constexpr int ES = 16 / (int)sizeof(S);  // elements of one 16-byte chunk, storage type
  static constexpr int ET = 16 / (int)sizeof(T);  // the same for the arithmetic type
  static constexpr int WS = BX + 2 * ES;          // staged S row: x0-ES .. x0+BX+ES-1
  static constexpr int WT = BX + 2 * ET;          // staged g_0 row: x0-ET .. x0+BX+ET-1
  static constexpr int NR = BY + 2;               // phase-A rows (with the halo rows)
  static constexpr int RW = BX + 2;               // ring columns (with the halo columns)
  static constexpr size_t F_OFF = 0;                                         // [19][BY][WS] S
  static constexpr size_t GM_OFF = F_OFF + (size_t)19 * BY * WS * sizeof(S);  // [6][NR][WS] S
  static constexpr size_t J_OFF = GM_OFF + (size_t)6 * NR * WS * sizeof(S);   // [3][BY][BX] T
  static constexpr size_t G0_OFF = J_OFF + (size_t)3 * BY * BX * sizeof(T);   // [2][NR][WT] T
  static constexpr size_t STAGE_BYTES = G0_OFF + (size_t)2 * NR * WT * sizeof(T);
  static constexpr size_t BAR_OFF = NST * STAGE_BYTES;
  static constexpr size_t RING_OFF = (BAR_OFF + NST * 8 + 127) / 128 * 128;
  static constexpr size_t RING_BYTES = (size_t)4 * NR * RW * sizeof(typename N3<T>::pair);
  static constexpr size_t SMEM_BYTES = RING_OFF + RING_BYTES;
  static constexpr int NROW_S = 19 * BY + 6 * NR;          // rows of stored values per stage
  static constexpr int NROW = NROW_S + 3 * BY + 2 * NR;    // and of the arithmetic type
  static constexpr int NPAD = 10 * BY + 10 * NR + 4 * NR;  // chunks left and right of them
  static_assert(BX % ES == 0 && BX % ET == 0, "strip width must be whole 16-byte chunks");
  static_assert(ES >= 2 && ET >= 2, "a chunk must cover the pull shift and the halo column");
  static_assert(STAGE_BYTES % 16 == 0 && GM_OFF % 16 == 0 && J_OFF % 16 == 0 &&
                    G0_OFF % 16 == 0 && (WS * sizeof(S)) % 16 == 0 && (WT * sizeof(T)) % 16 == 0,
                "stage regions and rows must keep 16-byte alignment");
};

template <typename T, typename S, int BX, int BY, int NST>
constexpr size_t strip_smem_bytes() {
  return StripShape<T, S, BX, BY, NST>::SMEM_BYTES;
}

template <typename T, typename S, int BX, int BY, int NST, int MINB>
__global__ void __launch_bounds__(BX* BY / 2, MINB)
    step3_strip_kernel(const Args3<T, S> a, long long wait_cycles) {
  using SH = StripShape<T, S, BX, BY, NST>;
  using Pair = typename N3<T>::pair;
  constexpr int NR = SH::NR, RW = SH::RW, ES = SH::ES, ET = SH::ET, WS = SH::WS, WT = SH::WT;
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* const bars = reinterpret_cast<uint64_t*>(smem + SH::BAR_OFF);
  Pair(*const ring)[NR][RW] = reinterpret_cast<Pair(*)[NR][RW]>(smem + SH::RING_OFF);

  const int tid = threadIdx.x;
  constexpr int NT = BX * BY / 2;
  // the thread's nodes: columns tx and tx + 1 (tx even) of row ty
  const int tx = 2 * (tid % (BX / 2)), ty = tid / (BX / 2), warp = tid >> 5, lane = tid & 31;
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int64_t P = a.plane;
  const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
  const int zb = blockIdx.z * a.zc;
  const int ze = min(zb + a.zc, nz);
  const int nplanes = ze - zb;
  const bool act = y0 + ty < ny;  // nx is a multiple of BX: every column is in the box
  // periodic wrap of row and plane indices (any number of periods: boxes may
  // be thinner than the rows and planes a CTA touches)
  auto wrapy = [&](int v) { return ((v % ny) + ny) % ny; };
  auto wrapz = [&](int v) { return ((v % nz) + nz) % nz; };

  const int par = a.parity, dst = par ^ 1;
  const S* __restrict__ fs = a.f[par];
  const S* __restrict__ gms = a.g[par];
  const T* __restrict__ g0s = a.g0[par];
  const T* __restrict__ g0ls = a.g0lo[par];
  const T* __restrict__ js = a.J[par];
  S* __restrict__ fd = a.f[dst];
  S* __restrict__ gmd = a.g[dst];
  T* __restrict__ g0d = a.g0[dst];
  T* __restrict__ g0ld = a.g0lo[dst];
  T* __restrict__ jd = a.J[dst];

  auto stage = [&](int k) { return smem + (size_t)(k % NST) * SH::STAGE_BYTES; };
  auto sF = [&](unsigned char* st, int i, int r) {
    return reinterpret_cast<S*>(st + SH::F_OFF) + ((size_t)i * BY + r) * WS;
  };
  auto sGM = [&](unsigned char* st, int m, int r) {  // mover m = 1..6, phase-A row r
    return reinterpret_cast<S*>(st + SH::GM_OFF) + ((size_t)(m - 1) * NR + r) * WS;
  };
  auto sJ = [&](unsigned char* st, int c, int r) {
    return reinterpret_cast<T*>(st + SH::J_OFF) + ((size_t)c * BY + r) * BX;
  };
  auto sG0 = [&](unsigned char* st, int h, int r) {  // h = 0: g_0, 1: its low part
    return reinterpret_cast<T*>(st + SH::G0_OFF) + ((size_t)h * NR + r) * WT;
  };
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) lbmk::mbar_init(&bars[s], NT);
    lbmk::fence_mbar_init();
  }

  // Copies of a stage (local plane k, plane z = zb + k): f and phi*u of the BY
  // rows of plane z, the g of the NR phase-A rows of plane z + 1.  The BX
  // columns of a row are 16-byte chunks that neighbouring threads copy; the
  // chunk left or right of them, where the row's population is read there
  // (wrapped at x = 0 and x = nx), is an item of its own.  A row and such an
  // item are described once per CTA (only the plane changes from stage to
  // stage): global address without the plane offset, byte offset inside a
  // stage, and the plane it reads (0..3: z-1 .. z+2).
  __shared__ uint4 rows[SH::NROW];
  __shared__ uint4 pads[SH::NPAD];
  auto desc = [&](const void* plane, int row, int x, int esz, size_t at, int dz) {
    const uint64_t src = reinterpret_cast<uint64_t>(plane) +
                         ((uint64_t)wrapy(y0 + row) * (uint32_t)nx + (uint32_t)x) * (uint32_t)esz;
    return make_uint4((uint32_t)src, (uint32_t)(src >> 32), (uint32_t)at, (uint32_t)dz);
  };
  for (int q = tid; q < SH::NROW; q += NT) {
    if (q < 19 * BY) {  // f_i of tile row r: row y0 + r - c_iy, plane z - c_iz
      const int i = q / BY, r = q % BY;
      rows[q] = desc(fs + (int64_t)i * P, r - bcy(i), x0, sizeof(S),
                     SH::F_OFF + (((size_t)i * BY + r) * WS + ES) * sizeof(S), 1 - bcz(i));
    } else if (q < SH::NROW_S) {  // mover m of phase-A row r: row y0-1+r-c_my, plane z+1-c_mz
      const int u = q - 19 * BY, m = u / NR + 1, r = u % NR;
      rows[q] = desc(gms + (int64_t)(m - 1) * P, r - 1 - bcy(m), x0, sizeof(S),
                     SH::GM_OFF + (((size_t)(m - 1) * NR + r) * WS + ES) * sizeof(S), 2 - bcz(m));
    } else if (q < SH::NROW_S + 3 * BY) {  // phi*u: row y0 + r, plane z
      const int u = q - SH::NROW_S, c = u / BY, r = u % BY;
      rows[q] = desc(js + (int64_t)c * P, r, x0, sizeof(T),
                     SH::J_OFF + ((size_t)c * BY + r) * BX * sizeof(T), 1);
    } else {  // g_0 (h = 0) and its low part: row y0 - 1 + r, plane z + 1
      const int u = q - SH::NROW_S - 3 * BY, h = u / NR, r = u % NR;
      rows[q] = desc(h == 0 ? g0s : g0ls, r - 1, x0, sizeof(T),
                     SH::G0_OFF + (((size_t)h * NR + r) * WT + ET) * sizeof(T), 2);
    }
  }
  for (int q = tid; q < SH::NPAD; q += NT) {
    if (q < 10 * BY) {  // f with c_x = 1: left, c_x = -1: right (i = 1, 7, 9, ...; 2, 8, 10, ...)
      const int u = q / BY, r = q % BY;
      const int i = u < 2 ? u + 1 : u + 5;
      const bool left = bcx(i) == 1;
      pads[q] = desc(fs + (int64_t)i * P, r - bcy(i), left ? (x0 - ES + nx) % nx : (x0 + BX) % nx,
                     sizeof(S),
                     SH::F_OFF + (((size_t)i * BY + r) * WS + (left ? 0 : ES + BX)) * sizeof(S),
                     1 - bcz(i));
    } else if (q < 10 * BY + 10 * NR) {  // movers: m = 1 left, m = 2 right, the others both
      const int u = (q - 10 * BY) / NR, r = (q - 10 * BY) % NR;
      const int m = u < 2 ? u + 1 : 3 + (u - 2) / 2;
      const bool left = u < 2 ? u == 0 : (u & 1) == 0;
      pads[q] = desc(gms + (int64_t)(m - 1) * P, r - 1 - bcy(m),
                     left ? (x0 - ES + nx) % nx : (x0 + BX) % nx, sizeof(S),
                     SH::GM_OFF + (((size_t)(m - 1) * NR + r) * WS + (left ? 0 : ES + BX)) * sizeof(S),
                     2 - bcz(m));
    } else {  // g_0 and its low part: both
      const int u = (q - 10 * BY - 10 * NR) / NR, r = (q - 10 * BY - 10 * NR) % NR;
      const int h = u >> 1;
      const bool left = (u & 1) == 0;
      pads[q] = desc(h == 0 ? g0s : g0ls, r - 1, left ? (x0 - ET + nx) % nx : (x0 + BX) % nx,
                     sizeof(T),
                     SH::G0_OFF + (((size_t)h * NR + r) * WT + (left ? 0 : ET + BX)) * sizeof(T), 2);
    }
  }
  __syncthreads();

  // Issue the copies of the next stage.  Every thread arrives once on the
  // stage's barrier, when its own copies have landed.  Stages are issued in
  // order, k = 0, 1, ...: zq is the wrapped index of plane z - 1 of the next.
  const uint32_t nxy = (uint32_t)nx * (uint32_t)ny;
  int zq = wrapz(zb - 1);
  constexpr int CS = BX / ES, CT = BX / ET;  // chunks of a row's BX columns
  static_assert(NT % CS == 0 && NT % CT == 0, "a thread keeps its chunk of the row");
  auto issue = [&](int k) {
    const uint32_t st = lbmk::smem_u32(stage(k));
    const int z1 = zq + 1 == nz ? 0 : zq + 1;
    const int z2 = z1 + 1 == nz ? 0 : z1 + 1;
    const int z3 = z2 + 1 == nz ? 0 : z2 + 1;
    const uint32_t o0 = (uint32_t)zq * nxy, o1 = (uint32_t)z1 * nxy, o2 = (uint32_t)z2 * nxy,
                   o3 = (uint32_t)z3 * nxy;
    auto copy = [&](const uint4& d, int esz, uint32_t chunk) {
      const uint32_t off = d.w & 2u ? (d.w & 1u ? o3 : o2) : (d.w & 1u ? o1 : o0);
      const uint64_t src = (((uint64_t)d.y << 32) | d.x) + (uint64_t)off * (uint32_t)esz;
      lbmk::copy16_g2s(st + d.z + chunk, src + chunk);
    };
#pragma unroll
    for (int q = tid; q < SH::NROW_S * CS; q += NT)
      copy(rows[q / CS], sizeof(S), (uint32_t)(tid % CS) * 16u);
#pragma unroll
    for (int q = tid; q < (SH::NROW - SH::NROW_S) * CT; q += NT)
      copy(rows[SH::NROW_S + q / CT], sizeof(T), (uint32_t)(tid % CT) * 16u);
#pragma unroll
    for (int q = tid; q < SH::NPAD; q += NT)
      copy(pads[q], q < 10 * BY + 10 * NR ? (int)sizeof(S) : (int)sizeof(T), 0u);
    lbmk::mbar_arrive_on_copies(&bars[k % NST]);
    zq = z1;
  };

  // pulled g at tile column xl (-1 .. BX) of phase-A row r from a staged plane
  auto staged_g = [&](unsigned char* st, int r, int xl, T (&G)[7], T& glo) {
    G[0] = sG0(st, 0, r)[xl + ET];
    glo = sG0(st, 1, r)[xl + ET];
#pragma unroll
    for (int m = 1; m < 7; ++m) G[m] = Conv<T, S>::ld(sGM(st, m, r) + (xl - bcx(m) + ES));
  };
  auto put = [&](int slot, int r, int xl, const T (&G)[7], T glo) {
    const T phi = phi_of(G, glo);
    Pair v;
    v.x = phi;
    v.y = psi3(phi, a.xi);
    ring[slot][r][xl + 1] = v;
  };

  // the same at columns xl and xl + 1 (xl even: what is not shifted is one
  // aligned load)
  auto staged_g2 = [&](unsigned char* st, int r, int xl, float2 (&G)[7], float2& glo) {
    G[0] = ld2<0>(sG0(st, 0, r) + xl + ET);
    glo = ld2<0>(sG0(st, 1, r) + xl + ET);
    G[1] = ld2<1>(sGM(st, 1, r) + xl + ES);
    G[2] = ld2<-1>(sGM(st, 2, r) + xl + ES);
#pragma unroll
    for (int m = 3; m < 7; ++m) G[m] = ld2<0>(sGM(st, m, r) + xl + ES);
  };
  auto put2 = [&](int slot, int r, int xl, const float2 (&G)[7], float2 glo) {
    const float2 phi = add2(
        add2(add2(add2(G[0], add2(G[1], G[2])), add2(G[3], G[4])), add2(G[5], G[6])), glo);
    ring[slot][r][xl + 1] = make_float2(phi.x, psi3(phi.x, a.xi));
    ring[slot][r][xl + 2] = make_float2(phi.y, psi3(phi.y, a.xi));
  };

  // The tile's halo ring, tile coordinates -1 .. BX and -1 .. BY: items h < BX
  // are node pairs of the rows below and above, the others single nodes of
  // the columns left and right (corners included).
  constexpr int NHI = BX + 2 * NR;
  auto halo_pair = [&](int h, int& hx, int& hy) {
    hx = 2 * (h % (BX / 2)), hy = h < BX / 2 ? -1 : BY;
  };
  auto halo_node = [&](int h, int& hx, int& hy) {
    const int u = h - BX;
    hx = u < NR ? -1 : BX, hy = (u < NR ? u : u - NR) - 1;
  };

  // a bound of 0 is tested before the prologue, which covers the copies' flight
  bool early = false;
  for (int k = 0; k < NST - 1 && k < nplanes; ++k) {
    issue(k);
    if (k == 0) early = wait_cycles <= 0 && !lbmk::mbar_test_wait(&bars[0], 0);
  }
  int issued_last = min(NST - 1, nplanes) - 1;
  int landed = -1;

  // ---- prologue: phase A of planes zb-1 and zb from global memory ----------
  float2 Gc[7], Gn[7], Gcl, Gnl;
  {
    auto pull = [&](int x, int y, int zl, T (&G)[7], T& gl) {  // tile coordinates
      Offs o;
      set_xy(o, (x0 + x + nx) % nx, wrapy(y0 + y), nx, ny);
      set_z(o, zl, nz, nxy);
      pull_g(g0s, g0ls, gms, P, o, G, gl);
    };
    for (int q = 0; q < 2; ++q) {
      const int zl = wrapz(zb - 1 + q), slot = (zb - 1 + q) & 3;
      T A[7], B[7], al, bl;
      pull(tx, ty, zl, A, al);
      pull(tx + 1, ty, zl, B, bl);
      put(slot, ty + 1, tx, A, al);
      put(slot, ty + 1, tx + 1, B, bl);
#pragma unroll
      for (int i = 0; i < 7; ++i) Gc[i] = make_float2(A[i], B[i]);  // of plane zb in the end
      Gcl = make_float2(al, bl);
      for (int h = tid; h < NHI; h += NT) {
        int hx, hy;
        if (h < BX) {
          halo_pair(h, hx, hy);
          pull(hx + 1, hy, zl, A, al);
          put(slot, hy + 1, hx + 1, A, al);
        } else {
          halo_node(h, hx, hy);
        }
        pull(hx, hy, zl, A, al);
        put(slot, hy + 1, hx, A, al);
      }
    }
  }

  const long long lim = wait_cycles;
  double vsum = 0.0;
  for (int k = 0; k < nplanes; ++k) {
    const int z = zb + k;
    unsigned char* st = stage(k);
    const bool bad = (k == 0 && early) ||
                     !lbmk::mbar_wait_bounded(&bars[k % NST], (uint32_t)((k / NST) & 1), lim);
    if (!bad) {
      landed = k;
      // phase A of plane z + 1 from the staged g rows
      staged_g2(st, ty + 1, tx, Gn, Gnl);
      put2((z + 1) & 3, ty + 1, tx, Gn, Gnl);
#pragma unroll
      for (int h = tid; h < NHI; h += NT) {
        int hx, hy;
        if (h < BX) {
          halo_pair(h, hx, hy);
          float2 H[7], hl;
          staged_g2(st, hy + 1, hx, H, hl);
          put2((z + 1) & 3, hy + 1, hx, H, hl);
        } else {
          halo_node(h, hx, hy);
          T H[7], hl;
          staged_g(st, hy + 1, hx, H, hl);
          put((z + 1) & 3, hy + 1, hx, H, hl);
        }
      }
    }
    if (__syncthreads_or(bad)) {
      // a wait gave up: report, wait for every stage issued but not yet seen
      // complete (its copies write into this CTA's shared memory), leave
      if (tid == 0) atomicOr(a.flags, kFlagTimeout3);
      for (int m = landed + 1; m <= issued_last; ++m)
        lbmk::mbar_wait_bounded(&bars[m % NST], (uint32_t)((m / NST) & 1), lbmk::kWaitCycles);
      return;
    }
    // the stage of plane k-1 is free: refill it with plane k-1+NST
    const int nxt = k + NST - 1;
    if (nxt < nplanes) {
      issue(nxt);
      issued_last = nxt;
    }
    if (act) {
      float2 F[19], jp[3];
#pragma unroll
      for (int i = 0; i < 19; ++i) {
        const S* const q = sF(st, i, ty) + tx + ES;
        F[i] = bcx(i) == 0 ? ld2<0>(q) : (bcx(i) == 1 ? ld2<1>(q) : ld2<-1>(q));
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) jp[c] = ld2<0>(sJ(st, c, ty) + tx);
      Pair2 N;
      {
        // (phi, psi) of columns tx-1 .. tx+2, rows ty-1 .. ty+1, planes z-1 .. z+1
        const int sm = (z + 3) & 3, s0 = z & 3, sp = (z + 1) & 3, j = ty + 1;
        float2 C[4], Nr[4], Sr[4], U[4], D[4], un[2], us[2], dn[2], ds[2];
        row4(&ring[s0][j][tx], C);
        row4(&ring[s0][j + 1][tx], Nr);
        row4(&ring[s0][j - 1][tx], Sr);
        row4(&ring[sp][j][tx], U);
        row4(&ring[sm][j][tx], D);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          un[n] = ring[sp][j + 1][tx + 1 + n];
          us[n] = ring[sp][j - 1][tx + 1 + n];
          dn[n] = ring[sm][j + 1][tx + 1 + n];
          ds[n] = ring[sm][j - 1][tx + 1 + n];
        }
        stencils2(C, Nr, Sr, U, D, un, us, dn, ds, N);
      }
      float2 J[3];
      const float2 fin = node3_pair<S>(a, F, Gc, Gcl, jp, N, J);
      if (!(isfinite(fin.x) && isfinite(fin.y))) atomicOr(a.flags, kFlagNonFinite);
      if (a.vol_part) vsum += (double)N.phi.x + (double)N.phi.y;
      const uint32_t node = ((uint32_t)z * (uint32_t)ny + (uint32_t)(y0 + ty)) * (uint32_t)nx +
                            (uint32_t)(x0 + tx);
#pragma unroll
      for (int c = 0; c < 3; ++c) *reinterpret_cast<float2*>(jd + c * P + node) = J[c];
      *reinterpret_cast<float2*>(g0d + node) = Gc[0];
      *reinterpret_cast<float2*>(g0ld + node) = Gcl;
#pragma unroll
      for (int m = 1; m < 7; ++m) st2(gmd + (m - 1) * P + node, Gc[m]);
#pragma unroll
      for (int q = 0; q < 19; ++q) st2(fd + q * P + node, F[q]);
    }
#pragma unroll
    for (int m = 0; m < 7; ++m) Gc[m] = Gn[m];
    Gcl = Gnl;
  }
  if (a.vol_part) {
    // fixed-order block reduction of the phi this CTA collided
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) vsum += __shfl_down_sync(0xffffffffu, vsum, off);
    __shared__ double wsum[NT / 32];
    if (lane == 0) wsum[warp] = vsum;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < NT / 32; ++w) t += wsum[w];
      a.vol_part[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
    }
  }
}

}  // namespace lbmk3
