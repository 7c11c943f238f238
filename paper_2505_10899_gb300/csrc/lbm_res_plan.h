// Tiling of a batch for the chip-resident kernel (lbm_resident.cuh): one tile
// per CTA, all CTAs on the chip at once.
#pragma once
#include <algorithm>
#include <cstdint>
#include <vector>

#include "../../include/lbm_api.h"
#include "launch.h"
#include "lbm_layout.h"

namespace lbmk {

constexpr int kResSMs = 152;
// Steps that pay for loading and storing the state, where nothing was measured.
constexpr int kResMinSteps = 4;
constexpr int kResMinTile = 64;  // nodes: tiles of 32, 64 and 128 measure alike

struct ResPlan {
  int variant = -1;  // -1: the batch does not fit
  uint32_t nslots = 0;
  std::vector<ResTile> tiles;
};

// Fewest tiles of at most m nodes (and the variant's cells and rim triples,
// `per` triples per rim node) that cover an nx x ny grid, tx by ty; among equal
// counts the shortest rim.  Tiles are at least 3 x 3.  False if there is none.
inline bool res_split(int nx, int ny, int m, const ResVariant& v, int per, int* tx, int* ty) {
  int best = INT32_MAX, rim = INT32_MAX;
  for (int a = 1; nx / a >= 3 && a <= kResSMs * v.per_sm; ++a) {
    const int w = (nx + a - 1) / a;
    const int hmax = std::min({m / w, v.pc / (w + 4) - 4, (v.nx - 8) / (2 * per) - w - 4});
    if (hmax < 3) continue;
    const int b = (ny + hmax - 1) / hmax;
    if (ny / b < 3) continue;
    const int r = w + (ny + b - 1) / b;
    if (a * b < best || (a * b == best && r < rim)) best = a * b, rim = r, *tx = a, *ty = b;
  }
  return best != INT32_MAX;
}

// The tiles with the fewest nodes per CTA that fit the chip at once, for the
// first of nv variants that holds the batch.  slots_h, slots_w: exchange slots
// of a tile per row and per column.
inline ResPlan res_tile(const lbm_params* c, int n, const ResVariant* variants, int nv, int per,
                        int slots_h, int slots_w) {
  ResPlan pl;
  int64_t nodes = 0;
  for (int k = 0; k < n; ++k) nodes += (int64_t)c[k].nx * c[k].ny;
  std::vector<int> tx(n), ty(n);
  for (int v = 0; v < nv; ++v) {
    const ResVariant X = variants[v];
    const int cap = X.nt * X.r, most = kResSMs * X.per_sm;
    if (n > most || nodes > (int64_t)most * cap) continue;
    bool fits = false;
    for (int m = (int)std::max<int64_t>(kResMinTile, (nodes + most - 1) / most); m <= cap && !fits;) {
      int64_t total = 0;
      for (int k = 0; k < n && total <= most; ++k)
        total += res_split(c[k].nx, c[k].ny, m, X, per, &tx[k], &ty[k]) ? (int64_t)tx[k] * ty[k]
                                                                        : most + 1;
      fits = total <= most;
      m = m == cap ? cap + 1 : std::min(cap, m + std::max(1, m / 32));
    }
    if (!fits) continue;
    pl.variant = v;
    for (int k = 0; k < n; ++k) {
      const int first = (int)pl.tiles.size();
      auto at = [](int i, int parts, int len) { return (int)((int64_t)i * len / parts); };
      for (int j = 0; j < ty[k]; ++j)
        for (int i = 0; i < tx[k]; ++i) {
          ResTile t{};
          t.c = k;
          t.x0 = at(i, tx[k], c[k].nx);
          t.y0 = at(j, ty[k], c[k].ny);
          t.w = at(i + 1, tx[k], c[k].nx) - t.x0;
          t.h = at(j + 1, ty[k], c[k].ny) - t.y0;
          t.slot = pl.nslots;
          pl.nslots += (uint32_t)(slots_h * t.h + slots_w * t.w);
          pl.tiles.push_back(t);
        }
      for (int j = 0; j < ty[k]; ++j)
        for (int i = 0; i < tx[k]; ++i) {
          ResTile& t = pl.tiles[first + j * tx[k] + i];
          const int jS = (j + ty[k] - 1) % ty[k], jN = (j + 1) % ty[k];
          const int iW = (i + tx[k] - 1) % tx[k], iE = (i + 1) % tx[k];
          auto other = [&](int jj, int ii) -> const ResTile& {
            return pl.tiles[first + jj * tx[k] + ii];
          };
          t.hS = other(jS, i).h;
          t.hN = other(jN, i).h;
          t.nb[kResW] = other(j, iW).slot;
          t.nb[kResW + 1] = other(jS, iW).slot;
          t.nb[kResW + 2] = other(jN, iW).slot;
          t.nb[kResE] = other(j, iE).slot;
          t.nb[kResE + 1] = other(jS, iE).slot;
          t.nb[kResE + 2] = other(jN, iE).slot;
          t.nb[kResS] = other(jS, i).slot;
          t.nb[kResN] = other(jN, i).slot;
        }
    }
    break;
  }
  return pl;
}

// Tiles of the step kernel (lbm_resident.cuh).
inline ResPlan res_plan(const lbm_params* c, int n) {
  const bool f64 = c[0].precision == LBM_F64, coupled = c[0].flow == LBM_FLOW_COUPLED;
  ResVariant v[kResVariants];
  for (int k = 0; k < kResVariants; ++k) v[k] = res_variant(f64, coupled, k);
  return res_tile(c, n, v, kResVariants, 4, 10, 8);
}

// Tiles of the reverse sweep (lbm_adjoint_resident.cuh): FP32, coupled flow.
constexpr ResVariant kResAdjoint = {512, 2, 1224, 896, 1};
inline ResPlan res_plan_adjoint(const lbm_params& c) {
  if (c.precision != LBM_F32 || c.flow != LBM_FLOW_COUPLED) return ResPlan{};
  return res_tile(&c, 1, &kResAdjoint, 1, 6, 12, 12);
}

}  // namespace lbmk
