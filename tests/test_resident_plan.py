"""CPU model of the exchange plans of the chip-resident kernels (csrc/lbm_resident.cuh and
lbm_adjoint_resident.cuh).

The tiling is the library's own (csrc/lbm_res_plan.h, compiled here for the host); the rim
tables that the kernel's threads build are restated.  For every tile: tables and cells within
their bounds, every slot within the exchange area and written by one triple only, every
received triple the one that the slot's sender puts there, and every population that a tile
pulls from outside itself received."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from conftest import ROOT

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
SHIM = r'''
#include "lbm_res_plan.h"
extern "C" int plan(const lbm_params* c, int n, int adjoint, int* out, int* nslots, int* var) {
  const lbmk::ResPlan p = adjoint ? lbmk::res_plan_adjoint(c[0]) : lbmk::res_plan(c, n);
  if (p.variant < 0) return 0;
  const lbmk::ResVariant v =
      adjoint ? lbmk::kResAdjoint
              : lbmk::res_variant(c[0].precision == LBM_F64, c[0].flow == LBM_FLOW_COUPLED, p.variant);
  var[0] = v.nt, var[1] = v.r, var[2] = v.pc, var[3] = v.nx, var[4] = v.per_sm;
  *nslots = (int)p.nslots;
  for (size_t i = 0; i < p.tiles.size(); ++i) {
    const lbmk::ResTile& t = p.tiles[i];
    const int v8[8] = {t.c, t.x0, t.y0, t.w, t.h, t.hS, t.hN, (int)t.slot};
    for (int k = 0; k < 8; ++k) out[16 * i + k] = v8[k];
    for (int k = 0; k < 8; ++k) out[16 * i + 8 + k] = (int)t.nb[k];
  }
  return (int)p.tiles.size();
}
'''


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    from paper_2505_10899_gb300 import build, lbm
    d = tmp_path_factory.mktemp("shim")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run([shutil.which("g++"), "-std=c++17", "-O1", "-shared", "-fPIC", "-I", build.CSRC,
                    "-I", os.path.join(ROOT, "include"), "-I", cuda, str(src), "-o", str(so)],
                   check=True)
    lib = ctypes.CDLL(str(so))

    def call(sizes, prec, flow="coupled", walls=0, adjoint=0):
        import workloads as W
        ps = [lbm.make_params(W.base_case(nx, ny, flow=flow, walls=walls), prec) for nx, ny in sizes]
        arr = (lbm.lbm_params * len(ps))(*ps)
        out = np.zeros(16 * 304, dtype=np.int32)
        ns, var = ctypes.c_int(), (ctypes.c_int * 5)()
        n = lib.plan(arr, len(ps), adjoint, out.ctypes.data_as(ctypes.c_void_p), ctypes.byref(ns), var)
        return out.reshape(-1, 16)[:n].tolist(), ns.value, tuple(var)
    return call


def send_table(t, coupled, wbot, wtop):
    c, x0, y0, w, h = t[:5]
    out = []
    for q in range(10 * h + 8 * w):
        if q < 10 * h:
            west = q < 5 * h
            u = q if west else q - 5 * h
            y, k = u // 5, u % 5
            x = (1 if k == 0 else 0) if west else (w - 2 if k == 0 else w - 1)
            fwd = west == (k == 4)
            tri = [0, 2, 4] if k == 1 else ([1, 5, 8] if fwd else [3, 6, 7])
            use = k < 3 or (k == 3 and coupled) or (k == 4 and ((wbot and y == 0) or (wtop and y == h - 1)))
        else:
            south = q < 10 * h + 4 * w
            u = q - 10 * h - (0 if south else 4 * w)
            x, k = u >> 2, u & 3
            y = (1 if k == 0 else 0) if south else (h - 2 if k == 0 else h - 1)
            tri = [0, 1, 3] if k == 1 else ([4, 7, 8] if south else [2, 5, 6])
            use = (k < 3 or coupled) and not (wbot if south else wtop)
        if use:
            out.append((t[7] + q, x, y, [p + 9 * (k == 3) for p in tri]))
    return out


def recv_table(t, coupled, wbot, wtop):
    c, x0, y0, w, h, hS, hN = t[:7]
    nb = t[8:16]
    out = []
    for q in range(10 * (h + 4) + 8 * w):
        if q < 10 * (h + 4):
            west = q < 5 * (h + 4)
            u = q if west else q - 5 * (h + 4)
            y, k = u // 5 - 2, u % 5
            lower, upper = y < 0, y >= h
            hn = hS if lower else (hN if upper else h)
            row = hn + y if lower else (y - h if upper else y)
            slot = nb[(0 if west else 3) + (1 if lower else (2 if upper else 0))]
            slot += (5 * hn if west else 0) + 5 * row + k
            x = (-2 if k == 0 else -1) if west else (w + 1 if k == 0 else w)
            fwd = west != (k == 4)
            tri = [0, 2, 4] if k == 1 else ([1, 5, 8] if fwd else [3, 6, 7])
            use = not (lower and wbot) and not (upper and wtop) and (
                k < 3 or (k == 3 and coupled and -1 <= y <= h) or
                (k == 4 and ((wbot and y == 0) or (wtop and y == h - 1))))
        else:
            south = q < 10 * (h + 4) + 4 * w
            u = q - 10 * (h + 4) - (0 if south else 4 * w)
            x, k = u >> 2, u & 3
            slot = nb[6] + 10 * hS + 4 * w + u if south else nb[7] + 10 * hN + u
            y = (-2 if k == 0 else -1) if south else (h + 1 if k == 0 else h)
            tri = [0, 1, 3] if k == 1 else ([2, 5, 6] if south else [4, 7, 8])
            use = (k < 3 or coupled) and not (wbot if south else wtop)
        if use:
            out.append((slot, x, y, [p + 9 * (k == 3) for p in tri]))
    return out


SIZES = [[(128, 64)], [(201, 101)], [(512, 256)], [(256, 256)], [(20, 3)], [(3, 20)], [(4, 9)],
         [(67, 5)], [(700, 97)], [(64, 64), (192, 40), (36, 52), (4, 9)], [(96, 96)] * 9, [(3, 3)]]


@pytest.mark.parametrize("prec,flow", [("f32", "coupled"), ("f64", "coupled"), ("f32", "vortex")])
@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("sizes", SIZES, ids=str)
def test_exchange_plan(plan, sizes, prec, flow, walls):
    if walls and flow == "vortex":
        pytest.skip("walls need the coupled flow")
    tiles, nslots, (nt, r, pc, cap, per_sm) = plan(sizes, prec, flow, walls)
    if not tiles:
        assert sum(x * y for x, y in sizes) > 60000  # only large grids are left out here
        return
    coupled = flow == "coupled"
    assert len(tiles) <= 152 * per_sm
    area = [np.zeros((ny, nx), int) for nx, ny in sizes]
    sent, tables = {}, []
    for t in tiles:
        c, x0, y0, w, h = t[:5]
        nx, ny = sizes[c]
        wbot, wtop = bool(walls and y0 == 0), bool(walls and y0 + h == ny)
        area[c][y0:y0 + h, x0:x0 + w] += 1
        assert w >= 3 and h >= 3 and w * h <= nt * r and (w + 4) * (h + 4) <= min(pc, 4096)
        S, V = send_table(t, coupled, wbot, wtop), recv_table(t, coupled, wbot, wtop)
        assert len(S) <= cap and len(V) <= cap and 4 * (w + h) <= cap
        for slot, x, y, tri in S:
            assert 0 <= slot < nslots and slot not in sent
            assert 0 <= x < w and 0 <= y < h
            sent[slot] = (c, x0 + x, y0 + y, tri)
        tables.append((t, wbot, wtop, V))
    assert all((a == 1).all() for a in area)  # the tiles partition every grid
    for t, wbot, wtop, V in tables:
        c, x0, y0, w, h = t[:5]
        nx, ny = sizes[c]
        have = set()
        for slot, x, y, tri in V:
            assert -2 <= x < w + 2 and -2 <= y < h + 2
            assert sent[slot] == (c, (x0 + x) % nx, (y0 + y) % ny, tri)
            have.update((x, y, p) for p in tri)
        # what the tile's collisions (f) and its phi, psi (g) pull
        for lo, hi, base in ((0, 0, 9),) * coupled + ((-1, 1, 0),):
            for y in range(lo, h + hi):
                if (wbot and y < 0) or (wtop and y >= h):
                    continue  # the ghost row is the wall row
                for x in range(lo, w + hi):
                    for i in range(9):
                        xs, ys, pl = x - CX[i], y - CY[i], i
                        if (wbot and ys < 0) or (wtop and ys >= h):
                            xs, ys, pl = x, y, OPP[i]
                        if not (0 <= xs < w and 0 <= ys < h):
                            assert (xs, ys, pl + base) in have, (t, xs, ys, pl + base)


def test_plan_leaves_out_what_does_not_fit(plan):
    assert not plan([(2, 64)], "f32")[0]          # narrower than a tile
    assert not plan([(1024, 1024)], "f32")[0]     # more nodes than the SMs hold
    assert not plan([(64, 64)] * 305, "f32")[0]   # more cases than CTAs


def ad_planes(k, dirs):
    if k < 4:  # 18..22 stencil adjoints, 23 phi adjoint
        return [21, 22, 23] if k & 1 else [18, 19, 20]
    return [d + (9 if k == 4 else 0) for d in dirs]


EAST, WEST, NORTH, SOUTH = [1, 5, 8], [3, 6, 7], [2, 5, 6], [4, 7, 8]


def ad_send(t, wbot, wtop):
    c, x0, y0, w, h = t[:5]
    out = []
    for q in range(12 * (h + w)):
        if q < 12 * h:
            side = 0 if q < 6 * h else 1
            u = q - side * 6 * h
            y, k = u // 6, u % 6
            far = int(k in (2, 3))
            x = far if side == 0 else w - 1 - far
        else:
            side = 2 if q < 12 * h + 6 * w else 3
            u = q - 12 * h - (side - 2) * 6 * w
            x, k = u // 6, u % 6
            far = int(k in (2, 3))
            y = far if side == 2 else h - 1 - far
            if wbot if side == 2 else wtop:
                continue
        out.append((t[7] + q, x, y, ad_planes(k, (EAST, WEST, NORTH, SOUTH)[side])))
    return out


def ad_recv(t, wbot, wtop):
    c, x0, y0, w, h, hS, hN = t[:7]
    nb = t[8:16]
    out = []
    for q in range(12 * (h + 4) + 12 * w):
        if q < 12 * (h + 4):
            side = 0 if q < 6 * (h + 4) else 1
            u = q - side * 6 * (h + 4)
            y, k = u // 6 - 2, u % 6
            lower, upper = y < 0, y >= h
            if (lower and wbot) or (upper and wtop):
                continue
            hn = hS if lower else (hN if upper else h)
            row = hn + y if lower else (y - h if upper else y)
            slot = nb[(0 if side == 0 else 3) + (1 if lower else (2 if upper else 0))]
            slot += (6 * hn if side == 0 else 0) + 6 * row + k
            far = int(k in (2, 3))
            x = -1 - far if side == 0 else w + far
            if k >= 4 and (y < -1 or y > h):
                continue
        else:
            side = 2 if q < 12 * (h + 4) + 6 * w else 3
            u = q - 12 * (h + 4) - (side - 2) * 6 * w
            x, k = u // 6, u % 6
            if wbot if side == 2 else wtop:
                continue
            slot = nb[6] + 12 * hS + 6 * w + u if side == 2 else nb[7] + 12 * hN + u
            far = int(k in (2, 3))
            y = -1 - far if side == 2 else h + far
        out.append((slot, x, y, ad_planes(k, (WEST, EAST, SOUTH, NORTH)[side])))
    return out


@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("size", [(128, 64), (201, 101), (512, 256), (20, 3), (3, 20), (67, 5),
                                  (700, 97), (3, 3)], ids=str)
def test_reverse_sweep_exchange_plan(plan, size, walls):
    nx, ny = size
    tiles, nslots, (nt, r, pc, cap, per_sm) = plan([size], "f32", "coupled", walls, 1)
    assert tiles and len(tiles) <= 152
    area, sent, tables = np.zeros((ny, nx), int), {}, []
    for t in tiles:
        c, x0, y0, w, h = t[:5]
        wbot, wtop = bool(walls and y0 == 0), bool(walls and y0 + h == ny)
        area[y0:y0 + h, x0:x0 + w] += 1
        assert w >= 3 and h >= 3 and w * h <= nt * r and w + 4 < 1024 and h + 4 < 1024
        assert (w + 4) * (h + 4) <= pc == 1224 and (w + 2) * (h + 2) <= 1088
        S, V = ad_send(t, wbot, wtop), ad_recv(t, wbot, wtop)
        assert len(S) <= cap and len(V) <= cap
        for slot, x, y, tri in S:
            assert 0 <= slot < nslots and slot not in sent and 0 <= x < w and 0 <= y < h
            sent[slot] = ((x0 + x) % nx, (y0 + y) % ny, tri)
        tables.append((t, wbot, wtop, V))
    assert (area == 1).all()
    for t, wbot, wtop, V in tables:
        c, x0, y0, w, h = t[:5]
        have = set()
        for slot, x, y, tri in V:
            assert sent[slot] == ((x0 + x) % nx, (y0 + y) % ny, tri)
            have.update((x, y, p) for p in tri)

        def need(x, y, p):
            assert (0 <= x < w and 0 <= y < h) or (x, y, p) in have, (t, x, y, p)
        rows = range(0 if wbot else -1, h if wtop else h + 1)
        for y in range(h):  # populations and phi totals that the own positions take
            for x in range(w):
                for i in range(9):
                    if (wbot and y == 0 and CY[i] == -1) or (wtop and y == h - 1 and CY[i] == 1):
                        continue  # bounced: the own opposite
                    xs, ys = x + CX[i], y + CY[i]
                    need(xs, ys, i), need(xs, ys, 9 + i)
                    assert -1 <= xs <= w and ys in rows
        for y in rows:  # stencil adjoints of the neighbours of every phi total
            for x in range(-1, w + 1):
                need(x, y, 23)
                for i in range(1, 9):
                    xs, ys = x - CX[i], y - CY[i]
                    if (wbot and ys < 0) or (wtop and ys >= h):
                        continue
                    for p in range(18, 23):
                        need(xs, ys, p)
