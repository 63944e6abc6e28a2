// lbpf_plan.h -- work decomposition of the step kernels (host code, plain C++).
//
// A step kernel block covers TILE_X interior columns and `by - 2` interior rows (one row
// for the one-row blocks of the 2D lattices) of the xy plane over a z-chunk of planes; a
// work item names one such tile.  This header also plans the one-launch step: the order
// in which the blocks of that launch take the phase-field and U/theta tiles, and which
// phase-field tiles each U/theta tile waits for.  It has no CUDA dependency, so the
// planner can be checked by a host program.
#pragma once

#include <algorithm>
#include <vector>

namespace lbpf {

constexpr int TILE_X = 30;  // interior columns per block row (block x = 32)

constexpr int NODE_THREADS = 128;  // largest block of the node-wise kernels

struct WorkItem {
  int sim;
  int x0, y0;  // first interior column of the tile
  int z0, z1;  // planes [z0, z1) written by this block
};

// Tiles of one simulation for blocks of `by` rows (tiles of `tile_x` columns) and z-chunks of
// `zchunk` planes, z-chunk major, then rows, then columns.
inline void build_items(int sim_index, int nx, int ny, int nz, int by, int zchunk, std::vector<WorkItem>& out,
                        int tile_x = TILE_X) {
  const int ty = by == 1 ? 1 : by - 2;  // interior rows per block: one-row blocks (2D) have no y halo
  for (int z0 = 0; z0 < nz; z0 += zchunk)
    for (int y0 = 0; y0 < ny; y0 += ty)
      for (int x0 = 0; x0 < nx; x0 += tile_x) out.push_back(WorkItem{sim_index, x0, y0, z0, std::min(nz, z0 + zchunk)});
}

// Blocks of one simulation's node-wise step: `span` consecutive nodes of a plane (x0 the first)
// over z-chunks of `zchunk` planes, z-chunk major.
inline void build_node_items(int sim_index, int nx, int ny, int nz, int span, int zchunk, std::vector<WorkItem>& out) {
  const int plane = nx * ny;
  for (int z0 = 0; z0 < nz; z0 += zchunk)
    for (int p0 = 0; p0 < plane; p0 += span)
      out.push_back(WorkItem{sim_index, p0, 0, z0, std::min(nz, z0 + zchunk)});
}

// Threads of a node-wise block, `nodes` nodes each, for a tiling of `by` rows (1: the 2D lattices, which
// have no rows to choose).  128 (the default, by = 8) against 256 on GB300: 32^3 FP64 64 against
// 69 us per step, 301^3 D3Q15/D3Q7/D3Q7 FP32 1835 against 1909 us, 256^3 FP16 the same.  `few`: planes (in
// 2D rows) of fewer nodes take whole warps only (few_warps).
inline int node_threads(int by, long long plane, int nodes, bool few) {
  const int most = by == 1 ? NODE_THREADS : 16 * by;
  const long long lanes = (plane + nodes - 1) / nodes;
  return few ? (int)std::min<long long>(most, (lanes + 31) / 32 * 32) : most;
}

// Whether the blocks of `planes` planes in all (in 2D rows) that are too small for a whole block take
// fewer warps.  In 2D with FP32 arithmetic always: 40 x 4000 FP32 25.0 us per step with 128 threads, 18.8 with 32;
// 16 x 8000 29.9, 22.9; 90 x 2000 18.1 with 128, 14.8 with 64.  In 3D and FP64, whose registers leave an SM
// few warps, only where there are more blocks than the chip holds at once.  Fewer than that are placed
// while the kernel ahead still runs, where it leaves room, and the more of them an SM takes the more
// uneven that is: D3Q19/D3Q19/D3Q7 FP64, 800 planes of 4 x 4, 31.8 us with 128 threads, 56.1 with 32, and 29.8 with
// 32 that were placed after the kernel ahead.  With 128 threads / whole warps: 8 x 8 FP64 3000 planes 122 / 111; 6 x 16
// FP32 600 15.1 / 20.5, 2000 34.2 / 29.0; 12 x 12 FP16 300 17.7 / 20.9, 1200 34.3 / 28.4; 2D D2Q9/D2Q5/D2Q5 FP64 64 x 500
// 24.2 / 32.6, 24 x 4000 42.2 / 39.5.
inline bool few_warps(bool two_d, int tbytes, int sbytes, long long planes) {
  if (two_d && tbytes == 4) return true;
  return planes >= (tbytes == 8 ? 3000 : sbytes == 4 ? 2000 : 1200);
}

// Blocks of `span` nodes of a node-wise kernel at one plane each.
inline long long node_blocks(int nx, int ny, int nz, int span) {
  return ((long long)nx * ny + span - 1) / span * nz;
}

// Planes per block of the node-wise step: one while `blocks` blocks of a plane each do not fill
// the chip several times over, then more, so that a block's start is shared by up to 16 planes
// and phi along z stays in registers.  Measured best (us per step): 48^3 1 plane 20 (4: 43),
// 128^3 FP32 4 planes 241 (16: 267), 256^3 FP16 16 planes 1630 (8: 1660, 32: 1720).
inline int node_zchunk(long long blocks, int nz) {
  const long long zc = blocks / 4000;
  return (int)std::max<long long>(1, std::min<long long>({zc, 16, (long long)nz}));
}

// Rows per block of the plane kernels: blocks are one warp each, 24 of which an SM holds, and run in
// waves, so a simulation of `tiles` blocks per row takes one wave where chunks of 8 to 48 rows make
// one, else chunks of 32 rows (two of which are recomputed).  2D FP16, us per step with chunks that
// count 30-column tiles / these: 2000^2 D2Q9/D2Q5/D2Q5 183 / 134 (half a wave / one), 3000^2 330 / 279
// (1.29 waves / one), D2Q9 x 3 466 / 384; 3400^2 in one wave of 54 rows FP32 D2Q9 x 3 666, in 32 rows 608.
inline int plane_zchunk(long long tiles, int nz) {
  const long long wave = 152 * 24, rows = (nz + std::max(1ll, wave / tiles) - 1) / std::max(1ll, wave / tiles);
  return (int)std::min<long long>(nz, rows <= 48 ? std::max<long long>(rows, 8) : 32);
}

struct TileGeom {
  int nx, ny, nz, zchunk;
};

// Ticket order and dependency lists of the one-launch step over `items` (tiles of TILE_X
// columns and ty rows, z-chunks of geo[sim].zchunk planes, as build_items makes them).  The
// U/theta tile of item j reads phi^{n+1} on columns [x0-2, x0+31], rows [y0-2, y0+by-1] and
// planes [z0-2, z1+1] (clamped to the grid): it depends on every phase-field tile that writes
// part of that box.  Phase-field tickets go by simulation, row tile, z-chunk, then column
// tile, so that the tiles a U/theta tile needs are close together in the order; each U/theta
// ticket follows the last of its phase-field tiles by `lag` phase-field tickets.  False if a
// tile of the box has no work item (a tiling that build_items did not make).
inline bool plan_one_launch(const std::vector<WorkItem>& items, const std::vector<TileGeom>& geo, int by, int lag,
                     std::vector<int>& order, std::vector<int>& dep_off, std::vector<int>& dep) {
  const int ty = by == 1 ? 1 : by - 2;
  const size_t ns = geo.size();
  std::vector<long long> base(ns + 1, 0);
  std::vector<int> nxt(ns), nyt(ns), nct(ns);
  for (size_t k = 0; k < ns; ++k) {
    nxt[k] = (geo[k].nx + TILE_X - 1) / TILE_X;
    nyt[k] = (geo[k].ny + ty - 1) / ty;
    nct[k] = (geo[k].nz + geo[k].zchunk - 1) / geo[k].zchunk;
    base[k + 1] = base[k] + (long long)nxt[k] * nyt[k] * nct[k];
  }
  auto cell = [&](int sim, int c, int r, int q) { return base[sim] + ((long long)r * nct[sim] + c) * nxt[sim] + q; };
  const int n = (int)items.size();
  std::vector<int> at((size_t)base[ns], -1);
  for (int j = 0; j < n; ++j) {
    const WorkItem& w = items[j];
    at[cell(w.sim, w.z0 / geo[w.sim].zchunk, w.y0 / ty, w.x0 / TILE_X)] = j;
  }
  // rank of each item's phase-field ticket: the cell order above
  std::vector<int> rank(n, -1), phi_order;
  phi_order.reserve(n);
  for (int a : at)
    if (a >= 0) {
      rank[a] = (int)phi_order.size();
      phi_order.push_back(a);
    }
  if ((int)phi_order.size() != n) return false;
  dep_off.assign(n + 1, 0);
  dep.clear();
  std::vector<std::vector<int>> after(n);
  for (int j = 0; j < n; ++j) {
    const WorkItem& w = items[j];
    const TileGeom& g = geo[w.sim];
    const int q0 = std::max(w.x0 - 2, 0) / TILE_X, q1 = std::min(w.x0 + 31, g.nx - 1) / TILE_X;
    const int ylo = std::max(w.y0 - 2, 0);
    const int r0 = ylo / ty, r1 = (by == 1 ? ylo : std::min(w.y0 + by - 1, g.ny - 1)) / ty;
    const int c0 = std::max(w.z0 - 2, 0) / g.zchunk, c1 = std::min(w.z1 + 1, g.nz - 1) / g.zchunk;
    int last = 0;
    for (int c = c0; c <= c1; ++c)
      for (int r = r0; r <= r1; ++r)
        for (int q = q0; q <= q1; ++q) {
          const int d = at[cell(w.sim, c, r, q)];
          if (d < 0) return false;
          dep.push_back(d);
          last = std::max(last, rank[d]);
        }
    dep_off[j + 1] = (int)dep.size();
    after[std::min(last + lag, n - 1)].push_back(j);
  }
  order.clear();
  order.reserve(2 * (size_t)n);
  for (int k = 0; k < n; ++k) {
    order.push_back(phi_order[k]);
    for (int j : after[k]) order.push_back(~j);
  }
  return true;
}

}  // namespace lbpf
