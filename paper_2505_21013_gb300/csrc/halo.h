// Host-side tables of the PCG's halo layout (SR_HALO, pcg_sr.cu): for each CTA
// of a launch, the rows of other CTAs that columns of its rows refer to, and
// every block's column in the CTA's local numbering.  Pure host code, so that
// the tables can be built and checked without a GPU.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

#include "kernels.h"

namespace ppn {

// BSR pattern of one scene of the launch (slot order); its rows are split
// into PCG_TILE-row tiles, all of them in the launch's tile table.
struct HaloPattern {
  int nv;
  const int64_t* row_ptr;  // nv + 1
  const int* col;          // row_ptr[nv], ascending per row
};

// Tables for `grid` CTAs over the launch's tile table (every tile of slot 0,
// then of slot 1, ...; CTA b owns tiles [b n / grid, (b + 1) n / grid)), laid
// out as PcgLaunch::halo_off, halo_col, halo_ref one after the other in `tab`:
//   [2 (grid + 1)]   first block and first halo row of each CTA, then the totals
//   [blocks]         local column of each block: own row item (tile index in the
//                    CTA x PCG_TILE + row within the tile), or n_items + the
//                    column's index in the CTA's halo list
//   [halo rows]      slot << HALO_ROW_BITS | row, ascending within each CTA
// Blocks are in the kernel's order: the CTA's tiles, their rows, each row's
// blocks.  Returns the most halo rows of one CTA; -1 when a scene has
// 2^HALO_ROW_BITS rows or more, there are more than HALO_MAX_SCENES scenes, or
// grid is outside [1, tiles].
inline int build_halo_tables(const std::vector<HaloPattern>& pats, int grid, std::vector<int>& tab) {
  const size_t ns = pats.size();
  if (ns == 0 || ns > (size_t)HALO_MAX_SCENES) return -1;
  std::vector<int> toff(ns + 1, 0);
  for (size_t k = 0; k < ns; ++k) {
    if (pats[k].nv <= 0 || pats[k].nv >= (1 << HALO_ROW_BITS)) return -1;
    toff[k + 1] = toff[k] + (pats[k].nv + PCG_TILE - 1) / PCG_TILE;
  }
  const int n_tiles = toff[ns];
  if (grid < 1 || grid > n_tiles) return -1;
  std::vector<std::vector<int>> mark(ns), hidx(ns);
  size_t n_blocks = 0;
  for (size_t k = 0; k < ns; ++k) {
    mark[k].assign(pats[k].nv, -1);
    hidx[k].resize(pats[k].nv);
    n_blocks += (size_t)pats[k].row_ptr[pats[k].nv];
  }
  const size_t col0 = 2 * ((size_t)grid + 1), ref0 = col0 + n_blocks;
  tab.assign(ref0, 0);
  size_t nc = 0;
  std::vector<int> hs;
  int maxh = 0;
  for (int b = 0; b < grid; ++b) {
    const int t0 = (int)(((long long)b * n_tiles) / grid), t1 = (int)(((long long)(b + 1) * n_tiles) / grid);
    const int n_items = (t1 - t0) * PCG_TILE;
    tab[2 * b] = (int)nc;
    tab[2 * b + 1] = (int)(tab.size() - ref0);
    int nh = 0;
    // the CTA's run of rows of each slot in turn: columns within it are its own, the others halo rows
    for (int t = t0, k = (int)(std::upper_bound(toff.begin(), toff.end(), t0) - toff.begin()) - 1; t < t1; ++k) {
      const HaloPattern& p = pats[k];
      const int te = std::min(t1, toff[k + 1]);
      const int r0 = (t - toff[k]) * PCG_TILE, re = (te - toff[k]) * PCG_TILE, item0 = (t - t0) * PCG_TILE;
      const int64_t q0 = p.row_ptr[r0], q1 = p.row_ptr[std::min(p.nv, re)];
      int *mk = mark[k].data(), *hx = hidx[k].data(), lo = p.nv, hi = -1;
      hs.clear();
      for (int64_t q = q0; q < q1; ++q) {
        const int j = p.col[q];
        if ((j < r0 || j >= re) && mk[j] != b) {
          mk[j] = b;
          hs.push_back(j);
          lo = std::min(lo, j);
          hi = std::max(hi, j);
        }
      }
      if (hi - lo < 16 * (int)hs.size()) {  // ascending: a scan of their range, unless they are few in a wide one
        size_t n = 0;
        for (int j = lo; j <= hi; ++j)
          if (mk[j] == b) hs[n++] = j;
      } else {
        std::sort(hs.begin(), hs.end());
      }
      for (int j : hs) {
        hx[j] = nh++;
        tab.push_back((k << HALO_ROW_BITS) | j);
      }
      for (int64_t q = q0; q < q1; ++q) {
        const int j = p.col[q];
        tab[col0 + nc++] = j >= r0 && j < re ? item0 + (j - r0) : n_items + hx[j];
      }
      t = te;
    }
    maxh = std::max(maxh, nh);
  }
  tab[2 * grid] = (int)nc;
  tab[2 * grid + 1] = (int)(tab.size() - ref0);
  return maxh;
}

}  // namespace ppn
