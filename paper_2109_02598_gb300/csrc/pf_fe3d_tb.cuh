// Shared by the 3D kernels that stream planes through two dependent levels (pf_fe3d_tb2.cu,
// pf_fe3d_two.cu): the per-site work of four sites and the split of the (row tile, plane) work
// over the CTAs.
#pragma once

#include <algorithm>

#include "pf_grid.h"
#include "pf_internal.h"

namespace pf {

template <int MODEL>
__device__ __forceinline__ void update4(const float4* c, const float4* lap, float4* res,
                                        const ModelParams& m) {
  if constexpr (MODEL == PF_MODEL_AC) {
    res[0].x = ac_update(c[0].x, lap[0].x, m);
    res[0].y = ac_update(c[0].y, lap[0].y, m);
    res[0].z = ac_update(c[0].z, lap[0].z, m);
    res[0].w = ac_update(c[0].w, lap[0].w, m);
  } else {
    gs_update(c[0].x, c[1].x, lap[0].x, lap[1].x, m, res[0].x, res[1].x);
    gs_update(c[0].y, c[1].y, lap[0].y, lap[1].y, m, res[0].y, res[1].y);
    gs_update(c[0].z, c[1].z, lap[0].z, lap[1].z, m, res[0].z, res[1].z);
    gs_update(c[0].w, c[1].w, lap[0].w, lap[1].w, m, res[0].w, res[1].w);
  }
}

// 7-point Laplacians of four sites: centre c, z-neighbours zm/zp, rows above/below and the
// two x-edge scalars of the centre row. Gray-Scott's stencil factor is carried in D_u and D_v
// (its lap_scale is 1), so its final multiply is left out, as lap_scaled does: the same bits,
// eight instructions fewer per float4 and level (GS 256^3: 503 -> 521 GLUPS). The sums run as
// packed FP32 pairs (lap3d_sum4: lap3d_sum's operations in its order, each lane's bits
// unchanged) while the update stays scalar, which splits the arithmetic between the heavy FMA
// pipe (the pairs) and both pipes (the scalars): GS 256^3 558 -> 596 GLUPS. Packing the
// update too loads the heavy pipe alone (measured slower before this change).
template <int MODEL>
__device__ __forceinline__ float4 lap3d_x4(const float4& c, const float4& ym, const float4& yp,
                                           const float4& zm, const float4& zp, float xm,
                                           float xp, float lap_scale) {
  float4 l = lap3d_sum4(c, xm, xp, ym, yp, zm, zp);
  if constexpr (MODEL != PF_MODEL_GS) l = mul4(lap_scale, l);  // lap_scaled
  return l;
}

// The work split with the shortest longest-CTA plane count (each segment streams `halo` planes
// besides its own), ROWS preferred when it is within one plane of the best, since it
// keeps neighbouring tiles in step over z. span_out: the longest CTA's plane count.
inline Tb2Sched tb2_schedule(int ncols, int nz, long long slots, long long* grid_out,
                             long long* span_out = nullptr, int halo = 4) {
  Tb2Sched s{};
  // ITEMS
  long long nchunks = slots / ncols;
  if (nchunks > nz / 4) nchunks = nz / 4;
  if (nchunks < 1) nchunks = 1;
  const int chunk_len = (int)((nz + nchunks - 1) / nchunks);
  nchunks = (nz + chunk_len - 1) / chunk_len;
  const long long items = (long long)ncols * nchunks;
  const long long item_grid = items < slots ? items : slots;
  const long long item_span = (items + item_grid - 1) / item_grid * (chunk_len + halo);
  // BALANCED: about units / slots + 8 planes (two segments at most when a range is under nz)
  const long long units = (long long)ncols * nz;
  const long long per = (units + slots - 1) / slots;
  const long long bal_span = per + (per < nz ? 2 * halo : halo * ((per + nz - 1) / nz + 1));
  const long long bal_grid = slots < units ? slots : units;
  // ROWS
  long long rows_span = -1, rows_L = 0;
  const long long F = slots / ncols, R = slots - F * ncols;
  for (long long L = 4; F >= 1 && L * F <= nz; ++L) {
    const long long Lp = nz - F * L;  // planes of the top row
    long long span = L + halo;
    if (Lp > 0) {
      if (R == 0) continue;
      const long long pu = ((long long)ncols * Lp + R - 1) / R;
      const long long segs = (pu + Lp - 1) / Lp + 1;
      span = std::max(span, pu + halo * segs);
    }
    if (rows_span < 0 || span < rows_span) {
      rows_span = span;
      rows_L = L;
    }
  }
  const long long best = std::min(item_span, slots > item_grid ? bal_span : item_span);
  long long span = item_span;
  if (rows_span > 0 && rows_span <= best + 1) {
    s.mode = kTb2Rows;
    span = rows_span;
    s.full_rows = (int)F;
    s.L = (int)rows_L;
    s.pdir = ((F - 1) & 1) ? 1 : -1;  // meet the last full row's chunk at its end
    *grid_out = (nz - F * rows_L) > 0 ? slots : F * ncols;
  } else if (bal_span < item_span && slots > item_grid) {
    s.mode = kTb2Balanced;
    span = bal_span;
    *grid_out = bal_grid;
  } else {
    s.mode = kTb2Items;
    *grid_out = item_grid;
  }
  if (span_out != nullptr) *span_out = span;
  s.nchunks = (int)nchunks;
  s.chunk_len = chunk_len;
  return s;
}

}  // namespace pf
