// Streaming a column tile of a 3D grid through shared memory, for the kernels that lay their
// threads out as (row, group of four columns) over rows of any length: the tile's place, the
// copies of a plane, and the walk over a CTA's segments of the work.
#pragma once

#include "pf_fe3d_tb.cuh"
#include "pf_tma.cuh"

namespace pf {

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// A thread's group in a row-major plane of rows of rw floats. cols: the columns after which the row
// repeats. Whole rows: nx, and a last group of nx % 4 columns holds the first columns behind them,
// periodic images that every level computes like the columns they repeat (their right neighbour
// is the column after the last image); strips: any, their outermost columns are not used.
struct GroupPos {
  int rw;       // floats per row: four per group
  int dm, dp;   // offsets of the group's x-neighbours from its first float
  bool nl, nr;  // take them from shared memory (a warp's or a row's end)
  __device__ __forceinline__ GroupPos(int G, int q, int cols) {
    rw = 4 * G;
    dm = q == 0 ? cols - 1 : -1;
    dp = q == G - 1 ? 4 - cols : 4;
    nl = (threadIdx.x & 31) == 0 || q == 0;
    nr = (threadIdx.x & 31) == 31 || q == G - 1;
  }
  // The values left of c.x and right of c.w in the row that `own` (the group) lies in: from the
  // neighbouring lanes, and from shared memory at the ends. Every lane of the warp calls it.
  __device__ __forceinline__ void edges(const float* own, const float4& c, float& xm,
                                        float& xp) const {
    xm = __shfl_up_sync(0xffffffffu, c.w, 1);
    xp = __shfl_down_sync(0xffffffffu, c.x, 1);
    if (nl) xm = own[dm];
    if (nr) xp = own[dp];
  }
};

// The copies of the planes of a column tile into shared memory, one plane after the other in
// direction dir: T + 2 H rows (T output rows; the first is row H) of every field, rows of 4 G
// floats, fields IN_FIELD apart. With R rows of threads (at least T / 2 + H), a thread copies its
// group of row r and of row R + r where there is one, from a pointer that moves on with the plane
// (the fields lie at constant distances).
// RAGGED > 0 (nx % 4 != 0): groups that are not four consecutive columns of the grid come as 4-byte
// copies: a whole row's last group, of a strip the columns within H of it at the ends of the rows;
// 1: at most one a thread, 2: several (short rows). Instantiations of their own: on aligned rows the state and the tests
// alone cost every warp 46 of 221 instructions a plane (one step of Gray-Scott), and the loop of
// 2 costs the others 4 to 10 %.
template <int NF, int H, int IN_FIELD, int RAGGED>
struct PlaneCopy {
  const float* pa;  // the group of row r of field 0, in the plane that is next
  int64_t db;           // from there to the group of row R + r
  int dst_a, dst_b, zin, dir, nz;
  int64_t step, wrap;   // to the next plane, and past the grid's last (or first) one
  bool has_a, has_b, warp_b;
  // the 4-byte copies: columns a row, left ones, first right one
  int nsc, nl, fr, items, sdst, xs, y0, T, rw;
  const float* ps;

  __device__ __forceinline__ const float* scalar_item(const FieldPtrs& in, const Geom& g, int i,
                                                      int& dst) const {
    const int k = i % nsc, rf = i / nsc;
    const int row = rf % (T + 2 * H), f = rf / (T + 2 * H);
    const int cx = k < nl ? k - H : fr + (k - nl);
    const float* base = in.f[0];
#pragma unroll
    for (int j = 1; j < NF; ++j)
      if (f == j) base = in.f[j];
    dst = f * IN_FIELD + row * rw + (cx - xs);
    return base + ((int64_t)zin * g.plane + (int64_t)wrap_index(y0 - H + row, g.ny) * g.pitch +
                   wrap_index(cx, g.nx));
  }

  // the tile of output columns [x0, x1), T rows from y0; lpad staged columns left of x0; the
  // first plane z
  __device__ __forceinline__ PlaneCopy(const FieldPtrs& in, const Geom& g, int x0_, int x1, int y0_,
                                       int lpad, int G, int T_, int R, int r, int q, bool live,
                                       int z, int dir_) {
    zin = wrap_index(z, g.nz);
    dir = dir_;
    nz = g.nz;
    step = dir > 0 ? g.plane : -g.plane;
    wrap = step - (dir > 0 ? g.plane : -g.plane) * g.nz;
    rw = 4 * G;
    dst_a = r * rw + 4 * q;
    dst_b = dst_a + R * rw;
    int cx = x0_ - lpad + 4 * q;
    if constexpr (RAGGED == 0) cx = wrap_index(cx, g.nx);  // a group wraps whole
    has_a = live && (RAGGED == 0 || (cx >= 0 && cx + 3 < g.nx));
    has_b = has_a && R + r < T_ + 2 * H;
    warp_b = __any_sync(0xffffffffu, has_b);
    const int ya = wrap_index(y0_ - H + r, g.ny), yb = wrap_index(y0_ - H + R + r, g.ny);
    const int64_t o = (int64_t)zin * g.plane + (int64_t)ya * g.pitch + (has_a ? cx : 0);
    db = (int64_t)(yb - ya) * g.pitch;
    pa = in.f[0] + o;
    if constexpr (RAGGED > 0) {
      xs = x0_ - lpad;
      y0 = y0_;
      T = T_;
      // strips: H columns left of the first one, and from the grid's last whole group to H past
      // the strip's last column
      nl = lpad > 0 && x0_ == 0 ? H : 0;
      fr = max(g.nx & ~3, xs);
      nsc = lpad > 0 ? nl + max(0, x1 + H - fr) : 4;
      items = NF * (T + 2 * H) * nsc;
      sdst = 0;
      ps = nullptr;
      if ((int)threadIdx.x < items) ps = scalar_item(in, g, threadIdx.x, sdst);
    }
  }

  // copy the next plane into the ring slot at st, and move on
  __device__ __forceinline__ void stage(const FieldPtrs& in, const Geom& g, float* st) {
    if (has_a) {
#pragma unroll
      for (int f = 0; f < NF; ++f) cp_async16(st + f * IN_FIELD + dst_a, pa + (in.f[f] - in.f[0]));
    }
    if (warp_b) {
      if (has_b) {
#pragma unroll
        for (int f = 0; f < NF; ++f) cp_async16(st + f * IN_FIELD + dst_b, pa + (db + (in.f[f] - in.f[0])));
      }
    }
    if constexpr (RAGGED > 0) {
      if (ps != nullptr) cp_async4(st + sdst, ps);
    }
    if constexpr (RAGGED == 2) {
      for (int k = threadIdx.x + blockDim.x; k < items; k += blockDim.x) {
        int d;
        const float* p = scalar_item(in, g, k, d);
        cp_async4(st + d, p);
      }
    }
    int64_t s = step;
    zin += dir;
    if ((unsigned)zin >= (unsigned)nz) {
      s = wrap;
      zin = dir > 0 ? 0 : nz - 1;
    }
    pa += s;
    if constexpr (RAGGED > 0)
      if (ps != nullptr) ps += s;
  }
};

// Store a thread's group of output columns gx .. gx + 3, those from x1 on as zeros: strips are a
// multiple of 4 wide, so they are the places behind the row's end, which stay zero that way (one
// vector store for every group: 4 to 6 % faster on ragged rows than column by column at their ends).
template <int NF, int RAGGED>
__device__ __forceinline__ void store_group(const FieldOut& out, int64_t off, float4 (&v)[NF],
                                            int gx, int x1) {
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    if constexpr (RAGGED > 0) {
      if (gx + 1 >= x1) v[f].y = 0.f;
      if (gx + 2 >= x1) v[f].z = 0.f;
      if (gx + 3 >= x1) v[f].w = 0.f;
    }
    *reinterpret_cast<float4*>(out.f[f] + off) = v[f];
  }
}

// A CTA's segments (column tile, z-range, direction) of the schedule.
struct SegmentWalk {
  int64_t pos = 0, pos_end = 0;
  int item, nfull;
  int col, zlo, zhi, dir;
  __device__ __forceinline__ SegmentWalk(const Tb2Sched& s, int ncols, int nz) {
    item = blockIdx.x;
    nfull = s.full_rows * ncols;
    if (s.mode == kTb2Balanced) {
      const int64_t units = (int64_t)ncols * nz;
      pos = units * blockIdx.x / gridDim.x;
      pos_end = units * (blockIdx.x + 1) / gridDim.x;
    } else if (s.mode == kTb2Rows && (int)blockIdx.x >= nfull) {
      const int64_t units = (int64_t)ncols * (nz - s.full_rows * s.L);
      const int p = blockIdx.x - nfull, np = gridDim.x - nfull;
      pos = units * p / np;
      pos_end = units * (p + 1) / np;
    }
  }
  // the next segment; false: none left (uniform over the CTA)
  __device__ __forceinline__ bool next(const Tb2Sched& s, int ncols, int nz) {
    const bool rows = s.mode == kTb2Rows;
    if (s.mode == kTb2Items || (rows && (int)blockIdx.x < nfull)) {
      do {
        if (item >= (rows ? nfull : ncols * s.nchunks)) return false;
        col = item % ncols;
        const int chunk = item / ncols;
        const int len = rows ? s.L : s.chunk_len;
        zlo = chunk * len;
        zhi = min(nz, zlo + len);
        dir = (chunk & 1) ? -1 : 1;
        item += rows ? nfull : gridDim.x;
      } while (zlo >= zhi);
      return true;
    }
    if (pos >= pos_end) return false;
    const int zbase = rows ? s.full_rows * s.L : 0;
    const int zlen = nz - zbase;
    col = (int)(pos / zlen);
    zlo = (int)(pos - (int64_t)col * zlen);
    zhi = (int)min((int64_t)zlen, zlo + (pos_end - pos));
    pos += zhi - zlo;
    zlo += zbase;
    zhi += zbase;
    dir = rows ? s.pdir : ((blockIdx.x & 1) ? -1 : 1);
    return true;
  }
};

// The PlaneCopy form for a tile: whether its 4-byte copies fit one a thread.
inline int copy_form(const Geom& g, const StreamTiles& p, int nf, int H, int threads) {
  const int row = p.lpad > 0 ? 2 * H + 3 : 4;  // copies a row (at most)
  return g.nx % 4 == 0 ? 0 : nf * (p.TY + 2 * H) * row <= threads ? 1 : 2;
}

// Tiles and work split of a grid for a kernel of at most nt threads, row-halo H, whose threads
// cover T = TY + trim rows. Rows of at most 4 maxg columns whole, longer ones in
// equal strips (ragged rows too: as strips with a halo group on either side and seven 4-byte copies
// a row they took 3 to 25 % longer, the longer the shorter the row); the tile height that makes the launch shortest by span * (c0 + warps): the
// longest CTA's plane count times a plane's time, linear in the CTA's warps above a fixed part
// for the barrier and the latencies behind it.
inline StreamPlan stream_plan(const Geom& g, long long sms, int nt, int maxg, int H, int trim,
                              int c0) {
  StreamPlan pl{};
  StreamTiles& p = pl.tiles;
  if (g.nx <= 4 * maxg) {
    p.G = (g.nx + 3) / 4;
    p.S = 1;
    p.w = g.nx;
  } else {
    const int wmax = 4 * maxg - 8;
    p.lpad = 4;
    p.S = (g.nx + wmax - 1) / wmax;
    p.w = ((g.nx + p.S - 1) / p.S + 3) / 4 * 4;
    p.S = (g.nx + p.w - 1) / p.w;
    p.G = (4 + p.w + H + 3) / 4;  // the halo group, w columns, and H more columns
  }
  const int tmax = std::min(nt / p.G - trim, g.ny);
  long long best = -1;
  int last = 0;
  for (int t = tmax; t >= 1; --t) {
    const int tiles = (g.ny + t - 1) / t;
    const int ty = (g.ny + tiles - 1) / tiles;  // spread evenly
    if (ty == last) continue;
    last = ty;
    long long gr = 0, span = 0;
    const long long ncols = (long long)p.S * tiles;
    if (pl.valid && ncols > 64 * sms) break;  // enough tiles: taller ones have less halo
    const Tb2Sched s = tb2_schedule((int)ncols, g.nz, sms, &gr, &span, 2 * H);
    const long long cost = span * (c0 + ((ty + trim) * p.G + 31) / 32);
    if (best < 0 || cost < best) {
      best = cost;
      p.TY = ty;
      pl.sched = s;
      pl.grid = (unsigned)gr;
      pl.valid = true;
    }
  }
  return pl;
}

}  // namespace pf
