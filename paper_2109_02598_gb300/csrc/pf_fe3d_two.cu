// 3D forward-Euler with the 7-point Laplacian on grids of any size: planes streamed through
// two dependent levels (Sec. 2.4.1 solver, Sec. 2.2.2 stencil, Sec. 3 models).
//   Allen-Cahn, Gray-Scott: level 1 is the first of two time steps, level 2 the second, so a
//     pass over HBM advances two steps;
//   Model B, Model C: level 1 is the chemical potential mu (of phi; of m), level 2 the step.
// Both reach two sites. The arithmetic is that of every other kernel (the same bits).
//
// A CTA takes a column tile (a strip of w output columns, TY rows) through a z-range. Its rows
// are laid out in groups of four columns, G per row, one thread per (level-1 row, group):
// thread t = r G + q, r = 0 .. TY + 1, so any row length fills the warps, and TY is as large
// as the threads allow (short rows: tall tiles). Per input plane, rows y0-2 .. y0+TY+1 of
// every field come into an NS-plane ring by cp.async, NS - 2 planes ahead: a 16-byte copy per
// thread and field for its group of row r (rows TY+2 and TY+3 by the threads of rows 0 and 1),
// from offsets within the plane that the thread computes once per tile. Iteration j computes
// level-1 plane j on rows y0-1 .. y0+TY from input planes j, j+1, j+2 (z-neighbours and centre
// in registers, y-neighbours from the ring) into one of two shared planes, then level 2 of
// output plane j - 2 from level-1 planes j - 2, j - 1, j (again the z-neighbours in registers);
// one CTA barrier per plane. x-neighbours come from the neighbouring lanes by shuffle, and at a
// warp's or a row's end from shared memory.
//   Whole rows (nx at most 256): G = nx / 4, rounded up; the row wraps in shared memory, and a
//     last group of nx % 4 columns is filled up with periodic images of the first ones.
//   Strips (longer rows): one halo group on the left, enough on the right for two columns,
//     staged at periodic columns; the level-1 values of a strip's outermost columns are wrong
//     and reach only columns that the strip does not store.
//   Groups that are not four consecutive columns of the grid (the ends of a row of nx % 4 != 0
//     columns) come as 4-byte copies of the columns the levels read.
//
// What bounds it (two time steps of Gray-Scott, 256^3, 640 threads, one CTA per SM): issue and
// the latencies behind the plane barrier; a plane takes 0.37 us + 0.035 us per warp. GLUPS
// against the general kernels it replaces (32x16 tiles, 4-byte copies or one plane in flight):
// GS 210x179x150 416 / 191, 256^3 585 / 200; AC 210x179x150 732 / 301, 256^3 1015 / 376; Model B
// 382 / 102 and 536 / 134; Model C 232 / 88 and 328 / 110 (TMA tiles, 256^3: 369, 716, 393,
// 165). NS = 5 planes leave three in flight over a plane's 1.1 us (4 and 6 measured the same).
// 640 threads: with 768 (80 registers) GS 256^3 gains 3 %, but AC, Models B and C lose 1 to
// 10 %; two CTAs of 320 threads per SM lose 17 % there (shorter tiles, more halo) and gain 2 to
// 5 % only below 100^3. The copies' pointer and the output offset advance from plane to plane
// (+5 to 13 % over computing them from j); the ring slots do not (offsets kept instead of slot
// numbers cost Gray-Scott 13 %, the compiler then reloading them), and level 2's rows are read
// after level 1 (before it: 1 to 4 % slower).
#include "pf_fe3d_stream.cuh"
#include "pf_grid.h"

#include <type_traits>

namespace pf {

namespace {

constexpr int kTwoThreads = 640;   // 20 warps: the most that leave a thread 96 registers
constexpr int kTwoStages = 5;      // input planes in the ring
constexpr int kTwoMaxGroups = 64;  // groups per row, halo groups included

template <int MODEL>
struct CfgTwo {
  static constexpr int NF = ModelTraits<MODEL>::NF;
  static constexpr bool kSteps = ModelTraits<MODEL>::R == 1;  // two time steps (else mu + step)
  static constexpr int NL1 = kSteps ? NF : 1;                 // fields of a level-1 plane
  static constexpr int NS = kTwoStages;
  static constexpr int IN_FIELD = 4 * kTwoThreads + 8 * kTwoMaxGroups;  // (TY + 4) rows of 4 G floats
  static constexpr int IN_STAGE = NF * IN_FIELD;
  static constexpr int L1_FIELD = 4 * kTwoThreads;                       // (TY + 2) rows
  static constexpr int L1_PLANE = NL1 * L1_FIELD;
  static constexpr size_t SMEM = (size_t)(NS * IN_STAGE + 2 * L1_PLANE) * 4;
};

// z-windows of one thread's column group, three slots each, slot = plane mod 3 (the plane loop
// is unrolled by three, so they are renamed instead of moved).
template <int MODEL>
struct TwoStream {
  using C = CfgTwo<MODEL>;
  static constexpr int NF = C::NF, NL1 = C::NL1;
  float4 iw[NF][3];   // input planes
  float4 lw[NL1][3];  // level-1 planes
  float4 lpsi;        // Model C: Laplacian of psi on the plane level 2 takes next

  // Level 1 of phase P: sc the ring's plane j + 1, sp its plane j + 2, both at the thread's own
  // group; l1w the level-1 plane at the group (written where live).
  template <int P>
  __device__ __forceinline__ void level1(const float* sc, const float* sp, float* l1w,
                                         const GroupPos& t, bool live, const ModelParams& m,
                                         float4& lpsi_next) {
    constexpr int S0 = P, S1 = (P + 1) % 3, S2 = (P + 2) % 3;
    float4 lap[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const float* F = sc + f * C::IN_FIELD;
      const float4 ym = ld4(F - t.rw), yp = ld4(F + t.rw);
      iw[f][S2] = ld4(sp + f * C::IN_FIELD);
      float xm, xp;
      t.edges(F, iw[f][S1], xm, xp);
      lap[f] = lap3d_x4<MODEL>(iw[f][S1], ym, yp, iw[f][S0], iw[f][S2], xm, xp, m.lap_scale);
    }
    if constexpr (C::kSteps) {
      float4 c[NF], res[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) c[f] = iw[f][S1];
      update4<MODEL>(c, lap, res, m);
#pragma unroll
      for (int f = 0; f < NF; ++f) lw[f][S0] = res[f];
    } else if constexpr (MODEL == PF_MODEL_CH) {
      lw[0][S0] = ch_mu4(iw[0][S1], lap[0], m);
    } else {
      lw[0][S0] = mc_mu4(iw[0][S1], iw[1][S1], lap[1], m);
      lpsi_next = lap[0];
    }
    if (live) {
#pragma unroll
      for (int f = 0; f < NL1; ++f) *reinterpret_cast<float4*>(l1w + f * C::L1_FIELD) = lw[f][S0];
    }
  }

  // Level 2 of output plane j - 2 (phase P): l1r the level-1 plane j - 1 at the thread's group,
  // ym / yp the offsets of the rows above and below.
  template <int P>
  __device__ __forceinline__ void level2(const float* l1r, int ym_off, int yp_off,
                                         const GroupPos& t, const ModelParams& m,
                                         float4 (&res)[NF]) {
    constexpr int S0 = P, S1 = (P + 1) % 3, S2 = (P + 2) % 3;
    float4 lap[NL1];
#pragma unroll
    for (int f = 0; f < NL1; ++f) {
      const float* F = l1r + f * C::L1_FIELD;
      const float4 ym = ld4(F + ym_off), yp = ld4(F + yp_off);
      float xm, xp;
      t.edges(F, lw[f][S2], xm, xp);
      lap[f] = lap3d_x4<MODEL>(lw[f][S2], ym, yp, lw[f][S1], lw[f][S0], xm, xp, m.lap_scale);
    }
    if constexpr (C::kSteps) {
      float4 c[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) c[f] = lw[f][S2];
      update4<MODEL>(c, lap, res, m);
    } else if constexpr (MODEL == PF_MODEL_CH) {
      res[0] = ch_update4(iw[0][S0], lap[0], m);
    } else {
      mc_update4(iw[0][S0], iw[1][S0], lpsi, lap[0], m, res[0], res[1]);
    }
  }
};

template <int MODEL, int RAGGED>
__global__ void __launch_bounds__(kTwoThreads, 1)
    fe3d_two_kernel(FieldPtrs in, FieldOut out, Geom g, ModelParams m, StreamTiles pl, Tb2Sched sc_) {
  using C = CfgTwo<MODEL>;
  constexpr int NF = C::NF, NS = C::NS;
  extern __shared__ __align__(16) float smem[];
  float* ring = smem;
  float* l1 = smem + NS * C::IN_STAGE;
  const int tid = threadIdx.x;
  const int G = pl.G, TY = pl.TY;
  canary_fill(smem, (size_t)NS * C::IN_STAGE + 2 * C::L1_PLANE);

  const bool live = tid < (TY + 2) * G;  // the last warp's spare threads repeat the last group
  const int t_ = live ? tid : (TY + 2) * G - 1;
  const int r = t_ / G, q = t_ - r * G;
  const GroupPos t(G, q, RAGGED > 0 && pl.lpad == 0 ? g.nx : 4 * G);
  const int o1 = r * t.rw + 4 * q;  // own group in a level-1 plane; in an input plane o1 + rw
  const int ym2 = r > 0 ? -t.rw : 0, yp2 = r < TY + 1 ? t.rw : 0;  // rows level 2 may read
  const bool inner = r >= 1 && r <= TY;
  const bool warp2 = __any_sync(0xffffffffu, inner && live);

  const int ncols = pl.S * ((g.ny + TY - 1) / TY);
  SegmentWalk seg(sc_, ncols, g.nz);
  TwoStream<MODEL> zs;
  chain_wait();
  while (seg.next(sc_, ncols, g.nz)) {
    const int col = seg.col, zlo = seg.zlo, zhi = seg.zhi, dir = seg.dir;
    const int n = zhi - zlo;  // output planes
    const int zfirst = dir > 0 ? zlo : zhi - 1;
    const int nin = n + 4;  // input planes zfirst - 2 dir .. zlast + 2 dir
    const int strip = col % pl.S;
    const int x0 = strip * pl.w, y0 = (col / pl.S) * TY;
    const int x1 = min(g.nx, x0 + pl.w);

    PlaneCopy<NF, 2, C::IN_FIELD, RAGGED> cp(in, g, x0, x1, y0, pl.lpad, G, TY, TY + 2, r, q, live,
                                             zfirst - 2 * dir, dir);

    // where this thread stores: its output row and columns
    const int gy = y0 + r - 1, gx = x0 - pl.lpad + 4 * q;
    const bool store = live && inner && gy < g.ny && gx >= x0 && gx < x1;
    int64_t off = (int64_t)zfirst * g.plane + (int64_t)gy * g.pitch + gx;
    const int64_t off_step = dir > 0 ? g.plane : -g.plane;

    __syncthreads();  // every thread is done with the last segment's planes
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      if (i < nin) cp.stage(in, g, ring + i * C::IN_STAGE);
      cp_async_commit();
    }
    cp_async_wait_group<NS - 2>();  // input planes 0 and 1
    __syncthreads();
    const int oi = o1 + t.rw;  // own group in an input plane
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      zs.iw[f][0] = ld4(ring + f * C::IN_FIELD + oi);
      zs.iw[f][1] = ld4(ring + C::IN_STAGE + f * C::IN_FIELD + oi);
    }
    int s0 = 0, s1 = 1, s2 = 2;  // ring slots of input planes j, j + 1, j + 2
    auto plane = [&](auto phase, int j) {
      constexpr int P = decltype(phase)::value;
      cp_async_wait_group<NS - 3>();  // input plane j + 2 has landed
      __syncthreads();                // ... for every thread, and plane j's slot is free
      if (j + NS < nin) cp.stage(in, g, ring + s0 * C::IN_STAGE);
      cp_async_commit();  // possibly empty: one group per iteration
      float* l1w = l1 + (j & 1) * C::L1_PLANE + o1;
      const float* l1r = l1 + ((j + 1) & 1) * C::L1_PLANE + o1;
      float4 lpsi_next = zs.lpsi;
      zs.template level1<P>(ring + s1 * C::IN_STAGE + oi, ring + s2 * C::IN_STAGE + oi, l1w, t,
                            live, m, lpsi_next);
      s0 = s1;
      s1 = s2;
      if (++s2 == NS) s2 = 0;
      if (j >= 2 && warp2) {
        float4 res[NF];
        zs.template level2<P>(l1r, ym2, yp2, t, m, res);
        if (store) store_group<NF, RAGGED>(out, off, res, gx, x1);
      }
      if (j >= 2) off += off_step;
      if constexpr (MODEL == PF_MODEL_C) zs.lpsi = lpsi_next;
    };
    const int nj = n + 2;
    for (int j = 0; j < nj; j += 3) {
      plane(std::integral_constant<int, 0>(), j);
      if (j + 1 >= nj) break;
      plane(std::integral_constant<int, 1>(), j + 1);
      if (j + 2 >= nj) break;
      plane(std::integral_constant<int, 2>(), j + 2);
    }
    cp_async_wait_all();  // (the last groups are empty)
  }
}

// The plan's fixed part, in warps. Fitted to 450 timed (grid, height) pairs of all four models,
// 64^3 to 256^3 (a plane of Gray-Scott 0.37 + 0.035 warps us, of Allen-Cahn 0.25 + 0.021); its
// choice was within 1 % of the best height on eight of nine grids (4 % on the ninth), where the
// tallest tile lost up to 55 % (64^3).
constexpr int kTwoPlaneWarps = 11;

template <int MODEL, int RAGGED>
cudaError_t launch_two_(pf_grid_s* gr, FieldPtrs in, FieldOut out, cudaStream_t st) {
  using C = CfgTwo<MODEL>;
  auto kern = fe3d_two_kernel<MODEL, RAGGED>;
  static unsigned long long attr_mask = 0;  // per instantiation and device
  cudaError_t e = ensure_smem_attr(kern, C::SMEM, &attr_mask);
  if (e != cudaSuccess) return e;
  const StreamTiles& p = gr->two.tiles;
  const int nt = ((p.TY + 2) * p.G + 31) / 32 * 32;
  return launch_chained(kern, gr->two.grid, nt, C::SMEM, st, in, out, grid_geom(gr), gr->params, p,
                        gr->two.sched);
}

template <int MODEL>
cudaError_t launch_two(pf_grid_s* gr, FieldPtrs in, FieldOut out, cudaStream_t st) {
  const StreamTiles& p = gr->two.tiles;
  switch (copy_form(grid_geom(gr), p, CfgTwo<MODEL>::NF, 2, (p.TY + 2) * p.G)) {
    case 0: return launch_two_<MODEL, 0>(gr, in, out, st);
    case 1: return launch_two_<MODEL, 1>(gr, in, out, st);
  }
  return launch_two_<MODEL, 2>(gr, in, out, st);
}

}  // namespace

// Depth 2 for Allen-Cahn and Gray-Scott, depth 1 for Models B and C.
cudaError_t launch_fe3d_two(pf_grid_s* gr, int src, int dst, cudaStream_t st) {
  if (!gr->two.valid) {
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, gr->device);
    if (e != cudaSuccess) return e;
    gr->two = stream_plan(grid_geom(gr), sms, kTwoThreads, kTwoMaxGroups, 2, 2, kTwoPlaneWarps);
  }
  FieldPtrs in{};
  FieldOut out{};
  for (int f = 0; f < gr->nf; ++f) {
    in.f[f] = gr->buf[src][f];
    out.f[f] = gr->buf[dst][f];
  }
  switch (gr->model) {
    case PF_MODEL_AC: return launch_two<PF_MODEL_AC>(gr, in, out, st);
    case PF_MODEL_GS: return launch_two<PF_MODEL_GS>(gr, in, out, st);
    case PF_MODEL_CH: return launch_two<PF_MODEL_CH>(gr, in, out, st);
    case PF_MODEL_C: return launch_two<PF_MODEL_C>(gr, in, out, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace pf
