// 3D forward-Euler, one step a launch, for the radius-1 updates on grids of any size
// (Sec. 2.4.1 solver): Allen-Cahn and Gray-Scott with the 7-, 19- and 27-point Laplacians
// (Sec. 2.2.2), and N coupled species with the 7-point one (Sec. 2.3). Planes stream through
// shared memory as in pf_fe3d_two.cu (its comment has the layout: one thread per row and group
// of four columns, rows of any length, an NS-plane cp.async ring from offsets a thread computes
// once per tile), with a halo of one row and one plane.
//
// Iteration j takes output plane j of the segment from input planes j, j + 1, j + 2; each kind
// of update keeps what it needs of them in registers, in slots named by plane mod 3 (the plane
// loop is unrolled by three, so they are renamed instead of moved):
//   7-point: the group's values on the three planes; rows above and below from the ring;
//   19- and 27-point: when a plane enters, its three rows are read once and its sums formed:
//     F = the site, E = (x-1 + x+1) + (y-1 + y+1), C = the four in-plane diagonals; then
//     faces = E(z) + (F(z-1) + F(z+1)), edges = C(z) + (E(z-1) + E(z+1)), corners =
//     C(z-1) + C(z+1), as lap3d_iso and lap3d_iso27 take them.
//
// Bound by latency at small sizes (a CTA takes only some ten planes a launch, behind a
// prologue) and by issue at large ones. Two CTAs per SM (one of 640 threads waits at its barrier
// with nothing else to run: 27-point 160^3 209 GLUPS, then 285 with two); three of 256 leave the
// species too few registers. GLUPS against the kernels it replaces, 160^3: Gray-Scott 27-point 158
// -> 302, 19-point 167 -> 312; Allen-Cahn 27-point 265 -> 485; three species 116 -> 186 (136 x 144
// x 160: 108 -> 176). Ragged rows (161^3): 255, 278, 392 and 153.
#include "pf_fe3d_stream.cuh"
#include "pf_grid.h"
#include "pf_rd.cuh"

#include <algorithm>
#include <type_traits>

namespace pf {

namespace {

constexpr int kOneMaxGroups = 64;
constexpr int kOnePlaneWarps = 11;  // the plan's fixed part (stream_plan)

// ---- the updates. A: kernel argument; NT: threads whose registers the update's state leaves
// room for; PHASES: 3 where the state is named by plane mod 3; LIVE: planes an iteration reads
// (2: j + 1 and j + 2; 3: j too); NS: planes in the ring

// 7-point windows of NF fields
template <int NF, int IN_FIELD>
struct Window7 {
  float4 w[NF][3];
  __device__ __forceinline__ void first(const float* p0, const float* p1) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      w[f][0] = ld4(p0 + f * IN_FIELD);
      w[f][1] = ld4(p1 + f * IN_FIELD);
    }
  }
  // neighbour sums (before the factor) on the plane at sc, with the one at sp entering
  template <int P>
  __device__ __forceinline__ void sums(const float* sc, const float* sp, const GroupPos& t,
                                       float4 (&l)[NF]) {
    constexpr int S0 = P, S1 = (P + 1) % 3, S2 = (P + 2) % 3;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const float* F = sc + f * IN_FIELD;
      const float4 ym = ld4(F - t.rw), yp = ld4(F + t.rw);
      w[f][S2] = ld4(sp + f * IN_FIELD);
      float xm, xp;
      t.edges(F, w[f][S1], xm, xp);
      l[f] = lap3d_sum4(w[f][S1], xm, xp, ym, yp, w[f][S0], w[f][S2]);
    }
  }
};

template <int MODEL>
struct Std7 {
  using A = ModelParams;
  static constexpr int NF = ModelTraits<MODEL>::NF, NT = 320, CTAS = 2;
  static constexpr int PHASES = 3, LIVE = 2, NS = 5;
  static constexpr int IN_FIELD = 4 * NT + 8 * kOneMaxGroups;
  Window7<NF, IN_FIELD> win;
  __device__ __forceinline__ void first(const float* p0, const float* p1, const GroupPos&) {
    win.first(p0, p1);
  }
  template <int P>
  __device__ __forceinline__ void step(const float*, const float* sc, const float* sp,
                                       const GroupPos& t, const A& m, float4 (&res)[NF]) {
    float4 l[NF], c[NF];
    win.template sums<P>(sc, sp, t, l);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      c[f] = win.w[f][(P + 1) % 3];
      if constexpr (MODEL != PF_MODEL_GS) l[f] = mul4(m.lap_scale, l[f]);  // lap_scaled
    }
    update4<MODEL>(c, l, res, m);
  }
};

// N species: the planes' values from shared memory every time (no register windows: the reaction
// is long, and with one phase it is in the kernel once)
template <int NF_>
struct Species {
  using A = RdParams;
  static constexpr int NF = NF_, NT = NF == 4 ? 256 : 320, CTAS = 2;
  static constexpr int PHASES = 1, LIVE = 3, NS = NF == 4 ? 4 : 5;
  static constexpr int IN_FIELD = 4 * NT + 8 * kOneMaxGroups;
  __device__ __forceinline__ void first(const float*, const float*, const GroupPos&) {}
  template <int P>
  __device__ __forceinline__ void step(const float* sb, const float* sc, const float* sp,
                                       const GroupPos& t, const A& p, float4 (&res)[NF]) {
    float4 l[NF], u[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const float* F = sc + f * IN_FIELD;
      u[f] = ld4(F);
      float xm, xp;
      t.edges(F, u[f], xm, xp);
      l[f] = lap3d_sum4(u[f], xm, xp, ld4(F - t.rw), ld4(F + t.rw), ld4(sb + f * IN_FIELD),
                        ld4(sp + f * IN_FIELD));
    }
    rd_sites4<NF>(u, l, p, res);
  }
};

template <int MODEL, int ST>
struct Iso {
  using A = ModelParams;
  static constexpr int NF = ModelTraits<MODEL>::NF, NT = NF == 2 ? 256 : 320, CTAS = 2;
  static constexpr int PHASES = 3, LIVE = 2, NS = 5;
  static constexpr int IN_FIELD = 4 * NT + 8 * kOneMaxGroups;
  float4 F[NF][3], E[NF][3], C[NF][3];

  template <int W>
  __device__ __forceinline__ void enter(const float* p, const GroupPos& t) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const float* q = p + f * IN_FIELD;
      const float4 b = ld4(q - t.rw), c = ld4(q), a = ld4(q + t.rw);
      float bm, bp, cm, cp, am, ap;
      t.edges(q - t.rw, b, bm, bp);
      t.edges(q, c, cm, cp);
      t.edges(q + t.rw, a, am, ap);
      auto pair = [](const float4& v, float m, float p_) {  // x-1 + x+1 of the four sites
        return make_float4(__fadd_rn(m, v.y), __fadd_rn(v.x, v.z), __fadd_rn(v.y, v.w),
                           __fadd_rn(v.z, p_));
      };
      F[f][W] = c;
      E[f][W] = add4(pair(c, cm, cp), add4(b, a));
      C[f][W] = add4(pair(b, bm, bp), pair(a, am, ap));
    }
  }
  __device__ __forceinline__ void first(const float* p0, const float* p1, const GroupPos& t) {
    enter<0>(p0, t);
    enter<1>(p1, t);
  }
  template <int P>
  __device__ __forceinline__ void step(const float*, const float*, const float* sp,
                                       const GroupPos& t, const A& m, float4 (&res)[NF]) {
    constexpr int S0 = P, S1 = (P + 1) % 3, S2 = (P + 2) % 3;
    enter<S2>(sp, t);
    float4 c[NF], l[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      c[f] = F[f][S1];
      const float4 faces = add4(E[f][S1], add4(F[f][S0], F[f][S2]));
      const float4 edges = add4(C[f][S1], add4(E[f][S0], E[f][S2]));
      float4 s;  // lap3d_iso, lap3d_iso27
      if constexpr (ST == PF_ST_ISO) {
        s = fma4(-24.0f, c[f], fma4(2.0f, faces, edges));
      } else {
        const float4 corners = add4(C[f][S0], C[f][S2]);
        s = fma4(-128.0f, c[f], fma4(14.0f, faces, fma4(3.0f, edges, corners)));
      }
      l[f] = s;
      if constexpr (MODEL != PF_MODEL_GS) l[f] = mul4(m.lap_scale, s);  // lap_scaled
    }
    update4<MODEL>(c, l, res, m);
  }
};

template <class U, int RAGGED>
__global__ void __launch_bounds__(U::NT, U::CTAS)
    fe3d_one_kernel(FieldPtrs in, FieldOut out, Geom g, typename U::A arg, StreamTiles pl,
                    Tb2Sched sc_) {
  constexpr int NF = U::NF, NS = U::NS, STAGE = NF * U::IN_FIELD;
  constexpr int AHEAD = NS + 2 - U::LIVE;  // planes staged before plane 0 is taken
  extern __shared__ __align__(16) float ring[];
  const int tid = threadIdx.x;
  const int G = pl.G, TY = pl.TY;
  canary_fill(ring, (size_t)NS * STAGE);
  const int R = max(TY, 2);       // rows of threads (a one-row tile's three input rows need two)
  const bool live = tid < R * G;  // the last warp's spare threads repeat the last group
  const int t_ = live ? tid : R * G - 1;
  const int r = t_ / G, q = t_ - r * G;
  const GroupPos t(G, q, RAGGED > 0 && pl.lpad == 0 ? g.nx : 4 * G);
  const int oi = (r + 1) * t.rw + 4 * q;  // own group in an input plane

  const int ncols = pl.S * ((g.ny + TY - 1) / TY);
  SegmentWalk seg(sc_, ncols, g.nz);
  U u;
  chain_wait();
  while (seg.next(sc_, ncols, g.nz)) {
    const int n = seg.zhi - seg.zlo, dir = seg.dir;  // output planes
    const int zfirst = dir > 0 ? seg.zlo : seg.zhi - 1;
    const int nin = n + 2;  // input planes zfirst - dir .. zlast + dir
    const int x0 = (seg.col % pl.S) * pl.w, y0 = (seg.col / pl.S) * TY;
    const int x1 = min(g.nx, x0 + pl.w);

    PlaneCopy<NF, 1, U::IN_FIELD, RAGGED> cp(in, g, x0, x1, y0, pl.lpad, G, TY, R, r, q, live,
                                             zfirst - dir, dir);
    // where this thread stores
    const int gy = y0 + r, gx = x0 - pl.lpad + 4 * q;
    const bool store = live && r < TY && gy < g.ny && gx >= x0 && gx < x1;
    int64_t off = (int64_t)zfirst * g.plane + (int64_t)gy * g.pitch + gx;
    const int64_t off_step = dir > 0 ? g.plane : -g.plane;

    __syncthreads();  // every thread is done with the last segment's planes
#pragma unroll
    for (int i = 0; i < AHEAD; ++i) {
      if (i < nin) cp.stage(in, g, ring + i * STAGE);
      cp_async_commit();
    }
    cp_async_wait_group<AHEAD - 2>();  // input planes 0 and 1
    __syncthreads();
    u.first(ring + oi, ring + STAGE + oi, t);
    int sn = AHEAD % NS, s0 = 0, s1 = 1, s2 = 2;  // ring slots of input planes j + AHEAD, j ..
    auto plane = [&](auto phase, int j) {
      constexpr int P = decltype(phase)::value;
      cp_async_wait_group<AHEAD - 3>();  // input plane j + 2 has landed
      __syncthreads();                   // ... for every thread, and slot sn is free
      if (j + AHEAD < nin) cp.stage(in, g, ring + sn * STAGE);
      cp_async_commit();  // possibly empty: one group per iteration
      float4 res[NF];
      u.template step<P>(ring + s0 * STAGE + oi, ring + s1 * STAGE + oi, ring + s2 * STAGE + oi, t,
                         arg, res);
      sn = U::LIVE == 3 ? s0 : s1;
      s0 = s1;
      s1 = s2;
      if (++s2 == NS) s2 = 0;
      if (store) store_group<NF, RAGGED>(out, off, res, gx, x1);
      off += off_step;
    };
    for (int j = 0; j < n; j += U::PHASES) {
      plane(std::integral_constant<int, 0>(), j);
      if constexpr (U::PHASES == 1) continue;
      if (j + 1 >= n) break;
      plane(std::integral_constant<int, 1>(), j + 1);
      if (j + 2 >= n) break;
      plane(std::integral_constant<int, 2>(), j + 2);
    }
    cp_async_wait_all();  // (the last groups are empty)
  }
}

template <class U, int RAGGED>
cudaError_t launch_one_(pf_grid_s* gr, FieldPtrs in, FieldOut out, const typename U::A& arg,
                       cudaStream_t st) {
  constexpr size_t smem = sizeof(float) * U::NS * U::NF * U::IN_FIELD;
  auto kern = fe3d_one_kernel<U, RAGGED>;
  static unsigned long long attr_mask = 0;  // per instantiation and device
  cudaError_t e = ensure_smem_attr(kern, smem, &attr_mask);
  if (e != cudaSuccess) return e;
  const StreamTiles& p = gr->one.tiles;
  const int nt = (std::max(p.TY, 2) * p.G + 31) / 32 * 32;
  return launch_chained(kern, gr->one.grid, nt, smem, st, in, out, grid_geom(gr), arg, p,
                        gr->one.sched);
}

template <class U>
cudaError_t launch_one(pf_grid_s* gr, FieldPtrs in, FieldOut out, const typename U::A& arg,
                       cudaStream_t st) {
  if (gr->one_key != U::NT) {  // the plan depends on the sides and the threads
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, gr->device);
    if (e != cudaSuccess) return e;
    gr->one = stream_plan(grid_geom(gr), (long long)sms * U::CTAS, U::NT, kOneMaxGroups, 1, 0,
                          kOnePlaneWarps);
    gr->one_key = U::NT;
  }
  const StreamTiles& p = gr->one.tiles;
  switch (copy_form(grid_geom(gr), p, U::NF, 1, std::max(p.TY, 2) * p.G)) {
    case 0: return launch_one_<U, 0>(gr, in, out, arg, st);
    case 1: return launch_one_<U, 1>(gr, in, out, arg, st);
  }
  return launch_one_<U, 2>(gr, in, out, arg, st);
}

template <int MODEL>
cudaError_t launch_stencil(pf_grid_s* gr, FieldPtrs in, FieldOut out, cudaStream_t st) {
  switch (gr->stencil) {
    case PF_ST_STD: return launch_one<Std7<MODEL>>(gr, in, out, gr->params, st);
    case PF_ST_ISO: return launch_one<Iso<MODEL, PF_ST_ISO>>(gr, in, out, gr->params, st);
    case PF_ST_ISO27: return launch_one<Iso<MODEL, PF_ST_ISO27>>(gr, in, out, gr->params, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_fe3d_one(pf_grid_s* gr, int src, int dst, cudaStream_t st) {
  FieldPtrs in{};
  FieldOut out{};
  for (int f = 0; f < gr->nf; ++f) {
    in.f[f] = gr->buf[src][f];
    out.f[f] = gr->buf[dst][f];
  }
  if (gr->model == PF_MODEL_AC) return launch_stencil<PF_MODEL_AC>(gr, in, out, st);
  if (gr->model == PF_MODEL_GS) return launch_stencil<PF_MODEL_GS>(gr, in, out, st);
  if (gr->model != PF_MODEL_RD) return cudaErrorInvalidValue;
  switch (gr->nf) {
    case 1: return launch_one<Species<1>>(gr, in, out, gr->rd, st);
    case 2: return launch_one<Species<2>>(gr, in, out, gr->rd, st);
    case 3: return launch_one<Species<3>>(gr, in, out, gr->rd, st);
    case 4: return launch_one<Species<4>>(gr, in, out, gr->rd, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace pf
