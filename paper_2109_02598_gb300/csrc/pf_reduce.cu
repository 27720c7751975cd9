// Deterministic reductions of a field: mass h^d sum(phi) and the discrete free energy
//   E = h^d sum_x [ 1/2 sum_i ((phi_{x+e_i} - phi_x)/h)^2 - c1/2 phi^2 + c2/4 phi^4 ],
// the energy whose discrete gradient flow is Model A (Sec. 3) with forward differences on
// the periodic grid, and Model C's (two fields). The result depends only on the grid's shape
// and its values, not on timing: each thread's sites and every order of addition are fixed.
//
// Arithmetic. This GPU's FP64 pipe does two operations per clock and SM against 128 in FP32,
// so an FP64 sum of an FP32 field is bound by it (two operations and conversions per site for
// the mass, twenty for the 3D energy). The sums run in FP32 without its rounding instead:
//   * differences, squares and fourth powers as unevaluated sums of three words (the error-free
//     sum and product of Knuth and Dekker; fma for the product's error), good to 2^-70 a site,
//     below FP64's 2^-53 site by site (with the third word left out, 2^-47: not made up for
//     where an energy lies in a few sites of a flat field);
//   * added into three-word accumulators by cascaded error-free sums, whose error, about
//     2^-72 of the sum, is below FP64's;
//   * on packed pairs of sites (add.rn.f32x2 and so on), one thread's words becoming one
//     double at its end. Threads' doubles are summed in FP64 (warp shuffles, shared memory,
//     one CTA over the CTAs' partials).
// The pairs need room: a group of sites whose largest value is outside [2^-20, 2^20] (2^100
// for the mass) and not zero is summed in FP64 as before, infinities with it; a NaN
// stays one either way.
//
// Work: a chunk is kRows consecutive rows of a group of four columns, one per thread (rows of
// fewer than 32 groups share a warp), so a row's y-neighbour is the chunk's next row and a
// chunk's loads are issued together; chunks are dealt round-robin over a fixed grid of two or
// three CTAs per SM. Small grids run in one CTA, which writes the result itself.
//
// Bound by issue (energies) and by latency at the CTAs' registers. A call with its
// synchronisation, before (FP64 sums; 64 of 256 threads busy on 256-wide rows; the result and
// the error word by two copies) -> now: mass 256^3 115 -> 35 us, 2048^2 43 -> 27, 128^2 29 -> 17;
// energy 256^3 659 -> 119 us, 2048^2 155 -> 38, 128^2 29 -> 18; Model C 128^3 361 -> 50 (the third
// words of squares and products are 10 to 16 % of these: 103, 34 and 46 without). Errors
// against 128-bit sums over 20 shapes and seven kinds of values (noise, smooth, 1e-9 to 3e6,
// mixed magnitudes) stay those of the FP64 sums: 4e-18 to 2e-17 on average for the mass, 5e-17
// to 1.4e-16 for the energies.
#include <algorithm>

#include "pf_internal.h"

namespace pf {

namespace {

constexpr int kNTR = 256;        // threads of a CTA of the two-kernel form
constexpr int kOneCta = 512;     // threads of the one-CTA form
constexpr int kNTS = 64;         // threads of a CTA of the FP64 form

// Energies of fewer sites are summed in FP64: many small CTAs of short FP64 work finish before the
// few that the words' sums would fill (a call on 128^2: 18 us against 29, Model C 21 against 49;
// from 40^3 on the times are the same).
constexpr int64_t kFp64Sites = 1 << 16;

constexpr int kMass = 0, kEnergy = 1, kEnergyC = 2;
template <int WHAT, bool FP64 = false>
struct RedTraits {
  static constexpr int kRows = FP64 ? 1 : WHAT == kMass ? 8 : WHAT == kEnergy ? 4 : 2;
  // CTAs of the two-kernel form: what 152 SMs hold at once (84 and 124-128 registers)
  static constexpr int kGrid = WHAT == kMass ? 3 * 152 : 2 * 152;
  static_assert(kGrid <= kReduceBlocks, "one partial per CTA");
};

struct RedArgs {
  const float* f[2];
  double c1, c2, c3, c4, c5, inv_h2, scale;
  double* partials;  // two-kernel form
  double* out;       // the result (device or mapped host)
  const int* err;    // device error word to pass on with the result, or nullptr
  int* err_out;
  int lw;            // log2 of the threads per row piece
  int segs;          // pieces per row
  int nyb;           // row blocks per plane
  int64_t chunks;    // segs * nyb * nz
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Sum of a value over the CTA (a multiple of 32 threads, at most 512); valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double t = 0.0;
  if (wid == 0) {
    t = (lane < (int)blockDim.x / 32) ? red[lane] : 0.0;
    t = warp_sum(t);
  }
  return t;
}

__device__ __forceinline__ void finish(const RedArgs& a, double t) {
  *a.out = t * a.scale;
  if (a.err != nullptr) *a.err_out = *a.err;
}

// ---- error-free arithmetic on two sites at once
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
// s + e = a + b exactly
__device__ __forceinline__ float2 two_sum(float2 a, float2 b, float2& e) {
  const float2 s = add2(a, b);
  const float2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
  return s;
}
// h + l = a b exactly.
__device__ __forceinline__ float2 product2(float2 a, float2 b, float2& l) {
  const float2 h = __fmul2_rn(a, b);
  l = __ffma2_rn(a, b, neg2(h));
  return h;
}
__device__ __forceinline__ float2 square2(float2 a, float2& l) { return product2(a, a, l); }
// h + l + r = (ah + al) b to 2^-72 for a pair (ah, al): al b meets the rounding of ah b in l, and
// what both leave goes to r, which callers add to an accumulator's last word.
__device__ __forceinline__ float2 product2(float2 ah, float2 al, float2 b, float2& l, float2& r) {
  float2 e, pe;
  const float2 h = product2(ah, b, l);
  const float2 p = product2(al, b, pe);
  l = two_sum(l, p, e);
  r = add2(e, pe);
  return h;
}
// h + l + r = (ah + al)^2 to 2^-72.
__device__ __forceinline__ float2 square2(float2 ah, float2 al, float2& l, float2& r) {
  float2 e, pe;
  const float2 h = square2(ah, l);
  const float2 p = product2(add2(ah, ah), al, pe);
  l = two_sum(l, p, e);
  r = __ffma2_rn(al, al, add2(e, pe));
  return h;
}

struct Sum3 {  // a0 + a1 + a2, one sum per half of the pair
  float2 a0 = {0.f, 0.f}, a1 = {0.f, 0.f}, a2 = {0.f, 0.f};
  __device__ __forceinline__ void add_low(float2 x) {  // below a0's last place
    float2 e;
    a1 = two_sum(a1, x, e);
    a2 = add2(a2, e);
  }
  __device__ __forceinline__ void add(float2 x) {
    float2 e;
    a0 = two_sum(a0, x, e);
    add_low(e);
  }
  __device__ __forceinline__ void add(float2 h, float2 l) {
    add(h);
    add_low(l);
  }
  __device__ __forceinline__ void add(float2 h, float2 l, float2 l2) {
    add(h, l);
    a2 = add2(a2, l2);
  }
  __device__ __forceinline__ double value() const {
    return (((double)a2.x + (double)a2.y) + ((double)a1.x + (double)a1.y)) +
           ((double)a0.x + (double)a0.y);
  }
};

__device__ __forceinline__ float at4(const float4& v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}
__device__ __forceinline__ float max4(const float4& v) {
  return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
}

// Four columns from x of a row of nx: one 16-byte load where they all lie in it and the rows
// are 16-byte aligned, else element by element, zero past the end.
template <bool VEC>
__device__ __forceinline__ float4 load4(const float* row, int x, int nx) {
  if (VEC && x + 3 < nx) return *reinterpret_cast<const float4*>(row + x);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (x < nx) v.x = row[x];
  if (x + 1 < nx) v.y = row[x + 1];
  if (x + 2 < nx) v.z = row[x + 2];
  if (x + 3 < nx) v.w = row[x + 3];
  return v;
}

// A chunk of one field: R + 1 rows of four columns, the x-neighbour right of each row and, in
// 3D, the rows of the next plane.
template <int R>
struct Rows {
  float4 v[R + 1], z[R];
  float after[R];
};

template <int R, bool VEC>
__device__ __forceinline__ void load_rows(const float* f, const Geom& g, int x, int y0, int zi,
                                          int nr, bool active, int lw, Rows<R>& c) {
  const float* pl = f + (int64_t)zi * g.plane;
  const float* pn = f + (int64_t)(zi + 1 == g.nz ? 0 : zi + 1) * g.plane;
  const bool in = active && x < g.nx;
#pragma unroll
  for (int r = 0; r <= R; ++r) {
    c.v[r] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int y = y0 + r < g.ny ? y0 + r : y0 + r - g.ny;
    if (in && r <= nr) c.v[r] = load4<VEC>(pl + (int64_t)y * g.pitch, x, g.nx);
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    c.z[r] = c.v[r];
    if (g.dim == 3 && in && r < nr) c.z[r] = load4<VEC>(pn + (int64_t)(y0 + r) * g.pitch, x, g.nx);
  }
  // right of the group: the next lane's first value, the row's next value at a piece's end,
  // the row's first value at the row's end (there it follows the last valid column)
  const int n = g.nx - x;  // valid columns
  const bool end = (threadIdx.x & ((1 << lw) - 1)) == (1 << lw) - 1;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    c.after[r] = __shfl_down_sync(0xffffffffu, c.v[r].x, 1);
    if (in && r < nr && (n <= 4 || end)) {
      const float e = pl[(int64_t)(y0 + r) * g.pitch + (n <= 4 ? 0 : x + 4)];
      if (n >= 4) c.after[r] = e;
      if (n == 1) c.v[r].y = e;
      if (n == 2) c.v[r].z = e;
      if (n == 3) c.v[r].w = e;
    }
  }
}

template <int R>
__device__ __forceinline__ float rows_max(const Rows<R>& c) {
  float m = 0.f;
#pragma unroll
  for (int r = 0; r <= R; ++r) m = fmaxf(m, max4(c.v[r]));
#pragma unroll
  for (int r = 0; r < R; ++r) m = fmaxf(m, fmaxf(max4(c.z[r]), fabsf(c.after[r])));
  return m;
}

// |grad|^2 h^2 of two sites (columns 2 q, 2 q + 1 of row r) as hi + lo + lo2, from the differences
// to the right, the next row and (3D) the next plane
template <int R>
__device__ __forceinline__ float2 grad2(const Rows<R>& c, int r, int q, bool three, float2& lo,
                                        float2& lo2) {
  const float4 &v = c.v[r], &y = c.v[r + 1], &z = c.z[r];
  const float2 p = q == 0 ? make_float2(v.x, v.y) : make_float2(v.z, v.w);
  const float2 px = q == 0 ? make_float2(v.y, v.z) : make_float2(v.w, c.after[r]);
  const float2 py = q == 0 ? make_float2(y.x, y.y) : make_float2(y.z, y.w);
  float2 dl, l, l2, e, r1, r2;
  float2 d = two_sum(px, neg2(p), dl);
  float2 s = square2(d, dl, lo, lo2);
  auto more = [&](const float2& pn) {
    d = two_sum(pn, neg2(p), dl);
    s = two_sum(s, square2(d, dl, l, l2), e);
    lo = two_sum(lo, l, r1);
    lo = two_sum(lo, e, r2);
    lo2 = add2(add2(lo2, l2), add2(r1, r2));
  };
  more(py);
  if (three) more(q == 0 ? make_float2(z.x, z.y) : make_float2(z.z, z.w));
  return s;
}

// Zero the halves of a pair past the row's last column (n valid columns from 2 q on).
__device__ __forceinline__ void mask2(float2& v, int n) {
  if (n < 2) v.y = 0.f;
  if (n < 1) v.x = 0.f;
}

__device__ __forceinline__ double energy_site(double p, double dx, double dy, double dz, int dim,
                                              double c1, double c2, double inv_h2) {
  double g2 = dx * dx + dy * dy;
  if (dim == 3) g2 += dz * dz;
  const double p2 = p * p;
  return 0.5 * g2 * inv_h2 - 0.5 * c1 * p2 + 0.25 * c2 * p2 * p2;
}

// FP64: an energy's chunks (one row of four columns each) all in FP64, for small grids.
template <int WHAT, bool VEC, bool FP64>
__global__ void __launch_bounds__(FP64 ? kNTS : kOneCta) reduce_kernel(const RedArgs a,
                                                                       const Geom g) {
  constexpr int R = RedTraits<WHAT, FP64>::kRows;
  __shared__ double red[kOneCta / 32];
  Sum3 sg, s2, s4, t2, t4, sx;  // |grad|^2 (both fields), psi^2, psi^4, m^2, m^4, psi^2 m
  double acc = 0.0;             // chunks summed in FP64
  // this thread's chunk (seg, yb, z), advanced by the grid's stride with carries
  const int lane_w = threadIdx.x & ((1 << a.lw) - 1);
  const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> a.lw;
  int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> a.lw;
  int seg = (int)(u % a.segs), yb, z, dseg, dyb, dz;
  {
    const int64_t t = u / a.segs, dt = stride / a.segs;
    yb = (int)(t % a.nyb);
    z = (int)(t / a.nyb);
    dseg = (int)(stride % a.segs);
    dyb = (int)(dt % a.nyb);
    dz = (int)(dt / a.nyb);
  }
  const bool three = g.dim == 3;
  // whole warps stay in the loop (shuffles): bounded by the warp's first chunk
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) >> a.lw; w < a.chunks;
       w += stride) {
    const bool active = u < a.chunks;
    const int x = 4 * ((seg << a.lw) + lane_w);
    const int y0 = yb * R;
    const int nr = min(R, g.ny - y0);
    if constexpr (WHAT == kMass) {
      float4 v[R];
      const float* pl = a.f[0] + (int64_t)z * g.plane;
      float m = 0.f;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        v[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (active && r < nr) v[r] = load4<VEC>(pl + (int64_t)(y0 + r) * g.pitch, x, g.nx);
      }
#pragma unroll
      for (int r = 0; r < R; ++r) m = fmaxf(m, max4(v[r]));
      if (m < 0x1p100f) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          sg.add(make_float2(v[r].x, v[r].y));
          s2.add(make_float2(v[r].z, v[r].w));
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r)
          acc += ((double)v[r].x + (double)v[r].y) + ((double)v[r].z + (double)v[r].w);
      }
    } else {
      Rows<R> p, q;
      load_rows<R, VEC>(a.f[0], g, x, y0, z, nr, active, a.lw, p);
      float m = rows_max(p);
      bool tiny = FP64 || (m < 0x1p-20f && m > 0.f);
      if constexpr (WHAT == kEnergyC) {
        load_rows<R, VEC>(a.f[1], g, x, y0, z, nr, active, a.lw, q);
        const float mq = rows_max(q);
        tiny = tiny || (mq < 0x1p-20f && mq > 0.f);
        m = fmaxf(m, mq);
      }
      const int n = active ? g.nx - x : 0;  // valid columns (4 or more: all)
      if (!FP64 && n > 0 && m < 0x1p20f && !tiny) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (r >= nr) break;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            float2 lo, lo2, l2, l4, r4;
            float2 hi = grad2(p, r, i, three, lo, lo2);
            float2 pv = i == 0 ? make_float2(p.v[r].x, p.v[r].y) : make_float2(p.v[r].z, p.v[r].w);
            if (n < 4) {
              mask2(hi, n - 2 * i);
              mask2(lo, n - 2 * i);
              mask2(lo2, n - 2 * i);
              mask2(pv, n - 2 * i);
            }
            sg.add(hi, lo, lo2);
            const float2 p2 = square2(pv, l2);
            s2.add(p2, l2);
            const float2 p4 = square2(p2, l2, l4, r4);
            s4.add(p4, l4, r4);
            if constexpr (WHAT == kEnergyC) {
              hi = grad2(q, r, i, three, lo, lo2);
              float2 qv = i == 0 ? make_float2(q.v[r].x, q.v[r].y) : make_float2(q.v[r].z, q.v[r].w);
              if (n < 4) {
                mask2(hi, n - 2 * i);
                mask2(lo, n - 2 * i);
                mask2(lo2, n - 2 * i);
                mask2(qv, n - 2 * i);
              }
              sg.add(hi, lo, lo2);
              float2 m2, m4;
              const float2 q2 = square2(qv, m2);
              t2.add(q2, m2);
              const float2 q4 = square2(q2, m2, m4, r4);
              t4.add(q4, m4, r4);
              float2 xl;  // psi^2 m
              const float2 x2 = product2(p2, l2, qv, xl, r4);
              sx.add(x2, xl, r4);
            }
          }
        }
      } else if (n > 0) {
        for (int r = 0; r < nr; ++r) {
          // (dynamic indices: this path is for values outside the pairs' range)
          float4 v = p.v[0], y = p.v[1], zz = p.z[0], v2{}, y2{}, z2{};
          float af = p.after[0], af2 = 0.f;
          if constexpr (WHAT == kEnergyC) {
            v2 = q.v[0];
            y2 = q.v[1];
            z2 = q.z[0];
            af2 = q.after[0];
          }
#pragma unroll
          for (int k = 1; k < R; ++k)
            if (r == k) {
              v = p.v[k];
              y = p.v[k + 1];
              zz = p.z[k];
              af = p.after[k];
              if constexpr (WHAT == kEnergyC) {
                v2 = q.v[k];
                y2 = q.v[k + 1];
                z2 = q.z[k];
                af2 = q.after[k];
              }
            }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (i >= n) break;
            const double pv = at4(v, i), xn = i == 3 ? af : at4(v, i + 1);
            acc += energy_site(pv, xn - pv, (double)at4(y, i) - pv, (double)at4(zz, i) - pv, g.dim,
                               a.c1, a.c2, a.inv_h2);
            if constexpr (WHAT == kEnergyC) {
              const double qv = at4(v2, i), qn = i == 3 ? af2 : at4(v2, i + 1);
              acc += energy_site(qv, qn - qv, (double)at4(y2, i) - qv, (double)at4(z2, i) - qv,
                                 g.dim, a.c3, a.c4, a.inv_h2) -
                     a.c5 * pv * pv * qv;
            }
          }
        }
      }
    }
    u += stride;
    seg += dseg;
    yb += dyb;
    z += dz;
    if (seg >= a.segs) {
      seg -= a.segs;
      ++yb;
    }
    if (yb >= a.nyb) {
      yb -= a.nyb;
      ++z;
    }
  }
  double v;
  if constexpr (WHAT == kMass)
    v = acc + (sg.value() + s2.value());
  else
    v = acc + (0.5 * a.inv_h2 * sg.value() - 0.5 * a.c1 * s2.value() + 0.25 * a.c2 * s4.value());
  if constexpr (WHAT == kEnergyC)
    v += -0.5 * a.c3 * t2.value() + 0.25 * a.c4 * t4.value() - a.c5 * sx.value();
  const double t = block_sum(v, red);
  if (threadIdx.x == 0) {
    if (gridDim.x == 1)
      finish(a, t);
    else
      a.partials[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(kReduceBlocks) reduce_final_kernel(const RedArgs a, int n) {
  __shared__ double red[kReduceBlocks / 32];
  const double t = block_sum((int)threadIdx.x < n ? a.partials[threadIdx.x] : 0.0, red);
  if (threadIdx.x == 0) finish(a, t);
}

template <int WHAT, bool FP64>
cudaError_t launch_form(RedArgs a, const Geom& g, cudaStream_t s) {
  using T = RedTraits<WHAT, FP64>;
  const int ng = (g.nx + 3) / 4;  // groups per row
  a.lw = 0;
  while (a.lw < 5 && (1 << a.lw) < ng) ++a.lw;
  a.segs = (ng + (1 << a.lw) - 1) >> a.lw;
  a.nyb = (g.ny + T::kRows - 1) / T::kRows;
  a.chunks = (int64_t)a.segs * a.nyb * g.nz;
  const bool vec = g.pitch % 4 == 0 && g.plane % 4 == 0 && ((uintptr_t)a.f[0] & 15) == 0 &&
                   ((uintptr_t)a.f[1] & 15) == 0;
  const int64_t threads = a.chunks << a.lw;
  // up to four chunks per thread of one CTA: one launch instead of two (FP64: small CTAs
  // instead, so that the work meets as many SMs' FP64 pipes as there are)
  int blocks = 1, nt = FP64 ? kNTS : kOneCta;
  if (FP64 || threads > 4 * kOneCta) {
    nt = FP64 ? kNTS : kNTR;
    blocks = (int)std::min<int64_t>((threads + nt - 1) / nt, T::kGrid);
  }
  if (vec)
    reduce_kernel<WHAT, true, FP64><<<blocks, nt, 0, s>>>(a, g);
  else
    reduce_kernel<WHAT, false, FP64><<<blocks, nt, 0, s>>>(a, g);
  if (blocks > 1) reduce_final_kernel<<<1, kReduceBlocks, 0, s>>>(a, blocks);
  return cudaGetLastError();
}

template <int WHAT>
cudaError_t launch(const RedArgs& a, const Geom& g, cudaStream_t s) {
  if constexpr (WHAT != kMass)
    if ((int64_t)g.nx * g.ny * g.nz < kFp64Sites) return launch_form<WHAT, true>(a, g, s);
  return launch_form<WHAT, false>(a, g, s);
}

}  // namespace

// Loads every kernel launch_reduce can choose (under lazy loading a kernel's first launch loads
// it, which may allocate and synchronise, and is not allowed while a stream is captured).
cudaError_t reduce_load_kernels() {
  const void* kernels[] = {reinterpret_cast<const void*>(reduce_kernel<kMass, true, false>),
                           reinterpret_cast<const void*>(reduce_kernel<kMass, false, false>),
                           reinterpret_cast<const void*>(reduce_kernel<kEnergy, true, false>),
                           reinterpret_cast<const void*>(reduce_kernel<kEnergy, false, false>),
                           reinterpret_cast<const void*>(reduce_kernel<kEnergy, true, true>),
                           reinterpret_cast<const void*>(reduce_kernel<kEnergy, false, true>),
                           reinterpret_cast<const void*>(reduce_final_kernel)};
  for (const void* k : kernels) {
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, k);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_reduce(int what, const Geom& g, const float* field, double c1, double c2,
                          double h, double* d_partials, double* d_out, cudaStream_t s,
                          const int* d_err, int* err_out) {
  RedArgs a{};
  a.f[0] = field;
  a.c1 = c1;
  a.c2 = c2;
  a.inv_h2 = 1.0 / (h * h);
  a.scale = g.dim == 3 ? h * h * h : h * h;
  a.partials = d_partials;
  a.out = d_out;
  a.err = d_err;
  a.err_out = err_out;
  return what == PF_REDUCE_MASS ? launch<kMass>(a, g, s) : launch<kEnergy>(a, g, s);
}

cudaError_t launch_reduce_energy_c(const Geom& g, const float* psi, const float* m,
                                   const double* c, double h, double* d_partials,
                                   double* d_out, cudaStream_t s, const int* d_err,
                                   int* err_out) {
  RedArgs a{};
  a.f[0] = psi;
  a.f[1] = m;
  a.c1 = c[0];
  a.c2 = c[1];
  a.c3 = c[2];
  a.c4 = c[3];
  a.c5 = c[4];
  a.inv_h2 = 1.0 / (h * h);
  a.scale = g.dim == 3 ? h * h * h : h * h;
  a.partials = d_partials;
  a.out = d_out;
  a.err = d_err;
  a.err_out = err_out;
  return launch<kEnergyC>(a, g, s);
}

}  // namespace pf
