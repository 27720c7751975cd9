// Discrete adjoint of the forward-Euler Gray-Scott time loop with sqrt(N) checkpointing.
//
// Forward map (Sec. 2.4.1 solver; Gray-Scott in its standard form, Sec. 1):
//   x^{n+1} = x^n + dt f(x^n; theta),  theta = (Du, Dv, F, k).
// For a loss L(x^N) with lambda^N = dL/dx^N, reverse-mode differentiation of the loop gives
//   lambda^n = lambda^{n+1} + dt J(x^n)^T lambda^{n+1},
//   dL/dtheta = sum_n dt (df/dtheta)(x^n)^T lambda^{n+1},   dL/dx^0 = lambda^0.
// With (u, v) = x^n and (a, b) = lambda^{n+1}, and the periodic Laplacian symmetric:
//   a' = a + dt [Du lap a - (v^2 + F) a + v^2 b]
//   b' = b + dt [Dv lap b - 2uv a + (2uv - F - k) b]
//   dL/dDu += dt sum a lap u,  dL/dDv += dt sum b lap v,
//   dL/dF  += dt sum [(1 - u) a - v b],  dL/dk += -dt sum v b.
//
// Model A (x' = x + dt (lap x + c1 x - c2 x^3)) and Model B (x' = x + dt M lap mu(x),
// mu = c2 x^3 - c1 x - lap x) take the same loop with their own reverse steps:
//   A: lambda^n = lambda + dt [lap lambda + (c1 - 3 c2 x^2) lambda];
//      sums S = (sum lambda x, sum lambda x^3), dL/d(c1, c2) = dt (S0, -S1).
//   B: w = lap lambda, lambda^n = lambda + dt M [(3 c2 x^2 - c1) w - lap w];
//      sums S = (sum w x, sum w x^3, sum w mu), dL/d(c1, c2, M) = dt (-M S0, M S1, S2).
//
// Memory/recompute: the forward pass stores x at every C-th step; the backward pass walks the
// segments from last to first and goes back through each in blocks of up to four steps (two for
// Model B) a launch, from the state at the block's first step; the states inside a block are
// recomputed on chip. The blocks' first states are stored where the library chooses C and they
// fit, else the segment's are recomputed from its checkpoint with the forward kernel
// (C ~ sqrt(N)). Parameter-gradient partials are summed per CTA in FP64 (each CTA owns one slot,
// so the order is fixed and the result deterministic) and added up in a fixed order at the end.
#include <atomic>
#include <cmath>

#include "pf_fe2d_tile.cuh"
#include "pf_grid.h"
#include "pf_internal.h"

namespace pf {

namespace {

// The forward pass keeps every block's first state where they fit, with those that the device's
// other handles keep this way, kAllStates bytes, and one part in kFreeParts of the memory that is
// free: a program may hold many handles (an autograd node is one each), and its other allocations
// do not wait for ours.
constexpr int64_t kAllStates = (int64_t)4 << 30;
constexpr int kFreeParts = 16;

constexpr int kATX = 64, kATY = 16;  // adjoint tile

// Warp sum of per-thread float partials, in float (a fixed tree, so the same bits on every
// run); the per-warp sums are added in double. FP64 arithmetic and conversions are a small
// fraction of FP32 throughput on this GPU: a double-precision shuffle tree in every CTA of
// every reverse step took most of the kernel's time.
__device__ __forceinline__ float warp_sum_f(float f) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) f = __fadd_rn(f, __shfl_down_sync(0xffffffffu, f, o));
  return f;
}

// Double-precision warp sum, for the final fixed-order sum over the CTAs' slots (once per
// reverse pass).
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// LEN reverse steps of Gray-Scott on a 64 x 16 tile in one launch, from the state x^s at the
// block's first step and lambda^{s+LEN}: both are staged with their halos (2 (LEN - 1) and LEN
// sites), the states x^{s+1} .. x^{s+LEN-1} are recomputed in shared memory on regions that
// shrink by a site a step (the forward step's functions, so its bits), and lambda goes back
// through them on regions of the tile plus j sites, j = LEN - 1 .. 0. So of the states only every
// LEN-th goes through memory, and a launch and its round trips through L2 are paid once per LEN
// steps. Groups past the grid's edge are computed as what they are, periodic images.
//
// The parameter-gradient terms are summed over the tile as a reverse step of its own would: per
// thread over its group of four sites, per warp (two rows of the tile) by a fixed tree, both in
// float, then in FP64 over the warps, and step after step into the CTA's slot, so the sums do not
// depend on how the steps are cut into blocks.
//
// Bound by the latency of its chain (staging, LEN - 1 forward and LEN reverse stages, each behind
// a barrier: about 8 us for four steps on a 64^2 grid, 12 at 512^2) and by shared memory on large
// grids. The reverse pass of 400 steps, against one launch per step with the states recomputed on
// a second stream: 512^2 2.09 -> 1.15 ms, 128^2 1.27 -> 0.75, 1024^2 4.7 -> 3.4, 2048^2 14.4 ->
// 12.3. 64 x 32 tiles (less halo, one CTA per SM): the same at 512^2, 20 to 45 % slower on smaller
// and larger grids.
template <int LEN>
struct AdjBlock {
  static constexpr int TY = kATY;
  static constexpr int TILE = 16 * TY;                           // groups of the tile
  static constexpr int H = LEN > 1 ? 2 * (LEN - 1) : 1;          // staged halo rows of the state
  static constexpr int HP = (H + 3) / 4 * 4;                     // and columns
  static constexpr int WS = kATX + 2 * HP, ROWS = TY + 2 * H;
  static constexpr int PL = WS * ROWS;                           // floats of a field
  static constexpr int SMEM_FLOATS = (2 * LEN + 4) * PL;         // the states, lambda twice
  // Threads: every region in one pass where 1024 do it: the first recomputed state, and the tile
  // with its widest ring (a group each)
  static constexpr int FIRST = LEN > 1 ? (TY + 2 * (H - 1)) * (kATX / 4 + 2 * ((H + 2) / 4)) : 0;
  static constexpr int RING = LEN > 1 ? 2 * (LEN - 1) * (kATX / 4 + 2) + 2 * TY : 0;
  static constexpr int WANT = FIRST > TILE + RING ? FIRST : TILE + RING;
  static constexpr int NT = WANT > 1024 ? 1024 : (WANT + 31) / 32 * 32;
  static_assert(NT >= TILE && (LEN == 1 || NT > TILE), "threads beside the tile's for its ring");
  static_assert(H >= LEN && HP >= 4, "lambda's halo fits the states' geometry");
  // offset of the group of tile row r, group q (four columns from 4 q)
  static __device__ __forceinline__ int at(int r, int q) { return (r + H) * WS + HP + 4 * q; }
};

template <int LEN>
__global__ void __launch_bounds__(AdjBlock<LEN>::NT)
    adj_gs2d_kernel(FieldPtrs x, FieldPtrs lam, FieldOut lam_out, Geom g, ModelParams m,
                    double* gpart) {
  using B = AdjBlock<LEN>;
  constexpr int TY = B::TY, WS = B::WS, PL = B::PL, NT = B::NT, H = B::H;
  extern __shared__ __align__(16) float sm[];  // state j: u at 2 j PL, v behind it
  constexpr int TILE = B::TILE, NW = TILE / 32;  // warps of the tile
  __shared__ float red[LEN][4][NW];
  __shared__ double step_sum[LEN][4];
  float* la = sm + 2 * LEN * PL;  // lambda: a, b; then the other buffer
  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * kATX, y0 = blockIdx.y * TY;
  canary_fill(sm, B::SMEM_FLOATS);
  chain_wait();
  // rows y0 - h .. y0 + TY + h - 1, columns x0 - hp .. x0 + 63 + hp of two fields
  auto stage = [&](const FieldPtrs& in, int h, int hp, float* dst) {
    const int gpr = (kATX + 2 * hp) / 4;
    for (int i = tid; i < (TY + 2 * h) * gpr; i += NT) {
      const int r = i / gpr, q = i - r * gpr - hp / 4;
      const int64_t row = (int64_t)wrap_index(y0 - h + r, g.ny) * g.pitch;
      const int gx = wrap_index(x0 + 4 * q, g.nx);
      float* d = dst + B::at(r - h, q);
      if (gx + 3 < g.nx && gx % 4 == 0) {
        cp_async16(d, in.f[0] + row + gx);
        cp_async16(d + PL, in.f[1] + row + gx);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int64_t o = row + wrap_index(gx + c, g.nx);
          cp_async4(d + c, in.f[0] + o);
          cp_async4(d + PL + c, in.f[1] + o);
        }
      }
    }
  };
  stage(x, H, B::HP, sm);
  stage(lam, LEN, 4, la);
  cp_async_wait_all();
  __syncthreads();
  // the block's states: x^{j+1} on the tile plus H - 1 - j sites
#pragma unroll
  for (int j = 0; j + 1 < LEN; ++j) {
    const float* s = sm + 2 * j * PL;
    float* d = sm + 2 * (j + 1) * PL;
    const int h = H - 1 - j;
    const int q0 = -((h + 3) / 4), gpr = kATX / 4 - 2 * q0;
    for (int i = tid; i < (TY + 2 * h) * gpr; i += NT) {
      const int r = i / gpr;
      const int p = B::at(r - h, i - r * gpr + q0);
      const float4 u = *reinterpret_cast<const float4*>(s + p);
      const float4 v = *reinterpret_cast<const float4*>(s + PL + p);
      const float4 lu = lap2d_x4<PF_ST_STD, PF_MODEL_GS>(s, p, WS, 1.0f);
      const float4 lv = lap2d_x4<PF_ST_STD, PF_MODEL_GS>(s + PL, p, WS, 1.0f);
      float4 un, vn;
      gs_update(u.x, v.x, lu.x, lv.x, m, un.x, vn.x);
      gs_update(u.y, v.y, lu.y, lv.y, m, un.y, vn.y);
      gs_update(u.z, v.z, lu.z, lv.z, m, un.z, vn.z);
      gs_update(u.w, v.w, lu.w, lv.w, m, un.w, vn.w);
      *reinterpret_cast<float4*>(d + p) = un;
      *reinterpret_cast<float4*>(d + PL + p) = vn;
    }
    __syncthreads();
  }
  // lambda back through them
  const int rr = tid / 16, jj = tid % 16;  // the thread's group of the tile
  const int gy = y0 + rr, gx = x0 + 4 * jj;
  const int nvalid = gy < g.ny ? (g.nx - gx < 4 ? (g.nx > gx ? g.nx - gx : 0) : 4) : 0;
#pragma unroll
  for (int j = LEN - 1; j >= 0; --j) {
    const float* s = sm + 2 * j * PL;
    const float* l = la + 2 * ((LEN - 1 - j) & 1) * PL;
    float* d = la + 2 * ((LEN - j) & 1) * PL;
    // lambda^{s+j} of the four sites at p
    auto back = [&](int p, float4& na, float4& nb) {
      const float4 u4 = *reinterpret_cast<const float4*>(s + p);
      const float4 v4 = *reinterpret_cast<const float4*>(s + PL + p);
      const float4 a4 = *reinterpret_cast<const float4*>(l + p);
      const float4 b4 = *reinterpret_cast<const float4*>(l + PL + p);
      const float4 la4 = lap2d_x4<PF_ST_STD, PF_MODEL_GS>(l, p, WS, 1.0f);
      const float4 lb4 = lap2d_x4<PF_ST_STD, PF_MODEL_GS>(l + PL, p, WS, 1.0f);
      auto site = [&](float u, float v, float a, float b, float lae, float lbe, float& ra,
                      float& rb) {
        const float vv = __fmul_rn(v, v);
        const float uv2 = __fmul_rn(2.0f, __fmul_rn(u, v));
        // a' = a + dt [Du la - (v^2 + F) a + v^2 b]
        float fa = __fmaf_rn(-__fadd_rn(vv, m.a2), a, __fmul_rn(vv, b));
        fa = __fmaf_rn(m.a0, lae, fa);
        // b' = b + dt [Dv lb - 2uv a + (2uv - F - k) b]
        float fb = __fmaf_rn(__fsub_rn(uv2, m.a3), b, -__fmul_rn(uv2, a));
        fb = __fmaf_rn(m.a1, lbe, fb);
        ra = __fmaf_rn(m.dt, fa, a);
        rb = __fmaf_rn(m.dt, fb, b);
      };
      site(u4.x, v4.x, a4.x, b4.x, la4.x, lb4.x, na.x, nb.x);
      site(u4.y, v4.y, a4.y, b4.y, la4.y, lb4.y, na.y, nb.y);
      site(u4.z, v4.z, a4.z, b4.z, la4.z, lb4.z, na.z, nb.z);
      site(u4.w, v4.w, a4.w, b4.w, la4.w, lb4.w, na.w, nb.w);
    };
    if (tid < TILE) {  // the tile, with the gradient terms
      const int p = B::at(rr, jj);
      float4 na, nb;
      back(p, na, nb);
      if (j > 0) {
        *reinterpret_cast<float4*>(d + p) = na;
        *reinterpret_cast<float4*>(d + PL + p) = nb;
      } else if (nvalid == 4) {
        const int64_t off = (int64_t)gy * g.pitch + gx;
        *reinterpret_cast<float4*>(lam_out.f[0] + off) = na;
        *reinterpret_cast<float4*>(lam_out.f[1] + off) = nb;
      } else if (nvalid > 0) {
        const int64_t off = (int64_t)gy * g.pitch + gx;
        const float ra[3] = {na.x, na.y, na.z}, rb[3] = {nb.x, nb.y, nb.z};
#pragma unroll
        for (int e = 0; e < 3; ++e)
          if (e < nvalid) {
            lam_out.f[0][off + e] = ra[e];
            lam_out.f[1][off + e] = rb[e];
          }
      }
      const float4 u4 = *reinterpret_cast<const float4*>(s + p);
      const float4 v4 = *reinterpret_cast<const float4*>(s + PL + p);
      const float4 a4 = *reinterpret_cast<const float4*>(l + p);
      const float4 b4 = *reinterpret_cast<const float4*>(l + PL + p);
      const float4 lu4 = lap2d_x4<PF_ST_STD, PF_MODEL_GS>(s, p, WS, 1.0f);
      const float4 lv4 = lap2d_x4<PF_ST_STD, PF_MODEL_GS>(s + PL, p, WS, 1.0f);
      float t[4] = {0.f, 0.f, 0.f, 0.f};  // Du, Dv, F, k
      auto term = [&](int e, float u, float v, float a, float b, float lu, float lv) {
        if (e < nvalid) {
          t[0] = __fmaf_rn(a, lu, t[0]);
          t[1] = __fmaf_rn(b, lv, t[1]);
          t[2] = __fadd_rn(t[2], __fsub_rn(__fmul_rn(__fsub_rn(1.0f, u), a), __fmul_rn(v, b)));
          t[3] = __fsub_rn(t[3], __fmul_rn(v, b));
        }
      };
      term(0, u4.x, v4.x, a4.x, b4.x, lu4.x, lv4.x);
      term(1, u4.y, v4.y, a4.y, b4.y, lu4.y, lv4.y);
      term(2, u4.z, v4.z, a4.z, b4.z, lu4.z, lv4.z);
      term(3, u4.w, v4.w, a4.w, b4.w, lu4.w, lv4.w);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float w = warp_sum_f(t[q]);
        if ((tid & 31) == 0) red[j][q][tid >> 5] = w;
      }
    } else if (j > 0) {  // the ring of j sites around it: rows above and below, a group a side
      constexpr int gpr = kATX / 4 + 2;
      const int nring = 2 * j * gpr + 2 * TY;
      for (int i = tid - TILE; i < nring; i += NT - TILE) {
        int r, q;
        if (i < 2 * j * gpr) {
          r = i / gpr;
          q = i - r * gpr - 1;
          r = r < j ? r - j : TY + r - j;
        } else {
          r = (i - 2 * j * gpr) >> 1;
          q = (i - 2 * j * gpr) & 1 ? kATX / 4 : -1;
        }
        const int p = B::at(r, q);
        float4 na, nb;
        back(p, na, nb);
        *reinterpret_cast<float4*>(d + p) = na;
        *reinterpret_cast<float4*>(d + PL + p) = nb;
      }
    }
    __syncthreads();
  }
  if (tid < 32) {  // the warps' sums per step (side by side: FP64 additions are slow), the steps'
    if (tid < 4 * LEN) {
      double v = 0.0;
#pragma unroll
      for (int w = 0; w < NW; ++w) v += (double)red[tid >> 2][tid & 3][w];
      step_sum[tid >> 2][tid & 3] = v;
    }
    __syncwarp();
    if (tid < 4) {
      double* slot = gpart + 4 * ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) + tid;
      double t = *slot;
#pragma unroll
      for (int j = LEN - 1; j >= 0; --j) t += step_sum[j][tid];
      *slot = t;
    }
  }
}

template <int LEN>
cudaError_t launch_gs_block(dim3 grid, const FieldPtrs& x, const FieldPtrs& lam,
                            const FieldOut& out, const Geom& g, const ModelParams& m,
                            double* gpart, cudaStream_t st) {
  using B = AdjBlock<LEN>;
  constexpr size_t smem = sizeof(float) * B::SMEM_FLOATS;
  static unsigned long long attr_mask = 0;  // per instantiation and device
  cudaError_t e = ensure_smem_attr(adj_gs2d_kernel<LEN>, smem, &attr_mask);
  if (e != cudaSuccess) return e;
  return launch_chained(adj_gs2d_kernel<LEN>, grid, B::NT, smem, st, x, lam, out, g, m, gpart);
}

// LEN reverse steps of Model A or B on a 64 x 16 tile in one launch: the block of
// adj_gs2d_kernel for one field. A step, forward or reverse, reaches R sites (Model B: 2, through
// mu and through w = lap lambda, which pass through one more plane of shared memory); Model B's
// blocks are two steps long, since four would stage a halo of 12. The gradient terms are summed
// per thread over four sites (every fourth row), per warp (half a row) in float, then in FP64.
//
// Bound by latency on small grids and by shared memory on large ones, as the Gray-Scott blocks.
// Reverse pass of 400 steps, against one launch per step with the states recomputed on a second
// stream: Model A 64^2 1.07 -> 0.55 ms, 512^2 1.42 -> 0.72, 2048^2 7.9 -> 5.8; Model B 64^2
// 1.28 -> 0.91, 512^2 2.09 -> 1.16, 2048^2 11.4 -> 8.9. 256 threads and four CTAs per SM: with a
// thread for every group of the widest region instead (544 and 416) 512^2 takes 0.93 and 1.53,
// 2048^2 6.2 and 10.1.
template <int MODEL, int LEN>
struct AdjBlock1 {
  static constexpr int R = MODEL == PF_MODEL_CH ? 2 : 1;
  static constexpr int NG = MODEL == PF_MODEL_CH ? 3 : 2;        // gradient sums
  static constexpr int HX = LEN > 1 ? 2 * R * (LEN - 1) : 1;     // staged halo of the state
  static constexpr int HL = R * LEN;                             // and of lambda
  static constexpr int H = HX > HL ? HX : HL;
  static constexpr int HP = (H + 3) / 4 * 4;
  static constexpr int WS = kATX + 2 * HP, ROWS = kATY + 2 * H;
  static constexpr int PL = WS * ROWS;
  static constexpr int NL = MODEL == PF_MODEL_CH ? 1 : 2;        // lambda buffers (B: in place)
  static constexpr int SMEM_FLOATS = (LEN + NL + (MODEL == PF_MODEL_CH ? 1 : 0)) * PL;
  static __device__ __forceinline__ int at(int r, int c) { return (r + H) * WS + HP + c; }
};

template <int MODEL, int LEN>
__global__ void __launch_bounds__(kNT2, 4)
    adj_one2d_kernel(FieldPtrs x, FieldPtrs lam, FieldOut lam_out, Geom g, ModelParams m,
                     double* gpart) {
  using B = AdjBlock1<MODEL, LEN>;
  constexpr bool CH = MODEL == PF_MODEL_CH;
  constexpr int WS = B::WS, PL = B::PL, NT = kNT2, R = B::R, NG = B::NG;
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) float sm[];  // state j at j PL
  __shared__ float red[LEN][NG][NW];
  __shared__ double step_sum[LEN][NG];
  float* la = sm + LEN * PL;         // lambda (Model A: twice)
  float* sw = la + B::NL * PL;       // Model B: mu, then w
  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * kATX, y0 = blockIdx.y * kATY;
  canary_fill(sm, B::SMEM_FLOATS);
  chain_wait();
  // f(p, r, q) for the groups of the tile and h sites around it
  auto region = [&](int h, auto f) {
    const int q0 = -((h + 3) / 4), gpr = kATX / 4 - 2 * q0;
    for (int i = tid; i < (kATY + 2 * h) * gpr; i += NT) {
      const int r = i / gpr - h, q = i % gpr + q0;
      f(B::at(r, 4 * q), r, q);
    }
  };
  auto stage = [&](const float* in, int h, float* dst) {
    region(h, [&](int p, int r, int q) {
      const float* row = in + (int64_t)wrap_index(y0 + r, g.ny) * g.pitch;
      const int gx = wrap_index(x0 + 4 * q, g.nx);
      if (gx + 3 < g.nx && gx % 4 == 0) {
        cp_async16(dst + p, row + gx);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) cp_async4(dst + p + c, row + wrap_index(gx + c, g.nx));
      }
    });
  };
  stage(x.f[0], B::HX, sm);
  stage(lam.f[0], B::HL, la);
  cp_async_wait_all();
  __syncthreads();
  // the block's states: x^{j+1} on the tile plus HX - R (j + 1) sites
#pragma unroll
  for (int j = 0; j + 1 < LEN; ++j) {
    const float* s = sm + j * PL;
    float* d = sm + (j + 1) * PL;
    const int h = B::HX - R * (j + 1);
    if constexpr (CH) {
      region(h + 1, [&](int p, int, int) {
        site4_mu<MODEL, PF_ST_STD>(s, p, WS, PL, m, sw);
      });
      __syncthreads();
    }
    region(h, [&](int p, int, int) {
      float4 v[1];
      site4_update<MODEL, PF_ST_STD>(s, sw, p, WS, PL, m, v);
      *reinterpret_cast<float4*>(d + p) = v[0];
    });
    __syncthreads();
  }
  // lambda back through them
  const float c2x3 = __fmul_rn(3.0f, m.a1);
#pragma unroll
  for (int j = LEN - 1; j >= 0; --j) {
    const float* s = sm + j * PL;
    const float* l = CH ? la : la + ((LEN - 1 - j) & 1) * PL;
    float* d = CH ? la : la + ((LEN - j) & 1) * PL;
    if constexpr (CH) {  // w = lap lambda^{s+j+1}
      region(R * j + 1, [&](int p, int, int) {
        *reinterpret_cast<float4*>(sw + p) = lap2d_x4(l, p, WS, m.lap_scale);
      });
      __syncthreads();
    }
    // lambda^{s+j} on the tile plus R j sites
    region(R * j, [&](int p, int r, int q) {
      const float4 p4 = *reinterpret_cast<const float4*>(s + p);
      const float4 l4 = *reinterpret_cast<const float4*>(l + p);
      float4 n;
      if constexpr (CH) {  // + dt M [(3 c2 x^2 - c1) w - lap w]
        const float4 w4 = *reinterpret_cast<const float4*>(sw + p);
        const float4 lw = lap2d_x4(sw, p, WS, m.lap_scale);
        auto site = [&](float ph, float la_, float w, float lwe) {
          const float sfac = __fmaf_rn(c2x3, __fmul_rn(ph, ph), -m.a0);
          return __fmaf_rn(m.a2, __fmaf_rn(sfac, w, -lwe), la_);
        };
        n = make_float4(site(p4.x, l4.x, w4.x, lw.x), site(p4.y, l4.y, w4.y, lw.y),
                        site(p4.z, l4.z, w4.z, lw.z), site(p4.w, l4.w, w4.w, lw.w));
      } else {  // + dt [lap lambda + (c1 - 3 c2 x^2) lambda]
        const float4 ll = lap2d_x4(l, p, WS, m.lap_scale);
        auto site = [&](float ph, float la_, float lle) {
          const float sfac = __fmaf_rn(-c2x3, __fmul_rn(ph, ph), m.a0);
          return __fmaf_rn(m.dt, __fmaf_rn(sfac, la_, lle), la_);
        };
        n = make_float4(site(p4.x, l4.x, ll.x), site(p4.y, l4.y, ll.y),
                        site(p4.z, l4.z, ll.z), site(p4.w, l4.w, ll.w));
      }
      if (j > 0) {
        *reinterpret_cast<float4*>(d + p) = n;
      } else {
        const int gy = y0 + r, gx = x0 + 4 * q;
        if (gy < g.ny && gx < g.nx) {
          float* o = lam_out.f[0] + (int64_t)gy * g.pitch + gx;
          if (gx + 3 < g.nx) {
            *reinterpret_cast<float4*>(o) = n;
          } else {
            const float e[3] = {n.x, n.y, n.z};
#pragma unroll
            for (int c = 0; c < 3; ++c)
              if (gx + c < g.nx) o[c] = e[c];
          }
        }
      }
    });
    float acc[NG] = {};  // the gradient terms
#pragma unroll
    for (int k = 0; k < kATX * kATY / NT; ++k) {
      const int rr = (tid + NT * k) / kATX, cc = tid % kATX;
      if (x0 + cc < g.nx && y0 + rr < g.ny) {
        const int p = B::at(rr, cc);
        const float ph = s[p], ph2 = __fmul_rn(ph, ph);
        if constexpr (CH) {
          const float w = sw[p];
          const float mu =
              ch_mu(ph, lap2d(ph, s[p - 1], s[p + 1], s[p - WS], s[p + WS], m.lap_scale), m);
          const float wp = __fmul_rn(w, ph);
          acc[0] = __fadd_rn(acc[0], wp);
          acc[1] = __fmaf_rn(wp, ph2, acc[1]);
          acc[2] = __fmaf_rn(w, mu, acc[2]);
        } else {
          const float lp = __fmul_rn(l[p], ph);
          acc[0] = __fadd_rn(acc[0], lp);
          acc[1] = __fmaf_rn(lp, ph2, acc[1]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const float w = warp_sum_f(acc[q]);
      if ((tid & 31) == 0) red[j][q][tid >> 5] = w;
    }
    __syncthreads();
  }
  if (tid < 32) {  // the warps' sums per step, then the steps'
    if (tid < NG * LEN) {
      double v = 0.0;
#pragma unroll
      for (int w = 0; w < NW; ++w) v += (double)red[tid / NG][tid % NG][w];
      step_sum[tid / NG][tid % NG] = v;
    }
    __syncwarp();
    if (tid < NG) {
      double* slot = gpart + 4 * ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) + tid;
      double t = *slot;
#pragma unroll
      for (int j = LEN - 1; j >= 0; --j) t += step_sum[j][tid];
      *slot = t;
    }
  }
}

template <int MODEL, int LEN>
cudaError_t launch_one_block(dim3 grid, const FieldPtrs& x, const FieldPtrs& lam,
                             const FieldOut& out, const Geom& g, const ModelParams& m,
                             double* gpart, cudaStream_t st) {
  using B = AdjBlock1<MODEL, LEN>;
  constexpr size_t smem = sizeof(float) * B::SMEM_FLOATS;
  static unsigned long long attr_mask = 0;  // per instantiation and device
  cudaError_t e = ensure_smem_attr(adj_one2d_kernel<MODEL, LEN>, smem, &attr_mask);
  if (e != cudaSuccess) return e;
  return launch_chained(adj_one2d_kernel<MODEL, LEN>, grid, kNT2, smem, st, x, lam, out, g, m,
                        gpart);
}

// One block of len reverse steps
cudaError_t launch_block(int model, int len, dim3 grid, const FieldPtrs& x, const FieldPtrs& lam,
                         const FieldOut& out, const Geom& g, const ModelParams& m, double* gpart,
                         cudaStream_t st) {
  constexpr int A = PF_MODEL_AC, B = PF_MODEL_CH;
  if (model == PF_MODEL_GS) {
    switch (len) {
      case 1: return launch_gs_block<1>(grid, x, lam, out, g, m, gpart, st);
      case 2: return launch_gs_block<2>(grid, x, lam, out, g, m, gpart, st);
      case 3: return launch_gs_block<3>(grid, x, lam, out, g, m, gpart, st);
      case 4: return launch_gs_block<4>(grid, x, lam, out, g, m, gpart, st);
    }
  } else if (model == PF_MODEL_AC) {
    switch (len) {
      case 1: return launch_one_block<A, 1>(grid, x, lam, out, g, m, gpart, st);
      case 2: return launch_one_block<A, 2>(grid, x, lam, out, g, m, gpart, st);
      case 3: return launch_one_block<A, 3>(grid, x, lam, out, g, m, gpart, st);
      case 4: return launch_one_block<A, 4>(grid, x, lam, out, g, m, gpart, st);
    }
  } else if (model == PF_MODEL_CH) {
    switch (len) {
      case 1: return launch_one_block<B, 1>(grid, x, lam, out, g, m, gpart, st);
      case 2: return launch_one_block<B, 2>(grid, x, lam, out, g, m, gpart, st);
    }
  }
  return cudaErrorInvalidValue;
}

// out[q] = sum over CTAs of gpart[4 * cta + q], in CTA order split over 256 threads.
__global__ void __launch_bounds__(256) adj_final_kernel(const double* gpart, int64_t nctas,
                                                        double* out) {
  __shared__ double red[4][256 / 32];
  double t[4] = {0, 0, 0, 0};
  const int64_t per = (nctas + 255) / 256;
  const int64_t c0 = per * threadIdx.x;
  const int64_t c1 = c0 + per < nctas ? c0 + per : nctas;
  for (int64_t c = c0; c < c1; ++c)
#pragma unroll
    for (int q = 0; q < 4; ++q) t[q] += gpart[4 * c + q];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    t[q] = warp_sum_d(t[q]);
    if (lane == 0) red[q][wid] = t[q];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double s = 0.0;
    for (int w = 0; w < 256 / 32; ++w) s += red[threadIdx.x][w];
    out[threadIdx.x] = s;
  }
}

// Steps per reverse launch: states at the blocks' first steps are stored or recomputed, those
// between live only inside a launch.
int block_len(int model) { return model == PF_MODEL_CH ? 2 : 4; }

// Reverse-step launch grid (the same tiles for every model).
dim3 adj_grid(const pf_grid_s* g) {
  const Geom q = grid_geom(g);
  return dim3((q.nx + kATX - 1) / kATX, (q.ny + kATY - 1) / kATY, 1);
}

float* ckpt_field(pf_grid_s* g, int64_t i, int f) {
  return g->adj.ckpt + (i * g->nf + f) * g->field_elems;
}
// States of a segment that are recomputed, and the j-th of them in buffer b.
int64_t seg_states(int64_t interval, int block) { return (interval + block - 1) / block - 1; }
float* seg_field(pf_grid_s* g, int b, int64_t j, int f) {
  const AdjointState& a = g->adj;
  return a.seg + ((b * seg_states(a.interval, a.block) + j) * g->nf + f) * g->field_elems;
}
float* lam_field(pf_grid_s* g, int b, int f) {
  return g->adj.lam + (b * g->nf + f) * g->field_elems;
}

int check_gs2d(pf_grid_s* g) {
  if (!g->model_set ||
      (g->model != PF_MODEL_GS && g->model != PF_MODEL_AC && g->model != PF_MODEL_CH)) {
    set_error("the adjoint needs a Gray-Scott, Allen-Cahn or Cahn-Hilliard model");
    return PF_ERR_STATE;
  }
  if (g->dim != 2) return invalid("the adjoint is implemented for 2D grids");
  if (g->stencil != PF_ST_STD) return invalid("the adjoint uses the standard 5-point stencil");
  return PF_OK;
}

}  // namespace

// Bytes that the live handles of a device hold in states stored by the library's choice.
static std::atomic<int64_t> g_stored[64];

// Count `need` bytes of this handle's checkpoints (in place of what it held) against the limits
// above; false, and nothing changed, where they do not fit.
static bool hold_states(pf_grid_s* g, double need) {
  AdjointState& a = g->adj;
  if (g->device < 0 || g->device >= 64 || need > (double)kAllStates) return false;
  size_t free_bytes = 0, total = 0;
  if (cudaMemGetInfo(&free_bytes, &total) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const int64_t want = (int64_t)need;
  if (want > ((int64_t)free_bytes + a.held) / kFreeParts) return false;
  std::atomic<int64_t>& sum = g_stored[g->device];
  int64_t now = sum.load();
  do {
    if (now - a.held + want > kAllStates) return false;
  } while (!sum.compare_exchange_weak(now, now - a.held + want));
  a.held = want;
  return true;
}

static void drop_states(pf_grid_s* g) {
  AdjointState& a = g->adj;
  if (a.held > 0) g_stored[g->device] -= a.held;
  a.held = 0;
}

void adjoint_release(pf_grid_s* g) {
  AdjointState& a = g->adj;
  drop_states(g);
  if (a.ckpt) cudaFree(a.ckpt);
  if (a.seg) cudaFree(a.seg);
  if (a.lam) cudaFree(a.lam);
  a = AdjointState();
}

// Enqueue the whole reverse pass on stream st: zero the gradient slots, then per segment from
// last to first recompute its blocks' first states from its checkpoint and run its reverse
// blocks, then sum the slots. *lb_out receives the buffer holding lambda^0.
//
// With two segment buffers the recomputation is a branch of its own (g->branch, forked from st and
// joined to it): segment s - 1 is recomputed into one buffer while segment s goes back from the
// other, so its launches hide behind the reverse blocks. A buffer is written again once the
// segment before last, its reader, is done; every kernel sees the same inputs as in one branch.
// (Reverse pass of 400 steps, in one branch and in two, ms: Gray-Scott 512^2 in intervals of 5
// 2.13 -> 1.43, of 20 1.62 -> 1.18; Model B 64^2 in 5 1.30 -> 0.91, 1024^2 3.84 -> 3.22; Gray-Scott
// 2048^2 in 20 14.04 -> 13.55.)
static cudaError_t enqueue_reverse(pf_grid_s* g, const ModelParams& m, cudaStream_t st,
                                   int* lb_out) {
  AdjointState& a = g->adj;
  const Geom q = grid_geom(g);
  const dim3 grid = adj_grid(g);
  const int64_t nctas = (int64_t)grid.x * grid.y;
  const int64_t C = a.interval;
  const int B = block_len(g->model);
  int tile = 0, depth = 1;
  plan2d(g, &tile, &depth);  // (depth: B)
  cudaError_t e = cudaMemsetAsync(a.gpart, 0, sizeof(double) * 4 * nctas, st);
  const bool two = a.seg_bufs == 2;
  cudaStream_t st2 = st;
  // per buffer: recomputed (on st2), its segment gone back through (on st); the branch's two ends
  struct Events {
    cudaEvent_t rec[2] = {}, rev[2] = {}, fork = nullptr, join = nullptr;
    cudaEvent_t* all[6] = {&rec[0], &rec[1], &rev[0], &rev[1], &fork, &join};
    ~Events() {
      for (cudaEvent_t* ev : all)
        if (*ev) cudaEventDestroy(*ev);
    }
  } ev;
  if (two) {
    if (e == cudaSuccess && g->branch == nullptr)
      e = cudaStreamCreateWithFlags(&g->branch, cudaStreamNonBlocking);
    for (cudaEvent_t* x : ev.all)
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(x, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(ev.fork, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(g->branch, ev.fork, 0);
    if (e != cudaSuccess) return e;
    st2 = g->branch;
  }
  int lb = 0;  // lambda ping-pong buffer holding the current adjoint state
  for (int64_t s = a.n_ckpt - 1; s >= 0 && e == cudaSuccess; --s) {
    const int64_t len = std::min(C, a.n_steps - s * C);
    const int64_t nb = (len + B - 1) / B;  // blocks
    const int buf = two ? (int)(s & 1) : 0;
    // first state of block b: the checkpoint, or recomputed
    auto state = [&](int64_t b, int f) -> float* {
      return b == 0 ? ckpt_field(g, s, f) : seg_field(g, buf, b - 1, f);
    };
    if (two && s + 2 < a.n_ckpt) e = cudaStreamWaitEvent(st2, ev.rev[buf], 0);
    for (int64_t b = 1; b < nb && e == cudaSuccess; ++b) {
      FieldPtrs in{};
      FieldOut out{};
      for (int f = 0; f < g->nf; ++f) {
        in.f[f] = state(b - 1, f);
        out.f[f] = state(b, f);
      }
      e = launch_2d(g, tile, B, in, out, m, st2);
    }
    if (two && e == cudaSuccess) e = cudaEventRecord(ev.rec[buf], st2);
    if (two && e == cudaSuccess) e = cudaStreamWaitEvent(st, ev.rec[buf], 0);
    for (int64_t b = nb - 1; b >= 0 && e == cudaSuccess; --b) {
      FieldPtrs xs{}, li{};
      FieldOut lo{};
      for (int f = 0; f < g->nf; ++f) {
        xs.f[f] = state(b, f);
        li.f[f] = lam_field(g, lb, f);
        lo.f[f] = lam_field(g, 1 - lb, f);
      }
      const int n = (int)std::min<int64_t>(B, len - b * B);
      e = launch_block(g->model, n, grid, xs, li, lo, q, m, a.gpart, st);
      lb = 1 - lb;
    }
    if (two && e == cudaSuccess) e = cudaEventRecord(ev.rev[buf], st);
  }
  if (two) {  // (also after an error, so that a capture can end)
    cudaError_t ej = cudaEventRecord(ev.join, st2);
    if (ej == cudaSuccess) ej = cudaStreamWaitEvent(st, ev.join, 0);
    if (e == cudaSuccess) e = ej;
  }
  if (e == cudaSuccess) {
    adj_final_kernel<<<1, 256, 0, st>>>(a.gpart, nctas, a.gout);
    e = cudaGetLastError();
  }
  *lb_out = lb;
  return e;
}

// Steps the grid's state from checkpoint 0 (set by the caller) through all n_steps, every segment
// from its checkpoint into the next one without a copy between; the result lands in a grid
// buffer. For the kernels that take any buffers; the on-chip ones run per segment, with copies,
// where segments are long enough for the state's way in and out of the chip (400 steps of GS 128^2
// with the cluster kernel: 0.45 ms in segments of 20, 1.03 in segments of 4, tiles 0.50 in either).
static int forward_segments(pf_grid_s* g, int64_t n_steps, int64_t C, int64_t n_ckpt) {
  int tile = 0, depth = 1;
  run_plan(g, &tile, &depth);
  const size_t state = sizeof(float) * g->nf * g->field_elems;
  const bool on_chip = tile == kTileCluster2D || tile == kTileBands2D;
  if (on_chip && C < 16) {
    plan2d(g, &tile, &depth);
  } else if (on_chip) {
    for (int64_t s = 0; s < n_ckpt; ++s) {
      if (s > 0)
        PF_CUDA_TRY(cudaMemcpyAsync(ckpt_field(g, s, 0), g->buf[g->cur][0], state,
                                    cudaMemcpyDeviceToDevice, g->stream));
      if (int rc = pf_step(g, std::min(C, n_steps - s * C))) return rc;
    }
    return PF_OK;
  }
  int last = g->cur;  // the grid buffer written last
  for (int64_t s = 0; s < n_ckpt; ++s) {
    FieldPtrs in{};
    for (int f = 0; f < g->nf; ++f) in.f[f] = ckpt_field(g, s, f);
    int64_t left = std::min(C, n_steps - s * C);
    while (left > 0) {
      int k = depth;
      while (k > left) k >>= 1;
      left -= k;
      FieldOut out{};
      const bool to_ckpt = left == 0 && s + 1 < n_ckpt;
      if (!to_ckpt) last = 1 - last;
      for (int f = 0; f < g->nf; ++f)
        out.f[f] = to_ckpt ? ckpt_field(g, s + 1, f) : g->buf[last][f];
      PF_CUDA_TRY(launch_2d(g, plan_tile(g, tile, k), k, in, out, g->params, g->stream));
      for (int f = 0; f < g->nf; ++f) in.f[f] = out.f[f];
    }
  }
  g->cur = last;
  return PF_OK;
}

}  // namespace pf

using namespace pf;

extern "C" {

int pf_adj_forward(pf_grid_t g, int64_t n_steps, int64_t ckpt_interval) {
  NvtxRange nvtx_("pf_adj_forward");
  if (int rc = check_grid(g)) return rc;
  if (int rc = check_gs2d(g)) return rc;
  if (n_steps < 1) return invalid("n_steps must be >= 1");
  if (ckpt_interval < 0) return invalid("ckpt_interval must be >= 0");
  AdjointState& a = g->adj;
  const size_t state = sizeof(float) * g->nf * g->field_elems;
  const int B = block_len(g->model);
  if (a.lam == nullptr) {  // lambda twice, the gradient slots of every CTA and the four sums
    const dim3 grid = adj_grid(g);
    const int64_t nctas = (int64_t)grid.x * grid.y;
    const size_t lam = (2 * state + 255) / 256 * 256;
    PF_CUDA_TRY(cudaMalloc(&a.lam, lam + sizeof(double) * (4 * nctas + 4)));
    PF_CUDA_TRY(cudaMemsetAsync(a.lam, 0, 2 * state, g->stream));
    a.gpart = reinterpret_cast<double*>(reinterpret_cast<char*>(a.lam) + lam);
    a.gout = a.gpart + 4 * nctas;
  }
  // The library's choice: every block's first state where they fit (hold_states; nothing to
  // recompute between blocks then), else sqrt(N) checkpoints. A request that was answered before
  // keeps its schedule: asked for anew in every pass of a training loop, a refused choice would
  // have the buffers freed and allocated again each time, and the reverse pass's graph with them.
  const int64_t root = (int64_t)std::ceil(std::sqrt((double)n_steps));
  const bool answered = a.n_ckpt > 0 && a.block == B && a.asked_steps == n_steps &&
                        a.asked_interval == ckpt_interval;
  int64_t C = ckpt_interval > 0 ? ckpt_interval : root;
  if (answered) {
    C = a.interval;
  } else if (ckpt_interval == 0 &&
             hold_states(g, (double)((n_steps + B - 1) / B) * (double)state)) {
    C = B;
  } else {
    drop_states(g);
  }
  if (C > n_steps) C = n_steps;
  int64_t n_ckpt = (n_steps + C - 1) / C;
  // (seg's size depends on the model's block length, and a grid's model may change)
  if (a.n_ckpt != n_ckpt || a.interval != C || a.block != B) {
    // (re)allocate for this schedule; a recorded pass or graph of the old one is void
    a.ready = 0;
    if (g->adj_exec) cudaGraphExecDestroy(g->adj_exec);
    g->adj_exec = nullptr;
    g->adj_exec_steps = -1;
    if (a.ckpt) cudaFree(a.ckpt);
    if (a.seg) cudaFree(a.seg);
    a.ckpt = nullptr;
    a.seg = nullptr;
    a.seg_bufs = 0;
    a.n_ckpt = 0;
    cudaError_t e = cudaMalloc(&a.ckpt, state * n_ckpt);
    if (e != cudaSuccess && ckpt_interval == 0 && C < root) {
      cudaGetLastError();  // no room for all of them
      drop_states(g);
      C = root < n_steps ? root : n_steps;
      n_ckpt = (n_steps + C - 1) / C;
      e = cudaMalloc(&a.ckpt, state * n_ckpt);
    }
    if (e != cudaSuccess) return cuda_fail(e, "pf_adj_forward checkpoints");
    if (C > B) {
      const size_t seg = state * seg_states(C, B);
      // (the library's own choice of sqrt(N) is made where memory is short: one buffer)
      a.seg_bufs = ckpt_interval > 0 && n_ckpt > 1 ? 2 : 1;
      if (a.seg_bufs == 2 && cudaMalloc(&a.seg, 2 * seg) != cudaSuccess) {
        cudaGetLastError();  // one segment after the other
        a.seg = nullptr;
        a.seg_bufs = 1;
      }
      if (a.seg_bufs == 1) PF_CUDA_TRY(cudaMalloc(&a.seg, seg));
    }
    a.n_ckpt = n_ckpt;
    a.interval = C;
    a.block = B;
  }
  a.asked_steps = n_steps;
  a.asked_interval = ckpt_interval;
  // (a grid buffer's fields lie one after the other, as a checkpoint's)
  PF_CUDA_TRY(cudaMemcpyAsync(ckpt_field(g, 0, 0), g->buf[g->cur][0], state,
                              cudaMemcpyDeviceToDevice, g->stream));
  if (int rc = forward_segments(g, n_steps, C, n_ckpt)) return rc;
  bool same = a.dt == g->dt;
  for (int i = 0; i < 4; ++i) same = same && a.coeffs[i] == g->coeffs[i];
  if (!same) {  // a recorded graph carries the old coefficients
    if (g->adj_exec) cudaGraphExecDestroy(g->adj_exec);
    g->adj_exec = nullptr;
    g->adj_exec_steps = -1;
  }
  for (int i = 0; i < 4; ++i) a.coeffs[i] = g->coeffs[i];
  a.dt = g->dt;
  a.n_steps = n_steps;
  a.model = g->model;
  a.ready = 1;
  return PF_OK;
}

int pf_adj_backward(pf_grid_t g, const float* dLdu_N, const float* dLdv_N, int on_device,
                    float* dLdu0, float* dLdv0, double* dtheta) {
  NvtxRange nvtx_("pf_adj_backward");
  if (int rc = check_grid(g)) return rc;
  if (int rc = check_gs2d(g)) return rc;
  AdjointState& a = g->adj;
  if (!a.ready) {
    set_error("pf_adj_backward: no recorded forward pass (call pf_adj_forward first)");
    return PF_ERR_STATE;
  }
  if (a.model != g->model) {  // the states, and what is kept of them, are another model's
    set_error("pf_adj_backward: the recorded forward pass is of another model (call "
              "pf_adj_forward after pf_set_model)");
    return PF_ERR_STATE;
  }
  if (dLdu_N == nullptr || (g->nf == 2 && dLdv_N == nullptr))
    return invalid("dL/dx_N must not be NULL");
  const ModelParams m = make_params(g->model, a.coeffs, a.dt, g->h);
  const size_t w = sizeof(float) * g->nx;
  const cudaMemcpyKind kin = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  const cudaMemcpyKind kout = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  const float* src[2] = {dLdu_N, dLdv_N};
  for (int f = 0; f < g->nf; ++f)
    PF_CUDA_TRY(cudaMemcpy2DAsync(lam_field(g, 0, f), sizeof(float) * g->pitch, src[f], w, w,
                                  (size_t)g->ny, kin, g->stream));
  // A first pass of a schedule is enqueued launch by launch; a second one is recorded as a graph,
  // which later ones replay (recording costs more than the launches it saves once).
  int lb = 0;
  const bool same = g->adj_exec_steps == a.n_steps && g->adj_exec_interval == a.interval;
  if (!same) {
    if (g->adj_exec) cudaGraphExecDestroy(g->adj_exec);
    g->adj_exec = nullptr;
    PF_CUDA_TRY(enqueue_reverse(g, m, g->stream, &lb));
    g->adj_exec_steps = a.n_steps;
    g->adj_exec_interval = a.interval;
  } else {
    if (g->adj_exec == nullptr) {
      if (g->capture == nullptr)
        PF_CUDA_TRY(cudaStreamCreateWithFlags(&g->capture, cudaStreamNonBlocking));
      PF_CUDA_TRY(cudaStreamBeginCapture(g->capture, cudaStreamCaptureModeRelaxed));
      cudaError_t e = enqueue_reverse(g, m, g->capture, &g->adj_exec_lb);
      cudaGraph_t graph = nullptr;
      cudaError_t e2 = cudaStreamEndCapture(g->capture, &graph);
      if (e != cudaSuccess || e2 != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        return cuda_fail(e != cudaSuccess ? e : e2, "pf_adj_backward graph capture");
      }
      e = cudaGraphInstantiate(&g->adj_exec, graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) {
        g->adj_exec = nullptr;
        return cuda_fail(e, "pf_adj_backward cudaGraphInstantiate");
      }
    }
    PF_CUDA_TRY(cudaGraphLaunch(g->adj_exec, g->stream));
    lb = g->adj_exec_lb;
  }
  PF_CUDA_TRY(cudaMemcpyAsync(g->sums_host(), a.gout, sizeof(double) * 4, cudaMemcpyDeviceToHost,
                              g->stream));
  float* dst[2] = {dLdu0, dLdv0};
  for (int f = 0; f < g->nf; ++f)
    if (dst[f] != nullptr)
      PF_CUDA_TRY(cudaMemcpy2DAsync(dst[f], w, lam_field(g, lb, f), sizeof(float) * g->pitch, w,
                                    (size_t)g->ny, kout, g->stream));
  PF_CUDA_TRY(cudaStreamSynchronize(g->stream));
  if (dtheta != nullptr) {
    const double* S = g->sums_host();
    if (g->model == PF_MODEL_GS) {
      // the kernel's Laplacians of u and v are unscaled (the parameters carry 1/h^2 in
      // D_u and D_v), so the sums for D_u and D_v take the factor here
      const double s = 1.0 / (g->h * g->h);
      for (int i = 0; i < 4; ++i) dtheta[i] = a.dt * S[i] * (i < 2 ? s : 1.0);
    } else if (g->model == PF_MODEL_AC) {
      dtheta[0] = a.dt * S[0];
      dtheta[1] = -a.dt * S[1];
    } else {
      const double M = a.coeffs[2];
      dtheta[0] = -a.dt * M * S[0];
      dtheta[1] = a.dt * M * S[1];
      dtheta[2] = a.dt * S[2];
    }
  }
  return PF_OK;
}

}  // extern "C"
