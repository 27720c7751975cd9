// N coupled species of reaction-diffusion type (any number of fields up to PF_MAX_FIELDS,
// Sec. 2.3's coupled equations of motion; Gray-Scott of Sec. 1 is the two-species case):
//   du_i/dt = D_i lap u_i + sum_m K[i][m] prod_j u_j^E[m][j]
// with up to kRdMonomials monomials of integer exponents 0..3, advanced by forward Euler
// (Sec. 2.4.1) with the 5-/7-point Laplacian (Sec. 2.2.2), every field from the same state.
//
// 2D kernel (3D: pf_fe3d_one.cu), fused per step: a CTA stages its tile plus a one-site periodic
// halo of every field in shared memory (rows with four halo columns a side, as 16-byte cp.async
// groups), then each thread takes four consecutive sites: every field's Laplacian, the reaction
// polynomial and the Euler update in registers (pf_rd.cuh), and one 16-byte store per field.
#include "pf_rd.cuh"
#include "pf_stage.cuh"

namespace pf {

namespace {

// Store four sites of every field at off (gx = their first column).
template <int NF>
__device__ __forceinline__ void rd_store4(const FieldOut& out, int64_t off, int gx, int nx,
                                          const float4 (&res)[NF]) {
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    if (gx + 3 < nx) {
      *reinterpret_cast<float4*>(out.f[f] + off) = res[f];
    } else {
      out.f[f][off] = res[f].x;
      if (gx + 1 < nx) out.f[f][off + 1] = res[f].y;
      if (gx + 2 < nx) out.f[f][off + 2] = res[f].z;
    }
  }
}

// ---- 2D: TX x TY tiles, rows staged with 4 halo columns each side (16-byte groups)
constexpr int kRd2Threads = 256;

template <int NF, int TX, int TY>
struct CfgRd2 {
  static constexpr int WS = TX + 8;      // staged row: columns x0-4 .. x0+TX+3
  static constexpr int HT = TY + 2;      // rows y0-1 .. y0+TY
  static constexpr int PL = WS * HT;     // floats per field
  static constexpr int GROUPS = (TX / 4) * TY;
};

template <int NF, int TX, int TY>
__global__ void __launch_bounds__(kRd2Threads) rd2d_kernel(FieldPtrs in, FieldOut out, Geom g,
                                                           RdParams p) {
  using C = CfgRd2<NF, TX, TY>;
  extern __shared__ __align__(16) float sm[];
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  canary_fill(sm, (size_t)NF * C::PL);
  chain_wait();
  stage_rows4<NF>(in, g, x0, y0, 0, C::WS, C::HT, C::PL, sm, kRd2Threads);
  cp_async_wait_all();
  __syncthreads();
  for (int q = threadIdx.x; q < C::GROUPS; q += kRd2Threads) {
    const int rr = q / (TX / 4), j = q - rr * (TX / 4);
    const int gy = y0 + rr, gx = x0 + 4 * j;
    if (gy >= g.ny || gx >= g.nx) continue;
    const int pc = (rr + 1) * C::WS + 4 + 4 * j;
    float4 u[NF], ls[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const float* s = sm + f * C::PL + pc;
      u[f] = *reinterpret_cast<const float4*>(s);
      const float4 ym = *reinterpret_cast<const float4*>(s - C::WS);
      const float4 yp = *reinterpret_cast<const float4*>(s + C::WS);
      ls[f] = lap2d_sum4(u[f], s[-1], s[4], ym, yp);
    }
    float4 res[NF];
    rd_sites4<NF>(u, ls, p, res);
    rd_store4<NF>(out, (int64_t)gy * g.pitch + gx, gx, g.nx, res);
  }
}

template <int NF>
cudaError_t launch_rd2d_nf(const Geom& g, FieldPtrs in, FieldOut out, const RdParams& p,
                           cudaStream_t s) {
  constexpr int TX = 64, TY = 16;
  using C = CfgRd2<NF, TX, TY>;
  const size_t smem = sizeof(float) * NF * C::PL;
  static unsigned long long attr_mask = 0;  // per instantiation and device
  cudaError_t e = ensure_smem_attr(rd2d_kernel<NF, TX, TY>, smem, &attr_mask);
  if (e != cudaSuccess) return e;
  const dim3 grid((g.nx + TX - 1) / TX, (g.ny + TY - 1) / TY);
  return launch_chained(rd2d_kernel<NF, TX, TY>, grid, kRd2Threads, smem, s, in, out, g, p);
}

}  // namespace

void rd_places(int nf, RdParams& p) {
  for (int m = 0; m < p.nmono; ++m) {
    int n = 0, f[3] = {0, 0, 0};  // degree and factors, ascending
    for (int j = 0; j < nf; ++j)
      for (int e = (p.E[m] >> (2 * j)) & 3; e > 0; --e, ++n)
        if (n < 3) f[n] = j;
    p.place[m] = n == 0   ? 0
                 : n == 1 ? 1 + f[0]
                 : n == 2 ? 1 + PF_MAX_FIELDS + rd_pair(f[0], f[1])
                 : n == 3 ? 15 + rd_triple(f[0], f[1], f[2])
                          : 35;
  }
}

cudaError_t launch_rd2d(const Geom& g, int nf, FieldPtrs in, FieldOut out, const RdParams& p,
                        cudaStream_t s) {
  switch (nf) {
    case 1: return launch_rd2d_nf<1>(g, in, out, p, s);
    case 2: return launch_rd2d_nf<2>(g, in, out, p, s);
    case 3: return launch_rd2d_nf<3>(g, in, out, p, s);
    case 4: return launch_rd2d_nf<4>(g, in, out, p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace pf
