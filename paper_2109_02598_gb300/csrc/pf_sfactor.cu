// Radially averaged structure factor of a phase indicator (analysis of the phase-separated
// systems of Sec. 3): rho = [psi > 0], rho_hat by a float64 transform, S = |rho_hat|^2 / N,
// binned by |k| with per-bin sums taken in a fixed order.
//
// The half spectrum holds each mode k with kx in (0, nx/2) once for itself and once for its
// mirror -k (equal |k|, equal S for a real rho), so those modes count twice; kx = 0 and the
// Nyquist plane of an even nx count once.  |k| and the bin index are float64, decided as the
// definition's correctly rounded operations in a fixed order would.
//
// Those operations (three wavenumbers, a square root and three divisions per mode) are FP64,
// of which an SM does two a clock: 1.8 ms for the 8.5 million modes of 256^3. Every one of
// them is monotone, so the bin of a mode is decided by its |k|^2 alone: a table kernel finds,
// per bin, the least double |k|^2 that the definition puts into it (by running the definition
// on neighbouring doubles) and the squared wavenumbers of each axis. A mode then costs two
// additions and two comparisons, and three operations for |rho_hat|^2 and its sum; 1/N and the
// weights are applied per bin. A lane keeps its kx and walks along ky, where |k|^2 changes
// slowly, adding into a register while the bin stays; when it changes, the warp's lanes add
// their sums to the warp's histogram in lane order. Fixed order throughout: the same bits on
// every run. The bin kernel, 256^3 and 32 bins: 1829 us before, 0.2 ms now (reading 135 MB);
// a whole call 4614 -> 3095 us, 4096^2 5260 -> 3660, 2048^2 1690 -> 1260, 128^3 1240 -> 1000, 64^2
// 460 -> 400, 16^2 340 either way (the transform and its plan are the rest).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "pf_cufft.h"
#include "pf_internal.h"

namespace pf {
int invalid(const char* fmt, ...);
}

namespace pf {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kMaxBins = 1024;
constexpr int kMaxBinBlocks = 2 * 152;

struct SfGeom {
  int rank;
  int64_t d[3];  // C order, x last
  int64_t nxh, nk, nsite;
  double h, kmax;
  int n_bins;
  // tables in device memory: squared wavenumbers of the axes (C order, x's half), and the
  // bins' least |k|^2 (n_bins, then infinity)
  double *k2[3], *least;
  // tasks of a warp: (z, chunk of cw columns of kx, segment of seg rows of ky)
  int nchunk, cw, seg, nseg;
  int64_t tasks;
};

__device__ __forceinline__ double fft_index(int64_t i, int64_t n) {
  return (double)(i <= (n - 1) / 2 ? i : i - n);
}

__device__ __forceinline__ double wavenumber(double f, int64_t n, double h) {
  const double val = __ddiv_rn(1.0, __dmul_rn((double)n, h));
  return __dmul_rn(2.0 * 3.141592653589793, __dmul_rn(f, val));
}

// Bin of a mode by the definition; -1 for k = 0, which is left out.
__device__ int bin_of(double s2, const SfGeom& g) {
  const double kmag = __dsqrt_rn(s2);
  if (!(kmag > 0.0)) return -1;
  const double fq = floor(__dmul_rn(__ddiv_rn(kmag, g.kmax), (double)g.n_bins));
  return fq >= (double)(g.n_bins - 1) ? g.n_bins - 1 : (int)fq;
}

// Bound by the latency of its FP64 chains, some 50 dependent operations a trial of bin_of: a block
// per SM, and eight lanes try a bin's limit at eight places at once (three trials after one another,
// where one lane's bisection over 128 doubles takes nine). 7 us on 16^2, 9 with an axis of 2^18.
constexpr int kTableBlocks = 152;
__global__ void __launch_bounds__(128) sf_table_kernel(SfGeom g) {
  const int64_t i = blockIdx.x * 128 + threadIdx.x;
  for (int a = 0; a < g.rank; ++a) {
    const int64_t n = g.d[a], m = a == g.rank - 1 ? g.nxh : n;
    for (int64_t j = i; j < m; j += (int64_t)gridDim.x * 128) {
      const double k = wavenumber(fft_index(j, n), n, g.h);
      g.k2[a][j] = __dmul_rn(k, k);
    }
  }
  if (i == 0) g.least[g.n_bins] = __longlong_as_double(0x7ff0000000000000ll);
  const int lane = threadIdx.x & 7;
  const unsigned group = 0xffu << (threadIdx.x & 24);  // the eight lanes of a bin
  for (int64_t b = i >> 3; b < g.n_bins; b += (int64_t)gridDim.x * 16) {
    // the least positive double whose bin is at least b: a search on the bit patterns of the
    // positive doubles (in their order), bin_of being monotone
    // bin(lo) < b <= bin(hi), taking bin(0) = -1: from 16 doubles either side of the bin's
    // lower edge squared (the roundings of both come to some ten), or from all of them where
    // that does not hold it
    const double edge = (double)b * g.kmax / (double)g.n_bins;
    const long long at = __double_as_longlong(edge * edge), top = 0x7ff0000000000000ll;
    long long lo = at - 16, hi = at + 16;
    auto below = [&](long long v) { return bin_of(__longlong_as_double(v), g) < (int)b; };
    const unsigned ends = __ballot_sync(group, below(lane == 0 ? lo : hi)) >> (threadIdx.x & 24);
    if (lo < 0 || !(ends & 1)) lo = 0;
    if (hi > top || (ends & 2)) hi = top;
    while (hi - lo > 1) {
      const long long step = (hi - lo + 6) / 8;  // eight places from lo + step, the last at hi - 1 or on
      const long long v = lo + (lane + 1) * step;
      const int n = __popc(__ballot_sync(group, v < hi && below(v)));
      hi = min(hi, lo + (n + 1) * step);
      lo += n * step;
    }
    if (lane == 0) g.least[b] = __longlong_as_double(hi);
  }
}

__global__ void indicator_kernel(const float* __restrict__ psi, int64_t pitch, int64_t nx,
                                 int64_t ny, int64_t nsite, double* __restrict__ rho) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nsite;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = i % nx, row = i / nx;  // row = z * ny + y
    rho[i] = psi[row * pitch + x] > 0.f ? 1.0 : 0.0;
  }
}

// Each warp takes tasks (z, kx chunk, ky segment) at a fixed stride into its own histogram;
// the block then sums its warps' histograms in warp order.
constexpr int kAhead = 8;  // ky rows loaded together
__global__ void __launch_bounds__(kThreads)
    sf_bin_kernel(const double2* __restrict__ rhat, SfGeom g, double* __restrict__ part_sum,
                  unsigned long long* __restrict__ part_cnt) {
  extern __shared__ unsigned char smem_raw[];
  double* wsum = reinterpret_cast<double*>(smem_raw);
  unsigned long long* wcnt =
      reinterpret_cast<unsigned long long*>(wsum + (size_t)kWarps * g.n_bins);
  for (int i = threadIdx.x; i < kWarps * g.n_bins; i += kThreads) {
    wsum[i] = 0.0;
    wcnt[i] = 0ull;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t nx = g.d[g.rank - 1], ny = g.d[g.rank - 2];
  double* my_sum = wsum + (size_t)warp * g.n_bins;
  unsigned long long* my_cnt = wcnt + (size_t)warp * g.n_bins;
  const double* ky2 = g.k2[g.rank - 2];
  for (int64_t task = (int64_t)blockIdx.x * kWarps + warp; task < g.tasks;
       task += (int64_t)gridDim.x * kWarps) {
    const int sg = (int)(task % g.nseg);
    const int64_t rest = task / g.nseg;
    const int chunk = (int)(rest % g.nchunk);
    const int64_t iz = rest / g.nchunk;
    const int64_t y0 = (int64_t)sg * g.seg, y1 = min(ny, y0 + g.seg);
    const int64_t ix = (int64_t)chunk * g.cw + lane;
    const bool on = lane < g.cw && ix < g.nxh;
    const int weight = on ? ((ix == 0 || 2 * ix == nx) ? 1 : 2) : 0;
    const double kx2 = g.k2[g.rank - 1][on ? ix : 0];
    const double kz2 = g.rank == 3 ? g.k2[0][iz] : 0.0;
    const double2* src = rhat + (iz * ny + y0) * g.nxh + (on ? ix : 0);
    // the lane's current bin, its limits [lo, hi), and the sum and count of the modes in it
    int bin = -1;
    double lo = 0.0, hi = 0.0, acc = 0.0;
    unsigned cnt = 0;
    auto flush = [&](bool need) {
      unsigned left = __ballot_sync(0xffffffffu, need && cnt > 0 && bin >= 0);
      while (left != 0) {
        const int src_lane = __ffs(left) - 1;
        left &= left - 1;
        if (lane == src_lane) {
          my_sum[bin] = __dadd_rn(my_sum[bin], weight == 2 ? acc + acc : acc);
          my_cnt[bin] += (unsigned long long)weight * cnt;
        }
        __syncwarp();
      }
      if (need) {
        acc = 0.0;
        cnt = 0;
      }
    };
    for (int64_t y = y0; y < y1; y += kAhead) {
      double2 r[kAhead];
#pragma unroll
      for (int k = 0; k < kAhead; ++k)
        r[k] = y + k < y1 && on ? src[(y - y0 + k) * g.nxh] : make_double2(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < kAhead; ++k) {
        if (y + k >= y1) break;  // uniform
        const double t = g.rank == 3 ? __dadd_rn(kz2, ky2[y + k]) : ky2[y + k];
        const double s2 = __dadd_rn(t, kx2);
        const bool moved = !(s2 >= lo && s2 < hi) && on;
        if (__any_sync(0xffffffffu, moved)) {
          flush(moved);
          if (moved) {
            if (s2 >= g.least[0]) {
              // near the root of |k|^2, then to the bin whose limits hold it
              bin = (int)(sqrt((float)s2) / (float)g.kmax * (float)g.n_bins);
              bin = bin < 0 ? 0 : bin > g.n_bins - 1 ? g.n_bins - 1 : bin;
              while (s2 < g.least[bin]) --bin;
              while (bin + 1 < g.n_bins && s2 >= g.least[bin + 1]) ++bin;
              lo = g.least[bin];
              hi = g.least[bin + 1];
            } else {  // k = 0
              bin = -1;
              lo = 0.0;
              hi = g.least[0];
            }
          }
        }
        acc = __dadd_rn(acc, __fma_rn(r[k].x, r[k].x, __dmul_rn(r[k].y, r[k].y)));
        cnt += 1;
      }
    }
    flush(on);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < g.n_bins; b += kThreads) {
    double s = 0.0;
    unsigned long long c = 0ull;
    for (int w = 0; w < kWarps; ++w) {
      s = __dadd_rn(s, wsum[(size_t)w * g.n_bins + b]);
      c += wcnt[(size_t)w * g.n_bins + b];
    }
    part_sum[(size_t)blockIdx.x * g.n_bins + b] = s;
    part_cnt[(size_t)blockIdx.x * g.n_bins + b] = c;
  }
}

// One warp per bin: the blocks' partials by lane, then a fixed tree.
__global__ void __launch_bounds__(kThreads)
    sf_final_kernel(const double* __restrict__ part_sum,
                    const unsigned long long* __restrict__ part_cnt, int nblocks, int n_bins,
                    double nsite, double* __restrict__ mean, long long* __restrict__ counts) {
  const int b = blockIdx.x * kWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (b >= n_bins) return;
  double s = 0.0;
  unsigned long long c = 0ull;
  for (int k = lane; k < nblocks; k += 32) {
    s = __dadd_rn(s, part_sum[(size_t)k * n_bins + b]);
    c += part_cnt[(size_t)k * n_bins + b];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s = __dadd_rn(s, __shfl_down_sync(0xffffffffu, s, o));
    c += __shfl_down_sync(0xffffffffu, c, o);
  }
  if (lane == 0) {
    mean[b] = c > 0 ? __ddiv_rn(__ddiv_rn(s, nsite), (double)c) : 0.0;
    counts[b] = (long long)c;
  }
}

unsigned long long g_bin_smem_mask = 0;

}  // namespace
}  // namespace pf

using namespace pf;

extern "C" int pf_structure_factor(int dim, const int64_t* n, int64_t pitch, const float* psi,
                                   double h, int n_bins, double* centres, double* mean,
                                   int64_t* counts, void* stream) {
  if (n == nullptr || psi == nullptr || centres == nullptr || mean == nullptr ||
      counts == nullptr)
    return invalid("pf_structure_factor: NULL argument");
  if (dim != 2 && dim != 3) return invalid("dim must be 2 or 3 (got %d)", dim);
  const int64_t nx = n[0], ny = n[1], nz = dim == 3 ? n[2] : 1;
  const int64_t lim = (int64_t)1 << 30;
  if (nx < 2 || ny < 1 || nz < 1 || nx > lim || ny > lim || nz > lim || nx * ny > lim ||
      nx * ny * nz > lim)
    return invalid("sizes must be nx >= 2, ny, nz >= 1, with at most 2^30 sites (got %lld x "
                   "%lld x %lld)", (long long)nx, (long long)ny, (long long)nz);
  if (pitch < nx || pitch > lim) return invalid("pitch %lld must be in [nx, 2^30]", (long long)pitch);
  if (!(h > 0.0) || !std::isfinite(h)) return invalid("h must be finite and > 0");
  if (n_bins < 1 || n_bins > kMaxBins) return invalid("n_bins must be in [1, %d]", kMaxBins);
  const CufftApi* api = cufft_api();
  if (api == nullptr) return PF_ERR_CUDA;
  cudaStream_t st = (cudaStream_t)stream;

  SfGeom g{};
  g.rank = dim;
  if (dim == 2) {
    g.d[0] = ny;
    g.d[1] = nx;
  } else {
    g.d[0] = nz;
    g.d[1] = ny;
    g.d[2] = nx;
  }
  g.nxh = nx / 2 + 1;
  g.nk = g.nxh * ny * nz;
  g.nsite = nx * ny * nz;
  g.h = h;
  g.kmax = (3.141592653589793 / h) * std::sqrt((double)dim);
  g.n_bins = n_bins;

  // tasks: even chunks of at most 32 columns of kx, and ky segments of at least kAhead rows, down
  // to where there are two tasks for each of the blocks' warps; on small grids of two rows, down
  // to a task per SM (their lanes meet a new bin in nearly every row, and add to the histogram
  // one after another: 64^2 in 256 bins 495 us a call with segments of 32 rows)
  g.nchunk = (int)((g.nxh + 31) / 32);
  g.cw = (int)((g.nxh + g.nchunk - 1) / g.nchunk);
  g.nseg = 1;
  for (;; g.nseg *= 2) {
    const int64_t rows = ny / (2 * g.nseg), tasks = (int64_t)g.nchunk * nz * g.nseg;
    if (!(rows >= kAhead && tasks < 2 * kWarps * kMaxBinBlocks) && !(rows >= 2 && tasks < 152)) break;
  }
  g.seg = (int)((ny + g.nseg - 1) / g.nseg);
  g.nseg = (int)((ny + g.seg - 1) / g.seg);
  g.tasks = (int64_t)g.nchunk * nz * g.nseg;
  int64_t nblocks = (g.tasks + kWarps - 1) / kWarps;
  if (nblocks > kMaxBinBlocks) nblocks = kMaxBinBlocks;

  // One allocation: rho (after its transform the tables), rho_hat, partial sums and counts, results.
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t b_rho = up(sizeof(double) * (size_t)std::max<int64_t>(
      g.nsite, nz + ny + g.nxh + n_bins + 1));
  const size_t b_hat = up(sizeof(double2) * (size_t)g.nk);
  const size_t b_part = up(sizeof(double) * (size_t)(nblocks * n_bins));
  const size_t b_res = up(sizeof(double) * (size_t)n_bins);
  unsigned char* mem = nullptr;
  cudaError_t e = cudaMalloc(&mem, b_rho + b_hat + 2 * b_part + 2 * b_res);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error("pf_structure_factor: out of device memory");
    return PF_ERR_OOM;
  }
  double* rho = reinterpret_cast<double*>(mem);
  double2* rhat = reinterpret_cast<double2*>(mem + b_rho);
  double* psum = reinterpret_cast<double*>(mem + b_rho + b_hat);
  unsigned long long* pcnt = reinterpret_cast<unsigned long long*>(mem + b_rho + b_hat + b_part);
  double* d_mean = reinterpret_cast<double*>(mem + b_rho + b_hat + 2 * b_part);
  long long* d_cnt = reinterpret_cast<long long*>(mem + b_rho + b_hat + 2 * b_part + b_res);

  double* tab = rho;
  for (int i = 0; i < dim; ++i) {
    g.k2[i] = tab;
    tab += i == dim - 1 ? g.nxh : g.d[i];
  }
  g.least = tab;

  cufftHandle plan = -1;
  int rc = cufft_plan(api, &plan, dim, g.d, CUFFT_D2Z, 1, 0, 0, 1, nullptr);
  if (rc == PF_OK) {
    int64_t blocks = (g.nsite + 255) / 256;
    if (blocks > 152 * 8) blocks = 152 * 8;
    indicator_kernel<<<(int)blocks, 256, 0, st>>>(psi, pitch, nx, ny, g.nsite, rho);
    e = cudaGetLastError();
    cufftResult r = CUFFT_SUCCESS;
    if (e == cudaSuccess) {
      r = api->set_stream(plan, st);
      if (r == CUFFT_SUCCESS) r = api->exec_d2z(plan, rho, reinterpret_cast<cufftDoubleComplex*>(rhat));
    }
    if (r != CUFFT_SUCCESS) {
      rc = cufft_fail(r, "pf_structure_factor transform");
    } else {
      const size_t smem = (size_t)kWarps * n_bins * (sizeof(double) + sizeof(unsigned long long));
      if (e == cudaSuccess)
        e = ensure_smem_attr(sf_bin_kernel, (size_t)kWarps * kMaxBins * 16, &g_bin_smem_mask);
      if (e == cudaSuccess) {
        sf_table_kernel<<<kTableBlocks, 128, 0, st>>>(g);
        sf_bin_kernel<<<(int)nblocks, kThreads, smem, st>>>(rhat, g, psum, pcnt);
        e = cudaGetLastError();
      }
      if (e == cudaSuccess) {
        sf_final_kernel<<<(n_bins + kWarps - 1) / kWarps, kThreads, 0, st>>>(
            psum, pcnt, (int)nblocks, n_bins, (double)g.nsite, d_mean, d_cnt);
        e = cudaGetLastError();
      }
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(mean, d_mean, sizeof(double) * n_bins, cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(counts, d_cnt, sizeof(int64_t) * n_bins, cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) rc = cuda_fail(e, "pf_structure_factor");
    }
  }
  if (plan != -1) api->destroy(plan);
  cudaStreamSynchronize(st);
  cudaFree(mem);
  if (rc != PF_OK) return rc;
  for (int b = 0; b < n_bins; ++b) centres[b] = ((double)b + 0.5) * g.kmax / (double)n_bins;
  return PF_OK;
}

extern "C" int pf_porod_fit(int n_bins, const double* centres, const double* mean,
                            const int64_t* counts, double k_lo, double k_hi, double* slope,
                            double* intercept, int* n_used) {
  if (centres == nullptr || mean == nullptr || counts == nullptr || slope == nullptr ||
      intercept == nullptr || n_used == nullptr)
    return invalid("pf_porod_fit: NULL argument");
  if (n_bins < 1) return invalid("n_bins must be >= 1");
  if (!(k_lo < k_hi)) return invalid("the window needs k_lo < k_hi");
  // two passes over the usable bins in bin order: the means, then the centred sums
  int n = 0;
  double sx = 0.0, sy = 0.0;
  auto usable = [&](int b) {
    return centres[b] >= k_lo && centres[b] <= k_hi && counts[b] > 0 && mean[b] > 0.0;
  };
  for (int b = 0; b < n_bins; ++b) {
    if (!usable(b)) continue;
    sx += std::log(centres[b]);
    sy += std::log(mean[b]);
    ++n;
  }
  if (n < 2) return invalid("fewer than two usable bins in [%g, %g]", k_lo, k_hi);
  const double xbar = sx / n, ybar = sy / n;
  double sxy = 0.0, sxx = 0.0;
  for (int b = 0; b < n_bins; ++b) {
    if (!usable(b)) continue;
    const double dx = std::log(centres[b]) - xbar;
    const double dy = std::log(mean[b]) - ybar;
    sxy += dx * dy;
    sxx += dx * dx;
  }
  if (!(sxx > 0.0)) return invalid("the usable bins share one centre");
  *slope = sxy / sxx;
  *intercept = ybar - *slope * xbar;
  *n_used = n;
  return PF_OK;
}
