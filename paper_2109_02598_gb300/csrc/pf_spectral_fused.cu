// Fused engine of the semi-implicit spectral solver (Sec. 2.4.2) for grids whose sides are
// powers of two: 2D with sides 4 .. 1024, and 3D with nx in 4 .. 1024 and ny nz small enough
// for one (y, z) slab to stay in a CTA's shared memory. Every step of a pf_spectral_step call
// runs inside one cooperative launch, with this file's own FFTs in shared memory.
//
// The state psi_hat [nz][ny][nxh] (and the tables) are those of the cuFFT engine; W (the f_hat
// slices of spec, which this engine uses as scratch) carries the data between the two phases
// of a step. In 2D it has the state's layout [y][kx]; in 3D it is held as [kx][z][y], so that
// a slab is contiguous and the strided accesses fall to the row phase, whose tasks spread
// them over many more SMs (the slab phase has one task per kx):
//   row phase   per x-row (z, y): the inverse transform along x of W's half spectrum, the
//               nonlinear terms, the forward transform along x, back into W. Two real rows
//               share one complex FFT: rows r and r+1 of a one-field model, or psi and m of
//               one row in Model C (whose nonlinear terms need both at the same site);
//   slab phase  per column kx (and field): the ny x nz slab of W at that kx, transformed
//               forward along y and then z -> f_hat; on the self-conjugate columns (kx = 0,
//               nx/2) its Hermitian part, pairing (kz, ky) with (-kz, -ky); the update
//               psi_hat <- A psi_hat + (B N) f_hat; and the inverse transform (z, then y) of
//               psi_hat / N back into W for the next row phase. In 2D the slab is one column.
// Each slab team owns fixed slabs for the whole launch and keeps their psi_hat and (A, B N) in
// shared memory: a prologue loads them and fills W from psi_hat; the last step writes
// psi_hat and work = psi_hat / N (as the cuFFT engine leaves them) back to global memory
// instead of the inverse transform. The phases are separated by a grid barrier (release /
// acquire atomics) whose waits are bounded by a clock budget: on timeout a CTA sets the
// error word and returns, so the launch always ends.
//
// A task (a row pair, or a slab) is done by a team of 32 .. 1024 threads of a CTA, chosen
// per phase so that each thread does one radix-8 butterfly per pass where the tasks still fit
// in one round on the SMs; a team synchronises on its own named barrier. The FFTs are
// Stockham passes between two shared-memory buffers: natural order in and out, no bit reversal,
// and every thread loads all of a butterfly's inputs before it computes. Both phases transform
// there and back, and a step is bound by the latency of that chain: a pass (about 1000 cycles
// with eight warps on an SM) is an exchange through shared memory and a barrier. So a transform is
// radix-8 passes and one of radix 8, 4 or 2, last on the way there and first on the way back, and
// those two passes are one, with the nonlinear terms or the update between them in registers; a
// 2D column's first pass reads global memory and its last one writes there. A 512-point row takes
// five exchanges, a column four (before: nine each, with the pointwise parts in passes of their
// own). A slab's transforms are batched passes: along y the slab's nz rows at once, along z its
// ny columns at once, consecutive lanes on consecutive FFTs of the batch; the slab's rows are
// padded to ny + 1 values in shared memory, so those lanes fall on distinct banks in both
// directions. Us a step, before and now: Model C 512^2 18.1 -> 10.4, 256^2 13.6 -> 8.0, Model B
// 512^2 14.2 -> 8.9, 64^3 17.6 -> 12.1, Model A 64^2 9.7 -> 6.4. What remains at 512^2: two grid
// barriers of 3300 and 4700 cycles (the wait for the other CTAs' stores and for the two columns
// that pair with themselves in it), loads and stores 5900, passes 9000.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "pf_spectral.h"
#include "pf_tma.cuh"

namespace pf {
int invalid(const char* fmt, ...);

namespace {

constexpr int kThreads = 1024;  // the widest CTA (launch bound); see fused_shape
constexpr int kMaxSide = 1024;

struct FusedArgs {
  float2* state;  // [nf][cs]
  float2* W;      // [nf][cs]
  float2* work;   // [nf][cs]
  const float2* table;
  const float2* twx;  // W_nx^j, j < nx
  const float2* twy;  // W_ny^j, j < ny
  const float2* twz;  // W_nz^j, j < nz (3D)
  int nx, ny, nz, nxh, lognx, logny, lognz, nf;
  int nrows;               // x-rows: ny nz
  int wr, wk;              // W: mode kx of x-row r at W + field cs + r wr + kx wk
  int rbuf, cbuf;          // float2s of one row team's / slab team's two FFT buffers
  int row_team, col_team;  // threads per task in the row and slab phases
  int cpt;                 // slabs owned per slab team
  int64_t cs;
  float inv_n;
  NlCoeffs k;
  int64_t steps;
  unsigned int* bar;  // count, generation, error
  long long budget;
};

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)),
                     __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}

// The threads that share one task: `size` threads (a power of two from 8) of one CTA, the
// `index`-th such group. Teams wider than a warp synchronise on named barrier index + 1; a
// warp, or a warp's 8- or 16-lane teams, on __syncwarp (the whole warp: its teams run the same
// control flow, see the row phase).
struct Team {
  int size, rank, index;
  __device__ __forceinline__ void sync() const {
    if (size <= 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(index + 1), "r"(size) : "memory");
  }
};

__device__ __forceinline__ Team make_team(int size) {
  Team t;
  t.size = size;
  t.rank = threadIdx.x % size;
  t.index = threadIdx.x / size;
  return t;
}

// 4-point DFT of (a, b, c, d): out[m] = sum_r x_r W_4^{r m}, W_4 = -i (forward) or +i.
template <bool INV>
__device__ __forceinline__ void dft4(const float2& a, const float2& b, const float2& c,
                                     const float2& d, float2* out) {
  const float2 a0 = make_float2(__fadd_rn(a.x, c.x), __fadd_rn(a.y, c.y));
  const float2 a1 = make_float2(__fsub_rn(a.x, c.x), __fsub_rn(a.y, c.y));
  const float2 a2 = make_float2(__fadd_rn(b.x, d.x), __fadd_rn(b.y, d.y));
  const float2 dd = make_float2(__fsub_rn(b.x, d.x), __fsub_rn(b.y, d.y));
  const float2 a3 = INV ? make_float2(-dd.y, dd.x) : make_float2(dd.y, -dd.x);
  out[0] = make_float2(__fadd_rn(a0.x, a2.x), __fadd_rn(a0.y, a2.y));
  out[1] = make_float2(__fadd_rn(a1.x, a3.x), __fadd_rn(a1.y, a3.y));
  out[2] = make_float2(__fsub_rn(a0.x, a2.x), __fsub_rn(a0.y, a2.y));
  out[3] = make_float2(__fsub_rn(a1.x, a3.x), __fsub_rn(a1.y, a3.y));
}

// R-point DFT in place, natural order in and out.
template <int R, bool INV>
__device__ __forceinline__ void dft(float2 (&v)[R]) {
  if constexpr (R == 8) {
    // two 4-point DFTs (even and odd inputs), the odd one twiddled by W_8^m, combined
    float2 e[4], o[4];
    dft4<INV>(v[0], v[2], v[4], v[6], e);
    dft4<INV>(v[1], v[3], v[5], v[7], o);
    const float c = 0.70710678118654752f;  // sqrt(1/2)
    const float2 o1 = o[1], o3 = o[3];
    if (!INV) {  // W_8 = c (1 - i), W_8^2 = -i, W_8^3 = -c (1 + i)
      o[1] = make_float2(__fmul_rn(c, __fadd_rn(o1.x, o1.y)), __fmul_rn(c, __fsub_rn(o1.y, o1.x)));
      o[2] = make_float2(o[2].y, -o[2].x);
      o[3] = make_float2(__fmul_rn(c, __fsub_rn(o3.y, o3.x)), -__fmul_rn(c, __fadd_rn(o3.x, o3.y)));
    } else {  // the conjugates: c (1 + i), i, c (-1 + i)
      o[1] = make_float2(__fmul_rn(c, __fsub_rn(o1.x, o1.y)), __fmul_rn(c, __fadd_rn(o1.x, o1.y)));
      o[2] = make_float2(-o[2].y, o[2].x);
      o[3] = make_float2(-__fmul_rn(c, __fadd_rn(o3.x, o3.y)), __fmul_rn(c, __fsub_rn(o3.x, o3.y)));
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      v[m] = make_float2(__fadd_rn(e[m].x, o[m].x), __fadd_rn(e[m].y, o[m].y));
      v[m + 4] = make_float2(__fsub_rn(e[m].x, o[m].x), __fsub_rn(e[m].y, o[m].y));
    }
  } else if constexpr (R == 4) {
    float2 x[4];
    dft4<INV>(v[0], v[1], v[2], v[3], x);
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = x[m];
  } else {
    const float2 a = v[0], b = v[1];
    v[0] = make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
    v[1] = make_float2(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y));
  }
}

template <int R>
constexpr int kLog2 = R == 8 ? 3 : R == 4 ? 2 : 1;

// Where element i of a single contiguous transform, and of a twiddle table, lies in shared memory:
// a place is left out after every eight, so that a first pass's stores (every eighth element from
// consecutive lanes) and the passes' twiddles (every 2^logt-th) fall on distinct banks (the tables
// alone, Model C 512^2: 11.2 -> 10.4 us a step).
__device__ __forceinline__ int padded(int i) { return i + (i >> 3); }
constexpr int64_t padded_size(int64_t n) { return n + n / 8; }

// v[r] *= W_n^{r k 2^logt} (INV: its conjugate); tw holds W_n^i = exp(-2 pi i / n), i < n,
// at padded(i)
template <int R, bool INV>
__device__ __forceinline__ void twiddle(float2 (&v)[R], int k, int logt, const float2* tw) {
#pragma unroll
  for (int r = 1; r < R; ++r) {
    float2 w = tw[padded((k * r) << logt)];
    if (INV) w.y = -w.y;
    v[r] = cmul(w, v[r]);
  }
}

// Butterfly t of a pass over 2^logb FFTs with 2^logq butterflies each: its FFT b and number j.
// BF: consecutive lanes take consecutive FFTs (whose elements are strided), else consecutive
// butterflies of one FFT.
template <bool BF>
__device__ __forceinline__ void butterfly(int t, int logq, int logb, int& b, int& j) {
  if (BF) {
    j = t >> logb;
    b = t - (j << logb);
  } else {
    b = t >> logq;
    j = t - (b << logq);
  }
}

// One Stockham pass of radix R over 2^logb FFTs of 2^logn points (stride 2^logns so far; FIRST:
// 0, no twiddles). Butterfly j of FFT b takes elements j + r n/R from ld(b, i), twiddles them by
// W_{ns R}^{(j mod ns) r}, and gives element (j - j mod ns) R + j mod ns + m ns of its DFT to
// st(b, i, value). INV: the inverse transform, unnormalised.
template <int R, bool INV, bool BF, bool FIRST, class LD, class ST>
__device__ __forceinline__ void fft_pass(int logn, int logns, int logb, const float2* tw,
                                         const Team& tm, const LD& ld, const ST& st) {
  const int logq = logn - kLog2<R>, q = 1 << logq, ns = 1 << logns;
  for (int t = tm.rank; t < 1 << (logq + logb); t += tm.size) {
    int b, j;
    butterfly<BF>(t, logq, logb, b, j);
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = ld(b, j + r * q);
    const int k = FIRST ? 0 : j & (ns - 1);
    if (!FIRST) twiddle<R, INV>(v, k, logn - logns - kLog2<R>, tw);
    dft<R, INV>(v);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int m = 0; m < R; ++m) st(b, base + m * ns, v[m]);
  }
}

// The last pass of one transform, op(b, i, value) on every element of its result, and the first
// pass of the transform back, in one: with the same radix the first pass's butterfly j takes just
// the elements j + m n/R that the last pass's butterfly j gives, so nothing passes through shared
// memory between them.
template <int R, bool INV, bool BF, class LD, class OP, class ST>
__device__ __forceinline__ void fft_there_and_back(int logn, int logb, const float2* tw,
                                                   const Team& tm, const LD& ld, const OP& op,
                                                   const ST& st) {
  const int logq = logn - kLog2<R>, q = 1 << logq;
  for (int t = tm.rank; t < 1 << (logq + logb); t += tm.size) {
    int b, j;
    butterfly<BF>(t, logq, logb, b, j);
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = ld(b, j + r * q);
    twiddle<R, INV>(v, j, 0, tw);
    dft<R, INV>(v);
#pragma unroll
    for (int m = 0; m < R; ++m) op(b, j + m * q, v[m]);
    dft<R, !INV>(v);
#pragma unroll
    for (int m = 0; m < R; ++m) st(b, j * R + m, v[m]);
  }
}

// A transform of 2^logn points is radix-8 passes and one of radix 2^odd_log(logn), last on the way
// there and first on the way back (logn >= 1).
__device__ __forceinline__ int odd_log(int logn) {
  const int l = logn % 3;
  return l == 0 ? 3 : l;
}

template <int R>
struct Radix {
  static constexpr int value = R;
};

template <class F>
__device__ __forceinline__ void with_radix(int log, const F& f) {
  if (log == 3) f(Radix<8>());
  else if (log == 2) f(Radix<4>());
  else f(Radix<2>());
}

__device__ __forceinline__ unsigned int ld_acquire(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier: bar[0] counts arrivals over the whole launch (target: the count that releases this
// one), bar[2] is the error word. An arrival is one reduction whose result nobody waits for, and
// every CTA polls the counter itself (a last arrival that reads the count and then publishes a
// generation is two more trips to L2: with 129 CTAs 4300 cycles a barrier, now 3300). Bounded:
// false after budget clocks without a release.
__device__ __forceinline__ bool grid_barrier(unsigned int* bar, unsigned int& target,
                                             long long budget) {
  target += gridDim.x;
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    // (release: with the CTA's writes, which the CTA barrier orders before this thread)
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const long long t0 = clock64();
    while ((int)(ld_acquire(bar) - target) < 0) {
      if (clock64() - t0 > budget) {
        atomicExch(bar + 2, 1u);
        ok = 0;
        break;
      }
    }
  }
  return __syncthreads_and(ok) != 0;
}

// At the end of a launch, also of one that gave up: the last CTA to leave (bar[1] counts them)
// sets the counters back for the next.
__device__ __forceinline__ void grid_leave(unsigned int* bar) {
  if (threadIdx.x == 0 && atomicAdd(bar + 1, 1u) + 1 == gridDim.x) {
    atomicExch(bar, 0u);
    atomicExch(bar + 1, 0u);
  }
}

template <int MODEL>
__device__ __forceinline__ void nl_pair(float2& z, const NlCoeffs& k) {
  if (MODEL == PF_MODEL_C) {
    nonlinear_site<MODEL>(z.x, z.y, k.c);
  } else {
    float unused = 0.f;
    nonlinear_site<MODEL>(z.x, unused, k.c);
    nonlinear_site<MODEL>(z.y, unused, k.c);
  }
}

// Row task: two real x-rows (field f1 row y1, field f2 row y2; a row index counts (z, y)
// rows, z slowest) whose half spectra are in W. A team with no task (valid false) runs the
// same steps on its own buffers without touching W, so that the warp it shares with other
// teams stays in step.
template <int MODEL>
__device__ __forceinline__ void row_task(const FusedArgs& a, int f1, int y1, int f2, int y2,
                                         bool valid, float2* b, float2* b2, const float2* twx,
                                         const Team& tm) {
  const int nx = a.nx, nh = nx >> 1;
  const int64_t ks = a.wk;  // mode stride of a row in W
  // both half spectra into b2 (X1 at [0, nh], X2 at [nh + 1, 2 nh + 1]; b2 holds nx + 2), all
  // of a thread's copies in flight before one wait
  const float2* X1g = a.W + f1 * a.cs + (int64_t)y1 * a.wr;
  const float2* X2g = a.W + f2 * a.cs + (int64_t)y2 * a.wr;
  for (int k = tm.rank; k <= nh && valid; k += tm.size) {
    cp_async8(b2 + k, X1g + k * ks);
    cp_async8(b2 + nh + 1 + k, X2g + k * ks);
  }
  cp_async_wait_all();
  tm.sync();
  // Z = X1 + i X2 over the full length, each extended by Hermitian symmetry; the imaginary
  // parts at k = 0 and nx/2 are dropped, as a complex-to-real transform does
  const float2* X1 = b2;
  const float2* X2 = b2 + nh + 1;
  auto z = [&](int, int k) {
    const bool up = k > nh;
    float2 p = X1[up ? nx - k : k], q = X2[up ? nx - k : k];
    if (k == 0 || k == nh) p.y = q.y = 0.f;
    if (up) {
      p.y = -p.y;
      q.y = -q.y;
    }
    return make_float2(__fsub_rn(p.x, q.y), __fadd_rn(p.y, q.x));
  };
  // the inverse transform, the nonlinear terms and the forward transform
  const int odd = odd_log(a.lognx);
  float2 *in = b2, *out = b;
  auto ld = [&](int, int i) { return in[padded(i)]; };
  auto st = [&](int, int i, float2 v) { out[padded(i)] = v; };
  auto turn = [&]() {
    tm.sync();
    float2* t = in;
    in = out;
    out = t;
  };
  if (a.lognx > odd) {
    fft_pass<8, true, false, true>(a.lognx, 0, 0, twx, tm, z, st);
    turn();
    for (int ns = 3; ns < a.lognx - odd; ns += 3) {
      fft_pass<8, true, false, false>(a.lognx, ns, 0, twx, tm, ld, st);
      turn();
    }
  } else {  // one pass in all
    for (int k = tm.rank; k < nx; k += tm.size) st(0, k, z(0, k));
    turn();
  }
  with_radix(odd, [&](auto r) {
    fft_there_and_back<decltype(r)::value, true, false>(
        a.lognx, 0, twx, tm, ld, [&](int, int, float2& v) { nl_pair<MODEL>(v, a.k); }, st);
  });
  turn();
  for (int ns = odd; ns < a.lognx; ns += 3) {
    fft_pass<8, false, false, false>(a.lognx, ns, 0, twx, tm, ld, st);
    turn();
  }
  const float2* Y = in;
  float2* F1 = a.W + f1 * a.cs + (int64_t)y1 * a.wr;
  float2* F2 = a.W + f2 * a.cs + (int64_t)y2 * a.wr;
  for (int k = tm.rank; k <= nh && valid; k += tm.size) {
    const float2 y = Y[padded(k)];
    const float2 r = Y[padded((nx - k) & (nx - 1))];  // Y(-k); conj taken below
    const float2 s = make_float2(__fadd_rn(y.x, r.x), __fsub_rn(y.y, r.y));  // Y + conj Y(-k)
    const float2 d = make_float2(__fsub_rn(y.x, r.x), __fadd_rn(y.y, r.y));  // Y - conj Y(-k)
    F1[k * ks] = make_float2(__fmul_rn(0.5f, s.x), __fmul_rn(0.5f, s.y));
    F2[k * ks] = make_float2(__fmul_rn(0.5f, d.y), __fmul_rn(-0.5f, d.x));  // -i d / 2
  }
  tm.sync();
}

// Slab task (field f, column kx): the ny x nz values W[f][z][y][kx], with the slab's psi_hat in
// st and (A, B N) in tb (shared memory, [kz][ky]). In 3D (D3) they are held in shared memory as
// [z][y] with rows of ny + 1 (the pad keeps a batched pass's lanes, one FFT each, on distinct
// banks) and transformed along y, then z; in 2D they are one column of ny values, which the first
// pass reads from global memory and the last one writes there.
// mode 0: prologue (W <- inverse(psi_hat / N)); mode 1: full step; mode 2: last step (psi_hat
// and work = psi_hat / N to global memory, no inverse transform).
template <bool D3>
__device__ __forceinline__ void slab_task(const FusedArgs& a, int f, int kx, int mode,
                                          float2* st, const float2* tb, float2* b, float2* b2,
                                          const float2* twy, const float2* twz, const Team& tm) {
  const int ny = a.ny, ns = ny * a.nz, rp = ny + 1;
  const int64_t base = f * a.cs + kx;  // the state's layout, [z][y][kx]
  const int64_t rstride = a.nxh;
  float2* Wg = a.W + f * a.cs + (int64_t)kx * a.wk;  // the slab in W (rows wr apart)
  // the axis transformed last on the way there (z; in 2D y) and the FFTs along it
  const int logn = D3 ? a.lognz : a.logny, logb = D3 ? a.logny : 0;
  const float2* tw = D3 ? twz : twy;
  const int odd = odd_log(logn);
  float2 *in = b, *out = b2;
  auto at = [&](int bb, int i) { return D3 ? bb + i * rp : padded(i); };
  auto ld = [&](int bb, int i) { return in[at(bb, i)]; };
  auto sm = [&](int bb, int i, float2 v) { out[at(bb, i)] = v; };
  auto ld_y = [&](int bb, int i) { return in[bb * rp + i]; };
  auto sm_y = [&](int bb, int i, float2 v) { out[bb * rp + i] = v; };
  auto turn = [&]() {
    tm.sync();
    float2* t = in;
    in = out;
    out = t;
  };
  const int odd_y = odd_log(a.logny);
  const bool direct = !D3 && logn > odd;  // 2D: global memory on either end
  if (mode != 0) {
    int s = 0;
    if (direct) {
      fft_pass<8, false, false, true>(
          logn, 0, 0, tw, tm, [&](int, int i) { return Wg[(int64_t)i * a.wr]; }, sm);
      turn();
      s = 3;
    } else {
      for (int i = tm.rank; i < ns; i += tm.size)
        cp_async8(b + (D3 ? i + (i >> a.logny) : padded(i)), Wg + (int64_t)i * a.wr);
      cp_async_wait_all();
      tm.sync();
    }
    if (D3) {  // forward along y: consecutive lanes take consecutive FFTs of the batch, here and below
      int sy = 0;
      if (a.logny > odd_y) {
        fft_pass<8, false, D3, true>(a.logny, 0, a.lognz, twy, tm, ld_y, sm_y);
        turn();
        for (sy = 3; sy < a.logny - odd_y; sy += 3) {
          fft_pass<8, false, D3, false>(a.logny, sy, a.lognz, twy, tm, ld_y, sm_y);
          turn();
        }
      }
      with_radix(odd_y, [&](auto r) {
        fft_pass<decltype(r)::value, false, D3, false>(a.logny, sy, a.lognz, twy, tm, ld_y, sm_y);
      });
      turn();
    }
    for (; s < logn - odd; s += 3) {
      fft_pass<8, false, D3, false>(logn, s, logb, tw, tm, ld, sm);
      turn();
    }
    // the update of the slab's value i = [kz][ky]; psi_hat / N
    auto update = [&](int i, const float2& fh) {
      const float2 p = st[i];
      const float2 t = tb[i];
      const float2 sn = make_float2(__fmaf_rn(t.x, p.x, __fmul_rn(t.y, fh.x)),
                                    __fmaf_rn(t.x, p.y, __fmul_rn(t.y, fh.y)));
      st[i] = sn;
      return make_float2(__fmul_rn(sn.x, a.inv_n), __fmul_rn(sn.y, a.inv_n));
    };
    auto value = [&](int bb, int i) { return D3 ? i * ny + bb : i; };
    const bool self = kx == 0 || 2 * kx == a.nx;
    if (mode == 1 && !self) {
      with_radix(odd, [&](auto r) {
        fft_there_and_back<decltype(r)::value, false, D3>(
            logn, logb, tw, tm, ld,
            [&](int bb, int i, float2& v) { v = update(value(bb, i), v); }, sm);
      });
    } else {
      with_radix(odd, [&](auto r) {
        fft_pass<decltype(r)::value, false, D3, false>(logn, s, logb, tw, tm, ld, sm);
      });
      turn();
      // f_hat, on a self-conjugate column its Hermitian part: (kz, ky) pairs with (-kz, -ky)
      auto fhat = [&](int bb, int i) {
        float2 u = ld(bb, i);
        if (self) {
          const float2 v = ld(D3 ? (ny - bb) & (ny - 1) : 0, ((1 << logn) - i) & ((1 << logn) - 1));
          u = make_float2(__fmul_rn(0.5f, __fadd_rn(u.x, v.x)),
                          __fmul_rn(0.5f, __fsub_rn(u.y, v.y)));
        }
        return u;
      };
      if (mode == 2) {
        for (int i = tm.rank; i < ns; i += tm.size) {
          const int kz = i >> a.logny, ky = i & (ny - 1);
          const float2 sc = update(i, D3 ? fhat(ky, kz) : fhat(0, i));
          a.state[base + i * rstride] = st[i];
          a.work[base + i * rstride] = sc;
        }
        tm.sync();
        return;
      }
      with_radix(odd, [&](auto r) {
        fft_pass<decltype(r)::value, true, D3, true>(
            logn, 0, logb, tw, tm,
            [&](int bb, int i) { return update(value(bb, i), fhat(bb, i)); }, sm);
      });
    }
  } else {
    with_radix(odd, [&](auto r) {
      fft_pass<decltype(r)::value, true, D3, true>(
          logn, 0, logb, tw, tm,
          [&](int bb, int i) {
            const float2 p = st[D3 ? i * ny + bb : i];
            return make_float2(__fmul_rn(p.x, a.inv_n), __fmul_rn(p.y, a.inv_n));
          },
          sm);
    });
  }
  turn();
  int s = odd;
  for (; s < logn - (direct ? 3 : 0); s += 3) {
    fft_pass<8, true, D3, false>(logn, s, logb, tw, tm, ld, sm);
    turn();
  }
  if (direct) {
    fft_pass<8, true, false, false>(logn, s, 0, tw, tm, ld, [&](int, int i, float2 v) {
      Wg[(int64_t)i * a.wr] = v;
    });
    tm.sync();
    return;
  }
  if (D3) {
    with_radix(odd_y, [&](auto r) {
      fft_pass<decltype(r)::value, true, D3, true>(a.logny, 0, a.lognz, twy, tm, ld_y, sm_y);
    });
    turn();
    for (int sy = odd_y; sy < a.logny; sy += 3) {
      fft_pass<8, true, D3, false>(a.logny, sy, a.lognz, twy, tm, ld_y, sm_y);
      turn();
    }
  }
  for (int i = tm.rank; i < ns; i += tm.size)
    Wg[(int64_t)i * a.wr] = in[D3 ? i + (i >> a.logny) : padded(i)];
  tm.sync();
}

template <int MODEL, bool D3>
__device__ __forceinline__ void spectral_fused(const FusedArgs& a) {
  extern __shared__ float2 smem[];
  unsigned int target = 0;
  const Team rt = make_team(a.row_team), ct = make_team(a.col_team);
  const int rteams = blockDim.x / a.row_team, cteams = blockDim.x / a.col_team;
  const int ns = a.ny * a.nz;
  float2* twx = smem;
  float2* twy = twx + padded_size(a.nx);
  float2* twz = twy + padded_size(a.ny);
  // the two phases' FFT buffers share one region: rteams x rbuf or cteams x cbuf
  float2* bufs = twz + padded_size(a.nz);
  const int bregion = rteams * a.rbuf > cteams * a.cbuf ? rteams * a.rbuf : cteams * a.cbuf;
  float2* res = bufs + bregion;  // cteams x cpt x (psi_hat, table) slabs
  float2* rb = bufs + (size_t)rt.index * a.rbuf;
  float2* rb2 = rb + padded_size(a.nx);
  float2* cb = bufs + (size_t)ct.index * a.cbuf;
  float2* st = res + (size_t)ct.index * a.cpt * 2 * ns;
  float2* tb = st + (size_t)a.cpt * ns;
  for (int j = threadIdx.x; j < a.nx; j += blockDim.x) twx[padded(j)] = a.twx[j];
  for (int j = threadIdx.x; j < a.ny; j += blockDim.x) twy[padded(j)] = a.twy[j];
  for (int j = threadIdx.x; j < a.nz; j += blockDim.x) twz[padded(j)] = a.twz[j];
  const int gct = blockIdx.x * cteams + ct.index, nct = gridDim.x * cteams;
  // row tasks: the CTAs' warps (or warp-wide teams) in turn, so that a phase with fewer tasks
  // than teams spreads them over every CTA; a warp of narrower teams takes consecutive tasks
  const int rtpw = a.row_team < 32 ? 32 / a.row_team : 1;  // row teams per warp
  const int nrt = gridDim.x * rteams;
  const int rt0 = ((rt.index / rtpw) * gridDim.x + blockIdx.x) * rtpw;  // this warp's first
  const int col_tasks = a.nf * a.nxh;
  const int row_tasks = MODEL == PF_MODEL_C ? a.nrows : (a.nrows >> 1);
  for (int i = 0; i < a.cpt; ++i) {
    const int t = gct + i * nct;
    if (t >= col_tasks) break;
    const int64_t base = (t / a.nxh) * a.cs + t % a.nxh;
    for (int k = ct.rank; k < ns; k += ct.size) {
      st[(size_t)i * ns + k] = a.state[base + (int64_t)k * a.nxh];
      tb[(size_t)i * ns + k] = a.table[base + (int64_t)k * a.nxh];
    }
  }
  __syncthreads();
  for (int i = 0; i < a.cpt; ++i) {
    const int t = gct + i * nct;
    if (t >= col_tasks) break;
    slab_task<D3>(a, t / a.nxh, t % a.nxh, 0, st + (size_t)i * ns, tb + (size_t)i * ns, cb,
              cb + a.cbuf / 2, twy, twz, ct);
  }
  if (!grid_barrier(a.bar, target, a.budget)) return;
  for (int64_t step = 0; step < a.steps; ++step) {
    // teams narrower than a warp take their rounds together: the warp's first team decides
    // the trip count, and a team past the last task runs without touching W
    for (int t0 = rt0; t0 < row_tasks; t0 += nrt) {
      const int t = t0 + rt.index % rtpw;
      const bool valid = t < row_tasks;
      if (MODEL == PF_MODEL_C) row_task<MODEL>(a, 0, t, 1, t, valid, rb, rb2, twx, rt);
      else row_task<MODEL>(a, 0, 2 * t, 0, 2 * t + 1, valid, rb, rb2, twx, rt);
    }
    if (!grid_barrier(a.bar, target, a.budget)) return;
    const int mode = step + 1 == a.steps ? 2 : 1;
    for (int i = 0; i < a.cpt; ++i) {
      const int t = gct + i * nct;
      if (t >= col_tasks) break;
      slab_task<D3>(a, t / a.nxh, t % a.nxh, mode, st + (size_t)i * ns, tb + (size_t)i * ns, cb,
                cb + a.cbuf / 2, twy, twz, ct);
    }
    if (mode == 1 && !grid_barrier(a.bar, target, a.budget)) return;
  }
}

template <int MODEL, bool D3>
__global__ void __launch_bounds__(kThreads) spectral_fused_kernel(FusedArgs a) {
  spectral_fused<MODEL, D3>(a);
  grid_leave(a.bar);
}

bool is_pow2(int64_t n) { return n > 0 && (n & (n - 1)) == 0; }

int ilog2(int64_t n) {
  int l = 0;
  while ((int64_t)1 << l < n) ++l;
  return l;
}

// Launch shape. For each CTA width (128 .. 1024 threads): per phase, the team size that gives
// one radix-8 butterfly per thread and pass, halved while that phase's tasks would need more
// than one round on the SMs; CTAs for the larger phase (at most one per SM, which keeps the
// grid barrier short); the slabs each slab team owns; and the shared memory that takes. The
// width whose phases need the fewest butterfly rounds per thread (task rounds times
// butterflies per thread) wins, the narrowest on a tie: warps that share an SM's issue slots
// lengthen every task's dependent chain. Where a width's slab teams do not fit, they are
// widened (fewer per CTA) until they do.
struct FusedShape {
  int threads, blocks, row_team, col_team, cpt, rbuf, cbuf;
  int rounds;  // the longer phase's task rounds per team
  size_t smem;
};

// Teams wider than a warp synchronise on named barriers 1 .. 15 (0 is the CTA's), so a CTA
// holds at most 15 of them: a 64-thread team in a 1024-thread CTA becomes a warp.
int team_for(int64_t n, int64_t tasks, int sms, int threads, int min_size = 32) {
  int64_t size = n / 8;
  if (size < min_size) size = min_size;
  if (size > threads) size = threads;
  while (size > 32 && (tasks + threads / size - 1) / (threads / size) > sms) size >>= 1;
  while (size > 32 && threads / size > 15) size >>= 1;
  return (int)size;
}

struct FusedDims {
  int64_t nx, ny, nz;
};

FusedDims fused_dims(const pf_spectral_s* s) {
  if (s->dim == 3) return {s->d[2], s->d[1], s->d[0]};
  return {s->d[1], s->d[0], 1};
}

FusedShape fused_shape_for(const pf_spectral_s* s, int sms, int threads, int col_team = 0) {
  const FusedDims d = fused_dims(s);
  const int64_t ns = d.ny * d.nz;  // values of a slab, and x-rows of a field
  const int64_t col_tasks = s->nf * (d.nx / 2 + 1);
  const int64_t row_tasks = s->model == PF_MODEL_C ? ns : ns / 2;
  FusedShape f{};
  f.threads = threads;
  // 3D: 8- or 16-lane teams for short rows (measured: Model C 64^3 22.2 -> 18.3 us per step);
  // 2D grids keep warp-wide teams (64^2 and 128^2 measured 0.6-1.0 us faster with them)
  f.row_team = team_for(d.nx, row_tasks, sms, f.threads, s->dim == 3 ? 8 : 32);
  f.col_team = col_team > 0 ? col_team : team_for(ns, col_tasks, sms, f.threads);
  const int64_t rteams = f.threads / f.row_team, cteams = f.threads / f.col_team;
  // row work counted in warps (a narrower team shares its warp's issue slots), so that short
  // rows still spread over as many SMs as warp-wide teams would
  const int64_t rwarps = f.threads / 32;
  const int64_t rtasks_per_warp = f.row_team < 32 ? 32 / f.row_team : 1;
  int64_t blocks = (row_tasks + rwarps * rtasks_per_warp - 1) / (rwarps * rtasks_per_warp);
  if (f.row_team < 32) blocks = std::max(blocks, (row_tasks + rwarps - 1) / rwarps);
  const int64_t cblocks = (col_tasks + cteams - 1) / cteams;
  if (cblocks > blocks) blocks = cblocks;
  if (blocks > sms) blocks = sms;
  f.blocks = (int)blocks;
  f.cpt = (int)((col_tasks + blocks * cteams - 1) / (blocks * cteams));
  // two padded rows; the second first takes both half spectra, nx + 2 values
  f.rbuf = (int)(padded_size(d.nx) + std::max(d.nx + 2, padded_size(d.nx)));
  // two padded slabs (rows of ny + 1) or, in 2D, columns
  f.cbuf = (int)(2 * (s->dim == 3 ? d.nz * (d.ny + 1) : padded_size(d.ny)));
  const int64_t region = std::max(rteams * f.rbuf, cteams * f.cbuf);
  const int64_t tables = padded_size(d.nx) + padded_size(d.ny) + padded_size(d.nz);
  f.smem = sizeof(float2) * (size_t)(tables + region + cteams * f.cpt * 2 * ns);
  const int64_t rrounds = (row_tasks + blocks * rteams - 1) / (blocks * rteams);
  const int64_t rb = (d.nx / 8 + f.row_team - 1) / f.row_team;  // butterflies per thread
  const int64_t cb = (ns / 8 + f.col_team - 1) / f.col_team;
  f.rounds = (int)(rrounds * std::max<int64_t>(rb, 1) + f.cpt * std::max<int64_t>(cb, 1));
  return f;
}

FusedShape fused_shape(const pf_spectral_s* s, int sms) {
  int optin = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    optin = 0;
  }
  FusedShape best = fused_shape_for(s, sms, 128);
  for (int threads : {256, 512, kThreads}) {
    FusedShape f = fused_shape_for(s, sms, threads);
    // wider slab teams (fewer per CTA) where their buffers and resident slabs do not fit
    while (f.smem > (size_t)optin && f.col_team < threads)
      f = fused_shape_for(s, sms, threads, 2 * f.col_team);
    const bool fits = f.smem <= (size_t)optin, best_fits = best.smem <= (size_t)optin;
    if ((fits && (!best_fits || f.rounds < best.rounds)) || (!fits && !best_fits && f.smem < best.smem))
      best = f;
  }
  return best;
}

template <int MODEL>
const void* fused_kernel_ptr(bool d3) {
  return d3 ? reinterpret_cast<const void*>(&spectral_fused_kernel<MODEL, true>)
            : reinterpret_cast<const void*>(&spectral_fused_kernel<MODEL, false>);
}

const void* kernel_for(int model, bool d3) {
  if (model == PF_MODEL_AC) return fused_kernel_ptr<PF_MODEL_AC>(d3);
  if (model == PF_MODEL_CH) return fused_kernel_ptr<PF_MODEL_CH>(d3);
  return fused_kernel_ptr<PF_MODEL_C>(d3);
}

unsigned long long g_attr_mask[6] = {};

}  // namespace

int device_limits(int* sms, int* smem_optin) {
  int dev = 0;
  PF_CUDA_TRY(cudaGetDevice(&dev));
  PF_CUDA_TRY(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
  PF_CUDA_TRY(cudaDeviceGetAttribute(smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  return PF_OK;
}

bool spectral_fused_supported(const pf_spectral_s* s) {
  const FusedDims d = fused_dims(s);
  if (!(is_pow2(d.nx) && is_pow2(d.ny) && is_pow2(d.nz) && d.nx >= 4 && d.nx <= kMaxSide &&
        d.ny >= 2 && d.ny <= kMaxSide && d.nz <= kMaxSide))
    return false;
  if (s->dim == 3 && d.nz < 2) return false;
  int sms = 0, optin = 0;
  if (device_limits(&sms, &optin) != PF_OK) return false;
  return fused_shape(s, sms).smem <= (size_t)optin;
}

int spectral_fused_prepare(pf_spectral_s* s) {
  if (s->fused_blocks > 0) return PF_OK;
  if (!spectral_fused_supported(s))
    return invalid("the fused engine takes power-of-two sides (nx in [4, 1024]) whose (y, z) "
                   "slab fits in a CTA's shared memory");
  const FusedDims d = fused_dims(s);
  std::vector<float2> tw((size_t)(d.nx + d.ny + d.nz));
  size_t o = 0;
  for (int64_t n : {d.nx, d.ny, d.nz}) {
    for (int64_t j = 0; j < n; ++j) {
      const double t = -2.0 * 3.141592653589793 * (double)j / (double)n;
      tw[o++] = make_float2((float)std::cos(t), (float)std::sin(t));
    }
  }
  cudaError_t e = cudaMalloc(&s->twiddle, sizeof(float2) * tw.size());
  if (e == cudaSuccess) e = cudaMalloc(&s->d_bar, 4 * sizeof(unsigned int));
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error("fused spectral engine: out of device memory");
    return PF_ERR_OOM;
  }
  PF_CUDA_TRY(cudaMemcpyAsync(s->twiddle, tw.data(), sizeof(float2) * tw.size(),
                              cudaMemcpyHostToDevice, s->stream));
  PF_CUDA_TRY(cudaMemsetAsync(s->d_bar, 0, 4 * sizeof(unsigned int), s->stream));
  PF_CUDA_TRY(cudaStreamSynchronize(s->stream));
  int sms = 0, optin = 0;
  if (int rc = device_limits(&sms, &optin)) return rc;
  const FusedShape f = fused_shape(s, sms);
  const bool d3 = s->dim == 3;
  const int mi = 2 * (s->model == PF_MODEL_AC ? 0 : (s->model == PF_MODEL_CH ? 1 : 2)) + d3;
  const void* kern = kernel_for(s->model, d3);
  int dev = 0;
  PF_CUDA_TRY(cudaGetDevice(&dev));
  // the limit is per kernel and device: set it once, to the device's opt-in maximum
  if (dev >= 64 || !(g_attr_mask[mi] & (1ull << dev))) {
    PF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    if (dev < 64) g_attr_mask[mi] |= 1ull << dev;
  }
  int per_sm = 0;
  PF_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, f.threads, f.smem));
  if (per_sm < 1) return invalid("fused spectral engine: the kernel does not fit on an SM");
  s->fused_blocks = f.blocks;
  s->fused_threads = f.threads;
  s->fused_row_team = f.row_team;
  s->fused_col_team = f.col_team;
  s->fused_cpt = f.cpt;
  s->fused_rbuf = f.rbuf;
  s->fused_cbuf = f.cbuf;
  s->fused_smem = f.smem;
  return PF_OK;
}

int spectral_fused_run(pf_spectral_s* s, int64_t n_steps) {
  if (n_steps <= 0) return PF_OK;
  if (int rc = spectral_fused_prepare(s)) return rc;
  const FusedDims d = fused_dims(s);
  FusedArgs a{};
  a.state = s->spec;
  a.W = s->spec + s->nf * s->cs;
  a.work = s->work;
  a.table = s->table;
  a.twx = s->twiddle;
  a.twy = s->twiddle + d.nx;
  a.twz = s->twiddle + d.nx + d.ny;
  a.nx = (int)d.nx;
  a.ny = (int)d.ny;
  a.nz = (int)d.nz;
  a.nxh = (int)(d.nx / 2 + 1);
  a.lognx = ilog2(d.nx);
  a.logny = ilog2(d.ny);
  a.lognz = ilog2(d.nz);
  a.nf = s->nf;
  a.nrows = (int)(d.ny * d.nz);
  a.wr = s->dim == 3 ? 1 : a.nxh;
  a.wk = s->dim == 3 ? a.nrows : 1;
  a.rbuf = s->fused_rbuf;
  a.cbuf = s->fused_cbuf;
  a.row_team = s->fused_row_team;
  a.col_team = s->fused_col_team;
  a.cpt = s->fused_cpt;
  a.cs = s->cs;
  a.inv_n = (float)(1.0 / (double)s->nsite);
  a.k = nl_coeffs(s);
  a.steps = n_steps;
  a.bar = s->d_bar;
  a.budget = kWaitBudgetCycles;
  void* args[] = {&a};
  PF_CUDA_TRY(cudaLaunchCooperativeKernel(kernel_for(s->model, s->dim == 3), dim3(s->fused_blocks),
                                          dim3(s->fused_threads), args, s->fused_smem,
                                          s->stream));
  return PF_OK;
}

int spectral_fused_check(pf_spectral_s* s) {
  if (s->d_bar == nullptr) return PF_OK;
  unsigned int flag = 0;
  PF_CUDA_TRY(cudaMemcpyAsync(&flag, s->d_bar + 2, sizeof(unsigned int), cudaMemcpyDeviceToHost,
                              s->stream));
  PF_CUDA_TRY(cudaStreamSynchronize(s->stream));
  if (flag != 0) {
    PF_CUDA_TRY(cudaMemsetAsync(s->d_bar, 0, 4 * sizeof(unsigned int), s->stream));
    set_error("a grid barrier wait of the fused spectral engine ran out; the state is invalid");
    return PF_ERR_TIMEOUT;
  }
  return PF_OK;
}

void spectral_fused_release(pf_spectral_s* s) {
  cudaFree(s->twiddle);
  cudaFree(s->d_bar);
  s->twiddle = nullptr;
  s->d_bar = nullptr;
}

}  // namespace pf
