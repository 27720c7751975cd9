// Staging of a tile's rows into shared memory with 16-byte cp.async copies, for the kernels
// that take four consecutive sites per thread: rows y0-1 .. y0+ht-2 of columns x0-4 ..
// x0+ws-5 of every field (a row of ws floats; ws - 8 output columns plus four halo columns a
// side, so each row's interior starts 16-byte aligned in shared memory and in the field).
#pragma once

#include "pf_internal.h"
#include "pf_tma.cuh"

namespace pf {

// Copy the rows of every field at plane offset zoff into dst (rows ws floats apart, fields pl
// floats apart): a 16-byte copy where a group of four columns, wrapped, is four consecutive ones
// on a 16-byte boundary, else four periodic 4-byte copies. Issues the copies and returns: the caller commits or waits.
template <int NF>
__device__ __forceinline__ void stage_rows4(const FieldPtrs& in, const Geom& g, int x0, int y0,
                                            int64_t zoff, int ws, int ht, int pl, float* dst,
                                            int nthreads) {
  const int ch4 = ws / 4;
  for (int i = threadIdx.x; i < ht * ch4; i += nthreads) {
    const int r = i / ch4, j = i - r * ch4;
    const int gy = wrap_index(y0 - 1 + r, g.ny);
    const int gx = wrap_index(x0 - 4 + 4 * j, g.nx);
    const int64_t row = zoff + (int64_t)gy * g.pitch;
    float* d = dst + r * ws + 4 * j;
    if (gx + 3 < g.nx && gx % 4 == 0) {
#pragma unroll
      for (int f = 0; f < NF; ++f) cp_async16(d + f * pl, in.f[f] + row + gx);
    } else {
#pragma unroll
      for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          cp_async4(d + f * pl + c, in.f[f] + row + wrap_index(gx + c, g.nx));
    }
  }
}

}  // namespace pf
