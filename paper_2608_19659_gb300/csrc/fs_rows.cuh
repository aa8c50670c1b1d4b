// Best SLO-feasible bin of every (class, TP) row of one realisation, shared by
// the allocation solver (fs_solve.cu) and the thresholds (fs_thresh.cu).
#pragma once

#include "fs_internal.cuh"

namespace fs {

// Rows over the 32 NW threads (t = warp, lane): lpr lanes per row (a power of
// two, at most 32), the row's bins dealt to them in chunks of four (16-byte
// loads) where the rows start on 16-byte boundaries, else one by one. A lane of
// a one-warp solve of 16 rows so takes half a row in a few loads; the eight warps
// of a latency-bound one take a chunk per thread. sC[rho] = the row's largest
// SLO-feasible capacity (0: none, -0 as +0), sB[rho] = the lowest bin that has it
// (-1: none). The caller synchronises before it reads them.
template <int NW>
__device__ __forceinline__ void best_rows(const Dims& d, const float* cap, const float* tail, const float* slo,
                                          int warp, int lane, float* sC, int* sB) {
  int lpr = 32;
  while (lpr > 1 && (lpr >> 1) * d.K4 >= 32 * NW) lpr >>= 1;
  const int sub = lane & (lpr - 1), rows = 32 / lpr;  // rows per warp and pass
  const bool vec = (d.B & 3) == 0 && ((reinterpret_cast<uintptr_t>(cap) | reinterpret_cast<uintptr_t>(tail)) & 15u) == 0;
  for (int first = 0; first < d.K4; first += NW * rows) {
    const int rho = first + warp * rows + lane / lpr;
    // key: capacity bits + 1 of a feasible bin (nonnegative floats order like
    // their bit patterns), 0 for none
    uint32_t key = 0u;
    int bin = 0x7fffffff;
    auto take = [&](int b, float c, float t, float L) {
      const uint32_t kb = t <= L ? __float_as_uint(__fadd_rn(c, 0.0f)) + 1u : 0u;
      if (kb > key) {  // (bins in ascending order: the first of equals stays)
        key = kb;
        bin = b;
      }
    };
    if (rho < d.K4) {
      const float L = slo[rho >> 2];
      const float* rc = cap + (size_t)rho * d.B;
      const float* rt = tail + (size_t)rho * d.B;
      if (vec) {
#pragma unroll 4
        for (int b = 4 * sub; b < d.B; b += 4 * lpr) {
          const float4 c = *reinterpret_cast<const float4*>(rc + b), t = *reinterpret_cast<const float4*>(rt + b);
          take(b, c.x, t.x, L);
          take(b + 1, c.y, t.y, L);
          take(b + 2, c.z, t.z, L);
          take(b + 3, c.w, t.w, L);
        }
      } else {
#pragma unroll 4
        for (int b = sub; b < d.B; b += lpr) take(b, rc[b], rt[b], L);
      }
    }
    uint32_t top = key;
    for (int o = lpr >> 1; o; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    int bb = key == top ? bin : 0x7fffffff;
    for (int o = lpr >> 1; o; o >>= 1) bb = min(bb, __shfl_xor_sync(0xffffffffu, bb, o));
    if (sub == 0 && rho < d.K4) {
      sC[rho] = top ? __uint_as_float(top - 1u) : 0.0f;
      sB[rho] = top ? bb : -1;
    }
  }
}

}  // namespace fs
