// Thresholds, rows and row tables of the base realisations A- and A+
// (Section 4.1), the scoring calls' view of the threshold solver, for sm_103a.
//
// The solver's threshold set Theta holds the positive fulfilments
// f(n, C_rho), n = 1..floor(G/tau) (cut at the first n with f = 1; a critical
// class's from its floor up) of every row rho = (class, TP degree), C_rho the
// row's best SLO-feasible capacity. Within a row they increase with n, so for
// any threshold t the number of a row's values below t is its cheapest cover
// of t less its first count n0. One evaluation of every row's cheapest cover
// of t = f(n, C_rho) therefore gives all that a scoring call needs of t:
//   - its rank in the sorted set (the sum of the rows' counts below t; equal
//     values are ordered by row, then by n), so no sort is needed;
//   - each class's cheapest cover, so whether t fits in G, and t* as the
//     largest threshold that does;
//   - for every row rho the word of the row table at that rank: bits 0-14 the
//     replicas rho may use once the other classes cover t (0 if one cannot),
//     bit 15 set if another row of rho's class covers t within that budget.
// The thresholds are independent of each other: blocks over them, a group of
// pow2 >= 4K lanes (at most 32) per threshold, a row per lane.
//
// What bounds it: dependent latencies (the cells' loads, a row's two covers,
// one cover per row and threshold); every block finds the rows for itself (a
// few kB from L2) rather than wait for another to hand them over. One block per
// realisation that sorts the values and probes them takes 19 us on the
// eight-class, 256-GPU grid against 7 (launch_thresh).
#include <cuda_runtime.h>

#include <algorithm>

#include "fs_internal.cuh"
#include "fs_rows.cuh"

namespace fs {

// FL: some class is critical (the model has floors).
template <bool FL>
__global__ void __launch_bounds__(kThreshThreads) k_thresh(Set set, int late) {
  const Dims& d = set.d;  // kernel-parameter space: no local copy
  const int r = blockIdx.x, p = r >> 1, sigma = r & 1;
  const int part = blockIdx.y, n_part = (int)gridDim.y;  // (a replay's realisations may pass 65535: along x)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kThreshThreads / 32;
  __shared__ float sC[256];
  __shared__ int sB[256], sN0[256], sOff[257];  // first count, offset of the row's values
  __shared__ float sLam[FS_MAX_CLASSES], sRl[FS_MAX_CLASSES], sDl[FS_MAX_CLASSES];
  __shared__ int sCover[kWarps][256];  // covers of one threshold (more than 32 rows)
  __shared__ uint32_t s_best;
  // late 1, 2: what is read here was complete before this kernel could start, and
  // nothing that may still run reads what is written here (launch_thresh), so the
  // wait for the previous kernel comes after the work: the last call's scenarios
  // overlap this call's thresholds and (2) the part of the preparation before its
  // wait, whose records are not those the scenarios read.
  if (late == 0) pdl_wait();
  if (late != 1) pdl_trigger();
  if (set.skip && set.skip[p] >= 0) return;
  const float* bp = set.bounds + (size_t)p * 4 * d.cells;
  const float* cap = bp + (size_t)(sigma ? CAP_HI : CAP_LO) * d.cells;
  const float* tail = bp + (size_t)(sigma ? TAIL_LO : TAIL_HI) * d.cells;

  for (int i = tid; i < d.K; i += kThreshThreads) {
    const float lam = set.lam[i];
    sLam[i] = lam;
    sRl[i] = __frcp_rn(lam);
    if (FL) sDl[i] = set.slo[d.K + i];
  }
  if (tid == 0) s_best = 0u;
  best_rows<kWarps>(d, cap, tail, set.slo, warp, lane, sC, sB);
  __syncthreads();
  // each row's values f(n), n = n0..len: the first at or above the class's
  // floor and positive, the last the first full one (or the row's cap)
  for (int rho = tid; rho < d.K4; rho += kThreshThreads) {
    const int i = rho >> 2, j = rho & 3, M = rep_cap(d, j);
    const float C = sC[rho], lam = sLam[i], rl = sRl[i], Mf = rep_capf(d, j);
    int n0 = 0, len = 0;
    if (sB[rho] >= 0 && M >= 1) {
      // (no floor, and every fulfilment positive: the first is that of one replica)
      const float lo_f = FL ? fmaxf(sDl[i], __int_as_float(1)) : __int_as_float(1);
      n0 = C > 0.0f && row_in_range(C, lam) && !(FL && sDl[i] > 0.0f) ? 1 : min_replicas(lo_f, C, lam, rl, Mf);
      const int ns = min_replicas(1.0f, C, lam, rl, Mf);
      if (n0) len = ns ? ns : M;
    }
    sN0[rho] = n0;
    sOff[rho + 1] = n0 ? len - n0 + 1 : 0;
  }
  __syncthreads();
  if (warp == 0) {  // inclusive scan of the row counts
    int carry = 0;
    for (int base = 0; base < d.K4; base += 32) {
      const int rho = base + lane;
      int incl = rho < d.K4 ? sOff[rho + 1] : 0;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (rho < d.K4) sOff[rho + 1] = carry + incl;
      carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) sOff[0] = 0;
  }
  __syncthreads();
  int total = sOff[d.K4];
  if (total > d.theta_cap) {  // cannot happen: a row holds at most floor(G/tau) values
    if (tid == 0) atomicOr(set.status, ST_THETA);
    total = d.theta_cap;
  }
  const size_t ps = (size_t)p * 2 + sigma;
  float* th = set.theta + ps * d.theta_cap;
  uint16_t* rt = d.K4 * total <= set.rt_cap ? set.rtab + ps * set.rt_cap : nullptr;
  if (part == 0) {
    for (int rho = tid; rho < d.K4; rho += kThreshThreads) {
      set.rowC[ps * d.K4 + rho] = sC[rho];
      set.rowB[ps * d.K4 + rho] = sB[rho];
    }
    if (tid == 0) set.ntheta[ps] = total;
    if (set.gp_span && tid < d.K) {
      set.gp_span[sigma * d.K + tid] = 0x7fffffff;
      set.gp_span[(2 + sigma) * d.K + tid] = -1;
    }
  }

  int lgs = 2;
  while ((1 << lgs) < d.K4 && lgs < 5) ++lgs;
  const int gsz = 1 << lgs, gl = lane & (gsz - 1), per = 32 >> lgs;  // thresholds of a warp at a time
  const int stride = n_part * kWarps * per;
  uint32_t best = 0u;  // the largest feasible threshold's bits
  for (int x0 = (part * kWarps + warp) * per; x0 < total; x0 += stride) {
    const int x = min(x0 + (lane >> lgs), total - 1);  // (a spare group repeats the last one)
    int row = 0, hi = d.K4 - 1;
    while (row < hi) {
      const int mid = (row + hi + 1) >> 1;
      if (sOff[mid] <= x) row = mid; else hi = mid - 1;
    }
    const float v = fulfil_r((float)(sN0[row] + (x - sOff[row])), sC[row], sLam[row >> 2], sRl[row >> 2]);
    int rank = 0, packed = 0, cost = kCostInf;
    for (int base = 0; base < d.K4; base += gsz) {
      const int rho = base + gl;
      cost = kCostInf;
      if (rho < d.K4) {
        const int i = rho >> 2, n0 = sN0[rho], cnt = sOff[rho + 1] - sOff[rho];
        const float C = sC[rho], lam = sLam[i], rl = sRl[i];
        const int n = min_replicas(FL ? fmaxf(v, sDl[i]) : v, C, lam, rl, rep_capf(d, rho & 3));
        if (n) cost = n << (rho & 3);
        if (rho == row) {
          rank += x - sOff[row];
        } else {
          int u = n ? n - n0 : cnt;  // the row's values below v
          if (n && rho < row)        // and, for an earlier row, equal ones
            while (u < cnt && fulfil_r((float)(n0 + u), C, lam, rl) == v) ++u;
          rank += u;
        }
      }
      if (d.K4 > 32) sCover[warp][rho & 255] = cost;
      int cm = min(cost, __shfl_xor_sync(0xffffffffu, cost, 1));
      cm = min(cm, __shfl_xor_sync(0xffffffffu, cm, 2));
      // uncovered classes are counted above bit 24 (a cost is at most G <=
      // 32767: 64 of them stay below 2^21)
      int s = rho < d.K4 ? (cm >= kCostInf ? (1 << 24) : cm) : 0;
      for (int o = 4; o < gsz; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      packed += s;
    }
    for (int o = 1; o < gsz; o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (packed <= d.G) best = max(best, __float_as_uint(v));
    const bool live = (uint32_t)rank < (uint32_t)total;  // (always, for checked inputs)
    if (gl == 0 && live) th[rank] = v;
    if (rt) {
      for (int base = 0; base < d.K4; base += gsz) {
        const int rho = base + gl, j = rho & 3;
        const int c = d.K4 > 32 ? sCover[warp][rho & 255] : cost;
        const int c1 = __shfl_xor_sync(0xffffffffu, c, 1), c2 = __shfl_xor_sync(0xffffffffu, c, 2),
                  c3 = __shfl_xor_sync(0xffffffffu, c, 3);
        const int other = min(c1, min(c2, c3)), cm = min(c, other);
        const int rest = packed - (cm >= kCostInf ? (1 << 24) : cm);
        const int A = (rest >> 24) ? -1 : d.G - rest;
        const int m = A >= (1 << j) ? min(A >> j, rep_cap(d, j)) : 0;
        if (rho < d.K4 && live)
          rt[(size_t)rank * d.K4 + rho] = (uint16_t)((uint32_t)m | (other < kCostInf && other <= A ? kRowOther : 0u));
      }
    }
  }
  if (set.tpart) {
    best = __reduce_max_sync(0xffffffffu, best);
    if (lane == 0) atomicMax(&s_best, best);
    __syncthreads();
    if (tid == 0) set.tpart[sigma * n_part + part] = __uint_as_float(s_best);
  }
  if (late) {
    pdl_wait();
    if (late == 1) pdl_trigger();
  }
}

// Measured (one GB300, calls in a row): the eight-class, 256-GPU grid (about 1300
// thresholds a realisation, 55 blocks each) 19.2 -> 7.3 us; with its tables, which
// one block left out above 8192 words, so that the preparation searched for each
// candidate, the preparation of 1024 candidates 60.6 -> 14 us: 1024 x 16 x 16384 scenarios
// 270 -> 206 us, 1024 x 8 x 60 116 -> 51 us; four classes, 64 GPUs 51 -> 45 us.
//
// late: for a scoring call n on the model's own device bounds, of at least one
// candidate, after another such call. What may still run when it starts is
// call n - 1's scenarios and reduction: that reduction let this kernel start, and
// was itself let start by the scenarios, after call n - 1's preparation and so
// (each waits for its predecessor) its thresholds had finished, which had waited
// for call n - 2's reduction. So
//   - the bounds are only written by copies, which are ordered after the calls
//     queued before them (a full barrier in the stream, flush_bounds on another);
//   - thresholds, rows and tables have no reader left: the preparation of call n -
//     1 was the last (a dump's scenarios read rows: not late after one; the goodput
//     stage and the replay are synchronous);
//   - the parts of t*, the sums and the counters, which call n - 1 still uses,
//     alternate between two sets, call n - 2's being free;
//   - late 2: so do the records, between two buffers (both calls' fit the second).
//     Late 1: one of them keeps its records in the first buffer whatever its turn,
//     so the preparation starts only after the wait.
// A call without candidates has no preparation and scenarios to hand that on: it
// and the call after it wait first. Calls are counted as they are queued; those that a stream capture
// records are counted by themselves (sequence_of).
cudaError_t launch_thresh(Set& set, int floors, int th_bound, cudaStream_t s, int late) {
  const Dims& d = set.d;
  const int bound = th_bound > 0 ? std::min(th_bound, d.theta_cap) : d.theta_cap;
  int gsz = 4;
  while (gsz < d.K4 && gsz < 32) gsz <<= 1;
  // about two thresholds per group: enough blocks that the evaluations' latency
  // is paid twice, few enough that the rows each block finds for itself stay cheap
  const int per_block = 2 * (kThreshThreads / gsz);
  const int nb = set.P > 1 ? 1 : std::max(1, std::min(kThreshBlocks, (bound + per_block - 1) / per_block));
  set.n_tpart = set.tpart ? nb : 0;
  return launch_pdl(floors ? k_thresh<true> : k_thresh<false>, dim3(2 * set.P, nb), dim3(kThreshThreads), 0, s, set,
                    late);
}

}  // namespace fs
