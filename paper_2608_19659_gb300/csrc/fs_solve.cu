// Allocation solver (Section 3, Eqs. 1-5; tier 2 of the objective) and the
// quantile table, for sm_103a.
//
// One warp (or, for a few realisations, one block of eight) solves one
// realisation (a capacity and a tail value per cell):
//   1. rows: for every (class i, TP index j) the best SLO-feasible bin
//      (largest capacity, then lowest bin; Eq. 5 gates l <= L_i) -> C_ij;
//   2. t*: the largest threshold t whose cheapest per-class covers fit in G,
//      the thresholds being the rows' positive fulfilments f(n, C_ij), n =
//      1..floor(G/tau_j). The covers of t change only just above a threshold,
//      so t fits exactly when the smallest threshold at or above it does, and
//      t* is found without a list of thresholds: a search over the bit
//      patterns of t, each probe one group of lanes (a row per lane, shuffles
//      for the per-class minimum over the four TP lanes and the sum). The
//      probes also count the thresholds below them, so the search ends when
//      one threshold is left between the last t that fits and the first that
//      does not: t* is the smallest threshold at or above the former;
//   3. choice at t*: per class the cheapest cover, ties to the lower TP.
// For a fixed (TP, n) a larger capacity never lowers f, so the best bin of
// each row is the option the tie rule (larger capacity, then lower bin) picks.
// Critical floors (tier 1 of the objective): options of a critical class i
// below delta_i are none, so it covers max(t, delta_i) at threshold t. Step 3
// also prices every critical class's cheapest cover of its floor: the floors
// are met when those fit in G together; with t* = 0 and the floors met, that
// cover is the class's allocation.
// What bounds it: the dependent chain of about a dozen probes (latency for a
// few realisations, issue slots for a batch). Measured, against a 256-thread block
// per realisation that lists and sorts the thresholds: see launch_solve.
#include <cuda_runtime.h>

#include <cstddef>

#include "fs_internal.cuh"
#include "fs_rows.cuh"

namespace fs {

__global__ void k_qtable(float* qn, int Q) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= Q) return;
  // Inverse CDF of the symmetric triangular law on [0, 1] at u = (k + 1/2) / Q:
  // 2x^2 = u below 1/2, 1 - 2(1-x)^2 = u above.
  const float u = __fdiv_rn(__fadd_rn(__int2float_rn(k), 0.5f), __int2float_rn(Q));
  float x;
  if (u < 0.5f) {
    x = __fsqrt_rn(__fmul_rn(u, 0.5f));
  } else {
    x = __fsub_rn(1.0f, __fsqrt_rn(__fmul_rn(__fsub_rn(1.0f, u), 0.5f)));
  }
  qn[k] = x;
}

// One realisation's state shared by its lanes (NW > 1, or more than 32 rows).
struct SolveSmem {
  float C[256], lam[FS_MAX_CLASSES], rl[FS_MAX_CLASSES], dl[FS_MAX_CLASSES];
  int bin[256];
  int4 end[16];  // per warp, alternate rounds: the search's ends and their sums
  fs_allocation out;
};

constexpr uint32_t kAboveOne = 0x3F800001u;  // the float pattern after 1

// Covers of threshold t by one aligned group of gsz lanes, lane gl taking rows
// gl, gl + gsz, ...: the classes' cheapest covers summed (an uncovered class
// counted as 2^24: a cost is at most G <= 32767, 64 of them stay below 2^21)
// and `below`, the rows' first covering counts summed (M + 1 for a row that
// does not cover t), which differ between two thresholds by the number of
// option fulfilments in between. Every lane of the group gets both.
template <bool FL>
__device__ __forceinline__ int group_cover(float t, const SolveSmem& sm, const Dims& d, int gl, int gsz, int* below) {
  int packed = 0, u = 0;
  for (int base = 0; base < d.K4; base += gsz) {
    const int rho = base + gl, j = rho & 3, i = rho >> 2;
    int cost = kCostInf;
    if (rho < d.K4) {
      const int n = min_replicas(FL ? fmaxf(t, sm.dl[i]) : t, sm.C[rho], sm.lam[i], sm.rl[i], rep_capf(d, j));
      u += n ? n : rep_cap(d, j) + 1;
      if (n) cost = n << j;
    }
    cost = min(cost, __shfl_xor_sync(0xffffffffu, cost, 1));
    cost = min(cost, __shfl_xor_sync(0xffffffffu, cost, 2));
    int v = rho < d.K4 ? (cost >= kCostInf ? (1 << 24) : cost) : 0;
    for (int off = 4; off < gsz; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    packed += v;
  }
  for (int off = 1; off < gsz; off <<= 1) u += __shfl_xor_sync(0xffffffffu, u, off);
  *below = u;
  return packed;
}

// A lane's row when every row has a lane of its own (at most 32 rows).
struct OneRow {
  float C, lam, rl, dl, M;
  int j;
  bool in, fast;  // a row; in Markstein's range
};

// min_replicas on it (the range test made once).
__device__ __forceinline__ int row_cover(const OneRow& r, float t) {
  if (!(r.M >= 1.0f)) return 0;
  if (!r.fast) return min_replicas_ieee(t, r.C, r.lam, r.M);
  return min_replicas_fast(t, r.C, r.lam, r.rl, r.M);
}

template <bool FL>
__device__ __forceinline__ int one_cover(float t, const OneRow& r, int gsz, int* below) {
  int cost = kCostInf, u = 0;
  if (r.in) {
    const int n = row_cover(r, FL ? fmaxf(t, r.dl) : t);
    u = n ? n : (int)r.M + 1;
    if (n) cost = n << r.j;
  }
  cost = min(cost, __shfl_xor_sync(0xffffffffu, cost, 1));
  cost = min(cost, __shfl_xor_sync(0xffffffffu, cost, 2));
  u += __shfl_xor_sync(0xffffffffu, u, 1);
  u += __shfl_xor_sync(0xffffffffu, u, 2);
  int v = r.in ? (cost >= kCostInf ? (1 << 24) : cost) : 0;
  for (int off = 4; off < gsz; off <<= 1) {
    v += __shfl_xor_sync(0xffffffffu, v, off);
    u += __shfl_xor_sync(0xffffffffu, u, off);
  }
  *below = u;
  return v;
}

// Estimates of t* (patterns in [1, that of 1], aim_lo <= aim_hi) that start the
// search; they only place the first probes. With replica counts real numbers,
// class i takes t min_j tau_j lambda_i / C_ij GPUs, so t* is at most G over the
// sum of those (aim_hi, with a margin for rounding); rounding the counts up adds
// at most the chosen TP degrees (aim_lo). One warp; every lane gets both.
__device__ __forceinline__ void search_aims(const SolveSmem& sm, const Dims& d, int lane, uint32_t& aim_lo,
                                            uint32_t& aim_hi) {
  float rate = 0.0f, extra = 0.0f;
  for (int base = 0; base < d.K4; base += 32) {
    const int rho = base + lane;
    const float inf = __int_as_float(0x7f800000);
    float c = inf;
    if (rho < d.K4 && sm.C[rho] > 0.0f) c = __fdividef(sm.lam[rho >> 2] * (float)(1 << (rho & 3)), sm.C[rho]);
    float m = fminf(c, __shfl_xor_sync(0xffffffffu, c, 1));
    m = fminf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    const uint32_t who = (__ballot_sync(0xffffffffu, c == m) >> (lane & 28)) & 15u;  // the class's cheapest degrees
    if ((lane & 3) == 0 && rho < d.K4) {
      rate += m;
      extra += (float)(1 << (__ffs(who | 8u) - 1));
    }
  }
  for (int o = 16; o; o >>= 1) {
    rate += __shfl_xor_sync(0xffffffffu, rate, o);
    extra += __shfl_xor_sync(0xffffffffu, extra, o);
  }
  const float G = (float)d.G;
  const float top = fminf(1.0f, __fdividef(G, rate) * 1.0001f);  // (0 when some class has no option)
  const float bottom = top * fmaxf(0.25f, 1.0f - __fdividef(extra, G));
  aim_hi = min(max(__float_as_uint(top), 1u), 0x3F800000u);
  aim_lo = min(max(__float_as_uint(bottom), 1u), aim_hi);
}

// FL: some class is critical (the model has floors). NW warps per realisation:
// 1 (four realisations a block) for batches, 8 for a few realisations, whose
// latency counts: the rows and the probes are then spread over the warps.
template <bool FL, int NW>
__global__ void __launch_bounds__(NW == 1 ? 128 : 32 * NW) k_solve(Set set, int n_real, const float* cap_x,
                                                                   const float* tail_x, fs_allocation* out_x,
                                                                   HostOut host) {
  constexpr int kPerBlock = NW == 1 ? 4 : 1;  // realisations per block
  __shared__ SolveSmem smem[kPerBlock];
  const Dims& d = set.d;  // kernel-parameter space: no local copy
  const int lane = threadIdx.x & 31, warp = NW == 1 ? 0 : (int)threadIdx.x >> 5;
  const int slot = NW == 1 ? (int)threadIdx.x >> 5 : 0, ltid = warp * 32 + lane;
  SolveSmem& sm = smem[slot];
  const int r = (int)blockIdx.x * kPerBlock + slot;
  pdl_wait();
  pdl_trigger();
  if (r >= n_real) return;
  auto sync = [] {
    if (NW == 1) __syncwarp();
    else __syncthreads();
  };

  const float* cap;
  const float* tail;
  fs_allocation* out;
  if (cap_x) {
    cap = cap_x + (size_t)r * d.cells;
    tail = tail_x + (size_t)r * d.cells;
    out = out_x + r;
  } else {
    const int p = r >> 1, sigma = r & 1;
    if (set.skip && set.skip[p] >= 0) return;
    const float* bp = set.bounds + (size_t)p * 4 * d.cells;
    cap = bp + (size_t)(sigma ? CAP_HI : CAP_LO) * d.cells;
    tail = bp + (size_t)(sigma ? TAIL_LO : TAIL_HI) * d.cells;
    out = set.base + r;
  }

  // 1. rows
  for (int i = ltid; i < d.K; i += 32 * NW) {
    const float lam = set.lam[i];
    sm.lam[i] = lam;
    sm.rl[i] = __frcp_rn(lam);
    if (FL) sm.dl[i] = set.slo[d.K + i];
  }
  best_rows<NW>(d, cap, tail, set.slo, warp, lane, sm.C, sm.bin);
  sync();

  // 2. t*: bit patterns [lo, hi) of nonnegative floats (ordered like the
  // values), lo feasible and hi not; every group probes one point a round.
  int lgs = 2;
  while ((1 << lgs) < d.K4 && lgs < 5) ++lgs;
  const int gsz = 1 << lgs, gl = lane & (gsz - 1);
  const int ng = NW << (5 - lgs), g = (warp << (5 - lgs)) + (lane >> lgs);
  // Ends not probed yet: 0 fits (nothing is bought) and the pattern above 1 does
  // not (no fulfilment exceeds 1); their sums never let the search end.
  uint32_t lo = 0u, hi = kAboveOne;
  int ulo = -(1 << 28), uhi = 1 << 28;
  uint32_t aim_lo, aim_hi;  // where the first probes go
  search_aims(sm, d, lane, aim_lo, aim_hi);
  const bool one = d.K4 <= gsz;  // (the same for every lane)
  OneRow mine;
  mine.in = gl < d.K4;
  mine.j = gl & 3;
  mine.C = mine.in ? sm.C[gl] : 0.0f;
  mine.lam = mine.in ? sm.lam[gl >> 2] : 1.0f;
  mine.rl = mine.in ? sm.rl[gl >> 2] : 1.0f;
  mine.dl = FL && mine.in ? sm.dl[gl >> 2] : 0.0f;
  mine.M = rep_capf(d, mine.j);
  mine.fast = row_in_range(mine.C, mine.lam);
  int oct = 22;  // an unprobed lower end is approached by points 2^oct patterns apart, growing
  for (int rd = 0; uhi - ulo > 1 && hi - lo > 1; ++rd) {
    uint32_t pt;
    if (rd == 0 || (ng == 1 && rd == 1 && lo == 0u)) {
      // between the two estimates; one group probes the upper, then the lower
      if (ng == 1) pt = rd == 0 ? aim_hi : min(aim_lo, hi - 1u);
      else pt = aim_lo + (uint32_t)(((uint64_t)g * (aim_hi - aim_lo)) / (uint32_t)(ng - 1));
    } else {
      const uint32_t span = hi - lo;
      const uint64_t reach = lo ? (uint64_t)span : min((uint64_t)span, (uint64_t)(ng + 1) << min(oct, 30));
      const uint32_t q = max(1u, (uint32_t)(reach / (uint32_t)(ng + 1)));
      const uint64_t off = (uint64_t)(g + 1) * q;
      pt = off < span ? hi - (uint32_t)off : lo;  // (past the lower end: that end again)
      oct += 2;
    }
    int u;
    const float tp = __uint_as_float(max(pt, 1u));
    const int cost = one ? one_cover<FL>(tp, mine, gsz, &u) : group_cover<FL>(tp, sm, d, gl, gsz, &u);
    const bool known = pt <= lo;
    const bool fits = known || cost <= d.G;
    // the largest point that fits and the smallest that does not
    uint32_t nlo = __reduce_max_sync(0xffffffffu, fits && !known ? pt : lo);
    uint32_t nhi = __reduce_min_sync(0xffffffffu, fits ? hi : min(pt, hi));
    const uint32_t bl = __ballot_sync(0xffffffffu, fits && !known && pt == nlo);
    const uint32_t bh = __ballot_sync(0xffffffffu, !fits && pt == nhi);
    int nul = __shfl_sync(0xffffffffu, u, bl ? __ffs(bl) - 1 : 0);
    int nuh = __shfl_sync(0xffffffffu, u, bh ? __ffs(bh) - 1 : 0);
    if (!bl) nul = ulo;
    if (!bh) nuh = uhi;
    if (NW > 1) {
      // (the arrays alternate between rounds: one barrier a round)
      const int w = (rd & 1) * NW;
      if (lane == 0) sm.end[w + warp] = make_int4((int)nlo, (int)nhi, nul, nuh);
      __syncthreads();
      const int4 e = sm.end[w + (lane & (NW - 1))];
      nlo = __reduce_max_sync(0xffffffffu, (uint32_t)e.x);
      nhi = __reduce_min_sync(0xffffffffu, (uint32_t)e.y);
      nul = __shfl_sync(0xffffffffu, e.z, __ffs(__ballot_sync(0xffffffffu, (uint32_t)e.x == nlo)) - 1);
      nuh = __shfl_sync(0xffffffffu, e.w, __ffs(__ballot_sync(0xffffffffu, (uint32_t)e.y == nhi)) - 1);
    }
    lo = nlo;
    hi = nhi;
    ulo = nul;
    uhi = nuh;
  }

  // 3. t* is the smallest option fulfilment at or above lo, and the covers at
  // t* are those at lo: per class the cheapest over its four TP lanes, lower
  // TP on ties; the same for the floor of a critical class. One warp.
  if (warp != 0) return;
  float tv = 2.0f;  // the smallest option fulfilment at or above lo
  int total = 0, ftotal = 0;
  bool fmiss = false;
  uint64_t mask = 0;
  fs_allocation& so = sm.out;
  const float t_lo = __uint_as_float(lo);
  if (FL) {  // the critical classes' floors
    for (int base = 0; base < d.K4; base += 32) {
      const int rho = base + lane, i = rho >> 2;
      int keyf = 0x7fffffff;
      const float dl = rho < d.K4 ? sm.dl[i] : 0.0f;
      if (dl > 0.0f) {
        const int n = min_replicas(dl, sm.C[rho], sm.lam[i], sm.rl[i], rep_capf(d, rho & 3));
        if (n) keyf = n << (rho & 3);
      }
      keyf = min(keyf, __shfl_xor_sync(0xffffffffu, keyf, 1));
      keyf = min(keyf, __shfl_xor_sync(0xffffffffu, keyf, 2));
      const bool head = (lane & 3) == 0 && dl > 0.0f;
      fmiss = fmiss || __any_sync(0xffffffffu, head && keyf == 0x7fffffff);
      ftotal += __reduce_add_sync(0xffffffffu, head && keyf != 0x7fffffff ? keyf : 0);
    }
  }
  const bool met = !FL || (!fmiss && ftotal <= d.G);
  // an empty allocation, then the model's classes
  uint64_t* words = reinterpret_cast<uint64_t*>(&so);
  constexpr int kBin0 = (int)(offsetof(fs_allocation, bin) / 8), kBin1 = (int)(offsetof(fs_allocation, replicas) / 8);
  for (int w = lane; w < (int)(sizeof(fs_allocation) / 8); w += 32) words[w] = w >= kBin0 && w < kBin1 ? ~0ull : 0ull;
  __syncwarp();
  for (int base = 0; base < d.K4; base += 32) {
    const int rho = base + lane, i = rho >> 2, j = rho & 3;
    int key = 0x7fffffff;
    bool has = false;
    if (rho < d.K4) {
      const float dl = FL ? sm.dl[i] : 0.0f;
      has = sm.bin[rho] >= 0;
      // at t* = 0 tier 1 alone: the critical classes' floors, when they can be met
      const float t = lo ? (FL ? fmaxf(t_lo, dl) : t_lo) : (met ? dl : 0.0f);
      const int n = t > 0.0f ? min_replicas(t, sm.C[rho], sm.lam[i], sm.rl[i], rep_capf(d, j)) : 0;
      if (n) {
        key = ((n << j) << 2) | j;
        tv = fminf(tv, fulfil_r((float)n, sm.C[rho], sm.lam[i], sm.rl[i]));
      }
    }
    key = min(key, __shfl_xor_sync(0xffffffffu, key, 1));
    key = min(key, __shfl_xor_sync(0xffffffffu, key, 2));
    const uint32_t bal = __ballot_sync(0xffffffffu, has);
    mask |= (uint64_t)__ballot_sync(0xffffffffu, lane < 8 && ((bal >> (4 * (lane & 7))) & 15u)) << (base >> 2);
    const bool head = j == 0 && key != 0x7fffffff;
    total += __reduce_add_sync(0xffffffffu, head ? key >> 2 : 0);
    if (head) {
      const int bj = key & 3, bn = (key >> 2) >> bj;
      so.tp[i] = (int8_t)(1 << bj);
      so.bin[i] = (int16_t)sm.bin[4 * i + bj];
      so.replicas[i] = (int16_t)bn;
      so.fulfil[i] = fulfil_r((float)bn, sm.C[4 * i + bj], sm.lam[i], sm.rl[i]);
    }
  }
  const float tstar = lo ? __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(tv))) : 0.0f;
  if (lane == 0) {
    so.t_star = tstar;
    so.total_gpus = total;
    so.has_option_mask = mask;
    so.ok = tstar > 0.0f ? 1 : 0;
    so.floors_met = met ? 1 : 0;
    so.goodput = 0.0;  // tier 3 is filled by the lexicographic solve
  }
  __syncwarp();
  uint64_t* dst = reinterpret_cast<uint64_t*>(out);
  uint64_t* dst2 = host.alloc ? reinterpret_cast<uint64_t*>(host.alloc + r) : nullptr;
  for (int w = lane; w < (int)(sizeof(fs_allocation) / 8); w += 32) {
    dst[w] = words[w];
    if (dst2) dst2[w] = words[w];
  }
  if (host.status && lane == 0) host.status[r] = *set.status;
}

// Watchdog self-test: wait on a barrier phase that nothing completes; the
// bounded wait gives up, records the timeout and the kernel returns.
__global__ void k_watchdog(uint32_t* status, uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) mbar_init(&bar, 1);
  __syncthreads();
  const bool ok = mbar_wait(&bar, 0u, limit_ns);
  if (!ok && threadIdx.x == 0) atomicOr(status, ST_TIMEOUT);
}

cudaError_t launch_watchdog(uint32_t* status, uint64_t limit_ns, cudaStream_t s) {
  note_launch();
  k_watchdog<<<1, 32, 0, s>>>(status, limit_ns);
  return cudaGetLastError();
}

cudaError_t launch_qtable(float* qn, int Q, cudaStream_t s) {
  note_launch();
  k_qtable<<<(Q + 255) / 256, 256, 0, s>>>(qn, Q);
  return cudaGetLastError();
}

// Measured (one GB300, calls in a row): 4096 realisations of the four-class,
// 64-GPU grid 71.7 -> 13.7 us (issue slots 56 % busy; the inputs' 8.4 MB take 1.3
// us at the memory's rate).
cudaError_t launch_solve(const Set& set, int n, const float* cap_x, const float* tail_x,
                         fs_allocation* out, LaunchCache& lc, cudaStream_t s, HostOut host) {
  if (n <= 0) return cudaSuccess;
  if (n <= kSolveWideMax)
    return launch_pdl(lc.floors ? k_solve<true, 8> : k_solve<false, 8>, dim3(n), dim3(256), 0, s, set, n, cap_x, tail_x,
                      out, host);
  return launch_pdl(lc.floors ? k_solve<true, 1> : k_solve<false, 1>, dim3((n + 3) / 4), dim3(128), 0, s, set, n, cap_x,
                    tail_x, out, host);
}

}  // namespace fs
