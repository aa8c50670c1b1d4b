// Tiers 3 and 4 of the lexicographic objective (Section 3) and the goodput
// gap (Fig. 4a; the third stage of Section 4.2's stage-wise gap), for sm_103a.
//
// Section 3 orders the objective: (1) critical floors, (2) max min_i r_i,
// (3) maximise total served goodput, (4) minimise fragmentation. The
// threshold solver (k_solve) settles tiers 1-2 (t*, floors met). Among the
// allocations that keep them optimal -- every class at r_i >= max(t*,
// delta_i) when t* > 0; at t* = 0 the critical classes at their floors and
// the others free; nothing at all when the floors cannot be met -- tier 3
// takes the most goodput, sum_i x_i with x_i = min(lambda_i, n c) (Eqs. 2
// and 4), each class's term in fixed point rint(x_i 2^20) so that sums are
// exact; tier 4 the fewest GPUs in use, then class by class the threshold
// solver's tie rules (no replicas first, lower TP, fewer replicas; the row's
// best bin carries the larger-capacity and lower-bin rules).
//
// For a fixed (TP, n) a larger capacity never lowers goodput or fulfilment,
// so one row per (class, TP) -- its best SLO-feasible bin -- carries every
// useful option, and replica counts past the first that serves the whole
// demand add GPUs and no goodput. The optimum is a programme over classes and
// GPUs left: S_i(g) = the best (goodput, -GPUs) of classes i..K-1 within g
// GPUs, S_K = 0, S_i(g) = max over class i's options (cost <= g) of their
// goodput plus S_{i+1}(g - cost).
//
// k_solve_lex: one warp (a block of 16 for a few) per realisation, threads over
//   g, one class per step, over the GPUs that the classes' cheapest options
//   leave; then a walk over the classes, lanes over a class's options, taking
//   the preferred option that keeps the optimum.
// k_score_goodput: the goodput stage of the Monte-Carlo score. Within a
//   segment (candidate e, outcome o) a scenario's goodput gap
//   |GP(A+') - GP(A-')| depends on its draw only through (c_y position,
//   tail gate), as its t* does: the block tabulates those values (a warp per
//   entry: each realisation's row capacity and t* as the scorer computes
//   them, then the programme over the classes with row r patched, lanes over
//   g), then draws every scenario's position and sums the entries.
// k_finalize_goodput: E[Gamma_gp,t+1 | e] = sum 2^-20 / (O S) / sum lambda,
//   the score Gamma_gp,t - E and the argmax (same order as the max-min stage).
#include <cuda_runtime.h>

#include "fs_finalize.cuh"
#include "fs_internal.cuh"
#include "fs_rows.cuh"
#include "fs_sample.cuh"

namespace fs {

// A class's served goodput in 2^-20 req/s: rint(min(lambda, fl(n c)) 2^20)
// (2^20 x is exact; the conversion rounds to nearest, ties to even).
__device__ __forceinline__ long long goodput_fx(float n, float c, float lam) {
  const float served = __fmul_rn(n, c);
  const float x = served < lam ? served : lam;
  return __float2ll_rn(__fmul_rn(x, 0x1p20f));
}

// One programme cell: goodput (-1: unreachable) and GPUs in use.
struct LexCell {
  long long gp;
  int gpus;
};

__device__ __forceinline__ bool lex_better(long long gpa, int gpusa, long long gpb, int gpusb) {
  return gpa > gpb || (gpa == gpb && gpusa < gpusb);
}

// --------------------------------------------------------------------------- tiers 3-4

// A programme value: goodput first, then fewest GPUs. Packed into one 64-bit
// word (goodput 2^16 less GPUs: both parts add, and more goodput or the same
// with fewer GPUs is the larger word) while goodput stays below 2^46, which the
// host knows from sum lambda <= 2^26; the two-word form otherwise.
template <bool PACK>
struct Lex;
template <>
struct Lex<true> {
  using T = long long;
  static __device__ __forceinline__ T make(long long gp, int gpus) { return (gp << 16) - gpus; }
  static __device__ __forceinline__ T add(T a, T b) { return a + b; }
  static __device__ __forceinline__ bool better(T a, T b) { return a > b; }
  static __device__ __forceinline__ bool same(T a, T b) { return a == b; }
  static __device__ __forceinline__ long long gp(T a) { return (a + 0xFFFF) >> 16; }
  static __device__ __forceinline__ T worst() { return -0x7FFFFFFFFFFFFFFFLL - 1; }
  static __device__ __forceinline__ T shfl_xor(T a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
};
template <>
struct Lex<false> {
  using T = LexCell;
  static __device__ __forceinline__ T make(long long gp, int gpus) { return LexCell{gp, gpus}; }
  static __device__ __forceinline__ T add(T a, T b) { return LexCell{a.gp + b.gp, a.gpus + b.gpus}; }
  static __device__ __forceinline__ bool better(T a, T b) { return lex_better(a.gp, a.gpus, b.gp, b.gpus); }
  static __device__ __forceinline__ bool same(T a, T b) { return a.gp == b.gp && a.gpus == b.gpus; }
  static __device__ __forceinline__ long long gp(T a) { return a.gp; }
  static __device__ __forceinline__ T worst() { return LexCell{-1, 0x7fffffff}; }
  static __device__ __forceinline__ T shfl_xor(T a, int o) {
    return LexCell{__shfl_xor_sync(0xffffffffu, a.gp, o), __shfl_xor_sync(0xffffffffu, a.gpus, o)};
  }
};

// First n in [1, M] with fl(n c) >= lambda (the whole demand served: further
// replicas add GPUs and no goodput), else M + 1; fl(n c) is nondecreasing in n.
// In range the answer is within one of ceil(lambda / c) and is reached from an
// estimate by steps of one, as in min_replicas; else by bisection.
__device__ __forceinline__ int first_full(float c, float lam, int M) {
  if (row_in_range(c, lam) && c > 0.0f) {
    const float Mf = (float)M;
    float n = fminf(fmaxf(ceilf(__fdividef(lam, c)), 1.0f), Mf);
    while (n > 1.0f && !(__fmul_rn(n - 1.0f, c) < lam)) n -= 1.0f;
    while (n <= Mf && __fmul_rn(n, c) < lam) n += 1.0f;
    return (int)n;
  }
  int a = 1, b = M + 1;
  while (a < b) {
    const int mid = (a + b) >> 1;
    if (!(__fmul_rn((float)mid, c) < lam)) b = mid;
    else a = mid + 1;
  }
  return a;
}

// Class i's options on row (i, tau = 2^j) at capacity C are the replica
// counts n in [1, M = G / tau] whose fulfilment reaches T (all of them when
// T = 0), up to the first that serves the whole demand. Both ends are monotone
// in n, so the options are one range [lo, hi]. lo = 0: none.
__device__ __forceinline__ void row_range(float C, bool ok, int M, float T, float lam, float rl, int& lo, int& hi) {
  lo = hi = 0;
  if (!ok || M < 1) return;
  lo = T > 0.0f ? min_replicas(T, C, lam, rl, (float)M) : 1;
  if (lo) hi = min(M, max(lo, first_full(C, lam, M)));
}

__device__ __forceinline__ float class_threshold(float t, float dl) { return t > 0.0f ? fmaxf(t, dl) : dl; }

// Dynamic shared memory of k_solve_lex per realisation: the rows (best
// capacity, its bin, its option range), the classes (cheapest option), one
// class's option values (opt of them; more are evaluated where they are used)
// and the programme's cells, when they fit (cells of them; else in scratch).
struct LexSmem {
  size_t rows, cls, opt, cells, total;
  int n_opt, n_cells;
};

__host__ __device__ inline LexSmem lex_smem(int K, int G, bool pack, int most_opt, size_t most_cell_bytes) {
  LexSmem m{};
  const size_t cell = pack ? 8 : sizeof(LexCell);
  auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
  m.n_opt = G + (G >> 1) + (G >> 2) + (G >> 3);
  if (m.n_opt > most_opt) m.n_opt = most_opt;
  const size_t all = (size_t)(K + 1) * (G + 1);
  m.n_cells = all * cell <= most_cell_bytes ? (int)all : 0;
  m.rows = 0;
  m.cls = up(m.rows + 16 * (size_t)(4 * K));
  m.opt = up(m.cls + 8 * (size_t)K);
  m.cells = up(m.opt + cell * (size_t)m.n_opt);
  m.total = up(m.cells + cell * (size_t)m.n_cells);
  return m;
}

constexpr int kLexWideWarps = 16;       // warps of a realisation when there are few
constexpr int kLexOptWarp = 512;        // option values kept per class (one warp, kLexWideWarps)
constexpr int kLexOptWide = 2048;
constexpr size_t kLexCellsWarp = 12 * 1024;   // bytes of programme cells in shared memory
constexpr size_t kLexCellsWide = 128 * 1024;

// NW warps per realisation: 1 (four realisations a block) for batches, 16 for
// a few realisations, whose latency counts.
//
// The programme runs over the GPUs left beyond what must be kept: class i's
// cheapest option costs m_i (0 when it may stay empty), so of G only slack = G -
// sum m_i can be spent freely, and S_i is needed (and reachable) for h = 0..slack
// GPUs above the cheapest options of classes i..K-1. An option of cost c takes e
// = c - m_i of them. Where t* is tight the slack is a few GPUs and a class's
// options with e <= slack are few; the table over all of [0, G] that stood here
// before, with a division per option and cell, took 66 us on 1000 realisations of
// the four-class, 64-GPU grid and 180 us on two of the eight-class, 256-GPU one
// (its last step, the walk forward, one thread's); measured now: see
// launch_solve_lex.
template <bool PACK, int NW>
__global__ void __launch_bounds__(NW == 1 ? 128 : 32 * NW) k_solve_lex(Set set, int n_real, const float* cap_x,
                                                                       const float* tail_x, fs_allocation* out_x,
                                                                       unsigned char* scratch, int r0, LexSmem lay) {
  using L = Lex<PACK>;
  using V = typename L::T;
  constexpr int kPerBlock = NW == 1 ? 4 : 1, kThreads = 32 * NW;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_slack[kPerBlock];
  __shared__ V s_top[NW];
  const Dims& d = set.d;
  const int lane = threadIdx.x & 31, warp = NW == 1 ? 0 : (int)threadIdx.x >> 5;
  const int slot = NW == 1 ? (int)threadIdx.x >> 5 : 0, tid = warp * 32 + lane;
  const int rel = (int)blockIdx.x * kPerBlock + slot, r = r0 + rel;
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
    const float* bp = set.bounds + (size_t)p * 4 * d.cells;
    cap = bp + (size_t)(sigma ? CAP_HI : CAP_LO) * d.cells;
    tail = bp + (size_t)(sigma ? TAIL_LO : TAIL_HI) * d.cells;
    out = set.base + r;
  }
  const float tstar = out->t_star;
  if (!out->floors_met) {  // tier 1 cannot hold: nothing is allocated (k_solve wrote the empty allocation)
    if (tid == 0) out->goodput = 0.0;
    return;
  }
  unsigned char* mem = smraw + (size_t)slot * lay.total;
  float* sC = reinterpret_cast<float*>(mem + lay.rows);
  int* sB = reinterpret_cast<int*>(sC + d.K4);
  int* sLo = sB + d.K4;
  int* sHi = sLo + d.K4;
  int* sMin = reinterpret_cast<int*>(mem + lay.cls);     // cheapest option's GPUs
  int* sEmpty = sMin + d.K;                               // 1: the class may stay empty
  V* sOpt = reinterpret_cast<V*>(mem + lay.opt);
  V* S = lay.n_cells ? reinterpret_cast<V*>(mem + lay.cells)
                     : reinterpret_cast<V*>(scratch) + (size_t)rel * (size_t)(d.K + 1) * (d.G + 1);
  best_rows<NW>(d, cap, tail, set.slo, warp, lane, sC, sB);
  sync();
  for (int rho = tid; rho < d.K4; rho += kThreads) {
    const int i = rho >> 2;
    const float lam = set.lam[i], T = class_threshold(tstar, set.slo[d.K + i]);
    int lo, hi;
    row_range(sC[rho], sB[rho] >= 0, rep_cap(d, rho & 3), T, lam, __frcp_rn(lam), lo, hi);
    sLo[rho] = lo;
    sHi[rho] = hi;
  }
  sync();
  if (warp == 0) {
    int sum = 0;
    for (int i = lane; i < d.K; i += 32) {
      const bool empty = !(tstar > 0.0f) && !(set.slo[d.K + i] > 0.0f);
      int m = empty ? 0 : kCostInf;
      for (int j = 0; j < kT && !empty; ++j)
        if (sLo[4 * i + j]) m = min(m, sLo[4 * i + j] << j);
      sMin[i] = m;
      sEmpty[i] = empty;
      sum += min(m, 1 << 24);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) s_slack[slot] = d.G - sum;
  }
  sync();
  const int slack = s_slack[slot], H = slack + 1;
  if (slack < 0) {  // cannot happen: t* and the floors were found feasible
    if (tid == 0) {
      atomicOr(set.status, ST_THETA);
      out->goodput = 0.0;
    }
    return;
  }
  // class i's options with e <= slack in the order of preference (no replicas,
  // lower TP, fewer replicas): x = 0.. over `empty`, then row j's lo..top
  struct Opts {
    int empty, e1, e2, e3, total, lo[kT], m;
  };
  auto options = [&](int i) {
    Opts o;
    o.empty = sEmpty[i];
    o.m = sMin[i];
    int cnt[kT];
#pragma unroll
    for (int j = 0; j < kT; ++j) {
      o.lo[j] = sLo[4 * i + j];
      cnt[j] = o.lo[j] ? max(0, min(sHi[4 * i + j], (slack + o.m) >> j) - o.lo[j] + 1) : 0;
    }
    o.e1 = o.empty + cnt[0];
    o.e2 = o.e1 + cnt[1];
    o.e3 = o.e2 + cnt[2];
    o.total = o.e3 + cnt[3];
    return o;
  };
  auto pick = [&](const Opts& o, int x, int& j, int& n) {
    if (x < o.empty) { j = 0; n = 0; }
    else if (x < o.e1) { j = 0; n = o.lo[0] + (x - o.empty); }
    else if (x < o.e2) { j = 1; n = o.lo[1] + (x - o.e1); }
    else if (x < o.e3) { j = 2; n = o.lo[2] + (x - o.e2); }
    else { j = 3; n = o.lo[3] + (x - o.e3); }
  };
  auto value = [&](int i, int j, int n) {
    return L::make(n ? goodput_fx((float)n, sC[4 * i + j], set.lam[i]) : 0, n << j);
  };
  for (int h = tid; h < H; h += kThreads) S[(size_t)d.K * H + h] = L::make(0, 0);
  sync();
  for (int i = d.K - 1; i >= 1; --i) {
    const V* nxt = S + (size_t)(i + 1) * H;
    V* cur = S + (size_t)i * H;
    const Opts o = options(i);
    const int kept = min(o.total, lay.n_opt);
    for (int x = tid; x < kept; x += kThreads) {
      int j, n;
      pick(o, x, j, n);
      sOpt[x] = value(i, j, n);
    }
    sync();
    for (int h = tid; h < H; h += kThreads) {
      V best = L::worst();
      if (o.empty) best = nxt[h];
      int x = o.empty;
#pragma unroll
      for (int j = 0; j < kT; ++j) {
        const int end = j == 0 ? o.e1 : j == 1 ? o.e2 : j == 2 ? o.e3 : o.total;
        int e = (o.lo[j] << j) - o.m;
        for (; x < end && e <= h; ++x, e += 1 << j) {
          const V v = L::add(x < kept ? sOpt[x] : value(i, j, (e + o.m) >> j), nxt[h - e]);
          if (L::better(v, best)) best = v;
        }
        x = end;
      }
      cur[h] = best;
    }
    sync();
  }
  // the first class: its best over all threads
  V top = L::worst();
  {
    const Opts o = options(0);
    for (int x = tid; x < o.total; x += kThreads) {
      int j, n;
      pick(o, x, j, n);
      const int e = (n << j) - o.m;
      if (e <= slack) {
        const V v = L::add(value(0, j, n), S[(size_t)H + slack - e]);
        if (L::better(v, top)) top = v;
      }
    }
    for (int off = 16; off; off >>= 1) {
      const V v = L::shfl_xor(top, off);
      if (L::better(v, top)) top = v;
    }
    if (NW > 1) {
      if (lane == 0) s_top[warp] = top;
      __syncthreads();
      if (warp != 0) return;
      top = s_top[lane & (NW - 1)];
      for (int off = 16; off; off >>= 1) {
        const V v = L::shfl_xor(top, off);
        if (L::better(v, top)) top = v;
      }
    }
  }
  // forward: class by class the first option, in the order of preference, that
  // keeps the optimum (lanes over the options). One warp.
  int left = slack, total = 0;
  V target = top;
  for (int i = 0; i < d.K; ++i) {
    const V* nxt = S + (size_t)(i + 1) * H;
    const Opts o = options(i);
    int j = 0, n = 0, e = 0;
    bool found = false;
    for (int x0 = 0; x0 < o.total && !found; x0 += 32) {
      const int x = x0 + lane;
      bool hit = false;
      if (x < o.total) {
        pick(o, x, j, n);
        e = (n << j) - o.m;
        hit = e <= left && L::same(L::add(value(i, j, n), nxt[left - e]), target);
      }
      const uint32_t bal = __ballot_sync(0xffffffffu, hit);
      if (bal) {
        const int src = __ffs(bal) - 1;
        j = __shfl_sync(0xffffffffu, j, src);
        n = __shfl_sync(0xffffffffu, n, src);
        e = __shfl_sync(0xffffffffu, e, src);
        found = true;
      }
    }
    if (lane == 0) {
      const bool some = found && n > 0;
      out->tp[i] = (int8_t)(some ? 1 << j : 0);
      out->bin[i] = (int16_t)(some ? sB[4 * i + j] : -1);
      out->replicas[i] = (int16_t)(some ? n : 0);
      out->fulfil[i] = some ? fulfil((float)n, sC[4 * i + j], set.lam[i]) : 0.0f;
    }
    if (found) {
      total += n << j;
      left -= e;
      target = nxt[left];
    }
  }
  if (lane == 0) {
    out->total_gpus = total;
    out->goodput = (double)L::gp(top) * 0x1p-20;
  }
}

// --------------------------------------------------------------------------- goodput stage

// rint(min(lambda, fl(n c)) 2^20), the same value as goodput_fx, for
// 0 <= min(...) <= 2^20 (the host requires sum lambda <= 2^20): x 2^-20 is
// exact there (or its rint is 0 either way), and fixed40 rounds its 2^40
// multiple to nearest, ties to even, without a float-to-int64 conversion.
__device__ __forceinline__ long long goodput_fx20(float n, float c, float lam) {
  const float served = __fmul_rn(n, c);
  const float x = served < lam ? served : lam;
  return (long long)fixed40(__fmul_rn(x, 0x1p-20f));
}

// The options of one row in a realisation: replica counts [lo, hi] (lo = 0:
// none) at capacity C, and the thresholds T in (a, b] for which they stay so.
struct RowOpt {
  float C;
  int lo, hi;
  float a, b;
};

// The row's range and the interval of thresholds that gives the same lo (and
// so the same hi): fulfil(lo - 1) < T <= fulfil(lo) for lo >= 1 (no lower end
// at lo = 1), T > fulfil(M) for lo = 0 (fulfil is nondecreasing in n).
__device__ __forceinline__ RowOpt row_opt(float C, bool ok, int M, float T, float lam, float rl) {
  RowOpt r{C, 0, 0, -INFINITY, INFINITY};
  row_range(C, ok, M, T, lam, rl, r.lo, r.hi);
  if (!ok || M < 1) return r;
  if (r.lo == 0) {
    r.a = fulfil((float)M, C, lam);
  } else {
    r.b = fulfil((float)r.lo, C, lam);
    if (r.lo > 1) r.a = fulfil((float)(r.lo - 1), C, lam);
  }
  return r;
}

// The best tier-3 goodput of every class but `skip` within g GPUs, for g in
// [0, G], at tiers 1-2 value t (-1: the floors of those classes cannot be
// met within g), by one warp: the programme over the classes (no replicas,
// when class i may stay empty: T_i = 0 and no floor; else one range of
// replica counts on each of its rows) with lanes over g. Also leaves in opt
// every row's range at t (those of `skip` for warp_best_with; row `fixed`,
// whose capacity varies, with no interval). dpa, dpb: the warp's two arrays
// of G + 1 cells. Returns the array that holds the result.
template <bool FL>
__device__ const long long* warp_other(const Dims& d, const float* sCs, const int* sOk, const float* sLam,
                                       const float* sRl, const float* sDl, int skip, int fixed, float t,
                                       RowOpt* opt, long long* dpa, long long* dpb) {
  const int lane = threadIdx.x & 31;
  __syncwarp();  // the previous result and ranges are no longer read
  for (int rho = lane; rho < d.K4; rho += 32) {
    const int i = rho >> 2;
    RowOpt r = row_opt(sCs[rho], sOk[rho] != 0, d.G >> (rho & 3), class_threshold(t, FL ? sDl[i] : 0.0f),
                       sLam[i], sRl[i]);
    if (rho == fixed) r.a = -INFINITY, r.b = INFINITY;
    opt[rho] = r;
  }
  for (int g = lane; g <= d.G; g += 32) dpa[g] = 0;
  __syncwarp();
  long long* cur = dpa;  // S_{i+1}
  long long* nxt = dpb;
  for (int i = d.K - 1; i >= 0; --i) {
    if (i == skip) continue;
    const float dl = FL ? sDl[i] : 0.0f;
    const bool may_empty = !(t > 0.0f) && !(dl > 0.0f);
    const float lam = sLam[i];
    for (int g = lane; g <= d.G; g += 32) {
      long long best = may_empty ? cur[g] : -1;
#pragma unroll
      for (int j = 0; j < kT; ++j) {
        const RowOpt ro = opt[4 * i + j];
        const int top = min(ro.hi, g >> j);
        for (int n = ro.lo; n <= top && n > 0; ++n) {
          const long long pv = cur[g - (n << j)];
          if (pv >= 0) {
            const long long v = goodput_fx20((float)n, ro.C, lam) + pv;
            best = v > best ? v : best;
          }
        }
      }
      nxt[g] = best;
    }
    __syncwarp();
    long long* x = cur;
    cur = nxt;
    nxt = x;
  }
  return cur;
}

// Whether the ranges in opt (left by warp_other at a value t0 with
// (t0 > 0) = pos) hold at t as well: then so do the programme's result and
// class i_r's other rows. One warp.
template <bool FL>
__device__ bool warp_ranges_hold(const Dims& d, const float* sDl, const RowOpt* opt, float t, bool pos) {
  const int lane = threadIdx.x & 31;
  bool ok = (t > 0.0f) == pos;
  for (int rho = lane; rho < d.K4; rho += 32) {
    const float T = class_threshold(t, FL ? sDl[rho >> 2] : 0.0f);
    ok = ok && opt[rho].a < T && T <= opt[rho].b;
  }
  return __all_sync(0xffffffffu, ok);
}

// Tier-3 goodput of one realisation with row rr at capacity Cr (its range
// [lor, hir] at t), at tiers 1-2 value t, given other = warp_other(..., skip
// = class of rr, t): the best over class i_r's choices (nothing, when it may
// stay empty; else n replicas on one of its rows) of its goodput plus the
// others' best within the GPUs left; -1 when the floors cannot be met. Lanes
// over the choices, one warp.
template <bool FL>
__device__ long long warp_best_with(const Dims& d, const float* sLam, const float* sDl, const RowOpt* opt, int rr,
                                    float Cr, int lor, int hir, float t, const long long* other) {
  const int lane = threadIdx.x & 31, ir = rr >> 2, jr = rr & 3;
  const float lam = sLam[ir];
  const float dl = FL ? sDl[ir] : 0.0f;
  int cnt[kT], lo[kT];
  float C[kT];
#pragma unroll
  for (int j = 0; j < kT; ++j) {
    const RowOpt ro = opt[4 * ir + j];
    lo[j] = j == jr ? lor : ro.lo;
    const int hi = j == jr ? hir : ro.hi;
    C[j] = j == jr ? Cr : ro.C;
    cnt[j] = lo[j] > 0 ? hi - lo[j] + 1 : 0;
  }
  long long best = (!(t > 0.0f) && !(dl > 0.0f)) ? other[d.G] : -1;
  const int e1 = cnt[0], e2 = e1 + cnt[1], e3 = e2 + cnt[2], total = e3 + cnt[3];
  for (int x = lane; x < total; x += 32) {
    int j, n;
    float Cj;
    if (x < e1) { j = 0; n = lo[0] + x; Cj = C[0]; }
    else if (x < e2) { j = 1; n = lo[1] + (x - e1); Cj = C[1]; }
    else if (x < e3) { j = 2; n = lo[2] + (x - e2); Cj = C[2]; }
    else { j = 3; n = lo[3] + (x - e3); Cj = C[3]; }
    const long long pv = other[d.G - (n << j)];
    if (pv >= 0) {
      const long long v = goodput_fx20((float)n, Cj, lam) + pv;
      best = v > best ? v : best;
    }
  }
  for (int off = 16; off; off >>= 1) {
    const long long o = __shfl_xor_sync(0xffffffffu, best, off);
    best = o > best ? o : best;
  }
  return best;
}

// t* of realisation sigma at row capacity C, from the candidate's table in
// global memory (the IEEE row term: every input).
template <bool FL>
__device__ __forceinline__ float tstar_global(const float* h, float C) {
  const int Lp = __float_as_int(h[H_LPAD]);
  const float* kap = h + kTableHeader;
  const float* thx = kap + Lp;
  const float* mnx = thx + Lp;
  int pos = 0;
  for (int step = __float_as_int(h[H_STEP0]); step > 0; step >>= 1) pos += kap[pos + step - 1] <= C ? step : 0;
  const float thb = thx[pos];
  const float m = mnx[pos];
  const float tr = m >= 1.0f ? fulfil(m, C, h[H_LAM]) : 0.0f;
  if (FL) return (tr > thb && tr >= h[H_DLT]) ? tr : thb;
  return tr > thb ? tr : thb;
}

// Shared memory of k_score_goodput: per table entry its gap (8 bytes), both
// realisations' row capacities (8) and values (16: t*, then the goodput),
// one flag byte; per warp its K4 row ranges and two programme arrays.
struct GoodputSmem {
  size_t gtab, cap, val, flag, warps, per_warp, total;
};

__host__ __device__ inline GoodputSmem goodput_smem(int K4, int G, int gt_len, int nwarp) {
  GoodputSmem m{};
  auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
  m.gtab = 0;
  m.cap = up(m.gtab + 8 * (size_t)gt_len);
  m.val = up(m.cap + 8 * (size_t)gt_len);
  m.flag = up(m.val + 16 * (size_t)gt_len);
  m.warps = up(m.flag + (size_t)gt_len);
  m.per_warp = up(sizeof(RowOpt) * (size_t)K4) + 16 * ((size_t)G + 1);
  m.total = m.warps + (size_t)nwarp * m.per_warp;
  return m;
}

// One block per segment (candidate e, outcome o) at a time. Entries: [0, W)
// open gate at position k; [W, 2W) closed gate at position k - W (under the
// prior), or W alone (closed, one value). A realisation's goodput depends on
// an entry only through its patched row capacity C' (t* is a function of
// C'), and consecutive entries often share C' (every position whose c_y lies
// at or below Cexcl, or is clamped by the refit): a run of equal C' takes one
// evaluation. The evaluation splits the programme at class i_r: the other
// classes' best within g GPUs depends on the entry only through the replica
// ranges that t* leaves their rows, which change at few values of t* in a
// segment, so a warp reruns that part only where a range changes and
// otherwise only combines it with class i_r's choices. Then the same draws
// and sums as the table path.
// MINB: resident blocks per SM the registers are capped for (2, or 4 for
// launches of many segments, whose throughput gains more from the occupancy
// than each block loses).
template <bool FL, bool RF, int MINB>
__global__ void __launch_bounds__(256, MINB) k_score_goodput(Set set, Items it, Plan pl, const float* rec,
                                                          uint64_t* sums) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const Dims& d = set.d;
  const int W = pl.W, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  const int gt_len = RF ? 2 * W : W + 1;
  const GoodputSmem lay = goodput_smem(d.K4, d.G, gt_len, nwarp);
  uint64_t* gtab = reinterpret_cast<uint64_t*>(smraw + lay.gtab);
  float* cap = reinterpret_cast<float*>(smraw + lay.cap);          // [2][gt_len]
  long long* val = reinterpret_cast<long long*>(smraw + lay.val);  // [2][gt_len]
  uint8_t* flag = smraw + lay.flag;  // bit 0 / 1: a run starts here (realisation 0 / 1); bit 2: reachable
  unsigned char* wbase = smraw + lay.warps + (size_t)warp * lay.per_warp;
  RowOpt* opt = reinterpret_cast<RowOpt*>(wbase);
  long long* dpa = reinterpret_cast<long long*>(wbase + ((sizeof(RowOpt) * (size_t)d.K4 + 15) & ~(size_t)15));
  long long* dpb = dpa + (d.G + 1);
  __shared__ float sC[2][256];
  __shared__ int sOk[2][256];
  __shared__ float sLam[FS_MAX_CLASSES], sRl[FS_MAX_CLASSES], sDl[FS_MAX_CLASSES];
  for (int x = tid; x < 2 * d.K4; x += blockDim.x) {
    const int sg = x / d.K4, rho = x - sg * d.K4;
    sC[sg][rho] = set.rowC[(size_t)sg * d.K4 + rho];
    sOk[sg][rho] = set.rowB[(size_t)sg * d.K4 + rho] >= 0;
  }
  for (int i = tid; i < d.K; i += blockDim.x) {
    sLam[i] = set.lam[i];
    sRl[i] = __frcp_rn(set.lam[i]);
    sDl[i] = FL ? set.slo[d.K + i] : 0.0f;
  }
  __syncthreads();
  const PhiloxKeys keys{};  // (the plan's round keys serve a one-problem launch)
  const long long n_seg = (long long)it.n * pl.O;
  for (long long seg = blockIdx.x; seg < n_seg; seg += gridDim.x) {
    const long long* other = nullptr;  // the warp's programme over the other classes, for this segment
    bool other_pos = false;
    int other_sg = 0;
    const int item = (int)(seg / pl.O), o = (int)(seg - (long long)item * pl.O);
    const float* r = rec + (size_t)item * pl.item_floats;
    const float* h0 = r;
    const float* h1 = r + d.slot_floats;
    const float* win = r + 2 * (size_t)d.slot_floats + (size_t)o * pl.Wp;
    const int cell = __float_as_int(h0[H_CELL]);
    if (cell < 0 || cell >= d.cells) continue;  // flagged by the preparation (uniform over the block)
    const int rr = cell / d.B;
    const uint32_t kgs = (uint32_t)__float_as_int(win[0]) << pl.sh;
    const uint32_t kgs16 = (uint32_t)min((unsigned long long)kgs << 16, 0xFFFFFFFFull);
    const bool any_open = kgs != 0u, any_closed = kgs16 != 0xFFFFFFFFu;
    const RowCap a0 = row_cap_of(h0), a1 = row_cap_of(h1);
    auto reachable = [&](int k) { return k < W ? any_open : any_closed; };
    // each entry's patched row capacity in both realisations
    for (int k = tid; k < gt_len; k += blockDim.x) {
      const bool g = k < W;
      const float cy = g ? win[4 + k] : (RF ? win[4 + k - W] : 0.0f);
      cap[k] = RF ? row_cap(a0, cy, g) : (g ? fmaxf(a0.pc, cy) : a0.pc);
      cap[gt_len + k] = RF ? row_cap(a1, cy, g) : (g ? fmaxf(a1.pc, cy) : a1.pc);
    }
    __syncthreads();
    // where runs of equal capacity start, and t* there
    for (int k = tid; k < gt_len; k += blockDim.x) {
      uint8_t f = 0;
      if (reachable(k)) {
        f = 4;
        const bool first = k == 0 || !reachable(k - 1);
        const float c0 = cap[k], c1 = cap[gt_len + k];
        if (first || __float_as_uint(c0) != __float_as_uint(cap[k - 1])) {
          f |= 1;
          val[k] = (long long)__float_as_uint(tstar_global<FL>(h0, c0));
        }
        if (first || __float_as_uint(c1) != __float_as_uint(cap[gt_len + k - 1])) {
          f |= 2;
          val[gt_len + k] = (long long)__float_as_uint(tstar_global<FL>(h1, c1));
        }
      }
      flag[k] = f;
    }
    __syncthreads();
    // the warps take chunks of 32 entries of one realisation in turn; a chunk's
    // first reachable entry starts a run. Every run start's row-r range comes
    // from its own lane; the others' programme is rerun only where a row's
    // range changes with t*
    {
      const int ir = rr >> 2, jr = rr & 3;
      const float lam_r = sLam[ir], rl_r = sRl[ir], dl_r = FL ? sDl[ir] : 0.0f;
      const int n_chunk = (gt_len + 31) >> 5;
      for (int task = warp; task < 2 * n_chunk; task += nwarp) {
        const int sg = task & 1, kk = ((task >> 1) << 5) + lane;
        const float* cs = cap + (size_t)sg * gt_len;
        long long* v = val + (size_t)sg * gt_len;
        const bool reach = kk < gt_len && (flag[kk] & 4);
        const bool start = reach && ((flag[kk] >> sg) & 1);
        const unsigned rb = __ballot_sync(0xffffffffu, reach);
        const bool head = start || (rb && lane == __ffs(rb) - 1);
        float c = 0.0f, t = 0.0f;
        int lor = 0, hir = 0;
        if (head) {  // t* stored where a run starts, else evaluated
          c = cs[kk];
          t = start ? __uint_as_float((uint32_t)v[kk]) : tstar_global<FL>(sg ? h1 : h0, c);
          row_range(c, true, d.G >> jr, class_threshold(t, dl_r), lam_r, rl_r, lor, hir);
        }
        unsigned heads = __ballot_sync(0xffffffffu, head);
        long long mine = 0;
        while (heads) {
          const int p = __ffs(heads) - 1;
          heads &= heads - 1;
          const float tp = __shfl_sync(0xffffffffu, t, p), cp = __shfl_sync(0xffffffffu, c, p);
          const int lop = __shfl_sync(0xffffffffu, lor, p), hip = __shfl_sync(0xffffffffu, hir, p);
          if (other == nullptr || other_sg != sg || !warp_ranges_hold<FL>(d, sDl, opt, tp, other_pos)) {
            other = warp_other<FL>(d, sC[sg], sOk[sg], sLam, sRl, sDl, ir, rr, tp, opt, dpa, dpb);
            other_pos = tp > 0.0f;
            other_sg = sg;
          }
          long long gv = warp_best_with<FL>(d, sLam, sDl, opt, rr, cp, lop, hip, tp, other);
          gv = gv < 0 ? 0 : gv;
          if (lane >= p) mine = gv;
        }
        if (reach) v[kk] = mine;
      }
    }
    __syncthreads();
    for (int k = tid; k < gt_len; k += blockDim.x) {
      if (!(flag[k] & 4)) continue;
      const long long g0 = val[k], g1 = val[gt_len + k];
      const unsigned long long gap = (unsigned long long)(g1 > g0 ? g1 - g0 : g0 - g1);
      gtab[k] = gap;
    }
    __syncthreads();
    unsigned long long v = sample_gtab<true, RF>(pl, keys, o, cell, 0, pl.calls, smem_u32(gtab), kgs16);
    for (int off = 16; off; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0 && v) atomicAdd(reinterpret_cast<unsigned long long*>(&sums[(size_t)seg]), v);
    __syncthreads();  // the tables are rebuilt for the next segment
  }
}

// E, score and argmax of the goodput stage for one problem (one CTA).
__global__ void k_finalize_goodput(Set set, Items it, Plan pl, const uint64_t* sums, double lam_sum, double* gap,
                                   double* score, double* gamma, int32_t* best, uint32_t* status_copy) {
  __shared__ Best sb[32];
  // every earlier kernel of the call has completed: the status word travels
  // with the outputs
  if (threadIdx.x == 0 && status_copy) *status_copy = *set.status;
  const Dims& d = set.d;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  const long long gm = __double2ll_rn(__dmul_rn(set.base[0].goodput, 0x1p20));
  const long long gpl = __double2ll_rn(__dmul_rn(set.base[1].goodput, 0x1p20));
  const long long gfix = gpl > gm ? gpl - gm : gm - gpl;
  const long long n = (long long)pl.O * pl.S;
  const double dn = __ll2double_rn(n);
  Best b = no_best();
  for (int q = tid; q < it.n; q += blockDim.x) {
    const int cell = it.cell[q];
    long long tot = 0;
    for (int o = 0; o < pl.O; ++o) tot += (long long)sums[(size_t)q * pl.O + o];
    const long long sc = gfix * n - tot;
    if (gap) gap[q] = __ddiv_rn(__ddiv_rn(__dmul_rn(__ll2double_rn(tot), 0x1p-20), dn), lam_sum);
    if (score) score[q] = __ddiv_rn(__ddiv_rn(__dmul_rn(__ll2double_rn(sc), 0x1p-20), dn), lam_sum);
    const Best c = make_best(sc, (cell / d.B) & 3, q, cell);
    if (better(c, b)) b = c;
  }
  b = warp_best(b);
  if (lane == 0) sb[warp] = b;
  __syncthreads();
  if (warp == 0) {
    b = warp_best(lane < nwarp ? sb[lane] : no_best());
    if (lane == 0) {
      if (best) *best = b.valid() ? b.cell : -1;
      if (gamma) *gamma = __ddiv_rn(__dmul_rn(__ll2double_rn(gfix), 0x1p-20), lam_sum);
    }
  }
}

// --------------------------------------------------------------------------- launchers

size_t lex_scratch_cells(const Dims& d) { return (size_t)(d.K + 1) * (d.G + 1); }

// Whether the programme of n realisations needs scratch in global memory.
static LexSmem lex_layout(const Dims& d, int n, bool pack) {
  return n <= kSolveWideMax ? lex_smem(d.K, d.G, pack, kLexOptWide, kLexCellsWide)
                            : lex_smem(d.K, d.G, pack, kLexOptWarp, kLexCellsWarp);
}

bool lex_needs_scratch(const Dims& d, int n, bool pack) { return lex_layout(d, n, pack).n_cells == 0; }

template <bool PACK, int NW>
static cudaError_t launch_lex(const Set& set, int n, const float* cap_x, const float* tail_x, fs_allocation* out,
                              void* scratch, int per_launch, const LexSmem& lay, cudaStream_t s) {
  constexpr int kPerBlock = NW == 1 ? 4 : 1;
  auto kern = k_solve_lex<PACK, NW>;
  const size_t smem = kPerBlock * lay.total;
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  for (int r0 = 0; r0 < n; r0 += per_launch) {
    const int m = n - r0 < per_launch ? n - r0 : per_launch;
    note_launch();
    kern<<<(m + kPerBlock - 1) / kPerBlock, NW == 1 ? 128 : 32 * NW, smem, s>>>(
        set, r0 + m, cap_x, tail_x, out, static_cast<unsigned char*>(scratch), r0, lay);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_solve_lex(const Set& set, int n, const float* cap_x, const float* tail_x, fs_allocation* out,
                             void* scratch, int per_launch, bool pack, cudaStream_t s) {
  const LexSmem lay = lex_layout(set.d, n, pack);
  auto go = n <= kSolveWideMax ? (pack ? launch_lex<true, kLexWideWarps> : launch_lex<false, kLexWideWarps>)
                               : (pack ? launch_lex<true, 1> : launch_lex<false, 1>);
  return go(set, n, cap_x, tail_x, out, scratch, per_launch, lay, s);
}

int goodput_threads(const Dims& d, const Plan& pl, bool rf, size_t* smem) {
  const int gt_len = rf ? 2 * pl.W : pl.W + 1;
  for (int nw = 8; nw >= 1; --nw) {
    const GoodputSmem m = goodput_smem(d.K4, d.G, gt_len, nw);
    if (m.total <= kGoodputSmemMax) {
      if (smem) *smem = m.total;
      return 32 * nw;
    }
  }
  return 0;
}

cudaError_t launch_score_goodput(const Set& set, const Items& it, const Plan& pl, const float* tables,
                                 uint64_t* sums, int floors, int sm_count, cudaStream_t s) {
  if (it.n <= 0) return cudaSuccess;
  const bool rf = set.prior == 1;
  size_t smem = 0;
  const int threads = goodput_threads(set.d, pl, rf, &smem);
  if (threads == 0) return cudaErrorInvalidValue;  // refused by the host before this point
  // many segments (beyond four waves of two blocks per SM): the instance with
  // registers for four blocks per SM (measured 5.94 -> 3.44 ms on the
  // eight-class workload, 0.375 -> 0.325 ms on the mid one at three times its
  // demands; the paper-scale call, one wave, slower: 0.17 -> 0.19 ms)
  const long long n_seg = (long long)it.n * pl.O;
  const bool wide = n_seg > 4LL * 2 * sm_count;
#define FS_GP(MB) \
  (floors ? (rf ? k_score_goodput<true, true, MB> : k_score_goodput<true, false, MB>) \
          : (rf ? k_score_goodput<false, true, MB> : k_score_goodput<false, false, MB>))
  auto kern = wide ? FS_GP(4) : FS_GP(2);
#undef FS_GP
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  // one block per segment: segments differ widely in cost (where row r sets
  // t*, its ranges change often), and the block scheduler evens them out
  const long long grid = n_seg < 0x7fffffffLL ? n_seg : 0x7fffffffLL;
  note_launch();
  kern<<<(unsigned)grid, threads, smem, s>>>(set, it, pl, tables, sums);
  return cudaGetLastError();
}

cudaError_t launch_finalize_goodput(const Set& set, const Items& it, const Plan& pl, const uint64_t* sums,
                                    double lam_sum, double* gap, double* score, double* gamma, int32_t* best,
                                    uint32_t* status_copy, cudaStream_t s) {
  note_launch();
  k_finalize_goodput<<<1, 256, 0, s>>>(set, it, pl, sums, lam_sum, gap, score, gamma, best, status_copy);
  return cudaGetLastError();
}

}  // namespace fs
