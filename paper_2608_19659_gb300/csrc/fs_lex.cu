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
// k_other, k_score_goodput: the goodput stage of the Monte-Carlo score. Within a
//   segment (candidate e, outcome o) a scenario's goodput gap
//   |GP(A+') - GP(A-')| depends on its draw only through (c_y position,
//   tail gate), as its t* does: the block tabulates those values, a thread per
//   entry, on top of tables of the other classes' best goodput that k_other
//   makes once per call, then draws every scenario's position and sums the
//   entries.
// k_finalize_goodput: E[Gamma_gp,t+1 | e] = sum 2^-20 / (O S) / sum lambda,
//   the score Gamma_gp,t - E and the argmax (same order as the max-min stage).
#include <cuda_runtime.h>

#include <algorithm>

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
// options with e <= slack are few. A table over all of [0, G] with a division per
// option and cell, and one thread's walk forward, takes 66 us on 1000 realisations
// of the four-class, 64-GPU grid and 180 us on two of the eight-class, 256-GPU one
// (this one: see launch_solve_lex).
template <bool PACK, int NW>
__global__ void __launch_bounds__(NW == 1 ? 128 : 32 * NW) k_solve_lex(Set set, int n_real, const float* cap_x,
                                                                       const float* tail_x, fs_allocation* out_x,
                                                                       unsigned char* scratch, int r0, LexSmem lay,
                                                                       HostOut host) {
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
    const float* bp = set.bounds + (size_t)p * 4 * d.cells;
    cap = bp + (size_t)(sigma ? CAP_HI : CAP_LO) * d.cells;
    tail = bp + (size_t)(sigma ? TAIL_LO : TAIL_HI) * d.cells;
    out = set.base + r;
  }
  const float tstar = out->t_star;
  // the first warp, once the allocation is complete: its copy for the host
  auto finish = [&]() {
    __syncwarp();
    if (host.alloc) {
      const uint64_t* src = reinterpret_cast<const uint64_t*>(out);
      uint64_t* dst = reinterpret_cast<uint64_t*>(host.alloc + r);
      for (int w = lane; w < (int)(sizeof(fs_allocation) / 8); w += 32) dst[w] = src[w];
    }
    if (host.status && lane == 0) host.status[r] = *set.status;
  };
  if (!out->floors_met) {  // tier 1 cannot hold: nothing is allocated (k_solve wrote the empty allocation)
    if (tid == 0) out->goodput = 0.0;
    if (warp == 0) finish();
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
    if (warp == 0) finish();
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
  finish();
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

// Value tables of one goodput call. A realisation's goodput depends on a
// scenario only through its patched row capacity C' (t* is a function of C').
// It splits at the candidate's class i_r: the best of class i_r's choices plus
// `other`, the best goodput of the other classes within the GPUs left, which
// depends on t* only through the replica ranges it leaves the other classes'
// rows. Those change only just above a threshold of the realisation, so `other`
// is the same for every t* in (theta_{k-1}, theta_k]: one table per
// (realisation, class, k), shared by every candidate of the class and every
// outcome. Row kk of a (realisation, class): 0 holds t* = 0, k + 1 holds t* in
// (theta_{k-1}, theta_k], total + 1 holds t* above every threshold. The
// preparation records the rows its candidates can reach (span), k_other fills
// them.
struct GoodputTables {
  int* span;            // [2 (least, most)][2][K] rows wanted per (realisation, class); least > most: none
  int* first;           // [2][K] first row of each in the pool (k_other)
  long long* base;      // [2] the base realisations' goodput, 2^-20 req/s
  long long* closed;    // [items][2] goodput at Cexcl: every scenario whose tail gate is closed
                        // (nullptr: few segments, each evaluates it itself)
  long long* rows;      // pool of rows of `stride` words
  int stride;           // G + 1 values by GPUs, then kT: the best without each row of the class
  int pool;             // rows the pool holds
  int c0, c1;           // classes of this pass (the pool may not hold every class's rows at once)
};

// First row of (sigma, class i) in the pool: the rows wanted by the pass's
// classes in order (a few dozen additions; every caller finds the same).
__device__ __forceinline__ int span_rows(const GoodputTables& g, int K, int sc) {
  const int lo = g.span[sc], hi = g.span[2 * K + sc];
  const int i = sc < K ? sc : sc - K;
  return i >= g.c0 && i < g.c1 && hi >= lo ? hi - lo + 1 : 0;
}

// Inclusive scan over the lanes (rows of the (realisation, class) pairs lane,
// lane + 32, .. < 2K handled by the caller).
__device__ __forceinline__ int warp_scan(int v, int lane) {
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// Tasks of k_other: one block per (realisation, class, row), and two more for
// the base realisations' goodput (t* itself, every class).
//
// A programme over the other classes within g GPUs, over the GPUs that their
// cheapest options leave (h = g - need; below need nothing reaches): options
// cost e = cost - cheapest of them. Threads over (h, TP degree): four lanes take
// a class's four rows for one h and merge by two shuffles. Then the best of class
// i's own rows at their base capacities on top, for candidates on another of its
// rows. What bounds it: the chain of K - 1 dependent steps of a task (some 800
// tasks on the eight-class, 256-GPU grid). A warp per task, lanes over h, took 35
// us there, a block 21 us.
constexpr int kOtherThreads = 128;

struct OtherSmem {
  size_t lohi, mins, opt, dp, total;
  int n_opt;
};

__host__ __device__ inline OtherSmem other_smem(int K, int G) {
  OtherSmem m{};
  auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
  m.n_opt = G + (G >> 1) + (G >> 2) + (G >> 3);
  m.lohi = up(16 * (size_t)(4 * K));             // base capacities [2][4K], feasible [2][4K]; option ranges [4K] x 2
  m.mins = up(m.lohi + 8 * (size_t)(4 * K));     // [K]
  m.opt = up(m.mins + 4 * (size_t)K);            // one class's option values
  m.dp = up(m.opt + 8 * (size_t)m.n_opt);        // two arrays of G + 1
  m.total = up(m.dp + 16 * ((size_t)G + 1));
  return m;
}

template <bool FL>
__global__ void __launch_bounds__(kOtherThreads) k_other(Set set, GoodputTables gt, OtherSmem lay) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const Dims& d = set.d;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ float sLam[FS_MAX_CLASSES], sRl[FS_MAX_CLASSES], sDl[FS_MAX_CLASSES];
  __shared__ int sBeg[2 * FS_MAX_CLASSES + 1];
  __shared__ long long sRow[kT];
  __shared__ int s_need;
  float* sC = reinterpret_cast<float*>(smraw);   // [2][K4]
  int* sOk = reinterpret_cast<int*>(sC + 2 * d.K4);
  int* sLo = reinterpret_cast<int*>(smraw + lay.lohi);
  int* sHi = sLo + d.K4;
  int* sMin = reinterpret_cast<int*>(smraw + lay.mins);
  long long* sOpt = reinterpret_cast<long long*>(smraw + lay.opt);
  long long* cur = reinterpret_cast<long long*>(smraw + lay.dp);
  long long* nxt = cur + (d.G + 1);
  pdl_wait();
  pdl_trigger();
  for (int x = tid; x < 2 * d.K4; x += kOtherThreads) {
    sC[x] = set.rowC[x];
    sOk[x] = set.rowB[x] >= 0;
  }
  for (int i = tid; i < d.K; i += kOtherThreads) {
    const float lam = set.lam[i];
    sLam[i] = lam;
    sRl[i] = __frcp_rn(lam);
    sDl[i] = FL ? set.slo[d.K + i] : 0.0f;
  }
  if (warp == 0) {  // first task of each (realisation, class)
    int carry = 0;
    for (int b = 0; b < 2 * d.K; b += 32) {
      const int sc = b + lane;
      const int v = sc < 2 * d.K ? span_rows(gt, d.K, sc) : 0;
      const int incl = warp_scan(v, lane);
      if (sc < 2 * d.K) {
        sBeg[sc + 1] = carry + incl;
        if (blockIdx.x == 0) gt.first[sc] = carry + incl - v;
      }
      carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) sBeg[0] = 0;
  }
  __syncthreads();
  const int rows = sBeg[2 * d.K];
  if (rows > gt.pool) {  // cannot happen: the host sized the pool for the most rows there can be
    if (blockIdx.x == 0 && tid == 0) atomicOr(set.status, ST_TABLE);
    return;
  }
  const int n_base = gt.c0 == 0 ? 2 : 0;  // (the first pass)
  for (int task = (int)blockIdx.x; task < rows + n_base; task += (int)gridDim.x) {
    const bool base = task >= rows;
    int sigma, cls, kk = 0;
    float t;
    if (base) {
      sigma = task - rows;
      cls = 0;
      t = base_tstar(set, 0, sigma);
    } else {
      int sc = 0, hi = 2 * d.K - 1;
      while (sc < hi) {
        const int mid = (sc + hi + 1) >> 1;
        if (sBeg[mid] <= task) sc = mid; else hi = mid - 1;
      }
      sigma = sc >= d.K ? 1 : 0;
      cls = sc - sigma * d.K;
      kk = gt.span[sc] + task - sBeg[sc];
      const int total = set.ntheta[sigma];
      const float* th = set.theta + (size_t)sigma * d.theta_cap;
      if (kk == 0) t = 0.0f;
      else if (kk <= total) t = th[kk - 1];
      else t = total ? __uint_as_float(__float_as_uint(th[total - 1]) + 1u) : __uint_as_float(1u);
    }
    // option ranges of every row at t, and each class's cheapest option
    const float* C = sC + sigma * d.K4;
    auto empty_ok = [&](int i) { return !(t > 0.0f) && !(FL && sDl[i] > 0.0f); };
    for (int rho = tid; rho < d.K4; rho += kOtherThreads) {
      const int i = rho >> 2;
      int lo, hi;
      row_range(C[rho], sOk[sigma * d.K4 + rho] != 0, rep_cap(d, rho & 3), class_threshold(t, FL ? sDl[i] : 0.0f),
                sLam[i], sRl[i], lo, hi);
      sLo[rho] = lo;
      sHi[rho] = hi;
    }
    __syncthreads();
    if (warp == 0) {
      int need = 0;
      for (int b = 0; b < d.K; b += 32) {
        const int i = b + lane;
        int m = 0;
        if (i < d.K) {
          if (!empty_ok(i)) {
            m = 1 << 24;  // (above every budget: 64 of them stay below 2^31)
            for (int j = 0; j < kT; ++j)
              if (sLo[4 * i + j]) m = min(m, sLo[4 * i + j] << j);
          }
          sMin[i] = m;
        }
        need += __reduce_add_sync(0xffffffffu, i < d.K && i != cls ? m : 0);
      }
      if (lane == 0) s_need = need;
    }
    __syncthreads();
    const int need = s_need;
    const int H = need <= d.G ? d.G - need + 1 : 0;  // GPUs above the cheapest options: 0..H-1
    for (int h = tid; h < H; h += kOtherThreads) cur[h] = 0;
    const int j = tid & 3;  // this thread's TP degree
    for (int i = 0; H > 0 && i < d.K; ++i) {
      if (i == cls) continue;
      const int m = sMin[i];
      int cnt[kT], beg[kT], all = 0;
#pragma unroll
      for (int q = 0; q < kT; ++q) {
        const int lo = sLo[4 * i + q];
        cnt[q] = lo ? max(0, min(sHi[4 * i + q], (H - 1 + m) >> q) - lo + 1) : 0;
        beg[q] = all;
        all += cnt[q];
      }
      for (int x = tid; x < all; x += kOtherThreads) {
        int q = 0;
#pragma unroll
        for (int y = 1; y < kT; ++y)
          if (x >= beg[y]) q = y;
        const int lo = sLo[4 * i + q], at = q == 0 ? 0 : q == 1 ? beg[1] : q == 2 ? beg[2] : beg[3];
        sOpt[x] = goodput_fx20((float)(lo + x - at), C[4 * i + q], sLam[i]);
      }
      __syncthreads();
      const int my_cnt = j == 0 ? cnt[0] : j == 1 ? cnt[1] : j == 2 ? cnt[2] : cnt[3];
      const long long* opt = sOpt + (j == 0 ? 0 : j == 1 ? beg[1] : j == 2 ? beg[2] : beg[3]);
      const int e0 = (sLo[4 * i + j] << j) - m;
      const bool empty = empty_ok(i);
      for (int h0 = 0; h0 < H; h0 += kOtherThreads / 4) {
        const int h = h0 + (tid >> 2);
        long long best = -1;
        if (h < H) {
          if (empty && j == 0) best = cur[h];
          int e = e0;
          for (int x = 0; x < my_cnt && e <= h; ++x, e += 1 << j) {
            const long long v = opt[x] + cur[h - e];
            best = v > best ? v : best;
          }
        }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
          const long long v = __shfl_xor_sync(0xffffffffu, best, o);
          best = v > best ? v : best;
        }
        if (j == 0 && h < H) nxt[h] = best;
      }
      __syncthreads();
      long long* x = cur;
      cur = nxt;
      nxt = x;
    }
    // (a lone class's programme is all zeros)
    if (H > 0) __syncthreads();
    // the class's own rows on top, a warp each: replicas over the lanes
    {
      long long best = -1;
      const int lo = sLo[4 * cls + warp];
      if (lo && H > 0) {
        const int top = min(sHi[4 * cls + warp], (H - 1) >> warp);
        for (int n = lo + lane; n <= top; n += 32) {
          const long long v = goodput_fx20((float)n, C[4 * cls + warp], sLam[cls]) + cur[H - 1 - (n << warp)];
          best = v > best ? v : best;
        }
      }
      for (int o = 16; o; o >>= 1) {
        const long long v = __shfl_xor_sync(0xffffffffu, best, o);
        best = v > best ? v : best;
      }
      if (lane == 0) sRow[warp] = best;
    }
    __syncthreads();
    const long long none = empty_ok(cls) && H > 0 ? cur[H - 1] : -1;  // no replicas for the class
    if (base) {
      long long best = none;
#pragma unroll
      for (int q = 0; q < kT; ++q) best = sRow[q] > best ? sRow[q] : best;
      if (tid == 0) gt.base[sigma] = best < 0 ? 0 : best;
    } else {
      // other[g] = cur[g - need], -1 below
      long long* row = gt.rows + (size_t)task * gt.stride;
      for (int g = tid; g <= d.G; g += kOtherThreads) row[g] = g >= need ? cur[g - need] : -1;
      if (tid < kT) {
        long long best = none;
#pragma unroll
        for (int q = 0; q < kT; ++q)
          if (q != tid && sRow[q] > best) best = sRow[q];
        row[d.G + 1 + tid] = best;
      }
    }
    __syncthreads();  // the next task's ranges and programme
  }
}

// What a scenario's goodput in one realisation needs besides C'.
struct GoodputCtx {
  const float* h;          // the candidate's table (header, kappa, theta, m) in global memory
  const long long* rows;   // other rows of (realisation, class), indexed by kk
  int stride, G, jr, M, lpad, step0, b0, fast;
  float lam, rl, dl;
};

// Tier-3 goodput at row capacity C (2^-20 req/s; 0 when the floors cannot be
// met): t* as the scorer finds it, then the best over row r's replica counts at
// C on top of the others' best, or the class's best without row r.
template <bool FL>
__device__ __forceinline__ long long goodput_at(const GoodputCtx& c, float C) {
  const float* kap = c.h + kTableHeader;
  int pos = 0;
  for (int step = c.step0; step > 0; step >>= 1) pos += kap[pos + step - 1] <= C ? step : 0;
  const float thb = kap[c.lpad + pos], m = kap[2 * c.lpad + pos];
  const float tr = m >= 1.0f ? (c.fast ? fulfil_fast(m, C, c.lam, c.rl) : fulfil(m, C, c.lam)) : 0.0f;
  const bool own = FL ? tr > thb && tr >= c.dl : tr > thb;
  const float t = own ? tr : thb;
  const long long* row = c.rows + (size_t)(c.b0 + 1 + pos + (own ? 1 : 0)) * c.stride;
  int lo, hi;
  row_range(C, true, c.M, class_threshold(t, FL ? c.dl : 0.0f), c.lam, c.rl, lo, hi);
  long long best = row[c.G + 1 + c.jr];
  if (lo) {
    const int top = min(hi, c.G >> c.jr);
    for (int n = lo; n <= top; ++n) {
      const long long pv = row[c.G - (n << c.jr)];
      if (pv >= 0) {
        const long long v = goodput_fx20((float)n, C, c.lam) + pv;
        best = v > best ? v : best;
      }
    }
  }
  return best < 0 ? 0 : best;
}

template <bool FL>
__device__ __forceinline__ GoodputCtx goodput_ctx(const Set& set, const GoodputTables& gt, const float* h, int sigma,
                                                  int rr) {
  const Dims& d = set.d;
  GoodputCtx c;
  const int i = rr >> 2;
  c.h = h;
  c.stride = gt.stride;
  c.G = d.G;
  c.jr = rr & 3;
  c.M = rep_cap(d, c.jr);
  c.lpad = __float_as_int(h[H_LPAD]);
  c.step0 = __float_as_int(h[H_STEP0]);
  c.b0 = __float_as_int(h[H_B0]);
  c.fast = __float_as_int(h[H_FAST]);
  c.lam = h[H_LAM];
  c.rl = h[H_RLAM];
  c.dl = FL ? h[H_DLT] : 0.0f;
  const int sc = sigma * d.K + i;
  c.rows = gt.rows + ((long long)gt.first[sc] - gt.span[sc]) * gt.stride;
  return c;
}

// Each candidate's goodput at Cexcl in both realisations, a thread each (without
// the prior): what every entry at or below Cexcl and every closed gate takes.
template <bool FL>
__global__ void __launch_bounds__(128) k_goodput_closed(Set set, Items it, Plan pl, const float* rec, GoodputTables gt) {
  pdl_wait();
  pdl_trigger();
  const Dims& d = set.d;
  const long long x = (long long)blockIdx.x * 128 + threadIdx.x;
  if (x >= 2LL * it.n) return;
  const int item = (int)(x >> 1), sigma = (int)x & 1;
  const float* h = rec + (size_t)item * pl.item_floats + (size_t)sigma * d.slot_floats;
  const int cell = __float_as_int(h[H_CELL]);
  if (cell < 0 || cell >= d.cells) return;  // flagged by the preparation
  const int rr = cell / d.B, ir = rr >> 2;
  if (ir < gt.c0 || ir >= gt.c1) return;    // another pass's class
  const GoodputCtx c = goodput_ctx<FL>(set, gt, h, sigma, rr);
  gt.closed[x] = goodput_at<FL>(c, h[H_CX]);
}

// One block per segment (candidate e, outcome o): entries [0, W) hold the gap
// with an open gate at position k, W with a closed one (under the prior [W, 2W),
// position k - W). A thread per entry; without the prior every entry at or
// below a realisation's Cexcl takes that realisation's closed-gate goodput. Then
// the same draws and sums as the table path.
template <bool FL, bool RF>
__global__ void __launch_bounds__(256, 4) k_score_goodput(Set set, Items it, Plan pl, const float* rec, uint64_t* sums,
                                                       GoodputTables gt) {
  extern __shared__ __align__(16) unsigned char smraw[];
  uint64_t* gtab = reinterpret_cast<uint64_t*>(smraw);
  __shared__ long long s_closed[2];
  __shared__ GoodputCtx s_ctx[2];
  const Dims& d = set.d;
  const int W = pl.W, tid = threadIdx.x, lane = tid & 31;
  pdl_wait();
  pdl_trigger();
  const PhiloxKeys keys{};  // (the plan's round keys serve a one-problem launch)
  const long long n_seg = (long long)it.n * pl.O;
  for (long long seg = blockIdx.x; seg < n_seg; seg += gridDim.x) {
    const int item = (int)(seg / pl.O), o = (int)(seg - (long long)item * pl.O);
    const float* h0 = rec + (size_t)item * pl.item_floats;
    const float* h1 = h0 + d.slot_floats;
    const float* win = h0 + 2 * (size_t)d.slot_floats + (size_t)o * pl.Wp;
    const int cell = __float_as_int(h0[H_CELL]);
    if (cell < 0 || cell >= d.cells) continue;  // flagged by the preparation (uniform over the block)
    const int rr = cell / d.B, ir = rr >> 2;
    if (ir < gt.c0 || ir >= gt.c1) continue;    // another pass's class (uniform)
    const uint32_t kgs = (uint32_t)__float_as_int(win[0]) << pl.sh;
    const uint32_t kgs16 = (uint32_t)min((unsigned long long)kgs << 16, 0xFFFFFFFFull);
    const bool any_open = kgs != 0u, any_closed = kgs16 != 0xFFFFFFFFu;
    if (lane == 0 && tid < 64) {
      const int sg = tid >> 5;
      const float* h = sg ? h1 : h0;
      s_ctx[sg] = goodput_ctx<FL>(set, gt, h, sg, rr);
      if (!RF) s_closed[sg] = gt.closed ? gt.closed[2 * (long long)item + sg] : goodput_at<FL>(s_ctx[sg], h[H_CX]);
    }
    __syncthreads();
    const long long c0 = s_closed[0], c1 = s_closed[1];
    const RowCap a0 = row_cap_of(h0), a1 = row_cap_of(h1);
    const int k0 = any_open ? 0 : W, k1 = RF ? (any_closed ? 2 * W : W) : W + 1;
    for (int k = k0 + tid; k < k1; k += blockDim.x) {
      const bool g = k < W;
      long long g0, g1;
      if (RF) {
        const float cy = win[4 + (g ? k : k - W)];
        g0 = goodput_at<FL>(s_ctx[0], row_cap(a0, cy, g));
        g1 = goodput_at<FL>(s_ctx[1], row_cap(a1, cy, g));
      } else {
        const float cy = g ? win[4 + k] : 0.0f;
        g0 = g && cy > a0.pc ? goodput_at<FL>(s_ctx[0], cy) : c0;
        g1 = g && cy > a1.pc ? goodput_at<FL>(s_ctx[1], cy) : c1;
      }
      gtab[k] = (unsigned long long)(g1 > g0 ? g1 - g0 : g0 - g1);
    }
    __syncthreads();
    unsigned long long v;
    if (!any_open || !any_closed)  // the gate is the same at every position
      v = sample_gtab<true, RF, false>(pl, keys, o, cell, 0, pl.calls, smem_u32(gtab) + (any_open ? 0u : 8u * (uint32_t)W),
                                       0u, (!RF && !any_open) ? pl.uniform_stride : pl.entry_bytes);
    else
      v = sample_gtab<true, RF, true>(pl, keys, o, cell, 0, pl.calls, smem_u32(gtab), kgs16);
    for (int off = 16; off; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0 && v) atomicAdd(reinterpret_cast<unsigned long long*>(&sums[(size_t)seg]), v);
    __syncthreads();  // the table is rebuilt for the next segment
  }
}

// E, score and argmax of the goodput stage for one problem, its candidates
// split over the blocks: each leaves its best in part[2 b ..], the last to take a
// ticket (work[1], zeroed by the preparation) merges them.
__global__ void k_finalize_goodput(Set set, Items it, Plan pl, const uint64_t* sums, const long long* base,
                                   double lam_sum, double* gap, double* score, double* gamma, int32_t* best,
                                   uint32_t* status_copy, uint64_t* part, uint64_t* sum_out) {
  __shared__ Best sb[32];
  __shared__ int s_last;
  pdl_wait();
  pdl_trigger();
  const Dims& d = set.d;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  const int nb = (int)gridDim.x, per = (it.n + nb - 1) / nb;
  const int beg = min(it.n, (int)blockIdx.x * per), end = min(it.n, beg + per);
  const long long gm = base[0], gpl = base[1];
  const long long gfix = gpl > gm ? gpl - gm : gm - gpl;
  const long long n = (long long)pl.O * pl.S;
  const double dn = __ll2double_rn(n);
  // x / n: a power of two's quotient is an exact scaling (no result is subnormal)
  const bool p2 = (n & (n - 1)) == 0;
  const double rn = p2 ? __longlong_as_double((1023LL - (63 - __clzll(n))) << 52) : 0.0;
  auto mean = [&](long long v) {
    const double x = __dmul_rn(__ll2double_rn(v), 0x1p-20);
    return __ddiv_rn(p2 ? __dmul_rn(x, rn) : __ddiv_rn(x, dn), lam_sum);
  };
  Best b = no_best();
  // lanes per candidate as in finalize_problem: four when split over blocks
  const int lpc = nb > 1 ? 4 : 1, sub = tid & (lpc - 1), step = (int)blockDim.x / lpc;
  for (int q0 = beg; q0 < end; q0 += step) {
    const int q = q0 + tid / lpc;
    const bool in = q < end;
    long long tot = 0;
    int cell = 0;
    if (in) {
      cell = __ldg(it.cell + q);
#pragma unroll 8
      for (int o = sub; o < pl.O; o += lpc) {
        const size_t x = (size_t)q * pl.O + o;
        const uint64_t v = __ldg(sums + x);
        tot += (long long)v;
        if (sum_out) sum_out[x] = v;  // (the caller's copy)
      }
    }
    for (int o = 1; o < lpc; o <<= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (!in) continue;
    const long long sc = gfix * n - tot;
    if (sub == 0 && gap) gap[q] = mean(tot);
    if (sub == lpc / 2 && score) score[q] = mean(sc);
    const Best c = make_best(sc, (cell / d.B) & 3, q, cell);
    if (better(c, b)) b = c;
  }
  b = warp_best(b);
  if (lane == 0) sb[warp] = b;
  __syncthreads();
  if (warp != 0) return;
  b = warp_best(lane < nwarp ? sb[lane] : no_best());
  if (nb > 1) {
    if (lane == 0) {
      part[2 * blockIdx.x] = (uint64_t)b.hi;
      part[2 * blockIdx.x + 1] = ((uint64_t)b.lo << 32) | (uint32_t)b.cell;
      __threadfence();
      s_last = atomicAdd(&set.work[1], 1ull) == (unsigned long long)(nb - 1);
    }
    __syncwarp();
    if (!s_last) return;
    __threadfence();
    b = no_best();
    for (int q = lane; q < nb; q += 32) {
      const uint64_t w = __ldcg(part + 2 * q + 1);
      const Best c{(long long)__ldcg(part + 2 * q), (uint32_t)(w >> 32), (int)(uint32_t)w};
      if (better(c, b)) b = c;
    }
    b = warp_best(b);
  }
  if (lane == 0) {
    if (best) *best = b.valid() ? b.cell : -1;
    if (gamma) *gamma = __ddiv_rn(__dmul_rn(__ll2double_rn(gfix), 0x1p-20), lam_sum);
    // every earlier kernel of the call has completed: the status word travels
    // with the outputs
    if (status_copy) *status_copy = *set.status;
  }
}

// --------------------------------------------------------------------------- launchers

size_t lex_scratch_cells(const Dims& d) { return (size_t)(d.K + 1) * (d.G + 1); }

// Whether the programme of n realisations needs scratch in global memory.
static LexSmem lex_layout(const Dims& d, int n, bool pack) {
  return n <= kLexWideMax ? lex_smem(d.K, d.G, pack, kLexOptWide, kLexCellsWide)
                            : lex_smem(d.K, d.G, pack, kLexOptWarp, kLexCellsWarp);
}

bool lex_needs_scratch(const Dims& d, int n, bool pack) { return lex_layout(d, n, pack).n_cells == 0; }

template <bool PACK, int NW>
static cudaError_t launch_lex(const Set& set, int n, const float* cap_x, const float* tail_x, fs_allocation* out,
                              void* scratch, int per_launch, const LexSmem& lay, cudaStream_t s, HostOut host) {
  constexpr int kPerBlock = NW == 1 ? 4 : 1;
  auto kern = k_solve_lex<PACK, NW>;
  const size_t smem = kPerBlock * lay.total;
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  for (int r0 = 0; r0 < n; r0 += per_launch) {
    const int m = n - r0 < per_launch ? n - r0 : per_launch;
    e = launch_pdl(kern, dim3((m + kPerBlock - 1) / kPerBlock), dim3(NW == 1 ? 128 : 32 * NW), smem, s, set, r0 + m,
                   cap_x, tail_x, out, static_cast<unsigned char*>(scratch), r0, lay, host);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Measured (one GB300): 1000 realisations of the four-class, 64-GPU grid 66.3 ->
// 9.3 us, two of the three-class, 40-GPU grid 25 -> 8.9 us (launch included).
cudaError_t launch_solve_lex(const Set& set, int n, const float* cap_x, const float* tail_x, fs_allocation* out,
                             void* scratch, int per_launch, bool pack, cudaStream_t s, HostOut host) {
  const LexSmem lay = lex_layout(set.d, n, pack);
  auto go = n <= kLexWideMax ? (pack ? launch_lex<true, kLexWideWarps> : launch_lex<false, kLexWideWarps>)
                               : (pack ? launch_lex<true, 1> : launch_lex<false, 1>);
  return go(set, n, cap_x, tail_x, out, scratch, per_launch, lay, s, host);
}

// Rows a (realisation, class) can want: t* = 0, every threshold, one above them.
static long long goodput_rows_per_class(const Dims& d, int th_bound) {
  const int bound = th_bound > 0 && th_bound < d.theta_cap ? th_bound : d.theta_cap;
  return 2LL * (bound + 2);
}

size_t goodput_pool_rows(const Dims& d, size_t most_bytes) {
  const long long per = goodput_rows_per_class(d, d.theta_cap);
  const long long row = 8LL * (d.G + 1 + kT);
  long long classes = (long long)most_bytes / (per * row);
  classes = classes < 1 ? 1 : classes > d.K ? d.K : classes;
  return (size_t)(classes * per);
}

size_t goodput_row_bytes(const Dims& d) { return 8 * (size_t)(d.G + 1 + kT); }

cudaError_t launch_score_goodput(const Set& set, const Items& it, const Plan& pl, const float* tables,
                                 uint64_t* sums, int* span, long long* base, void* pool, size_t pool_rows,
                                 int floors, int th_bound, int sm_count, cudaStream_t s) {
  const Dims& d = set.d;
  const bool rf = set.prior == 1;
  GoodputTables gt{};
  gt.span = span;
  gt.first = span + kGoodputSpanInts;
  gt.base = base;
  gt.rows = static_cast<long long*>(pool);
  gt.stride = d.G + 1 + kT;
  gt.pool = (int)pool_rows;
  const long long per = goodput_rows_per_class(d, th_bound);
  const int classes = (int)(gt.pool / per);  // classes a pass (all of them unless the pool is at its limit)
  if (classes < 1) return cudaErrorInvalidValue;
  const OtherSmem lay = other_smem(d.K, d.G);
  auto other = floors ? k_other<true> : k_other<false>;
  auto closed = floors ? k_goodput_closed<true> : k_goodput_closed<false>;
  const size_t smem = 8 * (size_t)(rf ? 2 * pl.W : pl.W + 1);
  auto kern = floors ? (rf ? k_score_goodput<true, true> : k_score_goodput<true, false>)
                     : (rf ? k_score_goodput<false, true> : k_score_goodput<false, false>);
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(other), lay.total);
  if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  // one block per segment: segments differ in cost, and the block scheduler
  // evens them out
  const long long n_seg = (long long)it.n * pl.O;
  // beyond a few waves of blocks the closed-gate goodputs are evaluated once per
  // candidate rather than by each of its segments (with the block-wide k_other 294 us
  // in all on the largest call, 352 us without both; 1.2 us more of a launch on the
  // paper-scale one, whose 512 segments are one wave)
  gt.closed = !rf && n_seg > 8LL * sm_count ? base + 2 : nullptr;
  const unsigned grid = (unsigned)(n_seg < 0x7fffffffLL ? n_seg : 0x7fffffffLL);
  // many segments: 128 threads (a segment's set-up is paid by fewer; the largest call
  // 288.7 -> 269.4 us); one wave keeps 256
  const int gthreads = gt.closed ? 128 : 256;
  for (gt.c0 = 0; gt.c0 < d.K; gt.c0 = gt.c1) {
    gt.c1 = gt.c0 + classes < d.K ? gt.c0 + classes : d.K;
    // a block per row wanted, as many as run at once (the count is not known
    // here; the rows are dealt to the blocks)
    const long long most = (long long)(gt.c1 - gt.c0) * per + 2;
    const long long fit = 8LL * sm_count;
    e = launch_pdl(other, dim3((unsigned)(most < fit ? most : fit)), dim3(kOtherThreads), lay.total, s, set, gt, lay);
    if (e == cudaSuccess && gt.closed)
      e = launch_pdl(closed, dim3((unsigned)((2LL * it.n + 127) / 128)), dim3(128), 0, s, set, it, pl, tables, gt);
    if (e != cudaSuccess) return e;
    if (it.n > 0) e = launch_pdl(kern, dim3(grid), dim3(gthreads), smem, s, set, it, pl, tables, sums, gt);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_finalize_goodput(const Set& set, const Items& it, const Plan& pl, const uint64_t* sums,
                                    const long long* base, double lam_sum, double* gap, double* score, double* gamma,
                                    int32_t* best, uint32_t* status_copy, uint64_t* part, uint64_t* sum_out,
                                    cudaStream_t s) {
  const int nb = std::max(1, finalize_blocks(it));
  return launch_pdl(k_finalize_goodput, dim3(nb), dim3(256), 0, s, set, it, pl, sums, base, lam_sum, gap, score, gamma,
                    best, status_copy, part, sum_out);
}

}  // namespace fs
