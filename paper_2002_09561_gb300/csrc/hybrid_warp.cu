// Hybrid SD / K-best (Sec. VI) in two kernels: one received vector per warp, and
// a CTA for each vector with many prefixes to finish.
//
// Most vectors need one K-best run: the best prefix's leaf shrinks the radius
// below every other prefix.  A run is a serial chain of levels, so what counts
// is how many run at once: select_run (select_run.cuh) needs no R in shared
// memory, so 28 vectors share an SM where the sorting form (kbest.cu), which
// stages R and sorts with CTA barriers, held one 100x100 vector on an SM of its
// own.  The master keeps no sorted list either: a pass over the P^d prefixes
// finds the best one inside the sphere after the last (128 evaluations a lane
// for 4,096 prefixes, 3 % of a run).  Four vectors in five have prefixes left after
// their first runs, one in eight more than 256; they go on in CTAs whose warps take a
// vector's prefixes in order under a shared radius.
// Vectors whose candidates tie for the last place kept go to the sorting form.
//
// Measured, whole calls with the QR (before: the CTA form for every vector):
// 4,000 vectors 100x100 64-QAM K = 32, depth 4, 20 to 32 dB 29.2 -> 17.3 ms (first
// runs 2.2 ms, large CTAs 3.3, small CTAs 1.8, QR 10); 2,000 vectors 96x96 16-QAM
// K = 48 13 -> 8; 1,000 vectors 12x12 64-QAM K = 8 0.57 -> 0.13.
#include <algorithm>
#include <cstddef>

#include "sd_common.cuh"
#include "select_run.cuh"

namespace mdx {
namespace {

constexpr int kWarps = 4;   // vectors per CTA of the first runs
constexpr int kRuns = 4;    // first runs at most, and the levels of those after the
constexpr int kMore = 64;   // first with a leaf
constexpr int kFew = 256;   // prefixes left: up to so many, a small CTA
constexpr int kSmall = 4;   // its warps
constexpr int kHelp = 8;    // large CTAs that may share a vector
constexpr int kOver = 1 << 30;
constexpr int kMany = 16;   // prefixes a warp runs at once at most
template <int SL>
constexpr int kLarge = SL == 1 ? 28 : 20;  // warps of a large CTA (registers: all of an SM's)

// The least (distance bits, prefix) above `after` among the prefixes inside
// the bound, and how many there are above it; digit l of a prefix is row
// n - 1 - l's index.
template <int P, int D>
__device__ __noinline__ uint64_t next_prefix_d(const float* __restrict__ Rg, const float* __restrict__ yg, int n,
                                               float alpha, float bnd, uint64_t after, int lane, int* count) {
  constexpr int kLog = P == 2 ? 1 : P == 4 ? 2 : 3;
  float R[D ? D : 1][D ? D : 1], y[D ? D : 1];  // R[l][m]: row n - 1 - l, column n - 1 - m
#pragma unroll
  for (int l = 0; l < D; ++l) {
    y[l] = yg[n - 1 - l];
#pragma unroll
    for (int m = 0; m <= l; ++m) R[l][m] = Rg[col_off(n - 1 - m) + n - 1 - l];
  }
  uint64_t best = kInfKey;
  int above = 0;
  for (int q = lane; q < 1 << (kLog * D); q += 32) {
    float a[D ? D : 1], ped = 0.0f;
#pragma unroll
    for (int l = 0; l < D; ++l) {
      a[l] = (float)(2 * ((q >> (kLog * l)) & (P - 1)) - (P - 1)) * alpha;
      float c = y[l];
#pragma unroll
      for (int m = 0; m < l; ++m) c = fmaf(-R[l][m], a[m], c);
      const float dd = fmaf(-R[l][l], a[l], c);
      ped = fmaf(dd, dd, ped);
    }
    if (ped < bnd) {
      const uint64_t key = ((uint64_t)__float_as_uint(ped) << 32) | (unsigned)q;
      if (key > after || after == kInfKey) {
        best = kmin(best, key);
        ++above;
      }
    }
  }
  *count = __reduce_add_sync(0xffffffffu, above);
  return warp_min_u64(best);
}

template <int P>
__device__ __forceinline__ uint64_t next_prefix(int D, const float* Rg, const float* yg, int n, float alpha, float bnd,
                                                uint64_t after, int lane, int* count) {
  switch (D) {
    case 0: return next_prefix_d<P, 0>(Rg, yg, n, alpha, bnd, after, lane, count);
    case 1: return next_prefix_d<P, 1>(Rg, yg, n, alpha, bnd, after, lane, count);
    case 2: return next_prefix_d<P, 2>(Rg, yg, n, alpha, bnd, after, lane, count);
    case 3: return next_prefix_d<P, 3>(Rg, yg, n, alpha, bnd, after, lane, count);
    default: return next_prefix_d<P, 4>(Rg, yg, n, alpha, bnd, after, lane, count);
  }
}

// The partial distance of one prefix, and its nibbles.
template <int P>
__device__ float prefix_distance(int D, int q, const float* __restrict__ Rg, const float* __restrict__ yg, int n,
                                 float alpha) {
  constexpr int kLog = P == 2 ? 1 : P == 4 ? 2 : 3;
  float ped = 0.0f;
  for (int l = 0; l < D; ++l) {
    float c = yg[n - 1 - l];
    for (int m = 0; m < l; ++m)
      c = fmaf(-Rg[col_off(n - 1 - m) + n - 1 - l], (float)(2 * ((q >> (kLog * m)) & (P - 1)) - (P - 1)) * alpha, c);
    const float dd = fmaf(-Rg[col_off(n - 1 - l) + n - 1 - l],
                          (float)(2 * ((q >> (kLog * l)) & (P - 1)) - (P - 1)) * alpha, c);
    ped = fmaf(dd, dd, ped);
  }
  return ped;
}
template <int P>
__device__ __forceinline__ uint32_t prefix_word(int D, unsigned q) {
  constexpr int kLog = P == 2 ? 1 : P == 4 ? 2 : 3;
  uint32_t word = 0;
  for (int l = 0; l < D; ++l) word |= ((q >> (kLog * l)) & (P - 1)) << (4 * l);
  return word;
}
template <int SL>
__device__ __forceinline__ float nearest_leaf(const float (&ped)[SL], int S, int lane) {
  float near = INFINITY;
#pragma unroll
  for (int t = 0; t < SL; ++t)
    if (lane + 32 * t < S) near = fminf(near, ped[t]);
  return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(near)));
}
// Survivor s's path as one index per row.
__device__ __forceinline__ void unpack_path(const uint32_t* x, int KS, int s, int n, uint8_t* cx, int lane) {
  for (int r = lane; r < n; r += 32) {
    const int d = n - 1 - r;
    cx[r] = (uint8_t)((x[(d >> 3) * KS + s] >> (4 * (d & 7))) & 15u);
  }
}
// A slot for a leaf at distance p, the list locked; -1: not among the best
// kCandMax (the list not locked).  Two equally near for the last place are noted
// (budget_hit: the least such distance).  The holder copies one path, so the wait is
// short; it is bounded all the same (then the vector is left: budget_hit -1).
__device__ int take_slot(SdVec* st, float p) {
  bool got = false;
  for (int it = 0; it < (1 << 16) && !got; ++it) {
    got = atomicCAS(&st->lock, 0, 1) == 0;
    if (!got) __nanosleep(64);
  }
  if (!got) {
    atomicExch(&st->budget_hit, -1);
    return -1;
  }
  __threadfence();
  int slot = *(volatile int*)&st->ncand;
  if (slot < kCandMax) {
    *(volatile int*)&st->ncand = slot + 1;
  } else {
    float worst = -1.0f;
    int equal = 0;
    for (int t = 0; t < kCandMax; ++t) {
      const float c = ((volatile float*)st->cand_ped)[t];
      equal = c > worst ? 1 : equal + (c == worst ? 1 : 0);
      if (c > worst) {
        worst = c;
        slot = t;
      }
    }
    if (p == worst || (p < worst && equal > 1)) {
      // (an arrival at the last one's distance, or one of several such leaves goes)
      const int hit = *(volatile int*)&st->budget_hit, tied = __float_as_int(worst);
      if (hit == 0 || (hit > 0 && tied < hit)) atomicCAS(&st->budget_hit, hit, tied);
    }
    if (!(p < worst)) {
      __threadfence();
      atomicExch(&st->lock, 0);
      return -1;
    }
  }
  ((volatile float*)st->cand_ped)[slot] = p;
  return slot;
}

// FP64 ||ybar - R x||^2 by one warp with the sums of the sorting form's eight
// warps (kbest.cu: columns j = w, w + 8, ... to partial w, partials added in
// order), so that both forms return the same bits.
__device__ double rescore_fp64_split(int n, int P, double alpha64, const double* __restrict__ R64,
                                     const double* __restrict__ y64, const uint8_t* x, int lane) {
  const double lv = (double)(2 * (lane < P ? lane : 0) - (P - 1)) * alpha64;
  double s = 0.0;
  for (int t = 0; 32 * t < n; ++t) {
    const int r = lane + 32 * t;
    double part[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) part[w] = w == 0 && r < n ? y64[r] : 0.0;
    for (int j0 = 32 * t; j0 < n; j0 += 8) {
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        const int j = j0 + w;
        const double xj = __shfl_sync(0xffffffffu, lv, (int)x[min(j, n - 1)]);
        if (j < n && r <= j) part[w] = fma(-R64[col_off(j) + r], xj, part[w]);
      }
    }
    double z = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) z += part[w];
    if (r < n) s = fma(z, z, s);
  }
  return __shfl_sync(0xffffffffu, warp_sum(s), 0);
}

// Re-scores the candidates within FP32 error of the best in FP64 and writes the
// vector's outputs (one warp).  restarts: the doublings of the initial radius
// until the best candidate is inside; the candidates outside then do not count.
__device__ void finish_hybrid(const SearchArgs& a, int v, const uint8_t* cx, int cs, const float* cped, int nc, float E,
                              long long nodes, long long flops, int lane) {
  const int n = a.n, P = a.P;
  float best = INFINITY;
  for (int t = 0; t < nc; ++t) best = fminf(best, cped[t]);
  float r = initial_r2(a, v);
  int restarts = 0;
  for (; !(best < prune_bound(r, E, n)) && r < INFINITY && restarts < 64; ++restarts) r *= 2.0f;
  if (!(best < prune_bound(r, E, n))) nc = 0;
  const float inside = prune_bound(r, E, n), keep = prune_bound(best, E, n);
  const double* R64 = a.R64 + (size_t)v * tri_stride64(n);
  const double* y64 = a.yb64 + (size_t)v * vec_stride64(n);
  int win = -1;
  double win_m = INFINITY;
  long long rescored = 0;
  for (int t = 0; t < nc; ++t) {
    if (!(cped[t] <= keep && cped[t] < inside)) continue;
    const uint8_t* px = cx + (size_t)t * cs;
    double m;
    if (a.flags & MDX_NO_RESCORE) {
      m = (double)cped[t];
    } else {
      m = rescore_fp64_split(n, P, a.alpha64, R64, y64, px, lane);
      ++rescored;
    }
    bool better = m < win_m;
    if (!better && m == win_m && win >= 0) {
      // tie: lexicographically smaller index vector, top row first
      const uint8_t* pw = cx + (size_t)win * cs;
      for (int j = n - 1; j >= 0; --j) {
        if (px[j] != pw[j]) {
          better = px[j] < pw[j];
          break;
        }
      }
    }
    if (better) {
      win = t;
      win_m = m;
    }
  }
  for (int j = lane; j < a.n_tx; j += 32) {
    const uint8_t* pw = cx + (size_t)(win < 0 ? 0 : win) * cs;
    a.sym_out[(size_t)v * a.n_tx + j] = win >= 0 ? (uint8_t)(pw[2 * j] * P + pw[2 * j + 1]) : 0;
  }
  if (lane == 0) {
    a.metric_out[v] = (win >= 0) ? win_m : (double)INFINITY;
    a.vstatus[v] = restarts > 0 ? MDX_V_EMPTY_RETRIED : MDX_V_OK;
    if (a.stats) {
      int64_t* st = a.stats + (size_t)v * kStats;
      st[0] = nodes;
      st[1] = nodes * P;
      st[2] = restarts;
      st[3] = rescored;
      st[4] = flops;
    }
  }
}

// The runs of m prefixes, lane i < m giving the i-th's distance and nibbles:
// select_run, again with ranks where it takes them.
template <int SL, int P>
__device__ __forceinline__ int prefix_run(const float* Rg, const float* yg, int n, int K, float alpha, int D, int m,
                                          float ped, uint32_t word, float bnd, const SelectWs& ws, int lane,
                                          Survivors<SL>& s, RunCost& cost) {
  int S = -1;
  for (int ranked = 0; ranked < 2 && S == -1; ++ranked) {
#pragma unroll
    for (int t = 0; t < SL; ++t) {
      s.ped[t] = ped;
      s.cur[t] = word;
    }
    if (D < n) {
      S = select_run<SL, P>(Rg, yg, n, K, alpha, D, m, bnd, ranked, ws, lane, s, cost);
    } else {
      ws.x[lane] = word;
      __syncwarp();
      S = m;
    }
  }
  return S;
}

// Leaves a vector to the sorting form.
__device__ void leave(const HybridWork& w, int v) {
  const unsigned int i = atomicAdd(&w.counts[1], 1u);
  reinterpret_cast<SdVec*>(w.state + (size_t)i * w.stride)->r2_start = __int_as_float(v);
}

// The leaves within lim join the candidates, nc of them, of which the
// kCandMax nearest are kept; tie: the least distance at which two were equally
// near for the last place (an arrival, or two kept of which one had to go).
template <int SL>
__device__ void add_leaves(const Survivors<SL>& w, int S, float lim, const SelectWs& ws, int n, SdVec* st, uint8_t* cx,
                           int cs, int& nc, float& tie, int lane) {
  for (int t = 0; t < SL; ++t) {
    unsigned who = __ballot_sync(0xffffffffu, lane + 32 * t < S && w.ped[t] <= lim);
    for (; who; who &= who - 1) {
      const int s = __ffs(who) - 1;
      const float p = __shfl_sync(0xffffffffu, w.ped[t], s);
      int slot = nc;
      if (nc < kCandMax) {
        ++nc;
      } else {
        __syncwarp();
        const unsigned c = lane < kCandMax ? __float_as_uint(st->cand_ped[lane]) : 0u;
        const unsigned worst = __reduce_max_sync(0xffffffffu, c);
        const unsigned last = __ballot_sync(0xffffffffu, c == worst && lane < kCandMax);
        if (p == __uint_as_float(worst) || (p < __uint_as_float(worst) && (last & (last - 1))))
          tie = fminf(tie, __uint_as_float(worst));
        if (!(p < __uint_as_float(worst))) continue;
        slot = __ffs(last) - 1;
      }
      if (lane == 0) st->cand_ped[slot] = p;
      unpack_path(ws.x, ws.KS, s + 32 * t, n, cx + (size_t)slot * cs, lane);
    }
  }
  __syncwarp();
}

template <int SL, int P>
__global__ void __launch_bounds__(32 * kWarps, SL == 1 ? 7 : 5)
    hybrid_warp_kernel(SearchArgs a, int ws_bytes, HybridWork w) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, v = blockIdx.x * kWarps + (threadIdx.x >> 5);
  const int n = a.n, K = a.K, D = a.depth;
  if (v >= a.batch) return;
  if (a.singular && a.singular[v]) {
    for (int j = lane; j < a.n_tx; j += 32) a.sym_out[(size_t)v * a.n_tx + j] = 0;
    if (lane == 0) {
      a.metric_out[v] = 0.0;
      a.vstatus[v] = MDX_V_SINGULAR;
      if (a.stats)
        for (int q = 0; q < kStats; ++q) a.stats[(size_t)v * kStats + q] = 0;
    }
    return;
  }
  const SelectWs ws = select_ws(smem + (size_t)(threadIdx.x >> 5) * ws_bytes, ws_bytes, nullptr, n, K);
  SdVec* st = reinterpret_cast<SdVec*>(w.state + (size_t)v * w.stride);
  uint8_t* cx = reinterpret_cast<uint8_t*>(st + 1);
  const int cs = path_pad(n);
  const float* Rg = a.R32 + (size_t)v * tri_stride32(n);
  const float* yg = a.yb32 + (size_t)v * vec_stride32(n);
  const float E = error_scale_warp(n, P, a.alpha, Rg, yg, lane);
  const float r0 = initial_r2(a, v);
  float r2 = r0;
  RunCost cost;
  cost.nodes = 1;
  int nc = 0, more = 0;
  float tie = INFINITY;
  // One prefix's run.
  auto run = [&](uint64_t key) {
    Survivors<SL> s;
    cost.nodes += 1;
    cost.flops += 2 * (D > 0 ? D - 1 : 0) + 4 * P;
    const int S = prefix_run<SL, P>(Rg, yg, n, K, a.alpha, D, 1, __uint_as_float((unsigned)(key >> 32)),
                                    prefix_word<P>(D, (unsigned)key), prune_bound(r2, E, n), ws, lane, s, cost);
    if (S <= 0) return;
    // the run's leaves within FP32 error of the best so far join the candidates
    const float near = nearest_leaf<SL>(s.ped, S, lane);
    if (near < r2) {
      r2 = near;
      // earlier ones may be out now
      const float lim = prune_bound(r2, E, n);
      __syncwarp();
      int kept = 0;
      for (int t = 0; t < nc; ++t) {
        const float p = st->cand_ped[t];
        if (p <= lim) {
          __syncwarp();
          if (lane == 0) st->cand_ped[kept] = p;
          if (kept != t)
            for (int i = lane; i < n; i += 32) cx[(size_t)kept * cs + i] = cx[(size_t)t * cs + i];
          ++kept;
        }
        __syncwarp();
      }
      nc = kept;
    }
    add_leaves<SL>(s, S, prune_bound(r2, E, n), ws, n, st, cx, cs, nc, tie, lane);
  };
  // The best prefix's run; without a leaf (or without a prefix) inside the
  // sphere, the run without a radius: doubling the radius until the sphere
  // holds a leaf ends with the best leaf there is, which is below this run's,
  // and finish_hybrid tells from its distance how often that is.  (Statistics
  // count the passes: such vectors are left.)
  uint64_t key = next_prefix<P>(D, Rg, yg, n, a.alpha, prune_bound(r2, E, n), kInfKey, lane, &more);
  if (key != kInfKey) run(key);
  if (nc == 0 && r0 < INFINITY) {
    if (a.stats) {
      if (lane == 0) leave(w, v);
      return;
    }
    r2 = INFINITY;
    if (key == kInfKey) key = next_prefix<P>(D, Rg, yg, n, a.alpha, INFINITY, kInfKey, lane, &more);
    if (key != kInfKey) run(key);
  }
  // The next ones in order: a first leaf can be far from the best, and the
  // radius of the best of a few spares the many warps that share the rest
  const int levels = cost.levels;
  uint64_t next = kInfKey;
  for (int t = 1; nc > 0; ++t) {
    next = next_prefix<P>(D, Rg, yg, n, a.alpha, prune_bound(r2, E, n), key, lane, &more);
    if (next == kInfKey || t == kRuns || cost.levels - levels >= kMore) break;
    run(next);
    key = next;
  }
  if (next != kInfKey) {  // more prefixes inside what is now the sphere
    if (lane == 0) {
      st->r2bits = __float_as_uint(r2);
      st->pending = more <= kFew ? 1 : kHelp;  // CTAs to come
      st->restarts = 0;                        // the next of the sorted prefixes
      st->lock = 0;
      st->ncand = nc;
      st->nodes = (unsigned long long)cost.nodes;
      st->peds = key;  // the prefixes up to it are done
      st->flops = (unsigned long long)cost.flops;
      // a tie that counts unless the radius shrinks past it (-1: left to the sorting form)
      st->budget_hit = tie < INFINITY ? __float_as_int(tie) : 0;
      st->E = E;
      if (more <= kFew)
        w.list[atomicAdd(&w.counts[0], 1u)] = v;
      else
        w.list[a.batch - 1 - (int)atomicAdd(&w.counts[3], 1u)] = v;
    }
    return;
  }
  if (tie <= prune_bound(r2, E, n) && tie < INFINITY) {
    if (lane == 0) leave(w, v);
    return;
  }
  __syncwarp();
  finish_hybrid(a, v, cx, cs, st->cand_ped, nc, E, cost.nodes, cost.flops, lane);
}

// The prefixes the first runs left inside the sphere: a vector to a CTA,
// sorted, the warps taking them in order (best-first, as the paper's master
// explores: the radius shrinks before the farther ones come up).  Up to kFew of
// them and small CTAs side by side, thousands and a CTA of all the SM's warps;
// once every such vector has its CTA, further ones join those still at work
// (each sorts for itself: the keys are unique, so all see one order, and take
// from one counter; 1,000 vectors 100x100: the slowest alone 4.1 ms).
// A warp runs several at a time (most of them end after a few levels): as many
// as the last run's peak lets expect to fit, half as many when they do not.
template <int SL, int P, int W>
__global__ void __launch_bounds__(32 * W, W == kSmall ? (SL == 1 ? 7 : 5) : 1)
    hybrid_share_kernel(SearchArgs a, int ws_bytes, int cap, HybridWork w) {
  constexpr int kLog = P == 2 ? 1 : P == 4 ? 2 : 3;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int at, nin, last, going;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = 32 * W;
  const int n = a.n, K = a.K, D = a.depth, np = 1 << (kLog * D);
  uint16_t* pidx = reinterpret_cast<uint16_t*>(smem);
  unsigned char* wsm = smem + ((size_t)cap * sizeof(uint16_t) + 15) / 16 * 16;
  uint64_t* keys = reinterpret_cast<uint64_t*>(wsm);  // before the runs
  const SelectWs ws = select_ws(wsm + (size_t)warp * ws_bytes, ws_bytes, nullptr, n, K);
  const int cs = path_pad(n);
  const int count = (int)w.counts[W == kSmall ? 0 : 3];
  for (;;) {
    if (tid == 0) {
      at = (int)atomicAdd(W == kSmall ? a.work_counter : &w.counts[4], 1u);
      nin = 0;
    }
    __syncthreads();
    if (at >= count * (W == kSmall ? 1 : kHelp)) break;
    const int v = w.list[W == kSmall ? at : a.batch - 1 - at % count];
    SdVec* st = reinterpret_cast<SdVec*>(w.state + (size_t)v * w.stride);
    uint8_t* cx = reinterpret_cast<uint8_t*>(st + 1);
    const float* Rg = a.R32 + (size_t)v * tri_stride32(n);
    const float* yg = a.yb32 + (size_t)v * vec_stride32(n);
    const float E = __ldcg(&st->E);
    const uint64_t done = __ldcg(&st->peds);
    auto bound = [&]() {
      return prune_bound(__uint_as_float(__shfl_sync(0xffffffffu, __ldcg(&st->r2bits), 0)), E, n);
    };
    RunCost cost;
    if (tid == 0) going = __ldcg(&st->restarts) < kOver;
    __syncthreads();
    if (going) {
      // (a warp that sees a smaller radius here leaves out prefixes outside it: up
      // to the first such one every CTA's order is the same, and the others are
      // outside as well)
      float bnd = bound();
      for (int q = tid; q < np; q += T) {
        const float p = prefix_distance<P>(D, q, Rg, yg, n, a.alpha);
        const uint64_t key = ((uint64_t)__float_as_uint(p) << 32) | (unsigned)q;
        if (p < bnd && key > done) keys[atomicAdd(&nin, 1)] = key;
      }
      __syncthreads();
      const int total = nin, Cs = pow2ceil(total < 2 ? 2 : total);
      for (int q = total + tid; q < Cs; q += T) keys[q] = kInfKey;
      __syncthreads();
      bitonic_sort(keys, Cs, tid, T);
      for (int q = tid; q < total; q += T) pidx[q] = (uint16_t)(keys[q] & 0xffffu);
      __syncthreads();
      int many = 1, t = 0, end = 0;  // the warp's prefixes
      for (;;) {
        if (t == end) {
          if (lane == 0) t = atomicAdd(&st->restarts, many);
          t = __shfl_sync(0xffffffffu, t, 0);
          end = min(t + many, total);
          if (t >= total) {
            if (lane == 0) atomicMax(&st->restarts, kOver);
            break;
          }
        }
        int m = min(many, end - t);
        bnd = bound();
        const int q = pidx[t + min(lane, m - 1)];
        const float dist = prefix_distance<P>(D, q, Rg, yg, n, a.alpha);
        const int in = __popc(__ballot_sync(0xffffffffu, lane < m && dist < bnd));  // in order: the first ones
        if (in < m) {  // and so is every later one
          if (lane == 0) atomicMax(&st->restarts, kOver);
          m = in;
          end = t + m;
          if (m == 0) break;
        }
        Survivors<SL> s;
        const int S = prefix_run<SL, P>(Rg, yg, n, K, a.alpha, D, m, dist, prefix_word<P>(D, (unsigned)q), bnd, ws, lane, s,
                                        cost);
        if (S == -2) {  // the same ones again, fewer at a time
          many = max(m >> 1, 1);
          continue;
        }
        cost.nodes += m;
        cost.flops += m * (2 * (D > 0 ? D - 1 : 0) + 4 * P);
        t += m;
        if (S <= 0) {
          // three quarters full at the last run's peak
          many = max(1, min(min(many + 1, kMany), 3 * K * m / (4 * max(cost.peak, 1))));
          continue;
        }
        const float near = nearest_leaf<SL>(s.ped, S, lane);
        unsigned was = 0;
        if (lane == 0) was = atomicMin(&st->r2bits, __float_as_uint(near));
        const float lim = prune_bound(fminf(near, __uint_as_float(__shfl_sync(0xffffffffu, was, 0))), E, n);
        // the leaves within FP32 error of the best so far join the candidates
        for (int j = 0; j < SL; ++j) {
          unsigned who = __ballot_sync(0xffffffffu, lane + 32 * j < S && s.ped[j] <= lim);
          for (; who; who &= who - 1) {
            const int i = __ffs(who) - 1;
            const float p = __shfl_sync(0xffffffffu, s.ped[j], i);
            int slot = -1;
            if (lane == 0) slot = take_slot(st, p);
            slot = __shfl_sync(0xffffffffu, slot, 0);
            if (slot < 0) continue;
            unpack_path(ws.x, ws.KS, i + 32 * j, n, cx + (size_t)slot * cs, lane);
            __threadfence();
            __syncwarp();
            if (lane == 0) atomicExch(&st->lock, 0);
          }
        }
      }
    }
    if (lane == 0) {
      atomicAdd(&st->nodes, (unsigned long long)cost.nodes);
      atomicAdd(&st->flops, (unsigned long long)cost.flops);
      __threadfence();
    }
    __syncthreads();
    if (tid == 0) {
      last = atomicSub(&st->pending, 1) == 1;
      __threadfence();
    }
    __syncthreads();
    if (warp == 0 && last) {
      // (nothing has read the candidates through this SM's L1)
      const int hit = __ldcg(&st->budget_hit);
      if (hit < 0 || (hit > 0 && __int_as_float(hit) <= bound())) {
        if (lane == 0) leave(w, v);
      } else {
        float* cped = reinterpret_cast<float*>(ws.ent);
        if (lane < kCandMax) cped[lane] = __ldcg(&st->cand_ped[lane]);
        __syncwarp();
        finish_hybrid(a, v, cx, cs, cped, __ldcg(&st->ncand), E, (long long)__ldcg(&st->nodes),
                      (long long)__ldcg(&st->flops), lane);
      }
    }
    __syncthreads();
  }
}

template <int SL, int P, int W>
cudaError_t launch_share(const SearchArgs& a, const HybridWork& w, int ws, int cap, int num_sms, cudaStream_t s) {
  const size_t sm = (sizeof(uint16_t) * (size_t)cap + 15) / 16 * 16 + std::max((size_t)ws * W, sizeof(uint64_t) * cap);
  int per_sm = 0;
  cudaError_t e =
      cudaFuncSetAttribute(hybrid_share_kernel<SL, P, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hybrid_share_kernel<SL, P, W>, 32 * W, sm);
  if (e != cudaSuccess) return e;
  hybrid_share_kernel<SL, P, W>
      <<<W == kSmall ? std::min(a.batch, std::max(per_sm, 1) * num_sms) : num_sms, 32 * W, sm, s>>>(a, ws, cap, w);
  return cudaGetLastError();
}

template <int SL, int P>
cudaError_t launch_hw(const SearchArgs& a, const HybridWork& w, int num_sms, cudaStream_t s) {
  const int ws = (int)((select_level_bytes(a.n, a.K) + select_path_bytes(a.n, a.K) + 15) / 16 * 16);
  const size_t sm = (size_t)ws * kWarps;
  cudaError_t e = cudaFuncSetAttribute(hybrid_warp_kernel<SL, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  hybrid_warp_kernel<SL, P><<<(a.batch + kWarps - 1) / kWarps, 32 * kWarps, sm, s>>>(a, ws, w);
  e = cudaGetLastError();
  const int np = 1 << ((P == 2 ? 1 : P == 4 ? 2 : 3) * a.depth);
  if (e == cudaSuccess && np > kFew) e = launch_share<SL, P, kLarge<SL>>(a, w, ws, np, num_sms, s);
  if (e == cudaSuccess && np > 1) e = launch_share<SL, P, kSmall>(a, w, ws, 2 * kFew, num_sms, s);
  return e;
}
template <int SL>
cudaError_t launch_hw_p(const SearchArgs& a, const HybridWork& w, int num_sms, cudaStream_t s) {
  if (a.P == 2) return launch_hw<SL, 2>(a, w, num_sms, s);
  if (a.P == 4) return launch_hw<SL, 4>(a, w, num_sms, s);
  return launch_hw<SL, 8>(a, w, num_sms, s);
}

}  // namespace

size_t hybrid_redo_offset() { return offsetof(SdVec, r2_start); }

// Runs for K <= 64, prefixes of at most four rows and no node budget (the
// budget counts the prefixes in the sorting form's order); else
// cudaErrorNotSupported, nothing launched.  Nor for statistics of a few vectors
// with the network's radius, which leaves one sphere in ten empty: their passes are
// counted by the sorting form, behind the runs here (20 vectors 100x100 64-QAM
// K = 32: 4.2 ms so, 3.0 by that form alone; 200: 11.2).
cudaError_t launch_hybrid_warp(const SearchArgs& a, const HybridWork& w, int num_sms, cudaStream_t s) {
  if (a.K > 64 || a.depth > 4 || a.budget > 0) return cudaErrorNotSupported;
  if (a.stats && a.radius_mode == RADIUS_PER_VECTOR && a.batch <= num_sms) return cudaErrorNotSupported;
  return a.K <= 32 ? launch_hw_p<1>(a, w, num_sms, s) : launch_hw_p<2>(a, w, num_sms, s);
}

}  // namespace mdx
