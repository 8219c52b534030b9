// Uneven batches: two persistent search kernels, side by side (walk_kernel for
// exact SDs, mixed_kernel for the others), over requests that differ in
// antennas, modulation, detector and K (the batching layer around the
// paper's detectors; the paper runs one system at a time).
//
// Every warp of a grid takes requests from a global counter, in the order
// the host chose (heaviest classes first), and searches each one alone:
//   exact SD   Algorithm 1 with Schnorr-Euchner child order (Sec. IV-A) and
//              incremental partial distances (Eq. inc), one warp walking the
//              whole tree (sd_walk);
//   K-best     Sec. VI, selection of the K best children per level
//              (select_run.cuh for K <= 64; for larger K a warp tournament over
//              the survivors' Schnorr-Euchner child streams, warp_kbest.cuh).
// What bounds a batch is the longest walk: one warp, one node after another,
// thousands of them, or one K-best level after another.  Both are therefore
// written for the latency of a step (see sd_walk), and the grid holds as many
// warps as the shared memory of a walk allows.
// Each warp owns a slice of the CTA's shared memory and a slot of global
// memory.  SD walks and K-best selections use what fits of them by themselves.
// For the other forms (natural-order and complex-tree SD, K > 64) the tuner
// decides per request class whether R and ybar are copied into the slice
// (MIX_STAGE_R) and whether the search state lives in the slice
// (MIX_STATE_SMEM) or in the global slot; the kernel uses generic pointers,
// so one code path serves every placement.  Leaves within the FP32 error
// bound of the best are re-scored in FP64 against the FP64 R and ybar.
#include <algorithm>

#include "mdx_internal.cuh"
#include "select_run.cuh"

namespace mdx {
namespace {

constexpr int kMixCand = 8;  // SD leaf candidates kept per request

__host__ __device__ inline size_t stage_bytes(int n) {
  return sizeof(float) * ((size_t)tri_stride32(n) + round_up(n, 4));
}

__host__ __device__ inline int mix_path_pad(int n) { return round_up(n, 16); }

__host__ __device__ inline size_t sd_state_bytes(int n) {
  const size_t n4 = (size_t)round_up(n, 4);
  const size_t b = sizeof(float) * (round_up(tri(n), 4) + 3 * n4) + sizeof(int) * n4 + sizeof(float) * kMixCand +
                   (size_t)mix_path_pad(n) * (1 + kMixCand);
  return (b + 15) / 16 * 16;
}

// Complex-tree SD: residual stack, per complex level {parent distance, c of
// row 2j+1, c of row 2j before x_{2j+1}, visited-children mask low word} and
// the mask's high word, level constants {R_{2j+1,2j+1}, R_{2j,2j+1}, R_{2j,2j}},
// candidates, path.
__host__ __device__ inline size_t sdc_state_bytes(int n) {
  const size_t M = (size_t)n / 2;
  const size_t b = sizeof(float) * round_up(tri(n), 4) + 16 * M + sizeof(unsigned) * round_up((int)M, 4) +
                   16 * M + sizeof(float) * kMixCand + (size_t)mix_path_pad(n) * (1 + kMixCand);
  return (b + 15) / 16 * 16;
}

__host__ __device__ inline size_t kb_state_bytes(int n, int K) {
  const size_t b = 16 + 2 * sizeof(float) * round_up(K, 4) + 2 * sizeof(uint16_t) * round_up(K, 8) +
                   2 * (size_t)path_stride(n) * K;
  return (b + 15) / 16 * 16;
}

__device__ float initial_r2(const MixedArgs& g, const MixedReq& q, int r) {
  float r2;
  if (q.radius_mode == RADIUS_PER_VECTOR) r2 = g.r2_vec[r];
  else if (q.radius_mode == RADIUS_NONE) r2 = INFINITY;
  else if (q.radius_mode == RADIUS_PAPER) r2 = (float)((double)q.n_rx * q.n_tx * g.noise_var[r]);
  else r2 = (float)q.radius_value;
  return (r2 > 0.0f) ? r2 : INFINITY;
}

// Picks, among nc candidate paths (stride cs bytes) with FP32 distances cped,
// the one of least FP64 metric (ties: smaller index vector, top row first)
// among those within the FP32 error bound of the best; writes the request's
// outputs.  All lanes call it.
__device__ void finish_request(const MixedArgs& g, const MixedReq& q, int r, const uint8_t* cx, int cs,
                               const float* cped, int nc, float E, int status, long long nodes, long long peds,
                               long long restarts, long long flops, int lane) {
  const int n = q.n, P = q.P;
  float best = INFINITY;
  for (int k = 0; k < nc; ++k) best = fminf(best, cped[k]);
  const float keep = prune_bound(best, E, n);
  const double* R64 = g.R64 + q.r_off64;
  const double* y64 = g.yb64 + q.y_off64;
  int win = -1;
  double win_m = INFINITY;
  long long rescored = 0;
  for (int k = 0; k < nc; ++k) {
    if (!(cped[k] <= keep)) continue;
    double m;
    if (g.flags & MDX_NO_RESCORE) {
      m = (double)cped[k];
    } else {
      m = rescore_fp64_warp(n, P, q.alpha64, R64, y64, cx + (size_t)k * cs, lane);
      ++rescored;
    }
    bool better = m < win_m;
    if (!better && m == win_m && win >= 0) {
      for (int j = n - 1; j >= 0; --j) {
        const int x1 = cx[(size_t)k * cs + j], x2 = cx[(size_t)win * cs + j];
        if (x1 != x2) {
          better = x1 < x2;
          break;
        }
      }
    }
    if (better) {
      win = k;
      win_m = m;
    }
  }
  uint8_t* so = g.sym_out + q.sym_off;
  for (int j = lane; j < q.n_tx; j += 32)
    so[j] = (win >= 0) ? (uint8_t)(cx[(size_t)win * cs + 2 * j] * P + cx[(size_t)win * cs + 2 * j + 1]) : 0;
  if (lane == 0) {
    g.metric_out[r] = (win >= 0) ? win_m : (double)INFINITY;
    g.vstatus[r] = status;
    if (g.stats) {
      int64_t* s = g.stats + (size_t)r * kStats;
      s[0] = nodes;
      s[1] = peds;
      s[2] = restarts;
      s[3] = rescored;
      s[4] = flops;
    }
  }
}

// Keeps the leaf xs at distance ped among the kMixCand best.
__device__ void keep_leaf(const uint8_t* xs, int n, float ped, uint8_t* cx, int cs, float* cped, int& ncand, int lane) {
  int at = -1;
  if (ncand < kMixCand) {
    at = ncand;
  } else {
    float worst = -1.0f;
    for (int t = 0; t < kMixCand; ++t)
      if (cped[t] > worst) {
        worst = cped[t];
        at = t;
      }
    if (!(ped < worst)) at = -1;
  }
  __syncwarp();
  if (at >= 0) {
    for (int rr = lane; rr < n; rr += 32) cx[(size_t)at * cs + rr] = xs[rr];
    if (lane == 0) cped[at] = ped;
    if (at == ncand) ++ncand;
  }
  __syncwarp();
}

// Unsorted depth-first search (children in natural index order, the variant
// the paper compares against, Sec. IV-A) of one request by one warp (ROWS =
// rows per lane, n <= 32 ROWS): lanes own rows, the residual of every row below
// the current level sits in a stack zs[level][row].  A child outside the sphere
// does not end its level, and pops go up one level at a time.
template <int ROWS>
__device__ void sd_natural(const MixedArgs& g, const MixedReq& q, int r, const float* Rc, const float* yb,
                           unsigned char* st, float E, int lane) {
  const int n = q.n, P = q.P, n4 = round_up(n, 4);
  const float alpha = q.alpha;
  float* zs = reinterpret_cast<float*>(st);
  float* lv_ped = zs + round_up(tri(n), 4);
  float* lv_c = lv_ped + n4;
  float* lv_rii = lv_c + n4;
  int* lv_k = reinterpret_cast<int*>(lv_rii + n4);
  float* cped = reinterpret_cast<float*>(lv_k + n4);
  uint8_t* xs = reinterpret_cast<uint8_t*>(cped + kMixCand);
  uint8_t* cx = xs + mix_path_pad(n);
  const int cs = mix_path_pad(n);

  for (int rr = lane; rr < n; rr += 32) lv_rii[rr] = Rc[col_off(rr) + rr];
  float r2_start = initial_r2(g, q, r);
  float r2 = r2_start;
  long long nodes = 0, peds = 0, flops = 0;
  int restarts = 0, ncand = 0;
  bool bh = false;
  for (;;) {
    // the root: z_r = ybar_r for every row
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      const int rr = lane + 32 * t;
      if (rr < n) zs[col_off(n - 1) + rr] = yb[rr];
    }
    __syncwarp();
    float bnd = prune_bound(r2, E, n);
    int i = n - 1, next = 0;
    float ped_par = 0.0f;
    float c = zs[col_off(i) + i];
    float rii = lv_rii[i];
    ++nodes;
    flops += 4 * P;
    for (;;) {
      if (next >= P) {
        if (i == n - 1) break;  // the root is exhausted
        ++i;                    // backtrack
        ped_par = lv_ped[i];
        c = lv_c[i];
        rii = lv_rii[i];
        next = lv_k[i];
        __syncwarp();  // the level's state is read before lane 0 writes it again
        continue;
      }
      const int k = next++;
      const float d = fmaf(-rii, (float)(2 * k - (P - 1)) * alpha, c);
      const float ped = fmaf(d, d, ped_par);
      ++peds;
      if (!(ped < bnd)) continue;
      if (i == 0) {
        if (lane == 0) xs[0] = (uint8_t)k;
        __syncwarp();
        keep_leaf(xs, n, ped, cx, cs, cped, ncand, lane);
        if (ped < r2) {
          r2 = ped;
          bnd = prune_bound(r2, E, n);
        }
        continue;
      }
      if (q.budget > 0 && nodes >= q.budget) {
        bh = true;
        break;
      }
      // descend into child k: push level i, update the residuals of the rows below
      const float av = (float)(2 * k - (P - 1)) * alpha;
      const float* zin = zs + col_off(i);
      const float* rc = Rc + col_off(i);
      const float cnext = fmaf(-rc[i - 1], av, zin[i - 1]);
      if (lane == 0) {
        lv_ped[i] = ped_par;
        lv_c[i] = c;
        lv_k[i] = next;
        xs[i] = (uint8_t)k;
      }
      float* zout = zs + col_off(i - 1);
#pragma unroll
      for (int t = 0; t < ROWS; ++t) {
        const int rr = lane + 32 * t;
        if (rr < i) zout[rr] = fmaf(-rc[rr], av, zin[rr]);
      }
      --i;
      __syncwarp();
      c = cnext;
      ped_par = ped;
      rii = lv_rii[i];
      next = 0;
      ++nodes;
      flops += 2 * (n - 1 - i) + 4 * P;
    }
    if (ncand == 0 && !bh && r2_start < INFINITY && restarts < 64) {
      // empty sphere: r^2 <- 2 r^2 and search again
      r2_start *= 2.0f;
      r2 = r2_start;
      ++restarts;
      continue;
    }
    break;
  }
  __syncwarp();
  const int status = bh ? MDX_V_BUDGET_EXCEEDED : (restarts > 0 ? MDX_V_EMPTY_RETRIED : MDX_V_OK);
  finish_request(g, q, r, cx, cs, cped, ncand, E, status, nodes, peds, restarts, flops, lane);
}

// Schnorr-Euchner orders of a level's children as nibbles, by the first child
// k0 and whether u lies above it: entry 2 k0 + (u > k0) for P = 2, 4, 8.  From
// k0 (the index nearest u) the order alternates sides, starting on u's side
// (below on a tie), until one side is used up: the order in which comparing
// |u - lo| <= |hi - u| takes them, since within the constellation those
// differences decide as in exact arithmetic (for u >= k0 both are multiples of
// ulp(u) no larger than u, so exact; below k0 rounding cannot pass the integer
// that separates them), and outside it only one side is left.
constexpr unsigned zigzag(int P, int k0, bool above) {
  unsigned w = (unsigned)k0;
  int lo = k0 - 1, hi = k0 + 1;
  for (int t = 1; t < P; ++t) {
    const bool low = lo >= 0 && (hi >= P || k0 - lo < hi - k0 || (k0 - lo == hi - k0 && !above));
    w |= (unsigned)(low ? lo-- : hi++) << (4 * t);
  }
  return w;
}
struct Zigzag {
  unsigned at[3][16];
  constexpr Zigzag() : at{} {
    for (int p = 0; p < 3; ++p)
      for (int k = 0; k < (2 << p); ++k) {
        at[p][2 * k] = zigzag(2 << p, k, false);
        at[p][2 * k + 1] = zigzag(2 << p, k, true);
      }
  }
};
__constant__ Zigzag kZigzag;

// Exact SD of one request by one warp (ROWS = rows per lane, n <= 32 ROWS).
// In Schnorr-Euchner order a visited node's next sibling is evaluated with it;
// outside the sphere it finishes the level (the bound only shrinks), and a pop
// goes straight to the nearest level above with a sibling left inside (each
// level keeps that return level).  A node whose nearest child is outside the
// sphere is counted but not entered.
//
// A walk is one dependent chain, so a step is kept short: every lane forms the
// chain's values itself; what a level's descent will need (its column's entries
// for the next rows, the residual two rows down, the next row's constants) is
// loaded when the level is reached, and the next row's interference is one FMA
// from it; each child is evaluated once, its sibling kept in the level's
// record; the child order is a table of nibbles; indexes become levels in the
// FP32 adder instead of by conversions.  The residuals of the current level
// are in registers (lanes own rows), a stack zs[level][row] holds the levels
// above for pops.  The lowest levels, where a walk spends its time, have R's
// columns and the stack in the slice (as many as fit), the levels above in
// global memory, so walks of every size leave the SM full; the placement is two
// selected pointers, since branches cost more (n = 128: 9.6 ms for the 7.4).
// Measured (333 requests of 64-QAM with the QR, walks up to 20,000 nodes; before:
// the rows' update, the sibling and the first child evaluated one after
// another, everything in global memory where the stack did not fit): n = 16
// 6.8 -> 4.6 ms, n = 128 10.6 -> 7.7, n = 200 19 -> 8.9.
__host__ __device__ inline size_t walk_record_bytes(int n) { return (sizeof(float4) + sizeof(float2)) * (size_t)n; }
__host__ __device__ inline size_t walk_slot_bytes(int n) {
  const size_t b = sizeof(float) * round_up(tri(n), 4) + sizeof(float) * kMixCand +
                   (size_t)mix_path_pad(n) * kMixCand;
  return (b + 15) / 16 * 16;
}

template <int ROWS>
__device__ void sd_walk(const MixedArgs& g, const MixedReq& q, int r, const float* __restrict__ Rg,
                        const float* __restrict__ yg, unsigned char* slot, float E, int lane) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* slice = smem + (size_t)(threadIdx.x >> 5) * g.slice_bytes;
  const int n = q.n, P = q.P;
  const float alpha = q.alpha, alpha2 = 2.0f * alpha, half = 0.5f * (float)(P - 1), mid = level_mid(P);
  const unsigned* zz = kZigzag.at[P == 2 ? 0 : P == 4 ? 1 : 2];
  // ---- placement (the slice holds the records at least)
  float* zg = reinterpret_cast<float*>(slot);
  float4* rec = reinterpret_cast<float4*>(slice);
  float2* cst = reinterpret_cast<float2*>(rec + n);
  float* cped = reinterpret_cast<float*>(slot + sizeof(float) * round_up(tri(n), 4));
  uint8_t* cx = reinterpret_cast<uint8_t*>(cped + kMixCand);
  const int cs = mix_path_pad(n);
  const int room = (g.slice_bytes - (int)walk_record_bytes(n)) / 8 - 3;
  int low = room > 0 ? min(n, (int)(0.5f * (sqrtf(8.0f * (float)room + 1.0f) - 1.0f))) : 0;  // levels in the slice
  while (low > 0 && tri(low) > room) --low;
  float* Rs = reinterpret_cast<float*>(cst + n);
  float* zl = Rs + round_up(tri(low), 4);
  for (int k = lane; k < tri(low); k += 32) Rs[k] = Rg[k];
  for (int rr = lane; rr < n; rr += 32) {
    const float d = Rg[col_off(rr) + rr];
    cst[rr] = make_float2(d, 0.5f / (alpha * d));
  }
  __syncwarp();

  float r2_start = initial_r2(g, q, r);
  float r2 = r2_start;
  const long long limit = q.budget > 0 ? q.budget : 0x7fffffffffffffffll;
  long long nodes = 0, peds = 0, flops = 0;
  int restarts = 0, ncand = 0;
  bool bh = false;
  for (;;) {
    float z[ROWS], rc[ROWS];  // residuals at the current level, its column
#pragma unroll
    for (int t = 0; t < ROWS; ++t) z[t] = lane + 32 * t < n ? yg[lane + 32 * t] : 0.0f;
    auto col = [&](int j) { return (j < low ? (const float*)Rs : Rg) + col_off(j); };
    auto res = [&](int j) { return (j < low ? zl : zg) + col_off(j); };
#pragma unroll
    for (int t = 0; t < ROWS; ++t)
      if (lane + 32 * t < n) res(n - 1)[lane + 32 * t] = z[t];
    __syncwarp();
    float bnd = prune_bound(r2, E, n);
    int i = n - 1, ret = n;  // ret: the level a pop goes to (n: none)
    float ped_par = 0.0f, c = yg[n - 1], z1 = yg[n - 2];
    float2 ri = cst[n - 1];
    float ra = 0.0f, rb = 0.0f, z2 = 0.0f;
    float2 nx = make_float2(0.0f, 0.0f);
    // what a descent from level i needs
    auto reach = [&]() {
      const float* rp = col(i);
      if (i > 0) {
        ra = rp[i - 1];
        nx = cst[i - 1];
      }
      if (i > 1) {
        rb = rp[i - 2];
        z2 = res(i)[i - 2];
      }
#pragma unroll
      for (int t = 0; t < ROWS; ++t) rc[t] = lane + 32 * t < i ? rp[lane + 32 * t] : 0.0f;
    };
    // the child nearest to u: its index, level and distance, and its order
    auto first = [&](float cc, float2 rr, float par, int& k, float& lev, float& ped, int& pat) {
      const float u = fmaf(cc, rr.y, half);
      const float kf =
          __fadd_ru(fminf(fmaxf(u - 0.5f, 0.0f), (float)(P - 1)), 8388608.0f) - 8388608.0f;
      k = __float_as_int(kf + 8388608.0f) & 15;
      lev = (kf - half) * alpha2;
      pat = 2 * k + (u > kf ? 1 : 0);
      const float d = fmaf(-rr.x, lev, cc);
      ped = fmaf(d, d, par);
    };
    int k, pat, idx = 1;
    float lev, ped;
    first(c, ri, 0.0f, k, lev, ped, pat);
    unsigned ord = zz[pat];
    ++nodes;
    flops += 4 * P;
    ++peds;
    bool inside = ped < bnd;
    if (inside) reach();
    while (inside) {
      // child k of level i, inside the sphere
      if (i == 0) {
        // leaf: keep it among the kMixCand best, shrink the radius
        int at = -1;
        if (ncand < kMixCand) {
          at = ncand;
        } else {
          float worst = -1.0f;
          for (int t = 0; t < kMixCand; ++t)
            if (cped[t] > worst) {
              worst = cped[t];
              at = t;
            }
          if (!(ped < worst)) at = -1;
        }
        __syncwarp();
        if (at >= 0) {
          for (int rr = lane; rr < n; rr += 32)
            cx[(size_t)at * cs + rr] = (uint8_t)(rr == 0 ? k : __float_as_int(rec[rr].w) & 15);
          if (lane == 0) cped[at] = ped;
          if (at == ncand) ++ncand;
        }
        __syncwarp();
        if (ped < r2) {
          r2 = ped;
          bnd = prune_bound(r2, E, n);
        }
      } else if (nodes >= limit) {
        bh = true;
        break;
      }
      // its next sibling: outside the sphere, nothing at this level is left
      const bool more = idx < P;
      const float lev2 = level_at(ord >> (4 * idx - 1), mid, alpha2);
      const float d2 = fmaf(-ri.x, lev2, c);
      const float ped2 = fmaf(d2, d2, ped_par);
      const bool done = !(more && ped2 < bnd);
      if (more && done) ++peds;
      if (i > 0) {
        // the next level's nearest child: outside the sphere it rules out every child
        const float cn = fmaf(-ra, lev, z1);
        int kn, patn;
        float levn, pedn;
        first(cn, nx, ped, kn, levn, pedn, patn);
        ++nodes;
        ++peds;
        flops += 2 * (n - i) + 4 * P;
        if (pedn < bnd) {
          // descend: push level i, update the residuals of the rows below
          rec[i] = make_float4(c, ped_par, ped2, __int_as_float(k | idx << 4 | pat << 8 | ret << 16));
          if (!done) ret = i;
          float* zo = res(i - 1);
#pragma unroll
          for (int t = 0; t < ROWS; ++t) {
            z[t] = fmaf(-rc[t], lev, z[t]);
            if (lane + 32 * t < i) zo[lane + 32 * t] = z[t];
          }
          z1 = fmaf(-rb, lev, z2);
          --i;
          c = cn;
          ri = nx;
          ped_par = ped;
          k = kn;
          lev = levn;
          ped = pedn;
          pat = patn;
          ord = zz[pat];
          idx = 1;
          __syncwarp();
          reach();
          continue;
        }
      }
      if (!done) {
        k = (int)(ord >> (4 * idx)) & 15;
        lev = lev2;
        ped = ped2;
        ++idx;
        ++peds;
        continue;
      }
      // back to the nearest level above with a child inside
      inside = false;
      float4 s4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      while (ret < n) {
        i = ret;
        s4 = rec[i];
        ret = __float_as_int(s4.w) >> 16;
        ++peds;
        if (s4.z < bnd) {
          inside = true;
          break;
        }
      }
      if (!inside) break;
      const int w = __float_as_int(s4.w);
      c = s4.x;
      ped_par = s4.y;
      ped = s4.z;
      idx = (w >> 4) & 15;
      pat = (w >> 8) & 15;
      ord = zz[pat];
      k = (int)(ord >> (4 * idx)) & 15;
      lev = level_at(ord >> (4 * idx - 1), mid, alpha2);
      ++idx;
      ri = cst[i];
      const float* zi = res(i);
#pragma unroll
      for (int t = 0; t < ROWS; ++t) z[t] = lane + 32 * t < i ? zi[lane + 32 * t] : 0.0f;
      z1 = i > 0 ? zi[i - 1] : 0.0f;
      // a level's record and residuals, read by lanes that did not write them, are
      // written again only after a pop: the reads so far come before
      __syncwarp();
      reach();
    }
    if (ncand == 0 && !bh && r2_start < INFINITY && restarts < 64) {
      // empty sphere: r^2 <- 2 r^2 and search again
      r2_start *= 2.0f;
      r2 = r2_start;
      ++restarts;
      __syncwarp();  // as after a pop
      continue;
    }
    break;
  }
  __syncwarp();
  const int status = bh ? MDX_V_BUDGET_EXCEEDED : (restarts > 0 ? MDX_V_EMPTY_RETRIED : MDX_V_OK);
  finish_request(g, q, r, cx, cs, cped, ncand, E, status, nodes, peds, restarts, flops, lane);
}

// Complex-tree exact SD of one request by one warp: one tree level per complex
// antenna j (real rows 2j+1, then 2j), Q = P^2 children.  The next child of a
// node is the unvisited one of least partial distance (ties to the lower q),
// found by a warp arg-min; a level is exhausted when that child leaves the
// sphere.  A descent updates the residuals of the rows below by both fixed
// rows; the rest (candidates, radius shrink and doubling, budget, FP64
// re-scoring) is as in sd_walk.
template <int ROWS>
__device__ void sdc_request(const MixedArgs& g, const MixedReq& q, int r, const float* Rc, const float* yb,
                            unsigned char* st, float E, int lane) {
  const int n = q.n, P = q.P, Q = P * P, M = n / 2;
  const float alpha = q.alpha;
  float* zs = reinterpret_cast<float*>(st);
  float4* lv = reinterpret_cast<float4*>(zs + round_up(tri(n), 4));
  unsigned* lv_hi = reinterpret_cast<unsigned*>(lv + M);
  float4* lv_r = reinterpret_cast<float4*>(lv_hi + round_up(M, 4));
  float* cped = reinterpret_cast<float*>(lv_r + M);
  uint8_t* xs = reinterpret_cast<uint8_t*>(cped + kMixCand);
  uint8_t* cx = xs + mix_path_pad(n);
  const int cs = mix_path_pad(n);
  for (int j = lane; j < M; j += 32) {
    const int r1 = 2 * j + 1, r0 = 2 * j;
    lv_r[j] = make_float4(Rc[col_off(r1) + r1], Rc[col_off(r1) + r0], Rc[col_off(r0) + r0], 0.0f);
  }
  float r2_start = initial_r2(g, q, r);
  float r2 = r2_start;
  long long nodes = 0, peds = 0, flops = 0;
  int restarts = 0, ncand = 0;
  bool bh = false;
  for (;;) {
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      const int rr = lane + 32 * t;
      if (rr < n) zs[col_off(n - 1) + rr] = yb[rr];
    }
    __syncwarp();
    float bnd = prune_bound(r2, E, n);
    int j = M - 1;
    float ped_par = 0.0f;
    float c1 = zs[col_off(n - 1) + n - 1], c0 = zs[col_off(n - 1) + n - 2];
    float4 rl = lv_r[j];
    unsigned long long mask = 0ull;
    ++nodes;
    peds += Q;
    flops += 10 * Q;
    for (;;) {
      // the unvisited child of least partial distance
      unsigned long long best = ~0ull;
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int qq = lane + 32 * t;
        if (qq < Q && !((mask >> qq) & 1ull)) {
          const int kre = qq / P, kim = qq - kre * P;
          const float aim = (float)(2 * kim - (P - 1)) * alpha, are = (float)(2 * kre - (P - 1)) * alpha;
          const float d1 = fmaf(-rl.x, aim, c1);
          const float p1 = fmaf(d1, d1, ped_par);
          const float d0 = fmaf(-rl.z, are, fmaf(-rl.y, aim, c0));
          const float pd = fmaf(d0, d0, p1);
          const unsigned long long key = ((unsigned long long)__float_as_uint(pd) << 32) | (unsigned)qq;
          if (key < best) best = key;
        }
      }
      best = warp_min_u64(best);
      const float ped = (best == ~0ull) ? INFINITY : __uint_as_float((unsigned)(best >> 32));
      if (!(ped < bnd)) {
        if (j == M - 1) break;  // the root is exhausted
        ++j;                    // backtrack
        const float4 s4 = lv[j];
        ped_par = s4.x;
        c1 = s4.y;
        c0 = s4.z;
        mask = (unsigned long long)__float_as_uint(s4.w) | ((unsigned long long)lv_hi[j] << 32);
        rl = lv_r[j];
        __syncwarp();  // the level's state is read before lane 0 writes it again
        continue;
      }
      const int qk = (int)(best & 0xffffffffu);
      mask |= 1ull << qk;
      const int kre = qk / P, kim = qk - kre * P;
      if (j == 0) {
        // leaf inside the sphere: keep it among the kMixCand best, shrink the radius
        if (lane == 0) {
          xs[1] = (uint8_t)kim;
          xs[0] = (uint8_t)kre;
        }
        __syncwarp();
        keep_leaf(xs, n, ped, cx, cs, cped, ncand, lane);
        if (ped < r2) {
          r2 = ped;
          bnd = prune_bound(r2, E, n);
        }
        continue;
      }
      if (q.budget > 0 && nodes >= q.budget) {
        bh = true;
        break;
      }
      // descend: push level j, update the residuals of rows 0..2j-1 by both fixed rows
      const float aim = (float)(2 * kim - (P - 1)) * alpha, are = (float)(2 * kre - (P - 1)) * alpha;
      if (lane == 0) {
        lv[j] = make_float4(ped_par, c1, c0, __uint_as_float((unsigned)mask));
        lv_hi[j] = (unsigned)(mask >> 32);
        xs[2 * j + 1] = (uint8_t)kim;
        xs[2 * j] = (uint8_t)kre;
      }
      const float* zin = zs + col_off(2 * j + 1);
      float* zout = zs + col_off(2 * j - 1);
      const float* ra = Rc + col_off(2 * j + 1);
      const float* rb = Rc + col_off(2 * j);
      float n1 = 0.0f, n0 = 0.0f;
#pragma unroll
      for (int t = 0; t < ROWS; ++t) {
        const int rr = lane + 32 * t;
        if (rr < 2 * j) {
          const float z = fmaf(-rb[rr], are, fmaf(-ra[rr], aim, zin[rr]));
          zout[rr] = z;
          if (rr == 2 * j - 1) n1 = z;
          if (rr == 2 * j - 2) n0 = z;
        }
      }
      --j;
      c1 = __shfl_sync(0xffffffffu, n1, (2 * j + 1) & 31);
      c0 = __shfl_sync(0xffffffffu, n0, (2 * j) & 31);
      __syncwarp();
      ped_par = ped;
      rl = lv_r[j];
      mask = 0ull;
      ++nodes;
      peds += Q;
      flops += 4 * (n - 2 - 2 * j) + 10 * Q;
    }
    if (ncand == 0 && !bh && r2_start < INFINITY && restarts < 64) {
      r2_start *= 2.0f;  // empty sphere: r^2 <- 2 r^2 and search again
      r2 = r2_start;
      ++restarts;
      continue;
    }
    break;
  }
  __syncwarp();
  const int status = bh ? MDX_V_BUDGET_EXCEEDED : (restarts > 0 ? MDX_V_EMPTY_RETRIED : MDX_V_OK);
  finish_request(g, q, r, cx, cs, cped, ncand, E, status, nodes, peds, restarts, flops, lane);
}

// K-best of one request by one warp (SPL survivor slots per lane, K <= 32 SPL).
template <int SPL>
__device__ void kb_request(const MixedArgs& g, const MixedReq& q, int r, const float* Rc, const float* yb,
                           unsigned char* st, float E, int lane) {
  const int n = q.n, P = q.P, K = q.K, pp = path_stride(n);
  unsigned int* r2w = reinterpret_cast<unsigned int*>(st);
  float* pa = reinterpret_cast<float*>(st + 16);
  float* pb = pa + round_up(K, 4);
  uint16_t* sel = reinterpret_cast<uint16_t*>(pb + round_up(K, 4));
  uint8_t* xa = reinterpret_cast<uint8_t*>(sel + 2 * round_up(K, 8));
  uint8_t* xb = xa + (size_t)pp * K;
  float r2 = initial_r2(g, q, r);
  long long nodes = 0, flops = 0;
  int restarts = 0, S = 0;
  uint8_t *xcur = xa, *xnxt = xb;
  float *pcur = pa, *pnxt = pb;
  for (;;) {
    xcur = xa;
    xnxt = xb;
    pcur = pa;
    pnxt = pb;
    if (lane == 0) {
      *r2w = __float_as_uint(r2);
      pa[0] = 0.0f;
    }
    __syncwarp();
    S = warp_kbest<SPL, false>(Rc, yb, n, P, K, pp, q.alpha, n - 1, r2w, E, sel, &xcur, &xnxt, &pcur, &pnxt, lane, &nodes,
                        &flops);
    __syncwarp();
    if (S > 0 || !(r2 < INFINITY) || restarts >= 64) break;
    r2 *= 2.0f;  // every survivor left the sphere: r^2 <- 2 r^2
    ++restarts;
  }
  const int nc = S < kCandMax ? S : kCandMax;
  finish_request(g, q, r, xcur, pp, pcur, nc, E, restarts > 0 ? MDX_V_EMPTY_RETRIED : MDX_V_OK, nodes,
                 nodes * P, restarts, flops, lane);
}

// The same by selection (K <= 32 SL).
template <int SL>
__device__ void kb_select(const MixedArgs& g, const MixedReq& q, int r, const float* Rg, const float* yg,
                          unsigned char* slice, unsigned char* slot, float E, int lane) {
  const int n = q.n, P = q.P, K = q.K, cs = mix_path_pad(n);
  const SelectWs ws = select_ws(slice, g.slice_bytes, slot, n, K);
  float* cped = reinterpret_cast<float*>(ws.ent);
  uint8_t* cx = slot + select_path_bytes(n, K);
  for (int ranked = 0; ranked < 2; ++ranked) {
    float r2 = initial_r2(g, q, r);
    RunCost cost;
    int restarts = 0, S = 0;
    Survivors<SL> v;
    for (;;) {
      const float bnd = prune_bound(r2, E, n);
#pragma unroll
      for (int t = 0; t < SL; ++t) {
        v.ped[t] = 0.0f;
        v.cur[t] = 0u;
      }
      if (P == 8) S = select_run<SL, 8>(Rg, yg, n, K, q.alpha, 0, 1, bnd, ranked, ws, lane, v, cost);
      else if (P == 4) S = select_run<SL, 4>(Rg, yg, n, K, q.alpha, 0, 1, bnd, ranked, ws, lane, v, cost);
      else S = select_run<SL, 2>(Rg, yg, n, K, q.alpha, 0, 1, bnd, ranked, ws, lane, v, cost);
      if (S != 0 || !(r2 < INFINITY) || restarts >= 64) break;
      r2 *= 2.0f;  // every survivor left the sphere: r^2 <- 2 r^2
      ++restarts;
    }
    if (S < 0 || !select_leaves<SL>(v, S, ranked, n, ws.x, ws.KS, cx, cs, cped, lane)) continue;
    finish_request(g, q, r, cx, cs, cped, min(S, kCandMax), E, restarts > 0 ? MDX_V_EMPTY_RETRIED : MDX_V_OK,
                   cost.nodes, cost.nodes * P, restarts, cost.flops, lane);
    break;
  }
}

// The next request of the launch's order to the calling warp (-1: none left),
// its descriptor in q; singular ones are answered here.
__device__ __forceinline__ int next_request(const MixedArgs& g, MixedReq& q, int lane) {
  for (;;) {
    unsigned int t = 0;
    if (lane == 0) t = atomicAdd(g.counter, 1u);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= (unsigned int)g.nreq) return -1;
    const int r = g.order ? g.order[t] : (int)t;
    if (g.reqs) {
      q = g.reqs[r];
    } else {
      q = g.uniform;
      q.r_off = (long long)r * tri_stride32(q.n);
      q.y_off = (long long)r * vec_stride32(q.n);
      q.r_off64 = (long long)r * tri_stride64(q.n);
      q.y_off64 = (long long)r * vec_stride64(q.n);
      q.sym_off = (long long)r * q.n_tx;
    }
    if (!g.singular[r]) return r;
    for (int j = lane; j < q.n_tx; j += 32) g.sym_out[q.sym_off + j] = 0;
    if (lane == 0) {
      g.metric_out[r] = 0.0;
      g.vstatus[r] = MDX_V_SINGULAR;
      if (g.stats)
        for (int k = 0; k < kStats; ++k) g.stats[(size_t)r * kStats + k] = 0;
    }
  }
}

// The walks have a kernel of their own: a step is a chain of a hundred
// instructions, and registers spilled for the other forms' sake lengthen it
// (the classes of sd_walk in one kernel with the selection: 6.5, 13.0, 14.9 ms).
__global__ void __launch_bounds__(512) walk_kernel(MixedArgs g) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
  unsigned char* gslot = g.gscratch + ((size_t)blockIdx.x * W + warp) * g.gslot_bytes;
  MixedReq q;
  for (int r; (r = next_request(g, q, lane)) >= 0; __syncwarp()) {
    const float* Rc = g.R32 + q.r_off;
    const float* yb = g.yb32 + q.y_off;
    const float E = error_scale_warp(q.n, q.P, q.alpha, Rc, yb, lane);
    if (q.n <= 32) sd_walk<1>(g, q, r, Rc, yb, gslot, E, lane);
    else if (q.n <= 64) sd_walk<2>(g, q, r, Rc, yb, gslot, E, lane);
    else if (q.n <= 128) sd_walk<4>(g, q, r, Rc, yb, gslot, E, lane);
    else sd_walk<7>(g, q, r, Rc, yb, gslot, E, lane);
  }
}

template <int KSPL>
__global__ void __launch_bounds__(512) mixed_kernel(MixedArgs g) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
  unsigned char* slice = smem + (size_t)warp * g.slice_bytes;
  unsigned char* gslot = g.gscratch + ((size_t)blockIdx.x * W + warp) * g.gslot_bytes;
  MixedReq q;
  for (int r; (r = next_request(g, q, lane)) >= 0; __syncwarp()) {
    const float* Rc = g.R32 + q.r_off;
    const float* yb = g.yb32 + q.y_off;
    if (q.algo == MDX_ALGO_KBEST && q.K <= 64) {
      const float E = error_scale_warp(q.n, q.P, q.alpha, Rc, yb, lane);
      if (q.K <= 32) kb_select<1>(g, q, r, Rc, yb, slice, gslot, E, lane);
      else kb_select<2>(g, q, r, Rc, yb, slice, gslot, E, lane);
      continue;
    }
    unsigned char* st = gslot;
    if (q.mode & MIX_STAGE_R) {
      const int ts = tri_stride32(q.n);
      float* sR = reinterpret_cast<float*>(slice);
      float* sy = sR + ts;
      const float4* src = reinterpret_cast<const float4*>(Rc);
      for (int k = lane; k < ts / 4; k += 32) reinterpret_cast<float4*>(sR)[k] = src[k];
      for (int k = lane; k < q.n; k += 32) sy[k] = yb[k];
      Rc = sR;
      yb = sy;
      if (q.mode & MIX_STATE_SMEM) st = slice + stage_bytes(q.n);
    } else if (q.mode & MIX_STATE_SMEM) {
      st = slice;
    }
    __syncwarp();
    const float E = error_scale_warp(q.n, q.P, q.alpha, Rc, yb, lane);
    if (q.algo == MIX_ALGO_SD_NATURAL) {
      if (q.n <= 32) sd_natural<1>(g, q, r, Rc, yb, st, E, lane);
      else if (q.n <= 64) sd_natural<2>(g, q, r, Rc, yb, st, E, lane);
      else if (q.n <= 128) sd_natural<4>(g, q, r, Rc, yb, st, E, lane);
      else sd_natural<7>(g, q, r, Rc, yb, st, E, lane);
    } else if (q.algo == MIX_ALGO_SD_COMPLEX) {
      if (q.n <= 32) sdc_request<1>(g, q, r, Rc, yb, st, E, lane);
      else if (q.n <= 64) sdc_request<2>(g, q, r, Rc, yb, st, E, lane);
      else if (q.n <= 128) sdc_request<4>(g, q, r, Rc, yb, st, E, lane);
      else sdc_request<7>(g, q, r, Rc, yb, st, E, lane);
    } else if constexpr (KSPL > 2) {
      if (q.K <= 128) kb_request<4>(g, q, r, Rc, yb, st, E, lane);
      else kb_request<8>(g, q, r, Rc, yb, st, E, lane);
    }
  }
}

cudaError_t prepare(const void* fn, int W, int slice_bytes, int num_sms, int* grid) {
  const int smem = W * slice_bytes;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, W * 32, (size_t)smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  *grid = per_sm * num_sms;
  return cudaSuccess;
}
const void* walk_fn() { return (const void*)walk_kernel; }
const void* mixed_fn(int max_K) { return max_K > 64 ? (const void*)mixed_kernel<8> : (const void*)mixed_kernel<2>; }

}  // namespace

size_t mixed_stage_bytes(int n) { return stage_bytes(n); }

size_t mixed_state_bytes(int algo, int n, int K, int P) {
  (void)P;
  if (algo == MIX_ALGO_SD_NATURAL) return sd_state_bytes(n);
  if (algo == MIX_ALGO_SD_COMPLEX) return sdc_state_bytes(n);
  return kb_state_bytes(n, K);
}

// Forms that use slice and slot by themselves: placement bits say nothing.
static bool self_placed(int algo, int K) { return algo == MDX_ALGO_SD || (algo == MDX_ALGO_KBEST && K <= 64); }

int mixed_greedy_mode(int algo, int n, int K, int P, int slice) {
  if (self_placed(algo, K)) return 0;
  const size_t stage = stage_bytes(n), state = mixed_state_bytes(algo, n, K, P);
  if (stage + state <= (size_t)slice) return MIX_STAGE_R | MIX_STATE_SMEM;
  if (state <= (size_t)slice) return MIX_STATE_SMEM;
  if (stage <= (size_t)slice) return MIX_STAGE_R;
  return 0;
}

bool mixed_mode_fits(int mode, int algo, int n, int K, int slice) {
  if (self_placed(algo, K)) return mode == 0;
  size_t need = 0;
  if (mode & MIX_STAGE_R) need += mixed_stage_bytes(n);
  if (mode & MIX_STATE_SMEM) need += mixed_state_bytes(algo, n, K, 0);
  return need <= (size_t)slice;
}

int mixed_least_slice(int algo, int n, int K) {
  if (algo == MDX_ALGO_SD) return (int)((walk_record_bytes(n) + 15) / 16 * 16);
  return self_placed(algo, K) ? (int)((select_level_bytes(n, K) + 15) / 16 * 16) : 0;
}

size_t mixed_slot_bytes(int mode, int algo, int n, int K) {
  if (algo == MDX_ALGO_SD) return walk_slot_bytes(n);
  if (self_placed(algo, K)) return (select_path_bytes(n, K) + (size_t)kCandMax * mix_path_pad(n) + 15) / 16 * 16;
  return (mode & MIX_STATE_SMEM) ? 16 : mixed_state_bytes(algo, n, K, 0);
}

int mixed_resident_warps(int W, int slice_bytes, int max_K, int num_sms) {
  int walks = 0, others = 0;
  cudaError_t e = prepare(walk_fn(), W, slice_bytes, num_sms, &walks);
  if (e == cudaSuccess) e = prepare(mixed_fn(max_K), W, slice_bytes, num_sms, &others);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return (walks + others) * W;
}

cudaError_t launch_mixed(const MixedArgs& a, int walks, int W, int max_K, int num_sms, const MixedFork& fork,
                         cudaStream_t s) {
  if (W < 1 || W > 16 || a.slice_bytes < 0 || (a.slice_bytes & 15)) return cudaErrorInvalidConfiguration;
  const size_t smem = (size_t)W * a.slice_bytes;
  const bool both = walks > 0 && a.nreq > walks;
  cudaError_t e = both ? cudaEventRecord(fork.begin, s) : cudaSuccess;
  int slots = 0;
  for (int form = 0; form < 2 && e == cudaSuccess; ++form) {
    MixedArgs g = a;
    g.nreq = form == 0 ? walks : a.nreq - walks;
    if (g.nreq <= 0) continue;
    if (form == 1) {
      if (a.order) g.order = a.order + walks;
      g.counter = a.counter + 1;
      g.gscratch = a.gscratch + (size_t)slots * a.gslot_bytes;
    }
    int grid = 0;
    e = prepare(form == 0 ? walk_fn() : mixed_fn(max_K), W, a.slice_bytes, num_sms, &grid);
    if (e != cudaSuccess) return e;
    slots += grid * W;
    const cudaStream_t on = form == 1 && both ? fork.side : s;
    if (on != s && (e = cudaStreamWaitEvent(on, fork.begin, 0)) != cudaSuccess) return e;
    if (form == 0) walk_kernel<<<grid, W * 32, smem, on>>>(g);
    else if (max_K > 64) mixed_kernel<8><<<grid, W * 32, smem, on>>>(g);
    else mixed_kernel<2><<<grid, W * 32, smem, on>>>(g);
    e = cudaGetLastError();
    if (e == cudaSuccess && on != s) e = cudaEventRecord(fork.end, on);
    if (e == cudaSuccess && on != s) e = cudaStreamWaitEvent(s, fork.end, 0);
  }
  return e;
}

}  // namespace mdx
