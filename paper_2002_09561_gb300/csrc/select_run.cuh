// A K-best run (Sec. VI) by one warp with the survivors selected instead of
// sorted: shared by the uneven-batch kernel and the hybrid.
//
// A level needs the set of the K smallest of the S P children, not their
// order: the order enters the result only where children at exactly the same
// FP32 distance straddle the cut (ties go to the lower parent rank, then to
// the Schnorr-Euchner rank).  So every lane keeps its survivors' children as
// 32-bit distance bits, the K-th smallest is found by a search on the bits,
// and the children up to it are compacted in lane order.  Where a tie straddles
// the cut, its children are taken in the order of their parents' distances,
// which is that of the ranks; only where those tie as well does the run start
// again with the ranks kept (a count of the smaller keys per survivor and
// level, some 30 % of a level).
//
// Survivor paths are nibbles in depth order (row n - 1 first), eight to a
// word, word w of all survivors together; a word is one step of the eight FMA
// chains of row_interference.  The word being filled stays in a register with
// the survivor's ancestor at the last full word, and only every eighth level
// are the full words reordered (in place, by a gather through the ancestors,
// which is also how they are read: the same word of any ancestors is in
// distinct banks or the same address).  R is not staged: the next row is
// fetched from global memory while a level runs.  A 100x100 run (n = 200, K =
// 32) needs 4.3 KB.
#pragma once

#include "warp_kbest.cuh"

namespace mdx {
namespace {

// The bits T such that exactly K of the warp's keys are <= T, or false if a
// tie straddles the K-th (T: the tie).  Invariant: n_lo < K keys are <= lo, n_hi >= K are
// <= hi.  (Six steps or so, since any value between the K-th and the next
// child will do.)
template <int N>
__device__ __forceinline__ bool select_cut(const unsigned (&key)[N], int K, unsigned lo, unsigned hi, int n_hi,
                                           unsigned& T) {
  int n_lo = 0;
  if (n_hi == K) {
    T = hi;
    return true;
  }
  for (int it = 0; hi - lo > 1u; ++it) {
    const unsigned gap = hi - lo;
    // where a uniform density would put the middle of the K-th gap, bisection
    // every third step and once the counts stop helping
    unsigned step = gap >> 1;
    if (it % 3 != 2) {
      const float f = ((float)(K - n_lo) + 0.5f) * __frcp_rn((float)(n_hi - n_lo) + 1.0f);
      step = (unsigned)((float)gap * fminf(f, 1.0f));
      step = min(max(step, 1u), gap - 1u);
    }
    const unsigned mid = lo + step;
    int c = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) c += key[j] <= mid ? 1 : 0;
    c = __reduce_add_sync(0xffffffffu, c);
    if (c == K) {
      T = mid;
      return true;
    }
    if (c < K) {
      lo = mid;
      n_lo = c;
    } else {
      hi = mid;
      n_hi = c;
    }
  }
  T = hi;
  return false;
}

// The cut of a level's children (all-ones: none) and how many it keeps; false:
// a tie straddles it.  SL survivors per lane, S in all, C children each.
template <int SL, int C>
__device__ __forceinline__ bool level_cut(const unsigned (&key)[SL * C], int S, int K, int lane, unsigned& T,
                                          int& kept) {
  T = 0xfffffffeu;
  int valid = 0;
  unsigned least = 0xffffffffu, most = 0u, own = 0u;
#pragma unroll
  for (int q = 0; q < SL; ++q) {
    unsigned low = 0xffffffffu;
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const unsigned x = key[q * C + k];
      valid += x != 0xffffffffu ? 1 : 0;
      low = min(low, x);
      most = max(most, x + 1u);  // (an empty key counts as 0)
    }
    least = min(least, low);
    if (lane + 32 * q < S) own = max(own, low);
  }
  valid = __reduce_add_sync(0xffffffffu, valid);
  kept = min(valid, K);
  if (valid <= K) return true;
  least = __reduce_min_sync(0xffffffffu, least);
  // the largest of the survivors' best children bounds the S smallest
  const unsigned far = __reduce_max_sync(0xffffffffu, own);
  unsigned hi = __reduce_max_sync(0xffffffffu, most) - 1u;
  int n_hi = valid;
  if (S >= K && far < hi) {
    int c = 0;
#pragma unroll
    for (int j = 0; j < SL * C; ++j) c += key[j] <= far ? 1 : 0;
    n_hi = __reduce_add_sync(0xffffffffu, c);
    hi = far;
  }
  return select_cut<SL * C>(key, K, least - 1u, hi, n_hi, T);
}

// The kept children in lane order: {parent | child << 16, distance bits}.
template <int SL, int C>
__device__ __forceinline__ void compact_level(const unsigned (&key)[SL * C], unsigned T, uint2* ent, int lane) {
  int at = 0;
  if (SL * C <= 16) {
    // as many ballots as a shuffle scan has instructions, but independent
#pragma unroll
    for (int j = 0; j < SL * C; ++j)
      at += __popc(__ballot_sync(0xffffffffu, key[j] <= T) & ((1u << lane) - 1u));
  } else {
    int mine = 0;
#pragma unroll
    for (int j = 0; j < SL * C; ++j) mine += key[j] <= T ? 1 : 0;
    at = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += t;
    }
    at -= mine;
  }
#pragma unroll
  for (int j = 0; j < SL * C; ++j) {
    if (key[j] <= T) {
      ent[at] = make_uint2((unsigned)(lane + 32 * (j / C)) | ((unsigned)(j % C) << 16), key[j]);
      ++at;
    }
  }
}

// PAM level 2 k - (P - 1) times alpha from the bits 1..4 of b (k << 1): an
// exact k - (P - 1) / 2 out of a float's low mantissa bits, then one rounding,
// the same as that of (float)(2 k - (P - 1)) * alpha.
constexpr unsigned kLevelMagic = 0x4a800000u;  // 2^22, half a unit per bit
__device__ __forceinline__ float level_at(unsigned b, float mid, float alpha2) {
  return (__uint_as_float((b & 0x1eu) | kLevelMagic) - mid) * alpha2;
}
__device__ __forceinline__ float level_mid(int P) { return 4194304.0f + 0.5f * (float)(P - 1); }

// A run's workspace: the level's row of R (in depth order, zeros behind) and
// the compacted children in shared memory, the full words of the paths there
// or in global memory.
struct SelectWs {
  float* row;
  uint2* ent;
  uint32_t* x;
  int KS;  // survivor slots
};
__host__ __device__ inline int select_slots(int K) { return round_up(K, 32); }
__host__ __device__ inline size_t select_level_bytes(int n, int K) {
  return sizeof(float) * round_up(n, 8) + sizeof(uint2) * (size_t)select_slots(K);
}
__host__ __device__ inline size_t select_path_bytes(int n, int K) {
  return sizeof(uint32_t) * (size_t)(round_up(n, 8) / 8) * (size_t)select_slots(K);
}
// In `room` bytes of shared memory, the paths in `other` if they do not fit.
__device__ __forceinline__ SelectWs select_ws(unsigned char* smem, int room, unsigned char* other, int n, int K) {
  SelectWs w;
  const size_t level = select_level_bytes(n, K);
  w.KS = select_slots(K);
  w.row = reinterpret_cast<float*>(smem);
  w.ent = reinterpret_cast<uint2*>(w.row + round_up(n, 8));
  w.x = reinterpret_cast<uint32_t*>(level + select_path_bytes(n, K) <= (size_t)room ? smem + level : other);
  return w;
}

// A lane's survivors: distance, rank (or the key it was chosen by, in place of
// one), ancestor at the last full word, and the word since.
template <int SL>
struct Survivors {
  float ped[SL];
  unsigned rank[SL];
  int anc[SL];
  uint32_t cur[SL];
};

// Interference of NQ survivors per lane at depth d (row_interference's chains
// and sums).
template <int NQ, int SL>
__device__ __forceinline__ void select_interference(const SelectWs& ws, const Survivors<SL>& v, int d, float y,
                                                    float mid, float alpha2, float (&c)[SL]) {
  float acc[NQ][8];
#pragma unroll
  for (int q = 0; q < NQ; ++q)
#pragma unroll
    for (int m = 0; m < 8; ++m) acc[q][m] = m == 0 ? y : 0.0f;
  // the next step's loads before this one's sums
  const float4* row = reinterpret_cast<const float4*>(ws.row);
  const int full = d >> 3, steps = (d + 7) >> 3;
  float4 r0 = row[0], r1 = row[1];
  uint32_t word[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) word[q] = full > 0 ? ws.x[v.anc[q]] : v.cur[q];
  for (int w = 1; w <= steps; ++w) {
    const float r[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
    uint32_t now[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) now[q] = word[q];
    if (w < steps) {
      r0 = row[2 * w];
      r1 = row[2 * w + 1];
#pragma unroll
      for (int q = 0; q < NQ; ++q) word[q] = w < full ? ws.x[w * ws.KS + v.anc[q]] : v.cur[q];
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
      for (int m = 0; m < 8; ++m)
        acc[q][m] = fmaf(-r[m], level_at(m ? now[q] >> (4 * m - 1) : now[q] << 1, mid, alpha2), acc[q][m]);
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q)
    c[q] = ((acc[q][0] + acc[q][1]) + (acc[q][2] + acc[q][3])) + ((acc[q][4] + acc[q][5]) + (acc[q][6] + acc[q][7]));
}
// The same for S <= 32 / G survivors, G lanes each (a level of few survivors
// is all latency): lane G s + p runs survivor s's chains p, p + G, ...
template <int G, int SL>
__device__ __forceinline__ float select_interference_few(const SelectWs& ws, const Survivors<SL>& v, int d, float y,
                                                         float mid, float alpha2, int S, int lane) {
  constexpr int M = 8 / G;
  const int s = lane / G < S ? lane / G : 0, p = lane % G;
  const int anc = __shfl_sync(0xffffffffu, v.anc[0], s);
  const uint32_t cur = __shfl_sync(0xffffffffu, v.cur[0], s);
  float acc[M];
#pragma unroll
  for (int m = 0; m < M; ++m) acc[m] = p + G * m == 0 ? y : 0.0f;
  const int full = d >> 3;
#pragma unroll 4
  for (int w = 0; w < full; ++w) {
    const uint32_t word = ws.x[w * ws.KS + anc] << 1;
#pragma unroll
    for (int m = 0; m < M; ++m)
      acc[m] = fmaf(-ws.row[8 * w + p + G * m], level_at(word >> (4 * (p + G * m)), mid, alpha2), acc[m]);
  }
  if (d & 7) {
#pragma unroll
    for (int m = 0; m < M; ++m)
      acc[m] = fmaf(-ws.row[8 * full + p + G * m], level_at((cur << 1) >> (4 * (p + G * m)), mid, alpha2), acc[m]);
  }
#pragma unroll
  for (int b = 1; b < 8; b <<= 1) {
#pragma unroll
    for (int m = 0; m < M; ++m) {
      if (b < G) acc[m] += __shfl_xor_sync(0xffffffffu, acc[m], b);
      else if ((m & (b / G)) == 0) acc[m] += acc[(m + b / G) % M];
    }
  }
  return __shfl_sync(0xffffffffu, acc[0], (lane * G) & 31);
}

// A child's key orders it as the sorting forms do: the largest distance among
// its siblings up to it in Schnorr-Euchner order, which is its own distance
// except where rounding breaks that order.  Same-side children cannot break it
// (every step is monotone), opposite ones only where 2 u is within 6e-6 of an
// integer (the roundings of u and of the distances, in units of the level
// spacing); from 2^-12 on nothing is compared.
template <int P>
__device__ __forceinline__ bool near_tie(float u) {
  const float t = 2.0f * u;
  return u > -1.0f && u < (float)P && !(fabsf(t - rintf(t)) >= 0x1p-12f);
}
template <int P>
__device__ __forceinline__ bool before(float u, int k2, int k) {  // k2 before k in Schnorr-Euchner order
  const float dk = fabsf(u - (float)k), d2 = fabsf(u - (float)k2);
  return d2 < dk || (d2 == dk && k2 < k);
}
template <int P>
__device__ __forceinline__ bool order_keys(float u, unsigned* key) {  // whether it changed one
  unsigned run[P];
  bool broken = false;
#pragma unroll
  for (int k = 0; k < P; ++k) {
    run[k] = key[k];
#pragma unroll
    for (int k2 = 0; k2 < P; ++k2)
      if (k2 != k && before<P>(u, k2, k)) run[k] = max(run[k], key[k2]);
    broken |= run[k] != key[k];
  }
#pragma unroll
  for (int k = 0; k < P; ++k) key[k] = run[k];
  return broken;
}

// Keeps, of the children at the distance T that a cut of K straddles, those
// that rank first: least parent rank, then Schnorr-Euchner order.  False if two
// of the parents have the same rank themselves.
template <int SL, int P>
__device__ __forceinline__ bool resolve_tie(unsigned (&key)[SL * P], unsigned T, int K, int S,
                                            const unsigned (&rank)[SL], const float (&u)[SL], int lane) {
  int less = 0;
  unsigned tied = 0;  // bit q P + k
#pragma unroll
  for (int j = 0; j < SL * P; ++j) {
    less += key[j] < T ? 1 : 0;
    if (key[j] == T) {
      tied |= 1u << j;
      key[j] = 0xffffffffu;
    }
  }
  const int need = K - __reduce_add_sync(0xffffffffu, less);
  for (int t = 0; t < need; ++t) {
    unsigned low = 0xffffffffu;
#pragma unroll
    for (int q = 0; q < SL; ++q)
      if ((tied >> (q * P)) & ((1u << P) - 1u)) low = min(low, rank[q]);
    const unsigned m = __reduce_min_sync(0xffffffffu, low);
    int parents = 0;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      const unsigned mine = (tied >> (q * P)) & ((1u << P) - 1u);
      if (mine && rank[q] == m) {
        ++parents;
        int first = -1;
#pragma unroll
        for (int k = 0; k < P; ++k)
          if (((mine >> k) & 1u) && (first < 0 || before<P>(u[q], k, first))) first = k;
#pragma unroll
        for (int k = 0; k < P; ++k)
          if (k == first) {
            key[q * P + k] = T;
            tied &= ~(1u << (q * P + k));
          }
      }
    }
    if (__reduce_add_sync(0xffffffffu, parents) != 1) return false;
  }
  return true;
}

// What runs have cost (nodes, flops, levels), and the last one's most survivors.
struct RunCost {
  long long nodes = 0, flops = 0;
  int levels = 0, peak = 0;
};

// A run from a node at depth d0 < 8 (rows n - 1 .. n - d0 fixed) inside the
// bound bnd: survivor 0 of v, its nibbles in cur.  Returns the number of
// leaves, their distances in v and their paths in ws.x; -1: a tie that only a
// run with ranks decides (ranked: v.rank counts from the best).  S > 1: that many runs from nodes 0 .. S - 1 at once, good for as long
// as all their survivors together are no more than K (then no run's cut
// applies); -2: they were more.
template <int SL, int P>
__device__ int select_run(const float* __restrict__ Rg, const float* __restrict__ yg, int n, int K, float alpha,
                          int d0, int S, float bnd, bool ranked, const SelectWs& ws, int lane, Survivors<SL>& v,
                          RunCost& cost) {
  const float mid = level_mid(P), alpha2 = 2.0f * alpha, uoff = 0.5f * (float)(P - 1);
  const int n8 = round_up(n, 8);
  float nxt[7];
  auto fetch = [&](int d) {  // the row at depth d
#pragma unroll
    for (int t = 0; t < 7; ++t) {
      const int dp = lane + 32 * t;
      if (32 * t < d) nxt[t] = dp < d ? Rg[col_off(n - 1 - dp) + n - 1 - d] : 0.0f;
    }
  };
  fetch(d0);
  float y = yg[n - 1 - d0], rii = Rg[col_off(n - 1 - d0) + n - 1 - d0];
#pragma unroll
  for (int q = 0; q < SL; ++q) {
    v.anc[q] = lane + 32 * q;
    v.rank[q] = 0u;
  }
  const bool joint = S > 1;
  int sum_nodes = 0, sum_flops = 0, peak = S, d = d0;  // (a run's fit 32 bits)
  for (; d < n && S > 0; ++d) {
#pragma unroll
    for (int t = 0; t < 7; ++t)
      if (32 * t < d && lane + 32 * t < n8) ws.row[lane + 32 * t] = nxt[t];
    __syncwarp();
    const float yi = y, r = rii, rinv = 0.5f / (alpha * r);
    if (d + 1 < n) {
      fetch(d + 1);
      y = yg[n - 2 - d];
      rii = Rg[col_off(n - 2 - d) + n - 2 - d];
    }
    float c[SL] = {};
    if (S <= 4)
      c[0] = select_interference_few<8, SL>(ws, v, d, yi, mid, alpha2, S, lane);
    else if (S <= 8)
      c[0] = select_interference_few<4, SL>(ws, v, d, yi, mid, alpha2, S, lane);
    else if (SL == 1 || S <= 32)
      select_interference<1, SL>(ws, v, d, yi, mid, alpha2, c);
    else
      select_interference<SL, SL>(ws, v, d, yi, mid, alpha2, c);
    unsigned key[SL * P];
    float u[SL];
    bool broken = false;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      u[q] = fmaf(c[q], rinv, uoff);
#pragma unroll
      for (int k = 0; k < P; ++k) key[q * P + k] = 0xffffffffu;
      if (lane + 32 * q < S) {
#pragma unroll
        for (int k = 0; k < P; ++k) {
          const float dd = fmaf(-r, (float)(2 * k - (P - 1)) * alpha, c[q]);
          const float p = fmaf(dd, dd, v.ped[q]);
          if (p < bnd) key[q * P + k] = __float_as_uint(p);
        }
        if (near_tie<P>(u[q])) broken |= order_keys<P>(u[q], key + q * P);
      }
    }
    sum_nodes += S;
    sum_flops += S * (2 * d + 4 * P);
    peak = max(peak, S);
    unsigned T;
    int kept;
    broken = __any_sync(0xffffffffu, broken);
    if (joint) {
      int valid = 0;
#pragma unroll
      for (int j = 0; j < SL * P; ++j) valid += key[j] != 0xffffffffu ? 1 : 0;
      kept = __reduce_add_sync(0xffffffffu, valid);
      T = 0xfffffffeu;
      if (kept > K) {
        S = -2;
        break;
      }
    } else if (!level_cut<SL, P>(key, S, K, lane, T, kept) &&
               !resolve_tie<SL, P>(key, T, K, S, v.rank, u, lane)) {
      S = -1;
      break;
    }
    compact_level<SL, P>(key, T, ws.ent, lane);
    __syncwarp();
    // ---- the new survivors, from their parents' registers
    const int sh = 4 * (d & 7);
    Survivors<SL> w;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      const uint2 e = lane + 32 * q < kept ? ws.ent[lane + 32 * q] : make_uint2(0u, 0u);
      const int par = (int)(e.x & 0xffffu);
      float cp = 0.0f, pp = 0.0f;
#pragma unroll
      for (int t = 0; t < SL; ++t) {
        const int at = __shfl_sync(0xffffffffu, v.anc[t], par & 31);
        const uint32_t ct = __shfl_sync(0xffffffffu, v.cur[t], par & 31);
        if (t == 0 || t == par >> 5) {
          w.anc[q] = at;
          w.cur[q] = ct;
        }
        if (broken) {
          const float cc = __shfl_sync(0xffffffffu, c[t], par & 31), pt = __shfl_sync(0xffffffffu, v.ped[t], par & 31);
          if (t == 0 || t == par >> 5) {
            cp = cc;
            pp = pt;
          }
        }
      }
      w.cur[q] = (sh ? w.cur[q] : 0u) | (e.x >> 16) << sh;
      w.ped[q] = __uint_as_float(e.y);
      w.rank[q] = e.y;
      if (broken) {  // the kept children's own distances
        const float dd = fmaf(-r, (float)(2 * (int)(e.x >> 16) - (P - 1)) * alpha, cp);
        w.ped[q] = fmaf(dd, dd, pp);
      }
    }
    if (ranked) {
      uint64_t mine[SL];
#pragma unroll
      for (int q = 0; q < SL; ++q) {
        const uint2 e = lane + 32 * q < kept ? ws.ent[lane + 32 * q] : make_uint2(0u, 0u);
        const int par = (int)(e.x & 0xffffu), k = (int)(e.x >> 16);
        unsigned pr = 0u;
        float up = 0.0f;
#pragma unroll
        for (int t = 0; t < SL; ++t) {
          const unsigned rt = __shfl_sync(0xffffffffu, v.rank[t], par & 31);
          const float ut = __shfl_sync(0xffffffffu, u[t], par & 31);
          if (t == par >> 5) {
            pr = rt;
            up = ut;
          }
        }
        unsigned se = 0;
        for (int k2 = 0; k2 < P; ++k2) se += k2 != k && before<P>(up, k2, k) ? 1u : 0u;
        mine[q] = (uint64_t)w.rank[q] << 32 | pr << 4 | se;  // (w.rank: the key so far)
        w.rank[q] = 0u;
      }
#pragma unroll
      for (int t = 0; t < SL; ++t)
        for (int i = 0; i < 32 && i + 32 * t < kept; ++i) {
          const uint64_t o = __shfl_sync(0xffffffffu, mine[t], i);
#pragma unroll
          for (int q = 0; q < SL; ++q) w.rank[q] += o < mine[q] ? 1u : 0u;
        }
    }
    v = w;
    if (sh == 28 || d == n - 1) {  // a full word, or the last one: the paths in survivor order
      const int full = d >> 3;
      constexpr int B = SL == 1 ? 4 : 2;
      for (int w0 = 0; w0 < full; w0 += B) {
        uint32_t t[B][SL];
#pragma unroll
        for (int b = 0; b < B; ++b)
#pragma unroll
          for (int q = 0; q < SL; ++q) t[b][q] = w0 + b < full ? ws.x[(w0 + b) * ws.KS + v.anc[q]] : 0u;
        __syncwarp();
#pragma unroll
        for (int b = 0; b < B; ++b)
#pragma unroll
          for (int q = 0; q < SL; ++q)
            if (w0 + b < full) ws.x[(w0 + b) * ws.KS + lane + 32 * q] = t[b][q];
      }
#pragma unroll
      for (int q = 0; q < SL; ++q) {
        ws.x[full * ws.KS + lane + 32 * q] = v.cur[q];
        v.anc[q] = lane + 32 * q;
      }
    }
    __syncwarp();
    S = kept;
  }
  if (S >= 0) {
    cost.nodes += sum_nodes;
    cost.flops += sum_flops;
  }
  cost.levels += d - d0;
  cost.peak = peak;
  return S;
}

// The first kCandMax leaves of a run: index paths by row to cx (stride cs),
// distances to cped.  False: a tie straddles the last one, and the run was
// without ranks.
template <int SL>
__device__ bool select_leaves(const Survivors<SL>& v, int S, bool ranked, int n, const uint32_t* x, int KS, uint8_t* cx,
                              int cs, float* cped, int lane) {
  unsigned key[SL];
#pragma unroll
  for (int q = 0; q < SL; ++q)
    key[q] = lane + 32 * q >= S ? 0xffffffffu : ranked ? v.rank[q] : __float_as_uint(v.ped[q]);
  const int nc = min(S, kCandMax);
  for (int t = 0; t < nc; ++t) {
    unsigned low = key[0];
#pragma unroll
    for (int q = 1; q < SL; ++q) low = min(low, key[q]);
    const unsigned m = __reduce_min_sync(0xffffffffu, low);
    const int who = __ffs(__ballot_sync(0xffffffffu, low == m)) - 1;
    int s = 0;
    float p = 0.0f;
#pragma unroll
    for (int q = SL - 1; q >= 0; --q)
      if (key[q] == m) {
        s = lane + 32 * q;
        p = v.ped[q];
      }
    s = __shfl_sync(0xffffffffu, s, who);
    p = __shfl_sync(0xffffffffu, p, who);
#pragma unroll
    for (int q = 0; q < SL; ++q)
      if (s == lane + 32 * q) key[q] = 0xffffffffu;  // taken
    if (lane == 0) cped[t] = p;
    for (int r = lane; r < n; r += 32) {
      const int d = n - 1 - r;
      cx[(size_t)t * cs + r] = (uint8_t)((x[(d >> 3) * KS + s] >> (4 * (d & 7))) & 15u);
    }
    if (t == kCandMax - 1 && !ranked) {
      bool same = false;
#pragma unroll
      for (int q = 0; q < SL; ++q) same |= key[q] == m;
      if (__any_sync(0xffffffffu, same)) return false;
    }
  }
  __syncwarp();
  return true;
}

}  // namespace
}  // namespace mdx
