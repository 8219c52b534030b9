// K-best (Sec. VI) with one received vector per warp, by selection instead of
// sorting.
//
// The selection is that of select_run.cuh (here ties go to the lower parent
// rank, then the lower child): every lane keeps the children of its survivors
// as 32-bit distance bits in registers (SL survivors of C children each), and a
// search on the bits (one compare and add per child and one warp reduction a
// step) finds the K-th smallest.  Sorting 64-bit
// keys, the ALU work that bound the CTA kernel (kbest.cu), disappears, and so
// do its CTA barriers.  Where a tie straddles a cut the parents' distances say
// which children stay; only where those are equal as well is the vector marked
// and left to that kernel, which sorts.
//
// Survivor paths are bytes 2k - (P - 1) in depth order (row n - 1 first, so
// that the rows fixed so far are a prefix), the stride an odd number of
// words.  Interference, partial distances, pruning, counts and re-scoring are
// the CTA kernel's operations in the same order: the same bits.
//
// Measured (whole calls with the QR, CTA kernel before): 16x16 16-QAM K = 64,
// 100,000 vectors 19.7 -> 5.2 ms; complex tree 16x16 64-QAM K = 32, 20,000
// vectors 14.8 -> 2.2 ms; 8x8 64-QAM K = 16 from host memory, 50,000 vectors
// 2.29 -> 1.2 ms.
#include "select_run.cuh"

namespace mdx {
namespace {

constexpr int kWarps = 4;  // vectors per CTA

struct KwLayout {
  int ts, stride;  // floats of R; bytes per path
  size_t off_yb, off_xa, off_xb, off_ent, off_x, warp_bytes;
  __host__ __device__ void init(int n, int K) {
    ts = tri_stride32(n);
    stride = path_stride(n);
    size_t o = sizeof(float) * (size_t)ts;
    off_yb = o;
    o += sizeof(float) * (size_t)round_up(n, 4);
    off_ent = o;
    o += sizeof(uint2) * (size_t)round_up(K, 32);
    off_xa = o;
    o += (size_t)stride * round_up(K, 32);
    off_xb = o;
    o += (size_t)stride * round_up(K, 32);
    off_x = (o + 3) / 4 * 4;
    o = off_x + kCandMax * sizeof(float) + (size_t)round_up(n, 4);
    warp_bytes = (o + 15) / 16 * 16;
  }
};

__device__ __forceinline__ float level_of(unsigned word, int b, float alpha) {
  return (float)(signed char)(word >> (8 * b)) * alpha;
}

// Interference of the row at depth d for the path xp (words, depth order), as
// row_interference (eight chains) ...
__device__ __forceinline__ float interference8(const float* Rc, const float* yb, const uint32_t* xp, int n, float alpha,
                                               int i, int d) {
  float acc[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) acc[m] = m == 0 ? yb[i] : 0.0f;
  int b = 0;
  for (; b + 8 <= d; b += 8) {
    const unsigned w0 = xp[b >> 2], w1 = xp[(b >> 2) + 1];
#pragma unroll
    for (int m = 0; m < 8; ++m)
      acc[m] = fmaf(-Rc[col_off(n - 1 - b - m) + i], level_of(m < 4 ? w0 : w1, m & 3, alpha), acc[m]);
  }
  if (b < d) {
    const unsigned w0 = xp[b >> 2], w1 = b + 4 < d ? xp[(b >> 2) + 1] : 0u;
#pragma unroll
    for (int m = 0; m < 8; ++m)
      if (b + m < d) acc[m] = fmaf(-Rc[col_off(n - 1 - b - m) + i], level_of(m < 4 ? w0 : w1, m & 3, alpha), acc[m]);
  }
#pragma unroll
  for (int s = 1; s < 8; s <<= 1)
#pragma unroll
    for (int m = 0; m < 8; ++m)
      if ((m & s) == 0 && (m & (s - 1)) == 0) acc[m] += acc[m + s];
  return acc[0];
}
// ... or as the CTA kernel's single chain for large K.
__device__ __forceinline__ float interference1(const float* Rc, const float* yb, const uint32_t* xp, int n, float alpha,
                                               int i, int d) {
  float c = yb[i];
  for (int b = 0; b < d; b += 4) {
    const unsigned w = xp[b >> 2];
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (b + m < d) c = fmaf(-Rc[col_off(n - 1 - b - m) + i], level_of(w, m, alpha), c);
  }
  return c;
}

// Keeps, of the children at the distance T that a cut of K straddles, those of
// the lower parent ranks, then the lower children.  Ranks go by distance, so the
// parents' distances tell; false where they are equal and it matters.  (A call
// on copies: in line its registers cost every level 2 %.)
template <int SL, int C>
__device__ __noinline__ bool resolve_cut_at(unsigned* key, unsigned T, int K, const float* ped) {
  int need = K;
  uint64_t tied[SL];
#pragma unroll
  for (int q = 0; q < SL; ++q) tied[q] = 0;
#pragma unroll
  for (int j = 0; j < SL * C; ++j) {
    need -= __popc(__ballot_sync(0xffffffffu, key[j] < T));
    if (key[j] == T) {
      tied[j / C] |= 1ull << (j % C);
      key[j] = 0xffffffffu;
    }
  }
  while (need > 0) {
    unsigned low = 0xffffffffu;
#pragma unroll
    for (int q = 0; q < SL; ++q)
      if (tied[q]) low = min(low, __float_as_uint(ped[q]));
    const unsigned m = __reduce_min_sync(0xffffffffu, low);
    int parents = 0, children = 0;
#pragma unroll
    for (int q = 0; q < SL; ++q)
      if (tied[q] && __float_as_uint(ped[q]) == m) {
        ++parents;
        children += __popcll(tied[q]);
      }
    children = __reduce_add_sync(0xffffffffu, children);
    if (children > need && __reduce_add_sync(0xffffffffu, parents) > 1) return false;
#pragma unroll
    for (int q = 0; q < SL; ++q)
      if (tied[q] && __float_as_uint(ped[q]) == m) {
        int left = need;
#pragma unroll
        for (int k = 0; k < C; ++k)
          if ((tied[q] >> k) & 1ull && left-- > 0) key[q * C + k] = T;
        tied[q] = 0;
      }
    need -= children;
  }
  return true;
}
template <int SL, int C>
__device__ __forceinline__ bool resolve_cut(unsigned (&key)[SL * C], unsigned T, int K, const float (&ped)[SL]) {
  unsigned k[SL * C];
  float p[SL];
#pragma unroll
  for (int j = 0; j < SL * C; ++j) k[j] = key[j];
#pragma unroll
  for (int q = 0; q < SL; ++q) p[q] = ped[q];
  if (!resolve_cut_at<SL, C>(k, T, K, p)) return false;
#pragma unroll
  for (int j = 0; j < SL * C; ++j) key[j] = k[j];
  return true;
}

// SL survivors per lane (K <= 32 SL), C children per survivor: the PAM size P
// of the real tree, or P^2 of the complex one.
template <int SL, int C, bool CPLX>
__global__ void __launch_bounds__(kWarps * 32) kbest_warp_kernel(SearchArgs a, KwLayout L, int eight) {
  constexpr int P = CPLX ? (C == 4 ? 2 : C == 16 ? 4 : 8) : C;
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int v = blockIdx.x * kWarps + warp;
  const int n = a.n, K = a.K;
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
  unsigned char* base = smem + (size_t)warp * L.warp_bytes;
  float* Rc = reinterpret_cast<float*>(base);
  float* yb = reinterpret_cast<float*>(base + L.off_yb);
  uint2* ent = reinterpret_cast<uint2*>(base + L.off_ent);  // {parent | child << 16, distance bits}
  unsigned char* xcur = base + L.off_xa;
  unsigned char* xnxt = base + L.off_xb;
  float* cped = reinterpret_cast<float*>(base + L.off_x);
  uint8_t* xnat = reinterpret_cast<uint8_t*>(cped + kCandMax);
  const double* R64 = a.R64 + (size_t)v * tri_stride64(n);
  const double* y64 = a.yb64 + (size_t)v * vec_stride64(n);
  {
    const float4* src = reinterpret_cast<const float4*>(a.R32 + (size_t)v * L.ts);
    for (int t = lane; t < L.ts / 4; t += 32) reinterpret_cast<float4*>(Rc)[t] = src[t];
    const float* ys = a.yb32 + (size_t)v * vec_stride32(n);
    for (int r = lane; r < n; r += 32) yb[r] = ys[r];
  }
  __syncwarp();
  const float E = error_scale_warp(n, P, a.alpha, Rc, yb, lane);
  const float alpha = a.alpha;
  float r2 = initial_r2(a, v);
  long long nodes = 0, flops = 0;
  int restarts = 0, S = 0;
  float ped[SL];
  bool tie = false;
  for (;;) {
    const float bnd = prune_bound(r2, E, n);
    S = 1;
#pragma unroll
    for (int q = 0; q < SL; ++q) ped[q] = 0.0f;
    constexpr int kStep = CPLX ? 2 : 1;  // rows per level
    for (int d = 0; d < n && S > 0; d += kStep) {
      const int i = n - 1 - d;
      // ---- the children's distance bits, ~0 outside the sphere or empty
      unsigned key[SL * C];
      const float rii = Rc[col_off(i) + i];
      float r01 = 0.0f, r00 = 0.0f;
      if (CPLX) {
        r01 = Rc[col_off(i) + i - 1];
        r00 = Rc[col_off(i - 1) + i - 1];
      }
#pragma unroll
      for (int q = 0; q < SL; ++q) {
        const int s = lane + 32 * q;
#pragma unroll
        for (int k = 0; k < C; ++k) key[q * C + k] = 0xffffffffu;
        if (32 * q >= S) continue;
        const uint32_t* xp = reinterpret_cast<const uint32_t*>(xcur + (size_t)(s < S ? s : 0) * L.stride);
        const float c = (!CPLX && eight) ? interference8(Rc, yb, xp, n, alpha, i, d)
                                         : interference1(Rc, yb, xp, n, alpha, i, d);
        const float c0 = CPLX ? interference1(Rc, yb, xp, n, alpha, i - 1, d) : 0.0f;
        if (s < S) {
#pragma unroll
          for (int k1 = 0; k1 < P; ++k1) {
            const float a1 = (float)(2 * k1 - (P - 1)) * alpha;
            const float d1 = fmaf(-rii, a1, c);
            const float p1 = fmaf(d1, d1, ped[q]);
            if (!CPLX) {
              if (p1 < bnd) key[q * C + k1] = __float_as_uint(p1);
            } else {
              const float t0 = fmaf(-r01, a1, c0);
#pragma unroll
              for (int k0 = 0; k0 < P; ++k0) {
                const float d0 = fmaf(-r00, (float)(2 * k0 - (P - 1)) * alpha, t0);
                const float p0 = fmaf(d0, d0, p1);
                if (p0 < bnd) key[q * C + k0 * P + k1] = __float_as_uint(p0);
              }
            }
          }
        }
      }
      nodes += S;
      flops += CPLX ? (long long)S * (4 * (n - 1 - i) + 10 * C) : (long long)S * (2 * (n - 1 - i) + 4 * C);
      unsigned T;
      int kept;
      if (!level_cut<SL, C>(key, S, K, lane, T, kept) && !resolve_cut<SL, C>(key, T, K, ped)) {
        tie = true;
        break;
      }
      compact_level<SL, C>(key, T, ent, lane);
      __syncwarp();
      // ---- the new survivors' paths: the parent's rows so far and the child's
      const int wd = d >> 2, sh = 8 * (d & 3);  // a complex level's two rows share a word (d is even)
#pragma unroll
      for (int q = 0; q < SL; ++q) {
        const int s = lane + 32 * q;
        if (s < kept) {
          const uint2 e = ent[s];
          const uint32_t* src = reinterpret_cast<const uint32_t*>(xcur + (size_t)(e.x & 0xffffu) * L.stride);
          uint32_t* dst = reinterpret_cast<uint32_t*>(xnxt + (size_t)s * L.stride);
          const int k = (int)(e.x >> 16);
          for (int w = 0; w < wd; ++w) dst[w] = src[w];
          uint32_t word = sh ? src[wd] & ((1u << sh) - 1u) : 0u;
          if (CPLX)
            word |= ((unsigned)(2 * (k % P) - (P - 1)) & 0xffu) << sh | ((unsigned)(2 * (k / P) - (P - 1)) & 0xffu) << (sh + 8);
          else
            word |= ((unsigned)(2 * k - (P - 1)) & 0xffu) << sh;
          dst[wd] = word;
          ped[q] = __uint_as_float(e.y);
        }
      }
      __syncwarp();
      unsigned char* t = xcur;
      xcur = xnxt;
      xnxt = t;
      S = kept;
    }
    if (tie || S > 0 || !(r2 < INFINITY) || restarts >= 64) break;
    r2 *= 2.0f;  // empty sphere: double the radius r^2
    ++restarts;
  }
  // ---- the best kCandMax leaves
  const int nc = min(S, kCandMax);
  int slot[kCandMax];
  float best = INFINITY;
#pragma unroll
  for (int t = 0; t < kCandMax; ++t) {
    slot[t] = 0;
    if (t < nc && !tie) {
      unsigned low = 0xffffffffu;
#pragma unroll
      for (int q = 0; q < SL; ++q)
        if (lane + 32 * q < S) low = min(low, __float_as_uint(ped[q]));
      const unsigned m = __reduce_min_sync(0xffffffffu, low);
      const int who = __ffs(__ballot_sync(0xffffffffu, low == m)) - 1;
      int s = 0;
#pragma unroll
      for (int q = SL - 1; q >= 0; --q)
        if (lane + 32 * q < S && __float_as_uint(ped[q]) == m) s = lane + 32 * q;
      slot[t] = __shfl_sync(0xffffffffu, s, who);
      if (lane == 0) cped[t] = __uint_as_float(m);
      if (t == 0) best = __uint_as_float(m);
#pragma unroll
      for (int q = 0; q < SL; ++q)
        if (slot[t] == lane + 32 * q) ped[q] = __uint_as_float(0xffffffffu);  // taken
      if (t == kCandMax - 1 && __uint_as_float(m) <= prune_bound(best, E, n)) {
        bool same = false;  // another leaf at the last one's distance, and it counts
#pragma unroll
        for (int q = 0; q < SL; ++q) same |= lane + 32 * q < S && __float_as_uint(ped[q]) == m;
        if (__any_sync(0xffffffffu, same)) tie = true;
      }
    }
  }
  if (tie) {
    // left to the sorting kernel
    if (lane == 0) const_cast<int*>(a.singular)[v] = kKbestRedo;
    return;
  }
  __syncwarp();
  const float keep = prune_bound(best, E, n);
  int win = -1;
  double win_m = INFINITY;
  long long rescored = 0;
#pragma unroll
  for (int t = 0; t < kCandMax; ++t) {
    if (t >= nc || !(cped[t] <= keep)) continue;
    const unsigned char* px = xcur + (size_t)slot[t] * L.stride;
    for (int r = lane; r < n; r += 32) xnat[r] = (uint8_t)(((int)(signed char)px[n - 1 - r] + (P - 1)) >> 1);
    __syncwarp();
    double m;
    if (a.flags & MDX_NO_RESCORE) {
      m = (double)cped[t];
    } else {
      m = rescore_fp64_warp(n, P, a.alpha64, R64, y64, xnat, lane);
      ++rescored;
    }
    bool better = m < win_m;
    if (!better && m == win_m && win >= 0) {
      // tie: lexicographically smaller index vector, top row first
      const unsigned char* pw = xcur + (size_t)win * L.stride;
      for (int d = 0; d < n; ++d) {
        const int w1 = (signed char)px[d], w2 = (signed char)pw[d];
        if (w1 != w2) {
          better = w1 < w2;
          break;
        }
      }
    }
    if (better) {
      win = slot[t];
      win_m = m;
    }
    __syncwarp();
  }
  for (int j = lane; j < a.n_tx; j += 32) {
    uint8_t q = 0;
    if (win >= 0) {
      const signed char* px = reinterpret_cast<const signed char*>(xcur + (size_t)win * L.stride);
      const int kre = (px[n - 1 - 2 * j] + (P - 1)) >> 1, kim = (px[n - 2 - 2 * j] + (P - 1)) >> 1;
      q = (uint8_t)(kre * P + kim);
    }
    a.sym_out[(size_t)v * a.n_tx + j] = q;
  }
  if (lane == 0) {
    a.metric_out[v] = (win >= 0) ? win_m : (double)INFINITY;
    a.vstatus[v] = restarts > 0 ? MDX_V_EMPTY_RETRIED : MDX_V_OK;
    if (a.stats) {
      int64_t* st = a.stats + (size_t)v * kStats;
      st[0] = nodes;
      st[1] = nodes * C;
      st[2] = restarts;
      st[3] = rescored;
      st[4] = flops;
    }
  }
}

template <int SL, int C, bool CPLX>
cudaError_t launch_kw(const SearchArgs& a, const KwLayout& L, bool eight, cudaStream_t s) {
  const size_t sm = L.warp_bytes * kWarps;
  const cudaError_t e =
      cudaFuncSetAttribute(kbest_warp_kernel<SL, C, CPLX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  kbest_warp_kernel<SL, C, CPLX><<<(a.batch + kWarps - 1) / kWarps, kWarps * 32, sm, s>>>(a, L, eight ? 1 : 0);
  return cudaGetLastError();
}

template <int C, bool CPLX>
cudaError_t launch_kw_k(const SearchArgs& a, const KwLayout& L, bool eight, cudaStream_t s) {
  if constexpr (C <= 64) {
    if (a.K <= 32) return launch_kw<1, C, CPLX>(a, L, eight, s);
  }
  if constexpr (2 * C <= 64) {
    if (a.K <= 64) return launch_kw<2, C, CPLX>(a, L, eight, s);
  }
  if constexpr (4 * C <= 64) {
    if (a.K <= 128) return launch_kw<4, C, CPLX>(a, L, eight, s);
  }
  if constexpr (8 * C <= 64) {
    if (a.K <= 256) return launch_kw<8, C, CPLX>(a, L, eight, s);
  }
  return cudaErrorNotSupported;
}

// Where a vector per warp (`warps` of them on an SM) is faster than the sorting
// CTA.  A warp takes its lanes' children one after another, so a vector alone
// takes longer where a lane has many survivors (large K of few children: the CTA
// sorts those on many threads); with the SMs full, the warp's fewer instructions
// win, except where its shared memory leaves an SM one CTA.  A cut of K <= 4 is a
// sort of a few keys.  Measured, time of the warp form over the sorting one, whole
// calls with the QR, 150 / 600 / 2,500 vectors:
//   real tree    K = 4 64-QAM 16 rows 1.10 / 1.14 / 1.10, 64 rows 1.17 / 1.12 / 1.20; 4-QAM 64 rows 0.91 / 0.95 / 1.10
//                K = 32 64 rows, 4-QAM 0.58 / 0.61 / 0.67, 64-QAM 0.60 / 0.57 / 0.51
//                K = 256 4-QAM 32 rows 1.56 / 0.98 / 0.77, 64 rows (a CTA on an SM) 2.25 / 1.29 / 1.54;
//                16-QAM 32 rows 1.27 / 0.50 / 0.37; 64-QAM 32 rows 0.85 / 0.27 / 0.20
//   complex tree K = 4 16 rows, 16-QAM 1.18 / 1.19 / 1.11, 64-QAM 1.23 / 1.14 / 0.99
//                K = 16 32 rows, 4-QAM 1.08 / 1.10 / 0.99, 16-QAM 1.06 / 0.94 / 0.61, 64-QAM 1.24 / 0.63 / 0.40
//                K = 32 32 rows, 4-QAM 0.92 / 0.93 / 0.75, 64-QAM 0.90 / 0.37 / 0.21
//                K = 128 32 rows, 4-QAM 1.47 / 0.96 / 0.71, 16-QAM 1.32 / 0.53 / 0.33
//                K = 48 4-QAM 96 rows (a CTA on an SM) 1.34 / 1.13 / 1.44
bool selection_pays(const SearchArgs& a, int warps, int num_sms) {
  const int K = a.K, P = a.P, per_sm = (a.batch + num_sms - 1) / num_sms;
  if (!(a.flags & MDX_COMPLEX_TREE)) {
    if (K <= 4) return P < 8 && a.n > 32;
    if (K > 128 && P < 8) return per_sm > 2 && !(P == 2 && warps <= 4);
    return true;
  }
  if (K <= 4) return P == 8 && per_sm > 8 && warps > 8;
  if (K <= 16 && P == 2) return per_sm > 8 && warps > 16;
  if (K > 16 && (P == 8 || (P == 2 && K <= 32))) return true;
  return per_sm > (P == 2 || warps <= 8 ? 2 : 1) && !(P == 2 && warps <= 4);
}

}  // namespace

// Runs where a lane's children fit in registers (64 distances), four vectors
// in an SM's shared memory, and where it pays; else cudaErrorNotSupported,
// nothing launched.
cudaError_t launch_kbest_warp(const SearchArgs& a, bool eight, int num_sms, cudaStream_t s) {
  KwLayout L;
  L.init(a.n, a.K);
  const int ctas = (int)(228 * 1024 / (L.warp_bytes * kWarps + 1024));
  if (L.warp_bytes * kWarps > 227 * 1024 || !selection_pays(a, ctas * kWarps, num_sms)) return cudaErrorNotSupported;
  if (a.flags & MDX_COMPLEX_TREE) {
    if (a.P == 2) return launch_kw_k<4, true>(a, L, eight, s);
    if (a.P == 4) return launch_kw_k<16, true>(a, L, eight, s);
    return launch_kw_k<64, true>(a, L, eight, s);
  }
  if (a.P == 2) return launch_kw_k<2, false>(a, L, eight, s);
  if (a.P == 4) return launch_kw_k<4, false>(a, L, eight, s);
  return launch_kw_k<8, false>(a, L, eight, s);
}

}  // namespace mdx
