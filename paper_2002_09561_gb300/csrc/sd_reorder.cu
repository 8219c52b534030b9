// Antenna order of exact sphere decoding: which vectors are searched with
// their antennas sorted, and in which order.
//
// The ML point does not depend on the order in which the tree takes the
// antennas, its cost does: with the strong antennas at the top (their rows of
// R, the last ones, have large diagonals) few children survive the first
// levels.  The order is that of the sorted QR decomposition (Wuebben et al.,
// "Efficient algorithm for decoding layered space-time codes", Electronics
// Letters 37, 2001): columns are taken for the QR by least residual norm.
// Visited nodes per vector on 16x16 16-QAM, network's radius (FP64 oracle):
// 4 dB 49.8 k -> 15.4 k, 6 dB 24.7 k -> 2.7 k, 8 dB 3.5 k -> 750, 10 dB
// 690 -> 160.
//
// The order costs a second QR (of the R at hand with its columns permuted,
// 15 ns a 16x16 vector of a full GPU, about 400 nodes' time), so each vector's
// tree is estimated first: the
// number of lattice points of each level's sublattice in the sphere, volume
// over determinant, capped by P^level (the Gaussian heuristic), for the
// smaller of the initial r^2 and 1.25 n_tx sigma^2 (a little over the expected
// ML distance, which the search's radius reaches soon).  Its correlation with
// the visited nodes is 0.5 .. 0.8 in logarithms, and the vectors that take
// longest are often those it underestimates.  Vectors above kReorderNodes are
// sorted, and searched first; the others keep their R.
//
// Measured (whole calls, ms; threshold none sorted / 1,000 / 100 / 40 / 10 / 0):
//   16x16 16-QAM, 4..20 dB, network's radius, 100,000 vectors
//                                        42.4 / 17.1 / 17.5 / 17.7 / 18.0 / 18.0
//   the same at 12..20 dB, paper radius  18.4 / 12.8 / 8.5 / 8.1 / 8.4 / 8.6
//   18..20 dB                            5.51 / 5.54 / 5.23 / 5.11 / 5.58 / 6.29
//   24x24 16-QAM, 18 dB, 8,000 vectors   9.2 / 8.0 / 5.6 / 4.1 / 3.8 / 3.8
//   20x18 16-QAM, 20..22 dB, 5,000       0.475 / 0.477 / 0.474 / 0.475 / 0.517 / 0.773
#include "mdx_internal.cuh"

namespace mdx {
namespace {

constexpr float kReorderNodes = 40.0f;
constexpr float kNoiseRadius = 1.25f;
constexpr float kMostNodes = 100.0f;  // log2: P^level passes FP32's range from 22 antennas of 64-QAM on

// log2 of the volume of the unit ball in k dimensions
__device__ __forceinline__ float log2_ball(int k) {
  const float h = 0.5f * (float)k;
  return 1.6514961f * h - 1.4426950f * lgammaf(h + 1.0f);  // log2(pi) h - log2(Gamma(h + 1))
}

// G lanes per vector, lane c owning complex column c (n_tx <= G).  The columns
// are orthogonalised in FP32 (the order is a heuristic; answers do not depend
// on it), the chosen column broadcast through shared memory.
template <int G>
__global__ void __launch_bounds__(128) reorder_select_kernel(ReorderArgs g) {
  __shared__ float2 piv[128 / G][G];
  const SearchArgs& a = g.a;
  const int lane = threadIdx.x & 31, c = lane % G, lead = lane - c, grp = threadIdx.x / G;
  const unsigned gmask = (G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u)) << lead;
  const int v = blockIdx.x * (128 / G) + grp;
  const int M = a.n_tx, n = a.n;
  const bool act = v < a.batch;
  const float* R = a.R32 + (size_t)(act ? v : 0) * tri_stride32(n);
  // ---- the tree's estimated size
  const bool mine = act && c < M;
  const float rcc = mine ? R[col_off(2 * c) + 2 * c] : 1.0f;
  const float ld = mine ? 1.0f + log2f(a.alpha * rcc) : 0.0f;  // log2 of one real row's spacing 2 alpha R_ii
  float below = 2.0f * ld;                                     // rows of antennas c .. M - 1
#pragma unroll
  for (int o = 1; o < G; o <<= 1) {
    const float t = __shfl_down_sync(gmask, below, o, G);
    if (c + o < G) below += t;
  }
  float r2 = act ? initial_r2(a, v) : 1.0f;
  if (act && a.noise_var) r2 = fminf(r2, kNoiseRadius * (float)M * (float)a.noise_var[v]);
  const float lr = 0.5f * log2f(r2), lp = log2f((float)a.P);
  float nodes = 0.0f;
  if (mine) {
    const int k = 2 * (M - c);  // both rows of antenna c, then its first alone
    const float b1 = fminf(lp * (float)k, log2_ball(k) + lr * (float)k - below);
    const float b0 = fminf(lp * (float)(k - 1), log2_ball(k - 1) + lr * (float)(k - 1) - (below - ld));
    nodes = exp2f(fminf(b1, kMostNodes)) + exp2f(fminf(b0, kMostNodes));
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) nodes += __shfl_xor_sync(gmask, nodes, o, G);
  // (a zero, infinite or NaN diagonal: left in natural order)
  const bool sound = __all_sync(gmask, !mine || (rcc > 0.0f && rcc < INFINITY));
  const bool pick = act && sound && nodes > kReorderNodes && !(a.singular && a.singular[v]);
  if (act && c == 0) g.sorted[v] = pick ? 1 : 0;
  // the search's order: the vectors chosen from the front, the others from the back
  const unsigned first = __ballot_sync(0xffffffffu, c == 0 && pick);
  const unsigned other = __ballot_sync(0xffffffffu, c == 0 && act && !pick);
  unsigned f0 = 0, o0 = 0;
  if (lane == 0) {
    if (first) f0 = atomicAdd(g.count, (unsigned)__popc(first));
    if (other) o0 = atomicAdd(g.count + 1, (unsigned)__popc(other));
  }
  f0 = __shfl_sync(0xffffffffu, f0, 0);
  o0 = __shfl_sync(0xffffffffu, o0, 0);
  if (act && c == 0) {
    const unsigned before = (1u << lane) - 1u;
    g.list[pick ? f0 + __popc(first & before) : a.batch - 1 - (o0 + __popc(other & before))] = v;
  }
  if (first == 0) return;
  // ---- the order
  float2 q[G];
  float norm = 0.0f;
#pragma unroll
  for (int r = 0; r < G; ++r) {
    q[r] = make_float2(0.0f, 0.0f);
    if (mine && r <= c) {
      const float* at = R + col_off(2 * c) + 2 * r;
      q[r].x = at[0];
      if (r < c) q[r].y = at[1];
    }
    norm = fmaf(q[r].x, q[r].x, fmaf(q[r].y, q[r].y, norm));
  }
  bool left = mine;
  for (int k = 0; k < M; ++k) {
    const unsigned key = left ? __float_as_uint(fmaxf(norm, 0.0f)) : 0xffffffffu;
    const unsigned least = __reduce_min_sync(gmask, key);
    const int p = __ffs(__ballot_sync(gmask, left && key == least) >> lead) - 1;
    if (p < 0) break;  // no column left (an inactive group)
    if (c == p) {
      const float s = norm > 0.0f ? rsqrtf(norm) : 0.0f;
#pragma unroll
      for (int r = 0; r < G; ++r) piv[grp][r] = make_float2(q[r].x * s, q[r].y * s);
      if (pick) {
        g.perm[(size_t)v * M + k] = (uint8_t)c;
        g.place[(size_t)v * M + c] = (uint8_t)k;
      }
      left = false;
    }
    __syncwarp(gmask);
    if (left) {
      float wr = 0.0f, wi = 0.0f;
#pragma unroll
      for (int r = 0; r < G; ++r) {
        const float2 u = piv[grp][r];
        wr = fmaf(u.x, q[r].x, fmaf(u.y, q[r].y, wr));
        wi = fmaf(u.x, q[r].y, fmaf(-u.y, q[r].x, wi));
      }
      norm = 0.0f;
#pragma unroll
      for (int r = 0; r < G; ++r) {
        const float2 u = piv[grp][r];
        q[r].x = fmaf(-u.x, wr, fmaf(u.y, wi, q[r].x));
        q[r].y = fmaf(-u.x, wi, fmaf(-u.y, wr, q[r].y));
        norm = fmaf(q[r].x, q[r].x, fmaf(q[r].y, q[r].y, norm));
      }
    }
    __syncwarp(gmask);
  }
}

}  // namespace

cudaError_t launch_reorder_select(const ReorderArgs& g, cudaStream_t s) {
  if (g.a.n_tx <= 16)
    reorder_select_kernel<16><<<(g.a.batch + 7) / 8, 128, 0, s>>>(g);
  else
    reorder_select_kernel<32><<<(g.a.batch + 3) / 4, 128, 0, s>>>(g);
  return cudaGetLastError();
}

}  // namespace mdx
