// Linear detectors, the controls the paper compares the tree searches with
// (Sec. III-A): zero forcing, x = H^+ y = R^-1 ybar (back substitution on the
// QR workspace), and MMSE, x = (H^H H + sigma^2 I)^-1 H^H y =
// (R^T R + sigma^2 I)^-1 R^T ybar.  Every real component of x is then sliced to
// the nearest PAM level (clipped to the grid) and the metric ||ybar - R x^||^2
// is evaluated in FP64 like the searches' final leaves.
//
// Up to 32 antennas (linear_group_kernel) both are a triangular solve: MMSE is
// the least-squares solution of [R; sigma I] x = [ybar; 0], whose QR the
// fixed-point kernels compute (qr.cu), where normal equations and a Cholesky
// factorisation would run on the FP64 unit (and square the condition number).
// Eight lanes per vector, complex rows r = gl + 8 t each, in FP64: bound by
// the FP64 unit (77 cycles a warp instruction), so the rows' reciprocals are
// formed once, in parallel, and four vectors share a warp.  100,000 16x16
// vectors: MMSE kernel 13.5 ms -> QR of the augmented systems and solve
// together 3.6 ms.  Larger systems, and those the fixed-point QR leaves
// (linear_kernel): one warp per vector, lanes over rows, MMSE by normal
// equations.
#include "mdx_internal.cuh"

namespace mdx {
namespace {

constexpr int kLinWarps = 4;

__host__ __device__ inline size_t lin_warp_bytes(int n, bool mmse) {
  size_t b = sizeof(double) * (size_t)round_up(n, 2) + (size_t)round_up(n, 16);  // x, sliced path
  if (mmse) b += sizeof(double) * ((size_t)n * n + (size_t)round_up(n, 2));       // G (row-major), rhs
  return (b + 15) / 16 * 16;
}

// z / d from rd = 1 / d, corrected by the remainder.
__device__ __forceinline__ double quotient(double z, double d, double rd) {
  const double q = z * rd;
  return fma(fma(-q, d, z), rd, q);
}

// Nearest PAM level of x (inv = 1 / alpha64).
__device__ __forceinline__ uint8_t slice_level(double x, double alpha64, double inv, int P) {
  const double u = 0.5 * (quotient(x, alpha64, inv) + (double)(P - 1));
  double k = floor(u + 0.5);
  k = k < 0.0 ? 0.0 : (k > (double)(P - 1) ? (double)(P - 1) : k);
  return (uint8_t)k;
}

// Back substitution R x = rhs (R column-packed upper triangular, FP64).
// rhs in x on entry, the solution on return; lanes own rows.
__device__ void back_substitute(int n, const double* R, double* x, int lane) {
  for (int i = n - 1; i >= 0; --i) {
    __syncwarp();
    const double xi = x[i] / R[col_off(i) + i];
    __syncwarp();
    const double* col = R + col_off(i);
    for (int r = lane; r < i; r += 32) x[r] = fma(-col[r], xi, x[r]);
    if (lane == 0) x[i] = xi;
  }
  __syncwarp();
}

// only (if not null): the vectors to solve, by a non-zero entry.
__global__ void __launch_bounds__(kLinWarps * 32) linear_kernel(SearchArgs a, int mmse, const int* only) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = a.n, P = a.P;
  unsigned char* base = smem + (size_t)warp * lin_warp_bytes(n, mmse != 0);
  double* x = reinterpret_cast<double*>(base);
  uint8_t* path = reinterpret_cast<uint8_t*>(x + round_up(n, 2));
  double* G = reinterpret_cast<double*>(path + round_up(n, 16));  // MMSE only
  double* rhs = G + (size_t)n * n;
  const double inv = 1.0 / a.alpha64;
  const int gw = blockIdx.x * kLinWarps + warp, nw = gridDim.x * kLinWarps;
  for (int v = gw; v < a.batch; v += nw) {
    if (only && !only[v]) continue;
    if (a.singular && a.singular[v]) {
      for (int j = lane; j < a.n_tx; j += 32) a.sym_out[(size_t)v * a.n_tx + j] = 0;
      if (lane == 0) {
        a.metric_out[v] = 0.0;
        a.vstatus[v] = MDX_V_SINGULAR;
        if (a.stats)
          for (int q = 0; q < kStats; ++q) a.stats[(size_t)v * kStats + q] = 0;
      }
      continue;
    }
    const double* R = a.R64 + (size_t)v * tri_stride64(n);
    const double* yb = a.yb64 + (size_t)v * vec_stride64(n);
    if (!mmse) {
      for (int r = lane; r < n; r += 32) x[r] = yb[r];
      back_substitute(n, R, x, lane);
    } else {
      const double s2 = a.noise_var[v];
      // G = R^T R + sigma^2 I (lower triangle), rhs = R^T ybar
      for (int e = lane; e < n * n; e += 32) {
        const int i = e / n, j = e % n;
        if (j > i) continue;
        const double* ci = R + col_off(i);
        const double* cj = R + col_off(j);
        double g = (i == j) ? s2 : 0.0;
        for (int k = 0; k <= j; ++k) g = fma(ci[k], cj[k], g);
        G[e] = g;
      }
      for (int i = lane; i < n; i += 32) {
        const double* ci = R + col_off(i);
        double b = 0.0;
        for (int k = 0; k <= i; ++k) b = fma(ci[k], yb[k], b);
        rhs[i] = b;
      }
      __syncwarp();
      // Cholesky G = L L^T in place (lower triangle), column by column
      for (int k = 0; k < n; ++k) {
        const double d = sqrt(G[k * n + k]);
        __syncwarp();
        for (int i = k + 1 + lane; i < n; i += 32) G[i * n + k] /= d;
        if (lane == 0) G[k * n + k] = d;
        __syncwarp();
        for (int e = lane; e < (n - k - 1) * (n - k - 1); e += 32) {
          const int i = k + 1 + e / (n - k - 1), j = k + 1 + e % (n - k - 1);
          if (j <= i) G[i * n + j] = fma(-G[i * n + k], G[j * n + k], G[i * n + j]);
        }
        __syncwarp();
      }
      // L z = rhs, then L^T x = z
      for (int i = 0; i < n; ++i) {
        const double zi = rhs[i] / G[i * n + i];
        __syncwarp();
        for (int r = i + 1 + lane; r < n; r += 32) rhs[r] = fma(-G[r * n + i], zi, rhs[r]);
        if (lane == 0) rhs[i] = zi;
        __syncwarp();
      }
      for (int i = n - 1; i >= 0; --i) {
        const double xi = rhs[i] / G[i * n + i];
        __syncwarp();
        for (int r = lane; r < i; r += 32) rhs[r] = fma(-G[i * n + r], xi, rhs[r]);
        if (lane == 0) rhs[i] = xi;
        __syncwarp();
      }
      for (int r = lane; r < n; r += 32) x[r] = rhs[r];
      __syncwarp();
    }
    for (int r = lane; r < n; r += 32) path[r] = slice_level(x[r], a.alpha64, inv, P);
    __syncwarp();
    const double m = rescore_fp64_warp(n, P, a.alpha64, R, yb, path, lane);
    for (int j = lane; j < a.n_tx; j += 32)
      a.sym_out[(size_t)v * a.n_tx + j] = (uint8_t)(path[2 * j] * P + path[2 * j + 1]);
    if (lane == 0) {
      a.metric_out[v] = m;
      a.vstatus[v] = MDX_V_OK;
      if (a.stats) {
        int64_t* s = a.stats + (size_t)v * kStats;
        s[0] = 0;
        s[1] = 0;
        s[2] = 0;
        s[3] = 1;
        s[4] = 0;
      }
    }
    __syncwarp();
  }
}

// T: complex rows per lane (n_tx <= 8 T).
template <bool kMmse, int T>
__global__ void __launch_bounds__(128) linear_group_kernel(AugArgs g) {
  const SearchArgs& a = g.a;
  const int lane = threadIdx.x & 31, gl = lane & 7, lead = lane & ~7;
  const int M = a.n_tx, n = a.n, P = a.P;
  const int v = blockIdx.x * 16 + (threadIdx.x >> 3);
  const bool act = v < a.batch && !(kMmse && g.bad[v]);
  const bool dead = act && a.singular && a.singular[v];
  const int vv = v < a.batch ? v : 0;
  const double* R64 = a.R64 + (size_t)vv * tri_stride64(n);
  const double* y64 = a.yb64 + (size_t)vv * vec_stride64(n);
  const double2* Ra = reinterpret_cast<const double2*>(g.R(vv));
  const double* da = g.diag(vv);
  double zr[T], zi[T], dg[T], rd[T];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int r = gl + 8 * t;
    zr[t] = zi[t] = 0.0;
    dg[t] = 1.0;
    if (r < M) {
      const double* yy = kMmse ? g.y(vv) : y64;
      zr[t] = yy[2 * r];
      zi[t] = yy[2 * r + 1];
      dg[t] = kMmse ? da[r] : R64[col_off(2 * r) + 2 * r];
    }
    rd[t] = 1.0 / dg[t];
  }
  // R x = z, from the last row up
  for (int i = M - 1; i >= 0; --i) {
    const int o = lead | (i & 7);
    double xr = 0.0, xi = 0.0;
#pragma unroll
    for (int t = 0; t < T; ++t)
      if (t == (i >> 3)) {
        xr = quotient(zr[t], dg[t], rd[t]);
        xi = quotient(zi[t], dg[t], rd[t]);
        if (gl == (i & 7)) {
          zr[t] = xr;
          zi[t] = xi;
        }
      }
    xr = __shfl_sync(0xffffffffu, xr, o);
    xi = __shfl_sync(0xffffffffu, xi, o);
#pragma unroll
    for (int t = 0; t < T; ++t) {
      if (8 * t >= i) continue;
      const int r = gl + 8 * t;
      if (r < i) {
        double2 c;
        if (kMmse) {
          c = Ra[i * (i - 1) / 2 + r];
        } else {
          const double* at = R64 + col_off(2 * i) + 2 * r;
          c = make_double2(at[0], at[1]);
        }
        zr[t] = fma(-c.x, xr, fma(c.y, xi, zr[t]));
        zi[t] = fma(-c.x, xi, fma(-c.y, xr, zi[t]));
      }
    }
  }
  // slice, then the residual ybar - R x^ on the natural R
  const double inv = 1.0 / a.alpha64;
  double lr[T], li[T];
  uint8_t sym[T];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int r = gl + 8 * t;
    const int kr = slice_level(zr[t], a.alpha64, inv, P), ki = slice_level(zi[t], a.alpha64, inv, P);
    sym[t] = (uint8_t)(kr * P + ki);
    lr[t] = (double)(2 * kr - (P - 1)) * a.alpha64;
    li[t] = (double)(2 * ki - (P - 1)) * a.alpha64;
    zr[t] = r < M ? y64[2 * r] : 0.0;
    zi[t] = r < M ? y64[2 * r + 1] : 0.0;
  }
  for (int j = 0; j < M; ++j) {
    double xr = 0.0, xi = 0.0;
#pragma unroll
    for (int t = 0; t < T; ++t)
      if (t == (j >> 3)) {
        xr = lr[t];
        xi = li[t];
      }
    xr = __shfl_sync(0xffffffffu, xr, lead | (j & 7));
    xi = __shfl_sync(0xffffffffu, xi, lead | (j & 7));
    const double* at = R64 + col_off(2 * j);
#pragma unroll
    for (int t = 0; t < T; ++t) {
      if (8 * t > j) continue;
      const int r = gl + 8 * t;
      if (r <= j) {
        const double cr = at[2 * r], ci = r < j ? at[2 * r + 1] : 0.0;
        zr[t] = fma(-cr, xr, fma(ci, xi, zr[t]));
        zi[t] = fma(-cr, xi, fma(-ci, xr, zi[t]));
      }
    }
  }
  double m = 0.0;
#pragma unroll
  for (int t = 0; t < T; ++t) m = fma(zr[t], zr[t], fma(zi[t], zi[t], m));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
  if (!act) return;
#pragma unroll
  for (int t = 0; t < T; ++t)
    if (gl + 8 * t < M) a.sym_out[(size_t)v * M + gl + 8 * t] = dead ? 0 : sym[t];
  if (gl == 0) {
    a.metric_out[v] = dead ? 0.0 : m;
    a.vstatus[v] = dead ? MDX_V_SINGULAR : MDX_V_OK;
    if (a.stats)
      for (int q = 0; q < kStats; ++q) a.stats[(size_t)v * kStats + q] = q == 3 && !dead ? 1 : 0;
  }
}

template <int T>
cudaError_t launch_linear_group(const AugArgs& g, bool mmse, cudaStream_t s) {
  const int grid = (g.a.batch + 15) / 16;
  if (mmse)
    linear_group_kernel<true, T><<<grid, 128, 0, s>>>(g);
  else
    linear_group_kernel<false, T><<<grid, 128, 0, s>>>(g);
  return cudaGetLastError();
}

}  // namespace

size_t linear_smem_bytes(int n, bool mmse) { return lin_warp_bytes(n, mmse) * kLinWarps; }

cudaError_t launch_linear(const AugArgs& g, bool mmse, int num_sms, cudaStream_t s) {
  const SearchArgs& a = g.a;
  if (a.batch <= 0) return cudaSuccess;
  const int* only = nullptr;
  if (a.n_tx <= kAugMaxTx) {
    cudaError_t e = mmse ? launch_qr_augmented(g, num_sms, s) : cudaSuccess;
    if (e != cudaSuccess) return e;
    e = a.n_tx <= 8    ? launch_linear_group<1>(g, mmse, s)
        : a.n_tx <= 16 ? launch_linear_group<2>(g, mmse, s)
                       : launch_linear_group<4>(g, mmse, s);
    if (e != cudaSuccess || !mmse) return e;
    only = g.bad;
  }
  const size_t smem = linear_smem_bytes(a.n, mmse);
  if (smem > 227 * 1024) return cudaErrorInvalidConfiguration;
  cudaError_t e = cudaFuncSetAttribute(linear_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, linear_kernel, kLinWarps * 32, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  long long grid = (long long)per_sm * num_sms;
  const long long need = (a.batch + kLinWarps - 1) / kLinWarps;
  if (grid > need) grid = need;
  linear_kernel<<<(int)grid, kLinWarps * 32, smem, s>>>(a, mmse ? 1 : 0, only);
  return cudaGetLastError();
}

}  // namespace mdx
