// Batched QR preprocessing (Sec. III-B): H = QR with a real positive diagonal
// and ybar = Q^H y, by complex Householder reflections applied to the
// augmented matrix [H | y] in 58-bit fixed point on the integer multiply-add pipe
// (fx64.cuh: this GPU's FP64 unit is thirty times slower per multiply-add
// instruction), with errors of a column's norm below those of FP64 arithmetic.
// Two forms: up to 32 receive antennas and enough matrices to fill the GPU,
// several matrices per warp held in registers (qr_small_kernel); otherwise one CTA
// per matrix in shared memory (qr_cta_kernel).  The few matrices that a fixed scale
// per column does not suit (a residual column below 2^-26 of its norm: singular or
// nearly so; last rows far below the first; infinities, NaN and exponents near the
// ends of the range) are factored by the FP64 forms (qr_small64, qr_one).  The
// complex R is written out in the real interleaved form (entry r_ab ->
// [[Re,-Im],[Im,Re]]) that the tree search uses.
//
// Measured (GB300; before: FP64 FMAs and FP64 MMA trailing updates): one 16x16
// matrix 384 -> 28 us, 100,000 of them 4.02 -> 1.42 ms, 3,000 64x64 7.52 ->
// 2.0 ms, 4,000 100x100 31.5 -> 9.9 ms; error of R against 64 bits 2.5e-15
// -> 1.9e-15 (64x64, of which the reference's own is most).
#include <algorithm>
#include <type_traits>

#include "fx64.cuh"
#include "mdx_internal.cuh"

namespace mdx {
namespace {

template <int LPC>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = LPC / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Output bases of one matrix (any pointer may be null).
struct QrDst {
  double* R64;
  double* yb64;
  float* R32;
  float* yb32;
  double* Rdense;
  double* ybdense;
  int* singular;
  // a re-factored R (SrcR): only R32 and yb32 are written, and where the
  // matrix needs the FP64 form the natural ones are restored and *sorted cleared
  uint8_t* sorted = nullptr;
  // the augmented system of MMSE (SrcAug): R above the diagonal as complex
  // numbers, column c at c (c - 1) / 2, its diagonal, Q^H y, and the mark
  longlong2* pk = nullptr;
  i64* pk_diag = nullptr;
  longlong2* pk_y = nullptr;
  int* pk_bad = nullptr;
};

// Phase fix and output of a factorised [R | ybar]: row k of R and ybar_k are
// multiplied by conj(alpha_k / |alpha_k|) so that R_kk = |alpha_k| > 0; R is
// written in the real interleaved form (entry r_ab -> [[Re,-Im],[Im,Re]]).
// getA(c, r) returns the complex entry of column c, row r (r < c for R, the
// ybar column is c = M).
// alpha and tau are overwritten: alpha_k by its phase alpha_k / |alpha_k|
// (1 if zero) and tau_k by |alpha_k|.
template <typename GetA>
__device__ void qr_writeout(int M, GetA getA, double2* alpha, double* tau, const QrDst& out) {
  const int tid = threadIdx.x;
  const int nthr = blockDim.x;
  for (int a = tid; a < M; a += nthr) {
    const double2 al = alpha[a];
    const double aa = hypot(al.x, al.y);
    alpha[a] = (aa > 0.0) ? make_double2(al.x / aa, al.y / aa) : make_double2(1.0, 0.0);
    tau[a] = aa;
  }
  __syncthreads();
  const int n = 2 * M;
  const int nb = M * (M + 1) / 2;  // complex entries (a, c) with a <= c
  for (int t = tid; t < nb; t += nthr) {
    // unrank t -> (a, c), a <= c, column-major over c
    int c = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);  // exact after the corrections below
    while (c * (c + 1) / 2 > t) --c;
    while ((c + 1) * (c + 2) / 2 <= t) ++c;
    const int a = t - c * (c + 1) / 2;
    const double2 ph = alpha[a];
    const double aa = tau[a];
    double re, im;
    if (a == c) {
      re = aa;
      im = 0.0;
    } else {
      const double2 r = getA(c, a);
      re = r.x * ph.x + r.y * ph.y;  // r * conj(ph)
      im = r.y * ph.x - r.x * ph.y;
    }
    const int r0 = 2 * a, c0 = 2 * c;
    // the 2x2 block [[re, -im], [im, re]] at rows r0..r0+1, columns c0..c0+1
    const double vals[4] = {re, -im, im, re};
    const int rows[4] = {r0, r0, r0 + 1, r0 + 1};
    const int cols[4] = {c0, c0 + 1, c0, c0 + 1};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int rr = rows[e], cc = cols[e];
      if (rr > cc) continue;  // below the diagonal (only in diagonal blocks)
      const double v = vals[e];
      if (out.R64) out.R64[col_off(cc) + rr] = v;
      if (out.R32) out.R32[col_off(cc) + rr] = (float)v;
      if (out.Rdense) out.Rdense[(size_t)rr * n + cc] = v;
    }
  }
  if (out.Rdense) {
    // zero the rest of the lower triangle
    for (int t = tid; t < n * n; t += nthr) {
      const int rr = t / n, cc = t % n;
      if (rr > cc) out.Rdense[t] = 0.0;
    }
  }
  for (int a = tid; a < M; a += nthr) {
    const double2 ph = alpha[a];
    const double2 r = getA(M, a);
    const double re = r.x * ph.x + r.y * ph.y, im = r.y * ph.x - r.x * ph.y;
    if (out.yb64) {
      out.yb64[2 * a] = re;
      out.yb64[2 * a + 1] = im;
    }
    if (out.yb32) {
      out.yb32[2 * a] = (float)re;
      out.yb32[2 * a + 1] = (float)im;
    }
    if (out.ybdense) {
      out.ybdense[2 * a] = re;
      out.ybdense[2 * a + 1] = im;
    }
  }
}

// Factorises one [H | y] (N x M complex, row-major; y of N) with the calling CTA.
template <int LPC>
__device__ void qr_one(int N, int M, const double2* __restrict__ Hb, const double2* __restrict__ yb,
                       const QrDst& out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* A = reinterpret_cast<double2*>(smem_raw);  // column-major, (M+1) columns of N
  double2* alpha = A + (size_t)(M + 1) * N;           // R_kk before the phase fix
  double* tau = reinterpret_cast<double*>(alpha + M);
  int* sing = reinterpret_cast<int*>(tau + M);

  const int tid = threadIdx.x;
  const int nthr = blockDim.x;
  const int lane_g = tid % LPC;  // lane within the column worker
  const int worker = tid / LPC;
  const int nworkers = nthr / LPC;

  // load [H | y] (global row-major complex) into column-major smem
  for (int t = tid; t < N * M; t += nthr) {
    const int r = t / M, c = t % M;
    A[(size_t)c * N + r] = Hb[t];
  }
  for (int r = tid; r < N; r += nthr) A[(size_t)M * N + r] = yb[r];
  if (tid == 0) *sing = 0;
  __syncthreads();

  for (int k = 0; k < M; ++k) {
    double2* col = A + (size_t)k * N;
    if (tid < 32) {
      // warp 0 forms the reflector; with LPC < 32 its workers all compute the same
      // sums, so full-warp shuffles stay uniform
      double s = 0.0;
      for (int i = k + lane_g; i < N; i += LPC) s += col[i].x * col[i].x + col[i].y * col[i].y;
      s = group_sum<LPC>(s);
      const double sigma = sqrt(s);
      const double2 x0 = col[k];
      const double ax0 = hypot(x0.x, x0.y);
      double2 al;
      double t = 0.0;
      if (sigma == 0.0) {
        al = make_double2(0.0, 0.0);
      } else {
        // alpha = -e^{i arg x0} sigma keeps v_0 = x0 - alpha free of cancellation
        const double2 ph = (ax0 > 0.0) ? make_double2(x0.x / ax0, x0.y / ax0) : make_double2(1.0, 0.0);
        al = make_double2(-ph.x * sigma, -ph.y * sigma);
        t = 1.0 / (sigma * (sigma + ax0));  // 2 / ||v||^2
      }
      __syncwarp();
      if (tid == 0) {
        alpha[k] = al;
        tau[k] = t;
        if (sigma == 0.0) *sing = 1;
        col[k] = make_double2(x0.x - al.x, x0.y - al.y);  // v_0; v_i = col[i] for i > k
      }
    }
    __syncthreads();
    const double t = tau[k];
    if (t != 0.0) {
      // every lane of a warp runs the same number of iterations (shuffles inside)
      for (int base = k + 1; base <= M; base += nworkers) {
        const int j = base + worker;
        const bool act = j <= M;
        double2* cj = A + (size_t)(act ? j : M) * N;
        double wr = 0.0, wi = 0.0;  // w = v^H a_j
        if (act) {
          for (int i = k + lane_g; i < N; i += LPC) {
            const double2 v = col[i], a = cj[i];
            if constexpr (LPC == 32) {
              wr += v.x * a.x + v.y * a.y;
              wi += v.x * a.y - v.y * a.x;
            } else {  // eight FP64 instructions an entry instead of twelve
              wr = fma(v.x, a.x, fma(v.y, a.y, wr));
              wi = fma(v.x, a.y, fma(-v.y, a.x, wi));
            }
          }
        }
        wr = group_sum<LPC>(wr) * t;
        wi = group_sum<LPC>(wi) * t;
        if (act) {
          for (int i = k + lane_g; i < N; i += LPC) {
            const double2 v = col[i];
            double2 a = cj[i];
            if constexpr (LPC == 32) {
              a.x -= v.x * wr - v.y * wi;
              a.y -= v.x * wi + v.y * wr;
            } else {
              a.x = fma(-v.x, wr, fma(v.y, wi, a.x));
              a.y = fma(-v.x, wi, fma(-v.y, wr, a.y));
            }
            cj[i] = a;
          }
        }
      }
    }
    __syncthreads();
  }

  qr_writeout(M, [&](int c, int r) { return A[(size_t)c * N + r]; }, alpha, tau, out);
  if (out.singular && tid == 0) *out.singular = *sing;
}

// One R entry z = R_kc (complex, after the phase fix) as double bit patterns
// in the real interleaved outputs: the block [[Re, -Im], [Im, Re]] at rows
// 2k.., columns 2c..
constexpr u64 kSignBit = 0x8000000000000000ull;
__device__ __forceinline__ float f32_of(u64 bits) {
  // the conversion instruction runs on the FP64 unit; needed only outside float's normal range
  const unsigned ex = (unsigned)(bits >> 52) & 0x7ffu;
  if (bits == 0 || (ex > 897u && ex < 1150u)) return __uint_as_float(f32_bits_of(bits));
  return (float)__longlong_as_double((i64)bits);
}
__device__ __forceinline__ void put_r(const QrDst& out, int n, int k, int c, u64 re, u64 im) {
  if (out.pk) {
    if (k == c)
      out.pk_diag[c] = (i64)re;
    else
      out.pk[c * (c - 1) / 2 + k] = make_longlong2((i64)re, (i64)im);
    return;
  }
  const int o0 = col_off(2 * c) + 2 * k, o1 = col_off(2 * c + 1) + 2 * k;
  const bool diag = k == c;  // the block's entry below the diagonal is not stored
  const u64 nim = im ? im ^ kSignBit : im;
  if (out.R64) {
    i64* R = reinterpret_cast<i64*>(out.R64);
    R[o0] = (i64)re;
    R[o1] = (i64)nim;
    R[o1 + 1] = (i64)re;
    if (!diag) R[o0 + 1] = (i64)im;
  }
  if (out.R32) {
    const float fr = f32_of(re), fi = f32_of(im);
    out.R32[o0] = fr;
    out.R32[o1] = im ? -fi : fi;
    out.R32[o1 + 1] = fr;
    if (!diag) out.R32[o0 + 1] = fi;
  }
  if (out.Rdense) {
    i64* D = reinterpret_cast<i64*>(out.Rdense) + (size_t)(2 * k) * n + 2 * c;
    D[0] = (i64)re;
    D[1] = (i64)nim;
    D[n] = diag ? 0 : (i64)im;
    D[n + 1] = (i64)re;
  }
}
__device__ __forceinline__ void put_y(const QrDst& out, int k, u64 re, u64 im) {
  if (out.pk) {
    out.pk_y[k] = make_longlong2((i64)re, (i64)im);
    return;
  }
  if (out.yb64) {
    reinterpret_cast<i64*>(out.yb64)[2 * k] = (i64)re;
    reinterpret_cast<i64*>(out.yb64)[2 * k + 1] = (i64)im;
  }
  if (out.yb32) {
    out.yb32[2 * k] = f32_of(re);
    out.yb32[2 * k + 1] = f32_of(im);
  }
  if (out.ybdense) {
    reinterpret_cast<i64*>(out.ybdense)[2 * k] = (i64)re;
    reinterpret_cast<i64*>(out.ybdense)[2 * k + 1] = (i64)im;
  }
}

// ---------------------------------------------------------------------------
// The FP64 form of a small system (n_rx <= 32), column by column in the
// left-looking order, L lanes per matrix: lane h of the group holds rows L q + h
// of the current column.  kMats matrices by the warp (32 / L, or one by its first
// group, the other lanes running along on zeros).  V, Tau: kMats qs_vo(M, N)
// reflector entries, the matrices innermost, and kMats M scalars of shared memory.
__host__ __device__ inline int qs_vo(int k, int N) { return k * N - k * (k - 1) / 2; }  // first entry of v_k
// Conversions between a positive normal double in [1e-30, 1e30] and a float
// estimate of it, done on the integer pipe (rebias the exponent, keep the top
// 23 fraction bits): an FP64 conversion would occupy the FP64 unit.
__device__ __forceinline__ float f32_estimate(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = ((hi >> 20) & 0x7ffu) - 1023u + 127u;
  return __uint_as_float((e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
}
__device__ __forceinline__ double f64_of(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned e = ((b >> 23) & 0xffu) - 127u + 1023u;
  return __hiloint2double((int)((e << 20) | ((b & 0x7fffffu) >> 3)), (int)((b & 7u) << 29));
}

// 1 / sqrt(x) for a positive x: a single-precision estimate y0 (relative
// error below 2^-21) refined by one third-order step of the binomial series
// (1 - e)^(-1/2) = 1 + e/2 + 3e^2/8 + O(e^3), e = 1 - x y0^2 (error below
// 2^-60 before rounding).
__device__ __forceinline__ double rsqrt64(double x) {
  if (!(x > 1e-30 && x < 1e30)) return 1.0 / sqrt(x);
  const double y = f64_of(rsqrtf(f32_estimate(x)));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y, e * fma(0.375, e, 0.5), y);
}
// 1 / d for a positive d: single-precision estimate refined by one
// third-order step of 1 / (1 - e) = 1 + e + e^2 + O(e^3), e = 1 - d y0.
__device__ __forceinline__ double rcp64(double d) {
  if (!(d > 1e-30 && d < 1e30)) return 1.0 / d;
  const double y = f64_of(__frcp_rn(f32_estimate(d)));
  const double e = fma(-d, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

template <int L, int kMats>
__device__ void qr_small64(int N, int M, bool act, const double2* __restrict__ Hb, const double2* __restrict__ yv,
                           const QrDst& out, double2* V, double* Tau) {
  constexpr int kQsSlots = 8;  // rows per lane (N <= 8 L)
  const int lane = threadIdx.x & 31, h = lane % L;
  const int n = 2 * M;
  V += lane / L % kMats;
  Tau += lane / L % kMats;
  double2 a[kQsSlots], ph[kQsSlots];
#pragma unroll
  for (int q = 0; q < kQsSlots; ++q) ph[q] = make_double2(1.0, 0.0);
  int sing = 0;
  for (int j = 0; j <= M; ++j) {
#pragma unroll
    for (int q = 0; q < kQsSlots; ++q) {
      const int r = L * q + h;
      a[q] = make_double2(0.0, 0.0);
      if (act && r < N) a[q] = (j < M) ? Hb[(size_t)r * M + j] : yv[r];
    }
    // reflectors 0 .. j-1: a <- a - v_k tau_k (v_k^H a) over rows k..N-1
    const int kend = j < M ? j : M;
    for (int k = 0; k < kend; ++k) {
      const double2* vk = V + (size_t)(qs_vo(k, N) - k) * kMats;  // entry r at vk[r kMats]
      double wr = 0.0, wi = 0.0;
#pragma unroll
      for (int q = 0; q < kQsSlots; ++q) {
        const int r = L * q + h;
        if (L * q + L - 1 < k || L * q >= N) continue;  // no lane of the group has this row
        if (r >= k && r < N) {
          const double2 v = vk[r * kMats];
          wr = fma(v.x, a[q].x, fma(v.y, a[q].y, wr));
          wi = fma(v.x, a[q].y, fma(-v.y, a[q].x, wi));
        }
      }
#pragma unroll
      for (int o = 1; o < L; o <<= 1) {
        wr += __shfl_xor_sync(0xffffffffu, wr, o);
        wi += __shfl_xor_sync(0xffffffffu, wi, o);
      }
      const double tk = Tau[k * kMats];
      wr *= tk;
      wi *= tk;
#pragma unroll
      for (int q = 0; q < kQsSlots; ++q) {
        const int r = L * q + h;
        if (L * q + L - 1 < k || L * q >= N) continue;
        if (r >= k && r < N) {
          const double2 v = vk[r * kMats];
          a[q].x = fma(-v.x, wr, fma(v.y, wi, a[q].x));
          a[q].y = fma(-v.x, wi, fma(-v.y, wr, a[q].y));
        }
      }
    }
    if (j < M) {
      // column j of R above the diagonal: rows k < j, final now, phase-fixed
#pragma unroll
      for (int q = 0; q < kQsSlots; ++q) {
        const int r = L * q + h;
        if (act && r < j) {
          const double re = a[q].x * ph[q].x + a[q].y * ph[q].y, im = a[q].y * ph[q].x - a[q].x * ph[q].y;
          put_r(out, n, r, j, (u64)__double_as_longlong(re), (u64)__double_as_longlong(im));
        }
      }
      // reflector j from rows j..N-1
      double s = 0.0;
      double2 x0 = make_double2(0.0, 0.0);
#pragma unroll
      for (int q = 0; q < kQsSlots; ++q) {
        const int r = L * q + h;
        if (r >= j && r < N) s = fma(a[q].x, a[q].x, fma(a[q].y, a[q].y, s));
        if (r == j) x0 = a[q];
      }
#pragma unroll
      for (int o = 1; o < L; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const int h0 = j % L;
      x0.x = __shfl_sync(0xffffffffu, x0.x, (lane & ~(L - 1)) | h0);
      x0.y = __shfl_sync(0xffffffffu, x0.y, (lane & ~(L - 1)) | h0);
      double sigma = 0.0, tj = 0.0;
      double2 phr = make_double2(1.0, 0.0), al = make_double2(0.0, 0.0);
      if (s > 0.0) {
        const double rs = rsqrt64(s);
        sigma = s * rs;
        const double qq = fma(x0.x, x0.x, x0.y * x0.y);
        double ax0 = 0.0;
        double2 p0 = make_double2(1.0, 0.0);
        if (qq > 0.0) {
          const double rq = rsqrt64(qq);
          ax0 = qq * rq;
          p0 = make_double2(x0.x * rq, x0.y * rq);
        }
        // alpha = -e^{i arg x0} sigma keeps v_j = x0 - alpha free of cancellation
        al = make_double2(-p0.x * sigma, -p0.y * sigma);
        phr = make_double2(-p0.x, -p0.y);
        tj = rcp64(sigma * (sigma + ax0));
      } else {
        sing = 1;
      }
      double2* vj = V + (size_t)(qs_vo(j, N) - j) * kMats;
#pragma unroll
      for (int q = 0; q < kQsSlots; ++q) {
        const int r = L * q + h;
        if (act && r >= j && r < N) vj[r * kMats] = (r == j) ? make_double2(x0.x - al.x, x0.y - al.y) : a[q];
        if (r == j) ph[q] = phr;
      }
      if (act && h == 0) Tau[j * kMats] = tj;
      if (act && h == h0) put_r(out, n, j, j, (u64)__double_as_longlong(sigma), 0);
    } else {
      // ybar = Q^H y: rows k < M of the y column, phase-fixed
#pragma unroll
      for (int q = 0; q < kQsSlots; ++q) {
        const int r = L * q + h;
        if (act && r < M) {
          const double re = a[q].x * ph[q].x + a[q].y * ph[q].y, im = a[q].y * ph[q].x - a[q].x * ph[q].y;
          put_y(out, r, (u64)__double_as_longlong(re), (u64)__double_as_longlong(im));
        }
      }
    }
    __syncwarp();
  }
  if (act) {
    if (out.Rdense)
      for (int t = h; t < n * n; t += L)
        if (t / n > t % n) out.Rdense[t] = 0.0;
    if (h == 0 && out.singular) *out.singular = sing;
  }
}


// Lanes per matrix (as few as hold the column in eight slots: every FP64
// instruction then serves many rows), and shared memory of `mats` matrices.
__host__ __device__ inline int qs64_lanes(int N) { return N <= 16 ? 2 : 4; }
__host__ __device__ inline size_t qs64_smem(int N, int M, int mats) {
  return (sizeof(double2) * (size_t)qs_vo(M, N) + sizeof(double) * (size_t)M) * mats;
}
// Factorises one [H | y] (n_rx <= 32) in FP64 with the calling CTA's first warp.
__device__ __noinline__ void qr_small64_one(int N, int M, const double* Hb, const double* yb, const QrDst& out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const double2* H2 = reinterpret_cast<const double2*>(Hb);
  const double2* y2 = reinterpret_cast<const double2*>(yb);
  if (threadIdx.x >= 32) return;
  double2* V = reinterpret_cast<double2*>(smem_raw);
  double* Tau = reinterpret_cast<double*>(V + qs_vo(M, N));
  if (qs64_lanes(N) == 2)
    qr_small64<2, 1>(N, M, threadIdx.x < 2, H2, y2, out, V, Tau);
  else
    qr_small64<4, 1>(N, M, threadIdx.x < 4, H2, y2, out, V, Tau);
}
__host__ __device__ inline size_t qr_one_smem(int N, int M) {
  return sizeof(double2) * ((size_t)(M + 1) * N + M) + sizeof(double) * M + sizeof(int) * 4;
}

// a conj(p) of a fixed-point entry and a phase p (limbs), as double bits.
__device__ __forceinline__ void fx_unphase(i64 ar, i64 ai, int4 p, int e, u64& re, u64& im) {
  const int4 a = fx_split(ar, ai);
  const i64 mr = wide_add(a.x, p.y, wide_add(a.y, p.x, wide_add(a.z, p.w, wide(a.w, p.z))));
  const i64 mi = wide_add(a.z, p.y, wide(a.w, p.x)) - wide_add(a.x, p.w, wide(a.y, p.z));
  re = fx_to_bits(wide(a.x, p.x) + wide(a.z, p.z) + ((mr + kFxHalf) >> kFxLimb), e);
  im = fx_to_bits(wide(a.z, p.x) - wide(a.x, p.z) + ((mi + kFxHalf) >> kFxLimb), e);
}

// u^H a summed over a lane's rows, one entry at a time (the low limbs'
// products, below a quarter of a unit each, are left out).  A wide multiply-add
// holds the multiplier for four cycles, so a complex product takes three real
// ones instead of four: with k1 = ur ar, k2 = ui ai and p = (ur + ui)(ai - ar),
// the real part is k1 + k2, the imaginary part p + k1 - k2.
struct FxDot {
  i64 k1h = 0, k1m = 0, k2h = 0, k2m = 0, ph = 0, pm = 0;
  __device__ __forceinline__ void add(int4 u, i64 ar, i64 ai) {
    const int4 a = fx_split(ar, ai);
    const int sh = u.x + u.z, sl = u.y + u.w, dh = a.z - a.x, dl = a.w - a.y;
    k1h = wide_add(u.x, a.x, k1h);
    k1m = wide_add(u.x, a.y, k1m);
    k1m = wide_add(u.y, a.x, k1m);
    k2h = wide_add(u.z, a.z, k2h);
    k2m = wide_add(u.z, a.w, k2m);
    k2m = wide_add(u.w, a.z, k2m);
    ph = wide_add(sh, dh, ph);
    pm = wide_add(sh, dl, pm);
    pm = wide_add(sl, dh, pm);
  }
  __device__ __forceinline__ i64 re() const { return (k1h + k2h) + ((k1m + k2m + kFxHalf) >> kFxLimb); }
  __device__ __forceinline__ i64 im() const {
    return (ph + (k1h - k2h)) + ((pm + (k1m - k2m) + kFxHalf) >> kFxLimb);
  }
};
// The multiplier w of an update a - u w, as limbs: -wr, wi and -(wr + wi).
struct FxMul {
  int nrh, nrl, ih, il, nsh, nsl;
  __device__ __forceinline__ FxMul(i64 wr, i64 wi)
      : nrh(fx_hi(-wr)), nrl(fx_lo(-wr)), ih(fx_hi(wi)), il(fx_lo(wi)), nsh(fx_hi(-wr) - fx_hi(wi)),
        nsl(fx_lo(-wr) - fx_lo(wi)) {}
};
// a - u w: with p1 = -ur wr, p2 = ui wi and p3 = -(ur + ui)(wr + wi), the real
// part gains p1 + p2, the imaginary part p3 - p1 + p2.
__device__ __forceinline__ void fx_axpy(int4 u, const FxMul& w, i64& ar, i64& ai) {
  const int sh = u.x + u.z, sl = u.y + u.w;
  const i64 h1 = wide(u.x, w.nrh), m1 = wide_add(u.y, w.nrh, wide(u.x, w.nrl));
  const i64 h2 = wide(u.z, w.ih), m2 = wide_add(u.w, w.ih, wide_add(u.z, w.il, kFxHalf));
  const i64 m3 = wide_add(sl, w.nsh, wide_add(sh, w.nsl, m2));
  ar += h1 + h2 + ((m1 + m2) >> kFxLimb);
  ai = wide_add(sh, w.nsh, ai) + (h2 - h1) + ((m3 - m1) >> kFxLimb);
}
// Sums of squares of a reflector column (see fx_reflector).
struct FxNorm {
  i64 hh = 0, md = 0;
  u64 ll = 0;
  __device__ __forceinline__ void add(i64 x) {
    const int h = fx_hi(x), l = fx_lo(x);
    hh = wide_add(h, h, hh);
    md = wide_add(h, l, md);
    ll = (u64)wide_add(l, l, (i64)ll);
  }
};
// The power of two 2^e (e returned) that scales a column of norm^2 ss 2^(2 ex - 2046),
// ex the largest exponent field in it: norm in [2^(e-1), 2^e).
__device__ __forceinline__ int fx_scale(int ex, float ss) {
  const int es = (int)(__float_as_uint(ss) >> 23) - 127;  // floor(log2 ss), ss >= 1
  return ex - 1023 + ((es + 2) >> 1);
}
__device__ __forceinline__ int ex_of(u64 bits) { return (int)(bits >> 52) & 0x7ff; }
// |x| 2^(1023 - ex) as a float (x's top 24 bits)
__device__ __forceinline__ float fx_rel(u64 bits, int ex) {
  const int d = ex - ex_of(bits);
  return d > 100 ? 0.0f : __uint_as_float(((unsigned)(127 - d) << 23) | ((unsigned)(bits >> 29) & 0x7fffffu));
}
// Columns outside these exponents are left to the FP64 form.
__device__ __forceinline__ bool fx_in_range(int ex) { return ex < 1023 + 400 && ex > 1023 - 400; }
// And so are channels whose last rows (M - 1 .. N - 1, from which R's last row
// comes) are below 2^-kFxGraded of the largest: a column's one scale leaves an
// entry 2^-k of its norm 58 - k bits, and Householder reflections in FP64 keep
// small rows' relative accuracy where they come last (pre-whitened antennas,
// strongest first).  Row-wise error of R, 8x8, rows graded evenly down to 2^-T, T =
// 4 / 6 / 8 / 10 / 20: fixed 0.9e-16 / 3.3e-16 / 0.9e-15 / 3.1e-15 / 3.4e-12, FP64 0.7e-15 to
// 1.4e-15 (2x2: equal at T = 6).  In any other order of the rows FP64 loses as many
// digits and is behind (T = 10, shuffled: 3.1e-15 and 3.6e-14).
constexpr int kFxGraded = 6;
template <int L>
__device__ __forceinline__ i64 lanes_sum(i64 v) {
#pragma unroll
  for (int o = 1; o < L; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// Small systems (n_rx <= 32), column by column in the left-looking order
// (column j receives reflectors 0..j-1, then forms its own), 32 / L matrices
// per warp with L lanes per matrix: lane L m + h holds rows r = L q + h
// (q < SL = ceil(n_rx / L)) of matrix m's current column in registers.  Bound
// by the integer pipes, so SL is a template parameter (no instruction for
// rows that do not exist) and the loop over the reflectors is cut at
// multiples of L, each piece compiled for the rows its reflectors still touch
// (half of them on average); after a piece the rows it finished are written
// out.  The reflectors' limbs live in shared memory, entry-major with the
// warp's matrices innermost (consecutive lanes read consecutive 16-byte
// entries); the phases of R's rows stay in the registers of the lanes owning
// them.
__host__ __device__ inline size_t qs_smem(int N, int M, int lanes) {
  return sizeof(int4) * (32 / lanes) * (size_t)qs_vo(M, N);
}

template <int L, int SL, int Q0>
__device__ __forceinline__ void qs_apply(i64 (&ar)[SL], i64 (&ai)[SL], const int4* u, int k, int N, int h) {
  static_assert(SL <= kFxEntries, "the accumulators' range");
  constexpr int stride = 32 / L;
  int4 uu[SL];
  FxDot d;
#pragma unroll
  for (int q = Q0; q < SL; ++q) {
    const int r = L * q + h;
    const bool in = (q > Q0 || r >= k) && r < N;
    uu[q] = in ? u[r * stride] : make_int4(0, 0, 0, 0);
    d.add(uu[q], ar[q], ai[q]);
  }
  const i64 wr = lanes_sum<L>(d.re()), wi = lanes_sum<L>(d.im());
  const FxMul w(wr, wi);
#pragma unroll
  for (int q = Q0; q < SL; ++q) fx_axpy(uu[q], w, ar[q], ai[q]);
}

// Reflectors L Q0 .. kend - 1 on column j (kend = j, or M for the y column
// j = M), in pieces of L; a finished piece's rows (and at the end those of the
// last, cut piece) are row entries of R or ybar and go out.
template <int L, int SL, int Q0>
struct QsSweep {
  static __device__ __forceinline__ void run(i64 (&ar)[SL], i64 (&ai)[SL], const int4 (&ph)[SL], const int4* U,
                                             int j, int N, int M, int e, bool act, int h, const QrDst& out) {
    constexpr int mats = 32 / L;
    const int k1 = min(j, L * (Q0 + 1));
    for (int k = L * Q0; k < k1; ++k)
      qs_apply<L, SL, Q0>(ar, ai, U + (qs_vo(k, N) - k) * mats, k, N, h);
    const int r = L * Q0 + h;
    if (act && r < j) {
      u64 re, im;
      fx_unphase(ar[Q0], ai[Q0], ph[Q0], e, re, im);
      if (j < M)
        put_r(out, 2 * M, r, j, re, im);
      else
        put_y(out, r, re, im);
    }
    if (j > L * (Q0 + 1)) QsSweep<L, SL, Q0 + 1>::run(ar, ai, ph, U, j, N, M, e, act, h, out);
  }
};
template <int L, int SL>
struct QsSweep<L, SL, SL> {
  static __device__ __forceinline__ void run(i64 (&)[SL], i64 (&)[SL], const int4 (&)[SL], const int4*, int, int, int,
                                             int, bool, int, const QrDst&) {}
};

// The matrix [H | y] to factor: entry (row r, column j), y being column M.
struct SrcH {  // row-major channel and received vector
  const longlong2* H;
  const longlong2* y;
  int M;
  __device__ __forceinline__ longlong2 operator()(int r, int j) const {
    return j < M ? H[(size_t)r * M + j] : y[r];
  }
};
struct SrcR {  // a factored R (real interleaved, column-packed) with its antennas permuted, and ybar
  const i64* R;
  const i64* y;
  const uint8_t* perm;
  int M;
  __device__ __forceinline__ longlong2 operator()(int r, int j) const {
    if (j == M) return make_longlong2(y[2 * r], y[2 * r + 1]);
    const int c = perm[j];
    const i64* at = R + col_off(2 * c) + 2 * r;
    return make_longlong2(r <= c ? at[0] : 0, r < c ? at[1] : 0);
  }
  __device__ void restore(const QrDst& out, int t0, int step) const {
    for (int t = t0; t < tri(2 * M); t += step) out.R32[t] = f32_of((u64)R[t]);
    for (int t = t0; t < 2 * M; t += step) out.yb32[t] = f32_of((u64)y[t]);
  }
};

struct SrcAug {  // [R; sigma I] and [ybar; 0] of a factored R: the regularised least squares of MMSE
  const i64* R;
  const i64* y;
  i64 sigma;
  int M;
  __device__ __forceinline__ longlong2 operator()(int r, int j) const {
    if (r >= M) return make_longlong2(r - M == j ? sigma : 0, 0);
    if (j == M) return make_longlong2(y[2 * r], y[2 * r + 1]);
    const i64* at = R + col_off(2 * j) + 2 * r;
    return make_longlong2(r <= j ? at[0] : 0, r < j ? at[1] : 0);
  }
};

// Whether the last rows are far below the first one (see kFxGraded).
__device__ __forceinline__ int entry_ex(const SrcH& src, int r, int c) {
  const longlong2 z = src(r, c);
  return max(ex_of((u64)z.x), ex_of((u64)z.y));
}
// Largest exponent of the rows from M - 1 on (lane h's of G), or one close enough to high.
__device__ __forceinline__ int last_rows_ex(const SrcH& src, int N, int high, int h, int G) {
  int low = 0;
  for (int e = h; e < (N - src.M + 1) * src.M && high - low >= kFxGraded; e += G)
    low = max(low, entry_ex(src, src.M - 1 + e / src.M, e % src.M));
  return low;
}

// A matrix left to the FP64 form is marked by -1 in its singular flag or,
// without one (mdx_qr), in the entry of the dense R below its first diagonal
// entry (zero in every finished R).
constexpr i64 kRedo = 1;
__device__ __forceinline__ void mark_redo(const QrDst& out, int n, bool bad) {
  if (out.singular)
    *out.singular = bad ? -1 : 0;
  else if (bad)
    reinterpret_cast<i64*>(out.Rdense)[n] = kRedo;
}
__device__ __forceinline__ bool is_redo(const QrDst& out, int n) {
  return out.singular ? *out.singular == -1 : reinterpret_cast<const i64*>(out.Rdense)[n] == kRedo;
}

// Factorises the matrix of this lane group (act: the group has one), or marks
// it for the FP64 form.  Every lane of the warp calls this
// with the same N, M (shuffles inside).
template <int L, int SL, typename Src>
__device__ void qr_small_pair(int N, int M, bool act, const Src& src, const QrDst& out, int4* U) {
  constexpr int mats = 32 / L;
  const int lane = threadIdx.x & 31, m = lane / L, h = lane % L;
  const int n = 2 * M;
  i64 ar[SL], ai[SL];
  int4 ph[SL];
#pragma unroll
  for (int q = 0; q < SL; ++q) ph[q] = make_int4(0, 0, 0, 0);
  U += m;
  bool bad = false;
  for (int j = 0; j <= M; ++j) {
    int ex = 0;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      const int r = L * q + h;
      longlong2 z = make_longlong2(0, 0);
      if (act && r < N) z = src(r, j);
      ar[q] = z.x;
      ai[q] = z.y;
      ex = max(ex, max(ex_of((u64)z.x), ex_of((u64)z.y)));
    }
#pragma unroll
    for (int o = 1; o < L; o <<= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
    float ss = 0.0f;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      const float fr = fx_rel((u64)ar[q], ex), fi = fx_rel((u64)ai[q], ex);
      ss = fmaf(fr, fr, fmaf(fi, fi, ss));
    }
#pragma unroll
    for (int o = 1; o < L; o <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    // an all-zero y is fine (any scale); an all-zero column of H is singular and caught below
    bad = bad || (ex != 0 && !fx_in_range(ex));
    const int e = fx_in_range(ex) ? fx_scale(ex, ss) : 0;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      ar[q] = fx_in_range(ex) ? fx_from((u64)ar[q], e) : 0;
      ai[q] = fx_in_range(ex) ? fx_from((u64)ai[q], e) : 0;
    }
    QsSweep<L, SL, 0>::run(ar, ai, ph, U, j, N, M, e, act && !bad, h, out);
    if (j < M) {
      // reflector j from rows j..N-1
      FxNorm s;
      i64 x0r = 0, x0i = 0;
#pragma unroll
      for (int q = 0; q < SL; ++q) {
        const bool in = L * q + h >= j && L * q + h < N;
        s.add(in ? ar[q] : 0);
        s.add(in ? ai[q] : 0);
        if (L * q + h == j) {
          x0r = ar[q];
          x0i = ai[q];
        }
      }
      const i64 hh = lanes_sum<L>(s.hh), md = lanes_sum<L>(s.md);
      const u64 ll = (u64)lanes_sum<L>((i64)(s.ll >> 3));
      const int h0 = (lane & ~(L - 1)) | (j % L);
      x0r = __shfl_sync(0xffffffffu, x0r, h0);
      x0i = __shfl_sync(0xffffffffu, x0i, h0);
      FxReflector f;
      f.s = 0;
      if (!fx_reflector(hh, md, ll, x0r, x0i, f)) bad = true;
      int4* uj = U + (qs_vo(j, N) - j) * mats;
#pragma unroll
      for (int q = 0; q < SL; ++q) {
        const int r = L * q + h;
        const bool first = r == j;
        if (r >= j && r < N)
          uj[r * mats] = bad ? make_int4(0, 0, 0, 0)
                             : fx_split(first ? f.ur : f.scale(ar[q]), first ? f.ui : f.scale(ai[q]));
        if (first) ph[q] = fx_split(-f.pr, -f.pi);
      }
      if (act && !bad && lane == h0) put_r(out, n, j, j, fx_to_bits((i64)f.sigma, e + f.s - 4), 0);
    }
    __syncwarp();
  }
  if (act) {
    if (out.Rdense)
      for (int t = h; t < n * n; t += L)
        if (t / n > t % n) out.Rdense[t] = 0.0;
  }
  __syncwarp();
  if (act && out.pk) {
    if (h == 0) *out.pk_bad = bad ? 1 : 0;
  } else if (act && out.sorted) {
    if constexpr (std::is_same<Src, SrcR>::value) {
      if (bad) src.restore(out, h, L);
    }
    if (bad && h == 0) *out.sorted = 0;
  } else if (act && h == 0) {
    mark_redo(out, n, bad);
  }
}

// Outputs of matrix b of a uniform batch (stride the library's per-vector layout).
__device__ __forceinline__ QrDst batch_dst(const QrOut& out, int b, int n) {
  QrDst d;
  d.R64 = out.R64 ? out.R64 + (size_t)b * tri_stride64(n) : nullptr;
  d.yb64 = out.yb64 ? out.yb64 + (size_t)b * vec_stride64(n) : nullptr;
  d.R32 = out.R32 ? out.R32 + (size_t)b * tri_stride32(n) : nullptr;
  d.yb32 = out.yb32 ? out.yb32 + (size_t)b * vec_stride32(n) : nullptr;
  d.Rdense = out.Rdense ? out.Rdense + (size_t)b * n * n : nullptr;
  d.ybdense = out.ybdense ? out.ybdense + (size_t)b * n : nullptr;
  d.singular = out.singular ? out.singular + b : nullptr;
  return d;
}
// One matrix of a launch: input, output, shape.  A uniform batch has ids =
// null; an uneven one lists its requests (all of one shape) in ids.
struct QrBatch {
  int count, N, M, num_sms;
  const int* ids;
  const MixedReq* reqs;
  const double* H;
  const double* y;
  QrOut out;
  __device__ __forceinline__ QrDst get(int i, const double*& Hb, const double*& yb) const {
    if (ids) {
      const int r = ids[i];
      const MixedReq& q = reqs[r];
      Hb = H + q.h_off;
      yb = y + q.yin_off;
      return QrDst{out.R64 + q.r_off64, out.yb64 + q.y_off64, out.R32 + q.r_off, out.yb32 + q.y_off,
                   nullptr,             nullptr,              out.singular + r};
    }
    Hb = H + (size_t)i * 2 * N * M;
    yb = y + (size_t)i * 2 * N;
    return batch_dst(out, i, 2 * M);
  }
};

template <int L, int SL>
__global__ void __launch_bounds__(32) qr_small_kernel(QrBatch g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i = blockIdx.x * (32 / L) + (threadIdx.x & 31) / L;
  const bool act = i < g.count;
  const double *Hb, *yb;
  const QrDst d = g.get(act ? i : 0, Hb, yb);
  const SrcH src{reinterpret_cast<const longlong2*>(Hb), reinterpret_cast<const longlong2*>(yb), g.M};
  qr_small_pair<L, SL>(g.N, g.M, act, src, d, reinterpret_cast<int4*>(smem_raw));
}

// The chosen vectors' R with their antennas in search order (see sd_reorder.cu).
__device__ __forceinline__ QrDst reorder_at(const ReorderArgs& g, int i, SrcR& src) {
  const int v = g.list[i], n = g.a.n, M = g.a.n_tx;
  src = SrcR{reinterpret_cast<const i64*>(g.a.R64 + (size_t)v * tri_stride64(n)),
             reinterpret_cast<const i64*>(g.a.yb64 + (size_t)v * vec_stride64(n)), g.perm + (size_t)v * M, M};
  QrDst d{};
  d.R32 = const_cast<float*>(g.a.R32) + (size_t)v * tri_stride32(n);
  d.yb32 = const_cast<float*>(g.a.yb32) + (size_t)v * vec_stride32(n);
  d.sorted = g.sorted + v;
  return d;
}
template <int L, int SL>
__global__ void __launch_bounds__(32) qr_reorder_small_kernel(ReorderArgs g, int few) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int count = (int)*g.count, i0 = blockIdx.x * (32 / L);
  if (count <= few || i0 >= count) return;
  const int i = i0 + (threadIdx.x & 31) / L;
  const bool act = i < count;
  SrcR src;
  const QrDst d = reorder_at(g, act ? i : i0, src);
  qr_small_pair<L, SL>(g.a.n_tx, g.a.n_tx, act, src, d, reinterpret_cast<int4*>(smem_raw));
}

// Whether matrix i was left to FP64, or has to be: last rows far below the first
// one, or a y of subnormal numbers, whose ybar is all zeros.  By a lane, which looks
// closer where two entries of each row or the first of ybar give reason to (all of
// them loaded at once); here so that qr_small_kernel keeps its registers.
__device__ __forceinline__ bool left_to_fp64(const QrBatch& g, int i) {
  const double *Hb, *yb;
  const QrDst d = g.get(i, Hb, yb);
  const SrcH src{reinterpret_cast<const longlong2*>(Hb), reinterpret_cast<const longlong2*>(yb), g.M};
  const int c = g.M > 1 ? 1 : 0;
  const int high = max(entry_ex(src, 0, 0), entry_ex(src, 0, c));
  const int low = max(entry_ex(src, g.M - 1, 0), entry_ex(src, g.M - 1, c));
  const double* y0 = d.yb64 ? d.yb64 : d.ybdense;  // (aligned to a double)
  const double yr = y0[0], yi = y0[1];
  const bool marked = is_redo(d, 2 * g.M), none = yr == 0.0 && yi == 0.0;
  if (!marked && !none && high - low < kFxGraded) return false;
  if (marked || high - last_rows_ex(src, g.N, high, 0, 1) >= kFxGraded) return true;
  bool some = false;
  for (int r = 0; none && r < 2 * g.N; ++r) some = some || yb[r] != 0.0;
  return some;
}

// The matrices that the fixed-point forms left, in FP64: n_rx <= 32, 32 / L of
// them per warp.  A warp looks through `per` matrices of the batch and factors
// the marked ones as it finds them, a warp full at a time: a batch of nothing but
// such matrices (keyhole or line-of-sight channels, copied columns) keeps the GPU
// as full as one kernel for all of them would.  Whole calls, a column twice in
// every matrix, us (128 matrices to a CTA, one after another, before / now; in
// brackets 1 % of them so): 10,000 of 16x16 52,117 / 726 (2,284 / 616), 100,000
// 157,397 / 5,305, 10,000 of 32x32 185,917 / 5,518; 1,000 of 64x64 130,993 / 3,283,
// of 100x100 346,849 / 11,686 (10,781 / 5,238).
template <int L>
__global__ void __launch_bounds__(32) qr_redo_small_kernel(QrBatch g, int per) {
  constexpr int mats = 32 / L;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int list[mats + 32];
  double2* V = reinterpret_cast<double2*>(smem_raw);
  double* Tau = reinterpret_cast<double*>(V + (size_t)mats * qs_vo(g.M, g.N));
  const int lane = threadIdx.x & 31, end = min(g.count, ((int)blockIdx.x + 1) * per);
  int base = blockIdx.x * per, have = 0;
  const double *Hb, *yb;
  for (;;) {
    for (; have < mats && base < end; base += 32) {
      const int i = base + lane;
      const bool mine = i < end && left_to_fp64(g, i);
      const unsigned who = __ballot_sync(0xffffffffu, mine);
      if (mine) list[have + __popc(who & ((1u << lane) - 1u))] = i;
      have += __popc(who);
    }
    if (have == 0) return;
    __syncwarp();
    const bool act = lane / L < have;
    const QrDst d = g.get(list[act ? lane / L : 0], Hb, yb);
    qr_small64<L, mats>(g.N, g.M, act, reinterpret_cast<const double2*>(Hb), reinterpret_cast<const double2*>(yb), d, V,
                        Tau);
    have = max(have - mats, 0);
    const int next = lane < have ? list[mats + lane] : 0;
    __syncwarp();
    if (lane < have) list[lane] = next;
    __syncwarp();
  }
}
// n_rx > 32: a CTA each, CTA b the marked ones among matrices b, b + grid, ...
// LPC lanes per column: 32 below 48 antennas; above, where a reduction over 32
// lanes would be half of a column's FP64 instructions, 8.
template <int LPC>
__global__ void __launch_bounds__(256) qr_redo_kernel(QrBatch g) {
  __shared__ unsigned marks[8];
  const double *Hb, *yb;
  for (int base = blockIdx.x; base < g.count; base += gridDim.x * 256) {
    const int i = base + threadIdx.x * gridDim.x;
    const unsigned who = __ballot_sync(0xffffffffu, i < g.count && left_to_fp64(g, i));
    if ((threadIdx.x & 31) == 0) marks[threadIdx.x >> 5] = who;
    __syncthreads();
    for (int w = 0; w < 8; ++w)
      for (unsigned left = marks[w]; left; left &= left - 1) {
        const QrDst d = g.get(base + (32 * w + __ffs(left) - 1) * gridDim.x, Hb, yb);
        qr_one<LPC>(g.N, g.M, reinterpret_cast<const double2*>(Hb), reinterpret_cast<const double2*>(yb), d);
        __syncthreads();
      }
    __syncthreads();  // the marks are read
  }
}

// ---------------------------------------------------------------------------
// One CTA per matrix, left-looking in a pipeline of warps.  A warp takes groups
// of 32 / L columns in ascending order (L lanes per column, rows L q + h of
// lane h in registers, y the last column), applies the reflectors of the
// groups before as they appear, then forms its own.  A reflector is published
// in shared memory under an mbarrier, so no warp waits for more than it reads:
// while one warp is on the chain (apply, norm, scalars of the next reflector),
// the others catch up on earlier ones.  Only the reflectors are in shared
// memory (a triangle of 16-byte limb entries, half of the matrix).  The loop
// over reflectors is compiled for the rows still touched in steps of 16.
//
// Bound by instruction issue (the multiply-add pipe 62-69 % busy on many
// matrices) and, for few matrices, by the chain.  Against the matrix in shared
// memory, right-looking, with one CTA barrier per column (us, before / now):
// one matrix 16x16 41 / 28, 32x32 78 / 58, 64x64 190 / 165; 608 matrices 32x32
// 176 / 92; 2,432 matrices 48x48 883 / 845, 64x64 1,673 / 1,609, 100x100
// 6,101 / 5,895.

struct QrCtaLayout {
  size_t off_ph, off_bar, off_flag, bytes;
  __host__ __device__ void init(int N, int M) {
    size_t o = sizeof(int4) * (size_t)qs_vo(M, N);
    off_ph = o;
    o += sizeof(int4) * (size_t)M;
    off_bar = o;
    o += sizeof(u64) * (size_t)M;
    off_flag = o;
    o += 16;
    bytes = o;
  }
};

__device__ __forceinline__ unsigned smem_at(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// Waits until the barrier's first phase is complete; false after a bounded
// number of tries.
__device__ __forceinline__ bool wait_published(const u64* bar) {
  for (int it = 0; it < (1 << 20); ++it) {
    unsigned done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(smem_at(bar))
        : "memory");
    if (done) return true;
  }
  return false;
}

// Slots per piece of the loop over reflectors: 16 rows, or a slot.
template <int L>
constexpr int qc_step = L < 16 ? 16 / L : 1;

// Reflector k (entries from row k on at u + r) on the rows L Q0 .. of the
// lanes' columns; masked: also rows above k among the piece's first slots.
template <int L, int SL, int Q0>
__device__ __forceinline__ void qc_apply(i64 (&ar)[SL], i64 (&ai)[SL], const int4* u, int k, int N, int h, bool act) {
  static_assert(SL <= kFxEntries, "the accumulators' range");
  FxDot d;
#pragma unroll
  for (int q = Q0; q < SL; ++q) {
    const int r = L * q + h;
    const bool in = (q >= Q0 + qc_step<L> || r >= k) && r < N;
    const int4 uu = in ? u[r] : make_int4(0, 0, 0, 0);
    d.add(uu, ar[q], ai[q]);
  }
  const i64 wr = lanes_sum<L>(d.re()), wi = lanes_sum<L>(d.im());
  const FxMul w(act ? wr : 0, act ? wi : 0);  // (0 leaves a column as it is)
#pragma unroll
  for (int q = Q0; q < SL; ++q) {
    const int r = L * q + h;
    const bool in = (q >= Q0 + qc_step<L> || r >= k) && r < N;
    const int4 uu = in ? u[r] : make_int4(0, 0, 0, 0);
    fx_axpy(uu, w, ar[q], ai[q]);
  }
}
template <int L, int SL, int Q0>
struct QcApply {  // one reflector, by the piece of k
  static __device__ __forceinline__ void run(i64 (&ar)[SL], i64 (&ai)[SL], const int4* u, int k, int N, int h,
                                             bool act) {
    if (k < L * (Q0 + qc_step<L>) || Q0 + qc_step<L> >= SL)
      qc_apply<L, SL, Q0>(ar, ai, u, k, N, h, act);
    else if constexpr (Q0 + qc_step<L> < SL)
      QcApply<L, SL, Q0 + qc_step<L>>::run(ar, ai, u, k, N, h, act);
  }
};

// Factorises the matrix with the calling CTA; false if it needs the FP64 form
// (the outputs are then unfinished).  rows: for last rows far below the first as
// well (warp 0 looks when it is done; the last columns are with other warps).
template <int L, int SL, typename Src>
__device__ bool qr_cta_one(int N, int M, const Src& src, const QrDst& out, bool rows) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int kCols = 32 / L;  // columns of a group
  QrCtaLayout lay;
  lay.init(N, M);
  int4* U = reinterpret_cast<int4*>(smem_raw);
  int4* ph = reinterpret_cast<int4*>(smem_raw + lay.off_ph);
  u64* bar = reinterpret_cast<u64*>(smem_raw + lay.off_bar);
  volatile int* flag = reinterpret_cast<volatile int*>(smem_raw + lay.off_flag);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int h = lane % L, sub = lane / L, n = 2 * M;
  if (tid == 0) *flag = 0;
  for (int k = tid; k < M; k += blockDim.x)
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_at(bar + k)) : "memory");
  __syncthreads();
  int avail = 0;  // reflectors known to be published
  for (int c0 = kCols * warp; c0 <= M; c0 += kCols * nw) {
    const int c = c0 + sub;
    const bool mine = c <= M;
    // ---- the column, at its scale
    i64 ar[SL], ai[SL];
    int ex = 0;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      const int r = L * q + h;
      longlong2 z = make_longlong2(0, 0);
      if (mine && r < N) z = src(r, c);
      ar[q] = z.x;
      ai[q] = z.y;
      ex = max(ex, max(ex_of((u64)z.x), ex_of((u64)z.y)));
    }
#pragma unroll
    for (int o = 1; o < L; o <<= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
    float ss = 0.0f;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      const float fr = fx_rel((u64)ar[q], ex), fi = fx_rel((u64)ai[q], ex);
      ss = fmaf(fr, fr, fmaf(fi, fi, ss));
    }
#pragma unroll
    for (int o = 1; o < L; o <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const bool fine = fx_in_range(ex);
    const int e = fine ? fx_scale(ex, ss) : 0;
    if (ex != 0 && !fine) *flag = 1;
    if (c == M && ex == 0) {  // y of subnormal numbers
      i64 bits = 0;
#pragma unroll
      for (int q = 0; q < SL; ++q) bits |= ar[q] << 1 | ai[q] << 1;
      if (bits) *flag = 1;
    }
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      ar[q] = fine ? fx_from((u64)ar[q], e) : 0;
      ai[q] = fine ? fx_from((u64)ai[q], e) : 0;
    }
    // ---- the reflectors of the groups before
    for (int k = 0; k < c0; ++k) {
      if (k >= avail) {
        if (!wait_published(bar + k)) *flag = 1;
        avail = k + 1;
      }
      QcApply<L, SL, 0>::run(ar, ai, U + qs_vo(k, N) - k, k, N, h, true);
    }
    // ---- the group's own
    u64 sigma = 0;
    int sexp = 0;
    for (int t = 0; t < kCols && c0 + t < M; ++t) {
      const int k = c0 + t;
      FxNorm s;
      i64 x0r = 0, x0i = 0;
#pragma unroll
      for (int q = 0; q < SL; ++q) {
        const int r = L * q + h;
        const bool in = r >= k && r < N;
        s.add(in ? ar[q] : 0);
        s.add(in ? ai[q] : 0);
        if (r == k) {
          x0r = ar[q];
          x0i = ai[q];
        }
      }
      const i64 hh = lanes_sum<L>(s.hh), md = lanes_sum<L>(s.md);
      const u64 ll = (u64)lanes_sum<L>((i64)(s.ll >> 3));
      const int h0 = (lane & ~(L - 1)) | (k % L);
      x0r = __shfl_sync(0xffffffffu, x0r, h0);
      x0i = __shfl_sync(0xffffffffu, x0i, h0);
      FxReflector f;
      const bool ok = fx_reflector(hh, md, ll, x0r, x0i, f);
      int4* u = U + qs_vo(k, N) - k;
      if (sub == t) {
#pragma unroll
        for (int q = 0; q < SL; ++q) {
          const int r = L * q + h;
          if (r >= k && r < N)
            u[r] = !ok ? make_int4(0, 0, 0, 0)
                       : r == k ? fx_split(f.ur, f.ui) : fx_split(f.scale(ar[q]), f.scale(ai[q]));
        }
        if (h == 0) {
          if (!ok) *flag = 1;
          ph[k] = fx_split(-f.pr, -f.pi);
        }
        sigma = f.sigma;
        sexp = f.s;
      }
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_at(bar + k)) : "memory");
      if (t < kCols - 1) QcApply<L, SL, 0>::run(ar, ai, u, k, N, h, sub > t);
    }
    avail = max(avail, min(c0 + kCols, M));
    // ---- out: rows above the diagonal (all their phases are published), the diagonal
    if (mine) {
#pragma unroll
      for (int q = 0; q < SL; ++q) {
        const int r = L * q + h;
        if (r < min(c, M)) {
          u64 re, im;
          fx_unphase(ar[q], ai[q], ph[r], e, re, im);
          if (c < M)
            put_r(out, n, r, c, re, im);
          else
            put_y(out, r, re, im);
        }
      }
      if (c < M && h == 0) put_r(out, n, c, c, fx_to_bits((i64)sigma, e + sexp - 4), 0);
    }
  }
  if constexpr (std::is_same<Src, SrcH>::value) {
    if (rows && warp == 0) {
      const int c = lane % M, high = __reduce_max_sync(0xffffffffu, entry_ex(src, 0, c));
      if (high - __reduce_max_sync(0xffffffffu, entry_ex(src, M - 1, c)) >= kFxGraded &&
          high - __reduce_max_sync(0xffffffffu, last_rows_ex(src, N, high, lane, 32)) >= kFxGraded)
        *flag = 1;
    }
  }
  __syncthreads();
  // (the barriers end here: the FP64 form takes this memory for other things)
  for (int k = tid; k < M; k += blockDim.x)
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_at(bar + k)) : "memory");
  if (*flag) return false;
  if (out.Rdense)
    for (int t = tid; t < n * n; t += blockDim.x)
      if (t / n > t % n) out.Rdense[t] = 0.0;
  return true;
}

template <int L, int SL, int T, int B>
__global__ void __launch_bounds__(T, B) qr_cta_kernel(QrBatch g, int here) {
  const double *Hb, *yb;
  const QrDst d = g.get(blockIdx.x, Hb, yb);
  const SrcH src{reinterpret_cast<const longlong2*>(Hb), reinterpret_cast<const longlong2*>(yb), g.M};
  const bool ok = qr_cta_one<L, SL>(g.N, g.M, src, d, here);
  __syncthreads();  // the zeroed triangle, before the mark in it; the shared memory, before the FP64 form
  if (!ok && here)
    qr_small64_one(g.N, g.M, Hb, yb, d);
  else if (threadIdx.x == 0)
    mark_redo(d, 2 * g.M, !ok);
}
template <int L, int SL>
__global__ void __launch_bounds__(288, 2) qr_reorder_cta_kernel(ReorderArgs g, int few) {
  const int count = (int)*g.count;
  if (count > few || (int)blockIdx.x >= count) return;
  SrcR src;
  const QrDst d = reorder_at(g, blockIdx.x, src);
  if (!qr_cta_one<L, SL>(g.a.n_tx, g.a.n_tx, src, d, false)) {
    __syncthreads();
    if (threadIdx.x == 0) *d.sorted = 0;
    src.restore(d, threadIdx.x, blockDim.x);
  }
}

// The augmented systems of a batch (2 M x M, see linear.cu).
__device__ __forceinline__ QrDst aug_at(const AugArgs& g, int v, SrcAug& src) {
  const int n = g.a.n, M = g.a.n_tx;
  src = SrcAug{reinterpret_cast<const i64*>(g.a.R64 + (size_t)v * tri_stride64(n)),
               reinterpret_cast<const i64*>(g.a.yb64 + (size_t)v * vec_stride64(n)),
               __double_as_longlong(sqrt(g.a.noise_var[v])), M};
  QrDst d{};
  d.pk = reinterpret_cast<longlong2*>(g.R(v));
  d.pk_diag = reinterpret_cast<i64*>(g.diag(v));
  d.pk_y = reinterpret_cast<longlong2*>(g.y(v));
  d.pk_bad = g.bad + v;
  return d;
}
template <int L, int SL>
__global__ void __launch_bounds__(32) qr_aug_small_kernel(AugArgs g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i = blockIdx.x * (32 / L) + (threadIdx.x & 31) / L;
  const bool act = i < g.a.batch;
  SrcAug src;
  const QrDst d = aug_at(g, act ? i : 0, src);
  qr_small_pair<L, SL>(2 * g.a.n_tx, g.a.n_tx, act, src, d, reinterpret_cast<int4*>(smem_raw));
}
template <int L, int SL>
__global__ void __launch_bounds__(288, 2) qr_aug_cta_kernel(AugArgs g) {
  SrcAug src;
  const QrDst d = aug_at(g, blockIdx.x, src);
  const bool ok = qr_cta_one<L, SL>(2 * g.a.n_tx, g.a.n_tx, src, d, false);
  if (threadIdx.x == 0) *d.pk_bad = ok ? 0 : 1;
}

size_t qr_cta_smem(int n_rx, int n_tx) {
  QrCtaLayout L;
  L.init(n_rx, n_tx);
  return n_rx <= 32 ? std::max(L.bytes, qs64_smem(n_rx, n_tx, 1)) : L.bytes;
}

// CTAs an SM's shared memory holds (a kilobyte each is the system's).
int smem_ctas(size_t bytes, int most) { return std::max(1, std::min(most, (int)(228 * 1024 / (bytes + 1024)))); }

template <int L>
cudaError_t launch_redo_small(const QrBatch& g, cudaStream_t s) {
  constexpr int mats = 32 / L;
  const size_t sm = qs64_smem(g.N, g.M, mats);
  const int warps = (g.count + mats - 1) / mats, most = g.num_sms * smem_ctas(sm + 256, 32);
  const int turns = (warps + most - 1) / most;
  cudaFuncSetAttribute(qr_redo_small_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  qr_redo_small_kernel<L><<<(warps + turns - 1) / turns, 32, sm, s>>>(g, turns * mats);
  return cudaGetLastError();
}
template <int LPC>
cudaError_t launch_redo_large(const QrBatch& g, cudaStream_t s) {
  const size_t sm = qr_one_smem(g.N, g.M);
  cudaFuncSetAttribute(qr_redo_kernel<LPC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  qr_redo_kernel<LPC><<<std::min(g.count, g.num_sms * smem_ctas(sm + 32, 4)), 256, sm, s>>>(g);
  return cudaGetLastError();
}
cudaError_t launch_redo(const QrBatch& g, cudaStream_t s) {
  if (g.N <= 32) return qs64_lanes(g.N) == 2 ? launch_redo_small<2>(g, s) : launch_redo_small<4>(g, s);
  return g.M < 48 ? launch_redo_large<32>(g, s) : launch_redo_large<8>(g, s);
}

template <int L, int SL>
cudaError_t launch_qs(const QrBatch& g, cudaStream_t s) {
  const size_t sm = qs_smem(g.N, g.M, L);
  cudaFuncSetAttribute(qr_small_kernel<L, SL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  qr_small_kernel<L, SL><<<(g.count + 32 / L - 1) / (32 / L), 32, sm, s>>>(g);
  return launch_redo(g, s);
}
// Threads of a CTA: a warp per 32 / L columns of [H | y], at most `most`.
int qc_threads(int L, int M, int most) { return 32 * std::min(M / (32 / L) + 1, most); }

template <int L, int SL, int T, int B>
cudaError_t launch_qc(const QrBatch& g, int most, cudaStream_t s) {
  const size_t sm = qr_cta_smem(g.N, g.M);
  cudaFuncSetAttribute(qr_cta_kernel<L, SL, T, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  // A small matrix left to FP64 is factored by its own CTA, which spares a launch
  // (5 us of 90 for 1,216 of 16x16): up to a matrix per scheduler that takes no
  // longer; for the few more of n_rx <= 16 that come here (all dependent, 1,216: 951
  // us, 480 by the launch) the ordinary call counts, above (1,824 of 32x32: 5.1 ms,
  // 1.7 by the launch) the others.
  const bool here = g.N <= 16 || (g.N <= 32 && g.count <= 4 * g.num_sms);
  qr_cta_kernel<L, SL, T, B><<<g.count, qc_threads(L, g.M, most), sm, s>>>(g, here);
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess || here ? e : launch_redo(g, s);
}

// Lanes per matrix of qr_small_kernel, or 0: qr_cta_kernel.  A warp of the
// small kernel takes as long for one matrix as for 32 / L, so few matrices go
// to a CTA each, and more lanes per matrix serve a half-empty GPU better than
// a full one, where the lanes' shared work (reflector scalars, reductions)
// counts.  Measured, us a call with 28 us of host time (CTA / 2 / 4 / 8 lanes):
//   16x16:  1,216 matrices 64 / 207 / 136 / 91, 9,728: - / 223 / 166 / 168,
//          38,912: - / 767 / 586 / 583
//   12x12:  9,728: 386 / 130 / 115 / 115, 38,912: 1,514 / 441 / 367 / 397
//    8x8:   1,216: 35 / 55 / 41 / 41, 9,728: 205 / 58 / 49 / 68,
//          38,912: 769 / 113 / 129 / 217
//   24x24:  1,216: 131 / - / 314 / 234, 4,864: 515 / - / 336 / 301,
//          38,912: 3,883 / - / 2,410 / 2,538
//   32x32:  2,432: 445 / - / 567 / 377, 9,728: 1,667 / - / 1,655 / 1,213
// (The lines in matrices per SM, of which this GPU has 152.)
int few_matrices(int n_rx, int num_sms) { return (n_rx <= 16 ? 8 : 12) * num_sms; }
int qr_form(int count, int n_rx, int num_sms) {
  if (n_rx > 32 || count <= few_matrices(n_rx, num_sms)) return 0;
  if (n_rx <= 4) return 2;
  if (n_rx <= 8) return count <= 108 * num_sms ? 4 : 2;
  if (n_rx <= 12) return count <= 64 * num_sms ? 8 : 4;
  if (n_rx > 16 && n_rx <= 24) return count <= 32 * num_sms ? 8 : 4;
  return 8;
}

template <int L, int SL>
cudaError_t launch_as(const AugArgs& g, cudaStream_t s) {
  const size_t sm = qs_smem(2 * g.a.n_tx, g.a.n_tx, L);
  cudaFuncSetAttribute(qr_aug_small_kernel<L, SL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  qr_aug_small_kernel<L, SL><<<(g.a.batch + 32 / L - 1) / (32 / L), 32, sm, s>>>(g);
  return cudaGetLastError();
}

template <int L, int SL>
cudaError_t launch_rs(const ReorderArgs& r, int few, cudaStream_t s) {
  const size_t sm = qs_smem(r.a.n_tx, r.a.n_tx, L);
  cudaFuncSetAttribute(qr_reorder_small_kernel<L, SL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  qr_reorder_small_kernel<L, SL><<<(r.a.batch + 32 / L - 1) / (32 / L), 32, sm, s>>>(r, few);
  return cudaGetLastError();
}

cudaError_t launch(const QrBatch& g, cudaStream_t s) {
  if (g.count <= 0) return cudaSuccess;
  const int N = g.N;
  switch (qr_form(g.count, N, g.num_sms)) {
    case 0: {
      // Few matrices: more warps each, for the chain; many: CTAs of fewer warps.
      const int w = g.count <= g.num_sms ? 9 : g.count <= 8 * g.num_sms ? 5 : 3;
      if (N <= 16) return launch_qc<16, 1, 288, 2>(g, std::min(w, 5), s);
      if (N <= 32) return launch_qc<16, 2, 288, 2>(g, w, s);
      if (N <= 48) return launch_qc<16, 3, 256, 3>(g, g.count <= g.num_sms ? 8 : 4, s);
      if (N <= 64) return launch_qc<32, 2, 256, 3>(g, 8, s);
      if (N <= 96) return launch_qc<32, 3, 256, 3>(g, 8, s);
      return launch_qc<32, 4, 384, 2>(g, 12, s);
    }
    case 2:
      if (N <= 4) return launch_qs<2, 2>(g, s);
      return launch_qs<2, 4>(g, s);
    case 4:
      if (N <= 8) return launch_qs<4, 2>(g, s);
      if (N <= 12) return launch_qs<4, 4>(g, s);
      return launch_qs<4, 6>(g, s);
    default:
      if (N <= 16) return launch_qs<8, 2>(g, s);
      return launch_qs<8, 4>(g, s);
  }
}

}  // namespace

// The number of vectors chosen is on the device: the CTA form's grid is for
// up to `few` of them (as in qr_form), the other's for the whole batch, and
// the one that does not apply returns at once.
cudaError_t launch_qr_reorder(const ReorderArgs& r, int num_sms, cudaStream_t s) {
  const int M = r.a.n_tx, few = few_matrices(M, num_sms);
  const size_t sm = qr_cta_smem(M, M);
  const int grid = std::min(r.a.batch, few), threads = qc_threads(8, M, 9);
  if (M <= 16) {
    qr_reorder_cta_kernel<8, 2><<<grid, threads, sm, s>>>(r, few);
  } else {
    qr_reorder_cta_kernel<8, 4><<<grid, threads, sm, s>>>(r, few);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || r.a.batch <= few) return e;
  if (M <= 8) return launch_rs<4, 2>(r, few, s);
  if (M <= 16) return launch_rs<8, 2>(r, few, s);
  if (M <= 24) return launch_rs<4, 6>(r, few, s);
  return launch_rs<8, 4>(r, few, s);
}

cudaError_t launch_qr_augmented(const AugArgs& g, int num_sms, cudaStream_t s) {
  const int M = g.a.n_tx;
  switch (qr_form(g.a.batch, 2 * M, num_sms)) {
    case 0: {
      const size_t sm = qr_cta_smem(2 * M, M);
      if (M <= 8) {
        qr_aug_cta_kernel<8, 2><<<g.a.batch, qc_threads(8, M, 9), sm, s>>>(g);
      } else if (M <= 16) {
        qr_aug_cta_kernel<8, 4><<<g.a.batch, qc_threads(8, M, 9), sm, s>>>(g);
      } else {
        qr_aug_cta_kernel<16, 4><<<g.a.batch, qc_threads(8, M, 9), sm, s>>>(g);
      }
      return cudaGetLastError();
    }
    case 2:
      if (M <= 2) return launch_as<2, 2>(g, s);
      return launch_as<2, 4>(g, s);
    case 4:
      if (M <= 4) return launch_as<4, 2>(g, s);
      if (M <= 8) return launch_as<4, 4>(g, s);
      return launch_as<4, 6>(g, s);
    default:
      if (M <= 8) return launch_as<8, 2>(g, s);
      return launch_as<8, 4>(g, s);
  }
}

cudaError_t launch_qr_gather(int count, int n_rx, int n_tx, const int* ids, const MixedReq* reqs,
                             const double* H, const double* y, QrOut out, int num_sms, cudaStream_t s) {
  return launch(QrBatch{count, n_rx, n_tx, num_sms, ids, reqs, H, y, out}, s);
}

cudaError_t launch_qr(int batch, int n_rx, int n_tx, const double* H, const double* y, QrOut out, int num_sms,
                      cudaStream_t s) {
  return launch(QrBatch{batch, n_rx, n_tx, num_sms, nullptr, nullptr, H, y, out}, s);
}

}  // namespace mdx
