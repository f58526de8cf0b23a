// Tridiagonal eigensolver used by the Lanczos drivers (internal header):
// Sturm-sequence multisection for the k lowest eigenvalues, inverse iteration
// with tridiagonal Gaussian elimination and partial pivoting for their
// vectors, one warp per pair; then Gram-Schmidt among (nearly) equal
// eigenvalues.  All in FP64.
//
// Bound by the latency and the rate of FP64 instructions along the matrix
// (GB300 issues about 1.6 FP64 lanes per SM and clock: 20 cycles per warp
// instruction), so the chains are kept short: the Sturm counts use the
// determinant recurrence (3 FP64 instructions per row and no division), the
// matrix and the factors sit in shared memory, the factor's reciprocals are
// taken by all lanes at once, and a pair's value and vector share one launch.
#pragma once

#include "ed_internal.h"
#include "fp64_short.h"

namespace ed {

constexpr int kTriSmemRows = 1024;   // matrices up to this size run from shared memory (6 doubles per row)

inline size_t tri_smem(int m) {
  return (size_t)6 * (m < 1 ? 1 : m < kTriSmemRows ? m : kTriSmemRows) * sizeof(double);
}

// Block-wide sum, result valid in thread 0.
__device__ inline double tri_block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  int nw = blockDim.x >> 5;
  if (w == 0) {
    v = (lane < nw) ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  __syncthreads();
  return v;
}

__device__ __forceinline__ int tri_exp(double v) { return __double2hiint(v) & 0x7ff00000; }

// 2^(-e) for the binary exponent field e of a normal double
__device__ __forceinline__ double tri_pow2_inv(int field) { return __hiloint2double(0x7fe00000 - field, 0); }

// Sturm count: eigenvalues below x of the matrix with rows ab[i] = (a_i, b_i^2),
// entries of magnitude below 2.  Determinants of the leading minors,
// p_i = (a_i - x) p_{i-1} - b_i^2 p_{i-2}, whose sign changes count the
// negative pivots; a pivot p_i / p_{i-1} below 2^-100 in magnitude counts as
// -2^-100 (a change of a_i far below rounding).  Every eight rows p is brought
// back to about 1 by an exact power of two, so that it cannot leave the range
// of a double (a row shrinks it by at most 2^-100 and multiplies it by less than
// 8: |a - x| < 4, b^2 < 4).
__device__ inline int sturm(const double2* __restrict__ ab, int m, double x) {
  double p0 = 1.0, p1 = ab[0].x - x;
  if (tri_exp(p1) + (100 << 20) < tri_exp(p0)) p1 = -0x1p-100;
  int cnt = p1 < 0.0 ? 1 : 0;
  auto row = [&](const double2 r) {
    double p = fma(r.x - x, p1, -(r.y * p0));
    if (tri_exp(p) + (100 << 20) < tri_exp(p1)) p = -p1 * 0x1p-100;
    cnt += (unsigned)(__double2hiint(p) ^ __double2hiint(p1)) >> 31;
    p0 = p1;
    p1 = p;
  };
  int i = 1;
  for (; i + 8 <= m; i += 8) {
#pragma unroll
    for (int q = 0; q < 8; ++q) row(ab[i + q]);
    const double sc = tri_pow2_inv(max(tri_exp(p0), tri_exp(p1)));
    p0 *= sc;
    p1 *= sc;
  }
  for (; i < m; ++i) row(ab[i]);
  return cnt;
}

__device__ __forceinline__ double tri_warp_min(double v) {
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ double tri_warp_max(double v) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Eigenvalue i (ascending) by 32-way multisection of the Gershgorin interval,
// one warp per value; ab is scratch for m rows.  The matrix is scaled by an
// exact power of two to a largest magnitude in [1, 2).
__device__ inline double tri_eig_one(const double* __restrict__ a, const double* __restrict__ b, int m, int i,
                                     double2* ab) {
  const int lane = threadIdx.x;
  double lo = INFINITY, hi = -INFINITY;
  for (int r = lane; r < m; r += 32) {
    const double off = (r > 0 ? fabs(b[r]) : 0.0) + (r + 1 < m ? fabs(b[r + 1]) : 0.0);
    lo = fmin(lo, a[r] - off);
    hi = fmax(hi, a[r] + off);
  }
  lo = tri_warp_min(lo);
  hi = tri_warp_max(hi);
  const double scale = fmax(fabs(lo), fabs(hi));
  const int ex = tri_exp(scale);
  // exact power-of-two scaling (none for a zero, tiny or huge matrix)
  const double inv = (ex > (30 << 20) && ex < (2000 << 20)) ? tri_pow2_inv(ex) : 1.0;
  for (int r = lane; r < m; r += 32) {
    const double br = r > 0 ? b[r] * inv : 0.0;
    ab[r] = make_double2(a[r] * inv, br * br);
  }
  __syncwarp();
  const double sc = scale * inv;
  lo = lo * inv - (1e-14 * sc + 1e-300);
  hi = hi * inv + (1e-14 * sc + 1e-300);
  for (int it = 0; it < 64; ++it) {
    if (hi - lo <= 4e-16 * fmax(fabs(lo), fabs(hi)) + 0x1p-62 * sc) break;
    const double x = lo + (hi - lo) * (double)(lane + 1) / 33.0;
    const int c = sturm(ab, m, x);
    // first lane whose point has more than i eigenvalues below it
    const unsigned above = __ballot_sync(0xffffffffu, c > i);
    const int f = above ? __ffs(above) - 1 : 32;
    const double nlo = (f == 0) ? lo : lo + (hi - lo) * (double)f / 33.0;
    const double nhi = (f == 32) ? hi : lo + (hi - lo) * (double)(f + 1) / 33.0;
    lo = nlo;
    hi = nhi;
  }
  __syncwarp();
  return 0.5 * (lo + hi) / inv;
}

// Vector of eigenvalue k = theta by inverse iteration: solve (T - theta I) x =
// x_prev by tridiagonal Gaussian elimination with partial pivoting (row
// interchanges as in LAPACK's gttrf/gtts2), three sweeps, one warp: lane 0 runs
// the recurrences, all lanes the rest.  wk holds 6 * m doubles of scratch.
// Output s[j], j < m, normalised, largest entry positive.  Quotients are rounded
// once: the factor's by a residual step; the back substitution's, by a pivot known
// ahead, as a product with the pivot's reciprocal in two parts (one dependent
// instruction more than with the rounded reciprocal, whose vectors have residuals
// 6% larger).  The low part's last bit holds the row's interchange.
__device__ inline void tri_vec_one(const double* __restrict__ a, const double* __restrict__ b, int m, double th, int k,
                                   double* wk, double* __restrict__ s) {
  const int lane = threadIdx.x;
  double* x = wk;
  double* dl = x + m;
  double* rd = dl + m;     // pivots, then the high parts of their reciprocals
  double* du = rd + m;
  double* du2 = du + m;
  double* rl = du2 + m;    // interchanges, then with them the low parts
  double anorm = 0.0;
  for (int r = lane; r < m; r += 32) {
    const double off = (r > 0 ? fabs(b[r]) : 0.0) + (r + 1 < m ? fabs(b[r + 1]) : 0.0);
    anorm = fmax(anorm, fabs(a[r]) + off);
    // the elimination reads the matrix from here
    x[r] = a[r] - th;
    dl[r] = r + 1 < m ? b[r + 1] : 0.0;
  }
  anorm = tri_warp_max(anorm);
  const double tiny = 2.2e-16 * fmax(anorm, 1e-300);
  __syncwarp();
  if (lane == 0) {
    double d = x[0], u = dl[0];   // the current row's diagonal and superdiagonal
    for (int r = 0; r + 1 < m; ++r) {
      const double sub = dl[r], nd = x[r + 1], nu = dl[r + 1];
      if (fabs(d) >= fabs(sub)) {
        const double f = (d != 0.0) ? quotient(sub, d) : 0.0;
        rd[r] = d;
        dl[r] = f;
        du[r] = u;
        du2[r] = 0.0;
        rl[r] = __longlong_as_double(0ll);
        d = nd - f * u;
        u = nu;
      } else {
        const double f = quotient(d, sub);
        rd[r] = sub;
        dl[r] = f;
        du[r] = nd;
        du2[r] = nu;
        rl[r] = __longlong_as_double(1ll);
        d = u - f * nd;
        u = -f * nu;
      }
    }
    rd[m - 1] = d;
    du[m - 1] = du2[m - 1] = rl[m - 1] = 0.0;
  }
  __syncwarp();
  for (int r = lane; r < m; r += 32) {
    double d = rd[r];
    if (fabs(d) < tiny) d = (d < 0 ? -tiny : tiny);
    const double y = 1.0 / d;
    rd[r] = y;
    rl[r] = __longlong_as_double((__double_as_longlong(fma(-d, y, 1.0) * y) & ~1ll) |
                                 (__double_as_longlong(rl[r]) & 1ll));
    x[r] = 1.0 + 0.01 * (double)((r * 7919 + k * 104729) % 97) / 97.0;
  }
  __syncwarp();
  for (int sweep = 0; sweep < 3; ++sweep) {
    if (lane == 0) {
      double t = x[0];
#pragma unroll 4
      for (int r = 0; r + 1 < m; ++r) {
        const double xn = x[r + 1], f = dl[r];
        const bool pv = __double2loint(rl[r]) & 1;
        const double keep = pv ? xn : t, go = pv ? t : xn;
        x[r] = keep;
        t = go - f * keep;
      }
      double x1 = fma(t, rd[m - 1], t * rl[m - 1]), x2 = 0.0;
      x[m - 1] = x1;
#pragma unroll 4
      for (int r = m - 2; r >= 0; --r) {
        const double num = x[r] - du2[r] * x2 - du[r] * x1;
        const double v = fma(num, rd[r], num * rl[r]);
        x[r] = v;
        x2 = x1;
        x1 = v;
      }
    }
    __syncwarp();
    double mx = 0.0;
    for (int r = lane; r < m; r += 32) mx = fmax(mx, fabs(x[r]));
    mx = tri_warp_max(mx);
    double inv = tri_pow2_inv(tri_exp(mx));   // to about 1, exactly
    double nrm = 0.0;
    for (int r = lane; r < m; r += 32) {
      const double v = x[r] * inv;
      x[r] = v;
      nrm += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
    const double root = sqrt(nrm);
    inv = nrm > 0 ? 1.0 / root : 0.0;
    for (int r = lane; r < m; r += 32) x[r] = quot_step(x[r], root, inv);   // rounded once: a single entry is 1
    __syncwarp();
  }
  // first entry of the largest magnitude positive
  double big = -1.0;
  int at = 0;
  for (int r = lane; r < m; r += 32)
    if (fabs(x[r]) > big) big = fabs(x[r]), at = r;
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, big, o);
    const int oa = __shfl_xor_sync(0xffffffffu, at, o);
    if (ob > big || (ob == big && oa < at)) big = ob, at = oa;
  }
  const double sg = x[at] < 0 ? -1.0 : 1.0;
  for (int r = lane; r < m; r += 32) s[r] = sg * x[r];
}

// Eigenpair i of T (alpha[0..m), beta[1..m)): theta[i] and S[i*ldS + j], one
// warp.  The scratch is the launch's shared memory (tri_smem(m) bytes) or, for
// matrices too large for it, `work` (6 * ldS doubles per pair).
__device__ inline void tri_pair_one(const double* __restrict__ a, const double* __restrict__ b, int m, int i,
                                    double* __restrict__ theta, double* __restrict__ S, int ldS,
                                    double* __restrict__ work, double* shm) {
  double* wk = m <= kTriSmemRows ? shm : work + (size_t)i * 6 * ldS;
  const double th = tri_eig_one(a, b, m, i, reinterpret_cast<double2*>(wk));
  if (threadIdx.x == 0) theta[i] = th;
  tri_vec_one(a, b, m, th, i, wk, S + (size_t)i * ldS);
}

// Orthogonalise eigenvectors of (nearly) equal eigenvalues in order, then
// residual estimates |beta_m s_{m-1,i}| and double-float copies.
__device__ inline void tri_finish_block(const double* __restrict__ theta, int k, int m, double beta_m,
                                        double* __restrict__ S, int ldS, float2* __restrict__ Sf,
                                        double* __restrict__ resid) {
  __shared__ double sh[32];
  double scale = 0.0;
  for (int i = 0; i < k; ++i) scale = fmax(scale, fabs(theta[i]));
  for (int i = 0; i < k; ++i) {
    double* si = S + (uint64_t)i * ldS;
    for (int j = 0; j < i; ++j) {
      if (fabs(theta[i] - theta[j]) > 1e-9 * fmax(scale, 1.0)) continue;
      double* sj = S + (uint64_t)j * ldS;
      double p = 0.0;
      for (int r = threadIdx.x; r < m; r += blockDim.x) p += si[r] * sj[r];
      p = tri_block_sum(p, sh);
      if (threadIdx.x == 0) sh[0] = p;
      __syncthreads();
      p = sh[0];
      __syncthreads();
      for (int r = threadIdx.x; r < m; r += blockDim.x) si[r] -= p * sj[r];
      __syncthreads();
      double q = 0.0;
      for (int r = threadIdx.x; r < m; r += blockDim.x) q += si[r] * si[r];
      q = tri_block_sum(q, sh);
      if (threadIdx.x == 0) sh[0] = q;
      __syncthreads();
      q = sh[0];
      __syncthreads();
      double inv = q > 0 ? 1.0 / sqrt(q) : 0.0;
      for (int r = threadIdx.x; r < m; r += blockDim.x) si[r] *= inv;
      __syncthreads();
    }
  }
  for (int i = 0; i < k; ++i) {
    for (int r = threadIdx.x; r < m; r += blockDim.x) Sf[(uint64_t)i * ldS + r] = df_from_double(S[(uint64_t)i * ldS + r]);
    if (threadIdx.x == 0) resid[i] = fabs(beta_m * S[(uint64_t)i * ldS + m - 1]);
  }
}

}  // namespace ed
