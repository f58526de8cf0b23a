// Thick-restart Lanczos (Wu & Simon, SIAM J. Matrix Anal. Appl. 22, 2000) for
// the k lowest eigenpairs of a sector Hamiltonian with a Krylov basis of at
// most m vectors.
//
// The paper's solver is the implicitly restarted Arnoldi method (abstract;
// Sec. 3).  For a symmetric H, an implicit restart whose shifts are the
// unwanted Ritz values keeps the span of the wanted Ritz vectors and the
// residual direction; a thick restart keeps that span explicitly:
//
//   after m steps   H V_m = V_m H_m + beta_m v_m e_m^T,   H_m Y = Y Theta,
//   keep u_i = V_m y_i (i < l) and v_l = v_m; the projected matrix becomes
//     [[diag(theta_0 .. theta_{l-1}), s], [s^T, alpha_l, beta_{l+1}], ...]
//   with s_i = beta_m Y[m-1][i] (an arrow on a tridiagonal), and the recurrence
//   continues from v_l with full CGS2 reorthogonalisation against every
//   basis vector (which also removes the s_i u_i components of H v_l).
//
// The projected eigenproblem (dense, symmetric, at most ED_MAX_BASIS rows) is
// solved on the device by cyclic Jacobi in one block, float sweeps finished in
// FP64; the basis rotation V_m Y is k_ritz.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <vector>

#include "lanczos_kernels.h"

namespace ed {

namespace {

constexpr int kMaxBasis = ED_MAX_BASIS;
constexpr int kJacThreads = 512;
constexpr int kJacPairs = kMaxBasis / 2;

// Row stride of a matrix of mp rows in shared memory (odd: rows fall into
// different banks).
__host__ __device__ inline int jac_ld(int mp) { return mp + 1; }
// Both the matrix and the vectors in shared memory up to this size; larger
// bases keep the vectors in global scratch.
constexpr int kJacSmemRows = 112;
inline size_t jac_smem(int m) {
  const int mp = m + (m & 1);
  const size_t one = (size_t)mp * jac_ld(mp) * sizeof(double);
  return (mp <= kJacSmemRows ? 2 : 1) * one + (size_t)kJacPairs * (kJacPairs + 1) / 2 * sizeof(uint16_t);
}

// tangent of the rotation that annihilates a_pq, from d = a_qq - a_pp and a = 2 a_pq
__device__ __forceinline__ float jac_tan(float d, float a) {
  const float tau = d / a;
  return (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
}
__device__ __forceinline__ void jac_cs(float t, float& c, float& s) {
  c = rsqrtf(1.f + t * t);
  s = t * c;
}
// cosine and sine of a given tangent to FP64 accuracy: two Newton steps from a
// float reciprocal root.  c^2 + s^2 = 1 is what keeps the vectors orthogonal and
// the values' sum: 1 / fl(sqrt(1 + t^2)) instead would round to 1 for every t^2
// below 2^-52 or so, always to the same side, and the values of a 40-row matrix
// end 8.6e-15 off where this is 1.5e-15.
__device__ __forceinline__ void jac_cs(double t, double& c, double& s) {
  const double d = fma(t, t, 1.0);
  double y = (double)rsqrtf((float)d);
  y = y * fma(-0.5 * d, y * y, 1.5);
  y = y * fma(-0.5 * d, y * y, 1.5);
  c = y;
  s = t * y;
}

// Rotations of one round, by the first np threads: pair i of round r in the
// round-robin order, identity where |a_pq| <= skip; inv scales the matrix to
// entries of about 1 for the float tangent.
template <class T>
__device__ __forceinline__ void jac_params(const T* A, int ld, int mp, int r, T skip, T inv, T* cs, T* sn, int* pq) {
  const int np = mp / 2, i = threadIdx.x;
  if (i >= np) return;
  const int a = (i == 0) ? 0 : ((i - 1 + r) % (mp - 1)) + 1;
  const int b = ((mp - 2 - i + r) % (mp - 1)) + 1;
  const int p = a < b ? a : b, q = a < b ? b : a;
  const T apq = A[p * ld + q];
  T c = T(1), s = T(0);
  if (fabs(apq) > skip) 
    jac_cs((T)jac_tan((float)((A[q * ld + q] - A[p * ld + p]) * inv), (float)(2 * apq * inv)), c, s);
  pq[i] = p << 8 | q;
  cs[i] = c;
  sn[i] = s;
}

// A <- J^T A J over the 2 x 2 blocks of the pairs i <= j (each block depends on
// its own four entries only, so a round needs no barrier inside), mirrored;
// Y, which holds the vectors as rows, <- J^T Y.
template <class T>
__device__ __forceinline__ void jac_rotate(T* A, T* Y, int ld, int mp, const uint16_t* tab, const T* cs, const T* sn,
                                           const int* pq) {
  const int np = mp / 2;
  for (int idx = threadIdx.x; idx < np * (np + 1) / 2; idx += kJacThreads) {
    const int i = tab[idx] >> 8, j = tab[idx] & 255;
    const T si = sn[i], sj = sn[j];
    if (si == T(0) && sj == T(0)) continue;
    const T ci = cs[i], cj = cs[j];
    const int pi = pq[i] >> 8, qi = pq[i] & 255, pj = pq[j] >> 8, qj = pq[j] & 255;
    const T pp = A[pi * ld + pj], pr = A[pi * ld + qj], qp = A[qi * ld + pj], qr = A[qi * ld + qj];
    const T a0 = ci * pp - si * qp, b0 = si * pp + ci * qp;   // rows of pair i
    const T a1 = ci * pr - si * qr, b1 = si * pr + ci * qr;
    const T r0 = cj * a0 - sj * a1, r1 = sj * a0 + cj * a1;   // columns of pair j
    const T r2 = cj * b0 - sj * b1, r3 = sj * b0 + cj * b1;
    A[pi * ld + pj] = r0;
    A[pi * ld + qj] = r1;
    A[qi * ld + qj] = r3;
    if (i == j) {
      A[qi * ld + pj] = r1;   // the pair's own block stays symmetric
    } else {
      A[qi * ld + pj] = r2;
      A[pj * ld + pi] = r0;
      A[qj * ld + pi] = r1;
      A[pj * ld + qi] = r2;
      A[qj * ld + qi] = r3;
    }
  }
  const int di = kJacThreads / mp, dr = kJacThreads - di * mp;
  int i = threadIdx.x / mp, r = threadIdx.x - i * mp;
  while (i < np) {
    const T s = sn[i];
    if (s != T(0)) {
      const T c = cs[i];
      const int p = pq[i] >> 8, q = pq[i] & 255;
      const T yp = Y[p * ld + r], yq = Y[q * ld + r];
      Y[p * ld + r] = c * yp - s * yq;
      Y[q * ld + r] = s * yp + c * yq;
    }
    i += di;
    r += dr;
    if (r >= mp) r -= mp, ++i;
  }
}

// Eigen-decomposition of the m x m symmetric matrix Ain (row-major, leading
// dimension lda): theta ascending, eigenvector i in S[i * ldS + r] (and its
// double-float split in Sf).  Yg is kMaxBasis^2 doubles of device scratch; S
// also serves as scratch.
//
// Cyclic Jacobi in one block (round-robin pairs, all disjoint rotations of a
// round at once).  A round of a 40 x 40 matrix is 5,600 FP64 multiply-adds, 2 us
// at GB300's 1.6 FP64 lanes per SM and clock, and 8 to 10 sweeps of 39 rounds
// are needed from scratch; in float a round takes 0.2 us.  So the sweeps run in
// float first, the vectors are made orthonormal in FP64 (two Newton-Schulz
// steps: Gram matrix in FP64, the small correction's product in float), the
// matrix is transformed by them in FP64, and FP64 sweeps finish from
// off-diagonals of about 1e-6 (two sweeps) to the same criterion as sweeps in
// FP64 throughout.
//
// The float sweeps work on the matrix less a diagonal entry, scaled to entries of at
// most 1: what float resolves follows the spread of the values, not how far
// from zero they lie.
//
// k > 0: a convergence check whose decomposition is not used further.  It ends
// after the float sweeps (110 us instead of 490 us) if one of the k lowest pairs
// is clearly not converged: beta |s_last| above twice tol max(1, |theta|) by more
// than beta times an estimate of the float component's error, with the k lowest
// float values and last components as the estimates.  To first order vector i
// takes up vector j by (what the sweeps leave at (i, j) + their rounding) / (their
// values' distance), so the estimate is the sum of that times |s_last| of j, and at
// least 1e-3; the rounding of some 10 m rotations of a row, 2^-24 each, is spread
// over the matrix (three times its mean square is taken).  A pair whose neighbour
// float cannot tell apart is not called open here, so that a check costs products
// only where it is open (values 2^14 from zero took 88 products instead of 44 with
// the 1e-3 alone).
__global__ void __launch_bounds__(kJacThreads) k_sym_jacobi(const double* __restrict__ Ain, int m, int lda,
                                                            double* __restrict__ theta, double* S,
                                                            float2* __restrict__ Sf, int ldS, double* Yg,
                                                            const double* __restrict__ beta, int k, double tol) {
  extern __shared__ __align__(16) unsigned char jsm[];
  const int mp = m + (m & 1);  // an odd size is padded by a zero row and column (index m)
  const int ld = jac_ld(mp), np = mp / 2;
  const size_t one = (size_t)mp * ld;
  double* A = reinterpret_cast<double*>(jsm);
  const bool ysm = mp <= kJacSmemRows;
  double* Y = ysm ? A + one : Yg;
  uint16_t* tab = reinterpret_cast<uint16_t*>(A + (ysm ? 2 : 1) * one);
  // float phase: the matrix and its vectors share the FP64 matrix's place
  float* Af = reinterpret_cast<float*>(A);
  float* Yf = Af + one;
  __shared__ double cs[kJacPairs], sn[kJacPairs];
  __shared__ float csf[kJacPairs], snf[kJacPairs];
  __shared__ int pq[kJacPairs];
  __shared__ double red[kJacThreads / 32];
  __shared__ int order[kMaxBasis];
  const int tid = threadIdx.x, nt = kJacThreads;
  const int lane = tid & 31, warp = tid >> 5, nw = nt / 32;
  auto block_sum = [&](double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < nw; ++w) t += red[w];
    __syncthreads();
    return t;
  };
  auto block_sumf = [&](float v) { return block_sum((double)v); };
  for (int i = tid; i < kMaxBasis; i += nt) order[i] = i;   // stays valid where values are not comparable (NaN)
  for (int i = warp; i < np; i += nw)
    for (int j = lane; j < np; j += 32)
      if (j >= i) tab[i * np - i * (i - 1) / 2 + (j - i)] = (uint16_t)(i << 8 | j);
  const double mid = Ain[(size_t)(m / 2) * (lda + 1)];
  double fro = 0.0, frof = 0.0, amax = 0.0;   // Frobenius norm, and that of the shifted matrix
  for (int i = warp; i < m; i += nw)
    for (int j = lane; j < m; j += 32)
      if (i != j) {
        const double v = Ain[(size_t)i * lda + j];
        frof += v * v;
        amax = fmax(amax, fabs(v));
      }
  fro = frof;
  for (int i = tid; i < m; i += nt) {
    const double d = Ain[(size_t)i * (lda + 1)], u = d - mid;
    fro += d * d;
    frof += u * u;
    amax = fmax(amax, fabs(u));
  }
  {   // both sums in one pass
    __shared__ double2 red2[kJacThreads / 32];
    for (int o = 16; o > 0; o >>= 1) {
      fro += __shfl_xor_sync(0xffffffffu, fro, o);
      frof += __shfl_xor_sync(0xffffffffu, frof, o);
    }
    if (lane == 0) red2[warp] = make_double2(fro, frof);
    __syncthreads();
    fro = frof = 0.0;
    for (int w = 0; w < nw; ++w) fro += red2[w].x, frof += red2[w].y;
  }
  for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if (lane == 0) red[warp] = amax;
  __syncthreads();
  for (int w = 0; w < nw; ++w) amax = fmax(amax, red[w]);
  __syncthreads();
  // ---- float sweeps on the shifted matrix scaled to entries of at most 1
  const double inv = amax > 0.0 ? 1.0 / amax : 0.0;
  for (int i = warp; i < mp; i += nw)
    for (int j = lane; j < mp; j += 32) {
      double v = (i < m && j < m) ? Ain[(size_t)i * lda + j] : 0.0;
      if (i == j && i < m) v -= mid;
      Af[i * ld + j] = (float)(v * inv);
      Yf[i * ld + j] = i == j ? 1.f : 0.f;
    }
  __syncthreads();
  frof *= inv * inv;
  for (int sweep = 0; sweep < 12 && m > 1; ++sweep) {
    float off = 0.f;
    for (int i = warp; i < m; i += nw)
      for (int j = lane; j < m; j += 32)
        if (i != j) off += Af[i * ld + j] * Af[i * ld + j];
    if (!(block_sumf(off) > 1e-11 * frof)) break;
    for (int r = 0; r < mp - 1; ++r) {
      jac_params<float>(Af, ld, mp, r, 0.f, 1.f, csf, snf, pq);
      __syncthreads();
      jac_rotate<float>(Af, Yf, ld, mp, tab, csf, snf, pq);
      __syncthreads();
    }
  }
  if (k > 0) {
    __shared__ int open;
    if (tid == 0) open = 0;
    __syncthreads();
    const double b = *beta;
    const float E = 3.f * 0x1p-24f * sqrtf(10.f / (float)m * (float)frof);
    for (int i = tid; i < m; i += nt) {
      const float key = Af[i * ld + i];
      int at = 0;
      float err = 0.f;
      for (int j = 0; j < m; ++j) {
        const float o = Af[j * ld + j];
        at += (o < key || (o == key && j < i)) ? 1 : 0;
        if (j != i) {
          const float e = fabsf(Af[i * ld + j]) + E, gap = fabsf(o - key);
          err += e < 0.5f * gap ? __fdividef(e, gap) * fabsf(Yf[j * ld + m - 1]) : 1.f;
        }
      }
      if (at < k) {
        const double th = fma((double)key, amax, mid), last = fabs((double)Yf[i * ld + m - 1]);
        theta[at] = th;
        S[(size_t)at * ldS + m - 1] = last;
        if (b * (last - fmax(1e-3, (double)err)) > 2.0 * tol * fmax(1.0, fabs(th))) open = 1;
      }
    }
    __syncthreads();
    if (open) return;
  }
  // ---- orthonormal vectors in FP64: twice Y += E Y with E = (I - Y Y^T) / 2
  for (int i = warp; i < mp; i += nw)
    for (int j = lane; j < mp; j += 32) Y[i * ld + j] = (double)Yf[i * ld + j];
  __syncthreads();
  for (int step = 0; step < 2; ++step) {
    for (int idx = tid; idx < m * m; idx += nt) {
      const int i = idx / m, j = idx - i * m;
      if (j > i) continue;
      double g = 0.0;
      for (int r = 0; r < m; ++r) g = fma(Y[i * ld + r], Y[j * ld + r], g);
      const float e = (float)(0.5 * ((i == j ? 1.0 : 0.0) - g));
      Af[i * ld + j] = e;
      Af[j * ld + i] = e;
    }
    __syncthreads();
    for (int i = warp; i < m; i += nw)
      for (int r = lane; r < m; r += 32) {
        float v = 0.f;
        for (int j = 0; j < m; ++j) v = fmaf(Af[i * ld + j], Yf[j * ld + r], v);
        Y[i * ld + r] += (double)v;
      }
    __syncthreads();
  }
  // ---- B = Y A Y^T through T[r][v] = sum_c A[r][c] Y[v][c] (kept in S); A is
  // an arrow on a tridiagonal, so most of its entries are zero
  for (int r = warp; r < m; r += nw)
    for (int v = lane; v < m; v += 32) {
      double t = 0.0;
      for (int c = 0; c < m; ++c) {
        const double arc = Ain[(size_t)r * lda + c];
        if (arc != 0.0) t = fma(arc, Y[v * ld + c], t);
      }
      S[(size_t)r * ldS + v] = t;
    }
  __syncthreads();
  for (int idx = tid; idx < mp * mp; idx += nt) {
    const int u = idx / mp, v = idx - u * mp;
    if (v > u) continue;
    double t = 0.0;
    if (u < m)
      for (int r = 0; r < m; ++r) t = fma(Y[u * ld + r], S[(size_t)r * ldS + v], t);
    A[u * ld + v] = t;
    A[v * ld + u] = t;
  }
  __syncthreads();
  // ---- FP64 sweeps
  const double skip = 1e-18 * sqrt(fro) / (double)m;   // below this a whole matrix of entries is under the criterion
  for (int sweep = 0; sweep < 60 && m > 1; ++sweep) {
    double off = 0.0;
    for (int i = warp; i < m; i += nw)
      for (int j = lane; j < m; j += 32)
        if (i != j) off += A[i * ld + j] * A[i * ld + j];
    off = block_sum(off);
    if (!(off > 1e-32 * fro)) break;
    for (int r = 0; r < mp - 1; ++r) {
      jac_params<double>(A, ld, mp, r, skip, inv, cs, sn, pq);
      __syncthreads();
      jac_rotate<double>(A, Y, ld, mp, tab, cs, sn, pq);
      __syncthreads();
    }
  }
  // ---- ascending order: a value's place is the number of values before it
  for (int i = tid; i < m; i += nt) {
    const double key = A[i * ld + i];
    int at = 0;
    for (int j = 0; j < m; ++j) {
      const double o = A[j * ld + j];
      at += (o < key || (o == key && j < i)) ? 1 : 0;
    }
    order[at] = i;
  }
  __syncthreads();
  for (int i = tid; i < m; i += nt) theta[i] = A[order[i] * ld + order[i]];
  for (int i = warp; i < m; i += nw)
    for (int r = lane; r < m; r += 32) {
      const double v = Y[order[i] * ld + r];
      S[(size_t)i * ldS + r] = v;
      Sf[(size_t)i * ldS + r] = df_from_double(v);
    }
}

// Projected matrix of the current basis (size rows): the kept Ritz values and
// their couplings s to basis vector l, then the Lanczos tridiagonal from l on.
__global__ void k_tr_project(double* __restrict__ Hp, int ld, int size, int l, const double* __restrict__ th,
                             const double* __restrict__ sv, Coefs c) {
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < size * size; idx += gridDim.x * blockDim.x) {
    const int i = idx / size, j = idx % size;
    double v = 0.0;
    if (i == j) v = (i < l) ? th[i] : c.alpha[i];
    else if (i < l && j == l) v = sv[i];
    else if (j < l && i == l) v = sv[j];
    else if (i >= l && j == i + 1) v = c.beta[j];
    else if (j >= l && i == j + 1) v = c.beta[i];
    Hp[(size_t)i * ld + j] = v;
  }
}

// After a restart with l kept vectors: theta and s_i = beta_m S[i][m-1].
__global__ void k_tr_keep(const double* __restrict__ theta, const double* __restrict__ S, int ldS, int m, int l,
                          Coefs c, double* __restrict__ th, double* __restrict__ sv) {
  for (int i = threadIdx.x; i < l; i += blockDim.x) {
    th[i] = theta[i];
    sv[i] = c.beta[m] * S[(size_t)i * ldS + m - 1];
  }
}

int jacobi(cudaStream_t st, const double* Hp, int m, int ld, double* theta, double* S, float2* Sf, int ldS,
           double* Y, const double* beta, int k, double tol) {
  // one cap for every size: concurrent solves of different basis sizes set the same value
  ED_TRY_CUDA(cudaFuncSetAttribute(k_sym_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)jac_smem(kJacSmemRows)));
  k_sym_jacobi<<<1, kJacThreads, jac_smem(m), st>>>(Hp, m, ld, theta, S, Sf, ldS, Y, beta, k, tol);
  ED_LAUNCH_CHECK();
  return ED_OK;
}

template <class V>
int trlan_impl(Sector* s, const ed_trlan_opts* o, double* evals, void* evecs, ed_trlan_info* info,
               cudaStream_t st) {
  auto t_start = std::chrono::steady_clock::now();
  Ctx* ctx = s->ctx;
  const uint64_t n = s->dim;
  const int k = o->k;
  const int kk = (int)std::min<uint64_t>((uint64_t)k, n);
  const int m = (int)std::min<uint64_t>((uint64_t)o->max_basis, n);
  int keep = o->keep > 0 ? o->keep : (m + kk) / 2;
  keep = std::max(kk, std::min(keep, m - 2));
  const int check_every = std::max(1, o->check_every);
  const int max_iter = std::max(1, o->max_iter);
  const size_t eb = sizeof(V);

  // basis V[0..m] (m + 1 vectors), w, rotation target T[0..keep)
  const int n_rot = (m >= 3) ? keep : 0;
  DevBuf vb, cb, hb;
  // slots padded to 32 elements, so that each starts 16-byte aligned
  const uint64_t ld = pad32(n);
  ED_TRY(vb.alloc(ctx, ((size_t)m + 2 + n_rot) * ld * eb));
  // four matrices (one of kMaxBasis + 1 columns) and three vectors beside the coefficients
  ED_TRY(cb.alloc(ctx, coef_bytes(m, 1) + (size_t)kMaxBasis * kMaxBasis * 8 * 4 + (size_t)kMaxBasis * 8 * 4));
  V* Vb = static_cast<V*>(vb.p);
  V* w = Vb + (size_t)(m + 1) * ld;
  V* T = w + ld;  // rotation target, keep vectors of n elements back to back
  Carve cv{static_cast<char*>(cb.p)};
  Coefs c = carve_coefs(cv, m);
  const int ldS = kMaxBasis;
  double* Hp = cv.take<double>((size_t)kMaxBasis * kMaxBasis);
  double* Y = cv.take<double>((size_t)kMaxBasis * jac_ld(kMaxBasis));
  double* Sd = cv.take<double>((size_t)kMaxBasis * ldS);
  float2* Sf = cv.take<float2>((size_t)kMaxBasis * ldS);
  double* theta = cv.take<double>(kMaxBasis);
  double* th = cv.take<double>(kMaxBasis);
  double* sv = cv.take<double>(kMaxBasis);

  Work<V> W;
  W.ctx = ctx;
  W.st = st;
  W.n = n;
  W.grid = (uint32_t)std::min<uint64_t>((n + kRedThreads - 1) / kRedThreads, (uint64_t)ctx->num_sms * 8);
  if (W.grid == 0) W.grid = 1;
  W.partial = ctx->d_red;
  W.c = c;
  ED_TRY(cgs_room(W, hb, m));
  uint32_t vgrid = (uint32_t)std::min<uint64_t>((n + 255) / 256, (uint64_t)ctx->num_sms * 16);
  if (vgrid == 0) vgrid = 1;
  auto vec = [&](int j) -> V* { return Vb + (size_t)j * ld; };

  k_init_coefs<<<1, 256, 0, st>>>(c, m + 2);
  if (o->v0) {
    ED_TRY_CUDA(cudaMemcpyAsync(w, o->v0, n * eb, cudaMemcpyDeviceToDevice, st));
  } else {
    k_random<V><<<vgrid, 256, 0, st>>>(w, n, o->seed);
  }
  ED_TRY(dot_to(W, (const V*)w, (const V*)w, OP_NORM_INV, 0));
  k_scale<V><<<vgrid, 256, 0, st>>>(w, vec(0), n, c, 0);
  ED_LAUNCH_CHECK();

  // one event pair per basis slot times the H*v launches; read at each check
  std::vector<cudaEvent_t> evs(2 * (size_t)m);
  for (auto& e : evs) ED_TRY_CUDA(cudaEventCreate(&e));
  struct EvGuard {
    std::vector<cudaEvent_t>* v;
    ~EvGuard() {
      for (auto e : *v) cudaEventDestroy(e);
    }
  } evguard{&evs};
  std::vector<int> pending;
  double apply_ms = 0.0;
  auto drain_timers = [&]() {
    for (int q : pending) {
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, evs[2 * q], evs[2 * q + 1]) == cudaSuccess) apply_ms += ms;
    }
    pending.clear();
  };

  const double thr = 1e-13;
  std::vector<double> h_theta(kMaxBasis), h_last(kMaxBasis), h_res(ED_MAX_K, 0.0);
  int l = 0, size = 0, iters = 0, restarts = 0, injections = 0, n_conv = 0;
  int status = ED_OK;
  bool done = false;
  int j = 0;  // next basis slot to extend from
  while (!done) {
    while (j < m) {
      ED_TRY(lanczos_step(s, W, (const V*)Vb, ld, j, j > l ? vec(j - 1) : nullptr, w, vec(j + 1), thr, evs[2 * j],
                          evs[2 * j + 1]));
      pending.push_back(j);
      ++iters;
      size = ++j;
      if (size < m && ((size - l) % check_every) != 0 && iters < max_iter) continue;
      // first vanished beta: the basis is an invariant subspace up to there
      int ex = -1;
      ED_TRY_CUDA(cudaMemcpyAsync(ctx->h_red, c.exhausted, sizeof(int), cudaMemcpyDeviceToHost, st));
      ED_TRY_CUDA(cudaStreamSynchronize(st));
      std::memcpy(&ex, ctx->h_red, sizeof(int));
      drain_timers();
      if (ex >= 0 && ex < size) size = j = ex;  // steps past it are discarded
      // projected eigenproblem of the current basis
      k_tr_project<<<(size * size + 255) / 256, 256, 0, st>>>(Hp, kMaxBasis, size, l, th, sv, c);
      ED_LAUNCH_CHECK();
      const int kc = std::min(kk, size);
      // the decomposition is used beyond the check at a restart, at the end and in an invariant subspace
      const bool check_only = size < m && iters < max_iter && ex < 0 && kc == kk;
      ED_TRY(jacobi(st, Hp, size, kMaxBasis, theta, Sd, Sf, ldS, Y, c.beta + size, check_only ? kc : 0, o->tol));
      double beta_next = 0.0;
      ED_TRY_CUDA(cudaMemcpyAsync(h_theta.data(), theta, kc * sizeof(double), cudaMemcpyDeviceToHost, st));
      ED_TRY_CUDA(cudaMemcpyAsync(&beta_next, c.beta + size, sizeof(double), cudaMemcpyDeviceToHost, st));
      ED_TRY_CUDA(cudaMemcpy2DAsync(h_last.data(), sizeof(double), Sd + (size - 1), (size_t)ldS * sizeof(double),
                                    sizeof(double), kc, cudaMemcpyDeviceToHost, st));
      ED_TRY_CUDA(cudaStreamSynchronize(st));
      n_conv = 0;
      for (int i = 0; i < kc; ++i) {
        h_res[i] = std::fabs(beta_next * h_last[i]);
        if (h_res[i] <= o->tol * std::max(1.0, std::fabs(h_theta[i])) && n_conv == i) ++n_conv;
      }
      if (ex >= 0) {
        // invariant subspace: its Ritz pairs are exact
        for (int i = 0; i < kc; ++i) h_res[i] = 0.0;
        n_conv = kc;
        if ((uint64_t)size >= n || kc >= kk) {
          done = true;
          break;
        }
        // fewer than k values in it: go on from a fresh direction orthogonal
        // to the basis, uncoupled from it (beta = 0)
        ++injections;
        k_random<V><<<vgrid, 256, 0, st>>>(w, n, o->seed + 7919ull * (uint64_t)injections);
        ED_TRY(cgs2(W, (const V*)Vb, ld, size, w));
        k_finish<<<1, kRedThreads, 0, st>>>(W.partial, (int)cgs_grid<V>(ctx, n), OP_NORM_INV, 1, c);
        k_scale<V><<<vgrid, 256, 0, st>>>(w, vec(size), n, c, 1);
        ED_LAUNCH_CHECK();
        const double zero = 0.0;
        const int neg = -1;
        ED_TRY_CUDA(cudaMemcpyAsync(c.beta + size, &zero, sizeof(double), cudaMemcpyHostToDevice, st));
        ED_TRY_CUDA(cudaMemcpyAsync(c.exhausted, &neg, sizeof(int), cudaMemcpyHostToDevice, st));
        ED_TRY_CUDA(cudaStreamSynchronize(st));
        continue;  // j == size: the next step starts from the new vector (a full basis restarts first)
      }
      if (kc >= kk && n_conv >= kk) {
        done = true;
        break;
      }
      if (iters >= max_iter) {
        status = ED_ERR_NOT_CONVERGED;
        done = true;
        break;
      }
    }
    if (done) break;
    // basis full: keep the `keep` lowest Ritz vectors and the residual direction
    if (n_rot == 0) {
      status = ED_ERR_NOT_CONVERGED;
      break;
    }
    ED_TRY(ritz(ctx, st, (const V*)Vb, ld, m, Sd, Sf, ldS, keep, T, n, 0));
    ED_TRY_CUDA(cudaMemcpy2DAsync(Vb, ld * eb, T, n * eb, n * eb, keep, cudaMemcpyDeviceToDevice, st));
    ED_TRY_CUDA(cudaMemcpyAsync(vec(keep), vec(m), n * eb, cudaMemcpyDeviceToDevice, st));
    k_tr_keep<<<1, 128, 0, st>>>(theta, Sd, ldS, m, keep, c, th, sv);
    ED_LAUNCH_CHECK();
    l = j = keep;
    ++restarts;
  }
  ED_TRY_CUDA(cudaStreamSynchronize(st));
  drain_timers();

  const int kc = std::min(kk, size);
  for (int i = 0; i < kc; ++i) evals[i] = h_theta[i];
  for (int i = kc; i < k; ++i) evals[i] = NAN;
  if (evecs && kc > 0) {
    // Sd holds the eigenvectors of the last projected matrix (size `size`)
    V* out = static_cast<V*>(evecs);
    ED_TRY(ritz(ctx, st, (const V*)Vb, ld, size, Sd, Sf, ldS, kc, out, n, 0));
  }
  ED_TRY_CUDA(cudaStreamSynchronize(st));
  if (info) {
    info->iters = iters;
    info->restarts = restarts;
    info->n_converged = std::min(n_conv, kc);
    for (int i = 0; i < ED_MAX_K; ++i) info->residual[i] = (i < kc) ? h_res[i] : 0.0;
    info->apply_ms = apply_ms;
    info->basis_bytes = ((size_t)m + 2 + n_rot) * ld * eb;
    info->total_ms =
        std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_start).count();
  }
  if (status != ED_OK) set_error("thick-restart Lanczos did not converge in %d products", max_iter);
  return status;
}

}  // namespace

int trlan_run(Sector* s, const ed_trlan_opts* o, double* evals, void* evecs, ed_trlan_info* info,
              cudaStream_t st) {
  if (!o || !evals) ED_INVALID("NULL argument");
  if (o->k < 1 || o->k > ED_MAX_K) ED_INVALID("k must be in 1..%d", ED_MAX_K);
  if (!(o->tol > 0.0)) ED_INVALID("tol must be positive");
  if (o->max_basis > ED_MAX_BASIS) ED_INVALID("max_basis must be at most %d", ED_MAX_BASIS);
  const uint64_t n = s->dim;
  const uint64_t kk = std::min<uint64_t>((uint64_t)o->k, n);
  if ((uint64_t)o->max_basis < std::min<uint64_t>(kk + 2, n))
    ED_INVALID("max_basis (%d) must be at least k + 2 (or the sector dimension)", o->max_basis);
  if (o->keep != 0 && (o->keep < (int)kk || o->keep > o->max_basis - 2))
    ED_INVALID("keep must be 0 or in k..max_basis-2");
  switch (s->prec) {
    case ED_PREC_FP64: return trlan_impl<double>(s, o, evals, evecs, info, st);
    case ED_PREC_DF64: return trlan_impl<float2>(s, o, evals, evecs, info, st);
    case ED_PREC_FP32: return trlan_impl<float>(s, o, evals, evecs, info, st);
  }
  ED_INVALID("unknown precision");
}

}  // namespace ed
