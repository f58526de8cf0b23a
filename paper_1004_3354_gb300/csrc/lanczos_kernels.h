// Lanczos building blocks shared by the solver drivers (lanczos.cu) and the
// request server (serve.cu): reductions, vector updates, the coefficient
// bookkeeping kernel, CGS2 and the tridiagonal solve.  Internal header; each
// translation unit gets its own copy (anonymous namespace).
#pragma once

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <vector>

#include "cgs_tile.h"
#include "ed_internal.h"
#include "fp64_short.h"
#include "tri_common.h"
#include "vec_ops.h"

namespace ed {

namespace {

// ------------------------------------------------ reductions
// partial[b] = sum over this block's elements of x*y (as double)
template <class V>
__global__ void __launch_bounds__(kRedThreads) k_dot(const V* __restrict__ x, const V* __restrict__ y,
                                                     uint64_t n, double* __restrict__ partial) {
  using A = typename AccOf<V>::T;
  __shared__ A sh[32];
  A acc{};
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x)
    dmac(acc, x[i], y[i]);
  acc = block_reduce(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = to_d(acc);
}

// ------------------------------------------------ coefficient bookkeeping
struct Coefs {
  double* alpha;    // [m+1]
  double* beta;     // [m+2], beta[0] = 0
  double* inv_d;    // 1 / beta (0 when beta vanished)
  float2* inv_f;
  double* h_d;      // -h (CGS projections)
  float2* h_f;
  double* scale;    // running max |alpha|, beta (two slots: k_scale_beta reads one and writes the other)
  int* exhausted;   // first step with a vanished beta, -1 if none
  double* out;      // generic scalar output slots
  // three-vector recurrence on unnormalised vectors q_j (v_j = sigma_j q_j):
  // q_{j+1} = ua_j H q_j + ub_j q_j + uc_j q_{j-1}
  double* sigma;
  double* ua_d;
  float2* ua_f;
  double* ub_d;
  float2* ub_f;
  double* uc_d;
  float2* uc_f;
  int* step;        // device step index for graph-replayed steps (slot < 0 / j < 0 read it)
};

enum FinishOp { OP_SUM, OP_NEGH, OP_NORM_INV, OP_SIGMA0 };

// Sum nb partials (one output per block of this kernel) and apply `op`.
__global__ void __launch_bounds__(kRedThreads) k_finish(const double* __restrict__ partial, int nb, int op,
                                                        int slot, Coefs c) {
  __shared__ double sh[32];
  int o = blockIdx.x;
  double v = 0.0;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) v += partial[(uint64_t)o * nb + i];
  v = block_reduce(v, sh);
  if (threadIdx.x != 0) return;
  switch (op) {
    case OP_SUM: c.out[slot + o] = v; break;
    case OP_NEGH:
      c.h_d[slot + o] = -v;
      c.h_f[slot + o] = df_from_double(-v);
      break;
    case OP_NORM_INV: {
      double b = sqrt(fmax(v, 0.0));
      double inv = b > 0.0 ? 1.0 / b : 0.0;
      c.out[slot] = b;
      c.inv_d[slot] = inv;
      c.inv_f[slot] = df_from_double(inv);
      break;
    }
    case OP_SIGMA0: {  // v = <q_0, q_0>
      double b = sqrt(fmax(v, 0.0));
      c.out[0] = b;
      c.sigma[0] = b > 0.0 ? 1.0 / b : 0.0;
      c.beta[0] = 0.0;
      break;
    }
  }
}

// ------------------------------------------------ vector updates
// q_out = ua y + ub q_j + uc q_{j-1} element by element in sixteen-byte
// vectors (every buffer 16-byte aligned); q_out may be the buffer of q_{j-1}.
// Returns the thread's share of <q_out, q_out> (NORM).
template <class V, bool NORM, class A>
__device__ __forceinline__ A lz_combine(const V* __restrict__ y, const V* __restrict__ qj, const V* qjm, V* qout,
                                        uint64_t n, A ua, A ub, A uc) {
  using W16 = Vec16<V>;
  using VT = typename W16::T;
  constexpr int N = W16::N;
  A nacc{};
  const uint64_t nv = n / N;
  const uint64_t g0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, gs = (uint64_t)gridDim.x * blockDim.x;
  auto one = [&](V yv, V q1, V q0) {
    A a{};
    hmac(a, ua, yv);
    hmac(a, ub, q1);
    if (qjm) hmac(a, uc, q0);
    const V q = store_v(a, qout);
    if (NORM) dmac(nacc, q, q);
    return q;
  };
  for (uint64_t t = g0; t < nv; t += gs) {
    const VT yv = reinterpret_cast<const VT*>(y)[t], v1 = reinterpret_cast<const VT*>(qj)[t];
    const VT v0 = qjm ? reinterpret_cast<const VT*>(qjm)[t] : VT{};
    VT o{};
#pragma unroll
    for (int i = 0; i < N; ++i) W16::set(o, i, one(W16::get(yv, i), W16::get(v1, i), W16::get(v0, i)));
    reinterpret_cast<VT*>(qout)[t] = o;
  }
  for (uint64_t i = nv * N + g0; i < n; i += gs) qout[i] = one(y[i], qj[i], qjm ? qjm[i] : V{});
  return nacc;
}

// beta_j and sigma_j = 1 / beta_j from v = |q_j|^2, sc the running scale.
__device__ __forceinline__ void lz_beta(double v, double& sc, double thr, double& beta, double& sigma, bool& dead) {
  double b = 0.0, y = 0.0;
  if (v > 0.0) root_inverse(v, b, y);
  sc = fmax(sc, b);
  dead = !(b > thr * fmax(sc, 1.0));
  beta = dead ? 0.0 : b;
  sigma = dead ? 0.0 : y;
}

// One three-vector step after H q_j (in y): alpha_j from the na partials of
// <q_j, H q_j>, beta_j from the previous step's nn partials of |q_j|^2
// (npart[(j - 1) & 1]), then q_{j+1} and the partials of its norm
// (npart[j & 1]).  Every block forms the step's numbers itself, so a step is two launches (H*v and this)
// where separate finishing launches made it four; block 0 keeps them.  j < 0:
// the step index in c.step (graph replays).
constexpr int kLzThreads = 1024;
struct NormPart {
  double* p[2];
};
template <class V>
__global__ void __launch_bounds__(kLzThreads) k_lz_step(const V* __restrict__ y, const V* __restrict__ qj,
                                                         const V* qjm, V* qout, uint64_t n, Coefs c, int j,
                                                         const double* __restrict__ apart, int na, NormPart npart,
                                                         double thr) {
  using A = typename AccOf<V>::T;
  __shared__ A sh[32];
  __shared__ double tot[2];
  __shared__ double ud[3];
  __shared__ A u[3];
  if (j < 0) j = *c.step;
  if (j == 0) qjm = nullptr;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp == 0) tot[0] = warp_total(apart, na, lane);
  if (warp == 1) tot[1] = warp_total(npart.p[(j + 1) & 1], j > 0 ? (int)gridDim.x : 0, lane);
  __syncthreads();
  if (threadIdx.x == 0) {
    double sc = c.scale[j & 1], beta = 0.0, sg = c.sigma[0];
    bool dead = false;
    if (j > 0) lz_beta(tot[1], sc, thr, beta, sg, dead);
    const double a = sg * sg * tot[0];
    ud[0] = sg;
    ud[1] = -a * sg;
    ud[2] = j > 0 ? -beta * c.sigma[j - 1] : 0.0;
    if (blockIdx.x == 0) {
      if (j > 0) {
        c.beta[j] = beta;
        c.sigma[j] = sg;
        if (dead && *c.exhausted < 0) *c.exhausted = j;
      }
      c.alpha[j] = a;
      c.scale[(j + 1) & 1] = fmax(sc, fabs(a));
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    const int i = threadIdx.x;
    h_split(u[i], ud[i]);
    if (blockIdx.x == 0) {
      (i == 0 ? c.ua_d : i == 1 ? c.ub_d : c.uc_d)[j] = ud[i];
      (i == 0 ? c.ua_f : i == 1 ? c.ub_f : c.uc_f)[j] = df_from_double(ud[i]);
    }
  }
  __syncthreads();
  A nacc = lz_combine<V, true, A>(y, qj, qjm, qout, n, u[0], u[1], u[2]);
  nacc = block_reduce(nacc, sh);
  if (threadIdx.x == 0) npart.p[j & 1][blockIdx.x] = to_d(nacc);
}

// beta_m, sigma_m and the exhaustion flag after m steps (m < 0: c.step), ahead of
// a convergence check; the next step forms the same numbers again, from the same
// sums in the same order.  One warp.
__global__ void k_lz_close(NormPart npart, int nn, Coefs c, int m, double thr) {
  if (m < 0) m = *c.step;
  if (m < 1) return;
  const double v = warp_total(npart.p[(m + 1) & 1], nn, threadIdx.x);
  if (threadIdx.x != 0) return;
  double sc = c.scale[m & 1], beta, sg;
  bool dead;
  lz_beta(v, sc, thr, beta, sg, dead);
  c.beta[m] = beta;
  c.sigma[m] = sg;
  if (dead && *c.exhausted < 0) *c.exhausted = m;
}

// q_{j+1} again from y = H q_j and the stored coefficients of step j.
template <class V>
__global__ void __launch_bounds__(kLzThreads) k_lz_regen(const V* __restrict__ y, const V* __restrict__ qj,
                                                          const V* qjm, V* qout, uint64_t n, Coefs c, int j) {
  using A = typename AccOf<V>::T;
  A ua, ub, uc;
  h_pick(ua, c.ua_d, c.ua_f, j);
  h_pick(ub, c.ub_d, c.ub_f, j);
  h_pick(uc, c.uc_d, c.uc_f, j);
  lz_combine<V, false, A>(y, qj, qjm, qout, n, ua, ub, uc);
}

// One block per SM: each sums the partials itself, and four blocks of 256
// threads spent 2 us of FP64 pipe on that (12.6 us per step at dim 853,776).
inline uint32_t lz_grid(const Ctx* c, uint64_t n) {
  const uint64_t g = (n + 2 * kLzThreads - 1) / (2 * kLzThreads), most = (uint64_t)c->num_sms;
  return (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>({g, most, 1024}));
}
// Norm partials in a context's reduction scratch, past the dot products' share.
inline NormPart lz_norm_part(double* red) { return NormPart{{red + 4096, red + 5120}}; }

// Sq[i*ldS + j] = S[i*ldS + j] * sigma[j] (Ritz coefficients on unnormalised q_j)
__global__ void k_scale_ritz(const double* __restrict__ S, const double* __restrict__ sigma, int m, int k, int ldS,
                             double* __restrict__ Sq, float2* __restrict__ Sqf) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m * k) return;
  int i = t / m, j = t % m;
  double v = S[(size_t)i * ldS + j] * sigma[j];
  Sq[(size_t)i * ldS + j] = v;
  Sqf[(size_t)i * ldS + j] = df_from_double(v);
}

// out = w * inv[slot]
template <class V>
__global__ void k_scale(const V* __restrict__ w, V* __restrict__ out, uint64_t n, Coefs c, int slot) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    typename AccOf<V>::T a{};
    amac(a, c.inv_d, c.inv_f, slot, w[i]);
    out[i] = store_v(a, out);
  }
}

// beta_{j+1} = |w| from its nb partials, and out = w / beta_{j+1} (zeros where
// beta vanished).  Every block sums the partials itself, in the same order, so
// that the step needs no launch for one number; block 0 keeps beta_{j+1}, the
// running scale (slot 1 - ph; every block reads slot ph) and the first
// vanished step.
template <class V>
__global__ void __launch_bounds__(kRedThreads) k_scale_beta(const V* __restrict__ w, V* __restrict__ out, uint64_t n,
                                                            const double* __restrict__ partial, int nb, Coefs c,
                                                            int slot, int ph, double thr) {
  using A = typename AccOf<V>::T;
  using W16 = Vec16<V>;
  using VT = typename W16::T;
  __shared__ A inv_s;
  double tot = 0.0;
  if (threadIdx.x < 32) tot = warp_total(partial, nb, threadIdx.x);
  if (threadIdx.x == 0) {
    double sc = c.scale[ph], beta, inv;
    bool dead;
    lz_beta(tot, sc, thr, beta, inv, dead);
    h_split(inv_s, inv);
    if (blockIdx.x == 0) {
      c.scale[1 - ph] = sc;
      if (dead && *c.exhausted < 0) *c.exhausted = slot;
      c.beta[slot] = beta;
    }
  }
  __syncthreads();
  const A inv = inv_s;
  const uint64_t nv = (n + W16::N - 1) / W16::N;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nv; t += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t e0 = t * W16::N;
    if (e0 + W16::N <= n) {
      const VT q = reinterpret_cast<const VT*>(w)[t];
      VT o{};
#pragma unroll
      for (int i = 0; i < W16::N; ++i) {
        A a{};
        hmac(a, inv, W16::get(q, i));
        W16::set(o, i, store_v(a, out));
      }
      reinterpret_cast<VT*>(out)[t] = o;
    } else {
      for (uint64_t e = e0; e < n; ++e) {
        A a{};
        hmac(a, inv, w[e]);
        out[e] = store_v(a, out);
      }
    }
  }
}

// v *= 1 / ||v|| (inv_d[slot] from OP_NORM_INV), in place.  Ritz vectors
// regenerated from a three-vector recurrence need it: once a converged Ritz
// value has a ghost copy (loss of orthogonality in finite precision, early
// with float vectors) sum_j S_j v_j keeps its direction but not unit norm.
template <class V>
__global__ void k_rescale(V* __restrict__ v, uint64_t n, Coefs c, int slot) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    typename AccOf<V>::T a{};
    amac(a, c.inv_d, c.inv_f, slot, v[i]);
    v[i] = store_v(a, v);
  }
}

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ void set_rand(double& o, float u) { o = (double)u; }
__device__ __forceinline__ void set_rand(float2& o, float u) { o = make_float2(u, 0.f); }
__device__ __forceinline__ void set_rand(float& o, float u) { o = u; }

// Seeded start vector: uniform(-1, 1) from a counter-based hash of (seed, i).
template <class V>
__global__ void k_random(V* __restrict__ v, uint64_t n, uint64_t seed) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t r = mix64(seed * 0x2545f4914f6cdd1dull + i);
    float u = (float)((r >> 40) * (1.0 / 16777216.0)) * 2.f - 1.f;
    set_rand(v[i], u);
  }
}

// out_i (+)= sum_{j<m} S[i*ldS + j] V_j for the eigenvectors i in [i0, i0 + KB),
// i < k: sixteen bytes of each V_j per thread (slots 16-byte aligned), eight in
// flight, the coefficients of 32 vectors at a time in shared memory.  av: every
// output row starts 16-byte aligned, else outputs go element by element.
// (One element per thread and load: 660 us for eight of 22 vectors of the
// N_s = 13 sector from a basis of 40, 1.4 TB/s.)
constexpr int kRitzChunk = 32;
template <class V, int KB>
__global__ void __launch_bounds__(256) k_ritz(const V* __restrict__ Vb, uint64_t stride, int m,
                                              const double* __restrict__ Sd, const float2* __restrict__ Sf, int ldS,
                                              int i0, int k, V* out, uint64_t n, int accumulate, int av) {
  using A = typename AccOf<V>::T;
  using W16 = Vec16<V>;
  using VT = typename W16::T;
  constexpr int N = W16::N;
  __shared__ A cs[kRitzChunk][KB];
  const int kn = min(KB, k - i0);
  const uint64_t nv = (n + N - 1) / N, gs = (uint64_t)gridDim.x * 256;
  const uint64_t rounds = (nv + gs - 1) / gs;   // the same for every thread: barriers inside
  for (uint64_t r = 0; r < rounds; ++r) {
    const uint64_t t = r * gs + (uint64_t)blockIdx.x * 256 + threadIdx.x;
    const bool on = t < nv;
    const bool whole = on && (t + 1) * N <= n;
    A acc[KB][N];
#pragma unroll
    for (int q = 0; q < KB; ++q) {
#pragma unroll
      for (int c = 0; c < N; ++c) acc[q][c] = A{};
      if (accumulate && q < kn && on) {
        const V* o = out + (uint64_t)(i0 + q) * n + t * N;
        if (av && whole) {
          const VT v = *reinterpret_cast<const VT*>(o);
#pragma unroll
          for (int c = 0; c < N; ++c) acc[q][c] = acc_of(W16::get(v, c));
        } else {
#pragma unroll
          for (int c = 0; c < N; ++c)
            if (t * N + c < n) acc[q][c] = acc_of(o[c]);
        }
      }
    }
    for (int j0 = 0; j0 < m; j0 += kRitzChunk) {
      const int jn = min(kRitzChunk, m - j0);
      __syncthreads();
      for (int i = threadIdx.x; i < jn * KB; i += 256) {
        const int j = i / KB, q = i % KB;
        A h{};
        if (q < kn) h_pick(h, Sd, Sf, (size_t)(i0 + q) * ldS + j0 + j);
        cs[j][q] = h;
      }
      __syncthreads();
      if (on) {
        const V* vb = Vb + (uint64_t)j0 * stride;
#pragma unroll 8
        for (int j = 0; j < jn; ++j) {
          VT v;
          if (whole) v = __ldg(reinterpret_cast<const VT*>(vb + (uint64_t)j * stride) + t);
          else v = tile_ld<V>(vb + (uint64_t)j * stride + t * N, 0, (uint32_t)(n - t * N));
#pragma unroll
          for (int q = 0; q < KB; ++q)
#pragma unroll
            for (int c = 0; c < N; ++c) hmac(acc[q][c], cs[j][q], W16::get(v, c));
        }
      }
    }
    if (on) {
#pragma unroll
      for (int q = 0; q < KB; ++q)
        if (q < kn) {
          V* o = out + (uint64_t)(i0 + q) * n + t * N;
          if (av && whole) {
            VT v{};
#pragma unroll
            for (int c = 0; c < N; ++c) W16::set(v, c, store_v(acc[q][c], out));
            *reinterpret_cast<VT*>(o) = v;
          } else {
#pragma unroll
            for (int c = 0; c < N; ++c)
              if (t * N + c < n) o[c] = store_v(acc[q][c], out);
          }
        }
    }
  }
}

// k_ritz over all k outputs, eight, two or one at a time (two double-float or
// FP64 elements of eight outputs fill the registers; a single output should not
// pay for eight).
template <class V>
int ritz(const Ctx* ctx, cudaStream_t st, const V* Vb, uint64_t stride, int m, const double* Sd, const float2* Sf, int ldS,
         int k, V* out, uint64_t n, int accumulate) {
  const uint64_t nv = (n + Vec16<V>::N - 1) / Vec16<V>::N;
  const uint32_t grid = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>((nv + 255) / 256, (uint64_t)ctx->num_sms * 8));
  const int av = (n * sizeof(V)) % 16 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0;
  for (int i0 = 0; i0 < k;) {
    if (k - i0 >= 3) {
      k_ritz<V, 8><<<grid, 256, 0, st>>>(Vb, stride, m, Sd, Sf, ldS, i0, k, out, n, accumulate, av);
      i0 += 8;
    } else if (k - i0 == 2) {
      k_ritz<V, 2><<<grid, 256, 0, st>>>(Vb, stride, m, Sd, Sf, ldS, i0, k, out, n, accumulate, av);
      i0 += 2;
    } else {
      k_ritz<V, 1><<<grid, 256, 0, st>>>(Vb, stride, m, Sd, Sf, ldS, i0, k, out, n, accumulate, av);
      i0 += 1;
    }
  }
  ED_LAUNCH_CHECK();
  return ED_OK;
}

__global__ void k_step_inc(int* step) { *step += 1; }

// ------------------------------------------------ tridiagonal eigensolver
// Eigenpair blockIdx.x (ascending), one warp per pair.
__global__ void __launch_bounds__(32) k_tri_pair(const double* __restrict__ a, const double* __restrict__ b, int m,
                                                 double* __restrict__ theta, double* __restrict__ S, int ldS,
                                                 double* __restrict__ work) {
  extern __shared__ __align__(16) double trish[];
  tri_pair_one(a, b, m, blockIdx.x, theta, S, ldS, work, trish);
}

__global__ void k_tri_finish(const double* __restrict__ theta, int k, int m, double beta_m, double* __restrict__ S,
                             int ldS, float2* __restrict__ Sf, double* __restrict__ resid) {
  tri_finish_block(theta, k, m, beta_m, S, ldS, Sf, resid);
}

// ------------------------------------------------ host-side driver
template <class V>
struct Work {
  Ctx* ctx;
  cudaStream_t st;
  uint64_t n;
  uint32_t grid;
  double* partial;  // ctx->d_red
  Coefs c;
  double* hpart = nullptr;  // projections' partials (reorthogonalised solvers) ...
  int hvecs = kCgsMaxVec;   // ... of this many basis vectors at once
  int ph = 0;               // which slot of c.scale is current
};

template <class V>
int dot_to(Work<V>& W, const V* x, const V* y, int op, int slot) {
  k_dot<V><<<W.grid, kRedThreads, 0, W.st>>>(x, y, W.n, W.partial);
  k_finish<<<1, kRedThreads, 0, W.st>>>(W.partial, (int)W.grid, op, slot, W.c);
  ED_LAUNCH_CHECK();
  return ED_OK;
}

// Full reorthogonalisation of w against the basis vectors [0, nvec), every slot
// and w starting on a 16-byte boundary: twice h = V^T w, w -= V h, with the
// three-term update of lz (if any) ahead of the first projection; W.partial
// gets the cgs_grid() partials of the final <w, w>.  Three launches over the
// basis instead of four: the first update and the second projection share one,
// in which a tile's second read comes from L2 while the blocks' tiles fit it (304
// blocks x 4 KB per vector: 125 MB at 100 vectors); with longer bases that
// launch costs 1.7 to 1.8 sweeps.
template <class V>
int cgs2(Work<V>& W, const V* Vb, uint64_t stride, int nvec, V* w, LzTerm<V> lz = LzTerm<V>()) {
  const uint32_t nb = cgs_grid<V>(W.ctx, W.n);
  const LzTerm<V> none;
  auto finish = [&](int k0, int kn) {
    k_finish<<<kn, kRedThreads, 0, W.st>>>(W.hpart, (int)nb, OP_NEGH, k0, W.c);
  };
  auto dots = [&](int k0, int kn, int rev, const LzTerm<V>& t) {
    k_cgs<V, false, true><<<nb, kCgsThreads, cgs_smem<V>(kn, false, true), W.st>>>(
        Vb + (uint64_t)k0 * stride, stride, kn, w, W.n, rev, nullptr, nullptr, W.hpart, nullptr, t);
    finish(k0, kn);
  };
  auto update = [&](int k0, int kn, int rev) {
    k_cgs<V, true, false><<<nb, kCgsThreads, cgs_smem<V>(kn, true, false), W.st>>>(
        Vb + (uint64_t)k0 * stride, stride, kn, w, W.n, rev, W.c.h_d + k0, W.c.h_f + k0, nullptr, W.partial, none);
  };
  if (nvec <= W.hvecs) {
    dots(0, nvec, 0, lz);
    k_cgs<V, true, true><<<nb, kCgsThreads, cgs_smem<V>(nvec, true, true), W.st>>>(
        Vb, stride, nvec, w, W.n, 1, W.c.h_d, W.c.h_f, W.hpart, nullptr, none);
    finish(0, nvec);
    update(0, nvec, 0);
  } else {   // more vectors than a block's shared memory, or the partials' place, serves at once: range by range
    for (int pass = 0; pass < 2; ++pass) {
      for (int k0 = 0; k0 < nvec; k0 += W.hvecs)
        dots(k0, std::min(W.hvecs, nvec - k0), 0, pass == 0 && k0 == 0 ? lz : none);
      for (int k0 = 0; k0 < nvec; k0 += W.hvecs) update(k0, std::min(W.hvecs, nvec - k0), 0);
    }
  }
  ED_LAUNCH_CHECK();
  return ED_OK;
}

// H v_j with the partials of <v_j, H v_j> in W.partial; *np of them.
template <class V>
int apply_dot(const Sector* s, Work<V>& W, const V* x, V* y, int* np) {
  if (has_rows(s)) return apply_fast(s, x, y, W.st, W.partial, np);
  ED_TRY(apply_h(s, x, y, W.st));
  k_dot<V><<<W.grid, kRedThreads, 0, W.st>>>(x, y, W.n, W.partial);
  ED_LAUNCH_CHECK();
  *np = (int)W.grid;
  return ED_OK;
}

// One reorthogonalised Lanczos step: w = H v, the three-term update (with vp
// unless NULL), CGS2 against [0, j], beta_{j+1} and v_{j+1} = w / beta_{j+1}.
// e0, e1 bracket the H*v.
template <class V>
int lanczos_step(const Sector* s, Work<V>& W, const V* Vb, uint64_t ld, int j, const V* vp, V* w, V* vnext, double thr,
                 cudaEvent_t e0, cudaEvent_t e1) {
  const V* vj = Vb + (uint64_t)j * ld;
  int np = 0;
  ED_TRY_CUDA(cudaEventRecord(e0, W.st));
  ED_TRY(apply_dot(s, W, vj, w, &np));
  ED_TRY_CUDA(cudaEventRecord(e1, W.st));
  LzTerm<V> lz;
  lz.v = vj;
  lz.vp = vp;
  lz.apart = W.partial;
  lz.na = np;
  lz.alpha = W.c.alpha + j;
  lz.beta = W.c.beta + j;
  lz.scale = W.c.scale + W.ph;
  ED_TRY(cgs2(W, Vb, ld, j + 1, w, lz));
  const uint32_t grid =
      (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>((W.n / Vec16<V>::N + 255) / 256, (uint64_t)W.ctx->num_sms * 4));
  k_scale_beta<V><<<grid, kRedThreads, 0, W.st>>>(w, vnext, W.n, W.partial, (int)cgs_grid<V>(W.ctx, W.n), W.c, j + 1,
                                                 W.ph, thr);
  ED_LAUNCH_CHECK();
  W.ph ^= 1;
  return ED_OK;
}

struct DevBuf {
  Ctx* ctx = nullptr;
  void* p = nullptr;
  size_t bytes = 0;
  int alloc(Ctx* c, size_t b) {
    ctx = c;
    bytes = b ? b : 1;
    return dev_alloc(c, &p, bytes);
  }
  ~DevBuf() {
    if (p) dev_free(ctx, p, bytes);
  }
};

// Room for the projections' partials of a basis of mmax + 1 vectors.  Where the
// budget has none beside the basis, the upper half of the context's reduction
// scratch takes those of a few vectors at a time (four sweeps instead of three).
template <class V>
int cgs_room(Work<V>& W, DevBuf& buf, int mmax) {
  const size_t nb = cgs_grid<V>(W.ctx, W.n);
  W.hvecs = kCgsMaxVec;
  const int st = buf.alloc(W.ctx, (size_t)std::min(mmax + 1, kCgsMaxVec) * nb * sizeof(double));
  W.hpart = static_cast<double*>(buf.p);
  if (st != ED_ERR_OOM) return st;
  set_error("");
  W.hpart = W.partial + kRedSlots / 2;
  W.hvecs = (int)std::max<size_t>(1, kRedSlots / 2 / nb);
  return ED_OK;
}

// Carves typed arrays out of one allocation (256-byte aligned).
struct Carve {
  char* base;
  size_t off = 0;
  template <class T>
  T* take(size_t n) {
    off = (off + 255) & ~(size_t)255;
    T* p = reinterpret_cast<T*>(base + off);
    off += n * sizeof(T);
    return p;
  }
};

size_t coef_bytes(int mmax, int k) {
  size_t m2 = (size_t)mmax + 2;
  return 256 * 64 + m2 * 8 * 24 + (size_t)k * m2 * 8 * 10 + 4096;
}

Coefs carve_coefs(Carve& cv, int mmax) {
  Coefs c;
  size_t m2 = (size_t)mmax + 2;
  c.alpha = cv.take<double>(m2);
  c.beta = cv.take<double>(m2);
  c.inv_d = cv.take<double>(m2);
  c.inv_f = cv.take<float2>(m2);
  c.h_d = cv.take<double>(m2);
  c.h_f = cv.take<float2>(m2);
  c.scale = cv.take<double>(2);
  c.exhausted = cv.take<int>(1);
  c.out = cv.take<double>(64);
  c.sigma = cv.take<double>(m2);
  c.ua_d = cv.take<double>(m2);
  c.ua_f = cv.take<float2>(m2);
  c.ub_d = cv.take<double>(m2);
  c.ub_f = cv.take<float2>(m2);
  c.uc_d = cv.take<double>(m2);
  c.uc_f = cv.take<float2>(m2);
  c.step = cv.take<int>(1);
  return c;
}

__global__ void k_init_coefs(Coefs c, int m2) {
  for (int i = threadIdx.x; i < m2; i += blockDim.x) {
    c.alpha[i] = 0;
    c.beta[i] = 0;
    c.inv_d[i] = 0;
    c.inv_f[i] = make_float2(0, 0);
    c.h_d[i] = 0;
    c.h_f[i] = make_float2(0, 0);
    c.sigma[i] = 0;
    c.ua_d[i] = c.ub_d[i] = c.uc_d[i] = 0;
    c.ua_f[i] = c.ub_f[i] = c.uc_f[i] = make_float2(0, 0);
  }
  if (threadIdx.x == 0) {
    c.scale[0] = c.scale[1] = 0.0;
    *c.exhausted = -1;
    *c.step = 0;
  }
}

// Solve the m x m tridiagonal problem for its k lowest pairs.
int tridiag(Ctx* ctx, cudaStream_t st, const Coefs& c, int m, int k, double beta_m, double* theta,
            double* S, float2* Sf, int ldS, double* resid, double* work) {
  k_tri_pair<<<k, 32, tri_smem(m), st>>>(c.alpha, c.beta, m, theta, S, ldS, work);
  k_tri_finish<<<1, 128, 0, st>>>(theta, k, m, beta_m, S, ldS, Sf, resid);
  ED_LAUNCH_CHECK();
  (void)ctx;
  return ED_OK;
}

template <class V>
int lanczos_impl(Sector* s, const ed_lanczos_opts* o, double* evals, void* evecs, ed_lanczos_info* info,
                 cudaStream_t st) {
  auto t_start = std::chrono::steady_clock::now();
  Ctx* ctx = s->ctx;
  const uint64_t n = s->dim;
  const int k = o->k;
  int mmax = (int)std::min<uint64_t>((uint64_t)o->max_iter, n);
  if (mmax < 1) mmax = 1;
  const int check_every = std::max(1, o->check_every);
  const int kk = std::min<int>(k, (int)n);

  // workspace: basis of mmax + 1 vectors, w
  size_t eb = sizeof(V);
  const int nvec_store = mmax + 1;
  DevBuf vb, cb, hb;
  // basis slots padded to 32 elements, so that each starts 16-byte aligned
  const uint64_t ld = pad32(n);
  ED_TRY(vb.alloc(ctx, ((size_t)nvec_store + 1) * ld * eb));
  ED_TRY(cb.alloc(ctx, coef_bytes(mmax, std::max(kk, 1))));
  V* Vbase = static_cast<V*>(vb.p);
  V* w = Vbase + (size_t)nvec_store * ld;
  Carve cv{static_cast<char*>(cb.p)};
  Coefs c = carve_coefs(cv, mmax);
  int ldS = mmax + 1;
  double* theta = cv.take<double>(ED_MAX_K);
  double* resid = cv.take<double>(ED_MAX_K);
  double* Sd = cv.take<double>((size_t)ldS * std::max(kk, 1));
  float2* Sf = cv.take<float2>((size_t)ldS * std::max(kk, 1));
  double* twork = cv.take<double>((size_t)6 * ldS * std::max(kk, 1));

  Work<V> W;
  W.ctx = ctx;
  W.st = st;
  W.n = n;
  W.grid = (uint32_t)std::min<uint64_t>((n + kRedThreads - 1) / kRedThreads, (uint64_t)ctx->num_sms * 8);
  if (W.grid == 0) W.grid = 1;
  W.partial = ctx->d_red;
  W.c = c;
  ED_TRY(cgs_room(W, hb, mmax));
  uint32_t vgrid = (uint32_t)std::min<uint64_t>((n + 255) / 256, (uint64_t)ctx->num_sms * 16);
  if (vgrid == 0) vgrid = 1;

  k_init_coefs<<<1, 256, 0, st>>>(c, mmax + 2);
  auto vec = [&](int j) -> V* { return Vbase + (size_t)j * ld; };

  // start vector
  if (o->v0) {
    ED_TRY_CUDA(cudaMemcpyAsync(w, o->v0, n * eb, cudaMemcpyDeviceToDevice, st));
  } else {
    k_random<V><<<vgrid, 256, 0, st>>>(w, n, o->seed);
  }
  ED_TRY(dot_to(W, (const V*)w, (const V*)w, OP_NORM_INV, 0));
  k_scale<V><<<vgrid, 256, 0, st>>>(w, vec(0), n, c, 0);
  ED_LAUNCH_CHECK();

  // one event pair per step to time the H*v launches
  std::vector<cudaEvent_t> evs(2 * (size_t)mmax);
  for (auto& e : evs) ED_TRY_CUDA(cudaEventCreate(&e));
  struct EvGuard {
    std::vector<cudaEvent_t>* v;
    ~EvGuard() {
      for (auto e : *v) cudaEventDestroy(e);
    }
  } evguard{&evs};
  double apply_ms = 0.0;
  int n_timed = 0;

  std::vector<double> h_theta(ED_MAX_K), h_res(ED_MAX_K);
  int m = 0;          // current Krylov dimension
  int n_conv = 0;
  double beta_last = 0.0;
  bool done = false;
  int status = ED_OK;
  int restarts = 0;
  const double thr = 1e-13;
  int j = 0;
  bool exhausted = false;
  while (!done) {
    exhausted = false;
    for (; j < mmax; ++j) {
      ED_TRY(lanczos_step(s, W, (const V*)Vbase, ld, j, j > 0 ? vec(j - 1) : nullptr, w, vec(j + 1), thr, evs[2 * j],
                          evs[2 * j + 1]));
      n_timed = std::max(n_timed, j + 1);
      m = j + 1;
      bool check = ((m % check_every) == 0) || (m == mmax) || (n <= 4096);
      if (!check) continue;
      // exhausted Krylov space?
      int ex = -1;
      ED_TRY_CUDA(cudaMemcpyAsync(ctx->h_red, c.exhausted, sizeof(int), cudaMemcpyDeviceToHost, st));
      ED_TRY_CUDA(cudaStreamSynchronize(st));
      std::memcpy(&ex, ctx->h_red, sizeof(int));
      if (ex >= 0) {
        m = ex;  // T is complete up to here; later steps are discarded
        exhausted = true;
        ++j;
        break;
      }
      int kc = std::min(kk, m);
      ED_TRY(tridiag(ctx, st, c, m, kc, 0.0, theta, Sd, Sf, ldS, resid, twork));
      // residuals use beta_{m}
      ED_TRY_CUDA(cudaMemcpyAsync(ctx->h_red, c.beta + m, sizeof(double), cudaMemcpyDeviceToHost, st));
      ED_TRY_CUDA(cudaMemcpyAsync(ctx->h_red + 1, theta, kc * sizeof(double), cudaMemcpyDeviceToHost, st));
      ED_TRY_CUDA(cudaStreamSynchronize(st));
      beta_last = ctx->h_red[0];
      std::memcpy(h_theta.data(), ctx->h_red + 1, kc * sizeof(double));
      // residual = beta_m * |last component|
      std::vector<double> last(kc);
      for (int i = 0; i < kc; ++i)
        ED_TRY_CUDA(cudaMemcpyAsync(&last[i], Sd + (size_t)i * ldS + m - 1, sizeof(double),
                                    cudaMemcpyDeviceToHost, st));
      ED_TRY_CUDA(cudaStreamSynchronize(st));
      n_conv = 0;
      for (int i = 0; i < kc; ++i) {
        h_res[i] = std::fabs(beta_last * last[i]);
        if (h_res[i] <= o->tol * std::max(1.0, std::fabs(h_theta[i])) && n_conv == i) ++n_conv;
      }
      if (kc >= kk && n_conv >= kk) {
        ++j;
        done = true;
        break;
      }
    }
    if (done) break;
    if (!exhausted && j >= mmax && m >= mmax) {
      status = ED_ERR_NOT_CONVERGED;
      break;
    }
    // Krylov space exhausted at m: finished if it spans the sector or we have
    // k values already; otherwise restart from a fresh orthogonal vector.
    {
      int kc = std::min(kk, m);
      ED_TRY(tridiag(ctx, st, c, m, kc, 0.0, theta, Sd, Sf, ldS, resid, twork));
      ED_TRY_CUDA(cudaMemcpyAsync(ctx->h_red, theta, kc * sizeof(double), cudaMemcpyDeviceToHost, st));
      ED_TRY_CUDA(cudaStreamSynchronize(st));
      std::memcpy(h_theta.data(), ctx->h_red, kc * sizeof(double));
      for (int i = 0; i < kc; ++i) h_res[i] = 0.0;
      n_conv = kc;
      beta_last = 0.0;
      if ((uint64_t)m >= n || m >= mmax || kc >= kk) {
        done = true;
        break;
      }
      // new random direction, orthogonalised against V[0..m)
      ++restarts;
      k_random<V><<<vgrid, 256, 0, st>>>(w, n, o->seed + 7919ull * restarts);
      ED_TRY(cgs2(W, (const V*)Vbase, ld, m, w));
      k_finish<<<1, kRedThreads, 0, st>>>(W.partial, (int)cgs_grid<V>(ctx, n), OP_NORM_INV, 1, c);
      k_scale<V><<<vgrid, 256, 0, st>>>(w, vec(m), n, c, 1);
      // beta[m] = 0 splits T; reset the exhaustion flag
      double zero = 0.0;
      int neg = -1;
      ED_TRY_CUDA(cudaMemcpyAsync(c.beta + m, &zero, sizeof(double), cudaMemcpyHostToDevice, st));
      ED_TRY_CUDA(cudaMemcpyAsync(c.exhausted, &neg, sizeof(int), cudaMemcpyHostToDevice, st));
      ED_TRY_CUDA(cudaStreamSynchronize(st));
      j = m;
    }
  }

  int kc = std::min(kk, m);
  for (int i = 0; i < kc; ++i) evals[i] = h_theta[i];
  for (int i = kc; i < k; ++i) evals[i] = NAN;
  if (info) {
    info->iters = m;
    info->n_converged = std::min(n_conv, kc);
    for (int i = 0; i < ED_MAX_K; ++i) info->residual[i] = (i < kc) ? h_res[i] : 0.0;
  }
  if (evecs && kc > 0) {
    // S for the final m
    ED_TRY(tridiag(ctx, st, c, m, kc, 0.0, theta, Sd, Sf, ldS, resid, twork));
    V* out = static_cast<V*>(evecs);
    ED_TRY(ritz(ctx, st, (const V*)Vbase, ld, m, Sd, Sf, ldS, kc, out, n, 0));
  }
  ED_TRY_CUDA(cudaStreamSynchronize(st));
  for (int q = 0; q < n_timed; ++q) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, evs[2 * q], evs[2 * q + 1]) == cudaSuccess) apply_ms += ms;
  }
  if (info) info->apply_ms = apply_ms;
  if (info)
    info->total_ms =
        std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_start).count();
  if (status != ED_OK) set_error("Lanczos did not converge in %d steps", mmax);
  return status;
}

}  // namespace

}  // namespace ed
