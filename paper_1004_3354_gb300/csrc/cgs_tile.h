// Classical Gram-Schmidt against a stored basis, tile by tile (internal
// header): the kernels of the full reorthogonalisation in ed_lanczos and
// ed_lanczos_tr.  Each translation unit gets its own copy.
//
// A tile is E = 32 * NV * N consecutive elements of every basis vector (N
// elements per sixteen bytes, NV vectors of sixteen bytes per lane: 512
// double-float or FP64 elements, 1024 floats).  A block of eight warps takes a
// tile through two phases:
//   owner phase  thread t owns the sixteen bytes t of the tile: the
//                recurrence's three-term update, or w += sum_k h_k V_k over all
//                k (coalesced, eight loads in flight), then the tile of the new
//                w goes to global and shared memory;
//   dot phase    warp i takes the vectors i, i + 8, ...: each lane holds its
//                part of the w tile in registers and sums products with V_k;
//                eight vectors are reduced together by a halving butterfly (9
//                exchanges instead of 40), and the block's sum per vector is
//                kept in shared memory over all its tiles.
// The work per vector and tile is one pass over 4 KB per warp, so nothing
// depends on how many vectors there are: one launch covers a whole projection
// where a launch per eight vectors over the whole grid left 3 elements per
// thread at dim 853,776.
#pragma once

#include "ed_internal.h"
#include "vec_ops.h"

namespace ed {

namespace {

constexpr int kCgsThreads = 256;
constexpr int kCgsWarps = kCgsThreads / 32;
constexpr int kCgsMaxVec = 2048;   // basis vectors of one launch (shared-memory coefficients and sums)

template <class V>
struct CgsTile {
  static constexpr int N = Vec16<V>::N;
  static constexpr int NV = kCgsThreads / 32;          // sixteen-byte vectors per lane
  static constexpr uint32_t E = 32 * NV * N;           // elements per tile
};

__device__ __forceinline__ void h_split(double& o, double h) { o = h; }
__device__ __forceinline__ void h_split(float2& o, double h) { o = df_from_double(h); }

// coefficient k in the accumulator's format, from its double or double-float copy
__device__ __forceinline__ void h_pick(double& o, const double* d, const float2*, size_t k) { o = d[k]; }
__device__ __forceinline__ void h_pick(float2& o, const double*, const float2* f, size_t k) { o = f[k]; }

// a += h * x, h in the accumulator's format
__device__ __forceinline__ void hmac(double& a, double h, double x) { a = fma(h, x, a); }
__device__ __forceinline__ void hmac(float2& a, float2 h, float2 x) { df_mac(a, h, x); }
__device__ __forceinline__ void hmac(float2& a, float2 h, float x) { df_mac1(a, h, x); }

// Sixteen bytes at vector index iv of a tile with `lim` valid elements; the
// elements past it read as zero (a slot's padding holds no defined values).
// RO: through the read-only path (not for w, which the kernel writes).
template <class V, bool RO = true>
__device__ __forceinline__ typename Vec16<V>::T tile_ld(const V* p, uint32_t iv, uint32_t lim) {
  using W16 = Vec16<V>;
  constexpr uint32_t N = W16::N;
  typename W16::T o{};
  if ((iv + 1) * N <= lim) {
    const typename W16::T* q = reinterpret_cast<const typename W16::T*>(p) + iv;
    o = RO ? __ldg(q) : *q;
  } else {
#pragma unroll
    for (uint32_t c = 0; c < N; ++c)
      if (iv * N + c < lim) W16::set(o, c, p[iv * N + c]);
  }
  return o;
}

// Sums over the warp of eight accumulators: lane l ends with the sum of
// accumulator cgs_q(l).
__device__ __forceinline__ int cgs_q(int lane) { return ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1); }

template <class A>
__device__ __forceinline__ A warp_sum8(A (&a)[8], int lane) {
#pragma unroll
  for (int h = 4; h >= 1; h >>= 1) {
    const int o = 4 * h;   // 16, 8, 4
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const A give = up ? a[i] : a[i + h], keep = up ? a[i + h] : a[i];
      a[i] = add_acc(keep, shfl_x(give, o));
    }
  }
  A v = a[0];
  v = add_acc(v, shfl_x(v, 2));
  return add_acc(v, shfl_x(v, 1));
}

// The dot phase: <V_k, wt> over one tile for the vectors k = warp, warp + 8,
// ... < nvec, added to hsum[k] (each k belongs to one warp).
template <class V, class A>
__device__ __forceinline__ void tile_dots(const V* __restrict__ vt, uint64_t stride, int nvec, const V* wt, uint32_t lim,
                                          A* hsum) {
  using W16 = Vec16<V>;
  using VT = typename W16::T;
  constexpr int N = W16::N, NV = CgsTile<V>::NV;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  VT wq[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) wq[i] = reinterpret_cast<const VT*>(wt)[i * 32 + lane];
  const bool full = lim == CgsTile<V>::E;
  for (int k0 = warp; k0 < nvec; k0 += 8 * kCgsWarps) {
    A acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      acc[q] = A{};
      const int k = k0 + q * kCgsWarps;
      if (k < nvec) {
        const V* vk = vt + (uint64_t)k * stride;
        VT v[NV];
        if (full) {
#pragma unroll
          for (int i = 0; i < NV; ++i) v[i] = __ldg(reinterpret_cast<const VT*>(vk) + i * 32 + lane);
#pragma unroll
          for (int i = 0; i < NV; ++i)
#pragma unroll
            for (int c = 0; c < N; ++c) dmac(acc[q], W16::get(v[i], c), W16::get(wq[i], c));
        } else {
#pragma unroll
          for (int i = 0; i < NV; ++i)
            if ((uint32_t)i * 32 * N < lim) v[i] = tile_ld(vk, i * 32 + lane, lim);
#pragma unroll
          for (int i = 0; i < NV; ++i)
            if ((uint32_t)i * 32 * N < lim) {
#pragma unroll
              for (int c = 0; c < N; ++c) dmac(acc[q], W16::get(v[i], c), W16::get(wq[i], c));
            }
        }
      }
    }
    const A s = warp_sum8(acc, lane);
    const int k = k0 + cgs_q(lane) * kCgsWarps;
    if ((lane & 3) == 0 && k < nvec) hsum[k] = add_acc(hsum[k], s);
  }
}

// Sum of nb doubles by one warp, the same in every lane.  Four sums per lane: a
// dependent FP64 addition takes about 100 cycles, and more warps would fill the
// FP64 pipe (20 cycles per warp instruction and SM) instead.
__device__ __forceinline__ double warp_total(const double* __restrict__ p, int nb, int lane) {
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (int i = lane; i < nb; i += 128) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i + 32 * q < nb) v[q] += p[i + 32 * q];
  }
  double s = (v[0] + v[1]) + (v[2] + v[3]);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Three-term update w -= alpha_j v_j + beta_j v_{j-1} ahead of the first
// projection, with alpha_j = the sum of the na partials of <v_j, H v_j>.
template <class V>
struct LzTerm {
  const V* v = nullptr;        // NULL: no three-term update
  const V* vp = nullptr;       // NULL: no v_{j-1} term
  const double* apart = nullptr;
  int na = 0;
  double* alpha = nullptr;     // alpha_j, written by block 0
  const double* beta = nullptr;
  double* scale = nullptr;     // running maximum of |alpha|, beta
};

// One tile (lim elements at w0, the same elements of the basis at vt).  UPD: w
// += sum_k hs_k V_k (hs: the negated projections); else with lv != NULL the
// three-term update w += na lv + nb lvp.  DOT: <V_k, w> of the updated w added
// to hsum[k], through the tile buffer wb (the caller alternates two: a warp
// still reading one tile's buffer holds the barrier of the next tile, past
// which the buffer is written again).  UPD without DOT: nacc += <w, w>.
template <class V, bool UPD, bool DOT, class A>
__device__ __forceinline__ void cgs_tile(const V* __restrict__ vt, uint64_t stride, int nvec, V* w0, uint32_t lim,
                                         const A* hs, A* hsum, V* wb, const V* __restrict__ lv,
                                         const V* __restrict__ lvp, A na, A nb, A& nacc) {
  using W16 = Vec16<V>;
  using VT = typename W16::T;
  constexpr int N = W16::N;
  const uint32_t t = threadIdx.x;
  VT wv{};
  if (t * N < lim) {
    wv = tile_ld<V, false>(w0, t, lim);
    if (UPD || lv) {
      A a[N];
#pragma unroll
      for (int c = 0; c < N; ++c) a[c] = acc_of(W16::get(wv, c));
      if (UPD) {
        if ((t + 1) * N <= lim) {
          const VT* vp = reinterpret_cast<const VT*>(vt) + t;
          const uint64_t sv = stride / N;
          int k = 0;
          for (; k + 8 <= nvec; k += 8) {
            VT v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = __ldg(vp + (uint64_t)(k + q) * sv);
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
              for (int c = 0; c < N; ++c) hmac(a[c], hs[k + q], W16::get(v[q], c));
          }
          for (; k < nvec; ++k) {
            const VT v = __ldg(vp + (uint64_t)k * sv);
#pragma unroll
            for (int c = 0; c < N; ++c) hmac(a[c], hs[k], W16::get(v, c));
          }
        } else {
          for (int k = 0; k < nvec; ++k) {
            const VT v = tile_ld<V>(vt + (uint64_t)k * stride, t, lim);
#pragma unroll
            for (int c = 0; c < N; ++c) hmac(a[c], hs[k], W16::get(v, c));
          }
        }
      } else {
        const VT v = tile_ld<V>(lv, t, lim);
#pragma unroll
        for (int c = 0; c < N; ++c) hmac(a[c], na, W16::get(v, c));
        if (lvp) {
          const VT u = tile_ld<V>(lvp, t, lim);
#pragma unroll
          for (int c = 0; c < N; ++c) hmac(a[c], nb, W16::get(u, c));
        }
      }
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const V o = store_v(a[c], w0);
        W16::set(wv, c, o);
        if (UPD && !DOT && t * N + c < lim) dmac(nacc, o, o);
      }
      if ((t + 1) * N <= lim) {
        reinterpret_cast<VT*>(w0)[t] = wv;
      } else {
#pragma unroll
        for (int c = 0; c < N; ++c)
          if (t * N + c < lim) w0[t * N + c] = W16::get(wv, c);
      }
    }
  }
  if (DOT) {
    reinterpret_cast<VT*>(wb)[t] = wv;
    __syncthreads();
    tile_dots<V, A>(vt, stride, nvec, wb, lim, hsum);
  }
}

// The projection of one vector: UPD, DOT and LzTerm as in cgs_tile, with the
// negated projections h; DOT writes the partials hpart[k * gridDim.x + b] of
// <V_k, w>, UPD without DOT the partials npart[b] of <w, w>.  rev walks the
// tiles from the last one, so that a kernel starts on what the one before it
// left in L2.
template <class V, bool UPD, bool DOT>
__global__ void __launch_bounds__(kCgsThreads, 2) k_cgs(const V* __restrict__ Vb, uint64_t stride, int nvec,
                                                        V* __restrict__ w, uint64_t n, int rev,
                                                        const double* __restrict__ h, const float2* __restrict__ hf,
                                                        double* __restrict__ hpart, double* __restrict__ npart,
                                                        LzTerm<V> lz) {
  using A = typename AccOf<V>::T;
  constexpr uint32_t E = CgsTile<V>::E;
  extern __shared__ __align__(16) unsigned char sm[];
  V* wt = reinterpret_cast<V*>(sm);                                   // two tiles of w
  A* hs = reinterpret_cast<A*>(sm + (DOT ? 2 * E * sizeof(V) : 0));   // coefficients (UPD)
  A* hsum = hs + (UPD ? nvec : 0);                                    // the block's sums (DOT)
  __shared__ A sha[32];
  const uint32_t t = threadIdx.x;
  if (lz.v) {
    double al = 0.0;
    if (t < 32) al = warp_total(lz.apart, lz.na, t);
    if (t == 0) {
      h_split(sha[0], -al);
      h_split(sha[1], lz.vp ? -*lz.beta : 0.0);
      if (blockIdx.x == 0) {
        *lz.alpha = al;
        *lz.scale = fmax(*lz.scale, fabs(al));
      }
    }
  }
  if (UPD)
    for (int k = t; k < nvec; k += kCgsThreads) h_pick(hs[k], h, hf, k);
  if (DOT)
    for (int k = t; k < nvec; k += kCgsThreads) hsum[k] = A{};
  __syncthreads();
  A na{}, nb{};   // -alpha_j, -beta_j
  if (lz.v) na = sha[0], nb = sha[1];
  A nacc{};
  const uint32_t tiles = (uint32_t)((n + E - 1) / E);
  int buf = 0;
  for (uint32_t ti = blockIdx.x; ti < tiles; ti += gridDim.x, buf ^= 1) {
    const uint64_t e0 = (uint64_t)(rev ? tiles - 1 - ti : ti) * E;
    const uint32_t lim = (uint32_t)(n - e0 < E ? n - e0 : E);
    cgs_tile<V, UPD, DOT, A>(Vb + e0, stride, nvec, w + e0, lim, hs, hsum, wt + buf * E, lz.v ? lz.v + e0 : nullptr,
                             lz.vp ? lz.vp + e0 : nullptr, na, nb, nacc);
  }
  if (DOT) {
    __syncthreads();
    for (int k = t; k < nvec; k += kCgsThreads) hpart[(uint64_t)k * gridDim.x + blockIdx.x] = to_d(hsum[k]);
  }
  if (UPD && !DOT) {
    nacc = block_reduce(nacc, sha);
    if (t == 0) npart[blockIdx.x] = to_d(nacc);
  }
}

template <class V>
size_t cgs_smem(int nvec, bool upd, bool dot) {
  const size_t ab = sizeof(typename AccOf<V>::T);
  return (dot ? 2 * (size_t)CgsTile<V>::E * sizeof(V) : 0) + (size_t)nvec * ab * ((upd ? 1 : 0) + (dot ? 1 : 0)) + 16;
}

// Blocks of a projection over n elements: two per SM (the kernels' register
// budget), no more than there are tiles.
template <class V>
uint32_t cgs_grid(const Ctx* c, uint64_t n) {
  const uint64_t tiles = (n + CgsTile<V>::E - 1) / CgsTile<V>::E;
  const uint64_t g = (uint64_t)c->num_sms * 2;
  return (uint32_t)(tiles < g ? (tiles ? tiles : 1) : g);
}

}  // namespace

}  // namespace ed
