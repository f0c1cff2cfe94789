// The separable nonlocal potential, Z += alpha C~ P with P = h (C~^H X): one pair of kernels for
// FP64, FP32 and complex blocks.
//
// The term reads, per projector, one row of X for each node of its support: the gathered rows bound
// it (FP32; in FP64 the pipe), and an atom's angular channels share one node list.  So projectors
// are taken in groups of up to four that follow one another with the same list (found when they are
// set): each row is read once for the group.  A group's support is split over the eight CTAs of a
// cluster, whose partial sums meet through distributed shared memory, in order: no workspace and no
// second launch.  Nodes and weights are staged in shared memory first; with them in the loop's
// chain of loads the grouped form took 88 us where the staged one takes 40 (27 atoms, 128 FP32
// columns, 885k DoFs; 57 us with one projector per CTA and a reduction launch).  64 complex64
// columns of 16 atoms at 176k DoFs: 26 us against 43; one FP64 column of one atom: 10.4 us against
// 23.5, and 4 against 18 for the update below, whose lanes no longer idle.  100 FP64 columns of 6
// atoms at 109k DoFs: coefficients and update 99 us against 104, on the FP64 pipe.
//
// X, Z and P are written by kernels that may still run when a CTA is placed (launch_after): plain loads,
// no __restrict__.  The tables were complete before.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "internal.h"

namespace dftfe {
namespace nl {

constexpr int kSplits = 8;   // CTAs of a cluster (the portable size), each one range of a support
constexpr int kWarps = 16, kChunk = 512;

// what a lane holds (V), how it is loaded, weighted and stored
struct F64 {
  using E = double; using V = double; using W = double; using S = double;
  static constexpr int kCols = 1, kLanes = 16;
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ V load(const E* p) { return *p; }
  static __device__ __forceinline__ void mad(V& s, W w, V x) { s = fma(w, x, s); }
  static __device__ __forceinline__ void add(V& s, V x) { s += x; }
  static __device__ __forceinline__ void madn(V& s, W w, V x) { s = fma(w, x, s); }
  static __device__ __forceinline__ V shfl(V x, int o) { return __shfl_xor_sync(~0u, x, o); }
  static __device__ __forceinline__ void store(E* p, double h, V x, int) { *p = h * x; }
  static __device__ __forceinline__ void update(E* p, double alpha, V x, V z, int) { *p = fma(alpha, x, z); }
};
// four columns per lane; X rows are padded to 32 columns, so the load stays inside.  Weights are
// narrowed once per entry (a conversion from FP64 costs a warp as much as 32 FP32 FMAs).
struct F32x4 {
  using E = float; using V = float4; using W = double; using S = float;
  static constexpr int kCols = 4, kLanes = 32;
  static __device__ __forceinline__ V zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ V load(const E* p) { return *reinterpret_cast<const float4*>(p); }
  static __device__ __forceinline__ void mad(V& s, S w, V x) {
    s.x = fmaf(w, x.x, s.x); s.y = fmaf(w, x.y, s.y); s.z = fmaf(w, x.z, s.z); s.w = fmaf(w, x.w, s.w);
  }
  static __device__ __forceinline__ void add(V& s, V x) { s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w; }
  static __device__ __forceinline__ void store(E* p, double h, V x, int left) {
    const float f = (float)h, v[4] = {f * x.x, f * x.y, f * x.z, f * x.w};
    for (int j = 0; j < 4; ++j)
      if (j < left) p[j] = v[j];
  }
  static __device__ __forceinline__ void madn(V& s, S w, V x) { mad(s, w, x); }
  static __device__ __forceinline__ void update(E* p, double alpha, V x, V z, int left) {
    const float a = (float)alpha;
    z.x = fmaf(a, x.x, z.x); z.y = fmaf(a, x.y, z.y); z.z = fmaf(a, x.z, z.z); z.w = fmaf(a, x.w, z.w);
    if (left >= 4) {
      *reinterpret_cast<float4*>(p) = z;
    } else {
      const float v[4] = {z.x, z.y, z.z, z.w};
      for (int j = 0; j < left; ++j) p[j] = v[j];
    }
  }
};
template <typename C>
struct Cplx {   // mad: conj(weight) x, madn: weight x
  using E = C; using V = C; using W = C; using S = C; using R = decltype(C::x);
  static constexpr int kCols = 1, kLanes = sizeof(R) == 8 ? 16 : 32;
  static __device__ __forceinline__ V zero() { V v; v.x = 0; v.y = 0; return v; }
  static __device__ __forceinline__ V load(const E* p) { return *p; }
  static __device__ __forceinline__ void mad(V& s, W w, V x) {
    s.x = fma(w.x, x.x, fma(w.y, x.y, s.x));
    s.y = fma(w.x, x.y, fma(-w.y, x.x, s.y));
  }
  static __device__ __forceinline__ void add(V& s, V x) { s.x += x.x; s.y += x.y; }
  static __device__ __forceinline__ V shfl(V x, int o) {
    x.x = __shfl_xor_sync(~0u, x.x, o);
    x.y = __shfl_xor_sync(~0u, x.y, o);
    return x;
  }
  static __device__ __forceinline__ void store(E* p, double h, V x, int) {
    x.x *= (R)h; x.y *= (R)h;
    *p = x;
  }
  static __device__ __forceinline__ void madn(V& s, W w, V x) {
    s.x = fma(w.x, x.x, fma(-w.y, x.y, s.x));
    s.y = fma(w.x, x.y, fma(w.y, x.x, s.y));
  }
  static __device__ __forceinline__ void update(E* p, double alpha, V x, V z, int) {
    z.x = fma((R)alpha, x.x, z.x);
    z.y = fma((R)alpha, x.y, z.y);
    *p = z;
  }
};

// sums of G projectors over `len` staged entries of their common support: LC lanes side by side over
// columns, 32 / LC entries at a time per warp.  Nodes and weights are in shared memory, so the
// rows are the only loads and eight of them are in flight per lane.
template <class T, int LC, int G>
__device__ __forceinline__ void sums(typename T::V (&acc)[kNlGroup], const typename T::E* X, int64_t ldx,
                                     const int32_t* node, const typename T::S (*val)[kChunk], int len) {
  constexpr int EL = 32 / LC;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 8
  for (int e = warp * EL + lane / LC; e < len; e += kWarps * EL) {
    const typename T::V x = T::load(X + (int64_t)node[e] * ldx);
#pragma unroll
    for (int j = 0; j < G; ++j) T::mad(acc[j], val[j][e], x);
  }
}

template <class T, int LC>
__global__ void __cluster_dims__(kSplits, 1, 1) __launch_bounds__(32 * kWarps)
    k_nl_coef(const typename T::E* X, int64_t ldx, int ncol, const int32_t* __restrict__ group,
              const int64_t* __restrict__ prow, const int32_t* __restrict__ pnode,
              const typename T::W* __restrict__ pval, const double* __restrict__ hcoup,
              typename T::E* P, int64_t ldP) {
  using V = typename T::V;
  constexpr size_t kRed = sizeof(V) * kNlGroup * kWarps * LC, kVal = sizeof(typename T::S) * kNlGroup * kChunk;
  __shared__ alignas(16) uint8_t buf[kRed > kVal ? kRed : kVal];
  auto val = reinterpret_cast<typename T::S(*)[kChunk]>(buf);       // while the rows are summed
  auto red = reinterpret_cast<V(*)[kWarps][LC]>(buf);               // then the warps' sums
  __shared__ V part[kNlGroup][LC];
  __shared__ int32_t node[kChunk];
  after_previous();
  auto cluster = cooperative_groups::this_cluster();
  const int g = blockIdx.x / kSplits, sidx = blockIdx.x % kSplits;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lc = lane % LC;
  const int c0 = (blockIdx.y * LC + lc) * T::kCols;
  const bool in = c0 < ncol;
  const int a0 = group[g], cnt = group[g + 1] - a0;
  const int64_t e0 = prow[a0], L = prow[a0 + 1] - e0, len = (L + kSplits - 1) / kSplits;
  const int64_t s0 = e0 + sidx * len, s1 = min(e0 + L, s0 + len);
  V acc[kNlGroup];
#pragma unroll
  for (int j = 0; j < kNlGroup; ++j) acc[j] = T::zero();
  for (int64_t c = s0; c < s1; c += kChunk) {
    const int n = (int)min((int64_t)kChunk, s1 - c);
    if (c != s0) __syncthreads();
    for (int t = threadIdx.x; t < n; t += 32 * kWarps) {
      node[t] = pnode[c + t];
      for (int j = 0; j < cnt; ++j) val[j][t] = (typename T::S)pval[c + t + j * L];
    }
    __syncthreads();
    if (in) switch (cnt) {
      case 1: sums<T, LC, 1>(acc, X + c0, ldx, node, val, n); break;
      case 2: sums<T, LC, 2>(acc, X + c0, ldx, node, val, n); break;
      case 3: sums<T, LC, 3>(acc, X + c0, ldx, node, val, n); break;
      default: sums<T, LC, 4>(acc, X + c0, ldx, node, val, n); break;
    }
  }
  if constexpr (LC < 32) {
#pragma unroll
    for (int o = LC; o < 32; o *= 2)
#pragma unroll
      for (int j = 0; j < kNlGroup; ++j) T::add(acc[j], T::shfl(acc[j], o));
  }
  __syncthreads();
  if (lane < LC)
#pragma unroll
    for (int j = 0; j < kNlGroup; ++j) red[j][warp][lane] = acc[j];
  __syncthreads();
  if (warp < cnt && lane < LC) {
    V t = red[warp][0][lane];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) T::add(t, red[warp][w][lane]);
    part[warp][lane] = t;
  }
  cluster.sync();
  if (sidx == 0 && warp < cnt && lane < LC && in) {
    V t = T::zero();
#pragma unroll
    for (int k = 0; k < kSplits; ++k) T::add(t, cluster.map_shared_rank(&part[0][0], k)[warp * LC + lane]);
    T::store(P + (int64_t)(a0 + warp) * ldP + c0, hcoup[a0 + warp], t, ncol - c0);
  }
  cluster.sync();   // the others' sums stay until they are read
}

// Z[node] += alpha sum_t w_t P[a_t] on the support nodes: LC lanes over columns per node, each row
// of Z read before its projectors are walked
template <class T, int LC>
__global__ void __launch_bounds__(256) k_nl_add(typename T::E* Z, int64_t ldz, int ncol,
                                                const int32_t* __restrict__ snode, const int64_t* __restrict__ srow,
                                                const int32_t* __restrict__ sproj,
                                                const typename T::S* __restrict__ sval,
                                                const typename T::E* P, int64_t ldP, int64_t nsup,
                                                double alpha) {
  after_previous();
  const int64_t s = blockIdx.x * (int64_t)(256 / LC) + threadIdx.x / LC;
  const int c = (blockIdx.y * LC + threadIdx.x % LC) * T::kCols;
  if (s >= nsup || c >= ncol) return;
  typename T::E* z = Z + (int64_t)snode[s] * ldz + c;
  const typename T::V zv = *reinterpret_cast<const typename T::V*>(z);
  typename T::V acc = T::zero();
  const int64_t t1 = srow[s + 1];
#pragma unroll 4
  for (int64_t t = srow[s]; t < t1; ++t)
    T::madn(acc, sval[t], *reinterpret_cast<const typename T::V*>(P + (int64_t)sproj[t] * ldP + c));
  T::update(z, alpha, acc, zv, ncol - c);
}

// P = h (C~^H X) on `stream`; ncol counts entries of E.  One column: the lanes of a warp lie over
// the support's entries instead of over columns.
template <class T>
void coef(dftfe_ham h, cudaStream_t stream, const typename T::E* X, int64_t ldx, int ncol,
          const typename T::W* pval, typename T::E* P, int64_t ldP) {
  static_assert(kNlGroup == 4, "the switch over group sizes");
  const unsigned gx = (unsigned)(h->npgroup * kSplits);
  if constexpr (T::kCols == 1) {
    if (ncol == 1) {
      launch_after(k_nl_coef<T, 1>, dim3(gx), 32 * kWarps, 0, stream, X, ldx, ncol, h->d_pgroup, h->d_prow,
                   h->d_pnode, pval, h->d_h, P, ldP);
      return;
    }
  }
  constexpr int kTile = T::kLanes * T::kCols;
  launch_after(k_nl_coef<T, T::kLanes>, dim3(gx, (unsigned)((ncol + kTile - 1) / kTile)), 32 * kWarps, 0, stream, X, ldx,
               ncol, h->d_pgroup, h->d_prow, h->d_pnode, pval, h->d_h, P, ldP);
}

template <class T>
void add(dftfe_ham h, cudaStream_t stream, typename T::E* Z, int64_t ldz, int ncol, const typename T::S* sval,
         const typename T::E* P, int64_t ldP, double alpha) {
  if (h->nsup == 0) return;      // every support is empty: the term is zero, and so would be the grid
  if constexpr (T::kCols == 1) {
    if (ncol == 1) {
      launch_after(k_nl_add<T, 1>, (unsigned)((h->nsup + 255) / 256), 256, 0, stream, Z, ldz, ncol, h->d_snode,
                   h->d_srow, h->d_sproj, sval, P, ldP, h->nsup, alpha);
      return;
    }
  }
  constexpr int kTile = T::kLanes * T::kCols, kNodes = 256 / T::kLanes;
  launch_after(k_nl_add<T, T::kLanes>,
               dim3((unsigned)((h->nsup + kNodes - 1) / kNodes), (unsigned)((ncol + kTile - 1) / kTile)), 256, 0,
               stream, Z, ldz, ncol, h->d_snode, h->d_srow, h->d_sproj, sval, P, ldP, h->nsup, alpha);
}

}  // namespace nl
}  // namespace dftfe
