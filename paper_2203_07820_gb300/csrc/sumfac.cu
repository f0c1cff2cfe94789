// Tensor-product form of H~_loc X (see sumfac.h): the cell kernel (FP64, FP32 and float pairs), the sums
// over shared faces, their launches for one system and for the batched passes, and the density
// at the quadrature points by the same contractions.
#include "internal.h"
#include "sumfac.h"
#include "tcgen05.h"

#include <algorithm>
#include <memory>
#include <mutex>
#include <type_traits>
#include <cmath>
#include <vector>

namespace dftfe {

// A CTA's item and work index, through shared memory (a single system's item comes by value, a
// batch's from its list).  Read after the next barrier.
template <typename T>
__device__ __forceinline__ int load_item(sf::Item<T>& it, const sf::Item<T>& one, const sf::Item<T>* items,
                                         const int2* work, int w) {
  static_assert(sizeof(sf::Item<T>) % 4 == 0, "copied by words");
  const int2 wk = items ? work[w] : make_int2(0, w);
  const uint32_t* src = reinterpret_cast<const uint32_t*>(items ? items + wk.x : &one);
  if (threadIdx.x < sizeof(sf::Item<T>) / 4) reinterpret_cast<uint32_t*>(&it)[threadIdx.x] = src[threadIdx.x];
  return wk.y;
}

// FP64 -> float pair and back with integer operations (one FP64 subtraction or addition each).
// As tc::narrow_f64, but magnitudes of 2^128 and more, infinities and NaNs among them, are held at
// 2^128's exponent, which FP32 reads as infinity or NaN (the clamp is one operation of the nine).  Every
// sum and product keeps that in the leading part, and it comes back as NaN.  The shifts and range
// tests are written for few operations: W of 373,248 DoFs x 256 columns 4.97 ms, as without the tests;
// with a test on each output beside tc::widen_f32 5.07 to 5.29.
__device__ __forceinline__ float narrow_held(double x) {
  const int hi = __double2hiint(x), t = (hi & 0x7fffffff) - 0x38000000;      // exponent 897: FP32's smallest normal
  const uint32_t lo = (uint32_t)__double2loint(x);
  const uint32_t f = __funnelshift_l(lo, (uint32_t)min(t, 0x0ff00000), 3) + ((lo >> 28) & 1u);
  return __uint_as_float((t < 0x100000 ? 0u : f) | ((uint32_t)hi & 0x80000000u));
}
// exact widening (sign and exponent moved by one arithmetic shift); FP32 subnormals become (next to)
// zero, exponent 255 is taken as 2^128
__device__ __forceinline__ double widen_held(float f) {
  const uint32_t u = __float_as_uint(f);
  const int h = (((int)u >> 3) & (int)0x8fffffff) + 0x38000000;
  return __hiloint2double((u & 0x7f800000u) ? h : 0, (int)(u << 29));
}
__device__ __forceinline__ sf::DF to_pair(double x) {
  const float hi = narrow_held(x);
  return sf::DF{hi, narrow_held(x - widen_held(hi))};
}
__device__ __forceinline__ double from_pair(sf::DF a) {
  const uint32_t u = __float_as_uint(a.hi);
  const int h = (((int)u >> 3) & (int)0x8fffffff) + 0x38000000;
  // a normal entry; otherwise zero, or NaN from exponent 255
  const int w = (u << 1) - 0x01000000u < 0xfe000000u ? h : (int)(u << 1) >> 5;
  return __hiloint2double(w, (int)(u << 29)) + widen_held(a.lo);
}
// For a column whose largest entry has biased exponent e (0: an all-zero column): 2^(e - 1022), its
// scale, or with -e the reciprocal (the ends of the range drawn in, so that both are normal numbers).
__device__ __forceinline__ double scale_of(int e) {
  const int m = min(max(abs(e), 2), 2044);
  return __longlong_as_double((long long)(e > 0 ? m + 1 : e < 0 ? 2045 - m : 1023) << 52);
}

// Where a work item lies: slots of one cell per CTA, columns of slots per row of cells, the first
// cell and its mesh position, the first slot column.  (The divisions of every thread otherwise.)
struct SfPlace {
  int cols, cell, cx, cy, cz, vcol;
};
template <typename T, int CB, int W>
__device__ __forceinline__ void find_place(const sf::Item<T>& it, int w, int sub, SfPlace& q) {
  const int nv = W ? (it.ncol + W - 1) / (W ? W : 1) : it.ncol;
  int cols = CB;                               // the power of two that holds nv
  while (cols > 1 && cols / 2 >= nv) cols /= 2;
  const int tiles = (nv + cols - 1) / cols;
  const int group = w / tiles;
  q.cols = cols;
  q.vcol = (w - group * tiles) * cols;
  q.cell = group * (CB / cols) + sub;
  const int cyz = q.cell / it.nx;
  q.cx = q.cell - cyz * it.nx;
  q.cz = cyz / it.ny;
  q.cy = cyz - q.cz * it.ny;
}

// eight or sixteen bytes from global to shared memory, asynchronously (zeros when !ok)
template <typename V> __device__ __forceinline__ void copy_async(V* dst, const void* src, bool ok) {
  if constexpr (sizeof(V) == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(ok ? 16 : 0)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(ok ? 8 : 0)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT> __device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// The cell kernel.  A work item is CB slots, a slot being W columns (one in FP64, a pair in FP32) of
// one cell: CB slots of one cell, or with fewer columns several cells (slot = sub-cell * slots per
// cell + column).  Thread (line, slot) applies one 1D contraction per stage to line `line` of its
// slot, the lines of a stage along x, y, z, y, x:
//   x  k = K u,                  T = L u      (k and u stay in registers)
//   y  R = kyx K u,              T = L T
//   z  R += kzx K u,             T = L^T (v . L T)
//   y                            T = L^T T
//   x  Z = s1 u + (s2 Xp + alpha (kappa_x (k + R) + L^T T)) on interior nodes; surface nodes go to
//      the face buffer, which k_sf_faces sums.
// s1 u is added last: s1 = -c alpha is of the size of the spectrum while H~ u of a wanted state is
// small, so the sums before it round at H~ u's size.  At a k-point (KPT, pairs = complex
// columns) -i k.grad adds g G (Im u, -Re u) to k and R.  U, R, T are
// [node][slot] in shared memory.  The kinetic contraction of a line on a shared face is left to
// the cell that holds the line at its low side; those lines come first, so whole warps skip it.
// CTAs are persistent: the next item's nodes are copied into U (asynchronously) once the z stage
// has read the last of it, this item's Xp during its first stages, the potential one stage ahead.
// FP64: bound by the FP64 pipe (2 FMA per clock and SM), about 350 operations per line of seven
// nodes against 2401 in the dense product.
//   W columns per thread and slot: 1 in FP64; 2 in FP32, or 4 (one CTA per SM at p = 6, twice the
//   independent work per thread, table entries and addresses shared) where it is the faster form
//   and the items fill the SMs: see quad_pays.
//   W = 0: FP64 blocks in and out, float pairs inside (Z = H~_loc X alone: alpha = 1, no recurrence).
template <int W> struct SfVec_;
template <> struct SfVec_<0> { using V = sf::DF; using C = sf::DF; };
template <> struct SfVec_<1> { using V = double; using C = double; };
template <> struct SfVec_<2> { using V = sf::F2; using C = sf::F2; };
template <> struct SfVec_<4> { using V = sf::F4; using C = sf::F2; };

template <int W, int N> struct SfCfg {
  static constexpr int CB = N >= 4 ? 8 : (N == 3 ? 16 : 32);
  static constexpr int LINES = N * N;
  static constexpr int THREADS = (LINES * CB + 31) / 32 * 32;
  static constexpr int NP = N == 4 || N == 6 ? N + 1 : N;       // x pitch: odd, so that the x lines of
  static constexpr int NODES = N * N * NP;                       // a warp fall into different banks
  static constexpr int INNER = (N - 2) * (N - 2) * (N - 2);
  static constexpr int UB = W == 4 ? 2 : 1;                      // buffers of U
  static constexpr int MINB = W == 4 ? (N == 7 ? 1 : 2)
                                     : N == 9 ? 1 : N >= 7 ? 2 : N == 6 ? 3 : N == 5 ? 4 : N == 3 ? 5 : 6;
  static constexpr size_t smem(bool nodal) {
    return ((size_t)(nodal ? 1 : 2) * NODES + UB * NODES + INNER) * CB * sizeof(typename SfVec_<W>::V);
  }
};

template <typename T, int W, int N, bool NODAL, bool KPT>
__global__ void __launch_bounds__(SfCfg<W, N>::THREADS, SfCfg<W, N>::MINB)
    k_sf_cell(const __grid_constant__ sf::Tables<typename SfVec_<W>::C, N> tab,
              const __grid_constant__ sf::AntiParity<typename SfVec_<W>::C, N> G,
              const __grid_constant__ sf::Item<T> one, const sf::Item<T>* __restrict__ items,
              const int2* __restrict__ work, int nwork) {
  using Cfg = SfCfg<W, N>;
  using V = typename SfVec_<W>::V;
  using C = typename SfVec_<W>::C;
  constexpr int CB = Cfg::CB, p = N - 1, UB = Cfg::UB, CW = W ? W : 1;      // columns per slot
  constexpr bool PAIRS = W == 0;
  const V vzero = V{};
  extern __shared__ double2 sfsm[];
  V* U = reinterpret_cast<V*>(sfsm);
  V* Unext = U + (UB - 1) * Cfg::NODES * CB;
  V* const R = U + UB * Cfg::NODES * CB;
  V* const P = R + Cfg::NODES * CB;                       // Xp on the interior nodes
  V* const B = P + Cfg::INNER * CB;                       // T
  __shared__ sf::Item<T> its[2];
  const int slot = threadIdx.x % CB, line = threadIdx.x / CB;
  const bool on = line < Cfg::LINES;
  // line -> its two transverse indices, the p x p lines owned by a cell first
  int i, j;
  if (line < p * p) {
    j = line / p;
    i = line - j * p;
  } else if (line < p * p + N) {
    j = p;
    i = line - p * p;
  } else {
    i = p;
    j = line - p * p - N;
  }
  const bool owned = i < p && j < p;
  const bool inside = owned && i > 0 && j > 0;
  constexpr int SY = Cfg::NP * CB, SZ = N * Cfg::NP * CB;  // node strides along y and z
  const int xl = (j * N + i) * SY + slot;                 // + a CB
  const int yl = j * SZ + i * CB + slot;                  // + b SY
  const int zl = j * SY + i * CB + slot;                  // + c SZ
  V* const Pl = P + (((j - 1) * (N - 2) + i - 1) * (N - 2) - 1) * CB + slot;   // + a CB (inside)
  const int fline = sf::surface_line<N>(i, j);
  // this thread's x line (., b = i, c = j) of a work item: cell, column, first row, row of a = p
  struct Place {
    int cell, col;
    bool ok;
    int64_t row;
    int last;
  };
  auto place = [&](const sf::Item<T>& it, const SfPlace& first, int w) {
    SfPlace f = first;
    int sub = slot;
    if (f.cols < CB) {                         // several cells: each slot its own
      sub = slot % f.cols;
      find_place<T, CB, CW>(it, w, slot / f.cols, f);
    }
    Place q;
    q.cell = f.cell;
    q.col = (f.vcol + sub) * CW;
    q.ok = on && f.cz < it.nz && q.col < it.ncol;
    int iy = f.cy * p + i, iz = f.cz * p + j;
    iy = iy == it.ny * p ? 0 : iy;
    iz = iz == it.nz * p ? 0 : iz;
    q.row = ((int64_t)iz * (it.ny * p) + iy) * (it.nx * p) + f.cx * p;
    q.last = f.cx + 1 < it.nx ? p : -f.cx * p;
    return q;
  };
  auto fetch = [&](V* U, const sf::Item<T>& it, const Place& q) {
    if (!on) return;
    const T* x = q.ok ? it.X + q.row * it.ldx + q.col : it.X;
#pragma unroll
    for (int a = 0; a < N; ++a)
      copy_async(&U[xl + a * CB], q.ok ? x + (a < p ? a : q.last) * it.ldx : x, q.ok);
  };
  // (Im u, -Re u) of a complex column
  auto turn = [&](V (&x)[N]) {
    if constexpr (KPT) {
#pragma unroll
      for (int a = 0; a < N; ++a) {
        if constexpr (W == 4) x[a] = V{{x[a].a.y, -x[a].a.x}, {x[a].b.y, -x[a].b.x}};
        else x[a] = V{x[a].y, -x[a].x};
      }
    }
  };
  __shared__ SfPlace first[2];
  auto load = [&](int buf, int w) {
    const int wl = load_item(its[buf], one, items, work, w);
    if (threadIdx.x == 0) find_place<T, CB, CW>(items ? items[work[w].x] : one, wl, 0, first[buf]);
    return wl;
  };
  int cur = 0;
  after_previous();
  int wloc = load(0, (int)blockIdx.x);
  __syncthreads();
  Place q = place(its[0], first[0], wloc);
  fetch(U, its[0], q);
  copy_commit();
  for (int w = blockIdx.x; w < nwork; w += gridDim.x, cur ^= 1) {
    const sf::Item<T>& it = its[cur];
    const bool more = w + (int)gridDim.x < nwork;
    copy_wait<0>();
    __syncthreads();
    Place next = q;
    if (more) wloc = load(cur ^ 1, w + (int)gridDim.x);
    if (q.ok && inside && it.Xp) {
      const T* xp = it.Xp + q.row * it.ldp + q.col;
#pragma unroll
      for (int a = 1; a < p; ++a) copy_async(Pl + a * CB, xp + a * it.ldp, true);
    }
    copy_commit();
    // scalars of the kernel's arithmetic: T, or float pairs (whose potential is stored as pairs)
    using E = std::conditional_t<PAIRS, sf::DF, T>;
    E vv[N];          // the potential of this thread's z line (plain loads: the kernel before may have formed it)
    {
      const E* v = reinterpret_cast<const E*>(it.v) + (int64_t)q.cell * (N * N * N) +
                   (NODAL ? (j * N + i) * N : j * N + i);
#pragma unroll
      for (int c = 0; c < N; ++c) {
        vv[c] = E{};
        if (q.ok) {
          if constexpr (PAIRS) {
            const float2 t = *reinterpret_cast<const float2*>(v + c * (NODAL ? 1 : N * N));
            vv[c] = sf::DF{t.x, t.y};
          } else {
            vv[c] = v[c * (NODAL ? 1 : N * N)];
          }
        }
      }
    }
    E kyx, kzx, kx;
    if constexpr (PAIRS) {
      kyx = to_pair(it.kyx);
      kzx = to_pair(it.kzx);
      kx = to_pair(it.kx);
    } else {
      kyx = it.kyx;
      kzx = it.kzx;
      kx = it.kx;
    }
    V u[N], r[N], k[N], e[(N + 1) / 2], o[N / 2], x0[UB == 1 && !PAIRS ? N : 1];
    if (on) {
#pragma unroll
      for (int a = 0; a < N; ++a) {
        u[a] = U[xl + a * CB];
        if constexpr (PAIRS) {
          // the copied FP64 entry, scaled by its column's power of two, becomes a pair
          double x = __hiloint2double(__float_as_int(u[a].lo), __float_as_int(u[a].hi));
          if (it.ex) x *= scale_of(-it.ex[q.ok ? q.col : 0]);
          u[a] = to_pair(x);
          U[xl + a * CB] = u[a];
        }
        if (UB == 1 && !PAIRS) x0[a] = u[a];
      }
      sf::split<V, N>(u, e, o);
      if (!NODAL) {
        sf::contract<C, V, N>(tab.L, e, o, r);
#pragma unroll
        for (int a = 0; a < N; ++a) B[xl + a * CB] = r[a];
      }
      if (owned) {
        sf::kinetic<N>(tab.K, u, e, o, k);
      } else {
#pragma unroll
        for (int a = 0; a < N; ++a) k[a] = vzero;
      }
      if (NODAL) {     // v u joins the kinetic sums, in their units
        E rk;
        if constexpr (PAIRS) rk = to_pair(1.0 / it.kx);
        else rk = T(1) / it.kx;
#pragma unroll
        for (int a = 0; a < N; ++a) k[a] = sf::fma(vv[a] * rk, u[a], k[a]);
      }
      if constexpr (KPT) {
        if (owned) {
          turn(u);
          sf::add_anti<C, T, V, N>(G, it.gx, u, k);
        }
      }
    }
    __syncthreads();
    if (more && UB == 2) {
      next = place(its[cur ^ 1], first[cur ^ 1], wloc);
      fetch(Unext, its[cur ^ 1], next);
    }
    // y line (a = i, ., c = j)
    if (on) {
      if (owned) {
#pragma unroll
        for (int b = 0; b < N; ++b) u[b] = U[yl + b * SY];
        sf::split<V, N>(u, e, o);
        sf::kinetic<N>(tab.K, u, e, o, r);
#pragma unroll
        for (int b = 0; b < N; ++b) r[b] = kyx * r[b];
        if constexpr (KPT) {
          turn(u);
          sf::add_anti<C, T, V, N>(G, it.gy, u, r);
        }
#pragma unroll
        for (int b = 0; b < N; ++b) R[yl + b * SY] = r[b];
      } else {
#pragma unroll
        for (int b = 0; b < N; ++b) R[yl + b * SY] = vzero;
      }
      if (!NODAL) {
#pragma unroll
        for (int b = 0; b < N; ++b) u[b] = B[yl + b * SY];
        sf::apply<C, V, N>(tab.L, u, r);
#pragma unroll
        for (int b = 0; b < N; ++b) B[yl + b * SY] = r[b];
      }
    }
    __syncthreads();
    // z line (a = i, b = j, .)
    if (on) {
      if (owned) {
#pragma unroll
        for (int c = 0; c < N; ++c) u[c] = U[zl + c * SZ];
        sf::split<V, N>(u, e, o);
        sf::kinetic<N>(tab.K, u, e, o, r);
#pragma unroll
        for (int c = 0; c < N; ++c) r[c] = sf::fma(kzx, r[c], R[zl + c * SZ]);
        if constexpr (KPT) {
          turn(u);
          sf::add_anti<C, T, V, N>(G, it.gz, u, r);
        }
#pragma unroll
        for (int c = 0; c < N; ++c) R[zl + c * SZ] = r[c];
      }
      if (!NODAL) {
#pragma unroll
        for (int c = 0; c < N; ++c) u[c] = B[zl + c * SZ];
        sf::apply<C, V, N>(tab.L, u, r);
#pragma unroll
        for (int c = 0; c < N; ++c) u[c] = vv[c] * r[c];
        sf::apply<C, V, N>(tab.Lt, u, r);
#pragma unroll
        for (int c = 0; c < N; ++c) B[zl + c * SZ] = r[c];
      }
    }
    __syncthreads();
    if (more && UB == 1) {                                // U is free: the next item's nodes
      next = place(its[cur ^ 1], first[cur ^ 1], wloc);
      fetch(U, its[cur ^ 1], next);
    }
    copy_commit();
    if (!NODAL) {
      if (on) {
#pragma unroll
        for (int b = 0; b < N; ++b) u[b] = B[yl + b * SY];
        sf::apply<C, V, N>(tab.Lt, u, r);
#pragma unroll
        for (int b = 0; b < N; ++b) B[yl + b * SY] = r[b];
      }
      __syncthreads();
    }
    if (q.ok) {
      if (NODAL) {
#pragma unroll
        for (int a = 0; a < N; ++a) r[a] = kx * (k[a] + R[xl + a * CB]);
      } else {
#pragma unroll
        for (int a = 0; a < N; ++a) u[a] = B[xl + a * CB];
        sf::apply<C, V, N>(tab.Lt, u, r);
#pragma unroll
        for (int a = 0; a < N; ++a) r[a] = sf::fma(kx, k[a] + R[xl + a * CB], r[a]);
      }
      T* const face = it.face + ((int64_t)q.cell * sf::surface_count<N>() + fline) * it.ldf + q.col;
      if constexpr (PAIRS) {
        const double sc = it.ex ? scale_of(it.ex[q.col]) : 1.0;
        T* z = it.Z + q.row * it.ldz + q.col;
#pragma unroll
        for (int a = 0; a < N; ++a) {
          const double y = from_pair(r[a]) * sc;
          if (!inside) face[a * it.ldf] = y;
          else if (a == 0 || a == p) face[a ? it.ldf : 0] = y;
          else z[a * it.ldz] = y;
        }
      } else if (!inside) {
#pragma unroll
        for (int a = 0; a < N; ++a) *reinterpret_cast<V*>(face + a * it.ldf) = r[a];
      } else {
        *reinterpret_cast<V*>(face) = r[0];
        *reinterpret_cast<V*>(face + it.ldf) = r[p];
        T* z = it.Z + q.row * it.ldz + q.col;
        const bool xp = it.Xp != nullptr;
        if (UB == 1) copy_wait<1>();                      // this thread's own Xp
        else if (more) copy_wait<1>();
        else copy_wait<0>();
#pragma unroll
        for (int a = 1; a < p; ++a) {
          const V y = xp ? sf::fma(it.alpha, r[a], it.s2 * Pl[a * CB]) : it.alpha * r[a];
          *reinterpret_cast<V*>(z + a * it.ldz) = sf::fma(it.s1, UB == 1 ? x0[a] : U[xl + a * CB], y);
        }
      }
    }
    q = next;
    if (UB == 2) {
      V* t = U;
      U = Unext;
      Unext = t;
    }
  }
}

// Nodes on cell surfaces: Z = s1 X + s2 Xp + alpha (sum of the face-buffer entries of the 2, 4 or 8
// cells that hold the node, z lowest first inside y inside x).  One CTA per cell takes the
// surface nodes it owns, VEC columns per thread; bound by memory: 200 us for the 1.03 GB of 16^3 cells x
// 128 FP32 columns at p = 6 (76 % of the copy bandwidth).  Five CTAs per SM: at four (52 to 56
// registers) 229 us.
template <typename T, int VEC> struct alignas(sizeof(T) * VEC) SfVec {
  T v[VEC];
};
template <typename T, int N, int VEC>
__global__ void __launch_bounds__(256, 5) k_sf_faces(const __grid_constant__ sf::Item<T> one,
                                                     const sf::Item<T>* __restrict__ items,
                                                     const int2* __restrict__ work) {
  using V = SfVec<T, VEC>;
  constexpr int p = N - 1, NS = sf::surface_count<N>(), NO = sf::owned_count<N>();
  __shared__ sf::Item<T> it;
  after_previous();
  const int cell = load_item(it, one, items, work, (int)blockIdx.x);
  __syncthreads();
  const int cyz = cell / it.nx, cx = cell - cyz * it.nx, cz = cyz / it.ny, cy = cyz - cz * it.ny;
  const int lx = cx ? cx - 1 : it.nx - 1, ly = cy ? cy - 1 : it.ny - 1, lz = cz ? cz - 1 : it.nz - 1;
  const int nv = (it.ncol + VEC - 1) / VEC;
  for (int t = threadIdx.x; t < NO * nv; t += blockDim.x) {
    const int s = t / nv, col = (t - s * nv) * VEC;
    int a, b, c;
    sf::owned_node<N>(s, a, b, c);
    V acc;
#pragma unroll
    for (int q = 0; q < VEC; ++q) acc.v[q] = T(0);
#pragma unroll
    for (int dx = 0; dx < 2; ++dx) {
      if (dx && a) continue;
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) {
        if (dy && b) continue;
#pragma unroll
        for (int dz = 0; dz < 2; ++dz) {
          if (dz && c) continue;
          // d = 0 with the index at the low side: the lower neighbour, which has the node at p
          const int ncx = a || dx ? cx : lx, ncy = b || dy ? cy : ly, ncz = c || dz ? cz : lz;
          const int na = a || dx ? a : p, nb = b || dy ? b : p, nc = c || dz ? c : p;
          const int64_t row = ((int64_t)ncz * it.ny + ncy) * it.nx + ncx;
          const V f = *reinterpret_cast<const V*>(
              it.face + (row * NS + sf::surface_index<N>(na, nb, nc)) * it.ldf + col);
#pragma unroll
          for (int q = 0; q < VEC; ++q) acc.v[q] += f.v[q];
        }
      }
    }
    const int64_t g = ((int64_t)(cz * p + c) * (it.ny * p) + (cy * p + b)) * (it.nx * p) + cx * p + a;
    const T* x = it.X + g * it.ldx + col;
    const T* xp = it.Xp ? it.Xp + g * it.ldp + col : nullptr;
    T* z = it.Z + g * it.ldz + col;
    if (VEC > 1 && col + VEC <= it.ncol) {       // VEC > 1: rows aligned to VEC entries
      V o;
      if (xp) {
        const V pv = *reinterpret_cast<const V*>(xp);
#pragma unroll
        for (int q = 0; q < VEC; ++q) o.v[q] = fma(it.alpha, acc.v[q], it.s2 * pv.v[q]);
      } else {
#pragma unroll
        for (int q = 0; q < VEC; ++q) o.v[q] = it.alpha * acc.v[q];
      }
      if (it.s1 != T(0)) {
        const V xv = *reinterpret_cast<const V*>(x);
#pragma unroll
        for (int q = 0; q < VEC; ++q) o.v[q] = fma(it.s1, xv.v[q], o.v[q]);
      }
      *reinterpret_cast<V*>(z) = o;
    } else {
#pragma unroll
      for (int q = 0; q < VEC; ++q)
        if (VEC == 1 || col + q < it.ncol) {
          const T y = xp ? fma(it.alpha, acc.v[q], it.s2 * xp[q]) : it.alpha * acc.v[q];
          z[q] = it.s1 != T(0) ? fma(it.s1, x[q], y) : y;
        }
    }
  }
}

__global__ void k_sf_narrow(const double* __restrict__ v, int64_t n, float* __restrict__ out) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < n) out[t] = (float)v[t];
}

// Electron density at the quadrature points of a cell (Alg. 3 steps 2-3): the columns of
// [Xo | Xfr] are interpolated by the contractions x, y, z of the cell kernel, CB columns at a time,
// squared and added with their weights (1, f - 1) on the thread that holds the z line, the next
// columns' nodes in flight meanwhile.  blockIdx.y: every gridDim.y-th column tile, into its own
// copy of rho (k_sf_density_sum adds the copies in order).  Bound by the FP64 pipe: 125
// operations per line of seven nodes and column against 2401 in the dense interpolation.
template <int N> struct SfDen {
  static constexpr int CB = SfCfg<1, N>::CB, THREADS = SfCfg<1, N>::THREADS;
  static constexpr int NODES = SfCfg<1, N>::NODES;
  static constexpr int MINB = N == 9 ? 1 : N >= 7 ? 2 : 3;
  static constexpr size_t smem() { return (size_t)2 * NODES * CB * sizeof(double); }
};
template <int N>
__global__ void __launch_bounds__(SfDen<N>::THREADS, SfDen<N>::MINB)
    k_sf_density(const __grid_constant__ sf::Parity<double, N> L, int nx, int ny, int nz,
                 const double* __restrict__ Xo, int64_t ldo, int ncol, const double* __restrict__ Xfr, int64_t ldf,
                 int nfr, const double* __restrict__ f_fr, double scale, double* __restrict__ rho, int64_t copy) {
  constexpr int CB = SfDen<N>::CB, p = N - 1, NP = SfCfg<1, N>::NP, SY = NP * CB, SZ = N * NP * CB;
  extern __shared__ double2 sfdn[];
  double* B = reinterpret_cast<double*>(sfdn);
  double* B2 = B + SfDen<N>::NODES * CB;
  const int slot = threadIdx.x % CB, line = threadIdx.x / CB;
  const bool on = line < N * N;
  const int j = line / N, i = line - j * N;
  const int cell = blockIdx.x, cyz = cell / nx, cx = cell - cyz * nx, cz = cyz / ny, cy = cyz - cz * ny;
  const int iy = cy * p + i == ny * p ? 0 : cy * p + i, iz = cz * p + j == nz * p ? 0 : cz * p + j;
  const int64_t row = ((int64_t)iz * (ny * p) + iy) * (nx * p) + cx * p;
  const int last = cx + 1 < nx ? p : -cx * p;
  const int xl = (j * N + i) * SY + slot, yl = j * SZ + i * CB + slot, zl = j * SY + i * CB + slot;
  const int total = ncol + nfr;
  double u[N], r[N], acc[N], un[N];
  auto read = [&](int c0) {
    const int col = c0 + slot;
    const bool ok = on && col < total;
    const double* x = col < ncol ? Xo + row * ldo + col : Xfr + row * ldf + (col - ncol);
    const int64_t ld = col < ncol ? ldo : ldf;
#pragma unroll
    for (int a = 0; a < N; ++a) un[a] = ok ? __ldg(x + (a < p ? a : last) * ld) : 0.0;
  };
#pragma unroll
  for (int c = 0; c < N; ++c) acc[c] = 0.0;
  const int step = CB * gridDim.y;
  read(CB * blockIdx.y);
  for (int c0 = CB * blockIdx.y; c0 < total; c0 += step) {
    const int col = c0 + slot;
    const double w = col < ncol ? 1.0 : col < total ? f_fr[col - ncol] - 1.0 : 0.0;
    if (on) {
      sf::apply<double, double, N>(L, un, r);
#pragma unroll
      for (int a = 0; a < N; ++a) B[xl + a * CB] = r[a];
    }
    if (c0 + step < total) read(c0 + step);
    __syncthreads();
    if (on) {
#pragma unroll
      for (int b = 0; b < N; ++b) u[b] = B[yl + b * SY];
      sf::apply<double, double, N>(L, u, r);
#pragma unroll
      for (int b = 0; b < N; ++b) B[yl + b * SY] = r[b];
    }
    __syncthreads();
    if (on) {
#pragma unroll
      for (int c = 0; c < N; ++c) u[c] = B[zl + c * SZ];
      sf::apply<double, double, N>(L, u, r);
#pragma unroll
      for (int c = 0; c < N; ++c) acc[c] = fma(w * r[c], r[c], acc[c]);
    }
    double* t = B;                  // the next tile writes the other buffer while z lines are read
    B = B2;
    B2 = t;
  }
#pragma unroll
  for (int c = 0; c < N; ++c) {
#pragma unroll
    for (int o = CB / 2; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
    if (on && slot == 0) rho[blockIdx.y * copy + (int64_t)cell * (N * N * N) + (c * N + j) * N + i] = scale * acc[c];
  }
}

__global__ void k_sf_density_sum(const double* __restrict__ part, int copies, int64_t n, double* __restrict__ rho) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  double s = 0.0;
  for (int k = 0; k < copies; ++k) s += part[k * n + t];
  rho[t] = s;
}

// v[c][q] = V[c][q] wref[q]
__global__ void k_sf_scale(const double* __restrict__ V, const double* __restrict__ wref, int nq, int64_t n,
                           double* __restrict__ out) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < n) out[t] = V[t] * wref[t % nq];
}

// ------------------------------------------------------------------ host side
// The potential quadrature must have p + 1 points per axis (the default Gauss rule) or sit on
// the nodes; other rules keep the dense cell products.
bool sf_applicable(const dftfe_mesh_s* m) { return m->nq1 == m->n1; }

// assembled 1D reference weights (both end nodes hold the sum of two elements' weights)
static std::vector<double> assembled_weights(const dftfe_mesh_s* m) {
  std::vector<double> w(m->gll.w);
  w.front() += m->gll.w.back();
  w.back() = w.front();
  return w;
}

// sum_q w_q l_i'(x_q) l_j'(x_q) / sqrt(w^_i w^_j)
static std::vector<double> kinetic1d(const dftfe_mesh_s* m) {
  const std::vector<double> wa = assembled_weights(m);
  const int N = m->n1;
  std::vector<double> K(N * N);
  for (int i = 0; i < N; ++i)
    for (int j = 0; j < N; ++j) {
      double s = 0.0;
      for (int q = 0; q < N; ++q) s += m->gll.w[q] * m->D[q * N + i] * m->D[q * N + j];
      K[i * N + j] = s / std::sqrt(wa[i] * wa[j]);
    }
  return K;
}

template <typename T, int N> static sf::Parity<T, N> parity(const std::vector<double>& A) {
  constexpr int H = N / 2, C = (N + 1) / 2;
  sf::Parity<T, N> r;
  for (int i = 0; i < C; ++i)
    for (int j = 0; j < C; ++j)
      sf::set(r.e[i][j], j < H ? 0.5 * (A[i * N + j] + A[i * N + N - 1 - j]) : A[i * N + j]);
  for (int i = 0; i < H; ++i)
    for (int j = 0; j < H; ++j) sf::set(r.o[i][j], 0.5 * (A[i * N + j] - A[i * N + N - 1 - j]));
  return r;
}

template <int N, typename C> static void kinetic_table(const dftfe_mesh_s* m, sf::Parity<C, N>& K) {
  K = parity<C, N>(kinetic1d(m));
}
template <int N> static void kinetic_table(const dftfe_mesh_s* m, sf::Differences<sf::F2, N>& D) {
  const std::vector<double> K = kinetic1d(m), wa = assembled_weights(m);
  std::vector<double> diag(N, 0.0);
  int q = 0;
  for (int i = 0; i < N; ++i)
    for (int j = i + 1; j < N; ++j, ++q) {
      const double rho = std::sqrt(wa[j] / wa[i]);
      sf::set(D.rho[q], -rho);
      sf::set(D.ki[q], K[i * N + j]);
      sf::set(D.kj[q], -K[i * N + j] / rho);
      const double off = rho + (double)D.rho[q].x;           // t on a constant is off sqrt(w^_i)
      diag[i] -= (double)D.ki[q].x * off;
      diag[j] -= (double)D.kj[q].x * off / rho;
    }
  for (int i = 0; i < N; ++i) sf::set(D.diag[i], diag[i]);
}

template <typename T, int N> static sf::Tables<T, N> tables(const dftfe_mesh_s* m) {
  const std::vector<double> wa = assembled_weights(m);
  std::vector<double> L(N * N), Lt(N * N);
  for (int i = 0; i < N; ++i)
    for (int j = 0; j < N; ++j) {
      L[i * N + j] = m->Lq[i * N + j] / std::sqrt(wa[j]);
      Lt[j * N + i] = L[i * N + j];
    }
  sf::Tables<T, N> t;
  t.L = parity<T, N>(L);
  t.Lt = parity<T, N>(Lt);
  kinetic_table<N>(m, t.K);
  return t;
}

void sf_init(dftfe_ham h) {
  auto* m = h->mesh;
  // reference weights of the scaled potential: w w' w'', over the assembled weights of the nodes
  // when the quadrature sits on them
  const std::vector<double> wa = assembled_weights(m);
  std::vector<double> w(m->nq);
  for (int q = 0; q < m->nq; ++q) {
    const int ix[3] = {q % m->nq1, (q / m->nq1) % m->nq1, q / (m->nq1 * m->nq1)};
    w[q] = 1.0;
    for (int d = 0; d < 3; ++d) w[q] *= m->vquad == 1 ? m->quad.w[ix[d]] / wa[ix[d]] : m->quad.w[ix[d]];
  }
  DFTFE_CHECK_CUDA(cudaMalloc(&h->d_sfw, sizeof(double) * m->nq));
  DFTFE_CHECK_CUDA(cudaMemcpy(h->d_sfw, w.data(), sizeof(double) * m->nq, cudaMemcpyHostToDevice));
  DFTFE_CHECK_CUDA(cudaMalloc(&h->d_sfv, sizeof(double) * m->Nc * m->nq));
  // 1D tables of the dense cell matrices: products of two basis functions at the quadrature
  // points, the kinetic matrix, the weight fractions of a cell's own nodes
  const int N = m->n1, nq = m->nq1;
  std::vector<double> tab;
  for (int q = 0; q < nq; ++q)
    for (int a = 0; a < N; ++a)
      for (int b = a; b < N; ++b) tab.push_back(m->Lq[q * N + a] * m->Lq[q * N + b] / std::sqrt(wa[a] * wa[b]));
  for (double k : kinetic1d(m)) tab.push_back(k);
  for (int a = 0; a < N; ++a) tab.push_back(m->gll.w[a] / wa[a]);
  DFTFE_CHECK_CUDA(cudaMalloc(&h->d_celltab, sizeof(double) * tab.size()));
  DFTFE_CHECK_CUDA(cudaMemcpy(h->d_celltab, tab.data(), sizeof(double) * tab.size(), cudaMemcpyHostToDevice));
}

void sf_set_potential(dftfe_ham h, const double* v_quad) {
  auto* m = h->mesh;
  const int64_t n = m->Nc * m->nq;
  DFTFE_LAUNCH(k_sf_scale, (unsigned)((n + 255) / 256), 256, 0, h->stream, v_quad, h->d_sfw, m->nq, n, h->d_sfv);
}

// columns of the face buffer: rows stay 16-byte aligned
static int face_ld(int ncol) { return (ncol + 7) / 8 * 8; }
size_t sf_face_elems(const dftfe_mesh_s* m, int ncol) {
  const int64_t n = m->n1, s = n * n * n - (n - 2) * (n - 2) * (n - 2);
  return (size_t)m->Nc * s * face_ld(ncol);
}

template <typename T>
static sf::Item<T> make_item(dftfe_ham h, const T* v, T* face, const T* X, int64_t ldx, const T* Xp, int64_t ldp, T* Z,
                             int64_t ldz, int ncol, double alpha, double s1, double s2) {
  auto* m = h->mesh;
  const double kx = 2.0 / (m->h[0] * m->h[0]), ky = 2.0 / (m->h[1] * m->h[1]), kz = 2.0 / (m->h[2] * m->h[2]);
  return sf::Item<T>{v, X, Xp, Z, face, ldx, ldp, ldz, ncol, face_ld(ncol), m->n[0], m->n[1], m->n[2],
                     (T)kx, (T)(ky / kx), (T)(kz / kx), (T)(h->kvec[0] * (2.0 / m->h[0]) / kx),
                     (T)(h->kvec[1] * (2.0 / m->h[1]) / kx), (T)(h->kvec[2] * (2.0 / m->h[2]) / kx), (T)alpha,
                     (T)s1, (T)s2, nullptr};
}

sf::Item<double> sf_item64(dftfe_ham h, double* face, const double* X, int64_t ldx, const double* Xp, int64_t ldp,
                           double* Z, int64_t ldz, int ncol, double alpha, double s1, double s2) {
  return make_item<double>(h, loc(h)->d_sfv, face, X, ldx, Xp, ldp, Z, ldz, ncol, alpha, s1, s2);
}

// work items of the cell kernel for one system
template <int W, int N> static int64_t cell_work(const dftfe_mesh_s* m, int ncol) {
  constexpr int CB = SfCfg<W, N>::CB, CW = W ? W : 1;
  const int nv = (ncol + CW - 1) / CW;
  int cols = CB;
  while (cols > 1 && cols / 2 >= nv) cols /= 2;
  return ((m->Nc + CB / cols - 1) / (CB / cols)) * ((nv + cols - 1) / cols);
}

// f(std::integral_constant<int, N>) for the mesh degree
template <typename F> static void with_n(int n1, F&& f) {
  switch (n1) {
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 7: f(std::integral_constant<int, 7>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
    case 9: f(std::integral_constant<int, 9>()); break;
    default: throw Error(DFTFE_ERR_ARG, "degree must be in 1..8");
  }
}

static_assert(sizeof(sf::Item<double>) <= 256, "items are passed by value");

template <typename T, int N> static sf::AntiParity<T, N> anti_table(const dftfe_mesh_s* m) {
  constexpr int H = N / 2, C = (N + 1) / 2;
  const std::vector<double> wa = assembled_weights(m);
  auto g = [&](int i, int j) { return m->gll.w[i] * m->D[i * N + j] / std::sqrt(wa[i] * wa[j]); };
  sf::AntiParity<T, N> r;
  for (int i = 0; i < H; ++i)
    for (int j = 0; j < C; ++j) sf::set(r.e[i][j], j < H ? 0.5 * (g(i, j) + g(i, N - 1 - j)) : g(i, j));
  for (int i = 0; i < C; ++i)
    for (int j = 0; j < H; ++j) sf::set(r.o[i][j], i < H ? 0.5 * (g(i, j) - g(i, N - 1 - j)) : g(i, j));
  return r;
}

__global__ void k_sf_pairs(const double* __restrict__ v, int64_t n, sf::DF* __restrict__ out) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < n) out[t] = to_pair(v[t]);
}

// the FP32 copy of the scaled potential (once per potential, in the owner of the operator)
const float* sf_potential32(dftfe_ham h) {
  dftfe_ham o = loc(h);
  const int64_t n = h->mesh->Nc * h->mesh->nq;
  float* v = (float*)ws_get(o, "sf_v32", sizeof(float) * n);
  if (o->sf32_version != o->potential_version) {
    DFTFE_LAUNCH(k_sf_narrow, (unsigned)((n + 255) / 256), 256, 0, h->stream, o->d_sfv, n, v);
    o->sf32_version = o->potential_version;
  }
  return v;
}

sf::Item<float> sf_item32(dftfe_ham h, const float* v, float* face, const float* X, int64_t ldx, const float* Xp,
                          int64_t ldp, float* Z, int64_t ldz, int ncol, double alpha, double s1, double s2) {
  return make_item<float>(h, v, face, X, ldx, Xp, ldp, Z, ldz, ncol, alpha, s1, s2);
}

int64_t sf_cell_work64(const dftfe_mesh_s* m, int ncol) {
  int64_t n = 0;
  with_n(m->n1, [&](auto k) { n = cell_work<1, decltype(k)::value>(m, ncol); });
  return n;
}
int64_t sf_cell_work32(const dftfe_mesh_s* m, int ncol, int width) {
  int64_t n = 0;
  with_n(m->n1, [&](auto k) {
    constexpr int N = decltype(k)::value;
    n = width == 4 ? cell_work<4, N>(m, ncol) : cell_work<2, N>(m, ncol);
  });
  return n;
}
// Columns per thread of the FP32 kernel (both widths give the same bits).  Four at p = 4 and 6, where
// they measured 10 to 12 % faster over 128 columns (12^3 cells, p = 6: 289 against 323 us a launch;
// 14^3, p = 4: 7 % of the filter), once there are eight items per resident CTA; with fewer the last
// wave costs more (8^3 cells, p = 6, 37 columns: 47 against 40 us).  p = 5 measured the same.
int sf_width32(int sm, int n1, int64_t items4) {
  return (n1 == 5 || n1 == 7) && items4 >= 8LL * sm * (n1 == 7 ? 1 : 2) ? 4 : 2;
}

template <typename T, int W, int N, bool NODAL, bool KPT>
static void launch_cell(cudaStream_t s, int sm, const sf::Tables<typename SfVec_<W>::C, N>& tab,
                        const sf::AntiParity<typename SfVec_<W>::C, N>& G, const sf::Item<T>& one,
                        const sf::Item<T>* items, const int2* work, int64_t n) {
  using Cfg = SfCfg<W, N>;
  if (n <= 0) return;
  DFTFE_REQUIRE(n < INT32_MAX / 2, "too many (cell, column tile) items for one launch");
  static const cudaError_t attr = cudaFuncSetAttribute(k_sf_cell<T, W, N, NODAL, KPT>,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::smem(NODAL));
  DFTFE_CHECK_CUDA(attr);
  // FP32: as many CTAs as stay resident, each walking its items with the next one's nodes in
  // flight; FP64: one CTA per item, since the FP64 pipe hides the loads and a fixed deal of long
  // items would leave it idle at the end
  const unsigned grid = (unsigned)(W <= 1 ? n : std::min<int64_t>(n, (int64_t)sm * Cfg::MINB));
  launch_after(k_sf_cell<T, W, N, NODAL, KPT>, grid, Cfg::THREADS, Cfg::smem(NODAL), s, tab, G, one, items, work,
               (int)n);
}

// 1D tables of a degree and quadrature rule, formed once per mesh (they depend on neither the box
// nor the potential)
template <typename C, int N> struct Tables1D {
  sf::Tables<C, N> tab;
  sf::AntiParity<C, N> G;
};
template <typename C, int N> static const Tables1D<C, N>& mesh_tables(const dftfe_mesh_s* m) {
  std::shared_ptr<void>& slot = m->sf_tables[std::is_same<C, double>::value ? 0 : std::is_same<C, sf::F2>::value ? 1 : 2];
  std::lock_guard<std::mutex> lock(m->sf_mutex);
  if (!slot) slot = std::make_shared<Tables1D<C, N>>(Tables1D<C, N>{tables<C, N>(m), anti_table<C, N>(m)});
  return *static_cast<const Tables1D<C, N>*>(slot.get());
}

void sf_launch64(cudaStream_t s, int sm, const dftfe_mesh_s* m, const sf::Item<double>& one,
                 const sf::Item<double>* items, const int2* cell_work, int64_t ncell_work, const int2* face_work,
                 int64_t nface_work) {
  with_n(m->n1, [&](auto k) {
    constexpr int N = decltype(k)::value;
    const auto& t = mesh_tables<double, N>(m);
    if (m->vquad == 1) launch_cell<double, 1, N, true, false>(s, sm, t.tab, t.G, one, items, cell_work, ncell_work);
    else launch_cell<double, 1, N, false, false>(s, sm, t.tab, t.G, one, items, cell_work, ncell_work);
    launch_after(k_sf_faces<double, N, 1>, (unsigned)nface_work, 256, 0, s, one, items, face_work);
  });
}

// kpoint: complex columns (all items of a launch alike); rows of every buffer of a multiple of 4
// floats, 16-byte aligned, with the columns padded to a multiple of 4; width: sf_width32 (the cell
// work list is that of the width)
void sf_launch32(cudaStream_t s, int sm, const dftfe_mesh_s* m, bool kpoint, int width, const sf::Item<float>& one,
                 const sf::Item<float>* items, const int2* cell_work, int64_t ncell_work, const int2* face_work,
                 int64_t nface_work) {
  with_n(m->n1, [&](auto k) {
    constexpr int N = decltype(k)::value;
    if constexpr (N <= 8) {      // split precision: at most 512 nodes per cell
      const auto& t = mesh_tables<sf::F2, N>(m);
      const bool nodal = m->vquad == 1;
      auto cell = [&](auto w) {
        constexpr int W = decltype(w)::value;
        if (nodal && kpoint) launch_cell<float, W, N, true, true>(s, sm, t.tab, t.G, one, items, cell_work, ncell_work);
        else if (nodal) launch_cell<float, W, N, true, false>(s, sm, t.tab, t.G, one, items, cell_work, ncell_work);
        else if (kpoint) launch_cell<float, W, N, false, true>(s, sm, t.tab, t.G, one, items, cell_work, ncell_work);
        else launch_cell<float, W, N, false, false>(s, sm, t.tab, t.G, one, items, cell_work, ncell_work);
      };
      if constexpr (N == 5 || N == 7) {
        if (width == 4) cell(std::integral_constant<int, 4>());
        else cell(std::integral_constant<int, 2>());
      } else {
        cell(std::integral_constant<int, 2>());
      }
      launch_after(k_sf_faces<float, N, 4>, (unsigned)nface_work, 256, 0, s, one, items, face_work);
    }
  });
}

// Z = s1 X + s2 Xp + alpha H~_loc X; at most kSfCols columns at a time, so the face buffer stays
// small against the block
void sf_local64(dftfe_ham h, const double* X, int64_t ldx, const double* Xp, int64_t ldp, double* Z, int64_t ldz,
                int ncol, double alpha, double s1, double s2) {
  auto* m = h->mesh;
  double* face = (double*)ws_get(h, "sf_face", sizeof(double) * sf_face_elems(m, std::min(ncol, kSfCols)));
  for (int c0 = 0; c0 < ncol; c0 += kSfCols) {
    const int nb = std::min(kSfCols, ncol - c0);
    ProfScope ps(h, "cell_gemm_fp64");
    sf_launch64(h->stream, h->sm_count, m, sf_item64(h, face, X + c0, ldx, Xp ? Xp + c0 : nullptr, ldp, Z + c0, ldz, nb, alpha, s1,
                                        s2),
                nullptr, nullptr, sf_cell_work64(m, nb), nullptr, m->Nc);
  }
}

// Y = H~_loc X from float pairs (FP64 blocks; about 2^-44 |H~||X|); ex: biased exponents of the columns'
// largest entries, by which they are scaled on the way (NULL: the entries lie well inside FP32's range;
// above it they come out as NaN)
void sf_local_pairs(dftfe_ham h, const double* X, int64_t ldx, double* Y, int64_t ldy, int ncol, const int* ex) {
  auto* m = h->mesh;
  dftfe_ham o = loc(h);
  const int64_t nvq = m->Nc * m->nq;
  sf::DF* v = (sf::DF*)ws_get(o, "sf_vdf", sizeof(sf::DF) * nvq);
  if (o->sfdf_version != o->potential_version) {
    DFTFE_LAUNCH(k_sf_pairs, (unsigned)((nvq + 255) / 256), 256, 0, h->stream, o->d_sfv, nvq, v);
    o->sfdf_version = o->potential_version;
  }
  double* face = (double*)ws_get(h, "sf_face", sizeof(double) * sf_face_elems(m, std::min(ncol, kSfCols)));
  for (int c0 = 0; c0 < ncol; c0 += kSfCols) {
    const int nb = std::min(kSfCols, ncol - c0);
    sf::Item<double> one = make_item<double>(h, (const double*)v, face, X + c0, ldx, (const double*)nullptr, 0, Y + c0, ldy,
                                             nb, 1.0, 0.0, 0.0);
    one.ex = ex ? ex + c0 : nullptr;
    ProfScope ps(h, "cell_gemm_df");
    with_n(m->n1, [&](auto k) {
      constexpr int N = decltype(k)::value;
      const auto& t = mesh_tables<sf::DF, N>(m);
      const int64_t n = cell_work<0, N>(m, nb);
      if (m->vquad == 1)
        launch_cell<double, 0, N, true, false>(h->stream, h->sm_count, t.tab, t.G, one, nullptr, nullptr, n);
      else
        launch_cell<double, 0, N, false, false>(h->stream, h->sm_count, t.tab, t.G, one, nullptr, nullptr, n);
      launch_after(k_sf_faces<double, N, 1>, (unsigned)m->Nc, 256, 0, h->stream, one, nullptr, nullptr);
    });
  }
}

// the density of sf_applicable meshes
void sf_density(dftfe_ham h, const double* Xo, int64_t ldo, int ncol, const double* Xfr, int64_t ldf, int nfr,
                const double* f_fr, double* rho) {
  auto* m = h->mesh;
  const double scale = 2.0 * 8.0 / (m->h[0] * m->h[1] * m->h[2]);     // M^-1/2 beyond the reference weights
  const int64_t n = m->Nc * m->nq;
  with_n(m->n1, [&](auto k) {
    constexpr int N = decltype(k)::value;
    using D = SfDen<N>;
    static const cudaError_t attr = cudaFuncSetAttribute(k_sf_density<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                         (int)D::smem());
    DFTFE_CHECK_CUDA(attr);
    // few cells: several CTAs per cell, up to one per column tile, so that every SM has a share
    const int64_t tiles = (ncol + nfr + D::CB - 1) / D::CB;
    const int copies = (int)std::max<int64_t>(1, std::min<int64_t>({tiles, 8, 4LL * D::MINB * h->sm_count / m->Nc}));
    double* part = copies > 1 ? (double*)ws_get(h, "sf_rho", sizeof(double) * n * copies) : rho;
    DFTFE_LAUNCH((k_sf_density<N>), dim3((unsigned)m->Nc, (unsigned)copies), D::THREADS, D::smem(), h->stream,
                 mesh_tables<double, N>(m).tab.L, m->n[0], m->n[1], m->n[2], Xo, ldo, ncol, Xfr, ldf, nfr, f_fr, scale, part, n);
    if (copies > 1)
      DFTFE_LAUNCH(k_sf_density_sum, (unsigned)((n + 255) / 256), 256, 0, h->stream, part, copies, n, rho);
  });
}

}  // namespace dftfe
