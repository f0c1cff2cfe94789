// Tensor-product (sum-factorised) form of the local operator, shared by the FP64 and FP32
// cell kernels (sumfac.cu) and the batched passes.
//
// On the structured periodic mesh the Loewdin cell matrix H~^c = D_c^-1/2 (K^c + V^c) D_c^-1/2
// is a sum of tensor products over the N = p + 1 GLL nodes of an axis:
//   kinetic   kappa_x K (x) 1 (x) 1 + kappa_y 1 (x) K (x) 1 + kappa_z 1 (x) 1 (x) K on the
//             mesh lines (GLL quadrature and the lumped mass are diagonal, so the weights of
//             the two other axes cancel; a line on a face shared by cells is applied by the
//             one cell that has it at its low side), kappa_d = 1/2 (2/h_d)^2,
//             K_ij = sum_q w_q l_i'(x_q) l_j'(x_q) / sqrt(w^_i w^_j), w^ the assembled weights;
//   potential (L (x) L (x) L)^T diag(v) (L (x) L (x) L), L_qa = l_a(x_q) / sqrt(w^_a) at the N
//             Gauss points, v = w_q w_q' w_q'' V(x_q) (mesh sizes cancel); diag(v) alone when the
//             potential quadrature sits on the nodes.
// Nine N-point contractions per node (three on the nodes) replace the N^3-point row of the
// dense matrix, and no cell matrix is read.  K, L and L^T are centrosymmetric, so a contraction
// runs on the even and odd parts of its line: N^2/2 products instead of N^2.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace dftfe {
namespace sf {

// Two FP32 columns of one thread (adjacent columns, or the real and imaginary part of one), and a
// table entry for them (both halves the same); the FP64 kernels take one column per thread.
struct alignas(8) F2 {
  float x, y;
};
struct alignas(16) F4 {
  F2 a, b;
};
// an unevaluated sum of two floats (about 48 bits), for FP64-accurate products on the FP32 pipes
struct alignas(8) DF {
  float hi, lo;
};
inline void set(DF& c, double v) {
  c.hi = (float)v;
  c.lo = (float)(v - (double)c.hi);
}
inline void set(double& c, double v) { c = v; }
inline void set(F2& c, double v) { c.x = c.y = (float)v; }

// parity blocks of a centrosymmetric N x N matrix A (A[N-1-i][N-1-j] = A[i][j]); with
// e_j = u_j + u_{N-1-j}, o_j = u_j - u_{N-1-j} (and the centre entry of odd N kept in e):
// (A u)_i = E_i + O_i, (A u)_{N-1-i} = E_i - O_i, E = e-block e, O = o-block o
template <typename T, int N> struct Parity {
  static constexpr int H = N / 2, C = (N + 1) / 2;
  T e[C][C];
  T o[H][H];
};
// K in difference form, for the FP32 kernels: the rows of K cancel on a constant (sum_j K_ij
// sqrt(w^_j) = 0), so with rho_ij = sqrt(w^_j / w^_i) and t_ij = u_j - rho_ij u_i (one rounding),
//   (K u)_i = sum_j K_ij t_ij, and the same t_ij serves row j with coefficient -K_ij / rho_ij;
// diag undoes what the rounding of rho to FP32 leaves on a constant, so that the form annihilates
// constants to far below FP32's precision.
// A smooth state has small differences, so the products round at their size and not at that of
// K u's large terms: rounding noise of one application of K on states below 1 Ha, in units of
// 2^-24 max(K) |u| (p = 4, 5, 6): 0.05, 0.05, 0.03 against 0.22, 0.24, 0.21 on the parity parts
// and 0.14, 0.13, 0.11 row by row; 3 N (N - 1) / 2 operations per line against N^2 / 2 + 2 N.
template <typename T, int N> struct Differences {
  static constexpr int PAIRS = N * (N - 1) / 2;
  T rho[PAIRS], ki[PAIRS], kj[PAIRS];     // pairs (i, j), i < j: -rho_ij, K_ij, -K_ij / rho_ij
  T diag[N];
};
template <typename T, int N> struct KineticOf { using Type = Parity<T, N>; };
template <int N> struct KineticOf<F2, N> { using Type = Differences<F2, N>; };
template <typename T, int N> struct Tables {
  Parity<T, N> L, Lt;
  typename KineticOf<T, N>::Type K;
};
// parity blocks of the k.grad matrix G_ij = w_i l_j'(x_i) / sqrt(w^_i w^_j), which changes sign
// under the reversal (G[N-1-i][N-1-j] = -G[i][j]): (G u)_i = E_i + O_i, (G u)_{N-1-i} = O_i - E_i
template <typename T, int N> struct AntiParity {
  static constexpr int H = N / 2, C = (N + 1) / 2;
  T e[H][C];
  T o[C][H];
};

// one system's operands of one application Z = s1 X + s2 Xp + alpha H~_loc X (Xp may be null;
// Z may be Xp: every entry is read before it is written, by the same thread)
template <typename T> struct Item {
  const T* v;                   // Nc x N^3 scaled potential
  const T* X;
  const T* Xp;
  T* Z;
  T* face;                      // Nc x (surface nodes of a cell) x ldf partial sums
  int64_t ldx, ldp, ldz;
  int ncol, ldf;
  int nx, ny, nz;
  T kx, kyx, kzx;               // kappa_x, kappa_y / kappa_x, kappa_z / kappa_x
  T gx, gy, gz;                 // k_d (2/h_d) / kappa_x (complex columns at a Bloch k-point)
  T alpha, s1, s2;
  const int* ex;                // float-pair form: biased exponents of the columns (or null)
};

#ifdef __CUDACC__
__device__ __forceinline__ uint64_t pack(F2 a) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ F2 unpack(uint64_t v) {
  F2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack(a)), "l"(pack(b)), "l"(pack(c)));
  return unpack(r);
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack(a)), "l"(pack(b)));
  return unpack(r);
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack(a)), "l"(pack(b)));
  return unpack(r);
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return fma(F2{-1.f, -1.f}, b, a); }
__device__ __forceinline__ F2 fma(float a, F2 b, F2 c) { return fma(F2{a, a}, b, c); }
__device__ __forceinline__ F2 operator*(float a, F2 b) { return F2{a, a} * b; }
// four columns
__device__ __forceinline__ F4 operator+(F4 a, F4 b) { return {a.a + b.a, a.b + b.b}; }
__device__ __forceinline__ F4 operator-(F4 a, F4 b) { return {a.a - b.a, a.b - b.b}; }
__device__ __forceinline__ F4 operator*(F2 c, F4 v) { return {c * v.a, c * v.b}; }
__device__ __forceinline__ F4 operator*(float c, F4 v) { return {c * v.a, c * v.b}; }
__device__ __forceinline__ F4 fma(F2 c, F4 v, F4 w) { return {fma(c, v.a, w.a), fma(c, v.b, w.b)}; }
__device__ __forceinline__ F4 fma(float c, F4 v, F4 w) { return {fma(c, v.a, w.a), fma(c, v.b, w.b)}; }
__device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }
// Float pairs: exact products (one FMA for the rounding error) plus the cross terms, Knuth's TwoSum for
// the leading parts.  The intrinsics keep the compiler from contracting them.
__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ DF tidy(DF a) {            // |lo| <= half an ulp of hi
  const float s = __fadd_rn(a.hi, a.lo);
  return {s, __fsub_rn(a.lo, __fsub_rn(s, a.hi))};
}
__device__ __forceinline__ DF operator*(DF a, DF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  return {p, __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -p)))};
}
__device__ __forceinline__ DF fma(DF a, DF b, DF c) {
  const DF p = a * b, s = two_sum(c.hi, p.hi);
  return {s.hi, __fadd_rn(__fadd_rn(c.lo, p.lo), s.lo)};
}
__device__ __forceinline__ DF operator+(DF a, DF b) {
  const DF s = two_sum(a.hi, b.hi);
  return tidy(DF{s.hi, __fadd_rn(__fadd_rn(a.lo, b.lo), s.lo)});
}
__device__ __forceinline__ DF operator-(DF a, DF b) { return a + DF{-b.hi, -b.lo}; }

// T: table entry, V: the thread's columns (both double, or both F2)
template <typename V, int N>
__device__ __forceinline__ void split(const V (&u)[N], V (&e)[(N + 1) / 2], V (&o)[N / 2]) {
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    e[i] = u[i] + u[N - 1 - i];
    o[i] = u[i] - u[N - 1 - i];
  }
  if (N & 1) e[N / 2] = u[N / 2];
}

// out = A u from the parity parts of u
template <typename T, typename V, int N>
__device__ __forceinline__ void contract(const Parity<T, N>& A, const V (&e)[(N + 1) / 2], const V (&o)[N / 2],
                                         V (&out)[N]) {
  constexpr int H = N / 2, C = (N + 1) / 2;
#pragma unroll
  for (int i = 0; i < C; ++i) {
    V E = A.e[i][0] * e[0];
#pragma unroll
    for (int j = 1; j < C; ++j) E = fma(A.e[i][j], e[j], E);
    if (i < H) {
      V O = A.o[i][0] * o[0];
#pragma unroll
      for (int j = 1; j < H; ++j) O = fma(A.o[i][j], o[j], O);
      out[i] = E + O;
      out[N - 1 - i] = E - O;
    } else {
      out[i] = E;
    }
  }
}

template <typename T, typename V, int N>
__device__ __forceinline__ void apply(const Parity<T, N>& A, const V (&u)[N], V (&out)[N]) {
  V e[(N + 1) / 2], o[N / 2];
  split<V, N>(u, e, o);
  contract<T, V, N>(A, e, o, out);
}

// out = K u (e, o: the parity parts of u, formed by the caller; the difference form needs u alone)
template <int N, typename V>
__device__ __forceinline__ void kinetic(const Parity<V, N>& K, const V (&)[N], const V (&e)[(N + 1) / 2],
                                        const V (&o)[N / 2], V (&out)[N]) {
  contract<V, V, N>(K, e, o, out);
}
template <int N, typename V>
__device__ __forceinline__ void kinetic(const Differences<F2, N>& K, const V (&u)[N], const V (&)[(N + 1) / 2],
                                        const V (&)[N / 2], V (&out)[N]) {
  int q = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) out[i] = K.diag[i] * u[i];
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = i + 1; j < N; ++j, ++q) {
      const V t = fma(K.rho[q], u[i], u[j]);
      out[i] = fma(K.ki[q], t, out[i]);
      out[j] = fma(K.kj[q], t, out[j]);
    }
}

// out += f G u
template <typename T, typename F, typename V, int N>
__device__ __forceinline__ void add_anti(const AntiParity<T, N>& G, F f, const V (&u)[N], V (&out)[N]) {
  constexpr int H = N / 2, C = (N + 1) / 2;
  V e[C], o[H];
  split<V, N>(u, e, o);
#pragma unroll
  for (int i = 0; i < C; ++i) {
    V O = G.o[i][0] * o[0];
#pragma unroll
    for (int j = 1; j < H; ++j) O = fma(G.o[i][j], o[j], O);
    if (i < H) {
      V E = G.e[i][0] * e[0];
#pragma unroll
      for (int j = 1; j < C; ++j) E = fma(G.e[i][j], e[j], E);
      out[i] = fma(f, E + O, out[i]);
      out[N - 1 - i] = fma(f, O - E, out[N - 1 - i]);
    } else {
      out[i] = fma(f, O, out[i]);
    }
  }
}

// Surface nodes of a cell, numbered x line by x line: the 4N - 4 lines that lie on the surface
// (line (b, c) with b or c at an end: N nodes each), then the two end nodes of the others.
template <int N> __host__ __device__ constexpr int surface_count() { return N * N * N - (N - 2) * (N - 2) * (N - 2); }
template <int N> __device__ __forceinline__ int surface_line(int b, int c) {     // first node of a line
  constexpr int p = N - 1;
  if (b > 0 && b < p && c > 0 && c < p) return (4 * N - 4) * N + ((c - 1) * (N - 2) + b - 1) * 2;
  return (c == 0 ? b : c == p ? N + b : 2 * N + (c - 1) * 2 + (b == p ? 1 : 0)) * N;
}
template <int N> __device__ __forceinline__ int surface_index(int a, int b, int c) {
  constexpr int p = N - 1;
  return surface_line<N>(b, c) + (b > 0 && b < p && c > 0 && c < p ? (a == p ? 1 : 0) : a);
}
// of these, the ones the cell owns (no index at the high side): p^3 - (p-1)^3
template <int N> __host__ __device__ constexpr int owned_count() {
  return (N - 1) * (N - 1) * (N - 1) - (N - 2) * (N - 2) * (N - 2);
}
template <int N> __device__ __forceinline__ void owned_node(int s, int& a, int& b, int& c) {
  constexpr int p = N - 1;
  if (s < p * p) {
    c = 0;
    b = s / p;
    a = s - b * p;
    return;
  }
  const int t = s - p * p;
  c = 1 + t / (2 * p - 1);
  const int r = t - (c - 1) * (2 * p - 1);
  b = r < p ? 0 : r - p + 1;
  a = r < p ? r : 0;
}

#endif  // __CUDACC__

}  // namespace sf
}  // namespace dftfe
