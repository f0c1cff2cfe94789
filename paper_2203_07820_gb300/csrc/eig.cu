// Dense eigensolver of the Rayleigh-Ritz step (a11; Alg. 2 step 2b-c), real symmetric and
// Hermitian: Householder tridiagonalisation, divide and conquer on the real tridiagonal matrix,
// back transformation.
//
//   k_tridiag      A = Q T Q^H by Householder reflectors, one cooperative launch: the rows of A stay
//                  in the shared memory of the CTAs (cyclic rows), and a column costs one grid
//                  barrier: the rank-2 update of the previous column and the product A v of the
//                  next one are a single pass over the rows, and every CTA forms v and w itself
//                  from the product and the pivot row that were exchanged.
//   k_dc_*         Cuppen's divide and conquer from single rows up (Golub & Van Loan, sec. 8.4;
//                  Gu & Eisenstat, SIAM J. Matrix Anal. Appl. 16, 1995: the coupling vector is
//                  recomputed from the computed roots, so the eigenvectors come out orthogonal).
//                  Merges of up to kDcBlock rows run whole in one CTA each, larger ones as one
//                  launch per phase.
//   k_wy, k_backtransform  z <- H_0 H_1 ... z for every eigenvector, one warp each, the vector in
//                  registers, four reflectors per pass.
//
// A cyclic Jacobi iteration (dense.cu) does 8 N^3 FP64 operations and 2 N grid barriers per sweep,
// for about eight sweeps; this form does about 9 N^3 in all and N barriers.
#include "internal.h"
#include "gridbar.h"

#include <algorithm>
#include <cmath>

namespace dftfe {
namespace eig {

constexpr double kEps = 1.1102230246251565e-16;   // 2^-53

// ------------------------------------------------------------------ scalars
__device__ __forceinline__ double zero_of(double) { return 0.0; }
__device__ __forceinline__ double2 zero_of(double2) { return make_double2(0.0, 0.0); }
__device__ __forceinline__ double conj_of(double a) { return a; }
__device__ __forceinline__ double2 conj_of(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double real_of(double a) { return a; }
__device__ __forceinline__ double real_of(double2 a) { return a.x; }
__device__ __forceinline__ bool is_real(double) { return true; }
__device__ __forceinline__ bool is_real(double2 a) { return a.y == 0.0; }
__device__ __forceinline__ double abs2(double a) { return a * a; }
__device__ __forceinline__ double abs2(double2 a) { return fma(a.x, a.x, a.y * a.y); }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ double2 mul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double top_of(double a) { return fabs(a); }
__device__ __forceinline__ double top_of(double2 a) { return fmax(fabs(a.x), fabs(a.y)); }
__device__ __forceinline__ double scale(double s, double a) { return s * a; }
__device__ __forceinline__ double2 scale(double s, double2 a) { return make_double2(s * a.x, s * a.y); }
// c + a b
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double2 mad(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
__device__ __forceinline__ double neg(double a) { return -a; }
__device__ __forceinline__ double2 neg(double2 a) { return make_double2(-a.x, -a.y); }
__device__ __forceinline__ double shfl_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double2 shfl_xor(double2 a, int o) {
  return make_double2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}
template <typename C> __device__ __forceinline__ C warp_sum(C v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = add(v, shfl_xor(v, o));
  return v;
}
// sum over a CTA of TT threads (every thread gets it; red holds TT / 32 entries)
template <typename C, int TT> __device__ __forceinline__ C block_total(C v, C* red) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  C t = red[0];
#pragma unroll
  for (int w = 1; w < TT / 32; ++w) t = add(t, red[w]);
  return t;
}

// The matrix is scaled by the power of two that brings its largest entry to [1/2, 1): exact, and neither
// the squares of the reflectors nor the thresholds of the divide and conquer, which are set against
// vectors of norm one, depend on the unit of A.  Biased exponent of that power from the bits of the
// largest entry (a matrix of zeros, or one that is not finite, is left alone; the ends of the range are
// drawn in, so that the power and its reciprocal are normal numbers).
__device__ __forceinline__ int scale_exponent(unsigned long long top) {
  const int e = (int)(top >> 52);
  return top == 0 || e == 2047 ? 1023 : min(max(2045 - e, 1), 2044);
}
__device__ __forceinline__ double pow2(int biased) { return __longlong_as_double((long long)biased << 52); }

// -------------------------------------------------------- tridiagonalisation
constexpr int kTriThreads = 128;    // one warp per sub-partition: scalar steps repeat in all of them for free
// Rows i = blockIdx.x, blockIdx.x + gridDim.x, ... of A (lower triangle read) live in shared
// memory.  Per column j, with the reflector H_j = I - tau v v^H, v_{j+1} = 1:
//   p = A v, w = tau p - (tau / 2)(tau p)^H v v, A <- A - v w^H - w v^H,
// d_j = A_jj, e_j = the real entry H_j leaves below it.  Exchange buffers are double-buffered by
// the parity of j: xp = p of this column, xr = row j + 1 before its update.
template <typename C>
__global__ void __launch_bounds__(kTriThreads) k_tridiag(const C* __restrict__ A, int N, C* __restrict__ V,
                                                         C* __restrict__ tau_out, double* __restrict__ d,
                                                         double* __restrict__ e, C* __restrict__ xp,
                                                         C* __restrict__ xr, jac::Barrier* bar, int* status) {
  extern __shared__ double2 tri_smem[];
  __shared__ C red[kTriThreads / 32];
  __shared__ double redd[kTriThreads / 32];
  const int G = gridDim.x, b = blockIdx.x;
  const int nrow = (N - b + G - 1) / G;
  C* const rows = reinterpret_cast<C*>(tri_smem);           // nrow x N
  C* const v = rows + (size_t)((N + G - 1) / G) * N;        // reflector of the column before
  C* const w = v + N;
  C* const x = w + N;                                       // pivot row, then the new reflector
  const C zero = zero_of(C());
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long top = 0;                // as bits: non-negative doubles order alike, NaN above all
  for (int r = 0; r < nrow; ++r) {
    const int i = b + r * G;
    for (int k = threadIdx.x; k < N; k += kTriThreads) {
      const C t = k <= i ? A[(size_t)i * N + k] : conj_of(A[(size_t)k * N + i]);
      rows[(size_t)r * N + k] = t;
      top = max(top, (unsigned long long)__double_as_longlong(top_of(t)));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  if (lane == 0 && top) atomicMax(&bar->top, top);
  for (int k = threadIdx.x; k < N; k += kTriThreads) v[k] = w[k] = zero;
  __syncthreads();
  if (b == 0)
    for (int k = threadIdx.x; k < N; k += kTriThreads) xr[N + k] = rows[k];     // read as column -1's
  if (!jac::grid_barrier(bar, status)) return;
  const double sc = pow2(scale_exponent(__ldcg(&bar->top)));
  for (int t = threadIdx.x; t < nrow * N; t += kTriThreads) rows[t] = scale(sc, rows[t]);
  __syncthreads();
  C tau = zero;
  for (int j = 0; j < N; ++j) {
    const int cur = j & 1, old = cur ^ 1;
    const C* const po = xp + (size_t)old * N;
    const C* const ro = xr + (size_t)old * N;
    // w of the column before, from its p (zero for j = 0: tau = 0)
    if (j > 0) {
      C s = zero;
      for (int k = j + threadIdx.x; k < N; k += kTriThreads) {
        const C pk = mul(tau, __ldcg(po + k));
        w[k] = pk;
        s = mad(conj_of(pk), v[k], s);
      }
      s = block_total<C, kTriThreads>(s, red);
      const C f = scale(-0.5, mul(tau, s));
      for (int k = j + threadIdx.x; k < N; k += kTriThreads) w[k] = mad(f, v[k], w[k]);
      __syncthreads();
    }
    // pivot row with that column's update; x_i = A_ij for i > j
    const C vj = j > 0 ? v[j] : zero, wj = j > 0 ? w[j] : zero;
    double nrm = 0.0;
    for (int k = j + threadIdx.x; k < N; k += kTriThreads) {
      C r = __ldcg(ro + k);
      if (j == 0) r = scale(sc, r);
      else r = mad(neg(vj), conj_of(w[k]), mad(neg(wj), conj_of(v[k]), r));
      x[k] = conj_of(r);
      if (k > j + 1) nrm += abs2(r);
    }
    nrm = block_total<double, kTriThreads>(nrm, redd);      // |x below its first entry|^2
    if (b == 0 && threadIdx.x == 0) d[j] = real_of(x[j]);
    if (j == N - 1) break;
    // reflector: H^H x = beta e_1, beta real (an entry with nothing below it may still need its phase
    // taken out, however small its imaginary part: squares would round that away).  Entries below
    // 1e-140 of the largest one count as zeros, so that their squares stay in range.
    const C a = x[j + 1];
    const double full = nrm + abs2(a);
    double beta = real_of(a);
    C inv = zero, tnew = zero;
    if (full > 1e-280 && (nrm > 0.0 || !is_real(a))) {
      const double rs = real_of(a) > 0.0 ? -rsqrt(full) : rsqrt(full);      // 1 / beta
      beta = full * rs;
      if constexpr (sizeof(C) == 16) {                      // inv = 1 / (alpha - beta)
        const C am = C{a.x - beta, a.y};
        const double q = 1.0 / abs2(am);
        inv = C{am.x * q, -am.y * q};
        tnew = C{(beta - a.x) * rs, -a.y * rs};
      } else {
        inv = 1.0 / (a - beta);
        tnew = (beta - a) * rs;
      }
    }
    const bool reflects = abs2(tnew) != 0.0;                // else H = I: v = 0
    __syncthreads();                                        // everyone has read x[j + 1]
    for (int k = j + 1 + threadIdx.x; k < N; k += kTriThreads) {
      if (k > j + 1) x[k] = mul(inv, x[k]);
      else if constexpr (sizeof(C) == 16) x[k] = C{reflects ? 1.0 : 0.0, 0.0};
      else x[k] = reflects ? 1.0 : 0.0;
    }
    __syncthreads();
    if (b == 0) {
      for (int k = threadIdx.x; k < N; k += kTriThreads) V[(size_t)j * N + k] = k > j ? x[k] : zero;
      if (threadIdx.x == 0) {
        e[j] = beta;
        tau_out[j] = tnew;
      }
    }
    // own rows below j: the update of the column before and the product with the new reflector
    C* const pc = xp + (size_t)cur * N;
    C* const rc = xr + (size_t)cur * N;
    const int rfirst = b > j ? 0 : (j - b) / G + 1;
    for (int r = rfirst + warp; r < nrow; r += kTriThreads / 32) {
      const int i = b + r * G;
      C* const row = rows + (size_t)r * N;
      const C nv = j > 0 ? neg(v[i]) : zero, nw = j > 0 ? neg(w[i]) : zero;
      C s = zero;
      for (int k = j + 1 + lane; k < N; k += 32) {
        C t = row[k];
        if (j > 0) t = mad(nv, conj_of(w[k]), mad(nw, conj_of(v[k]), t));
        row[k] = t;
        s = mad(t, x[k], s);
        if (i == j + 1) __stcg(rc + k, t);
      }
      s = warp_sum(s);
      if (lane == 0) __stcg(pc + i, s);
    }
    tau = tnew;
    __syncthreads();
    for (int k = j + 1 + threadIdx.x; k < N; k += kTriThreads) v[k] = x[k];
    if (G > 1) {
      if (!jac::grid_barrier(bar, status)) return;
    } else {
      __threadfence();
      __syncthreads();
    }
  }
}

// ----------------------------------------------------------- divide and conquer
// Workspace, indexed by row of the whole matrix; a merge of rows [s, e) uses its own range.
struct Dc {
  int N;
  double *d, *e;                  // tridiagonal; d becomes the blocks' eigenvalues
  double *Qa, *Qb;                // eigenvectors as rows (Qa: input of the level, Qb: output)
  double *pole, *z, *lam, *mu, *zh, *out, *S;
  int *col, *typ, *org, *src, *K;
  double* rho;
};
// sum and maximum over the CTA
template <int TT> __device__ double dc_max(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = red[0];
  for (int w = 1; w < TT / 32; ++w) t = fmax(t, red[w]);
  return t;
}
// total order on all doubles (NaNs included), for the sort
__device__ __forceinline__ long long dc_key(double v) {
  const long long b = __double_as_longlong(v);
  return b < 0 ? (long long)(0x8000000000000000ull - (unsigned long long)b) : b;
}

constexpr int kDcThreads = 256;

// T_1, T_2 of every split: each off-diagonal entry is taken out of the two diagonal entries it
// couples, T = diag(T_1, T_2) + |e| u u^T, u = (0 .. 1, sign e, .. 0)
__global__ void k_dc_init(Dc w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= w.N) return;
  const double l = i > 0 ? fabs(w.e[i - 1]) : 0.0, r = i < w.N - 1 ? fabs(w.e[i]) : 0.0;
  w.out[i] = w.d[i] - l - r;
}
__global__ void k_dc_start(Dc w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= w.N) return;
  w.d[i] = w.out[i];
  w.Qa[(size_t)i * w.N + i] = 1.0;
}

// Sort the merge's poles, deflate: poles whose coupling is negligible keep their eigenvector; of two
// poles too close to separate one is rotated free of the coupling.  Serial over the sorted poles
// (one thread), with the common decisions made in parallel before.
__device__ void dc_prepare(const Dc& w, int s, int mid, int e, double* sm) {
  const int n = e - s, N = w.N;
  double* ds = sm;                 // sorted poles
  double* zs = ds + n;
  double* rc = zs + n;             // rotations: cosine, sine
  double* rs = rc + n;
  int* cs = reinterpret_cast<int*>(rs + n);   // row of Q of each sorted pole
  int* fl = cs + n;                // bit 0: negligible coupling, bit 1: close to the pole before
  int* ra = fl + n;                // rotations: the two rows
  int* rb = ra + n;
  __shared__ double red[kDcThreads / 32];
  __shared__ int nrot, kk;
  double dm = 0.0, zm = 0.0;
  const double off = w.e[mid - 1], rho = 2.0 * fabs(off), sg = off < 0.0 ? -1.0 : 1.0;
  for (int t = threadIdx.x; t < n; t += kDcThreads) {
    const double dt = w.d[s + t];
    const long long key = dc_key(dt);
    int r = 0;
    for (int q = 0; q < n; ++q) {
      const long long kq = dc_key(w.d[s + q]);
      r += kq < key || (kq == key && q < t);
    }
    const double zt = (s + t < mid ? w.Qa[(size_t)(s + t) * N + mid - 1] : sg * w.Qa[(size_t)(s + t) * N + mid]) *
                      0.70710678118654752440;
    ds[r] = dt;
    zs[r] = zt;
    cs[r] = s + t;
    dm = fmax(dm, fabs(dt));
    zm = fmax(zm, fabs(zt));
  }
  dm = dc_max<kDcThreads>(dm, red);
  zm = dc_max<kDcThreads>(zm, red);
  const double tol = 16.0 * kEps * fmax(dm, zm);
  __syncthreads();
  for (int r = threadIdx.x; r < n; r += kDcThreads) fl[r] = rho * fabs(zs[r]) <= tol ? 1 : 0;
  __syncthreads();
  for (int r = threadIdx.x; r < n; r += kDcThreads) {
    if (fl[r] & 1) continue;
    int q = r - 1;
    while (q >= 0 && (fl[q] & 1)) --q;
    if (q < 0) continue;
    const double zz = fma(zs[r], zs[r], zs[q] * zs[q]);
    if (fabs((ds[r] - ds[q]) * zs[r] * zs[q]) <= tol * zz) atomicOr(&fl[r], 2);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int K = 0, D = 0, nr = 0, prev = -1;
    bool moved = false;              // prev's coupling changed since the parallel decisions
    for (int r = 0; r < n; ++r) {
      if (fl[r] & 1) {               // deflated as it is: value and row from the end of the lists
        w.out[e - 1 - D] = ds[r];
        w.src[e - 1 - D] = cs[r];
        ++D;
        continue;
      }
      bool close = (fl[r] & 2) != 0;
      if (prev >= 0 && moved) {
        const double zz = fma(zs[r], zs[r], zs[prev] * zs[prev]);
        close = fabs((ds[r] - ds[prev]) * zs[r] * zs[prev]) <= tol * zz;
      }
      if (prev >= 0 && close) {
        // rotate the rows of prev and r so that prev's coupling vanishes
        const double tau = sqrt(fma(zs[r], zs[r], zs[prev] * zs[prev]));
        const double c = zs[r] / tau, sn = -zs[prev] / tau;
        zs[r] = tau;
        const double dp = ds[prev], dr = ds[r];
        ds[r] = dp * sn * sn + dr * c * c;
        ra[nr] = cs[prev];
        rb[nr] = cs[r];
        rc[nr] = c;
        rs[nr] = sn;
        ++nr;
        w.out[e - 1 - D] = dp * c * c + dr * sn * sn;
        w.src[e - 1 - D] = cs[prev];
        ++D;
        prev = r;
        moved = true;
        continue;
      }
      if (prev >= 0) {
        w.pole[s + K] = ds[prev];
        w.z[s + K] = zs[prev];
        w.col[s + K] = cs[prev];
        ++K;
      }
      prev = r;
      moved = false;
    }
    if (prev >= 0) {
      w.pole[s + K] = ds[prev];
      w.z[s + K] = zs[prev];
      w.col[s + K] = cs[prev];
      ++K;
    }
    w.K[s] = K;
    w.rho[s] = rho;
    nrot = nr;
    kk = K;
  }
  __syncthreads();
  // 1: rows of the first half only, 2: of the second half only, 3: both (rotated)
  for (int t = s + threadIdx.x; t < e; t += kDcThreads) w.typ[t] = t < mid ? 1 : 2;
  __syncthreads();
  for (int q = 0; q < nrot; ++q) {
    double* x = w.Qa + (size_t)ra[q] * N;
    double* y = w.Qa + (size_t)rb[q] * N;
    const double c = rc[q], sn = rs[q];
    for (int t = s + threadIdx.x; t < e; t += kDcThreads) {
      const double a = x[t], b = y[t];
      x[t] = c * a + sn * b;
      y[t] = c * b - sn * a;
    }
    if (threadIdx.x == 0) {
      const int m = w.typ[ra[q]] | w.typ[rb[q]];
      w.typ[ra[q]] = m;
      w.typ[rb[q]] = m;
    }
    __syncthreads();
  }
  // the type rides in the top bits of the row index
  for (int k = threadIdx.x; k < kk; k += kDcThreads) w.col[s + k] |= w.typ[w.col[s + k]] << 28;
}

// four sums over a warp at once (every lane gets all four): the halving steps share their adds
template <typename F> __device__ __forceinline__ void warp_sum4(F& a, F& b, F& c, F& d) {
  const int lane = threadIdx.x & 31;
  const bool h16 = lane & 16, h8 = lane & 8;
  const F x0 = (h16 ? c : a) + __shfl_xor_sync(0xffffffffu, h16 ? a : c, 16);
  const F x1 = (h16 ? d : b) + __shfl_xor_sync(0xffffffffu, h16 ? b : d, 16);
  F y = (h8 ? x1 : x0) + __shfl_xor_sync(0xffffffffu, h8 ? x0 : x1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
  a = __shfl_sync(0xffffffffu, y, 0);
  b = __shfl_sync(0xffffffffu, y, 8);
  c = __shfl_sync(0xffffffffu, y, 16);
  d = __shfl_sync(0xffffffffu, y, 24);
}

// Iterate for the zero of f(x) = 1 + rho sum_j z_j^2 / (gap_j - x) in [lo, hi] (one warp; f increases):
// each step fits c + s / (gap_a - x) + t / (gap_b - x) to the sums left and right of the interval
// (the "middle way" of Li, LAPACK Working Note 89) and falls back to Newton, then bisection when
// it leaves the bracket or the bracket shrinks slowly.  get(j, gap, z) delivers the terms.
template <typename F, typename Get>
__device__ __forceinline__ F dc_solve(const Get& get, int K, int k, F rho, F lo, F hi, F mu, F eps, int most) {
  const int lane = threadIdx.x & 31;
  const bool last = k == K - 1;
  F ga, gb, zu, zk;
  get(last ? k - 1 : k, ga, zu);
  get(last ? k : k + 1, gb, zk);               // last: zk belongs to pole k
  F width = hi - lo;
  for (int it = 0; it < most; ++it) {
    F fl = 0, fr = 0, gl = 0, gr = 0;          // sums up to the interval and beyond, derivatives
    for (int j = lane; j < K; j += 32) {
      F g, z;
      get(j, g, z);
      const F t = z / (g - mu);
      if (j <= k) {
        fl += z * t;
        gl += t * t;
      } else {
        fr += z * t;
        gr += t * t;
      }
    }
    warp_sum4(fl, fr, gl, gr);
    fl *= rho;
    fr *= rho;
    gl *= rho;
    gr *= rho;
    const F f = F(1) + fl + fr;
    const F mag = F(1) + fabs(fl) + fabs(fr) + fabs(mu) * (gl + gr);
    if (fabs(f) <= F(4) * eps * mag || !(hi - lo > F(2) * eps * fmax(fabs(lo), fabs(hi)))) break;
    if (f < F(0)) lo = mu;
    else hi = mu;
    F next = F(0.5) * (lo + hi);
    if (!(it % 3 == 2 && hi - lo > F(0.5) * width)) {
      const F da = ga - mu, db = gb - mu;
      F c;
      if (last) {                              // both fitted poles lie left of the root
        const F tl = zk / db, gk = rho * tl * tl;
        c = f - da * (gl - gk) - db * gk;
      } else {
        c = f - da * gl - db * gr;
      }
      const F a = (da + db) * f - da * db * (gl + gr), b = da * db * f;
      const F disc = sqrt(fmax(F(0), a * a - F(4) * b * c));
      F eta;
      if (last) eta = a >= F(0) ? (a + disc) / (F(2) * c) : F(2) * b / (a - disc);
      else eta = a <= F(0) ? (a - disc) / (F(2) * c) : F(2) * b / (a + disc);
      F cand = mu + eta;
      if (!(cand > lo && cand < hi)) cand = mu - f / (gl + gr);
      if (cand > lo && cand < hi) next = cand;
    }
    if (it % 3 == 2) width = hi - lo;
    if (next == mu) break;
    mu = next;
  }
  return mu;
}

// Root k of a merge (one warp): lambda = pole[org] + mu, org the nearer end of the root's interval.
// The iteration starts in FP32 on the differences from the origin (FP64 operations cost a warp 64
// clocks each) and a few FP64 steps finish it; buf: 2 K floats of the warp.
__device__ void dc_root(const Dc& w, int s, int k, int lane, float* buf) {
  const int K = w.K[s];
  const double rho = w.rho[s];
  const double* pole = w.pole + s;
  const double* z = w.z + s;
  const bool last = k == K - 1;
  double gap;                                  // length of the root's interval
  if (last) {
    double zz = 0.0;
    for (int j = lane; j < K; j += 32) zz = fma(z[j], z[j], zz);
    gap = rho * warp_sum(zz);
  } else {
    gap = pole[k + 1] - pole[k];
  }
  if (K == 1) {
    if (lane == 0) {
      w.org[s] = s;
      w.mu[s] = gap;
      w.lam[s] = pole[0] + gap;
    }
    return;
  }
  // the sign at the middle of the interval picks the origin (in FP32: near the middle either will do)
  float* gb = buf;
  float* zb = buf + K;
  const double inv = 1.0 / gap;                // gaps in units of the interval: no FP32 range to watch
  float fm = 0.f;
  const float rz = (float)(rho * inv);
  for (int j = lane; j < K; j += 32) {
    gb[j] = (float)((pole[j] - pole[k]) * inv);
    zb[j] = (float)z[j];
    fm += zb[j] * zb[j] / (gb[j] - 0.5f);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) fm += __shfl_xor_sync(0xffffffffu, fm, o);
  const bool left = last || 1.f + rz * fm >= 0.f;
  const int org = left ? k : k + 1;
  if (!left)
    for (int j = lane; j < K; j += 32) gb[j] = (float)((pole[j] - pole[k + 1]) * inv);
  __syncwarp();
  auto get32 = [&](int j, float& g, float& zz) {
    g = gb[j];
    zz = zb[j];
  };
  const float m32 = dc_solve<float>(get32, K, k, rz, left ? 0.f : -1.f, left ? 1.f : 0.f,
                                    last ? 0.5f : left ? 0.25f : -0.25f, 6e-8f, 24);
  const double lo = left ? 0.0 : -gap, hi = left ? gap : 0.0;
  double mu = (double)m32 * gap;
  if (!(mu > lo && mu < hi)) mu = 0.5 * (lo + hi);
  const double o = pole[org];
  auto get64 = [&](int j, double& g, double& zz) {
    g = pole[j] - o;
    zz = z[j];
  };
  mu = dc_solve<double>(get64, K, k, rho, lo, hi, mu, kEps, 120);
  if (lane == 0) {
    w.org[s + k] = s + org;
    w.mu[s + k] = mu;
    w.lam[s + k] = o + mu;
  }
}

// pole_j - lambda_k without cancellation
__device__ __forceinline__ double dc_gap(const Dc& w, int j, int k) { return (w.pole[j] - w.pole[w.org[k]]) - w.mu[k]; }

// the coupling entry for which the computed roots are exact (one warp)
__device__ void dc_coupling(const Dc& w, int s, int j, int lane) {
  const int K = w.K[s];
  double p = 1.0;
  for (int k = lane; k < K; k += 32) {
    const double g = -dc_gap(w, s + j, s + k);
    p *= k == j ? g : g / (w.pole[s + k] - w.pole[s + j]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) p *= __shfl_xor_sync(0xffffffffu, p, o);
  if (lane == 0) w.zh[s + j] = copysign(sqrt(fabs(p)), w.z[s + j]);
}

// row k of S: the merge's eigenvector k in the basis of its poles (one warp)
__device__ void dc_vector(const Dc& w, int s, int k, int lane) {
  const int K = w.K[s];
  double* row = w.S + (size_t)(s + k) * w.N + s;
  double nn = 0.0;
  for (int j = lane; j < K; j += 32) {
    const double t = w.zh[s + j] / dc_gap(w, s + j, s + k);
    row[j] = t;
    nn = fma(t, t, nn);
  }
  nn = 1.0 / sqrt(warp_sum(nn));
  for (int j = lane; j < K; j += 32) row[j] *= nn;
  if (lane == 0) w.out[s + k] = w.lam[s + k];
}

// output rows [r0, r0 + 16) x components [c0, c0 + 32) of a merge: S times the poles' rows, deflated
// rows copied.  128 threads, 4 rows x 1 component each.  Poles that are zero on these components
// (of the other half) are left out.
constexpr int kDcTr = 16, kDcTc = 32;
__device__ void dc_tile(const Dc& w, int s, int mid, int e, int r0, int c0, int t) {
  const int K = w.K[s], N = w.N;
  const int c = c0 + (t & 31), q = t >> 5;
  const int skip = c0 + kDcTc <= mid ? 2 : c0 >= mid ? 1 : 0;      // pole type that is zero here
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const bool ok = c < e;
  const int r = s + r0 + 4 * q;
  if (r0 < K) {
    const double* S0 = w.S + (size_t)r * N + s;
    const int nu = min(4, s + K - r);                // rows of this thread that are eigenvectors
    for (int j0 = 0; j0 < K; j0 += 4) {
      int cj[4];
      double x[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) cj[v] = j0 + v < K ? w.col[s + j0 + v] : skip << 28;
#pragma unroll
      for (int v = 0; v < 4; ++v)
        x[v] = ok && (cj[v] >> 28) != skip && j0 + v < K ? w.Qa[(size_t)(cj[v] & 0xfffffff) * N + c] : 0.0;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        if (j0 + v >= K || (cj[v] >> 28) == skip) continue;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (u < nu) acc[u] = fma(S0[(size_t)u * N + j0 + v], x[v], acc[u]);
      }
    }
  }
  if (!ok) return;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = r + u;
    if (i >= e) break;
    w.Qb[(size_t)i * N + c] = i < s + K ? acc[u] : w.Qa[(size_t)w.src[i] * N + c];
  }
}

// merge m of the level with half blocks of h rows
__device__ __forceinline__ bool dc_range(const Dc& w, int m, int h, int& s, int& mid, int& e) {
  s = 2 * h * m;
  mid = s + h;
  e = min(w.N, s + 2 * h);
  return mid < e;
}
// a block without a partner: unchanged
__device__ void dc_carry(const Dc& w, int s, int e) {
  const int n = e - s;
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const size_t i = (size_t)(s + t / n) * w.N + s + t % n;
    w.Qb[i] = w.Qa[i];
  }
}

constexpr int kDcBlock = 16;         // rows of a merge that one CTA does whole
__global__ void __launch_bounds__(kDcThreads) k_dc_merge(Dc w, int h) {
  extern __shared__ double dcs[];
  int s, mid, e;
  if (!dc_range(w, blockIdx.x, h, s, mid, e)) {
    dc_carry(w, s, e);
    return;
  }
  dc_prepare(w, s, mid, e, dcs);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, K = w.K[s];
  __shared__ float buf[kDcThreads / 32][2 * kDcBlock];
  for (int k = warp; k < K; k += kDcThreads / 32) {
    dc_root(w, s, k, lane, buf[warp]);
    __syncwarp();
  }
  __syncthreads();
  for (int j = warp; j < K; j += kDcThreads / 32) dc_coupling(w, s, j, lane);
  __syncthreads();
  for (int k = warp; k < K; k += kDcThreads / 32) dc_vector(w, s, k, lane);
  __syncthreads();
  const int n = e - s, tr = (n + kDcTr - 1) / kDcTr, tc = (n + kDcTc - 1) / kDcTc;
  for (int t = threadIdx.x / 128; t < tr * tc; t += kDcThreads / 128)
    dc_tile(w, s, mid, e, (t / tc) * kDcTr, s + (t % tc) * kDcTc, threadIdx.x % 128);
  __syncthreads();
  for (int t = s + threadIdx.x; t < e; t += kDcThreads) w.d[t] = w.out[t];
}
__global__ void __launch_bounds__(kDcThreads) k_dc_prepare(Dc w, int h) {
  extern __shared__ double dcs[];
  int s, mid, e;
  if (dc_range(w, blockIdx.x, h, s, mid, e)) dc_prepare(w, s, mid, e, dcs);
}
// phase 0: roots, 1: coupling, 2: vectors; one warp per row of the matrix
template <int PHASE> __global__ void __launch_bounds__(128) k_dc_rows(Dc w, int h) {
  extern __shared__ float dcf[];
  const int i = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= w.N) return;
  int s, mid, e;
  if (!dc_range(w, i / (2 * h), h, s, mid, e)) return;
  if (i - s >= w.K[s]) return;
  if (PHASE == 0) dc_root(w, s, i - s, lane, dcf + (size_t)(threadIdx.x >> 5) * 2 * (e - s));
  else if (PHASE == 1) dc_coupling(w, s, i - s, lane);
  else dc_vector(w, s, i - s, lane);
}
__global__ void __launch_bounds__(128) k_dc_gemm(Dc w, int h) {
  int s, mid, e;
  const bool merge = dc_range(w, blockIdx.z, h, s, mid, e);
  if (!merge) {
    if (blockIdx.x == 0 && blockIdx.y == 0) dc_carry(w, s, e);
    return;
  }
  const int r0 = blockIdx.y * kDcTr, c0 = s + blockIdx.x * kDcTc;
  if (s + r0 >= e || c0 >= e) return;
  dc_tile(w, s, mid, e, r0, c0, threadIdx.x);
  if (blockIdx.x == 0)
    for (int t = s + r0 + threadIdx.x; t < min(e, s + r0 + kDcTr); t += 128) w.d[t] = w.out[t];
}

// --------------------------------------------------------- back transformation
// Reflectors in groups of four: H_j H_j+1 H_j+2 H_j+3 = I - V T V^H with T upper triangular (the compact
// WY form of Schreiber & Van Loan), so the four inner products of a group share one pass and one
// reduction.  tri[4 g + a][b] = T of group g (10 entries used).
template <typename C>
__global__ void __launch_bounds__(32) k_wy(const C* __restrict__ V, const C* __restrict__ tau, int N, int nref,
                                           C* __restrict__ tri) {
  const int j0 = 4 * blockIdx.x, lane = threadIdx.x;
  const C zero = zero_of(C());
  C dot[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) dot[a][b] = zero;
  for (int k = j0 + lane; k < N; k += 32) {
    C v[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) v[a] = j0 + a < nref ? V[(size_t)(j0 + a) * N + k] : zero;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = a + 1; b < 4; ++b) dot[a][b] = mad(conj_of(v[a]), v[b], dot[a][b]);
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = a + 1; b < 4; ++b) dot[a][b] = warp_sum(dot[a][b]);
  if (lane) return;
  // column b of T: T_bb = tau_b, T_ab = -tau_b sum_c T_ac (v_c^H v_b), c = a .. b - 1
  C T[4][4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const C tb = j0 + b < nref ? tau[j0 + b] : zero;
    T[b][b] = tb;
#pragma unroll
    for (int a = 0; a < b; ++a) {
      C s = zero;
#pragma unroll
      for (int c = a; c < b; ++c) s = mad(T[a][c], dot[c][b], s);
      T[a][b] = neg(mul(tb, s));
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) tri[(size_t)(j0 + a) * 4 + b] = b >= a ? T[a][b] : zero;
}

__device__ __forceinline__ void sum4(double (&s)[4]) { warp_sum4(s[0], s[1], s[2], s[3]); }
__device__ __forceinline__ void sum4(double2 (&s)[4]) {
  warp_sum4(s[0].x, s[0].y, s[1].x, s[1].y);
  warp_sum4(s[2].x, s[2].y, s[3].x, s[3].y);
}

// z <- H_0 (H_1 (... z)) for one eigenvector per warp: Z row (real, N) -> out row (N); the vector stays
// in registers (lane l holds components l + 32 q), the reflectors stream from L2.  The eigenvalues go
// back to the matrix's scale here.
template <typename C, int E>
__global__ void __launch_bounds__(64) k_backtransform(const double* __restrict__ Z, const C* __restrict__ V,
                                                      const C* __restrict__ tri, int N, int nref,
                                                      C* __restrict__ out, const jac::Barrier* __restrict__ bar,
                                                      double* __restrict__ d) {
  const int lane = threadIdx.x & 31, i = blockIdx.x * 2 + (threadIdx.x >> 5);
  if (i >= N) return;
  if (lane == 0) d[i] *= pow2(2046 - scale_exponent(bar->top));
  C z[E];
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int k = lane + 32 * q;
    const double t = k < N ? Z[(size_t)i * N + k] : 0.0;
    if constexpr (sizeof(C) == 16) z[q] = C{t, 0.0};
    else z[q] = t;
  }
  for (int j0 = (nref - 1) / 4 * 4; j0 >= 0; j0 -= 4) {
    const C* v[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) v[a] = V + (size_t)min(j0 + a, nref - 1) * N;   // beyond the last: T is zero there
    C s[4], t[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) s[a] = zero_of(C());
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const int k = lane + 32 * q;
      if (32 * q + 31 <= j0) continue;                 // the reflectors are zero up to j0 (warp-uniform)
#pragma unroll
      for (int a = 0; a < 4; ++a) s[a] = mad(conj_of(k < N ? __ldg(v[a] + k) : zero_of(C())), z[q], s[a]);
    }
    sum4(s);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      t[a] = zero_of(C());
#pragma unroll
      for (int b = a; b < 4; ++b) t[a] = mad(__ldg(tri + (size_t)(j0 + a) * 4 + b), s[b], t[a]);
      t[a] = neg(t[a]);
    }
#pragma unroll
    for (int q = 0; q < E; ++q) {                      // the reflectors again, from L1
      const int k = lane + 32 * q;
      if (32 * q + 31 <= j0) continue;
#pragma unroll
      for (int a = 0; a < 4; ++a) z[q] = mad(t[a], k < N ? __ldg(v[a] + k) : zero_of(C()), z[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int k = lane + 32 * q;
    if (k < N) out[(size_t)i * N + k] = z[q];
  }
}

// ------------------------------------------------------------------- host side
static int tri_grid(dftfe_ham h, int N) {
  // one CTA up to 40 rows (no grid barrier: 5.5 us a column at 32 rows); beyond that enough CTAs that a
  // column's pass over the rows costs no more than the barrier (64 rows: 8.6 us a column in one
  // CTA, 5.6 us in five; 320 rows: 8.7 us in 64, 7.0 us in 128)
  return N <= 40 ? 1 : (int)std::min<int64_t>(h->sm_count, std::max<int64_t>(2, (int64_t)N * N / 800));
}
template <typename C> static size_t tri_smem(int N, int G) {
  return sizeof(C) * ((size_t)((N + G - 1) / G) * N + 3 * (size_t)N);
}

template <typename C, int E>
static void launch_back(cudaStream_t s, const Dc& w, const C* V, const C* tri, int nref, C* out,
                        const jac::Barrier* bar) {
  DFTFE_LAUNCH((k_backtransform<C, E>), (unsigned)((w.N + 1) / 2), 64, 0, s, w.Qa, V, tri, w.N, nref, out, bar, w.d);
}

}  // namespace eig

constexpr size_t kTriMaxSmem = 220 * 1024;
bool tridiag_applicable(dftfe_ham h, int N, bool cplx) {
  const int G = eig::tri_grid(h, N);
  return N <= 2048 && (cplx ? N <= 1024 : true) &&
         (cplx ? eig::tri_smem<double2>(N, G) : eig::tri_smem<double>(N, G)) <= kTriMaxSmem;
}

// A (lower triangle) -> eigenvalues in d (unsorted), eigenvectors as rows of VT
template <typename C>
void tridiag_eig(dftfe_ham h, const C* A, int N, double* d, C* VT, int* d_status) {
  using namespace eig;
  cudaStream_t st = h->stream;
  const size_t NN = (size_t)N * N;
  const bool cplx = sizeof(C) == 16;
  // doubles: e, pole, z, lam, mu, zh, out, rho (8 N), Q a, Q b, S (3 N^2); C: V (N^2), tau, exchange, WY (9 N)
  double* ws = (double*)ws_get(h, "eig_dc", sizeof(double) * (3 * NN + 8 * (size_t)N));
  C* wc = (C*)ws_get(h, cplx ? "eig_refl_z" : "eig_refl", sizeof(C) * (NN + 9 * (size_t)N + 16));
  int* wi = (int*)ws_get(h, "eig_idx", sizeof(int) * 5 * (size_t)N);
  jac::Barrier* bar = (jac::Barrier*)ws_get(h, "eig_bar", sizeof(jac::Barrier));
  C *V = wc, *tau = wc + NN, *xp = tau + N, *xr = xp + 2 * (size_t)N, *tri = xr + 2 * (size_t)N;
  Dc w;
  w.N = N;
  w.d = d;
  w.Qa = ws;
  w.Qb = ws + NN;
  w.S = ws + 2 * NN;
  double* v1 = ws + 3 * NN;
  w.e = v1;
  w.pole = v1 + N;
  w.z = v1 + 2 * (size_t)N;
  w.lam = v1 + 3 * (size_t)N;
  w.mu = v1 + 4 * (size_t)N;
  w.zh = v1 + 5 * (size_t)N;
  w.out = v1 + 6 * (size_t)N;
  w.rho = v1 + 7 * (size_t)N;
  w.col = wi;
  w.typ = wi + N;
  w.org = wi + 2 * (size_t)N;
  w.src = wi + 3 * (size_t)N;
  w.K = wi + 4 * (size_t)N;
  jac::init_barrier(st, bar, h->wait_limit, (unsigned int)h->wait_missing);
  DFTFE_CHECK_CUDA(cudaMemsetAsync(d_status, 0, sizeof(int), st));
  DFTFE_CHECK_CUDA(cudaMemsetAsync(ws, 0, sizeof(double) * 2 * NN, st));
  {
    const int G = tri_grid(h, N);
    const size_t sh = tri_smem<C>(N, G);
    DFTFE_CHECK_CUDA(cudaFuncSetAttribute(k_tridiag<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTriMaxSmem));
    int n = N;
    double* e = w.e;
    void* args[] = {&A, &n, &V, &tau, &d, &e, &xp, &xr, &bar, &d_status};
    DFTFE_CHECK_CUDA(cudaLaunchCooperativeKernel((const void*)k_tridiag<C>, dim3(G), dim3(kTriThreads), args, sh, st));
    g_launches.fetch_add(1, std::memory_order_relaxed);
  }
  const unsigned nb = (unsigned)((N + 127) / 128);
  DFTFE_LAUNCH(k_dc_init, nb, 128, 0, st, w);
  DFTFE_LAUNCH(k_dc_start, nb, 128, 0, st, w);
  for (int hh = 1; hh < N; hh *= 2) {
    const unsigned merges = (unsigned)((N + 2 * hh - 1) / (2 * hh));
    const int n = std::min(N, 2 * hh);
    const size_t sh = (size_t)n * (4 * sizeof(double) + 4 * sizeof(int));
    if (n <= kDcBlock) {
      DFTFE_LAUNCH(k_dc_merge, merges, kDcThreads, sh, st, w, hh);
    } else {
      DFTFE_CHECK_CUDA(cudaFuncSetAttribute(k_dc_rows<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(100 * 1024)));
      DFTFE_CHECK_CUDA(cudaFuncSetAttribute(k_dc_prepare, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(100 * 1024)));
      DFTFE_LAUNCH(k_dc_prepare, merges, kDcThreads, sh, st, w, hh);
      const unsigned rows = (unsigned)((N + 3) / 4);
      DFTFE_LAUNCH(k_dc_rows<0>, rows, 128, (size_t)n * 8 * sizeof(float), st, w, hh);
      DFTFE_LAUNCH(k_dc_rows<1>, rows, 128, 0, st, w, hh);
      DFTFE_LAUNCH(k_dc_rows<2>, rows, 128, 0, st, w, hh);
      DFTFE_LAUNCH(k_dc_gemm, dim3((unsigned)((n + kDcTc - 1) / kDcTc), (unsigned)((n + kDcTr - 1) / kDcTr), merges),
                   128, 0, st, w, hh);
    }
    std::swap(w.Qa, w.Qb);
  }
  const int nref = std::max(N - 1, 1);          // N = 1: one reflector that is the identity
  if (N == 1) {
    DFTFE_CHECK_CUDA(cudaMemsetAsync(V, 0, sizeof(C), st));
    DFTFE_CHECK_CUDA(cudaMemsetAsync(tau, 0, sizeof(C), st));
  }
  DFTFE_LAUNCH(k_wy<C>, (unsigned)((nref + 3) / 4), 32, 0, st, V, tau, N, nref, tri);
  const int E = (N + 31) / 32;
  if (E <= 2) launch_back<C, 2>(st, w, V, tri, nref, VT, bar);
  else if (E <= 4) launch_back<C, 4>(st, w, V, tri, nref, VT, bar);
  else if (E <= 8) launch_back<C, 8>(st, w, V, tri, nref, VT, bar);
  else if (E <= 16) launch_back<C, 16>(st, w, V, tri, nref, VT, bar);
  else if (E <= 32) launch_back<C, 32>(st, w, V, tri, nref, VT, bar);
  else if constexpr (sizeof(C) == 8) launch_back<C, 64>(st, w, V, tri, nref, VT, bar);
}
template void tridiag_eig<double>(dftfe_ham, const double*, int, double*, double*, int*);
template void tridiag_eig<double2>(dftfe_ham, const double2*, int, double*, double2*, int*);

}  // namespace dftfe
