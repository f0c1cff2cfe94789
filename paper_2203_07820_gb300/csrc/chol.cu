// Blocked Cholesky factorisation S = L L^T and triangular inverse Z = L^-T for the
// Cholesky-Gram-Schmidt step (Sec. 3.2, Alg. 2 steps 2a and 3b), FP64, on all SMs.
//
// Right-looking, 32 x 32 blocks (textbook blocked Cholesky): for every block column k
//   1. factor the diagonal block A_kk = L_kk L_kk^T and invert it (one CTA, shared memory),
//   2. L_ik = A_ik L_kk^-T for the blocks below it (one CTA per block),
//   3. A_ij -= L_ik L_jk^T for the trailing lower blocks k < j <= i (one CTA per block).
// The inverse is then formed by doubling from the inverted diagonal blocks (k_tri_inv_pair) and
// written transposed as Z = L^-T (upper triangular), with L's strict upper triangle
// zeroed.  A pivot not above 1e-14 times its original diagonal entry (or not finite)
// records DFTFE_ERR_NOT_SPD; the later steps still run on finite stand-in values, so the
// caller reads the status once after the factorisation.
#include "internal.h"

namespace dftfe {

namespace chol {
constexpr int NB = 32;

__device__ __forceinline__ int rows_of(int blk, int N) { return min(NB, N - blk * NB); }

// load the 32 x 32 block (bi, bj) of A (row-major, N x N) into s (zero outside N)
__device__ __forceinline__ void load_block(const double* A, int N, int bi, int bj, double (*s)[NB + 1]) {
  for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) {
    const int r = t / NB, c = t % NB;
    const int gi = bi * NB + r, gj = bj * NB + c;
    s[r][c] = (gi < N && gj < N) ? A[(int64_t)gi * N + gj] : 0.0;
  }
}
}  // namespace chol

// original diagonal (for the pivot test) and a cleared status word
__global__ void k_chol_save_diag(const double* __restrict__ A, int N, double* __restrict__ d0, int* status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) d0[i] = A[(int64_t)i * N + i];
  if (i == 0) *status = 0;
}

// step 1: factor and invert the diagonal block k.  Column by column, with the inverse formed alongside
// (right-looking forward substitution on the identity): one reciprocal square root per column and no
// division, since the FP64 pipe's latency sets the pace (80 us a block with a division per
// entry and one thread per column of the inverse).
__global__ void __launch_bounds__(256) k_chol_diag(double* __restrict__ A, int N, int k, const double* __restrict__ d0,
                                                   double* __restrict__ Linv, int* status) {
  using namespace chol;
  __shared__ double a[NB][NB + 1];
  __shared__ double y[NB][NB + 1];
  __shared__ double rpiv;
  const int nb = rows_of(k, N), off = k * NB;
  load_block(A, N, k, k, a);
  for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) y[t / NB][t % NB] = t / NB == t % NB ? 1.0 : 0.0;
  __syncthreads();
  for (int j = 0; j < nb; ++j) {
    if (threadIdx.x == 0) {
      const double d = a[j][j], dorig = d0[off + j];
      if (!(d > 1e-14 * dorig) || !(dorig > 0.0) || !isfinite(d)) {
        atomicExch(status, (int)DFTFE_ERR_NOT_SPD);
        rpiv = 1.0;                                   // finite stand-in; the status stays set
        a[j][j] = 1.0;
      } else {
        rpiv = rsqrt(d);
        a[j][j] = d * rpiv;
      }
    }
    __syncthreads();
    if (threadIdx.x < NB) {
      const int i = threadIdx.x;
      if (i > j && i < nb) a[i][j] *= rpiv;
    } else if (threadIdx.x < 2 * NB) {
      const int c = threadIdx.x - NB;
      if (c <= j) y[j][c] *= rpiv;
    }
    __syncthreads();
    // trailing lower triangle of the block, and the rows of the inverse below j
    const int m = nb - j - 1;
    for (int t = threadIdx.x; t < m * NB; t += blockDim.x) {
      const int i = j + 1 + t / NB, l = t % NB;
      const double lij = a[i][j];
      if (l > j) {
        if (l <= i) a[i][l] = fma(-lij, a[l][j], a[i][l]);
      } else {
        y[i][l] = fma(-lij, y[j][l], y[i][l]);
      }
    }
    __syncthreads();
  }
  for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) {
    const int r = t / NB, c = t % NB;
    if (r < nb && c < nb) {
      A[(int64_t)(off + r) * N + off + c] = c <= r ? a[r][c] : 0.0;
      Linv[(int64_t)(off + r) * N + off + c] = y[r][c];
    }
  }
}

// step 2: L_ik = A_ik L_kk^-T for the blocks i > k (block i = k + 1 + blockIdx.x)
__global__ void __launch_bounds__(256) k_chol_panel(double* __restrict__ A, int N, int k, const double* __restrict__ Linv) {
  using namespace chol;
  __shared__ double p[NB][NB + 1];
  __shared__ double li[NB][NB + 1];
  const int bi = k + 1 + blockIdx.x;
  load_block(A, N, bi, k, p);
  load_block(Linv, N, k, k, li);
  __syncthreads();
  for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) {
    const int r = t / NB, c = t % NB;
    double s = 0.0;
#pragma unroll 8
    for (int l = 0; l <= c; ++l) s = fma(p[r][l], li[c][l], s);     // L_kk^-1 is lower
    const int gi = bi * NB + r, gj = k * NB + c;
    if (gi < N && gj < N) A[(int64_t)gi * N + gj] = s;
  }
}

// step 3: A_ij -= L_ik L_jk^T for k < j <= i (blockIdx.x enumerates the lower pairs)
__global__ void __launch_bounds__(256) k_chol_update(double* __restrict__ A, int N, int k) {
  using namespace chol;
  __shared__ double li[NB][NB + 1];
  __shared__ double lj[NB][NB + 1];
  // pair index t -> (i, j), i >= j, both counted from k + 1
  const int t = blockIdx.x;
  int i = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
  while (i * (i + 1) / 2 > t) --i;
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  const int j = t - i * (i + 1) / 2;
  const int bi = k + 1 + i, bj = k + 1 + j;
  load_block(A, N, bi, k, li);
  load_block(A, N, bj, k, lj);
  __syncthreads();
  for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
    const int r = e / NB, c = e % NB;
    const int gi = bi * NB + r, gj = bj * NB + c;
    if (gi >= N || gj >= N || (bi == bj && c > r)) continue;
    double s = 0.0;
#pragma unroll 8
    for (int l = 0; l < NB; ++l) s = fma(li[r][l], lj[c][l], s);
    A[(int64_t)gi * N + gj] -= s;
  }
}

// inverse by doubling: with the diagonal blocks of h rows inverted, pairs of them give
//   [[A, 0], [C, B]]^-1 = [[A^-1, 0], [-B^-1 C A^-1, B^-1]],
// two products per doubling (PHASE 0: T = C A^-1, PHASE 1: -B^-1 T), each spread over 16 x 16 tiles
// on all SMs (a block row at a time, one CTA per block of the row, took N / 32 launches of up to N / 32
// serial 32^3 products: 1.14 ms at N = 512).
constexpr int TI = 16;
template <int PHASE>
__global__ void __launch_bounds__(TI * TI) k_tri_inv_pair(const double* __restrict__ L, int N, int h,
                                                          double* __restrict__ Linv, double* __restrict__ T) {
  __shared__ double p[TI][TI + 1];
  __shared__ double q[TI][TI + 1];
  const int s = 2 * h * blockIdx.x, mid = s + h, r0 = mid + TI * blockIdx.y, c0 = s + TI * blockIdx.z;
  if (mid >= N || r0 >= min(N, mid + h)) return;
  const int tr = threadIdx.x / TI, tc = threadIdx.x % TI;
  const int r = r0 + tr, c = c0 + tc, end = min(N, mid + h);
  // PHASE 0: sum over k in [s, mid), A^-1 lower: k >= c0; PHASE 1: k in [mid, end), B^-1 lower: k <= r0 + 15
  const int k0 = PHASE == 0 ? c0 : mid, k1 = PHASE == 0 ? mid : min(end, r0 + TI);
  double acc = 0.0;
  for (int k = k0; k < k1; k += TI) {
    const double* P = PHASE == 0 ? L : Linv;
    const double* Q = PHASE == 0 ? Linv : T;
    p[tr][tc] = r < end && k + tc < k1 ? P[(int64_t)r * N + k + tc] : 0.0;
    q[tr][tc] = k + tr < k1 ? Q[(int64_t)(k + tr) * N + c] : 0.0;
    __syncthreads();
#pragma unroll
    for (int l = 0; l < TI; ++l) acc = fma(p[tr][l], q[l][tc], acc);
    __syncthreads();
  }
  if (r < end) {
    if (PHASE == 0) T[(int64_t)r * N + c] = acc;
    else Linv[(int64_t)r * N + c] = -acc;
  }
}

// Z = (L^-1)^T (upper triangular, zero below the diagonal); L's strict upper triangle zeroed
__global__ void k_tri_finish(double* __restrict__ L, const double* __restrict__ Linv, double* __restrict__ Z, int N) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)N * N) return;
  const int r = (int)(t / N), c = (int)(t % N);
  Z[t] = c >= r ? Linv[(int64_t)c * N + r] : 0.0;
  if (c > r) L[t] = 0.0;
}

static unsigned nblk_c(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

void cholesky_blocked(dftfe_ham h, double* A, int N, int* d_status) {
  using namespace chol;
  cudaStream_t s = h->stream;
  const int nbk = (N + NB - 1) / NB;
  double* d0 = (double*)ws_get(h, "chol_d0", sizeof(double) * (size_t)N);
  double* Linv = (double*)ws_get(h, "chol_linv", sizeof(double) * (size_t)N * N);
  ProfScope ps(h, "potrf");
  DFTFE_LAUNCH(k_chol_save_diag, nblk_c(N), 256, 0, s, A, N, d0, d_status);
  for (int k = 0; k < nbk; ++k) {
    DFTFE_LAUNCH(k_chol_diag, 1, 256, 0, s, A, N, k, d0, Linv, d_status);
    const int below = nbk - k - 1;
    if (below == 0) break;
    DFTFE_LAUNCH(k_chol_panel, below, 256, 0, s, A, N, k, Linv);
    DFTFE_LAUNCH(k_chol_update, below * (below + 1) / 2, 256, 0, s, A, N, k);
  }
}

void tri_inverse_blocked(dftfe_ham h, double* L, double* Z, int N) {
  using namespace chol;
  cudaStream_t s = h->stream;
  const int nbk = (N + NB - 1) / NB;
  double* Linv = (double*)ws_get(h, "chol_linv", sizeof(double) * (size_t)N * N);
  ProfScope ps(h, "trtri");
  for (int hb = 1; hb < nbk; hb *= 2) {           // Z is the scratch of the products until it is written
    const int hh = hb * NB;
    const dim3 grid((unsigned)((N + 2 * hh - 1) / (2 * hh)), (unsigned)(hh / TI), (unsigned)(hh / TI));
    DFTFE_LAUNCH(k_tri_inv_pair<0>, grid, TI * TI, 0, s, L, N, hh, Linv, Z);
    DFTFE_LAUNCH(k_tri_inv_pair<1>, grid, TI * TI, 0, s, L, N, hh, Linv, Z);
  }
  DFTFE_LAUNCH(k_tri_finish, nblk_c((int64_t)N * N), 256, 0, s, L, Linv, Z, N);
}

}  // namespace dftfe
