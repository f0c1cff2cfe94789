// Mesh (a1), cell Hamiltonians (a2) and nonlocal projector setup (a3).
//
// a1 (Sec. 2.3): structured periodic hexahedral mesh of GLL spectral elements, the
//    cell -> global map and the lumped diagonal mass M (text after Eq. hep).  On a
//    uniform periodic mesh M = M1x (x) M1y (x) M1z with M1 the 1D lumped mass, which
//    is how the device builds it.
// a2 (Sec. 4.2, Eq. quadLocal): H~^c = D_c^-1/2 (K^c + V^c) D_c^-1/2 (Eq. hep, Eq. celldgemm),
//    V^c one axis at a time from the tensor-product quadrature, the GLL stiffness K^c =
//    1/2 int grad N . grad N as its Kronecker terms.
// a3 (Eq. nonlocalHamDiscrete, Alg. 4): C_ja = M_jj chi_a(x_j) (GLL collocation), stored
//    as C~ = M^1/2 chi in CSR by projector and by node.
#include "internal.h"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace dftfe {

std::atomic<int64_t> g_launches{0};
static thread_local std::string t_last_error;
void set_error(const std::string& msg) { t_last_error = msg; }
void clear_error() { t_last_error.clear(); }
const char* last_error() { return t_last_error.c_str(); }


void* DevBuf::get(size_t need) {
  if (need <= bytes && ptr) return ptr;
  if (ptr) {
    cudaFree(ptr);
    ptr = nullptr;
    bytes = 0;
  }
  size_t alloc = std::max<size_t>(need, 256);
  DFTFE_CHECK_CUDA(cudaMalloc(&ptr, alloc));
  bytes = alloc;
  return ptr;
}
void DevBuf::release() {
  if (ptr) cudaFree(ptr);
  ptr = nullptr;
  bytes = 0;
}

// buffers that live only inside one pass tail (CholGS, Rayleigh-Ritz, residuals): in a batched
// pass they come from the batch's shared tail workspace
static bool tail_buffer(const char* name) {
  static const char* const names[] = {"S", "Zinv", "gram_part", "Hhat", "Q", "W", "chol_d0", "chol_linv",
                                      "eig_V", "eigz_V", "eig_vec", "eig_perm", "eig_dc", "eig_refl", "eig_refl_z",
                                      "eig_idx", "resid_part", "coldot_part",
                                      "gram32_part", "rotmix_Zf", "rotmix_zd", "Hz", "Qz", "rot_tc_tiles",
                                      "rot_tc_zd", "rot_tc_out", "gram_tc_part", "slices_x", "slices_xe"};
  for (const char* n : names)
    if (std::strcmp(n, name) == 0) return true;
  return false;
}

void* ws_get(dftfe_ham h, const char* name, size_t bytes) {
  DevBuf& b = (h->tail_ws && tail_buffer(name)) ? (*h->tail_ws)[name] : h->ws[name];
  if (bytes > b.bytes && b.ptr) DFTFE_CHECK_CUDA(cudaStreamSynchronize(h->stream));
  return b.get(bytes);
}

ProfScope::ProfScope(dftfe_ham ham, const char* name) : h(ham) {
  if (!h || !h->profiling) return;
  t = &h->timers[name];
  if (t->used == t->events.size()) {
    cudaEvent_t a, b;
    DFTFE_CHECK_CUDA(cudaEventCreate(&a));
    DFTFE_CHECK_CUDA(cudaEventCreate(&b));
    t->events.push_back({a, b});
  }
  auto& ev = t->events[t->used++];
  e1 = ev.second;
  DFTFE_CHECK_CUDA(cudaEventRecord(ev.first, h->stream));
}
ProfScope::~ProfScope() {
  if (t) {
    cudaEventRecord(e1, h->stream);
    t->launches++;
  }
}

// ------------------------------------------------------------------ kernels

// cell_map[c*nc + (a + n1*(b + n1*cc))] = global node of local (a, b, cc) in cell c
__global__ void k_cell_map(int32_t* map, int64_t Nc, int n1, int p, int nx, int ny,
                           int64_t gx, int64_t gy, int64_t gz) {
  const int nc = n1 * n1 * n1;
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= Nc * nc) return;
  int64_t c = t / nc;
  int l = (int)(t % nc);
  int a = l % n1, b = (l / n1) % n1, cc = l / (n1 * n1);
  int64_t cx = c % nx, cy = (c / nx) % ny, cz = c / ((int64_t)nx * ny);
  int64_t ix = (cx * p + a) % gx, iy = (cy * p + b) % gy, iz = (cz * p + cc) % gz;
  map[t] = (int32_t)(ix + gx * (iy + gy * iz));
}

// M_jj = m1x[ix] m1y[iy] m1z[iz]; also M^-1/2.
__global__ void k_mass(double* mass, double* minvsqrt, const double* m1x, const double* m1y,
                       const double* m1z, int64_t gx, int64_t gy, int64_t M) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= M) return;
  int64_t ix = j % gx, iy = (j / gx) % gy, iz = j / (gx * gy);
  double m = m1x[ix] * m1y[iy] * m1z[iz];
  mass[j] = m;
  minvsqrt[j] = 1.0 / sqrt(m);
}

// Dense cell matrices H~^c = D_c^-1/2 (K^c + V^c) D_c^-1/2 from the tensor-product form of Eq.
// quadLocal: with B[q][aa'] = l_a(x_q) l_a'(x_q) / sqrt(w^_a w^_a') (pairs a <= a', w^ the
// assembled 1D weights) and v = w_q w_q' w_q'' V,
//   V^c[(abc), (a'b'c')] = sum_qx,qy,qz B[qx][aa'] B[qy][bb'] B[qz][cc'] v[qz][qy][qx],
// one axis at a time: per pair cc' the sums over qz, qx and qy, then the two (N^2 x N^2) blocks
// (c, c') and (c', c) are written in runs of N^2 with the kinetic term added.  About 200,000
// multiply-adds per cell at p = 6 against 20 million for the product table times V of Eq.
// gemmLoc (and no 162 MB table), so the writes of the matrices bound it.  One CTA takes one
// cell and every gridDim.y-th pair cc'.
struct CellTab {
  const double* B;        // nq1 x npair
  const double* K;        // N x N: the 1D kinetic matrix without its mesh factor
  const double* om;       // N: w_a / w^_a
  double kx, ky, kz;      // 1/2 (2/h_d)^2
};
__global__ void __launch_bounds__(256) k_cell_matrices(const double* __restrict__ v, CellTab tab, int N, int nq,
                                                       int nodal, double* __restrict__ Hc) {
  extern __shared__ double cms[];
  const int np = N * (N + 1) / 2, n2 = N * N, nc = n2 * N;
  double* sv = cms;                        // nq^3
  double* sB = sv + nq * nq * nq;          // nq x np
  double* sK = sB + nq * np;               // n2
  double* som = sK + n2;                   // N
  double* t1 = som + N;                    // nq x nq (qy, qx)
  double* t2 = t1 + nq * nq;               // np x nq (aa', qy)
  double* t3 = t2 + np * nq;               // np x np (aa', bb')
  uint8_t* pr = reinterpret_cast<uint8_t*>(t3 + np * np);   // n2: pair index of (a, a')
  const int64_t cell = blockIdx.x;
  for (int t = threadIdx.x; t < nq * nq * nq; t += 256) sv[t] = v[cell * nq * nq * nq + t];
  for (int t = threadIdx.x; t < nq * np; t += 256) sB[t] = tab.B[t];
  for (int t = threadIdx.x; t < n2; t += 256) {
    sK[t] = tab.K[t];
    const int a = min(t / N, t % N), b = max(t / N, t % N);
    pr[t] = (uint8_t)(a * N - a * (a - 1) / 2 + b - a);
  }
  for (int t = threadIdx.x; t < N; t += 256) som[t] = tab.om[t];
  __syncthreads();
  double* H = Hc + cell * (int64_t)nc * nc;
  int c = 0, cp = 0;
  for (int P = 0; P < np; ++P, ++cp) {
    if (cp == N) {
      ++c;
      cp = c;
    }
    if (P % (int)gridDim.y != (int)blockIdx.y) continue;
    if (!nodal) {
      for (int t = threadIdx.x; t < nq * nq; t += 256) {
        double s = 0.0;
        for (int q = 0; q < nq; ++q) s = fma(sB[q * np + P], sv[q * nq * nq + t], s);
        t1[t] = s;
      }
      __syncthreads();
      for (int t = threadIdx.x; t < np * nq; t += 256) {
        const int a = t / nq, qy = t - a * nq;
        double s = 0.0;
        for (int q = 0; q < nq; ++q) s = fma(sB[q * np + a], t1[qy * nq + q], s);
        t2[t] = s;
      }
      __syncthreads();
      for (int t = threadIdx.x; t < np * np; t += 256) {
        const int a = t / np, b = t - a * np;
        double s = 0.0;
        for (int q = 0; q < nq; ++q) s = fma(sB[q * np + b], t2[a * nq + q], s);
        t3[t] = s;
      }
      __syncthreads();
    }
    // rows (a, b, c), columns (a', b', c'), and the transposed block
    for (int t = threadIdx.x; t < n2 * n2; t += 256) {
      const int r = t / n2, k = t - r * n2;
      const int b = r / N, a = r - b * N, b2 = k / N, a2 = k - b2 * N;
      double h = nodal ? 0.0 : t3[pr[a * N + a2] * np + pr[b * N + b2]];
      if (c == cp) {
        if (nodal && r == k) h = sv[c * n2 + r];
        if (b == b2) h = fma(tab.kx * sK[a * N + a2], som[b] * som[c], h);
        if (a == a2) h = fma(tab.ky * sK[b * N + b2], som[a] * som[c], h);
      }
      if (r == k) h = fma(tab.kz * sK[c * N + cp], som[a] * som[b], h);
      H[(int64_t)(c * n2 + r) * nc + cp * n2 + k] = h;
      if (c != cp) H[(int64_t)(cp * n2 + r) * nc + c * n2 + k] = h;
    }
    __syncthreads();
  }
}

__global__ void k_scale_by_sqrt_mass(double* out, const double* chi, const int32_t* node,
                                     const double* mass, int64_t n) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < n) out[t] = sqrt(mass[node[t]]) * chi[t];
}

__global__ void k_gather_vals(double* out, float* out32, const double* in, const int64_t* perm, int64_t n) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  out[t] = in[perm[t]];
  out32[t] = (float)in[perm[t]];
}

static unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

template <class T>
static T* dev_upload(const std::vector<T>& v, cudaStream_t s) {
  T* p = nullptr;
  DFTFE_CHECK_CUDA(cudaMalloc(&p, std::max<size_t>(v.size(), 1) * sizeof(T)));
  if (!v.empty())
    DFTFE_CHECK_CUDA(cudaMemcpyAsync(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, s));
  return p;
}

static void free_nonlocal(dftfe_ham h) {
  cudaFree(h->d_h); cudaFree(h->d_prow); cudaFree(h->d_pnode); cudaFree(h->d_pval);
  cudaFree(h->d_snode); cudaFree(h->d_srow); cudaFree(h->d_sproj); cudaFree(h->d_sval);
  cudaFree(h->d_nptr_all); cudaFree(h->d_sperm); cudaFree(h->d_pval_z); cudaFree(h->d_sval_z);
  cudaFree(h->d_pval_z32); cudaFree(h->d_sval_z32); cudaFree(h->d_pgroup);
  cudaFree(h->d_sval32);
  h->d_sval32 = nullptr;
  h->d_pgroup = nullptr;
  h->npgroup = 0;
  h->d_pval_z32 = nullptr; h->d_sval_z32 = nullptr;
  h->d_h = nullptr; h->d_prow = nullptr; h->d_pnode = nullptr; h->d_pval = nullptr;
  h->d_snode = nullptr; h->d_srow = nullptr; h->d_sproj = nullptr; h->d_sval = nullptr;
  h->d_nptr_all = nullptr; h->d_sperm = nullptr; h->d_pval_z = nullptr; h->d_sval_z = nullptr;
  h->nproj = 0;
  h->nsup = 0;
  h->nnz = 0;
  h->kpoint_nl = false;   // the phased projector values belong to the old CSR
}

}  // namespace dftfe

using namespace dftfe;

extern "C" dftfe_status dftfe_mesh_create(const dftfe_mesh_desc* d, dftfe_mesh* out) {
  ABI_BEGIN
  DFTFE_REQUIRE(d && out, "null argument");
  DFTFE_REQUIRE(d->degree >= 1 && d->degree <= 8, "degree must be in 1..8");
  DFTFE_REQUIRE(d->vquad == 0 || d->vquad == 1, "vquad must be 0 or 1");
  DFTFE_REQUIRE(d->nq1d >= 0 && d->nq1d <= 12, "nq1d must be in 0..12");
  for (int a = 0; a < 3; ++a) {
    DFTFE_REQUIRE(d->ncell[a] >= 2, "need at least 2 cells per axis");
    DFTFE_REQUIRE(d->L[a] > 0 && std::isfinite(d->L[a]), "box lengths must be positive");
    DFTFE_REQUIRE(d->periodic[a] == 1, "only fully periodic meshes are supported");
  }
  auto* m = new dftfe_mesh_s();
  m->p = d->degree;
  m->n1 = m->p + 1;
  m->nc = m->n1 * m->n1 * m->n1;
  m->vquad = d->vquad;
  m->nq1d = d->nq1d ? d->nq1d : m->p + 1;
  m->nq1 = m->vquad == 1 ? m->n1 : m->nq1d;
  m->nq = m->nq1 * m->nq1 * m->nq1;
  m->M = 1;
  m->Nc = 1;
  for (int a = 0; a < 3; ++a) {
    m->L[a] = d->L[a];
    m->n[a] = d->ncell[a];
    m->g[a] = (int64_t)d->ncell[a] * m->p;
    m->h[a] = d->L[a] / d->ncell[a];
    m->M *= m->g[a];
    m->Nc *= m->n[a];
  }
  if (m->M >= (int64_t)INT32_MAX) {
    delete m;
    throw Error(DFTFE_ERR_ARG, "more than 2^31-1 DoFs");
  }
  m->detJ = m->h[0] * m->h[1] * m->h[2] / 8.0;
  m->gll = gll_rule(m->p);
  m->quad = m->vquad == 1 ? m->gll : gauss_rule(m->nq1);
  m->D = derivative_matrix(m->gll.x);
  m->Lq = lagrange_at(m->gll.x, m->quad.x);
  for (int a = 0; a < 3; ++a) {
    m->m1[a].assign(m->g[a], 0.0);
    for (int c = 0; c < m->n[a]; ++c)
      for (int i = 0; i <= m->p; ++i)
        m->m1[a][(c * (int64_t)m->p + i) % m->g[a]] += m->gll.w[i] * m->h[a] / 2.0;
  }
  *out = m;
  ABI_END
}

extern "C" dftfe_status dftfe_mesh_info(dftfe_mesh m, int64_t* ndofs, int64_t* ncells,
                                        int* nodes_per_cell, int* quad_per_cell) {
  ABI_BEGIN
  DFTFE_REQUIRE(m, "null mesh");
  if (ndofs) *ndofs = m->M;
  if (ncells) *ncells = m->Nc;
  if (nodes_per_cell) *nodes_per_cell = m->nc;
  if (quad_per_cell) *quad_per_cell = m->nq;
  ABI_END
}

extern "C" dftfe_status dftfe_mesh_coords(dftfe_mesh m, double* node_xyz, double* quad_xyz) {
  ABI_BEGIN
  DFTFE_REQUIRE(m, "null mesh");
  if (node_xyz) {
    for (int64_t j = 0; j < m->M; ++j) {
      int64_t idx[3] = {j % m->g[0], (j / m->g[0]) % m->g[1], j / (m->g[0] * m->g[1])};
      for (int a = 0; a < 3; ++a) {
        int64_t cell = idx[a] / m->p;
        int loc = (int)(idx[a] % m->p);
        node_xyz[3 * j + a] = cell * m->h[a] + (m->gll.x[loc] + 1.0) * m->h[a] / 2.0;
      }
    }
  }
  if (quad_xyz) {
    const int nq1 = m->nq1;
    for (int64_t c = 0; c < m->Nc; ++c) {
      int64_t cc[3] = {c % m->n[0], (c / m->n[0]) % m->n[1], c / ((int64_t)m->n[0] * m->n[1])};
      for (int q = 0; q < m->nq; ++q) {
        int qi[3] = {q % nq1, (q / nq1) % nq1, q / (nq1 * nq1)};
        for (int a = 0; a < 3; ++a)
          quad_xyz[(c * m->nq + q) * 3 + a] = cc[a] * m->h[a] + (m->quad.x[qi[a]] + 1.0) * m->h[a] / 2.0;
      }
    }
  }
  ABI_END
}

extern "C" dftfe_status dftfe_mesh_destroy(dftfe_mesh m) {
  ABI_BEGIN
  delete m;
  ABI_END
}

// ----------------------------------------------------------------- ABI: ham
// A ham over mesh m on `stream`; with src, one that uses src's local operator (no cell
// matrices or packed basis products of its own).
static dftfe_ham create_ham(dftfe_mesh m, void* stream, dftfe_ham src) {
  auto* h = new dftfe_ham_s();
  try {
    h->mesh = m;
    h->local_src = src;
    h->stream = (cudaStream_t)stream;
    DFTFE_CHECK_CUDA(cudaGetDevice(&h->device));
    DFTFE_CHECK_CUDA(cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device));
    cudaStream_t s = h->stream;
    const int nc = m->nc, n1 = m->n1;
    // a1: map and lumped mass
    DFTFE_CHECK_CUDA(cudaMalloc(&h->d_map, sizeof(int32_t) * m->Nc * nc));
    DFTFE_LAUNCH(k_cell_map, nblk(m->Nc * nc), 256, 0, s, h->d_map, m->Nc, n1, m->p, m->n[0],
                 m->n[1], m->g[0], m->g[1], m->g[2]);
    DFTFE_CHECK_CUDA(cudaMalloc(&h->d_mass, sizeof(double) * m->M));
    DFTFE_CHECK_CUDA(cudaMalloc(&h->d_minvsqrt, sizeof(double) * m->M));
    {
      double* m1[3];
      for (int a = 0; a < 3; ++a) m1[a] = dev_upload(m->m1[a], s);
      DFTFE_LAUNCH(k_mass, nblk(m->M), 256, 0, s, h->d_mass, h->d_minvsqrt, m1[0], m1[1], m1[2],
                   m->g[0], m->g[1], m->M);
      DFTFE_CHECK_CUDA(cudaStreamSynchronize(s));
      for (int a = 0; a < 3; ++a) cudaFree(m1[a]);
    }
    // colouring: per axis 2 colours (even count) or 3 (odd count, last cell apart)
    {
      int ncol_ax[3];
      for (int a = 0; a < 3; ++a) ncol_ax[a] = (m->n[a] % 2 == 0) ? 2 : 3;
      h->ncolours = ncol_ax[0] * ncol_ax[1] * ncol_ax[2];
      std::vector<std::vector<int32_t>> lists(h->ncolours);
      for (int64_t c = 0; c < m->Nc; ++c) {
        int64_t cc[3] = {c % m->n[0], (c / m->n[0]) % m->n[1], c / ((int64_t)m->n[0] * m->n[1])};
        int k[3];
        for (int a = 0; a < 3; ++a)
          k[a] = (ncol_ax[a] == 3 && cc[a] == m->n[a] - 1) ? 2 : (int)(cc[a] % 2);
        lists[k[0] + ncol_ax[0] * (k[1] + ncol_ax[1] * k[2])].push_back((int32_t)c);
      }
      std::vector<int32_t> flat;
      h->colour_off.assign(1, 0);
      for (auto& l : lists) {
        flat.insert(flat.end(), l.begin(), l.end());
        h->colour_off.push_back((int64_t)flat.size());
      }
      h->d_colour_cells = dev_upload(flat, s);
    }
    // a2 reference tables: the basis at the quadrature points (density)
    {
      std::vector<double> Nq((size_t)m->nq * nc);
      for (int q = 0; q < m->nq; ++q) {
        const int qa = q % m->nq1, qb = (q / m->nq1) % m->nq1, qc = q / (m->nq1 * m->nq1);
        for (int j = 0; j < nc; ++j) {
          const int a = j % n1, b = (j / n1) % n1, c = j / (n1 * n1);
          Nq[(size_t)q * nc + j] = m->Lq[qa * n1 + a] * m->Lq[qb * n1 + b] * m->Lq[qc * n1 + c];
        }
      }
      h->d_Nq = dev_upload(Nq, s);
    }
    if (!src) sf_init(h);
    if (!src) DFTFE_CHECK_CUDA(cudaMalloc(&h->d_Hc, sizeof(double) * m->Nc * (int64_t)nc * nc));
  } catch (...) {
    h->local_src = nullptr;
    dftfe_ham_destroy(h);
    throw;
  }
  if (src) src->sharers++;
  return h;
}

extern "C" dftfe_status dftfe_ham_create(dftfe_mesh m, void* stream, dftfe_ham* out) {
  ABI_BEGIN
  DFTFE_REQUIRE(m && out, "null argument");
  *out = create_ham(m, stream, nullptr);
  ABI_END
}

extern "C" dftfe_status dftfe_ham_create_shared(dftfe_ham src, dftfe_ham* out) {
  ABI_BEGIN
  DFTFE_REQUIRE(src && out, "null argument");
  DFTFE_REQUIRE(!src->local_src, "src must own its local operator (not itself made by dftfe_ham_create_shared)");
  int dev = -1;
  DFTFE_CHECK_CUDA(cudaGetDevice(&dev));
  DFTFE_REQUIRE(dev == src->device, "the current device must be src's");
  *out = create_ham(src->mesh, (void*)src->stream, src);
  ABI_END
}

extern "C" dftfe_status dftfe_ham_set_potential(dftfe_ham h, const double* v_quad) {
  ABI_BEGIN
  DFTFE_REQUIRE(h && v_quad, "null argument");
  if (h->local_src)
    throw Error(DFTFE_ERR_STATE, "this ham uses another ham's local operator: set the potential on that ham");
  auto* m = h->mesh;
  sf_set_potential(h, v_quad);
  {
    ProfScope ps(h, "dhm_gemm");
    const int N = m->n1, np = N * (N + 1) / 2, nq = m->nq1;
    const CellTab tab{h->d_celltab, h->d_celltab + nq * np, h->d_celltab + nq * np + N * N,
                      2.0 / (m->h[0] * m->h[0]), 2.0 / (m->h[1] * m->h[1]), 2.0 / (m->h[2] * m->h[2])};
    const size_t sh = sizeof(double) * ((size_t)nq * nq * nq + nq * np + N * N + N + nq * nq + np * nq + np * np) +
                      (size_t)N * N;
    // enough CTAs for a few per SM when there are few cells
    const int split = (int)std::max<int64_t>(1, std::min<int64_t>(np, 6LL * h->sm_count / m->Nc));
    DFTFE_LAUNCH(k_cell_matrices, dim3((unsigned)m->Nc, (unsigned)split), 256, sh, h->stream, h->d_sfv, tab, N, nq,
                 m->vquad == 1 ? 1 : 0, h->d_Hc);
  }
  h->has_potential = true;
  h->potential_version++;
  ABI_END
}

extern "C" dftfe_status dftfe_ham_set_nonlocal(dftfe_ham h, int nproj, const double* hcoup,
                                               const int64_t* rowptr, const int64_t* node,
                                               const double* chi) {
  ABI_BEGIN
  DFTFE_REQUIRE(h, "null ham");
  DFTFE_REQUIRE(nproj >= 0, "nproj must be >= 0");
  auto* m = h->mesh;
  if (nproj == 0) {
    DFTFE_CHECK_CUDA(cudaStreamSynchronize(h->stream));
    free_nonlocal(h);
    return DFTFE_OK;
  }
  DFTFE_REQUIRE(hcoup && rowptr && node && chi, "null CSR input");
  DFTFE_REQUIRE(rowptr[0] == 0, "rowptr[0] must be 0");
  for (int a = 0; a < nproj; ++a) DFTFE_REQUIRE(rowptr[a + 1] >= rowptr[a], "rowptr not monotone");
  const int64_t nnz = rowptr[nproj];
  for (int64_t e = 0; e < nnz; ++e)
    DFTFE_REQUIRE(node[e] >= 0 && node[e] < m->M, "projector node index out of range");
  // node-major transpose (counting sort over the support nodes)
  std::vector<int32_t> pnode(nnz);
  for (int64_t e = 0; e < nnz; ++e) pnode[e] = (int32_t)node[e];
  std::vector<int64_t> order(nnz);
  for (int64_t e = 0; e < nnz; ++e) order[e] = e;
  std::stable_sort(order.begin(), order.end(), [&](int64_t x, int64_t y) { return node[x] < node[y]; });
  std::vector<int32_t> snode, sproj(nnz);
  std::vector<int64_t> srow;
  std::vector<int64_t> eproj(nnz);
  for (int a = 0; a < nproj; ++a)
    for (int64_t e = rowptr[a]; e < rowptr[a + 1]; ++e) eproj[e] = a;
  for (int64_t t = 0; t < nnz; ++t) {
    int64_t e = order[t];
    if (snode.empty() || snode.back() != (int32_t)node[e]) {
      snode.push_back((int32_t)node[e]);
      srow.push_back(t);
    }
    sproj[t] = (int32_t)eproj[e];
  }
  srow.push_back(nnz);
  // runs of projectors with one node list (an atom's angular channels)
  std::vector<int32_t> group{0};
  for (int a = 1; a < nproj; ++a) {
    const int64_t b = rowptr[group.back()], len = rowptr[group.back() + 1] - b;
    if (a - group.back() < kNlGroup && rowptr[a + 1] - rowptr[a] == len &&
        std::equal(node + rowptr[a], node + rowptr[a + 1], node + b))
      continue;
    group.push_back(a);
  }
  group.push_back(nproj);
  DFTFE_CHECK_CUDA(cudaStreamSynchronize(h->stream));
  free_nonlocal(h);
  cudaStream_t s = h->stream;
  h->nproj = nproj;
  h->nnz = nnz;
  h->nsup = (int64_t)snode.size();
  h->d_h = dev_upload(std::vector<double>(hcoup, hcoup + nproj), s);
  h->npgroup = (int)group.size() - 1;
  h->d_pgroup = dev_upload(group, s);
  h->d_prow = dev_upload(std::vector<int64_t>(rowptr, rowptr + nproj + 1), s);
  h->d_pnode = dev_upload(pnode, s);
  double* d_chi = dev_upload(std::vector<double>(chi, chi + nnz), s);
  DFTFE_CHECK_CUDA(cudaMalloc(&h->d_pval, sizeof(double) * std::max<int64_t>(nnz, 1)));
  if (nnz)
    DFTFE_LAUNCH(k_scale_by_sqrt_mass, nblk(nnz), 256, 0, s, h->d_pval, d_chi, h->d_pnode,
                 h->d_mass, nnz);
  h->d_snode = dev_upload(snode, s);
  h->d_srow = dev_upload(srow, s);
  {
    // the same node-major entries indexed by every node (empty ranges off the supports)
    std::vector<int64_t> nall(m->M + 1, 0);
    for (size_t k = 0; k < snode.size(); ++k) nall[(size_t)snode[k] + 1] = srow[k + 1] - srow[k];
    for (int64_t g = 0; g < m->M; ++g) nall[g + 1] += nall[g];
    h->d_nptr_all = dev_upload(nall, s);
  }
  h->d_sproj = dev_upload(sproj, s);
  // node-major position t holds projector-major entry sperm[t] (kept for the k-point values)
  h->d_sperm = dev_upload(order, s);
  DFTFE_CHECK_CUDA(cudaMalloc(&h->d_sval, sizeof(double) * std::max<int64_t>(nnz, 1)));
  DFTFE_CHECK_CUDA(cudaMalloc(&h->d_sval32, sizeof(float) * std::max<int64_t>(nnz, 1)));
  if (nnz) DFTFE_LAUNCH(k_gather_vals, nblk(nnz), 256, 0, s, h->d_sval, h->d_sval32, h->d_pval, h->d_sperm, nnz);
  DFTFE_CHECK_CUDA(cudaStreamSynchronize(s));
  cudaFree(d_chi);
  ABI_END
}

extern "C" dftfe_status dftfe_ham_destroy(dftfe_ham h) {
  ABI_BEGIN
  if (!h) return DFTFE_OK;
  if (h->sharers > 0)
    throw Error(DFTFE_ERR_STATE, "hams made by dftfe_ham_create_shared still use this ham: destroy them first");
  if (h->local_src) h->local_src->sharers--;
  cudaStreamSynchronize(h->stream);
  free_graphs(h);
  if (h->h_pass) cudaFreeHost(h->h_pass);
  free_nonlocal(h);
  cudaFree(h->d_map); cudaFree(h->d_mass); cudaFree(h->d_minvsqrt);
  cudaFree(h->d_colour_cells); cudaFree(h->d_node_ptr); cudaFree(h->d_node_slot); 
  cudaFree(h->d_sfw); cudaFree(h->d_sfv);
  cudaFree(h->d_celltab); cudaFree(h->d_Hc); cudaFree(h->d_Nq); cudaFree(h->d_ktab); cudaFree(h->d_ktab32);
  for (auto& kv : h->ws) kv.second.release();
  for (auto& kv : h->timers)
    for (auto& ev : kv.second.events) {
      cudaEventDestroy(ev.first);
      cudaEventDestroy(ev.second);
    }
  delete h;
  ABI_END
}

extern "C" dftfe_status dftfe_ham_export(dftfe_ham h, double* mass, int32_t* cell_map, int64_t c0,
                                         int64_t count, double* cell_mats) {
  ABI_BEGIN
  DFTFE_REQUIRE(h, "null ham");
  auto* m = h->mesh;
  cudaStream_t s = h->stream;
  if (mass)
    DFTFE_CHECK_CUDA(cudaMemcpyAsync(mass, h->d_mass, sizeof(double) * m->M, cudaMemcpyDeviceToDevice, s));
  if (cell_map)
    DFTFE_CHECK_CUDA(cudaMemcpyAsync(cell_map, h->d_map, sizeof(int32_t) * m->Nc * m->nc,
                                     cudaMemcpyDeviceToDevice, s));
  if (cell_mats) {
    DFTFE_REQUIRE(c0 >= 0 && count >= 0 && c0 + count <= m->Nc, "cell range out of bounds");
    DFTFE_REQUIRE(loc(h)->has_potential, "no potential set");
    const int64_t n2 = (int64_t)m->nc * m->nc;
    DFTFE_CHECK_CUDA(cudaMemcpyAsync(cell_mats, loc(h)->d_Hc + c0 * n2, sizeof(double) * count * n2,
                                     cudaMemcpyDeviceToDevice, s));
  }
  ABI_END
}

extern "C" int64_t dftfe_launch_count(void) { return g_launches.load(); }
extern "C" const char* dftfe_last_error(void) { return dftfe::last_error(); }
