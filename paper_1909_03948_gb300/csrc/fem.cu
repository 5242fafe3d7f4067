// fem.cu -- operators of the discretised log-coefficient Poisson problem.
//
// Coefficient:  kappa_e = mean_{v in e} e^{m_v}  (exact element integral of the
//               P1 interpolant of e^m, divided by |e|).
// Stiffness K(kappa): only axis (path) edges couple (see common.cuh), with
//               edge weight w = (|e|/h^2) sum_{e contains the edge} kappa_e; stored
//               as a 5-point (2D) / 7-point (3D) symmetric stencil.  Dirichlet
//               rows (last coordinate 0 or N) become identity rows and their
//               couplings are removed; the removed couplings times the Dirichlet
//               data form the lifting right-hand side (Section 5.1.3 boundary
//               conditions).
// Multigrid coarse operators: the meshes are nested (the fine simplices refine
//               the coarse ones, 2^D children each) and P1 interpolation is the
//               prolongation, so the Galerkin operator P^T K(kappa) P is the coarse
//               FE stiffness with kappa_coarse = mean of the children's kappa.
// Prior A = gamma K(1) + delta M (Section 5.1.1, eq. (PoissonPrior), Theta = I,
//               zero Neumann) and mass M couple along all 2^D - 1 Kuhn edge
//               directions (7-point / 15-point).
// C X   = K(kappa_hat) u, kappa_hat_e = mean_{v in e}(e^m X)_v   (Appendix A,
//               eq. (incrementals1): the term (mhat e^m grad u, grad p~)).
// C^T W = e^{m_v}/(D+1) sum_{e ni v} |e| grad u . grad W          (Appendix A,
//               eqs. (firstcontrol), (incrementals3)).
// B     = P1 interpolation at the observation points (Section 5.1.1).
// C_M   = rectangular factor of M from a degree-2 element rule (Appendix C,
//               eq. (rect_decomp)).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <vector>

#include "dfloat.cuh"
#include "internal.h"
#include "philox.cuh"

namespace hp {

// children of each coarse simplex: (fine cell offset mask) | (fine perm << 3)
__constant__ int c_child2[2][4];
__constant__ int c_child3[6][8];

// quadrature: barycentric coordinate of vertex k at point q (degree-2 rules)
__constant__ double c_quad2[3][3] = {{0.5, 0.5, 0.0}, {0.0, 0.5, 0.5}, {0.5, 0.0, 0.5}};

static std::mutex g_children_mutex;
static int g_children_ready = 0;

// The coarse simplex (cell C, perm pi) = {x in C : x_{pi_0} >= x_{pi_1} >= ...}
// (local coordinates); a fine simplex belongs to it iff its centroid does.
static void compute_children(int D, std::vector<std::vector<int>> &out) {
  std::vector<std::vector<int>> perms;
  std::vector<int> a(D);
  for (int i = 0; i < D; ++i) a[i] = i;
  do perms.push_back(a);
  while (std::next_permutation(a.begin(), a.end()));
  out.assign(perms.size(), {});
  for (size_t cp = 0; cp < perms.size(); ++cp) {
    for (int o = 0; o < (1 << D); ++o) {
      for (size_t fp = 0; fp < perms.size(); ++fp) {
        double s[3] = {0, 0, 0};
        for (int ax = 0; ax < D; ++ax) s[ax] = (o >> ax) & 1;
        for (int j = 0; j < D; ++j) s[perms[fp][j]] += double(D - j) / double(D + 1);
        bool in = true;
        for (int j = 0; j + 1 < D; ++j) in = in && (s[perms[cp][j]] > s[perms[cp][j + 1]]);
        if (in) out[cp].push_back(o | (int(fp) << 3));
      }
    }
  }
}

static int ensure_children() {
  std::lock_guard<std::mutex> lock(g_children_mutex);
  if (g_children_ready) return 0;
  std::vector<std::vector<int>> c2, c3;
  compute_children(2, c2);
  compute_children(3, c3);
  int t2[2][4], t3[6][8];
  for (int p = 0; p < 2; ++p) {
    if (c2[p].size() != 4) return set_error(HP_ERR_INVALID, "internal: 2D refinement table");
    for (int q = 0; q < 4; ++q) t2[p][q] = c2[p][q];
  }
  for (int p = 0; p < 6; ++p) {
    if (c3[p].size() != 8) return set_error(HP_ERR_INVALID, "internal: 3D refinement table");
    for (int q = 0; q < 8; ++q) t3[p][q] = c3[p][q];
  }
  HP_CUDA(cudaMemcpyToSymbol(c_child2, t2, sizeof(t2)));
  HP_CUDA(cudaMemcpyToSymbol(c_child3, t3, sizeof(t3)));
  g_children_ready = 1;
  return 0;
}

// ---------------------------------------------------------------------------
// element coefficients
// ---------------------------------------------------------------------------
template <int D>
__global__ void k_elem_kappa_fine(GridDesc g, const double *__restrict__ E, double *__restrict__ kappa,
                                  long nelems) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < nelems; e += (long)gridDim.x * blockDim.x) {
    const long cell = e / MeshT<D>::NPERM;
    const int p = (int)(e % MeshT<D>::NPERM);
    int c[3];
    c[0] = (int)(cell % g.N);
    const long t = cell / g.N;
    c[1] = D == 2 ? (int)t : (int)(t % g.N);
    c[2] = D == 2 ? 0 : (int)(t / g.N);
    const long base = c[0] + (long)g.np * (c[1] + (long)g.np * c[2]);
    double s = 0.0;
#pragma unroll
    for (int k = 0; k <= D; ++k) s += E[base + mask_offset(g, MeshT<D>::chain(p, k))];
    kappa[e] = s / (D + 1);
  }
}

template <int D>
__global__ void k_elem_kappa_coarsen(GridDesc gc, GridDesc gf, const double *__restrict__ kf,
                                     double *__restrict__ kc, long nelems_c) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < nelems_c; e += (long)gridDim.x * blockDim.x) {
    const long cell = e / MeshT<D>::NPERM;
    const int p = (int)(e % MeshT<D>::NPERM);
    int c[3];
    c[0] = (int)(cell % gc.N);
    const long t = cell / gc.N;
    c[1] = D == 2 ? (int)t : (int)(t % gc.N);
    c[2] = D == 2 ? 0 : (int)(t / gc.N);
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < (1 << D); ++q) {
      const int code = D == 2 ? c_child2[p][q] : c_child3[p][q];
      const int o = code & 7, fp = code >> 3;
      int fc[3] = {2 * c[0] + (o & 1), 2 * c[1] + ((o >> 1) & 1), 2 * c[2] + ((o >> 2) & 1)};
      s += kf[cell_linear<D>(gf, fc) * MeshT<D>::NPERM + fp];
    }
    kc[e] = s / (1 << D);
  }
}

// ---------------------------------------------------------------------------
// stencils
// ---------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ bool is_dirichlet(const GridDesc &g, const int v[3]) {
  return v[D - 1] == 0 || v[D - 1] == g.N;
}

template <int D>
__device__ __forceinline__ double edge_weight(const GridDesc &g, const double *__restrict__ kappa, const int v[3],
                                              int b) {
  double s = 0.0;
  for_elems_with<D>(g, v, b, [&](const int c[3], int p, int k) {
    s += kappa[cell_linear<D>(g, c) * MeshT<D>::NPERM + p];
  });
  return s * vol_over_h2<D>(g.h);
}

template <int D>
__global__ void k_build_K(GridDesc g, const double *__restrict__ kappa, double *diag, double *invdiag, double *c,
                          float *diag32, float *invdiag32, float *c32, double *lift, double u_top,
                          double u_bottom) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.n; i += (long)gridDim.x * blockDim.x) {
    int v[3];
    node_coords<D>(g, i, v);
    const bool dv = is_dirichlet<D>(g, v);
    double dsum = 0.0, lf = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      double wf = 0.0, wb = 0.0;
      int vn[3] = {v[0], v[1], v[2]};
      if (v[a] < g.N) {
        wf = edge_weight<D>(g, kappa, v, 1 << a);
        vn[a] = v[a] + 1;
        const bool dn = is_dirichlet<D>(g, vn);
        const double cf = (dv || dn) ? 0.0 : -wf;
        c[(long)a * g.n + i] = cf;
        c32[(long)a * g.n + i] = (float)cf;
        if (!dv && dn) lf += wf * (vn[D - 1] == g.N ? u_top : u_bottom);
      } else {
        c[(long)a * g.n + i] = 0.0;
        c32[(long)a * g.n + i] = 0.0f;
      }
      if (v[a] > 0) {
        int vb[3] = {v[0], v[1], v[2]};
        vb[a] = v[a] - 1;
        wb = edge_weight<D>(g, kappa, vb, 1 << a);
        if (!dv && is_dirichlet<D>(g, vb)) lf += wb * (vb[D - 1] == g.N ? u_top : u_bottom);
      }
      dsum += wf + wb;
    }
    const double dg = dv ? 1.0 : dsum;
    diag[i] = dg;
    invdiag[i] = 1.0 / dg;
    diag32[i] = (float)dg;
    invdiag32[i] = (float)(1.0 / dg);
    if (lift) lift[i] = dv ? 0.0 : lf;
  }
}

// 2D stiffness in FP32, one 16-byte record per node for the tiled stencil kernels:
// {diag, 1 / diag, coupling to x + 1, coupling to y + 1}
__global__ void k_pack_K2(long n, const float *__restrict__ diag, const float *__restrict__ invdiag,
                          const float *__restrict__ c, float4 *__restrict__ pk) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    pk[i] = make_float4(diag[i], invdiag[i], c[i], c[n + i]);
}

// 3D stiffness in FP32 for the tiled kernels: one 16-byte record per node {diag, 1 / diag,
// coupling to x + 1, coupling to y + 1}, and the coupling to z + 1 in rows padded to a
// multiple of 4 nodes (a tensor map's row stride must be a multiple of 16 bytes)
__global__ void k_pack_K3(GridDesc g, const float *__restrict__ diag, const float *__restrict__ invdiag,
                          const float *__restrict__ c, float4 *__restrict__ pk, float *__restrict__ cz) {
  const long n = g.n, ldr = (g.np + 3) / 4 * 4;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    pk[i] = make_float4(diag[i], invdiag[i], c[i], c[n + i]);
    const long x = i % g.np, row = i / g.np;
    cz[row * ldr + x] = c[2 * n + i];
  }
}

template <int D>
__device__ __forceinline__ int count_elems(const GridDesc &g, const int v[3], int b) {
  int n = 0;
  for_elems_with<D>(g, v, b, [&](const int *, int, int) { ++n; });
  return n;
}

// Symmetric anisotropy tensor: t[0..2] = (T00, T11, T22), t[3..5] = (T01, T02, T12).
struct Theta6 {
  double t[6];
};
__device__ __forceinline__ double theta_ab(const Theta6 &T, int a, int b) {
  if (a == b) return T.t[a];
  const int lo = a < b ? a : b, hi = a < b ? b : a;
  return lo == 0 ? (hi == 1 ? T.t[3] : T.t[4]) : T.t[5];
}

// Gradient (in units of 1/h) of the barycentric function of chain vertex t of Kuhn simplex p:
// with pi_t the axis added at step t, lambda_0 = 1 - x_{pi_1}, lambda_t = x_{pi_t} - x_{pi_{t+1}},
// lambda_D = x_{pi_D} in the cell's local coordinates.
template <int D>
__device__ __forceinline__ void kuhn_grad(int p, int t, double gv[3]) {
  gv[0] = gv[1] = gv[2] = 0.0;
  if (t >= 1) gv[__ffs(MeshT<D>::chain(p, t) ^ MeshT<D>::chain(p, t - 1)) - 1] += 1.0;
  if (t < D) gv[__ffs(MeshT<D>::chain(p, t + 1) ^ MeshT<D>::chain(p, t)) - 1] -= 1.0;
}

// A = gamma K(Theta) + delta M + cR M_boundary (all nodes, no Dirichlet rows), assembled per
// node from the simplices that contain it (each node keeps its diagonal and its forward
// couplings along the 2^D - 1 Kuhn edge directions) and from the boundary facets that
// contain it (the facets of a face of the cube are the Kuhn triangulation of that face).
// With Theta = I and cR = 0 this is gamma K(1) + delta M with zero Neumann.
template <int D>
__global__ void k_build_A(GridDesc g, double gamma, double delta, double cR, Theta6 Th, double *diag,
                          double *invdiag, double *c, float *diag32, float *invdiag32, float *c32) {
  constexpr int NF = (1 << D) - 1;
  const double vh2 = vol_over_h2<D>(g.h);
  const double mc = elem_vol<D>(g.h) / ((D + 1) * (D + 2));
  const double fvol = D == 2 ? g.h : 0.5 * g.h * g.h;   // boundary facet measure
  const double fm = fvol / (D * (D + 1));                // off-diagonal boundary facet mass
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.n; i += (long)gridDim.x * blockDim.x) {
    int v[3];
    node_coords<D>(g, i, v);
    double cf[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) cf[f] = 0.0;
    double dg = 0.0;
    for_elems_with<D>(g, v, 0, [&](const int *, int p, int k) {
      double gk[3];
      kuhn_grad<D>(p, k, gk);
      for (int t = k; t <= D; ++t) {
        double gt[3];
        kuhn_grad<D>(p, t, gt);
        double e = 0.0;
        for (int a = 0; a < D; ++a)
          for (int b = 0; b < D; ++b) e += gk[a] * theta_ab(Th, a, b) * gt[b];
        const double val = gamma * vh2 * e + delta * mc * (t == k ? 2.0 : 1.0);
        if (t == k)
          dg += val;
        else
          cf[(MeshT<D>::chain(p, t) ^ MeshT<D>::chain(p, k)) - 1] += val;
      }
    });
    if (cR != 0.0) {
      for (int a = 0; a < D; ++a) {
        if (v[a] != 0 && v[a] != g.N) continue;
        int ax[2] = {0, 0}, na = 0;
        for (int o = 0; o < D; ++o)
          if (o != a) ax[na++] = o;
        for (int s0 = 0; s0 < 2; ++s0)
          for (int s1 = 0; s1 < (D == 3 ? 2 : 1); ++s1) {
            int cc[3] = {v[0], v[1], v[2]};
            cc[ax[0]] -= s0;
            if (D == 3) cc[ax[1]] -= s1;
            if (cc[ax[0]] < 0 || cc[ax[0]] >= g.N) continue;
            if (D == 3 && (cc[ax[1]] < 0 || cc[ax[1]] >= g.N)) continue;
            const int vm = (s0 << ax[0]) | (D == 3 ? (s1 << ax[1]) : 0);  // v - cc as a corner mask
            for (int perm = 0; perm < (D == 3 ? 2 : 1); ++perm) {
              const int p1 = D == 3 ? ax[perm] : ax[0];
              const int m[3] = {0, 1 << p1, D == 3 ? ((1 << p1) | (1 << ax[1 - perm])) : 0};
              int k = -1;
              for (int t = 0; t < D; ++t)
                if (m[t] == vm) k = t;
              if (k < 0) continue;
              dg += cR * 2.0 * fm;
              for (int t = k + 1; t < D; ++t) cf[(m[t] ^ m[k]) - 1] += cR * fm;
            }
          }
      }
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      c[(long)f * g.n + i] = cf[f];
      c32[(long)f * g.n + i] = (float)cf[f];
    }
    diag[i] = dg;
    invdiag[i] = 1.0 / dg;
    diag32[i] = (float)dg;
    invdiag32[i] = (float)(1.0 / dg);
  }
}

// max over nodes of (diag_i + sum_j |s_ij|) / diag_i: a bound of the spectrum of diag^-1 S
template <int D>
__global__ void k_gersh(GridDesc g, const double *__restrict__ diag, const double *__restrict__ c, int nf, bool full,
                        unsigned long long *out) {
  double mx = 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.n; i += (long)gridDim.x * blockDim.x) {
    int v[3];
    node_coords<D>(g, i, v);
    double sum = fabs(diag[i]);
    for (int f = 0; f < nf; ++f) {
      const int b = full ? f + 1 : (1 << f);
      bool fw = true, bw = true;
      for (int a = 0; a < D; ++a)
        if ((b >> a) & 1) {
          fw = fw && (v[a] < g.N);
          bw = bw && (v[a] > 0);
        }
      const long off = mask_offset(g, b);
      if (fw) sum += fabs(c[(long)f * g.n + i]);
      if (bw) sum += fabs(c[(long)f * g.n + i - off]);
    }
    mx = fmax(mx, sum / diag[i]);
  }
  // positive doubles order like their bit patterns
  atomicMax(out, (unsigned long long)__double_as_longlong(mx));
}

int gershgorin_bound(hp_problem *P, const GridDesc &g, const Stencil<double> &S, double *out) {
  unsigned long long *d = reinterpret_cast<unsigned long long *>(P->sc.tmp.p);
  HP_TRY(P->sc.tmp.ensure(64));
  d = reinterpret_cast<unsigned long long *>(P->sc.tmp.p);
  HP_CUDA(cudaMemsetAsync(d, 0, sizeof(unsigned long long), P->st));
  const int nb = (int)std::min<long>((g.n + 255) / 256, 1024);
  if (g.dim == 2)
    k_gersh<2><<<nb, 256, 0, P->st>>>(g, S.diag, S.c, S.nf, S.full, d);
  else
    k_gersh<3><<<nb, 256, 0, P->st>>>(g, S.diag, S.c, S.nf, S.full, d);
  count_launch();
  unsigned long long h = 0;
  HP_CUDA(cudaMemcpyAsync(&h, d, sizeof(h), cudaMemcpyDeviceToHost, P->st));
  HP_CUDA(cudaStreamSynchronize(P->st));
  double v;
  std::memcpy(&v, &h, sizeof(v));
  *out = v;
  return 0;
}

// ---------------------------------------------------------------------------
// dense coarse-grid inverse
// ---------------------------------------------------------------------------
template <int D>
__global__ void k_dense_from_stencil(GridDesc g, const double *diag, const double *c, int nf, bool full,
                                     double *A) {
  const long nc = g.n;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < nc; i += (long)gridDim.x * blockDim.x) {
    int v[3];
    node_coords<D>(g, i, v);
    A[i * nc + i] = diag[i];
    for (int f = 0; f < nf; ++f) {
      const int b = full ? f + 1 : (1 << f);
      bool fwd = true;
      for (int a = 0; a < D; ++a)
        if ((b >> a) & 1) fwd = fwd && (v[a] < g.N);
      if (!fwd) continue;
      const long j = i + mask_offset(g, b);
      const double w = c[(long)f * g.n + i];
      A[i * nc + j] = w;
      A[j * nc + i] = w;
    }
  }
}

// In-place lower Cholesky of a dense SPD matrix (row-major), one block.
__global__ void k_dense_cholesky(double *A, int nc, int *status) {
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int k = 0; k < nc; ++k) {
    if (threadIdx.x == 0) {
      const double d = A[(long)k * nc + k];
      if (!(d > 0.0) || !isfinite(d)) bad = 1;
      A[(long)k * nc + k] = (d > 0.0) ? sqrt(d) : 1.0;
    }
    __syncthreads();
    const double dk = A[(long)k * nc + k];
    for (int i = k + 1 + threadIdx.x; i < nc; i += blockDim.x) A[(long)i * nc + k] /= dk;
    __syncthreads();
    const int m = nc - k - 1;
    for (long t = threadIdx.x; t < (long)m * m; t += blockDim.x) {
      const int i = k + 1 + (int)(t / m), j = k + 1 + (int)(t % m);
      if (j <= i) A[(long)i * nc + j] -= A[(long)i * nc + k] * A[(long)j * nc + k];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *status = bad;
}

// Column j of the inverse from the Cholesky factor, one thread per column.  The inverse is
// symmetric, so thread j keeps its column as row j of the output, x[i] at inv[i * nc + j]:
// the threads of a warp then touch consecutive addresses at every step (and all read the same
// L entry), and the substitutions start at row j (rows above it are zero in L^-1 e_j).
__global__ void k_dense_inverse(const double *L, int nc, double *inv, float *inv32) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nc) return;
  for (int i = 0; i < j; ++i) inv[(long)i * nc + j] = 0.0;
  for (int i = j; i < nc; ++i) {  // L y = e_j
    double s = (i == j) ? 1.0 : 0.0;
    for (int k = j; k < i; ++k) s -= L[(long)i * nc + k] * inv[(long)k * nc + j];
    inv[(long)i * nc + j] = s / L[(long)i * nc + i];
  }
  for (int i = nc - 1; i >= 0; --i) {  // L^T x = y
    double s = inv[(long)i * nc + j];
    for (int k = i + 1; k < nc; ++k) s -= L[(long)k * nc + i] * inv[(long)k * nc + j];
    inv[(long)i * nc + j] = s / L[(long)i * nc + i];
  }
  for (int i = 0; i < nc; ++i) inv32[(long)i * nc + j] = (float)inv[(long)i * nc + j];
}

// FP32 coarse factorisation for the FP32 inner solves (the only consumer of inv32 when the
// refinement runs in FP32): one CTA, the lower triangle packed in shared memory (row i at
// offset i (i + 1) / 2), filled from the stencil.  Cholesky in panels of CH_B columns:
//   diagonal block: thread (lane i, warp j) holds entry (i, j); one barrier per column;
//   rows below: a thread per row solves its CH_B entries in registers;
//   trailing triangle: 4 x 4 tiles per thread against the panel, kept transposed so that a
//     tile's two operands are one 16-byte load each per column.
// Every entry takes its updates in ascending column order, then the division or the root, as
// the unblocked right-looking form does, so the factor has the same bits.  That form was bound
// by its three barriers and its index arithmetic per column: 1,200 us for 17^2 nodes.
constexpr int CH_B = 32;
__host__ __device__ __forceinline__ constexpr int tri_at(int i, int j) { return i * (i + 1) / 2 + j; }
static size_t chol32_smem(long nc) {  // the triangle and the transposed panel
  return sizeof(float) * ((size_t)(nc * (nc + 1) / 2 + 3) / 4 * 4 + (size_t)CH_B * ((nc + 3) / 4 * 4));
}

template <int D>
__global__ void __launch_bounds__(1024) k_dense_cholesky32(GridDesc g, const float *__restrict__ diag,
                                                           const float *__restrict__ c, int nf, bool full,
                                                           float *__restrict__ Lg, int *status) {
  extern __shared__ __align__(16) float tri[];
  __shared__ float colb[2][CH_B];
  __shared__ int bad;
  const int nc = (int)g.n, nt = nc * (nc + 1) / 2, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ldp = (nc + 3) / 4 * 4;
  float *PT = tri + (nt + 3) / 4 * 4;  // PT[k][r]: column k of the panel, rows past the panel
  if (tid == 0) bad = 0;
  for (int t = tid; t < nt; t += 1024) tri[t] = 0.f;
  __syncthreads();
  for (int i = tid; i < nc; i += 1024) {
    int v[3];
    node_coords<D>(g, i, v);
    tri[tri_at(i, i)] = diag[i];
    for (int f = 0; f < nf; ++f) {
      const int b = full ? f + 1 : (1 << f);
      bool fwd = true;
      for (int a = 0; a < D; ++a)
        if ((b >> a) & 1) fwd = fwd && (v[a] < g.N);
      if (fwd) tri[tri_at(i + (int)mask_offset(g, b), i)] = c[(long)f * nc + i];
    }
  }
  __syncthreads();
  for (int k0 = 0; k0 < nc; k0 += CH_B) {
    const int kb = min(CH_B, nc - k0), r0 = k0 + kb, R = nc - r0;
    // diagonal block
    const bool held = lane >= w && lane < kb;
    float a = held ? tri[tri_at(k0 + lane, k0 + w)] : 0.f;
    for (int k = 0; k < kb; ++k) {
      if (w == k) {
        const float d = __shfl_sync(0xffffffffu, a, k);
        const float dk = d > 0.f ? sqrtf(d) : 1.f;
        if (lane == k && (!(d > 0.f) || !isfinite(d))) bad = 1;
        a = lane == k ? dk : a / dk;
        colb[k & 1][lane] = a;
      }
      __syncthreads();
      if (w > k && lane >= w) a = fmaf(-colb[k & 1][lane], colb[k & 1][w], a);
    }
    if (held) tri[tri_at(k0 + lane, k0 + w)] = a;
    __syncthreads();
    // rows below
    if (tid < R) {
      float v[CH_B];
      float *row = tri + tri_at(r0 + tid, k0);
#pragma unroll
      for (int k = 0; k < CH_B; ++k) v[k] = row[k];  // R > 0: the panel is full
#pragma unroll
      for (int k = 0; k < CH_B; ++k) {
        v[k] = v[k] / tri[tri_at(k0 + k, k0 + k)];
#pragma unroll
        for (int m = k + 1; m < CH_B; ++m) v[m] = fmaf(-v[k], tri[tri_at(k0 + m, k0 + k)], v[m]);
      }
#pragma unroll
      for (int k = 0; k < CH_B; ++k) {
        row[k] = v[k];
        PT[k * ldp + tid] = v[k];
      }
    }
    __syncthreads();
    // trailing triangle (rows past R of the panel hold stale values that are never stored)
    const int nb = (R + 3) / 4;
    for (int t = tid; t < nb * (nb + 1) / 2; t += 1024) {
      int ti = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
      while (ti * (ti + 1) / 2 > t) --ti;
      while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
      const int tj = t - ti * (ti + 1) / 2;
      float acc[4][4];
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = 4 * ti + p, j = 4 * tj + q;
          acc[p][q] = i < R && j <= i ? tri[tri_at(r0 + i, r0 + j)] : 0.f;
        }
#pragma unroll 8
      for (int k = 0; k < CH_B; ++k) {
        const float4 x = *reinterpret_cast<const float4 *>(PT + k * ldp + 4 * ti);
        const float4 y = *reinterpret_cast<const float4 *>(PT + k * ldp + 4 * tj);
        const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(-xv[p], yv[q], acc[p][q]);
      }
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = 4 * ti + p, j = 4 * tj + q;
          if (i < R && j <= i) tri[tri_at(r0 + i, r0 + j)] = acc[p][q];
        }
    }
    __syncthreads();
  }
  for (int t = tid; t < nt; t += 1024) Lg[t] = tri[t];
  if (tid == 0) *status = bad;
}

// Column j of the inverse from the packed L, one warp per column: the forward substitution
// L y = e_j from row j on (rows above are zero), then L^T x = y, each row's sum split over
// the 32 lanes and reduced.  L is held in shared memory: a row is a chain of loads, lane sums,
// five shuffles and a division, and with L read from L2 the chains took 500 us.  x goes out
// as row j of inv32 (the inverse is symmetric) and its entries from j on as column j of tri32;
// with sym, the entries from j on as row and column j of inv32, so that the square and the
// triangle hold the same numbers (see col_holds_triangle).
constexpr int CI_W = 16;  // columns per CTA
static size_t inv32_smem(long nc) {
  return sizeof(float) * ((size_t)(nc * (nc + 1) / 2 + 3) / 4 * 4 + (size_t)CI_W * nc);
}

__global__ void __launch_bounds__(32 * CI_W) k_dense_inverse32(const float *__restrict__ Lg, int nc,
                                                               float *__restrict__ inv32, float *__restrict__ tri32,
                                                               bool sym) {
  extern __shared__ __align__(16) float L[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nt4 = (nc * (nc + 1) / 2 + 3) / 4;
  for (int t = threadIdx.x; t < nt4; t += 32 * CI_W)
    reinterpret_cast<float4 *>(L)[t] = reinterpret_cast<const float4 *>(Lg)[t];
  __syncthreads();
  const int j = blockIdx.x * CI_W + w;
  if (j >= nc) return;
  float *x = L + 4 * nt4 + w * nc;
  for (int i = lane; i < nc; i += 32) x[i] = 0.f;
  __syncwarp();
  for (int i = j; i < nc; ++i) {
    const float *row = L + tri_at(i, 0);
    float sum = 0.f;
#pragma unroll 3
    for (int k = j + lane; k < i; k += 32) sum = fmaf(row[k], x[k], sum);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) x[i] = ((i == j ? 1.f : 0.f) - sum) / row[i];
    __syncwarp();
  }
  for (int i = nc - 1; i >= 0; --i) {
    float sum = 0.f;
#pragma unroll 3
    for (int k = i + 1 + lane; k < nc; k += 32) sum = fmaf(L[tri_at(k, i)], x[k], sum);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) x[i] = (x[i] - sum) / L[tri_at(i, i)];
    __syncwarp();
  }
  for (int i = lane; i < nc; i += 32) {
    if (i >= j || !sym) inv32[(long)j * nc + i] = x[i];
    if (i < j) continue;
    if (sym) inv32[(long)i * nc + j] = x[i];
    tri32[tri_at(i, j)] = x[i];
  }
}

// lower triangle of the symmetric FP32 inverse, row i at i (i + 1) / 2 (the one-CTA coarse
// solve holds it in shared memory: half the square); sym: and into the upper one
__global__ void k_pack_tri(float *inv, int nc, float *__restrict__ tri, bool sym) {
  const int i = blockIdx.x;
  for (int j = threadIdx.x; j <= i; j += blockDim.x) {
    const float v = inv[(long)j * nc + i];
    tri[(long)i * (i + 1) / 2 + j] = v;
    if (sym) inv[(long)i * nc + j] = v;
  }
}

int coarse_setup(hp_problem *P, OpKind op) {
  const Level &lc = P->lv[P->L - 1];
  CoarseInv &C = op == OP_K ? P->cK : P->cA;
  const Stencil<double> &S = op == OP_K ? lc.K64 : lc.A64;
  const long nc = lc.g.n;
  int *dstat = P->sc.active.as<int>();
  const bool sym = col_holds_triangle(P, op);
  constexpr size_t SMEM32 = 222 * 1024;
  if (P->precision == HP_FP32_IR && std::max(chol32_smem(nc), inv32_smem(nc)) <= SMEM32) {
    // only inv32 is used by FP32 inner solves: factor and invert in FP32 (inv64 is
    // rebuilt by hp_set_precision if the plain FP64 path is selected later)
    static std::atomic<unsigned long long> attr_set{0};
    int dev = 0;
    HP_CUDA(cudaGetDevice(&dev));
    if (dev >= 64 || !(attr_set.load(std::memory_order_acquire) & (1ull << dev))) {
      for (const void *k : {(const void *)k_dense_cholesky32<2>, (const void *)k_dense_cholesky32<3>,
                            (const void *)k_dense_inverse32})
        HP_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM32));
      if (dev < 64) attr_set.fetch_or(1ull << dev, std::memory_order_release);
    }
    float *L32 = reinterpret_cast<float *>(C.inv64);  // scratch: the FP64 inverse is not kept in this mode
    const Stencil<float> &S32 = op == OP_K ? lc.K32 : lc.A32;
    if (P->dim == 2)
      k_dense_cholesky32<2><<<1, 1024, chol32_smem(nc), P->st>>>(lc.g, S32.diag, S32.c, S32.nf, S32.full, L32, dstat);
    else
      k_dense_cholesky32<3><<<1, 1024, chol32_smem(nc), P->st>>>(lc.g, S32.diag, S32.c, S32.nf, S32.full, L32, dstat);
    k_dense_inverse32<<<(int)((nc + CI_W - 1) / CI_W), 32 * CI_W, inv32_smem(nc), P->st>>>(L32, (int)nc, C.inv32,
                                                                                           C.tri32, sym);
    C.fp64_valid = false;
    count_launch(2);
  } else {
    HP_CUDA(cudaMemsetAsync(C.dense, 0, sizeof(double) * nc * nc, P->st));
    const int nb = (int)std::min<long>((nc + 255) / 256, 1024);
    if (P->dim == 2)
      k_dense_from_stencil<2><<<nb, 256, 0, P->st>>>(lc.g, S.diag, S.c, S.nf, S.full, C.dense);
    else
      k_dense_from_stencil<3><<<nb, 256, 0, P->st>>>(lc.g, S.diag, S.c, S.nf, S.full, C.dense);
    k_dense_cholesky<<<1, 1024, 0, P->st>>>(C.dense, (int)nc, dstat);
    k_dense_inverse<<<(int)((nc + 31) / 32), 32, 0, P->st>>>(C.dense, (int)nc, C.inv64, C.inv32);
    k_pack_tri<<<(int)nc, 128, 0, P->st>>>(C.inv32, (int)nc, C.tri32, sym);
    C.fp64_valid = true;
    count_launch(4);
  }
  int h = 0;
  HP_CUDA(cudaMemcpyAsync(&h, dstat, sizeof(int), cudaMemcpyDeviceToHost, P->st));
  HP_CUDA(cudaStreamSynchronize(P->st));
  HP_CUDA(cudaGetLastError());
  if (h) return set_error(HP_ERR_NONFINITE, "coarse-grid operator is not SPD (non-finite coefficient?)");
  return 0;
}

// ---------------------------------------------------------------------------
// setup
// ---------------------------------------------------------------------------
static int alloc_stencil(Stencil<double> &S64, Stencil<float> &S32, long n, int nf, bool full) {
  S64.nf = S32.nf = nf;
  S64.full = S32.full = full;
  HP_CUDA(cudaMalloc(&S64.diag, sizeof(double) * n));
  HP_CUDA(cudaMalloc(&S64.invdiag, sizeof(double) * n));
  HP_CUDA(cudaMalloc(&S64.c, sizeof(double) * n * nf));
  HP_CUDA(cudaMalloc(&S32.diag, sizeof(float) * n));
  HP_CUDA(cudaMalloc(&S32.invdiag, sizeof(float) * n));
  HP_CUDA(cudaMalloc(&S32.c, sizeof(float) * n * nf));
  return 0;
}

static int grid_blocks(long n) { return (int)std::max<long>(1, std::min<long>((n + 255) / 256, 8192)); }

int build_hierarchy_geometry(hp_problem *P) {
  HP_TRY(ensure_children());
  const int D = P->dim;
  const int ncmax = D == 2 ? 16 : 4;  // coarsest grid: <= 17^2 or 5^3 nodes, dense inverse
  int N = P->N, L = 1;
  while (N % 2 == 0 && N > ncmax && L < HP_MAXL) {
    N /= 2;
    ++L;
  }
  long nc = 1;
  for (int a = 0; a < D; ++a) nc *= (N + 1);
  if (nc > 1600)
    return set_error(HP_ERR_INVALID, "coarsest multigrid grid too large: N must be 2^k times a small factor");
  P->L = L;
  const int nfK = D, nfA = (1 << D) - 1;
  const int nperm = D == 2 ? 2 : 6;
  for (int l = 0; l < L; ++l) {
    Level &lv = P->lv[l];
    lv.g.dim = D;
    lv.g.N = P->N >> l;
    lv.g.np = lv.g.N + 1;
    lv.g.mnp = (unsigned)((1ull << 32) / (unsigned long long)lv.g.np);
    lv.g.n = 1;
    for (int a = 0; a < D; ++a) lv.g.n *= lv.g.np;
    lv.g.h = 1.0 / lv.g.N;
    lv.nelems = nperm;
    for (int a = 0; a < D; ++a) lv.nelems *= lv.g.N;
    HP_CUDA(cudaMalloc(&lv.kappa, sizeof(double) * lv.nelems));
    HP_TRY(alloc_stencil(lv.K64, lv.K32, lv.g.n, nfK, false));
    if (tile_grid(lv.g)) HP_CUDA(cudaMalloc(&lv.K32.pk, sizeof(float4) * lv.g.n));
    if (tile3_grid(lv.g)) {
      const long ldr = (lv.g.np + 3) / 4 * 4;
      const size_t bytes = sizeof(float4) * lv.g.n + sizeof(float) * ldr * lv.g.np * lv.g.np;
      HP_CUDA(cudaMalloc(&lv.K32.pk, bytes));
      HP_CUDA(cudaMemset(lv.K32.pk, 0, bytes));  // the row padding of the z couplings stays zero
    }
    HP_TRY(alloc_stencil(lv.A64, lv.A32, lv.g.n, nfA, true));
    const int nb = grid_blocks(lv.g.n);
    Theta6 th;
    for (int q = 0; q < 6; ++q) th.t[q] = P->theta[q];
    const double cR = P->gamma * P->robin_beta;
    if (D == 2)
      k_build_A<2><<<nb, 256, 0, P->st>>>(lv.g, P->gamma, P->delta, cR, th, lv.A64.diag, lv.A64.invdiag, lv.A64.c,
                                          lv.A32.diag, lv.A32.invdiag, lv.A32.c);
    else
      k_build_A<3><<<nb, 256, 0, P->st>>>(lv.g, P->gamma, P->delta, cR, th, lv.A64.diag, lv.A64.invdiag, lv.A64.c,
                                          lv.A32.diag, lv.A32.invdiag, lv.A32.c);
    count_launch();
  }
  // mass matrix on the fine grid
  const Level &l0 = P->lv[0];
  HP_TRY(alloc_stencil(P->M64, P->M32, l0.g.n, nfA, true));
  const Theta6 eye{{1.0, 1.0, 1.0, 0.0, 0.0, 0.0}};
  if (D == 2)
    k_build_A<2><<<grid_blocks(l0.g.n), 256, 0, P->st>>>(l0.g, 0.0, 1.0, 0.0, eye, P->M64.diag, P->M64.invdiag,
                                                         P->M64.c, P->M32.diag, P->M32.invdiag, P->M32.c);
  else
    k_build_A<3><<<grid_blocks(l0.g.n), 256, 0, P->st>>>(l0.g, 0.0, 1.0, 0.0, eye, P->M64.diag, P->M64.invdiag,
                                                         P->M64.c, P->M32.diag, P->M32.invdiag, P->M32.c);
  count_launch();
  // coarse inverses
  const long ncn = P->lv[L - 1].g.n;
  for (CoarseInv *C : {&P->cK, &P->cA}) {
    C->nc = (int)ncn;
    HP_CUDA(cudaMalloc(&C->dense, sizeof(double) * ncn * ncn));
    HP_CUDA(cudaMalloc(&C->inv64, sizeof(double) * ncn * ncn));
    HP_CUDA(cudaMalloc(&C->inv32, sizeof(float) * ncn * ncn));
    const size_t tb = sizeof(float) * (size_t)((ncn * (ncn + 1) / 2 + 3) / 4 * 4);
    HP_CUDA(cudaMalloc(&C->tri32, tb));
    HP_CUDA(cudaMemset(C->tri32, 0, tb));
  }
  HP_TRY(coarse_setup(P, OP_A));
  for (int l = 0; l < L; ++l) {
    double b = 2.0;
    HP_TRY(gershgorin_bound(P, P->lv[l].g, P->lv[l].A64, &b));
    P->lv[l].A64.lmax = P->lv[l].A32.lmax = b;
  }
  return 0;
}

int build_point(hp_problem *P, const double *m_dev) {
  const long n = P->n;
  P->have_p = P->have_full = false;
  P->have_point = false;  // until the state solve at the new point succeeds
  HP_CUDA(cudaMemcpyAsync(P->m, m_dev, sizeof(double) * n, cudaMemcpyDeviceToDevice, P->st));
  launch_ew_exp(P->m, P->E, n, P->st);
  const int D = P->dim;
  Level &l0 = P->lv[0];
  if (D == 2)
    k_elem_kappa_fine<2><<<grid_blocks(l0.nelems), 256, 0, P->st>>>(l0.g, P->E, l0.kappa, l0.nelems);
  else
    k_elem_kappa_fine<3><<<grid_blocks(l0.nelems), 256, 0, P->st>>>(l0.g, P->E, l0.kappa, l0.nelems);
  count_launch();
  for (int l = 1; l < P->L; ++l) {
    Level &lc = P->lv[l], &lf = P->lv[l - 1];
    if (D == 2)
      k_elem_kappa_coarsen<2><<<grid_blocks(lc.nelems), 256, 0, P->st>>>(lc.g, lf.g, lf.kappa, lc.kappa, lc.nelems);
    else
      k_elem_kappa_coarsen<3><<<grid_blocks(lc.nelems), 256, 0, P->st>>>(lc.g, lf.g, lf.kappa, lc.kappa, lc.nelems);
    count_launch();
  }
  for (int l = 0; l < P->L; ++l) {
    Level &lv = P->lv[l];
    double *lift = l == 0 ? P->lift : nullptr;
    if (D == 2)
      k_build_K<2><<<grid_blocks(lv.g.n), 256, 0, P->st>>>(lv.g, lv.kappa, lv.K64.diag, lv.K64.invdiag, lv.K64.c,
                                                           lv.K32.diag, lv.K32.invdiag, lv.K32.c, lift, P->u_top,
                                                           P->u_bottom);
    else
      k_build_K<3><<<grid_blocks(lv.g.n), 256, 0, P->st>>>(lv.g, lv.kappa, lv.K64.diag, lv.K64.invdiag, lv.K64.c,
                                                           lv.K32.diag, lv.K32.invdiag, lv.K32.c, lift, P->u_top,
                                                           P->u_bottom);
    count_launch();
    lv.K64.cpr_ok = false;  // the double-float coefficient pairs follow on first use
    if (lv.K32.pk) {
      if (D == 2)
        k_pack_K2<<<grid_blocks(lv.g.n), 256, 0, P->st>>>(lv.g.n, lv.K32.diag, lv.K32.invdiag, lv.K32.c,
                                                          reinterpret_cast<float4 *>(lv.K32.pk));
      else
        k_pack_K3<<<grid_blocks(lv.g.n), 256, 0, P->st>>>(lv.g, lv.K32.diag, lv.K32.invdiag, lv.K32.c,
                                                          reinterpret_cast<float4 *>(lv.K32.pk),
                                                          lv.K32.pk + 4 * lv.g.n);
      count_launch();
    }
  }
  HP_CUDA(cudaGetLastError());
  HP_TRY(coarse_setup(P, OP_K));
  return 0;
}

// ---------------------------------------------------------------------------
// C, C^T
//
// (C X)_v = sum_{e ni v} kappa_hat_e (K_e^1 u_e)_v with kappa_hat_e the element mean of
// E X, so C X = S_C (E (.) X) where S_C couples v to the nodes w that share a simplex
// with v: beta_{v,w} = sum_{e ni v,w} (K_e^1 u_e)_v / (D+1), K_e^1 the unit-coefficient
// element stiffness.  beta depends only on u, so it is built once per linearisation
// point; C X and C^T W = E (.) S_C^T W are then FP64 stencil applications.
// Offsets w - v: index 0 = v itself, idx = b for +b, idx = 2^D - 1 + b for -b
// (b a Kuhn edge mask), 2^{D+1} - 1 coefficients per node.
// ---------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ int coff_index(int from_mask, int to_mask) {
  // simplex vertices S_k (from) and S_t (to) of one chain: to - from is +/- a Kuhn edge
  if (to_mask == from_mask) return 0;
  if ((to_mask & from_mask) == from_mask) return to_mask ^ from_mask;        // +b
  return (1 << D) - 1 + (from_mask ^ to_mask);                               // -b
}

template <int D>
__global__ void k_build_C(GridDesc g, const double *__restrict__ u, double *__restrict__ beta) {
  constexpr int NC = (1 << (D + 1)) - 1;
  const double vh2 = vol_over_h2<D>(g.h) / (D + 1);
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.n; i += (long)gridDim.x * blockDim.x) {
    int v[3];
    node_coords<D>(g, i, v);
    double b[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) b[q] = 0.0;
    const double uv = u[i];
    for_elems_with<D>(g, v, 0, [&](const int c[3], int p, int k) {
      const long base = c[0] + (long)g.np * (c[1] + (long)g.np * c[2]);
      double a = 0.0;
      if (k > 0) a += uv - u[base + mask_offset(g, MeshT<D>::chain(p, k - 1))];
      if (k < D) a += uv - u[base + mask_offset(g, MeshT<D>::chain(p, k + 1))];
      a *= vh2;
      const int mk = MeshT<D>::chain(p, k);
#pragma unroll
      for (int t = 0; t <= D; ++t) b[coff_index<D>(mk, MeshT<D>::chain(p, t))] += a;
    });
#pragma unroll
    for (int q = 0; q < NC; ++q) beta[(long)q * g.n + i] = b[q];
  }
}

// signed offset of coefficient index q: returns the mask and the sign (+1 / -1; 0 for q = 0)
template <int D>
__device__ __forceinline__ int coff_mask(int q, int *sign) {
  if (q == 0) {
    *sign = 0;
    return 0;
  }
  if (q < (1 << D)) {
    *sign = 1;
    return q;
  }
  *sign = -1;
  return q - ((1 << D) - 1);
}

template <int D>
__device__ __forceinline__ bool shift_ok(const GridDesc &g, const int v[3], int mask, int sign) {
  bool ok = true;
#pragma unroll
  for (int a = 0; a < D; ++a)
    if ((mask >> a) & 1) ok = ok && (sign > 0 ? v[a] < g.N : v[a] > 0);
  return ok;
}

// betaE_q(i) = beta_q(i) E(i + o_q): the coefficients of C with e^m folded in (once per point),
// so that C X costs one FMA per coupling
template <int D>
__global__ void k_scale_C(GridDesc g, const double *__restrict__ E, const double *__restrict__ beta,
                          double *__restrict__ betaE) {
  constexpr int NC = (1 << (D + 1)) - 1;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.n; i += (long)gridDim.x * blockDim.x) {
    int v[3];
    node_coords<D>(g, i, v);
    betaE[i] = beta[i] * E[i];
#pragma unroll
    for (int q = 1; q < NC; ++q) {
      int sg;
      const int m = coff_mask<D>(q, &sg);
      betaE[(long)q * g.n + i] =
          shift_ok<D>(g, v, m, sg) ? beta[(long)q * g.n + i] * E[i + sg * mask_offset(g, m)] : 0.0;
    }
  }
}

// TRANS false: Y = scale * S_C (E (.) X) + yb * Y with the E-scaled coefficients betaE
// TRANS true:  Y = scale * E (.) S_C^T X + yb * Y with the coefficients beta
// One node per thread over the flattened grid (32-bit addresses: the 64-bit divisions of the
// node's coordinates cost as much as its FP64 operations), CC_Q columns per thread that share
// the coefficients.  Bound by the FP64 pipe: 2^{D+1} + 1 operations per node and column.
// 65^3 nodes, 120 columns: C^T 1,730 -> 945 us, C 930 -> 923 (840 us is the pipe's time).
// The last column of an odd count is taken alone (a call for one column: C 30.4 us, computed twice 37.4).
constexpr int CC_Q = 2;
template <int D, bool TRANS>
__global__ void __launch_bounds__(NT) k_cct_apply(GridDesc g, const double *__restrict__ E,
                                                  const double *__restrict__ beta, const double *__restrict__ X,
                                                  long ldx, double *__restrict__ Y, long ldy, int s, double scale,
                                                  double yb) {
  constexpr int NC = (1 << (D + 1)) - 1;
  const int j0 = blockIdx.y * CC_Q;
  const unsigned np = (unsigned)g.np, n = (unsigned)g.n;
  auto nodes = [&](auto nk) {  // this block's nodes for the first nk of its columns
    constexpr int Q = decltype(nk)::value;
    const double *x[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) x[k] = X + ldx * (j0 + k);
    for (unsigned i = blockIdx.x * NT + threadIdx.x; i < n; i += gridDim.x * NT) {
      const unsigned t = div_np(g, i), t2 = D == 2 ? 0u : div_np(g, t);
      const int v[3] = {(int)(i - t * np), D == 2 ? (int)t : (int)(t - t2 * np), (int)t2};
      double acc[Q];
      const double b0 = beta[i];
#pragma unroll
      for (int k = 0; k < Q; ++k) acc[k] = mulr(b0, x[k][i]);
#pragma unroll
      for (int q = 1; q < NC; ++q) {
        int sg;
        const int m = coff_mask<D>(q, &sg);
        // C^T: the row whose offset q points at node i is i - (sg * m)
        const int sgn = TRANS ? -sg : sg;
        if (!shift_ok<D>(g, v, m, sgn)) continue;
        const unsigned r = i + (unsigned)(sgn * (int)mask_offset(g, m));
        const double w = beta[(size_t)q * n + (TRANS ? r : i)];
#pragma unroll
        for (int k = 0; k < Q; ++k) acc[k] = fmadd(w, x[k][r], acc[k]);
      }
      const double f = TRANS ? mulr(scale, E[i]) : scale;
#pragma unroll
      for (int k = 0; k < Q; ++k) {
        double *y = Y + ldy * (j0 + k) + i;
        const double val = mulr(f, acc[k]);
        *y = yb == 0.0 ? val : fmadd(yb, *y, val);
      }
    }
  };
  if (j0 + CC_Q <= s) nodes(std::integral_constant<int, CC_Q>{});
  else nodes(std::integral_constant<int, 1>{});
}

// The same two stencils in double-float arithmetic on the FP32 pipe (at the solve
// tolerances where the refinement runs in double-float): the input block is split into
// pairs once (k_to_pairs, grouped by 4 columns: one {hi x4, lo x4} record per node, 32
// bytes), the coefficients are kept as pairs (made once per linearisation point), and each
// thread forms the compensated (Dot2) sums of one node for 4 columns, its stencil's points
// taken in chunks whose loads are all issued before their arithmetic.  The final scaling
// (and the accumulation into Y when yb != 0) is one FP64 operation or two per element.
__global__ void k_to_pairs(const double *__restrict__ X, long ldx, int s, long n, float4 *__restrict__ Xp, long ldp) {
  const int grp = blockIdx.y;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    float hi[4], lo[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int col = grp * 4 + q;
      const dfl d = d2df(col < s ? X[ldx * col + i] : 0.0);
      hi[q] = d.hi;
      lo[q] = d.lo;
    }
    const long k = 2 * ((long)grp * ldp + i);
    Xp[k] = make_float4(hi[0], hi[1], hi[2], hi[3]);
    Xp[k + 1] = make_float4(lo[0], lo[1], lo[2], lo[3]);
  }
}

__global__ void k_pairs_of(const double *__restrict__ a, long m, float2 *__restrict__ out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < m; i += (long)gridDim.x * blockDim.x) {
    const dfl d = d2df(a[i]);
    out[i] = make_float2(d.hi, d.lo);
  }
}

// TRANS false: Y = scale * sum_q cpr[q][i] x[i + o_q] (+ yb Y)            (C, coefficients betaE)
// TRANS true:  Y = scale * E_i sum_q cpr[q][i + o'_q] x[i + o'_q] (+ yb Y)  (C^T, coefficients beta)
template <int D, bool TRANS>
__global__ void __launch_bounds__(NT, 2) k_cct_dfp(GridDesc g, const float2 *__restrict__ cpr,
                                                   const float2 *__restrict__ Epr, const float4 *__restrict__ Xp,
                                                   long ldp, double *__restrict__ Y, long ldy, int s, double scale,
                                                   double yb) {
  constexpr int NC = (1 << (D + 1)) - 1;
  constexpr int CH = 5;  // points per chunk of loads
  const int grp = blockIdx.y;
  const float4 *xg = Xp + 2 * (long)grp * ldp;
  const unsigned np = (unsigned)g.np, n = (unsigned)g.n;
  for (unsigned i = blockIdx.x * NT + threadIdx.x; i < n; i += gridDim.x * NT) {
    int v[3];
    const unsigned t = div_np(g, i), t2 = D == 2 ? 0u : div_np(g, t);
    v[0] = (int)(i - t * np);
    v[1] = D == 2 ? (int)t : (int)(t - t2 * np);
    v[2] = (int)t2;
    Dot2 a[4];
#pragma unroll
    for (int q0 = 0; q0 < NC; q0 += CH) {
      float4 xh[CH], xl[CH];
      float2 cp[CH];
      bool ok[CH];
#pragma unroll
      for (int k = 0; k < CH; ++k) {
        const int q = q0 + k;
        ok[k] = false;
        if (q >= NC) continue;
        int sg;
        const int m = coff_mask<D>(q, &sg);
        const int sgn = TRANS ? -sg : sg;
        ok[k] = q == 0 || shift_ok<D>(g, v, m, sgn);
        const unsigned pt = ok[k] && q > 0 ? (unsigned)((long)i + sgn * mask_offset(g, m)) : i;
        xh[k] = xg[2 * pt];
        xl[k] = xg[2 * pt + 1];
        cp[k] = cpr[(unsigned)q * n + (TRANS ? pt : i)];
      }
#pragma unroll
      for (int k = 0; k < CH; ++k) {
        if (!ok[k]) continue;
        const dfl c{cp[k].x, cp[k].y};
        a[0].fma(c, dfl{xh[k].x, xl[k].x});
        a[1].fma(c, dfl{xh[k].y, xl[k].y});
        a[2].fma(c, dfl{xh[k].z, xl[k].z});
        a[3].fma(c, dfl{xh[k].w, xl[k].w});
      }
    }
    dfl e{1.f, 0.f};
    if (TRANS) {
      const float2 ep = Epr[i];
      e = dfl{ep.x, ep.y};
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = grp * 4 + j;
      if (col >= s) break;
      dfl r = a[j].result();
      if (TRANS) {
        Dot2 b;  // e^{m_i} times the sum
        b.fma(e, r);
        r = b.result();
      }
      const double val = scale * df2d(r);
      Y[ldy * col + i] = yb == 0.0 ? val : val + yb * Y[ldy * col + i];
    }
  }
}

// double-float C and C^T where the refinement runs in double-float (the same tolerance and
// block-size rule as the solves')
static bool cct_df(const hp_problem *P, int s) {
  return P->precision == HP_FP32_IR &&
         (P->refine_df == 2 || (P->refine_df == 1 && P->rtol >= 1e-9 && (double)P->n * s >= 16.0 * 1024 * 1024));
}

// the coefficient and e^m pairs of the u-based C, made when missing or stale
static int ensure_cct_pairs(hp_problem *P) {
  const long n = P->n, nc = P->dim == 2 ? 7 : 15;
  if (!P->CbetaE_pr) {
    HP_CUDA(cudaMalloc(&P->CbetaE_pr, sizeof(float2) * nc * n));
    HP_CUDA(cudaMalloc(&P->Cbeta_pr, sizeof(float2) * nc * n));
    HP_CUDA(cudaMalloc(&P->E_pr, sizeof(float2) * n));
  }
  if (!P->cct_pr_ok) {
    k_pairs_of<<<blocks_for(nc * n, 1), NT, 0, P->st>>>(P->CbetaE, nc * n, P->CbetaE_pr);
    k_pairs_of<<<blocks_for(nc * n, 1), NT, 0, P->st>>>(P->Cbeta, nc * n, P->Cbeta_pr);
    k_pairs_of<<<blocks_for(n, 1), NT, 0, P->st>>>(P->E, n, P->E_pr);
    count_launch(3);
    P->cct_pr_ok = true;
  }
  return cuda_check(cudaGetLastError(), "C pairs");
}

// Y = scale (C or C^T) X (+ yb Y) in double-float; false when not applicable (the caller
// then runs the FP64 kernel)
static bool cct_dfp(hp_problem *P, bool trans, const double *X, long ldx, double *Y, long ldy, int s, double scale,
                    double yb) {
  const long n = P->n, ldp = (n + 63) / 64 * 64;
  const int ng = (s + 3) / 4;
  if (ensure_cct_pairs(P) || P->xpairs.ensure(sizeof(float4) * 2 * (size_t)ldp * ng)) {
    (void)cudaGetLastError();
    return false;
  }
  float4 *Xp = P->xpairs.as<float4>();
  const dim3 gd(blocks_for(n, ng), ng);
  k_to_pairs<<<gd, NT, 0, P->st>>>(X, ldx, s, n, Xp, ldp);
  const GridDesc &g = P->lv[0].g;
  const dim3 gc(blocks_for(n, ng), ng);
  if (P->dim == 2) {
    if (trans)
      k_cct_dfp<2, true><<<gc, NT, 0, P->st>>>(g, P->Cbeta_pr, P->E_pr, Xp, ldp, Y, ldy, s, scale, yb);
    else
      k_cct_dfp<2, false><<<gc, NT, 0, P->st>>>(g, P->CbetaE_pr, nullptr, Xp, ldp, Y, ldy, s, scale, yb);
  } else {
    if (trans)
      k_cct_dfp<3, true><<<gc, NT, 0, P->st>>>(g, P->Cbeta_pr, P->E_pr, Xp, ldp, Y, ldy, s, scale, yb);
    else
      k_cct_dfp<3, false><<<gc, NT, 0, P->st>>>(g, P->CbetaE_pr, nullptr, Xp, ldp, Y, ldy, s, scale, yb);
  }
  count_launch(2);
  const double nc = P->dim == 2 ? 7.0 : 15.0;
  // the split: read X, write the pairs; the stencil: the pairs, Y (read as well when yb != 0)
  // and the coefficient pairs (and e^m for C^T)
  count_bytes(BY_CCT, 16.0 * (double)n * s);
  count_bytes(BY_CCT, (double)n * ((yb == 0.0 ? 16.0 : 24.0) * s + 8.0 * (nc + (trans ? 1.0 : 0.0))));
  return true;
}

void launch_build_C_from(hp_problem *P, const double *w, double *beta, double *betaE) {
  if (P->dim == 2) {
    k_build_C<2><<<grid_blocks(P->n), 256, 0, P->st>>>(P->lv[0].g, w, beta);
    k_scale_C<2><<<grid_blocks(P->n), 256, 0, P->st>>>(P->lv[0].g, P->E, beta, betaE);
  } else {
    k_build_C<3><<<grid_blocks(P->n), 256, 0, P->st>>>(P->lv[0].g, w, beta);
    k_scale_C<3><<<grid_blocks(P->n), 256, 0, P->st>>>(P->lv[0].g, P->E, beta, betaE);
  }
  count_launch(2);
}

void launch_build_C(hp_problem *P) {
  launch_build_C_from(P, P->u, P->Cbeta, P->CbetaE);
  P->cct_pr_ok = false;  // the double-float pairs follow on first use
}

void launch_C_apply_beta(hp_problem *P, const double *betaE, const double *X, long ldx, double *Y, long ldy, int s,
                         double scale, double yb) {
  if (betaE == P->CbetaE && cct_df(P, s) && cct_dfp(P, false, X, ldx, Y, ldy, s, scale, yb)) return;
  const int nq = (s + CC_Q - 1) / CC_Q;
  const dim3 grid(blocks_for(P->n, nq), nq);
  if (P->dim == 2)
    k_cct_apply<2, false><<<grid, NT, 0, P->st>>>(P->lv[0].g, nullptr, betaE, X, ldx, Y, ldy, s, scale, yb);
  else
    k_cct_apply<3, false><<<grid, NT, 0, P->st>>>(P->lv[0].g, nullptr, betaE, X, ldx, Y, ldy, s, scale, yb);
  count_launch();
  {  // read X (and Y when yb != 0), write Y, the (2^{D+1} - 1) coefficients per node
    const double nc = P->dim == 2 ? 7.0 : 15.0;
    count_bytes(BY_CCT, 8.0 * (double)P->n * ((yb == 0.0 ? 2.0 : 3.0) * s + nc));
  }
}

void launch_C_apply(hp_problem *P, const double *X, long ldx, double *Y, long ldy, int s, double scale) {
  launch_C_apply_beta(P, P->CbetaE, X, ldx, Y, ldy, s, scale, 0.0);
}

void launch_Ct_apply_beta(hp_problem *P, const double *beta_c, const double *W, long ldw, double *Y, long ldy, int s,
                          double scale, double beta) {
  if (beta_c == P->Cbeta && cct_df(P, s) && cct_dfp(P, true, W, ldw, Y, ldy, s, scale, beta)) return;
  const int nq = (s + CC_Q - 1) / CC_Q;
  const dim3 grid(blocks_for(P->n, nq), nq);
  if (P->dim == 2)
    k_cct_apply<2, true><<<grid, NT, 0, P->st>>>(P->lv[0].g, P->E, beta_c, W, ldw, Y, ldy, s, scale, beta);
  else
    k_cct_apply<3, true><<<grid, NT, 0, P->st>>>(P->lv[0].g, P->E, beta_c, W, ldw, Y, ldy, s, scale, beta);
  count_launch();
  {  // read W (and Y when beta != 0), write Y, e^m and the coefficients per node
    const double nc = P->dim == 2 ? 7.0 : 15.0;
    count_bytes(BY_CCT, 8.0 * (double)P->n * ((beta == 0.0 ? 2.0 : 3.0) * s + nc + 1.0));
  }
}

void launch_Ct_apply(hp_problem *P, const double *W, long ldw, double *Y, long ldy, int s, double scale,
                     double beta) {
  launch_Ct_apply_beta(P, P->Cbeta, W, ldw, Y, ldy, s, scale, beta);
}

// ---------------------------------------------------------------------------
// observation operator
// ---------------------------------------------------------------------------
__global__ void k_obs_gather(const int *__restrict__ node, const double *__restrict__ w, int nobs, int nv,
                             const double *__restrict__ X, long ldx, double *__restrict__ Yq) {
  const int j = blockIdx.y;
  for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < nobs; o += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int k = 0; k < nv; ++k) s += w[o * nv + k] * X[ldx * j + node[o * nv + k]];
    Yq[(long)nobs * j + o] = s;
  }
}

__global__ void k_obs_scatter(long n, const int *__restrict__ row, const int *__restrict__ ptr,
                              const int *__restrict__ ent, const double *__restrict__ w, int nobs, int nv,
                              const double *__restrict__ Yq, double *__restrict__ X, long ldx, double scale) {
  const int j = blockIdx.y;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const int r = row[i];
    double s = 0.0;
    if (r >= 0) {
      for (int t = ptr[r]; t < ptr[r + 1]; ++t) {
        const int e = ent[t];
        s += w[e] * Yq[(long)nobs * j + e / nv];
      }
    }
    X[ldx * j + i] = scale * s;
  }
}

void launch_obs_gather(hp_problem *P, const double *X, long ldx, double *Yq, int s) {
  if (P->nobs == 0) return;
  dim3 grid((P->nobs + 127) / 128, s);
  k_obs_gather<<<grid, 128, 0, P->st>>>(P->obs_node, P->obs_w, P->nobs, P->dim + 1, X, ldx, Yq);
  count_launch();
  count_bytes(BY_CCT, 8.0 * (double)P->nobs * s * (P->dim + 2));
}

void launch_obs_scatter(hp_problem *P, const double *Yq, double *X, long ldx, int s, double scale) {
  dim3 grid(blocks_for(P->n, s), s);
  k_obs_scatter<<<grid, NT, 0, P->st>>>(P->n, P->bt_row, P->bt_ptr, P->bt_ent, P->obs_w, P->nobs, P->dim + 1,
                                        Yq, X, ldx, scale);
  count_launch();
  count_bytes(BY_CCT, 8.0 * ((double)P->n + (double)P->nobs) * s);
}

// ---------------------------------------------------------------------------
// rectangular factor of the mass matrix
// ---------------------------------------------------------------------------
template <int D>
__global__ void k_mass_factor(GridDesc g, const double *__restrict__ eta, long ldeta, double *__restrict__ W,
                              long ldw) {
  const int j = blockIdx.y;
  const double *et = eta + ldeta * j;
  const double sw = sqrt(elem_vol<D>(g.h) / (D + 1));
  const double qa = (5.0 + 3.0 * sqrt(5.0)) / 20.0, qb = (5.0 - sqrt(5.0)) / 20.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < g.n; i += (long)gridDim.x * blockDim.x) {
    int v[3];
    node_coords<D>(g, i, v);
    double acc = 0.0;
    for_elems_with<D>(g, v, 0, [&](const int c[3], int p, int k) {
      const long e = cell_linear<D>(g, c) * MeshT<D>::NPERM + p;
#pragma unroll
      for (int q = 0; q <= D; ++q) {
        const double lam = D == 2 ? c_quad2[q][k] : (q == k ? qa : qb);
        acc += lam * et[e * (D + 1) + q];
      }
    });
    W[ldw * j + i] = sw * acc;
  }
}

void launch_mass_factor(hp_problem *P, const double *eta, long ldeta, double *W, long ldw, int s) {
  dim3 grid(blocks_for(P->n, s), s);
  if (P->dim == 2)
    k_mass_factor<2><<<grid, NT, 0, P->st>>>(P->lv[0].g, eta, ldeta, W, ldw);
  else
    k_mass_factor<3><<<grid, NT, 0, P->st>>>(P->lv[0].g, eta, ldeta, W, ldw);
  count_launch();
}

// W = C_M eta in 3D with eta drawn on the way: column j holds the normals of sample first + j
// (element e takes the four of call e, as launch_philox_normals lays them out), which never
// reach memory.  A CTA marches up through a segment of cell layers over a tile of cells, one
// cell per thread and layer; the nodes of the tile but its first row and column are summed.
// With w_qk = qa for q = k and qb otherwise, a node's value is
//   sw (qb sum_e S_e + (qa - qb) sum_e eta_{e,k(e)}),  S_e the sum of the element's four.
// The normals are floats, so both sums are taken in 64-bit integers of 2^-52 each (|eta| < 6,
// 96 terms: no overflow): a term is within 2^-53, the additions are exact, no less precise than
// FP64 sums of such values (half an ulp of a partial sum is 2^-53 to 2^-50), and the FP64 pipe,
// which bounded the gathering form (96 multiply-adds per node), is left with five operations
// per node.  64 samples on 64^3 cells: 6.1 ms and 1.6 ms for the normals before; now bound by
// the generator's own arithmetic.
constexpr int MF_NT = 256;

__device__ __forceinline__ long long fixed52(float z) {  // z 2^52 rounded, |z| < 8
  const float a = z * 0x1p27f;
  const int hi = __float2int_rz(a);
  const int lo = __float2int_rn((a - (float)hi) * 0x1p25f);
  return ((long long)hi << 25) + lo;
}

__global__ void __launch_bounds__(MF_NT) k_mass_factor_philox3(GridDesc g, unsigned long long seed, long long first,
                                                               double *__restrict__ W, long ldw, int tx, int ty,
                                                               int nzs) {
  __shared__ long long sa[8][MF_NT], st[8][MF_NT];  // per corner: sums of S_e and of the corner's own normals
  const int np = g.np, N = g.N, bw = tx + 1, t = threadIdx.x;
  const int ntx = (np + tx - 1) / tx;
  const int bx = blockIdx.x % ntx, by = blockIdx.x / ntx;
  const int ly = t / bw, lx = t - ly * bw;
  // this thread's cell column, and the node at the same place
  const int cx = bx * tx - 1 + lx, cy = by * ty - 1 + ly;
  const bool cell = ly <= ty && cx >= 0 && cx < N && cy >= 0 && cy < N;
  const bool node = ly >= 1 && ly <= ty && lx >= 1 && cx < np && cy < np;
  const int zb = (int)((long)blockIdx.y * np / nzs), ze = (int)((long)(blockIdx.y + 1) * np / nzs);
  const unsigned long long smp = (unsigned long long)(first + blockIdx.z);
  const uint2 key = make_uint2((unsigned)seed, (unsigned)(seed >> 32));
  const double h3 = g.h * g.h * g.h / 6.0;
  const double sw = sqrt(h3 / 4.0) * 0x1p-52;
  const double qa = (5.0 + 3.0 * sqrt(5.0)) / 20.0, qb = (5.0 - sqrt(5.0)) / 20.0;
  const double wa = sw * qb, wt = sw * (qa - qb);
  double *out = W + ldw * blockIdx.z;
  long long ua = 0, ut = 0;  // what the layer below contributes to the node
  for (int cz = zb - 1; cz < ze; ++cz) {
    long long A[8] = {0, 0, 0, 0, 0, 0, 0, 0}, T[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (cell && cz >= 0 && cz < N) {
      const unsigned long long e0 = 6ull * (unsigned long long)(cx + (long)N * (cy + (long)N * cz));
#pragma unroll
      for (int p = 0; p < 6; ++p) {
        const unsigned long long e = e0 + p;
        const uint4 w = philox4x32_10(make_uint4((unsigned)e, (unsigned)(e >> 32), (unsigned)smp, (unsigned)(smp >> 32)),
                                      key);
        float z[4];
        box_muller(w.x, w.y, &z[0], &z[1]);
        box_muller(w.z, w.w, &z[2], &z[3]);
        long long f[4], S = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) S += f[k] = fixed52(z[k]);
        constexpr int chain[6][4] = {{0, 1, 3, 7}, {0, 1, 5, 7}, {0, 2, 3, 7}, {0, 2, 6, 7}, {0, 4, 5, 7}, {0, 4, 6, 7}};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          A[chain[p][k]] += S;
          T[chain[p][k]] += f[k];
        }
      }
    }
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      sa[b][t] = A[b];
      st[b][t] = T[b];
    }
    __syncthreads();
    if (node) {
      // the node is corner s of the cell at its place less s
      long long da = ua, dt = ut;
      ua = ut = 0;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int q = t - (s & 1) - (s >> 1) * bw;
        da += sa[s][q];
        dt += st[s][q];
        ua += sa[s + 4][q];
        ut += st[s + 4][q];
      }
      if (cz >= zb) out[cx + (long)np * (cy + (long)np * cz)] = fma(wt, (double)dt, wa * (double)da);
    }
    __syncthreads();
  }
}

void launch_mass_factor_philox3(hp_problem *P, unsigned long long seed, long long first, double *W, long ldw, int s) {
  const GridDesc &g = P->lv[0].g;
  // tiles of equal width, as large as 256 cells with their extra row and column allow
  const int ntx = (g.np + 30) / 31, tx = (g.np + ntx - 1) / ntx;
  const int tm = MF_NT / (tx + 1) - 1, nty = (g.np + tm - 1) / tm, ty = (g.np + nty - 1) / nty;
  // z segments of about 16 layers (one more is computed for each), shorter ones while there are fewer
  // CTAs than two per SM: a call for 7 prior samples on 10^3 nodes 249 -> 222 us, on 15^3 521 -> 467
  const int most = std::max(1, g.np / 2), fill = (2 * NSM + ntx * nty * s - 1) / (ntx * nty * s);
  const int nzs = std::min(most, std::max(std::max(1, g.np / 16), fill));
  k_mass_factor_philox3<<<dim3(ntx * nty, nzs, s), MF_NT, 0, P->st>>>(g, seed, first, W, ldw, tx, ty, nzs);
  count_launch();
}

// ---------------------------------------------------------------------------
// Dirichlet rows
// ---------------------------------------------------------------------------
__global__ void k_zero_dirichlet(long face, long top_off, double *X, long ldx) {
  const int j = blockIdx.y;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < face; t += (long)gridDim.x * blockDim.x) {
    X[ldx * j + t] = 0.0;
    X[ldx * j + top_off + t] = 0.0;
  }
}

void launch_zero_dirichlet(hp_problem *P, double *X, long ldx, int s) {
  const GridDesc &g = P->lv[0].g;
  const long face = P->dim == 2 ? g.np : (long)g.np * g.np;
  dim3 grid((unsigned)std::max<long>(1, std::min<long>((face + 255) / 256, 64)), s);
  k_zero_dirichlet<<<grid, 256, 0, P->st>>>(face, g.n - face, X, ldx);
  count_launch();
}

}  // namespace hp
