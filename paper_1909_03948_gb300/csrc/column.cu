// column.cu -- multigrid work of one right-hand side inside one CTA.
//
// A level of up to COL_MAXN nodes fits in one SM's shared memory with every vector that its
// V-cycle (or its whole PCG) needs, and its stencil's coefficients fit in the CTA's
// registers.  The steps of the cycle are then separated by block barriers instead of kernel
// launches (2.2 to 2.8 us each inside a CUDA graph, which is what bounded these levels: each
// of their kernels moves far less than it takes to launch).  Two kernels share the code:
//   k_vtail   the V-cycle from level l0 down and back, one CTA per column: the coarse end
//             of a larger problem's preconditioner (one launch in place of nine per level);
//   k_colpcg  the whole PCG of a column, for problems whose finest level already fits: the
//             columns are independent, so each CTA iterates until its own column converges.
// One column per CTA (not a group of four) because these launches are short of CTAs, not of
// bandwidth: 60 columns occupy 60 of the 152 SMs.  One SM's issue rate bounds the kernels, so
// the sweeps are laid out for few instructions per node: in 2D a thread owns NPT vertically
// consecutive nodes of one grid column, whose values and coefficients stay in its registers
// through a leg's sweeps; only the neighbours to the left and right (and the ends of the
// strip) come from shared memory.
//
// Vectors are FP32 in shared memory with `pad` zeros on both sides of the flattened grid, so
// that a stencil needs no boundary tests: a coupling that leaves the grid is zero (the
// stencils store it so), a neighbour index that leaves the array reads the padding, and one
// that wraps to another row meets a zero coupling.  Every value is formed by the operations
// of the per-level kernels in their order, so a solve has the same bits either way (the square
// coarse inverse is made symmetric to the last bit where its triangle may be held here).
#include <algorithm>
#include <atomic>
#include <cstring>
#include <type_traits>

#include "dfloat.cuh"
#include "internal.h"

namespace hp {

// threads per CTA: 2D strips need at most 896 (71 columns of 12 strips), which leaves 72
// registers each; 3D takes all 1024
template <int D> constexpr int col_nt() { return D == 2 ? 896 : 1024; }
constexpr int COL_NPT = 6;            // most nodes per thread on the finest level held
constexpr int COL_SMEM = 220 * 1024;  // dynamic shared memory (227 KB less the static part)

extern __shared__ __align__(16) float col_sm[];

template <int D, bool FULL> struct ColShape {
  static constexpr int NF = FULL ? (1 << D) - 1 : D;
  // coefficients per node (diagonal, its inverse, both directions of each coupling) and
  // whether a thread of the flattened mapping keeps those of its NPT nodes in registers over
  // a leg (64 registers per thread at 1024 threads; otherwise every sweep reads them through L1)
  static constexpr int NC = 2 + 2 * NF;
  template <int NPT> static constexpr bool in_regs() { return NC * NPT <= 40; }
};

// offset of coupling f on a grid of np nodes per axis
template <int D, bool FULL> __device__ __forceinline__ int col_off(int np, int f) {
  const int b = FULL ? f + 1 : (1 << f);
  return (b & 1) + ((b >> 1) & 1) * np + (D == 3 ? ((b >> 2) & 1) * np * np : 0);
}

// A thread's view of a level's stencil: everything the sweeps need held in registers (the
// level's description lives in the kernel's parameters, and reading it through a reference
// again after every store to shared memory costs more than the sweep).
template <int D, bool FULL, int NPT> struct ColCoef {
  static constexpr int NF = ColShape<D, FULL>::NF;
  static constexpr bool REG = ColShape<D, FULL>::template in_regs<NPT>();
  static constexpr int NR = REG ? NPT : 1;
  float d[NR], iv[NR], cf[NR][NF], cb[NR][NF];
  int n, off[NF];
  const float *__restrict__ diag, *__restrict__ invdiag, *__restrict__ c;
  __device__ __forceinline__ explicit ColCoef(const ColLevel &l)
      : n(l.n), diag(l.diag), invdiag(l.invdiag), c(l.c) {
#pragma unroll
    for (int f = 0; f < NF; ++f) off[f] = col_off<D, FULL>(l.np, f);
    if constexpr (REG) {
#pragma unroll
      for (int k = 0; k < NPT; ++k) load_node(k, min((int)threadIdx.x + k * col_nt<D>(), n - 1));
    }
  }
  __device__ __forceinline__ void load_node(int k, int id) {
    d[k] = __ldg(diag + id);
    iv[k] = __ldg(invdiag + id);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      cf[k][f] = __ldg(c + f * n + id);
      // a backward neighbour before the array's start is padding (zero): any finite
      // coefficient serves there
      cb[k][f] = __ldg(c + f * n + max(id - off[f], 0));
    }
  }
  // S x at the thread's node k (id)
  __device__ __forceinline__ float apply(int k, int id, int x) {
    if constexpr (!REG) load_node(0, id);
    const int q = REG ? k : 0;
    const float *xi = col_sm + x + id;
    float acc = mulr(d[q], xi[0]);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      acc = fmadd(cf[q][f], xi[off[f]], acc);
      acc = fmadd(cb[q][f], xi[-off[f]], acc);
    }
    return acc;
  }
  __device__ __forceinline__ float inv(int k, int id) const { return REG ? iv[k] : __ldg(invdiag + id); }
};

// runs body(k, id) for the nodes of this thread (NPT the least number that covers n)
template <int D, int NPT, class F> __device__ __forceinline__ void col_nodes(int n, F &&body) {
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    const int id = (int)threadIdx.x + k * col_nt<D>();
    if (k < NPT - 1 || id < n) body(k, id);
  }
}

// y[id] = val(k, id) for the nodes of this thread, every value formed before the first store
// (the stores would otherwise hold back the next node's loads), then a barrier
template <int D, int NPT, class F> __device__ __forceinline__ void col_set(int n, int y, F &&val) {
  float out[NPT];
  col_nodes<D, NPT>(n, [&](int k, int id) { out[k] = val(k, id); });
  col_nodes<D, NPT>(n, [&](int k, int id) { col_sm[y + id] = out[k]; });
  __syncthreads();
}

// Two sweeps from zero (the arithmetic of k_st's M_JAC2): e1 = w1 D^-1 r,
// y = e1 + w2 D^-1 (r - S e1), the neighbours entering as (c w1 / diag) r
template <int D, bool FULL, int NPT>
__device__ __forceinline__ void col_two_sweeps(ColCoef<D, FULL, NPT> &C, float w1, float w2, int r, int y) {
  col_set<D, NPT>(C.n, y, [&](int k, int id) {
    if constexpr (!C.REG) C.load_node(0, id);
    const int q = C.REG ? k : 0;
    const float *ri = col_sm + r + id;
    const float rc = ri[0], e1 = mulr(mulr(w1, C.iv[q]), rc);
    float acc = mulr(C.d[q], e1);
#pragma unroll
    for (int f = 0; f < C.NF; ++f) {
      const int o = C.off[f];
      acc = fmadd(mulr(mulr(C.cf[q][f], w1), __ldg(C.invdiag + min(id + o, C.n - 1))), ri[o], acc);
      acc = fmadd(mulr(mulr(C.cb[q][f], w1), __ldg(C.invdiag + max(id - o, 0))), ri[-o], acc);
    }
    return fmadd(mulr(w2, C.iv[q]), addr(rc, -acc), e1);
  });
}

// y = x + w D^-1 (r - S x)
template <int D, bool FULL, int NPT>
__device__ __forceinline__ void col_sweep(ColCoef<D, FULL, NPT> &C, int x, int r, int y, float w) {
  col_set<D, NPT>(C.n, y, [&](int k, int id) {
    const float sx = C.apply(k, id, x);
    return fmadd(mulr(w, C.inv(k, id)), addr(col_sm[r + id], -sx), col_sm[x + id]);
  });
}

// Pre-smoothing of a level from zero and the residual.  R, A, B: the places of the level's
// right-hand side and two iterates; the smoothed iterate ends in A when nu is even, in B when
// odd, the residual in the other.
template <int D, bool FULL, int NPT>
__device__ __noinline__ void col_down(const ColLevel &l) {
  ColCoef<D, FULL, NPT> C(l);
  const int nu = l.nu, R = l.offr;
  const float w[4] = {l.w[0], l.w[1], l.w[2], l.w[3]};
  int x = l.offa, y = l.offb;
  if (nu >= 2) {
    col_two_sweeps<D, FULL, NPT>(C, w[0], w[1], R, x);
#pragma unroll
    for (int s = 2; s < 4; ++s) {
      if (s >= nu) break;
      col_sweep<D, FULL, NPT>(C, x, R, y, w[s]);
      const int t = x;
      x = y;
      y = t;
    }
  } else {
    x = l.offb;
    y = l.offa;
    col_set<D, NPT>(C.n, x, [&](int k, int id) { return mulr(mulr(w[0], C.inv(k, id)), col_sm[R + id]); });
  }
  col_set<D, NPT>(C.n, y, [&](int k, int id) { return addr(col_sm[R + id], -C.apply(k, id, x)); });
}

// Post-smoothing of nu sweeps: the iterate is in A for even nu, else in B, and ends in A.
template <int D, bool FULL, int NPT>
__device__ __noinline__ void col_up(const ColLevel &l) {
  ColCoef<D, FULL, NPT> C(l);
  const int nu = l.nu, R = l.offr;
  const float w[4] = {l.w[0], l.w[1], l.w[2], l.w[3]};
  int x = (nu & 1) ? l.offb : l.offa, y = (nu & 1) ? l.offa : l.offb;
#pragma unroll
  for (int s = 3; s >= 0; --s) {
    if (s >= nu) continue;
    col_sweep<D, FULL, NPT>(C, x, R, y, w[s]);
    const int t = x;
    x = y;
    y = t;
  }
}

// A thread's strip of a 2D level: nodes (x, y0 .. y0 + m - 1).
template <bool FULL, int NPT> struct ColStrip {
  int np, at, m;  // nodes per row, index of the first node, valid nodes (0: a thread without one)
  // diagonal, its inverse, couplings to x + 1 and x - 1, to y + 1 (cy[k + 1]) and y - 1 (cy[k]),
  // and (FULL) to (x + 1, y + 1) and (x - 1, y - 1); zero for nodes that do not exist
  float d[NPT], iv[NPT], cx[NPT], cxm[NPT], cy[NPT + 1], cd[FULL ? NPT : 1], cdm[FULL ? NPT : 1];
  __device__ __forceinline__ explicit ColStrip(const ColLevel &l) : np(l.np) {
    const int t = threadIdx.x, s = t / np, y0 = s * NPT, n = l.n;
    at = y0 * np + (t - s * np);
    m = min(NPT, max(0, np - y0));
    const float *c = l.c;
    // every load is issued unconditionally at a clamped index (a load under a condition waits
    // for the one before it), and what does not exist is cleared afterwards
    auto at_or = [&](const float *p, int id) { return __ldg(p + min(max(id, 0), n - 1)); };
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int id = at + k * np;
      d[k] = at_or(l.diag, id);
      iv[k] = at_or(l.invdiag, id);
      cx[k] = at_or(c, id);
      cxm[k] = at_or(c, id - 1);
      cy[k + 1] = at_or(c + n, id);
      if constexpr (FULL) {
        cd[k] = at_or(c + 2 * n, id);
        cdm[k] = at_or(c + 2 * n, id - np - 1);
      }
    }
    cy[0] = at_or(c + n, at - np);
    if (at < np) cy[0] = 0.f;
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int id = at + k * np;
      if (k >= m) d[k] = iv[k] = cx[k] = cxm[k] = cy[k + 1] = 0.f;
      if (id < 1) cxm[k] = 0.f;
      if constexpr (FULL) {
        if (k >= m) cd[k] = cdm[k] = 0.f;
        if (id < np + 1) cdm[k] = 0.f;
      }
    }
  }
  // the strip's values of the vector at v
  __device__ __forceinline__ void get(int v, float x[NPT]) const {
#pragma unroll
    for (int k = 0; k < NPT; ++k) x[k] = k < m ? col_sm[v + at + k * np] : 0.f;
  }
  __device__ __forceinline__ void put(int v, const float x[NPT]) const {
#pragma unroll
    for (int k = 0; k < NPT; ++k)
      if (k < m) col_sm[v + at + k * np] = x[k];
  }
  // y_k = S x at the strip's nodes for the vector at v, whose own values are x; the weights of
  // the neighbours' values come from wx/wxm/wy/wym/wd/wdm (k), the centre's product is c0[k]
  template <class WX, class WXM, class WY, class WYM, class WD, class WDM>
  __device__ __forceinline__ void stencil(int v, const float x[NPT], const float c0[NPT], float y[NPT], WX &&wx,
                                          WXM &&wxm, WY &&wy, WYM &&wym, WD &&wd, WDM &&wdm) const {
    if (m == 0) return;
    const float *p = col_sm + v + at;
    float xr[NPT + 1], xl[NPT + 1];  // columns x + 1 (rows 0 .. NPT) and x - 1 (rows -1 .. NPT - 1)
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      xr[k] = k < m ? p[k * np + 1] : 0.f;
      xl[k + 1] = k < m ? p[k * np - 1] : 0.f;
    }
    // the row past a full strip (a partial one ends at the grid's last row: no coupling)
    const bool more = m == NPT;
    const float up = more ? p[NPT * np] : 0.f, dn = p[-np];
    if constexpr (FULL) {
      xr[NPT] = more ? p[NPT * np + 1] : 0.f;
      xl[0] = p[-np - 1];
    }
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      float acc = c0[k];
      acc = fmadd(wx(k), xr[k], acc);
      acc = fmadd(wxm(k), xl[k + 1], acc);
      acc = fmadd(wy(k), k + 1 < NPT ? x[k + 1 < NPT ? k + 1 : 0] : up, acc);
      acc = fmadd(wym(k), k > 0 ? x[k > 0 ? k - 1 : 0] : dn, acc);
      if constexpr (FULL) {
        acc = fmadd(wd(k), xr[k + 1], acc);
        acc = fmadd(wdm(k), xl[k], acc);
      }
      y[k] = acc;
    }
  }
  __device__ __forceinline__ void apply(int v, const float x[NPT], float y[NPT]) const {
    float c0[NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) c0[k] = mulr(d[k], x[k]);
    stencil(
        v, x, c0, y, [&](int k) { return cx[k]; }, [&](int k) { return cxm[k]; }, [&](int k) { return cy[k + 1]; },
        [&](int k) { return cy[k]; }, [&](int k) { return cd[FULL ? k : 0]; }, [&](int k) { return cdm[FULL ? k : 0]; });
  }
};

// x <- x + w D^-1 (r - S x) of the vector at v into the vector at t
template <bool FULL, int NPT>
__device__ __forceinline__ void strip_sweep(const ColStrip<FULL, NPT> &C, float x[NPT], const float r[NPT], int v,
                                            int t, float w) {
  float sx[NPT];
  C.apply(v, x, sx);
#pragma unroll
  for (int k = 0; k < NPT; ++k) x[k] = fmadd(mulr(w, C.iv[k]), addr(r[k], -sx[k]), x[k]);
  C.put(t, x);
  __syncthreads();
}

// the 2D legs (see col_down and col_up)
template <bool FULL, int NPT> __device__ __noinline__ void strip_down(const ColLevel &l) {
  const ColStrip<FULL, NPT> C(l);
  const int nu = l.nu;
  const float w[4] = {l.w[0], l.w[1], l.w[2], l.w[3]};
  float r[NPT], x[NPT], sx[NPT];
  C.get(l.offr, r);
  int v = l.offa, t = l.offb;
  if (nu >= 2) {
    // inverse diagonals of the neighbouring columns, rows -1 .. NPT (outside the grid, where
    // the coupling is zero, any value serves); the strip's own column is in C.iv
    float ir[NPT + 2], il[NPT + 2];
    const int np = C.np;
    auto inv_at = [&](int id) { return __ldg(l.invdiag + min(max(id, 0), l.n - 1)); };
#pragma unroll
    for (int k = 0; k < NPT + 2; ++k) {
      ir[k] = inv_at(C.at + (k - 1) * np + 1);
      il[k] = inv_at(C.at + (k - 1) * np - 1);
    }
    const float iu = inv_at(C.at + NPT * np), id = inv_at(C.at - np);
    // couplings times w1 / diag of the neighbour
    auto wt = [&](float c, float i) { return mulr(mulr(c, w[0]), i); };
    float e1[NPT], c0[NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      e1[k] = mulr(mulr(w[0], C.iv[k]), r[k]);
      c0[k] = mulr(C.d[k], e1[k]);
    }
    C.stencil(
        l.offr, r, c0, sx, [&](int k) { return wt(C.cx[k], ir[k + 1]); }, [&](int k) { return wt(C.cxm[k], il[k + 1]); },
        [&](int k) { return wt(C.cy[k + 1], k + 1 < NPT ? C.iv[k + 1 < NPT ? k + 1 : 0] : iu); },
        [&](int k) { return wt(C.cy[k], k > 0 ? C.iv[k > 0 ? k - 1 : 0] : id); },
        [&](int k) { return wt(C.cd[FULL ? k : 0], ir[k + 2]); }, [&](int k) { return wt(C.cdm[FULL ? k : 0], il[k]); });
#pragma unroll
    for (int k = 0; k < NPT; ++k) x[k] = fmadd(mulr(w[1], C.iv[k]), addr(r[k], -sx[k]), e1[k]);
    C.put(v, x);
    __syncthreads();
#pragma unroll
    for (int s = 2; s < 4; ++s) {
      if (s >= nu) break;
      strip_sweep<FULL, NPT>(C, x, r, v, t, w[s]);
      const int q = v;
      v = t;
      t = q;
    }
  } else {
    v = l.offb;
    t = l.offa;
#pragma unroll
    for (int k = 0; k < NPT; ++k) x[k] = mulr(mulr(w[0], C.iv[k]), r[k]);
    C.put(v, x);
    __syncthreads();
  }
  C.apply(v, x, sx);
#pragma unroll
  for (int k = 0; k < NPT; ++k) x[k] = addr(r[k], -sx[k]);
  C.put(t, x);
  __syncthreads();
}

template <bool FULL, int NPT> __device__ __noinline__ void strip_up(const ColLevel &l) {
  const ColStrip<FULL, NPT> C(l);
  const int nu = l.nu;
  const float w[4] = {l.w[0], l.w[1], l.w[2], l.w[3]};
  int v = (nu & 1) ? l.offb : l.offa, t = (nu & 1) ? l.offa : l.offb;
  float r[NPT], x[NPT];
  C.get(l.offr, r);
  C.get(v, x);
#pragma unroll
  for (int s = 3; s >= 0; --s) {
    if (s >= nu) continue;
    strip_sweep<FULL, NPT>(C, x, r, v, t, w[s]);
    const int q = v;
    v = t;
    t = q;
  }
}

// node coordinates
template <int D> __device__ __forceinline__ void col_coords(const GridDesc &g, unsigned id, int v[3]) {
  const unsigned t = div_np(g, id), t2 = D == 2 ? 0u : div_np(g, t);
  v[0] = (int)(id - t * (unsigned)g.np);
  v[1] = D == 2 ? (int)t : (int)(t - t2 * (unsigned)g.np);
  v[2] = (int)t2;
}

// rc = P^T rf (see k_restrict)
template <int D>
__device__ __forceinline__ void col_restrict(const ColLevel &lf, const ColLevel &lc, int rf_, int zero_dirichlet) {
  const float *rf = col_sm + rf_;
  float *rc = col_sm + lc.offr;
  const GridDesc g = lc.g;
  const int n = lc.n, N = g.N, npf = lf.np;
  for (int I = threadIdx.x; I < n; I += blockDim.x) {
    int J[3];
    col_coords<D>(g, I, J);
    float out = 0.f;
    if (!(zero_dirichlet && (J[D - 1] == 0 || J[D - 1] == N))) {
      const int f0 = 2 * (J[0] + npf * (J[1] + (D == 3 ? npf * J[2] : 0)));
      out = rf[f0];
#pragma unroll
      for (int b = 1; b < (1 << D); ++b) {
        bool fw = true, bw = true;
#pragma unroll
        for (int a = 0; a < D; ++a)
          if ((b >> a) & 1) {
            fw = fw && (J[a] < N);
            bw = bw && (J[a] > 0);
          }
        const int o = col_off<D, true>(npf, b - 1);
        if (fw) out = fmadd(0.5f, rf[f0 + o], out);
        if (bw) out = fmadd(0.5f, rf[f0 - o], out);
      }
    }
    rc[I] = out;
  }
  __syncthreads();
}

// ef += P ec (see k_prolong_add)
template <int D>
__device__ __forceinline__ void col_prolong(const ColLevel &lf, const ColLevel &lc, int ef_) {
  const float *ec = col_sm + lc.offa;
  float *ef = col_sm + ef_;
  const GridDesc g = lf.g;
  const int n = lf.n, npc = lc.np;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int v[3];
    col_coords<D>(g, i, v);
    const int b = (v[0] & 1) | ((v[1] & 1) << 1) | ((v[2] & 1) << 2);
    const int ic = (v[0] >> 1) + npc * ((v[1] >> 1) + npc * (v[2] >> 1));
    float val = ec[ic];
    if (b) val = mulr(0.5f, addr(val, ec[ic + col_off<D, true>(npc, b - 1)]));
    ef[i] = addr(ef[i], val);
  }
  __syncthreads();
}

// E = inv R with the dense inverse of the coarsest level (symmetric, nc x nc).  The sums keep
// k_coarse_apply's order: eight shares of the columns (k = share, share + 8, ...), added in
// order.  A warp takes 32 rows of one share at a time.
//   HELD: the lower triangle (row i at i (i + 1) / 2) lies in shared memory: below the
//     diagonal block the 32 lanes read words at triangular-number distances (which all differ
//     in their bank), above it consecutive words;
//   else the matrix is read from L2, CO_RUN loads in flight per warp (17^2 nodes, two such runs
//     per share and one more load: 334 KB in 9,700 clocks; with the loads under conditions,
//     which serialised them, 30,000).
// rp: R in share order ([share][q], k = share + 8 q), so that four values are one load.
constexpr int CO_RUN = 18;
template <bool HELD> __device__ __noinline__ void col_coarse(const float *inv, int tri, const ColLevel &l, int offs) {
  const int nc = l.n, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int nch = (nc + 31) / 32, qp = 4 * nch;  // q < qp covers nc
  float *rp = col_sm + offs, *red = rp + 8 * qp;
  for (int t = threadIdx.x; t < 8 * qp; t += blockDim.x) {
    const int k = t / qp + 8 * (t % qp);
    rp[t] = k < nc ? col_sm[l.offr + k] : 0.f;
  }
  __syncthreads();
  for (int item = w; item < 8 * nch; item += nw) {
    const int ch = item >> 3, share = item & 7, i = min(ch * 32 + lane, nc - 1);
    const float *rs = rp + share * qp;
    const int qn = (nc - share + 7) / 8;  // terms of this share
    float acc = 0.f;
    if (HELD) {
      const float *row = col_sm + tri + i * (i + 1) / 2 + share;
      auto four = [&](int q, auto &&at) {  // q .. q + 3, the last of them checked
        const float4 r4 = *reinterpret_cast<const float4 *>(rs + q);
        const float r[4] = {r4.x, r4.y, r4.z, r4.w};
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = q + j < qn ? at(q + j) : 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (q + j < qn) acc = fmadd(v[j], r[j], acc);
      };
#pragma unroll 4
      for (int q = 0; q < 4 * ch; q += 4) {  // columns below this block of rows
        const float4 r4 = *reinterpret_cast<const float4 *>(rs + q);
        const float v0 = row[8 * q], v1 = row[8 * q + 8], v2 = row[8 * q + 16], v3 = row[8 * q + 24];
        acc = fmadd(v0, r4.x, acc);
        acc = fmadd(v1, r4.y, acc);
        acc = fmadd(v2, r4.z, acc);
        acc = fmadd(v3, r4.w, acc);
      }
      four(4 * ch, [&](int q) {
        const int k = share + 8 * q;
        return k <= i ? row[8 * q] : col_sm[tri + k * (k + 1) / 2 + i];
      });
#pragma unroll 2
      for (int q = 4 * ch + 4; q < qn; q += 4)
        four(q, [&](int qq) {
          const int k = share + 8 * qq;
          return col_sm[tri + k * (k + 1) / 2 + i];
        });
    } else {
      // runs of unconditional loads, all in flight before the first is used
      const float *p = inv + share * nc + i;
      int q = 0;
      for (; q + CO_RUN <= qn; q += CO_RUN) {
        float v[CO_RUN];
#pragma unroll
        for (int j = 0; j < CO_RUN; ++j) v[j] = __ldg(p + (q + j) * 8 * nc);
#pragma unroll
        for (int j = 0; j < CO_RUN; ++j) acc = fmadd(v[j], rs[q + j], acc);
      }
      for (; q < qn; ++q) acc = fmadd(__ldg(p + q * 8 * nc), rs[q], acc);
    }
    red[item * 32 + lane] = acc;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    const float *r = red + (i >> 5) * 256 + (i & 31);
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) s = addr(s, r[32 * q]);
    col_sm[l.offa + i] = s;
  }
  __syncthreads();
}

// starts the asynchronous copy of the coarse inverse's triangle to shared memory
__device__ __forceinline__ void col_copy_tri(const ColArgs &a) {
  for (int i = 4 * threadIdx.x; i < a.tn; i += 4 * blockDim.x) {
    const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(col_sm + a.offt + i));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(a.tri + i) : "memory");
  }
}

// the two legs of a level, with the least number of nodes per thread that covers it
template <int D, bool FULL, bool UP> __device__ __forceinline__ void col_leg(const ColLevel &l) {
  auto go = [&](auto k) {
    constexpr int N = decltype(k)::value;
    if constexpr (D == 2) {
      if (UP) strip_up<FULL, N>(l);
      else strip_down<FULL, N>(l);
    } else {
      if (UP) col_up<D, FULL, N>(l);
      else col_down<D, FULL, N>(l);
    }
  };
  switch (l.npt) {
    case 1: go(std::integral_constant<int, 1>{}); break;
    case 2: go(std::integral_constant<int, 2>{}); break;
    case 3: go(std::integral_constant<int, 3>{}); break;
    case 4: go(std::integral_constant<int, 4>{}); break;
    case 5: go(std::integral_constant<int, 5>{}); break;
    default: go(std::integral_constant<int, COL_NPT>{});
  }
}

// The V-cycle on levels l0 .. L-1 in shared memory: right-hand side in R of level l0, the
// correction in its A.
template <int D, bool FULL> __device__ __forceinline__ void col_vcycle(const ColArgs &a) {
  for (int l = a.l0; l + 1 < a.L; ++l) {
    col_leg<D, FULL, false>(a.lv[l]);
    col_restrict<D>(a.lv[l], a.lv[l + 1], (a.lv[l].nu & 1) ? a.lv[l].offa : a.lv[l].offb, a.zero_dirichlet);
  }
  if (a.tn) {
    asm volatile("cp.async.wait_all;" ::: "memory");  // visible after the barrier in col_coarse
    col_coarse<true>(nullptr, a.offt, a.lv[a.L - 1], a.offc);
  } else {
    col_coarse<false>(a.inv, 0, a.lv[a.L - 1], a.offc);
  }
  for (int l = a.L - 2; l >= a.l0; --l) {
    col_prolong<D>(a.lv[l], a.lv[l + 1], (a.lv[l].nu & 1) ? a.lv[l].offb : a.lv[l].offa);
    col_leg<D, FULL, true>(a.lv[l]);
  }
}

// zeros everywhere but in the coarse inverse's place, whose copy is started
__device__ __forceinline__ void col_begin(const ColArgs &a) {
  if (a.tn) col_copy_tri(a);
  for (int i = threadIdx.x; i < a.nclear; i += blockDim.x) col_sm[i] = 0.f;
  __syncthreads();
}

// the arguments in shared memory: the out-of-line legs read their level's description by
// address, which from the parameter space is a trip to L2 for every field's first use
__device__ __forceinline__ void col_args_to_smem(const ColArgs &from, ColArgs &to) {
  static_assert(sizeof(ColArgs) % 4 == 0, "copied by words");
  for (int i = threadIdx.x; i < (int)(sizeof(ColArgs) / 4); i += blockDim.x)
    reinterpret_cast<int *>(&to)[i] = reinterpret_cast<const int *>(&from)[i];
  __syncthreads();
}

template <int D, bool FULL>
__global__ void __launch_bounds__(col_nt<D>()) k_vtail(const __grid_constant__ ColArgs args) {
  __shared__ __align__(16) unsigned char args_raw[sizeof(ColArgs)];
  ColArgs &a = *reinterpret_cast<ColArgs *>(args_raw);
  col_args_to_smem(args, a);
  const int col = blockIdx.x;
  col_begin(a);
  const long base = (long)(col / a.vw) * a.gs + col % a.vw;
  const ColLevel &l = a.lv[a.l0];
  float *R = col_sm + l.offr;
  for (int i = threadIdx.x; i < l.n; i += blockDim.x) R[i] = a.r[base + (long)i * a.vw];
  __syncthreads();
  col_vcycle<D, FULL>(a);
  const float *A = col_sm + l.offa;
  for (int i = threadIdx.x; i < l.n; i += blockDim.x) a.x[base + (long)i * a.vw] = A[i];
}

// Sums over the CTA.  The FP32 part of a sum is always over 32 neighbouring nodes (a warp of
// the multi-kernel PCG's partials, lane order and tree the same); those sums go to shared
// memory and one warp adds them error-free in pairs of floats (two_sum, about 48 bits), and
// one thread turns the total into the scalars that every thread then reads (fin, which
// writes shared memory).  FP64 instructions issue at 1/64 of the FP32 rate and each takes
// tens of clocks: the same sums and the quotient in FP64 took 3 us per product.
__device__ __forceinline__ float col_warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;  // lane 0
}

template <class F> __device__ __forceinline__ void col_total(const float *seg, int m, F &&fin) {
  __syncthreads();
  if (threadIdx.x < 32) {
    float s = 0.f, c = 0.f;
    for (int i = threadIdx.x; i < m; i += 32) {
      const dfl t = two_sum(s, seg[i]);
      s = t.hi;
      c = addr(c, t.lo);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const dfl t = two_sum(s, __shfl_xor_sync(0xffffffffu, s, o));
      c = addr(addr(c, __shfl_xor_sync(0xffffffffu, c, o)), t.lo);
      s = t.hi;
    }
    if (threadIdx.x == 0) fin(two_sum(s, c));
  }
  __syncthreads();
}

// a / b of pairs, rounded to a float (the quotient of the leading floats and one correction)
__device__ __forceinline__ float df_ratio(dfl a, dfl b) {
  const float q = __fdiv_rn(a.hi, b.hi);
  const float r = addr(fmadd(-q, b.hi, a.hi), fmadd(-q, b.lo, a.lo));
  return addr(q, __fdiv_rn(r, b.hi));
}

// <a, b> with FP32 sums over 32-node segments of the grid's rows (as k_st's dots)
template <class F>
__device__ __forceinline__ void col_row_dot(int np, int rows, const float *a, const float *b, float *seg, F &&fin) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int m = 0;
  for (int x0 = 0; x0 < np; x0 += 32, m += rows) {
    const bool in = x0 + lane < np;
#pragma unroll 4
    for (int row = w; row < rows; row += nw) {
      const int id = row * np + x0 + lane;
      const float v = col_warp_sum(in ? mulr(a[id], b[id]) : 0.f);
      if (lane == 0) seg[m + row] = v;
    }
  }
  col_total(seg, m, fin);
}

// the scalars of a column's PCG, in shared memory
struct ColScal {
  dfl rz;
  double stop;  // |r|^2 at which the column has converged
  float alpha, beta;
  int active;
};

// PCG of one column from x = 0: right-hand side a.r, solution a.x; the steps and stopping
// test of pcg_body.  a.jacobi: diagonal scaling as the preconditioner (the mass matrix).
template <int D, bool FULL, int NPT>
__device__ __forceinline__ void col_pcg(const ColArgs &a, int col, ColScal &sc) {
  const ColLevel &l = a.lv[0];
  const int n = l.n, np = l.np, rows = D == 2 ? np : np * np, vw = a.vw;
  const float *__restrict__ src = a.r + (long)(col / vw) * a.gs + col % vw;
  float *__restrict__ dst = a.x + (long)(col / vw) * a.gs + col % vw;
  float *R = col_sm + l.offr, *Z = col_sm + l.offa, *X = col_sm + a.offx, *P = col_sm + a.offp,
        *seg = col_sm + a.offs;
  float *Q = Z;  // z is not needed once p has it
  const bool jacobi = a.jacobi, dense = a.L == 1;
  const int maxit = a.maxit;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float part[NPT];
  auto flat_dot = [&](auto &&fin) {  // of the threads' part, 32 consecutive nodes per segment
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const float v = col_warp_sum(part[k]);
      if (lane == 0) seg[k * nw + w] = v;
    }
    col_total(seg, NPT * nw, fin);
  };
#pragma unroll
  for (int k = 0; k < NPT; ++k) part[k] = 0.f;
  col_nodes<D, NPT>(n, [&](int k, int id) {
    const float r = src[(long)id * vw];
    R[id] = r;
    part[k] = mulr(r, r);
  });
  flat_dot([&](dfl b) {
    const double bb = df2d(b);
    sc.rz = dfl{0.f, 0.f};
    sc.stop = (a.tol2col ? a.tol2col[col] : a.tol2) * bb;
    sc.active = bb > 0.0 && (a.open == nullptr || a.open[col] != 0.0);
  });
  int it = 0;
  for (; sc.active && it < maxit; ++it) {
    auto set_beta = [&](dfl rz) {
      sc.beta = it > 0 && sc.rz.hi != 0.f ? df_ratio(rz, sc.rz) : 0.f;
      sc.rz = rz;
    };
    if (jacobi || dense) {
      if (!jacobi) col_vcycle<D, FULL>(a);  // the coarse solve alone
      col_nodes<D, NPT>(n, [&](int k, int id) {
        const float r = R[id], z = jacobi ? mulr(__ldg(l.invdiag + id), r) : Z[id];
        Z[id] = z;
        part[k] = mulr(r, z);
      });
      flat_dot(set_beta);
    } else {
      col_vcycle<D, FULL>(a);
      col_row_dot(np, rows, R, Z, seg, set_beta);
    }
    const float beta = sc.beta;
    col_nodes<D, NPT>(n, [&](int, int id) { P[id] = fmadd(beta, P[id], Z[id]); });
    __syncthreads();
    {  // q = S p (one application: the coefficients are not worth keeping)
      ColCoef<D, FULL, 16> C(l);
      col_set<D, NPT>(n, l.offa, [&](int k, int id) { return C.apply(k, id, a.offp); });
    }
    col_row_dot(np, rows, P, Q, seg, [&](dfl pq) { sc.alpha = pq.hi > 0.f ? df_ratio(sc.rz, pq) : 0.f; });
    const float alpha = sc.alpha;
    col_nodes<D, NPT>(n, [&](int k, int id) {
      X[id] = fmadd(alpha, P[id], X[id]);
      const float r = fmadd(-alpha, Q[id], R[id]);
      R[id] = r;
      part[k] = mulr(r, r);
    });
    flat_dot([&](dfl rr) { sc.active = df2d(rr) > sc.stop; });
  }
  // no copy outlives the CTA: a column without an iteration has not waited for the triangle yet
  asm volatile("cp.async.wait_all;" ::: "memory");
  col_nodes<D, NPT>(n, [&](int, int id) { dst[(long)id * vw] = X[id]; });
  if (threadIdx.x == 0) atomicMax(a.iter, it);
}

template <int D, bool FULL>
__global__ void __launch_bounds__(col_nt<D>()) k_colpcg(const __grid_constant__ ColArgs args) {
  __shared__ __align__(16) unsigned char args_raw[sizeof(ColArgs)];
  ColArgs &a = *reinterpret_cast<ColArgs *>(args_raw);
  col_args_to_smem(args, a);
  __shared__ ColScal sc;
  const int col = blockIdx.x;
  if (col >= a.s) {  // the empty columns of the last group
    const long base = (long)(col / a.vw) * a.gs + col % a.vw;
    for (int i = threadIdx.x; i < a.lv[0].n; i += blockDim.x) a.x[base + (long)i * a.vw] = 0.f;
    return;
  }
  col_begin(a);
  switch ((a.lv[0].n + col_nt<D>() - 1) / col_nt<D>()) {
    case 1: col_pcg<D, FULL, 1>(a, col, sc); break;
    case 2: col_pcg<D, FULL, 2>(a, col, sc); break;
    case 3: col_pcg<D, FULL, 3>(a, col, sc); break;
    case 4: col_pcg<D, FULL, 4>(a, col, sc); break;
    case 5: col_pcg<D, FULL, 5>(a, col, sc); break;
    default: col_pcg<D, FULL, COL_NPT>(a, col, sc);
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// shared-memory layout of levels l0 .. L-1 (and x, p, segment sums of a PCG, the coarse
// solve's scratch, and the coarse inverse's triangle for a PCG where it fits: a V-cycle alone
// would have to fetch it for one use); false if the levels do not fit
template <int D> static bool col_layout(ColArgs &a, bool pcg) {
  constexpr long CAP = COL_SMEM / (long)sizeof(float);
  long off = 0;
  auto take = [&](long n, long pad) {  // every vector starts on a 16-byte boundary
    off += (pad + 3) / 4 * 4;
    const long o = off;
    off = (off + n + pad + 3) / 4 * 4;
    return (int)o;
  };
  for (int l = a.l0; l < a.L; ++l) {
    ColLevel &v = a.lv[l];
    v.offr = take(v.n, v.pad);
    v.offa = take(v.n, v.pad);
    v.offb = l + 1 < a.L ? take(v.n, v.pad) : 0;
    for (v.npt = 1; v.npt < COL_NPT + 1; ++v.npt)
      if (D == 2 ? v.np * ((v.np + v.npt - 1) / v.npt) <= col_nt<D>() : v.n <= v.npt * col_nt<D>()) break;
    if (l + 1 < a.L && v.npt > COL_NPT) return false;
  }
  if (a.lv[a.l0].n > COL_NPT * col_nt<D>()) return false;
  if (pcg) {
    const ColLevel &v = a.lv[0];
    a.offx = take(v.n, 0);
    a.offp = take(v.n, v.pad);
    // segment sums of the dots: 32-node row segments, or the threads' nodes by warps
    a.offs = take(std::max((v.n / v.np) * ((v.np + 31) / 32), COL_NPT * col_nt<D>() / 32), 0);
  }
  const long nc = a.lv[a.L - 1].n, nch = (nc + 31) / 32;
  if (!a.jacobi) a.offc = take(8 * 4 * nch + 8 * nch * 32, 0);
  a.nclear = (int)off;
  a.tn = 0;
  const long tn = (nc * (nc + 1) / 2 + 3) / 4 * 4;
  if (!a.jacobi && pcg && a.tri && off + tn <= CAP) {
    a.tn = (int)tn;
    a.offt = take(tn, 0);
  }
  a.nfloats = (int)off;
  return off <= CAP;
}

static void col_launch(void (*k)(const ColArgs), const ColArgs &a, int dim, int cols, cudaStream_t st) {
  // the opt-in shared-memory size, once per kernel and device (setting it twice is harmless)
  static std::atomic<unsigned long long> done[8];
  static void (*const ks[8])(const ColArgs) = {k_vtail<2, false>, k_vtail<2, true>, k_vtail<3, false>, k_vtail<3, true>,
                                               k_colpcg<2, false>, k_colpcg<2, true>, k_colpcg<3, false>,
                                               k_colpcg<3, true>};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  for (int i = 0; i < 8; ++i) {
    if (ks[i] != k) continue;
    if (dev >= 64 || !(done[i].load(std::memory_order_acquire) & (1ull << dev))) {
      if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, COL_SMEM) != cudaSuccess) return;
      if (dev < 64) done[i].fetch_or(1ull << dev, std::memory_order_release);
    }
  }
  k<<<cols, dim == 2 ? col_nt<2>() : col_nt<3>(), sizeof(float) * a.nfloats, st>>>(a);
  count_launch();
}

bool col_fits(const ColArgs &in, bool pcg) {
  ColArgs a = in;
  return a.lv[a.l0].n <= COL_MAXN && (a.lv[a.l0].g.dim == 2 ? col_layout<2>(a, pcg) : col_layout<3>(a, pcg));
}

bool col_holds(const ColArgs &in) {
  ColArgs a = in;
  return a.lv[0].n <= COL_MAXN && (a.lv[0].g.dim == 2 ? col_layout<2>(a, true) : col_layout<3>(a, true)) && a.tn > 0;
}

void launch_vtail(ColArgs a, int dim, bool full, int cols, cudaStream_t st) {
  (void)(dim == 2 ? col_layout<2>(a, false) : col_layout<3>(a, false));
  col_launch(dim == 2 ? (full ? k_vtail<2, true> : k_vtail<2, false>)
                      : (full ? k_vtail<3, true> : k_vtail<3, false>),
             a, dim, cols, st);
}

void launch_colpcg(ColArgs a, int dim, bool full, int cols, cudaStream_t st) {
  (void)(dim == 2 ? col_layout<2>(a, true) : col_layout<3>(a, true));
  col_launch(dim == 2 ? (full ? k_colpcg<2, true> : k_colpcg<2, false>)
                      : (full ? k_colpcg<3, true> : k_colpcg<3, false>),
             a, dim, cols, st);
}

}  // namespace hp
