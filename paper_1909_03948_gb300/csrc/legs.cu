// legs.cu -- the two legs of a 2D multigrid level as one kernel each (FP32).
//
//   k_leg_down  pre-smoothing of nu sweeps from zero, the residual and its restriction:
//               reads r, writes the smoothed iterate and the coarse right-hand side;
//   k_leg_up    prolongation of the coarse correction and nu post-smoothing sweeps (and, on
//               the finest level, the partial sums of <r, z>): reads the iterate, the coarse
//               correction and r, writes the level's correction.
// A CTA owns a tile of LEG_X x LEG_Y nodes of one column group and computes it from a region
// with a halo of one node per stencil applied after the load, so that its sweeps need barriers
// only; halo nodes are computed by several CTAs.  As separate kernels the same steps are four
// or five launches each: on the levels below the finest those cost 1.6 to 3 us apiece and move
// next to nothing, on the finest (257^2 nodes, 60 columns, L2-resident) every one of them
// reads and writes whole blocks through L2.
//
// A thread owns LEG_N vertically consecutive nodes of one column of the region; their values,
// right-hand sides and coefficients stay in its registers, and only the neighbours to the left
// and right (and the ends of the strip) come from shared memory.  That is what bounds the
// kernel: per node and sweep two 16-byte loads and one store (and two fifths for the ends)
// against nine through L1 in the row kernel.  Nodes outside the grid have zero coefficients
// and stay zero; at the region's edge a wrong neighbour (the next row's first node, or the
// zero padding) spoils one more layer of the halo with every sweep and never reaches the
// tile.  Every value, and every FP32 partial sum of <r, z>, is formed by the operations of the
// per-level kernels in their order, so both forms have the same bits.
#include <algorithm>
#include <atomic>

#include "internal.h"

namespace hp {

constexpr int LEG_X = 32, LEG_Y = 16;  // the last tile in a direction also takes the last node
static_assert(LEG_X * LEG_Y == LEG_TILE, "the fill of the tiles");
constexpr int LEG_N = 5;               // nodes per thread
constexpr int LEG_NT = 224;            // threads at most (three sweeps: 41 columns of 5 strips)

template <int VW> struct LegV;  // VW values of one node
template <> struct LegV<1> {
  float v[1];
  __device__ __forceinline__ static LegV ld(const float *p) { return {{*p}}; }
  __device__ __forceinline__ void st(float *p) const { *p = v[0]; }
};
template <> struct LegV<4> {
  float v[4];
  __device__ __forceinline__ static LegV ld(const float *p) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    return {{t.x, t.y, t.z, t.w}};
  }
  __device__ __forceinline__ void st(float *p) const {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};

template <int VW, bool FULL> struct LegStrip {
  using V = LegV<VW>;
  int W, at;            // region columns; place of the strip's first node in a region vector
  int gx, gy;           // its grid coordinates
  bool in[LEG_N];       // inside the grid
  // diagonal, its inverse, couplings to x + 1 and x - 1, to y + 1 (cy[k + 1]) and y - 1
  // (cy[k]), and (FULL) to (x + 1, y + 1) and (x - 1, y - 1)
  float d[LEG_N], iv[LEG_N], cx[LEG_N], cxm[LEG_N], cy[LEG_N + 1], cd[FULL ? LEG_N : 1], cdm[FULL ? LEG_N : 1];
  // clamped index of grid node (x, y): every load is issued unconditionally (a load under a
  // condition waits for the one before it) and what does not exist is cleared afterwards
  __device__ __forceinline__ static int node(const LegArgs &a, int x, int y) {
    return min(max(x, 0), a.np - 1) + a.np * min(max(y, 0), a.np - 1);
  }
  __device__ __forceinline__ void init(const LegArgs &a, int x0, int y0, int halo, int strip, int col) {
    const int np = a.np, n = np * np;
    W = a.W;
    at = strip * LEG_N * W + col;
    gx = x0 - halo + col;
    gy = y0 - halo + strip * LEG_N;
    const float *c = a.c;
#pragma unroll
    for (int k = 0; k < LEG_N; ++k) {
      const int id = node(a, gx, gy + k), il = node(a, gx - 1, gy + k);
      d[k] = __ldg(a.diag + id);
      iv[k] = __ldg(a.invdiag + id);
      cx[k] = __ldg(c + id);
      cxm[k] = __ldg(c + il);
      cy[k + 1] = __ldg(c + n + id);
      if constexpr (FULL) {
        cd[k] = __ldg(c + 2 * n + id);
        cdm[k] = __ldg(c + 2 * n + node(a, gx - 1, gy + k - 1));
      }
    }
    cy[0] = __ldg(c + n + node(a, gx, gy - 1));
    const bool inx = gx >= 0 && gx < np;
    if (!inx || gy <= 0) cy[0] = 0.f;
#pragma unroll
    for (int k = 0; k < LEG_N; ++k) {
      in[k] = inx && gy + k >= 0 && gy + k < np;
      if (!in[k]) d[k] = iv[k] = cx[k] = cy[k + 1] = 0.f;
      if (!in[k] || gx == 0) cxm[k] = 0.f;
      if constexpr (FULL) {
        if (!in[k]) cd[k] = 0.f;
        if (!in[k] || gx == 0 || gy + k == 0) cdm[k] = 0.f;
      }
    }
  }
  // strip values of the block at base (group's first value), zero outside the grid
  __device__ __forceinline__ void load(const LegArgs &a, const float *base, V x[LEG_N]) const {
#pragma unroll
    for (int k = 0; k < LEG_N; ++k) x[k] = V::ld(base + (long)node(a, gx, gy + k) * VW);
#pragma unroll
    for (int k = 0; k < LEG_N; ++k)
#pragma unroll
      for (int q = 0; q < VW; ++q) x[k].v[q] = in[k] ? x[k].v[q] : 0.f;
  }
  __device__ __forceinline__ void put(float *v, const V x[LEG_N]) const {
#pragma unroll
    for (int k = 0; k < LEG_N; ++k) x[k].st(v + (at + k * W) * VW);
  }
  // For each node k in turn: sx = c0(k) + the neighbours' weighted values of the vector at v,
  // whose own values are x; then x[k] = fin(k, x[k], sx) (the strip's neighbours see the old
  // values).
  template <class C0, class WR, class WL, class WU, class WD, class WE, class WF, class FIN>
  __device__ __forceinline__ void stencil(const float *v, V x[LEG_N], C0 &&c0, WR &&wr, WL &&wl, WU &&wu, WD &&wd,
                                          WE &&we, WF &&wf, FIN &&fin) const {
    const float *p = v + at * VW;
    V below = V::ld(p - W * VW), rk = V::ld(p + VW), lm;
    const V above = V::ld(p + LEG_N * W * VW);
    if constexpr (FULL) lm = V::ld(p - (W + 1) * VW);
#pragma unroll
    for (int k = 0; k < LEG_N; ++k) {
      const V l = V::ld(p + (k * W - 1) * VW);
      V rn;
      if (FULL || k + 1 < LEG_N) rn = V::ld(p + ((k + 1) * W + 1) * VW);
      V sx = c0(k);
      const float a0 = wr(k), a1 = wl(k), a2 = wu(k), a3 = wd(k);
#pragma unroll
      for (int q = 0; q < VW; ++q) {
        float t = sx.v[q];
        t = fmadd(a0, rk.v[q], t);
        t = fmadd(a1, l.v[q], t);
        t = fmadd(a2, k + 1 < LEG_N ? x[k + 1 < LEG_N ? k + 1 : 0].v[q] : above.v[q], t);
        t = fmadd(a3, below.v[q], t);
        if constexpr (FULL) {
          t = fmadd(we(k), rn.v[q], t);
          t = fmadd(wf(k), lm.v[q], t);
        }
        sx.v[q] = t;
      }
      below = x[k];
      x[k] = fin(k, x[k], sx);
      rk = rn;
      if constexpr (FULL) lm = l;
    }
  }
  template <class FIN> __device__ __forceinline__ void apply(const float *v, V x[LEG_N], FIN &&fin) const {
    stencil(
        v, x,
        [&](int k) {
          V t;
#pragma unroll
          for (int q = 0; q < VW; ++q) t.v[q] = mulr(d[k], x[k].v[q]);
          return t;
        },
        [&](int k) { return cx[k]; }, [&](int k) { return cxm[k]; }, [&](int k) { return cy[k + 1]; },
        [&](int k) { return cy[k]; }, [&](int k) { return cd[FULL ? k : 0]; }, [&](int k) { return cdm[FULL ? k : 0]; },
        fin);
  }
  // x <- x + w D^-1 (r - S x), from the vector at v into the vector at t
  __device__ __forceinline__ void sweep(const float *v, float *t, V x[LEG_N], const V r[LEG_N], float w) const {
    apply(v, x, [&](int k, const V &xk, const V &sx) {
      V o;
      const float wi = mulr(w, iv[k]);
#pragma unroll
      for (int q = 0; q < VW; ++q) o.v[q] = fmadd(wi, addr(r[k].v[q], -sx.v[q]), xk.v[q]);
      return o;
    });
    put(t, x);
  }
};

// zeros before and after a region vector (its first and last row's neighbours)
template <int VW> __device__ __forceinline__ void leg_pad(const LegArgs &a, float *v) {
  const int pad = (a.W + 1) * VW, len = a.W * a.strips * LEG_N * VW;
  for (int i = threadIdx.x; i < pad; i += blockDim.x) {
    v[i - pad] = 0.f;
    v[len + i] = 0.f;
  }
}

template <int VW, bool FULL>
__global__ void __launch_bounds__(LEG_NT, VW == 4 ? 2 : 3) k_leg_down(const __grid_constant__ LegArgs a) {
  using V = LegV<VW>;
  extern __shared__ __align__(16) float leg_sm[];
  const int np = a.np, halo = a.nu + 1;
  const int tx = blockIdx.x % a.ntx, ty = blockIdx.x / a.ntx, x0 = tx * LEG_X, y0 = ty * LEG_Y;
  const int xe = tx == a.ntx - 1 ? np : x0 + LEG_X, ye = ty == a.nty - 1 ? np : y0 + LEG_Y;  // tile's end
  const int t = threadIdx.x, strip = t / a.W, col = t - strip * a.W;
  const bool mine = strip < a.strips;
  const long grp = blockIdx.y;
  float *A = leg_sm + a.pad * VW, *B = A + a.vec * VW;
  LegStrip<VW, FULL> C;
  V r[LEG_N], x[LEG_N];
  leg_pad<VW>(a, A);
  leg_pad<VW>(a, B);
  const float w0 = a.w[0];
  float *v = A, *o = B;
  // The coefficients are older than the kernel before this one.  One column's CTAs load them
  // ahead of the wait; blocks run several rounds of CTAs, where all loads at once are better
  // (the uneven batch 25.2 -> 24.7 ms).
  if (VW > 1) pdl_enter();
  if (mine) C.init(a, x0, y0, halo, strip, col);
  if (VW == 1) pdl_enter();
  if (mine) C.load(a, a.r + grp * a.gs, r);
  if (a.nu >= 2) {
    // two sweeps from zero (k_st's M_JAC2): e1 = w1 D^-1 r, x = e1 + w2 D^-1 (r - S e1), the
    // neighbours entering as (c w1 / diag) r
    float ir[LEG_N + 2], il[LEG_N + 2];  // inverse diagonals of the columns x + 1, x - 1, rows -1 .. LEG_N
    float iu = 0.f, id = 0.f;
    if (mine) {
#pragma unroll
      for (int k = 0; k < LEG_N + 2; ++k) {
        ir[k] = __ldg(a.invdiag + C.node(a, C.gx + 1, C.gy + k - 1));
        il[k] = __ldg(a.invdiag + C.node(a, C.gx - 1, C.gy + k - 1));
      }
      iu = __ldg(a.invdiag + C.node(a, C.gx, C.gy + LEG_N));
      id = __ldg(a.invdiag + C.node(a, C.gx, C.gy - 1));
      C.put(B, r);
    }
    __syncthreads();
    if (mine) {
      const float w1 = a.w[1];
      auto wt = [&](float c, float i) { return mulr(mulr(c, w0), i); };
#pragma unroll
      for (int k = 0; k < LEG_N; ++k) x[k] = r[k];
      C.stencil(
          B, x,
          [&](int k) {
            V s;
            const float wi = mulr(w0, C.iv[k]);
#pragma unroll
            for (int q = 0; q < VW; ++q) s.v[q] = mulr(C.d[k], mulr(wi, r[k].v[q]));
            return s;
          },
          [&](int k) { return wt(C.cx[k], ir[k + 1]); }, [&](int k) { return wt(C.cxm[k], il[k + 1]); },
          [&](int k) { return wt(C.cy[k + 1], k + 1 < LEG_N ? C.iv[k + 1 < LEG_N ? k + 1 : 0] : iu); },
          [&](int k) { return wt(C.cy[k], k > 0 ? C.iv[k > 0 ? k - 1 : 0] : id); },
          [&](int k) { return wt(C.cd[FULL ? k : 0], ir[k + 2]); },
          [&](int k) { return wt(C.cdm[FULL ? k : 0], il[k]); },
          [&](int k, const V &rk, const V &sx) {
            V e;
            const float wi = mulr(w0, C.iv[k]), wi2 = mulr(w1, C.iv[k]);
#pragma unroll
            for (int q = 0; q < VW; ++q) e.v[q] = fmadd(wi2, addr(rk.v[q], -sx.v[q]), mulr(wi, rk.v[q]));
            return e;
          });
      C.put(A, x);
    }
    __syncthreads();
    for (int s = 2; s < a.nu; ++s) {
      if (mine) C.sweep(v, o, x, r, a.w[s]);
      __syncthreads();
      float *q = v;
      v = o;
      o = q;
    }
  } else {
    if (mine) {
#pragma unroll
      for (int k = 0; k < LEG_N; ++k) {
        const float wi = mulr(w0, C.iv[k]);
#pragma unroll
        for (int q = 0; q < VW; ++q) x[k].v[q] = mulr(wi, r[k].v[q]);
      }
      C.put(A, x);
    }
    __syncthreads();
  }
  // the tile's smoothed iterate, then the residual in place of it
  if (mine) {
    float *out = a.x + grp * a.gs;
    const bool inx = C.gx >= x0 && C.gx < xe;
#pragma unroll
    for (int k = 0; k < LEG_N; ++k) {
      const int y = C.gy + k;
      if (inx && y >= y0 && y < ye) x[k].st(out + (long)(C.gx + np * y) * VW);
    }
    C.apply(v, x, [&](int k, const V &, const V &sx) {
      V e;
#pragma unroll
      for (int q = 0; q < VW; ++q) e.v[q] = addr(r[k].v[q], -sx.v[q]);
      return e;
    });
    C.put(o, x);
  }
  __syncthreads();
  // restriction (see k_restrict) to the coarse nodes under the tile
  const int npc = a.npc, Nc = npc - 1, cx0 = x0 / 2, cy0 = y0 / 2, cw = (xe - x0 + 1) / 2, ch = (ye - y0 + 1) / 2;
  float *rc = a.rc + grp * a.gsc;
  for (int i = threadIdx.x; i < cw * ch; i += blockDim.x) {
    const int jy = i / cw, jx = i - jy * cw, Jx = cx0 + jx, Jy = cy0 + jy;
    V out;
#pragma unroll
    for (int q = 0; q < VW; ++q) out.v[q] = 0.f;
    if (!(a.zero_dirichlet && (Jy == 0 || Jy == Nc))) {
      const float *p = o + ((2 * jy + halo) * a.W + 2 * jx + halo) * VW;
      out = V::ld(p);
#pragma unroll
      for (int b = 1; b < 4; ++b) {
        const bool fw = (!(b & 1) || Jx < Nc) && (!(b & 2) || Jy < Nc);
        const bool bw = (!(b & 1) || Jx > 0) && (!(b & 2) || Jy > 0);
        const int off = ((b & 1) + ((b >> 1) & 1) * a.W) * VW;
        if (fw) {
          const V f = V::ld(p + off);
#pragma unroll
          for (int q = 0; q < VW; ++q) out.v[q] = fmadd(0.5f, f.v[q], out.v[q]);
        }
        if (bw) {
          const V f = V::ld(p - off);
#pragma unroll
          for (int q = 0; q < VW; ++q) out.v[q] = fmadd(0.5f, f.v[q], out.v[q]);
        }
      }
    }
    out.st(rc + (long)(Jx + npc * Jy) * VW);
  }
}

template <int VW, bool FULL, bool DOT>
__global__ void __launch_bounds__(LEG_NT, VW == 4 ? 2 : 3) k_leg_up(const __grid_constant__ LegArgs a) {
  using V = LegV<VW>;
  extern __shared__ __align__(16) float leg_sm[];
  const int np = a.np, npc = a.npc, halo = a.nu;
  const int tx = blockIdx.x % a.ntx, ty = blockIdx.x / a.ntx, x0 = tx * LEG_X, y0 = ty * LEG_Y;
  const int xe = tx == a.ntx - 1 ? np : x0 + LEG_X, ye = ty == a.nty - 1 ? np : y0 + LEG_Y;
  const int t = threadIdx.x, strip = t / a.W, col = t - strip * a.W;
  const bool mine = strip < a.strips;
  const long grp = blockIdx.y;
  float *v = leg_sm + a.pad * VW, *o = v + a.vec * VW;
  LegStrip<VW, FULL> C;
  V r[LEG_N], x[LEG_N];
  leg_pad<VW>(a, v);
  leg_pad<VW>(a, o);
  if (VW > 1) pdl_enter();  // as in k_leg_down
  if (mine) C.init(a, x0, y0, halo, strip, col);
  if (VW == 1) pdl_enter();
  if (mine) {
    C.load(a, a.xin + grp * a.gs, x);
    C.load(a, a.r + grp * a.gs, r);
    // x += P e_c (see k_prolong_add): e_c at the coarse node below, or the mean with its
    // neighbour along the odd directions
    const float *ec = a.ec + grp * a.gsc;
    V e0[LEG_N], e1[LEG_N];
    const int X = min(max(C.gx, 0), np - 1);
#pragma unroll
    for (int k = 0; k < LEG_N; ++k) {
      const int Y = min(max(C.gy + k, 0), np - 1), ic = (X >> 1) + npc * (Y >> 1);
      e0[k] = V::ld(ec + (long)ic * VW);
      e1[k] = V::ld(ec + (long)(ic + (X & 1) + (Y & 1) * npc) * VW);
    }
#pragma unroll
    for (int k = 0; k < LEG_N; ++k) {
      const bool mean = (X & 1) || ((C.gy + k) & 1);
#pragma unroll
      for (int q = 0; q < VW; ++q) {
        const float val = mean ? mulr(0.5f, addr(e0[k].v[q], e1[k].v[q])) : e0[k].v[q];
        x[k].v[q] = C.in[k] ? addr(x[k].v[q], val) : 0.f;
      }
    }
    C.put(v, x);
  }
  __syncthreads();
  for (int s = a.nu - 1; s >= 0; --s) {
    if (mine) C.sweep(v, o, x, r, a.w[s]);
    __syncthreads();
    float *q = v;
    v = o;
    o = q;
  }
  if (mine) {
    float *out = a.x + grp * a.gs;
    const bool inx = C.gx >= x0 && C.gx < xe;
#pragma unroll
    for (int k = 0; k < LEG_N; ++k) {
      const int y = C.gy + k;
      if (inx && y >= y0 && y < ye) x[k].st(out + (long)(C.gx + np * y) * VW);
      if (DOT) {
#pragma unroll
        for (int q = 0; q < VW; ++q) x[k].v[q] = mulr(r[k].v[q], x[k].v[q]);
      }
    }
    if (DOT) C.put(o, x);  // the products
  }
  if (DOT) {
    // FP32 sums over the 32 nodes of a row that a warp of the row kernel holds (the tiles are
    // aligned with them), everything above in FP64
    __shared__ double sh[LEG_NT / 32][VW];
    __syncthreads();
    const int lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
    double acc[VW];
#pragma unroll
    for (int q = 0; q < VW; ++q) acc[q] = 0.0;
    for (int row = w; row < ye - y0; row += nw) {
      const float *p = o + ((row + halo) * a.W + halo) * VW;
      V u;
#pragma unroll
      for (int q = 0; q < VW; ++q) u.v[q] = 0.f;
      if (x0 + lane < xe && lane < LEG_X) u = V::ld(p + lane * VW);
#pragma unroll
      for (int q = 0; q < VW; ++q) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) u.v[q] += __shfl_down_sync(0xffffffffu, u.v[q], d);
      }
      if (lane == 0) {
#pragma unroll
        for (int q = 0; q < VW; ++q) {
          acc[q] += (double)u.v[q];
          if (xe - x0 > LEG_X) acc[q] += (double)p[LEG_X * VW + q];  // the last column is a segment of its own
        }
      }
    }
    if (lane == 0) {
#pragma unroll
      for (int q = 0; q < VW; ++q) sh[w][q] = acc[q];
    }
    __syncthreads();
    if (t < VW && grp * VW + t < a.s) {
      double s = 0.0;
      for (int i = 0; i < nw; ++i) s += sh[i][t];
      a.part[(grp * VW + t) * gridDim.x + blockIdx.x] = s;
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int leg_tiles(const GridDesc &g) {
  const int ntx = std::max(1, (g.np - 1 + LEG_X - 1) / LEG_X), nty = std::max(1, (g.np - 1 + LEG_Y - 1) / LEG_Y);
  return ntx * nty;
}

void launch_leg(LegArgs a, const GridDesc &g, bool full, bool up, int vw, int s, cudaStream_t st) {
  const int halo = up ? a.nu : a.nu + 1;
  a.np = g.np;
  a.npc = g.N / 2 + 1;
  a.s = s;
  a.ntx = std::max(1, (g.np - 1 + LEG_X - 1) / LEG_X);
  a.nty = std::max(1, (g.np - 1 + LEG_Y - 1) / LEG_Y);
  a.W = LEG_X + 1 + 2 * halo;
  a.strips = (LEG_Y + 1 + 2 * halo + LEG_N - 1) / LEG_N;
  a.pad = (a.W + 1 + 3) / 4 * 4;
  a.vec = (a.W * a.strips * LEG_N + 2 * a.pad + 3) / 4 * 4;
  const int nt = (a.W * a.strips + 31) / 32 * 32;
  const size_t shm = sizeof(float) * (size_t)vw * 2 * a.vec;
  using K = void (*)(const LegArgs);
  const bool dot = a.part != nullptr;
  K k;
  if (vw == 4)
    k = full ? (up ? (dot ? (K)k_leg_up<4, true, true> : (K)k_leg_up<4, true, false>) : (K)k_leg_down<4, true>)
             : (up ? (dot ? (K)k_leg_up<4, false, true> : (K)k_leg_up<4, false, false>) : (K)k_leg_down<4, false>);
  else
    k = full ? (up ? (dot ? (K)k_leg_up<1, true, true> : (K)k_leg_up<1, true, false>) : (K)k_leg_down<1, true>)
             : (up ? (dot ? (K)k_leg_up<1, false, true> : (K)k_leg_up<1, false, false>) : (K)k_leg_down<1, false>);
  pdl_launch(k, dim3(a.ntx * a.nty, (s + vw - 1) / vw), nt, shm, st, a);
  count_launch();
}

}  // namespace hp
