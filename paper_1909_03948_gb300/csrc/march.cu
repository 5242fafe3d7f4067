// march.cu -- 3D stencils over all Kuhn edges (15 points: the prior A and the mass M) on
// grouped FP32 blocks, marching through z.
//
// A CTA takes an xy tile of MA_X x MA_Y nodes (the last tile in a direction also takes the
// last node) of one group of four columns and marches through a segment of planes; a thread
// owns one (x, y).  Planes of x arrive in a ring of four shared-memory slots by 16-byte
// asynchronous copies (zeros outside the grid), two planes ahead of their use.  Of the 15
// points of a node three lie above it, six around it in its plane and its diagonals, three
// below: a thread reads each plane's forward neighbours (+x, +y, +x+y) once, when the plane
// is the one above, and its backward neighbours once, when the plane is its own, and carries
// both in registers to the step that needs them again.  That is 7 shared-memory loads per node
// where the row kernel has 15 global ones.
// A and M have constant coefficients, so away from the first and last two planes a node's
// coefficients do not depend on z: a thread keeps its 16 in registers for the segment and
// reads them again at those planes only.
//
// Bound: half its time is shared-memory and issue slots (41 wavefronts and about 150
// instructions per warp and plane), the rest the barrier per plane at 20 warps per SM: 65^3 nodes
// with 120 columns take 99 us for the matvec of 264 MB (the row kernel 170 us).  A ring of six
// planes gained 4 us, loading b a plane ahead or unrolling the march twice cost registers and
// 10 to 30 %.  The operations per node are the row kernel's in its order; the
// inner-product partial sums are grouped by tile.
#include <algorithm>

#include "internal.h"

namespace hp {

constexpr int MA_X = 32, MA_Y = 8, MA_NT = 320;       // a last tile has up to 33 x 9 nodes
constexpr int MA_BX = MA_X + 3, MA_BY = MA_Y + 3;     // its box with the halo
constexpr int MA_SLOTS = 4, MA_AHEAD = MA_SLOTS - 2;  // planes in flight beyond the current one

struct F4 {
  float v[4];
  __device__ __forceinline__ static F4 ld(const float4 *p) {
    const float4 t = *p;
    return {{t.x, t.y, t.z, t.w}};
  }
  __device__ __forceinline__ void st(float4 *p) const { *p = make_float4(v[0], v[1], v[2], v[3]); }
};

__device__ __forceinline__ void f4_axpy(F4 &s, float a, const F4 &x) {
#pragma unroll
  for (int q = 0; q < 4; ++q) s.v[q] = fmadd(a, x.v[q], s.v[q]);
}

template <int MODE>
__global__ void __launch_bounds__(MA_NT, 2) k_march_full(const __grid_constant__ MarchArgs a) {
  pdl_enter();
  constexpr bool HAS_B = MODE == MA_RESID || MODE == MA_JACOBI || MODE == MA_JACOBI_DOT || MODE == MA_CHEB;
  constexpr bool DOT = MODE == MA_APPLY_DOT || MODE == MA_JACOBI_DOT;
  __shared__ __align__(16) float4 ring[MA_SLOTS][MA_BX * MA_BY];
  const int np = a.np, N = np - 1, plane = np * np, n = plane * np, t = threadIdx.x;
  int q = blockIdx.x;
  const int tx = q % a.ntx;
  q /= a.ntx;
  const int ty = q % a.nty, tz = q / a.nty;
  const int x0 = tx * MA_X, y0 = ty * MA_Y;
  const int wx = tx == a.ntx - 1 ? np - x0 : MA_X, hy = ty == a.nty - 1 ? np - y0 : MA_Y;
  const int zb = (int)((long)tz * np / a.nzs), ze = (int)((long)(tz + 1) * np / a.nzs);
  // MA_CHEB: iterate j lies in X when n - j is even and in Y otherwise; Y of the step is the
  // iterate before X's
  const bool odd = MODE == MA_CHEB && ((a.ctl->n - a.ctl->it) & 1);
  const float cw = MODE == MA_CHEB ? a.ctl->omega : 0.f;
  const bool first = MODE == MA_CHEB && a.ctl->it == 0;  // a plain step: no iterate before X's
  const float *X = (odd ? a.Y : a.X) + blockIdx.y * a.gx;
  float *Y = (odd ? const_cast<float *>(a.X) : a.Y) + blockIdx.y * a.gy;
  const int bw = wx + 2;
  const int ly = t / wx, lx = t - ly * wx;
  const bool mine = ly < hy;
  const int x = x0 + lx, y = y0 + ly, at = (ly + 1) * bw + lx + 1;
  // this thread's two nodes of the box: place in a slot, place in a plane, inside the grid
  int bi[2], bo[2];
  bool bin[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    bi[k] = t + k * MA_NT;
    const int by = bi[k] / bw, bx = bi[k] - by * bw, gx = x0 - 1 + bx, gy = y0 - 1 + by;
    bin[k] = gx >= 0 && gx < np && gy >= 0 && gy < np;
    bo[k] = bin[k] ? gx + np * gy : 0;
    if (by >= hy + 2) bi[k] = -1;
  }
  const uint32_t ring0 = static_cast<uint32_t>(__cvta_generic_to_shared(&ring[0][0]));
  auto issue = [&](int p) {  // plane p into its slot (p & 3)
    const bool inz = p >= 0 && p < np;
    const float *base = X + 4 * (long)(inz ? p : 0) * plane;
    const uint32_t slot = ring0 + (unsigned)(p & (MA_SLOTS - 1)) * (MA_BX * MA_BY * 16u);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (bi[k] >= 0) {
        const uint32_t dst = slot + 16u * bi[k];
        const float *src = base + 4 * bo[k];
        const int bytes = inz && bin[k] ? 16 : 0;  // 0: the 16 bytes are filled with zeros
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // couplings: cf[f] forward, cb[f] backward along the Kuhn edge with mask f + 1 (M_JAC2:
  // times omega / diag of the neighbour)
  float d = 0.f, iv = 0.f, cf[7], cb[7];
  const int xy = min(x, N) + np * min(y, N);
  auto coefficients = [&](int p) {
    const int id = xy + p * plane;
    d = __ldg(a.diag + id);
    iv = __ldg(a.invdiag + id);
    float nf[7], nb[7];
#pragma unroll
    for (int f = 0; f < 7; ++f) {
      const int b = f + 1, o = (b & 1) + ((b >> 1) & 1) * np + ((b >> 2) & 1) * plane;
      cf[f] = __ldg(a.c + (long)f * n + id);
      cb[f] = __ldg(a.c + (long)f * n + max(id - o, 0));
      if (MODE == MA_JAC2) {
        nf[f] = __ldg(a.invdiag + min(id + o, n - 1));
        nb[f] = __ldg(a.invdiag + max(id - o, 0));
      }
    }
#pragma unroll
    for (int f = 0; f < 7; ++f) {
      const int b = f + 1;
      // a coupling that leaves the grid is not there
      const bool fw = (!(b & 1) || x < N) && (!(b & 2) || y < N) && (!(b & 4) || p < N);
      const bool bk = (!(b & 1) || x > 0) && (!(b & 2) || y > 0) && (!(b & 4) || p > 0);
      if (MODE == MA_JAC2) {
        cf[f] = mulr(mulr(cf[f], a.omega), nf[f]);
        cb[f] = mulr(mulr(cb[f], a.omega), nb[f]);
      }
      if (!fw) cf[f] = 0.f;
      if (!bk) cb[f] = 0.f;
    }
  };
#pragma unroll
  for (int k = -1; k < MA_AHEAD; ++k) issue(zb + k);
  asm volatile("cp.async.wait_group %0;" ::"n"(MA_AHEAD - 1) : "memory");  // planes zb - 1 and zb
  __syncthreads();
  F4 cm, c0, F0[3], Bm[3];
  {
    const float4 *s = ring[(zb - 1) & (MA_SLOTS - 1)] + at, *s0 = ring[zb & (MA_SLOTS - 1)] + at;
    if (mine) {
      cm = F4::ld(s);
      Bm[0] = F4::ld(s - 1);
      Bm[1] = F4::ld(s - bw);
      Bm[2] = F4::ld(s - bw - 1);
      c0 = F4::ld(s0);
      F0[0] = F4::ld(s0 + 1);
      F0[1] = F4::ld(s0 + bw);
      F0[2] = F4::ld(s0 + bw + 1);
    }
  }
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  const float4 *bp = reinterpret_cast<const float4 *>(a.B + blockIdx.y * a.gb) + xy;
  for (int p = zb; p < ze; ++p) {
    // into the slot of plane p - 2, which every thread has left at the last barrier
    issue(p + MA_AHEAD);
    const long o4 = (long)xy + (long)p * plane;
    F4 bb, xo;
    if (HAS_B && mine) bb = F4::ld(bp + (long)p * plane);
    if (MODE == MA_CHEB && mine && !first) xo = F4::ld(reinterpret_cast<const float4 *>(Y) + o4);
    if (mine && (p == zb || p <= 2 || p >= N - 1)) coefficients(p);
    asm volatile("cp.async.wait_group %0;" ::"n"(MA_AHEAD - 1) : "memory");  // plane p + 1 is there
    __syncthreads();
    if (mine) {
      const float4 *s = ring[p & (MA_SLOTS - 1)] + at, *s1 = ring[(p + 1) & (MA_SLOTS - 1)] + at;
      const F4 cp = F4::ld(s1);
      F4 F1[3], B0[3];
      F1[0] = F4::ld(s1 + 1);
      F1[1] = F4::ld(s1 + bw);
      F1[2] = F4::ld(s1 + bw + 1);
      B0[0] = F4::ld(s - 1);
      B0[1] = F4::ld(s - bw);
      B0[2] = F4::ld(s - bw - 1);
      F4 e1, sx, out;
      if (MODE == MA_JAC2) {
        const float wi = mulr(a.omega, iv);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          e1.v[k] = mulr(wi, c0.v[k]);
          sx.v[k] = mulr(d, e1.v[k]);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) sx.v[k] = mulr(d, c0.v[k]);
      }
      f4_axpy(sx, cf[0], F0[0]);
      f4_axpy(sx, cb[0], B0[0]);
      f4_axpy(sx, cf[1], F0[1]);
      f4_axpy(sx, cb[1], B0[1]);
      f4_axpy(sx, cf[2], F0[2]);
      f4_axpy(sx, cb[2], B0[2]);
      f4_axpy(sx, cf[3], cp);
      f4_axpy(sx, cb[3], cm);
      f4_axpy(sx, cf[4], F1[0]);
      f4_axpy(sx, cb[4], Bm[0]);
      f4_axpy(sx, cf[5], F1[1]);
      f4_axpy(sx, cb[5], Bm[1]);
      f4_axpy(sx, cf[6], F1[2]);
      f4_axpy(sx, cb[6], Bm[2]);
      if (MODE == MA_JAC2) {
        const float wi2 = mulr(a.omega2, iv);
#pragma unroll
        for (int k = 0; k < 4; ++k) out.v[k] = fmadd(wi2, addr(c0.v[k], -sx.v[k]), e1.v[k]);
      } else if (HAS_B && MODE == MA_RESID) {
#pragma unroll
        for (int k = 0; k < 4; ++k) out.v[k] = addr(bb.v[k], -sx.v[k]);
      } else if (HAS_B) {
        const float wi = mulr(a.omega, iv);
#pragma unroll
        for (int k = 0; k < 4; ++k) out.v[k] = fmadd(wi, addr(bb.v[k], -sx.v[k]), c0.v[k]);
        if (MODE == MA_CHEB && !first) {
#pragma unroll
          for (int k = 0; k < 4; ++k) out.v[k] = fmadd(cw, addr(out.v[k], -xo.v[k]), xo.v[k]);
        }
      } else {
        out = sx;
      }
      if (DOT) {
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] = fmadd(HAS_B ? bb.v[k] : c0.v[k], out.v[k], acc[k]);
      }
      out.st(reinterpret_cast<float4 *>(Y) + o4);
      cm = c0;
      c0 = cp;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        F0[k] = F1[k];
        Bm[k] = B0[k];
      }
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");  // no copy outlives the CTA
  if (DOT) {  // warp sums in FP32, across warps in FP64
    __shared__ double sh[MA_NT / 32][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float u = acc[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) u += __shfl_down_sync(0xffffffffu, u, o);
      if ((t & 31) == 0) sh[t >> 5][k] = (double)u;
    }
    __syncthreads();
    if (t < 4 && blockIdx.y * 4 + t < (unsigned)a.s) {
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < MA_NT / 32; ++w) s += sh[w][t];
      a.part[(blockIdx.y * 4l + t) * gridDim.x + blockIdx.x] = s;
    }
  }
}

static int ntx_of(const GridDesc &g) { return std::max(1, (g.np - 1 + MA_X - 1) / MA_X); }
static int nty_of(const GridDesc &g) { return std::max(1, (g.np - 1 + MA_Y - 1) / MA_Y); }
static_assert(MA_X * MA_Y == MARCH_TILE, "the fill of the tiles");
int march_tiles(const GridDesc &g) { return ntx_of(g) * nty_of(g); }

// CTAs per group: xy tiles times z segments -- of about 16 planes, or 8 while that leaves the
// GPU's two CTAs per SM with fewer than two rounds
static int march_segs(const GridDesc &g, int ng, int tiles) {
  const int n16 = std::max(1, g.np / 16), n8 = std::max(1, g.np / 8);
  return (long)tiles * n16 * ng >= 4 * NSM ? n16 : n8;
}

int launch_march(MarchArgs a, const GridDesc &g, int mode, int s, cudaStream_t st) {
  const int ng = (s + 3) / 4;
  a.np = g.np;
  a.s = s;
  a.ntx = ntx_of(g);
  a.nty = nty_of(g);
  a.nzs = march_segs(g, ng, a.ntx * a.nty);
  const dim3 gr(a.ntx * a.nty * a.nzs, ng);
  switch (mode) {
    case MA_APPLY_DOT: pdl_launch(k_march_full<MA_APPLY_DOT>, gr, MA_NT, 0, st, a); break;
    case MA_RESID: pdl_launch(k_march_full<MA_RESID>, gr, MA_NT, 0, st, a); break;
    case MA_JACOBI: pdl_launch(k_march_full<MA_JACOBI>, gr, MA_NT, 0, st, a); break;
    case MA_JACOBI_DOT: pdl_launch(k_march_full<MA_JACOBI_DOT>, gr, MA_NT, 0, st, a); break;
    case MA_CHEB: pdl_launch(k_march_full<MA_CHEB>, gr, MA_NT, 0, st, a); break;
    default: pdl_launch(k_march_full<MA_JAC2>, gr, MA_NT, 0, st, a);
  }
  count_launch();
  return (int)gr.x;
}

}  // namespace hp
