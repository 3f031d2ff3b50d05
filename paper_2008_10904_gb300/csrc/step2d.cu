// Step form of the structured-grid marches (real state), and its 2-D kernels.
//
// For a linear time-invariant system one classical RK4 step with the forcing sampled at t_n,
// t_n + h/2 and t_n + h is exactly (B = h A)
//     u_{n+1} = u + B (u + B/2 (u + B/3 (u + B/4 u))) + g_n,
//     g_n = (h/6) [P1 f(t_n) + P2 f(t_n + h/2) + f(t_n + h)],
//     P1 = I + B + B^2/2 + B^3/4,   P2 = 4 I + 2 B + B^2/2.
// With f(t) = sum_j fhat_j e^{i w_j t}, g_n = sum_j c_j e^{i w_j t_n} with
//     c_j = (h/6) [(1 + 4 s_j + z_j) + (1 + 2 s_j) B + (1 + s_j)/2 B^2 + 1/4 B^3] fhat_j,
// s_j = e^{i w_j h/2}, z_j = s_j^2 (the dense kind's coefficients, dense_kernels.cu).  So the march
// needs the forcing at one time per step instead of three stage times (half of the synthesis, and
// one forcing pass per step instead of four), no stage reads a forcing, and the four stages keep no
// accumulator: w1 = u + h/4 A u, w2 = u + h/3 A w1, w3 = u + h/2 A w2, u' = u + h A w3 + g.
// The operator's coefficients are the ones the stage kernels use.  c_j costs three operator
// applications per march, a few passes over the coefficient block.
//
// Rows of the state, forcing and snapshot tiles and of the transformed coefficients are padded to a
// multiple of four cells (zeros), so that every grid takes the 16-byte loads and the pipelined
// contractions; `march_finish` drops the padding.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "rsv_ops.h"

namespace rsv {
namespace {

// ---------------------------------------------------------------------------
// Coefficient transform: three passes t <- a f + B t (complex a, real B on both parts)
// ---------------------------------------------------------------------------
template <typename R>
struct Grid3 {
  int nx, nxp, ny, nz;         // nz = 1 and one component in 2-D
  int64_t ncell, ncellp;       // cells of one component, without and with the row padding
  R i2dx, nx2, ny2, nz2;       // 1 / (2 dx), visc / dx^2, visc / dy^2, visc / dz^2
  const R *f0, *f1, *f2, *f3;  // ADR2D: U(y), r(y); ADV3D: U, dU/dx, dU/dy, dU/dz per cell
  int sponge_cells;
  R sponge_amp, sponge_inv;    // amplitude, 1 / sponge_cells
  R h;
};

template <typename R>
__device__ __forceinline__ R sponge2d(int i, int j, const Grid3<R>& g) {
  const int d = min(min(i, g.nx - 1 - i), min(j, g.ny - 1 - j));
  if (d >= g.sponge_cells) return R(0);
  const R t = R(g.sponge_cells - d) * g.sponge_inv;
  return g.sponge_amp * t * t;
}

template <typename R>
__device__ __forceinline__ cpx<R> ld_or0(const cpx<R>* p, bool ok) {
  return ok ? *p : mk<R>(0, 0);
}

// One pass for the frequencies j0 .. j0 + gridDim.y - 1 and the vectors gridDim.z of a 2-D block:
// out = scale (a_j f + B t), with a_j = (1, s_j, z_j) . coef.  f has the caller's layout (stride
// f_stride per frequency), t and out the padded one.
template <typename R, bool ADJ>
__global__ void __launch_bounds__(256) coef2d_kernel(Grid3<R> g, int j0, const cpx<R>* __restrict__ f, int64_t f_stride,
                                                     const cpx<R>* __restrict__ t, int64_t t_stride, bool t_is_f,
                                                     cpx<R>* __restrict__ out, int64_t o_stride,
                                                     const cpx<R>* __restrict__ tw, const int64_t* __restrict__ pj,
                                                     int sgn, int64_t m4, R c1, R cs, R cz, R bscale, R scale) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) % g.nxp, j = (blockIdx.x * blockDim.x + threadIdx.x) / g.nxp;
  if (j >= g.ny) return;
  const int w = blockIdx.y, v = blockIdx.z;
  cpx<R>* o = out + (int64_t)w * o_stride + (int64_t)v * g.ncellp + (int64_t)j * g.nxp + i;
  if (i >= g.nx) {
    *o = mk<R>(0, 0);
    return;
  }
  const cpx<R> s = tw[phase_index(sgn * pj[j0 + w], 1, m4)], z = tw[phase_index(sgn * pj[j0 + w], 2, m4)];
  const cpx<R> a = mk<R>(c1 + cs * s.re + cz * z.re, cs * s.im + cz * z.im);
  const cpx<R> fv = f[(int64_t)(j0 + w) * f_stride + (int64_t)v * g.ncell + (int64_t)j * g.nx + i];
  const int pitch = t_is_f ? g.nx : g.nxp;
  const cpx<R>* x = t_is_f ? f + (int64_t)(j0 + w) * f_stride + (int64_t)v * g.ncell
                           : t + (int64_t)w * t_stride + (int64_t)v * g.ncellp;
  x += (int64_t)j * pitch + i;
  const cpx<R> c = *x, we = ld_or0(x - 1, i > 0), ea = ld_or0(x + 1, i < g.nx - 1), so = ld_or0(x - pitch, j > 0),
               no = ld_or0(x + pitch, j < g.ny - 1);
  const R ux = (ADJ ? -g.f0[j] : g.f0[j]) * g.i2dx;
  const R cw = ux + g.nx2, ce = g.nx2 - ux;
  const R cc = R(-2) * (g.nx2 + g.ny2) + g.f1[j] - sponge2d<R>(i, j, g);
  const R hb = g.h * bscale;
  const R br = hb * (cw * we.re + ce * ea.re + g.ny2 * (so.re + no.re) + cc * c.re);
  const R bi = hb * (cw * we.im + ce * ea.im + g.ny2 * (so.im + no.im) + cc * c.im);
  const cpx<R> af = a * fv;
  *o = mk<R>(scale * (af.re + br), scale * (af.im + bi));
}

template <typename R, bool ADJ>
__global__ void __launch_bounds__(256) coef3d_kernel(Grid3<R> g, int j0, const cpx<R>* __restrict__ f, int64_t f_stride,
                                                     const cpx<R>* __restrict__ t, int64_t t_stride, bool t_is_f,
                                                     cpx<R>* __restrict__ out, int64_t o_stride,
                                                     const cpx<R>* __restrict__ tw, const int64_t* __restrict__ pj,
                                                     int sgn, int64_t m4, R c1, R cs, R cz, R bscale, R scale) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int i = (int)(e % g.nxp);
  const int64_t jk = e / g.nxp;
  const int j = (int)(jk % g.ny), kz = (int)(jk / g.ny);
  if (kz >= g.nz) return;
  const int w = blockIdx.y, v = blockIdx.z;
  cpx<R>* o = out + (int64_t)w * o_stride + (int64_t)v * 3 * g.ncellp + e;
  if (i >= g.nx) {
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c * g.ncellp] = mk<R>(0, 0);
    return;
  }
  const cpx<R> s = tw[phase_index(sgn * pj[j0 + w], 1, m4)], z = tw[phase_index(sgn * pj[j0 + w], 2, m4)];
  const cpx<R> a = mk<R>(c1 + cs * s.re + cz * z.re, cs * s.im + cz * z.im);
  const cpx<R>* fv = f + (int64_t)(j0 + w) * f_stride + (int64_t)v * 3 * g.ncell;
  const int64_t q = jk * g.nx + i;                       // cell in the fields and in f
  const int64_t pitch = t_is_f ? g.nx : g.nxp, plane = pitch * g.ny, cells = t_is_f ? g.ncell : g.ncellp;
  const cpx<R>* x = (t_is_f ? fv : t + (int64_t)w * t_stride + (int64_t)v * 3 * g.ncellp) + (t_is_f ? q : e);
  const R Uc = g.f0[q], Uw = i > 0 ? g.f0[q - 1] : R(0), Ue = i < g.nx - 1 ? g.f0[q + 1] : R(0);
  const R Ux = g.f1[q], Uy = g.f2[q], Uz = g.f3[q];
  const R cw = g.nx2 + g.i2dx * (ADJ ? -Uw : Uc), ce = g.nx2 - g.i2dx * (ADJ ? -Ue : Uc);
  const R cc = R(-2) * (g.nx2 + g.ny2 + g.nz2);
  cpx<R> xc[3], b[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const cpx<R>* p = x + c * cells;
    const cpx<R> we = ld_or0(p - 1, i > 0), ea = ld_or0(p + 1, i < g.nx - 1);
    const cpx<R> so = ld_or0(p - pitch, j > 0), no = ld_or0(p + pitch, j < g.ny - 1);
    const cpx<R> bo = ld_or0(p - plane, kz > 0), to = ld_or0(p + plane, kz < g.nz - 1);
    xc[c] = *p;
    b[c].re = cw * we.re + ce * ea.re + g.ny2 * (so.re + no.re) + g.nz2 * (bo.re + to.re) + cc * xc[c].re;
    b[c].im = cw * we.im + ce * ea.im + g.ny2 * (so.im + no.im) + g.nz2 * (bo.im + to.im) + cc * xc[c].im;
  }
  if (ADJ) {
    b[0] = b[0] - Ux * xc[0];
    b[1] = b[1] - Uy * xc[0];
    b[2] = b[2] - Uz * xc[0];
  } else {
    b[0] = b[0] - (Ux * xc[0] + Uy * xc[1] + Uz * xc[2]);
  }
  const R hb = g.h * bscale;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const cpx<R> af = a * fv[c * g.ncell + q];
    o[c * g.ncellp] = mk<R>(scale * (af.re + hb * b[c].re), scale * (af.im + hb * b[c].im));
  }
}

template <typename R>
Grid3<R> grid3_of(rsv_operator op) {
  Grid3<R> g;
  g.nx = op->nx;
  g.nxp = (op->nx + 3) / 4 * 4;
  g.ny = op->ny;
  g.nz = op->kind == RSV_OP_ADV3D ? op->nz : 1;
  g.ncell = (int64_t)g.nx * g.ny * g.nz;
  g.ncellp = (int64_t)g.nxp * g.ny * g.nz;
  // formed in R from the rounded spacings, as the stage kernels form them
  const R dx = (R)op->c_dx, dy = (R)op->c_dy, dz = op->kind == RSV_OP_ADV3D ? (R)op->c_dz : R(1), nu = (R)op->visc;
  g.i2dx = R(0.5) / dx;
  g.nx2 = nu * (R(1) / (dx * dx));
  g.ny2 = nu * (R(1) / (dy * dy));
  g.nz2 = nu * (R(1) / (dz * dz));
  g.f0 = (const R*)op->fld[0];
  g.f1 = (const R*)op->fld[1];
  g.f2 = (const R*)op->fld[2];
  g.f3 = (const R*)op->fld[3];
  g.sponge_cells = op->sponge_cells;
  g.sponge_amp = (R)op->sponge_amp;
  g.sponge_inv = op->sponge_cells > 0 ? R(1) / R(op->sponge_cells) : R(0);
  g.h = (R)op->h;
  return g;
}

// ---------------------------------------------------------------------------
// 2-D, FP32: one whole step per launch, streaming along y in registers.
//
// A warp owns a strip of 120 cells in x (lane l: four consecutive cells; lanes 0 and 31 are the halo
// of four cells, one per stage) and a run of rows, and walks up the rows: with row r of u just
// loaded it evaluates w1 on row r - 1, w2 on r - 2, w3 on r - 3 and u' on r - 4.  Rows live in
// registers (x neighbours across lanes by shuffles), so there is no barrier and no shared-memory
// traffic but the per-warp ring that stages u and g by 16-byte asynchronous copies.  A run starts
// four rows early and ends four late; what it computes there is not stored.  Rows outside the grid
// have zero coefficients, so they stay zero.  Issue slots bound it, not bytes: per row and warp 96
// arithmetic instructions of about 150.
// ---------------------------------------------------------------------------
constexpr int kStripCells = 120, kStreamWarps = 2, kRing = 8, kAhead = 6, kMaxRun = 128;

struct Stream2D {
  int nx, nxp, ny, kg;
  int strips, runs, run_rows;
  int64_t vstride;
  const float *U, *r;
  float i2dx, nx2, ny2, h, h2, h3, h4;   // h / m for the stages' factors
  int sponge_cells;
  float sponge_amp, sponge_inv;
  int adj;
};

__device__ __forceinline__ void cp16_zfill(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

struct F4 {
  float v[4];
};

// The rows of one warp.  WALL: the strip or the run reaches a wall or its sponge.
template <bool WALL>
__device__ __forceinline__ void stream2d_rows(const Stream2D& P, const float* __restrict__ u, const float* __restrict__ g,
                                              float* __restrict__ out, float* __restrict__ ysnap, float4 (*ring)[2][32],
                                              const float4* rowc, const float* rowt, int ya, int yb, int gx, int lane,
                                              int64_t base) {
  const bool in_x = gx >= 0 && gx < P.nxp;
  const bool owner = lane >= 1 && lane <= 30 && gx < P.nxp;
  const bool forced = g != nullptr;
  bool cell[4];
  float sx[4];   // sponge depth of the lane's columns (0: none)
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int i = gx + c;
    cell[c] = i >= 0 && i < P.nx;
    const int d = min(i, P.nx - 1 - i);
    sx[c] = cell[c] && d < P.sponge_cells ? (float)(P.sponge_cells - d) * P.sponge_inv : 0.f;
  }
  // row r of u (from ya - 4) and row r - 4 of g go to ring slot (r - ya + 4) mod kRing
  const int64_t off = base + (in_x ? gx : 0);
  const float* pu = u + off + (int64_t)(ya - 4) * P.nxp;
  const float* pg = (forced ? g : u) + off + (int64_t)(ya - 8) * P.nxp;
  const uint32_t slot0 = (uint32_t)__cvta_generic_to_shared(&ring[0][0][lane]);
  const int iters = yb - ya + 8;
  auto prefetch = [&](int i) {   // iteration i: row ya - 4 + i
    if (i < iters) {
      const uint32_t d = slot0 + (uint32_t)(i & (kRing - 1)) * (2 * 32 * 16);
      const int r = ya - 4 + i;
      const bool oku = in_x && r >= 0 && r < P.ny;
      cp16_zfill(d, oku ? pu : u, oku);
      if (forced && i >= 8) cp16_zfill(d + 32 * 16, in_x ? pg : u, in_x);
    }
    pu += P.nxp;
    pg += P.nxp;
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int q = 0; q < kAhead; ++q) prefetch(q);
  F4 ur[6], w1[3], w2[3], w3[3];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
#pragma unroll
    for (int q = 0; q < 6; ++q) ur[q].v[c] = 0.f;
#pragma unroll
    for (int q = 0; q < 3; ++q) w1[q].v[c] = w2[q].v[c] = w3[q].v[c] = 0.f;
  }
  // u0 + f A x on a row from the rows below, at and above it; e: the row's index in rowc
  auto stage = [&](const F4& xb, const F4& xc, const F4& xt, const F4& u0, int e, float f) -> F4 {
    const float4 rc = rowc[e];   // west, east, diagonal, north / south
    const float left = __shfl_up_sync(0xffffffffu, xc.v[3], 1), right = __shfl_down_sync(0xffffffffu, xc.v[0], 1);
    F4 o;
    const float ty = WALL ? rowt[e] : 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float cc = rc.z;
      if (WALL) {
        const float t = fmaxf(sx[c], ty);
        cc = rc.z - P.sponge_amp * t * t;
      }
      float a = rc.w * (xb.v[c] + xt.v[c]);
      a = fmaf(rc.x, c == 0 ? left : xc.v[c - 1], a);
      a = fmaf(rc.y, c == 3 ? right : xc.v[c + 1], a);
      a = fmaf(cc, xc.v[c], a);
      o.v[c] = fmaf(f, a, u0.v[c]);
      if (WALL) o.v[c] = cell[c] ? o.v[c] : 0.f;
    }
    return o;
  };
  float* po = out + base + (int64_t)ya * P.nxp + gx;
  float* py = ysnap + base + (int64_t)ya * P.nxp + gx;   // used only when ysnap is given
  for (int i0 = 0; i0 < iters; i0 += 6) {
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int i = i0 + q;
      if (i >= iters) break;
      asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
      const float4(&slot)[2][32] = ring[i & (kRing - 1)];
      const float4 nu4 = slot[0][lane];
      ur[q].v[0] = nu4.x;
      ur[q].v[1] = nu4.y;
      ur[q].v[2] = nu4.z;
      ur[q].v[3] = nu4.w;
      float4 gv = make_float4(0.f, 0.f, 0.f, 0.f);
      if (forced && i >= 8) gv = slot[1][lane];
      prefetch(i + kAhead);
      // rows: u[r - d] in ur[(q - d) mod 6], w_s[r - d] in w_s[(q - d) mod 3]; rowc[e] holds row ya - 8 + e
      w1[(q + 2) % 3] = stage(ur[(q + 4) % 6], ur[(q + 5) % 6], ur[q], ur[(q + 5) % 6], i + 3, P.h4);
      w2[(q + 1) % 3] = stage(w1[q % 3], w1[(q + 1) % 3], w1[(q + 2) % 3], ur[(q + 4) % 6], i + 2, P.h3);
      w3[q % 3] = stage(w2[(q + 2) % 3], w2[q % 3], w2[(q + 1) % 3], ur[(q + 3) % 6], i + 1, P.h2);
      if (i >= 8) {
        const F4 o = stage(w3[(q + 1) % 3], w3[(q + 2) % 3], w3[q % 3], ur[(q + 2) % 6], i, P.h);
        if (owner) {
          *reinterpret_cast<float4*>(po) = make_float4(o.v[0] + gv.x, o.v[1] + gv.y, o.v[2] + gv.z, o.v[3] + gv.w);
          if (ysnap) {
            const F4& y = ur[(q + 2) % 6];
            __stcs(reinterpret_cast<float4*>(py), make_float4(y.v[0], y.v[1], y.v[2], y.v[3]));
          }
        }
        po += P.nxp;
        py += P.nxp;
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

__global__ void __launch_bounds__(32 * kStreamWarps, 8) adr2d_stream_kernel(Stream2D P, const float* __restrict__ u,
                                                                           const float* __restrict__ g,
                                                                           float* __restrict__ out,
                                                                           float* __restrict__ ysnap) {
  __shared__ float4 ring[kStreamWarps][kRing][2][32];   // rows of u and g
  __shared__ float4 rowc[kMaxRun + 16];                 // rows ya - 8 .. yb + 7: west, east, diagonal, north / south
  __shared__ float rowt[kMaxRun + 16];                  // sponge depth of the row
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int run = blockIdx.y;
  const int ya = run * P.run_rows, yb = min(P.ny, ya + P.run_rows);
  // row coefficients of the run (constant over the march: read before the previous launch is waited for)
  for (int e = threadIdx.x; e < yb - ya + 16; e += blockDim.x) {
    const int j = ya - 8 + e;
    float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
    float t = 0.f;
    if (j >= 0 && j < P.ny) {
      const float ux = (P.adj ? -__ldg(P.U + j) : __ldg(P.U + j)) * P.i2dx;
      c = make_float4(ux + P.nx2, P.nx2 - ux, -2.f * (P.nx2 + P.ny2) + __ldg(P.r + j), P.ny2);
      const int d = min(j, P.ny - 1 - j);
      t = d < P.sponge_cells ? (float)(P.sponge_cells - d) * P.sponge_inv : 0.f;
    }
    rowc[e] = c;
    rowt[e] = t;
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int item = blockIdx.x * kStreamWarps + warp;    // vector and strip
  if (item >= P.strips * P.kg) return;
  const int v = item % P.kg, strip = item / P.kg;
  const int x0 = strip * kStripCells - 4, x1 = x0 + 128;   // the warp's cells
  const int64_t base = (int64_t)v * P.vstride;
  const int sc = max(P.sponge_cells, 0);
  const bool wall = x0 < sc || x1 > P.nx - sc || ya - 4 < sc || yb + 4 > P.ny - sc;
  if (wall)
    stream2d_rows<true>(P, u, g, out, ysnap, ring[warp], rowc, rowt, ya, yb, x0 + 4 * lane, lane, base);
  else
    stream2d_rows<false>(P, u, g, out, ysnap, ring[warp], rowc, rowt, ya, yb, x0 + 4 * lane, lane, base);
}

// Rows per run: the run length with the least estimated time.  A row costs a warp about 450 cycles of
// its own dependent chain, and the SM about 45 cycles of issue slots per resident warp (16 at most).
int stream2d_run_rows(int items, int ny, int sms) {
  int best = std::min(ny, kMaxRun);
  double best_t = 1e300;
  for (int runs = (ny + kMaxRun - 1) / kMaxRun; runs <= std::min(65535, std::max(1, ny / 4)); ++runs) {
    const int rows = (ny + runs - 1) / runs;
    const int nr = (ny + rows - 1) / rows;
    const double warps = std::ceil((double)items * nr / std::max(1, sms));
    const double t = (rows + 8) * std::max(450.0 * std::ceil(warps / 16.0), 45.0 * warps);
    if (t < best_t) {
      best_t = t;
      best = rows;
    }
  }
  return best;
}

// ---------------------------------------------------------------------------
// One stage per launch (FP64): out = u + f A x (+ g).  FP64 arithmetic bounds it: the constants come
// ready from the host and a point costs six FP64 operations (seven in the sponge).
// ---------------------------------------------------------------------------
template <typename R, bool LAST>
__global__ void __launch_bounds__(128) adr2d_horner_kernel(Grid3<R> g, bool adj, const R* x, const R* u,
                                                           const R* __restrict__ gf, R* out, R* __restrict__ ysnap,
                                                           R f) {
  const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 4 + threadIdx.y;
  const int64_t base = (int64_t)blockIdx.z * g.ncellp;
  const bool in = i < g.nx && j < g.ny;
  R cw = 0, ce = 0, cc = 0;
  if (in) {   // constant over the march: read before the previous launch is waited for
    const R ux = (adj ? -g.f0[j] : g.f0[j]) * g.i2dx;
    cw = ux + g.nx2;
    ce = g.nx2 - ux;
    cc = R(-2) * (g.nx2 + g.ny2) + g.f1[j];
    if (min(min(i, g.nx - 1 - i), min(j, g.ny - 1 - j)) < g.sponge_cells) cc -= sponge2d<R>(i, j, g);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!in) return;
  const int64_t p = base + (int64_t)j * g.nxp + i;
  const R* q = x + p;
  const R c = q[0];
  const R w = i > 0 ? q[-1] : R(0), e = i < g.nx - 1 ? q[1] : R(0);
  const R s = j > 0 ? q[-g.nxp] : R(0), n = j < g.ny - 1 ? q[g.nxp] : R(0);
  const R u0 = u == x ? c : u[p];
  R a = g.ny2 * (s + n);
  a = fma(cw, w, a);
  a = fma(ce, e, a);
  a = fma(cc, c, a);
  R o = fma(f, a, u0);
  if (LAST && gf != nullptr) o += gf[p];
  out[p] = o;
  if (ysnap != nullptr) ysnap[p] = u0;
}

template <typename F, typename... A>
cudaError_t launch_pdl(F kernel, dim3 grid, dim3 block, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace

template <typename R>
cudaError_t step_coefs_grid(rsv_operator op, const void* fhat, int64_t f_stride, int kg, bool adjoint, void* out,
                            void* tmp, int64_t tmp_freqs) {
  const Grid3<R> g = grid3_of<R>(op);
  const int comps = op->kind == RSV_OP_ADV3D ? 3 : 1;
  const int64_t rows = (int64_t)kg * comps * g.ncellp;
  const cpx<R>* f = (const cpx<R>*)fhat;
  const cpx<R>* tw = (const cpx<R>*)op->d_tw;
  const int sgn = adjoint ? -1 : 1;
  const int64_t m4 = 4 * op->n_t;
  for (int j0 = 0; j0 < op->n_omega; j0 += (int)tmp_freqs) {
    const int nf = (int)std::min<int64_t>(tmp_freqs, op->n_omega - j0);
    const dim3 grid((unsigned)((g.ncellp + 255) / 256), (unsigned)nf, (unsigned)kg);
    cpx<R>* o = (cpx<R>*)out + (int64_t)j0 * rows;
    cpx<R>* t = (cpx<R>*)tmp;
    // c = (h/6) (a0 f + B (a1 f + B (a2 f + 1/4 B f)))
    auto pass = [&](bool first, const cpx<R>* in, cpx<R>* dst, R c1, R cs, R cz, R bs, R sc) {
      if (comps == 3) {
        auto k = adjoint ? coef3d_kernel<R, true> : coef3d_kernel<R, false>;
        k<<<grid, 256, 0, op->stream>>>(g, j0, f, f_stride, in, rows, first, dst, rows, tw, op->d_pj, sgn, m4, c1, cs, cz, bs, sc);
      } else {
        auto k = adjoint ? coef2d_kernel<R, true> : coef2d_kernel<R, false>;
        k<<<grid, 256, 0, op->stream>>>(g, j0, f, f_stride, in, rows, first, dst, rows, tw, op->d_pj, sgn, m4, c1, cs, cz, bs, sc);
      }
    };
    pass(true, nullptr, o, R(0.5), R(0.5), R(0), R(0.25), R(1));
    pass(false, o, t, R(1), R(2), R(0), R(1), R(1));
    pass(false, t, o, R(1), R(4), R(1), R(1), R(op->h / 6.0));
  }
  return cudaGetLastError();
}

// S steps of the 2-D kind; the state ping-pongs between u and its second buffer.
template <typename R>
cudaError_t step_march_2d(rsv_operator op, const MarchTile& t, void* state, const void* G, void* Y) {
  const Grid3<R> g = grid3_of<R>(op);
  const int64_t rows = (int64_t)t.kg * g.ncellp;
  R* cur = static_cast<R*>(state);
  R* nxt = cur + rows;
  cudaError_t e = cudaSuccess;
  if constexpr (sizeof(R) == 4) {
    Stream2D P;
    P.nx = g.nx;
    P.nxp = g.nxp;
    P.ny = g.ny;
    P.kg = t.kg;
    P.strips = (g.nx + kStripCells - 1) / kStripCells;
    P.run_rows = stream2d_run_rows(P.strips * t.kg, g.ny, op->sm_count);
    P.runs = (g.ny + P.run_rows - 1) / P.run_rows;
    P.vstride = g.ncellp;
    P.U = g.f0;
    P.r = g.f1;
    P.i2dx = g.i2dx;
    P.nx2 = g.nx2;
    P.ny2 = g.ny2;
    P.h = g.h;
    P.h2 = g.h / 2.f;
    P.h3 = g.h / 3.f;
    P.h4 = g.h / 4.f;
    P.sponge_cells = g.sponge_cells;
    P.sponge_amp = g.sponge_amp;
    P.sponge_inv = g.sponge_inv;
    P.adj = t.adjoint ? 1 : 0;
    const dim3 grid((unsigned)((P.strips * t.kg + kStreamWarps - 1) / kStreamWarps), (unsigned)P.runs);
    for (int s = 0; s < t.steps && e == cudaSuccess; ++s) {
      const float* gs = (G != nullptr && t.n0 + s < t.n_forced) ? static_cast<const float*>(G) + (size_t)s * rows : nullptr;
      float* ys = (Y != nullptr && s >= t.y_first) ? static_cast<float*>(Y) + (size_t)s * rows : nullptr;
      e = launch_pdl(adr2d_stream_kernel, grid, dim3(32 * kStreamWarps), op->stream, P, (const float*)cur, gs, nxt, ys);
      std::swap(cur, nxt);
    }
    if (e == cudaSuccess && cur != static_cast<R*>(state))
      e = cudaMemcpyAsync(state, cur, sizeof(R) * rows, cudaMemcpyDeviceToDevice, op->stream);
  } else {
    R* w = nxt + rows;
    const dim3 grid((unsigned)((g.nx + 31) / 32), (unsigned)((g.ny + 3) / 4), (unsigned)t.kg), block(32, 4);
    for (int s = 0; s < t.steps && e == cudaSuccess; ++s) {
      const R* gs = (G != nullptr && t.n0 + s < t.n_forced) ? static_cast<const R*>(G) + (size_t)s * rows : nullptr;
      R* ys = (Y != nullptr && s >= t.y_first) ? static_cast<R*>(Y) + (size_t)s * rows : nullptr;
      const R* none = nullptr;
      R* nosnap = nullptr;
      e = launch_pdl(adr2d_horner_kernel<R, false>, grid, block, op->stream, g, t.adjoint, (const R*)cur, (const R*)cur, none, nxt, ys, g.h / R(4));
      if (e == cudaSuccess) e = launch_pdl(adr2d_horner_kernel<R, false>, grid, block, op->stream, g, t.adjoint, (const R*)nxt, (const R*)cur, none, w, nosnap, g.h / R(3));
      if (e == cudaSuccess) e = launch_pdl(adr2d_horner_kernel<R, false>, grid, block, op->stream, g, t.adjoint, (const R*)w, (const R*)cur, none, nxt, nosnap, g.h / R(2));
      // the last stage reads its own point of u only: in place
      if (e == cudaSuccess) e = launch_pdl(adr2d_horner_kernel<R, true>, grid, block, op->stream, g, t.adjoint, (const R*)nxt, (const R*)cur, gs, cur, nosnap, g.h);
    }
  }
  if (e == cudaSuccess) e = check_finite(op, state, rows, true);
  return e;
}

template cudaError_t step_coefs_grid<float>(rsv_operator, const void*, int64_t, int, bool, void*, void*, int64_t);
template cudaError_t step_coefs_grid<double>(rsv_operator, const void*, int64_t, int, bool, void*, void*, int64_t);
template cudaError_t step_march_2d<float>(rsv_operator, const MarchTile&, void*, const void*, void*);
template cudaError_t step_march_2d<double>(rsv_operator, const MarchTile&, void*, const void*, void*);

}  // namespace rsv
