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
// contractions; `launch_finish` drops the padding.
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

// a_j = c1 + cs s_j + cz z_j (one thread per block: the 64-bit remainders of the phases are slow)
template <typename R>
__device__ cpx<R> coef_factor(const cpx<R>* tw, int64_t p, int64_t m4, R c1, R cs, R cz) {
  const cpx<R> s = tw[phase_index(p, 1, m4)], z = tw[phase_index(p, 2, m4)];
  return mk<R>(c1 + cs * s.re + cz * z.re, cs * s.im + cz * z.im);
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
  __shared__ cpx<R> sa;
  const int w = blockIdx.y, v = blockIdx.z;
  if (threadIdx.x == 0) sa = coef_factor<R>(tw, sgn * pj[j0 + w], m4, c1, cs, cz);
  __syncthreads();
  const cpx<R> a = sa;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) % g.nxp, j = (blockIdx.x * blockDim.x + threadIdx.x) / g.nxp;
  if (j >= g.ny) return;
  cpx<R>* o = out + (int64_t)w * o_stride + (int64_t)v * g.ncellp + (int64_t)j * g.nxp + i;
  if (i >= g.nx) {
    *o = mk<R>(0, 0);
    return;
  }
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
  __shared__ cpx<R> sa;
  const int w = blockIdx.y, v = blockIdx.z;
  if (threadIdx.x == 0) sa = coef_factor<R>(tw, sgn * pj[j0 + w], m4, c1, cs, cz);
  __syncthreads();
  const cpx<R> a = sa;
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;   // a component's cells number less than 2^31
  const unsigned jk = e / (unsigned)g.nxp;
  const int i = (int)(e - jk * (unsigned)g.nxp), j = (int)(jk % (unsigned)g.ny), kz = (int)(jk / (unsigned)g.ny);
  if (kz >= g.nz) return;
  cpx<R>* o = out + (int64_t)w * o_stride + (int64_t)v * 3 * g.ncellp + e;
  if (i >= g.nx) {
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c * g.ncellp] = mk<R>(0, 0);
    return;
  }
  const cpx<R>* fv = f + (int64_t)(j0 + w) * f_stride + (int64_t)v * 3 * g.ncell;
  const int64_t q = (int64_t)jk * g.nx + i;              // cell in the fields and in f
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
// loaded it evaluates w1 on row r - 1, w2 on r - 2, w3 on r - 3 and u' on r - 4.  The rows of a
// stencil live in registers (x neighbours across lanes by shuffles), so there is no barrier and no
// shared-memory traffic but the per-warp ring that stages u and g by 16-byte asynchronous copies.  A
// run starts four rows early and ends four late; what it computes there is not stored.  Rows and
// columns outside the grid have zero factors, so they stay zero.  Issue slots bound it, not bytes: the
// stage factors h / m are multiplied into the row coefficients, so that a cell costs one addition and
// four multiply-adds per stage.
//
// The rows of all (vector, strip) columns are one list that is cut into equal chunks, one per warp
// (block of one warp) and as many as the GPU holds at once; a chunk that crosses from one column to
// the next runs as two runs.  1024 x 512 x 16 vectors: 28 us per step with 16 warps per SM (12: 33, 8: 43),
// against 103 us for the two stage-pair kernels; 96 MB of DRAM traffic per step.
// ---------------------------------------------------------------------------
constexpr int kStripCells = 120, kGroups = 3, kMaxChunk = 256, kWarpsPerSm = 16;

struct Stream2D {
  int nx, nxp, ny, kg;
  int strips, chunk;
  int64_t total;             // rows of all columns
  int64_t vstride;
  const float *U, *r;
  float i2dx, nx2, ny2;
  float f[4];                // h / 4, h / 3, h / 2, h: the stages' factors
  int sponge_cells;
  float sponge_amp, sponge_inv;
  int adj;
};

// Copies 16 bytes, or writes zeros without reading.
__device__ __forceinline__ void cp16_zfill(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

struct F4 {
  float v[4];
};
__device__ __forceinline__ F4 lds4(uint32_t a) {
  F4 o;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(o.v[0]), "=f"(o.v[1]), "=f"(o.v[2]), "=f"(o.v[3]) : "r"(a) : "memory");
  return o;
}

constexpr uint32_t kSlotBytes = 2 * 32 * 16;                       // a row of u and a row of g
constexpr uint32_t kRingBytes = kGroups * 3 * kSlotBytes;
// per row of the run (with 8 rows before and after it): 4 stages x (west, east, diagonal, north / south) x h / m,
// then the sponge depths
constexpr uint32_t kRowBytes = 4 * 16;
constexpr size_t stream2d_smem(int chunk) { return kRingBytes + (size_t)(chunk + 16) * (kRowBytes + 4); }

// One run: rows [ya, yb) of a column.  WALL: the strip reaches a wall in x or its sponge (elsewhere the
// row's sponge rate is part of the row's diagonal coefficient).
template <bool WALL>
__device__ __forceinline__ void stream2d_rows(const Stream2D& P, const float* __restrict__ u, const float* __restrict__ g,
                                              float* __restrict__ out, float* __restrict__ ysnap, uint32_t ring,
                                              uint32_t rows, const float* rowt, int ya, int yb, int gx, int lane,
                                              int64_t base) {
  const bool in_x = gx >= 0 && gx < P.nxp;
  const bool owner = lane >= 1 && lane <= 30 && gx < P.nxp;
  const bool forced = g != nullptr;
  float sx[4], sg[4];   // sponge depth and rate of the lane's columns (0: none)
  float m[4];           // 1 inside the grid, 0 outside
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int i = gx + c;
    const bool in = i >= 0 && i < P.nx;
    const int d = min(i, P.nx - 1 - i);
    m[c] = in ? 1.f : 0.f;
    sx[c] = in && d < P.sponge_cells ? (float)(P.sponge_cells - d) * P.sponge_inv : 0.f;
    sg[c] = P.sponge_amp * sx[c] * sx[c];
  }
  const bool edge_x = WALL && __any_sync(0xffffffffu, m[0] * m[1] * m[2] * m[3] == 0.f);
  // iteration i loads row ya - 4 + i of u and row ya - 8 + i of g; three groups of three ring slots:
  // the current three iterations', the previous three's and the next three's
  const int iters = yb - ya + 8;
  const int u_lo = max(0, 4 - ya), u_n = min(iters, P.ny - ya + 4) - u_lo;   // iterations whose row is inside the grid
  const int64_t off = base + (in_x ? gx : 0);
  const float* pu = u + off + (int64_t)(ya - 4) * P.nxp;
  const float* pg = (forced ? g : u) + off + (int64_t)(ya - 8) * P.nxp;
  auto prefetch = [&](int i, uint32_t dst) {
    cp16_zfill(dst, pu, in_x && (unsigned)(i - u_lo) < (unsigned)u_n);
    if (forced) cp16_zfill(dst + 32 * 16, pg, in_x && i >= 8 && i < iters);
    pu += P.nxp;
    pg += P.nxp;
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  uint32_t cur = ring + 16 * lane, prev = cur + 3 * kSlotBytes, next = cur + 6 * kSlotBytes;
#pragma unroll
  for (int q = 0; q < 3; ++q) prefetch(q, cur + q * kSlotBytes);
  F4 ur[3], w1[3], w2[3], w3[3];
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int c = 0; c < 4; ++c) ur[q].v[c] = w1[q].v[c] = w2[q].v[c] = w3[q].v[c] = 0.f;
  // u0 + h/m A x on a row from the rows below, at and above it; e: the row's index in the table
  auto stage = [&](const F4& xb, const F4& xc, const F4& xt, const F4& u0, int e, int st) -> F4 {
    const F4 rc = lds4(rows + (uint32_t)e * kRowBytes + 16 * st);   // west, east, diagonal, north / south
    const float left = __shfl_up_sync(0xffffffffu, xc.v[3], 1), right = __shfl_down_sync(0xffffffffu, xc.v[0], 1);
    float cc[4] = {rc.v[2], rc.v[2], rc.v[2], rc.v[2]};
    if (WALL) {
      const float ty = rowt[e];   // the rate of the nearer wall: the larger depth
#pragma unroll
      for (int c = 0; c < 4; ++c) cc[c] = fmaf(-P.f[st], sx[c] > ty ? sg[c] : P.sponge_amp * ty * ty, rc.v[2]);
    }
    F4 o;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float a = fmaf(rc.v[3], xb.v[c] + xt.v[c], u0.v[c]);
      a = fmaf(rc.v[0], c == 0 ? left : xc.v[c - 1], a);
      a = fmaf(rc.v[1], c == 3 ? right : xc.v[c + 1], a);
      o.v[c] = fmaf(cc[c], xc.v[c], a);
    }
    if (edge_x) {
#pragma unroll
      for (int c = 0; c < 4; ++c) o.v[c] = m[c] != 0.f ? o.v[c] : 0.f;
    }
    return o;
  };
  float* po = out + base + (int64_t)(ya - 8) * P.nxp + gx;
  float* py = ysnap + base + (int64_t)(ya - 8) * P.nxp + gx;   // used only when ysnap is given
  for (int i0 = 0; i0 < iters; i0 += 3) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int i = i0 + q;
      if (i >= iters) break;
      asm volatile("cp.async.wait_group 2;" ::: "memory");
      ur[q] = lds4(cur + q * kSlotBytes);
      // rows r - 3 and r - 4 of u are read again from the ring
      const F4 u3 = lds4(prev + q * kSlotBytes);
      const F4 u4 = lds4(q == 0 ? next + 2 * kSlotBytes : prev + (q - 1) * kSlotBytes);
      const F4 gv = lds4(cur + q * kSlotBytes + 32 * 16);
      prefetch(i + 3, next + q * kSlotBytes);
      // rows: u[r - d], w_s[r - d] in slot (q - d) mod 3; the table's row e is row ya - 8 + e
      w1[(q + 2) % 3] = stage(ur[(q + 1) % 3], ur[(q + 2) % 3], ur[q], ur[(q + 2) % 3], i + 3, 0);
      w2[(q + 1) % 3] = stage(w1[q], w1[(q + 1) % 3], w1[(q + 2) % 3], ur[(q + 1) % 3], i + 2, 1);
      w3[q] = stage(w2[(q + 2) % 3], w2[q], w2[(q + 1) % 3], u3, i + 1, 2);
      const F4 o = stage(w3[(q + 1) % 3], w3[(q + 2) % 3], w3[q], u4, i, 3);
      if (owner && i >= 8) {
        float4 v = make_float4(o.v[0], o.v[1], o.v[2], o.v[3]);
        if (forced) v = make_float4(v.x + gv.v[0], v.y + gv.v[1], v.z + gv.v[2], v.w + gv.v[3]);
        *reinterpret_cast<float4*>(po) = v;
        if (ysnap) __stcs(reinterpret_cast<float4*>(py), make_float4(u4.v[0], u4.v[1], u4.v[2], u4.v[3]));
      }
      po += P.nxp;
      py += P.nxp;
    }
    const uint32_t t = prev;
    prev = cur;
    cur = next;
    next = t;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
}

__global__ void __launch_bounds__(32, kWarpsPerSm) adr2d_stream_kernel(Stream2D P, const float* __restrict__ u,
                                                                      const float* __restrict__ g,
                                                                      float* __restrict__ out,
                                                                      float* __restrict__ ysnap) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x;
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem_raw), rows = ring + kRingBytes;
  float4* rowc = reinterpret_cast<float4*>(smem_raw + kRingBytes);
  float* rowt = reinterpret_cast<float*>(rowc + 4 * (P.chunk + 16));
  int64_t at = (int64_t)blockIdx.x * P.chunk;
  const int64_t end = min(P.total, at + P.chunk);
  bool waited = false;
  while (at < end) {
    const int col = (int)(at / P.ny);
    const int ya = (int)(at - (int64_t)col * P.ny), yb = (int)min((int64_t)P.ny, ya + (end - at));
    const int v = col % P.kg, strip = col / P.kg;
    const int x0 = strip * kStripCells - 4, x1 = x0 + 128;   // the warp's cells
    const int sc = max(P.sponge_cells, 0);
    const bool wall = x0 < sc || x1 > P.nx - sc;
    // row coefficients of the run (constant over the march: read before the previous launch is waited for)
    for (int e = lane; e < yb - ya + 16; e += 32) {
      const int j = ya - 8 + e;
      float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
      float t = 0.f;
      if (j >= 0 && j < P.ny) {
        const float ux = (P.adj ? -__ldg(P.U + j) : __ldg(P.U + j)) * P.i2dx;
        const int d = min(j, P.ny - 1 - j);
        t = d < P.sponge_cells ? (float)(P.sponge_cells - d) * P.sponge_inv : 0.f;
        c = make_float4(ux + P.nx2, P.nx2 - ux, -2.f * (P.nx2 + P.ny2) + __ldg(P.r + j), P.ny2);
        if (!wall) c.z -= P.sponge_amp * t * t;
      }
#pragma unroll
      for (int st = 0; st < 4; ++st)
        rowc[4 * e + st] = make_float4(P.f[st] * c.x, P.f[st] * c.y, P.f[st] * c.z, P.f[st] * c.w);
      rowt[e] = t;
    }
    __syncwarp();
    if (!waited) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      waited = true;
    }
    const int64_t base = (int64_t)v * P.vstride;
    if (wall)
      stream2d_rows<true>(P, u, g, out, ysnap, ring, rows, rowt, ya, yb, x0 + 4 * lane, lane, base);
    else
      stream2d_rows<false>(P, u, g, out, ysnap, ring, rows, rowt, ya, yb, x0 + 4 * lane, lane, base);
    at += yb - ya;
  }
}

// ---------------------------------------------------------------------------
// One stage per launch (FP64): out = u + f A x (+ g).  FP64 arithmetic bounds it (one warp instruction
// per 19 cycles and SM), so the row coefficients times h / m come ready from a table built per march
// tile: a point costs one addition and four multiply-adds, one more in the sponge and for the forcing.
// ---------------------------------------------------------------------------
template <typename R>
struct RowTab {
  R w, e, c, y;   // west, east, diagonal, north / south
};

// rows [4 stages][ny] of the table, then the sponge rates of the columns [nx] and of the rows [ny]
template <typename R>
__global__ void row_table_kernel(Grid3<R> g, bool adj, RowTab<R>* __restrict__ rows, R* __restrict__ sp) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  auto rate = [&](int d) {
    if (d >= g.sponge_cells) return R(0);
    const R t = R(g.sponge_cells - d) * g.sponge_inv;
    return g.sponge_amp * t * t;
  };
  if (e < g.ny) {
    const R ux = (adj ? -g.f0[e] : g.f0[e]) * g.i2dx;
    for (int st = 0; st < 4; ++st) {
      const R f = g.h / R(4 - st);
      RowTab<R> t;
      t.w = f * (ux + g.nx2);
      t.e = f * (g.nx2 - ux);
      t.c = f * (R(-2) * (g.nx2 + g.ny2) + g.f1[e]);
      t.y = f * g.ny2;
      rows[st * g.ny + e] = t;
    }
    sp[g.nx + e] = rate(min(e, g.ny - 1 - e));
  }
  if (e < g.nx) sp[e] = rate(min(e, g.nx - 1 - e));
}

template <typename R, bool LAST>
__global__ void __launch_bounds__(128) adr2d_horner_kernel(Grid3<R> g, const RowTab<R>* __restrict__ rows,
                                                           const R* __restrict__ sp, R f, const R* x, const R* u,
                                                           const R* __restrict__ gf, R* out, R* __restrict__ ysnap) {
  const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 4 + threadIdx.y;
  const int64_t p = (int64_t)blockIdx.z * g.ncellp + (int64_t)j * g.nxp + i;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (i >= g.nx || j >= g.ny) return;
  const RowTab<R> t = rows[j];
  const R* q = x + p;
  const R c = q[0];
  const R w = i > 0 ? q[-1] : R(0), e = i < g.nx - 1 ? q[1] : R(0);
  const R s = j > 0 ? q[-g.nxp] : R(0), n = j < g.ny - 1 ? q[g.nxp] : R(0);
  const R u0 = u == x ? c : u[p];
  R cc = t.c;
  const int dx = min(i, g.nx - 1 - i), dy = min(j, g.ny - 1 - j);
  if (min(dx, dy) < g.sponge_cells) cc = fma(-f, sp[dx < dy ? i : g.nx + j], cc);   // the nearer wall's rate
  R o = fma(t.y, s + n, u0);
  o = fma(t.w, w, o);
  o = fma(t.e, e, o);
  o = fma(cc, c, o);
  if (LAST && gf != nullptr) o += gf[p];
  out[p] = o;
  if (ysnap != nullptr) ysnap[p] = u0;
}

template <typename F, typename... A>
cudaError_t launch_pdl(F kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
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
    P.total = (int64_t)P.strips * t.kg * g.ny;
    // one chunk per resident warp, of 4 rows at least (a run pays 8 rows for its start and end)
    const int64_t warps = (int64_t)std::max(1, op->sm_count) * kWarpsPerSm;
    P.chunk = (int)std::min<int64_t>(kMaxChunk, std::max<int64_t>(4, (P.total + warps - 1) / warps));
    P.vstride = g.ncellp;
    P.U = g.f0;
    P.r = g.f1;
    P.i2dx = g.i2dx;
    P.nx2 = g.nx2;
    P.ny2 = g.ny2;
    for (int m = 0; m < 4; ++m) P.f[m] = g.h / (float)(4 - m);
    P.sponge_cells = g.sponge_cells;
    P.sponge_amp = g.sponge_amp;
    P.sponge_inv = g.sponge_inv;
    P.adj = t.adjoint ? 1 : 0;
    const unsigned blocks = (unsigned)((P.total + P.chunk - 1) / P.chunk);
    for (int s = 0; s < t.steps && e == cudaSuccess; ++s) {
      const float* gs = (G != nullptr && t.n0 + s < t.n_forced) ? static_cast<const float*>(G) + (size_t)s * rows : nullptr;
      float* ys = (Y != nullptr && s >= t.y_first) ? static_cast<float*>(Y) + (size_t)s * rows : nullptr;
      e = launch_pdl(adr2d_stream_kernel, dim3(blocks), dim3(32), stream2d_smem(P.chunk), op->stream, P, (const float*)cur, gs, nxt,
                     ys);
      std::swap(cur, nxt);
    }
    if (e == cudaSuccess && cur != static_cast<R*>(state))
      e = cudaMemcpyAsync(state, cur, sizeof(R) * rows, cudaMemcpyDeviceToDevice, op->stream);
  } else {
    R* w = nxt + rows;
    RowTab<R>* tab = reinterpret_cast<RowTab<R>*>(w + rows);
    R* sp = reinterpret_cast<R*>(tab + 4 * (size_t)g.ny);
    const dim3 grid((unsigned)((g.nx + 31) / 32), (unsigned)((g.ny + 3) / 4), (unsigned)t.kg), block(32, 4);
    row_table_kernel<R><<<(unsigned)((std::max(g.nx, g.ny) + 127) / 128), 128, 0, op->stream>>>(g, t.adjoint, tab, sp);
    e = cudaGetLastError();
    auto stage = [&](auto kernel, int st, const R* x, const R* u, const R* gs, R* o, R* ys) {
      if (e == cudaSuccess)
        e = launch_pdl(kernel, grid, block, 0, op->stream, g, (const RowTab<R>*)(tab + (size_t)st * g.ny), (const R*)sp,
                       g.h / R(4 - st), x, u, gs, o, ys);
    };
    for (int s = 0; s < t.steps && e == cudaSuccess; ++s) {
      const R* gs = (G != nullptr && t.n0 + s < t.n_forced) ? static_cast<const R*>(G) + (size_t)s * rows : nullptr;
      R* ys = (Y != nullptr && s >= t.y_first) ? static_cast<R*>(Y) + (size_t)s * rows : nullptr;
      stage(adr2d_horner_kernel<R, false>, 0, cur, cur, nullptr, nxt, ys);
      stage(adr2d_horner_kernel<R, false>, 1, nxt, cur, nullptr, w, nullptr);
      stage(adr2d_horner_kernel<R, false>, 2, w, cur, nullptr, nxt, nullptr);
      stage(adr2d_horner_kernel<R, true>, 3, nxt, cur, gs, cur, nullptr);   // reads its own point of u only: in place
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
