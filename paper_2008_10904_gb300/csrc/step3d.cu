// 3-D kernels of the step form (see step2d.cu), FP32: two launches per step, two stages each.
//
//   half 1:  w1 = u + h/4 A u    on the tile + 1 halo cell in x, y (shared memory)
//            w2 = u + h/3 A w1   on the tile
//   half 2:  w3 = u + h/2 A w2   on the tile + 1 halo cell
//            u' = u + h A w3 + g on the tile
//
// A CTA owns a 64 x 8 tile in (x, y) of one vector and a run of planes in z, and streams through z:
// the first stage's input (u or w2) sits in a ring of four planes with two halo cells in x and y
// (three in use, the next arriving by asynchronous copies), the first stage's result in a ring of
// three planes with one halo cell.  At plane p the first stage is evaluated on plane p + 1 and the
// second on plane p, one barrier apart.  Per step the state-sized arrays cross HBM six times (half 1:
// u read, w2 written, plus the snapshot on analysed steps; half 2: w2, u and g read, u' written)
// against eleven for the stage pairs with accumulator and forcing (stencil_kernels.cu).  Cells outside
// the grid hold zero (homogeneous Dirichlet), in both rings.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <mutex>

#include "rsv_ops.h"

namespace rsv {
namespace {

constexpr int kTX = 64, kTY = 8, kThreads = 256;
constexpr int kUW = kTX + 8, kUH = kTY + 4;     // input ring: x from X0 - 4 (16-byte aligned), y halo 2
constexpr int kXW = kTX + 2, kXH = kTY + 2;     // intermediate ring: halo 1
constexpr int kUP = kUW * kUH, kXP = kXW * kXH;
constexpr int kRow4 = kUW / 4;
constexpr int kS1 = (kXP + kThreads - 1) / kThreads, kS2 = kTX * kTY / kThreads;
constexpr size_t kSmem = sizeof(float) * (4 * 3 * (size_t)kUP + 3 * 3 * (size_t)kXP);

struct Half3D {
  int nx, nxp, ny, nz, kg, zruns;
  int64_t vstride;            // 3 * nxp * ny * nz
  float cdx, nx2, ny2, nz2;   // 1 / (2 dx), visc / d^2
  const float4* f4;           // base flow per cell: U, dU/dx, dU/dy, dU/dz (rows padded to nxp)
  const float *U, *Ux, *Uy, *Uz;
  const float* in;            // u (half 1) or w2 (half 2)
  const float* u;             // half 2: u
  const float* g;             // half 2: g_n (nullable)
  float* out;                 // w2 or u'
  float* ysnap;               // half 1: snapshot of u (nullable)
  float f1, f2;               // factors of the two stages
};

// Base flow at one cell: forward advection uses U at the cell, the transposed one U at the x neighbours.
struct Flow {
  float Uc, Uw, Ue, Ux, Uy, Uz;
};

template <bool ADJ>
__device__ __forceinline__ Flow load_flow(const Half3D& P, int q, int i, bool ok) {
  Flow b;
  if (!ADJ) {   // one 16-byte load of the interleaved fields (the transposed one measured slower so)
    const float4 v = ok ? __ldg(P.f4 + q) : make_float4(0.f, 0.f, 0.f, 0.f);
    b.Uc = v.x;
    b.Uw = b.Ue = 0.f;
    b.Ux = v.y;
    b.Uy = v.z;
    b.Uz = v.w;
    return b;
  }
  b.Uc = 0.f;
  b.Uw = (ok && i > 0) ? __ldg(P.U + q - 1) : 0.f;
  b.Ue = (ok && i < P.nx - 1) ? __ldg(P.U + q + 1) : 0.f;
  b.Ux = ok ? __ldg(P.Ux + q) : 0.f;
  b.Uy = ok ? __ldg(P.Uy + q) : 0.f;
  b.Uz = ok ? __ldg(P.Uz + q) : 0.f;
  return b;
}

// 7-point operator at index e of component planes with rows of width W (below, centre, above).
template <bool ADJ, int W, int PLANE>
__device__ __forceinline__ void op3d(const float* __restrict__ xb, const float* __restrict__ xc,
                                     const float* __restrict__ xt, int e, const Flow& b, const Half3D& P, float k[3]) {
  float cen[3];
  const float cc = -2.f * (P.nx2 + P.ny2 + P.nz2);
  const float cw = P.nx2 + P.cdx * (ADJ ? -b.Uw : b.Uc), ce = P.nx2 - P.cdx * (ADJ ? -b.Ue : b.Uc);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float* p = xc + c * PLANE;
    cen[c] = p[e];
    float a = P.nz2 * (xb[c * PLANE + e] + xt[c * PLANE + e]);
    a = fmaf(P.ny2, p[e - W] + p[e + W], a);
    a = fmaf(cw, p[e - 1], a);
    a = fmaf(ce, p[e + 1], a);
    k[c] = fmaf(cc, cen[c], a);
  }
  if (ADJ) {
    k[0] = fmaf(-b.Ux, cen[0], k[0]);
    k[1] = fmaf(-b.Uy, cen[0], k[1]);
    k[2] = fmaf(-b.Uz, cen[0], k[2]);
  } else {
    k[0] = fmaf(-b.Ux, cen[0], fmaf(-b.Uy, cen[1], fmaf(-b.Uz, cen[2], k[0])));
  }
}

__device__ __forceinline__ void cp16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

template <bool ADJ, bool SECOND>
__global__ void __launch_bounds__(kThreads, 2) adv3d_half_kernel(Half3D P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* ring = reinterpret_cast<float*>(smem_raw);   // [4 planes][3 comps][kUP]
  float* mid = ring + 4 * 3 * kUP;                      // [3 planes][3 comps][kXP]
  const int nx = P.nx, ny = P.ny, nz = P.nz;
  const int plane = P.nxp * ny, ncell = plane * nz;
  int b = blockIdx.x;          // vector fastest: neighbouring tiles of all vectors in flight together
  const int v = b % P.kg;
  b /= P.kg;
  const int ntx = (nx + kTX - 1) / kTX, nty = (ny + kTY - 1) / kTY;
  const int X0 = (b % ntx) * kTX;
  b /= ntx;
  const int Y0 = (b % nty) * kTY;
  const int cz = b / nty;
  const int z0 = (int)((int64_t)cz * nz / P.zruns), z1 = (int)((int64_t)(cz + 1) * nz / P.zruns);
  const int64_t base = (int64_t)v * P.vstride;
  const float* __restrict__ in = P.in + base;
  const float* __restrict__ pu = SECOND ? P.u + base : nullptr;
  const float* __restrict__ pg = SECOND && P.g ? P.g + base : nullptr;
  float* __restrict__ out = P.out + base;
  float* __restrict__ ysnap = !SECOND && P.ysnap ? P.ysnap + base : nullptr;
  const int tid = threadIdx.x;
  // launched as a programmatic dependent: resident early, waits here before any memory access
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // per-thread cells, fixed over the planes: (x, y) offset (-1 outside the grid), x index, ring index
  int xy1[kS1], gi1[kS1], eu1[kS1];
#pragma unroll
  for (int sl = 0; sl < kS1; ++sl) {
    const int e = tid + sl * kThreads;
    const int lx = e % kXW, ly = e / kXW;
    const int gi = X0 - 1 + lx, gj = Y0 - 1 + ly;
    const bool ok = e < kXP && gi >= 0 && gi < nx && gj >= 0 && gj < ny;
    xy1[sl] = ok ? gj * P.nxp + gi : -1;
    gi1[sl] = gi;
    eu1[sl] = e < kXP ? (ly + 1) * kUW + lx + 3 : kUW + 3;   // a slot past the region evaluates the first cell
  }
  int xy2[kS2], gi2[kS2];
#pragma unroll
  for (int sl = 0; sl < kS2; ++sl) {
    const int e = tid + sl * kThreads;
    const int gi = X0 + e % kTX, gj = Y0 + e / kTX;
    xy2[sl] = (gi < nx && gj < ny) ? gj * P.nxp + gi : -1;
    gi2[sl] = gi;
  }

  // plane kz of the input into ring slot kz & 3, 16-byte chunks wholly inside or outside the padded grid
  auto load_plane = [&](int kz) {
    float* dst = ring + (size_t)(kz & 3) * 3 * kUP;
    const bool zin = kz >= 0 && kz < nz;
    for (int e = tid; e < 3 * kUH * kRow4; e += kThreads) {
      const int row = e / kRow4, ch = e - row * kRow4;
      const int c = row / kUH, ly = row - c * kUH;
      const int gj = Y0 - 2 + ly, gx = X0 - 4 + 4 * ch;
      float* d = dst + c * kUP + ly * kUW + 4 * ch;
      if (zin && gj >= 0 && gj < ny && gx >= 0 && gx < P.nxp)
        cp16(d, in + c * ncell + kz * plane + gj * P.nxp + gx);
      else
        *reinterpret_cast<float4*>(d) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  struct In1 {
    float u[kS1][3];
    Flow b[kS1];
  };
  struct In2 {
    float u[kS2][3], g[kS2][3];
    Flow b[kS2];
  };
  auto fetch1 = [&](int kz, In1& r) {
    const bool zin = kz >= 0 && kz < nz;
#pragma unroll
    for (int sl = 0; sl < kS1; ++sl) {
      const bool ok = zin && xy1[sl] >= 0;
      const int q = kz * plane + xy1[sl];
#pragma unroll
      for (int c = 0; c < 3; ++c) r.u[sl][c] = (SECOND && ok) ? __ldg(pu + q + c * ncell) : 0.f;
      r.b[sl] = load_flow<ADJ>(P, q, gi1[sl], ok);
    }
  };
  auto fetch2 = [&](int kz, In2& r) {
    const bool zin = kz >= z0 && kz < z1;
#pragma unroll
    for (int sl = 0; sl < kS2; ++sl) {
      const bool ok = zin && xy2[sl] >= 0;
      const int q = kz * plane + xy2[sl];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        r.u[sl][c] = (SECOND && ok) ? __ldg(pu + q + c * ncell) : 0.f;
        r.g[sl][c] = (SECOND && ok && pg) ? __ldcs(pg + q + c * ncell) : 0.f;
      }
      r.b[sl] = load_flow<ADJ>(P, q, gi2[sl], ok);
    }
  };
  // first stage on plane kz, tile + 1 halo cell, as one straight-line block masked afterwards
  auto first_stage = [&](int kz, const In1& r) {
    float* dst = mid + (size_t)(((kz % 3) + 3) % 3) * 3 * kXP;
    const float* xb = ring + (size_t)((kz - 1) & 3) * 3 * kUP;
    const float* xc = ring + (size_t)(kz & 3) * 3 * kUP;
    const float* xt = ring + (size_t)((kz + 1) & 3) * 3 * kUP;
    const bool zin = kz >= 0 && kz < nz;
#pragma unroll
    for (int sl = 0; sl < kS1; ++sl) {
      const int e = tid + sl * kThreads;
      const bool ok = zin && xy1[sl] >= 0;
      float k[3];
      op3d<ADJ, kUW, kUP>(xb, xc, xt, eu1[sl], r.b[sl], P, k);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float uu = SECOND ? r.u[sl][c] : xc[c * kUP + eu1[sl]];
        const float o = ok ? fmaf(P.f1, k[c], uu) : 0.f;
        if (e < kXP) dst[c * kXP + e] = o;
      }
    }
  };
  // second stage on plane kz, the tile: every slot is evaluated, only the stores are masked
  auto second_stage = [&](int kz, const In2& r) {
    const float* mb = mid + (size_t)((((kz - 1) % 3) + 3) % 3) * 3 * kXP;
    const float* mc = mid + (size_t)(kz % 3) * 3 * kXP;
    const float* mt = mid + (size_t)((kz + 1) % 3) * 3 * kXP;
    const float* uc = ring + (size_t)(kz & 3) * 3 * kUP;
#pragma unroll
    for (int sl = 0; sl < kS2; ++sl) {
      const int e = tid + sl * kThreads;
      const int tx = e % kTX, ty = e / kTX;
      const int q = kz * plane + xy2[sl];
      float k[3];
      op3d<ADJ, kXW, kXP>(mb, mc, mt, (ty + 1) * kXW + tx + 1, r.b[sl], P, k);
      if (xy2[sl] < 0) continue;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float uu = SECOND ? r.u[sl][c] : uc[c * kUP + (ty + 2) * kUW + tx + 4];
        float o = fmaf(P.f2, k[c], uu);
        if (SECOND) o += r.g[sl][c];
        out[q + c * ncell] = o;
        if (!SECOND && ysnap) __stcs(ysnap + q + c * ncell, uu);
      }
    }
  };

  In1 s1;
  In2 s2;
  for (int kz = z0 - 2; kz <= z0 + 1; ++kz) load_plane(kz);
  fetch1(z0 - 1, s1);
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  first_stage(z0 - 1, s1);
  fetch1(z0, s1);
  fetch2(z0, s2);
  for (int p = z0 - 1; p < z1; ++p) {
    // plane p + 2 has landed; the slot of plane p - 1 is free and receives plane p + 3
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (p + 3 <= z1 + 1) load_plane(p + 3);
    first_stage(p + 1, s1);
    if (p + 2 <= z1) fetch1(p + 2, s1);   // in flight during the barrier and the second stage
    __syncthreads();
    if (p >= z0) {
      second_stage(p, s2);
      if (p + 1 < z1) fetch2(p + 1, s2);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Runs in z: as many CTAs as fill whole waves of the resident CTAs (runs of at least 4 planes).
int zruns_for(int per_run, int nz, int resident) {
  int best = 1;
  double best_t = 1e300;
  for (int nr = 1; nr <= std::min(64, std::max(1, nz / 4)); ++nr) {
    const double waves = std::ceil((double)per_run * nr / std::max(resident, 1));
    const double t = waves * ((nz + nr - 1) / nr + 4.0);   // planes of the longest run and its prologue
    if (t < best_t) {
      best_t = t;
      best = nr;
    }
  }
  return best;
}

template <bool ADJ, bool SECOND>
cudaError_t launch_half(rsv_operator op, Half3D P) {
  // the shared-memory opt-in and the residency are per device, set up once under a lock
  static std::mutex mu;
  static int resident_dev[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  int resident = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 0 || dev >= 64 || resident_dev[dev] == 0) {
      cudaError_t e = cudaFuncSetAttribute(adv3d_half_kernel<ADJ, SECOND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kSmem);
      int per_sm = 0;
      if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, adv3d_half_kernel<ADJ, SECOND>, kThreads, kSmem);
      if (e != cudaSuccess) return e;
      resident = std::max(1, per_sm) * std::max(1, op->sm_count);
      if (dev >= 0 && dev < 64) resident_dev[dev] = resident;
    } else {
      resident = resident_dev[dev];
    }
  }
  const int ntx = (P.nx + kTX - 1) / kTX, nty = (P.ny + kTY - 1) / kTY;
  { const char* zr = getenv("RSV_ZR"); P.zruns = zr ? atoi(zr) : zruns_for(ntx * nty * P.kg, P.nz, resident); }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ntx * nty) * (unsigned)P.zruns * (unsigned)P.kg);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = op->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, adv3d_half_kernel<ADJ, SECOND>, P);
}

}  // namespace

// S steps of the 3-D kind, FP32; the state ping-pongs between its buffer and a second one.
cudaError_t step_march_3d(rsv_operator op, const MarchTile& t, void* state, const void* G, void* Y) {
  Half3D P = {};
  P.nx = op->nx;
  P.nxp = (op->nx + 3) / 4 * 4;
  P.ny = op->ny;
  P.nz = op->nz;
  P.kg = t.kg;
  P.vstride = (int64_t)3 * P.nxp * P.ny * P.nz;
  const float dx = (float)op->c_dx, dy = (float)op->c_dy, dz = (float)op->c_dz, nu = (float)op->visc;
  P.cdx = 0.5f / dx;
  P.nx2 = nu * (1.f / (dx * dx));
  P.ny2 = nu * (1.f / (dy * dy));
  P.nz2 = nu * (1.f / (dz * dz));
  P.f4 = (const float4*)op->fldp[4];
  P.U = (const float*)op->fldp[0];
  P.Ux = (const float*)op->fldp[1];
  P.Uy = (const float*)op->fldp[2];
  P.Uz = (const float*)op->fldp[3];
  const int64_t rows = (int64_t)t.kg * P.vstride;
  float* cur = static_cast<float*>(state);
  float* nxt = cur + rows;
  float* w2 = nxt + rows;
  const float h = (float)op->h;
  cudaError_t e = cudaSuccess;
  for (int s = 0; s < t.steps && e == cudaSuccess; ++s) {
    Half3D A = P;
    A.in = cur;
    A.out = w2;
    A.ysnap = (Y != nullptr && s >= t.y_first) ? static_cast<float*>(Y) + (size_t)s * rows : nullptr;
    A.f1 = h / 4.f;
    A.f2 = h / 3.f;
    Half3D B = P;
    B.in = w2;
    B.u = cur;
    B.g = (G != nullptr && t.n0 + s < t.n_forced) ? static_cast<const float*>(G) + (size_t)s * rows : nullptr;
    B.out = nxt;
    B.f1 = h / 2.f;
    B.f2 = h;
    e = t.adjoint ? launch_half<true, false>(op, A) : launch_half<false, false>(op, A);
    if (e == cudaSuccess) e = t.adjoint ? launch_half<true, true>(op, B) : launch_half<false, true>(op, B);
    std::swap(cur, nxt);
  }
  if (e == cudaSuccess && cur != static_cast<float*>(state))
    e = cudaMemcpyAsync(state, cur, sizeof(float) * rows, cudaMemcpyDeviceToDevice, op->stream);
  if (e == cudaSuccess) e = check_finite(op, state, rows, true);
  return e;
}

}  // namespace rsv
