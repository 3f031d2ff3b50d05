// 3-D kernels of the step form (see step2d.cu), FP32: two launches per step, two stages each.
//
//   half 1:  w1 = u + h/4 A u    on the tile + 1 halo cell in x, y (shared memory)
//            w2 = u + h/3 A w1   on the tile
//   half 2:  w3 = u + h/2 A w2   on the tile + 1 halo cell
//            u' = u + h A w3 + g on the tile
//
// A CTA owns a 64 x 12 tile in (x, y) of one vector and a run of planes in z, and streams through z.  A
// thread owns four consecutive x cells of one row of every plane: its own column of the planes below, at
// and above comes from registers, and only the y neighbours (16-byte loads) and the x neighbours at the
// ends of shuffles come from shared memory.  Nine warps evaluate the first stage (18 groups x 16 rows with
// the halo), six the second on the tile, two planes behind; the planes between them pass through a ring
// of three, one barrier per plane.  All operands arrive by 16-byte asynchronous copies issued a plane
// ahead; the base flow and u are copied once and read by both stages.  Both stages in the same threads
// (nine warps at 168 registers) were bound by the latency of 2.25 warps per scheduler: 162 us per step at
// 256 x 128 x 128; one cell per thread with scalar shared-memory operands took 143 us.
//
// Per step the state-sized arrays cross HBM six times (half 1: u read, w2 written, plus the snapshot on
// analysed steps; half 2: w2, u and g read, u' written) against eleven for the stage pairs with
// accumulator and forcing (stencil_kernels.cu).  Cells outside the grid hold zero (homogeneous Dirichlet).
//
// Rounding.  What is systematic in it acts like a change of the operator and adds up over a march, so the stage factors
// are formed in FP64 and rounded once, the diagonal is exactly minus the sum of the diffusion factors, advection is a
// difference of its own (added to the diffusion, it was rounded at its own size, and rows of the operator kept a rest
// of 1e-8 per step), and the last stage adds one rounded increment to u, as a stage-time march does.  Error against
// FP64, contractions on the CUDA cores: 128 x 64 x 64 over four windows of 643 steps 2e-7 (3e-7 by the stage-time
// kernels, 6e-7 with merged factors), leading gains of 256 x 128 x 128 2.5e-6 (2.5e-6, 5.4e-6).  It costs 1.6% of
// the march, two additions per value and stage.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "rsv_ops.h"

namespace rsv {
namespace {

constexpr int kTX = 64, kTY = 12;
constexpr int kGX = kTX / 4 + 2, kRY = kTY + 4;   // groups of a row with the halo, rows with the halo
constexpr int kT1 = kGX * kRY;                    // first-stage threads (288)
constexpr int kT2 = kTX / 4 * kTY;                // second-stage threads (192)
constexpr int kThreads = kT1 + kT2;
constexpr int kMidRing = 3, kFlowRing = 4, kGRing = 2;
constexpr int in_ring(bool second) { return second ? 3 : 5; }   // half 1's second stage reads u from it
constexpr size_t half_smem(bool second) {
  return sizeof(float4) * (kT1 * (size_t)(3 * in_ring(second) + 3 * kMidRing + 4 * kFlowRing + (second ? 3 * kFlowRing : 0)) +
                           (second ? (size_t)kT2 * 3 * kGRing : 0));
}
static_assert(half_smem(true) <= 232448 && half_smem(false) <= 232448, "3-D rings exceed the shared memory of a CTA");

// Factors of one stage, formed in FP64 from f = h / m and rounded once: a relative error of them acts like one of
// the operator itself, and adds up over a march.  d is exactly minus twice the sum of x, y and z: what is missing
// there acts as damping or growth, all the longer the slower the flow.
struct Stage3D {
  float f, x, y, z, c, d;     // f; f visc / dx^2, ... / dy^2, ... / dz^2; f / (2 dx); -2 (x + y + z)
};

struct Half3D {
  int nx, nxp, ny, nz, kg, zruns;
  int64_t vstride;            // 3 * nxp * ny * nz
  const float *U, *Ux, *Uy, *Uz;   // base flow, rows padded to nxp
  const float* in;            // u (half 1) or w2 (half 2)
  const float* u;             // half 2: u
  const float* g;             // half 2: g_n (nullable)
  float* out;                 // w2 or u'
  float* ysnap;               // half 1: snapshot of u (nullable)
  Stage3D s1, s2;             // the two stages
};

struct V4 {
  float v[4];
};
__device__ __forceinline__ V4 zero4() {
  V4 o;
  o.v[0] = o.v[1] = o.v[2] = o.v[3] = 0.f;
  return o;
}
__device__ __forceinline__ V4 v4(float4 x) {
  V4 o;
  o.v[0] = x.x;
  o.v[1] = x.y;
  o.v[2] = x.z;
  o.v[3] = x.w;
  return o;
}
__device__ __forceinline__ float4 f4(const V4& x) { return make_float4(x.v[0], x.v[1], x.v[2], x.v[3]); }
struct C3 {
  V4 c[3];
};
// Base flow of a group: U with its two x neighbours (transposed advection), gradient.
struct Flow {
  V4 U, Ux, Uy, Uz;
  float Ul, Ur;
};

// u0 + f A x of one group (INC: f A x, so that the increment is rounded before it meets the state): below, centre
// and above in registers, rows so and no from shared memory, the cells l and r beside the group.
template <bool ADJ, bool INC>
__device__ __forceinline__ void stage3d(const Stage3D& S, const C3& xb, const C3& xc, const C3& xt,
                                        const float4 so[3], const float4 no[3], const float l[3], const float r[3],
                                        const Flow& w, const C3& u0, C3& o) {
  const float f = S.f;
  float au[4];   // advection, apart from the diffusion: added up, the two would be rounded at the size of the larger
#pragma unroll
  for (int k = 0; k < 4; ++k) au[k] = S.c * w.U.v[k];
  const float al = S.c * w.Ul, ar = S.c * w.Ur;   // transposed only
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const V4 s = v4(so[c]), n = v4(no[c]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float we = k == 0 ? l[c] : xc.c[c].v[k - 1], ea = k == 3 ? r[c] : xc.c[c].v[k + 1];
      const float zz = xb.c[c].v[k] + xt.c[c].v[k];
      float a = INC ? S.z * zz : fmaf(S.z, zz, u0.c[c].v[k]);
      a = fmaf(S.y, s.v[k] + n.v[k], a);
      a = fmaf(S.x, we + ea, a);
      a = fmaf(S.d, xc.c[c].v[k], a);
      if (ADJ) {
        a = fmaf(-(k == 0 ? al : au[k - 1]), we, a);
        o.c[c].v[k] = fmaf(k == 3 ? ar : au[k + 1], ea, a);
      } else {
        o.c[c].v[k] = fmaf(au[k], we - ea, a);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (ADJ) {
      const float fx0 = -f * xc.c[0].v[k];
      o.c[0].v[k] = fmaf(w.Ux.v[k], fx0, o.c[0].v[k]);
      o.c[1].v[k] = fmaf(w.Uy.v[k], fx0, o.c[1].v[k]);
      o.c[2].v[k] = fmaf(w.Uz.v[k], fx0, o.c[2].v[k]);
    } else {
      const float d = fmaf(w.Ux.v[k], xc.c[0].v[k], fmaf(w.Uy.v[k], xc.c[1].v[k], w.Uz.v[k] * xc.c[2].v[k]));
      o.c[0].v[k] = fmaf(-f, d, o.c[0].v[k]);
    }
  }
}

// Copies 16 bytes, or writes zeros without reading.
__device__ __forceinline__ void cp16_zfill(float4* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void plane_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory"); }

template <bool ADJ, bool SECOND>
__global__ void __launch_bounds__(kThreads, 1) adv3d_half_kernel(Half3D P) {
  constexpr int kIn = in_ring(SECOND);
  extern __shared__ __align__(16) float4 smem_raw[];
  // rings of planes, one slot per first-stage thread
  float4 (*s_in)[3][kT1] = reinterpret_cast<float4 (*)[3][kT1]>(smem_raw);          // [kIn] input
  float4 (*s_mid)[3][kT1] = s_in + kIn;                                             // [kMidRing] first stage's result
  float4 (*s_w)[4][kT1] = reinterpret_cast<float4 (*)[4][kT1]>(s_mid + kMidRing);   // [kFlowRing] base flow
  float4 (*s_u)[3][kT1] = reinterpret_cast<float4 (*)[3][kT1]>(s_w + kFlowRing);    // [kFlowRing] half 2: u
  float4 (*s_g)[3][kT2] = reinterpret_cast<float4 (*)[3][kT2]>(s_u + kFlowRing);    // [kGRing] half 2: g
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
  const bool second = threadIdx.x >= kT1;              // this thread's stage
  const int t2 = threadIdx.x - kT1, lane = threadIdx.x & 31;
  const int gx = second ? t2 % (kTX / 4) + 1 : threadIdx.x % kGX, ry = second ? t2 / (kTX / 4) + 2 : threadIdx.x / kGX;
  const int at = ry * kGX + gx;                        // the group's slot in the planes
  const int x = X0 - 4 + 4 * gx, y = Y0 - 2 + ry;
  const bool in_xy = x >= 0 && x < P.nxp && y >= 0 && y < ny;
  const int xy = in_xy ? y * P.nxp + x : 0;
  bool cell[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) cell[c] = in_xy && x + c < nx;
  const bool inner = X0 >= 4 && X0 + kTX + 4 <= nx && Y0 >= 2 && Y0 + kTY + 2 <= ny;   // no cell of the tile outside
  // launched as a programmatic dependent: resident early, waits here before any memory access
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  auto in_z = [&](int kz) { return kz >= 0 && kz < nz; };
  auto get3 = [&](const float4 (*s)[kT1]) -> C3 {
    C3 r;
#pragma unroll
    for (int c = 0; c < 3; ++c) r.c[c] = v4(s[c][at]);
    return r;
  };
  auto get_w = [&](const float4 (*s)[kT1]) -> Flow {
    Flow w;
    w.U = v4(s[0][at]);
    w.Ux = v4(s[1][at]);
    w.Uy = v4(s[2][at]);
    w.Uz = v4(s[3][at]);
    w.Ul = w.Ur = 0.f;
    return w;
  };
  // neighbours of the thread's group in plane s: rows beside it (row 0 and the last one: results unused) and
  // cells beside it, from the neighbouring lanes where they hold them
  const int up = ry + 1 < kRY ? at + kGX : at, dn = ry > 0 ? at - kGX : at;
  const bool edge_l = second ? gx == 1 || lane == 0 : lane == 0, edge_r = second ? gx == kTX / 4 || lane == 31 : lane == 31;
  auto around = [&](const float4 (*s)[kT1], const C3& xc, float4 so[3], float4 no[3], float l[3], float r[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      so[c] = s[c][dn];
      no[c] = s[c][up];
      l[c] = __shfl_up_sync(0xffffffffu, xc.c[c].v[3], 1);
      r[c] = __shfl_down_sync(0xffffffffu, xc.c[c].v[0], 1);
      if (edge_l) l[c] = at > 0 ? s[c][at - 1].w : 0.f;
      if (edge_r) r[c] = at + 1 < kT1 ? s[c][at + 1].x : 0.f;
    }
  };
  const C3 zero = {{zero4(), zero4(), zero4()}};
  // Iteration i = z0 - 1 .. z1 + 1: the first stage on plane i (to z1), the second on plane i - 2 (from z0).
  // Ring slots of plane k: (k - z0 + 2) mod the ring's length, kept as running indices.
  const int last = z1 + 1;
  if (!second) {
    const float* in = P.in + base + xy;
    const float* pu = SECOND ? P.u + base + xy : nullptr;
    auto copy3 = [&](float4 (*s)[kT1], const float* p, int kz, bool ok) {
#pragma unroll
      for (int c = 0; c < 3; ++c) cp16_zfill(&s[c][at], ok ? p + c * ncell + kz * plane : P.in, ok);
    };
    auto copy_in = [&](int kz, int slot) { copy3(s_in[slot], in, kz, in_xy && in_z(kz) && kz <= z1 + 1); };
    auto copy_wu = [&](int kz, int slot) {
      const bool ok = in_xy && in_z(kz) && kz <= z1;
      const int64_t q = ok ? kz * plane + xy : 0;
      cp16_zfill(&s_w[slot][0][at], P.U + q, ok);
      cp16_zfill(&s_w[slot][1][at], P.Ux + q, ok);
      cp16_zfill(&s_w[slot][2][at], P.Uy + q, ok);
      cp16_zfill(&s_w[slot][3][at], P.Uz + q, ok);
      if (SECOND) copy3(s_u[slot], pu, kz, ok);
    };
    // planes z0 - 2 .. z0 of the input and plane z0 - 1 of the rest; slot of plane z0 - 2 + k is k
    copy_in(z0 - 2, 0);
    copy_in(z0 - 1, 1);
    copy_in(z0, 2);
    copy_wu(z0 - 1, 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    C3 xin[3];
    xin[0] = get3(s_in[0]);
    xin[1] = get3(s_in[1]);
    plane_barrier();
    int si = 1, sm = 1, sw = 1;    // slots of plane i in the input, result and flow rings
    for (int i0 = z0 - 1; i0 <= last; i0 += 3) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int i = i0 + q;        // planes i - 1, i, i + 1 in xin[q], xin[q + 1], xin[q + 2]
        if (i > last) break;
        if (i <= z1) {
          asm volatile("cp.async.wait_group 0;" ::: "memory");
          const int sn = si + 1 < kIn ? si + 1 : 0, sn2 = sn + 1 < kIn ? sn + 1 : 0;   // planes i + 1, i + 2
          const int wn = sw + 1 < kFlowRing ? sw + 1 : 0;
          xin[(q + 2) % 3] = get3(s_in[sn]);
          copy_in(i + 2, sn2);
          copy_wu(i + 1, wn);
          asm volatile("cp.async.commit_group;" ::: "memory");
          const C3& c = xin[(q + 1) % 3];
          float4 so[3], no[3];
          float l[3], r[3];
          around(s_in[si], c, so, no, l, r);
          C3 o;
          Flow w = get_w(s_w[sw]);
          if (ADJ) {   // U of the x neighbours: this plane's copies of other warps may still be on their way
            w.Ul = __shfl_up_sync(0xffffffffu, w.U.v[3], 1);
            w.Ur = __shfl_down_sync(0xffffffffu, w.U.v[0], 1);
            const bool ok = in_xy && in_z(i);
            if (lane == 0) w.Ul = ok && x > 0 ? __ldg(P.U + i * plane + xy - 1) : 0.f;
            if (lane == 31) w.Ur = ok && x + 4 < P.nxp ? __ldg(P.U + i * plane + xy + 4) : 0.f;
          }
          stage3d<ADJ, false>(P.s1, xin[q], c, xin[(q + 2) % 3], so, no, l, r, w, SECOND ? get3(s_u[sw]) : c, o);
          if (!inner || !in_z(i)) {
            const bool zin = in_z(i);
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
              for (int e = 0; e < 4; ++e) o.c[k].v[e] = zin && cell[e] ? o.c[k].v[e] : 0.f;
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) s_mid[sm][k][at] = f4(o.c[k]);
          si = sn;
          sw = wn;
          sm = sm + 1 < kMidRing ? sm + 1 : 0;
        }
        plane_barrier();
      }
    }
  } else {
    float* out = P.out + base + xy;
    float* ysnap = !SECOND && P.ysnap ? P.ysnap + base + xy : nullptr;
    const float* pg = SECOND && P.g ? P.g + base + xy : nullptr;
    auto copy_g = [&](int kz) {
      if (SECOND) {
        const bool ok = in_xy && pg != nullptr && kz >= z0 && kz < z1;
#pragma unroll
        for (int c = 0; c < 3; ++c) cp16_zfill(&s_g[kz & 1][c][t2], ok ? pg + c * ncell + kz * plane : P.in, ok);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    copy_g(z0);
    C3 mid[3] = {zero, zero, zero};
    plane_barrier();
    // slots of plane i - 2 in the result, flow and input rings, of plane i - 1 in the result ring
    int sm = kMidRing - 1, sw = kFlowRing - 1, si = kIn - 1;
    for (int i0 = z0 - 1; i0 <= last; i0 += 3) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int i = i0 + q;        // planes i - 3, i - 2, i - 1 of the first stage's result in mid[q], mid[q + 1], mid[q + 2]
        if (i > last) break;
        const int sm1 = sm + 1 < kMidRing ? sm + 1 : 0;
        if (i >= z0) mid[(q + 2) % 3] = get3(s_mid[sm1]);
        const int k2 = i - 2;
        if (k2 >= z0) {
          asm volatile("cp.async.wait_group 0;" ::: "memory");
          const C3& c = mid[(q + 1) % 3];
          float4 so[3], no[3];
          float l[3], r[3];
          around(s_mid[sm], c, so, no, l, r);
          const C3 u0 = SECOND ? get3(s_u[sw]) : get3(s_in[si]);
          C3 o;
          Flow w = get_w(s_w[sw]);
          if (ADJ) {
            w.Ul = s_w[sw][0][at - 1].w;
            w.Ur = s_w[sw][0][at + 1].x;
          }
          stage3d<ADJ, SECOND>(P.s2, mid[q], c, mid[(q + 2) % 3], so, no, l, r, w, u0, o);
          if (in_xy) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              V4 gv = zero4();
              if (SECOND) gv = v4(s_g[k2 & 1][k][t2]);
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                if (SECOND) o.c[k].v[e] = u0.c[k].v[e] + (o.c[k].v[e] + gv.v[e]);
                if (!inner) o.c[k].v[e] = cell[e] ? o.c[k].v[e] : 0.f;
              }
              *reinterpret_cast<float4*>(out + k * ncell + k2 * plane) = f4(o.c[k]);
              if (!SECOND && ysnap) __stcs(reinterpret_cast<float4*>(ysnap + k * ncell + k2 * plane), f4(u0.c[k]));
            }
          }
          copy_g(k2 + 1);
        }
        sm = sm1;
        sw = sw + 1 < kFlowRing ? sw + 1 : 0;
        si = si + 1 < kIn ? si + 1 : 0;
        plane_barrier();
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Runs in z for the least planes of work on one SM (one CTA each), runs of at least 4 planes.
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
cudaError_t launch_half(rsv_operator op, const Half3D& P) {
  const int ntx = (P.nx + kTX - 1) / kTX, nty = (P.ny + kTY - 1) / kTY;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ntx * nty) * (unsigned)P.zruns * (unsigned)P.kg);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = half_smem(SECOND);
  cfg.stream = op->stream;
  cudaError_t e = cudaFuncSetAttribute(adv3d_half_kernel<ADJ, SECOND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)half_smem(SECOND));
  if (e != cudaSuccess) return e;
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
  auto factors = [&](double f) {
    const double x = f * op->visc / (op->c_dx * op->c_dx), y = f * op->visc / (op->c_dy * op->c_dy),
                 z = f * op->visc / (op->c_dz * op->c_dz), sum = x + y + z;
    // the diffusion factors on the FP32 grid of their sum (at most 2e-7 off for like spacings), so that it is exact
    const double unit = sum > 0.0 ? std::ldexp(1.0, std::ilogb(sum) - 23) : 1.0;
    auto on_grid = [&](double v) { return (float)(unit * std::nearbyint(v / unit)); };
    const float fx = on_grid(x), fy = on_grid(y), fz = on_grid(z);
    return Stage3D{(float)f, fx, fy, fz, (float)(0.5 * f / op->c_dx), -2.f * (fx + fy + fz)};
  };
  const Stage3D st[4] = {factors(op->h / 4), factors(op->h / 3), factors(op->h / 2), factors(op->h)};
  P.U = (const float*)op->fldp[0];
  P.Ux = (const float*)op->fldp[1];
  P.Uy = (const float*)op->fldp[2];
  P.Uz = (const float*)op->fldp[3];
  P.zruns = zruns_for(((P.nx + kTX - 1) / kTX) * ((P.ny + kTY - 1) / kTY) * P.kg, P.nz, std::max(1, op->sm_count));
  const int64_t rows = (int64_t)t.kg * P.vstride;
  float* cur = static_cast<float*>(state);
  float* nxt = cur + rows;
  float* w2 = nxt + rows;
  cudaError_t e = cudaSuccess;
  for (int s = 0; s < t.steps && e == cudaSuccess; ++s) {
    Half3D A = P;
    A.in = cur;
    A.out = w2;
    A.ysnap = (Y != nullptr && s >= t.y_first) ? static_cast<float*>(Y) + (size_t)s * rows : nullptr;
    A.s1 = st[0];
    A.s2 = st[1];
    Half3D B = P;
    B.in = w2;
    B.u = cur;
    B.g = (G != nullptr && t.n0 + s < t.n_forced) ? static_cast<const float*>(G) + (size_t)s * rows : nullptr;
    B.out = nxt;
    B.s1 = st[2];
    B.s2 = st[3];
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
