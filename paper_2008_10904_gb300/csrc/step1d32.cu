// Step form (see step2d.cu) of FP32 RK4 marches of the 1-D kind: (instance, vector) segments packed into
// CTAs, four contiguous points per lane.
//
//   w1 = u + h/4 A u,  w2 = u + h/3 A w1,  w3 = u + h/2 A w2,  u' = u + h A w3 + g_n
//
// A pack is a run of slots: segments start on multiples of four slots and are followed by at least one
// empty slot, which holds zero (the Dirichlet ends).  A warp owns 120 slots and evaluates 128 (lanes 0 and
// 31 are halos of four slots, one per stage): the four stages of a step exchange neighbours by shuffles
// only, and once per step the warps' edge points pass through shared memory (one barrier; none in a pack of
// one warp).  A lane's points belong to one segment, whose off-diagonal couplings are constant, so the
// coefficients take 12 registers.  The forcing arrives kRing - 1 steps ahead through a ring of asynchronous
// copies.  The tiles (forcing, snapshots, transformed coefficients, accumulators) keep the packs' slot
// order, so that every access is a 16-byte one and the contractions always take their pipelined kernel.
// One forcing per step instead of stage times halves the forcing tile and its synthesis.  FP32 issue bounds
// it (about 62 multiply-adds per point and step, issue 49% with one CTA per SM and one barrier per step): 64
// instances of 256 to 2048 points, 8 vectors, 10822 steps march in 25.4 ms and are synthesised in 8.3 ms; one
// stage per barrier, a point per thread and three forcings per step took 44.7 and 16.7 ms.
#include <algorithm>
#include <cstdlib>
#include <functional>
#include <queue>
#include <utility>
#include <vector>

#include "rsv_ops.h"

namespace rsv {
namespace {

using cf = cpx<float>;

constexpr int kOwn = 120;                  // slots owned by a warp
constexpr int kMaxWarps = 32;
constexpr int kMaxSlots = kMaxWarps * kOwn;
constexpr int kRing = 4;                   // steps of forcing in shared memory, kRing - 1 ahead

struct Step32 {
  const cf* lo;
  const cf* di;
  const cf* up;
  const int64_t* inst_off;
  const int32_t* inst_of_point;
  const int32_t* off;         // [packs + 1]: first slot of each pack, multiples of 4
  const int32_t* first;       // [slots / 4]: row of the group's first point, -1 for an empty group
  int64_t rows;               // slots of all packs
  int64_t n;                  // points per vector
  float h;
  int steps;
  int64_t n0, n_forced;
  int y_first;
};

__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__global__ void __launch_bounds__(32 * kMaxWarps, 1) gl1d_step32_kernel(Step32 P, cf* __restrict__ u,
                                                                       const cf* __restrict__ G, cf* __restrict__ Y,
                                                                       int* __restrict__ flag) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  // per warp: forcing ring [kRing][30 lanes x 32 bytes], then the edges [2][warps][2][4]
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem_raw) + (uint32_t)warp * (kRing * kOwn * 8);
  const unsigned char* ring_p = smem_raw + (size_t)warp * (kRing * kOwn * 8);
  float4* edge = reinterpret_cast<float4*>(smem_raw + (size_t)warps * (kRing * kOwn * 8));
  const int slot = warp * kOwn - 4 + 4 * lane;                 // the lane's first slot
  const bool own = lane >= 1 && lane <= 30;
  const int32_t off = P.off[blockIdx.x];
  const bool inside = slot >= 0 && slot < P.off[blockIdx.x + 1] - off;
  const int32_t row = inside ? P.first[(off + slot) / 4] : -1;
  cf x[4], lo, up, di[4];
  float f[4];                                                    // h inside the segment, 0 outside
  const cf zero = mk<float>(0.f, 0.f);
  lo = up = zero;
  const int64_t base = (int64_t)off + slot;   // the lane's row of the tiles
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    x[c] = di[c] = zero;
    f[c] = 0.f;
  }
  if (row >= 0) {
    const int64_t p = row % P.n;
    const int inst = P.inst_of_point[p];
    const int64_t a = P.inst_off[inst], b = P.inst_off[inst + 1];
    lo = P.lo[b - 1];                                            // constant but for the zero at the first point
    up = P.up[a];                                                // ... and at the last one
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (p + c >= b) break;
      di[c] = P.di[p + c];
      f[c] = P.h;
      x[c] = u[base + c];
    }
  }
  const float2* Gp = reinterpret_cast<const float2*>(G) + base;
  auto prefetch = [&](int s) {   // the forcing of step s
    if (s < P.steps && G != nullptr && P.n0 + s < P.n_forced && own && inside) {
      const float2* src = Gp + (int64_t)s * P.rows;
      const uint32_t dst = ring + (uint32_t)(s & (kRing - 1)) * (kOwn * 8) + (uint32_t)(lane - 1) * 32;
      cp16(dst, src);
      cp16(dst + 16, src + 2);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < kRing - 1; ++s) prefetch(s);
  // w = x + f A v (f = h / m inside the segment)
  auto stage = [&](const cf v[4], float m, cf w[4]) {
    cf l, r;
    l.re = __shfl_up_sync(0xffffffffu, v[3].re, 1);
    l.im = __shfl_up_sync(0xffffffffu, v[3].im, 1);
    r.re = __shfl_down_sync(0xffffffffu, v[0].re, 1);
    r.im = __shfl_down_sync(0xffffffffu, v[0].im, 1);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      cf a = di[c] * v[c];
      cfma(a, lo, c == 0 ? l : v[c - 1]);
      cfma(a, up, c == 3 ? r : v[c + 1]);
      const float ff = f[c] * m;
      w[c] = mk<float>(fmaf(ff, a.re, x[c].re), fmaf(ff, a.im, x[c].im));
    }
  };
  for (int s = 0; s < P.steps; ++s) {
    prefetch(s + kRing - 1);   // into the entry of step s - 1, whose values are consumed
    if (warps > 1) {           // halos: the neighbouring warps' first and last owned points
      float4* e = edge + (size_t)(s & 1) * warps * 4;
      if (lane == 1 || lane == 30) {
        float4* d = e + warp * 4 + (lane == 30 ? 2 : 0);
        d[0] = make_float4(x[0].re, x[0].im, x[1].re, x[1].im);
        d[1] = make_float4(x[2].re, x[2].im, x[3].re, x[3].im);
      }
      __syncthreads();
      const int nb = lane == 0 ? warp - 1 : lane == 31 ? warp + 1 : -1;
      if (nb >= 0 && nb < warps) {
        const float4* q = e + nb * 4 + (lane == 0 ? 2 : 0);
        const float4 v0 = q[0], v1 = q[1];
        x[0] = mk<float>(v0.x, v0.y);
        x[1] = mk<float>(v0.z, v0.w);
        x[2] = mk<float>(v1.x, v1.y);
        x[3] = mk<float>(v1.z, v1.w);
      }
    }
    if (Y != nullptr && s >= P.y_first && own && inside) {
      float4* y = reinterpret_cast<float4*>(Y + (int64_t)s * P.rows + base);
      __stcs(y, make_float4(x[0].re, x[0].im, x[1].re, x[1].im));
      __stcs(y + 1, make_float4(x[2].re, x[2].im, x[3].re, x[3].im));
    }
    cf w[4], v[4];
    stage(x, 0.25f, w);
    stage(w, 1.f / 3.f, v);
    stage(v, 0.5f, w);
    stage(w, 1.f, v);
    asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 1) : "memory");   // this lane's step-s copies landed
    float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), g1 = g0;
    if (G != nullptr && P.n0 + s < P.n_forced && own && inside) {
      const float4* q = reinterpret_cast<const float4*>(ring_p + (size_t)(s & (kRing - 1)) * (kOwn * 8) + (lane - 1) * 32);
      g0 = q[0];
      g1 = q[1];
    }
    x[0] = mk<float>(v[0].re + g0.x, v[0].im + g0.y);
    x[1] = mk<float>(v[1].re + g0.z, v[1].im + g0.w);
    x[2] = mk<float>(v[2].re + g1.x, v[2].im + g1.y);
    x[3] = mk<float>(v[3].re + g1.z, v[3].im + g1.w);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (own && inside) {
    bool bad = false;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      u[base + c] = x[c];
      const double q = (double)x[c].re * (double)x[c].re + (double)x[c].im * (double)x[c].im;
      bad = bad || !(q < 1e300);
    }
    if (bad) atomicExch(flag, 1);   // NaN or overflow
  }
}

// c_j = (h/6) [(1 + 4 s + z) + (1 + 2 s) B + (1 + s)/2 B^2 + 1/4 B^3] f_j of one row per thread (the row's seven
// neighbours from L1), into its slot.
__global__ void __launch_bounds__(256) coef32_kernel(Step32 P, int64_t rows, const int32_t* __restrict__ slot_of_row,
                                                     const cf* __restrict__ f, int64_t f_stride, cf* __restrict__ out,
                                                     const cf* __restrict__ tw, const int64_t* __restrict__ pj, int sgn,
                                                     int64_t m4) {
  __shared__ cf co[3];
  const int j = blockIdx.y;
  if (threadIdx.x == 0) {
    const cf s = tw[phase_index(sgn * pj[j], 1, m4)], z = tw[phase_index(sgn * pj[j], 2, m4)];
    co[0] = mk<float>(1.f + 4.f * s.re + z.re, 4.f * s.im + z.im);
    co[1] = mk<float>(1.f + 2.f * s.re, 2.f * s.im);
    co[2] = mk<float>(0.5f + 0.5f * s.re, 0.5f * s.im);
  }
  __syncthreads();
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= rows) return;
  const int64_t p = r % P.n;
  const int inst = P.inst_of_point[p];
  const int64_t a = P.inst_off[inst] - p, b = P.inst_off[inst + 1] - p;   // the segment relative to the row
  const cf* x = f + (int64_t)j * f_stride + r;
  const cf zero = mk<float>(0.f, 0.f);
  cf v[7], t[7];
#pragma unroll
  for (int d = -3; d <= 3; ++d) v[d + 3] = t[d + 3] = (d >= a && d < b) ? x[d] : zero;
  // t <- a f + c B t on a window shrinking by one point per side: c = 1/4, 1, 1
#pragma unroll
  for (int k = 2; k >= 0; --k) {
    cf w[7];
#pragma unroll
    for (int d = -3; d <= 3; ++d) w[d + 3] = zero;
#pragma unroll
    for (int d = -2; d <= 2; ++d) {
      if (d < -k || d > k || d < a || d >= b) continue;
      cf e = P.di[p + d] * t[d + 3];
      cfma(e, P.lo[p + d], t[d + 2]);
      cfma(e, P.up[p + d], t[d + 4]);
      w[d + 3] = co[k] * v[d + 3] + (k == 2 ? 0.25f * P.h : P.h) * e;
    }
#pragma unroll
    for (int d = 0; d < 7; ++d) t[d] = w[d];
  }
  out[(int64_t)j * P.rows + slot_of_row[r]] = (P.h / 6.f) * t[3];
}

__global__ void slot_sumsq_kernel(const cf* __restrict__ u, const int32_t* __restrict__ slot_of_row, int64_t n,
                                  double* __restrict__ out) {
  double acc = 0.0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const cf x = u[slot_of_row[(int64_t)blockIdx.y * n + p]];
    acc += (double)x.re * (double)x.re + (double)x.im * (double)x.im;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  __shared__ double part[8];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
    atomicAdd(out + blockIdx.y, t);
  }
}

size_t step32_smem(int warps) { return (size_t)warps * (kRing * kOwn * 8 + 2 * 4 * sizeof(float4)); }

struct Seg {
  int64_t len;
  int inst, v;
};
int64_t up4(int64_t x) { return (x + 3) / 4 * 4; }

// Segments, longest first, each to the least loaded of n_bins packs of cap slots; load: the next free start.
bool fill_packs(const std::vector<Seg>& segs, int64_t cap, int n_bins, std::vector<std::vector<Seg>>& packs) {
  using Load = std::pair<int64_t, int>;
  std::priority_queue<Load, std::vector<Load>, std::greater<Load>> heap;
  packs.assign((size_t)n_bins, {});
  for (int b = 0; b < n_bins; ++b) heap.push({0, b});
  for (const Seg& s : segs) {
    const Load top = heap.top();
    if (top.first + s.len > cap) return false;
    heap.pop();
    packs[(size_t)top.second].push_back(s);
    heap.push({up4(top.first + s.len + 1), top.second});
  }
  packs.erase(std::remove_if(packs.begin(), packs.end(), [](const std::vector<Seg>& p) { return p.empty(); }), packs.end());
  return true;
}

Step32 geom32(rsv_operator op, bool adjoint) {
  Step32 g = {};
  const int b = adjoint ? 3 : 0;
  g.lo = (const cf*)op->tri[b];
  g.di = (const cf*)op->tri[b + 1];
  g.up = (const cf*)op->tri[b + 2];
  g.inst_off = (const int64_t*)op->d_inst_off;
  g.inst_of_point = (const int32_t*)op->d_inst_of_point;
  g.off = (const int32_t*)op->p32.off;
  g.first = (const int32_t*)op->p32.first;
  g.rows = op->p32.slots;
  g.n = op->n;
  g.h = (float)op->h;
  return g;
}

}  // namespace

// FP32 RK4 marches of instances that fit a pack.
bool step32_taken(rsv_operator op, int k) {
  return op->kind == RSV_OP_GL1D && op->prec == RSV_PREC_FP32 && op->scheme == RSV_SCHEME_RK4 &&
         op->gl_max_n <= kMaxSlots && (int64_t)k * op->n < ((int64_t)1 << 29) && k <= 65535;
}

// Packs of the kg vectors of a group (kept until another group size comes).  As many pairs as SMs or fewer:
// one per pack.  More: packs of 1024 q slots (q = 1 to 4, at least the longest instance), the q whose packs
// fill the fewest waves of resident CTAs, the smaller on a tie.  RSV_GL1D_PPT forces q; RSV_GL1D_PACK=0
// keeps one pair per pack.
rsv_status step32_packs(rsv_operator op, int kg) {
  Pack32& P = op->p32;
  if (P.kg == kg) return RSV_OK;
  std::vector<Seg> segs;
  int64_t slots = 0;
  for (int v = 0; v < kg; ++v)
    for (int i = 0; i < op->n_inst; ++i) {
      segs.push_back({op->inst_len[i], i, v});
      slots += up4(op->inst_len[i] + 1);
    }
  std::stable_sort(segs.begin(), segs.end(), [](const Seg& a, const Seg& b) { return a.len > b.len; });
  std::vector<std::vector<Seg>> packs;
  int q_best = 0, wave = 0;
  const char* ep = getenv("RSV_GL1D_PACK");
  if (op->n_inst == 1 || (int64_t)segs.size() <= op->sm_count || (ep != nullptr && ep[0] == '0')) {
    for (const Seg& s : segs) packs.push_back({s});
  } else {
    const char* env = getenv("RSV_GL1D_PPT");
    const int q_min = (op->gl_max_n + 1023) / 1024, forced = env ? atoi(env) : 0;
    const bool force = forced >= q_min && forced <= 4;
    int64_t best_waves = 0;
    for (int q = force ? forced : q_min; q <= (force ? forced : 4); ++q) {
      const int64_t cap = std::min<int64_t>(1024 * q, kMaxSlots);
      int per_sm = 0;
      const int warps = (int)((cap + kOwn - 1) / kOwn);
      cudaError_t e = cudaFuncSetAttribute(gl1d_step32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)step32_smem(kMaxWarps));
      if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gl1d_step32_kernel, 32 * warps, step32_smem(warps));
      if (e != cudaSuccess) return cuda_fail(e, "pack occupancy");
      const int wave_q = op->sm_count * std::max(1, per_sm);
      std::vector<std::vector<Seg>> pk;
      int64_t waves = std::max<int64_t>(1, (slots + wave_q * cap - 1) / (wave_q * cap));
      while (!fill_packs(segs, cap, (int)(waves * wave_q), pk)) ++waves;   // ends: one segment per pack fits
      if (q_best == 0 || waves < best_waves) {
        q_best = q;
        wave = wave_q;
        best_waves = waves;
        packs.swap(pk);
      }
    }
  }
  // one host block: slot of each row, row of each group of four slots, first slot of each pack
  const int64_t rows = (int64_t)kg * op->n;
  std::vector<int32_t> slot(rows), first, off;
  int64_t widest = 0;
  for (const auto& pk : packs) {
    const int64_t base = (int64_t)first.size() * 4;
    int64_t pos = 0;
    off.push_back((int32_t)base);
    for (const Seg& s : pk) {
      const int64_t r0 = (int64_t)s.v * op->n + op->inst_off[s.inst];
      first.resize((size_t)(base + pos) / 4, -1);
      for (int64_t j = 0; j < s.len; ++j) {
        slot[r0 + j] = (int32_t)(base + pos + j);
        if (j % 4 == 0) first.push_back((int32_t)(r0 + j));
      }
      pos = up4(pos + s.len + 1);
    }
    widest = std::max(widest, (int64_t)first.size() * 4 - base);
  }
  off.push_back((int32_t)(first.size() * 4));
  const size_t n_slot = slot.size(), n_first = first.size();
  slot.insert(slot.end(), first.begin(), first.end());
  slot.insert(slot.end(), off.begin(), off.end());
  P.kg = 0;
  rsv_status st = ensure(op->ws_p32, slot.size() * sizeof(int32_t));
  if (st != RSV_OK) return st;
  int32_t* d = static_cast<int32_t*>(op->ws_p32.ptr);
  cudaError_t e = cudaMemcpyAsync(d, slot.data(), slot.size() * sizeof(int32_t), cudaMemcpyHostToDevice, op->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(op->stream);   // the host block goes out of scope
  if (e != cudaSuccess) return cuda_fail(e, "packs");
  P.kg = kg;
  P.packs = (int)packs.size();
  P.warps = (int)((widest + kOwn - 1) / kOwn);
  P.slots = (int64_t)n_first * 4;
  P.q = q_best;
  P.wave = wave;
  P.slot = d;
  P.first = d + n_slot;
  P.off = d + n_slot + n_first;
  return RSV_OK;
}

rsv_status step32_coefficients(rsv_operator op, const void* fhat, int64_t f_stride, int kg, bool adjoint, void* out) {
  const Step32 g = geom32(op, adjoint);
  const int64_t rows = (int64_t)kg * op->n;
  cudaError_t e = cudaMemsetAsync(out, 0, (size_t)op->n_omega * g.rows * sizeof(cf), op->stream);   // empty slots
  if (e == cudaSuccess) {
    coef32_kernel<<<dim3((unsigned)((rows + 255) / 256), (unsigned)op->n_omega), 256, 0, op->stream>>>(
        g, rows, (const int32_t*)op->p32.slot, (const cf*)fhat, f_stride, (cf*)out, (const cf*)op->d_tw, op->d_pj,
        adjoint ? -1 : 1, 4 * op->n_t);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? RSV_OK : cuda_fail(e, "forcing transform");
}

cudaError_t step_march_1d32(rsv_operator op, const MarchTile& t, void* state, const void* G, void* Y) {
  Step32 g = geom32(op, t.adjoint);
  g.steps = t.steps;
  g.n0 = t.n0;
  g.n_forced = t.n_forced;
  g.y_first = t.y_first;
  const size_t smem = step32_smem(op->p32.warps);
  cudaError_t e = cudaFuncSetAttribute(gl1d_step32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)step32_smem(kMaxWarps));
  if (e != cudaSuccess) return e;
  gl1d_step32_kernel<<<(unsigned)op->p32.packs, 32 * (unsigned)op->p32.warps, smem, op->stream>>>(
      g, (cf*)state, (const cf*)G, (cf*)Y, op->d_flag);
  return cudaGetLastError();
}

// Squared 2-norms of the kg vectors of the packed state (out zeroed here).
cudaError_t step32_sq_norms(rsv_operator op, int kg, double* d_out) {
  cudaError_t e = cudaMemsetAsync(d_out, 0, sizeof(double) * kg, op->stream);
  if (e != cudaSuccess) return e;
  const unsigned bx = (unsigned)std::min<int64_t>((op->n + 255) / 256, std::max(1, 2 * op->sm_count / std::max(kg, 1)));
  slot_sumsq_kernel<<<dim3(std::max(bx, 1u), (unsigned)kg), 256, 0, op->stream>>>(
      (const cf*)op->ws_state.ptr, (const int32_t*)op->p32.slot, op->n, d_out);
  return cudaGetLastError();
}

}  // namespace rsv
