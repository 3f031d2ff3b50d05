// FP64 synthesis and analysis at whole steps (step form), using the symmetry of the time points.
//
//   F[tau][r]    = sum_j c_j[r] exp(i w_j t_tau)            (real state: sum_j cw_j Re(...))
//   acc[j][r]   += sum_s Y[s][r] exp(-i w_j t_s)
//
// FP64 arithmetic bounds both (one warp instruction per 19 cycles and SM), so they are arranged for the
// fewest operations: the times are taken in pairs around a centre t_c,
//   F(t_c +- d) = a -+ i' b,  a = sum_j c'_j cos(w_j d),  b = sum_j c'_j sin(w_j d),  c'_j = c_j exp(i w_j t_c),
//   sum_s       = exp(-i w_j t_c) sum_d [(Y(t_c + d) + Y(t_c - d)) cos(w_j d) - i (Y(t_c + d) - Y(t_c - d)) sin(w_j d)],
// four multiply-adds per frequency and pair of times instead of eight (real state: two instead of
// four).  A warp owns 32 rows (one per lane) and 16 times (synthesis) or 8 frequencies and a run of
// 64-step slices (analysis), so that small blocks of rows still spread over the GPU.  Analysis runs of
// one (row, frequency) are summed in a fixed order from a partial-sum buffer.
#include <algorithm>

#include "rsv_ops.h"

namespace rsv {
namespace {

constexpr int kPairs = 8;          // synthesis: 16 times per warp
constexpr int kWarps = 4;
constexpr int kJ = 8;              // analysis: frequencies per warp
constexpr int kSlice = 64;         // analysis: steps per slice
constexpr int kHalf = kSlice / 2;

using cd = cpx<double>;

template <bool REAL>
__global__ void __launch_bounds__(32 * kWarps) synth64_kernel(TileGeom g, int n_tau, int row_groups, int chunks,
                                                              const cd* __restrict__ c, const cd* __restrict__ tw,
                                                              const int64_t* __restrict__ pj,
                                                              const float* __restrict__ cw, void* __restrict__ Fout) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cd* off = reinterpret_cast<cd*>(smem_raw);                      // [n_omega][kPairs]: cos, sin of w_j d
  cd* rot = off + (size_t)g.n_omega * kPairs;                     // [kWarps][n_omega]: exp(i w_j t_c) (x cw_j)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int hs = g.tau_stride / 2;                                // half of a time step in half steps
  for (int e = threadIdx.x; e < g.n_omega * kPairs; e += blockDim.x) {
    const int j = e / kPairs, d = e % kPairs;
    off[e] = tw[phase_index(g.sgn * pj[j], (int64_t)(2 * d + 1) * hs, g.m4)];
  }
  const int64_t item = (int64_t)blockIdx.x * kWarps + warp;       // times fastest: neighbours share their rows
  const int64_t rg = item / chunks;
  const int tau0 = (int)(item % chunks) * 2 * kPairs;
  if (rg < row_groups) {
    for (int j = lane; j < g.n_omega; j += 32) {
      const int64_t t_c = 2 * g.n0 + (int64_t)tau0 * g.tau_stride + (int64_t)(2 * kPairs - 1) * hs;
      cd w = tw[phase_index(g.sgn * pj[j], t_c, g.m4)];
      if (REAL) w = (double)cw[j] * w;
      rot[warp * g.n_omega + j] = w;
    }
  }
  __syncthreads();
  if (rg >= row_groups) return;
  const int64_t r = rg * 32 + lane;
  const bool ok = r < g.rows;
  const cd* cr = c + (ok ? r : 0);
  const cd* ro = rot + warp * g.n_omega;
  cd a[kPairs], b[kPairs];
#pragma unroll
  for (int d = 0; d < kPairs; ++d) a[d] = b[d] = mk<double>(0, 0);
  cd x = cr[0];
  for (int j = 0; j < g.n_omega; ++j) {
    const cd nx = j + 1 < g.n_omega ? cr[(int64_t)(j + 1) * g.coef_stride] : x;   // in flight during this frequency
    const cd y = ro[j] * x;
#pragma unroll
    for (int d = 0; d < kPairs; ++d) {
      const cd w = off[j * kPairs + d];
      a[d].re = fma(y.re, w.re, a[d].re);
      b[d].im = fma(y.im, w.im, b[d].im);
      if (!REAL) {
        a[d].im = fma(y.im, w.re, a[d].im);
        b[d].re = fma(y.re, w.im, b[d].re);
      }
    }
    x = nx;
  }
  if (!ok) return;
#pragma unroll
  for (int d = 0; d < kPairs; ++d) {
    const int tp = tau0 + kPairs + d, tm = tau0 + kPairs - 1 - d;
    if (REAL) {
      double* F = reinterpret_cast<double*>(Fout);
      if (tp < n_tau) F[(int64_t)tp * g.rows + r] = a[d].re - b[d].im;
      if (tm < n_tau) F[(int64_t)tm * g.rows + r] = a[d].re + b[d].im;
    } else {
      cd* F = reinterpret_cast<cd*>(Fout);
      if (tp < n_tau) F[(int64_t)tp * g.rows + r] = mk<double>(a[d].re - b[d].im, a[d].im + b[d].re);
      if (tm < n_tau) F[(int64_t)tm * g.rows + r] = mk<double>(a[d].re + b[d].im, a[d].im - b[d].re);
    }
  }
}

// part == nullptr: one run per (rows, frequencies), added to acc; otherwise run p writes part[p][j][r].
template <bool REAL>
__global__ void __launch_bounds__(32 * kWarps) analysis64_kernel(TileGeom g, const void* __restrict__ Yin, int s0, int s1,
                                                                 int row_groups, int runs, int slices_per_run,
                                                                 const cd* __restrict__ tw,
                                                                 const int64_t* __restrict__ pj, cd* __restrict__ acc,
                                                                 int64_t acc_stride, cd* __restrict__ part) {
  __shared__ cd off[kHalf][kJ];                 // cos, sin of w_j d, d = (2 l + 1) h / 2
  __shared__ cd rot[kJ];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = blockDim.x >> 5;
  const int j0 = blockIdx.y * kJ, nj = min(kJ, g.n_omega - j0);
  const int run = blockIdx.z;
  for (int e = threadIdx.x; e < kHalf * kJ; e += blockDim.x) {
    const int l = e / kJ, q = e % kJ;
    off[l][q] = q < nj ? tw[phase_index(g.sgn * pj[j0 + q], 2 * l + 1, g.m4)] : mk<double>(0, 0);
  }
  const int64_t r = ((int64_t)blockIdx.x * nw + warp) * 32 + lane;
  const bool ok = r < g.rows;
  const double* yr = reinterpret_cast<const double*>(Yin) + (ok ? r : 0);
  const cd* yc = reinterpret_cast<const cd*>(Yin) + (ok ? r : 0);
  auto load = [&](int s) -> cd {
    if (s < s0 || s >= s1) return mk<double>(0, 0);
    return REAL ? mk<double>(yr[(int64_t)s * g.rows], 0.0) : yc[(int64_t)s * g.rows];
  };
  cd sum[kJ];
#pragma unroll
  for (int q = 0; q < kJ; ++q) sum[q] = mk<double>(0, 0);
  for (int sl = 0; sl < slices_per_run; ++sl) {
    const int sa = s0 + (run * slices_per_run + sl) * kSlice;
    if (sa >= s1) break;
    __syncthreads();
    for (int q = threadIdx.x; q < nj; q += blockDim.x)
      rot[q] = tw[phase_index(g.sgn * pj[j0 + q], 2 * (g.n0 + sa) + kSlice - 1, g.m4)];   // exp(i w_j t_c)
    __syncthreads();
    cd a[kJ], b[kJ];
#pragma unroll
    for (int q = 0; q < kJ; ++q) a[q] = b[q] = mk<double>(0, 0);
    // pairs (sa + 31 - l, sa + 32 + l) with at least one step inside
    const int l0 = max(0, kHalf - (s1 - sa));
    cd ym = load(sa + kHalf - 1 - l0), yp = load(sa + kHalf + l0);
    for (int l = l0; l < kHalf; ++l) {
      const cd nm = load(sa + kHalf - 2 - l), np = l + 1 < kHalf ? load(sa + kHalf + l + 1) : mk<double>(0, 0);
      const cd p = yp + ym, m = yp - ym;
#pragma unroll
      for (int q = 0; q < kJ; ++q) {
        const cd w = off[l][q];
        a[q].re = fma(p.re, w.re, a[q].re);
        b[q].re = fma(m.re, w.im, b[q].re);
        if (!REAL) {
          a[q].im = fma(p.im, w.re, a[q].im);
          b[q].im = fma(m.im, w.im, b[q].im);
        }
      }
      ym = nm;
      yp = np;
    }
    // += exp(-i w t_c) (a - i b)
#pragma unroll
    for (int q = 0; q < kJ; ++q) {
      const cd z = REAL ? mk<double>(a[q].re, -b[q].re) : mk<double>(a[q].re + b[q].im, a[q].im - b[q].re);
      if (q < nj) cfma_conj(sum[q], rot[q], z);
    }
  }
  if (!ok) return;
#pragma unroll
  for (int q = 0; q < kJ; ++q) {
    if (q >= nj) break;
    if (part != nullptr) {
      part[((int64_t)run * g.n_omega + j0 + q) * g.rows + r] = sum[q];
    } else {
      cd* p = acc + (int64_t)(j0 + q) * acc_stride + r;
      *p = *p + sum[q];
    }
  }
}

__global__ void add_parts_kernel(const cd* __restrict__ part, int runs, int n_omega, int64_t rows, cd* __restrict__ acc,
                                 int64_t acc_stride) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (r >= rows) return;
  cd s = acc[(int64_t)j * acc_stride + r];
  for (int p = 0; p < runs; ++p) s = s + part[((int64_t)p * n_omega + j) * rows + r];
  acc[(int64_t)j * acc_stride + r] = s;
}

}  // namespace

// Synthesis at n_tau whole-step times (tau_stride even), FP64.
cudaError_t synth64(rsv_operator op, const TileGeom& g, const void* coef, void* F) {
  const int n_tau = g.n_tau;
  if (n_tau <= 0) return cudaSuccess;
  const int64_t rg = (g.rows + 31) / 32;
  const int chunks = (n_tau + 2 * kPairs - 1) / (2 * kPairs);
  const size_t smem = sizeof(cd) * (size_t)g.n_omega * (kPairs + kWarps);
  if (smem > 200 * 1024)   // more than about a thousand frequencies: the general kernel
    return launch_synth<double>(g, coef, op->d_tw, op->d_pj, op->d_cw, op->real_state, F, op->stream);
  const unsigned blocks = (unsigned)((rg * chunks + kWarps - 1) / kWarps);
  auto k = op->real_state ? synth64_kernel<true> : synth64_kernel<false>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  k<<<blocks, 32 * kWarps, smem, op->stream>>>(g, n_tau, (int)rg, chunks, (const cd*)coef, (const cd*)op->d_tw, op->d_pj,
                                               op->d_cw, F);
  return cudaGetLastError();
}

// Runs an analysis of `steps` steps is split into: enough warps for four per SM and scheduler with a
// single vector of `points` points, few enough that a run has at least two slices.  Not a function of the
// vectors in the group: the order of the sums is the same however a block is cut into groups, and the
// partial sums of a smaller group fit where a larger one's did.
static int analysis64_runs(rsv_operator op, int64_t points, int steps) {
  const int64_t warps = ((points + 31) / 32) * ((op->n_omega + kJ - 1) / kJ);
  const int slices = (steps + kSlice - 1) / kSlice;
  const int64_t want = (16 * (int64_t)std::max(1, op->sm_count) + warps - 1) / warps;
  return (int)std::max<int64_t>(1, std::min<int64_t>(want, slices / 2));
}

size_t analysis64_part_bytes(rsv_operator op, int64_t rows, int64_t points, int steps) {
  const int runs = analysis64_runs(op, points, steps);
  return runs > 1 ? (size_t)runs * op->n_omega * rows * sizeof(cd) : 0;
}

// acc += the Fourier sums of the tile steps [s0, s1) of vectors of `points` points; part: a buffer of part_bytes,
// analysis64_part_bytes(s1 - s0) or more (InvalidValue otherwise).
cudaError_t analysis64(rsv_operator op, const TileGeom& g, int64_t points, const void* Y, int s0, int s1,
                       cpx<double>* acc, int64_t acc_stride, void* part, size_t part_bytes) {
  if (s1 <= s0) return cudaSuccess;
  if (analysis64_part_bytes(op, g.rows, points, s1 - s0) > part_bytes) return cudaErrorInvalidValue;
  const int slices = (s1 - s0 + kSlice - 1) / kSlice;
  int runs = analysis64_runs(op, points, s1 - s0);
  const int per = (slices + runs - 1) / runs;
  runs = (slices + per - 1) / per;
  const int64_t rg = (g.rows + 31) / 32;
  const int nw = (int)std::min<int64_t>(kWarps, rg);
  const dim3 grid((unsigned)((rg + nw - 1) / nw), (unsigned)((g.n_omega + kJ - 1) / kJ), (unsigned)runs);
  cd* pb = runs > 1 ? static_cast<cd*>(part) : nullptr;
  auto k = op->real_state ? analysis64_kernel<true> : analysis64_kernel<false>;
  k<<<grid, 32 * nw, 0, op->stream>>>(g, Y, s0, s1, (int)rg, runs, per, (const cd*)op->d_tw, op->d_pj, acc, acc_stride, pb);
  if (runs > 1)
    add_parts_kernel<<<dim3((unsigned)((g.rows + 127) / 128), (unsigned)g.n_omega), 128, 0, op->stream>>>(
        pb, runs, g.n_omega, g.rows, acc, acc_stride);
  return cudaGetLastError();
}

}  // namespace rsv
