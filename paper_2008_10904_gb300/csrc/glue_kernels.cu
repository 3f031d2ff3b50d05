// Per-frequency block algebra of the randomized SVD: Gram matrices of the
// k-vector blocks and recombination of a block by a small matrix.  Products
// are formed in the storage precision of the blocks; the Gram sums across
// 256-point slabs are FP64, and the small matrices are formed in FP64 on the
// host and applied in the block's precision.
//
//   gram:    G[j][i][a][b] = sum_{p in instance i} conj(X[j][a][p]) X[j][b][p]
//   combine: Out[j][b][p]  = sum_a In[j][a][p] M[j][inst(p)][a][b]   (M in the block's precision)
//
// gram gives the CholeskyQR factor (Q = X R^{-1}, R^H R = G) and the small
// Hermitian eigenproblem W^H W = B B^H of the final SVD step.
#include "rsv_internal.h"

namespace rsv {
namespace {

constexpr int kMaxK = 32;

// One CTA per (frequency, instance, chunk of points).  The CTA stages the k vectors of 256 points at a
// time in shared memory (each value read once from HBM, the next slab in flight during the current one).  The k x k Gram is Hermitian and cut into
// tiles of T x T pairs on and above the diagonal, one or a few per warp: a lane holds the T x T sums of
// its points (every 32nd), so that 2 T loads feed T^2 complex multiply-adds.  The lanes' sums over a slab
// (8 points each) are added up across the warp by a halving exchange that leaves one of the 2 T^2 values
// per lane, which goes on in FP64 across the slabs.  One FP64 atomic per value and chunk.  k = 16, 4.2 M points, FP32: 0.22 ms (one pair per thread: 0.70).
constexpr int kSlab = 256;
constexpr int kSlabsPerCta = 8;
constexpr int kGramWarps = 12;

template <typename R>
constexpr int gram_tile() { return sizeof(R) == 4 ? 4 : 2; }

// v[0 .. N-1] of every lane summed over the warp; lane l returns the sum of value l mod N.
template <int N, typename R>
__device__ __forceinline__ R warp_scatter_sum(R* v, int lane) {
#pragma unroll
  for (int h = N / 2; h >= 1; h /= 2) {   // lanes with bit h keep the upper half
    const bool up = (lane & h) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const R send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
    }
  }
  R r = v[0];
#pragma unroll
  for (int o = N; o < 32; o *= 2) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

template <typename R>
__global__ void __launch_bounds__(32 * kGramWarps) gram_kernel(const cpx<R>* __restrict__ X, int k, int64_t n,
                                                              const int64_t* __restrict__ inst_off, int n_inst,
                                                              cpx<double>* __restrict__ G) {
  constexpr int T = gram_tile<R>(), NV = 2 * T * T;
  constexpr int kMaxOwn = sizeof(R) == 4 ? 3 : 12;                 // tiles per warp at k = 32
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<R>* slabs = reinterpret_cast<cpx<R>*>(smem_raw);             // [2][kt T][kSlab], rows from k on zero
  const int inst = blockIdx.y;
  const int j = blockIdx.z;
  const int64_t p0 = inst_off[inst], p1 = inst_off[inst + 1];
  const int64_t c0 = p0 + (int64_t)blockIdx.x * kSlab * kSlabsPerCta;
  if (c0 >= p1) return;
  const cpx<R>* Xj = X + (int64_t)j * k * n;
  const int kt = (k + T - 1) / T, tiles = kt * (kt + 1) / 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int slab_len = kt * T * kSlab;
  for (int e = threadIdx.x; e < (kt * T - k) * kSlab; e += blockDim.x)
    slabs[k * kSlab + e] = slabs[slab_len + k * kSlab + e] = mk<R>(0, 0);
  // asynchronous copies of slab sl into its buffer (zeros past the instance's end); nothing past the chunk
  auto copy_slab = [&](int sl) {
    const int64_t s0 = c0 + (int64_t)sl * kSlab;
    if (sl < kSlabsPerCta && s0 < p1) {
      const int cnt = (int)min((int64_t)kSlab, p1 - s0);
      cpx<R>* dst = slabs + (sl & 1) * slab_len;
      for (int e = threadIdx.x; e < k * kSlab; e += blockDim.x) {
        const int a = e / kSlab, pp = e % kSlab;
        const cpx<R>* src = Xj + (int64_t)a * n + s0 + (pp < cnt ? pp : 0);
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + e)),
                     "l"(src), "n"(sizeof(cpx<R>)), "r"(pp < cnt ? (int)sizeof(cpx<R>) : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  copy_slab(0);
  // this warp's tiles warp, warp + nw, ...: rows ta, columns tb >= ta
  auto tile_of = [&](int t, int* ta, int* tb) {
    int a = 0;
    while (t >= kt - a) t -= kt - a++;
    *ta = a * T;
    *tb = (a + t) * T;
  };
  double tot[kMaxOwn];
#pragma unroll
  for (int q = 0; q < kMaxOwn; ++q) tot[q] = 0.0;
  for (int sl = 0; sl < kSlabsPerCta; ++sl) {
    const int64_t s0 = c0 + (int64_t)sl * kSlab;
    if (s0 >= p1) break;
    const int cnt = (int)min((int64_t)kSlab, p1 - s0);
    copy_slab(sl + 1);                                             // into the buffer read before the last barrier
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const cpx<R>* xs = slabs + (sl & 1) * slab_len;
#pragma unroll
    for (int q = 0; q < kMaxOwn; ++q) {
      const int t = warp + q * nw;
      if (t >= tiles) break;
      int ta, tb;
      tile_of(t, &ta, &tb);
      R v[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = R(0);
      const cpx<R>* xa = xs + ta * kSlab + lane;
      const cpx<R>* xb = xs + tb * kSlab + lane;
      for (int pp = 0; pp < cnt; pp += 32) {                      // points past cnt are zero
        cpx<R> a[T], b[T];
#pragma unroll
        for (int i = 0; i < T; ++i) {
          a[i] = xa[i * kSlab + pp];
          b[i] = xb[i * kSlab + pp];
        }
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
          for (int l = 0; l < T; ++l) {
            R& re = v[2 * (i * T + l)];
            R& im = v[2 * (i * T + l) + 1];
            re = fma(a[i].re, b[l].re, fma(a[i].im, b[l].im, re));
            im = fma(a[i].re, b[l].im, fma(-a[i].im, b[l].re, im));
          }
      }
      tot[q] += (double)warp_scatter_sum<NV>(v, lane);
    }
    __syncthreads();
  }
  double* g = reinterpret_cast<double*>(G + ((int64_t)j * n_inst + inst) * k * k);
#pragma unroll
  for (int q = 0; q < kMaxOwn; ++q) {
    const int t = warp + q * nw;
    if (t >= tiles) break;
    int ta, tb;
    tile_of(t, &ta, &tb);
    const double s = tot[q];
    if (lane >= NV) continue;
    const int pair = lane >> 1, a = ta + pair / T, b = tb + pair % T;
    if (a >= k || b >= k) continue;
    atomicAdd(g + 2 * (a * k + b) + (lane & 1), s);
    if (ta != tb) atomicAdd(g + 2 * (b * k + a) + (lane & 1), (lane & 1) ? -s : s);   // the mirrored tile
  }
}

// KA: ka rounded up to 4, 8, 16 or 32 (the point's inputs in registers).  A block without instances of its
// own keeps the matrix of its frequency in shared memory.
template <typename R, int KA>
__global__ void __launch_bounds__(256) combine_kernel(const cpx<R>* In, int ka, int kb, int64_t n,
                                                     const int32_t* __restrict__ inst_of_point, int n_inst,
                                                     const cpx<R>* __restrict__ M, cpx<R>* Out,
                                                     int64_t out_k) {
  __shared__ cpx<R> sM[kMaxK * KA];                                // [b][a], zero past ka
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  const cpx<R>* Mj = M + (int64_t)j * n_inst * ka * kb;
  if (n_inst == 1) {
    for (int e = threadIdx.x; e < kb * KA; e += blockDim.x) {
      const int b = e / KA, a = e % KA;
      sM[e] = a < ka ? Mj[a * kb + b] : mk<R>(0, 0);
    }
    __syncthreads();
  }
  if (p >= n) return;
  // arithmetic in the element precision R (FP64 blocks: FP64; FP32 blocks: FP32)
  cpx<R> x[KA];
#pragma unroll
  for (int a = 0; a < KA; ++a) x[a] = a < ka ? In[((int64_t)j * ka + a) * n + p] : mk<R>(0, 0);
  // In and Out may alias: every input of this point is in registers now.
  if (n_inst == 1) {
    for (int b = 0; b < kb; ++b) {
      cpx<R> s = mk<R>(0, 0);
#pragma unroll
      for (int a = 0; a < KA; ++a)
        if (sizeof(R) == 4 || a < ka) cfma(s, x[a], sM[b * KA + a]);
      Out[((int64_t)j * out_k + b) * n + p] = s;
    }
    return;
  }
  Mj += (int64_t)inst_of_point[p] * ka * kb;
  for (int b = 0; b < kb; ++b) {
    cpx<R> s = mk<R>(0, 0);
#pragma unroll
    for (int a = 0; a < KA; ++a)
      if (a < ka) cfma(s, x[a], Mj[a * kb + b]);
    Out[((int64_t)j * out_k + b) * n + p] = s;
  }
}

}  // namespace

template <typename R>
cudaError_t launch_gram(const void* X, int n_omega, int k, int64_t n, const int64_t* inst_off, int n_inst,
                        int64_t max_len, cpx<double>* G, cudaStream_t st) {
  if (k > kMaxK) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(G, 0, sizeof(cpx<double>) * (size_t)n_omega * n_inst * k * k, st);
  if (e != cudaSuccess) return e;
  // chunks per instance: enough for the longest instance (short instances return early)
  const int64_t per_cta = (int64_t)kSlab * kSlabsPerCta;
  dim3 grid((unsigned)((max_len + per_cta - 1) / per_cta), (unsigned)n_inst, (unsigned)n_omega);
  constexpr int T = gram_tile<R>();
  const int kt = (k + T - 1) / T, tiles = kt * (kt + 1) / 2;
  const size_t smem = 2 * sizeof(cpx<R>) * (size_t)kt * T * kSlab;
  if (smem > 48 * 1024) {
    e = cudaFuncSetAttribute(gram_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  gram_kernel<R><<<grid, 32 * (tiles < kGramWarps ? tiles : kGramWarps), smem, st>>>((const cpx<R>*)X, k, n, inst_off, n_inst, G);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_combine(const void* In, int n_omega, int ka, int kb, int64_t n, const int32_t* inst_of_point,
                           int n_inst, const void* M, void* Out, int64_t out_k, cudaStream_t st) {
  if (ka > kMaxK || kb > kMaxK) return cudaErrorInvalidValue;
  dim3 grid((unsigned)((n + 255) / 256), (unsigned)n_omega);
  auto k = ka <= 4 ? combine_kernel<R, 4> : ka <= 8 ? combine_kernel<R, 8> : ka <= 16 ? combine_kernel<R, 16> : combine_kernel<R, 32>;
  k<<<grid, 256, 0, st>>>((const cpx<R>*)In, ka, kb, n, inst_of_point, n_inst, (const cpx<R>*)M, (cpx<R>*)Out, out_k);
  return cudaGetLastError();
}

template cudaError_t launch_gram<double>(const void*, int, int, int64_t, const int64_t*, int, int64_t,
                                        cpx<double>*, cudaStream_t);
template cudaError_t launch_gram<float>(const void*, int, int, int64_t, const int64_t*, int, int64_t, cpx<double>*,
                                       cudaStream_t);
template cudaError_t launch_combine<double>(const void*, int, int, int, int64_t, const int32_t*, int, const void*,
                                           void*, int64_t, cudaStream_t);
template cudaError_t launch_combine<float>(const void*, int, int, int, int64_t, const int32_t*, int, const void*,
                                          void*, int64_t, cudaStream_t);

}  // namespace rsv
