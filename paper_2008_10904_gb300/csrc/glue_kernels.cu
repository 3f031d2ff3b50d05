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

// FP64: one CTA per (frequency, instance, chunk of points).  The CTA stages the k vectors of 256 (128) points at a
// time in shared memory (each value read once from HBM, the next slab in flight during the current one).  The
// k x k Gram is Hermitian and cut into tiles of T x T pairs on and above the diagonal, one or a few per warp: a
// lane holds the T x T sums of its points (every 32nd), so that 2 T loads feed T^2 complex multiply-adds.  The
// lanes' sums over a slab are added up across the warp by a halving exchange that leaves one of the 2 T^2
// values per lane.  One FP64 atomic per value and chunk.
constexpr int kSlab = 256;
constexpr int kSlabsPerCta = 8;
constexpr int kGramWarps = 12;
// Two slabs of more than 28 vectors exceed the shared memory of a CTA: these take slabs of half the points.
constexpr int kWideK = 28, kWideSlab = kSlab / 2;
constexpr size_t gram64_smem(int rows, int slab) { return 2 * sizeof(cpx<double>) * (size_t)rows * slab; }
static_assert(gram64_smem(kWideK, kSlab) <= 232448 && gram64_smem(kMaxK, kWideSlab) <= 232448, "FP64 Gram slabs");

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

__device__ __forceinline__ void gram_tile_of(int t, int kt, int T, int* ta, int* tb) {   // rows ta, columns tb >= ta
  int a = 0;
  while (t >= kt - a) t -= kt - a++;
  *ta = a * T;
  *tb = (a + t) * T;
}

template <int kSlab64, int kSlabs64>   // points per slab, slabs per CTA
__global__ void __launch_bounds__(32 * kGramWarps) gram64_kernel(const cpx<double>* __restrict__ X, int k, int64_t n,
                                                                const int64_t* __restrict__ inst_off, int n_inst,
                                                                cpx<double>* __restrict__ G) {
  using R = double;
  constexpr int T = 2, NV = 2 * T * T;
  constexpr int kMaxOwn = 12;                                       // tiles per warp at k = 32
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<R>* slabs = reinterpret_cast<cpx<R>*>(smem_raw);             // [2][kt T][kSlab64], rows from k on zero
  const int inst = blockIdx.y;
  const int j = blockIdx.z;
  const int64_t p0 = inst_off[inst], p1 = inst_off[inst + 1];
  const int64_t c0 = p0 + (int64_t)blockIdx.x * kSlab64 * kSlabs64;
  if (c0 >= p1) return;
  const cpx<R>* Xj = X + (int64_t)j * k * n;
  const int kt = (k + T - 1) / T, tiles = kt * (kt + 1) / 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int slab_len = kt * T * kSlab64;
  for (int e = threadIdx.x; e < (kt * T - k) * kSlab64; e += blockDim.x)
    slabs[k * kSlab64 + e] = slabs[slab_len + k * kSlab64 + e] = mk<R>(0, 0);
  // asynchronous copies of slab sl into its buffer (zeros past the instance's end); nothing past the chunk
  auto copy_slab = [&](int sl) {
    const int64_t s0 = c0 + (int64_t)sl * kSlab64;
    if (sl < kSlabs64 && s0 < p1) {
      const int cnt = (int)min((int64_t)kSlab64, p1 - s0);
      cpx<R>* dst = slabs + (sl & 1) * slab_len;
      for (int e = threadIdx.x; e < k * kSlab64; e += blockDim.x) {
        const int a = e / kSlab64, pp = e % kSlab64;
        const cpx<R>* src = Xj + (int64_t)a * n + s0 + (pp < cnt ? pp : 0);
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + e)),
                     "l"(src), "n"(sizeof(cpx<R>)), "r"(pp < cnt ? (int)sizeof(cpx<R>) : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  copy_slab(0);
  // this warp's tiles warp, warp + nw, ...
  double tot[kMaxOwn];
#pragma unroll
  for (int q = 0; q < kMaxOwn; ++q) tot[q] = 0.0;
  for (int sl = 0; sl < kSlabs64; ++sl) {
    const int64_t s0 = c0 + (int64_t)sl * kSlab64;
    if (s0 >= p1) break;
    const int cnt = (int)min((int64_t)kSlab64, p1 - s0);
    copy_slab(sl + 1);                                             // into the buffer read before the last barrier
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const cpx<R>* xs = slabs + (sl & 1) * slab_len;
#pragma unroll
    for (int q = 0; q < kMaxOwn; ++q) {
      const int t = warp + q * nw;
      if (t >= tiles) break;
      int ta, tb;
      gram_tile_of(t, kt, T, &ta, &tb);
      R v[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = R(0);
      const cpx<R>* xa = xs + ta * kSlab64 + lane;
      const cpx<R>* xb = xs + tb * kSlab64 + lane;
      for (int pp = 0; pp < cnt; pp += 32) {                      // points past cnt are zero
        cpx<R> a[T], b[T];
#pragma unroll
        for (int i = 0; i < T; ++i) {
          a[i] = xa[i * kSlab64 + pp];
          b[i] = xb[i * kSlab64 + pp];
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
    gram_tile_of(t, kt, T, &ta, &tb);
    const double s = tot[q];
    if (lane >= NV) continue;
    const int pair = lane >> 1, a = ta + pair / T, b = tb + pair % T;
    if (a >= k || b >= k) continue;
    atomicAdd(g + 2 * (a * k + b) + (lane & 1), s);
    if (ta != tb) atomicAdd(g + 2 * (b * k + a) + (lane & 1), (lane & 1) ? -s : s);   // the mirrored tile
  }
}

// FP32: sums over a slab of 256 points in FP32, point after point, then FP64 across slabs.  That order is part of
// the result (another one moves the triangular factors by 3e-8), and it is a chain of 512 multiply-adds, so the
// parallelism is across slabs and pairs: a lane takes a slab of its own and a 4 x 4 tile of pairs, 8 loads per
// point for 64 multiply-adds in 32 independent chains.  A CTA holds 32 slabs, eight points of each at a time in
// shared memory (rows of 9, so that the lanes' loads fall in different banks; the next eight in flight).
// 16 x 16 x 262,144: 1.40 ms per CholeskyQR2 call (a pair per thread with all loads its own: 3.1).
constexpr int kG32Pts = 8, kG32Ld = kG32Pts + 1;

template <int kOwnTiles>   // tiles per warp
__global__ void __launch_bounds__(32 * kGramWarps) gram32_kernel(const cpx<float>* __restrict__ X, int k, int64_t n,
                                                                const int64_t* __restrict__ inst_off, int n_inst,
                                                                cpx<double>* __restrict__ G) {
  constexpr int T = 4, NV = 2 * T * T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<float>* bufs = reinterpret_cast<cpx<float>*>(smem_raw);      // [2][kt T][32 slabs][kG32Ld], rows from k on zero
  const int inst = blockIdx.y;
  const int j = blockIdx.z;
  const int64_t p0 = inst_off[inst], p1 = inst_off[inst + 1];
  const int64_t c0 = p0 + (int64_t)blockIdx.x * kSlab * 32;
  if (c0 >= p1) return;
  const cpx<float>* Xj = X + (int64_t)j * k * n;
  const int kt = (k + T - 1) / T, tiles = kt * (kt + 1) / 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int buf_len = kt * T * 32 * kG32Ld;
  for (int e = threadIdx.x; e < (kt * T - k) * 32 * kG32Ld; e += blockDim.x)
    bufs[k * 32 * kG32Ld + e] = bufs[buf_len + k * 32 * kG32Ld + e] = mk<float>(0.f, 0.f);
  const int rounds = (int)((min((int64_t)kSlab, p1 - c0) + kG32Pts - 1) / kG32Pts);
  // points [8 s, 8 s + 8) of every slab, zeros past the instance's end
  auto copy_round = [&](int s) {
    if (s < rounds) {
      cpx<float>* dst = bufs + (s & 1) * buf_len;
      for (int e = threadIdx.x; e < k * 32 * kG32Pts; e += blockDim.x) {
        const int a = e / (32 * kG32Pts), sl = e / kG32Pts % 32, pp = e % kG32Pts;
        const int64_t p = c0 + (int64_t)sl * kSlab + s * kG32Pts + pp;
        const bool in = p < p1;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(dst + (a * 32 + sl) * kG32Ld + pp)),
                     "l"(Xj + (int64_t)a * n + (in ? p : c0)), "r"(in ? 8 : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  copy_round(0);
  float v[kOwnTiles][NV];
  int ta[kOwnTiles], tb[kOwnTiles];
#pragma unroll
  for (int q = 0; q < kOwnTiles; ++q) {
    ta[q] = tb[q] = 0;
    if (warp + q * nw < tiles) gram_tile_of(warp + q * nw, kt, T, &ta[q], &tb[q]);
#pragma unroll
    for (int i = 0; i < NV; ++i) v[q][i] = 0.f;
  }
  for (int s = 0; s < rounds; ++s) {
    copy_round(s + 1);                                             // into the buffer read before the last barrier
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const cpx<float>* xs = bufs + (s & 1) * buf_len + lane * kG32Ld;
#pragma unroll
    for (int q = 0; q < kOwnTiles; ++q) {
      if (warp + q * nw >= tiles) break;
      const cpx<float>* xa = xs + ta[q] * 32 * kG32Ld;
      const cpx<float>* xb = xs + tb[q] * 32 * kG32Ld;
#pragma unroll
      for (int pp = 0; pp < kG32Pts; ++pp) {
        cpx<float> a[T], b[T];
#pragma unroll
        for (int i = 0; i < T; ++i) {
          a[i] = xa[i * 32 * kG32Ld + pp];
          b[i] = xb[i * 32 * kG32Ld + pp];
        }
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
          for (int l = 0; l < T; ++l) {
            float& re = v[q][2 * (i * T + l)];
            float& im = v[q][2 * (i * T + l) + 1];
            re = fmaf(a[i].re, b[l].re, fmaf(a[i].im, b[l].im, re));
            im = fmaf(a[i].re, b[l].im, fmaf(-a[i].im, b[l].re, im));
          }
      }
    }
    __syncthreads();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  double* g = reinterpret_cast<double*>(G + ((int64_t)j * n_inst + inst) * k * k);
#pragma unroll
  for (int q = 0; q < kOwnTiles; ++q) {
    if (warp + q * nw >= tiles) break;
    double d[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) d[i] = (double)v[q][i];
    const double t = warp_scatter_sum<NV>(d, lane);                // value `lane` over the slabs
    const int pair = lane >> 1, a = ta[q] + pair / T, b = tb[q] + pair % T;
    if (a >= k || b >= k) continue;
    atomicAdd(g + 2 * (a * k + b) + (lane & 1), t);
    if (ta[q] != tb[q]) atomicAdd(g + 2 * (b * k + a) + (lane & 1), (lane & 1) ? -t : t);   // the mirrored tile
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
  constexpr bool f32 = sizeof(R) == 4;
  constexpr int T = f32 ? 4 : 2;
  const int64_t per_cta = (int64_t)kSlab * (f32 ? 32 : kSlabsPerCta);
  dim3 grid((unsigned)((max_len + per_cta - 1) / per_cta), (unsigned)n_inst, (unsigned)n_omega);
  const int kt = (k + T - 1) / T, tiles = kt * (kt + 1) / 2;
  const bool wide = kt * T > kWideK;
  const size_t smem =
      f32 ? 2 * sizeof(cpx<R>) * (size_t)kt * T * 32 * kG32Ld : gram64_smem(kt * T, wide ? kWideSlab : kSlab);
  void (*kernel)(const cpx<R>*, int, int64_t, const int64_t*, int, cpx<double>*);
  if constexpr (f32)
    kernel = tiles <= kGramWarps ? gram32_kernel<1> : gram32_kernel<3>;
  else
    kernel = wide ? gram64_kernel<kWideSlab, kSlabsPerCta * kSlab / kWideSlab> : gram64_kernel<kSlab, kSlabsPerCta>;
  if (smem > 48 * 1024) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  const int warps = tiles > kGramWarps ? kGramWarps : f32 && tiles < 4 ? 4 : tiles;   // FP32: four share the copies
  kernel<<<grid, 32 * warps, smem, st>>>((const cpx<R>*)X, k, n, inst_off, n_inst, G);
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
