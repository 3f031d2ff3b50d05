// Tensor-core (tcgen05) RK4 step of the dense propagator, FP32 mode.
//
//   u_{n+1} = u_n + D u_n + F_n      (D = RK4 step polynomial minus identity, see dense_kernels.cu)
//
// D u is computed as the real GEMM  [Dr; Di] (2n x n)  x  [Ur | Ui] (n x 2kg):
// rows 2 r of a CTA's A tile are 64 rows of Re D, rows 2 r + 1 the same rows
// of Im D, and  Re(Du) = DrUr - DiUi,  Im(Du) = DrUi + DiUr.  Operands are
// split into TF32 pairs (x = hi + lo, hi = tf32(x)) and three MMAs
// (hi*hi + hi*lo + lo*hi) give FP32-level products with FP32 accumulation in
// tensor memory.
//
// Grid: one cluster of CS = n/128 CTAs per block of 64 complex rows; CTA rank
// j of a cluster owns the K slice of 128 complex columns [128 j, 128 j + 128).
// Each CTA bulk-copies its pre-arranged A tile (hi, lo: 2 x 64 KB) and its X
// slice (hi, lo: 2 x 32 KB) into shared memory, issues 16 K-steps x 3 MMAs
// (M = 128, N = 64, K = 8) from one thread, reads the 128 x 64 partial from
// tensor memory and exchanges it through distributed shared memory: CTA j
// sums over the cluster the partials of its 64/CS complex rows and
// writes the new state, the snapshot, and the TF32 split of the new state
// in the operand layout of the next step.  All waits are bounded; a timeout
// sets the error flag.
#include <cuda_runtime.h>

#include <cstdlib>

#include "rsv_ops.h"
#include "tc_ptx.h"

namespace rsv {
namespace {

constexpr int kTileK = 128;                         // complex columns per K slice
constexpr int kTileRows = 64;                       // complex rows per cluster
constexpr int kM = 128, kN = 64;                    // MMA shape (real rows, 2 x 32 vector columns)
constexpr uint32_t kATileFloats = kM * kTileK;      // 16384 floats = 64 KB
constexpr uint32_t kXTileFloats = kN * kTileK;      // 8192 floats = 32 KB
constexpr uint32_t kSmemBytes = 4 * kATileFloats + 4 * kATileFloats + 4 * kXTileFloats + 4 * kXTileFloats + 64;
constexpr uint32_t kWaitTries = 1u << 24;
constexpr int kRedLd = kN + 1;

struct TcStepArgs {
  const float* A;     // [n/64][CS][2][kATileFloats]
  const float* Xin;   // [CS][2][kXTileFloats]
  float* Xout;
  const cpx<float>* uin;   // [kg][n]
  cpx<float>* uout;
  const cpx<float>* F;     // nullable
  cpx<float>* Y;           // nullable
  int n, kg, cs;
  int* err;
};

__global__ void __launch_bounds__(256, 1) dense_tc_step_kernel(TcStepArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  float* A_hi = reinterpret_cast<float*>(smem);
  float* A_lo = A_hi + kATileFloats;
  float* X_hi = A_lo + kATileFloats;
  float* X_lo = X_hi + kXTileFloats;
  uint64_t* bars = reinterpret_cast<uint64_t*>(X_lo + kXTileFloats);  // [0] loads, [1] mma
  uint32_t* tbase = reinterpret_cast<uint32_t*>(bars + 2);
  float* red = A_hi;  // reused for the 128 x 64 partial once the MMAs have completed

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t mb = tc::cluster_id_x();
  const uint32_t j = tc::cluster_rank();
  if (tid == 0) {
    tc::mbar_init(&bars[0], 1);
    tc::mbar_init(&bars[1], 1);
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc(tbase, 64);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tbase;

  if (tid == 0) {
    const float* at = a.A + ((size_t)mb * a.cs + j) * 2 * kATileFloats;
    const float* xt = a.Xin + (size_t)j * 2 * kXTileFloats;
    tc::mbar_arrive_expect_tx(&bars[0], 4 * (2 * kATileFloats + 2 * kXTileFloats));
    tc::bulk_g2s(A_hi, at, 4 * kATileFloats, &bars[0]);
    tc::bulk_g2s(A_lo, at + kATileFloats, 4 * kATileFloats, &bars[0]);
    tc::bulk_g2s(X_hi, xt, 4 * kXTileFloats, &bars[0]);
    tc::bulk_g2s(X_lo, xt + kXTileFloats, 4 * kXTileFloats, &bars[0]);
  }
  bool ok = tc::mbar_wait(&bars[0], 0, kWaitTries);
  if (tid == 0) {
    if (ok) {
      const uint32_t idesc = tc::idesc_tf32(kM, kN);
      const uint32_t lbo = 128, sbo_a = (kTileK / 4) * 128, sbo_x = (kTileK / 4) * 128;
#pragma unroll 1
      for (int ks = 0; ks < kTileK / 8; ++ks) {
        const uint64_t ah = tc::smem_desc(reinterpret_cast<char*>(A_hi) + ks * 256, lbo, sbo_a);
        const uint64_t al = tc::smem_desc(reinterpret_cast<char*>(A_lo) + ks * 256, lbo, sbo_a);
        const uint64_t xh = tc::smem_desc(reinterpret_cast<char*>(X_hi) + ks * 256, lbo, sbo_x);
        const uint64_t xl = tc::smem_desc(reinterpret_cast<char*>(X_lo) + ks * 256, lbo, sbo_x);
        tc::mma_tf32(tmem, ah, xh, idesc, ks > 0);
        tc::mma_tf32(tmem, ah, xl, idesc, true);
        tc::mma_tf32(tmem, al, xh, idesc, true);
      }
      tc::mma_commit(&bars[1]);
    } else {
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&bars[1])) : "memory");
    }
  }
  ok = tc::mbar_wait(&bars[1], 0, kWaitTries) && ok;
  tc::tc_fence_after();
  if (warp < 4) {
    const int row = 32 * warp + lane;
#pragma unroll
    for (int c = 0; c < kN; c += 16) {
      float v[16];
      tc::tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + c, v);
#pragma unroll
      for (int q = 0; q < 16; ++q) red[row * kRedLd + c + q] = ok ? v[q] : 0.f;
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::cluster_sync();

  // cluster reduction + RK4 update: CTA j owns complex rows [rpc j, rpc j + rpc) of the
  // cluster's 64-row block (rpc = 64 / cs), i.e. stacked rows 2 iloc and 2 iloc + 1
  {
    const int rpc = kTileRows / a.cs;
    for (int pidx = tid; pidx < rpc * 32; pidx += blockDim.x) {
      const int ii = pidx >> 5;
      const int v = pidx & 31;
      const int iloc = rpc * (int)j + ii;
      float pr = 0.f, pi = 0.f;
      {
        float rr[8], ri[8], ir[8], ix[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) {
          if (p < a.cs) {
            rr[p] = tc::ld_peer_f32(tc::map_peer(&red[2 * iloc * kRedLd + v], p));
            ri[p] = tc::ld_peer_f32(tc::map_peer(&red[2 * iloc * kRedLd + 32 + v], p));
            ir[p] = tc::ld_peer_f32(tc::map_peer(&red[(2 * iloc + 1) * kRedLd + v], p));
            ix[p] = tc::ld_peer_f32(tc::map_peer(&red[(2 * iloc + 1) * kRedLd + 32 + v], p));
          }
        }
#pragma unroll
        for (int p = 0; p < 8; ++p) {
          if (p < a.cs) {
            pr += rr[p] - ix[p];
            pi += ri[p] + ir[p];
          }
        }
      }
      const int i = (int)mb * kTileRows + iloc;
      if (v < a.kg && i < a.n) {
        const int64_t e = (int64_t)v * a.n + i;
        const cpx<float> u0 = a.uin[e];
        cpx<float> u1 = mk<float>(u0.re + pr, u0.im + pi);
        if (a.F) u1 = u1 + a.F[e];
        a.uout[e] = u1;
        if (a.Y) a.Y[e] = u0;
        const int js = i / kTileK, kk = i % kTileK;
        float* xo = a.Xout + (size_t)js * 2 * kXTileFloats;
        const float hr = tc::to_tf32(u1.re), hi = tc::to_tf32(u1.im);
        const uint32_t o_re = tc::kmajor_offset(v, kk, kTileK) / 4, o_im = tc::kmajor_offset(32 + v, kk, kTileK) / 4;
        xo[o_re] = hr;
        xo[kXTileFloats + o_re] = u1.re - hr;
        xo[o_im] = hi;
        xo[kXTileFloats + o_im] = u1.im - hi;
      }
    }
  }
  tc::cluster_sync();
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, 64);
  if (!ok && tid == 0) atomicExch(a.err, 2);
}

// ---------------------------------------------------------------------------
// Persistent variant (no clusters): one launch marches a whole time tile with
// MB * CS CTAs, one per SM, all resident at once.  CTA (mb, j) keeps the A
// tile of row block mb and K slice j in shared memory for the whole tile.
//
// Two hand-offs per step pass through L2: the partial sums of a row block's CS
// CTAs to the owners of its rows, and the owners' new state to the CTAs of its
// K slice.  Every value travels with the number of its step in one 8-byte word
// (16-byte accesses carry two of them), and the receiver loads until the numbers
// are right: no counter, no fence and no copy stands between a store and the load
// that wants it.  Per step, with C = 32 or 64 real columns (16 or 32 vectors):
//   1. the eight worker warps load the state slice (128 x C), split it into TF32
//      hi / lo and store it as the K-major operand, one K half after the other;
//   2. warp 8 issues two MMAs per K-step, A_hi x [X_hi | X_lo] (N = 2 C) and
//      A_lo x X_hi (N = C), the first half's while the second is converted: the A
//      tile is read from shared memory twice, for all vectors at once;
//   3. the workers sum the three product groups out of tensor memory, combine them to
//      Re (D u) and Im (D u) and store the CTA's 64 x C partial;
//   4. as owner of 64/CS rows of its row block, each thread loads its rows of the
//      CS partials, all in flight at once, sums them in order, applies the RK4
//      update u <- u + D u + F (u stays in registers for the whole tile), writes
//      the snapshot and the new state.
// Both buffers alternate by step parity.  A CTA stores step n + 2's values only
// after it has received the state n + 2, which depends on every CTA's partials of
// step n + 1 and those on every owner's state n + 1: all loads of step n are over.
// The numbers start at 1; the buffers are zeroed at the start of a march.  Loads
// that wait are bounded in time and stop once any CTA has set the error flag.
// A step is a chain of latencies: n = 1024, 32 vectors, 13188 steps march in
// 57 ms.  With counters (fence, add, poll and bulk copy per hand-off) and two
// chains of 16 vectors that took turns on the tensor cores 88 ms; of 6.7 us per
// step 1.4 us were fences, 1.8 us polls and 2 us products.  Partials of separate Re D and
// Im D rows, twice as many words: 66 ms.
// ---------------------------------------------------------------------------
constexpr int kMaxCols = 64;                               // real columns: (re, im) of 32 vectors
constexpr int kWorkers = 256;
constexpr int kMarchThreads = kWorkers + 32;               // and the warp that issues the products
constexpr uint32_t kXsFloats = kTileK * kMaxCols * 2;      // a slice's words: [K / 2][C] x 2 (value, number)
constexpr uint32_t kPartFloats = kM * kMaxCols;            // a partial's words: [C / 4][64 rows x 2 vectors] x (re, im)
constexpr uint32_t kSmemPersistent = 4 * (2 * kATileFloats + 2 * kMaxCols * kTileK) + 256;

struct TcMarchArgs {
  const float* A;
  float* X;                 // [2][CS][kXsFloats]
  float* part;              // [2][MB][CS][kPartFloats]
  cpx<float>* u;            // [2][kg][n]: state at n0 in slot n0 & 1, written back to slot (n0 + steps) & 1
  const cpx<float>* F;      // [steps][kg][n] or null
  cpx<float>* Y;            // [steps][kg][n] or null
  int64_t n0;
  int steps;
  int64_t n_forced;
  int y_first;
  int n, kg, cs;
  int* err;
  uint64_t wait_ns;         // limit of each wait on another CTA's values
  int stall;                // test hook: the first state wait of the tile wants a number nobody writes
};

// Two (value, number) words, each of them one access of 8 bytes.
__device__ __forceinline__ void words_store(float* p, float v0, float v1, uint32_t number) {
  const uint64_t hi = (uint64_t)number << 32;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(hi | __float_as_uint(v0)),
               "l"(hi | __float_as_uint(v1))
               : "memory");
}
__device__ __forceinline__ void words_load(const float* p, uint64_t w[2]) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(p) : "memory");
}
__device__ __forceinline__ float word_value(uint64_t w) { return __uint_as_float((uint32_t)w); }

// Load again what has not got its number yet, until all have; false on the time limit or another CTA's error.
template <int M, typename At>
__device__ __forceinline__ bool words_wait(uint64_t (*w)[2], int count, uint32_t number, At at, const volatile int* err,
                                           uint64_t limit_ns) {
  uint64_t t0 = 0;
  for (uint32_t tries = 0;; ++tries) {
    bool all = true;
#pragma unroll
    for (int i = 0; i < M; ++i) {
      if (i < count && ((uint32_t)(w[i][0] >> 32) != number || (uint32_t)(w[i][1] >> 32) != number)) {
        all = false;
        words_load(at(i), w[i]);
      }
    }
    if (all) return true;
    if ((tries & 15) == 15) {
      if (*err != 0) return false;
      const uint64_t now = tc::global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) return false;
    }
  }
}

template <int C, int kMaxGroups>   // real columns; groups of eight owner rows at most (1: CS = 8)
__global__ void __launch_bounds__(kMarchThreads, 1) dense_tc_march_kernel(TcMarchArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  float* A_hi = reinterpret_cast<float*>(smem);
  float* A_lo = A_hi + kATileFloats;
  float* X_sm = A_lo + kATileFloats;                                    // [K half][hi rows [0, C), lo rows [C, 2 C)][64]
  uint64_t* bars = reinterpret_cast<uint64_t*>(X_sm + 2 * kMaxCols * kTileK);   // A; X halves; products
  uint32_t* tbase = reinterpret_cast<uint32_t*>(bars + 4);
  volatile int* dead = reinterpret_cast<volatile int*>(tbase + 1);   // a wait of this CTA has run out: no values from here on
  constexpr uint32_t kHalf = 2 * C * (kTileK / 2);                       // floats of a K half of the operand

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // known to be the warp's: uniform registers
  const int MB = a.n / kTileRows;
  const int mb = blockIdx.x / a.cs;
  const int j = blockIdx.x % a.cs;
  const volatile int* errv = a.err;
  if (tid == 0) {
    tc::mbar_init(&bars[0], 1);
    tc::mbar_init(&bars[1], kWorkers / 32);
    tc::mbar_init(&bars[2], kWorkers / 32);
    tc::mbar_init(&bars[3], 1);
    *dead = 0;
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc(tbase, 256);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tbase;
  if (tid == 0) {
    const float* at = a.A + ((size_t)mb * a.cs + j) * 2 * kATileFloats;
    tc::mbar_arrive_expect_tx(&bars[0], 4 * 2 * kATileFloats);
    tc::bulk_g2s(A_hi, at, 4 * kATileFloats, &bars[0]);
    tc::bulk_g2s(A_lo, at + kATileFloats, 4 * kATileFloats, &bars[0]);
  }
  bool ok = tc::mbar_wait(&bars[0], 0, 0xFFFFFFFFu);   // this CTA's own copy: never abandoned early
  __syncthreads();
  uint64_t* bar_x = &bars[1];       // one per K half
  uint64_t* bar_m = &bars[3];
  const uint64_t own_ns = 2 * a.wait_ns + tc::kWaitLimitNs;   // waits on this CTA's own warps outlast theirs on others

  if (warp == kWorkers / 32) {
    // 2. products, issued by a converged warp (descriptors in uniform registers)
    const uint32_t idesc_hx = tc::idesc_tf32(kM, 2 * C);   // A_hi x [X_hi | X_lo]
    const uint32_t idesc_lx = tc::idesc_tf32(kM, C);       // A_lo x X_hi
    const uint64_t ah = tc::smem_desc(A_hi, 128, (kTileK / 4) * 128), al = tc::smem_desc(A_lo, 128, (kTileK / 4) * 128);
    const uint64_t xx = tc::smem_desc(X_sm, 128, (kTileK / 8) * 128);
    for (int s = 0; s < a.steps; ++s) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool here = tc::mbar_wait(bar_x + h, (uint32_t)(s & 1), 0xFFFFFFFFu, nullptr, own_ns);
        ok = __all_sync(0xffffffffu, here) && ok;
        tc::tc_fence_after();
        if (ok && lane == 0 && *dead == 0) {
#pragma unroll
          for (int ks = 0; ks < kTileK / 16; ++ks) {
            const uint64_t x = xx + h * (kHalf / 4) + ks * 16;
            tc::mma_tf32(tmem, ah + (8 * h + ks) * 16, x, idesc_hx, h + ks > 0);
            tc::mma_tf32(tmem + 2 * C, al + (8 * h + ks) * 16, x, idesc_lx, h + ks > 0);
          }
        }
        __syncwarp();
      }
      if (lane == 0) tc::mma_commit(bar_m);
      __syncwarp();
    }
  } else {
    const int64_t rows = (int64_t)a.kg * a.n;
    // owner pairs: rows [rpc j, rpc j + rpc) of the row block, eight at a time, x 16 or 32 vectors
    const int groups = kTileRows / a.cs / 8;
    const int vg = 4 * warp + (lane >> 3);
    const bool owner = 4 * warp < C / 2;                          // a whole warp
    const int il0 = (kTileRows / a.cs) * j + (lane & 7);          // row of group 0 in the row block
    cpx<float> u_own[kMaxGroups];
#pragma unroll
    for (int q = 0; q < kMaxGroups; ++q) {
      const int i = mb * kTileRows + il0 + 8 * q;
      u_own[q] = (owner && q < groups && vg < a.kg) ? a.u[(size_t)(a.n0 & 1) * rows + (int64_t)vg * a.n + i]
                                                    : mk<float>(0.f, 0.f);
    }
    // State words of a slice: [K / 4][pair of the four][C] x (two K values); two neighbouring rows swap their
    // halves, so that each stores one column's two values.
    auto write_x = [&](int par, int i, cpx<float> u1, uint32_t number) {
      const bool odd = lane & 1;
      const float got = __shfl_xor_sync(0xffffffffu, odd ? u1.re : u1.im, 1);
      const int kk = i % kTileK, c = 2 * vg + (odd ? 1 : 0);
      float* x = a.X + ((size_t)par * a.cs + i / kTileK) * kXsFloats;
      words_store(x + ((kk >> 1) * C + c) * 4, odd ? got : u1.re, odd ? u1.im : got, number);
    };
    if (a.n0 == 0 && owner) {  // publish the initial state (later tiles find it from the previous tile)
#pragma unroll
      for (int q = 0; q < kMaxGroups; ++q)
        if (q < groups) write_x(0, mb * kTileRows + il0 + 8 * q, u_own[q], 1u);
    }
    constexpr int kUnits = (kTileK / 2) * C / 4 / kWorkers;   // groups of four K values of a half per thread: 2 or 4
    const int col = tid % C, kq0 = tid / C;
    // Every warp runs every step; after an error the waits return at once and the flag reports the failure.
    for (int s = 0; s < a.steps; ++s) {
      const int64_t n = a.n0 + s;
      const int par = (int)(n & 1);
      const uint32_t number = (uint32_t)(n + 1);
      // forcing of this step for the owned pairs: loads in flight during the products
      const cpx<float>* Fs = (a.F != nullptr && n < a.n_forced) ? a.F + (size_t)s * rows : nullptr;
      cpx<float> fv[kMaxGroups];
#pragma unroll
      for (int q = 0; q < kMaxGroups; ++q) {
        const int i = mb * kTileRows + il0 + 8 * q;
        fv[q] = mk<float>(0.f, 0.f);
        if (Fs != nullptr && owner && q < groups && vg < a.kg) {
          const float2 f = __ldcs(reinterpret_cast<const float2*>(Fs + (int64_t)vg * a.n + i));
          fv[q] = mk<float>(f.x, f.y);
        }
      }
      // 1. the state slice of this step
      {
        const float* xs = a.X + ((size_t)par * a.cs + j) * kXsFloats;
        const uint32_t want = number + ((a.stall && s == 0) ? (1u << 30) : 0u);
        auto at = [&](int h, int i) {   // load i of half h: unit i / 2, K pair i % 2
          return xs + (((kTileK / 8) * h + kq0 + (kWorkers / C) * (i >> 1)) * 2 + (i & 1)) * C * 4 + col * 4;
        };
        uint64_t w[2][2 * kUnits][2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < 2 * kUnits; ++i) words_load(at(h, i), w[h][i]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (!words_wait<2 * kUnits>(w[h], 2 * kUnits, want, [&](int i) { return at(h, i); }, errv, a.wait_ns)) {
            atomicExch(a.err, 2);
            *dead = 1;
          }
#pragma unroll
          for (int t = 0; t < kUnits; ++t) {
            float v[4], hi[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              v[e] = word_value(w[h][2 * t + (e >> 1)][e & 1]);
              hi[e] = tc::to_tf32(v[e]);
            }
            const int kk = 4 * (kq0 + (kWorkers / C) * t);
            float* x = X_sm + h * kHalf;
            *reinterpret_cast<float4*>(x + tc::kmajor_offset(col, kk, kTileK / 2) / 4) =
                make_float4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<float4*>(x + tc::kmajor_offset(C + col, kk, kTileK / 2) / 4) =
                make_float4(v[0] - hi[0], v[1] - hi[1], v[2] - hi[2], v[3] - hi[3]);
          }
          tc::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar_x + h)) : "memory");
        }
      }
      ok = tc::mbar_wait(bar_m, (uint32_t)(s & 1), 0xFFFFFFFFu, nullptr, own_ns) && ok;
      const bool live = ok && *dead == 0;   // else zeros go out and the state stays
      __syncwarp();
      tc::tc_fence_after();
      // 3. partial: hi*hi + hi*lo + lo*hi, one row and half of the columns per thread
      {
        constexpr int W = C / 2;
        const int row = 32 * (warp & 3) + lane, c0 = W * (warp >> 2);
        const uint32_t tl = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
        float x0[W], x1[W], x2[W];
        if constexpr (W == 32) {
          tc::tmem_ld32(tl, x0);
          tc::tmem_ld32(tl + C, x1);
          tc::tmem_ld32(tl + 2 * C, x2);
        } else {
          tc::tmem_ld16(tl, x0);
          tc::tmem_ld16(tl + C, x1);
          tc::tmem_ld16(tl + 2 * C, x2);
        }
        tc::tc_fence_before();
        // Neighbouring lanes hold a row of Re D and of Im D: they swap the products of one vector each, and the
        // sums of half as many values go out
        const bool odd = lane & 1;
        float* pb = a.part + (((size_t)par * MB + mb) * a.cs + j) * kPartFloats + ((size_t)(c0 / 4) * kM + row) * 4;
#pragma unroll
        for (int c = 0; c < W; c += 4) {
          float y[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) y[e] = x0[c + e] + x1[c + e] + x2[c + e];
          const float g0 = __shfl_xor_sync(0xffffffffu, odd ? y[0] : y[2], 1);
          const float g1 = __shfl_xor_sync(0xffffffffu, odd ? y[1] : y[3], 1);
          const float re = odd ? g0 - y[3] : y[0] - g1, im = odd ? g1 + y[2] : y[1] + g0;
          words_store(pb + (size_t)(c / 4) * kM * 4, live ? re : 0.f, live ? im : 0.f, number);
        }
      }
      // 4. owner: its rows of all partials of the row block for this step
      if (owner) {
        cpx<float>* Ys = (a.Y != nullptr && s >= a.y_first) ? a.Y + (size_t)s * rows : nullptr;
        const float* pbase = a.part + ((size_t)par * MB + mb) * a.cs * kPartFloats;
#pragma unroll
        for (int q = 0; q < kMaxGroups; ++q) {
          if (q < groups) {
            const int iloc = il0 + 8 * q;
            auto at = [&](int p) {
              return pbase + (size_t)p * kPartFloats + ((size_t)(vg >> 1) * kM + 2 * iloc + (vg & 1)) * 4;
            };
            uint64_t w[8][2];
#pragma unroll
            for (int p = 0; p < 8; ++p)
              if (p < a.cs) words_load(at(p), w[p]);
            bool got = live;
            if (!words_wait<8>(w, a.cs, number, at, errv, a.wait_ns)) {
              atomicExch(a.err, 2);
              *dead = 1;
              got = false;
            }
            __syncwarp();
            float pr = 0.f, pi = 0.f;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
              if (p < a.cs) {
                pr += word_value(w[p][0]);
                pi += word_value(w[p][1]);
              }
            }
            const int i = mb * kTileRows + iloc;
            const cpx<float> u0 = u_own[q];
            cpx<float> u1 = mk<float>(u0.re + pr + fv[q].re, u0.im + pi + fv[q].im);
            if (vg >= a.kg) u1 = mk<float>(0.f, 0.f);
            if (!got) u1 = u0;
            write_x(1 - par, i, u1, number + 1);
            if (Ys != nullptr && vg < a.kg)
              __stcs(reinterpret_cast<float2*>(Ys + (int64_t)vg * a.n + i), make_float2(u0.re, u0.im));
            u_own[q] = u1;
          }
        }
      }
    }
    // state at the end of the tile
    const int64_t nend = a.n0 + a.steps;
#pragma unroll
    for (int q = 0; q < kMaxGroups; ++q) {
      const int i = mb * kTileRows + il0 + 8 * q;
      if (owner && q < groups && vg < a.kg) a.u[(size_t)(nend & 1) * rows + (int64_t)vg * a.n + i] = u_own[q];
    }
  }
  if (!ok && lane == 0) atomicExch(a.err, 2);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

void (*march_kernel(int n, int kg))(TcMarchArgs) {
  if (n / kTileK == 8) return kg <= 16 ? dense_tc_march_kernel<32, 1> : dense_tc_march_kernel<64, 1>;
  return kg <= 16 ? dense_tc_march_kernel<32, 8> : dense_tc_march_kernel<64, 8>;
}

// Partial words of all CTAs, two step parities.
size_t part_bytes(int n) { return (size_t)2 * (n / kTileRows) * (n / kTileK) * kPartFloats * sizeof(float); }

// A tiles from the FP64 matrix (conj-transposed for the adjoint): tile (mb, j) rows
// r even: Re M[64 mb + r / 2][128 j + k], r odd: Im; hi/lo TF32 split.
__global__ void arrange_a_kernel(int n, int cs, const cpx<double>* __restrict__ M, bool conj_t, float* __restrict__ out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // over (mb, j, r, k)
  const int64_t total = (int64_t)(n / kTileRows) * cs * kM * kTileK;
  if (e >= total) return;
  const int k = (int)(e % kTileK);
  const int r = (int)((e / kTileK) % kM);
  const int j = (int)((e / ((int64_t)kTileK * kM)) % cs);
  const int mb = (int)(e / ((int64_t)kTileK * kM * cs));
  const int row = mb * kTileRows + (r >> 1), col = j * kTileK + k;
  const cpx<double> m = conj_t ? conjg(M[(int64_t)col * n + row]) : M[(int64_t)row * n + col];
  const double x = (r & 1) == 0 ? m.re : m.im;
  const float hi = tc::to_tf32((float)x);
  const float lo = (float)(x - (double)hi);
  float* tile = out + ((size_t)mb * cs + j) * 2 * kATileFloats;
  const uint32_t o = tc::kmajor_offset(r, k, kTileK) / 4;
  tile[o] = hi;
  tile[kATileFloats + o] = lo;
}

}  // namespace

// Shapes of the tensor-core kernels: n a multiple of 128 with CS = n / 128 K slices, and
// CS dividing the 64 rows of a row block (each of the CS CTAs of a row block owns
// 64 / CS of its rows): CS in {1, 2, 4, 8}, n in {128, 256, 512, 1024}.  Other n take
// the CUDA-core step.
static bool tc_shape_ok(int n) {
  if (n % kTileK != 0) return false;
  const int cs = n / kTileK;
  return cs >= 1 && cs <= 8 && kTileRows % cs == 0;
}

bool dense_tc_supported(rsv_operator op, int kg) {
  if (op->prec != RSV_PREC_FP32 || op->kind != RSV_OP_DENSE) return false;
  if (op->tc_disabled) return false;
  if (!tc_shape_ok((int)op->n) || kg > 32) return false;
  return op->tc_tiles[0] != nullptr;
}

size_t dense_tc_scratch_bytes(rsv_operator op) {
  return (size_t)2 * (op->n / kTileK) * 2 * kXTileFloats * sizeof(float);
}

// Build the hi/lo A tiles of D and D^H (after the FP64 propagator build).
rsv_status dense_tc_prepare(rsv_operator op, const void* d64_direct) {
  const int n = (int)op->n;
  if (op->prec != RSV_PREC_FP32 || !tc_shape_ok(n) || op->tc_disabled) return RSV_OK;
  const int cs = n / kTileK;
  const size_t floats = (size_t)(n / kTileRows) * cs * 2 * kATileFloats;
  for (int d = 0; d < 2; ++d) {
    if (!op->tc_tiles[d]) {
      cudaError_t e = cudaMalloc(&op->tc_tiles[d], floats * sizeof(float));
      if (e != cudaSuccess) return cuda_fail(e, "tensor-core tiles");
      op->dev.push_back(op->tc_tiles[d]);
    }
    const int64_t total = (int64_t)(n / kTileRows) * cs * kM * kTileK;
    arrange_a_kernel<<<(unsigned)((total + 255) / 256), 256, 0, op->stream>>>(
        n, cs, (const cpx<double>*)d64_direct, d == 1, (float*)op->tc_tiles[d]);
  }
  cudaError_t e = cudaFuncSetAttribute(dense_tc_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmemBytes);
  for (auto* k : {march_kernel(n, 16), march_kernel(n, 32)})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemPersistent);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "tensor-core tiles");
  // The persistent tile kernel needs all of its CTAs resident at once (one per SM).
  op->tc_persistent = false;
  const int MB = n / kTileRows;
  if (!op->tc_acc) {
    e = cudaMalloc(&op->tc_acc, part_bytes(n));
    if (e == cudaSuccess) op->dev.push_back(op->tc_acc);
    if (e != cudaSuccess) return cuda_fail(e, "tensor-core march buffers");
  }
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, march_kernel(n, 32), kMarchThreads, kSmemPersistent);
  if (e != cudaSuccess) {
    cudaGetLastError();
    per_sm = 0;
  }
  op->tc_max_clusters = per_sm * op->sm_count;  // resident CTAs
  const char* env = getenv("RSV_DENSE_PERSISTENT");
  op->tc_persistent = per_sm * op->sm_count >= MB * cs && !(env != nullptr && env[0] == '0');
  return RSV_OK;
}

// State words of the persistent kernel (two step parities).
size_t dense_tc_chain_x_bytes(rsv_operator op) { return (size_t)2 * (op->n / kTileK) * kXsFloats * sizeof(float); }

// A whole tile of steps in one persistent launch (requires op->tc_persistent).
cudaError_t dense_tc_march_tile(rsv_operator op, int kg, bool adjoint, int64_t n0, int steps, int64_t n_forced,
                                int y_first, void* state, const void* F, void* Y, void* xbuf) {
  const int n = (int)op->n;
  const int cs = n / kTileK;
  const int MB = n / kTileRows;
  TcMarchArgs a;
  a.A = (const float*)op->tc_tiles[adjoint ? 1 : 0];
  a.X = (float*)xbuf;
  a.part = (float*)op->tc_acc;
  a.u = (cpx<float>*)state;
  a.F = (const cpx<float>*)F;
  a.Y = (cpx<float>*)Y;
  a.n0 = n0;
  a.steps = steps;
  a.n_forced = n_forced;
  a.y_first = y_first;
  a.n = n;
  a.kg = kg;
  a.cs = cs;
  a.err = op->d_flag;
  a.wait_ns = op->wait_limit_ns;
  a.stall = op->test_stall_wait ? 1 : 0;
  cudaError_t e = cudaSuccess;
  if (n0 == 0) {
    e = cudaMemsetAsync(xbuf, 0, dense_tc_chain_x_bytes(op), op->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(op->tc_acc, 0, part_bytes(n), op->stream);
  }
  if (e != cudaSuccess) return e;
  march_kernel(n, kg)<<<MB * cs, kMarchThreads, kSmemPersistent, op->stream>>>(a);
  return cudaGetLastError();
}

// One step; xbuf holds two X operand sets (ping-pong by step parity).
cudaError_t dense_tc_step(rsv_operator op, int kg, bool adjoint, int64_t step, const void* uin, void* uout,
                          const void* F, void* Y, void* xbuf) {
  const int n = (int)op->n;
  const int cs = n / kTileK;
  const size_t xset = (size_t)cs * 2 * kXTileFloats;
  TcStepArgs a;
  a.A = (const float*)op->tc_tiles[adjoint ? 1 : 0];
  a.Xin = (const float*)xbuf + (size_t)(step & 1) * xset;
  a.Xout = (float*)xbuf + (size_t)((step + 1) & 1) * xset;
  a.uin = (const cpx<float>*)uin;
  a.uout = (cpx<float>*)uout;
  a.F = (const cpx<float>*)F;
  a.Y = (cpx<float>*)Y;
  a.n = n;
  a.kg = kg;
  a.cs = cs;
  a.err = op->d_flag;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((n / kTileRows) * cs), 1, 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = op->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, dense_tc_step_kernel, a);
}

}  // namespace rsv
