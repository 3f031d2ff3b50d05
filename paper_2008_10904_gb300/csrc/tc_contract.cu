// Forcing synthesis and DFT analysis on the tensor cores (FP32 mode).
//
// Both contractions of a time tile are real GEMMs after expanding complex
// numbers into (re, im) pairs:
//   synthesis  F[tau][r]     = sum_j W[tau][j] C[j][r]          (Sec. 2.3, Eq. forceFseries)
//   analysis   acc[j][r]    += sum_s conj(W[s][j]) Y[s][r]       (Sec. 2.1, Eq. fourier)
// with W the exact twiddles of the tile.  The M dimension is the long one
// (state rows r, 128 per CTA), N the output columns (stage times or
// frequencies, re/im expanded, <= 512, accumulated in tensor memory), and K
// the contracted one (frequencies or tile steps, re/im expanded).
//
// The twiddle operand B (N x K) is the same for every CTA: one small kernel
// builds it per tile in global memory, already TF32 hi/lo split and in the
// K-major no-swizzle operand layout, 16 K-columns per chunk.  Each CTA streams
// K in chunks of 16 through two shared-memory stages: threads read its 128
// rows of the long operand (coalesced along r), split them into TF32 hi/lo
// and store them K-major; one thread bulk-copies the B chunk and issues the
// MMAs (3 per K-step: hi*hi, hi*lo, lo*hi).  The epilogue reads tensor memory
// (one row per thread) and writes F, or adds the tile's sums into the FP64
// accumulators.  Waits are bounded; a timeout sets the error flag.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "rsv_ops.h"
#include "tc_ptx.h"

namespace rsv {
namespace {

constexpr int kRowsCta = 128;
constexpr int kKc = 16;                              // K columns per chunk
constexpr int kMaxN = 512;
constexpr uint32_t kAStageFloats = kRowsCta * kKc;   // per hi / lo
constexpr uint32_t kBStageFloats = kMaxN * kKc;      // per hi / lo (N padded to 512)
constexpr uint32_t kSmem = 4 * 2 * (2 * kAStageFloats + 2 * kBStageFloats) + 128;
constexpr uint32_t kTries = 1u << 24;

enum Mode { SYNTH_C = 0, SYNTH_R = 1, ANAL_C = 2, ANAL_R = 3 };

struct ContractArgs {
  int mode;
  int64_t rows;
  int N;                   // output columns (multiple of 16, <= 512)
  int K;                   // contracted columns (multiple of 16)
  int n_tau;               // synthesis: stage times in this call
  int tau0;                // synthesis: first stage time of this call
  int n_omega;
  const void* src;         // coefficients [n_omega][coef_stride] or snapshots [steps][rows]
  int64_t src_stride;
  int s0, s1;              // analysis: valid tile steps [s0, s1)
  const float* B;          // [K / 16][sub-tile of up to 256 columns][hi, lo][columns x 16] pre-split twiddles
  void* out;               // synthesis: F [n_tau][rows]; analysis: acc (cpx<double>) [n_omega][acc_stride]
  int64_t acc_stride;
  int seg;                 // K chunks summed in one tensor-memory accumulator (pipelined kernel)
  int* err;
};

// The long operand of one K chunk as this thread's share, loaded into registers:
// complex modes: 4 (re, im) pairs = 4 rows x one contracted pair index each;
// real analysis: 8 values.  Zero outside the valid range.
struct AShare {
  float v[8];
};

__device__ __forceinline__ void load_share(const ContractArgs& a, int64_t r0, int kc, int tid, AShare& sh) {
  if (a.mode == ANAL_R) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = tid + 256 * q;
      const int kk = e >> 7, rr = e & 127;
      const int s = kc * kKc + kk;
      const int64_t r = r0 + rr;
      sh.v[q] = (r < a.rows && s >= a.s0 && s < a.s1) ? __ldg(reinterpret_cast<const float*>(a.src) + (int64_t)s * a.rows + r)
                                                        : 0.f;
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int e = tid + 256 * q;
    const int jj = e >> 7, rr = e & 127;
    const int idx = kc * (kKc / 2) + jj;  // frequency (synthesis) or tile step (analysis)
    const int64_t r = r0 + rr;
    bool valid = r < a.rows;
    int64_t off;
    if (a.mode == ANAL_C) {
      valid = valid && idx >= a.s0 && idx < a.s1;
      off = (int64_t)idx * a.rows + r;
    } else {
      valid = valid && idx < a.n_omega;
      off = (int64_t)idx * a.src_stride + r;
    }
    const float2 c = valid ? __ldg(reinterpret_cast<const float2*>(a.src) + off) : make_float2(0.f, 0.f);
    sh.v[2 * q] = c.x;
    sh.v[2 * q + 1] = c.y;
  }
}

__device__ __forceinline__ void store_share(const ContractArgs& a, int tid, const AShare& sh, float* A_hi, float* A_lo) {
  if (a.mode == ANAL_R) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = tid + 256 * q;
      const int kk = e >> 7, rr = e & 127;
      const float hi = tc::to_tf32(sh.v[q]);
      const uint32_t o = tc::kmajor_offset(rr, kk, kKc) / 4;
      A_hi[o] = hi;
      A_lo[o] = sh.v[q] - hi;
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int e = tid + 256 * q;
    const int jj = e >> 7, rr = e & 127;
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      const float x = sh.v[2 * q + part];
      const float hi = tc::to_tf32(x);
      const uint32_t o = tc::kmajor_offset(rr, 2 * jj + part, kKc) / 4;
      A_hi[o] = hi;
      A_lo[o] = x - hi;
    }
  }
}

__global__ void __launch_bounds__(256, 1) tc_contract_kernel(ContractArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  float* sA = reinterpret_cast<float*>(smem);                    // [2 stages][hi, lo][kAStageFloats]
  float* sB = sA + 2 * 2 * kAStageFloats;                        // [2 stages][hi, lo][kBStageFloats]
  uint64_t* bars = reinterpret_cast<uint64_t*>(sB + 2 * 2 * kBStageFloats);  // [0,1] B loaded, [2,3] MMA done
  uint32_t* tbase = reinterpret_cast<uint32_t*>(bars + 4);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t r0 = (int64_t)blockIdx.x * kRowsCta;
  if (tid == 0) {
    for (int b = 0; b < 4; ++b) tc::mbar_init(&bars[b], 1);
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc(tbase, 512);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tbase;
  const int chunks = a.K / kKc;
  const uint32_t sbo_a = (kKc / 4) * 128, sbo_b = (kKc / 4) * 128;
  const uint32_t bchunk_bytes = 4u * (uint32_t)a.N * kKc;  // one of hi / lo, only the N used rows
  bool ok = true;
  uint32_t mma_phase[2] = {0, 0};
  uint32_t load_phase[2] = {0, 0};
  AShare nxt;
  load_share(a, r0, 0, tid, nxt);
  for (int kc = 0; kc < chunks; ++kc) {
    const int st = kc & 1;
    float* A_hi = sA + st * 2 * kAStageFloats;
    float* A_lo = A_hi + kAStageFloats;
    float* B_hi = sB + st * 2 * kBStageFloats;
    float* B_lo = B_hi + kBStageFloats;
    const AShare cur = nxt;
    if (kc + 1 < chunks) load_share(a, r0, kc + 1, tid, nxt);  // in flight during this chunk
    if (kc >= 2) {  // the MMAs of chunk kc - 2 read this stage
      ok = tc::mbar_wait(&bars[2 + st], mma_phase[st], kTries) && ok;
      mma_phase[st] ^= 1;
    }
    if (tid == 0) {
      const float* bsrc = a.B + (size_t)kc * 2 * a.N * kKc;
      tc::mbar_arrive_expect_tx(&bars[st], 2 * bchunk_bytes);
      for (int nh = 0; nh < a.N; nh += 256) {
        const int nf = min(256, a.N - nh) * kKc;
        tc::bulk_g2s(B_hi + nh * kKc, bsrc, 4 * nf, &bars[st]);
        tc::bulk_g2s(B_lo + nh * kKc, bsrc + nf, 4 * nf, &bars[st]);
        bsrc += 2 * nf;
      }
    }
    store_share(a, tid, cur, A_hi, A_lo);
    tc::fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0) {
      ok = tc::mbar_wait(&bars[st], load_phase[st], kTries) && ok;
      tc::tc_fence_after();
      if (ok) {
        for (int ks = 0; ks < kKc / 8; ++ks) {
          const uint64_t ah = tc::smem_desc(reinterpret_cast<char*>(A_hi) + ks * 256, 128, sbo_a);
          const uint64_t al = tc::smem_desc(reinterpret_cast<char*>(A_lo) + ks * 256, 128, sbo_a);
          for (int nh = 0; nh < a.N; nh += 256) {
            const int nn = min(256, a.N - nh);
            const uint32_t idesc = tc::idesc_tf32(128, (uint32_t)nn);
            const uint64_t bh = tc::smem_desc(reinterpret_cast<char*>(B_hi) + ks * 256 + (nh / 8) * sbo_b, 128, sbo_b);
            const uint64_t bl = tc::smem_desc(reinterpret_cast<char*>(B_lo) + ks * 256 + (nh / 8) * sbo_b, 128, sbo_b);
            const uint32_t d = tmem + (uint32_t)nh;
            tc::mma_tf32(d, ah, bh, idesc, kc > 0 || ks > 0);
            tc::mma_tf32(d, ah, bl, idesc, true);
            tc::mma_tf32(d, al, bh, idesc, true);
          }
        }
        tc::mma_commit(&bars[2 + st]);
      } else {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&bars[2 + st])) : "memory");
      }
    }
    load_phase[st] ^= 1;
  }
  // wait for the last chunks' MMAs
  for (int st = 0; st < 2; ++st) {
    const int issued = chunks > st ? (chunks - 1 - st) / 2 + 1 : 0;   // commits on this stage
    const int waited = chunks > st + 2 ? (chunks - 1 - st) / 2 : 0;   // waits done in the loop
    if (issued > waited) ok = tc::mbar_wait(&bars[2 + st], mma_phase[st], kTries) && ok;
  }
  tc::tc_fence_after();
  // epilogue: warps 0-3 own TMEM lanes (rows) 0-127
  if (warp < 4) {
    const int64_t r = r0 + 32 * warp + lane;
    for (int c = 0; c < a.N; c += 16) {
      float v[16];
      tc::tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c, v);
      if (!ok || r >= a.rows) continue;
      if (a.mode == SYNTH_C) {
        cpx<float>* F = reinterpret_cast<cpx<float>*>(a.out);
#pragma unroll
        for (int q = 0; q < 16; q += 2) {
          const int tau = (c + q) >> 1;
          if (tau < a.n_tau) F[(int64_t)(a.tau0 + tau) * a.rows + r] = mk<float>(v[q], v[q + 1]);
        }
      } else if (a.mode == SYNTH_R) {
        float* F = reinterpret_cast<float*>(a.out);
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const int tau = c + q;
          if (tau < a.n_tau) F[(int64_t)(a.tau0 + tau) * a.rows + r] = v[q];
        }
      } else {
        // 8 complex accumulators per TMEM load: issue the 8 FP64 reads before any add / write
        cpx<double>* __restrict__ acc = reinterpret_cast<cpx<double>*>(a.out);
        double2 old[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int j = (c >> 1) + q;
          old[q] = j < a.n_omega ? __ldcg(reinterpret_cast<const double2*>(acc + (int64_t)j * a.acc_stride + r))
                                 : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int j = (c >> 1) + q;
          if (j < a.n_omega)
            __stcg(reinterpret_cast<double2*>(acc + (int64_t)j * a.acc_stride + r),
                   make_double2(old[q].x + (double)v[2 * q], old[q].y + (double)v[2 * q + 1]));
        }
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
  if (!ok && tid == 0) atomicExch(a.err, 2);
}

// ---------------------------------------------------------------------------
// Pipelined persistent variant (long operand streamed by bulk copies).
//
// One CTA per SM walks the 128-row tiles blockIdx.x, blockIdx.x + gridDim.x, ...
// with warp roles connected by mbarrier rings:
//   warp 12 (one thread) producer: copies each K chunk of the long operand in its
//                        storage precision into an 8-deep raw ring, one tensor
//                        copy per chunk;
//   warp 14 (one thread) producer: bulk-copies the chunk's pre-split twiddles
//                        into a 4-deep B ring, one copy per chunk;
//   warps 0-3            converters: one row each, raw value -> TF32 hi / lo, into
//                        tensor memory where at most 96 columns leave room for it
//                        (4 stages), else in the K-major operand layout in shared
//                        memory (2 stages);
//   warp 13              MMA issuer: 3 TF32 MMAs per K-step and N half into the
//                        tile's tensor-memory accumulator, commits release the
//                        operand stages and, after the last chunk, the tile;
//   warps 4-11           epilogue: two warps per tensor-memory lane quadrant,
//                        each taking half of the columns, 32 columns per load;
//                        tensor memory -> F, or += FP64 accumulators; then
//                        release the accumulator for the next tile.
// The chunk sequence runs on across tiles, so the next tile's operands stream
// in during the current tile's epilogue.  Every wait is bounded and also
// returns once another role has aborted; on abort the producer and the MMA
// issuer drain what they issued (bounded) before the CTA frees tensor memory.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int round16c(int x) { return (x + 15) / 16 * 16; }

// Ring depths: the twiddle operand of every sub-tile streams from L2 (about 512 KB per row tile), so
// its ring is four chunks deep; a slot holds one sub-tile's 256 rows (hi and lo), half of a global
// chunk.  The raw long-operand ring is eight chunks deep.  Total 224.25 KB of shared memory.
constexpr int kRawRing = 8;
constexpr int kAStages = 2;
constexpr int kBRing = 4;
constexpr uint32_t kBRingFloats = 256 * kKc;          // per hi / lo: one sub-tile's rows
constexpr uint32_t kRawBytes = kRowsCta * kKc * 4;   // 128 rows x 16 real K values
constexpr int kPipeThreads = 480;                    // 15 warps, roles below

struct PipeBars {
  uint64_t raw_full[kRawRing], raw_empty[kRawRing];
  uint64_t a_full[kBRing], b_full[kBRing];
  uint64_t empty[kBRing];               // products of chunk g done: empty[g % kBRing]
  uint64_t acc_full[2], acc_empty[2];   // two tensor-memory accumulators of 256 columns
  int abort_flag;
};

// the barriers sit behind the operand rings; their reserve is sizeof(PipeBars) rounded up
constexpr uint32_t kPipeBarBytes = (uint32_t)((sizeof(PipeBars) + 127) / 128 * 128);
constexpr uint32_t kPipeSmem =
    kRawRing * kRawBytes + kAStages * 2 * kAStageFloats * 4 + kBRing * 2 * kBRingFloats * 4 + kPipeBarBytes;
// dynamic shared memory plus up to 1 KB for the static variable and the 1024-byte alignment
static_assert(kPipeSmem + 1024 <= 232448, "pipelined contraction exceeds the shared memory of a CTA");

__device__ __forceinline__ bool pwait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  return tc::mbar_wait(bar, parity, 0xFFFFFFFFu, abort_flag);
}

// One warp waits for two barriers; the same answer in every lane.
__device__ __forceinline__ bool pwait2(uint64_t* b0, uint32_t p0, uint64_t* b1, uint32_t p1, volatile int* abort_flag) {
  uint64_t t0 = 0;
  for (uint32_t i = 0;; ++i) {
    const bool d0 = tc::mbar_try(b0, p0), d1 = tc::mbar_try(b1, p1);
    if (__all_sync(0xffffffffu, d0 && d1)) return true;
    if ((i & 63) == 63) {
      const uint64_t now = tc::global_ns();
      if (t0 == 0) t0 = now;
      if (__any_sync(0xffffffffu, *abort_flag != 0 || now - t0 > tc::kWaitLimitNs)) return false;
    }
  }
}

__device__ __forceinline__ void pabort(PipeBars* pb, int* err) {
  *reinterpret_cast<volatile int*>(&pb->abort_flag) = 1;
  atomicExch(err, 2);
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}

// Raw layout of one chunk in shared memory: complex modes [8][128] float2 (pair index jj = frequency or
// step within the chunk), real analysis [16][128] float: one box of the tensor map, 8 KB.  Rows and pair
// indices outside the operand come as zeros; snapshots of steps that are not analysed are masked by the
// converters.  (Row slices by single bulk copies of 512 or 1024 bytes took about 94 cycles each, 1500 per
// chunk, and bounded the analysis: 54 ms of the 2-D 1024 x 512 x 16 march.)
__device__ __forceinline__ void issue_raw(const ContractArgs& a, const CUtensorMap* map, int64_t r0, int kc,
                                          unsigned char* raw, uint64_t* bar) {
  const bool real = a.mode == ANAL_R;
  tc::mbar_arrive_expect_tx(bar, kRawBytes);
  tc::tensor_g2s(raw, map, (int32_t)(real ? r0 : 2 * r0), kc * (real ? kKc : kKc / 2), bar);
}

// FP32 -> TF32, round to nearest with ties away from zero, as to_tf32 (integer instructions; a NaN's
// remainder x - hi is NaN still).
__device__ __forceinline__ float tf32_hi(float x) { return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u); }

// One row of a chunk.  A warp converts a chunk per scheduler, so its instruction count is the chunk's time:
// chunks that are valid as a whole take no test per value.
__device__ __forceinline__ void load_row(const ContractArgs& a, bool row_ok, int kc, int rr, const unsigned char* raw,
                                         float x[kKc]) {
  if (a.mode == ANAL_R) {
    const float* rv = reinterpret_cast<const float*>(raw) + rr;
    const int s = kc * kKc;
#pragma unroll
    for (int kk = 0; kk < kKc; ++kk) x[kk] = rv[kk * kRowsCta];
    if (!(row_ok && s >= a.s0 && s + kKc <= a.s1)) {
#pragma unroll
      for (int kk = 0; kk < kKc; ++kk) x[kk] = (row_ok && s + kk >= a.s0 && s + kk < a.s1) ? x[kk] : 0.f;
    }
  } else {
    const float2* rv = reinterpret_cast<const float2*>(raw) + rr;
    const int idx = kc * (kKc / 2);
    const int lo = a.mode == ANAL_C ? a.s0 : 0, hi = a.mode == ANAL_C ? a.s1 : a.n_omega;
#pragma unroll
    for (int jj = 0; jj < kKc / 2; ++jj) {
      const float2 c = rv[jj * kRowsCta];
      x[2 * jj] = c.x;
      x[2 * jj + 1] = c.y;
    }
    if (!(row_ok && idx >= lo && idx + kKc / 2 <= hi)) {
#pragma unroll
      for (int k = 0; k < kKc; ++k) x[k] = (row_ok && idx + k / 2 >= lo && idx + k / 2 < hi) ? x[k] : 0.f;
    }
  }
}
__device__ __forceinline__ void store_row(const float x[kKc], int rr, float* A_hi, float* A_lo) {
  // K-major core matrices: 4 consecutive K values of one row are one 16-byte vector
#pragma unroll
  for (int q = 0; q < kKc / 4; ++q) {
    float4 h, l;
    h.x = tf32_hi(x[4 * q]);
    h.y = tf32_hi(x[4 * q + 1]);
    h.z = tf32_hi(x[4 * q + 2]);
    h.w = tf32_hi(x[4 * q + 3]);
    l = make_float4(x[4 * q] - h.x, x[4 * q + 1] - h.y, x[4 * q + 2] - h.z, x[4 * q + 3] - h.w);
    const uint32_t o = tc::kmajor_offset(rr, 4 * q, kKc) / 4;
    *reinterpret_cast<float4*>(A_hi + o) = h;
    *reinterpret_cast<float4*>(A_lo + o) = l;
  }
}

// The same in tensor memory: columns [0, 16) high parts, [16, 32) low parts.
__device__ __forceinline__ void store_row_tmem(float x[kKc], uint32_t ta) {
  float h[kKc];
#pragma unroll
  for (int k = 0; k < kKc; ++k) {
    h[k] = tf32_hi(x[k]);
    x[k] -= h[k];
  }
  tc::tmem_st16(ta, h);
  tc::tmem_st16(ta + 16, x);
  tc::tmem_wait_st();
}

// FP32 -> FP64 with integer instructions, for zero and normal values (exact).  FP64 instructions issue once
// per 19 cycles and SM, conversions among them, and the accumulation needs one FP64 addition per value
// anyway: converting there as well held the FP64 pipe 48% busy and the epilogue at twice its loads' time.
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x), m = u & 0x7fffffffu;
  const uint32_t hi = m == 0u ? 0u : (m >> 3) + 0x38000000u;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}

// FP64 accumulators of 16 output columns from column c on (8 frequencies) of row r.
__device__ __forceinline__ void load_acc16(const ContractArgs& a, int64_t r, int c, double2 old[8]) {
  const double2* acc = reinterpret_cast<const double2*>(a.out);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int j = (c >> 1) + q;
    old[q] = (r < a.rows && j < a.n_omega) ? __ldcs(acc + (int64_t)j * a.acc_stride + r) : make_double2(0.0, 0.0);
  }
}
// += v, the columns' sums over the tile or a segment of it.
__device__ __forceinline__ void add_acc16(double2 old[8], const float v[16]) {
  uint32_t top = 0, low = 0xffffffffu;
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const uint32_t m = __float_as_uint(v[q]) & 0x7fffffffu;
    top = max(top, m);
    low = min(low, m - 1u);               // zero counts as the largest
  }
  const bool plain = top < 0x7f800000u && low >= 0x007fffffu;   // no infinity, NaN or denormal value
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    old[q].x += plain ? widen(v[2 * q]) : (double)v[2 * q];
    old[q].y += plain ? widen(v[2 * q + 1]) : (double)v[2 * q + 1];
  }
}
__device__ __forceinline__ void store_acc16(const ContractArgs& a, int64_t r, int c, const double2 old[8]) {
  if (r >= a.rows) return;
  double2* acc = reinterpret_cast<double2*>(a.out);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int j = (c >> 1) + q;
    if (j < a.n_omega) __stcs(acc + (int64_t)j * a.acc_stride + r, old[q]);
  }
}

// Accumulator columns [c0, c1) of row r (output columns coff + c) to F, 32 columns per tensor-memory load.
template <int W>
__device__ __forceinline__ void epilogue_cols(const ContractArgs& a, int64_t r, uint32_t tq, int cl, int coff,
                                              bool row_ok) {
  float v[32];
  if (W == 32) tc::tmem_ld32(tq + (uint32_t)cl, v);
  else tc::tmem_ld16(tq + (uint32_t)cl, v);
  if (!row_ok) return;
  const int c = coff + cl;
  // whole groups of stage times step a pointer; only the last one tests each
  if (a.mode == SYNTH_C) {
    const int tau = c >> 1;
    float2* F = reinterpret_cast<float2*>(a.out) + (int64_t)(a.tau0 + tau) * a.rows + r;
    if (tau + W / 2 <= a.n_tau) {
#pragma unroll
      for (int q = 0; q < W; q += 2, F += a.rows) __stcs(F, make_float2(v[q], v[q + 1]));
    } else {
#pragma unroll
      for (int q = 0; q < W; q += 2, F += a.rows)
        if (tau + q / 2 < a.n_tau) __stcs(F, make_float2(v[q], v[q + 1]));
    }
  } else {
    float* F = reinterpret_cast<float*>(a.out) + (int64_t)(a.tau0 + c) * a.rows + r;
    if (c + W <= a.n_tau) {
#pragma unroll
      for (int q = 0; q < W; ++q, F += a.rows) __stcs(F, v[q]);
    } else {
#pragma unroll
      for (int q = 0; q < W; ++q, F += a.rows)
        if (c + q < a.n_tau) __stcs(F, v[q]);
    }
  }
}

__device__ __forceinline__ void epilogue_tile(const ContractArgs& a, int64_t r, uint32_t tq, int c0, int c1,
                                              int coff) {
  const bool row_ok = r < a.rows;
  int c = c0;
  for (; c + 32 <= c1; c += 32) epilogue_cols<32>(a, r, tq, c, coff, row_ok);
  if (c < c1) epilogue_cols<16>(a, r, tq, c, coff, row_ok);
}

// kTA: the converted operand in tensor memory (at most 96 columns of a segment, one column sub-tile).  In shared
// memory a chunk of an analysis with 64 columns moves 76 KB: raw in and out, converted in, read by three
// products each, twiddles; at 128 bytes per cycle that is most of its time.  In tensor memory 36 KB are left:
// analysis of the 2-D 1024 x 512 x 16 march 26.4 -> 23.8 ms, of 64 1-D instances x 8 vectors 14.4 -> 12.8 ms.
constexpr uint32_t kTaCols = 96;                       // columns of a segment's accumulator
constexpr uint32_t kTaBase = 4 * kTaCols;              // two accumulators of two segments, then the operand's stages
static_assert(kTaBase + kBRing * 2 * kKc <= 512, "tensor memory");

template <bool kTA>
__global__ void __launch_bounds__(kPipeThreads, 1) tc_contract_pipe_kernel(ContractArgs a,
                                                                           const __grid_constant__ CUtensorMap raw_map) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* raw = smem;                                                     // [kRawRing][kRawBytes]
  float* sA = reinterpret_cast<float*>(smem + kRawRing * kRawBytes);             // [kAStages][hi, lo][..]
  float* sB = sA + kAStages * 2 * kAStageFloats;                                 // [kBRing][hi, lo][..]
  PipeBars* pb = reinterpret_cast<PipeBars*>(sB + kBRing * 2 * kBRingFloats);
  __shared__ uint32_t tbase;
  volatile int* abort_flag = &pb->abort_flag;

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // known to be the warp's: uniform registers
  if (tid == 0) {
    for (int i = 0; i < kRawRing; ++i) {
      tc::mbar_init(&pb->raw_full[i], 1);
      tc::mbar_init(&pb->raw_empty[i], 128);
    }
    for (int i = 0; i < kBRing; ++i) {
      tc::mbar_init(&pb->a_full[i], 128);
      tc::mbar_init(&pb->b_full[i], 1);
      tc::mbar_init(&pb->empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&pb->acc_full[i], 1);
      tc::mbar_init(&pb->acc_empty[i], 256);
    }
    pb->abort_flag = 0;
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc(&tbase, 512);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tbase;
  const int chunks = a.K / kKc;
  const int64_t tiles = (a.rows + kRowsCta - 1) / kRowsCta;
  // Each row tile runs as one or two column sub-tiles of at most 256 columns; sub-tiles alternate
  // between the two accumulators, so the products of one overlap the epilogue of the previous one.
  const int nsub = !kTA && a.N > 256 ? 2 : 1;
  constexpr uint32_t kSegCols = kTA ? kTaCols : 128u, kBufCols = 2 * kSegCols;
  constexpr int kStages = kTA ? kBRing : kAStages;     // of the converted operand

  if (warp == 12) {
    if (lane == 0) {  // producer of the long operand
      uint32_t g = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        const int64_t r0 = t * kRowsCta;
        for (int h = 0; h < nsub && ok; ++h) {   // the second sub-tile re-reads the rows from L2
          for (int kc = 0; kc < chunks; ++kc, ++g) {
            const uint32_t rs = g % kRawRing, ru = g / kRawRing;
            if (ru > 0 && !pwait(&pb->raw_empty[rs], (ru - 1) & 1, abort_flag)) { ok = false; break; }
            issue_raw(a, &raw_map, r0, kc, raw + rs * kRawBytes, &pb->raw_full[rs]);
          }
        }
      }
      if (!ok) {
        pabort(pb, a.err);
        for (uint32_t q = 0; q < kRawRing && q < g; ++q) {  // the last copies land on their full barriers
          const uint32_t gg = g - 1 - q;
          tc::mbar_wait(&pb->raw_full[gg % kRawRing], (gg / kRawRing) & 1, kTries);
        }
      }
    }
  } else if (warp == 14) {
    if (lane == 0) {  // producer of the twiddle operand (the same chunks for every tile)
      uint32_t g = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        for (int h = 0; h < nsub && ok; ++h) {
          // a sub-tile's rows of a chunk, hi and lo, are one contiguous run of 8-row core-matrix groups
          const int nn = h == 0 ? min(256, a.N) : a.N - 256;
          const uint32_t bytes = 4u * (uint32_t)nn * kKc;
          for (int kc = 0; kc < chunks; ++kc, ++g) {
            const uint32_t bs = g % kBRing, bu = g / kBRing;
            if (bu > 0 && !pwait(&pb->empty[bs], (bu - 1) & 1, abort_flag)) { ok = false; break; }
            tc::mbar_arrive_expect_tx(&pb->b_full[bs], 2 * bytes);
            tc::bulk_g2s(sB + bs * 2 * kBRingFloats, a.B + ((size_t)kc * a.N + 256 * h) * 2 * kKc, 2 * bytes, &pb->b_full[bs]);
          }
        }
      }
      if (!ok) {
        pabort(pb, a.err);
        for (uint32_t q = 0; q < kBRing && q < g; ++q) {
          const uint32_t gg = g - 1 - q;
          tc::mbar_wait(&pb->b_full[gg % kBRing], (gg / kBRing) & 1, kTries);
        }
      }
    }
  } else if (warp == 13) {
    // MMA issuer: the whole warp walks the chunks, so that addresses and descriptors stay in uniform
    // registers: with the loop in one lane a chunk's six products took 680 cycles to issue (those analyses
    // 31.0 and 16.4 ms, 28.8 and 15.6 with one wait and one copy less per chunk, 26.4 and 14.4 like this)
    uint32_t g = 0, tt = 0;
    bool ok = true;
    const bool issue = lane == 0;
    const uint64_t desc_a = tc::smem_desc(sA, 128, (kKc / 4) * 128), desc_b = tc::smem_desc(sB, 128, (kKc / 4) * 128);
    for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      for (int h = 0; h < nsub; ++h, ++tt) {
        const uint32_t buf = tt & 1, use = tt >> 1;
        if (use > 0 && !__all_sync(0xffffffffu, pwait(&pb->acc_empty[buf], (use - 1) & 1, abort_flag))) { ok = false; break; }
        tc::tc_fence_after();
        const int nn = h == 0 ? min(256, a.N) : a.N - 256;
        const uint32_t idesc = tc::idesc_tf32(128, (uint32_t)nn);
        const uint32_t d = tmem + buf * kBufCols;
        for (int kc = 0; kc < chunks; ++kc, ++g) {
          const uint32_t as = g % kStages, au = g / kStages;
          const uint32_t bs = g % kBRing, bu = g / kBRing;
          if (!pwait2(&pb->a_full[as], au & 1, &pb->b_full[bs], bu & 1, abort_flag)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const int seg0 = kc >= a.seg ? a.seg : 0;            // first chunk of the segment
          const uint32_t ds = d + (seg0 > 0 ? kSegCols : 0u);
          // start addresses (16-byte units) are the descriptors' low bits
          const uint64_t ah = desc_a + as * (2 * kAStageFloats / 4), al = ah + kAStageFloats / 4;
          const uint64_t bh = desc_b + bs * (2 * kBRingFloats / 4), bl = bh + nn * (kKc / 4);
          if (kTA) {
            const uint32_t ta = tmem + kTaBase + as * (2 * kKc);
            if (issue) {
              tc::mma_tf32_ta(ds, ta, bh, idesc, kc > seg0);
              tc::mma_tf32_ta(ds, ta, bl, idesc, true);
              tc::mma_tf32_ta(ds, ta + kKc, bh, idesc, true);
              tc::mma_tf32_ta(ds, ta + 8, bh + 16, idesc, true);
              tc::mma_tf32_ta(ds, ta + 8, bl + 16, idesc, true);
              tc::mma_tf32_ta(ds, ta + kKc + 8, bh + 16, idesc, true);
              tc::mma_commit(&pb->empty[bs]);
            }
          } else if (issue) {
            tc::mma_tf32(ds, ah, bh, idesc, kc > seg0);
            tc::mma_tf32(ds, ah, bl, idesc, true);
            tc::mma_tf32(ds, al, bh, idesc, true);
            tc::mma_tf32(ds, ah + 16, bh + 16, idesc, true);
            tc::mma_tf32(ds, ah + 16, bl + 16, idesc, true);
            tc::mma_tf32(ds, al + 16, bh + 16, idesc, true);
            tc::mma_commit(&pb->empty[bs]);   // frees both operands
          }
          __syncwarp();
        }
        if (!ok) break;
        if (issue) tc::mma_commit(&pb->acc_full[buf]);
        __syncwarp();
      }
    }
    if (!ok && issue) {
      pabort(pb, a.err);
      // every MMA issued so far completes before tensor memory is freed: a commit after them
      // completes the next phase of the current sub-tile's accumulator barrier
      tc::mma_commit(&pb->acc_full[tt & 1]);
      tc::mbar_wait(&pb->acc_full[tt & 1], (tt >> 1) & 1, kTries);
    }
  } else if (warp < 4) {  // converters: one row each
    const int rr = tid;
    uint32_t g = 0;
    bool ok = true;
    for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const int64_t r0 = t * kRowsCta;
      for (int h = 0; h < nsub && ok; ++h) {
        for (int kc = 0; kc < chunks; ++kc, ++g) {
          const uint32_t rs = g % kRawRing, ru = g / kRawRing;
          const uint32_t as = g % kStages, gp = g - kStages;   // gp: the chunk that used the stage before
          bool got = pwait(&pb->raw_full[rs], ru & 1, abort_flag);
          if (got && g >= kStages) got = pwait(&pb->empty[gp % kBRing], (gp / kBRing) & 1, abort_flag);
          if (kTA) got = __all_sync(0xffffffffu, got);   // the stores to tensor memory take whole warps
          if (!got) { ok = false; break; }
          float x[kKc];
          load_row(a, r0 + rr < a.rows, kc, rr, raw + rs * kRawBytes, x);
          if (kTA) {
            tc::tc_fence_after();
            store_row_tmem(x, tmem + kTaBase + as * (2 * kKc) + ((uint32_t)(32 * warp) << 16));
            tc::tc_fence_before();
          } else {
            float* A_hi = sA + as * 2 * kAStageFloats;
            store_row(x, rr, A_hi, A_hi + kAStageFloats);
            tc::fence_proxy_async_smem();
          }
          mbar_arrive(&pb->a_full[as]);
          mbar_arrive(&pb->raw_empty[rs]);
        }
      }
    }
    if (!ok) pabort(pb, a.err);
  } else if (warp >= 4 && warp < 12) {  // epilogue: TMEM lane quadrant warp % 4, one half of the columns
    const int q = warp & 3;
    const bool anal = a.mode == ANAL_C || a.mode == ANAL_R;
    uint32_t tt = 0;
    bool ok = true;
    // first column of this warp's half and one past its last in column sub-tile h
    auto half_cols = [&](int h, int* c0, int* c1) {
      const int nn = h == 0 ? min(256, a.N) : a.N - 256;
      const int half = round16c((nn + 1) / 2);
      *c0 = warp < 8 ? 0 : half;
      *c1 = warp < 8 ? half : nn;
    };
    // analysis: the accumulators of the next 16 columns, of this tile or the next one, are in flight while
    // the current ones are added to and while the tile's products are waited for
    double2 nxt[8];
    if (anal) {
      int c0, c1;
      half_cols(0, &c0, &c1);
      if (c0 < c1) load_acc16(a, (int64_t)blockIdx.x * kRowsCta + 32 * q + lane, c0, nxt);
    }
    for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      for (int h = 0; h < nsub; ++h, ++tt) {
        const uint32_t buf = tt & 1;
        if (!pwait(&pb->acc_full[buf], (tt >> 1) & 1, abort_flag)) { ok = false; break; }
        tc::tc_fence_after();
        int c0, c1;
        half_cols(h, &c0, &c1);
        const int64_t r = t * kRowsCta + 32 * q + lane;
        const uint32_t tq = tmem + ((uint32_t)(32 * q) << 16) + buf * kBufCols;
        if (anal) {
          for (int c = c0; c < c1; c += 16) {
            double2 old[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) old[i] = nxt[i];
            if (c + 16 < c1) {
              load_acc16(a, r, 256 * h + c + 16, nxt);
            } else {
              int hn = h + 1, n0 = 0, n1 = 0;
              if (hn < nsub) half_cols(hn, &n0, &n1);
              const bool same = n0 < n1;   // the next sub-tile of this tile has columns for this warp
              if (!same) half_cols(hn = 0, &n0, &n1);
              load_acc16(a, same ? r : r + (int64_t)gridDim.x * kRowsCta, 256 * hn + n0, nxt);
            }
            float v[16];
            tc::tmem_ld16(tq + (uint32_t)c, v);
            add_acc16(old, v);
            if (a.seg < chunks) {   // the tile's second segment
              tc::tmem_ld16(tq + kSegCols + (uint32_t)c, v);
              add_acc16(old, v);
            }
            store_acc16(a, r, 256 * h + c, old);
          }
        } else {
          epilogue_tile(a, r, tq, c0, c1, 256 * h);
        }
        tc::tc_fence_before();
        mbar_arrive(&pb->acc_empty[buf]);
      }
    }
    if (!ok) pabort(pb, a.err);
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// B operand of the tile: element (nrow, k) in chunk k / 16, TF32 hi / lo, K-major.
__global__ void build_b_kernel(ContractArgs a, TileGeom g, const cpx<float>* __restrict__ tw,
                               const int64_t* __restrict__ pj, const float* __restrict__ cw, float* __restrict__ B) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)a.N * a.K) return;
  const int nrow = (int)(e / a.K), k = (int)(e % a.K);
  float val = 0.f;
  {
    switch (a.mode) {
      case SYNTH_C: {
        const int tau = nrow >> 1, q = nrow & 1, j = k >> 1, part = k & 1;
        if (tau < a.n_tau && j < a.n_omega) {
          const cpx<float> w = tw[phase_index(g.sgn * pj[j], 2 * g.n0 + (int64_t)(a.tau0 + tau) * g.tau_stride, g.m4)];
          // Fr = sum (Tr Cr - Ti Ci), Fi = sum (Ti Cr + Tr Ci)
          val = q == 0 ? (part == 0 ? w.re : -w.im) : (part == 0 ? w.im : w.re);
        }
        break;
      }
      case SYNTH_R: {
        const int tau = nrow, j = k >> 1, part = k & 1;
        if (tau < a.n_tau && j < a.n_omega) {
          const cpx<float> w = tw[phase_index(g.sgn * pj[j], 2 * g.n0 + (int64_t)(a.tau0 + tau) * g.tau_stride, g.m4)];
          val = cw[j] * (part == 0 ? w.re : -w.im);
        }
        break;
      }
      case ANAL_C: {
        const int j = nrow >> 1, q = nrow & 1, s = k >> 1, part = k & 1;
        if (j < a.n_omega && s >= a.s0 && s < a.s1) {
          const cpx<float> w = tw[phase_index(g.sgn * pj[j], 2 * (g.n0 + s), g.m4)];
          // conj(w) y: re = Tr yr + Ti yi, im = Tr yi - Ti yr
          val = q == 0 ? (part == 0 ? w.re : w.im) : (part == 0 ? -w.im : w.re);
        }
        break;
      }
      default: {
        const int j = nrow >> 1, q = nrow & 1, s = k;
        if (j < a.n_omega && s >= a.s0 && s < a.s1) {
          const cpx<float> w = tw[phase_index(g.sgn * pj[j], 2 * (g.n0 + s), g.m4)];
          val = q == 0 ? w.re : -w.im;
        }
      }
    }
  }
  const float hi = tc::to_tf32(val);
  const int kc = k / kKc, kk = k % kKc;
  const int h0 = nrow < 256 ? 0 : 256, nn = min(256, a.N - h0);
  float* part = B + ((size_t)kc * a.N + h0) * 2 * kKc;
  const uint32_t o = tc::kmajor_offset(nrow - h0, kk, kKc) / 4;
  part[o] = hi;
  part[(uint32_t)nn * kKc + o] = val - hi;
}

int round16(int x) { return (x + 15) / 16 * 16; }

// The driver's tensor-map encoder (null when there is none), through the runtime: no link to the driver.
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled encode_tiled() {
  static const EncodeTiled fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
    return reinterpret_cast<EncodeTiled>(p);
  }();
  return fn;
}

// Tensor map of the long operand for the pipelined kernel: FP32 values, rows fastest, boxes of one K chunk
// by 128 rows.  False where the operand does not fit one: its base and its row stride in memory must be
// multiples of 16 bytes and a row of it shorter than 2^31 values.
bool pipe_enabled(rsv_operator op) {
  static const int env = [] {
    const char* e = getenv("RSV_CONTRACT_PIPE");
    return e != nullptr && e[0] == '0' ? 0 : 1;
  }();
  return env && op->sm_count > 0 && encode_tiled() != nullptr;
}
bool raw_map_of(const ContractArgs& a, const TileGeom& g, rsv_operator op, CUtensorMap* map) {
  if (!pipe_enabled(op)) return false;
  const bool real = a.mode == ANAL_R, anal = real || a.mode == ANAL_C;
  const cuuint64_t vals = (cuuint64_t)a.rows * (real ? 1 : 2);
  const cuuint64_t stride = (cuuint64_t)(anal ? a.rows : a.src_stride) * (real ? 4 : 8);
  if ((reinterpret_cast<uintptr_t>(a.src) & 15u) != 0 || stride % 16 != 0 || vals >= ((cuuint64_t)1 << 31) ||
      stride >= ((cuuint64_t)1 << 40))
    return false;
  const cuuint64_t dims[2] = {vals, (cuuint64_t)(anal ? g.steps : a.n_omega)};
  const cuuint32_t box[2] = {(cuuint32_t)(kRowsCta * (real ? 1 : 2)), (cuuint32_t)(real ? kKc : kKc / 2)};
  const cuuint32_t unit[2] = {1, 1};
  return encode_tiled()(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(a.src), dims, &stride, box, unit,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t run(ContractArgs& a, const TileGeom& g, rsv_operator op) {
  const size_t bbytes = (size_t)a.K * 2 * a.N * sizeof(float);
  if (ensure(op->ws_tcb, bbytes) != RSV_OK) return cudaErrorMemoryAllocation;
  a.B = (const float*)op->ws_tcb.ptr;
  a.err = op->d_flag;
  // Tensor memory sums in FP32 with truncation, a bias that grows with the length of the sum: 2.9e-6 of a
  // march's result with 254 values, 5.2e-6 with 512.  So an analysis of more than 256 values whose columns
  // leave room takes two accumulators per tile, added up in FP64.
  const int chunks = a.K / kKc;
  const bool anal = a.mode == ANAL_C || a.mode == ANAL_R;
  a.seg = anal && a.N <= 128 && chunks > 16 ? std::max(16, (chunks + 1) / 2) : chunks;
  const int64_t total = (int64_t)a.N * a.K;
  build_b_kernel<<<(unsigned)((total + 255) / 256), 256, 0, op->stream>>>(a, g, (const cpx<float>*)op->d_tw, op->d_pj,
                                                                          op->d_cw, (float*)op->ws_tcb.ptr);
  // the shared-memory opt-in is a per-device attribute: set it before every launch (cheap next
  // to a launch that moves gigabytes), so that any device and any thread gets it
  cudaError_t ae = cudaFuncSetAttribute(tc_contract_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  // the converted operand in tensor memory where the accumulators leave room for it
  const bool ta = a.N <= (int)kTaCols;
  auto* pipe = ta ? tc_contract_pipe_kernel<true> : tc_contract_pipe_kernel<false>;
  if (ae == cudaSuccess) ae = cudaFuncSetAttribute(pipe, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPipeSmem);
  if (ae != cudaSuccess) return ae;
  const int64_t tiles = (a.rows + kRowsCta - 1) / kRowsCta;
  CUtensorMap map;
  if (raw_map_of(a, g, op, &map)) {
    const unsigned blocks = (unsigned)std::min<int64_t>(tiles, (int64_t)op->sm_count);
    pipe<<<blocks, kPipeThreads, kPipeSmem, op->stream>>>(a, map);
  } else {
    tc_contract_kernel<<<(unsigned)tiles, 256, kSmem, op->stream>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace

bool tc_contract_supported(rsv_operator op, bool synth) {
  if (op->prec != RSV_PREC_FP32 || op->tc_contract_disabled) return false;
  return synth || round16(2 * op->n_omega) <= kMaxN;
}

bool tc_contract_segments(rsv_operator op) {
  return tc_contract_supported(op, false) && pipe_enabled(op) && round16(2 * op->n_omega) <= 128;
}

// Stage times are processed in calls of at most 512 output columns (256 complex).
cudaError_t tc_synth(rsv_operator op, const TileGeom& g, const void* fhat, void* F) {
  const int total = g.n_tau > 0 ? g.n_tau : 2 * g.steps + 1;
  const int per_call = op->real_state ? kMaxN : kMaxN / 2;
  cudaError_t e = cudaSuccess;
  for (int t0 = 0; t0 < total && e == cudaSuccess; t0 += per_call) {
    ContractArgs a = {};
    a.mode = op->real_state ? SYNTH_R : SYNTH_C;
    a.rows = g.rows;
    a.tau0 = t0;
    a.n_tau = std::min(per_call, total - t0);
    a.n_omega = g.n_omega;
    a.N = op->real_state ? round16(a.n_tau) : round16(2 * a.n_tau);
    a.K = round16(2 * g.n_omega);
    a.src = fhat;
    a.src_stride = g.coef_stride;
    a.out = F;
    e = run(a, g, op);
  }
  return e;
}

cudaError_t tc_analysis(rsv_operator op, const TileGeom& g, const void* Y, int s0, int s1, cpx<double>* acc,
                        int64_t acc_stride) {
  ContractArgs a = {};
  a.mode = op->real_state ? ANAL_R : ANAL_C;
  a.rows = g.rows;
  a.n_omega = g.n_omega;
  a.N = round16(2 * g.n_omega);
  a.K = op->real_state ? round16(g.steps) : round16(2 * g.steps);
  a.s0 = s0;
  a.s1 = s1;
  a.src = Y;
  a.out = acc;
  a.acc_stride = acc_stride;
  return run(a, g, op);
}

}  // namespace rsv
