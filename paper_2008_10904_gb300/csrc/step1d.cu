// Step form of FP64 1-D marches of few (instance, vector) pairs: jumps over several steps.
//
// For three-point operators the unforced step is a banded matrix T_1 (RK4: 9 diagonals;
// Crank-Nicolson: 2 (I - h/2 A)^-1 - I, whose entries decay exponentially from the diagonal), and so
// is p steps' T_p = T_1^p.  With the forcing transformed as in step2d.cu (Crank-Nicolson:
// c_j = (I - h/2 A)^-1 (h/2) (1 + z_j) fhat_j),
//     u_{n+p} = T_p u_n + sum_j c^(p)_j e^{i w_j t_n},   c^(p)_j = sum_{i<p} z_j^i T_1^{p-1-i} c_j.
// Such a march is a serial chain on few points, bound by FP64 issue (one warp instruction per 64
// cycles and scheduler whatever its lanes do, one per 19 cycles and SM) and by the exchange between
// CTAs.  A jump has about as many products as one step has (T_p has 8 p + 1 diagonals but for moderate
// steps far fewer entries above rounding), one exchange instead of one per step, and needs the forcing
// at one time per p steps.  The steps between two jumps are needed in the analysed window only; there
// they are marched from the jumps' states, all jumps side by side over the whole GPU (fill kernels).
//
// The band of T_p is bounded from the coefficients on the host (products of non-negative bounds of the
// diagonals): what lies outside sums to less than 2^-61 per row.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <mutex>
#include <vector>

#include "rsv_ops.h"

namespace rsv {

static bool jump_cluster16_ok();

namespace {

namespace cg = cooperative_groups;
using cd = cpx<double>;

constexpr int kGroups = 4;                       // term groups of a point (fixed: the order of the sums)
constexpr int kLanes = 2 * kGroups;              // lanes of a point: (re, im) x groups
constexpr int kMaxP = 16;                        // longest jump
constexpr int kMaxPoints = 1024;                 // points of an instance
constexpr int kMaxThreads = 1024;

struct Band {
  const cd* lo;
  const cd* di;
  const cd* up;
  const int64_t* inst_off;
  int64_t n;
  double h;
  int wl, wr, ld;             // T_p: diagonals -wl .. wr, at most ld columns per row
  // Crank-Nicolson factors ([levels][n] each, pivots [n])
  const cd* cr_lo;
  const cd* cr_up;
  const cd* cr_inv;
  int levels;
};

// First column and column count of row i of T_p on an instance of len points.
__device__ __forceinline__ int row_cols(int len, int wl, int wr) { return min(wl + wr + 1, len); }
__device__ __forceinline__ int row_first(int i, int len, int wl, int nt) { return max(0, min(i - wl, len - nt)); }

// ---------------------------------------------------------------------------
// One unforced step of the points of one CTA's instance.  RK4: x <- x + B (x + B/2 (x + B/3 (x + B/4 x)));
// Crank-Nicolson: x <- 2 (I - h/2 A)^-1 x - x by cyclic reduction.  One point per thread; s: [2][len + 2]
// shared values, buffer toggled per exchange.
// ---------------------------------------------------------------------------
struct Point {
  cd lo, di, up, inv;
  int64_t at;                 // index of the point in the operator's arrays
  int i, len;
  bool on;
};

__device__ __forceinline__ Point load_point(const Band& b, int64_t off, int len) {
  Point p;
  p.i = threadIdx.x;
  p.len = len;
  p.on = p.i < len;
  p.at = off + (p.on ? p.i : 0);
  const cd zero = mk<double>(0, 0);
  p.lo = p.on ? b.lo[p.at] : zero;
  p.di = p.on ? b.di[p.at] : zero;
  p.up = p.on ? b.up[p.at] : zero;
  p.inv = (p.on && b.levels > 0) ? b.cr_inv[p.at] : zero;
  return p;
}

template <bool REALC>
__device__ __forceinline__ void cmac(cd& a, cd w, cd x) {
  if (REALC) {
    a.re = fma(w.re, x.re, a.re);
    a.im = fma(w.re, x.im, a.im);
  } else {
    cfma(a, w, x);
  }
}

__device__ __forceinline__ cd neg(cd x) { return mk<double>(-x.re, -x.im); }

template <bool REALC>
__device__ __forceinline__ cd apply_a(const Point& p, cd x, cd* s, int& buf) {
  cd* b = s + buf * (p.len + 2);
  if (p.on) b[1 + p.i] = x;
  if (threadIdx.x == 0) b[0] = b[p.len + 1] = mk<double>(0, 0);
  __syncthreads();
  cd a = mk<double>(0, 0);
  if (p.on) {
    cmac<REALC>(a, p.lo, b[p.i]);
    cmac<REALC>(a, p.di, x);
    cmac<REALC>(a, p.up, b[p.i + 2]);
  }
  buf ^= 1;
  return a;
}

// (I - h/2 A)^-1 x
template <bool REALC>
__device__ __forceinline__ cd solve_cn(const Band& b, const Point& p, cd x, cd* s, int& buf) {
  for (int l = 0; l < b.levels; ++l) {
    const int sd = 1 << l;
    cd* q = s + buf * (p.len + 2);
    if (p.on) q[p.i] = x;
    __syncthreads();
    if (p.on) {
      const int64_t k = (int64_t)l * b.n + p.at;
      if (p.i - sd >= 0) cmac<REALC>(x, neg(b.cr_lo[k]), q[p.i - sd]);
      if (p.i + sd < p.len) cmac<REALC>(x, neg(b.cr_up[k]), q[p.i + sd]);
    }
    buf ^= 1;
  }
  cd o = mk<double>(0, 0);
  if (p.on) cmac<REALC>(o, p.inv, x);
  return o;
}

template <bool CN, bool REALC>
__device__ __forceinline__ cd one_step(const Band& b, const Point& p, cd x, cd* s, int& buf) {
  if (CN) {
    const cd y = solve_cn<REALC>(b, p, x, s, buf);
    return mk<double>(fma(2.0, y.re, -x.re), fma(2.0, y.im, -x.im));
  }
  cd w = x;
#pragma unroll
  for (int m = 4; m >= 1; --m) {
    const cd a = apply_a<REALC>(p, w, s, buf);
    const double f = b.h / (double)m;
    w = mk<double>(fma(f, a.re, x.re), fma(f, a.im, x.im));
  }
  return w;
}

// T_p column by column: the CTA of column j marches the unit vector e_j p steps and stores its entry
// (i, j) in the rows whose window holds column j.  T: [n][ld].
template <bool CN, bool REALC>
__global__ void __launch_bounds__(kMaxPoints) band_build_kernel(Band b, int p, int inst, cd* __restrict__ T) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cd* s = reinterpret_cast<cd*>(smem_raw);
  const int64_t off = b.inst_off[inst];
  const int len = (int)(b.inst_off[inst + 1] - off);
  const int j = blockIdx.x;
  if (j >= len) return;
  const Point pt = load_point(b, off, len);
  int buf = 0;
  cd x = mk<double>(pt.i == j ? 1.0 : 0.0, 0.0);
  for (int k = 0; k < p; ++k) x = one_step<CN, REALC>(b, pt, x, s, buf);
  if (!pt.on) return;
  const int nt = row_cols(len, b.wl, b.wr), f = row_first(pt.i, len, b.wl, nt);
  if (j >= f && j < f + nt) T[(off + pt.i) * b.ld + (j - f)] = x;
}

// Forcing coefficients c_j and, with p > 1, c^(p)_j of one (frequency, instance, vector) per CTA.
template <bool CN, bool REALC>
__global__ void __launch_bounds__(kMaxPoints) coef1d_kernel(Band b, int p, int n_inst, const cd* __restrict__ f,
                                                            int64_t f_stride, const cd* __restrict__ tw,
                                                            const int64_t* __restrict__ pj, int sgn, int64_t m4,
                                                            cd* __restrict__ c1, cd* __restrict__ cp, int64_t stride) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cd* s = reinterpret_cast<cd*>(smem_raw);
  const int inst = blockIdx.x % n_inst, v = blockIdx.x / n_inst, j = blockIdx.y;
  const int64_t off = b.inst_off[inst];
  const int len = (int)(b.inst_off[inst + 1] - off);
  const Point pt = load_point(b, off, len);
  const int64_t r = (int64_t)v * b.n + pt.at;
  const cd sj = tw[phase_index(sgn * pj[j], 1, m4)], zj = tw[phase_index(sgn * pj[j], 2, m4)];
  const cd fv = pt.on ? f[(int64_t)j * f_stride + r] : mk<double>(0, 0);
  const cd one = mk<double>(1, 0);
  int buf = 0;
  cd c;
  if (CN) {
    c = solve_cn<REALC>(b, pt, (0.5 * b.h) * ((one + zj) * fv), s, buf);
  } else {   // (h/6) [(1 + 4 s + z) f + B ((1 + 2 s) f + B ((1 + s)/2 f + 1/4 B f))]
    cd t = (0.5 * (one + sj)) * fv + (0.25 * b.h) * apply_a<REALC>(pt, fv, s, buf);
    t = (one + 2.0 * sj) * fv + b.h * apply_a<REALC>(pt, t, s, buf);
    c = (b.h / 6.0) * ((one + 4.0 * sj + zj) * fv + b.h * apply_a<REALC>(pt, t, s, buf));
  }
  if (pt.on) c1[(int64_t)j * stride + r] = c;
  if (p <= 1) return;
  cd x = c, z = c;
  for (int k = 1; k < p; ++k) {   // x <- T_1 x + z^k c
    z = zj * z;
    x = one_step<CN, REALC>(b, pt, x, s, buf) + z;
  }
  if (pt.on) cp[(int64_t)j * stride + r] = x;
}

// ---------------------------------------------------------------------------
// The serial chain: one cluster of CS CTAs per (instance, vector) pair.  A CTA owns a contiguous chunk
// of points and their rows of T_p in shared memory; eight lanes per point each sum a quarter of the
// row's products for the real or the imaginary part.  Every CTA keeps the whole state (double
// buffered): after a jump each CTA stores its points into the shared memory of all CTAs whose rows
// reach them, and one cluster barrier ends the jump.
// ---------------------------------------------------------------------------
struct Jump {
  Band b;
  int p, jumps;               // jumps of p steps (T_p), or single steps (T_1) with p = 1
  int64_t rows;
  const cd* T;
  const cd* G;                // [jumps][rows], nullable
  cd* u;                      // [rows]
  cd* Y;                      // state at the start of jump m to Y[m p] (nullable)
  int* flag;
  int cs;
};

template <bool REALC>
__global__ void __launch_bounds__(kMaxThreads, 1) gl1d_jump_kernel(Jump a) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int CS = a.cs;
  const int rank = CS > 1 ? (int)cluster.block_rank() : 0;
  const int inst = blockIdx.x / CS, v = blockIdx.y;
  const int64_t off = a.b.inst_off[inst];
  const int len = (int)(a.b.inst_off[inst + 1] - off);
  const int ch = (len + CS - 1) / CS;
  const int p0 = min(rank * ch, len), cnt = min(ch, len - p0);
  const int nt = row_cols(len, a.b.wl, a.b.wr);
  const int tg = (nt + kGroups - 1) / kGroups;               // terms per group
  double* su = reinterpret_cast<double*>(smem_raw);           // [2][len][2]
  // this CTA's rows of T: [cnt][kGroups * tg], zeros past nt
  double* sT = su + 4 * (size_t)len;
  for (int e = threadIdx.x; e < cnt * kGroups * tg; e += blockDim.x) {
    const int pt = e / (kGroups * tg), k = e % (kGroups * tg);
    const cd t = k < nt ? a.T[(off + p0 + pt) * a.b.ld + k] : mk<double>(0, 0);
    if (REALC) {
      sT[e] = t.re;
    } else {
      sT[2 * e] = t.re;
      sT[2 * e + 1] = t.im;
    }
  }
  const int64_t r0 = (int64_t)v * a.b.n + off;
  for (int e = threadIdx.x; e < 2 * len; e += blockDim.x) su[e] = reinterpret_cast<const double*>(a.u + r0)[e];
  const int pt = threadIdx.x / kLanes, comp = threadIdx.x & 1, grp = (threadIdx.x >> 1) & (kGroups - 1);
  const bool on = pt < cnt;
  const int i = p0 + (on ? pt : 0);
  const int first = row_first(i, len, a.b.wl, nt);
  const int k0 = grp * tg, k1 = min(k0 + tg, nt);            // this lane's terms
  const double* Tr = sT + ((size_t)(on ? pt : 0) * kGroups * tg + k0) * (REALC ? 1 : 2);
  const double sign = comp == 0 ? -1.0 : 1.0;
  // CTAs that read point i: the owners of the rows [i - wr, i + wl] (and their clamped windows)
  int lo_rank = 0, hi_rank = 0;
  if (CS > 1 && on) {
    const int ra = i - (nt == len ? len : a.b.wr), rb = i + (nt == len ? len : a.b.wl);
    // rows near the ends have clamped windows of nt columns: they reach up to nt - 1 points away
    const int a_lo = (i < nt) ? 0 : max(0, ra), b_hi = (i >= len - nt) ? len - 1 : min(len - 1, rb);
    lo_rank = a_lo / ch;
    hi_rank = b_hi / ch;
  }
  const int64_t gr = 2 * (r0 + i) + comp;
  const double* G = reinterpret_cast<const double*>(a.G);
  double* Y = reinterpret_cast<double*>(a.Y);
  const bool head = on && grp == 0;
  if (CS > 1) cluster.sync();
  else __syncthreads();
  int buf = 0;
  double g = (head && G && a.jumps > 0) ? G[gr] : 0.0, val = su[2 * i + comp];
  for (int m = 0; m < a.jumps; ++m) {
    const double ng = (head && G && m + 1 < a.jumps) ? G[(int64_t)(m + 1) * 2 * a.rows + gr] : 0.0;
    if (head && Y) Y[(int64_t)m * a.p * 2 * a.rows + gr] = val;
    const double* x = su + buf * 2 * len + 2 * first;
    double acc = g;
    if (on) {
      if (REALC) {
        for (int k = k0; k < k1; ++k) acc = fma(Tr[k - k0], x[2 * k + comp], acc);
      } else {
        double ai = 0.0;
        for (int k = k0; k < k1; ++k) {
          acc = fma(Tr[2 * (k - k0)], x[2 * k + comp], acc);
          ai = fma(Tr[2 * (k - k0) + 1], x[2 * k + 1 - comp], ai);
        }
        acc = fma(sign, ai, acc);
      }
    }
    // the four groups' sums: lanes r, r ^ 2, r ^ 4
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    val = acc;
    buf ^= 1;
    if (on) {
      double* dst = su + buf * 2 * len + 2 * i + comp;
      if (CS > 1) {
        for (int c = lo_rank + grp; c <= hi_rank; c += kGroups) *cluster.map_shared_rank(dst, c) = acc;
      } else if (grp == 0) {
        *dst = acc;
      }
    }
    if (CS > 1) cluster.sync();
    else __syncthreads();
    g = ng;
  }
  if (head) {
    reinterpret_cast<double*>(a.u)[gr] = val;
    if (!(val * val < 1e300)) atomicExch(a.flag, 1);   // NaN or overflow
  }
  if (CS > 1) cluster.sync();   // no CTA leaves while another may still store into its shared memory
}

// The steps between two jumps: the CTA of (jump m, pair) marches p - 1 steps from Y[m p].
template <bool CN, bool REALC>
__global__ void __launch_bounds__(kMaxPoints) fill_kernel(Band b, int p, int n_inst, int64_t rows, int y_first,
                                                          const cd* __restrict__ G, cd* __restrict__ Y) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cd* s = reinterpret_cast<cd*>(smem_raw);
  const int inst = blockIdx.y % n_inst, v = blockIdx.y / n_inst;
  const int s0 = blockIdx.x * p;
  if (s0 + p <= y_first) return;               // none of these steps is analysed
  const int64_t off = b.inst_off[inst];
  const int len = (int)(b.inst_off[inst + 1] - off);
  const Point pt = load_point(b, off, len);
  const int64_t r = (int64_t)v * b.n + pt.at;
  cd x = pt.on ? Y[(int64_t)s0 * rows + r] : mk<double>(0, 0);
  int buf = 0;
  for (int k = 0; k + 1 < p; ++k) {
    const cd g = (pt.on && G) ? G[(int64_t)(s0 + k) * rows + r] : mk<double>(0, 0);
    x = one_step<CN, REALC>(b, pt, x, s, buf) + g;
    if (pt.on) Y[(int64_t)(s0 + k + 1) * rows + r] = x;
  }
}

// ---------------------------------------------------------------------------
// Host: band bounds, jump length, launches
// ---------------------------------------------------------------------------
using Laurent = std::vector<double>;            // bounds of the diagonals -w .. w, centre at size / 2

// Bound of the product's diagonals up to wmax (a matrix of wmax + 1 points has no others).
Laurent conv(const Laurent& a, const Laurent& b, int wmax) {
  const int wa = (int)a.size() / 2, wb = (int)b.size() / 2, w = std::min(wa + wb, wmax);
  Laurent o(2 * (size_t)w + 1, 0.0);
  for (int i = -wa; i <= wa; ++i) {
    if (a[i + wa] == 0.0) continue;
    for (int j = std::max(-wb, -w - i); j <= std::min(wb, w - i); ++j) o[i + j + w] += a[i + wa] * b[j + wb];
  }
  return o;
}

// The bound of p steps without its outermost ends.  What is dropped of p steps' bound b reaches kMaxP steps'
// at most (kMaxP / p) |b|^(kMaxP / p - 1) times (|b|: the sum over the diagonals, 1 or more), which stays below 2^-70.
Laurent trimmed(const Laurent& b, int p) {
  double norm = 0;
  for (double x : b) norm += x;
  const double m = (double)kMaxP / p, tol = std::ldexp(1.0, -70) / (m * std::pow(norm, m - 1.0));
  const int w = (int)b.size() / 2;
  int c = w;
  double s = 0;
  while (c > 0 && s + b[w - c] + b[w + c] < tol) {
    s += b[w - c] + b[w + c];
    --c;
  }
  return Laurent(b.begin() + (w - c), b.begin() + (w + c + 1));
}

// Non-negative bounds of T_1's diagonals; empty when there is none (Crank-Nicolson matrix not
// dominated by its diagonal).
Laurent step_bound(rsv_operator op, bool adjoint) {
  double lo = 0, di = 0, up = 0, piv = 1e300;
  const int64_t n = op->n;
  const double hh = 0.5 * op->h;
  for (int64_t p = 0; p < n; ++p) {
    const double* t = op->tri_host.data();
    const int b = adjoint ? 3 : 0;
    auto mod = [&](int a) { return std::hypot(t[2 * ((size_t)(b + a) * n + p)], t[2 * ((size_t)(b + a) * n + p) + 1]); };
    lo = std::max(lo, mod(0));
    di = std::max(di, mod(1));
    up = std::max(up, mod(2));
    const double dr = t[2 * ((size_t)(b + 1) * n + p)], dimg = t[2 * ((size_t)(b + 1) * n + p) + 1];
    piv = std::min(piv, std::hypot(1.0 - hh * dr, hh * dimg));
  }
  if (op->scheme == RSV_SCHEME_CN) {
    // |(D - O)^-1| <= (piv - a S^-1 - c S)^-1: entries K r^d to the one side, K q^d to the other
    const double a = hh * lo, c = hh * up;
    if (!(piv > 1.0001 * (a + c))) return {};
    const double disc = std::sqrt(piv * piv - 4.0 * a * c);
    const double r = 2.0 * a / (piv + disc), q = 2.0 * c / (piv + disc), K = 1.0 / disc;
    const int w = op->gl_max_n - 1;
    Laurent o(2 * (size_t)w + 1);
    for (int d = 0; d <= w; ++d) {     // row i, column i - d: entries decay with the lower couplings
      o[w - d] = 2.0 * K * std::pow(r, d);
      o[w + d] = 2.0 * K * std::pow(q, d);
    }
    o[w] += 1.0;
    return trimmed(o, 1);
  }
  const Laurent B = {op->h * lo, op->h * di, op->h * up};
  Laurent t = {1.0};
  for (int m = 4; m >= 1; --m) {
    t = conv(B, t, 4);
    for (double& x : t) x /= m;
    t[t.size() / 2] += 1.0;
  }
  return t;
}

// Smallest (wl, wr) outside which the bounds sum to less than 2^-62 (2^-61 with what `trimmed` dropped, five times
// 2^-70 at most).
void band_of(const Laurent& b, int* wl, int* wr) {
  const int w = (int)b.size() / 2;
  const double tol = std::ldexp(1.0, -63);
  double s = 0;
  int l = w, r = w;
  while (l > 0 && s + b[w - l] < tol) s += b[w - l--];
  s = 0;
  while (r > 0 && s + b[w + r] < tol) s += b[w + r--];
  *wl = l;
  *wr = r;
}

int chunk_of(int max_n, int cs) { return (max_n + cs - 1) / cs; }

size_t jump_smem(int max_n, int cs, int nt, bool realc) {
  const int tg = (nt + kGroups - 1) / kGroups;
  return sizeof(double) * (4 * (size_t)max_n + (size_t)chunk_of(max_n, cs) * kGroups * tg * (realc ? 1 : 2));
}

Band band_geom(rsv_operator op, bool adjoint) {
  Band b;
  const int k = adjoint ? 3 : 0;
  b.lo = (const cd*)op->tri[k];
  b.di = (const cd*)op->tri[k + 1];
  b.up = (const cd*)op->tri[k + 2];
  b.inst_off = (const int64_t*)op->d_inst_off;
  b.n = op->n;
  b.h = op->h;
  b.cr_lo = b.cr_up = b.cr_inv = nullptr;
  b.levels = 0;
  if (op->scheme == RSV_SCHEME_CN) {
    const int L = op->pcr_levels;
    const cd* base = (const cd*)op->pcr + (size_t)(adjoint ? 1 : 0) * (2 * L + 1) * op->n;
    b.cr_lo = base;
    b.cr_up = base + (size_t)L * op->n;
    b.cr_inv = base + (size_t)2 * L * op->n;
    b.levels = L;
  }
  b.wl = b.wr = b.ld = 0;
  return b;
}

Band with_band(const rsv_operator op, Band b, int wl, int wr) {
  b.wl = wl;
  b.wr = wr;
  b.ld = std::min(wl + wr + 1, op->gl_max_n);
  return b;
}

int point_threads(rsv_operator op) { return (op->gl_max_n + 31) / 32 * 32; }
size_t point_smem(rsv_operator op) { return sizeof(cd) * 2 * (size_t)(op->gl_max_n + 2); }

// Calls fn with the (Crank-Nicolson, real coefficients) instance of a kernel template.
#define RSV_BY_SCHEME(op, KERNEL) \
  ((op)->scheme == RSV_SCHEME_CN ? ((op)->tri_real ? KERNEL<true, true> : KERNEL<true, false>) \
                                 : ((op)->tri_real ? KERNEL<false, true> : KERNEL<false, false>))

// Cluster size of a march of `pairs` pairs: the chunks of the longest instance are 16 points or more and
// all pairs' clusters fit the GPU at once; a size the device cannot hold falls back to 8.
int jump_cluster(rsv_operator op, int pairs) {
  const int n = op->gl_max_n;
  int cs = n >= 128 ? 16 : n >= 64 ? 4 : 1;
  if (cs == 16 && ((int64_t)pairs * 16 > op->sm_count || !jump_cluster16_ok())) cs = 8;
  return cs;
}

}  // namespace

// Clusters of 16 CTAs exceed the portable size: asked once per device whether the kernel may have them.
static bool jump_cluster16_ok() {
  static std::mutex mu;
  static int state[64] = {0};   // 0 not asked, 1 yes, 2 no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  std::lock_guard<std::mutex> lock(mu);
  if (state[dev] == 0) {
    bool ok = true;
    for (auto k : {gl1d_jump_kernel<true>, gl1d_jump_kernel<false>}) {
      ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
           cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) == cudaSuccess;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(16);
      cfg.blockDim = dim3(512);
      cfg.dynamicSmemBytes = 200 * 1024;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 16;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int clusters = 0;
      ok = ok && cudaOccupancyMaxActiveClusters(&clusters, k, &cfg) == cudaSuccess && clusters > 0;
    }
    if (!ok) cudaGetLastError();
    state[dev] = ok ? 1 : 2;
  }
  return state[dev] == 1;
}

// Plan of the jumps of one direction (kept until the frequencies change): jump length and bands.  The
// length is the one with the least estimated cycles per step: a jump's products (76 cycles per warp
// instruction with four warps, 19 per further warp) and its exchange.
const JumpPlan& jump_plan(rsv_operator op, bool adjoint) {
  JumpPlan& pl = op->jump[adjoint ? 1 : 0];
  if (pl.state != 0) return pl;
  pl.state = 2;
  const int max_n = op->gl_max_n;
  if (max_n > kMaxPoints) return pl;
  const Laurent one = step_bound(op, adjoint);
  if (one.empty()) return pl;
  Laurent t = one;
  const int cs = max_n >= 128 ? 16 : max_n >= 64 ? 4 : 1;
  const int warps = (chunk_of(max_n, cs) * kLanes + 31) / 32;
  double best = 1e300;
  for (int p = 1; p <= kMaxP; p *= 2) {
    int wl, wr;
    band_of(t, &wl, &wr);
    wl = std::min(wl, max_n - 1);
    wr = std::min(wr, max_n - 1);
    const int nt = std::min(wl + wr + 1, max_n);
    const int terms = (nt + kGroups - 1) / kGroups;
    const double cyc = (terms * (op->tri_real ? 1 : 2) + 3) * std::max(76.0, 19.0 * warps) + (cs > 1 ? 600.0 : 100.0);
    if (p == 1) {
      pl.wl1 = wl;
      pl.wr1 = wr;
    }
    if (jump_smem(max_n, std::min(cs, 8), nt, op->tri_real) <= 200 * 1024 && cyc / p < best) {
      best = cyc / p;
      pl.p = p;
      pl.wl = wl;
      pl.wr = wr;
    }
    if (p < kMaxP) t = trimmed(conv(t, t, max_n - 1), 2 * p);
  }
  if (best < 1e300 && jump_smem(max_n, std::min(cs, 8), std::min(pl.wl1 + pl.wr1 + 1, max_n), op->tri_real) <= 200 * 1024)
    pl.state = 1;
  return pl;
}

// Whether FP64 1-D marches of k vectors take the jumps: few pairs (as many as clusters of eight fit four
// times over), instances of up to 1024 points.
bool jump_taken(rsv_operator op, int k) {
  static const bool env = [] {
    const char* e = getenv("RSV_GL1D_CLUSTER");
    return !(e != nullptr && e[0] == '0');
  }();
  if (!env || !op->have_freq || op->kind != RSV_OP_GL1D || op->prec != RSV_PREC_FP64 || op->gl_max_n > kMaxPoints) return false;
  if ((int64_t)op->n_inst * k > op->sm_count || k > 65535) return false;
  return jump_plan(op, false).state == 1 && jump_plan(op, true).state == 1;
}

// Builds T_p and T_1 of the direction on the operator's stream (once per frequency grid).
static rsv_status jump_bands(rsv_operator op, bool adjoint) {
  jump_plan(op, adjoint);
  JumpPlan& pl = op->jump[adjoint ? 1 : 0];
  if (pl.built) return RSV_OK;
  const int ldp = std::min(pl.wl + pl.wr + 1, op->gl_max_n), ld1 = std::min(pl.wl1 + pl.wr1 + 1, op->gl_max_n);
  const size_t np = (size_t)op->n * ldp * sizeof(cd), n1 = (size_t)op->n * ld1 * sizeof(cd);
  rsv_status s = ensure(op->ws_band[adjoint ? 1 : 0], np + n1);
  if (s != RSV_OK) return s;
  pl.Tp = op->ws_band[adjoint ? 1 : 0].ptr;
  pl.T1 = static_cast<char*>(pl.Tp) + np;
  cudaError_t e = cudaMemsetAsync(pl.Tp, 0, np + n1, op->stream);
  const Band g = band_geom(op, adjoint);
  auto k = RSV_BY_SCHEME(op, band_build_kernel);
  for (int i = 0; i < op->n_inst && e == cudaSuccess; ++i) {
    const unsigned cols = (unsigned)op->inst_len[i];
    k<<<cols, point_threads(op), point_smem(op), op->stream>>>(with_band(op, g, pl.wl, pl.wr), pl.p, i, (cd*)pl.Tp);
    k<<<cols, point_threads(op), point_smem(op), op->stream>>>(with_band(op, g, pl.wl1, pl.wr1), 1, i, (cd*)pl.T1);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return cuda_fail(e, "step matrices");
  pl.built = true;
  return RSV_OK;
}

rsv_status jump_coefficients(rsv_operator op, const void* fhat, int64_t f_stride, int kg, bool adjoint, void* c1, void* cp) {
  rsv_status s = jump_bands(op, adjoint);
  if (s != RSV_OK) return s;
  const JumpPlan& pl = op->jump[adjoint ? 1 : 0];
  auto k = RSV_BY_SCHEME(op, coef1d_kernel);
  k<<<dim3((unsigned)(op->n_inst * kg), (unsigned)op->n_omega), point_threads(op), point_smem(op), op->stream>>>(
      band_geom(op, adjoint), pl.p, op->n_inst, (const cd*)fhat, f_stride, (const cd*)op->d_tw, op->d_pj, adjoint ? -1 : 1,
      4 * op->n_t, (cd*)c1, (cd*)cp, (int64_t)kg * op->n);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? RSV_OK : cuda_fail(e, "forcing transform");
}

static cudaError_t launch_jump(rsv_operator op, Jump a, int kg) {
  const int n = op->gl_max_n;
  a.cs = jump_cluster(op, op->n_inst * kg);
  op->gl_cluster = a.cs > 1 ? a.cs : 0;
  const int nt = std::min(a.b.wl + a.b.wr + 1, n);
  const size_t smem = jump_smem(n, a.cs, nt, op->tri_real);
  auto k = op->tri_real ? gl1d_jump_kernel<true> : gl1d_jump_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.cs * op->n_inst), (unsigned)kg);
  cfg.blockDim = dim3((unsigned)((chunk_of(n, a.cs) * kLanes + 31) / 32 * 32));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = op->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)a.cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, a);
}

// Steps [n0, n0 + steps) of the state, all forced or all unforced: synthesis of the jumps' and (analysed
// or left-over) single steps' forcing, the jumps, the left-over single steps, the fill.  Y (nullable):
// snapshots of the tile's steps, complete from y_first on.
cudaError_t jump_march(rsv_operator op, TileGeom g, bool adjoint, int kg, int steps, bool forced, int y_first,
                       const void* c1, const void* cp, void* state, void* G, void* Y) {
  const JumpPlan& pl = op->jump[adjoint ? 1 : 0];
  const int p = pl.p, jumps = steps / p, rest = steps - jumps * p;
  const size_t row = (size_t)g.rows * sizeof(cd);
  char* G1 = static_cast<char*>(G);                     // [steps][rows] (fill, rest) ...
  char* Gp = G1 + (size_t)(Y != nullptr ? steps : rest) * row;   // ... then [jumps][rows]
  cudaError_t e = cudaSuccess;
  const int64_t n0 = g.n0;
  if (forced && jumps > 0) {
    TileGeom q = g;
    q.n_tau = jumps;
    q.tau_stride = 2 * p;
    ProfScope ps(op, PROF_SYNTH);
    e = synth64(op, q, p > 1 ? cp : c1, Gp);
  }
  if (e == cudaSuccess && forced && (rest > 0 || (Y != nullptr && p > 1))) {
    TileGeom q = g;
    const int skip = Y != nullptr ? 0 : jumps * p;
    q.n0 = n0 + skip;
    q.n_tau = steps - skip;
    q.tau_stride = 2;
    ProfScope ps(op, PROF_SYNTH);
    e = synth64(op, q, c1, G1);
  }
  ProfScope ps(op, PROF_MARCH, (jumps > 0) + (rest > 0) + (Y != nullptr && p > 1 && jumps > 0));
  Jump a;
  a.rows = g.rows;
  a.u = (cd*)state;
  a.flag = op->d_flag;
  const Band b = band_geom(op, adjoint);
  if (e == cudaSuccess && jumps > 0) {
    a.b = with_band(op, b, pl.wl, pl.wr);
    a.T = (const cd*)pl.Tp;
    a.p = p;
    a.jumps = jumps;
    a.G = forced ? (const cd*)Gp : nullptr;
    a.Y = (cd*)Y;
    e = launch_jump(op, a, kg);
  }
  if (e == cudaSuccess && rest > 0) {
    a.b = with_band(op, b, pl.wl1, pl.wr1);
    a.T = (const cd*)pl.T1;
    a.p = 1;
    a.jumps = rest;
    a.G = forced ? (const cd*)(G1 + (Y != nullptr ? (size_t)jumps * p * row : 0)) : nullptr;
    a.Y = Y != nullptr ? (cd*)Y + (size_t)jumps * p * g.rows : nullptr;
    e = launch_jump(op, a, kg);
  }
  if (e == cudaSuccess && Y != nullptr && p > 1 && jumps > 0) {
    auto k = RSV_BY_SCHEME(op, fill_kernel);
    k<<<dim3((unsigned)jumps, (unsigned)(op->n_inst * kg)), point_threads(op), point_smem(op), op->stream>>>(
        b, p, op->n_inst, g.rows, y_first, forced ? (const cd*)G1 : nullptr, (cd*)Y);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace rsv
