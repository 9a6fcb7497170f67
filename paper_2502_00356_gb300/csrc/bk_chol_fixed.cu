// The Gaussian log-likelihood of bk_loglik.cu with its Cholesky factorisation in
// 64-bit fixed point: products of 64-bit integers on the integer pipe inside a
// panel of 64 columns, and the trailing update on the tensor cores, where every
// integer is split into digits that FP16 holds exactly and FP32 sums exactly.
// GB300's FP64 pipe does 2 FMAs per clock and SM: a 64 x 64 x 64 FP64 product
// takes an SM 66 us there, 2.8 us this way, and the FP64 factorisation of n =
// 8,000 ran at 0.9 of that pipe's rate (190 ms).
//
// Scaling.  With 2^{2 s_i} the power of four above a_ii, the matrix N_ij = a_ij
// 2^{60 - s_i - s_j} has |N_ij| < 2^60 whenever the matrix is positive definite
// (|a_ij| <= sqrt(a_ii a_jj)), and so have its Schur complements and the rows
// of its factor x_ij = L_ij 2^{60 - s_i}, |x| < 2^60, sum_j x_ij^2 = N_ii 2^60.
// The lower triangle is converted in place and factored as integers in units
// of 2^-60; every finished panel is written back as FP64.  Rounding is 2^-60 to
// 2^-57 of sqrt(a_ii a_jj) a step, against FP64's 2^-53 of the numbers at hand.
// An input outside those bounds, a pivot that is not positive, or a row of L
// longer than its diagonal allows means that the matrix is not positive definite.
// All three are tested, so that no integer wraps around unnoticed.  What stands
// below a pivot D is held at 2^62 sqrt(D 2^-60) before it is scaled (clamped), so
// that such an x shows, and the blocks of the forward substitution, which read all
// of L off the pivots' path, sum the squares of its rows (add_square).  A row of a
// positive definite matrix sums to less than 2^120; one of up to 2 2^120 has left
// the differences of 2^60 and such sums below 2^63.  (The same tests beside the pivots,
// in the panel's registers: n = 1,000 792 us, n = 8,000 11.0 ms; this way 678 us and
// 10.12 ms; without them 675 us and 10.01 ms.)
//
// Digits.  x = sum_s d_s 2^{54 - 9 s}, s = 0 .. 6, d_s in [-256, 255] (|d_0| <=
// 64): exact.  A product of two rows is sum_g 2^{48 - 9 g} S_g in units of 2^-60,
// S_g = sum_{s + t = g} sum_k d_s(i,k) d_t(j,k); S_0 .. S_7 are kept, 34 digit
// products as FP16 MMAs of K = 64 with FP32 accumulation (what is left out is
// below a tenth of a unit; without S_7 it was 13 units a step, which summed to
// FP64's own error at n = 8,000).  Sums of integers below 2^24 are exact in
// FP32: with the row norms above, |S_g| <= g 2^22 + 2^19, which passes 2^24 only
// for S_5 to S_7, where a lost unit weighs 2^-57.
//
// Launches.  Per panel of 64 columns: chol_panel_kernel (every block factors
// the diagonal tile for itself and solves its own rows below it) and
// chol_update_kernel (trailing tiles of 128 x 64, one persistent CTA per SM);
// the forward substitution rides along one panel behind, in a few extra blocks
// of the panel kernel.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "bk_internal.h"
#include "bk_math64.cuh"
#include "bk_tc.cuh"

namespace bk {
namespace {

constexpr int kNB = 64;          // panel width
constexpr int kFrac = 60;        // fraction bits
constexpr int kSlices = 7;
constexpr int kGroups = 8;       // digit-sum groups S_0 .. S_7
constexpr int kRowBlock = 128;   // rows of an MMA tile and of a slice block
// One row block's digits: [slice][row][64 halves], K-major with the 128-byte
// swizzle (a row is 128 bytes; its 16-byte chunk q sits at q xor (row mod 8)).
// Without a swizzle an MMA of 128 x 64 x 16 took 75 cycles of operand fetch.
constexpr int kSliceBytes = kRowBlock * kNB * 2;           // 16,384
constexpr int kBlockBytes = kSlices * kSliceBytes;         // 114,688
constexpr int kPanelThreads = 512;
constexpr int kEpiWarps = 16;
constexpr int kEpiCols = kNB / (kEpiWarps / 4);            // columns of an epilogue thread
constexpr int kUpdThreads = (kEpiWarps + 2) * 32;          // epilogue, MMA, copies
constexpr long long kWaitCycles = 2000000000LL;            // bound of every barrier wait, about 1 s

constexpr int kNotPd = 1, kGaveUp = 2;   // not positive definite; a wait that gave up

// The workspace.
struct CholWork {
  int* flag;       // kNotPd, kGaveUp
  int* scale;      // s_i
  double* diag;    // two 64 x 64 factors, column-major: panel k's at k mod 2
  double* part;    // per panel: sum log L_ii, sum y_i^2
  float* squares;  // per row: the squares of its part of the panels taken off z so far
  unsigned char* slices;
};
size_t round256(size_t v) { return (v + 255) / 256 * 256; }
struct CholLayout {
  size_t scale, diag, part, squares, slices, total;
};
CholLayout chol_layout(int64_t n) {
  CholLayout l;
  l.scale = 256;
  l.diag = l.scale + round256((size_t)n * sizeof(int));
  l.part = l.diag + 2 * kNB * kNB * sizeof(double);
  l.squares = l.part + round256((size_t)((n + kNB - 1) / kNB) * 2 * sizeof(double));
  l.slices = l.squares + round256((size_t)n * sizeof(float));
  l.total = l.slices + (size_t)((n + kRowBlock - 1) / kRowBlock) * kBlockBytes;
  return l;
}

// Each kernel of the chain is launched while the one before it still runs, waits
// here for that one's end (and so for all before it), and then lets the next one
// come: the launches' latency, about 2 us each, is hidden.
__device__ __forceinline__ void chain() {
  asm volatile("griddepcontrol.wait;\n griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ double qnan() { return __longlong_as_double(0x7ff8000000000000LL); }

// a 2^{60 - s_i - s_j} as an integer (rounded); false when it is not below 2^60.
__device__ __forceinline__ bool to_fixed(double a, int s2, long long& v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(a);
  int e = (int)((b >> 52) & 0x7ff);
  unsigned long long sig = (b & 0xfffffffffffffULL) | 0x10000000000000ULL;
  if (e == 0) {  // subnormal
    sig ^= 0x10000000000000ULL;
    const int lz = __clzll((long long)sig) - 11;
    sig <<= lz;  // (0 stays 0)
    e = sig ? 1 - lz : 1;
  }
  const int sh = e - 1075 + kFrac - s2;
  if (e == 0x7ff || (sh >= kFrac - 52 && sig)) return false;  // |a| >= 2^{s_i + s_j}, infinite, NaN
  unsigned long long m = 0;
  if (sh >= 0) m = sig << (sh & 63);
  else if (sh >= -54) m = (sig + (1ULL << (-sh - 1))) >> -sh;
  v = (long long)b < 0 ? -(long long)m : (long long)m;
  return true;
}

// x 2^{s - 60} as a double, rounded to nearest, without the FP64 pipe.
__device__ __forceinline__ double from_fixed(long long x, int s) {
  if (x == 0) return 0.0;
  const unsigned long long m = (unsigned long long)(x < 0 ? -x : x);
  const int lz = __clzll((long long)m);           // the leading bit to bit 63
  const unsigned long long q = (m << lz >> 11) + (m << lz >> 10 & 1);  // [2^52, 2^53]
  const int e = 63 - lz - kFrac + s + 1023;       // the exponent field
  if (e <= 0 || e >= 2046) return scalbn((double)x, s - kFrac);
  const long long r = (long long)(q + ((unsigned long long)(e - 1) << 52));
  return __longlong_as_double(x < 0 ? (r | (long long)0x8000000000000000ULL) : r);
}

// A fixed-point number as two signed words, x = h 2^32 + l, so that products
// accumulate by signed 32 x 32 + 64-bit multiply-adds.
struct Limbs {
  int l, h;
};
__device__ __forceinline__ Limbs limbs(long long x) {
  const int l = (int)x;
  return Limbs{l, (int)(x >> 32) + (l < 0 ? 1 : 0)};
}
__device__ __forceinline__ long long value(Limbs a) { return ((long long)a.h << 32) + a.l; }
// Accumulates x y / 2^60 in two parts (high products, crossed products), rounded
// to nearest at the end.  The products of the low words (below 4 units, of
// either sign) are left out, except where x and y may be the same number
// (add_low): there they are positive, and a pivot's logarithm would show it.
struct Acc {
  long long hh = 0, hl = 0;
  __device__ __forceinline__ void add(Limbs x, Limbs y) {
    hh = mad_wide(x.h, y.h, hh);
    hl = mad_wide(x.h, y.l, hl);
    hl = mad_wide(x.l, y.h, hl);
  }
  __device__ __forceinline__ void add_low(Limbs x, Limbs y) { hl += __mulhi(x.l, y.l); }
  __device__ __forceinline__ long long sum() const { return (hh << 4) + ((hl + (1LL << 27)) >> 28); }
};

__device__ __forceinline__ long long shfl64(long long v, int src) {
  const int lo = __shfl_sync(0xffffffffu, (int)v, src), hi = __shfl_sync(0xffffffffu, (int)(v >> 32), src);
  return ((long long)hi << 32) | (unsigned)lo;
}

// For a pivot D in (0, 2^60): t and rho (60 fraction bits, in [1, 2)) with
// 1/sqrt(D 2^-60) = 2^t rho 2^-60.  The FP32 root gives 2^t y, y of 24 bits within
// 2^-22; with delta = D 2^{2t - 60}, e = 1 - delta y^2 is read exactly to 2^-62 from
// the middle 64 bits of the product (it is small, the high bits are known), and
// rho = y (1 + e/2 + 3 e^2/8) leaves 2^-61.
__device__ __forceinline__ long long rsqrt_fixed(long long D, int& t) {
  // D as a float: its upper 32 bits hold 24 of them unless the pivot is small (a
  // 64-bit conversion takes 94 cycles, this one 20)
  const float f = D >= (1LL << 52) ? __uint2float_rn((unsigned)(D >> 28)) * 0x1p28f : __ll2float_rn(D);
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const unsigned yb = max(__float_as_uint(y), 0x30800000u);         // at least 2^-30
  t = (int)(yb >> 23) - 97;
  const unsigned Y = (yb & 0x7fffffu) | 0x800000u;                  // y 2^23
  const unsigned long long y2 = (unsigned long long)Y * Y;          // y^2 2^46
  const unsigned long long dn = (unsigned long long)D << (2 * t);   // delta 2^60
  const unsigned d0 = (unsigned)dn, d1 = (unsigned)(dn >> 32), p0 = (unsigned)y2, p1 = (unsigned)(y2 >> 32);
  unsigned long long T = __umulhi(d0, p0);                          // (dn y2 >> 32) mod 2^64
  T = (unsigned long long)d0 * p1 + T;
  T = (unsigned long long)d1 * p0 + T;
  T += (unsigned long long)(d1 * p1) << 32;
  const long long e = -((long long)T >> 12);                        // e 2^62
  const int es = (int)(e >> 10);
  const long long h = (e >> 1) + 3 * (((long long)es * es) >> 45);  // (e/2 + 3 e^2/8) 2^62
  const long long p = mad_wide((int)(h >> 16), (int)Y, ((h & 0xffff) * (long long)Y) >> 16);
  return ((long long)Y << 37) + (p >> 9);
}

// v, held between about -2^{62 - t} and 2^{62 - t}; t <= 30.
__device__ __forceinline__ long long clamped(long long v, int t) {
  const int top = 0x40000000 >> t;
  const int h = min(max((int)(v >> 32), -top), top);
  return ((long long)h << 32) | (unsigned)v;
}
// (v 2^t) rho / 2^60 for a clamped v.
__device__ __forceinline__ long long mul_rho(long long v, int t, Limbs rho) {
  Acc a;
  a.add(limbs(v << t), rho);
  return a.sum();
}

// sum + (L 2^-s)^2 in FP32 without the FP64 pipe, nothing for L below 2^{s - 60}.
constexpr float kMaxSquares = 2.0f;
__device__ __forceinline__ float add_square(float sum, double L, int s) {
  const unsigned hi = (unsigned)__double2hiint(L) & 0x7fffffffu;
  const int e = (int)(hi >> 20) - s;  // (infinite and NaN entries: the flag is set already)
  const float x = __uint_as_float(((unsigned)(e - 1023 + 127) << 23) | ((hi & 0xfffffu) << 3));
  return e > 1023 - 60 ? fmaf(x, x, sum) : sum;
}

// Scales, y = z, the flag, the sums of squares.
__global__ void __launch_bounds__(256) chol_prep_kernel(const double* __restrict__ a, int64_t ld,
                                                        int64_t n, const double* __restrict__ z,
                                                        double* __restrict__ y, CholWork w) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double d = a[i + i * ld];
  const long long bits = __double_as_longlong(d);
  const int e = bits >> 52 ? (int)(bits >> 52) - 1023 : -1011 - __clzll(bits);  // (subnormal)
  if (bits <= 0 || e == 1024) {
    atomicOr(w.flag, kNotPd);
    w.scale[i] = 0;
  } else {
    w.scale[i] = (e >> 1) + 1;
  }
  w.squares[i] = 0.0f;
  y[i] = z[i];
}

// Panel q's share of the forward substitution and of the sums, by one block:
// y_q <- L_qq^{-1} (y_q - L_{q,q-1} y_{q-1}), sum log L_ii, sum y_i^2, and L_qq
// into the matrix.  Earlier panels' parts of y_q were taken off before, and their
// squares are summed.
__device__ __forceinline__ void finish_panel(double* __restrict__ a, int64_t ld, int64_t n, int64_t q,
                                             double* __restrict__ y, const CholWork& w, double* sh) {
  const int64_t o = q * kNB;
  const int b = (int)(n - o < kNB ? n - o : kNB);
  const int tid = threadIdx.x, lane = tid & 31;
  double* const L = sh;                       // 64 x 65
  double* const part = sh + kNB * (kNB + 1);  // 8 x 64
  float* const squares = reinterpret_cast<float*>(part + 8 * kNB);  // 8 x 64
  for (int e = tid; e < kNB * kNB; e += kPanelThreads) {
    const int r = e & 63, c = e >> 6;
    const double v = w.diag[(q & 1) * (kNB * kNB) + e];
    L[c * (kNB + 1) + r] = v;
    if (r < b && c <= r) a[(o + r) + (o + c) * ld] = v;
  }
  {
    const int r = tid & 63, h = tid >> 6;
    double s = 0.0;
    float sum = 0.0f;
    if (q > 0 && r < b) {
      const int scale = w.scale[o + r];
#pragma unroll
      for (int c = 8 * h; c < 8 * h + 8; ++c) {
        const double v = a[(o + r) + (o - kNB + c) * ld];
        s = fma(v, y[o - kNB + c], s);
        sum = add_square(sum, v, scale);
      }
    }
    part[h * kNB + r] = s;
    squares[h * kNB + r] = sum;
  }
  __syncthreads();
  if (tid < 32) {  // rows lane and lane + 32
    double v0 = lane < b ? y[o + lane] : 0.0, v1 = lane + 32 < b ? y[o + lane + 32] : 0.0;
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      s0 += part[h * kNB + lane];
      s1 += part[h * kNB + lane + 32];
    }
    v0 -= s0;
    v1 -= s1;
    const double d0 = L[lane * (kNB + 2)], d1 = L[(lane + 32) * (kNB + 2)];
    const double i0 = 1.0 / d0, i1 = 1.0 / d1;
#pragma unroll 4
    for (int c = 0; c < 32; ++c) {
      const double yc = __shfl_sync(0xffffffffu, v0 * i0, c);
      if (lane == c) v0 = yc;
      if (lane > c) v0 = fma(-L[c * (kNB + 1) + lane], yc, v0);
      v1 = fma(-L[c * (kNB + 1) + lane + 32], yc, v1);
    }
#pragma unroll 4
    for (int c = 0; c < 32; ++c) {
      const double yc = __shfl_sync(0xffffffffu, v1 * i1, c);
      if (lane == c) v1 = yc;
      if (lane > c) v1 = fma(-L[(c + 32) * (kNB + 1) + lane + 32], yc, v1);
    }
    if (lane < b) y[o + lane] = v0;
    if (lane + 32 < b) y[o + lane + 32] = v1;
    double sq = (lane < b ? v0 * v0 : 0.0) + (lane + 32 < b ? v1 * v1 : 0.0);
    double ld_ = (lane < b ? log(d0) : 0.0) + (lane + 32 < b ? log(d1) : 0.0);
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      sq += __shfl_xor_sync(0xffffffffu, sq, s);
      ld_ += __shfl_xor_sync(0xffffffffu, ld_, s);
    }
    if (lane == 0) {
      w.part[2 * q] = ld_;
      w.part[2 * q + 1] = sq;
    }
  } else if (tid >= kPanelThreads / 2) {
    const int r = (tid - kPanelThreads / 2) >> 2, g = tid & 3;
    if (r < b) {
      const int scale = w.scale[o + r];
      float sum = squares[2 * g * kNB + r] + squares[(2 * g + 1) * kNB + r];
      if (g == 0) sum += w.squares[o + r];
      for (int c = g; c < r; c += 4) sum = add_square(sum, L[c * (kNB + 1) + r], scale);
      const unsigned quad = 15u << (tid & 28);
      sum += __shfl_xor_sync(quad, sum, 1);
      sum += __shfl_xor_sync(quad, sum, 2);
      if (sum > kMaxSquares) atomicOr(w.flag, kNotPd);
    }
  }
}

// ---------------------------------------------------------------------------
// A panel.  Block b < row_blocks factors the diagonal tile (rows 0 .. 63 of its
// shared array) and solves rows_per_block rows below it (rows 64 .., none for the
// last block, which writes the tile instead) against it, in
// column groups of 8.  The pivots are one serial chain (about 400 cycles a
// column: root, scaling, update of the next pivot), so everything else is
// arranged around it.  Four (kSolve) solving warps, one on each of the SM's
// schedulers, all factor the group's 8 x 8 block in their lanes 0 .. 7, and the other
// 24 lanes of each carry one row further down through the same instructions: the
// rows are solved at no extra time, without a barrier.  The group's update (rank
// 8) of the next group's columns happens in the solving warps' registers; the
// other warps apply it to the columns after those while the solving warps are at
// the next group: one barrier a group.  The factored 8 x 8 blocks have a place of
// their own: all solving warps read a group's block between the same two barriers
// as one of them has its factor, so nothing is written where they read.  Four warps carry 96 rows, the tile's 56 and
// 32 below it; where more are needed to fill one wave of the SMs a fifth warp
// takes 64 below it, which shares a scheduler and slows the chain.  A product
// costs three wide multiply-adds of 8 cycles a warp and scheduler (an FP64 FMA 64),
// which bounds the first groups: the rest of their update goes out evenly, by
// pairs of a row group and a column.  Of the blocks beyond row_blocks the first
// finishes panel k - 1 (finish_panel) and the others take panel k - 2's part off
// the forward substitution of the rows from here on, 256 rows each.
constexpr int kFollow = 24;
constexpr int solve_rows(int solve) { return solve == 4 ? 32 : 64; }  // rows below the tile
struct PanelSmem {
  long long S[2 * kNB][kNB + 1];   // two's complement before, limbs after a column is done
  long long D[kNB][8];             // the diagonal 8 x 8 blocks' factors (limbs), row by row
  int scale[2 * kNB];
  int bad;
};

__device__ __forceinline__ Limbs as_limbs(long long raw) {
  return Limbs{(int)raw, (int)(raw >> 32)};
}
__device__ __forceinline__ long long raw_limbs(Limbs x) {
  return ((long long)x.h << 32) | (unsigned)x.l;
}

// What the row's own square keeps of the low words (Acc::add_low over a group).
__device__ __forceinline__ long long low_square(const Limbs (&x)[8]) {
  long long low = 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) low += __mulhi(x[c].l, x[c].l);
  return low;
}

template <bool kFirst, int kSolve>
__global__ void __launch_bounds__(kPanelThreads, 1) chol_panel_kernel(
    double* __restrict__ a, int64_t ld, int64_t n, int64_t k, int row_blocks, int rows_per_block,
    double* __restrict__ y, CholWork w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PanelSmem& sm = *reinterpret_cast<PanelSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t o = k * kNB;
  chain();
  if ((int)blockIdx.x == row_blocks) {
    finish_panel(a, ld, n, k - 1, y, w, reinterpret_cast<double*>(smem_raw));
    return;
  }
  if ((int)blockIdx.x > row_blocks) {  // y_r -= L_{r,k-2} y_{k-2} for the rows from o on
    double* const ys = reinterpret_cast<double*>(smem_raw);
    const int64_t po = o - 2 * kNB;
    if (tid < kNB) ys[tid] = y[po + tid];
    __syncthreads();
    const int64_t r = o + (int64_t)((int)blockIdx.x - row_blocks - 1) * 256 + (tid & 255);
    const int h = tid >> 8;
    float* const squares = reinterpret_cast<float*>(ys + kNB + 256);
    double s = 0.0;
    float sum = 0.0f;
    if (r < n) {
      const int scale = w.scale[r];
#pragma unroll 8
      for (int c = 32 * h; c < 32 * h + 32; ++c) {
        const double v = a[r + (po + c) * ld];
        s = fma(v, ys[c], s);
        sum = add_square(sum, v, scale);
      }
    }
    if (h == 1) {
      ys[kNB + (tid & 255)] = s;
      squares[tid & 255] = sum;
    }
    __syncthreads();
    if (h == 0 && r < n) {
      y[r] -= s + ys[kNB + tid];
      w.squares[r] += sum + squares[tid];
    }
    return;
  }
  const int b = (int)(n - o < kNB ? n - o : kNB);
  const int64_t r0 = o + kNB + (int64_t)blockIdx.x * rows_per_block;
  int own = 0;
  if (r0 < n) own = (int)(n - r0 < rows_per_block ? n - r0 : rows_per_block);
  {
    // All 16 loads of a thread go out before the first is waited for: four at a
    // time, behind the scales, they took 3 us (now 1.8).
    const int row = tid & 127, q = tid >> 7;
    const bool diag = row < kNB;
    const int64_t r = diag ? o + row : r0 + row - kNB;
    const bool in = diag ? row < b : row - kNB < own;
    constexpr int kEach = kNB / (kPanelThreads / 128);
    double x[kEach];
#pragma unroll
    for (int i = 0; i < kEach; ++i) {
      const int c = q + i * (kPanelThreads / 128);
      x[i] = in && c < b && (!diag || c <= row) ? a[r + (o + c) * ld] : 0.0;
    }
    if (tid == 0) sm.bad = *w.flag != 0;
    if (tid < 2 * kNB) sm.scale[tid] = in ? w.scale[r] : 0;
    if constexpr (kFirst) __syncthreads();
    bool ok = true;
#pragma unroll
    for (int i = 0; i < kEach; ++i) {
      const int c = q + i * (kPanelThreads / 128);
      long long v;
      if constexpr (kFirst) {
        v = 0;
        if (in && c < b && (!diag || c <= row))
          ok = to_fixed(x[i], sm.scale[row] + sm.scale[c], v) && ok;
      } else {
        v = __double_as_longlong(x[i]);
      }
      if (diag && c == row && row >= b) v = 1LL << 58;  // identity beyond the matrix
      sm.S[row][c] = v;
    }
    if (kFirst && !ok) {
      sm.bad = 1;
      atomicOr(w.flag, kNotPd);
    }
  }
  __syncthreads();
  const int groups = own > 32 ? 4 : own > 0 ? 3 : 2;  // row groups of 32
  const int follow = 8 + kFollow * warp + lane - 8;   // a solving lane's row (lanes 8 .. 31)
  for (int c0 = 0; c0 < kNB; c0 += 8) {
    // solving warps whose rows are all done (the tile's first ones) join the others
    const int retired = min(c0 / kFollow, kSolve - 1);
    if (warp < kSolve && warp >= retired) {
      const int row = lane < 8 ? c0 + lane : follow;
      long long v[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = sm.S[row][c0 + c];
      if (c0 > 0) {  // the previous group's update of these columns
        const int p0 = c0 - 8;
        Limbs x[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) x[c] = as_limbs(sm.S[row][p0 + c]);
        const long long low = low_square(x);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          Acc acc;
          acc.hl = j == lane ? low : 0;
#pragma unroll
          for (int c = 0; c < 8; ++c) acc.add(x[c], as_limbs(sm.S[c0 + j][p0 + c]));
          v[j] -= acc.sum();
        }
      }
      bool bad = false;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        long long D = shfl64(v[c], c);
        if (D <= 0 || D >= (1LL << 60)) {
          bad = true;
          D = 1LL << 58;
        }
        int t;
        const Limbs rho = limbs(rsqrt_fixed(D, t));
        const Limbs x = limbs(mul_rho(clamped(v[c], t), t, rho));
        v[c] = raw_limbs(x);
#pragma unroll
        for (int j = c + 1; j < 8; ++j) {
          const Limbs xj{__shfl_sync(0xffffffffu, x.l, j), __shfl_sync(0xffffffffu, x.h, j)};
          Acc p;
          p.add(x, xj);
          p.add_low(x, xj);
          v[j] -= p.sum();
        }
      }
      if (lane >= 8 ? follow >= c0 + 8 : warp == kSolve - 1) {
        long long* const dst = lane >= 8 ? &sm.S[row][c0] : sm.D[row];
#pragma unroll
        for (int c = 0; c < 8; ++c) dst[c] = v[c];
      }
      if (bad && lane == 0) sm.bad = 1;
    } else if (c0 > 0) {
      // the rest of the previous group's update: columns from c0 + 8 on
      const int rest = kPanelThreads / 32 - kSolve + retired, u = warp < kSolve ? warp : warp - kSolve + retired;
      const int p0 = c0 - 8, j0 = c0 + 8;
      // items: row group 0 with columns j0 .. 31, then groups 1, 2, 3 with j0 .. 63
      const int first = max(32 - j0, 0), each = kNB - j0, items = first + (groups - 1) * each;
      int have = -1;
      Limbs x[8];
      long long low = 0;
      const int i0 = items * u / rest, i1 = items * (u + 1) / rest;
      for (int i = i0; i < i1; ++i) {
        const int rg = i < first ? 0 : 1 + (i - first) / each;
        const int j = j0 + (i < first ? i : (i - first) % each), row = 32 * rg + lane;
        if (rg != have) {
          have = rg;
#pragma unroll
          for (int c = 0; c < 8; ++c) x[c] = as_limbs(sm.S[row][p0 + c]);
          low = low_square(x);
        }
        Acc acc;
        acc.hl = row == j ? low : 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) acc.add(x[c], as_limbs(sm.S[j][p0 + c]));
        sm.S[row][j] -= acc.sum();
      }
    }
    __syncthreads();
  }
  const bool bad = sm.bad != 0;
  if ((int)blockIdx.x == row_blocks - 1) {
    if (bad && tid == 0) atomicOr(w.flag, kNotPd);
    for (int e = tid; e < kNB * kNB; e += kPanelThreads) {
      const int r = e & 63, c = e >> 6;
      double v = r == c ? 1.0 : 0.0;
      if (r < b && c <= r) {
        const long long x = c >= (r & ~7) ? sm.D[r][c & 7] : sm.S[r][c];
        v = bad ? qnan() : from_fixed(value(as_limbs(x)), sm.scale[r]);
      }
      w.diag[(k & 1) * (kNB * kNB) + e] = v;
    }
  }
  if (own == 0) return;
  {
    const int row = tid & 63, q = tid >> 6;  // one row (of own), one chunk of 8 columns
    if (row < own) {
      const int64_t r = r0 + row;
      long long x[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        x[c] = value(as_limbs(sm.S[kNB + row][8 * q + c]));
        a[r + (o + 8 * q + c) * ld] = bad ? qnan() : from_fixed(x[c], sm.scale[kNB + row]);
        // digits are read from x + sum_s 256 2^{54 - 9 s}, so that each is a bit field
        x[c] += 0x4020100804020100LL;
      }
      unsigned char* const dst =
          w.slices + (r / kRowBlock) * kBlockBytes + (r % kRowBlock) * 128 + ((q ^ (int)(r & 7)) << 4);
#pragma unroll
      for (int s = 0; s < kSlices; ++s) {
        unsigned u[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const unsigned d0 = (unsigned)(x[2 * p] >> (54 - 9 * s)) & 511u;
          const unsigned d1 = (unsigned)(x[2 * p + 1] >> (54 - 9 * s)) & 511u;
          // the halves 1024 + field, less 1024 + 256
          const unsigned packed = 0x64006400u | d0 | (d1 << 16);
          const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&packed),
                                    __halves2half2(__ushort_as_half(0x6500), __ushort_as_half(0x6500)));
          u[p] = *reinterpret_cast<const unsigned*>(&h);
        }
        *reinterpret_cast<uint4*>(dst + s * kSliceBytes) = make_uint4(u[0], u[1], u[2], u[3]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The trailing update N_ij -= x_i x_j^T over the panel's 64 columns, in tiles of
// 128 rows x 64 columns: the rows' seven slices (112 KB) stay in shared memory
// along a row of tiles, the columns' (56 KB) are double-buffered, both by bulk
// copies from one warp.  The 34 digit products (K = 64) go into eight accumulators of
// 64 TMEM columns, S_0 .. S_7 side by side, so that slice s of the rows times slices
// t .. t + c - 1 of the columns is one MMA of N = 64 c into S_{s+t} and the next: 48 of
// them, 4,352 cycles.  As 136 MMAs of N = 64 they took 60 to 68 cycles each, rows in
// shared memory or in TMEM, against 32 of arithmetic.  S_g is complete after slice
// g, and sixteen warps drain it into 64-bit integers while the products go on, the
// next tile's too.  The drain (about 700 cycles a sum) and the entries' loads and
// stores bound it: a tile among many takes 4.1 us (5.9 with 136 MMAs, a conversion
// of every sum and eight warps), at n = 8,000 two thirds of HBM's rate for the entries;
// the next tile's are prefetched into L2 (n = 8,000 without: 10.48 ms, with: 10.14).
struct UpdBarriers {
  uint64_t full_a[kSlices], full_b[2], free_b[2], done[kGroups], drained[kGroups], last;
  uint32_t tmem;
};
constexpr int kBBytes = kBlockBytes / 2;
constexpr size_t kUpdSmem = (size_t)kBlockBytes + 2 * kBBytes + sizeof(UpdBarriers);

__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          tc::smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(tc::smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
// Waits for the phase of *bar with this parity; false after kWaitCycles.
__device__ __forceinline__ bool wait_phase(uint64_t* bar, uint32_t parity) {
  const long long start = clock64();
  while (!tc::mbar_wait(bar, parity, 64))
    if (clock64() - start > kWaitCycles) return false;
  return true;
}
__device__ __forceinline__ void arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc ? 1u : 0u)
      : "memory");
}

// Descriptor of a K-major operand with the 128-byte swizzle: rows of 128 bytes,
// groups of 8 rows 1,024 bytes apart (bits 32-45), swizzle mode 2 in bits 61-63;
// otherwise as desc_kmajor.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)64 << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// v[j] = TMEM[lane][column + j], j = 0 .. 15 (complete after ld_wait).
__device__ __forceinline__ void ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// Waits for the loads; the registers pass through, so that no use moves ahead.
__device__ __forceinline__ void ld_wait(uint32_t (&a)[kEpiCols]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < kEpiCols; ++j) asm volatile("" : "+r"(a[j]));
}

// *p when c < cols, else 0, and the store of it: volatile, so that a column of
// accesses keeps one running pointer instead of one each per column (the
// registers spilled, and with 224 KB of shared memory in use spills miss L1).
__device__ __forceinline__ long long load_if(const double* p, int c, int cols) {
  long long v;
  asm volatile(
      "{\n .reg .pred q;\n setp.lt.s32 q, %2, %3;\n mov.b64 %0, 0;\n @q ld.global.b64 %0, [%1];\n}\n"
      : "=l"(v)
      : "l"(p), "r"(c), "r"(cols)
      : "memory");
  return v;
}
__device__ __forceinline__ void store_if(double* p, long long v, int c, int cols) {
  asm volatile("{\n .reg .pred q;\n setp.lt.s32 q, %2, %3;\n @q st.global.b64 [%0], %1;\n}\n" ::"l"(p),
               "l"(v), "r"(c), "r"(cols)
               : "memory");
}

// Sums of magnitude below 2^22 become integers by adding 1.5 2^23, whose bits they
// then follow (a conversion has an eighth of the addition's rate); what those bits
// add to an entry, S_1's in the upper word and S_6's and S_7's below, goes off at once.
constexpr float kMagic = 12582912.0f;
constexpr unsigned kMagicBits = 0x4B400000u;
constexpr unsigned long long kMagicSum =
    ((unsigned long long)(kMagicBits << 7) << 32) + 2ULL * kMagicBits;

// One lane of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(p));
  return p != 0;
}

// Tiles of step k: row block I takes column blocks k + 1 .. min(2 I + 1, nt - 1).
__host__ __device__ inline int row_tiles(int I, int k, int nt) {
  return (2 * I + 1 < nt - 1 ? 2 * I + 1 : nt - 1) - k;
}

template <bool kFirst>
__global__ void __launch_bounds__(kUpdThreads, 1) chol_update_kernel(
    double* __restrict__ a, int64_t ld, int64_t n, int64_t k, int64_t tiles, CholWork w) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* const A = smem;
  unsigned char* const B = smem + kBlockBytes;
  UpdBarriers& bar = *reinterpret_cast<UpdBarriers*>(smem + kBlockBytes + 2 * kBBytes);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    for (int s = 0; s < kSlices; ++s) tc::mbar_init(&bar.full_a[s], 1);
    tc::mbar_init(&bar.full_b[0], 1);
    tc::mbar_init(&bar.full_b[1], 1);
    tc::mbar_init(&bar.free_b[0], 1);
    tc::mbar_init(&bar.free_b[1], 1);
    for (int g = 0; g < kGroups; ++g) {
      tc::mbar_init(&bar.done[g], 1);
      tc::mbar_init(&bar.drained[g], kEpiWarps);
    }
    tc::mbar_init(&bar.last, 1);
  }
  if (warp == kEpiWarps) tc::tmem_alloc(&bar.tmem, 512);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tm = bar.tmem;
  chain();
  const int nt = (int)((n + kNB - 1) / kNB), ki = (int)k, workers = (int)gridDim.x;
  const int t0 = (int)(tiles * blockIdx.x / workers), t1 = (int)(tiles * (blockIdx.x + 1) / workers);
  int I = (ki + 1) / 2, left = t0;  // the first tile's row block and place in it
  while (left >= row_tiles(I, ki, nt)) left -= row_tiles(I++, ki, nt);
  int J = ki + 1 + left;
  auto next_tile = [&]() {
    if (++J - ki - 1 >= row_tiles(I, ki, nt)) {
      ++I;
      J = ki + 1;
    }
  };
  if (warp == kEpiWarps + 1) {
    if (lane == 0) {  // the copies: tile t's into buffer t mod 2 once tile t - 2's products are complete
      int cur = -1, loads = 0, it = 0;
      bool ok = true;
      for (; it < t1 - t0; ++it) {
        const int buf = it & 1;
        if (it > 1) ok = wait_phase(&bar.free_b[buf], (uint32_t)((it >> 1) - 1) & 1u);
        if (!ok) break;
        // the column block is half of a 128-row block in each slice
        const unsigned char* src = w.slices + (size_t)(J / 2) * kBlockBytes + (J & 1) * (kSliceBytes / 2);
        expect_tx(&bar.full_b[buf], kBBytes);
        for (int s = 0; s < kSlices; ++s)
          bulk_copy(B + buf * kBBytes + s * (kSliceBytes / 2), src + s * kSliceBytes, kSliceBytes / 2,
                    &bar.full_b[buf]);
        if (I != cur) {  // each of the rows' slices once tile t - 1 is through with it
          src = w.slices + (size_t)I * kBlockBytes;
          for (int s = 0; s < kSlices; ++s) {
            if (it > 0) ok = ok && wait_phase(&bar.done[s], (uint32_t)(it - 1) & 1u);
            if (!ok) break;
            expect_tx(&bar.full_a[s], kSliceBytes);
            bulk_copy(A + s * kSliceBytes, src + s * kSliceBytes, kSliceBytes, &bar.full_a[s]);
          }
          ++loads;
          cur = I;
        }
        next_tile();
      }
      if (!ok) atomicOr(w.flag, kGaveUp);
      // copies in flight land before the block ends
      for (int s = 0; s < kSlices && loads > 0; ++s) wait_phase(&bar.full_a[s], (uint32_t)(loads - 1) & 1u);
      for (int b = 0; b < 2; ++b)
        if (it > b) wait_phase(&bar.full_b[b], (uint32_t)((it - b - 1) >> 1) & 1u);
    }
  } else if (warp == kEpiWarps) {
    // The whole warp runs the loop and one elected lane issues, so that the
    // descriptors stay in uniform registers: issued from a branch on the lane
    // number, an MMA cost 110 cycles of moves.
    constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(kRowBlock >> 4) << 24);
    const uint64_t a0 = desc_sw128(tc::smem_addr(A)), b0 = desc_sw128(tc::smem_addr(B));
    int cur = -1, loads = 0;
    bool ok = true;
    for (int it = 0; it < t1 - t0 && ok; ++it) {
      const int buf = it & 1;
      const uint32_t before = (uint32_t)(it - 1) & 1u;
      const bool rows = I != cur;
      loads += rows;
      cur = I;
      ok = wait_phase(&bar.full_b[buf], (uint32_t)(it >> 1) & 1u);
      uint64_t at = a0, bt = b0 + (uint32_t)(buf * (kBBytes >> 4));
      asm volatile("" : "+l"(at), "+l"(bt));  // or all descriptors are kept across tiles
#pragma unroll
      for (int s = 0; s < kSlices; ++s) {
        if (rows) ok = wait_phase(&bar.full_a[s], (uint32_t)(loads - 1) & 1u) && ok;
        const int slices = min(kSlices, kGroups - s);  // of the columns: t = 0 .. slices - 1
#pragma unroll
        for (int t = 0; t < slices;) {
          // S_7 begins with slices 1 and 6, which take an MMA of their own
          const int c = min(s == 1 && t < 6 ? 6 - t : slices - t, 4);
          const bool begin = s == 0 || (s == 1 && t == 6);
          if (begin && it > 0) {
            for (int g = s + t; g < s + t + c; ++g) ok = wait_phase(&bar.drained[g], before) && ok;
          }
          ok = __all_sync(0xffffffffu, ok);
          if (ok) {
            tc::fence_after();
            if (elect_one()) {
#pragma unroll
              for (int q = 0; q < kNB / 16; ++q)  // 32 bytes along K inside the swizzled rows
                mma_f16(tm + (s + t) * kNB, at + (uint32_t)(s * (kSliceBytes >> 4) + 2 * q),
                        bt + (uint32_t)(t * (kSliceBytes >> 5) + 2 * q),
                        kIdesc | ((uint32_t)(c * (kNB >> 3)) << 17), !begin || q > 0);
            }
            __syncwarp();
          }
          t += c;
        }
        if (ok && elect_one()) {
          tc::commit(&bar.done[s]);
          if (s == kSlices - 1) {
            tc::commit(&bar.done[kGroups - 1]);
            tc::commit(&bar.free_b[buf]);
          }
        }
        __syncwarp();
      }
      next_tile();
    }
    // products in flight end before the accumulators are given back
    if (elect_one()) {
      if (!ok) atomicOr(w.flag, kGaveUp);
      tc::commit(&bar.last);
    }
    __syncwarp();
    wait_phase(&bar.last, 0);
  } else {
    const int row = 32 * (warp & 3) + lane, c0 = kEpiCols * (warp >> 2);
    const uint32_t taddr = tm + ((uint32_t)(32 * (warp & 3)) << 16) + c0;
    bool ok = true;
    for (int it = 0; it < t1 - t0 && ok; ++it) {
      const int r = I * kRowBlock + row, cb = J * kNB + c0;
      double* const p0 = a + r + cb * ld;
      // entries of the lower triangle: this thread's column c exists when cb + c <= r
      const int cols = r < n ? min(r - cb + 1, kEpiCols) : 0;
      long long acc[kEpiCols];
      double* p = p0;
#pragma unroll
      for (int c = 0; c < kEpiCols; ++c, p += ld) acc[c] = load_if(p, c, cols);
      if (it + 1 < t1 - t0) {  // the next tile's entries into L2, two lines of 16 rows per column
        int nI = I, nJ = J;
        if (++nJ - ki - 1 >= row_tiles(I, ki, nt)) {
          ++nI;
          nJ = ki + 1;
        }
        const int64_t pr = (int64_t)nI * kRowBlock + 32 * (warp & 3) + 16 * (lane & 1), pc = nJ * kNB + c0 + (lane >> 1);
        if (pr < n && pc < n && pc <= pr + 15) asm volatile("prefetch.global.L2 [%0];" ::"l"(a + pr + pc * ld));
      }
      if constexpr (kFirst) {
        const int sr = r < n ? w.scale[r] : 0;
#pragma unroll
        for (int c = 0; c < kEpiCols; ++c) {
          long long f = 0;
          if (c < cols && !to_fixed(__longlong_as_double(acc[c]), sr + w.scale[cb + c], f)) atomicOr(w.flag, kNotPd);
          acc[c] = f;
        }
      }
      unsigned top[kEpiCols];  // S_0 and S_1's part of the upper words
#pragma unroll
      for (int g = 0; g < kGroups; ++g) {
        ok = wait_phase(&bar.done[g], (uint32_t)it & 1u) && ok;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc::fence_after();
        uint32_t v[kEpiCols];
#pragma unroll
        for (int c = 0; c < kEpiCols; c += 16) ld16(taddr + g * kNB + c, v + c);
        ld_wait(v);
        tc::fence_before();
        __syncwarp();
        if (lane == 0) arrive(&bar.drained[g]);
#pragma unroll
        for (int c = 0; c < kEpiCols; ++c) {
          const float S = __uint_as_float(v[c]);
          if (g == 0) top[c] = __float_as_uint(S + kMagic) << 16;  // |S_0| <= 2^18
          else if (g == 1) top[c] += __float_as_uint(S + kMagic) << 7;  // <= 2^21
          else if (g >= 6) acc[c] -= __float_as_uint(fmaf(S, g == 6 ? 0x1p-6f : 0x1p-15f, kMagic));
          else acc[c] = mad_wide(__float2int_rn(S), -(1 << (48 - 9 * g)), acc[c]);
          if (g == 1) acc[c] += kMagicSum - ((unsigned long long)top[c] << 32);
        }
      }
      if (ok) {
        p = p0;
        asm volatile("" : "+l"(p));  // or the loads' addresses are kept for the stores
#pragma unroll
        for (int c = 0; c < kEpiCols; ++c, p += ld) store_if(p, acc[c], c, cols);
      }
      next_tile();
    }
    if (!ok && lane == 0) atomicOr(w.flag, kGaveUp);
  }
  tc::fence_before();
  __syncthreads();
  if (warp == kEpiWarps) tc::tmem_dealloc(tm, 512);
}

// The last panel's finish, then out = [l, log det, z^T a^{-1} z] from the panels' sums.
__global__ void __launch_bounds__(kPanelThreads) chol_finish_kernel(
    double* __restrict__ a, int64_t ld, int64_t n, int64_t nt, double* __restrict__ y,
    double* __restrict__ out, CholWork w, unsigned long long* __restrict__ ctr) {
  __shared__ double sh[kNB * (kNB + 1) + 12 * kNB];
  chain();
  finish_panel(a, ld, n, nt - 1, y, w, sh);
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  double ld_ = 0.0, q = 0.0;
  for (int64_t k = lane; k < nt; k += 32) {
    ld_ += w.part[2 * k];
    q += w.part[2 * k + 1];
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    ld_ += __shfl_xor_sync(0xffffffffu, ld_, s);
    q += __shfl_xor_sync(0xffffffffu, q, s);
  }
  if (lane != 0) return;
  if (const int flag = *w.flag; flag != 0) {
    ld_ = q = qnan();
    if (ctr != nullptr) atomicAdd(ctr + BK_CTR_FAIL, (flag & kGaveUp) != 0 ? 1ull << 32 : 1ull);
  }
  out[1] = 2.0 * ld_;
  out[2] = q;
  out[0] = -0.5 * (q + 2.0 * ld_ + (double)n * 1.8378770664093454836);  // log 2 pi
}

template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), int64_t grid, int block, size_t smem, cudaStream_t s,
                           A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, (P)args...);
}

// Shared memory beyond 48 KB: opted in once per device.
cudaError_t set_chol_smem() {
  static std::atomic<bool> done[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  e = cudaFuncSetAttribute(chol_panel_kernel<true, 4>, attr, (int)sizeof(PanelSmem));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(chol_panel_kernel<true, 5>, attr, (int)sizeof(PanelSmem));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(chol_panel_kernel<false, 4>, attr, (int)sizeof(PanelSmem));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(chol_panel_kernel<false, 5>, attr, (int)sizeof(PanelSmem));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(chol_update_kernel<true>, attr, (int)kUpdSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(chol_update_kernel<false>, attr, (int)kUpdSmem);
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
  return e;
}

}  // namespace

size_t loglik_workspace_bytes(int64_t n) { return chol_layout(n).total; }

cudaError_t launch_loglik_fixed(double* a, int64_t n, int64_t ld, const double* z, double* y,
                                double* out, unsigned long long* ctr, void* work, cudaStream_t s) {
  cudaError_t e = set_chol_smem();
  if (e != cudaSuccess) return e;
  const CholLayout l = chol_layout(n);
  unsigned char* const base = (unsigned char*)work;
  const CholWork w{(int*)base, (int*)(base + l.scale), (double*)(base + l.diag),
                   (double*)(base + l.part), (float*)(base + l.squares), base + l.slices};
  if ((e = cudaMemsetAsync(w.flag, 0, sizeof(int), s)) != cudaSuccess) return e;
  chol_prep_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, ld, n, z, y, w);
  const int64_t nt = (n + kNB - 1) / kNB, R = (n + kRowBlock - 1) / kRowBlock;
  const int64_t sms = current_sm_count();
  for (int64_t k = 0; k < nt; ++k) {
    const int64_t below = n - (k + 1) * kNB;  // rows below the panel
    const bool wide = below > (sms - 8) * solve_rows(4);  // a few blocks stay for the substitution
    const int rows = solve_rows(wide ? 5 : 4);
    // the last one has no rows of its own and writes the diagonal tile
    const int row_blocks = 1 + (below > 0 ? (int)((below + rows - 1) / rows) : 0);
    const int extra = k == 0 ? 0 : k == 1 ? 1 : 1 + (int)((n - k * kNB + 255) / 256);
    const auto panel = k == 0 ? (wide ? chol_panel_kernel<true, 5> : chol_panel_kernel<true, 4>)
                              : (wide ? chol_panel_kernel<false, 5> : chol_panel_kernel<false, 4>);
    e = launch_chained(panel, row_blocks + extra, kPanelThreads, sizeof(PanelSmem), s, a, ld, n, k,
                       row_blocks, rows, y, w);
    if (e != cudaSuccess) return e;
    if (below <= 0) break;
    int64_t tiles = 0;
    for (int I = (int)(k + 1) / 2; I < R; ++I) tiles += row_tiles(I, (int)k, (int)nt);
    const auto update = k == 0 ? chol_update_kernel<true> : chol_update_kernel<false>;
    e = launch_chained(update, tiles < sms ? tiles : sms, kUpdThreads, kUpdSmem, s, a, ld, n, k, tiles, w);
    if (e != cudaSuccess) return e;
  }
  return launch_chained(chol_finish_kernel, 1, kPanelThreads, 0, s, a, ld, n, nt, y, out, w, ctr);
}

}  // namespace bk
