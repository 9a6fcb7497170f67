// The Matern entry as a function of r^2 alone.  One call's (sigma^2, beta, nu)
// are fixed, so that M(r) = sigma^2 2^{1-nu}/Gamma(nu) x^nu K_nu(x), x = r/beta,
// is one smooth function of r^2.  A small kernel tabulates it once per call,
// on intervals of r^2, by polynomials whose coefficients come from the integral
// of Sec. IV-B; an entry then costs its squared distance, one table record
// and a fixed-point Horner scheme instead of its own quadrature (about 120
// instructions against about 1,500).
//
// The integral.  With t = tau - log x,
//   x^nu K_nu(x) = F_nu(s) = 1/2 int_{-inf}^{inf} e^{nu tau - e^tau/2} e^{-s e^{-tau}/2} dtau,
// s = x^2: the trapezoid rule on a grid of tau that does not depend on x turns
// F_nu into a sum of decaying exponentials of s,
//   F_nu(s) = sum_j w_j e^{-s v_j},  v_j = e^{-tau_j}/2,
// whose derivatives -2 F_nu' = F_{nu-1} = sum_j 2 v_j w_j e^{-s v_j} alternate in
// sign: expanded about the right end of an interval in the distance u to it,
// every coefficient is positive, c_k = (W/2)^k/k! F_{nu-k} for an interval of
// width W, and nothing cancels (FP32 records expand about the left end, with
// alternating signs, which their intervals can afford).  F_nu and F_{nu-1} come from the sums, the
// rest from K's recurrence in the order, s F_{mu-1} = F_{mu+1} - 2 mu F_mu.
//
// The intervals.  Every binade of r^2 is cut into 2^m equal parts, so that an
// interval's number and the position inside it are bit fields of r^2.  m = 7
// up to x = 2 (the series about s in powers of W/s <= 2^-7 past the branch
// point at s = 0), 8 and 9 up to x = 8 and from there growing with x so that
// x W/(2 s) <= 1/64, the ratio of the series of e^{-x}: degree 6 then leaves
// less than 4e-16 of M (checked in the orders' ratio K_{nu-7}/K_nu too).  The
// FP32 records take two or more bits less and degree 3 (an economised
// quartic; 1e-8 at worst, for nu = 0.02, else below 5e-9, checked against K).
// Fewer and wider intervals mean fewer cache lines a warp's load touches.  Binades with x^2 in [2^-18, 2^14) are covered (x from 2.8e-3
// to 90 at least); entries outside take the direct evaluation.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "bk_forms.cuh"
#include "bk_matern_common.cuh"
#include "bk_math64.cuh"

namespace bk {

constexpr float kInfF = __builtin_huge_valf();
constexpr int kTabTile = 64;  // tile edge of the writers that use a table
constexpr int kTauMax = 384;
static __device__ const double kTauTab[2 * kTauMax + 1] = {
#include "bk_tau_table.inc"
};

// Binades of x^2: q = kTabQ0 .. kTabQ0 + kTabOct - 1 (x^2 = f 2^q with the
// significand f of 1/beta^2, so the binades of r^2 map onto them one to one).
constexpr int kTabQ0 = -18, kTabOct = 31;

// Layout of a table for FP64 or FP32 records: log2 of the intervals in binade
// o = q - kTabQ0, and the first of them.
template <bool F32>
struct TabLayout {
  static constexpr int kRecord = F32 ? 16 : 32;  // bytes
  __host__ __device__ static constexpr int bits(int o) {
    const int q = o + kTabQ0;
    if (F32) return q < 2 ? 5 : q < 4 ? 6 : (q + 8) >> 1;
    return q < 0 ? 7 : q < 3 ? 8 : q < 5 ? 9 : (q + 13) >> 1;
  }
  __host__ __device__ static constexpr int first(int o) {
    int b = 0;
    for (int i = 0; i < o; ++i) b += 1 << bits(i);
    return b;
  }
  static constexpr int kBins = first(kTabOct);
  // FP32 tables end in two records without a value, for what lies outside them,
  // and 256 words by the exponent of r^2 (tab_octave32).
  static constexpr int kExtra = F32 ? 2 : 0, kWords = F32 ? 256 : 0;
  static constexpr size_t kBytes = (size_t)(kBins + kExtra) * kRecord + kWords * sizeof(int);
};
using TabLayout64 = TabLayout<false>;
using TabLayout32 = TabLayout<true>;

// Scales of the fixed-point coefficients: c_k is held in units of 2^-S_k of
// the record's power of two 2^E, the value's upper bound.
//  FP64 record, 32 bytes (two 16-byte loads):
//   words 0-1  c_0 (units 2^-62, its low 11 bits zero) + the exponent word,
//   words 2-3  c_1 (2^-67) with c_6 (2^-54) in its low 12 bits,
//   words 4-5  c_2 (2^-74) with c_5 (2^-54) in its low 19 bits,
//   words 6-7  c_3 (2^-51), c_4 (2^-54).
//  The bits that share a word with c_1 and c_2 lie below 2^-55 of the value and
//  are left in place.
// The top bit of c_0 stays free: the value may round up to 2^E itself.  An
// exponent word of 0 marks an interval without a usable polynomial.
//  An FP32 record is a cubic in four floats; a constant of NaN marks an interval
//  without one.
constexpr int kS0 = 62, kS1 = 67, kS2 = 74, kS3 = 51, kS4 = 54;
constexpr int kTabNodes = 485;                  // tau = -24 .. 6.25 in steps of 1/16

// Whether (sigma^2, beta, nu) are inside the tables' domain: orders for which
// the node grid holds the integral, and scales that keep every value, the FP32
// squared distances included, a normal number.
__host__ __device__ inline bool tab_domain(double sigma2, double beta, double nu) {
  return nu >= 0.02 && nu <= 10.0 && beta >= 1e-8 && beta <= 1e8 && sigma2 >= 1e-20 &&
         sigma2 <= 1e20;
}

// Whether a matrix of rows x cols entries is worth a table (see
// entry_table_pays).
__host__ __device__ inline bool entry_table_size(int64_t rows, int64_t cols) {
  constexpr int64_t kLeast = (int64_t)1 << 19;
  return rows > 0 && cols > 0 && rows >= (kLeast + cols - 1) / cols;
}

// One instance of a batch: its descriptor, checked, and its constants.
struct BatchInstance {
  const double* locs;
  void* out;
  int64_t n, ld;
  int64_t table;  // whether its entries come from a table
  MaternParams mp;
};

// The biased exponent of the first binade of r^2: 1/beta^2 = f 2^k, q = e + k.
__device__ __forceinline__ unsigned tab_first_binade(double inv_beta) {
  const int k = (int)((__double2hiint(inv_beta * inv_beta) >> 20) & 0x7ff) - 1023;
  return (unsigned)(kTabQ0 - k + 1023);
}

// The power of two of 1/beta that scales coordinates for FP32 records, 1/beta^2 =
// f 4^h with f in [1, 4), and whether f >= 2.
struct TabScale {
  int h, odd;
};
__device__ __forceinline__ TabScale tab_scale(double inv_beta) {
  const int h = ((__double2hiint(inv_beta) >> 20) & 0x7ff) - 1023;
  const int k = ((__double2hiint(inv_beta * inv_beta) >> 20) & 0x7ff) - 1023;
  return TabScale{h, k - 2 * h};
}

// The word of FP32 exponent field ex: 32 (first interval less the leading bits) +
// shift; 31, which leads to the last two records, outside the table.
__device__ __forceinline__ int tab_octave32(int ex, int odd) {
  using L = TabLayout32;
  const int q = ex - 127 + odd, o = q - kTabQ0;
  int first = L::kBins, sh = 31;
#pragma unroll
  for (int k = 0; k < kTabOct; ++k) {
    if (k == o) {
      sh = 23 - L::bits(k);
      first = L::first(k) - (ex << L::bits(k));
    }
  }
  return (int)((unsigned)first << 5) | sh;
}

// ---------------------------------------------------------------------------
// Building a table.  A block of 1,024 threads first evaluates the node weights
// (all tau of the grid, for this nu) into shared memory; then eight lanes per
// interval sum F_nu and F_{nu-1} at its right end over the nodes that matter
// there (about 25 to 100, the most near x = 0), and 128 threads write the 128
// records.  One block per SM covers the FP64 table; a block's intervals are
// grid-strided, so that every block gets the same share of costly ones.  The
// FP64 pipe bounds it, so the exponentials run on the integer pipe (exp2s_int)
// and the recurrence, which needs one thread per interval, on full warps.
constexpr int kTabLanes = 8;
constexpr int kTabThreads = 1024;
constexpr int kTabBinsPerBlock = kTabThreads / kTabLanes;
struct TabBuildSmem {
  double v[kTabNodes], w[kTabNodes], w2[kTabNodes];
  double f0[kTabBinsPerBlock], f1[kTabBinsPerBlock];
  float box[kTabThreads / 32][4];
};

// c 2^scale for c >= 0, rounded to nearest, on the integer pipe.
__device__ __forceinline__ unsigned long long tab_fix(double c, int scale) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(c);
  const int sh = (int)(b >> 52) - 1075 + scale;
  const unsigned long long sig = (b & 0xfffffffffffffULL) | 0x10000000000000ULL;
  if (sh >= 0) return sig << sh;
  return sh < -54 ? 0ULL : (sig + (1ULL << (-sh - 1))) >> -sh;
}

// Node weights for the order nu, log c = log(sigma^2 2^{1-nu}/Gamma(nu)) in
// them: w = (1/16)/2 c e^{nu tau - e^tau/2}, w2 = w e^{-tau}, and v =
// -e^{-tau}/2 in the units of exp2s_int (times 4096/ln 2).
__device__ __forceinline__ void tab_nodes(TabBuildSmem& sm, double nu, double log_c) {
  for (int i = threadIdx.x; i < kTabNodes; i += blockDim.x) {
    const int j = i - kTauMax;  // tau = j/16
    const double ep = kTauTab[j + kTauMax], en = kTauTab[kTauMax - j];
    const double a = fma(nu, 0.0625 * (double)j, -0.5 * ep) + log_c;
    const double w = 0.03125 * exp_units_full(a * kExpScale, kExp2Tab);
    sm.v[i] = (-0.5 * kExpScale) * en;
    sm.w[i] = w;
    sm.w2[i] = w * en;
  }
}

// The interval's binade, the position in it and the expansion point: its
// right end less one FP64 ulp (its largest double), for FP32 records its left end.
template <bool F32>
__device__ __forceinline__ void tab_interval(int bin, unsigned e0, int& o, int& m, double& s_ref) {
  using L = TabLayout<F32>;
  constexpr int kFlat = -kTabQ0, kFlatBits = L::bits(0);  // binades below x = 1 are cut alike
  int i = bin & ((1 << kFlatBits) - 1);
  o = min(bin >> kFlatBits, kFlat);
  m = kFlatBits;
#pragma unroll
  for (int k = kFlat; k < kTabOct; ++k) {
    if (bin >= L::first(k)) {
      o = k;
      i = bin - L::first(k);
      m = L::bits(k);
    }
  }
  s_ref = __longlong_as_double((long long)(((unsigned long long)(e0 + o) << 52) +
                                           ((unsigned long long)(F32 ? i : i + 1) << (52 - m)) -
                                           (F32 ? 0ULL : 1ULL)));
}

// An upper bound of every squared distance between two sets of locations, from
// their common bounding box (FP32, rounded outwards); infinite when a
// coordinate is not finite.  Every thread of the block calls it.
__device__ __forceinline__ double tab_r2_bound(float (*s_box)[4], const double* __restrict__ locs1,
                                               int64_t m, const double* __restrict__ locs2, int64_t n) {
  float lo[2] = {kInfF, kInfF}, hi[2] = {-kInfF, -kInfF};
  for (int set = 0; set < 2; ++set) {
    const double* const l = set ? locs2 : locs1;
    const int64_t len = set ? n : m;
    if (set && locs2 == locs1) break;
    for (int64_t i = threadIdx.x; i < len; i += blockDim.x) {
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        const float v = f32_trunc(l[d * len + i]);
        if (!isfinite(v)) hi[d] = kInfF;
        lo[d] = fminf(lo[d], v);
        hi[d] = fmaxf(hi[d], v);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
      hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
    }
  }
  if ((threadIdx.x & 31) == 0) {
    float* const b = s_box[threadIdx.x >> 5];
    b[0] = lo[0];
    b[1] = lo[1];
    b[2] = hi[0];
    b[3] = hi[1];
  }
  __syncthreads();
  const float* const b = s_box[threadIdx.x & ((blockDim.x >> 5) - 1)];
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    lo[d] = b[d];
    hi[d] = b[2 + d];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
      hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
    }
  }
  // truncation took at most 2^-23 of a coordinate's magnitude from each end
  float r2 = 0.0f;
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    const float e = (hi[d] - lo[d]) + 0x1p-21f * (fabsf(hi[d]) + fabsf(lo[d])) + 1e-30f;
    r2 = fmaf(e, e, r2);
  }
  return widen_f(r2 * 1.001f);
}

// Writes the record of one interval from F_nu and F_{nu-1} at its expansion
// point (unless the interval lies beyond r2_max).
template <bool F32>
__device__ __forceinline__ void tab_record(int bin, double nu, unsigned e0, double ib, double b2,
                                           double b2lo, double r2_max, double f0, double f1,
                                           unsigned char* __restrict__ table) {
  using L = TabLayout<F32>;
  int o, m;
  double s_ref;
  tab_interval<F32>(bin, e0, o, m, s_ref);
  if (!bits_le(__hiloint2double((int)((e0 + o) << 20), 0), r2_max)) return;
  const double s = fma(s_ref, b2, s_ref * b2lo);
  // c_k = q^k/k! s^k F_{nu-k}, q = W/(2 s) in units of r^2: c_0 = F_nu, c_1 = q s F_{nu-1},
  // c_{k+1} = s q^2/(k (k+1)) c_{k-1} - 2 (nu - k) q/(k+1) c_k
  const double q = __longlong_as_double((long long)(e0 + o - m - 1) << 52) * rcp_nr2(s_ref);
  constexpr int kDeg = F32 ? 4 : 6;
  double c[kDeg + 1];
  c[0] = f0;
  const double sq = s * q;
  c[1] = sq * f1;
  const double sq2 = sq * q;
#pragma unroll
  for (int k = 1; k < kDeg; ++k)
    c[k + 1] = fma(sq2 * (1.0 / (k * (k + 1))), c[k - 1], (q * ((-2.0 / (k + 1)) * (nu - k))) * c[k]);
  if constexpr (F32) {
    // F = c_0 - c_1 u + c_2 u^2 - c_3 u^3 + c_4 u^4, u^4 replaced by its cubic best
    // approximation on [0, 1], u^4 ~ 2 u^3 - 5/4 u^2 + u/4 - 1/128
    const double a0 = fma(-1.0 / 128.0, c[4], c[0]);
    const float f = (float)a0;
    // The constant's rounding error d is spread over the interval, d (1 - 15/2 u +
    // 15 u^2 - 35/4 u^3): the cubic of least square mean among those that are d at 0.
    const double d = a0 - (double)f;
    const double a1 = fma(7.5, d, fma(0.25, c[4], -c[1])), a2 = fma(-15.0, d, fma(-1.25, c[4], c[2])),
                 a3 = fma(8.75, d, fma(2.0, c[4], -c[3]));
    // in units of the scaled square, in which the interval's width is 2^w
    const int w = o + kTabQ0 - tab_scale(ib).odd - m;
    const double iw = __hiloint2double((1023 - w) << 20, 0);
    const bool ok = f >= 0x1p-120f && f <= 0x1p50f;
    reinterpret_cast<float4*>(table)[bin] = make_float4(ok ? f : __int_as_float(0x7fc00000), (float)(a1 * iw),
                                                        (float)(a2 * (iw * iw)), (float)(a3 * (iw * iw * iw)));
  } else {
  double vmax = c[kDeg];  // the value at the left end, the largest of the interval
#pragma unroll
  for (int k = kDeg - 1; k >= 0; --k) vmax += c[k];
  const int ev = (int)((unsigned)__double2hiint(vmax) >> 20);  // 2048 and above: negative
  const int E = ev - 1022;                                     // vmax in [2^{E-1}, 2^E)
  // signs, and the bounds that the scales were chosen for (c_k < 2^{E-b})
  auto below = [&](int k, int b) { return (int)((unsigned)__double2hiint(c[k]) >> 20) < ev + 1 - b; };
  bool ok = ev > 60 && ev < 1980;
  // exponent words: the exponent field of 2^{E-1} less the leading bit that the
  // significand adds
  uint4* rec = reinterpret_cast<uint4*>(table + (size_t)bin * L::kRecord);
    ok = ok && below(0, 0) && below(1, 5) && below(2, 12) && below(3, 20) && below(4, 23) &&
         below(5, 35) && below(6, 42);
    const unsigned long long c0 = (tab_fix(c[0], kS0 - 11 - E) << 11) | (ok ? (unsigned)(E + 1021) : 0u);
    const unsigned long long c1 = (tab_fix(c[1], kS1 - E) & ~0xfffULL) | (tab_fix(c[6], kS4 - E) & 0xfffULL);
    const unsigned long long c2 = (tab_fix(c[2], kS2 - E) & ~0x7ffffULL) | (tab_fix(c[5], kS4 - E) & 0x7ffffULL);
    rec[0] = make_uint4((unsigned)c0, (unsigned)(c0 >> 32), (unsigned)c1, (unsigned)(c1 >> 32));
    rec[1] = make_uint4((unsigned)c2, (unsigned)(c2 >> 32), (unsigned)tab_fix(c[3], kS3 - E),
                        (unsigned)tab_fix(c[4], kS4 - E));
  }
}

template <bool F32>
__device__ __forceinline__ void tab_build_block(TabBuildSmem& sm, const MaternParams& mp, int block,
                                                int blocks, double r2_max,
                                                unsigned char* __restrict__ table) {
  using L = TabLayout<F32>;
  tab_nodes(sm, mp.nu, mp.log_pref);
  __syncthreads();
  const unsigned e0 = tab_first_binade(mp.inv_beta);
  // x^2 = s_ref/beta^2, with the rounding of 1/beta and of its square taken back
  const double ib = mp.inv_beta, b2 = ib * ib;
  const double b2lo = fma(ib, ib, -b2) + 2.0 * ib * (fma(-ib, mp.beta, 1.0) * ib);
  const float nuf = f32_trunc(mp.nu);
  if (F32 && block == 0) {
    if (threadIdx.x < L::kExtra)
      reinterpret_cast<float4*>(table)[L::kBins + threadIdx.x] =
          make_float4(__int_as_float(0x7fc00000), 0.0f, 0.0f, 0.0f);
    if (threadIdx.x < L::kWords)
      reinterpret_cast<int*>(table + (size_t)(L::kBins + L::kExtra) * L::kRecord)[threadIdx.x] =
          tab_octave32((int)threadIdx.x, tab_scale(ib).odd);
  }
  for (int k0 = 0; k0 * blocks + block < L::kBins; k0 += kTabBinsPerBlock) {
    if (k0 > 0) __syncthreads();  // the previous round's sums have been read
    const int k = (int)threadIdx.x / kTabLanes, lane = threadIdx.x % kTabLanes;
    int o, m;
    double s_ref;
    tab_interval<F32>(min((k0 + k) * blocks + block, L::kBins - 1), e0, o, m, s_ref);
    const double s = fma(s_ref, b2, s_ref * b2lo);
    const bool use = bits_le(__hiloint2double((int)((e0 + o) << 20), 0), r2_max);
    double f0 = 0.0, f1 = 0.0;
    int step = 1;
    if (use) {
      // Nodes with terms above e^-36 of the largest (e^-24 for FP32 records): tau
      // = log x + t, x (cosh t - 1) - nu t below that to the right, x (cosh t - 1)
      // to the left, and nu (log x + t) above its negative.  The step is 1/16
      // times 1 to 4, the largest that keeps the trapezoid rule's error below
      // 3e-16 (1e-10) up to the binade's end (checked against 30-digit values).
      constexpr float kCut = F32 ? 24.0f : 36.0f;
      const float xf = sqrtf(f32_trunc(s)), lx = __logf(xf), rx = 1.0f / xf;
      const float ar = fmaf(kCut + 6.0f * nuf, rx, 1.0f), al = fmaf(kCut, rx, 1.0f);
      const float tr = __logf(ar + sqrtf(fmaf(ar, ar, -1.0f))), tl = __logf(al + sqrtf(fmaf(al, al, -1.0f)));
      const int q = o + kTabQ0;
      step = F32 ? (q <= 4 && nuf <= 5.0f ? 4 : q <= 6 ? 3 : q <= 8 ? 2 : 1)
                           : (q <= 4 && nuf <= 2.5f ? 3 : q <= 8 ? 2 : 1);
      const int j0 = max((int)floorf(16.0f * fmaxf(lx - tl, -kCut / nuf - 6.0f)), -kTauMax);
      const int j1 = min((int)ceilf(16.0f * (lx + tr)), kTabNodes - 1 - kTauMax);
#pragma unroll 2
      for (int j = j0 + step * lane; j <= j1; j += step * kTabLanes) {
        const double u = s * sm.v[j + kTauMax];
        if ((unsigned)__double2hiint(u) < 0xc14fe000u) {  // u > -4.18e6: the term's factor above e^-707
          const double e = exp2s_int(u, kExp2Tab);
          f0 = fma(sm.w[j + kTauMax], e, f0);
          f1 = fma(sm.w2[j + kTauMax], e, f1);
        }
      }
    }
    const unsigned mask = 0xffu << (threadIdx.x & 24);
#pragma unroll
    for (int d = 1; d < kTabLanes; d <<= 1) {
      f0 += __shfl_xor_sync(mask, f0, d);
      f1 += __shfl_xor_sync(mask, f1, d);
    }
    if (lane == 0) {
      sm.f0[k] = (double)step * f0;
      sm.f1[k] = (double)step * f1;
    }
    __syncthreads();
    const int bin = (k0 + (int)threadIdx.x) * blocks + block;
    if (threadIdx.x < kTabBinsPerBlock && bin < L::kBins)
      tab_record<F32>(bin, mp.nu, e0, ib, b2, b2lo, r2_max, sm.f0[threadIdx.x], sm.f1[threadIdx.x], table);
  }
}

// ---------------------------------------------------------------------------
// Evaluating an entry.

// (a u) >> 64 for a, u < 2^63, without the product of the low words (less
// than one unit low).
__device__ __forceinline__ unsigned long long mulhi63(unsigned long long a, unsigned long long u) {
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, uh = (unsigned)(u >> 32), ul = (unsigned)u;
  unsigned long long t = (unsigned long long)al * uh;
  t = (unsigned long long)ah * ul + t;
  return (unsigned long long)ah * uh + (t >> 32);
}

// The octave table of the FP64 evaluation, one int2 per binade in shared memory:
// {shift of r^2's leading word, first interval less the binade's leading bits}.
__device__ __forceinline__ void tab_stage_octaves(int2* s_oct, unsigned e0) {
  using L = TabLayout64;
  if (threadIdx.x < kTabOct) {
    const int o = threadIdx.x, sh = 20 - L::bits(o);
    s_oct[o] = make_int2(sh, L::first(o) - (int)((e0 + o) << (20 - sh)));
  }
}

// M for the squared distance r2 (a double), false when r2 lies outside the
// table (zero and NaN among it).
__device__ __forceinline__ bool tab_entry64(const unsigned char* __restrict__ table,
                                            const int2* s_oct, unsigned e0, double r2, double& out) {
  const unsigned hi = (unsigned)__double2hiint(r2), lo = (unsigned)__double2loint(r2);
  const unsigned o = (hi >> 20) - e0;
  const bool in = o < (unsigned)kTabOct;
  const int2 oc = s_oct[in ? o : 0];
  const int idx = in ? (int)(hi >> oc.x) + oc.y : 0;
  const uint4* rec = reinterpret_cast<const uint4*>(table) + 2 * idx;
  const uint4 a = __ldg(rec), b = __ldg(rec + 1);
  // distance to the expansion point in units of the interval: 64 fraction bits
  const unsigned long long v = (~(((unsigned long long)hi << 32) | lo)) << (32 - oc.x);
  const unsigned u32 = (unsigned)(v >> 32);
  const unsigned long long u = v >> 1;
  unsigned A = (b.x & 0x7ffffu) + __umulhi(a.z & 0xfffu, u32);
  A = b.w + __umulhi(A, u32);
  A = b.z + (__umulhi(A, u32) >> (kS4 - kS3));
  const unsigned long long A2 =
      (((unsigned long long)b.y << 32) | b.x) + (((unsigned long long)A * u32) >> (kS3 + 32 - kS2));
  const unsigned long long A1 = (((unsigned long long)a.w << 32) | a.z) + (mulhi63(A2, u) >> (kS2 - kS1 - 1));
  unsigned long long F =
      (((unsigned long long)a.y << 32) | (a.x & ~0x7ffu)) + (mulhi63(A1, u) >> (kS1 - kS0 - 1));
  // F 2^{E-62}, F in [2^60, 2^62]
  const unsigned ex = a.x & 0x7ffu;
  unsigned ew = ex;
  if ((unsigned)(F >> 32) < 0x20000000u) {
    F <<= 1;
    --ew;
  }
  F = (F + 256ULL) >> 9;
  out = __hiloint2double((int)((unsigned)(F >> 32) + (ew << 20)), (int)(unsigned)F);
  return in && ex != 0u;
}

// ---------------------------------------------------------------------------
// FP32 entries: about 35 instructions, most of them on the FP32 pipe (with
// double-float differences of global coordinates and a fixed-point Horner
// scheme it was 125, 60 of them on the integer pipe: n = 40,000 took 3.60 ms,
// now 1.67).  The record loads bound it now: a warp's 32 distances touch about
// nine cache lines.  A matrix's rms error is 2.6e-8, against 2.5e-8 of rounding alone.
//
// Coordinates.  A tile's coordinates are held relative to its first row's point, in
// units of 2^h of 1/beta, each as two floats: a multiple of Q = E/1024, E a power
// of two above every difference between a row and a column, and the rest to
// Q 2^-25.  Differences of the first parts and sums of their squares are then
// exact without error terms; what the second parts add is rounded to 2^-33 E of
// the distance.
//
// Intervals.  The FP32 bits of the square t = x^2/f index, by their exponent, a
// word of shift and first interval in shared memory, 256 of them so that no
// range check is needed: what lies outside the table has a shift of 31, which
// leads to one of the two records without a value.
struct TabPoints32 {
  float4 p[2 * kTabTile];  // rows, then columns: {x first part, x rest, y first part, y rest}
  int oct[256];            // tab_octave32
  unsigned extent[4];
};

// Stages a tile's points and octaves; every thread of the block calls it (the
// caller synchronises before the last readers of sm and after).  False: the
// tile spans more than the coordinates' precision allows (or is not finite).
template <int THREADS>
__device__ __forceinline__ bool tab_stage32(TabPoints32& sm, const double* __restrict__ locs1, int64_t m,
                                            const double* __restrict__ locs2, int64_t n, int64_t r0,
                                            int64_t c0, const MaternParams& mp,
                                            const unsigned char* __restrict__ table) {
  static_assert(THREADS >= 2 * kTabTile, "one thread per point");
  const int tid = threadIdx.x, lane = tid & 31;
  double wx = 0.0, wy = 0.0;
  if (tid < 2 * kTabTile) {
    const bool row = tid < kTabTile;
    const double* const l = row ? locs1 : locs2;
    const int64_t len = row ? m : n, i = row ? r0 + tid : c0 + (tid - kTabTile);
    if (i < len) {
      wx = l[i] - locs1[r0];
      wy = l[len + i] - locs1[m + r0];
    }
    const unsigned a = max((unsigned)__double2hiint(wx) & 0x7fffffffu, (unsigned)__double2hiint(wy) & 0x7fffffffu);
    const unsigned warp_max = __reduce_max_sync(0xffffffffu, a);
    if (lane == 0) sm.extent[tid >> 5] = warp_max;
  }
  __syncthreads();
  // 2^e above the sum of the rows' and the columns' largest coordinate
  const unsigned hr = max(sm.extent[0], sm.extent[1]), hc = max(sm.extent[2], sm.extent[3]);
  const unsigned a = max(hr, hc), b = min(hr, hc);
  const unsigned sum = ((a & 0xfffffu) | 0x100000u) + (((b & 0xfffffu) | 0x100000u) >> min((a >> 20) - (b >> 20), 31u)) + 3u;
  const int e = (int)(a >> 20) - 1022 + (sum >> 21 ? 1 : 0);
  const TabScale sc = tab_scale(mp.inv_beta);
  const int es = max(e + sc.h, -40);
  // d ln M/dx is at most 1 for nu >= 1/2, 1 + 1/x below; x is off by 2^{es-32} at
  // most, and M may be by 2^-26 (its rounding to FP32 is 2^-24)
  using L = TabLayout32;
  const int ex_min = mp.nu >= 0.5 ? 0 : 2 * es - 12 + 127 - sc.odd;
  const int* const words = reinterpret_cast<const int*>(table + (size_t)(L::kBins + L::kExtra) * L::kRecord);
#pragma unroll
  for (int k = tid; k < L::kWords; k += THREADS) sm.oct[k] = k < ex_min ? (L::kBins << 5) | 31 : __ldg(words + k);
  if (tid < 2 * kTabTile) {
    // one FP64 fma to an integer in units of 2^{es-35}
    const double scale = __hiloint2double((1023 + sc.h - es + 35) << 20, 0);
    const float u1 = __int_as_float((127 + es - 10) << 23), u2 = __int_as_float((127 + es - 35) << 23);
    const long long kMagic = 0x4338000000000000LL;  // 1.5 2^52
    auto split = [&](double w, float& f1, float& f2) {
      const long long k = __double_as_longlong(fma(w, scale, __longlong_as_double(kMagic))) - kMagic;
      const int k1 = (int)((k + (1 << 24)) >> 25), k2 = (int)(k - ((long long)k1 << 25));
      f1 = (float)k1 * u1;
      f2 = (float)k2 * u2;
    };
    float4 p;
    split(wx, p.x, p.y);
    split(wy, p.z, p.w);
    sm.p[tid] = p;
  }
  return es <= 6;
}

// M between the points a and b; NaN when they lie outside the table.
__device__ __forceinline__ float tab_entry32(const unsigned char* __restrict__ table, const int* s_oct,
                                             const float4& a, const float4& b) {
  const float dx = b.x - a.x, lx = b.y - a.y, dy = b.z - a.z, ly = b.w - a.w;
  const float h = fmaf(dx, dx, dy * dy);                                           // exact
  const float l = fmaf(ly, fmaf(2.0f, dy, ly), lx * fmaf(2.0f, dx, lx));
  const float t = h + l, lo = (h - t) + l;
  const unsigned tb = __float_as_uint(t);
  const unsigned w = (unsigned)s_oct[(tb >> 23) & 255u];
  const unsigned lead = __funnelshift_r(tb, 0u, w);                                // tb >> (w & 31)
  const float4 c = __ldg(reinterpret_cast<const float4*>(table) + ((int)lead + ((int)w >> 5)));
  const float u = (t - __uint_as_float(__funnelshift_l(0u, lead, w))) + lo;        // from the left end
  return fmaf(fmaf(fmaf(c.w, u, c.z), u, c.y), u, c.x);
}

// The direct evaluation of one entry, for pairs outside the table; out of
// line, so that the common path keeps its registers.
static __device__ __noinline__ double matern_direct64(const Loc& a, const Loc& b,
                                                      const MaternParams& mp) {
  Tally tl{0u, 0u, 0u, 0u, 0u, 0u, 0u};
  unsigned evals = 0;
  const FormF64 f{kExp2Tab, false, 0.0};
  return f.matern(a, b, mp, tl, evals);
}
static __device__ __noinline__ float matern_direct32(const Loc& a, const Loc& b,
                                                     const MaternParams& mp) {
  Tally tl{0u, 0u, 0u, 0u, 0u, 0u, 0u};
  unsigned evals = 0;
  const FormF32 f{kExp2Tab};
  return f.matern_out<float>(a, b, mp, tl, evals);
}

struct TabPoints64 {
  double2 c[kTabTile];   // columns' coordinates
  int2 oct[kTabOct];
};
template <bool F32, typename OutT>
struct TabTileSmem {
  std::conditional_t<F32, TabPoints32, TabPoints64> pts;
  OutT tile[kTabTile][kTabTile + 1];
};

// The transposed block (J, I) of a tile: columns cb .. cb + width - 1 of sm.tile as rows.
template <typename OutT, int WARPS>
__device__ __forceinline__ void tab_transpose(const OutT (*tile)[kTabTile + 1], int64_t r0, int64_t m,
                                              int64_t c0, int64_t n, int cb, int width,
                                              OutT* __restrict__ out, int64_t ld) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (r0 + kTabTile <= m && c0 + kTabTile <= n && width == kTabTile) {
    OutT* po = out + (c0 + lane) + (r0 + warp) * ld;
#pragma unroll
    for (int c = 0; c < kTabTile; c += WARPS, po += WARPS * ld) {
      po[0] = tile[warp + c][lane];
      po[32] = tile[warp + c][lane + 32];
    }
  } else if (width == kTabTile) {
    for (int c = warp; c < kTabTile; c += WARPS) {
      const int64_t j = r0 + c;  // column r0 + c of block (J, I): row c of the tile
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t i = c0 + lane + 32 * h;
        if (i < n && j < m) out[i + j * ld] = tile[c][lane + 32 * h];
      }
    }
  } else {
    for (int t = threadIdx.x; t < kTabTile * width; t += WARPS * 32) {
      const int c = t / width, i = cb + t % width;
      if (c0 + i < n && r0 + c < m) out[(c0 + i) + (r0 + c) * ld] = tile[c][i];
    }
  }
}

// One entry by the direct evaluation.
template <bool F32, typename OutT>
__device__ __forceinline__ OutT tab_direct(const double* __restrict__ locs1, int64_t m, int64_t i,
                                           const double* __restrict__ locs2, int64_t n, int64_t j,
                                           const MaternParams& mp) {
  Loc p, q;
  p.x = locs1[i];
  p.y = locs1[m + i];
  q.x = locs2[j];
  q.y = locs2[n + j];
  if constexpr (F32) {
    split_f(p.x, p.xh, p.xl);
    split_f(p.y, p.yh, p.yl);
    split_f(q.x, q.xh, q.xl);
    split_f(q.y, q.yh, q.yl);
    return matern_direct32(p, q, mp);
  } else {
    return to_out<OutT>(matern_direct64(p, q, mp));
  }
}

// One 64 x 64 tile (I, J) of M between locs1 (rows) and locs2 (columns) by a
// block of WARPS warps: lane i of warp w takes rows i and i + 32 of columns w,
// w + WARPS, ..., two rows at a time so that the loads of one entry overlap the
// arithmetic of the other.  kSym: the transposed block (J, I) is written too.
// use_table false: every entry by the direct evaluation.  part, width: the block
// takes columns part * width .. + width - 1 only (width 16 or 64), where whole
// tiles would leave SMs without a block.
template <bool F32, typename OutT, bool kSym, int WARPS>
__device__ __forceinline__ void tab_tile(TabTileSmem<F32, OutT>& sm, const unsigned char* __restrict__ table,
                                         unsigned e0, const double* __restrict__ locs1, int64_t m,
                                         const double* __restrict__ locs2, int64_t n, int64_t I,
                                         int64_t J, const MaternParams& mp, OutT* __restrict__ out,
                                         int64_t ld, int part = 0, int width = kTabTile,
                                         bool use_table = true) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = I * kTabTile, c0 = J * kTabTile;
  const bool in0 = r0 + lane < m, in1 = r0 + lane + 32 < m;
  const int cb = part * width, cw = cb + warp;  // the part's first column, the warp's
  const int cols = (int)(n - c0 < cb + width ? n - c0 : cb + width);
  OutT* const p0 = out + (r0 + lane) + (c0 + cw) * ld;
  if constexpr (F32) {
    use_table = use_table && tab_stage32<WARPS * 32>(sm.pts, locs1, m, locs2, n, r0, c0, mp, table);
    __syncthreads();
    const float4 a0 = sm.pts.p[lane], a1 = sm.pts.p[lane + 32];
    float nan = 0.0f;  // NaN once an entry lies outside the table
    if (use_table) {
      OutT* po = p0;
      auto column = [&](int c) {
        const float4 b = sm.pts.p[kTabTile + c];
        const float v0 = tab_entry32(table, sm.pts.oct, a0, b), v1 = tab_entry32(table, sm.pts.oct, a1, b);
        nan = fmaf(v1, 0.0f, fmaf(v0, 0.0f, nan));
        if (in0) po[0] = v0;
        if (in1) po[32] = v1;
        if constexpr (kSym) {
          sm.tile[lane][c] = v0;
          sm.tile[lane + 32][c] = v1;
        }
        po += WARPS * ld;
      };
      if (cols == kTabTile && width == kTabTile) {
#pragma unroll 4
        for (int c = 0; c < kTabTile; c += WARPS) column(warp + c);
      } else {
        for (int c = cw; c < cols; c += WARPS) column(c);
      }
    }
    if (!use_table || nan != nan) {  // coincident, very near or far pairs
      for (int k = 0; cw + (k >> 1) * WARPS < cols; ++k) {
        const int c = cw + (k >> 1) * WARPS, i = lane + 32 * (k & 1);
        OutT* const po = p0 + 32 * (k & 1) + (c - cw) * ld;
        if (r0 + i >= m) continue;
        if (use_table) {
          const float v = *po;
          if (v == v) continue;
        }
        const OutT v = tab_direct<true, OutT>(locs1, m, r0 + i, locs2, n, c0 + c, mp);
        *po = v;
        if constexpr (kSym) sm.tile[i][c] = v;
      }
    }
  } else {
    if (threadIdx.x < kTabTile) {
      const int64_t j = c0 + threadIdx.x;
      sm.pts.c[threadIdx.x] = j < n ? make_double2(locs2[j], locs2[n + j]) : make_double2(0.0, 0.0);
    }
    double ax[2], ay[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t i = r0 + lane + 32 * h;
      ax[h] = i < m ? locs1[i] : 0.0;
      ay[h] = i < m ? locs1[m + i] : 0.0;
    }
    __syncthreads();
    OutT* po = p0;
    unsigned bad = 0;  // entries outside the table: bits 2 k and 2 k + 1 of column cw + k WARPS
    int k = 0;
#pragma unroll 2
    for (int c = cw; c < (use_table ? cols : 0); c += WARPS, ++k) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const double2 b = sm.pts.c[c];
        const double dx = b.x - ax[h], dy = b.y - ay[h];
        double d;
        const bool ok = tab_entry64(table, sm.pts.oct, e0, fma(dx, dx, dy * dy), d);
        const OutT v = to_out<OutT>(d);
        bad |= (ok ? 0u : 1u) << (2 * k + h);
        if (h ? in1 : in0) po[32 * h] = v;
        if constexpr (kSym) sm.tile[lane + 32 * h][c] = v;
      }
      po += WARPS * ld;
    }
    if (!use_table)
      for (int c = cw; c < cols; c += WARPS, ++k) bad |= 3u << (2 * k);
    while (bad != 0) {  // coincident, very near or far pairs: written again by the direct evaluation
      const int b = __ffs((int)bad) - 1, c = cw + (b >> 1) * WARPS, i = lane + 32 * (b & 1);
      bad &= bad - 1;
      if (r0 + i >= m) continue;
      const OutT v = tab_direct<false, OutT>(locs1, m, r0 + i, locs2, n, c0 + c, mp);
      out[(r0 + i) + (c0 + c) * ld] = v;
      if constexpr (kSym) sm.tile[i][c] = v;
    }
  }
  if constexpr (kSym) {
    if (I != J) tab_transpose<OutT, WARPS>(sm.tile, r0, m, c0, n, cb, width, out, ld);
  }
}

}  // namespace bk
