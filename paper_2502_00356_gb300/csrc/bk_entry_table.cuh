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
// interval's number and the position inside it are bit fields of r^2.  FP64: m =
// 6 up to x = 0.7 (the series about s in powers of W/s <= 2^-6 past the branch
// point at s = 0), 7 up to x = 4 and from there growing with x so that x W/(2 s)
// <= 1/45, the ratio of the series of e^{-x}: degree 6, with u^7 economised,
// leaves 1e-17 of M, and the coefficients fit the record's fields (both checked
// with K's ratios for nu = 0.02 to 10).  FP32: one or two bits less and a cubic
// (an economised quartic; 1e-8 at worst, for nu = 0.02, else below 5e-9).
// Few and wide intervals mean few cache lines for a warp's record loads, which
// bound the writers.  Binades with x^2 from f 2^-18 to f 2^13, f in [1, 2) by beta
// (tab_scale), are covered: x from 2.0e-3 .. 2.8e-3 to 90 .. 128.  Entries outside
// take the direct evaluation, or are zero.
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
    if (F32) return q < 1 ? 5 : q < 4 ? 6 : q < 7 ? 7 : (q + 9) >> 1;
    return q < -1 ? 6 : q < 4 ? 7 : (q + 12) >> 1;
  }
  __host__ __device__ static constexpr int first(int o) {
    int b = 0;
    for (int i = 0; i < o; ++i) b += 1 << bits(i);
    return b;
  }
  static constexpr int kBins = first(kTabOct);
  // Tables end in two records without a value (NaN), for what lies outside them,
  // one of zero, for what underflows, and the words of tab_octave.
  static constexpr int kNaN = kBins, kZero = kBins + 2, kExtra = 3;
  static constexpr int kWords = F32 ? 256 : 128;
  static constexpr size_t kBytes = (size_t)(kBins + kExtra) * kRecord + kWords * sizeof(int);
  // In front of an FP64 table, for the entries beyond it: the plain form's
  // e^{-2 nu h} on kCoshTab's steps (n = 4,001, beta = 0.002, most entries between
  // x = 90 and 700: 980 us without it, 920 with; the per-entry writer 810).  Its
  // first entry is negative when it was not filled.
  static constexpr size_t kFront = F32 ? 0 : (size_t)kCoshTabSize * sizeof(double);
  static constexpr size_t kStride = (kFront + kBytes + 255) / 256 * 256;
};
using TabLayout64 = TabLayout<false>;
using TabLayout32 = TabLayout<true>;

// Scales of the fixed-point coefficients: c_k is held in units of 2^-S_k of
// the record's power of two 2^E, the value's upper bound.
//  FP64 record, two 16-byte parts in two arrays (side by side, a warp's loads
//  touched twice the cache lines, and those bound the writer):
//   words 0-1  c_0 (units 2^-62, its low 11 bits zero) + the exponent word,
//   words 2-3  c_1 (2^-68) with c_6 (2^-54) in its low 15 bits,
//   words 4-5  c_2 (2^-75) with c_5 (2^-54) in its low 22 bits,
//   words 6-7  c_3 (2^-51), c_4 (2^-54).
//  The bits that share a word with c_1 and c_2 are left in place; the bits above
//  them are chosen so that the whole word is nearest (within 2^-54 of the value).
// The top bit of c_0 stays free: the value may round up to 2^E itself.
//  An FP32 record is a cubic in four floats.
// An interval without a usable polynomial has a record whose value is NaN.
constexpr int kS0 = 62, kS1 = 68, kS2 = 75, kS3 = 51, kS4 = 54;
constexpr int kLow6 = 15, kLow5 = 22;  // bits of c_6, c_5
// c_0 and exponent word of a record whose value is NaN: 3/2 2^61 with the largest exponent.
constexpr unsigned kNaNLow = 2046u, kNaNHigh = 0x30000000u;
constexpr int kTabNodes = 485;                  // tau = -24 .. 6.25 in steps of 1/16

// Whether (sigma^2, beta, nu) are inside the tables' domain: orders for which
// the node grid holds the integral, and scales that keep every value, the FP32
// squared distances and coefficients included, a normal number.
constexpr double kTabMax32 = 0x1p50;  // the largest value of an FP32 record
__host__ __device__ inline bool tab_domain(bool f32, double sigma2, double beta, double nu) {
  return nu >= 0.02 && nu <= 10.0 && beta >= 1e-8 && beta <= 1e8 && sigma2 >= 1e-20 &&
         sigma2 <= (f32 ? kTabMax32 : 1e20);
}

// One instance of a batch: its descriptor, checked, and its constants.
struct BatchInstance {
  const double* locs;
  void* out;
  int64_t n, ld;
  int64_t table;  // whether its entries come from a table
  MaternParams mp;
};

// 1/beta^2 = f 2^{2 h + odd} with f in [1, 2) (to 2^-19 at the ends, by the leading
// bits of 1/beta); 2^h scales coordinates.
struct TabScale {
  int h, odd;
};
__device__ __forceinline__ TabScale tab_scale(double inv_beta) {
  const int hi = __double2hiint(inv_beta);
  return TabScale{((hi >> 20) & 0x7ff) - 1023, (hi & 0xfffff) >= 0x6a09f};  // sqrt 2
}

// The biased exponent of the first binade of r^2: q = its exponent + 2 h + odd.
__device__ __forceinline__ unsigned tab_first_binade(double inv_beta) {
  const TabScale sc = tab_scale(inv_beta);
  return (unsigned)(kTabQ0 - 2 * sc.h - sc.odd + 1023);
}

// Shift and first interval of a binade of r^2 as one word, 32 (first interval less
// the binade's leading bits) + shift.  FP32: k is the exponent field of the
// scaled square, whose bits the word shifts; FP64: k = q + 64, for a square
// normalised to bit 31.  Outside the table a shift of 31 leads to the two records
// without a value (the bits left are 0 or 1), or where M underflows (below 2^-160, 2^-1080) to that of zero.
template <bool F32>
__device__ __forceinline__ int tab_octave(int k, const MaternParams& mp) {
  using L = TabLayout<F32>;
  const int q = F32 ? k - 127 + tab_scale(mp.inv_beta).odd : k - 64, o = q - kTabQ0;
  int first = L::kNaN, sh = 31;
#pragma unroll
  for (int i = 0; i < kTabOct; ++i) {
    if (i == o) {
      sh = (F32 ? 23 : 31) - L::bits(i);
      first = L::first(i) - ((F32 ? k : 1) << L::bits(i));
    }
  }
  if (o >= kTabOct && (!F32 || k < 255)) {
    // log M <= log c + (nu - 1/2) log x - x + (4 nu^2 - 1)/(8 x) + 0.23
    const float x = exp2f(0.5f * (float)q), nu = f32_trunc(mp.nu);
    const float m = f32_trunc(mp.log_pref) + fmaxf(nu - 0.5f, 0.0f) * 0.34657359f * (float)q - x + 1.5f;
    if (m < (F32 ? -111.0f : -749.0f)) first = L::kZero - (F32 ? 0 : 1);  // (the shifted bits are 1)
  }
  return (int)((unsigned)first << 5) | sh;
}

// ---------------------------------------------------------------------------
// Building a table.  A block of 1,024 threads first evaluates the node weights
// (all tau of the grid, for this nu) into shared memory; then eight lanes per
// interval sum F_nu and F_{nu-1} at its expansion point over the nodes that matter
// there (about 25 to 100, the most near x = 0), and one thread each writes the
// records.  The FP64 pipe bounds it (an operation of one warp takes 17 cycles of
// the SM), so the exponentials run on the integer pipe (exp2s_int), every SM takes
// part, a block's intervals grid-strided so that each gets the same share of
// costly ones, warps without an interval do nothing, one thread computes 1/beta^2
// for all, and a sum over lanes costs one addition a step for both values (n = 777:
// 28.9 us with 1/beta^2 in every thread and two additions, 26.6 so).  Small matrices leave most
// intervals out (r2_max): then latency bounds it, and 16 or 32 lanes share one
// (n = 777: eight took 21,000 cycles for the sums).
constexpr int kTabThreads = 1024;
constexpr int kTabGroups = kTabThreads / 8;  // at most
struct TabBuildSmem {
  double v[kTabNodes], w[kTabNodes], w2[kTabNodes];
  double f0[kTabGroups], f1[kTabGroups];
  double b2, b2lo;  // 1/beta^2
  float box[kTabThreads / 64][4];
};

// c 2^scale for c >= 0, rounded to nearest, on the integer pipe.
__device__ __forceinline__ unsigned long long tab_fix(double c, int scale) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(c);
  const int sh = (int)(b >> 52) - 1075 + scale;
  const unsigned long long sig = (b & 0xfffffffffffffULL) | 0x10000000000000ULL;
  if (sh >= 0) return sig << sh;
  return sh < -54 ? 0ULL : (sig + (1ULL << (-sh - 1))) >> -sh;
}

// j/16 for |j| < 2^19, without a conversion.
__device__ __forceinline__ double tab_tau(int j) {
  return __hiloint2double(0x42f80000, j + (1 << 30)) - __hiloint2double(0x42f80000, 1 << 30);  // 1.5 2^48 + j/16
}

// Node weights for the order nu, log c = log(sigma^2 2^{1-nu}/Gamma(nu)) in
// them: w = (1/16)/2 c e^{nu tau - e^tau/2}, w2 = w e^{-tau}, and v =
// -e^{-tau}/2 in the units of exp2s_int (times 4096/ln 2).
__device__ __forceinline__ void tab_nodes(TabBuildSmem& sm, double nu, double log_c) {
  if (const int i = threadIdx.x; i < kTabNodes) {
    const int j = i - kTauMax;  // tau = j/16
    const double ep = kTauTab[j + kTauMax], en = kTauTab[kTauMax - j];
    const double a = fma(nu, tab_tau(j), fma(-0.5, ep, log_c));
    const double w = 0.03125 * exp_units_full(a * kExpScale, kExp2Tab);
    sm.v[i] = (-0.5 * kExpScale) * en;
    sm.w[i] = w;
    sm.w2[i] = w * en;
  }
}

// The interval's binade o, log2 m of the binade's intervals, and the expansion
// point: its right end, for FP32 records its left end.
template <bool F32>
__device__ __forceinline__ void tab_interval(int bin, unsigned e0, int& o, int& m, double& s_ref) {
  using L = TabLayout<F32>;
  constexpr int kFlat = -kTabQ0 - 2, kFlatBits = L::bits(0);  // binades below x = 1/2 are cut alike
  static_assert(L::first(kFlat + 1) == (kFlat + 1) << kFlatBits, "up to kFlat");
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
                                           ((unsigned long long)(F32 ? i : i + 1) << (52 - m))));
}

// An upper bound of every squared distance between two sets of locations, from
// their common bounding box (FP32, rounded outwards); infinite when a
// coordinate is not finite.  The block's upper half of the threads scans the
// locations (the lower half is at the node weights) ...
constexpr int kTabScanThreads = kTabThreads / 2;
__device__ __forceinline__ void tab_scan(float (*s_box)[4], const double* __restrict__ locs1, int64_t m,
                                         const double* __restrict__ locs2, int64_t n) {
  float lo[2] = {kInfF, kInfF}, hi[2] = {-kInfF, -kInfF};
  for (int set = 0; set < 2; ++set) {
    const double* const l = set ? locs2 : locs1;
    const int64_t len = set ? n : m;
    if (set && locs2 == locs1 && n == m) break;
#pragma unroll 4
    for (int64_t i = threadIdx.x % kTabScanThreads; i < len; i += kTabScanThreads) {
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
    float* const b = s_box[threadIdx.x % kTabScanThreads >> 5];
    b[0] = lo[0];
    b[1] = lo[1];
    b[2] = hi[0];
    b[3] = hi[1];
  }
}
// ... and after a barrier every thread reads the bound.
__device__ __forceinline__ double tab_r2_bound(const float (*s_box)[4]) {
  const float* const b = s_box[threadIdx.x % (kTabScanThreads / 32)];
  float r2 = 0.0f;
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    float lo = b[d], hi = b[2 + d];
#pragma unroll
    for (int o = kTabScanThreads / 64; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    // truncation took at most 2^-23 of a coordinate's magnitude from each end
    const float e = (hi - lo) + 0x1p-21f * (fabsf(hi) + fabsf(lo)) + 1e-30f;
    r2 = fmaf(e, e, r2);
  }
  return widen_f(r2 * 1.001f);
}

// Writes the record of one interval from F_nu and F_{nu-1} at its expansion
// point.
template <bool F32>
__device__ __forceinline__ void tab_record(int bin, double nu, unsigned e0, double ib, double b2,
                                           double b2lo, double f0, double f1,
                                           unsigned char* __restrict__ table) {
  using L = TabLayout<F32>;
  int o, m;
  double s_ref;
  tab_interval<F32>(bin, e0, o, m, s_ref);
  const double s = fma(s_ref, b2, s_ref * b2lo);
  // c_k = q^k/k! s^k F_{nu-k}, q = W/(2 s) in units of r^2: c_0 = F_nu, c_1 = q s F_{nu-1},
  // c_{k+1} = s q^2/(k (k+1)) c_{k-1} - 2 (nu - k) q/(k+1) c_k
  const double q = __longlong_as_double((long long)(e0 + o - m - 1) << 52) * rcp_nr2(s_ref);
  constexpr int kDeg = F32 ? 4 : 7;
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
    const bool ok = f >= 0.0f && f <= (float)kTabMax32;  // (subnormal values keep their absolute accuracy)
    reinterpret_cast<float4*>(table)[bin] = make_float4(ok ? f : __int_as_float(0x7fc00000), (float)(a1 * iw),
                                                        (float)(a2 * (iw * iw)), (float)(a3 * (iw * iw * iw)));
  } else {
    // u^7 replaced by its best approximation of degree 6 on [0, 1] (off by 2^-13)
    constexpr double kU7[7] = {1.0 / 8192, -98.0 / 8192, 1568.0 / 8192, -9408.0 / 8192, 26880.0 / 8192, -39424.0 / 8192, 28672.0 / 8192};
#pragma unroll
    for (int k = 0; k < 7; ++k) c[k] = fmax(fma(kU7[k], c[7], c[k]), 0.0);
    // t_k = c_k + c_{k+1} + ...; t_0 is the value at the left end, the largest of the interval
    double t[7];
    t[6] = c[6];
#pragma unroll
    for (int k = 5; k >= 0; --k) t[k] = t[k + 1] + c[k];
    const int ev = (int)((unsigned)__double2hiint(t[0]) >> 20);  // 2048 and above: negative
    const int E = ev - 1022;                                     // t_0 in [2^{E-1}, 2^E)
    // the bounds that the scales were chosen for (t_k < 2^{E-b}); NaN fails them
    auto below = [&](int k, int b) { return (int)((unsigned)__double2hiint(t[k]) >> 20) < ev + 1 - b; };
    const bool ok = ev > 60 && ev < 1980 && below(1, 5) && below(2, 12) && below(3, 19) && below(4, 22) &&
                    below(5, 32) && below(6, 39);
    // c, its low bits replaced by low, to nearest
    auto share = [](unsigned long long c, unsigned long long low, int bits) {
      const unsigned long long half = 1ULL << (bits - 1);
      return (c + half > low ? (c + half - low) >> bits << bits : 0ULL) | low;
    };
    // the exponent word: the exponent field of 2^{E-1} less the leading bit that
    // the significand adds
    const unsigned long long c0 = ok ? (tab_fix(c[0], kS0 - 11 - E) << 11) | (unsigned)(E + 1021)
                                     : ((unsigned long long)kNaNHigh << 32) | kNaNLow;
    const unsigned long long c1 = share(tab_fix(c[1], kS1 - E), tab_fix(c[6], kS4 - E), kLow6);
    const unsigned long long c2 = share(tab_fix(c[2], kS2 - E), tab_fix(c[5], kS4 - E), kLow5);
    uint4* const rec = reinterpret_cast<uint4*>(table) + bin;
    rec[0] = make_uint4((unsigned)c0, (unsigned)(c0 >> 32), ok ? (unsigned)c1 : 0u, ok ? (unsigned)(c1 >> 32) : 0u);
    rec[L::kBins + L::kExtra] = ok ? make_uint4((unsigned)c2, (unsigned)(c2 >> 32), (unsigned)tab_fix(c[3], kS3 - E),
                             (unsigned)tab_fix(c[4], kS4 - E))
                : make_uint4(0u, 0u, 0u, 0u);
  }
}

// Block `block` of `blocks`: its share of the table.  scan: the locations bound
// the distances, and binades beyond the bound are left out.
template <bool F32>
__device__ __forceinline__ void tab_build_block(TabBuildSmem& sm, const MaternParams& mp, int block,
                                                int blocks, bool scan, const double* __restrict__ locs1,
                                                int64_t m_locs, const double* __restrict__ locs2,
                                                int64_t n_locs, unsigned char* __restrict__ table) {
  using L = TabLayout<F32>;
  static_assert(kTabNodes <= kTabThreads - kTabScanThreads, "nodes and scan side by side");
  if (threadIdx.x < kTabThreads - kTabScanThreads) tab_nodes(sm, mp.nu, mp.log_pref);
  else if (scan) tab_scan(sm.box, locs1, m_locs, locs2, n_locs);
  if (threadIdx.x == kTabThreads - 1) {
    // x^2 = s_ref/beta^2, with the rounding of 1/beta and of its square taken back
    const double ib = mp.inv_beta, b2 = ib * ib;
    sm.b2 = b2;
    sm.b2lo = fma(ib, ib, -b2) + 2.0 * ib * (fma(-ib, mp.beta, 1.0) * ib);
  }
  __syncthreads();
  const double r2_max = scan ? tab_r2_bound(sm.box) : kInf;
  const unsigned e0 = tab_first_binade(mp.inv_beta);
  const double ib = mp.inv_beta, b2 = sm.b2, b2lo = sm.b2lo;
  const float nuf = f32_trunc(mp.nu);
  if (block == blocks - 1) {
    if (threadIdx.x < L::kExtra) {
      uint4* const rec = reinterpret_cast<uint4*>(table) + L::kBins + threadIdx.x;
      if constexpr (F32) {
        *rec = make_uint4(threadIdx.x < 2 ? 0x7fc00000u : 0u, 0u, 0u, 0u);
      } else {
        rec[0] = threadIdx.x < 2 ? make_uint4(kNaNLow, kNaNHigh, 0u, 0u) : make_uint4(1u, 0u, 0u, 0u);
        rec[L::kBins + L::kExtra] = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    if (threadIdx.x < L::kWords)
      reinterpret_cast<int*>(table + (size_t)(L::kBins + L::kExtra) * L::kRecord)[threadIdx.x] =
          tab_octave<F32>((int)threadIdx.x, mp);
  }
  // the intervals of binades up to r2_max's
  const int o_top = (int)((unsigned)__double2hiint(r2_max) >> 20) - (int)e0, o_max = min(o_top, kTabOct - 1);
  if constexpr (!F32) {
    double* const front = reinterpret_cast<double*>(table - L::kFront);
    if (o_top >= kTabOct) {  // distances beyond the table
      for (int i = block + blocks * (int)threadIdx.x; i < kCoshTabSize; i += blocks * kTabThreads)
        front[i] = decay_entry(mp.nu, i, kExp2Tab);
    } else if (block == 0 && threadIdx.x == 0) {
      front[0] = -1.0;
    }
  }
  int bins = 0;
#pragma unroll
  for (int o = 0; o < kTabOct; ++o)
    if (o <= o_max) bins = L::first(o + 1);
  const int lanes = bins <= blocks * (kTabThreads / 32) ? 32 : bins <= blocks * (kTabThreads / 16) ? 16 : 8;
  const int groups = kTabThreads / lanes;
  for (int k0 = 0; k0 * blocks + block < bins; k0 += groups) {
    if (k0 > 0) __syncthreads();  // the previous round's sums have been read
    const int k = (int)threadIdx.x / lanes, lane = (int)threadIdx.x & (lanes - 1), bin = (k0 + k) * blocks + block;
    if (bin < bins) {
      double f0 = 0.0, f1 = 0.0;
      int o, m;
      double s_ref;
      tab_interval<F32>(bin, e0, o, m, s_ref);
      const double s = fma(s_ref, b2, s_ref * b2lo);
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
      const int step = F32 ? (q <= 4 && nuf <= 5.0f ? 4 : q <= 6 ? 3 : q <= 8 ? 2 : 1)
                           : (q <= 4 && nuf <= 2.5f ? 3 : q <= 8 ? 2 : 1);
      const int j0 = max((int)floorf(16.0f * fmaxf(lx - tl, -kCut / nuf - 6.0f)), -kTauMax);
      const int j1 = min((int)ceilf(16.0f * (lx + tr)), kTabNodes - 1 - kTauMax);
#pragma unroll 2
      for (int j = j0 + step * lane; j <= j1; j += step * lanes) {
        const double u = s * sm.v[j + kTauMax];
        if ((unsigned)__double2hiint(u) < 0xc14fe000u) {  // u > -4.18e6: the term's factor above e^-707
          const double e = exp2s_int(u, kExp2Tab);
          f0 = fma(sm.w[j + kTauMax], e, f0);
          f1 = fma(sm.w2[j + kTauMax], e, f1);
        }
      }
      const unsigned mask = lanes == 32 ? 0xffffffffu : ((1u << lanes) - 1u) << (threadIdx.x & 31 & -lanes);
      // half of the lanes go on with F_nu, half with F_{nu-1}
      const int half = lanes >> 1;
      const bool second = (lane & half) != 0;
      double f = second ? f1 : f0;
      f += __shfl_xor_sync(mask, second ? f0 : f1, half);
      for (int d = 1; d < half; d <<= 1) f += __shfl_xor_sync(mask, f, d);
      if ((lane & (half - 1)) == 0) {
        const double h = step == 1 ? 1.0 : step == 2 ? 2.0 : step == 3 ? 3.0 : 4.0;
        (second ? sm.f1 : sm.f0)[k] = h * f;
      }
    }
    __syncthreads();
    const int rec = (k0 + (int)threadIdx.x) * blocks + block;
    if ((int)threadIdx.x < groups && rec < bins)
      tab_record<F32>(rec, mp.nu, e0, ib, b2, b2lo, sm.f0[threadIdx.x], sm.f1[threadIdx.x], table);
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

// Coordinates.  A tile's coordinates are held relative to its first row's point.
// With 2^e above every difference between a row and a column:
//  FP64 entries: integers in units of 2^{e-61} (exact but for that rounding), as
//   two words, x = x_1 2^30 + x_2 with |x_2| <= 2^29, so that a difference is two
//   subtractions without a carry and r^2, in units of 2^{2 e - 62} and 29 bits
//   below, six multiply-adds: sum x_1^2 + 2^-29 (sum x_1 x_2 + 2^-31 sum x_2^2).
//   The FP64 pipe, whose four operations bounded the writer before (64 cycles of
//   an SM for 32 entries), is left alone.
//  FP32 entries: two floats in units of 2^h of 1/beta, a multiple of Q = 2^{e-10}
//   and the rest to Q 2^-25.  Differences of the first parts and sums of their
//   squares are exact; what the second parts add is rounded to 2^{e-33} of r.
// In x, then, r is off by at most X 2^-60 (X 2^-32) with X = 2^e/beta, and M by that
// times |d log M/dx|, at most 1 for nu >= 1/2 and 1 + 1/x below: binades for
// which that passes 2^-51 (2^-26) are left to the direct evaluation.
template <bool F32>
struct TabPoints {
  static constexpr int kOct = F32 ? 256 : 64;
  std::conditional_t<F32, float4, int4> p[2 * kTabTile];  // rows, then columns: {x_1, x_2, y_1, y_2}
  int oct[kOct];  // words by FP32 exponent field, or by leading zeros of r^2's upper word
  unsigned extent[4];
};

// (a b >> 32) + c
__device__ __forceinline__ int mad_hi(int a, int b, int c) {
  int r;
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

// v 2^s modulo 2^64, rounded.
__device__ __forceinline__ long long fix_mod(double v, int s) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int ex = (int)(b >> 52) & 0x7ff, sh = ex - 1075 + s;
  const unsigned long long sig = ex ? (b & 0xfffffffffffffULL) | 0x10000000000000ULL : 0ULL;
  unsigned long long r = 0;
  if (sh >= 0) r = sh < 64 ? sig << sh : 0ULL;
  else if (sh > -56) r = (sig + (1ULL << (-sh - 1))) >> -sh;
  return (long long)b < 0 ? -(long long)r : (long long)r;
}

// Loads of a table by kernels that are launched while an earlier grid may still
// write it, which they wait for first: plain loads, as the read-only path (ld.global.nc)
// is for memory that nothing writes while the kernel lives.  A record's address comes
// from a word, a word's load is volatile: neither moves ahead of the wait.
__device__ __forceinline__ uint4 load_record(const uint4* p) {
  uint4 v;
  asm("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 load_record(const float4* p) {
  float4 v;
  asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ int load_word(const int* p) {
  int v;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Stages a tile's points and words; every thread of the block calls it (the caller
// synchronises before, when sm was read, and after).  False: the tile spans
// more than any table could use, or is not finite.
template <bool F32, int THREADS>
__device__ __forceinline__ bool tab_stage(TabPoints<F32>& sm, const double* __restrict__ locs1, int64_t m,
                                          const double* __restrict__ locs2, int64_t n, int64_t r0,
                                          int64_t c0, const MaternParams& mp,
                                          const unsigned char* table) {
  static_assert(THREADS >= 2 * kTabTile, "one thread per point");
  using L = TabLayout<F32>;
  const int tid = threadIdx.x, lane = tid & 31;
  double x = 0.0, y = 0.0, px = 0.0, py = 0.0, wx = 0.0, wy = 0.0;
  if (tid < 2 * kTabTile) {
    const bool row = tid < kTabTile;
    const double* const l = row ? locs1 : locs2;
    const int64_t len = row ? m : n, i = row ? r0 + tid : c0 + (tid - kTabTile);
    px = locs1[r0];
    py = locs1[m + r0];
    x = i < len ? l[i] : px;
    y = i < len ? l[len + i] : py;
    wx = x - px;
    wy = y - py;
    const unsigned a = max((unsigned)__double2hiint(wx) & 0x7fffffffu, (unsigned)__double2hiint(wy) & 0x7fffffffu);
    const unsigned warp_max = __reduce_max_sync(0xffffffffu, a);
    if (lane == 0) sm.extent[tid >> 5] = warp_max;
  }
  __syncthreads();
  // 2^e above the sum of the rows' and the columns' largest coordinate
  const unsigned hr = max(sm.extent[0], sm.extent[1]), hc = max(sm.extent[2], sm.extent[3]);
  const unsigned a = max(hr, hc), b = min(hr, hc);
  const unsigned sum = ((a & 0xfffffu) | 0x100000u) + (((b & 0xfffffu) | 0x100000u) >> min((a >> 20) - (b >> 20), 31u)) + 3u;
  const TabScale sc = tab_scale(mp.inv_beta);
  const int es = max((int)(a >> 20) - 1022 + (sum >> 21 ? 1 : 0) + sc.h, -40);  // scaled: 2^es
  const int* const words = reinterpret_cast<const int*>(table + (size_t)(L::kBins + L::kExtra) * L::kRecord);
  constexpr int kNone = (L::kNaN << 5) | 31;
  const int q_min = es > (F32 ? 6 : 9) ? kTabQ0 + kTabOct : mp.nu >= 0.5 ? kTabQ0 : 2 * es - (F32 ? 12 : 18);
  if constexpr (F32) {
    const int ex_min = q_min + 127 - sc.odd;
#pragma unroll
    for (int k = tid; k < TabPoints<F32>::kOct; k += THREADS) sm.oct[k] = k < ex_min ? kNone : load_word(words + k);
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
  } else {
    if (tid < TabPoints<F32>::kOct) {
      const int q = 1 - tid + 2 * es + sc.odd;  // tid leading zeros
      sm.oct[tid] = tid == 0 || tid >= 32 || q < q_min ? kNone : load_word(words + min(max(q + 64, 0), L::kWords - 1));
    }
    if (tid < 2 * kTabTile) {
      const int s = 61 - (es - sc.h);
      auto split = [&](double v, double p, int& i1, int& i2) {
        const long long k = fix_mod(v, s) - fix_mod(p, s);
        i1 = (int)((k + (1 << 29)) >> 30);
        i2 = (int)(k - ((long long)i1 << 30));
      };
      int4 p;
      split(x, px, p.x, p.y);
      split(y, py, p.z, p.w);
      sm.p[tid] = p;
    }
  }
  return es <= 20;
}

// M between the points a and b; NaN when they lie outside the table.  FP64: about
// 95 instructions, 16 of them wide products of 8 cycles a warp and scheduler; with
// the FP64 pipe's distance n = 20,000 took 1,616 us, now 1,040 (bytes: 480).
__device__ __forceinline__ double tab_entry(const unsigned char* table, const int* s_oct,
                                            const int4& p, const int4& q) {
  const int dx = q.x - p.x, lx = q.y - p.y, dy = q.z - p.z, ly = q.w - p.w;
  const long long mid = mad_wide(2, mad_hi(ly, ly, mad_hi(lx, lx, 0)), mad_wide(dy, ly, mad_wide(dx, lx, 0LL)));
  const unsigned long long r2 = (unsigned long long)(mad_wide(dy, dy, mad_wide(dx, dx, 0LL)) + (mid >> 29));
  // the leading bit to bit 63; the position below the interval's right end, 64 fraction bits
  const unsigned rl = (unsigned)r2, rh = (unsigned)(r2 >> 32);
  const int lz = __clz((int)rh);
  const unsigned h = __funnelshift_l(rl, rh, lz), l = __funnelshift_l((unsigned)mid << 3, rl, lz);
  const unsigned w = (unsigned)s_oct[lz];
  using L = TabLayout64;
  const uint4* const rec = reinterpret_cast<const uint4*>(table) + ((int)__funnelshift_r(h, 0u, w) + ((int)w >> 5));
  const uint4 a = load_record(rec), b = load_record(rec + (L::kBins + L::kExtra));
  const unsigned u32 = __funnelshift_r(~l, ~h, w);
  const unsigned long long u = (((unsigned long long)u32 << 32) | __funnelshift_r(0u, ~l, w)) >> 1;
  unsigned A = (b.x & ((1u << kLow5) - 1u)) + __umulhi(a.z & ((1u << kLow6) - 1u), u32);
  A = b.w + __umulhi(A, u32);
  A = b.z + (__umulhi(A, u32) >> (kS4 - kS3));
  const unsigned long long A2 =
      (((unsigned long long)b.y << 32) | b.x) + (((unsigned long long)A * u32) >> (kS3 + 32 - kS2));
  const unsigned long long A1 = (((unsigned long long)a.w << 32) | a.z) + (mulhi63(A2, u) >> (kS2 - kS1 - 1));
  unsigned long long F =
      (((unsigned long long)a.y << 32) | (a.x & ~0x7ffu)) + (mulhi63(A1, u) >> (kS1 - kS0 - 1));
  // F 2^{E-62}, F in [2^60, 2^62]
  unsigned ew = a.x & 0x7ffu;
  if ((unsigned)(F >> 32) < 0x20000000u) {
    F <<= 1;
    --ew;
  }
  F = (F + 256ULL) >> 9;
  return __hiloint2double((int)((unsigned)(F >> 32) + (ew << 20)), (int)(unsigned)F);
}

// The same in FP32: about 35 instructions, most of them on the FP32 pipe (with
// double-float differences of global coordinates and a fixed-point Horner
// scheme it was 125, 60 of them on the integer pipe: n = 40,000 took 3.60 ms,
// now 1.67).  The record loads bound it: a warp's 32 distances touch about
// nine cache lines.  A matrix's rms error is 2.6e-8, against 2.5e-8 of rounding alone.
__device__ __forceinline__ float tab_entry(const unsigned char* table, const int* s_oct,
                                           const float4& a, const float4& b) {
  const float dx = b.x - a.x, lx = b.y - a.y, dy = b.z - a.z, ly = b.w - a.w;
  const float h = fmaf(dx, dx, dy * dy);                                           // exact
  const float l = fmaf(ly, fmaf(2.0f, dy, ly), lx * fmaf(2.0f, dx, lx));
  const float t = h + l, lo = (h - t) + l;
  const unsigned tb = __float_as_uint(t);
  const unsigned w = (unsigned)s_oct[(tb >> 23) & 255u];
  const unsigned lead = __funnelshift_r(tb, 0u, w);                                // tb >> (w & 31)
  const float4 c = load_record(reinterpret_cast<const float4*>(table) + ((int)lead + ((int)w >> 5)));
  const float u = (t - __uint_as_float(__funnelshift_l(0u, lead, w))) + lo;        // from the left end
  // at least 0: where a record's coefficients are subnormal numbers the cubic may
  // end a few of their units below (a NaN stays)
  float v;
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(v) : "f"(fmaf(fmaf(fmaf(c.w, u, c.z), u, c.y), u, c.x)));
  return v;
}

// Keeps a NaN among the values it has seen.
struct NanSeen {
  float f = 0.0f;
  int hi = 0;
  __device__ __forceinline__ void see(float v) { f = fmaf(v, 0.0f, f); }
  __device__ __forceinline__ void see(double v) { hi = max(hi, __double2hiint(v)); }
  __device__ __forceinline__ bool any() const { return f != f || hi >= 0x7ff00000; }
};

// The direct evaluation of one entry, for pairs outside the table; out of
// line, so that the common path keeps its registers.
static __device__ __noinline__ double matern_direct64(double px, double py, double qx, double qy,
                                                      const MaternParams& mp, const double* decay) {
  Tally tl{0u, 0u, 0u, 0u, 0u, 0u, 0u};
  unsigned evals = 0;
  const FormF64 f{kExp2Tab, false, 0.0, decay};
  Loc a, b;
  a.x = px;
  a.y = py;
  b.x = qx;
  b.y = qy;
  return f.matern(a, b, mp, tl, evals);
}
static __device__ __noinline__ float matern_direct32(const Loc& a, const Loc& b,
                                                     const MaternParams& mp) {
  Tally tl{0u, 0u, 0u, 0u, 0u, 0u, 0u};
  unsigned evals = 0;
  const FormF32 f{kExp2Tab};
  return f.matern_out<float>(a, b, mp, tl, evals);
}

template <bool F32, typename OutT>
struct TabTileSmem {
  TabPoints<F32> pts;
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

// log M at most, for x >= 1: log c + (nu - 1/2) log x - x + (4 nu^2 - 1)/(8 x) + 0.23.
__device__ __forceinline__ float tab_log_bound(float x, const MaternParams& mp) {
  return fmaf(fmaxf(f32_trunc(mp.nu) - 0.5f, 0.0f), __logf(x), f32_trunc(mp.log_pref)) - x + 1.5f;
}

// One entry by the direct evaluation, 0 where it underflows (below 2^-1080, 2^-152).
template <bool F32, typename OutT>
__device__ __forceinline__ OutT tab_direct(const double* __restrict__ locs1, int64_t m, int64_t i,
                                           const double* __restrict__ locs2, int64_t n, int64_t j,
                                           const MaternParams& mp, const double* decay) {
  const double px = locs1[i], py = locs1[m + i], qx = locs2[j], qy = locs2[n + j];
  const double wx = qx - px, wy = qy - py;
  if (wx == 0.0 && wy == 0.0) return (OutT)mp.sigma2;  // the diagonal, without a call
  const float dx = f32_trunc(wx), dy = f32_trunc(wy), x = sqrtf(fmaf(dx, dx, dy * dy)) * mp.inv_beta_f;
  if (x > 64.0f && x < 1e6f && tab_log_bound(x, mp) < (sizeof(OutT) == 4 ? -106.0f : -749.0f)) return (OutT)0;
  if constexpr (F32) {
    Loc p, q;
    split_f(px, p.xh, p.xl);
    split_f(py, p.yh, p.yl);
    split_f(qx, q.xh, q.xl);
    split_f(qy, q.yh, q.yl);
    return matern_direct32(p, q, mp);
  } else {
    return to_out<OutT>(matern_direct64(px, py, qx, qy, mp, *decay > 0.0 ? decay : nullptr));
  }
}

// One 64 x 64 tile (I, J) of M between locs1 (rows) and locs2 (columns) by a
// block of WARPS warps: lane i of warp w takes rows i and i + 32 of columns w,
// w + WARPS, ..., two rows at a time so that the loads of one entry overlap the
// arithmetic of the other.  kSym: the transposed block (J, I) is written too.
// part, width: the block takes columns part * width .. + width - 1 only (width 16, 32 or 64: tile_width),
// where whole tiles would leave SMs without a block.
template <bool F32, typename OutT, bool kSym, int WARPS>
__device__ __forceinline__ void tab_tile(TabTileSmem<F32, OutT>& sm, const unsigned char* table,
                                         const double* __restrict__ locs1, int64_t m,
                                         const double* __restrict__ locs2, int64_t n, int64_t I,
                                         int64_t J, const MaternParams& mp, OutT* __restrict__ out,
                                         int64_t ld, int part = 0, int width = kTabTile) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = I * kTabTile, c0 = J * kTabTile;
  const bool in0 = r0 + lane < m, in1 = r0 + lane + 32 < m;
  const int cb = part * width, cw = cb + warp;  // the part's first column, the warp's
  const int cols = (int)(n - c0 < cb + width ? n - c0 : cb + width);
  OutT* const p0 = out + (r0 + lane) + (c0 + cw) * ld;
  const bool use_table = tab_stage<F32, WARPS * 32>(sm.pts, locs1, m, locs2, n, r0, c0, mp, table);
  __syncthreads();
  const auto a0 = sm.pts.p[lane], a1 = sm.pts.p[lane + 32];
  NanSeen nan;
  if (use_table) {
    OutT* po = p0;
    auto column = [&](int c) {
      const auto b = sm.pts.p[kTabTile + c];
      const auto v0 = tab_entry(table, sm.pts.oct, a0, b), v1 = tab_entry(table, sm.pts.oct, a1, b);
      nan.see(v0);
      nan.see(v1);
      const OutT w0 = (OutT)v0, w1 = (OutT)v1;
      if (in0) po[0] = w0;
      if (in1) po[32] = w1;
      if constexpr (kSym) {
        sm.tile[lane][c] = w0;
        sm.tile[lane + 32][c] = w1;
      }
      po += WARPS * ld;
    };
    if (cols == kTabTile && width == kTabTile) {
#pragma unroll (F32 ? 4 : kSym ? 2 : 4)  // (20,000 x 2,003: 211.5 us with 2, 209 with 4)
      for (int c = 0; c < kTabTile; c += WARPS) column(warp + c);
    } else {
      for (int c = cw; c < cols; c += WARPS) column(c);
    }
  }
  if (!use_table || nan.any()) {  // coincident, very near or far pairs: written again by the direct evaluation
    for (int k = 0; cw + (k >> 1) * WARPS < cols; ++k) {
      const int c = cw + (k >> 1) * WARPS, i = lane + 32 * (k & 1);
      OutT* const po = p0 + 32 * (k & 1) + (c - cw) * ld;
      if (r0 + i >= m) continue;
      if (use_table) {
        OutT v;
        if constexpr (kSym) v = sm.tile[i][c];  // (the matrix may be host memory)
        else v = *po;
        if (v == v) continue;
      }
      const OutT v = tab_direct<F32, OutT>(locs1, m, r0 + i, locs2, n, c0 + c, mp,
                                           reinterpret_cast<const double*>(table - TabLayout<F32>::kFront));
      *po = v;
      if constexpr (kSym) sm.tile[i][c] = v;
    }
  }
  if constexpr (kSym) {
    if (I != J) tab_transpose<OutT, WARPS>(sm.tile, r0, m, c0, n, cb, width, out, ld);
  }
}

}  // namespace bk
