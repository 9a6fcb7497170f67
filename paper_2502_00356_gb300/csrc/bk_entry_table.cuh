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
// width W, and nothing cancels.  F_nu and F_{nu-1} come from the sums, the
// rest from K's recurrence in the order, s F_{mu-1} = F_{mu+1} - 2 mu F_mu.
//
// The intervals.  Every binade of r^2 is cut into 2^m equal parts, so that an
// interval's number and the position inside it are bit fields of r^2.  m = 7
// up to x = 2 (the series about s in powers of W/s <= 2^-7 past the branch
// point at s = 0), 8 and 9 up to x = 8 and from there growing with x so that
// x W/(2 s) <= 1/64, the ratio of the series of e^{-x}: degree 6 then leaves
// less than 4e-16 of M (checked in the orders' ratio K_{nu-7}/K_nu too).  The
// FP32 records take one to four bits less and degree 3 (an economised
// quartic, 2e-9).  Binades with x^2 in [2^-18, 2^14) are covered (x from 2.8e-3
// to 90 at least); entries outside take the direct evaluation.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "bk_forms.cuh"
#include "bk_matern_common.cuh"
#include "bk_math64.cuh"

namespace bk {

constexpr float kInfF = __builtin_huge_valf();
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
    if (F32) return q < 0 ? 6 : q < 5 ? 7 : (q + 9) >> 1;
    return q < 0 ? 7 : q < 3 ? 8 : q < 5 ? 9 : (q + 13) >> 1;
  }
  __host__ __device__ static constexpr int first(int o) {
    int b = 0;
    for (int i = 0; i < o; ++i) b += 1 << bits(i);
    return b;
  }
  static constexpr int kBins = first(kTabOct);
  static constexpr size_t kBytes = (size_t)kBins * kRecord;
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
//  FP32 record, 16 bytes: c_0 (2^-31), c_1 (2^-34), c_2 (2^-39), and c_3 (2^-32)
//   in the upper 20 bits of the word that holds the exponent.
// The top bit of c_0 stays free: the value may round up to 2^E itself.  An
// exponent word of 0 marks an interval without a usable polynomial.
constexpr int kS0 = 62, kS1 = 67, kS2 = 74, kS3 = 51, kS4 = 54;
constexpr int kT0 = 31, kT1 = 34, kT2 = 39, kT3 = 44;
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
// right end less one FP64 ulp (its largest double), for FP32 records less half
// an FP32 ulp.
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
                                           ((unsigned long long)(i + 1) << (52 - m)) -
                                           (F32 ? 1ULL << 28 : 1ULL)));
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
__device__ __forceinline__ void tab_record(int bin, double nu, unsigned e0, double b2, double b2lo,
                                           double r2_max, double f0, double f1,
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
    // c_4 u^4 replaced by its cubic best approximation on [0, 1],
    // u^4 ~ 2 u^3 - 5/4 u^2 + u/4 - 1/128
    c[3] = fma(2.0, c[4], c[3]);
    c[2] = fmax(fma(-1.25, c[4], c[2]), 0.0);
    c[1] = fma(0.25, c[4], c[1]);
    c[0] = fma(-1.0 / 128.0, c[4], c[0]);
  }
  constexpr int kTop = F32 ? 3 : 6;
  double vmax = c[kTop];  // the value at the left end, the largest of the interval
#pragma unroll
  for (int k = kTop - 1; k >= 0; --k) vmax += c[k];
  const int ev = (int)((unsigned)__double2hiint(vmax) >> 20);  // 2048 and above: negative
  const int E = ev - 1022;                                     // vmax in [2^{E-1}, 2^E)
  // signs, and the bounds that the scales were chosen for (c_k < 2^{E-b})
  auto below = [&](int k, int b) { return (int)((unsigned)__double2hiint(c[k]) >> 20) < ev + 1 - b; };
  bool ok = ev > 60 && ev < 1980;
  // exponent words: the exponent field of 2^{E-1} less the leading bit that the
  // significand adds
  uint4* rec = reinterpret_cast<uint4*>(table + (size_t)bin * L::kRecord);
  if constexpr (F32) {
    ok = ok && below(0, 0) && below(1, 3) && below(2, 8) && below(3, 13) && E > -120 && E < 120;
    rec[0] = make_uint4((unsigned)tab_fix(c[0], kT0 - E), (unsigned)tab_fix(c[1], kT1 - E),
                        (unsigned)tab_fix(c[2], kT2 - E),
                        ((unsigned)tab_fix(c[3], kT3 - 12 - E) << 12) | (ok ? (unsigned)(E + 125) : 0u));
  } else {
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
      tab_record<F32>(bin, mp.nu, e0, b2, b2lo, r2_max, sm.f0[threadIdx.x], sm.f1[threadIdx.x], table);
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

// The octave table of the evaluation, one int2 per binade in shared memory:
// {shift of r^2's (or the FP32 r^2's) leading word, first interval less the
// binade's leading bits}.
template <bool F32>
__device__ __forceinline__ void tab_stage_octaves(int2* s_oct, unsigned e0) {
  using L = TabLayout<F32>;
  if (threadIdx.x < kTabOct) {
    const int o = threadIdx.x, m = L::bits(o);
    if constexpr (F32) {  // FP32 word: biased exponent 127, 23 significand bits
      const int sh = 23 - m;
      s_oct[o] = make_int2(sh, L::first(o) - ((((int)e0 - 1023 + 127 + o) << 23) >> sh));
    } else {
      const int sh = 20 - m;
      s_oct[o] = make_int2(sh, L::first(o) - (int)((e0 + o) << (20 - sh)));
    }
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

// The same in FP32: the squared distance as a double-float.
__device__ __forceinline__ bool tab_entry32(const unsigned char* __restrict__ table,
                                            const int2* s_oct, unsigned e0, DF r2, float& out) {
  const unsigned hb = (unsigned)__float_as_int(r2.hi);
  const unsigned o = (hb >> 23) - (e0 - 1023u + 127u);
  const bool in = o < (unsigned)kTabOct;
  const int2 oc = s_oct[in ? o : 0];
  const int idx = in ? (int)(hb >> oc.x) + oc.y : 0;
  const uint4 a = __ldg(reinterpret_cast<const uint4*>(table) + idx);
  // distance to the expansion point: the bits of hi, half a unit, less lo.
  // |lo| <= half an ulp of hi = 2^{8+m} units of 2^-32 of the interval, cut
  // just below it so that u stays inside 32 bits.  Conversions between FP32 and
  // integers by magic numbers and bit fields: as instructions they took the
  // FP64 pipe here, 53 % busy.
  const int m = 23 - oc.x;
  const float scale = __int_as_float((int)((127 + 32 + m + 127) << 23) - (int)(hb & 0x7f800000u));
  const int d = __float_as_int(fmaf(r2.lo, scale * (1.0f - 0x1p-12f), 12582912.0f)) - 0x4b400000;
  const unsigned u = ((~hb) << (9 + m)) + (1u << (8 + m)) - (unsigned)d;
  unsigned A = a.z + (__umulhi(a.w & 0xfffff000u, u) >> (kT3 - kT2));
  A = a.y + (__umulhi(A, u) >> (kT2 - kT1));
  unsigned F = a.x + (__umulhi(A, u) >> (kT1 - kT0));
  // F 2^{E-31}, F in [2^29, 2^31]
  const unsigned ex = a.w & 0xfffu;
  unsigned ew = ex;
  if (F < 0x40000000u) {
    F <<= 1;
    --ew;
  }
  out = __int_as_float((int)(((F + 64u) >> 7) + (ew << 23)));
  return in && ex != 0u;
}

// The squared distance as a double-float, hi the rounded sum (|lo| <= half
// an ulp): exact FP32 differences of the hi parts, products by the FMA.
__device__ __forceinline__ DF df_dist2(float axh, float axl, float ayh, float ayl, float bxh,
                                       float bxl, float byh, float byl) {
  const DF dx = two_sum(bxh, -axh), dy = two_sum(byh, -ayh);
  const float lx = dx.lo + (bxl - axl), ly = dy.lo + (byl - ayl);
  const float px = dx.hi * dx.hi, py = dy.hi * dy.hi;
  const float ex = fmaf(lx, fmaf(2.0f, dx.hi, lx), fmaf(dx.hi, dx.hi, -px));
  const float ey = fmaf(ly, fmaf(2.0f, dy.hi, ly), fmaf(dy.hi, dy.hi, -py));
  const DF s = two_sum(px, py);
  return quick_two_sum(s.hi, s.lo + (ex + ey));
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

constexpr int kTabTile = 64;  // tile edge of the writers that use a table

template <typename OutT>
struct TabTileSmem {
  double2 c[kTabTile];   // columns' coordinates
  float4 cf[kTabTile];   // the same as floats {x hi, x lo, y hi, y lo}
  int2 oct[kTabOct];
  OutT tile[kTabTile][kTabTile + 1];
};

// A coordinate as two floats (hi + lo) on the integer pipe.  What those do not
// hold (tiny, huge, not finite) becomes NaN, which no table contains: its
// entries take the direct evaluation.  (A branch to conversions instead was
// executed by every thread: 200 FP64-pipe instructions a tile, half its time.)
__device__ __forceinline__ void split_bits(double v, float& h, float& l) {
  bool ok;
  const DF d = df_from_bits(v, ok);
  const bool zero = ((__double2hiint(v) << 1) | __double2loint(v)) == 0;
  h = ok ? d.hi : zero ? 0.0f : __int_as_float(0x7fc00000);
  l = ok ? d.lo : 0.0f;
}

// One 64 x 64 tile (I, J) of M between locs1 (rows) and locs2 (columns) by a
// block of WARPS warps: lane i of warp w takes rows i and i + 32 of columns w,
// w + WARPS, ..., two rows at a time so that the loads of one entry overlap the
// arithmetic of the other.  kSym: the transposed block (J, I) is written too.
// The caller has staged sm.oct; the block is synchronised here after staging.
// use_table false: every entry by the direct evaluation.  part, width: the block takes columns part * width .. + width - 1 only (width
// 16 or 64), where whole tiles would leave SMs without a block.
template <bool F32, typename OutT, bool kSym, int WARPS>
__device__ __forceinline__ void tab_tile(TabTileSmem<OutT>& sm, const unsigned char* __restrict__ table,
                                         unsigned e0, const double* __restrict__ locs1, int64_t m,
                                         const double* __restrict__ locs2, int64_t n, int64_t I,
                                         int64_t J, const MaternParams& mp, OutT* __restrict__ out,
                                         int64_t ld, int part = 0, int width = kTabTile,
                                         bool use_table = true) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = I * kTabTile, c0 = J * kTabTile;
  if (threadIdx.x < kTabTile) {
    const int64_t j = c0 + threadIdx.x;
    const double x = j < n ? locs2[j] : 0.0, y = j < n ? locs2[n + j] : 0.0;
    sm.c[threadIdx.x] = make_double2(x, y);
    if constexpr (F32) {
      float4 f;
      split_bits(x, f.x, f.y);
      split_bits(y, f.z, f.w);
      sm.cf[threadIdx.x] = f;
    }
  }
  double ax[2], ay[2];
  float axh[2], axl[2], ayh[2], ayl[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int64_t i = r0 + lane + 32 * h;
    ax[h] = i < m ? locs1[i] : 0.0;
    ay[h] = i < m ? locs1[m + i] : 0.0;
    if constexpr (F32) {
      split_bits(ax[h], axh[h], axl[h]);
      split_bits(ay[h], ayh[h], ayl[h]);
    }
  }
  __syncthreads();
  const bool in0 = r0 + lane < m, in1 = r0 + lane + 32 < m;
  const int cb = part * width, cw = cb + warp;  // the part's first column, the warp's
  OutT* po = out + (r0 + lane) + (c0 + cw) * ld;
  const int cols = (int)(n - c0 < cb + width ? n - c0 : cb + width);
  unsigned bad = 0;  // entries outside the table: bits 2 k and 2 k + 1 of column cw + k WARPS
  int k = 0;
#pragma unroll 2
  for (int c = cw; c < (use_table ? cols : 0); c += WARPS, ++k) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      OutT v;
      bool ok;
      if constexpr (F32) {
        const float4 b = sm.cf[c];
        const DF r2 = df_dist2(axh[h], axl[h], ayh[h], ayl[h], b.x, b.y, b.z, b.w);
        ok = tab_entry32(table, sm.oct, e0, r2, v);
      } else {
        const double2 b = sm.c[c];
        const double dx = b.x - ax[h], dy = b.y - ay[h];
        double d;
        ok = tab_entry64(table, sm.oct, e0, fma(dx, dx, dy * dy), d);
        v = to_out<OutT>(d);
      }
      bad |= (ok ? 0u : 1u) << (2 * k + h);
      if (h ? in1 : in0) po[32 * h] = v;
      if constexpr (kSym) sm.tile[lane + 32 * h][c] = v;
    }
    po += WARPS * ld;
  }
  if (!use_table)
    for (int c = cw; c < cols; c += WARPS, ++k) bad |= 3u << (2 * k);
  if (bad != 0) {  // coincident, very near or far pairs: written again by the direct evaluation
    while (bad != 0) {
      const int b = __ffs((int)bad) - 1, c = cw + (b >> 1) * WARPS, i = lane + 32 * (b & 1);
      bad &= bad - 1;
      if (r0 + i >= m) continue;
      Loc p, q;
      p.x = locs1[r0 + i];
      p.y = locs1[m + r0 + i];
      q.x = sm.c[c].x;
      q.y = sm.c[c].y;
      OutT v;
      if constexpr (F32) {
        split_f(p.x, p.xh, p.xl);
        split_f(p.y, p.yh, p.yl);
        split_f(q.x, q.xh, q.xl);
        split_f(q.y, q.yh, q.yl);
        v = matern_direct32(p, q, mp);
      } else {
        v = to_out<OutT>(matern_direct64(p, q, mp));
      }
      out[(r0 + i) + (c0 + c) * ld] = v;
      if constexpr (kSym) sm.tile[i][c] = v;
    }
  }
  if constexpr (kSym) {
    if (I == J) return;
    __syncthreads();
    if (width == kTabTile) {
#pragma unroll 4
      for (int c = warp; c < kTabTile; c += WARPS) {
        const int64_t j = r0 + c;  // column r0 + c of block (J, I): row c of the tile
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int64_t i = c0 + lane + 32 * h;
          if (i < n && j < m) out[i + j * ld] = sm.tile[c][lane + 32 * h];
        }
      }
    } else {
      for (int t = threadIdx.x; t < kTabTile * width; t += WARPS * 32) {
        const int c = t / width, i = cb + t % width;
        if (c0 + i < n && r0 + c < m) out[(c0 + i) + (r0 + c) * ld] = sm.tile[c][i];
      }
    }
  }
}

}  // namespace bk
