// The Matern tile writers that evaluate their entries from a per-call table
// (bk_entry_table.cuh): the table's kernel, the symmetric writer and the m x n
// block writer, and the rule that takes a call to them.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "bk_entry_table.cuh"
#include "bk_internal.h"
#include "bk_tiles.cuh"

namespace bk {
namespace {

// The table of one call.  Up to kTabScan locations, every block first bounds
// the distances (1.5 us there), and the binades beyond the bound are left out:
// for x up to 14 that is two thirds of the intervals.
constexpr int64_t kTabScan = 8192;
template <bool F32>
__global__ void __launch_bounds__(kTabThreads) entry_table_kernel(
    const __grid_constant__ MaternParams mp, const double* __restrict__ locs1, int64_t m,
    const double* __restrict__ locs2, int64_t n, unsigned char* __restrict__ table) {
  __shared__ TabBuildSmem sm;
  asm volatile("griddepcontrol.launch_dependents;");
  tab_build_block<F32>(sm, mp, (int)blockIdx.x, (int)gridDim.x, m + n <= 2 * kTabScan, locs1, m, locs2, n,
                       table);
}

// One 64 x 64 tile per block of 256 threads; lane i of warp w evaluates rows
// i and i + 32 against columns w, w + 8, w + 16, ...  Block (I, J) is stored straight
// from registers (a warp writes 32 consecutive rows of one column); for a
// symmetric matrix the tile also goes through shared memory to block (J, I).
// col_base as in matern_sym_kernel, in tiles of 64.  FP32 entries wait on their
// record's load more than on anything else (n = 40,000: 4 blocks an SM 1,883 us,
// 6 1,699, 8 1,988, spilling a few registers outside the loop); FP64 entries
// do not gain from more (n = 20,000: 3 blocks 1,139, 4 1,079, 5 1,081, 6 1,142; now
// 1,673 and 1,040).
template <bool F32, typename OutT, bool kSym>
__global__ void __launch_bounds__(256, F32 ? 6 : 4) matern_table_kernel(
    const unsigned char* table, const double* __restrict__ locs1, int64_t m,
    const double* __restrict__ locs2, int64_t n, const __grid_constant__ MaternParams mp,
    OutT* __restrict__ out, int64_t ld, int64_t tiles_m, int64_t col_base, int width) {
  __shared__ TabTileSmem<F32, OutT> sm;
  // launched while the table's kernel may still run (launch_writer)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const unsigned parts = kTabTile / width, tile = blockIdx.x / parts, part = blockIdx.x % parts;
  int64_t I, J;
  if constexpr (kSym) {
    if (col_base < 0) tri_tile(tile, I, J);
    else col_tile(col_base + tile, tiles_m, I, J);
  } else {
    I = tile % tiles_m;
    J = tile / tiles_m;
  }
  tab_tile<F32, OutT, kSym, 8>(sm, table, locs1, m, locs2, n, I, J, mp, out, ld, (int)part, width);
}

// ---- batched: every instance's constants and table in one launch, all tiles in
// the next, instances without a table in a third (bk_batched.cu) ----
// One short block for each instance that cannot have a table, then `share` blocks
// for each of the others: its constants, which the first block also stores, and the
// block's share of the table.  (A kernel of their own for the constants
// cost 2 us; 300 matrices of n = 300 take 2 % more without it, in FP32 8 %.)
template <bool F32>
__global__ void __launch_bounds__(kTabThreads) batched_table_kernel(
    const bk_matern_desc* __restrict__ descs, const __grid_constant__ BatchTable t, int share) {
  __shared__ TabBuildSmem sm;
  __shared__ BatchInstance b;
  asm volatile("griddepcontrol.launch_dependents;");
  const int rest = t.count - t.with_table, id = (int)blockIdx.x - rest;
  const int k = t.order[id >= 0 ? id / share : t.count + id];
  const int block = id >= 0 ? id % share : 0, blocks = id >= 0 ? share : 1;
  if (threadIdx.x == 0) {
    const bk_matern_desc d = descs[k];
    // a descriptor that does not match the plan is skipped (n = 0)
    const bool ok = d.n == t.sizes[k] && d.ld >= d.n && d.locs != nullptr && d.out != nullptr &&
                    d.beta > 0.0 && d.nu > 0.0 && d.sigma2 >= 0.0;
    b.locs = d.locs;
    b.out = d.out;
    b.n = ok ? d.n : 0;
    b.ld = d.ld;
    b.table = ok && t.prefix[k + 1] > t.prefix[k] && tab_domain(F32, d.sigma2, d.beta, d.nu);
    b.mp = matern_params(d.sigma2, d.beta, d.nu);
  }
  __syncthreads();
  if (block == 0) {
    constexpr int kWords = (int)(sizeof(BatchInstance) / 8);
    if (threadIdx.x < kWords)
      reinterpret_cast<long long*>((BatchInstance*)t.instances + k)[threadIdx.x] =
          reinterpret_cast<const long long*>(&b)[threadIdx.x];
    if (threadIdx.x == 0) t.direct[k] = b.n > 0 && !b.table;
    if (blockIdx.x == 0 && threadIdx.x < 2) t.next[threadIdx.x] = 0ull;
  }
  unsigned char* const table = (unsigned char*)t.tables + (size_t)k * TabLayout<F32>::kStride;
  if (!b.table) {  // for the per-entry kernel: the plain form's e^{-2 nu h}
    if constexpr (!F32) {
      for (int i = block * kTabThreads + (int)threadIdx.x; t.decay && b.n > 0 && i < kCoshTabSize; i += blocks * kTabThreads)
        reinterpret_cast<double*>(table)[i] = decay_entry(b.mp.nu, i, kExp2Tab);
    }
    return;
  }
  tab_build_block<F32>(sm, b.mp, block, blocks, b.n <= kTabScan, b.locs, b.n, b.locs, b.n,
                       table + TabLayout<F32>::kFront);
}

// Persistent kernel as matern_batched_kernel, in tiles of 64 of the instances that
// may have a table; one that has none (parameters outside the domain) is passed over.
template <bool F32, typename OutT, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 32 / WARPS) matern_batched_table_kernel(
    const BatchInstance* inst, int count, const int64_t* __restrict__ prefix,
    int64_t limit, unsigned long long* __restrict__ next, int chunk,
    const unsigned char* tables) {
  __shared__ TabTileSmem<F32, OutT> sm;
  __shared__ BatchInstance cur;
  __shared__ int64_t item;
  int k = -1;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  while (true) {
    __syncthreads();  // shared data of the previous round is no longer read
    if (threadIdx.x == 0) item = (int64_t)atomicAdd(next, (unsigned long long)chunk);
    __syncthreads();
    const int64_t base = item;
    if (base >= limit) break;
    const int64_t end = min(base + (int64_t)chunk, limit);
    for (int64_t w = base; w < end; ++w) {
      const int kw = find_instance(prefix, count, w);
      __syncthreads();
      if (kw != k) {
        k = kw;
        constexpr int kWords = (int)(sizeof(BatchInstance) / 8);
        static_assert(sizeof(BatchInstance) % 8 == 0 && kWords <= 128, "copied by the block's threads");
        if (threadIdx.x < kWords)
          reinterpret_cast<long long*>(&cur)[threadIdx.x] =
              reinterpret_cast<const long long*>(inst + k)[threadIdx.x];
        __syncthreads();
      }
      if (!cur.table) {
        if (threadIdx.x == 0) atomicMax(next, (unsigned long long)__ldg(prefix + k + 1));
        w = min(__ldg(prefix + k + 1), end) - 1;
        continue;
      }
      int64_t I, J;
      tri_tile(w - __ldg(prefix + k), I, J);
      tab_tile<F32, OutT, true, WARPS>(sm, tables + (size_t)k * TabLayout<F32>::kStride + TabLayout<F32>::kFront,
                                       cur.locs, cur.n, cur.locs, cur.n, I, J, cur.mp, (OutT*)cur.out, cur.ld);
    }
  }
}

}  // namespace

size_t entry_table_bytes(bool f32) { return f32 ? TabLayout32::kStride : TabLayout64::kStride; }

// A matrix is worth a table, which costs about 13 us,
// from 2^19 entries on (n = 725) in every form, as the writers without one are bound
// by one entry's latency there.  n = 800, beta = 0.1, nu = 0.8: 27 us with it, without
// 66 (FP64), 44 (FP32), 34 (learned); blocks of 520,000 entries 24 with it, without
// 80, 44, 31.  Smaller ones keep the direct path, whose results do not depend on
// whether the caller has scratch memory.  Stored to host memory FP64 and FP32 gain too
// (n = 800: 53 and 36 us, without 75 and 49 to 61); the learned form takes 36 (38) at
// n = 800, 47 (42) at 900, 44 (41) at 1,024, 57 (58) at 1,280, 85 (88) at 1,450, and
// keeps the rule, so that a matrix is the same wherever it is stored.
bool entry_table_pays(int64_t rows, int64_t cols) {
  constexpr int64_t kLeast = (int64_t)1 << 19;
  return rows > 0 && cols > 0 && rows >= (kLeast + cols - 1) / cols;
}

bool entry_table_applies(const bk_opts& o, bk_dtype out_t, double sigma2, double beta, double nu) {
  return o.d_counters == nullptr && o.window != BK_WIN_FIXED && o.series_below == 0.0 &&
         o.search_f64 == 0 && tab_domain(o.compute == BK_F32 && out_t == BK_F32, sigma2, beta, nu);
}

namespace {

// Whole tiles where they fill the SMs' four slots once, else quarters of 16
// columns (n = 777: 91 tiles on 152 SMs, 14.8 us whole).  Over the link to host
// memory a part's transposed columns of 16 rows are pieces of lines, so halves there
// (FP32: n = 850 48.5 us in quarters, 44.6 in halves; n = 1,280 61.0, 56.5), and
// whole tiles where the matrix's columns do not start on 32 bytes, from 1.5 tiles an
// SM on (n = 1,450 99.7 us in quarters, 87.4 in halves, 85.2 whole; n = 1,837 147.8,
// 131.3, 123.3; FP64 218, 199, 194; but FP64 n = 2,048 199 in halves, 205 whole).
int tile_width(int64_t ntiles, bool host, int64_t column_bytes) {
  const int64_t sms = current_sm_count();
  if (ntiles >= 4 * sms) return kTabTile;
  if (!host) return kTabTile / 4;
  return column_bytes % 32 != 0 && 2 * ntiles >= 3 * sms ? kTabTile : kTabTile / 2;
}

template <typename... P, typename... A>
cudaError_t launch_writer(void (*kernel)(P...), unsigned grid, cudaStream_t s, A... args) {
  return launch_next(kernel, dim3(grid), 256, s, args...);
}

template <bool F32>
cudaError_t build_table(const MaternParams& mp, const double* locs1, int64_t m,
                        const double* locs2, int64_t n, unsigned char* table, cudaStream_t s) {
  entry_table_kernel<F32><<<current_sm_count(), kTabThreads, 0, s>>>(mp, locs1, m, locs2, n, table);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_matern_sym_table(const double* locs, int64_t n, double sigma2, double beta,
                                    double nu, void* out, int64_t ld, bk_dtype out_t,
                                    bk_dtype compute, void* table, cudaStream_t s,
                                    const SymRange& range) {
  const MaternParams mp = matern_params_host(sigma2, beta, nu);
  const bool f32 = compute == BK_F32 && out_t == BK_F32;
  unsigned char* const tab = (unsigned char*)table + (f32 ? TabLayout32::kFront : TabLayout64::kFront);
  if (range.fill_table) {
    const cudaError_t e = f32 ? build_table<true>(mp, locs, n, locs, n, tab, s)
                              : build_table<false>(mp, locs, n, locs, n, tab, s);
    if (e != cudaSuccess) return e;
  }
  const int64_t nb = (n + kTabTile - 1) / kTabTile;
  int64_t ntiles = nb * (nb + 1) / 2, col_base = -1;
  if (range.j1 >= 0) {
    const int64_t j0 = range.j0 < 0 ? 0 : range.j0, j1 = range.j1 < nb ? range.j1 : nb;
    if (j1 <= j0) return cudaSuccess;
    col_base = j0 * nb - j0 * (j0 - 1) / 2;
    ntiles = (j1 * nb - j1 * (j1 - 1) / 2) - col_base;
  }
  if (ntiles > 2147483647) return cudaErrorInvalidConfiguration;
  const int width = tile_width(ntiles, range.host, ld * (out_t == BK_F64 ? 8 : 4));
  const unsigned grid = (unsigned)(ntiles * (kTabTile / width));
  if (f32)
    return launch_writer(matern_table_kernel<true, float, true>, grid, s, tab, locs, n, locs, n, mp,
                         (float*)out, ld, nb, col_base, width);
  if (out_t == BK_F32)
    return launch_writer(matern_table_kernel<false, float, true>, grid, s, tab, locs, n, locs, n, mp,
                         (float*)out, ld, nb, col_base, width);
  return launch_writer(matern_table_kernel<false, double, true>, grid, s, tab, locs, n, locs, n, mp,
                       (double*)out, ld, nb, col_base, width);
}

cudaError_t launch_matern_block_table(const double* locs1, int64_t m, const double* locs2, int64_t n,
                                      double sigma2, double beta, double nu, void* out, int64_t ld,
                                      bk_dtype out_t, bk_dtype compute, void* table, cudaStream_t s) {
  const MaternParams mp = matern_params_host(sigma2, beta, nu);
  const bool f32 = compute == BK_F32 && out_t == BK_F32;
  unsigned char* const tab = (unsigned char*)table + (f32 ? TabLayout32::kFront : TabLayout64::kFront);
  const cudaError_t e = f32 ? build_table<true>(mp, locs1, m, locs2, n, tab, s)
                            : build_table<false>(mp, locs1, m, locs2, n, tab, s);
  if (e != cudaSuccess) return e;
  const int64_t tm = (m + kTabTile - 1) / kTabTile, tn = (n + kTabTile - 1) / kTabTile;
  if (tm * tn > 2147483647) return cudaErrorInvalidConfiguration;
  const int width = tile_width(tm * tn, false, 0);
  const unsigned grid = (unsigned)(tm * tn * (kTabTile / width));
  if (f32)
    return launch_writer(matern_table_kernel<true, float, false>, grid, s, tab, locs1, m, locs2, n, mp,
                         (float*)out, ld, tm, -1, width);
  if (out_t == BK_F32)
    return launch_writer(matern_table_kernel<false, float, false>, grid, s, tab, locs1, m, locs2, n, mp,
                         (float*)out, ld, tm, -1, width);
  return launch_writer(matern_table_kernel<false, double, false>, grid, s, tab, locs1, m, locs2, n, mp,
                       (double*)out, ld, tm, -1, width);
}


size_t batched_instance_bytes() { return sizeof(BatchInstance); }

namespace {

template <bool F32, typename OutT>
cudaError_t launch_batched_table_t(const BatchTable& b, const bk_matern_desc* descs, int64_t limit, int warps,
                                   int ctas_per_sm, int chunk, cudaStream_t s) {
  // The instances' tables in one wave of blocks, one on an SM, beside a few of the
  // other instances' (many of those leave the SMs again at once); at least four each,
  // so that the node weights, once per block, stay a small part of it.
  const int sms = current_sm_count(), rest = b.count - b.with_table;
  const int share = std::max((sms - (rest <= sms / 4 ? rest : 0)) / b.with_table, 4);
  batched_table_kernel<F32><<<(unsigned)(rest + share * b.with_table), kTabThreads, 0, s>>>(descs, b, share);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_next(warps == 4 ? matern_batched_table_kernel<F32, OutT, 4> : matern_batched_table_kernel<F32, OutT, 8>,
                     dim3((unsigned)(sms * ctas_per_sm)), warps * 32, s, (const BatchInstance*)b.instances, b.count,
                     b.prefix, limit, b.next, chunk, (const unsigned char*)b.tables);
}

}  // namespace

cudaError_t launch_batched_table(const BatchTable& b, const bk_matern_desc* descs, bool f32,
                                 bk_dtype out_t, int64_t limit, int warps, int ctas_per_sm, int chunk,
                                 cudaStream_t s) {
  if (f32) return launch_batched_table_t<true, float>(b, descs, limit, warps, ctas_per_sm, chunk, s);
  if (out_t == BK_F32) return launch_batched_table_t<false, float>(b, descs, limit, warps, ctas_per_sm, chunk, s);
  return launch_batched_table_t<false, double>(b, descs, limit, warps, ctas_per_sm, chunk, s);
}

int batched_table_max_ctas(bool f32, bk_dtype out_t, int warps) {
  const void* fn =
      f32 ? (warps == 4 ? (const void*)matern_batched_table_kernel<true, float, 4>
                        : (const void*)matern_batched_table_kernel<true, float, 8>)
      : out_t == BK_F32 ? (warps == 4 ? (const void*)matern_batched_table_kernel<false, float, 4>
                                      : (const void*)matern_batched_table_kernel<false, float, 8>)
                        : (warps == 4 ? (const void*)matern_batched_table_kernel<false, double, 4>
                                      : (const void*)matern_batched_table_kernel<false, double, 8>);
  int blocks = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, warps * 32, 0) != cudaSuccess) return 1;
  return blocks < 1 ? 1 : blocks;
}

}  // namespace bk
