// Batched persistent Matern writer (a maximum-likelihood parameter sweep
// issues many covariance matrices of uneven n with per-instance
// (sigma^2, beta, nu); Sec. III-A motivates regenerating them every
// likelihood evaluation).  One launch covers every lower-triangle tile of
// every instance: CTAs take tiles from a device counter, so instances of any
// size share the machine without a launch per matrix.  The plan owns the
// work list (tile prefix sums per instance) and the counter; the hot call is
// one memset + one launch, or with entry tables (bk_entry_table.cu) three launches,
// all capturable in a CUDA graph.
#include <cuda_runtime.h>

#include <algorithm>
#include <cerrno>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <sys/stat.h>
#include <vector>

#include "bk_internal.h"
#include "bk_forms.cuh"
#include "bk_tiles.cuh"

namespace bk {

template <typename OutT>
struct BatchSmem {
  SymTileSmem<OutT> tile;
  const double* locs;
  OutT* out;
  int64_t n, ld, item;
  MaternParams mp;
  const double* wnu;  // the instance's table of e^{-2 nu h}, or null
};

// Persistent kernel: each CTA repeatedly takes `chunk` consecutive tiles from
// *next (scratch, zeroed before the launch) until `limit` tiles are taken.
// kChosen: only the instances with direct[k] != 0 (a plan with entry tables;
// launched while the kernels that write direct and the tables may still run).
template <class Form, typename OutT, int WARPS, bool kChosen>
__global__ void __launch_bounds__(WARPS * 32, Form::kMinBlocks * 8 / WARPS) matern_batched_kernel(
    const Form form, const bk_matern_desc* __restrict__ descs, int count, const int64_t* __restrict__ prefix,
    const int64_t* __restrict__ sizes, int64_t limit, unsigned long long* __restrict__ next,
    int chunk, unsigned long long* __restrict__ ctr, const double* wnu_tabs, int64_t wnu_stride, const int* direct) {
  if constexpr (kChosen) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int any = 0;
    for (int k = (int)threadIdx.x; k < count; k += WARPS * 32) any |= direct[k];
    if (!__syncthreads_or(any)) return;
  }
  __shared__ BatchSmem<OutT> sm;
  __shared__ double s_tab[Form::kStageTable ? kExpTabSize : 1];
  const Form f = bind_table(form, s_tab);
  Tally tl{0u, 0u, 0u, 0u, 0u, 0u, 0u};
  unsigned evals = 0;
  int cur = -1;
  while (true) {
    __syncthreads();  // shared data of the previous round is no longer read
    if (threadIdx.x == 0) sm.item = (int64_t)atomicAdd(next, (unsigned long long)chunk);
    __syncthreads();
    const int64_t base = sm.item;
    if (base >= limit) break;
    const int64_t end = min(base + (int64_t)chunk, limit);
    for (int64_t w = base; w < end; ++w) {
      const int k = find_instance(prefix, count, w);
      if constexpr (kChosen) {
        if (!direct[k]) {  // past all of this instance's tiles
          if (threadIdx.x == 0) atomicMax(next, (unsigned long long)__ldg(prefix + k + 1));
          w = min(__ldg(prefix + k + 1), end) - 1;
          continue;
        }
      }
      if (k != cur) {
        __syncthreads();
        if (threadIdx.x == 0) {
          bk_matern_desc d = descs[k];
          // a descriptor that does not match the plan is skipped (n = 0) and counted
          const bool ok = d.n == __ldg(sizes + k) && d.ld >= d.n && d.locs != nullptr &&
                          d.out != nullptr && d.beta > 0.0 && d.nu > 0.0 && d.sigma2 >= 0.0;
          if (!ok) {
            d.n = 0;
            if (ctr != nullptr) atomicAdd(ctr + BK_CTR_FAIL, 1ull);
          }
          sm.locs = d.locs;
          sm.out = (OutT*)d.out;
          sm.n = d.n;
          sm.ld = d.ld;
          sm.mp = matern_params(d.sigma2, d.beta, d.nu);  // a1, once per instance run
          sm.wnu = (wnu_tabs != nullptr) ? wnu_tabs + k * wnu_stride : nullptr;
        }
        __syncthreads();
        cur = k;
      }
      int64_t I, J;
      tri_tile(w - __ldg(prefix + k), I, J);
      __syncthreads();
      if constexpr (Form::kDecayTable) {
        Form fk = f;
        fk.wnu = sm.wnu;
        sym_tile<Form, OutT, WARPS>(fk, sm.tile, sm.locs, sm.n, I, J, sm.mp, sm.out, sm.ld, tl,
                                    evals);
      } else {
        sym_tile<Form, OutT, WARPS>(f, sm.tile, sm.locs, sm.n, I, J, sm.mp, sm.out, sm.ld, tl,
                                    evals);
      }
    }
  }
  flush_tally(ctr, tl, evals);
}

// Fills each instance's table of e^{-2 nu h} on kCoshTab's steps from its
// descriptor's nu (instances with a bad descriptor are skipped by the tile
// kernel whatever their table holds).
__global__ void __launch_bounds__(256) batched_decay_kernel(const bk_matern_desc* __restrict__ descs,
                                                              int count, double* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)count * kCoshTabSize) return;
  const int k = (int)(i / kCoshTabSize), j = (int)(i % kCoshTabSize);
  const double nu = descs[k].nu;
  out[i] = decay_entry(nu > 0.0 ? nu : 0.0, j, kExp2Tab);
}

}  // namespace bk

// ---------------------------------------------------------------------------
// Plan and launch (host)

struct bk_plan {
  int device;
  int32_t count;
  bk_dtype dtype;
  bk_opts opts;
  int64_t total_tiles;
  int64_t* d_prefix;               // count + 1 tile offsets (device)
  int64_t* d_sizes;                // count instance sizes (device)
  unsigned long long* d_next;      // two tile counters (device scratch)
  double* d_wnu;                   // count x kCoshTabSize: e^{-2 nu h} per instance, or null
  // with entry tables (else null): tiles of 64 of the instances that may have one
  // and their offsets, the instances' constants, their tables, and a flag for each
  // instance that the per-entry kernel takes
  int64_t table_tiles;
  int with_table;                  // instances that may have a table, first in d_order
  int* d_order;
  int64_t* d_table_prefix;
  void* d_inst;
  void* d_tables;
  int* d_direct;
  int warps, ctas_per_sm, chunk;   // launch shape
  int tuned;                       // 1 when the shape came from the autotuner or its cache
  double tuned_ms;
  std::string key;
};

namespace bk {
namespace {

template <class Form>
Form make_form(const bk_plan*) { return Form{}; }
template <>
FormF64 make_form<FormF64>(const bk_plan* p) {
  return FormF64{nullptr, p->opts.search_f64 != 0, 0.0};
}
template <>
FormF64Series make_form<FormF64Series>(const bk_plan* p) {
  return FormF64Series{nullptr, p->opts.search_f64 != 0, p->opts.series_below};
}
template <>
FormF64Fixed make_form<FormF64Fixed>(const bk_plan* p) {
  return FormF64Fixed{nullptr, p->opts.fixed_t1, p->opts.fixed_bins, p->opts.series_below};
}
template <>
FormF32Learned make_form<FormF32Learned>(const bk_plan* p) {
  return FormF32Learned{learned_view(p->opts.learned)};
}

template <class Form, typename OutT, int WARPS>
cudaError_t launch_batched_t(const bk_plan* p, const bk_matern_desc* d, int64_t limit,
                             int ctas_per_sm, int chunk, cudaStream_t s) {
  const int grid = current_sm_count() * ctas_per_sm;
  matern_batched_kernel<Form, OutT, WARPS, false><<<grid, WARPS * 32, 0, s>>>(
      make_form<Form>(p), d, p->count, p->d_prefix, p->d_sizes, limit, p->d_next, chunk, p->opts.d_counters,
      Form::kDecayTable ? p->d_wnu : nullptr, kCoshTabSize, nullptr);
  return cudaGetLastError();
}

// The instances of a plan with tables that have none, in the plan's form.
template <class Form, typename OutT>
cudaError_t launch_batched_rest(const bk_plan* p, const bk_matern_desc* d, int64_t limit, cudaStream_t s) {
  const size_t stride = entry_table_bytes(p->opts.compute == BK_F32 && p->dtype == BK_F32);
  return launch_next(matern_batched_kernel<Form, OutT, 8, true>, dim3((unsigned)(current_sm_count() * 2)), 256, s,
                     make_form<Form>(p), d, p->count, (const int64_t*)p->d_prefix, (const int64_t*)p->d_sizes, limit,
                     p->d_next + 1, 1, (unsigned long long*)nullptr,
                     Form::kDecayTable ? (const double*)p->d_tables : nullptr, (int64_t)(stride / sizeof(double)),
                     (const int*)p->d_direct);
}
template <class Form>
cudaError_t launch_batched_rest(const bk_plan* p, const bk_matern_desc* d, int64_t limit, cudaStream_t s) {
  return p->dtype == BK_F64 ? launch_batched_rest<Form, double>(p, d, limit, s)
                            : launch_batched_rest<Form, float>(p, d, limit, s);
}

template <class Form, typename OutT>
cudaError_t launch_batched_w(const bk_plan* p, const bk_matern_desc* d, int64_t limit, int warps,
                             int ctas_per_sm, int chunk, cudaStream_t s) {
  if (warps == 4) return launch_batched_t<Form, OutT, 4>(p, d, limit, ctas_per_sm, chunk, s);
  return launch_batched_t<Form, OutT, 8>(p, d, limit, ctas_per_sm, chunk, s);
}

// FP32 records: FP32 arithmetic into FP32 matrices.
bool plan_table_f32(const bk_plan* p) { return p->opts.compute == BK_F32 && p->dtype == BK_F32; }

cudaError_t launch_batched(const bk_plan* p, const bk_matern_desc* d, int64_t limit, int warps,
                           int ctas_per_sm, int chunk, cudaStream_t s) {
  if (p->d_tables != nullptr) {
    const BatchTable b{p->count, p->with_table, p->d_order, p->d_table_prefix, p->d_sizes, p->d_next, p->d_direct, p->d_inst, p->d_tables,
                       p->opts.compute == BK_F64};
    const int64_t tiles = limit < p->total_tiles
                              ? std::max<int64_t>(1, (int64_t)((double)p->table_tiles * limit / p->total_tiles))
                              : p->table_tiles;
    const cudaError_t e = launch_batched_table(b, d, plan_table_f32(p), p->dtype, tiles, warps, ctas_per_sm, chunk, s);
    if (e != cudaSuccess) return e;
    return p->opts.window == BK_WIN_LEARNED ? launch_batched_rest<FormF32Learned>(p, d, limit, s)
           : p->opts.compute == BK_F64      ? launch_batched_rest<FormF64>(p, d, limit, s)
                                            : launch_batched_rest<FormF32>(p, d, limit, s);
  }
  cudaError_t e = cudaMemsetAsync(p->d_next, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  if (p->d_wnu != nullptr) {
    const int64_t cells = (int64_t)p->count * kCoshTabSize;
    batched_decay_kernel<<<(unsigned)((cells + 255) / 256), 256, 0, s>>>(d, p->count, p->d_wnu);
  }
  const bool f64 = (p->opts.compute == BK_F64);
  const bool learned = (p->opts.window == BK_WIN_LEARNED);
  if (p->opts.window == BK_WIN_FIXED)
    return (p->dtype == BK_F64)
               ? launch_batched_w<FormF64Fixed, double>(p, d, limit, warps, ctas_per_sm, chunk, s)
               : launch_batched_w<FormF64Fixed, float>(p, d, limit, warps, ctas_per_sm, chunk, s);
  if (f64 && p->opts.series_below > 0.0)
    return (p->dtype == BK_F64)
               ? launch_batched_w<FormF64Series, double>(p, d, limit, warps, ctas_per_sm, chunk, s)
               : launch_batched_w<FormF64Series, float>(p, d, limit, warps, ctas_per_sm, chunk, s);
  if (p->dtype == BK_F64) {
    if (learned)
      return launch_batched_w<FormF32Learned, double>(p, d, limit, warps, ctas_per_sm, chunk, s);
    return f64 ? launch_batched_w<FormF64, double>(p, d, limit, warps, ctas_per_sm, chunk, s)
               : launch_batched_w<FormF32, double>(p, d, limit, warps, ctas_per_sm, chunk, s);
  }
  if (learned)
    return launch_batched_w<FormF32Learned, float>(p, d, limit, warps, ctas_per_sm, chunk, s);
  return f64 ? launch_batched_w<FormF64, float>(p, d, limit, warps, ctas_per_sm, chunk, s)
             : launch_batched_w<FormF32, float>(p, d, limit, warps, ctas_per_sm, chunk, s);
}

int max_ctas_per_sm(const bk_plan* p, int warps) {
  if (p->d_tables != nullptr) return batched_table_max_ctas(plan_table_f32(p), p->dtype, warps);
  int blocks = 0;
  const void* fn = nullptr;
  const bool f64 = (p->opts.compute == BK_F64);
  if (p->opts.window == BK_WIN_FIXED) {
    if (p->dtype == BK_F64)
      fn = (warps == 4) ? (const void*)matern_batched_kernel<FormF64Fixed, double, 4, false>
                        : (const void*)matern_batched_kernel<FormF64Fixed, double, 8, false>;
    else
      fn = (warps == 4) ? (const void*)matern_batched_kernel<FormF64Fixed, float, 4, false>
                        : (const void*)matern_batched_kernel<FormF64Fixed, float, 8, false>;
  } else if (f64 && p->opts.series_below > 0.0) {
    if (p->dtype == BK_F64)
      fn = (warps == 4) ? (const void*)matern_batched_kernel<FormF64Series, double, 4, false>
                        : (const void*)matern_batched_kernel<FormF64Series, double, 8, false>;
    else
      fn = (warps == 4) ? (const void*)matern_batched_kernel<FormF64Series, float, 4, false>
                        : (const void*)matern_batched_kernel<FormF64Series, float, 8, false>;
  } else if (p->opts.window == BK_WIN_LEARNED) {
    if (p->dtype == BK_F64)
      fn = (warps == 4) ? (const void*)matern_batched_kernel<FormF32Learned, double, 4, false>
                        : (const void*)matern_batched_kernel<FormF32Learned, double, 8, false>;
    else
      fn = (warps == 4) ? (const void*)matern_batched_kernel<FormF32Learned, float, 4, false>
                        : (const void*)matern_batched_kernel<FormF32Learned, float, 8, false>;
  } else if (p->dtype == BK_F64) {
    if (warps == 4) fn = f64 ? (const void*)matern_batched_kernel<FormF64, double, 4, false>
                             : (const void*)matern_batched_kernel<FormF32, double, 4, false>;
    else fn = f64 ? (const void*)matern_batched_kernel<FormF64, double, 8, false>
                  : (const void*)matern_batched_kernel<FormF32, double, 8, false>;
  } else {
    if (warps == 4) fn = f64 ? (const void*)matern_batched_kernel<FormF64, float, 4, false>
                             : (const void*)matern_batched_kernel<FormF32, float, 4, false>;
    else fn = f64 ? (const void*)matern_batched_kernel<FormF64, float, 8, false>
                  : (const void*)matern_batched_kernel<FormF32, float, 8, false>;
  }
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, warps * 32, 0) != cudaSuccess)
    return 1;
  return std::max(1, blocks);
}

// ---- autotune cache: one line per key: "<key> <warps> <ctas_per_sm> <chunk> <ms>"
std::mutex g_cache_mutex;

std::string cache_path() {
  const char* env = std::getenv("BK_AUTOTUNE_CACHE");
  if (env != nullptr) return std::string(env);
  const char* xdg = std::getenv("XDG_CACHE_HOME");
  const char* home = std::getenv("HOME");
  std::string dir;
  if (xdg != nullptr && *xdg) dir = std::string(xdg) + "/libbesselk";
  else if (home != nullptr && *home) dir = std::string(home) + "/.cache/libbesselk";
  else return std::string();
  return dir + "/autotune.txt";
}

bool cache_lookup(const std::string& key, int& warps, int& cps, int& chunk, double& ms) {
  std::lock_guard<std::mutex> lk(g_cache_mutex);
  const std::string path = cache_path();
  if (path.empty()) return false;
  FILE* f = std::fopen(path.c_str(), "r");
  if (f == nullptr) return false;
  char kbuf[256];
  int w, c, ch;
  double m;
  bool found = false;
  while (std::fscanf(f, "%255s %d %d %d %lf", kbuf, &w, &c, &ch, &m) == 5) {
    if (key == kbuf) {  // the last entry for a key wins
      warps = w;
      cps = c;
      chunk = ch;
      ms = m;
      found = true;
    }
  }
  std::fclose(f);
  return found;
}

void cache_store(const std::string& key, int warps, int cps, int chunk, double ms) {
  std::lock_guard<std::mutex> lk(g_cache_mutex);
  const std::string path = cache_path();
  if (path.empty()) return;
  const size_t slash = path.find_last_of('/');
  if (slash != std::string::npos) {  // create the directory chain (best effort)
    std::string dir = path.substr(0, slash);
    for (size_t pos = 1; pos <= dir.size(); ++pos)
      if (pos == dir.size() || dir[pos] == '/') mkdir(dir.substr(0, pos).c_str(), 0755);
  }
  FILE* f = std::fopen(path.c_str(), "a");
  if (f == nullptr) return;
  std::fprintf(f, "%s %d %d %d %.6f\n", key.c_str(), warps, cps, chunk, ms);
  std::fclose(f);
}

void free_tables(bk_plan* p) {
  cudaFree(p->d_table_prefix);
  cudaFree(p->d_inst);
  cudaFree(p->d_direct);
  cudaFree(p->d_tables);
  cudaFree(p->d_order);
  p->d_order = nullptr;
  p->d_table_prefix = nullptr;
  p->d_inst = p->d_tables = nullptr;
  p->d_direct = nullptr;
}

// Whether an instance of a plan with tables is worth one.  Many tables are built
// side by side, in 2.4 us each (FP32 1.1): 300 instances of n = 300 take 763 us with
// them and 2,263 without, in FP32 347 and 859, with the learned window 347 and 753;
// 20 of them 88 and 176, 49 and 54, 49 and 62.  FP32 arithmetic into FP64 matrices
// needs FP64 tables: 20 of n = 300 88 us with, 71 without (learned 65), 40 of n = 400
// 200 and 219 (195), 40 of n = 500 212 and 310 (279).
bool batch_instance_pays(int64_t n, const bk_opts& o, bk_dtype out_t) {
  return n >= (o.compute == BK_F32 && out_t == BK_F64 ? 480 : 256);
}
// Whether a batch is worth tables: by the entries of the instances that are worth one,
// in units of 2^19, as tables cost the call about 40 us (FP32 30).  Times in us with
// tables and without: one matrix of n = 750 42, 60 (FP64), 31, 24 (FP32), 30, 21
// (learned); of n = 1,000 42, 92; 32, 33; 32, 30; FP32 arithmetic into FP64, n = 1,000
// 42, 34, n = 1,250 44, 44.  Beside smaller instances, which take a launch of their own
// then: n = 900 beside one of 30 73, 86 (FP64); n = 1,100 beside one of 100 82, 108;
// 48, 42; 47, 40; two of n = 900 81, 137; 49, 51; 48, 48; n = 2,000 beside 200 of 100
// 349, 519; 155, 185; 143, 167; FP32 into FP64 n = 1,500 beside one of 200 61, 59, three
// of n = 1,000 65, 82.
bool batch_pays(const int64_t* sizes, int32_t count, const bk_opts& o, bk_dtype out_t) {
  double entries = 0.0;
  bool smaller = false;
  for (int32_t k = 0; k < count; ++k) {
    if (batch_instance_pays(sizes[k], o, out_t)) entries += (double)sizes[k] * (double)sizes[k];
    else smaller = smaller || sizes[k] > 0;
  }
  const int least = o.compute == BK_F64 ? 1 : out_t == BK_F32 ? (smaller ? 3 : 2) : (smaller ? 5 : 3);
  return entries >= 524288.0 * least;
}

std::string make_key(const bk_plan* p) {
  cudaDeviceProp prop;
  std::string name = "gpu";
  if (cudaGetDeviceProperties(&prop, p->device) == cudaSuccess) name = prop.name;
  for (char& c : name)
    if (c == ' ') c = '_';
  int bucket = 0;
  while ((1LL << bucket) < (p->d_tables != nullptr ? p->table_tiles : p->total_tiles)) ++bucket;
  char buf[256];
  std::snprintf(buf, sizeof(buf), "%s|out%d|compute%d|win%d|tiles2^%d%s", name.c_str(),
                (int)p->dtype, (int)p->opts.compute, (int)p->opts.window, bucket,
                p->d_tables != nullptr ? "|table" : "");
  return std::string(buf);
}

}  // namespace
}  // namespace bk

using namespace bk;

extern "C" {

bk_status bk_batched_plan_create(bk_plan** plan, const int64_t* sizes, int32_t count,
                                 bk_dtype dtype, const bk_opts* opts) {
  if (plan == nullptr) return set_error(BK_ERR_INVALID_ARG, "plan is NULL");
  *plan = nullptr;
  if (count < 1) return set_error(BK_ERR_INVALID_ARG, "count must be >= 1");
  if (sizes == nullptr) return set_error(BK_ERR_INVALID_ARG, "sizes is NULL");
  if (dtype != BK_F64 && dtype != BK_F32)
    return set_error(BK_ERR_INVALID_ARG, "dtype: unknown value %d", (int)dtype);
  bk_opts o;
  bk_opts_default(&o);
  if (opts != nullptr) o = *opts; else o.compute = dtype;
  const bk_status st = check_opts(&o);
  if (st != BK_OK) return st;
  for (int32_t k = 0; k < count; ++k)
    if (sizes[k] < 0) return set_error(BK_ERR_INVALID_ARG, "sizes[%d] < 0", (int)k);
  std::vector<int64_t> prefix((size_t)count + 1, 0), table_prefix((size_t)count + 1, 0);
  std::vector<int> order;
  // Entry tables (bk_entry_table.cuh) for the forms that have them, where the batch
  // is worth them and they fit 1 GiB.  The parameters are only known at each call:
  // instances outside the tables' domain, and those too small for one, are the
  // per-entry kernel's.
  const bool table_f32 = o.compute == BK_F32 && dtype == BK_F32;
  const size_t table_bytes = (size_t)count * entry_table_bytes(table_f32);
  const bool tables = count <= 65535 && table_bytes <= ((size_t)1 << 30) &&
                      entry_table_applies(o, dtype, 1.0, 1.0, 1.0) && batch_pays(sizes, count, o, dtype);
  for (int32_t k = 0; k < count; ++k) {
    const int64_t nb = (sizes[k] + kTile - 1) / kTile, nt = batch_instance_pays(sizes[k], o, dtype) ? (sizes[k] + 63) / 64 : 0;
    prefix[(size_t)k + 1] = prefix[(size_t)k] + nb * (nb + 1) / 2;
    table_prefix[(size_t)k + 1] = table_prefix[(size_t)k] + nt * (nt + 1) / 2;
    if (nt > 0) order.push_back(k);
  }
  const int with_table = (int)order.size();
  for (int32_t k = 0; k < count; ++k)
    if (table_prefix[(size_t)k + 1] == table_prefix[(size_t)k]) order.push_back(k);
  bk_plan* p = new bk_plan();
  p->count = count;
  p->dtype = dtype;
  p->opts = o;
  p->total_tiles = prefix.back();
  p->d_prefix = nullptr;
  p->d_sizes = nullptr;
  p->d_next = nullptr;
  p->d_wnu = nullptr;
  p->table_tiles = table_prefix.back();
  p->with_table = with_table;
  p->d_order = nullptr;
  p->d_table_prefix = nullptr;
  p->d_inst = nullptr;
  p->d_tables = nullptr;
  p->d_direct = nullptr;
  p->warps = 8;
  p->chunk = 1;
  p->tuned = 0;
  p->tuned_ms = 0.0;
  cudaError_t e = cudaGetDevice(&p->device);
  if (e == cudaSuccess) e = cudaMalloc((void**)&p->d_prefix, prefix.size() * sizeof(int64_t));
  if (e == cudaSuccess) e = cudaMalloc((void**)&p->d_sizes, (size_t)count * sizeof(int64_t));
  if (e == cudaSuccess) e = cudaMalloc((void**)&p->d_next, 2 * sizeof(unsigned long long));
  if (e == cudaSuccess)
    e = cudaMemcpy(p->d_prefix, prefix.data(), prefix.size() * sizeof(int64_t),
                   cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(p->d_sizes, sizes, (size_t)count * sizeof(int64_t), cudaMemcpyHostToDevice);
  if (e == cudaSuccess && tables) {
    const size_t offsets = table_prefix.size() * sizeof(int64_t);
    if (cudaMalloc((void**)&p->d_table_prefix, offsets) != cudaSuccess ||
        cudaMalloc(&p->d_inst, (size_t)count * batched_instance_bytes()) != cudaSuccess ||
        cudaMalloc((void**)&p->d_direct, (size_t)count * sizeof(int)) != cudaSuccess ||
        cudaMalloc((void**)&p->d_order, (size_t)count * sizeof(int)) != cudaSuccess ||
        cudaMalloc(&p->d_tables, table_bytes) != cudaSuccess) {
      (void)cudaGetLastError();  // without them the per-entry kernel takes every instance
      free_tables(p);
    } else {
      e = cudaMemcpy(p->d_table_prefix, table_prefix.data(), offsets, cudaMemcpyHostToDevice);
      if (e == cudaSuccess)
        e = cudaMemcpy(p->d_order, order.data(), (size_t)count * sizeof(int), cudaMemcpyHostToDevice);
    }
  }
  // per-instance tables of e^{-2 nu h} for the searched-window FP64 forms
  // (without them, or for more than 4,096 instances, the kernel computes the
  // values itself)
  if (e == cudaSuccess && p->d_tables == nullptr && o.compute == BK_F64 && o.window != BK_WIN_FIXED &&
      o.window != BK_WIN_LEARNED && count <= 4096) {
    if (cudaMalloc((void**)&p->d_wnu, (size_t)count * kCoshTabSize * sizeof(double)) != cudaSuccess) {
      (void)cudaGetLastError();
      p->d_wnu = nullptr;
    }
  }
  if (e != cudaSuccess) {
    cudaFree(p->d_prefix);
    cudaFree(p->d_sizes);
    cudaFree(p->d_next);
    free_tables(p);
    delete p;
    return (e == cudaErrorMemoryAllocation) ? set_error(BK_ERR_NOMEM, "plan: out of device memory")
                                            : check_cuda(e, "bk_batched_plan_create");
  }
  p->ctas_per_sm = std::min(p->d_tables != nullptr ? 4 : 2, max_ctas_per_sm(p, p->warps));
  p->key = make_key(p);
  int w, c, ch;
  double ms;
  if (cache_lookup(p->key, w, c, ch, ms) && (w == 4 || w == 8) && c >= 1 && ch >= 1 &&
      c <= max_ctas_per_sm(p, w)) {
    p->warps = w;
    p->ctas_per_sm = c;
    p->chunk = ch;
    p->tuned = 1;
    p->tuned_ms = ms;
  }
  *plan = p;
  return BK_OK;
}

bk_status bk_batched_plan_destroy(bk_plan* plan) {
  if (plan == nullptr) return BK_OK;
  cudaFree(plan->d_prefix);
  cudaFree(plan->d_sizes);
  cudaFree(plan->d_next);
  cudaFree(plan->d_wnu);
  free_tables(plan);
  delete plan;
  return BK_OK;
}

bk_status bk_batched_plan_info(const bk_plan* plan, int64_t* total_tiles, int* warps,
                               int* ctas_per_sm, int* chunk, int* tuned) {
  if (plan == nullptr) return set_error(BK_ERR_INVALID_ARG, "plan is NULL");
  if (total_tiles) *total_tiles = plan->total_tiles;
  if (warps) *warps = plan->warps;
  if (ctas_per_sm) *ctas_per_sm = plan->ctas_per_sm;
  if (chunk) *chunk = plan->chunk;
  if (tuned) *tuned = plan->tuned;
  return BK_OK;
}

bk_status bk_matern_batched(const bk_matern_desc* d_descs, int32_t count, bk_dtype dtype,
                            const bk_plan* plan, bk_stream_t stream) {
  if (plan == nullptr) return set_error(BK_ERR_INVALID_ARG, "plan is NULL");
  if (count != plan->count)
    return set_error(BK_ERR_INVALID_ARG, "count %d does not match the plan (%d)", (int)count,
                     (int)plan->count);
  if (dtype != plan->dtype) return set_error(BK_ERR_INVALID_ARG, "dtype does not match the plan");
  if (d_descs == nullptr) return set_error(BK_ERR_INVALID_ARG, "d_descs is NULL");
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != plan->device)
    return set_error(BK_ERR_INVALID_ARG, "the plan belongs to device %d", plan->device);
  if (plan->total_tiles == 0) return BK_OK;
  return check_cuda(launch_batched(plan, d_descs, plan->total_tiles, plan->warps,
                                   plan->ctas_per_sm, plan->chunk, (cudaStream_t)stream),
                    "bk_matern_batched launch");
}

bk_status bk_batched_autotune(bk_plan* plan, const bk_matern_desc* d_descs, int64_t sample_tiles,
                              bk_stream_t stream) {
  if (plan == nullptr || d_descs == nullptr)
    return set_error(BK_ERR_INVALID_ARG, "plan and d_descs must be non-NULL");
  if (plan->total_tiles == 0) return BK_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t limit = (sample_tiles > 0) ? std::min(sample_tiles, plan->total_tiles)
                                           : plan->total_tiles;
  cudaEvent_t a, b;
  if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess)
    return check_cuda(cudaGetLastError(), "bk_batched_autotune events");
  float best = 1e30f;
  int bw = plan->warps, bc = plan->ctas_per_sm, bch = plan->chunk;
  const int warps_c[2] = {4, 8};
  const int chunk_c[2] = {1, 4};
  bk_status st = BK_OK;
  for (int wi = 0; wi < 2 && st == BK_OK; ++wi) {
    // CTAs per SM: 1, 2, 4, ... below the occupancy limit, and the limit itself
    const int maxc = std::min(max_ctas_per_sm(plan, warps_c[wi]), 8);
    for (int c = 1; c <= maxc && st == BK_OK; c = (c * 2 > maxc && c < maxc) ? maxc : c * 2) {
      for (int ci = 0; ci < 2 && st == BK_OK; ++ci) {
        float ms = 0.0f;
        for (int rep = 0; rep < 2; ++rep) {  // the first run warms the shape up
          cudaEventRecord(a, s);
          cudaError_t e = launch_batched(plan, d_descs, limit, warps_c[wi], c, chunk_c[ci], s);
          cudaEventRecord(b, s);
          if (e == cudaSuccess) e = cudaEventSynchronize(b);
          if (e != cudaSuccess) {
            st = check_cuda(e, "bk_batched_autotune");
            break;
          }
          cudaEventElapsedTime(&ms, a, b);
        }
        if (st == BK_OK && ms < best) {
          best = ms;
          bw = warps_c[wi];
          bc = c;
          bch = chunk_c[ci];
        }
      }
    }
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  if (st != BK_OK) return st;
  plan->warps = bw;
  plan->ctas_per_sm = bc;
  plan->chunk = bch;
  plan->tuned = 1;
  plan->tuned_ms = best;
  cache_store(plan->key, bw, bc, bch, best);
  return BK_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free batched entry point (bk_matern_batched_static).
//
// bk_batched_plan_create calls cudaMalloc for the work list and the tile
// counter.  Some callers cannot allocate device memory where they build
// their matrices: code running inside a framework that owns all device
// memory through its own pool (a cudaMalloc there can fail, or stall other
// streams while the driver maps memory), and real-time or embedded services
// that forbid allocation after start-up.  For them the same batched work runs
// with its scratch in the fixed array below, which is part of the loaded
// library image: every GPU that loads the library holds it until the process
// exits.  It fits kStaticMaxInstances instances.

namespace bk {
namespace {

constexpr int kStaticMaxInstances = 4096;
// Word layout of the scratch (8-byte words; each part starts on 256 bytes):
// [0] tile counter, [kStaticPrefixOff ...] count + 1 tile offsets,
// [kStaticSizesOff ...] count instance sizes.
constexpr int kStaticPrefixOff = 32;
constexpr int kStaticSizesOff = ((kStaticPrefixOff + kStaticMaxInstances + 1 + 31) / 32) * 32;
constexpr int kStaticWords = kStaticSizesOff + kStaticMaxInstances;

static __device__ __align__(256) unsigned long long g_static_scratch[kStaticWords];

// One block: reads each descriptor's n, writes the sizes and the tile prefix
// sums, and zeroes the tile counter (the scratch keeps the previous call's
// contents, so everything is rewritten here every call).
__global__ void __launch_bounds__(1024) static_batch_prep_kernel(
    const bk_matern_desc* __restrict__ descs, int count, unsigned long long* __restrict__ scratch) {
  int64_t* prefix = (int64_t*)(scratch + kStaticPrefixOff);
  int64_t* sizes = (int64_t*)(scratch + kStaticSizesOff);
  __shared__ int64_t part[1024];
  const int per = (count + (int)blockDim.x - 1) / (int)blockDim.x;
  const int k0 = (int)threadIdx.x * per, k1 = min(count, k0 + per);
  int64_t local = 0;
  for (int k = k0; k < k1; ++k) {
    const int64_t n = descs[k].n;
    sizes[k] = n;
    const int64_t nb = (n > 0) ? (n + kTile - 1) / kTile : 0;
    local += nb * (nb + 1) / 2;
  }
  part[threadIdx.x] = local;
  __syncthreads();
  for (int off = 1; off < (int)blockDim.x; off <<= 1) {  // inclusive scan of the partial sums
    const int64_t v = ((int)threadIdx.x >= off) ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int64_t run = (threadIdx.x == 0) ? 0 : part[threadIdx.x - 1];
  for (int k = k0; k < k1; ++k) {
    prefix[k] = run;
    const int64_t n = sizes[k];
    const int64_t nb = (n > 0) ? (n + kTile - 1) / kTile : 0;
    run += nb * (nb + 1) / 2;
  }
  if (threadIdx.x == blockDim.x - 1) prefix[count] = part[blockDim.x - 1];
  if (threadIdx.x == 0) scratch[0] = 0ull;
}

// The persistent kernel of bk_matern_batched, with its work list, tile total
// and counter taken from the static scratch (filled by the preparation
// kernel earlier on the same stream).
template <class Form, typename OutT, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, Form::kMinBlocks * 8 / WARPS) matern_batched_static_kernel(
    const bk_matern_desc* __restrict__ descs, int count, unsigned long long* __restrict__ scratch) {
  const int64_t* prefix = (const int64_t*)(scratch + kStaticPrefixOff);
  const int64_t limit = prefix[count];
  __shared__ BatchSmem<OutT> sm;
  __shared__ double s_tab[Form::kStageTable ? kExpTabSize : 1];
  const Form f = bind_table(Form{}, s_tab);
  Tally tl{0u, 0u, 0u, 0u, 0u, 0u, 0u};
  unsigned evals = 0;
  int cur = -1;
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) sm.item = (int64_t)atomicAdd(scratch, 1ull);
    __syncthreads();
    const int64_t w = sm.item;
    if (w >= limit) break;
    const int k = find_instance(prefix, count, w);
    if (k != cur) {
      __syncthreads();
      if (threadIdx.x == 0) {
        bk_matern_desc d = descs[k];
        // sizes[k] was copied from this descriptor by the preparation kernel,
        // so only the descriptor's own fields need checking here.  There are
        // no counters on this path: a skipped descriptor leaves its output
        // untouched and is not reported.
        const bool ok = d.n >= 0 && d.ld >= d.n && d.locs != nullptr && d.out != nullptr &&
                        d.beta > 0.0 && d.nu > 0.0 && d.sigma2 >= 0.0;
        if (!ok) d.n = 0;  // an invalid descriptor is skipped
        sm.locs = d.locs;
        sm.out = (OutT*)d.out;
        sm.n = d.n;
        sm.ld = d.ld;
        sm.mp = matern_params(d.sigma2, d.beta, d.nu);
      }
      __syncthreads();
      cur = k;
    }
    int64_t I, J;
    tri_tile(w - prefix[k], I, J);
    __syncthreads();
    sym_tile<Form, OutT, WARPS>(f, sm.tile, sm.locs, sm.n, I, J, sm.mp, sm.out, sm.ld, tl,
                                evals);
  }
}

// Device address of the scratch on the current device.  The array's name in
// host code is only a host-side handle, so the address is looked up with
// cudaGetSymbolAddress on every call (a host-side lookup once the library's
// device code is loaded on the device; the first call on a device also loads
// it there).  Not caching it keeps the address right after the context is
// torn down and created again (cudaDeviceReset), when the array may move.
bk_status static_scratch_address(unsigned long long** out) {
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
  if (e != cudaSuccess) return check_cuda(e, "bk_matern_batched_static: cudaGetSymbolAddress");
  *out = (unsigned long long*)p;
  return BK_OK;
}

}  // namespace
}  // namespace bk

extern "C" bk_status bk_matern_batched_static(const bk_matern_desc* d_descs, int32_t count,
                                              bk_dtype dtype, bk_stream_t stream) {
  using namespace bk;
  if (count < 1 || count > kStaticMaxInstances)
    return set_error(BK_ERR_INVALID_ARG,
                     "bk_matern_batched_static: count must be in [1, %d] (got %d); use a plan "
                     "(bk_batched_plan_create) for larger batches",
                     kStaticMaxInstances, (int)count);
  if (d_descs == nullptr) return set_error(BK_ERR_INVALID_ARG, "d_descs is NULL");
  if (dtype != BK_F64 && dtype != BK_F32)
    return set_error(BK_ERR_INVALID_ARG, "dtype: unknown value %d", (int)dtype);
  unsigned long long* scratch = nullptr;
  bk_status st = static_scratch_address(&scratch);
  if (st != BK_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  static_batch_prep_kernel<<<1, 1024, 0, s>>>(d_descs, count, scratch);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return check_cuda(e, "bk_matern_batched_static: preparation launch");
  const int grid = current_sm_count() * 2;
  if (dtype == BK_F64)
    matern_batched_static_kernel<FormF64, double, 8><<<grid, 256, 0, s>>>(d_descs, count, scratch);
  else
    matern_batched_static_kernel<FormF32, float, 8><<<grid, 256, 0, s>>>(d_descs, count, scratch);
  return check_cuda(cudaGetLastError(), "bk_matern_batched_static launch");
}
