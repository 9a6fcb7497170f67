// Internal declarations shared by the library's translation units (not part
// of the public C-ABI in include/bk.h).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "bk.h"

namespace bk {

// Number of SMs of the current device (cached per device ordinal).
int current_sm_count();

// Records a message for bk_last_error() on this thread and returns `st`.
bk_status set_error(bk_status st, const char* fmt, ...);

// Converts a CUDA error into BK_ERR_CUDA with a message (BK_OK if none).
bk_status check_cuda(cudaError_t e, const char* what);

// A range of block-columns [j0, j1) of a symmetric matrix (64-wide blocks),
// written in block-column order; j1 < 0 means the whole matrix.  fill_table:
// whether a launch refills the caller's tables (e^{-2 nu h}, or the entry
// table; a caller writing several ranges of one matrix fills them with the
// first).  host: the matrix is in host memory.
struct SymRange {
  int64_t j0 = 0, j1 = -1;
  bool fill_table = true;
  bool host = false;
};

// ---- plain FP64 form (bk_plain.cu) ----
cudaError_t launch_eval_f64(const double* x, const double* nu, void* out, void* log_out,
                            bk_dtype out_t, int64_t n, const bk_opts& o, cudaStream_t s);

// Full symmetric n x n matrix: lower-triangle tiles, each written twice.
cudaError_t launch_matern_sym_f64(const double* locs, int64_t n, double sigma2, double beta,
                                  double nu, void* out, int64_t ld, bk_dtype out_t,
                                  const bk_opts& o, cudaStream_t s,
                                  const SymRange& range = SymRange{});

// General m x n block between two location sets.
cudaError_t launch_matern_block_f64(const double* locs1, int64_t m, const double* locs2,
                                    int64_t n, double sigma2, double beta, double nu, void* out,
                                    int64_t ld, bk_dtype out_t, const bk_opts& o, cudaStream_t s);

// K, dK/dx, dK/dnu of the plain form (outputs may be null).
cudaError_t launch_eval_grad_f64(const double* x, const double* nu, double* k, double* dkdx,
                                 double* dkdnu, int64_t n, const bk_opts& o, cudaStream_t s);

// The Gaussian log-likelihood steps (Cholesky, log det, forward
// substitution, reduction) on `s`; see bk_gaussian_loglik.
cudaError_t launch_loglik(double* a, int64_t n, int64_t ld, const double* z, double* y,
                          double* out, unsigned long long* ctr, cudaStream_t s);

// The same with the Cholesky factorisation in fixed point (bk_chol_fixed.cu);
// work: loglik_workspace_bytes(n), 256-byte aligned.
size_t loglik_workspace_bytes(int64_t n);
cudaError_t launch_loglik_fixed(double* a, int64_t n, int64_t ld, const double* z, double* y,
                                double* out, unsigned long long* ctr, void* work, cudaStream_t s);

// ---- writers with a per-call entry table (bk_entry_table.cu) ----
// Bytes of a table with FP64 or FP32 records.
size_t entry_table_bytes(bool f32);
// Whether a matrix of this size is worth a table, and whether the options and
// parameters are inside the tables' domain.
bool entry_table_pays(int64_t rows, int64_t cols);
bool entry_table_applies(const bk_opts& o, bk_dtype out_t, double sigma2, double beta, double nu);
// A batch of matrices with tables (bk_batched.cu's plans): device arrays of
// the plan, `instances` of batched_instance_bytes() and `tables` of
// entry_table_bytes() per instance, prefix sums over the tiles of 64 of the
// instances that may have a table, two tile counters (the second of the per-entry
// kernel), and what that kernel is to take: direct[k] != 0 for valid instances
// without a table, whose e^{-2 nu h} then stand in place of the table (decay).
struct BatchTable {
  int count;
  int with_table;    // instances that may have one
  const int* order;  // all instances, those first
  const int64_t* prefix;
  const int64_t* sizes;
  unsigned long long* next;
  int* direct;
  void* instances;
  void* tables;
  bool decay;
};
size_t batched_instance_bytes();
cudaError_t launch_batched_table(const BatchTable& b, const bk_matern_desc* descs, bool f32,
                                 bk_dtype out_t, int64_t limit, int warps, int ctas_per_sm, int chunk,
                                 cudaStream_t s);
int batched_table_max_ctas(bool f32, bk_dtype out_t, int warps);

// The scratch of one Matern call: the plain form's e^{-2 nu h} table, or the entry
// table when the matrix is worth one.  matern_scratch returns the place of the entry
// table when the call takes it, else null, with o.d_cosh_table set to the scratch
// when it fits and the caller gave none.
constexpr size_t kDecayTableBytes = (size_t)BK_COSH_TABLE_LEN * sizeof(double);
size_t matern_scratch_bytes(bool table);
void* matern_scratch(bk_opts& o, bk_dtype out_t, int64_t rows, int64_t cols, double sigma2, double beta, double nu,
                     void* d_work, size_t work_bytes);
// The writers of launch_matern_sym_* and launch_matern_block_* with a table in
// device memory (16-byte aligned, entry_table_bytes of the records: FP32 when
// compute and output are FP32).
cudaError_t launch_matern_sym_table(const double* locs, int64_t n, double sigma2, double beta,
                                    double nu, void* out, int64_t ld, bk_dtype out_t,
                                    bk_dtype compute, void* table, cudaStream_t s,
                                    const SymRange& range = SymRange{});
cudaError_t launch_matern_block_table(const double* locs1, int64_t m, const double* locs2, int64_t n,
                                      double sigma2, double beta, double nu, void* out, int64_t ld,
                                      bk_dtype out_t, bk_dtype compute, void* table, cudaStream_t s);

// Option checks shared by every entry point that takes bk_opts (sets the
// error message and returns the status).
bk_status check_opts(const bk_opts* o);

// Lanes per evaluation of the FP32 forms' bare evaluations: opts.lanes, else
// bk_eval_autotune's choice for the current device, else the default.
int eval_lanes(const bk_opts& o, bk_dtype out_dtype);

// ---- FP32 precision form (bk_fp32.cu) ----
cudaError_t launch_eval_f32(const double* x, const double* nu, void* out, void* log_out,
                            bk_dtype out_t, int64_t n, unsigned long long* ctr, cudaStream_t s,
                            int lanes);
cudaError_t launch_matern_sym_f32(const double* locs, int64_t n, double sigma2, double beta,
                                  double nu, void* out, int64_t ld, bk_dtype out_t,
                                  unsigned long long* ctr, cudaStream_t s,
                                  const SymRange& range = SymRange{});
cudaError_t launch_matern_block_f32(const double* locs1, int64_t m, const double* locs2,
                                    int64_t n, double sigma2, double beta, double nu, void* out,
                                    int64_t ld, bk_dtype out_t, unsigned long long* ctr,
                                    cudaStream_t s);

// ---- learned window (bk_learned.cu); `m` must have weights (learned_ready)
bool learned_ready(const bk_learned* m);
cudaError_t launch_eval_learned(const bk_learned* m, const double* x, const double* nu, void* out,
                                void* log_out, bk_dtype out_t, int64_t n, unsigned long long* ctr,
                                cudaStream_t s, int lanes);
cudaError_t launch_matern_sym_learned(const bk_learned* m, const double* locs, int64_t n,
                                      double sigma2, double beta, double nu, void* out, int64_t ld,
                                      bk_dtype out_t, unsigned long long* ctr, cudaStream_t s,
                                      const SymRange& range = SymRange{});
cudaError_t launch_matern_block_learned(const bk_learned* m, const double* locs1, int64_t m_,
                                        const double* locs2, int64_t n, double sigma2,
                                        double beta, double nu, void* out, int64_t ld,
                                        bk_dtype out_t, unsigned long long* ctr, cudaStream_t s);

}  // namespace bk
