// Host-side internal interfaces between the C ABI (api.cu) and the kernel translation
// units.  Not part of the public boundary.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/qless.h"

namespace ql {

// Epilogue selected for the root of a TSQR / the last CTA of a Gram pass.
enum Epilogue : int { kEpiR = 0, kEpiLstsq = 1 };

struct TsqrCall {
  int64_t m = 0;
  int n = 0;            // columns factored (n + 1 for least squares)
  int nA = 0;           // columns taken from A; column nA (if < n) comes from b
  const void* A = nullptr;
  int64_t lda = 0;
  const void* b = nullptr;
  ql_dtype dtype = QL_F64;
  int epilogue = kEpiR;
  double* R = nullptr;  // kEpiR: n x n output (ldr)
  int64_t ldr = 0;
  double* x = nullptr;  // kEpiLstsq: solution (n - 1 entries)
  double* resnorm = nullptr;
  double* Rext = nullptr;  // kEpiLstsq: optional n x n R_ext (ld n)
  int32_t* info = nullptr;
  void* ws = nullptr;
  size_t ws_bytes = 0;
  cudaStream_t stream = nullptr;
  int ctas_per_sm = 0;  // 0: occupancy maximum
  int max_ctas = 0;     // 0: no limit (testing the R-tree with few leaves)
  int variant = -1;     // thread layout (row-block height) for n > 8: -1 environment default, 0..2
  int arity = 0;        // R-tree arity: 0 the column class's default, else 2 .. default
  bool householder = false;  // Householder tiles only (no exact Gram pass)
};

// Upper bound of the TSQR workspace for n columns (any m); householder: without the exact
// Gram pass.
size_t tsqr_workspace_bytes(int n, bool householder = false);
// The exact Gram pass as a TSQR call's first launch (gram.cu): workspace, the leading bytes
// of it to clear, and the launch.
size_t xgram_tsqr_bytes(int n);
size_t xgram_tsqr_clear_bytes(int n);
ql_status xgram_tsqr_launch(const TsqrCall& c, void* base);
// Whether ql_tsqr_qless of m rows and n columns starts with that pass.
bool tsqr_exact_route(int64_t m, int n);
// Columns of the workspace-free entry point (tsqr_noalloc.cu), always on Householder tiles.
constexpr int kNoAllocMaxN = 16;
// Launch the double-float TSQR (or FP64 when arith == QL_ARITH_F64) and, after a
// double-float launch, the gated FP64 fallback.
ql_status tsqr_launch(const TsqrCall& c, ql_arith arith);

struct GramCall {
  int64_t m = 0;
  int n = 0;
  int nA = 0;
  const void* A = nullptr;
  int64_t lda = 0;
  const void* b = nullptr;
  ql_dtype dtype = QL_F64;
  int method = QL_CHOLQR2;  // QL_CHOLQR2 or QL_SVQB2
  int epilogue = kEpiR;
  double* R = nullptr;
  int64_t ldr = 0;
  double* Z = nullptr;
  double rank_tol = 0.0;
  double* x = nullptr;
  double* resnorm = nullptr;
  double* Rext = nullptr;
  int32_t* info = nullptr;
  void* ws = nullptr;
  size_t ws_bytes = 0;
  cudaStream_t stream = nullptr;
};
size_t gram_workspace_bytes(int n);
ql_status gram_launch(const GramCall& c, ql_arith arith);

// SM count of the current device (cached per device).
int device_sm_count();
// The current device's index below kMaxDevices, for what is set up or cached once per device (a
// kernel's shared-memory limit and occupancy hold for the device that was current).
constexpr int kMaxDevices = 64;
int device_slot();
ql_arith current_arith();

// Largest n any entry point accepts.
constexpr int kApiMaxN = 64;
// Argument checks shared by the entry points (no device work): m >= 0, 1 <= n <= nmax, a
// known dtype, ld >= max(m, 1), X non-null when m > 0 (QL_ERR_ARG), X aligned to its
// element size (QL_ERR_ALIGN).
bool elem_aligned(const void* p, ql_dtype dt);
ql_status check_matrix(int64_t m, int64_t n, const void* X, ql_dtype dt, int64_t ld, int nmax);
// Output triangle R: non-null with ldr >= n (QL_ERR_ARG), 8-byte aligned (QL_ERR_ALIGN).
ql_status check_r(const double* R, int64_t ldr, int64_t n);
// Whether the tensor-core kernels are used (double-float mode): the exact pass, of TSQR calls too,
// and the later Gram passes from 9 columns; the environment variable QL_GRAM_SIMT=1 selects the
// Householder tiles and the SIMT Gram kernels instead.
bool tc_gram_enabled();
// First Gram pass of the Gram methods' 16-, 32- and 64-column classes, and the batched form, on the
// exact kernel (default; QL_GRAM_PIPE=0 selects the per-tile kernels, for comparison; TSQR calls and
// the Gram methods of up to 8 columns stay on the exact kernel).
bool pipe_gram_enabled();
// QL_GRAM_PIPE2=0: the later Gram passes of n <= 32 run on the per-tile mma.sync kernel instead
// of the pipelined one (A/B comparisons).
bool pipe_gram2_enabled();
// Tensor maps of the columns of [A b] for the pipelined Gram pass: A as a rank-2 tensor (rows
// innermost, stride lda; boxes of 128 bytes of rows x all its columns, 128-byte swizzle) and
// b as one unswizzled column; rows past m read as zeros.  tmB may be null (no b).  False, with the maps left
// unset, if the data does not allow tensor copies (a column not 16-byte aligned, m >= 2^31)
// or the driver offers no encoder; the caller then reads X without them.
bool pipe_tensor_maps(CUtensorMap* tmA, CUtensorMap* tmB, const void* A, const void* b, int dtype, int64_t m, int nA,
                      int64_t lda);

// Tensor map of the exact Gram pass (xgram.cuh): A as rank 3 (128 bytes of rows, columns, row
// blocks; 128-byte swizzle) whose box is a whole tile of 4096 / nc rows x nc columns (columns
// past nA read as zeros).  False if the data does not allow tensor copies of its full tiles
// (a column, or b unless it is null, not 16-byte aligned; m >= 2^31).
bool xg_tensor_map(CUtensorMap* map, int nc, const void* A, const void* b, int dtype, int64_t m, int nA, int64_t lda);

// Thread-layout variant of the TSQR kernels (environment QL_TSQR_CFG, 0 = default).
int tsqr_variant();

// Launch a kernel that may start while its predecessor in the stream still runs; it calls
// pdl_wait (common.cuh) before it touches anything the predecessor writes.
template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kern)(P...), int grid, int block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}
// Zero `bytes` (a multiple of 16, at a 16-byte boundary) on the stream, by a kernel that lets
// the next one start early.
ql_status clear_async(void* p, size_t bytes, cudaStream_t st);

// Counts every kernel this library launches (reported by ql_launch_count()).
void count_launch();
// dst = the first nonzero {status, index} pair among src[0 .. count) (one tiny launch).
ql_status first_status_async(int32_t* dst, const int32_t* src, int count, cudaStream_t stream);

// Autotune table lookup for an (m, n, dtype, kappa) class: method, TSQR CTAs per SM, thread
// layout and R-tree arity (null outputs are skipped).
bool tune_lookup(int64_t m, int64_t n, ql_dtype dt, double kappa, int* method, int* ctas, int* variant = nullptr,
                 int* arity = nullptr);

// Batched path, asynchronous plan upload through pinned staging (serving loop).
ql_status batch_prepare_async(int32_t count, const ql_problem* probs, void* ws, size_t ws_bytes, cudaStream_t st,
                              unsigned char* pinned, size_t pinned_bytes);
size_t batch_plan_upload_bytes(int32_t count, const ql_problem* probs);

}  // namespace ql
