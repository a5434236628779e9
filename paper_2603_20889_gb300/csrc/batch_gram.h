// Grouped tensor-core Gram passes of the batched form (see batch_gram.cu).
#pragma once

#include "gram_launch.cuh"

namespace ql {

// One Gram-method problem of a grouped launch: its single-call arguments (float storage has
// the same layout), the first work index of its chunks in the launch and their number, and
// the tensor maps of its columns for the pipelined first pass (see pipe_tensor_maps).
struct GramGroupItem {
  GramArgs<double> args;
  int64_t work_begin;
  int nchunks;
  int tma;          // tmA (and tmB for least squares) are valid
  CUtensorMap tmA;  // 64-byte aligned: the item array is uploaded as it is laid out here
  CUtensorMap tmB;
};

// One problem of the grouped exact Gram launch (xgram.cuh): the arguments of a single call, the
// tensor map of its tiles, its column class and storage, and its chunks' place in the work list.
struct XgItem {
  GramArgs<double> args;
  int64_t work_begin;
  int nchunks;
  int nc;           // 4, 8, 16, 32 or 64
  int dtype;
  CUtensorMap map;  // 64-byte aligned
};
// One persistent launch over every problem's chunks.  acc: the 128-bit sums, one block of
// xg_acc_bytes(largest nc) per CTA; grid: the number of CTAs (blocks).
ql_status xgram_group_launch(int* counter, const XgItem* items, int count, int64_t total, int grid, double* acc,
                             int max_nc, cudaStream_t st);
constexpr size_t xg_acc_bytes(int nc) { return (size_t)nc * 128 * 16; }

// One persistent launch over `count` items (total work = their chunks) of column class nc
// (16, 32 or 64) and storage dtype, for pass 1 (Gram of X) or 2 (Gram of X M).
ql_status gram_group_launch(int nc, int dtype, int pass, int* counter, const GramGroupItem* items, int count,
                            int64_t total, cudaStream_t st);
// Rows per tile of the grouped kernels of column class nc.
int gram_group_tile_rows(int nc);

}  // namespace ql
