// Grouped exact Gram launch of the batched form: every CTA claims (problem, chunk) work items
// from one atomic counter and runs the single-call body (xgram.cuh) of the problem's column
// class and storage on that chunk's tiles; the last chunk of a problem factors its Gram matrix
// and writes R.  One launch serves every class, so a batch of any mix costs one launch, and the
// factorisation of one problem overlaps with the tiles of the others.
#include "batch_gram.h"
#include "xgram.cuh"

namespace ql {

template <int NC, typename S>
QL_DEV void xg_item(const XgItem& it, int chunk, uint32_t tbase, PipeBars& bars, double* acc) {
  GramArgs<S> a = *reinterpret_cast<const GramArgs<S>*>(&it.args);
  a.w.fbuf = acc;
  xgram_body<NC, S>(a, chunk, it.nchunks, tbase, bars, &it.map, 0);
}
template <typename S>
QL_DEV void xg_dispatch(const XgItem& it, int chunk, uint32_t tbase, PipeBars& bars, double* acc) {
  switch (it.nc) {
    case 4: xg_item<4, S>(it, chunk, tbase, bars, acc); break;
    case 8: xg_item<8, S>(it, chunk, tbase, bars, acc); break;
    case 16: xg_item<16, S>(it, chunk, tbase, bars, acc); break;
    case 32: xg_item<32, S>(it, chunk, tbase, bars, acc); break;
    default: xg_item<64, S>(it, chunk, tbase, bars, acc); break;
  }
}

constexpr size_t kGroupBytes = (XgSmem<64, double>::kBytes + 15) / 16 * 16 + 32;
static_assert(kGroupBytes <= 232448, "shared memory of one SM");

// Last item whose work_begin <= v (items ordered by work_begin).
QL_DEV int item_of(const XgItem* items, int count, int64_t v) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (items[mid].work_begin <= v)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

__global__ void __launch_bounds__(XgShape<64>::T, 1)
    xgram_group_kernel(int* counter, const XgItem* items, int count, int64_t total, double* acc, int max_nc) {
  extern __shared__ __align__(1024) unsigned char smem_umma[];
  int64_t* s_work = reinterpret_cast<int64_t*>(smem_umma + kGroupBytes - 32);
  int* s_item = reinterpret_cast<int*>(s_work + 1);
  // tensor memory and the barriers once per CTA, at the same place in every class
  const uint32_t tbase = xg_cta_begin<64, double>(smem_umma);
  PipeBars bars;
  double* my_acc = acc + (size_t)blockIdx.x * (xg_acc_bytes(max_nc) / sizeof(double));
  while (bars.ok) {  // a CTA whose bounded wait gave up takes no more work
    if (threadIdx.x == 0) {
      const int64_t v = atomicAdd(counter, 1);
      *s_work = v;
      *s_item = item_of(items, count, v);
    }
    __syncthreads();
    const int64_t w = *s_work;
    const XgItem& it = items[*s_item];
    __syncthreads();
    if (w >= total) break;
    const int chunk = (int)(w - it.work_begin);
    if (it.dtype == QL_F64)
      xg_dispatch<double>(it, chunk, tbase, bars, my_acc);
    else
      xg_dispatch<float>(it, chunk, tbase, bars, my_acc);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
  if (!bars.ok && threadIdx.x == 0) {
    // Should every CTA give up, nobody would claim the rest and its problems would have neither an
    // answer nor a redo: hand what is left to the gated launch.
    for (int64_t v = atomicAdd(counter, 1); v < total; v = atomicAdd(counter, 1)) {
      const GramArgs<double>& a = items[item_of(items, count, v)].args;
      gram_request_redo(a.redo, a.redo_any, 1, a.method == QL_TSQR ? kRedoDF : kRedoF64);
    }
  }
  tc_fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 0) tmem_dealloc(tbase, 512);
}

ql_status xgram_group_launch(int* counter, const XgItem* items, int count, int64_t total, int grid, double* acc,
                             int max_nc, cudaStream_t st) {
  if (count < 1 || total < 1) return QL_OK;
  static std::mutex mu;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (cudaFuncSetAttribute(xgram_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGroupBytes) !=
        cudaSuccess)
      return QL_ERR_CUDA;
  }
  count_launch();
  xgram_group_kernel<<<grid, XgShape<64>::T, kGroupBytes, st>>>(counter, items, count, total, acc, max_nc);
  return cudaPeekAtLastError() == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

}  // namespace ql
