// Host launcher of the Q-less Householder TSQR (paper Sec. 3.2, Algorithms 2-4).
//
// One persistent launch per call: CTA i factors tiles [t0_i, t1_i) of X into its triangle
// (tsqr.cuh), stores it as leaf i of a binary R-tree and climbs the tree; the CTA that
// completes the root writes R (or solves the least-squares problem of [A b]).  When the
// double-float launch finds data outside its exponent range it leaves R unwritten and
// raises a flag; the FP64 launch queued behind it runs only in that case.
#include <atomic>
#include <cstdlib>

#include "tsqr_launch.cuh"

namespace ql {

int tsqr_variant() {
  static const int v = [] {
    const char* e = std::getenv("QL_TSQR_CFG");
    return e ? std::atoi(e) : 0;
  }();
  return v;
}

int device_slot() {
  int dev = 0;
  return cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices ? 0 : dev;
}

int device_sm_count() {
  // cached per device: a process may drive GPUs with different SM counts
  static std::atomic<int> sms[kMaxDevices] = {};
  const int dev = device_slot();
  int v = sms[dev].load(std::memory_order_relaxed);
  if (v > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 1;
  sms[dev].store(v, std::memory_order_relaxed);
  return v;
}

static __global__ void __launch_bounds__(256) clear_kernel(uint4* p, unsigned n) {
  pdl_release();
  const unsigned i = blockIdx.x * 256 + threadIdx.x;
  if (i < n) p[i] = make_uint4(0, 0, 0, 0);
}
ql_status clear_async(void* p, size_t bytes, cudaStream_t st) {
  const unsigned n = (unsigned)(bytes / 16);
  count_launch();
  clear_kernel<<<(n + 255) / 256, 256, 0, st>>>(static_cast<uint4*>(p), n);
  return cudaPeekAtLastError() == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

// Workspace: the exact Gram pass's block (its head, the flags, is shared by every launch of
// the call) unless the call is Householder only, then the tree's counters and slots.
constexpr size_t kFlagBytes = 512;

static size_t counter_bytes() {
  const size_t cnt = tree_counters(device_sm_count() * kMaxCtasPerSm);
  return (cnt * sizeof(int) + 255) / 256 * 256;
}

size_t tsqr_workspace_bytes(int n, bool householder) {
  if (n < 1 || n > kMaxN) return 0;
  const size_t leaves = (size_t)device_sm_count() * kMaxCtasPerSm;
  return counter_bytes() + (householder || n < 2 ? kFlagBytes : xgram_tsqr_bytes(n)) +
         tree_slots((int)leaves) * (size_t)n * n * sizeof(double);
}

// Whether the exact Gram pass (xgram.cuh) takes a TSQR call.  Below the line one Householder tile
// per CTA and a one-level tree are the shorter chain.  Measured, Householder and exact, us:
//   R:             3 columns 2048 rows 22.7, 24;  4096 24.7, 24;  8192 27.1, 25;  16384 35, 25
//                  4 columns 2048 rows 25.6, 25;  4096 28.3, 25;  16384 45, 25
//                  5 columns  100 rows 28.8, 27;  2048 39, 28
//   least squares: 3 columns 4096 rows 27, 30;    8192 32, 30;    16384 39, 30
//                  4 columns 4096 rows 32, 31;    8192 35, 31
//                  5 columns 1024 rows 30, 36;    2048 40, 34
//                  6 columns 1024 rows 33, 38;    2048 44, 37;    9 columns 100 rows 48, 45
// One or two columns stay with the norm and the Householder tiles: the 4-column class works for two
// columns that are not there (m = 2^25, n = 2 288 us against 378).  With fewer rows than columns the
// exact pass would factor twice (dependent columns), where a single tile is quick.
static bool exact_route(const TsqrCall& c, ql_arith arith) {
  if (c.householder || arith == QL_ARITH_F64 || !tc_gram_enabled() || c.n < 3 || c.m < c.n) return false;
  if (c.epilogue == kEpiR) return c.n >= 5 || c.m >= (1 << 12);
  return c.n >= 7 || c.m >= (c.n >= 5 ? 1 << 11 : 1 << 13);
}

bool tsqr_exact_route(int64_t m, int n) {
  TsqrCall c;
  c.m = m;
  c.n = n;
  return exact_route(c, current_arith());
}

template <typename S>
static ql_status tsqr_launch_s(const TsqrCall& c, const TreeView& tv, bool exact, ql_arith arith) {
  if (arith == QL_ARITH_F64) return dispatch<S, ArithF64>(c, tv, 0);
  ql_status st = dispatch<S, ArithDF>(c, tv, exact ? 2 : 0);
  if (st != QL_OK) return st;
  return dispatch<S, ArithF64>(c, tv, 1);
}

ql_status tsqr_launch(const TsqrCall& c, ql_arith arith) {
  if (c.n < 1 || c.n > kMaxN) return QL_ERR_ARG;
  if (!c.ws || c.ws_bytes < tsqr_workspace_bytes(c.n, c.householder)) return QL_ERR_WORKSPACE;
  const bool exact = exact_route(c, arith);
  // [tree counters][flags (head of the exact pass's block)][slots]
  unsigned char* ws = static_cast<unsigned char*>(c.ws);
  const size_t cb = counter_bytes(), xb = c.householder || c.n < 2 ? kFlagBytes : xgram_tsqr_bytes(c.n);
  TreeView tv;
  tv.counters = reinterpret_cast<int*>(ws);
  tv.flags = reinterpret_cast<int*>(ws + cb);
  tv.slots = reinterpret_cast<double*>(ws + cb + xb);
  tv.leaves = 0;
  if (exact) {
    ql_status st = clear_async(ws, cb + xgram_tsqr_clear_bytes(c.n), c.stream);
    if (st == QL_OK) st = xgram_tsqr_launch(c, ws + cb);
    if (st != QL_OK) return st;
  } else if (cudaMemsetAsync(ws, 0, cb + kFlagBytes, c.stream) != cudaSuccess) {
    return QL_ERR_CUDA;
  }
  return c.dtype == QL_F64 ? tsqr_launch_s<double>(c, tv, exact, arith) : tsqr_launch_s<float>(c, tv, exact, arith);
}

}  // namespace ql
