// Q reconstruction: Q = X R^{-1}, the orthonormal factor of X = Q R from the R that any of
// the Q-less calls returned (the explicit Q of Sec. 1 that block iterative solvers use).
//
// One launch.  Every CTA inverts R (FP64, shared memory; n <= 64 so this is cheap); then each
// warp streams blocks of 64 rows by itself: a thread owns two adjacent rows, fetches them eight
// columns at a time (16-byte loads, all in flight at once), converts them once to double-float
// (its own words of shared memory, so no barrier and the warps drift apart), and forms its rows
// of Q = X M eight columns at a time from the M rows above the diagonal, two columns per packed
// FP32 instruction.  A block whose X or whose M lies outside the double-float exponent range is
// formed in FP64 instead (decided per warp), so no second launch and no workspace are needed.
//
// Bound: 13 FP32 operations per product and row (m = 2^23, n = 16: 378 us at the measured FP32
// rate, against 323 us of HBM).  Measured there 1638 us with one row per thread, a column fetched
// at a time and block-wide tiles, 1190 us now; 4000000 x 32 2393 -> 1430 us, 2097152 x 64 5015 ->
// 3994 us, 4000001 x 8 381 -> 263 us; few rows, spread over the SMs, 1000 x 31 68 -> 61 us; FP32
// 1048576 x 64 1760 -> 1305 us.  What is left is latency (fixed-latency stalls at 5 to 24
// warps per SM) and the conversions of X and of the results (three FP64-pipe instructions each,
// 640 us of that pipe at n = 16, overlapped; assembling the doubles with integer instructions
// instead measured slower, 1605 us).
#include <mutex>

#include "df2.cuh"
#include "internal.h"
#include "small_dense.cuh"

namespace ql {

template <typename S>
struct QformArgs {
  int64_t m;
  int n;
  const S* X;
  int64_t ldx;
  const double* R;
  int64_t ldr;
  S* Q;
  int64_t ldq;
  int32_t* info;
  int64_t tiles;  // blocks of 64 rows
  int cta_step, warp_step;  // first block of a warp = CTA x cta_step + warp x warp_step
  int pair;       // two adjacent rows of every column can be read and written in one access
};

template <int NC, typename S>
struct QformSmem {
  // one CTA per SM of as many warps as the shared memory holds (32 and 16 KB each for FP64) at 64
  // and 32 columns, else three of eight warps
  static constexpr int T = NC == 64 ? (sizeof(S) == 8 ? 160 : 320) : (NC == 32 ? 384 : 256);
  static constexpr int kCtas = NC <= 16 ? 3 : 1;
  static constexpr int LDM = NC + 1;                         // odd stride: column walks of the inverse
  static constexpr size_t kM = 8 * (size_t)NC * LDM;         // FP64 M = R^{-1}
  static constexpr size_t kMd = 8 * (size_t)NC * NC;         // double-float M, [k][column pair]
  static constexpr size_t kX = 2 * sizeof(S) * (size_t)NC * T;  // two rows per thread, [k][thread]: (hi, lo) or FP32
  static constexpr size_t kOffMd = (kM + 15) / 16 * 16;
  static constexpr size_t kOffX = kOffMd + kMd;
  static constexpr size_t kOffMisc = kOffX + kX;
  static constexpr size_t kBytes = kOffMisc + 64;
  static_assert(kBytes <= 232448, "shared memory of one SM");
  static_assert(kX >= 8 * (size_t)NC * LDM, "R fits in the row area");
};

template <int NC, typename S>
__global__ void __launch_bounds__(QformSmem<NC, S>::T, QformSmem<NC, S>::kCtas) qform_kernel(QformArgs<S> a) {
  using Sm = QformSmem<NC, S>;
  constexpr int T = Sm::T, LDM = Sm::LDM;
  extern __shared__ __align__(16) unsigned char smem[];
  double* Mf = reinterpret_cast<double*>(smem);
  df2* Md = reinterpret_cast<df2*>(smem + Sm::kOffMd);
  using X2 = typename std::conditional<sizeof(S) == 8, float4, float2>::type;  // both rows: (hi, lo) each, or FP32
  X2* xs = reinterpret_cast<X2*>(smem + Sm::kOffX);
  int* misc = reinterpret_cast<int*>(smem + Sm::kOffMisc);
  const int tid = threadIdx.x, n = a.n;

  // ---- M = R^{-1} (FP64).  A zero diagonal entry (rank-deficient R) gives no inverse.
  double* Rs = reinterpret_cast<double*>(smem + Sm::kOffX);  // the tile area is free here
  if (tid == 0) misc[0] = NC + 1;
  __syncthreads();
  for (int e = tid; e < n * n; e += T) {
    const int i = e % n, j = e / n;
    const double r = i <= j ? __ldcg(a.R + (int64_t)j * a.ldr + i) : 0.0;
    Rs[i * LDM + j] = r;
    if (i == j && !(r != 0.0)) atomicMin(&misc[0], i + 1);
  }
  __syncthreads();
  const int zi = misc[0];
  if (zi <= n) {  // Q would not be finite: NaN columns from the first zero pivot on, and the status
    const int64_t k = gridDim.x;
    const int64_t r0 = a.tiles * blockIdx.x / k * 64, r1 = min(a.m, a.tiles * (blockIdx.x + 1) / k * 64);
    for (int j = 0; j < n; ++j)
      for (int64_t r = r0 + tid; r < r1; r += T) a.Q[j * a.ldq + r] = (S)__longlong_as_double(0x7ff8000000000000ll);
    if (blockIdx.x == 0 && tid == 0 && a.info) {
      a.info[0] = QL_ERR_NOT_SPD;
      a.info[1] = zi;
    }
    return;
  }
  tri_upper_inverse<T>(Rs, LDM, Mf, LDM, n);
  // double-float copy (zero below the diagonal and past n) and its range verdict
  bool mbad = false;
  for (int e = tid; e < NC * NC / 2; e += T) {
    const int k = e / (NC / 2), j0 = 2 * (e % (NC / 2));
    df m2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = j0 + h;
      const double v = (k < n && j < n && k <= j) ? Mf[k * LDM + j] : 0.0;
      if (v != 0.0) {
        const int E = (int)((__double_as_longlong(v) >> 52) & 0x7ff);
        if (E < 1023 - 60 || E > 1023 + 60) mbad = true;
      }
      m2[h] = df_from_double_rn(v);
    }
    Md[e] = df2{f2_make(m2[0].hi, m2[1].hi), f2_make(m2[0].lo, m2[1].lo)};
  }
  const bool m_f64 = __syncthreads_or(mbad);
  if (blockIdx.x == 0 && tid == 0 && a.info) {
    a.info[0] = QL_OK;
    a.info[1] = 0;
  }

  // ---- row blocks of 64 rows (tiles), one warp each
  const int lane = tid & 31;
  const int64_t nw = (int64_t)gridDim.x * (T / 32);
  X2* mine = xs + tid;  // column k of this thread's rows at mine[k T]
  using S2 = typename std::conditional<sizeof(S) == 8, double2, float2>::type;
  for (int64_t t = (int64_t)blockIdx.x * a.cta_step + (tid >> 5) * a.warp_step; t < a.tiles; t += nw) {
    const int64_t row = t * 64 + 2 * lane;
    const bool live0 = row < a.m, live1 = row + 1 < a.m;
    const bool whole = a.pair && t * 64 + 64 <= a.m;  // uniform in the warp
    bool xbad = false;
#pragma unroll 1
    for (int c0 = 0; c0 < n; c0 += 8) {
      S2 v[8];
      if (whole) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c0 + u < n) v[u] = __ldcs(reinterpret_cast<const S2*>(a.X + (c0 + u) * a.ldx + row));
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          v[u].x = c0 + u < n && live0 ? __ldg(a.X + (c0 + u) * a.ldx + row) : S(0);
          v[u].y = c0 + u < n && live1 ? __ldg(a.X + (c0 + u) * a.ldx + row + 1) : S(0);
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (c0 + u >= n) break;
        int E0, E1;
        const df v0 = load_df(v[u].x, E0), v1 = load_df(v[u].y, E1);
        if ((E0 != 0 && (E0 < kDfEminLimit || E0 > kDfEmaxLimit)) || (E1 != 0 && (E1 < kDfEminLimit || E1 > kDfEmaxLimit)))
          xbad = true;
        if constexpr (sizeof(S) == 8)
          mine[(c0 + u) * T] = make_float4(v0.hi, v0.lo, v1.hi, v1.lo);
        else
          mine[(c0 + u) * T] = make_float2(v0.hi, v1.hi);
      }
    }
    const bool f64 = __any_sync(0xffffffffu, xbad) || m_f64;
    if (!f64) {
#pragma unroll 1
      for (int jb = 0; jb < n; jb += 8) {
        df2 acc[2][4];  // [row][column pair]
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) acc[h][jj] = df2{0, 0};
        const int kend = min(n, jb + 8);  // M is upper triangular: rows past column jb + 7 are zero
#pragma unroll (NC <= 16 ? 1 : 2)
        for (int kk = 0; kk < kend; ++kk) {
          const X2 x = mine[kk * T];
          df2n x0, x1;
          if constexpr (sizeof(S) == 8) {
            x0 = df2_factor(df2{f2_make(x.x, x.x), f2_make(x.y, x.y)});
            x1 = df2_factor(df2{f2_make(x.z, x.z), f2_make(x.w, x.w)});
          } else {
            x0 = df2_factor(df2{f2_make(x.x, x.x), 0});
            x1 = df2_factor(df2{f2_make(x.y, x.y), 0});
          }
          const df2* mrow = Md + kk * (NC / 2) + jb / 2;
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const df2 mv = mrow[jj];
            df2_acc_fma(acc[0][jj], x0, mv);
            df2_acc_fma(acc[1][jj], x1, mv);
          }
        }
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
          if (jb + jj >= n) break;
          S2 o;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            df c[2];
            df2_rows(acc[h][jj / 2], c[0], c[1]);
            const df q = c[jj & 1];
            const S r = sizeof(S) == 8 ? (S)((double)q.hi + (double)q.lo) : (S)__fadd_rn(q.hi, q.lo);
            (h == 0 ? o.x : o.y) = r;
          }
          S* out = a.Q + (jb + jj) * a.ldq + row;
          if (whole) {
            __stcs(reinterpret_cast<S2*>(out), o);
          } else {
            if (live0) out[0] = o.x;
            if (live1) out[1] = o.y;
          }
        }
      }
    } else {
      // FP64 for this block: outside the double-float range, or M is
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        const int64_t r = row + h;
        if (r >= a.m) break;
        for (int jb = 0; jb < n; jb += 8) {
          double acc[8];
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) acc[jj] = 0.0;
          const int kend = min(n, jb + 8);
#pragma unroll 1
          for (int kk = 0; kk < kend; ++kk) {
            const double xk = (double)a.X[kk * a.ldx + r];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj)
              acc[jj] = fma(xk, (jb + jj < n && kk <= jb + jj) ? Mf[kk * LDM + jb + jj] : 0.0, acc[jj]);
          }
#pragma unroll
          for (int jj = 0; jj < 8; ++jj)
            if (jb + jj < n) a.Q[(jb + jj) * a.ldq + r] = (S)acc[jj];
        }
      }
    }
  }
}

template <int NC, typename S>
static ql_status qform_launch_one(QformArgs<S> a, cudaStream_t stream) {
  using Sm = QformSmem<NC, S>;
  auto kern = qform_kernel<NC, S>;
  static bool ready_on[kMaxDevices] = {};
  bool& ready = ready_on[device_slot()];
  static std::mutex mu;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!ready) {
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sm::kBytes) != cudaSuccess)
        return QL_ERR_CUDA;
      ready = true;
    }
  }
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, Sm::T, Sm::kBytes) != cudaSuccess) return QL_ERR_CUDA;
  // A block of rows costs its SM's FP64 pipe 3 n conversions each way per row, so with fewer blocks
  // than warps they are spread over the SMs, a warp or a few in each CTA, instead of filling the
  // warps of a few CTAs
  // (and, while one CTA per SM has the warps, one copy of R^{-1} is formed per SM)
  const int64_t sms = device_sm_count();
  int64_t g = sms * (occ < 1 ? 1 : occ);
  const bool spread = a.tiles < g * (Sm::T / 32);
  if (a.tiles <= sms * (Sm::T / 32)) g = sms;
  if (g > a.tiles) g = a.tiles;
  if (g < 1) g = 1;
  a.cta_step = spread ? 1 : Sm::T / 32;
  a.warp_step = spread ? (int)g : 1;
  count_launch();
  kern<<<(int)g, Sm::T, Sm::kBytes, stream>>>(a);
  return cudaPeekAtLastError() == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

template <typename S>
static ql_status qform_dispatch(QformArgs<S> a, cudaStream_t stream) {
  a.tiles = (a.m + 63) / 64;
  if (a.tiles < 1) a.tiles = 1;
  auto aligned = [](const void* p) { return reinterpret_cast<uintptr_t>(p) % (2 * sizeof(S)) == 0; };
  a.pair = aligned(a.X) && aligned(a.Q) && a.ldx % 2 == 0 && a.ldq % 2 == 0 ? 1 : 0;
  const int n = a.n;
  if (n <= 8) return qform_launch_one<8, S>(a, stream);
  if (n <= 16) return qform_launch_one<16, S>(a, stream);
  if (n <= 32) return qform_launch_one<32, S>(a, stream);
  return qform_launch_one<64, S>(a, stream);
}

// dst <- the first nonzero {status, index} pair of src[0 .. count) (or {QL_OK, 0})
__global__ void first_status_kernel(int32_t* dst, const int32_t* src, int count) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  int32_t s = 0, i = 0;
  for (int c = 0; c < count; ++c)
    if (src[2 * c] != 0) {
      s = src[2 * c];
      i = src[2 * c + 1];
      break;
    }
  dst[0] = s;
  dst[1] = i;
}

ql_status first_status_async(int32_t* dst, const int32_t* src, int count, cudaStream_t stream) {
  count_launch();
  first_status_kernel<<<1, 32, 0, stream>>>(dst, src, count);
  return cudaPeekAtLastError() == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

}  // namespace ql

using namespace ql;

extern "C" ql_status ql_q_from_r(int64_t m, int64_t n, const void* X, ql_dtype dtype, int64_t ldx, const double* R,
                                 int64_t ldr, void* Q, int64_t ldq, int32_t* info, void* stream) {
  if (m < 0 || n < 1 || n > kMaxN || (dtype != QL_F64 && dtype != QL_F32) || ldx < (m > 1 ? m : 1) ||
      ldq < (m > 1 ? m : 1) || (m > 0 && (!X || !Q)) || !R || ldr < n)
    return QL_ERR_ARG;
  const size_t el = dtype == QL_F64 ? 8 : 4;
  if ((reinterpret_cast<uintptr_t>(X) % el) || (reinterpret_cast<uintptr_t>(Q) % el) ||
      (reinterpret_cast<uintptr_t>(R) % 8))
    return QL_ERR_ALIGN;
  cudaStream_t st = (cudaStream_t)stream;
  if (dtype == QL_F64) {
    QformArgs<double> a{m, (int)n, static_cast<const double*>(X), ldx, R, ldr, static_cast<double*>(Q), ldq, info, 0, 0, 0, 0};
    return qform_dispatch(a, st);
  }
  QformArgs<float> a{m, (int)n, static_cast<const float*>(X), ldx, R, ldr, static_cast<float*>(Q), ldq, info, 0, 0, 0, 0};
  return qform_dispatch(a, st);
}
