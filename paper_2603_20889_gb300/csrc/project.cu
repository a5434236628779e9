// Two-phase orthogonalisation (the "two-phase problem" QR = (I - Y Y^T) X with
// re-orthogonalisation that Sec. 2 discusses for the Gram methods): for Y (m x k) with
// orthonormal columns and X (m x n),
//   C1 = Y^T X,  W1 = X - Y C1,  C2 = Y^T W1,  W = W1 - Y C2,  C = C1 + C2,
// so that W = (I - Y Y^T) X to working precision even when X is nearly in range(Y).  The R
// of the orthogonalised block is then any of the Q-less calls on W.
//
// Six launches (cross product, its reduction, update; twice).  The cross product Y^T V is a
// reduction over the m rows: every CTA accumulates 4 x 4 blocks of the k x n product over its row
// tiles in double-float, two rows per packed FP32 instruction (half the issue slots; two CTAs per
// SM, so that one loads while the other multiplies), and writes one FP64 partial;
// cross_reduce_kernel sums the partials in a fixed order (reproducible), an entry per thread over
// many CTAs, where the last CTA used to sum all of them.  The update W = V - Y C streams blocks of
// 64 rows, a warp each, two adjacent rows per thread and two columns per packed instruction; few
// blocks are spread over the SMs (see qform.cu).  Tiles outside the double-float exponent range run
// in FP64.  With few rows the later launches wait on the device for their predecessors (programmatic
// dependent launches): 1000 rows, k = 8, n = 1 57 -> 44 us.
//
// Both are bound by the FP32 pipes, 13 operations per product and row: k = n = 64, m = 2^19
// 0.71 ms each; measured 1.34 + 0.05 ms (cross product and reduction) and 1.67 ms (update).  QR
// of 524288 x 128, with two of each: 15.3 -> 9.8 ms.
#include <mutex>

#include "df2.cuh"
#include "internal.h"
#include "small_dense.cuh"

namespace ql {

constexpr int kProjT = 256;
constexpr int kProjB = 64;   // rows per tile of the cross product

struct ProjWs {
  double* cprev;     // C of the first pass (k x n, ld n)
  double* cpass;     // C of the current pass, read by the update (k x n, ld n)
  double* partials;  // one KC x NC partial per CTA
};

template <typename S>
struct ProjArgs {
  int64_t m;
  int k, n;
  const S* Y;
  int64_t ldy;
  const S* V;  // X (pass 1) or W1 (pass 2)
  int64_t ldv;
  S* W;
  int64_t ldw;
  double* C;  // output coefficients (k x n, ld ldc)
  int64_t ldc;
  int pass;
  ProjWs w;
  int64_t tiles;
  int cta_step, warp_step;  // update: first block of a warp = CTA x cta_step + warp x warp_step
};

QL_DEV bool df_range_ok_dev(int E) { return E == 0 || (E >= kDfEminLimit && E <= kDfEmaxLimit); }


// ---- C = Y^T V over the rows: one partial per CTA
template <int KC, int NC, typename S>
__global__ void __launch_bounds__(kProjT, 2) cross_kernel(ProjArgs<S> a) {
  constexpr int T = kProjT, B = kProjB;
  constexpr int NBLK = (KC / 4) * (NC / 4);  // 4 x 4 blocks of C
  constexpr int SL = T / NBLK >= 1 ? T / NBLK : 1;
  static_assert(NBLK <= T, "one block per thread at least");
  extern __shared__ __align__(16) unsigned char smem[];
  df2* Ys = reinterpret_cast<df2*>(smem);  // [KC][B / 2] row pairs
  df2* Vs = Ys + KC * (B / 2);             // [NC][B / 2]
  double* red = reinterpret_cast<double*>(smem);  // [SL][KC][NC] at the end
  const int tid = threadIdx.x, k = a.k, n = a.n;
  pdl_release();
  pdl_wait();
  const int blk = tid / SL, slice = tid % SL;
  const bool active = blk < NBLK;
  const int bi = active ? (blk / (NC / 4)) * 4 : 0, bj = active ? (blk % (NC / 4)) * 4 : 0;

  df2 acc[4][4];
  double acc64[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[i][j] = df2{0, 0};
      acc64[i][j] = 0.0;
    }
  const int64_t nb = gridDim.x, bid = blockIdx.x;
  const int64_t t0 = a.tiles * bid / nb, t1 = a.tiles * (bid + 1) / nb;
  for (int64_t t = t0; t < t1; ++t) {
    const int64_t row0 = t * B;
    bool bad = false;
#pragma unroll 8
    for (int e = tid; e < (KC + NC) * (B / 2); e += T) {
      const int c = e / (B / 2), r = e % (B / 2);
      const int64_t row = row0 + 2 * r;
      const bool isY = c < KC, used = isY ? c < k : c - KC < n;
      const S* p = (isY ? a.Y + c * a.ldy : a.V + (c - KC) * a.ldv) + row;
      S x0 = S(0), x1 = S(0);
      if (used) {
        if (row < a.m) x0 = p[0];
        if (row + 1 < a.m) x1 = p[1];
      }
      int E0, E1;
      const df v0 = load_df(x0, E0), v1 = load_df(x1, E1);
      if (!df_range_ok_dev(E0) || !df_range_ok_dev(E1)) bad = true;
      Ys[e] = df2{f2_make(v0.hi, v1.hi), f2_make(v0.lo, v1.lo)};
    }
    const bool f64 = __syncthreads_or(bad);
    if (active) {
      if (!f64) {
#pragma unroll 1
        for (int r = slice; r < B / 2; r += SL) {
          df2 v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = Vs[(bj + j) * (B / 2) + r];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const df2n y = df2_factor(Ys[(bi + i) * (B / 2) + r]);
#pragma unroll
            for (int j = 0; j < 4; ++j) df2_acc_fma(acc[i][j], y, v[j]);
          }
        }
      } else {  // FP64 for this tile, straight from global memory
        for (int r = slice; r < B; r += SL) {
          const int64_t row = row0 + r;
          if (row >= a.m) break;
          double y[4], v[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) y[i] = bi + i < k ? (double)a.Y[(bi + i) * a.ldy + row] : 0.0;
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = bj + j < n ? (double)a.V[(bj + j) * a.ldv + row] : 0.0;
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc64[i][j] = fma(y[i], v[j], acc64[i][j]);
        }
      }
    }
    __syncthreads();
  }
  // combine the row parities and the slices and store this CTA's partial (FP64)
  if (active) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        df e, o;
        df2_rows(acc[i][j], e, o);
        red[((size_t)slice * KC + bi + i) * NC + bj + j] = (df_to_double(e) + df_to_double(o)) + acc64[i][j];
      }
  }
  __syncthreads();
  double* part = a.w.partials + (size_t)bid * KC * NC;
  for (int e = tid; e < KC * NC; e += T) {
    double s = 0.0;
    for (int sl = 0; sl < SL; ++sl) s += red[(size_t)sl * KC * NC + e];
    part[e] = s;
  }
}

// ---- the fixed-order sum of the nb partials: C of this pass and the running total
constexpr int kReduceT = 64;
template <typename S>
__global__ void __launch_bounds__(kReduceT) cross_reduce_kernel(ProjArgs<S> a, int kc, int nc, int nb) {
  pdl_release();
  pdl_wait();
  const int e = blockIdx.x * kReduceT + threadIdx.x, i = e / nc, j = e % nc;
  if (e >= kc * nc || i >= a.k || j >= a.n) return;
  const double* p = a.w.partials + e;
  const size_t step = (size_t)kc * nc;
  double s = 0.0;
#pragma unroll 16
  for (int b = 0; b < nb; ++b) s += __ldg(p + b * step);
  a.w.cpass[i * a.n + j] = s;
  const double tot = a.pass == 1 ? s : a.w.cprev[i * a.n + j] + s;
  if (a.pass == 1) a.w.cprev[i * a.n + j] = s;
  a.C[j * a.ldc + i] = tot;
}

// ---- W = V - Y C (C of this pass): blocks of 64 rows, a warp each, two adjacent rows per thread
// and two columns per packed instruction (as qform_kernel)
template <int KC>
__host__ __device__ constexpr int update_threads() {
  return KC == 64 ? 160 : 256;
}
template <int KC, int NC, typename S>
__global__ void __launch_bounds__(update_threads<KC>(), 1) update_kernel(ProjArgs<S> a) {
  constexpr int T = update_threads<KC>();
  extern __shared__ __align__(16) unsigned char smem[];
  df2* Cd = reinterpret_cast<df2*>(smem);                                        // [KC][NC / 2] column pairs
  float4* mine = reinterpret_cast<float4*>(Cd + KC * NC / 2) + threadIdx.x;     // column i of this thread's rows at mine[i T]
  const int tid = threadIdx.x, lane = tid & 31, k = a.k, n = a.n;
  pdl_release();
  pdl_wait();
  bool cbad = false;
  for (int e = tid; e < KC * NC / 2; e += T) {
    const int i = e / (NC / 2), j0 = 2 * (e % (NC / 2));
    df c2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double c = (i < k && j0 + h < n) ? __ldcg(a.w.cpass + i * n + j0 + h) : 0.0;
      const int E = (int)((__double_as_longlong(c) >> 52) & 0x7ff);
      if (c != 0.0 && (E < 1023 - 80 || E > 1023 + 80)) cbad = true;  // products with Y stay normal floats
      c2[h] = df_from_double_rn(c);
    }
    Cd[e] = df2{f2_make(c2[0].hi, c2[1].hi), f2_make(c2[0].lo, c2[1].lo)};
  }
  const bool c64 = __syncthreads_or(cbad);
  auto fp64_entry = [&](int64_t row, int j) {
    double s = (double)a.V[j * a.ldv + row];
    for (int i = 0; i < k; ++i) s = fma(-(double)a.Y[i * a.ldy + row], __ldcg(a.w.cpass + i * n + j), s);
    a.W[j * a.ldw + row] = (S)s;
  };
  const int64_t nw = (int64_t)gridDim.x * (T / 32);
  for (int64_t t = (int64_t)blockIdx.x * a.cta_step + (tid >> 5) * a.warp_step; t < a.tiles; t += nw) {
    const int64_t row = t * 64 + 2 * lane;
    const bool live0 = row < a.m, live1 = row + 1 < a.m;
    bool bad = false;
#pragma unroll 1
    for (int i0 = 0; i0 < k; i0 += 8) {
      S x[8][2];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const S* p = a.Y + (i0 + u) * a.ldy + row;
        x[u][0] = i0 + u < k && live0 ? __ldg(p) : S(0);
        x[u][1] = i0 + u < k && live1 ? __ldg(p + 1) : S(0);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (i0 + u >= k) break;
        int E0, E1;
        const df y0 = load_df(x[u][0], E0), y1 = load_df(x[u][1], E1);
        if (!df_range_ok_dev(E0) || !df_range_ok_dev(E1)) bad = true;
        mine[(i0 + u) * T] = make_float4(y0.hi, y0.lo, y1.hi, y1.lo);
      }
    }
    const bool f64 = __any_sync(0xffffffffu, bad) || c64;
#pragma unroll 1
    for (int jb = 0; jb < n; jb += 8) {
      if (!f64) {
        // V's entries first: their fetch hides behind the products (W may be V itself)
        S v[2][8];
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
          v[0][jj] = jb + jj < n && live0 ? a.V[(jb + jj) * a.ldv + row] : S(0);
          v[1][jj] = jb + jj < n && live1 ? a.V[(jb + jj) * a.ldv + row + 1] : S(0);
        }
        df2 acc[2][4];  // [row][column pair]
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) acc[h][jj] = df2{0, 0};
#pragma unroll 2
        for (int i = 0; i < k; ++i) {
          const float4 x = mine[i * T];
          const df2n y0 = df2_factor(df2{f2_make(x.x, x.x), f2_make(x.y, x.y)});
          const df2n y1 = df2_factor(df2{f2_make(x.z, x.z), f2_make(x.w, x.w)});
          const df2* crow = Cd + i * (NC / 2) + jb / 2;
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const df2 c = crow[jj];
            df2_acc_fma(acc[0][jj], y0, c);
            df2_acc_fma(acc[1][jj], y1, c);
          }
        }
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
          const int j = jb + jj;
          if (j >= n) break;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (h == 0 ? !live0 : !live1) continue;
            df c[2];
            df2_rows(acc[h][jj / 2], c[0], c[1]);
            int E;
            const df vv = load_df(v[h][jj], E);
            if (df_range_ok_dev(E)) {
              const df w = df_sub(vv, c[jj & 1]);
              if constexpr (sizeof(S) == 8)
                a.W[j * a.ldw + row + h] = (double)w.hi + (double)w.lo;
              else
                a.W[j * a.ldw + row + h] = __fadd_rn(w.hi, w.lo);
            } else {  // this entry alone is out of range: FP64
              fp64_entry(row + h, j);
            }
          }
        }
      } else {
        for (int jj = 0; jj < 8 && jb + jj < n; ++jj) {
          if (live0) fp64_entry(row, jb + jj);
          if (live1) fp64_entry(row + 1, jb + jj);
        }
      }
    }
  }
}

static int cls(int v) { return v <= 8 ? 8 : v <= 16 ? 16 : v <= 32 ? 32 : 64; }

template <int KC, int NC>
struct ProjSmem {
  static constexpr int NBLK = (KC / 4) * (NC / 4);
  static constexpr int SL = kProjT / NBLK >= 1 ? kProjT / NBLK : 1;
  static constexpr size_t kTile = 8 * (size_t)(KC + NC) * kProjB, kRed = 8 * (size_t)SL * KC * NC;
  static constexpr size_t kCross = kTile > kRed ? kTile : kRed;
  static constexpr size_t kUpdate = 8 * (size_t)KC * NC + 16 * (size_t)KC * update_threads<KC>();
  static_assert(kUpdate <= 232448, "shared memory of one SM");
};

constexpr int kCrossCtasPerSm = 2;
static size_t proj_parts_bytes() { return (size_t)device_sm_count() * kCrossCtasPerSm * 64 * 64 * sizeof(double); }

size_t project_workspace_bytes(int k, int n) {
  if (k < 1 || k > kMaxN || n < 1 || n > kMaxN) return 0;
  return 256 + 2 * (size_t)kMaxN * kMaxN * sizeof(double) + proj_parts_bytes();
}

template <int KC, int NC, typename S>
static ql_status proj_run(ProjArgs<S> a, cudaStream_t st) {
  using Sm = ProjSmem<KC, NC>;
  auto ck = cross_kernel<KC, NC, S>;
  auto uk = update_kernel<KC, NC, S>;
  static bool ready_on[kMaxDevices] = {};
  bool& ready = ready_on[device_slot()];
  static std::mutex mu;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!ready) {
      if (cudaFuncSetAttribute(ck, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sm::kCross) != cudaSuccess ||
          cudaFuncSetAttribute(uk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sm::kUpdate) != cudaSuccess)
        return QL_ERR_CUDA;
      ready = true;
    }
  }
  constexpr int UT = update_threads<KC>();
  int occ = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, uk, UT, Sm::kUpdate) != cudaSuccess) return QL_ERR_CUDA;
  const int64_t ctiles = (a.m + kProjB - 1) / kProjB, utiles = (a.m + 63) / 64;
  int64_t gc = (int64_t)device_sm_count() * kCrossCtasPerSm, gu = (int64_t)device_sm_count() * (occ < 1 ? 1 : occ);
  if (gc > ctiles) gc = ctiles;
  const bool spread = utiles < gu * (UT / 32);  // as in qform.cu: the conversions' FP64 pipes
  if (gu > utiles) gu = utiles;
  // (a choice between the two orders inside the kernel slowed its loop: 6.1 -> 6.36 ms)
  a.cta_step = spread ? 1 : UT / 32;
  a.warp_step = spread ? (int)gu : 1;
  if (gc < 1) gc = 1;
  if (gu < 1) gu = 1;
  const S* X = a.V;
  const int64_t ldx = a.ldv;
  for (int pass = 1; pass <= 2; ++pass) {
    a.pass = pass;
    if (pass == 2) {  // the second phase projects the first one's result again
      a.V = a.W;
      a.ldv = a.ldw;
    } else {
      a.V = X;
      a.ldv = ldx;
    }
    a.tiles = ctiles;
    count_launch();
    // The first kernel is an ordinary launch (its inputs are the caller's).  With few rows the others
    // start while their predecessor runs and wait for its end before they touch memory; with many
    // they are ordinary launches too (as dependent ones k = n = 64, m = 2^19 took 6.5 instead of 6.1 ms).
    if (pass == 1 || !spread) {
      ck<<<(int)gc, kProjT, Sm::kCross, st>>>(a);
      if (cudaPeekAtLastError() != cudaSuccess) return QL_ERR_CUDA;
    } else if (launch_dependent(ck, (int)gc, kProjT, Sm::kCross, st, a) != cudaSuccess) {
      return QL_ERR_CUDA;
    }
    count_launch();
    constexpr int gr = (KC * NC + kReduceT - 1) / kReduceT;
    if (!spread) {
      cross_reduce_kernel<S><<<gr, kReduceT, 0, st>>>(a, KC, NC, (int)gc);
      if (cudaPeekAtLastError() != cudaSuccess) return QL_ERR_CUDA;
    } else if (launch_dependent(cross_reduce_kernel<S>, gr, kReduceT, 0, st, a, KC, NC, (int)gc) != cudaSuccess) {
      return QL_ERR_CUDA;
    }
    a.tiles = utiles;
    count_launch();
    if (!spread) {
      uk<<<(int)gu, UT, Sm::kUpdate, st>>>(a);
      if (cudaPeekAtLastError() != cudaSuccess) return QL_ERR_CUDA;
    } else if (launch_dependent(uk, (int)gu, UT, Sm::kUpdate, st, a) != cudaSuccess) {
      return QL_ERR_CUDA;
    }
  }
  return QL_OK;
}

template <typename S>
static ql_status proj_dispatch(ProjArgs<S> a, cudaStream_t st) {
  const int kc = cls(a.k), nc = cls(a.n);
#define QL_PROJ_CASE(K, N) \
  if (kc == K && nc == N) return proj_run<K, N, S>(a, st);
#define QL_PROJ_ROW(K) QL_PROJ_CASE(K, 8) QL_PROJ_CASE(K, 16) QL_PROJ_CASE(K, 32) QL_PROJ_CASE(K, 64)
  QL_PROJ_ROW(8) QL_PROJ_ROW(16) QL_PROJ_ROW(32) QL_PROJ_ROW(64)
#undef QL_PROJ_ROW
#undef QL_PROJ_CASE
  return QL_ERR_ARG;
}

}  // namespace ql

using namespace ql;

extern "C" {

size_t ql_project_workspace_bytes(int64_t k, int64_t n) { return project_workspace_bytes((int)k, (int)n); }

ql_status ql_project_out(int64_t m, int64_t k, const void* Y, int64_t ldy, int64_t n, const void* X, int64_t ldx,
                         ql_dtype dtype, void* W, int64_t ldw, double* C, int64_t ldc, void* ws, size_t ws_bytes,
                         void* stream) {
  const int64_t lmin = m > 1 ? m : 1;
  if (m < 0 || k < 1 || k > kMaxN || n < 1 || n > kMaxN || (dtype != QL_F64 && dtype != QL_F32) || ldy < lmin ||
      ldx < lmin || ldw < lmin || ldc < k || !C || (m > 0 && (!Y || !X || !W)))
    return QL_ERR_ARG;
  const size_t el = dtype == QL_F64 ? 8 : 4;
  if ((reinterpret_cast<uintptr_t>(Y) % el) || (reinterpret_cast<uintptr_t>(X) % el) ||
      (reinterpret_cast<uintptr_t>(W) % el) || (reinterpret_cast<uintptr_t>(C) % 8))
    return QL_ERR_ALIGN;
  if (!ws || ws_bytes < project_workspace_bytes((int)k, (int)n)) return QL_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  unsigned char* b = static_cast<unsigned char*>(ws);
  ProjWs w;
  w.cprev = reinterpret_cast<double*>(b + 256);
  w.cpass = w.cprev + (size_t)kMaxN * kMaxN;
  w.partials = w.cpass + (size_t)kMaxN * kMaxN;
  if (dtype == QL_F64) {
    ProjArgs<double> a{m, (int)k, (int)n, static_cast<const double*>(Y), ldy, static_cast<const double*>(X), ldx,
                       static_cast<double*>(W), ldw, C, ldc, 1, w, 0, 0, 0};
    return proj_dispatch(a, st);
  }
  ProjArgs<float> a{m, (int)k, (int)n, static_cast<const float*>(Y), ldy, static_cast<const float*>(X), ldx,
                    static_cast<float*>(W), ldw, C, ldc, 1, w, 0, 0, 0};
  return proj_dispatch(a, st);
}

}  // extern "C"
