// Dense ||A x||^2 for rows of up to 2048 entries in native arithmetic (FP64, FP32):
// forward and fused value-and-gradient, several rows per team and step.
//
// What bounds it: FP32, the stream of A from HBM; FP64, GB300's 2 DFMA a clock and SM
// (two DFMA an entry are 2.7 times the HBM time of its 8 bytes).  Neither leaves room
// for a reduction of its own per row: a butterfly over a warp is five adds a lane and
// row, more than the row's own work when a lane holds a few columns.  So a team (W
// warps, column j = lane + 32 W k in lane registers, k < CPL) takes R rows at once:
//   - the R rows' loads are issued together (R * CPL of them in flight a lane);
//   - one transposed butterfly reduces the R dot products: each exchange hands half of
//     the rows to the other half of the lanes, R - 1 adds and then log2(32 / R) for R
//     rows (R = 4: 6 adds instead of 20), and ybar = 2 fbar y is one multiplication for
//     all R rows;
//   - only teams wider than a warp (n > 256) exchange through shared memory, once per
//     R rows.
// CPL is ceil(n / (32 W)) at compile time, so that no column slot but the last is
// tested or idle.  Groups of R rows go round-robin over all teams of the grid; xbar is
// accumulated in registers, combined over the CTA's teams in team order and, for grids
// of one CTA, written as the gradient; larger grids write a row of partials per CTA,
// summed in a fixed order by the CTA that finishes last (few partials) or by
// qf_reduce_kernel: bitwise reproducible.
//
// Measured (value and gradient, one call, against one row a team and step with a butterfly
// per row): FP64 150001 x 255 857 -> 160 us (its DFMAs take 122), FP32 400000 x 100
// 121 -> 36.6 us (its bytes take 23.6).
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "kg_device.cuh"
#include "kg_internal.h"
#include "kg_pair.cuh"

namespace kg {

constexpr int QR_THREADS = 256;
constexpr int QR_WARPS = QR_THREADS / 32;

template <typename T>
struct QrArgs {
  const T* A;
  const T* x;
  int64_t m;
  int n;
  const T* seed;     // nullable device scalar (fbar)
  T* partials;       // FUSED, more than one CTA: [gridDim.x][n]
  double* fpart;     // per-CTA f partials
  unsigned* counter; // arrival counter of the last-CTA reductions
  T* y;              // EVAL, nullable: forward row values
  T* f;              // EVAL, one CTA or `last`: output (nullable when FUSED)
  T* gx;             // FUSED, one CTA or `last`: output
  T* gA;             // FUSED, nullable: gradient w.r.t. A
  int accumulate;
  int last;          // FUSED: the last CTA sums the partials
};

// Sum of the R rows' values over a warp: lane l ends with the total of row
// l / (32 / R), the same bits on all lanes of that row.
template <int R, typename T>
__device__ __forceinline__ T reduce_rows(T (&d)[R]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int w = R / 2; w > 0; w >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const T keep = up ? d[i + w] : d[i], send = up ? d[i] : d[i + w];
      d[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (; o > 0; o >>= 1) d[0] += __shfl_xor_sync(0xffffffffu, d[0], o);
  return d[0];
}

// FP64: two CTAs an SM (128 registers, R * CPL doubles of A in them); FP32: three.
template <typename T, int W, int CPL, int R, bool FUSED>
__global__ void __launch_bounds__(QR_THREADS, sizeof(T) == 8 ? 2 : 3) qf_rows_kernel(QrArgs<T> a) {
  constexpr int TEAM = 32 * W, NT = QR_WARPS / W, G = 32 / R;  // G lanes hold a row's total
  static_assert(W <= G, "the cross-warp butterfly stays inside a row's lanes");
  __shared__ T xbs[FUSED ? QR_THREADS * CPL : 1];
  __shared__ T red[W > 1 ? 2 * QR_WARPS * R : 1];
  __shared__ double fred[32];
  __shared__ bool s_last;
  const int n = a.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / W, lt = threadIdx.x % TEAM;
  auto col_in = [&](int k) { return k < CPL - 1 || lt + k * TEAM < n; };

  T xv[CPL], xb[CPL];
#pragma unroll
  for (int k = 0; k < CPL; ++k) {
    xv[k] = col_in(k) ? a.x[lt + k * TEAM] : T(0);
    xb[k] = T(0);
  }
  const T fb2 = FUSED ? T(2) * load_seed(a.seed) : T(0);
  FSum<T> fsum;  // of row lane / G of every group (counted once per row below)

  // group g of R rows goes to team g / gridDim.x of CTA g % gridDim.x, round by round
  const int64_t groups = (a.m + R - 1) / R;
  const int64_t nteams = (int64_t)gridDim.x * NT;
  int par = 0;
  // the trip count is that of the CTA's first team: teams of W > 1 meet at a CTA barrier
  for (int64_t g0 = blockIdx.x; g0 < groups; g0 += nteams, par ^= 1) {
    const int64_t grp = g0 + (int64_t)team * gridDim.x;
    const int64_t r0 = grp * R;
    if (W == 1 && grp >= groups) break;
    const int rows = grp < groups ? (int)(a.m - r0 < R ? a.m - r0 : R) : 0;
    const T* Ar = a.A + (rows > 0 ? r0 : 0) * (int64_t)n + lt;
    T av[R][CPL];
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
      for (int k = 0; k < CPL; ++k)
        av[r][k] = r < rows && col_in(k) ? ld_stream(Ar + k * TEAM) : T(0);
      Ar += n;
    }
    T d[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      d[r] = av[r][0] * xv[0];
#pragma unroll
      for (int k = 1; k < CPL; ++k) d[r] = fma(av[r][k], xv[k], d[r]);
    }
    T tot = reduce_rows<R>(d);
    const int row = lane / G;
    if constexpr (W > 1) {
      T* rd = red + par * QR_WARPS * R + team * W * R;
      if (lane % G == 0) rd[(warp % W) * R + row] = tot;
      __syncthreads();
      tot = rd[(lane % W) * R + row];
#pragma unroll
      for (int o = W / 2; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if (row >= rows) tot = T(0);  // past the end: 0 times an infinite x is no row's value
    fsum.add(tot);
    if constexpr (!FUSED) {
      if (a.y && row < rows && lane % G == 0 && (W == 1 || warp % W == 0)) a.y[r0 + row] = tot;
    } else {
      const T ybl = fb2 * tot;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const T yb = __shfl_sync(0xffffffffu, ybl, r * G);
#pragma unroll
        for (int k = 0; k < CPL; ++k) xb[k] = fma(yb, av[r][k], xb[k]);
        if (a.gA && r < rows) {
          T* gr = a.gA + (r0 + r) * (int64_t)n + lt;
#pragma unroll
          for (int k = 0; k < CPL; ++k)
            if (col_in(k)) {
              const T v = yb * xv[k];
              gr[k * TEAM] = a.accumulate ? gr[k * TEAM] + v : v;
            }
        }
      }
    }
  }

  // the CTA's f: one lane per row of a group, one warp per team
  const double fcta =
      block_sum(lane % G == 0 && (W == 1 || warp % W == 0) ? fsum.get() : 0.0, fred);
  if constexpr (!FUSED) {
    finish_sum<T>(fcta, a.fpart, a.counter, a.f, 0, fred);
    return;
  } else {
#pragma unroll
    for (int k = 0; k < CPL; ++k) xbs[team * TEAM * CPL + lt + k * TEAM] = xb[k];
    __syncthreads();
    const bool one = gridDim.x == 1;
    T* out = one ? a.gx : a.partials + (int64_t)blockIdx.x * n;
    for (int j = threadIdx.x; j < n; j += QR_THREADS) {
      T s = xbs[j];
#pragma unroll
      for (int t = 1; t < NT; ++t) s += xbs[t * TEAM * CPL + j];
      out[j] = one && a.accumulate ? out[j] + s : s;
    }
    if (threadIdx.x == 0) {
      if (one) {
        if (a.f) *a.f = (T)fcta;
      } else {
        a.fpart[blockIdx.x] = fcta;
      }
    }
    if (one || !a.last) return;
    // few partials: the CTA that arrives last sums them, thread (cx, pg) partials pg,
    // pg + PG, ... of column cx, the PG sums then in pg order
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(a.counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int parts = gridDim.x;
    int cw = 32;
    while (cw < n && cw < QR_THREADS) cw *= 2;
    const int pgs = QR_THREADS / cw, cx = threadIdx.x % cw, pg = threadIdx.x / cw;
    for (int jb = 0; jb < n; jb += cw) {
      const int j = jb + cx;
      T s = T(0);
      if (j < n) {
#pragma unroll 8
        for (int c = pg; c < parts; c += pgs) s += __ldcg(a.partials + (int64_t)c * n + j);
      }
      __syncthreads();
      xbs[threadIdx.x] = s;
      __syncthreads();
      if (pg == 0 && j < n) {
        for (int q = 1; q < pgs; ++q) s += xbs[q * cw + cx];
        a.gx[j] = a.accumulate ? a.gx[j] + s : s;
      }
    }
    double fs = 0.0;
    for (int i = threadIdx.x; i < parts; i += QR_THREADS) fs += __ldcg(a.fpart + i);
    fs = block_sum(fs, fred);
    if (threadIdx.x == 0) {
      if (a.f) *a.f = (T)fs;
      *a.counter = 0u;
    }
  }
}

// ---------------------------------------------------------------- host ----
// Warps per team for rows of n entries (8 columns a lane at most); team: the
// caller's threads per team (0: the smallest that holds the row).
static int qr_warps(int64_t n, int team) {
  if (team) return team / 32;
  int w = 1;
  while ((int64_t)256 * w < n) w *= 2;
  return w;
}

// Rows per step: R * CPL values of A in a lane's registers, up to 32; a team of 8 warps
// takes 4 rows (the cross-warp butterfly needs W lanes a row).
constexpr int qr_rows(int cpl, int w) { return cpl <= 4 && w < 8 ? 8 : 4; }

// Calls go(kernel, rows per step, teams per CTA) with the kernel of this row length.
template <typename T, bool FUSED, int W, typename Go>
static void qr_with_cpl(int64_t n, const Go& go) {
  switch ((n + 32 * W - 1) / (32 * W)) {
#define KG_CPL(c) \
  case c: go(qf_rows_kernel<T, W, c, qr_rows(c, W), FUSED>, qr_rows(c, W), QR_WARPS / W); break;
    KG_CPL(1) KG_CPL(2) KG_CPL(3) KG_CPL(4) KG_CPL(5) KG_CPL(6) KG_CPL(7) KG_CPL(8)
#undef KG_CPL
  }
}

template <typename T, bool FUSED, typename Go>
static void qr_with_kernel(int64_t n, int team, const Go& go) {
  switch (qr_warps(n, team)) {
    case 1: qr_with_cpl<T, FUSED, 1>(n, go); break;
    case 2: qr_with_cpl<T, FUSED, 2>(n, go); break;
    case 4: qr_with_cpl<T, FUSED, 4>(n, go); break;
    case 8: qr_with_cpl<T, FUSED, 8>(n, go); break;
  }
}

bool qf_rows_supported(int64_t n) { return n <= 2048; }

// One wave of resident CTAs, or fewer when every team has a group of rows.
template <typename T>
static int qr_grid_t(int64_t m, int64_t n, int team) {
  int64_t grid = 1;
  qr_with_kernel<T, true>(n, team, [&](auto kern, int rows, int teams) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, QR_THREADS, 0) != cudaSuccess || occ < 1) {
      cudaGetLastError();
      occ = 1;
    }
    const int64_t step = (int64_t)rows * teams;
    grid = std::min<int64_t>((m + step - 1) / step, (int64_t)num_sms() * occ);
  });
  return (int)std::max<int64_t>(1, grid);
}

int qf_rows_grid(int dtype, int64_t m, int64_t n, int team) {
  return dtype == KG_F64 ? qr_grid_t<double>(m, n, team) : qr_grid_t<float>(m, n, team);
}

template <typename T, bool FUSED>
static cudaError_t launch_rows(int grid, int team, const QrArgs<T>& a, cudaStream_t s) {
  prof_begin(s, FUSED ? "qf_rows_kernel<fused>" : "qf_rows_kernel<eval>");
  qr_with_kernel<T, FUSED>(a.n, team, [&](auto kern, int, int) { kern<<<grid, QR_THREADS, 0, s>>>(a); });
  prof_end(s);
  count_launch();
  return cudaGetLastError();
}

// The last CTA sums the partials itself up to this many bytes of them: about 32 loads a
// thread, less than a second launch takes.
constexpr int64_t QR_LAST_BYTES = 64 << 10;

template <typename T>
kg_status qf_rows_eval(const QfRowsCall<T>& c, cudaStream_t s) {
  QrArgs<T> a{};
  a.A = c.A;
  a.x = c.x;
  a.m = c.m;
  a.n = (int)c.n;
  a.fpart = c.fpart;
  a.counter = c.counter;
  a.y = c.y;
  a.f = c.f;
  cudaError_t e = launch_rows<T, false>(c.grid, c.team, a, s);
  return e == cudaSuccess ? KG_OK : cuda_fail(e, "qf forward kernel");
}

template <typename T>
kg_status qf_rows_grad(const QfRowsCall<T>& c, cudaStream_t s) {
  QrArgs<T> a{};
  a.A = c.A;
  a.x = c.x;
  a.m = c.m;
  a.n = (int)c.n;
  a.seed = c.seed;
  a.partials = c.partials;
  a.fpart = c.fpart;
  a.counter = c.counter;
  a.f = c.f;
  a.gx = c.gx;
  a.gA = c.gA;
  a.accumulate = c.accumulate;
  a.last = c.counter && (int64_t)c.grid * c.n * (int64_t)sizeof(T) <= QR_LAST_BYTES;
  cudaError_t e = launch_rows<T, true>(c.grid, c.team, a, s);
  if (e != cudaSuccess) return cuda_fail(e, "qf fused kernel");
  if (c.grid == 1 || a.last) return KG_OK;
  return qf_reduce_partials<T>(c.partials, c.grid, a.n, c.fpart, c.grid, c.gx, c.f, c.accumulate, s);
}

template kg_status qf_rows_eval<double>(const QfRowsCall<double>&, cudaStream_t);
template kg_status qf_rows_eval<float>(const QfRowsCall<float>&, cudaStream_t);
template kg_status qf_rows_grad<double>(const QfRowsCall<double>&, cudaStream_t);
template kg_status qf_rows_grad<float>(const QfRowsCall<float>&, cudaStream_t);

}  // namespace kg
