// Dense ||A x||^2 in native arithmetic (FP64, FP32): forward and fused value-and-gradient,
// several rows per team and step.
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
// CPL is fixed at compile time, ceil(n / (32 W)) up to n = 4096 and even above, so that
// at most the last two column slots are tested or idle.  Groups of R rows go round-robin over
// all teams of the grid, each team by itself: with a barrier of the whole CTA the teams without
// a group kept the FP64 unit busy with zeros (300 x 1024 value 8.3 -> 5.5 us, 610 x 1000 value
// and gradient 18.8 -> 12.7, 3000 x 1000 29.4 -> 23.4, together with f summed by the warps that
// hold it instead of the whole CTA).  xbar is accumulated in registers, combined over the CTA's
// teams in team order and, for grids of one CTA, written as the gradient; larger grids write a
// row of partials per CTA, summed in a fixed order by the CTA that finishes last (few partials)
// or by qf_reduce_kernel: bitwise reproducible.
//
// Measured (value and gradient, one call, against one row a team and step with a butterfly
// per row): FP64 150001 x 255 857 -> 158 us (its DFMAs take 122), 20000 x 2051 963 -> 248
// (131), 10000 x 5001 484 -> 242 (160), 10000 x 9999 478 -> 478 (320); FP32 400000 x 100
// 121 -> 35.9 us (its bytes take 23.6), 40000 x 1024 96.8 -> 31 (24), 20000 x 4095
// 157 -> 72 (48).
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "kg_device.cuh"
#include "kg_internal.h"
#include "kg_pair.cuh"

namespace kg {

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

// One kernel's shape: W warps a team, CPL columns a lane (the first FULL of them inside every
// row that runs it), R rows a step.  Teams of up to 8 warps share CTAs of 256 threads, a team
// of 16 is a CTA.  XS: x in shared memory, where a lane's columns leave no registers for it.
template <int W_, int CPL_, int FULL_, int R_, bool XS_>
struct QrShape {
  static constexpr int W = W_, CPL = CPL_, FULL = FULL_, R = R_;
  static constexpr bool XS = XS_;
  static constexpr int THREADS = W_ > 8 ? 512 : 256, WARPS = THREADS / 32, NT = WARPS / W_;
};

// FP64: 16 warps an SM (128 registers, R * CPL doubles of A in them); FP32 teams of up to 8
// warps: 24.
template <typename T, typename S, bool FUSED>
__global__ void __launch_bounds__(S::THREADS, S::THREADS == 512 ? 1 : sizeof(T) == 8 ? 2 : 3)
    qf_rows_kernel(QrArgs<T> a) {
  constexpr int W = S::W, CPL = S::CPL, R = S::R, NT = S::NT, THREADS = S::THREADS, WARPS = S::WARPS;
  constexpr int TEAM = 32 * W, G = 32 / R, WG = W < G ? W : G;  // G lanes hold a row's total
  __shared__ T xbs[FUSED ? (NT > 1 ? THREADS * CPL : THREADS) : 1];
  __shared__ T red[W > 1 ? 2 * WARPS * R : 1];
  __shared__ double fred[32];
  __shared__ bool s_last;
  extern __shared__ __align__(16) unsigned char dyn[];
  T* xs = reinterpret_cast<T*>(dyn);  // XS: [CPL][THREADS], each thread its own entries
  const int n = a.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / W, lt = threadIdx.x % TEAM;
  auto col_in = [&](int k) { return k < S::FULL || lt + k * TEAM < n; };

  T xr[S::XS ? 1 : CPL], xb[CPL];
#pragma unroll
  for (int k = 0; k < CPL; ++k) {
    const T v = col_in(k) ? a.x[lt + k * TEAM] : T(0);
    if constexpr (S::XS) xs[k * THREADS + threadIdx.x] = v;
    else xr[k] = v;
    xb[k] = T(0);
  }
  auto xv = [&](int k) {
    if constexpr (S::XS) return xs[k * THREADS + threadIdx.x];
    else return xr[k];
  };
  const T fb2 = FUSED ? T(2) * load_seed(a.seed) : T(0);
  FSum<T> fsum;  // of row lane / G of every group (counted once per row below)

  // group g of R rows goes to team g / gridDim.x of CTA g % gridDim.x, round by round
  const unsigned groups = (unsigned)((a.m + R - 1) / R);  // m < 2^31
  const int64_t first = blockIdx.x + (int64_t)team * gridDim.x, all = (int64_t)gridDim.x * NT;
  const unsigned step = all < groups ? (unsigned)all : groups;
  int par = 0;
  // each team by itself: one that runs out of groups leaves the FP64 unit to the others
  for (unsigned grp = first < groups ? (unsigned)first : groups; grp < groups; grp += step, par ^= 1) {
    const int64_t r0 = (int64_t)grp * R;
    const int rows = (int)(a.m - r0 < R ? a.m - r0 : R);
    const T* Ar = a.A + r0 * (int64_t)n + lt;
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
      d[r] = av[r][0] * xv(0);
#pragma unroll
      for (int k = 1; k < CPL; ++k) d[r] = fma(av[r][k], xv(k), d[r]);
    }
    T tot = reduce_rows<R>(d);
    const int row = lane / G;
    if constexpr (W > 1) {
      T* rd = red + par * WARPS * R + team * W * R;
      if (lane % G == 0) rd[(warp % W) * R + row] = tot;
      if constexpr (NT == 1) __syncthreads();
      else named_barrier(1 + team, TEAM);
      tot = rd[(lane % WG) * R + row];
#pragma unroll
      for (int i = G; i < W; i += G) tot += rd[(i + lane % G) * R + row];
#pragma unroll
      for (int o = WG / 2; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    // past the end there is no row: neither 0 times an infinite x nor, below, an infinite seed
    // times 0 is one's value
    if (row >= rows) tot = T(0);
    if (W == 1 || warp % W == 0) fsum.add(tot);  // one warp of the team: an FP64 instruction a row
    if constexpr (!FUSED) {
      if (a.y && row < rows && lane % G == 0 && (W == 1 || warp % W == 0)) a.y[r0 + row] = tot;
    } else {
      const T ybl = row < rows ? fb2 * tot : T(0);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const T yb = R == 1 ? ybl : __shfl_sync(0xffffffffu, ybl, r * G);
#pragma unroll
        for (int k = 0; k < CPL; ++k) xb[k] = fma(yb, av[r][k], xb[k]);
        if (a.gA && r < rows) {
          T* gr = a.gA + (r0 + r) * (int64_t)n + lt;
#pragma unroll
          for (int k = 0; k < CPL; ++k)
            if (col_in(k)) {
              const T v = yb * xv(k);
              gr[k * TEAM] = a.accumulate ? gr[k * TEAM] + v : v;
            }
        }
      }
    }
  }

  // the CTA's f, in thread 0: one lane per row of a group, one warp per team (a sum over the
  // whole CTA would occupy the FP64 unit for 1.3 us in CTAs of 16 warps)
  double fcta = 0.0;
  if (W == 1 || warp % W == 0) {
    double fs = fsum.get();
#pragma unroll
    for (int o = G; o < 32; o <<= 1) fs += __shfl_xor_sync(0xffffffffu, fs, o);
    if (lane == 0) fred[team] = fs;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    fcta = fred[0];
#pragma unroll
    for (int t = 1; t < NT; ++t) fcta += fred[t];
  }
  if constexpr (!FUSED) {
    finish_sum_warp<T>(fcta, a.fpart, a.counter, a.f);
    return;
  } else {
    const bool one = gridDim.x == 1;
    T* out = one ? a.gx : a.partials + (int64_t)blockIdx.x * n;
    if constexpr (NT == 1) {
#pragma unroll
      for (int k = 0; k < CPL; ++k) {
        const int j = lt + k * TEAM;
        if (col_in(k)) out[j] = one && a.accumulate ? out[j] + xb[k] : xb[k];
      }
    } else {
#pragma unroll
      for (int k = 0; k < CPL; ++k) xbs[team * TEAM * CPL + lt + k * TEAM] = xb[k];
      __syncthreads();
      for (int j = threadIdx.x; j < n; j += THREADS) {
        T s = xbs[j];
#pragma unroll
        for (int t = 1; t < NT; ++t) s += xbs[t * TEAM * CPL + j];
        out[j] = one && a.accumulate ? out[j] + s : s;
      }
    }
    if (threadIdx.x == 0) {
      if (one) {
        if (a.f) *a.f = (T)fcta;
      } else {
        a.fpart[blockIdx.x] = fcta;
      }
    }
    if (one || !a.last) return;
    // few partials of few columns: the CTA that arrives last sums them, thread (j, pg)
    // partials pg, pg + PG, ... of column j, the PG sums then in pg order
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(a.counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int parts = gridDim.x;
    int cw = 32;
    while (cw < n) cw *= 2;  // n <= 128 here
    const int pgs = THREADS / cw, j = threadIdx.x % cw, pg = threadIdx.x / cw;
    T s = T(0);
    if (j < n) {
#pragma unroll 8
      for (int c = pg; c < parts; c += pgs) s += __ldcg(a.partials + (int64_t)c * n + j);
    }
    __syncthreads();
    xbs[threadIdx.x] = s;
    __syncthreads();
    if (pg == 0 && j < n) {
      for (int q = 1; q < pgs; ++q) s += xbs[q * cw + j];
      a.gx[j] = a.accumulate ? a.gx[j] + s : s;
    }
    if (warp == 0) {
      double fs = 0.0;
      for (int i = lane; i < parts; i += 8 * 32) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = i + 32 * u < parts ? __ldcg(a.fpart + i + 32 * u) : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u) fs += v[u];
      }
      fs = warp_sum(fs);
      if (lane == 0) {
        if (a.f) *a.f = (T)fs;
        *a.counter = 0u;
      }
    }
  }
}

// ---------------------------------------------------------------- host ----
// Calls go(shape) with the shape for rows of n entries.  team: the caller's threads per team
// (0: the smallest that holds the row in 8 columns a lane; 512 threads above 2048 entries).
//   up to 8 warps:  8 columns a lane at most, 8 rows a step up to 4 of them, else 4 (a team
//                   of 8 warps: 4), R * CPL <= 32 values of A in a lane's registers;
//   16 warps:       n <= 4096 4 rows a step, then x in shared memory and 2 rows (FP32 4) to
//                   8192 entries, 1 (FP32 2) to 12288, where the forward, which keeps no row
//                   for a reverse, still takes 2 (FP32 4).
//   FP64 rows of more than 128 entries, at most two an SM, are taken one a step by teams of two
//   warps or more: several rows on one team leave the other SMs idle while its FP64 unit works
//   through them, and the rows missing from a step cost the unit as much as rows (value and
//   gradient of 100 x 2001 11.7 us, 9.0 with a row a step; of 150 x 256 9.6 and 7.1; the value
//   of 80 x 12288 12.1 and 8.9).  Rows of up to 256 entries on one CTA stay with its eight
//   one-warp teams (31 x 129 5.9 us, 6.7 one a step).
template <typename T, int W, typename Go>
static void qr_small(int64_t n, const Go& go) {
  switch ((n + 32 * W - 1) / (32 * W)) {
#define KG_CPL(c) \
  case c: go(QrShape<W, c, c - 1, (c <= 4 && W < 8 ? 8 : 4), false>{}); break;
    KG_CPL(1) KG_CPL(2) KG_CPL(3) KG_CPL(4) KG_CPL(5) KG_CPL(6) KG_CPL(7) KG_CPL(8)
#undef KG_CPL
  }
}

template <typename T, bool FUSED, typename Go>
static void qr_with_shape(int64_t m, int64_t n, int team, const Go& go) {
  constexpr int R2 = sizeof(T) == 8 ? 2 : 4, R1 = FUSED ? R2 / 2 : R2, R0 = sizeof(T) == 8 ? 1 : R1;
  int w = team / 32;
  if (!team)
    for (w = 1; (int64_t)256 * w < n && w < 16;) w *= 2;
  const bool few = sizeof(T) == 8 && m <= 2 * (int64_t)num_sms() && (w >= 2 || (!team && n > 128 && m * n > 4096));
  if (few && n <= 8192) {
    switch (w) {
      case 1: return go(QrShape<2, 4, 0, 1, false>{});
      case 2: return go(QrShape<2, 8, 0, 1, false>{});
      case 4: return go(QrShape<4, 8, 0, 1, false>{});
      case 8: return go(QrShape<8, 8, 0, 1, false>{});
    }
    return n <= 4096 ? go(QrShape<16, 8, 0, 1, false>{}) : go(QrShape<16, 16, 8, 1, true>{});
  }
  switch (w) {
    case 1: return qr_small<T, 1>(n, go);
    case 2: return qr_small<T, 2>(n, go);
    case 4: return qr_small<T, 4>(n, go);
    case 8: return qr_small<T, 8>(n, go);
  }
  const int64_t c = (n + 511) / 512;
  if (c <= 4) return go(QrShape<16, 4, 0, 4, false>{});  // a caller's team of 512 only
  if (c == 5) return go(QrShape<16, 5, 4, 4, false>{});
  if (c == 6) return go(QrShape<16, 6, 5, 4, false>{});
  if (c == 7) return go(QrShape<16, 7, 6, 4, false>{});
  if (c == 8) return go(QrShape<16, 8, 7, 4, false>{});
  if (c <= 10) return go(QrShape<16, 10, 8, R2, true>{});
  if (c <= 12) return go(QrShape<16, 12, 10, R2, true>{});
  if (c <= 14) return go(QrShape<16, 14, 12, R2, true>{});
  if (c <= 16) return go(QrShape<16, 16, 14, R2, true>{});
  if (few) {
    if (c <= 18) return go(QrShape<16, 18, 16, R0, true>{});
    if (c <= 20) return go(QrShape<16, 20, 18, R0, true>{});
    if (c <= 22) return go(QrShape<16, 22, 20, R0, true>{});
    return go(QrShape<16, 24, 22, R0, true>{});
  }
  if (c <= 18) return go(QrShape<16, 18, 16, R1, true>{});
  if (c <= 20) return go(QrShape<16, 20, 18, R1, true>{});
  if (c <= 22) return go(QrShape<16, 22, 20, R1, true>{});
  return go(QrShape<16, 24, 22, R1, true>{});
}

template <typename T, typename S>
constexpr size_t qr_smem() { return S::XS ? sizeof(T) * S::CPL * S::THREADS : 0; }

// One wave of resident CTAs, or fewer when a quarter of an SM's warps (one a scheduler,
// which its FP64 unit needs no more than) or a whole CTA has a group of rows.
//   - The gradient of up to 4096 entries is one CTA's, which writes it itself, when its teams
//     need at most 2 rounds (FP64) or 5: 64 x 64 5.6 us and 7.1 with several CTAs, 128 x 8 6.6
//     and 6.4, 256 x 8 10.6 and 6.5; FP32 300 x 8 5.0 and 5.5, 512 x 8 6.9 and 5.3.
//   - The forward has no partials to sum: several CTAs are as fast at 8 rows and faster above
//     (FP32 300 x 8 5.0 and 3.9).  In FP64 it spreads its groups over the SMs, one FP64 unit
//     each: 150 x 16 7.6 -> 4.6, 4 x 700 5.9 -> 4.3.
template <typename T>
static int qr_grid_t(int64_t m, int64_t n, int team, bool eval) {
  int64_t grid = 1;
  const bool spread = eval && sizeof(T) == 8;
  qr_with_shape<T, true>(m, n, team, [&](auto shape) {
    using S = decltype(shape);
    constexpr int one = S::R * S::NT * (sizeof(T) == 8 ? 2 : 5);  // rows of one CTA
    if (!eval && m * n <= 4096 && m <= one) return;
    int occ = 0;
    auto kern = qf_rows_kernel<T, S, true>;
    if (set_smem_once(kern, qr_smem<T, S>()) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, S::THREADS, qr_smem<T, S>()) != cudaSuccess ||
        occ < 1) {
      cudaGetLastError();
      occ = 1;
    }
    const int64_t step = (int64_t)S::R * std::max(1, 4 / S::W);
    grid = std::min<int64_t>((m + step - 1) / step, (int64_t)num_sms() * occ);
    if (spread) grid = std::max(grid, std::min<int64_t>((m + S::R - 1) / S::R, num_sms()));
  });
  return (int)std::max<int64_t>(1, grid);
}

int qf_rows_grid(int dtype, int64_t m, int64_t n, int team, bool eval) {
  return dtype == KG_F64 ? qr_grid_t<double>(m, n, team, eval) : qr_grid_t<float>(m, n, team, eval);
}

template <typename T, bool FUSED>
static cudaError_t launch_rows(int grid, int team, const QrArgs<T>& a, cudaStream_t s) {
  cudaError_t e = cudaErrorInvalidValue;
  prof_begin(s, FUSED ? "qf_rows_kernel<fused>" : "qf_rows_kernel<eval>");
  qr_with_shape<T, FUSED>(a.m, a.n, team, [&](auto shape) {
    using S = decltype(shape);
    auto kern = qf_rows_kernel<T, S, FUSED>;
    if (S::XS && (e = set_smem_once(kern, qr_smem<T, S>())) != cudaSuccess) return;
    kern<<<grid, S::THREADS, qr_smem<T, S>(), s>>>(a);
    e = cudaGetLastError();
  });
  prof_end(s);
  count_launch();
  return e;
}

// The last CTA sums the partials itself up to this many bytes of them and this many columns,
// one pass of at least two threads a column: 200 x 60 FP64 7.0 us, with a second launch 8.6;
// 30 x 501, two passes, 12.7 and 8.2.
constexpr int64_t QR_LAST_BYTES = 64 << 10, QR_LAST_N = 128;

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
  a.last = c.counter && c.n <= QR_LAST_N && (int64_t)c.grid * c.n * (int64_t)sizeof(T) <= QR_LAST_BYTES;
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
