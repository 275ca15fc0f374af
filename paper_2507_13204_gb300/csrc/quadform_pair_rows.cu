// Dense ||A x||^2 in float pairs for rows of 1024 to 4096 entries (the forward: to 8192):
// forward and one-launch value-and-gradient, several rows a step.
//
// Streamed a row at a time (quadform_pair.cu), a step's CTA barrier and its two
// reductions cost more than the 8 to 32 KB row's own arithmetic.  Here a CTA of 8 warps
// takes R rows at once, as the native kernels of quadform_rows.cu do: thread t holds the
// column pairs jp = t + 256 k (k < KP) in packed pairs, the rows' loads are issued
// together (64 KB a CTA in flight, two CTAs an SM; the next step's rows are prefetched
// into L2), and one transposed butterfly, one barrier and one butterfly over the warps'
// sums reduce all R dot products.  R KP entry pairs of A stay in registers for the
// reverse: R = 4 up to 4 column pairs a thread (n <= 2048), then 2 with x in shared
// memory.  xbar accumulates in registers.  Steps go round-robin over the grid.
//
// Measured (value and gradient, device time, against a row at a time): 2000 x 1500 21.4 ->
// 11.1 us, 40000 x 1024 236 -> 68, 40000 x 2048 294 -> 121 (5.4 TB/s), 20000 x 2500
// 141 -> 81; the forward 206 -> 51, 238 -> 100 (6.5 TB/s), 135 -> 66.  The rest of the
// gradient is issue: 24 packed and scalar FP32 operations an entry.
//
// The CTAs' partials are summed in a fixed order: behind a bounded grid barrier in the
// same (cooperative) launch, every CTA taking its share of the columns, or by a second
// kernel with the same bits when the grid cannot be resident at once.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "kg_device.cuh"
#include "kg_internal.h"
#include "kg_pair.cuh"
#include "kg_pair2.cuh"

namespace kg {

constexpr int PR_NGRAD = 4096;  // longest row of the gradient, and of CTAs of 256 threads
constexpr int PR_NEVAL = 8192;  // longest row of the forward, in CTAs of 512 threads above PR_NGRAD
constexpr int PR_RT = 256;      // threads that sum the partials

struct PrArgs {
  const double* A;  // FP64 rows, or (PREP) rows of float pairs, two entries as (h0, h1, l0, l1)
  const double* x;
  int64_t m;
  int n;            // even
  const double* seed;
  float4* partials;  // [grid][n / 2] of (s0, l0, s1, l1)
  double* fpart;
  unsigned* counter;
  double* f;
  double* gx;
  int accumulate;
  unsigned* err;
};

__device__ __forceinline__ Acc pr_shfl(Acc a, int o) {
  Acc b;
  b.s = __shfl_xor_sync(0xffffffffu, a.s, o);
  b.l = __shfl_xor_sync(0xffffffffu, a.l, o);
  return b;
}

// Columns [j0, j1) (pairs) of the gradient from the CTAs' partials, by 256 threads: thread
// (cx, py) adds partials py, py + 256 / CX, ... of pair cx of each block of CX, the lanes of
// a warp that hold the same pair add by a butterfly, and the eight warps' sums are added in
// order.  The order depends on neither the CTA nor the range.
template <int CX>
__device__ __forceinline__ void pr_reduce_block(const float4* partials, int nparts, int np2, int j0, int j1,
                                                double* gx, int accumulate, Acc (*red)[16][2]) {
  constexpr int PY = PR_RT / CX;
  const int cx = threadIdx.x % CX, py = threadIdx.x / CX, warp = threadIdx.x >> 5;
  for (int jb = j0; jb < j1; jb += CX) {
    const int jp = jb + cx;
    Acc s0 = acc_zero(), s1 = acc_zero();
    if (jp < j1) {
      for (int c = py; c < nparts; c += 8 * PY) {
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c + PY * u < nparts) v[u] = __ldcg(partials + (int64_t)(c + PY * u) * np2 + jp);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c + PY * u < nparts) {
            s0 = acc_add(s0, Acc{v[u].x, v[u].y});
            s1 = acc_add(s1, Acc{v[u].z, v[u].w});
          }
      }
    }
#pragma unroll
    for (int o = CX; o < 32; o <<= 1) {
      s0 = acc_add(s0, pr_shfl(s0, o));
      s1 = acc_add(s1, pr_shfl(s1, o));
    }
    if ((threadIdx.x & 31) < CX) {
      red[warp][cx][0] = s0;
      red[warp][cx][1] = s1;
    }
    __syncthreads();
    if (threadIdx.x < CX && jp < j1) {
      Acc t0 = red[0][cx][0], t1 = red[0][cx][1];
#pragma unroll
      for (int w = 1; w < PR_RT / 32; ++w) {
        t0 = acc_add(t0, red[w][cx][0]);
        t1 = acc_add(t1, red[w][cx][1]);
      }
      const double g0 = pair_to_double(acc_pair(t0)), g1 = pair_to_double(acc_pair(t1));
      double2* o = reinterpret_cast<double2*>(gx) + jp;
      if (accumulate) {
        const double2 old = *o;
        *o = make_double2(old.x + g0, old.y + g1);
      } else {
        *o = make_double2(g0, g1);
      }
    }
    __syncthreads();
  }
}

// Few partials leave each CTA many columns: 16 pairs a block then (75 partials of 1024
// pairs in 5 us with blocks of 4, the tail of a 300 x 2048 gradient), 4 otherwise, so that
// one round of loads takes up to 512 partials.
__device__ __forceinline__ void pr_reduce_columns(const float4* partials, int nparts, int np2, int j0, int j1,
                                                  double* gx, int accumulate, Acc (*red)[16][2]) {
  if (nparts <= 128) pr_reduce_block<16>(partials, nparts, np2, j0, j1, gx, accumulate, red);
  else pr_reduce_block<4>(partials, nparts, np2, j0, j1, gx, accumulate, red);
}

__device__ __forceinline__ void pr_reduce_f(const double* fpart, int nparts, double* f, double* scratch) {
  double fs = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) fs += __ldcg(fpart + i);
  fs = block_sum(fs, scratch);
  if (threadIdx.x == 0) *f = fs;
}

// Sum of the R rows' values over a warp: lane l ends with the total of row l / (32 / R).
template <int R>
__device__ __forceinline__ Acc pr_reduce_rows(Acc (&d)[R]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int w = R / 2; w > 0; w >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) d[i] = acc_add(up ? d[i + w] : d[i], pr_shfl(up ? d[i] : d[i + w], o));
  }
#pragma unroll
  for (; o > 0; o >>= 1) d[0] = acc_add(d[0], pr_shfl(d[0], o));
  return d[0];
}

// NTH threads, KP column pairs a thread, R rows a step.  XS: x is kept in shared memory (a
// thread of more than 4 column pairs has no registers left for it).
template <int NTH, int KP, int R, bool XS, bool FUSED, bool PREP, bool GRIDRED>
__global__ void __launch_bounds__(NTH, 512 / NTH) qf_pair_rows_kernel(PrArgs a) {
  constexpr int W = NTH / 32, G = 32 / R;  // G lanes hold a row's total
  __shared__ Acc sums[2][W][R];
  __shared__ Acc red[FUSED ? W : 1][16][2];
  __shared__ double fred[FUSED ? 32 : 1];
  __shared__ int go;
  extern __shared__ __align__(16) float4 xs[];  // XS: [KP][NTH]
  const int np2 = a.n >> 1, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  auto in_row = [&](int k) { return k < KP - 1 || t + k * NTH < np2; };
  Pair2 xr[XS ? 1 : KP];
  Acc2 xb[KP];
  bool bad = false;
#pragma unroll
  for (int k = 0; k < KP; ++k) {
    const double2 xv = t + k * NTH < np2 ? reinterpret_cast<const double2*>(a.x)[t + k * NTH]
                                         : make_double2(0.0, 0.0);
    bad |= !pair_in_range(xv.x) || !pair_in_range(xv.y);
    const Pair p0 = split_f64(xv.x), p1 = split_f64(xv.y);
    if constexpr (XS) xs[k * NTH + t] = pair2_entry(p0, p1);  // read by this thread only
    else xr[k] = pair2_of(p0, p1);
    xb[k] = acc2_zero();
  }
  auto xp = [&](int k) {
    if constexpr (XS) return pair2_load(xs + k * NTH + t);
    else return xr[k];
  };
  Pair fb2{2.f, 0.f};
  if (FUSED) {
    const double fb = a.seed ? *a.seed : 1.0;
    bad |= !pair_in_range(2.0 * fb);
    fb2 = split_f64(2.0 * fb);
  }
  if (bad) set_error(a.err, ERRBIT_RANGE);
  Acc facc = acc_zero();

  const int64_t steps = (a.m + R - 1) / R;
  int par = 0, done = 0;
  for (int64_t g = blockIdx.x; g < steps; g += gridDim.x, par ^= 1) {
    const int64_t r0 = g * R;
    const int rows = (int)(a.m - r0 < R ? a.m - r0 : R);
    if (t == 0 && g + gridDim.x < steps) {
      const int64_t rn = (g + gridDim.x) * R;
      const int64_t cnt = a.m - rn < R ? a.m - rn : R;
      prefetch_l2_bulk(a.A + rn * a.n, (uint32_t)(cnt * a.n * 8));
    }
    Pair2 av[R][KP];
    if constexpr (PREP) {
      const float4* Ar = reinterpret_cast<const float4*>(a.A) + r0 * np2 + t;
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int k = 0; k < KP; ++k) {
          ulonglong2 q = make_ulonglong2(0ull, 0ull);
          if (r < rows && in_row(k)) q = __ldcs(reinterpret_cast<const ulonglong2*>(Ar + k * NTH));
          av[r][k] = Pair2{F2{q.x}, F2{q.y}};
        }
        Ar += np2;
      }
    } else {
      const double2* Ar = reinterpret_cast<const double2*>(a.A) + r0 * np2 + t;
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int k = 0; k < KP; ++k) {
          double2 q = make_double2(0.0, 0.0);
          if (r < rows && in_row(k)) q = __ldcs(Ar + k * NTH);
          av[r][k] = pair2_of(split_f64(q.x), split_f64(q.y));
        }
        Ar += np2;
      }
    }
    Acc d[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      Acc2 y = acc2_prod(av[r][0], xp(0));
#pragma unroll
      for (int k = 1; k < KP; ++k) acc2_fma(y, av[r][k], xp(k));
      d[r] = acc2_sum(y);
    }
    Acc tot = pr_reduce_rows<R>(d);
    const int row = lane / G;
    if (lane % G == 0) sums[par][warp][row] = tot;
    __syncthreads();
    tot = sums[par][lane % (W < G ? W : G)][row];
#pragma unroll
    for (int i = G; i < W; i += G) tot = acc_add(tot, sums[par][i + lane % G][row]);
#pragma unroll
    for (int o = (W < G ? W : G) / 2; o > 0; o >>= 1) tot = acc_add(tot, pr_shfl(tot, o));
    const Pair y = acc_pair(tot);  // rows past the end: zero
    if (warp == 0) {
      const Pair y2 = pair_mul(y, y);
      facc = acc_add(facc, Acc{y2.h, y2.l});
    }
    ++done;
    if constexpr (FUSED) {
      const Pair ybl = pair_mul(fb2, y);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const Pair2 yb = pair2_dup(Pair{__shfl_sync(0xffffffffu, ybl.h, r * G),
                                        __shfl_sync(0xffffffffu, ybl.l, r * G)});
#pragma unroll
        for (int k = 0; k < KP; ++k) acc2_fma(xb[k], av[r][k], yb);
      }
      if ((done & 3) == 0) {
#pragma unroll
        for (int k = 0; k < KP; ++k) acc2_renorm(xb[k]);
      }
    }
    if ((done & 7) == 7) acc_renorm(facc);
  }

  // the CTA's f: warp 0's rows, one lane each, in pairs (an FP64 sum over the CTA is 0.7 us)
  if (warp == 0) {
#pragma unroll
    for (int o = G; o < 32; o <<= 1) facc = acc_add(facc, pr_shfl(facc, o));
  }
  const double fcta = acc_to_double(facc);  // in thread 0
  if constexpr (!FUSED) {
    finish_sum_warp<double>(fcta, a.fpart, a.counter, a.f);
  } else {
    float4* out = a.partials + (int64_t)blockIdx.x * np2;
#pragma unroll
    for (int k = 0; k < KP; ++k)
      if (in_row(k)) {
        const Pair p0 = acc_pair(acc2_x(xb[k])), p1 = acc_pair(acc2_y(xb[k]));
        out[t + k * NTH] = make_float4(p0.h, p0.l, p1.h, p1.l);
      }
    if (t == 0) a.fpart[blockIdx.x] = fcta;
    if constexpr (GRIDRED) {
      __syncthreads();
      if (t == 0) go = grid_arrive_and_wait(a.counter + 2, a.err, ERRBIT_TIMEOUT);
      __syncthreads();
      if (go) {
        const int nparts = gridDim.x, b = blockIdx.x;
        const int j0 = (int)((int64_t)b * np2 / nparts), j1 = (int)((int64_t)(b + 1) * np2 / nparts);
        pr_reduce_columns(a.partials, nparts, np2, j0, j1, a.gx, a.accumulate, red);
        if (b == 0 && a.f) pr_reduce_f(a.fpart, nparts, a.f, fred);
      }
      if (t == 0) grid_depart(a.counter + 2, a.counter + 3);
    }
  }
}

// The same sums as a second, dependent launch: block b takes 16 column pairs.
__global__ void __launch_bounds__(PR_RT) qf_pair_rows_reduce_kernel(PrArgs a, int nparts) {
  __shared__ Acc red[PR_RT / 32][16][2];
  __shared__ double fred[32];
  grid_dependency_wait();
  const int np2 = a.n >> 1, j0 = 16 * blockIdx.x;
  pr_reduce_columns(a.partials, nparts, np2, j0, min(j0 + 16, np2), a.gx, a.accumulate, red);
  if (blockIdx.x == 0 && a.f) pr_reduce_f(a.fpart, nparts, a.f, fred);
}

// ---------------------------------------------------------------- host ----
struct PrShape {
  int threads, kp, rows;
  bool xs;
};

// Threads, column pairs a thread and rows a step for rows of n entries.
static PrShape pr_shape(int64_t n) {
  const int th = n <= PR_NGRAD ? 256 : 512;
  const int kp = (int)((n / 2 + th - 1) / th);
  return PrShape{th, kp, kp <= 4 ? 4 : 2, kp > 4};
}

template <bool FUSED, bool PREP, bool GRIDRED, typename Go>
static void pr_with_kernel(int64_t n, const Go& go) {
  const PrShape sh = pr_shape(n);
#define KG_PR(T, K)                    \
  if (sh.threads == T && sh.kp == K)   \
    return go(qf_pair_rows_kernel<T, K, (K <= 4 ? 4 : 2), (K > 4), FUSED, PREP, GRIDRED>);
  KG_PR(256, 2) KG_PR(256, 3) KG_PR(256, 4) KG_PR(256, 5) KG_PR(256, 6) KG_PR(256, 7) KG_PR(256, 8)
  if constexpr (!FUSED) {
    KG_PR(512, 5) KG_PR(512, 6) KG_PR(512, 7) KG_PR(512, 8)
  }
#undef KG_PR
}

static size_t pr_smem(int64_t n) {
  const PrShape sh = pr_shape(n);
  return sh.xs ? (size_t)sh.kp * sh.threads * 16 : 0;
}

template <typename K>
static int pr_resident(K kern, int64_t n) {
  int occ = 0;
  if (set_smem_once(kern, pr_smem(n)) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, pr_shape(n).threads, pr_smem(n)) != cudaSuccess) {
    cudaGetLastError();
    occ = 0;
  }
  return occ;
}

// Rows of 2050 to 4096 entries run here when there are 4 rows an SM, the gradient of more than
// 3600 entries when there are 8: 610 x 2560 takes 10.6 us here and 13.2 by the warp-specialized
// kernel, 850 x 3584 13.8 and 14.5, 700 x 3700 15.7 and 13.5, 1216 x 4096 16.0 and 16.6, 2432 x
// 4096 22.8 and 25.4, 20000 x 4096 115 and 134.  Longer rows: the gradient is the warp-
// specialized kernel's (10000 x 5000 91 against 87 there, 10000 x 8000 129 against 107), the
// forward this one's (74.7 against 87, 101 against 105).
bool qf_pair_rows_supported(int64_t m, int64_t n, bool eval) {
  if (n <= 2048) return true;
  return n <= (eval ? PR_NEVAL : PR_NGRAD) && m >= (eval || n <= 3600 ? 4 : 8) * (int64_t)num_sms();
}

// One wave of resident CTAs, or one a step.  Fewer, so that all CTAs take as many steps (305
// steps on 153 CTAs instead of 304), left SMs with half their warps: 610 x 4096 16.7 -> 13.8 us,
// 610 x 2560 11.9 -> 10.6, 1400 x 1500 11.8 -> 10.8; more partials cost at most 0.3 us.
int qf_pair_rows_grid(const kg_problem* p) {
  int occ = 0;
  pr_with_kernel<true, true, true>(p->n, [&](auto k) { occ = pr_resident(k, p->n); });
  const int rows = pr_shape(p->n).rows;
  const int64_t steps = (p->m + rows - 1) / rows;
  return (int)std::min(steps, (int64_t)num_sms() * std::max(occ, 1));
}

// Whether the gradient runs as one cooperative launch.  A grid of at most 64 CTAs leaves
// each too many columns to sum: a second launch then.
bool qf_pair_rows_coop_fits(const kg_problem* p) {
  if (const char* env = std::getenv("KG_TEST_NO_COOP"))
    if (std::atoi(env) == 1) return false;
  if (p->qf.grid <= 64) return false;
  int dev = 0, coop = 0, occ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
    return false;
  if (p->aprep) pr_with_kernel<true, true, true>(p->n, [&](auto k) { occ = pr_resident(k, p->n); });
  else pr_with_kernel<true, false, true>(p->n, [&](auto k) { occ = pr_resident(k, p->n); });
  return (int64_t)occ * num_sms() >= p->qf.grid;
}

static PrArgs pr_args(kg_problem* p, const void* x, const void* seed, void* f) {
  PrArgs a{};
  a.A = static_cast<const double*>(p->aprep ? p->aprep : p->data0);
  a.x = static_cast<const double*>(x);
  a.m = p->m;
  a.n = (int)p->n;
  a.seed = static_cast<const double*>(seed);
  a.partials = static_cast<float4*>(p->partials);
  a.fpart = p->fpart;
  a.counter = p->counter;
  a.f = static_cast<double*>(f);
  a.err = p->err;
  return a;
}

template <bool FUSED, bool GRIDRED>
static cudaError_t launch_pr(const kg_problem* p, const PrArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p->qf.grid);
  cfg.blockDim = dim3(pr_shape(p->n).threads);
  cfg.dynamicSmemBytes = pr_smem(p->n);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = GRIDRED ? 1 : 0;
  cudaError_t e = cudaErrorInvalidValue;
  auto go = [&](auto k) {
    if ((e = set_smem_once(k, cfg.dynamicSmemBytes)) == cudaSuccess) e = cudaLaunchKernelEx(&cfg, k, a);
  };
  if (p->aprep) pr_with_kernel<FUSED, true, GRIDRED>(p->n, go);
  else pr_with_kernel<FUSED, false, GRIDRED>(p->n, go);
  count_launch();
  return e;
}

kg_status qf_pair_rows_eval(kg_problem* p, const void* x, void* f, cudaStream_t s) {
  prof_begin(s, "qf_pair_rows_kernel<eval>");
  cudaError_t e = launch_pr<false, false>(p, pr_args(p, x, nullptr, f), s);
  prof_end(s);
  return e == cudaSuccess ? KG_OK : cuda_fail(e, "qf pair forward kernel");
}

kg_status qf_pair_rows_grad(kg_problem* p, const void* x, void* f, void* gx, const void* seed,
                            int accumulate, cudaStream_t s) {
  PrArgs a = pr_args(p, x, seed, f);
  a.gx = static_cast<double*>(gx);
  a.accumulate = accumulate;
  cudaError_t e;
  if (p->qf.coop) {
    prof_begin(s, "qf_pair_rows_kernel<fused, grid reduction>");
    e = launch_pr<true, true>(p, a, s);
    prof_end(s);
    if (e == cudaSuccess) return KG_OK;
    if (e != cudaErrorCooperativeLaunchTooLarge) return cuda_fail(e, "qf pair fused kernel");
    cudaGetLastError();  // the grid is not resident at once here: two launches from now on
    p->qf.coop = 0;
  }
  prof_begin(s, "qf_pair_rows_kernel<fused>");
  e = launch_pr<true, false>(p, a, s);
  prof_end(s);
  if (e != cudaSuccess) return cuda_fail(e, "qf pair fused kernel");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((p->n / 2 + 15) / 16));
  cfg.blockDim = dim3(PR_RT);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, qf_pair_rows_reduce_kernel, a, p->qf.grid);
  count_launch();
  return e == cudaSuccess ? KG_OK : cuda_fail(e, "qf pair reduce kernel");
}

}  // namespace kg
