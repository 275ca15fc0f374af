// Row passes of the sparse ||A x||^2 (forward, fused atomic scatter, row pass of the CSC
// strategy) a block of consecutive rows at a time.
//
// What bounds them is random access to L2: one gather of x and, with the atomic scatter, one
// reduction into xbar per stored entry.  A team of lanes per row (spquadform.cu) leaves
// lanes idle at every row's end and walks a long row a few gathers at a time, then again
// for its reverse.  Here a CTA takes RB rows with their (at most CAP) stored entries:
//   A  thread t takes entries t, t + 256, ...: their columns and values stream in full
//      lines, all their gathers are in flight together, whatever the rows' lengths; the
//      products go to shared memory, columns, values and gathered x stay in registers;
//   B  TW lanes per row add the row's products (fixed order) and publish ybar_i; they also
//      note each entry's row;
//   C  thread t scatters its entries of A with their rows' ybar (full warps: the FP64 add
//      that ends a float-pair product costs the FP64 unit the same for one lane as for 32).
// Two CTA barriers a block; three or four CTAs an SM overlap their phases.  A block with
// more than CAP entries (long rows) is walked by a warp per row instead.
//
// Measured against the row teams: 300001 x 200003, 1..60 entries a row, FP32, both gradients
// (row pass and CSC gather) 140 -> 112 us; 2^20 x 2^20, 8..24 a row, FP64 atomic gradient
// 186 -> 177 us, of which 135 are its 16.8e6 gathers and reductions at the measured L2
// rates and the rest mostly the matrix itself, 201 MB through the same L2.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "kg_device.cuh"
#include "kg_internal.h"
#include "kg_pair.cuh"

namespace kg {

constexpr int SS_THREADS = 256;
constexpr int SS_K = 6;                      // entries a thread
constexpr int SS_CAP = SS_THREADS * SS_K;    // entries a block
enum { SS_EVAL = 0, SS_ATOMIC = 1, SS_ROWPASS = 2 };
// CTAs an SM.  Gathers and reductions together slow each other down at L2 when more of
// them are outstanding: the 2^20-row FP64 gradient takes 211, 177, 181 us with 2, 3 and 4
// (249 with 5 of 1280 entries); the row pass, which only gathers, 119 and 112 with 3 and 4.
constexpr int ss_ctas(int mode) { return mode == SS_ATOMIC ? 3 : 4; }
enum { SS_F32 = 0, SS_F64 = 1, SS_PAIR = 2 };

template <int AR> struct SsTypes;
// val: a stored value; sum: a row sum; ent: an entry's product, or its factors
template <> struct SsTypes<SS_F32> { using T = float; using val = float; using sum = float; using ent = float2; };
template <> struct SsTypes<SS_F64> { using T = double; using val = double; using sum = double; using ent = double2; };
template <> struct SsTypes<SS_PAIR> { using T = double; using val = float2; using sum = Acc; using ent = Acc; };

template <int AR>
struct SsArgs {
  using T = typename SsTypes<AR>::T;
  const int* rowptr;
  const int* col;
  const typename SsTypes<AR>::val* val;
  const T* x;
  int64_t m;
  const T* seed;
  T* gx;
  T* gval;
  void* y;  // ROWPASS: T, or float2 pairs
  int accumulate;
  double* fpart;
  unsigned* counter;
  T* f;
  unsigned* err;
};

// One entry: the gathered x (pairs: split) and its contribution to the row sum.
template <int AR>
__device__ __forceinline__ typename SsTypes<AR>::val ss_x(typename SsTypes<AR>::T x, bool& bad) {
  if constexpr (AR == SS_PAIR) {
    bad |= !pair_in_range(x);
    const Pair p = split_f64(x);
    return make_float2(p.h, p.l);
  } else {
    return x;
  }
}

template <int AR>
__device__ __forceinline__ void ss_add(typename SsTypes<AR>::sum& s, typename SsTypes<AR>::val v,
                                       typename SsTypes<AR>::val x) {
  if constexpr (AR == SS_PAIR) acc_fma(s, v.x, v.y, x.x, x.y);
  else s = fma(v, x, s);
}

template <int AR>
__device__ __forceinline__ typename SsTypes<AR>::sum ss_team_sum(typename SsTypes<AR>::sum s, int tw) {
  for (int o = tw >> 1; o > 0; o >>= 1) {
    if constexpr (AR == SS_PAIR)
      s = acc_add(s, Acc{__shfl_xor_sync(0xffffffffu, s.s, o), __shfl_xor_sync(0xffffffffu, s.l, o)});
    else
      s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  return s;
}

template <int AR, int MODE, int TW>
__global__ void __launch_bounds__(SS_THREADS, ss_ctas(MODE)) spq_stream_kernel(SsArgs<AR> a) {
  using T = typename SsTypes<AR>::T;
  using val = typename SsTypes<AR>::val;
  using sum = typename SsTypes<AR>::sum;
  using ent = typename SsTypes<AR>::ent;
  // ybar, and y before it is doubled: a T, or a pair
  using yv = std::conditional_t<AR == SS_PAIR, float2, T>;
  constexpr int RB = SS_THREADS / TW;
  __shared__ ent ents[SS_CAP];
  __shared__ uint8_t rid[MODE == SS_EVAL ? 1 : SS_CAP];
  __shared__ yv ybs[MODE == SS_EVAL ? 1 : RB];
  __shared__ double red[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int trow = tid / TW, tl = tid % TW;
  bool bad = false;
  Pair fb2p{0.f, 0.f};
  T fb2 = T(0);
  if constexpr (MODE != SS_EVAL) {
    fb2 = T(2) * load_seed(a.seed);
    if constexpr (AR == SS_PAIR) {
      bad |= !pair_in_range(fb2);
      fb2p = split_f64(fb2);
    }
  }
  std::conditional_t<AR == SS_PAIR, Acc, FSum<T>> fa{};
  int nf = 0;
  // y of a row from its sum: counts it in f, stores it (ROWPASS) and returns ybar
  auto finish_row = [&](int64_t i, sum s) {
    yv yb{};
    if constexpr (AR == SS_PAIR) {
      const Pair y = acc_pair(s);
      const Pair y2 = pair_mul(y, y);
      fa = acc_add(fa, Acc{y2.h, y2.l});
      if ((++nf & 31) == 0) acc_renorm(fa);
      if constexpr (MODE == SS_ROWPASS) static_cast<float2*>(a.y)[i] = make_float2(y.h, y.l);
      const Pair b = pair_mul(fb2p, y);
      yb = make_float2(b.h, b.l);
    } else {
      fa.add(s);
      if constexpr (MODE == SS_ROWPASS) static_cast<T*>(a.y)[i] = s;
      yb = fb2 * s;
    }
    return yb;
  };
  auto times = [&](val v, yv yb) -> T {
    if constexpr (AR == SS_PAIR) return pair_to_double_fast(pair_mul(Pair{v.x, v.y}, Pair{yb.x, yb.y}));
    else return v * yb;
  };
  auto scatter = [&](int p, int c, val v, val x, yv yb) {
    if constexpr (MODE == SS_ATOMIC) red_add(a.gx + c, times(v, yb));
    if (a.gval) {
      const T g = times(x, yb);
      a.gval[p] = a.accumulate ? a.gval[p] + g : g;
    }
  };

  const int64_t nblk = (a.m + RB - 1) / RB;
  auto bound = [&](int64_t blk) { return __ldg(a.rowptr + (blk * RB < a.m ? blk * RB : a.m)); };
  int pb = blockIdx.x < nblk ? bound(blockIdx.x) : 0, pe = blockIdx.x < nblk ? bound(blockIdx.x + 1) : 0;
  for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    const int64_t row0 = blk * RB;
    const int cnt = pe - pb, p0 = pb;
    const int nrow = (int)(a.m - row0 < RB ? a.m - row0 : RB);
    const bool act = trow < nrow;
    const int q0 = act ? __ldg(a.rowptr + row0 + trow) - p0 : 0;
    const int q1 = act ? __ldg(a.rowptr + row0 + trow + 1) - p0 : 0;
    if (blk + gridDim.x < nblk) {  // the next block's bounds, behind this one's work
      pb = bound(blk + gridDim.x);
      pe = bound(blk + gridDim.x + 1);
    }
    if (cnt <= SS_CAP) {
      int c[SS_K];
      val v[SS_K], xv[SS_K];
#pragma unroll
      for (int k = 0; k < SS_K; ++k) {
        const int e = tid + k * SS_THREADS;
        c[k] = e < cnt ? __ldcs(a.col + p0 + e) : 0;  // column 0 for padding (n >= 1)
        v[k] = e < cnt ? __ldcs(a.val + p0 + e) : val{};
      }
#pragma unroll
      for (int k = 0; k < SS_K; ++k) {
        bool out = false;  // of range: an entry's x counts, the padding's does not
        xv[k] = ss_x<AR>(__ldg(a.x + c[k]), out);
        bad |= out && tid + k * SS_THREADS < cnt;
      }
#pragma unroll
      for (int k = 0; k < SS_K; ++k) {
        const int e = tid + k * SS_THREADS;
        if (e < cnt) {
          if constexpr (AR == SS_PAIR) ents[e] = acc_prod(v[k].x, v[k].y, xv[k].x, xv[k].y);
          else ents[e] = ent{v[k], xv[k]};
        }
      }
      __syncthreads();
      sum s{};
      for (int e = q0 + tl; e < q1; e += TW) {
        if constexpr (AR == SS_PAIR) s = acc_add(s, ents[e]);
        else s = fma(ents[e].x, ents[e].y, s);
        if constexpr (MODE != SS_EVAL) rid[e] = (uint8_t)trow;
      }
      s = ss_team_sum<AR>(s, TW);
      if (act && tl == 0) {
        const yv yb = finish_row(row0 + trow, s);
        if constexpr (MODE != SS_EVAL) ybs[trow] = yb;
      }
      __syncthreads();
      if constexpr (MODE != SS_EVAL) {
        if (MODE == SS_ATOMIC || a.gval) {
#pragma unroll
          for (int k = 0; k < SS_K; ++k) {
            const int e = tid + k * SS_THREADS;
            if (e < cnt) scatter(p0 + e, c[k], v[k], xv[k], ybs[rid[e]]);
          }
        }
      }
    } else {
      for (int r = warp; r < nrow; r += SS_THREADS / 32) {
        const int e0 = __ldg(a.rowptr + row0 + r), e1 = __ldg(a.rowptr + row0 + r + 1);
        sum s{};
#pragma unroll 4
        for (int p = e0 + lane; p < e1; p += 32)
          ss_add<AR>(s, __ldg(a.val + p), ss_x<AR>(__ldg(a.x + __ldg(a.col + p)), bad));
        s = ss_team_sum<AR>(s, 32);
        yv yb{};
        if (lane == 0) yb = finish_row(row0 + r, s);
        if constexpr (MODE != SS_EVAL) {
          if constexpr (AR == SS_PAIR)
            yb = make_float2(__shfl_sync(0xffffffffu, yb.x, 0), __shfl_sync(0xffffffffu, yb.y, 0));
          else
            yb = __shfl_sync(0xffffffffu, yb, 0);
          if (MODE == SS_ATOMIC || a.gval) {
#pragma unroll 4
            for (int p = e0 + lane; p < e1; p += 32) {
              const int cp = __ldg(a.col + p);
              const val x = a.gval ? ss_x<AR>(__ldg(a.x + cp), bad) : val{};
              scatter(p, cp, __ldg(a.val + p), x, yb);
            }
          }
        }
      }
    }
  }
  if (bad) set_error(a.err, ERRBIT_RANGE);
  double fs;
  if constexpr (AR == SS_PAIR) fs = acc_to_double(fa);
  else fs = fa.get();
  finish_sum<T>(block_sum(fs, red), a.fpart, a.counter, a.f, 0, red);
}

// ---------------------------------------------------------------- host ----
// Lanes per row for `avg` stored entries a row: 256 / TW rows have at most 1229 entries on
// average, a fifth below the block's capacity; 0 when 8 rows do not fit.
int spq_stream_team(double avg) {
  int tw = 1;
  while (tw <= 32 && avg > 4.8 * tw) tw *= 2;
  return tw <= 32 ? tw : 0;
}

// Whether a call's row pass runs here (measured against the row teams).  FP32 gathers are
// cheap enough for narrow teams to keep as many in flight: the forward and the row pass stay
// with them (2^20 rows, 8..24 entries: 80 us there, 103 here; 300001, 1..60: 46, 59), the
// atomic gradient of rows of up to 38 entries runs here (170 -> 158 us, 104 -> 90; 40..60
// entries on 5000 columns 193 -> 209), and so does every gradient w.r.t. the values, whose
// long rows a team walks entry by entry.  FP64 rows of up to 76 entries run here (gradients
// 185 -> 175 us, 113 -> 101, 143 -> 134, forwards 122 -> 119, 79 -> 65; 100..200 entries
// 37.0 -> 39.1, CSC).  Of more than 20 blocks an SM the row teams keep
//   - thin blocks, of fewer than 700 entries because TW has just doubled (100000 rows; 350000
//     rows): the forward in pairs (39 entries a row 27.6 us there, 37.1 here; 21 a row 64 and
//     90), its row pass from TW = 8 (39 a row 51.7 and 57.3), the native atomic gradient from
//     TW = 8 (42 a row 54 and 59, 21 a row 107 and 124);
//   - the forward in pairs of TW = 16, which has no reverse to keep the entries for (60 entries
//     a row 40.4 and 45.0);
//   - the native atomic gradient with values of TW = 32 (120 a row 138 and 182).
// Fewer blocks hide less latency there (20000 rows of 39 15.0 us and 12.9, the forward).
bool spq_stream_takes(const kg_problem* p, int mode, bool gval) {
  const int tw = p->sq_stream;
  if (!tw) return false;
  if (p->dtype == KG_F32) return gval || (mode == SS_ATOMIC && tw <= 8);
  const int rb = SS_THREADS / tw;
  const bool many = (p->m + rb - 1) / rb > 20 * (int64_t)num_sms();
  const bool thin = many && tw > 1 && (double)p->nnz / (double)p->m * rb < 700.0;
  if (p->arith == KG_ARITH_PAIR) {
    if (gval) return true;
    if (mode == SS_EVAL) return tw <= (many ? 8 : 16) && !thin;
    return tw <= 16 && !(mode == SS_ROWPASS && tw >= 8 && thin);
  }
  if (mode == SS_ATOMIC) return tw <= (gval && !many ? 32 : 16) && !(tw >= 8 && thin);
  return gval || tw <= 16;
}

template <int AR, int MODE, typename Go>
static void ss_with_kernel(int tw, const Go& go) {
  switch (tw) {
    case 1: go(spq_stream_kernel<AR, MODE, 1>); break;
    case 2: go(spq_stream_kernel<AR, MODE, 2>); break;
    case 4: go(spq_stream_kernel<AR, MODE, 4>); break;
    case 8: go(spq_stream_kernel<AR, MODE, 8>); break;
    case 16: go(spq_stream_kernel<AR, MODE, 16>); break;
    case 32: go(spq_stream_kernel<AR, MODE, 32>); break;
  }
}

// One wave of at most `ctas` CTAs an SM (the kernels' launch bound).
static int ss_grid(int64_t m, int tw, int ctas) {
  const int rb = SS_THREADS / tw;
  return (int)std::max<int64_t>(1, std::min<int64_t>((m + rb - 1) / rb, ctas * (int64_t)num_sms()));
}
int spq_stream_grid(int64_t m, int tw) { return ss_grid(m, tw, 4); }  // the largest of them

template <int AR>
static cudaError_t ss_launch(const kg_problem* p, int mode, const SpqStreamCall& c, cudaStream_t s) {
  using T = typename SsTypes<AR>::T;
  SsArgs<AR> a{};
  a.rowptr = static_cast<const int*>(p->data0);
  a.col = static_cast<const int*>(p->data1);
  a.val = static_cast<const typename SsTypes<AR>::val*>(AR == SS_PAIR ? p->aprep : p->data2);
  a.x = static_cast<const T*>(c.x);
  a.m = p->m;
  a.seed = static_cast<const T*>(c.seed);
  a.gx = static_cast<T*>(c.gx);
  a.gval = static_cast<T*>(c.gval);
  a.y = p->y;
  a.accumulate = c.accumulate;
  a.fpart = p->fpart;
  a.counter = p->counter;
  a.f = static_cast<T*>(c.f);
  a.err = p->err;
  const int grid = ss_grid(p->m, p->sq_stream, ss_ctas(mode));
  auto go = [&](auto k) { k<<<grid, SS_THREADS, 0, s>>>(a); };
  if (mode == SS_EVAL) ss_with_kernel<AR, SS_EVAL>(p->sq_stream, go);
  else if (mode == SS_ATOMIC) ss_with_kernel<AR, SS_ATOMIC>(p->sq_stream, go);
  else ss_with_kernel<AR, SS_ROWPASS>(p->sq_stream, go);
  return cudaGetLastError();
}

// mode: 0 forward, 1 fused atomic gradient, 2 row pass of the CSC strategy.
cudaError_t spq_stream(const kg_problem* p, int mode, const SpqStreamCall& c, cudaStream_t s) {
  if (p->arith == KG_ARITH_PAIR) return ss_launch<SS_PAIR>(p, mode, c, s);
  return p->dtype == KG_F64 ? ss_launch<SS_F64>(p, mode, c, s) : ss_launch<SS_F32>(p, mode, c, s);
}

}  // namespace kg
