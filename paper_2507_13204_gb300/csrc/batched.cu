// Batched value-and-gradient of many independent problems in ONE persistent
// kernel launch, replayed from a CUDA graph (the paper's Sec. 5 second
// restriction: the generated gradient doubles the kernel launches and host
// synchronisation points; here a whole batch of gradients is one launch).
//
// Work: every instance is cut into tiles -- row tiles for the dense quadratic
// form, element tiles for the tet energy -- and the (instance, tile) items are
// sorted longest-first into a device work table.  Each CTA of the persistent
// grid claims items from a device queue head (one atomicAdd per item) until
// the table is exhausted.
//   dense tile:  rows [r0, r0 + R): y_i by a row team (4 .. 256 threads,
//                about 8 columns a thread), four rows a step, ybar_i = 2 y_i,
//                private xbar partial of the tile written to the instance's
//                partial buffer; the next step's rows are prefetched into L2;
//                pair arithmetic runs on packed column pairs (kg_pair2.cuh);
//   tet tile:    elements [e0, e0 + T): f_e and the scatter of c_e into gu (zeroed
//                by a small kernel earlier in the graph): one global reduction per
//                contribution, or warp-combined first with the WARP strategy.
// A dense instance of few tiles is summed into gx and f by the CTA that finishes
// its last tile (a per-instance arrival counter); one of more than B_SUM_TILES
// tiles by sum items of 256 columns at the end of the table, which wait for that
// counter.  The last CTA to leave resets the queue head and the counters, so the graph
// can be replayed as is: no tile is running any more then, also when a sum item's
// bounded wait gave up before its instance's last tile.
//
// Tile sizes R and T are chosen per (kind, size bucket) by an autotuner that
// times candidates on the instances of the batch at kg_batch_create and keeps
// the choices in a JSON cache keyed by GPU name, kind, dtype and bucket.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <map>
#include <mutex>
#include <new>
#include <sstream>
#include <string>
#include <type_traits>
#include <vector>

#include <sys/stat.h>

#include "kg_device.cuh"
#include "kg_internal.h"
#include "kg_pair.cuh"
#include "kg_pair2.cuh"
#include "kg_tet_elem.cuh"

namespace kg {

enum { BK_DENSE = 1, BK_TET = 2 };
constexpr int BT = 256;   // threads per CTA
constexpr int BW = BT / 32;
constexpr int B_CPT = 8;  // dense: columns per team thread (n <= 8 * team)
constexpr int B_MAXN = 2048;

struct BInst {
  int kind;
  int n;      // dense: columns; tet: vertices
  int64_t m;  // dense: rows; tet: elements
  int ntiles;
  int team;   // dense: threads of a row team
  int pitch;  // dense, pair batches: n rounded up to even: entries of a copy's or a partial's row
  int prep;   // pair batches: d0 (dense A) or d1 (tet G) is the prepared float-pair copy
  const void* d0;
  const void* d1;
  const void* x;
  void* f;
  void* gx;
  void* partials;  // dense: [ntiles][n] of T, or (pair) [ntiles][pitch] of Acc
  double* fpart;   // [ntiles]
  unsigned* done;  // tiles done
  int nsum;        // dense: items that sum the partials (0: the last tile's CTA does)
};

// Rows (dense) or elements (tet) [start, start + count) of tile `tile`; or, tile < 0, a sum
// item: columns [start, start + count) of a dense instance's gradient.
struct BItem {
  int inst, tile;
  int64_t start;
  int count;
};

struct BArgs {
  const BInst* insts;
  const BItem* items;
  int nitems, ninst;
  unsigned* head;  // [0] queue head, [1] CTAs that left, [2] sum items give up at once
  unsigned* done;  // [ninst] the instances' counters
  unsigned* err;
  const float4* logtab;
  LogConsts K;
  int warpc;  // tet tiles: warp-combined atomics (else one per contribution)
};

// ------------------------------------------------------------- device ----
// L2 prefetch of the whole 16-byte units inside [p, p + bytes) (never beyond).
__device__ __forceinline__ void prefetch_range_l2(const void* p, size_t bytes) {
  uintptr_t a = (reinterpret_cast<uintptr_t>(p) + 15) & ~uintptr_t(15);
  const uintptr_t b = (reinterpret_cast<uintptr_t>(p) + bytes) & ~uintptr_t(15);
  while (a < b) {
    const uint32_t chunk = (uint32_t)((b - a) < (uintptr_t(1) << 16) ? (b - a) : (uintptr_t(1) << 16));
    prefetch_l2_bulk(reinterpret_cast<const void*>(a), chunk);
    a += chunk;
  }
}

// The bytes of rows [r, r + rows) of a dense instance (one step's) into L2.
__device__ __forceinline__ void prefetch_rows_l2(const BInst& I, int64_t r, int64_t rows, size_t es) {
  const int64_t pitch = I.prep ? I.pitch : I.n;
  prefetch_range_l2(static_cast<const unsigned char*>(I.d0) + r * pitch * es, (size_t)(rows * pitch) * es);
}

// Barrier over the TEAM threads of one row team: the whole CTA for TEAM = BT,
// otherwise hardware barrier 1 + team (TEAM = 64 or 128).
template <int TEAM>
__device__ __forceinline__ void team_barrier(int team) {
  if constexpr (TEAM == BT) __syncthreads();
  else named_barrier(1 + team, TEAM);
}

// Rows [w.start, w.start + w.count) of a dense instance in native arithmetic, B_NR rows per
// team and step: their loads go out together and one transposed butterfly reduces them all
// (a butterfly per row is five FP64 adds a lane for eight columns' products).  Returns the
// tile's f.  CPT > 0: ceil(n / TEAM) columns a thread, no test but the last one's; 0: at run
// time (teams of 4).
constexpr int B_NR = 4;

template <typename T, int TEAM, int CPT>
__device__ double dense_tile(const BInst& I, const BItem& w, unsigned char* wsp, double* red) {
  constexpr int R = B_NR, WL = TEAM < 32 ? TEAM : 32, GL = WL / R;  // lanes of a row's total in a warp
  constexpr int NT = BT / TEAM, KM = CPT ? CPT : B_CPT, TW = TEAM > 32 ? TEAM / 32 : 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = I.n;
  const T* __restrict__ A = static_cast<const T*>(I.d0);
  const T* __restrict__ x = static_cast<const T*>(I.x);
  const int lt = tid % TEAM, team = tid / TEAM;
  auto col_in = [&](int k) { return (CPT && k < CPT - 1) || lt + k * TEAM < n; };
  T xv[KM], xbn[KM];
#pragma unroll
  for (int k = 0; k < KM; ++k) {
    xv[k] = col_in(k) ? x[lt + k * TEAM] : T(0);
    xbn[k] = T(0);
  }
  FSum<T> fn;
  const int row = (lane % WL) / GL;  // whose total this lane holds
  const int64_t r1 = w.start + w.count;
  const int steps = (w.count + R * NT - 1) / (R * NT);
  for (int c = 0; c < steps; ++c) {
    if (tid == 0 && c + 1 < steps) {
      const int64_t rn = w.start + (int64_t)(c + 1) * R * NT;
      prefetch_rows_l2(I, rn, r1 - rn < R * NT ? r1 - rn : R * NT, sizeof(T));
    }
    const int64_t r0 = w.start + ((int64_t)c * NT + team) * R;
    const int rows = r0 < r1 ? (int)(r1 - r0 < R ? r1 - r0 : R) : 0;
    const T* Ar = A + (rows > 0 ? r0 : w.start) * (int64_t)n + lt;
    T av[R][KM], d[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
      for (int k = 0; k < KM; ++k) av[r][k] = r < rows && col_in(k) ? __ldcs(Ar + k * TEAM) : T(0);
      Ar += n;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      d[r] = av[r][0] * xv[0];
#pragma unroll
      for (int k = 1; k < KM; ++k) d[r] = fma(av[r][k], xv[k], d[r]);
    }
    int o = WL / 2;
#pragma unroll
    for (int q = R / 2; q > 0; q >>= 1, o >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < q; ++i)
        d[i] = (up ? d[i + q] : d[i]) + __shfl_xor_sync(0xffffffffu, up ? d[i] : d[i + q], o);
    }
#pragma unroll
    for (; o > 0; o >>= 1) d[0] += __shfl_xor_sync(0xffffffffu, d[0], o);
    T tot = d[0];
    if constexpr (TEAM > 32) {
      static_assert(TW <= GL, "the butterfly over the warps stays inside a row's lanes");
      T* rt = reinterpret_cast<T*>(red) + ((c & 1) * BW + team * TW) * R;  // [TW][R]
      if (lane % GL == 0) rt[(warp % TW) * R + row] = tot;
      team_barrier<TEAM>(team);
      tot = rt[(lane % TW) * R + row];
#pragma unroll
      for (int q = TW / 2; q > 0; q >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, q);
    }
    if (row >= rows) tot = T(0);  // past the tile's end: 0 times an infinite x is no row's value
    if (TEAM <= 32 || warp % TW == 0) fn.add(tot);
    const T ybl = T(2) * tot;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const T yb = __shfl_sync(0xffffffffu, ybl, (lane & ~(WL - 1)) + r * GL);
#pragma unroll
      for (int k = 0; k < KM; ++k) xbn[k] = fma(yb, av[r][k], xbn[k]);
    }
  }
  // combine the teams' partials in team order and store the tile's partial
  __syncthreads();
  T* out = static_cast<T*>(I.partials) + (int64_t)w.tile * n;
  if constexpr (NT == 1) {
#pragma unroll
    for (int k = 0; k < KM; ++k)
      if (col_in(k)) out[lt + k * TEAM] = xbn[k];
  } else {
    T* ws = reinterpret_cast<T*>(wsp);
#pragma unroll
    for (int k = 0; k < KM; ++k) ws[team * TEAM * B_CPT + lt + k * TEAM] = xbn[k];
    __syncthreads();
    for (int j = tid; j < n; j += BT) {
      T s = ws[j];
      for (int t2 = 1; t2 < NT; ++t2) s += ws[t2 * TEAM * B_CPT + j];
      out[j] = s;
    }
  }
  // f: each row's total once, one lane of the team's first warp
  const bool counts = lane % GL == 0 && (TEAM <= 32 || warp % TW == 0);
  const double f = block_sum(counts ? fn.get() : 0.0, red);
  __syncthreads();
  return f;
}

// ---- dense tiles of pair batches: B_NR rows per team and step, columns in packed pairs ----
// Team thread lt holds the column pairs jp = lt + k TEAM, k < KM (odd n: the last
// pair's second column is a zero).

// x in float pairs for the thread's column pairs.
template <int TEAM, int KM>
__device__ __forceinline__ void pair_load_x(const BInst& I, Pair2 (&xp)[KM], Acc2 (&xb)[KM], bool& bad) {
  const double* __restrict__ x = static_cast<const double*>(I.x);
  const int lt = threadIdx.x % TEAM;
#pragma unroll
  for (int k = 0; k < KM; ++k) {
    const int j = 2 * (lt + k * TEAM);
    const double x0 = j < I.n ? x[j] : 0.0, x1 = j + 1 < I.n ? x[j + 1] : 0.0;
    bad |= !pair_in_range(x0) || !pair_in_range(x1);
    xp[k] = pair2_of(split_f64(x0), split_f64(x1));
    xb[k] = acc2_zero();
  }
}

// The end of a pair tile: the teams' partials combined in team order, two column
// pairs of every thread at a time through B_WS entries, and the tile's f (fp: the
// thread's sum, zero where it counts no row).
constexpr int B_WS = 1024;  // Acc entries of the combine buffer (8 KB)

template <int TEAM, int KM>
__device__ double pair_tile_end(const BInst& I, const BItem& w, const Acc2 (&xb)[KM], Acc fp,
                                unsigned char* wsp, double* red) {
  constexpr int NT = BT / TEAM, H = 2;
  static_assert(2 * BT * H <= B_WS, "the combine buffer holds two column pairs of all threads");
  const int tid = threadIdx.x, lt = tid % TEAM, team = tid / TEAM;
  const int np2 = I.pitch / 2;
  auto entry = [](Acc2 c) {
    const Acc a = acc2_x(c), b = acc2_y(c);
    return make_float4(a.s, a.l, b.s, b.l);
  };
  float4* out = reinterpret_cast<float4*>(I.partials) + (int64_t)w.tile * np2;
  if constexpr (NT == 1) {
#pragma unroll
    for (int k = 0; k < KM; ++k)
      if (lt + k * TEAM < np2) out[lt + k * TEAM] = entry(xb[k]);
  } else {
    float4* ws = reinterpret_cast<float4*>(wsp);  // [NT][TEAM * H]
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      if (half * H * TEAM >= np2) break;
#pragma unroll
      for (int kk = 0; kk < H; ++kk)  // column pairs k >= KM are past the row's end: not read
        if (half * H + kk < KM) ws[team * TEAM * H + lt + kk * TEAM] = entry(xb[half * H + kk < KM ? half * H + kk : 0]);
      __syncthreads();
      for (int jj = tid; jj < TEAM * H; jj += BT) {
        const int jp = jj + half * H * TEAM;
        if (jp < np2) {
          float4 e = ws[jj];
          Acc a{e.x, e.y}, b{e.z, e.w};
          for (int t2 = 1; t2 < NT; ++t2) {
            e = ws[t2 * TEAM * H + jj];
            a = acc_add(a, Acc{e.x, e.y});
            b = acc_add(b, Acc{e.z, e.w});
          }
          out[jp] = make_float4(a.s, a.l, b.s, b.l);
        }
      }
      __syncthreads();
    }
  }
  Acc* ra = reinterpret_cast<Acc*>(red);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) fp = acc_add(fp, shfl_xor_acc2(fp, o));
  __syncthreads();
  if ((tid & 31) == 0) ra[tid >> 5] = fp;
  __syncthreads();
  Acc tot = ra[0];
  for (int q = 1; q < BW; ++q) tot = acc_add(tot, ra[q]);
  __syncthreads();
  return acc_to_double(tot);
}

// Rows [w.start, w.start + w.count) of an instance of a pair batch, as the native tiles:
// B_NR rows per team and step, their loads together (up to 64 KB a CTA in flight), one
// transposed butterfly and, for teams wider than a warp, one barrier for all of them; the
// next step's rows are prefetched into L2.  PREP: from the float-pair copy, 16 bytes a column
// pair; otherwise FP64 data, split on every load, in the same order (the same bits).
// KP > 0: ceil(pitch / 2 / TEAM) column pairs a thread, no test but the last one's; 0: at run
// time.  Returns the tile's f.
// Bound by instruction issue and the loads' latency, 2 CTAs an SM.  Against two rows a step
// through a shared-memory ring of bulk copies (a CTA barrier a step, a shared-memory pass):
// 128 dense (n to 2048) + 16 tet instances 178 -> 156 us, 32 + 4 49.7 -> 43.0, 16 + 2
// 45.3 -> 33.0; 4096 + 512 4.13 -> 3.51 ms (17.87 GB, 0.75 of the copy peak).
template <int TEAM, int KP, bool PREP>
__device__ double dense_tile_pair(const BInst& I, const BItem& w, unsigned char* wsp, double* red, bool& bad) {
  constexpr int R = B_NR, WL = TEAM < 32 ? TEAM : 32, GL = WL / R;  // lanes of a row's total in a warp
  constexpr int NT = BT / TEAM, KM = KP ? KP : B_CPT / 2, TW = TEAM > 32 ? TEAM / 32 : 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lt = tid % TEAM, team = tid / TEAM;
  const int n = I.n, np2 = I.pitch / 2;
  auto in_row = [&](int k) { return (KP && k < KP - 1) || lt + k * TEAM < np2; };
  Pair2 xp[KM];
  Acc2 xb[KM];
  pair_load_x<TEAM>(I, xp, xb, bad);
  Acc fp = acc_zero();
  const int row = (lane % WL) / GL;  // whose total this lane holds
  const bool counts = lane % GL == 0 && (TEAM <= 32 || warp % TW == 0);
  const int64_t r1 = w.start + w.count;
  const int steps = (w.count + R * NT - 1) / (R * NT);
  for (int c = 0; c < steps; ++c) {
    if (tid == 0 && c + 1 < steps) {
      const int64_t rn = w.start + (int64_t)(c + 1) * R * NT;
      prefetch_rows_l2(I, rn, r1 - rn < R * NT ? r1 - rn : R * NT, 8);
    }
    const int64_t r0 = w.start + ((int64_t)c * NT + team) * R;
    const int rows = r0 < r1 ? (int)(r1 - r0 < R ? r1 - r0 : R) : 0;
    const int64_t first = rows > 0 ? r0 : w.start;
    Pair2 av[R][KM];
    if constexpr (PREP) {
      const ulonglong2* Ar = static_cast<const ulonglong2*>(I.d0) + first * np2 + lt;
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int k = 0; k < KM; ++k) {
          const ulonglong2 q = r < rows && in_row(k) ? __ldcs(Ar + k * TEAM) : make_ulonglong2(0ull, 0ull);
          av[r][k] = Pair2{F2{q.x}, F2{q.y}};
        }
        Ar += np2;
      }
    } else {
      const double* Ar = static_cast<const double*>(I.d0) + first * n;
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int k = 0; k < KM; ++k) {
          const int j = 2 * (lt + k * TEAM);
          const double v0 = r < rows && j < n ? __ldcs(Ar + j) : 0.0;
          const double v1 = r < rows && j + 1 < n ? __ldcs(Ar + j + 1) : 0.0;
          av[r][k] = pair2_of(split_f64(v0), split_f64(v1));
        }
        Ar += n;
      }
    }
    Acc d[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      Acc2 y = acc2_prod(av[r][0], xp[0]);
#pragma unroll
      for (int k = 1; k < KM; ++k) acc2_fma(y, av[r][k], xp[k]);
      d[r] = acc2_sum(y);
    }
    int o = WL / 2;
#pragma unroll
    for (int q = R / 2; q > 0; q >>= 1, o >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < q; ++i)
        d[i] = acc_add(up ? d[i + q] : d[i], shfl_xor_acc2(up ? d[i] : d[i + q], o));
    }
#pragma unroll
    for (; o > 0; o >>= 1) d[0] = acc_add(d[0], shfl_xor_acc2(d[0], o));
    Acc tot = d[0];
    if constexpr (TEAM > 32) {
      static_assert(TW <= GL, "the butterfly over the warps stays inside a row's lanes");
      Acc* rt = reinterpret_cast<Acc*>(red) + ((c & 1) * BW + team * TW) * R;  // [TW][R]
      if (lane % GL == 0) rt[(warp % TW) * R + row] = tot;
      team_barrier<TEAM>(team);
      tot = rt[(lane % TW) * R + row];
#pragma unroll
      for (int q = TW / 2; q > 0; q >>= 1) tot = acc_add(tot, shfl_xor_acc2(tot, q));
    }
    const Pair y = acc_pair(tot);  // rows past the tile's end: zero
    if (TEAM <= 32 || warp % TW == 0) {
      const Pair y2 = pair_mul(y, y);
      fp = acc_add(fp, Acc{y2.h, y2.l});
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int src = (lane & ~(WL - 1)) + r * GL;
      const Pair2 yb = pair2_dup(Pair{2.0f * __shfl_sync(0xffffffffu, y.h, src),
                                      2.0f * __shfl_sync(0xffffffffu, y.l, src)});  // exact
#pragma unroll
      for (int k = 0; k < KM; ++k) acc2_fma(xb[k], av[r][k], yb);
    }
    if ((c & 3) == 3) {
      acc_renorm(fp);
#pragma unroll
      for (int k = 0; k < KM; ++k) acc2_renorm(xb[k]);
    }
  }
  __syncthreads();
  return pair_tile_end<TEAM>(I, w, xb, counts ? fp : acc_zero(), wsp, red);
}

// Elements [w.start, w.start + w.count) of a tet instance; returns the tile's f.
template <typename T, bool PAIR, bool WARPC, bool PREP>
__device__ double tet_tile(const BInst& I, const BItem& w, const float4* tab, const LogConsts& K,
                           double* red, bool& bad) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int4* conn = static_cast<const int4*>(I.d0);
  const T* G = static_cast<const T*>(I.d1);
  const T* u = static_cast<const T*>(I.x);
  T* gu = static_cast<T*>(I.gx);
  LogSum lsum = log_sum_zero();
  T fn = T(0);
  const int64_t e1 = w.start + w.count;
  if constexpr (!WARPC) {  // one atomic per contribution
    for (int64_t e = w.start + tid; e < e1; e += BT) {
      const int4 c = __ldcs(conn + e);
      if constexpr (PAIR) {
        elem_pair<TS_GRAD, AtomicSink<double>, PREP>(
            c, reinterpret_cast<const double*>(G) + e * 12, reinterpret_cast<const double*>(u),
            Pair{2.0f, 0.0f}, tab, K, lsum, AtomicSink<double>{reinterpret_cast<double*>(gu)}, nullptr,
            bad);
      } else {
        elem_native<T, TS_GRAD>(c, G + e * 12, u, T(1), fn, AtomicSink<T>{gu}, nullptr);
      }
    }
  }
  // WARPC: block-uniform loop, so that every lane reaches the warp-level combine
  for (int64_t e0 = w.start; WARPC && e0 < e1; e0 += BT) {
    const int64_t e = e0 + tid;
    const bool act = e < e1;
    T cv[4];
    Pair cpr[4];
    int4 c = make_int4(-1, -1, -1, -1);
    if (act) {
      c = __ldcs(conn + e);
      if constexpr (PAIR) {
        elem_pair<TS_GRAD, CollectSink<T>, PREP>(
            c, reinterpret_cast<const double*>(G) + e * 12, reinterpret_cast<const double*>(u),
            Pair{2.0f, 0.0f}, tab, K, lsum, CollectSink<T>{cv, cpr}, nullptr, bad);
      } else {
        elem_native<T, TS_GRAD>(c, G + e * 12, u, T(1), fn, CollectSink<T>{cv, cpr}, nullptr);
      }
    }
    const int key[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if constexpr (PAIR) {
        warp_combine(act, key[k], Acc{cpr[k].h, cpr[k].l},
                     [](Acc x, Acc y) { return acc_add(x, y); },
                     [&](int v, Acc tot) {
                       red_add(reinterpret_cast<double*>(gu) + v, pair_to_double_fast(acc_pair(tot)));
                     });
      } else {
        warp_combine(act, key[k], cv[k], [](T x, T y) { return x + y; },
                     [&](int v, T tot) { red_add(gu + v, tot); });
      }
    }
  }
  __syncthreads();
  if constexpr (PAIR) {
    Acc fp = log_sum_get(lsum, tab, K);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fp = acc_add(fp, shfl_xor_acc2(fp, o));
    Acc* ra = reinterpret_cast<Acc*>(red);
    if (lane == 0) ra[warp] = fp;
    __syncthreads();
    Acc tot = ra[0];
    for (int q = 1; q < BW; ++q) tot = acc_add(tot, ra[q]);
    __syncthreads();
    return acc_to_double(tot);
  } else {
    const double t = block_sum((double)fn, red);
    __syncthreads();
    return t;
  }
}

// Calls go.template run<TEAM>() with the instance's team width.
template <typename Go>
__device__ __forceinline__ double with_team(int team, const Go& go) {
  switch (team) {
    case 4: return go.template run<4>();
    case 8: return go.template run<8>();
    case 16: return go.template run<16>();
    case 32: return go.template run<32>();
    case 64: return go.template run<64>();
    case 128: return go.template run<128>();
    default: return go.template run<BT>();
  }
}

template <typename T>
struct NativeTile {
  const BInst& I;
  const BItem& w;
  unsigned char* wsp;
  double* red;
  // the team is the smallest power of two (>= 4) with 8 columns a thread, so above 4
  // threads a team thread has 5 to 8
  template <int TEAM>
  __device__ __forceinline__ double run() const {
    if constexpr (TEAM > 4) {
      switch ((I.n + TEAM - 1) / TEAM) {
        case 5: return dense_tile<T, TEAM, 5>(I, w, wsp, red);
        case 6: return dense_tile<T, TEAM, 6>(I, w, wsp, red);
        case 7: return dense_tile<T, TEAM, 7>(I, w, wsp, red);
        default: return dense_tile<T, TEAM, 8>(I, w, wsp, red);
      }
    } else {
      return dense_tile<T, TEAM, 0>(I, w, wsp, red);
    }
  }
};

template <bool PREP>
struct PairTile {
  const BInst& I;
  const BItem& w;
  unsigned char* wsp;
  double* red;
  bool& bad;
  // the team is the smallest power of two (>= 4) with 4 column pairs a thread, so
  // above 4 threads a team thread has 3 or 4
  template <int TEAM>
  __device__ __forceinline__ double run() const {
    if constexpr (TEAM > 4 && PREP) {
      const int kp = (I.pitch / 2 + TEAM - 1) / TEAM;
      if (kp == 4) return dense_tile_pair<TEAM, 4, PREP>(I, w, wsp, red, bad);
      if (kp == 3) return dense_tile_pair<TEAM, 3, PREP>(I, w, wsp, red, bad);
    }
    return dense_tile_pair<TEAM, 0, PREP>(I, w, wsp, red, bad);
  }
};

// The instance's f from its tile partials: lane l of warp 0 adds tiles l, l + 32, ..., then
// a butterfly (call with warp 0 only).
template <typename T>
__device__ __forceinline__ void sum_f(const BInst& I) {
  double fs = 0.0;
#pragma unroll 4
  for (int t = threadIdx.x; t < I.ntiles; t += 32) fs += __ldcg(I.fpart + t);
  fs = warp_sum(fs);
  if (threadIdx.x == 0 && I.f) *static_cast<T*>(I.f) = (T)fs;
}

// Columns [j0, j0 + cols) of a dense instance's gradient: a thread per column adds the
// tile partials in tile order, eight loads in flight.
template <typename T, bool PAIR>
__device__ void sum_columns(const BInst& I, int j0, int cols) {
  using P = std::conditional_t<PAIR, float2, T>;
  using S = std::conditional_t<PAIR, Acc, T>;
  const P* parts = static_cast<const P*>(I.partials);
  const int64_t pitch = PAIR ? I.pitch : I.n;
  for (int j = j0 + threadIdx.x; j < j0 + cols; j += BT) {
    S s{};
    for (int t = 0; t < I.ntiles; t += 8) {
      P v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = t + u < I.ntiles ? __ldcg(parts + (t + u) * pitch + j) : P{};
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if constexpr (PAIR) s = acc_add(s, Acc{v[u].x, v[u].y});
        else s += v[u];
      }
      if constexpr (PAIR)
        if ((t & 24) == 24) acc_renorm(s);
    }
    if constexpr (PAIR) static_cast<double*>(I.gx)[j] = pair_to_double_fast(acc_pair(s));
    else static_cast<T*>(I.gx)[j] = s;
  }
}

template <typename T, bool PAIR>
__global__ void __launch_bounds__(BT, 2) batched_kernel(BArgs a) {
  // [PAIR: log table][combine buffer][red]
  extern __shared__ __align__(16) unsigned char smem[];
  float4* tab = reinterpret_cast<float4*>(smem);
  unsigned char* wsp = smem + (PAIR ? kLogTableSize * sizeof(float4) : 0);
  double* red = reinterpret_cast<double*>(wsp + (PAIR ? B_WS * sizeof(Acc) : (size_t)BT * B_CPT * 8));
  __shared__ int s_item, s_last;
  // PAIR: the item and its instance, registers being short in the tiles.  The native kernels
  // hold them in registers (32 dense + 4 tet FP32 instances: 29.0 us, 33.3 in shared memory)
  __shared__ BItem s_w;
  __shared__ BInst s_I;
  const int tid = threadIdx.x;
  if constexpr (PAIR) {
    for (int i = tid; i < kLogTableSize; i += BT) tab[i] = a.logtab[i];
  }
  bool bad = false;
  // items are claimed one ahead: the next one's first rows go into L2 during this one
  if (tid == 0) s_item = (int)atomicAdd(&a.head[0], 1u);
  __syncthreads();
  int it = s_item;
  for (;;) {
    __syncthreads();  // every thread has read s_item
    if (it >= a.nitems) break;
    if (tid == 0) {
      const int nit = (int)atomicAdd(&a.head[0], 1u);
      s_item = nit;
      if (nit < a.nitems) {
        const BItem wn = a.items[nit];
        const BInst& In = a.insts[wn.inst];
        if (In.kind == BK_DENSE && wn.tile >= 0) {
          const int64_t rows = B_NR * (BT / In.team);
          prefetch_rows_l2(In, wn.start, rows < wn.count ? rows : wn.count, sizeof(T));
        }
      }
    }
    BItem wr;
    BInst Ir;
    if constexpr (PAIR) {
      if (tid == 32) {
        s_w = a.items[it];
        s_I = a.insts[s_w.inst];
      }
      __syncthreads();
    } else {
      wr = a.items[it];
      Ir = a.insts[wr.inst];
    }
    const BItem& w = PAIR ? s_w : wr;
    const BInst& I = PAIR ? s_I : Ir;
    if (w.tile < 0) {
      // every tile item comes before the sum items and is held by a running CTA (this
      // one has none left), so the wait ends
      if (tid == 0) {
        const bool give_up = a.head[2] != 0u;
        const uint64_t t0 = global_ns();
        unsigned arrived = ld_acquire_u32(I.done);
        s_last = 1;
        while (give_up || arrived < (unsigned)I.ntiles) {
          if (give_up || global_ns() - t0 > kWaitLimitNs) {
            set_error(a.err, ERRBIT_TIMEOUT);
            s_last = 0;
            break;
          }
          arrived = ld_acquire_u32(I.done);
        }
        __threadfence();
      }
      __syncthreads();
      if (s_last) {
        if (w.start == 0 && tid < 32) sum_f<T>(I);
        sum_columns<T, PAIR>(I, (int)w.start, w.count);
      }
      it = s_item;
      continue;
    }
    // a tet tile's contiguous data into L2 while the first loads are in flight (dense tiles
    // prefetch a step ahead: whole tiles of every CTA exceed L2 and are evicted before use)
    if (tid == 0 && I.kind == BK_TET) {
      prefetch_range_l2(static_cast<const int4*>(I.d0) + w.start, (size_t)w.count * 16);
      prefetch_range_l2(static_cast<const T*>(I.d1) + w.start * 12, (size_t)w.count * 12 * sizeof(T));
    }
    double ft;
    const bool prep = PAIR && I.prep;
    if (I.kind == BK_DENSE) {
      if constexpr (PAIR)
        ft = prep ? with_team(I.team, PairTile<true>{I, w, wsp, red, bad})
                  : with_team(I.team, PairTile<false>{I, w, wsp, red, bad});
      else
        ft = with_team(I.team, NativeTile<T>{I, w, wsp, red});
    } else {
      if (a.warpc)
        ft = prep ? tet_tile<T, PAIR, true, true>(I, w, tab, a.K, red, bad)
                  : tet_tile<T, PAIR, true, false>(I, w, tab, a.K, red, bad);
      else
        ft = prep ? tet_tile<T, PAIR, false, true>(I, w, tab, a.K, red, bad)
                  : tet_tile<T, PAIR, false, false>(I, w, tab, a.K, red, bad);
    }
    if (tid == 0) I.fpart[w.tile] = ft;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(I.done, 1u) == (unsigned)I.ntiles - 1u;
    __syncthreads();
    if (s_last && I.nsum == 0) {
      __threadfence();
      if (tid < 32) sum_f<T>(I);
      if (I.kind == BK_DENSE) sum_columns<T, PAIR>(I, 0, I.n);
    }
    it = s_item;  // written by thread 0 before the barriers above
  }
  if (bad) set_error(a.err, ERRBIT_RANGE);
  // the last CTA to leave resets the queue and the counters for the next replay
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(&a.head[1], 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) {
    for (int i = tid; i < a.ninst; i += BT) a.done[i] = 0u;
    if (tid < 3) a.head[tid] = 0u;
  }
}

// The float pairs of m rows of n (odd) doubles, n + 1 entries a row, the last a zero.
__global__ void pair_rows_kernel(const double* __restrict__ A, float4* __restrict__ out, int64_t m, int n) {
  const int np2 = (n + 1) / 2;
  const int64_t count = m * np2, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
    const int64_t r = i / np2;
    const int j = 2 * (int)(i - r * np2);
    const double* a = A + r * n + j;
    out[i] = pair2_entry(split_f64(a[0]), split_f64(j + 1 < n ? a[1] : 0.0));
  }
}

template <typename T>
__global__ void batched_zero_kernel(const BInst* __restrict__ insts, const int* __restrict__ ids,
                                    int count) {
  for (int k = blockIdx.x; k < count; k += gridDim.x) {
    const BInst I = insts[ids[k]];
    T* g = static_cast<T*>(I.gx);
    for (int j = threadIdx.x; j < I.n; j += blockDim.x) g[j] = T(0);
  }
}

}  // namespace kg

// ------------------------------------------------------------------ host --
using namespace kg;

namespace {

size_t batched_smem(bool pair) {
  if (pair) return kLogTableSize * sizeof(float4) + B_WS * sizeof(Acc) + 64 * sizeof(double);
  return (size_t)BT * B_CPT * 8 + 64 * sizeof(double);
}

int bucket_of(int64_t v) {
  int b = 0;
  while ((int64_t(1) << (b + 1)) <= v) ++b;
  return b;
}

// ---- tuning cache: one JSON object of "key": value lines ----
std::mutex g_tune_mu;

std::string cache_path() {
  if (const char* p = std::getenv("KG_TUNE_CACHE")) return p;
  const char* home = std::getenv("HOME");
  return std::string(home ? home : ".") + "/.cache/kg_tune.json";
}

std::map<std::string, int> cache_read() {
  std::map<std::string, int> m;
  std::ifstream in(cache_path());
  std::string line;
  while (std::getline(in, line)) {
    const size_t q1 = line.find('"'), q2 = line.find('"', q1 + 1), c = line.find(':', q2 + 1);
    if (q1 == std::string::npos || q2 == std::string::npos || c == std::string::npos) continue;
    m[line.substr(q1 + 1, q2 - q1 - 1)] = std::atoi(line.c_str() + c + 1);
  }
  return m;
}

void cache_write(const std::map<std::string, int>& m) {
  const std::string path = cache_path();
  const size_t slash = path.rfind('/');
  if (slash != std::string::npos) {  // create the parent directories
    const std::string dir = path.substr(0, slash);
    for (size_t i = 1; i <= dir.size(); ++i)
      if (i == dir.size() || dir[i] == '/') mkdir(dir.substr(0, i).c_str(), 0755);
  }
  const std::string tmp = path + ".tmp";
  std::ofstream out(tmp);
  if (!out) return;
  out << "{\n";
  size_t i = 0;
  for (const auto& kv : m) out << "  \"" << kv.first << "\": " << kv.second << (++i < m.size() ? ",\n" : "\n");
  out << "}\n";
  out.close();
  std::rename(tmp.c_str(), path.c_str());
}

}  // namespace

namespace {

// ---- plans: instances cut into tiles ----
struct Plan {
  std::vector<BInst> insts;
  std::vector<BItem> items;
  std::vector<BItem> sums;       // after all tiles, in the order of their instances' size
  std::vector<int> tet_ids;
  std::vector<size_t> part_off;  // byte offset of each dense instance's partials
  std::vector<size_t> fpart_off; // index of each instance's first f partial
  size_t part_bytes = 0, fparts = 0;
};

struct Tuning {
  std::map<int, int> dense_rows;   // bucket -> rows per item
  std::map<int, int> tet_elems;    // bucket -> elements per item
};

int default_rows(int n) { return n <= 64 ? 128 : n <= 256 ? 64 : (n <= 1024 ? 16 : 8); }
int default_elems(int64_t) { return 4096; }

// Bytes a work item streams, the tets' weighted by their lower rate.
double item_cost(const kg_problem* p, int64_t count, size_t es) {
  return p->kind == KG_QUADFORM ? (double)count * p->n * es : 1.7 * (double)count * (16.0 + 12.0 * es);
}

// Dense instances of more tiles than this are summed by items of their own, by all CTAs
// that have no tile left: the last tile's CTA alone reads 256 columns of 8 partials in
// about a microsecond, 48 partials of 2035 columns in 50, at the end of the batch.
constexpr int B_SUM_TILES = 16;
// No tile is larger than a CTA's share of the batch / B_SHARE, so that a batch of few
// large instances still fills the grid: the autotuner's tiles (up to 256 rows, right for
// batches of thousands) gave 128 dense and 16 tet instances two items a CTA.  Measured on
// that batch, 630 MB, shares of 2, 3, 4 and 6 (medians of six tunings): float pairs 160, 156,
// 159 and 164 us, FP32 79, 81, 83 and 92, native FP64 462, 419, 426 and 421; 32 + 4 instances
// 66, 68, 69 and 69, 16 + 2 do not differ (their tiles are at the 4 steps make_plan leaves).
constexpr int B_SHARE = 3;

// prep[i]: the float-pair copy of problem i's A (dense) or G (tet) that the
// batch streams, or NULL (the FP64 data, split per load).  grid > 0: tiles are
// cut so that none exceeds a CTA's share of these instances / B_SHARE.
Plan make_plan(const std::vector<kg_problem*>& probs, const std::vector<const void*>& prep,
               const std::vector<int>& ids, const Tuning& tu, bool pair, size_t es, int grid) {
  Plan P;
  double cap = 0.0;
  if (grid > 0) {
    for (int i : ids) cap += item_cost(probs[i], probs[i]->m, es);
    cap /= (double)B_SHARE * grid;
  }
  struct Cost {
    double c;
    BItem it;
  };
  std::vector<Cost> all;
  for (int idx = 0; idx < (int)ids.size(); ++idx) {
    const kg_problem* p = probs[ids[idx]];
    BInst I{};
    I.kind = p->kind == KG_QUADFORM ? BK_DENSE : BK_TET;
    I.n = (int)p->n;
    I.pitch = (int)(p->n + (p->n & 1));
    I.m = p->m;
    I.d0 = p->data0;
    I.d1 = p->data1;
    if (pair && prep[ids[idx]]) {  // stream the prepared float pairs
      I.prep = 1;
      if (p->kind == KG_QUADFORM) I.d0 = prep[ids[idx]];
      else I.d1 = prep[ids[idx]];
    }
    int64_t per;
    if (I.kind == BK_DENSE) {
      auto f = tu.dense_rows.find(bucket_of(p->n));
      per = f != tu.dense_rows.end() ? f->second : default_rows((int)p->n);
      // row team: about B_CPT columns per thread (4 .. 256 threads)
      I.team = 4;
      while (I.team < BT && (int64_t)I.team * B_CPT < p->n) I.team *= 2;
    } else {
      auto f = tu.tet_elems.find(bucket_of(p->m));
      per = f != tu.tet_elems.end() ? f->second : default_elems(p->m);
      I.team = 0;
      P.tet_ids.push_back(idx);
    }
    if (cap > 0.0) {  // whole steps of the row teams or of the CTA's threads, 4 at least
      const int64_t unit = I.kind == BK_DENSE ? B_NR * (BT / I.team) : BT;
      const int64_t most = (int64_t)(cap / item_cost(p, unit, es)) * unit;
      per = std::min(per, std::max(most, 4 * unit));
    }
    I.ntiles = (int)((I.m + per - 1) / per);
    if (I.kind == BK_DENSE && I.ntiles > B_SUM_TILES) {
      for (int j = 0; j < I.n; j += BT) {
        P.sums.push_back(BItem{idx, -1, j, std::min(BT, I.n - j)});
        ++I.nsum;
      }
    }
    P.fpart_off.push_back(P.fparts);
    P.fparts += I.ntiles;
    P.part_off.push_back(P.part_bytes);
    if (I.kind == BK_DENSE) {
      const size_t b = (size_t)I.ntiles * (pair ? I.pitch * sizeof(Acc) : I.n * es);
      P.part_bytes += (b + 255) & ~size_t(255);
    }
    for (int t = 0; t < I.ntiles; ++t) {
      BItem it{idx, t, (int64_t)t * per, (int)std::min<int64_t>(per, I.m - (int64_t)t * per)};
      all.push_back({item_cost(p, it.count, es), it});
    }
    P.insts.push_back(I);
  }
  std::stable_sort(all.begin(), all.end(), [](const Cost& a, const Cost& b) { return a.c > b.c; });
  for (const auto& c : all) P.items.push_back(c.it);
  // instances whose tiles come first are summed first
  std::stable_sort(P.sums.begin(), P.sums.end(), [&](const BItem& a, const BItem& b) {
    return P.insts[a.inst].m * P.insts[a.inst].n > P.insts[b.inst].m * P.insts[b.inst].n;
  });
  P.items.insert(P.items.end(), P.sums.begin(), P.sums.end());
  return P;
}

// Device copy of a plan with its workspaces; x/f/gx filled per call.
struct DevPlan {
  BInst* insts = nullptr;
  BItem* items = nullptr;
  int* tet_ids = nullptr;
  unsigned* head = nullptr;
  unsigned* done = nullptr;
  unsigned char* parts = nullptr;
  double* fpart = nullptr;
  int nitems = 0, ntet = 0, ninst = 0;
  std::vector<void*> allocs;
  void release() {
    for (void* p : allocs) cudaFree(p);
    allocs.clear();
  }
};

kg_status devplan_alloc(DevPlan& D, Plan& P, cudaStream_t s) {
  auto al = [&](void** ptr, size_t bytes, const char* what) -> kg_status {
    cudaError_t e = dev_alloc(ptr, bytes);
    if (e != cudaSuccess) return fail(KG_ERR_OOM, std::string("batch workspace: ") + what);
    D.allocs.push_back(*ptr);
    return KG_OK;
  };
  kg_status rc;
  D.ninst = (int)P.insts.size();
  D.nitems = (int)P.items.size();
  D.ntet = (int)P.tet_ids.size();
  if ((rc = al((void**)&D.insts, sizeof(BInst) * P.insts.size(), "descriptors")) != KG_OK) return rc;
  if ((rc = al((void**)&D.items, sizeof(BItem) * P.items.size(), "work table")) != KG_OK) return rc;
  if ((rc = al((void**)&D.tet_ids, sizeof(int) * std::max<size_t>(1, P.tet_ids.size()), "tet ids")) != KG_OK) return rc;
  if ((rc = al((void**)&D.head, 16, "queue head")) != KG_OK) return rc;
  if ((rc = al((void**)&D.done, sizeof(unsigned) * P.insts.size(), "arrival counters")) != KG_OK) return rc;
  if ((rc = al((void**)&D.parts, std::max<size_t>(256, P.part_bytes), "partials")) != KG_OK) return rc;
  if ((rc = al((void**)&D.fpart, sizeof(double) * std::max<size_t>(1, P.fparts), "f partials")) != KG_OK) return rc;
  for (int i = 0; i < D.ninst; ++i) {
    P.insts[i].partials = D.parts + P.part_off[i];
    P.insts[i].fpart = D.fpart + P.fpart_off[i];
    P.insts[i].done = D.done + i;
  }
  cudaError_t e;
  if ((e = cudaMemsetAsync(D.head, 0, 16, s)) != cudaSuccess) return cuda_fail(e, "batch set-up");
  if ((e = cudaMemsetAsync(D.done, 0, sizeof(unsigned) * P.insts.size(), s)) != cudaSuccess)
    return cuda_fail(e, "batch set-up");
  if ((e = cudaMemcpyAsync(D.items, P.items.data(), sizeof(BItem) * P.items.size(),
                           cudaMemcpyHostToDevice, s)) != cudaSuccess)
    return cuda_fail(e, "batch set-up");
  if (!P.tet_ids.empty() &&
      (e = cudaMemcpyAsync(D.tet_ids, P.tet_ids.data(), sizeof(int) * P.tet_ids.size(),
                           cudaMemcpyHostToDevice, s)) != cudaSuccess)
    return cuda_fail(e, "batch set-up");
  return KG_OK;
}

int batched_grid(bool pair) {
  int per = 0, dev = 0;
  cudaGetDevice(&dev);
  const size_t smem = batched_smem(pair);
  cudaError_t e;
  if (pair)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, batched_kernel<double, true>, BT, smem);
  else
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, batched_kernel<double, false>, BT, smem);
  if (e != cudaSuccess || per < 1) per = 2;
  return num_sms() * std::min(per, 4);
}

// The float-pair copy of m rows of n doubles, rows padded to whole column pairs.
kg_status pair_prepare_rows(const double* src, void* dst, int64_t m, int64_t n, cudaStream_t s) {
  if (n % 2 == 0) return pair_prepare(src, dst, m * n, s);
  const int64_t count = m * ((n + 1) / 2);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((count + 255) / 256, (int64_t)num_sms() * 8));
  pair_rows_kernel<<<grid, 256, 0, s>>>(src, static_cast<float4*>(dst), m, (int)n);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? KG_OK : cuda_fail(e, "prepare float pairs");
}

// Launches the zero kernel (tet gradients) and the persistent kernel on s.
static void launch_batched(int dtype, bool pair, int grid, size_t smem, cudaStream_t s, const BArgs& a) {
  if (dtype == KG_F64) {
    if (pair) batched_kernel<double, true><<<grid, BT, smem, s>>>(a);
    else batched_kernel<double, false><<<grid, BT, smem, s>>>(a);
  } else {
    batched_kernel<float, false><<<grid, BT, smem, s>>>(a);
  }
}

kg_status launch_plan(const DevPlan& D, int dtype, bool pair, bool warp, unsigned* err,
                      cudaStream_t s, int grid) {
  cudaError_t e = cudaSuccess;
  if (D.ntet > 0) {
    const int zg = std::min(D.ntet, num_sms() * 4);
    if (dtype == KG_F64) batched_zero_kernel<double><<<zg, 256, 0, s>>>(D.insts, D.tet_ids, D.ntet);
    else batched_zero_kernel<float><<<zg, 256, 0, s>>>(D.insts, D.tet_ids, D.ntet);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "batched zero kernel");
  }
  BArgs a{};
  a.insts = D.insts;
  a.items = D.items;
  a.nitems = D.nitems;
  a.ninst = D.ninst;
  a.head = D.head;
  a.done = D.done;
  a.err = err;
  a.K = log_consts();
  if (pair) {
    kg_status rc = logtab_for_device(&a.logtab);
    if (rc != KG_OK) return rc;
  }
  a.warpc = warp ? 1 : 0;
  launch_batched(dtype, pair, grid, batched_smem(pair), s, a);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "batched kernel");
  return KG_OK;
}

}  // namespace

struct kg_batch {
  std::vector<kg_problem*> probs;
  std::vector<const void*> prep;  // per problem: the float-pair copy streamed, or NULL
  std::vector<void*> own_preps;   // the copies the batch made itself
  int dtype = KG_F64;
  bool pair = false;
  bool warp = false;  // tet scatter: warp-combined atomics (false: one atomic per contribution)
  size_t es = 8;
  Plan plan;
  DevPlan dev;
  unsigned* err = nullptr;
  int grid = 0;
  Tuning tune;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  std::vector<const void*> last_x, last_f, last_gx;
  bool ptrs_valid = false;
  cudaStream_t last_stream = nullptr;
  std::string gpu;
};

namespace {

std::string gpu_name() {
  int dev = 0;
  cudaDeviceProp pr{};
  if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&pr, dev) != cudaSuccess)
    return "unknown";
  std::string s = pr.name;
  for (char& c : s)
    if (c == '"' || c == '|') c = '_';
  return s;
}

// Times the persistent kernel on the instances `ids` with tuning `tu`.
kg_status time_plan(kg_batch* b, const std::vector<int>& ids, const Tuning& tu, cudaStream_t s,
                    void* xbuf, void* gbuf, float* ms) {
  Plan P = make_plan(b->probs, b->prep, ids, tu, b->pair, b->es, b->grid);
  DevPlan D;
  kg_status rc = devplan_alloc(D, P, s);
  if (rc == KG_OK) {
    size_t off = 0;
    for (auto& I : P.insts) {
      I.x = static_cast<unsigned char*>(xbuf) + off;
      I.gx = static_cast<unsigned char*>(gbuf) + off;
      I.f = nullptr;
      off += ((size_t)I.n * b->es + 255) & ~size_t(255);
    }
    cudaError_t e = cudaMemcpyAsync(D.insts, P.insts.data(), sizeof(BInst) * P.insts.size(),
                                    cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) rc = cuda_fail(e, "autotune");
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (rc == KG_OK && (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess))
      rc = fail(KG_ERR_CUDA, "autotune events");
    float best = 1e30f;
    for (int r = 0; rc == KG_OK && r < 4; ++r) {
      cudaEventRecord(e0, s);
      rc = launch_plan(D, b->dtype, b->pair, b->warp, b->err, s, b->grid);
      cudaEventRecord(e1, s);
      if (rc == KG_OK && (e = cudaEventSynchronize(e1)) != cudaSuccess) rc = cuda_fail(e, "autotune");
      float t = 0.f;
      if (rc == KG_OK && r > 0 && cudaEventElapsedTime(&t, e0, e1) == cudaSuccess) best = std::min(best, t);
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    *ms = best;
  }
  cudaStreamSynchronize(s);
  D.release();
  return rc;
}

// Chooses rows (dense) / elements (tet) per item for every size bucket of the
// batch: each candidate runs on a sample of the bucket's instances large
// enough that the largest candidate still gives four items per CTA of the
// persistent grid (or on all of them); the largest tile within 3% of the
// fastest wins.  A smaller sample favours small tiles for want of parallelism
// that the whole batch has (make_plan cuts them to a CTA's share anyway): there
// the largest within 10% wins, in float pairs and FP32 (128 dense and 16 tet
// instances: pairs 157 to 159 us over six tunings, 156 to 166 within 3%; FP32
// 81 and 82).  Native FP64 is bound by its FP64 unit, whose work larger tiles
// spread less evenly: 3% there as well (419 us, 459 within 10%).  Choices are
// cached by GPU name, kind, dtype, arithmetic and bucket.
kg_status autotune(kg_batch* b, cudaStream_t s) {
  std::map<std::pair<int, int>, std::vector<int>> groups;  // (kind, bucket) -> instance ids
  for (int i = 0; i < (int)b->probs.size(); ++i) {
    const kg_problem* p = b->probs[i];
    const int kind = p->kind == KG_QUADFORM ? BK_DENSE : BK_TET;
    groups[{kind, bucket_of(kind == BK_DENSE ? p->n : p->m)}].push_back(i);
  }
  std::lock_guard<std::mutex> lk(g_tune_mu);
  std::map<std::string, int> cache = cache_read();
  bool dirty = false;
  // "k6": dense tiles take four rows a step, native FP64 the largest within 3%
  const std::string prefix = b->gpu + "|k6|" + (b->dtype == KG_F64 ? "f64" : "f32") + "|" +
                             (b->pair ? "pair" : "native") + "|";
  const std::vector<int> dense_cands{4, 8, 16, 32, 64, 128, 256}, tet_cands{1024, 2048, 4096, 8192, 16384};
  std::map<std::pair<int, int>, std::vector<int>> sample;
  for (auto& g : groups) {
    const int64_t biggest = g.first.first == BK_DENSE ? dense_cands.back() : tet_cands.back();
    std::vector<int>& ids = sample[g.first];
    int64_t items = 0;
    for (int i : g.second) {
      ids.push_back(i);
      items += (b->probs[i]->m + biggest - 1) / biggest;
      if (items >= 4 * (int64_t)b->grid) break;
    }
  }
  // scratch x / gx for the timing runs (zeros are valid inputs for both kinds)
  size_t need = 0;
  for (auto& g : sample) {
    size_t sz = 0;
    for (int i : g.second) sz += ((size_t)b->probs[i]->n * b->es + 255) & ~size_t(255);
    need = std::max(need, sz);
  }
  void *xbuf = nullptr, *gbuf = nullptr;
  if (dev_alloc(&xbuf, need) != cudaSuccess || dev_alloc(&gbuf, need) != cudaSuccess) {
    cudaFree(xbuf);
    return fail(KG_ERR_OOM, "autotune scratch");
  }
  cudaMemsetAsync(xbuf, 0, need, s);
  kg_status rc = KG_OK;
  for (auto& g : groups) {
    const int kind = g.first.first, bucket = g.first.second;
    const std::string key = prefix + (kind == BK_DENSE ? "dense|" : "tet|") + std::to_string(bucket);
    auto hit = cache.find(key);
    if (hit != cache.end()) {
      (kind == BK_DENSE ? b->tune.dense_rows : b->tune.tet_elems)[bucket] = hit->second;
      continue;
    }
    const std::vector<int>& ids = sample[g.first];
    const std::vector<int>& cands = kind == BK_DENSE ? dense_cands : tet_cands;
    std::vector<float> ms(cands.size(), 0.f);
    for (size_t i = 0; i < cands.size() && rc == KG_OK; ++i) {
      Tuning tu;
      (kind == BK_DENSE ? tu.dense_rows : tu.tet_elems)[bucket] = cands[i];
      rc = time_plan(b, ids, tu, s, xbuf, gbuf, &ms[i]);
    }
    if (rc != KG_OK) break;
    int64_t items = 0;
    for (int i : ids) items += (b->probs[i]->m + cands.back() - 1) / cands.back();
    const bool fp64 = b->dtype == KG_F64 && !b->pair;
    const float slack = fp64 || items >= 4 * (int64_t)b->grid ? 1.03f : 1.10f;
    const float least = *std::min_element(ms.begin(), ms.end());
    int best = cands[0];
    for (size_t i = 0; i < cands.size(); ++i)
      if (ms[i] <= slack * least) best = cands[i];
    (kind == BK_DENSE ? b->tune.dense_rows : b->tune.tet_elems)[bucket] = best;
    cache[key] = best;
    dirty = true;
  }
  cudaFree(xbuf);
  cudaFree(gbuf);
  if (rc == KG_OK && dirty) cache_write(cache);
  return rc;
}

void batch_free(kg_batch* b) {
  if (!b) return;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->dev.release();
  for (void* q : b->own_preps) cudaFree(q);
  if (b->err) cudaFree(b->err);
  delete b;
}

}  // namespace

extern "C" {

kg_status kg_batch_create(kg_batch** out, kg_problem* const* probs, int count,
                          const kg_options* opt, kg_stream stream) {
  if (!out) return fail(KG_ERR_INVALID_ARG, "kg_batch_create: out is NULL");
  *out = nullptr;
  if (!probs || count < 1) return fail(KG_ERR_INVALID_ARG, "kg_batch_create: no problems");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  kg_batch* b = new (std::nothrow) kg_batch();
  if (!b) return fail(KG_ERR_OOM, "kg_batch_create: host allocation");
  b->probs.assign(probs, probs + count);
  b->dtype = b->probs[0] ? b->probs[0]->dtype : KG_F64;
  b->es = b->dtype == KG_F64 ? 8 : 4;
  kg_status rc = KG_OK;
  const int strat = opt ? opt->strategy : KG_STRATEGY_AUTO;
  if (strat != KG_STRATEGY_AUTO && strat != KG_STRATEGY_WARP && strat != KG_STRATEGY_ATOMIC)
    rc = fail(KG_ERR_UNSUPPORTED, "kg_batch_create: strategy must be AUTO, WARP or ATOMIC");
  b->warp = strat == KG_STRATEGY_WARP;  // AUTO: plain atomics (measured ~3% faster here)
  for (kg_problem* p : b->probs) {
    if (rc != KG_OK) break;
    if (!p) rc = fail(KG_ERR_INVALID_ARG, "kg_batch_create: NULL problem");
    else if (p->dtype != b->dtype) rc = fail(KG_ERR_INVALID_ARG, "kg_batch_create: mixed dtypes");
    else if (p->kind == KG_QUADFORM && p->n > B_MAXN)
      rc = fail(KG_ERR_UNSUPPORTED, "kg_batch_create: dense instances need n <= 2048");
    else if (p->kind != KG_QUADFORM && p->kind != KG_TETENERGY)
      rc = fail(KG_ERR_UNSUPPORTED, "kg_batch_create: QUADFORM and TETENERGY only");
    if (rc != KG_OK) break;
  }
  if (rc == KG_OK && dev_alloc((void**)&b->err, 16) != cudaSuccess)
    rc = fail(KG_ERR_OOM, "kg_batch_create: error word");
  if (rc == KG_OK) cudaMemsetAsync(b->err, 0, 16, s);
  // FP64 arithmetic of the batch: pairs when every instance's data is in range
  if (rc == KG_OK && b->dtype == KG_F64) {
    const int want = opt ? opt->arith : KG_ARITH_AUTO;
    bool pair = want != KG_ARITH_NATIVE;
    for (kg_problem* p : b->probs) {
      if (!pair) break;
      if (p->arith == KG_ARITH_PAIR) continue;
      if (p->kind == KG_TETENERGY) {
        pair = false;
        break;
      }
      bool ok = false;
      if ((rc = pair_range_ok(p, static_cast<const double*>(p->data0), p->m * p->n, s, &ok)) != KG_OK)
        break;
      pair = ok;
    }
    if (rc == KG_OK && want == KG_ARITH_PAIR && !pair)
      rc = fail(KG_ERR_UNSUPPORTED, "kg_batch_create: some data is outside the pair range");
    b->pair = pair;
  }
  // the float-pair copies: the instances' own, else (dense instances whose
  // kg_create took none, n < 1024) one the batch makes, largest first, within
  // opt->tape_budget_bytes (0: 1 GiB)
  b->prep.assign(count, nullptr);
  if (rc == KG_OK && b->pair) {
    size_t budget = opt && opt->tape_budget_bytes ? opt->tape_budget_bytes : (size_t(1) << 30);
    std::vector<int> order;
    for (int i = 0; i < count; ++i) {
      kg_problem* p = b->probs[i];
      if (p->aprep && p->arith == KG_ARITH_PAIR) b->prep[i] = p->aprep;
      else if (p->kind == KG_QUADFORM) order.push_back(i);
    }
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
      return b->probs[a]->m * b->probs[a]->n > b->probs[c]->m * b->probs[c]->n;
    });
    for (int i : order) {
      kg_problem* p = b->probs[i];
      // rows of odd n are padded by a zero to whole column pairs
      const size_t bytes = 8 * (size_t)p->m * (size_t)(p->n + (p->n & 1));
      if (bytes > budget) continue;
      void* q = nullptr;
      if (dev_alloc(&q, bytes) != cudaSuccess) {
        rc = fail(KG_ERR_OOM, "kg_batch_create: float-pair copy of A");
        break;
      }
      b->own_preps.push_back(q);
      if ((rc = pair_prepare_rows(static_cast<const double*>(p->data0), q, p->m, p->n, s)) != KG_OK) break;
      b->prep[i] = q;
      budget -= bytes;
    }
  }
  if (rc == KG_OK) {
    b->gpu = gpu_name();
    b->grid = batched_grid(b->pair);
    if (b->pair) {
      const float4* t = nullptr;
      rc = logtab_for_device(&t);
    }
    const char* no_tune = std::getenv("KG_NO_AUTOTUNE");
    if (rc == KG_OK && !(no_tune && no_tune[0] == '1')) rc = autotune(b, s);
  }
  if (rc == KG_OK) {
    std::vector<int> ids(count);
    for (int i = 0; i < count; ++i) ids[i] = i;
    b->plan = make_plan(b->probs, b->prep, ids, b->tune, b->pair, b->es, b->grid);
    rc = devplan_alloc(b->dev, b->plan, s);
  }
  // for tests: the sum items of the first replay give up instead of waiting
  const char* give_up = std::getenv("KG_TEST_BATCH_GIVE_UP");
  if (rc == KG_OK && give_up && give_up[0] == '1') {
    const unsigned one = 1u;
    cudaError_t e = cudaMemcpyAsync(b->dev.head + 2, &one, sizeof(one), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) rc = cuda_fail(e, "kg_batch_create");
  }
  if (rc == KG_OK) {
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) rc = cuda_fail(e, "kg_batch_create");
  }
  if (rc != KG_OK) {
    batch_free(b);
    return rc;
  }
  b->last_stream = s;
  *out = b;
  return KG_OK;
}

static kg_status batch_update_ptrs(kg_batch* b, const void* const* x, void* const* f,
                                   void* const* gx, cudaStream_t s) {
  const int n = (int)b->probs.size();
  for (int i = 0; i < n; ++i)
    if (!x[i] || !gx[i]) return fail(KG_ERR_INVALID_ARG, "kg_grad_batched: NULL x or gx entry");
  bool same = b->ptrs_valid;
  for (int i = 0; same && i < n; ++i)
    same = b->last_x[i] == x[i] && b->last_f[i] == f[i] && b->last_gx[i] == gx[i];
  if (same) return KG_OK;
  b->last_x.assign(x, x + n);
  b->last_f.assign(f, f + n);
  b->last_gx.assign(gx, gx + n);
  for (int i = 0; i < n; ++i) {
    b->plan.insts[i].x = x[i];
    b->plan.insts[i].f = f[i];
    b->plan.insts[i].gx = gx[i];
  }
  cudaError_t e = cudaMemcpyAsync(b->dev.insts, b->plan.insts.data(), sizeof(BInst) * n,
                                  cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return cuda_fail(e, "kg_grad_batched: descriptor update");
  b->ptrs_valid = true;
  return KG_OK;
}

kg_status kg_grad_batched(kg_batch* b, const void* const* x, void* const* f, void* const* gx,
                          kg_stream stream) {
  reset_launch_count();
  if (!b || !x || !f || !gx) return fail(KG_ERR_INVALID_ARG, "kg_grad_batched: NULL argument");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  b->last_stream = s;
  kg_status rc = batch_update_ptrs(b, x, f, gx, s);
  if (rc != KG_OK) return rc;
  cudaError_t e;
  if (!b->exec) {  // capture the launch sequence once, replay it afterwards
    cudaStream_t cs = nullptr;
    if ((e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking)) != cudaSuccess)
      return cuda_fail(e, "kg_grad_batched: capture stream");
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      rc = launch_plan(b->dev, b->dtype, b->pair, b->warp, b->err, cs, b->grid);
      cudaError_t e2 = cudaStreamEndCapture(cs, &b->graph);
      if (rc == KG_OK && e2 != cudaSuccess) rc = cuda_fail(e2, "kg_grad_batched: end capture");
    } else {
      rc = cuda_fail(e, "kg_grad_batched: begin capture");
    }
    cudaStreamDestroy(cs);
    if (rc != KG_OK) return rc;
    if ((e = cudaGraphInstantiate(&b->exec, b->graph, 0)) != cudaSuccess) {
      b->exec = nullptr;
      return cuda_fail(e, "kg_grad_batched: instantiate");
    }
  }
  prof_begin(s, "batched_kernel (graph)");
  e = cudaGraphLaunch(b->exec, s);
  prof_end(s);
  if (e != cudaSuccess) return cuda_fail(e, "kg_grad_batched: launch");
  count_launch(b->dev.ntet > 0 ? 2 : 1);
  return KG_OK;
}

kg_status kg_grad_batched_loop(kg_batch* b, const void* const* x, void* const* f, void* const* gx,
                               kg_stream stream) {
  if (!b || !x || !f || !gx) return fail(KG_ERR_INVALID_ARG, "kg_grad_batched_loop: NULL argument");
  int launches = 0;
  for (size_t i = 0; i < b->probs.size(); ++i) {
    kg_status rc = kg_grad(b->probs[i], x[i], f[i], gx[i], nullptr, nullptr, 0, stream);
    if (rc != KG_OK) return rc;
    launches += kg_last_launch_count();
  }
  reset_launch_count();
  count_launch(launches);
  return KG_OK;
}

kg_status kg_batch_get_config(const kg_batch* b, int* arith, int* items, int* grid) {
  if (!b) return fail(KG_ERR_INVALID_ARG, "kg_batch_get_config: NULL batch");
  if (arith) *arith = b->pair ? KG_ARITH_PAIR : KG_ARITH_NATIVE;
  if (items) *items = b->dev.nitems - (int)b->plan.sums.size();
  if (grid) *grid = b->grid;
  return KG_OK;
}

kg_status kg_batch_sync(kg_batch* b) {
  if (!b) return fail(KG_ERR_INVALID_ARG, "kg_batch_sync: NULL batch");
  cudaError_t e = cudaStreamSynchronize(b->last_stream);
  if (e != cudaSuccess) return cuda_fail(e, "kg_batch_sync");
  unsigned h = 0;
  if ((e = cudaMemcpy(&h, b->err, sizeof(h), cudaMemcpyDeviceToHost)) != cudaSuccess)
    return cuda_fail(e, "kg_batch_sync");
  if (h) cudaMemset(b->err, 0, sizeof(unsigned));
  if (h & ERRBIT_RANGE)
    return fail(KG_ERR_RANGE, "device: an input is outside the float-pair range");
  if (h & ERRBIT_TIMEOUT) return fail(KG_ERR_TIMEOUT, "device: a bounded wait gave up");
  return KG_OK;
}

void kg_batch_destroy(kg_batch* b) {
  if (!b) return;
  cudaStreamSynchronize(b->last_stream);
  batch_free(b);
}

}  // extern "C"
