// Integer outputs of the implicit plan P_ij = exp(u_i + v_j - gamma C_ij) (Sec. 2.1,
// Eq. lagrangian-closed-form): the row argmax and the support {P_ij > tau}.
//
// Every decision is taken on an FP64 exponent formed by a fixed sequence of
// correctly rounded operations (__dmul_rn / __dadd_rn / __dsub_rn are never
// contracted into an FMA), so the results are bit-exact against any IEEE-754
// evaluation of the same sequence:
//   C_ij  = (double)C_ij                       dense cost (exact promotion)
//   C_ij  = s_C * D_ij, D_ij = ((x_i0 - y_j0)^2 + (x_i1 - y_j1)^2) + ...
//                                             points, summed in coordinate order
//   gC_ij = gamma * C_ij
//   argmax: t_ij = v_j - gC_ij        (u_i is constant along row i, exp increasing)
//   support: t_ij = (u_i + v_j) - gC_ij > log_tau
// One warp owns a row; ties of the argmax go to the lowest column index.
#pragma once
#include "common.cuh"

namespace eot {
namespace pint {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kTile = 128;  // other-side points staged per tile (point costs)
constexpr int kMaxD = 64;

// (value, index) pair of a running argmax: an index < 0 marks an empty pair.
// `b` wins over `a` if it is larger, or equal with a lower index.
__device__ __forceinline__ void argmax_merge(double& av, int64_t& ai, double bv, int64_t bi) {
  if (bi < 0) return;
  if (ai < 0 || bv > av || (bv == av && bi < ai)) {
    av = bv;
    ai = bi;
  }
}

template <int MODE>  // MODE 0: argmax of v_j - gC_ij; MODE 1: count of (u_i + v_j) - gC_ij > log_tau
struct Acc {
  double best = 0.0;
  int64_t idx = -1;
  long long cnt = 0;
  __device__ __forceinline__ void add(double ui, double vj, double gC, int64_t j, double log_tau) {
    if constexpr (MODE == 0) {
      const double t = __dsub_rn(vj, gC);
      // a lane visits its columns in increasing order: a later column replaces the
      // held one only if strictly larger
      if (idx < 0 || t > best) {
        best = t;
        idx = j;
      }
    } else {
      const double t = __dsub_rn(__dadd_rn(ui, vj), gC);
      cnt += (t > log_tau) ? 1 : 0;
    }
  }
  // warp-wide combine
  __device__ __forceinline__ void reduce() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if constexpr (MODE == 0) {
        const double bv = __shfl_xor_sync(0xffffffffu, best, o);
        const long long bi = __shfl_xor_sync(0xffffffffu, (long long)idx, o);
        argmax_merge(best, idx, bv, (int64_t)bi);
      } else {
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
      }
    }
  }
  // the same; lane 0 writes row i's result
  __device__ __forceinline__ void finish(int64_t i, int lane, int64_t* idx_out, int64_t* counts,
                                         unsigned long long* total) {
    reduce();
    if (lane != 0) return;
    if constexpr (MODE == 0) {
      idx_out[i] = idx < 0 ? 0 : idx;
    } else {
      if (counts) counts[i] = (int64_t)cnt;
      if (total) atomicAdd(total, (unsigned long long)cnt);
    }
  }
};

// Dense cost (float or double), row-major with leading dimension ldc.
template <class T, int MODE>
__global__ void __launch_bounds__(kThreads) plan_int_dense_kernel(int64_t n, int64_t m, const T* C, int64_t ldc,
                                                                  const double* u, const double* v, double gamma,
                                                                  double log_tau, int64_t* idx_out,
                                                                  int64_t* counts, unsigned long long* total) {
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * kWarps + warp;
  if (i >= n) return;
  const T* crow = C + i * ldc;
  const double ui = MODE == 1 ? u[i] : 0.0;
  Acc<MODE> acc;
  for (int64_t j = lane; j < m; j += 32) {
    const double gC = __dmul_rn(gamma, (double)__ldg(crow + j));
    acc.add(ui, __ldg(v + j), gC, j, log_tau);
  }
  acc.finish(i, lane, idx_out, counts, total);
}

// Point costs: C_ij = s_C * sum_k (x_ik - y_jk)^2 in coordinate order. The CTA's
// 8 rows share tiles of kTile other-side points, staged coordinate-major in
// shared memory (lanes read consecutive points: no bank conflicts); each warp
// keeps its row's coordinates, promoted to FP64, in shared memory (broadcast reads).
template <int MODE>
__global__ void __launch_bounds__(kThreads) plan_int_points_kernel(int64_t n, int64_t m, int d, const float* X,
                                                                   const float* Y, double sC, const double* u,
                                                                   const double* v, double gamma, double log_tau,
                                                                   int64_t* idx_out, int64_t* counts,
                                                                   unsigned long long* total) {
  __shared__ float ys[kMaxD][kTile];
  __shared__ double xs[kWarps][kMaxD];
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * kWarps + warp;
  const bool rv = i < n;
  for (int k = lane; k < d; k += 32) xs[warp][k] = rv ? (double)X[i * d + k] : 0.0;
  const double ui = (MODE == 1 && rv) ? u[i] : 0.0;
  Acc<MODE> acc;
  for (int64_t j0 = 0; j0 < m; j0 += kTile) {
    const int tw = (int)min((int64_t)kTile, m - j0);
    __syncthreads();
    // the tile's tw * d floats are contiguous in Y: coalesced loads, transposed store
    for (int q = threadIdx.x; q < tw * d; q += kThreads) {
      const int jj = q / d, k = q - jj * d;
      ys[k][jj] = Y[(j0 + jj) * d + k];
    }
    __syncthreads();
    if (!rv) continue;
    for (int jj = lane; jj < tw; jj += 32) {
      double D = 0.0;
      for (int k = 0; k < d; ++k) {
        const double df = __dsub_rn(xs[warp][k], (double)ys[k][jj]);
        D = __dadd_rn(D, __dmul_rn(df, df));
      }
      const double gC = __dmul_rn(gamma, __dmul_rn(sC, D));
      acc.add(ui, __ldg(v + j0 + jj), gC, j0 + jj, log_tau);
    }
  }
  if (rv) acc.finish(i, lane, idx_out, counts, total);
}

// ---- FP32 screening -------------------------------------------------------
//
// The decisions above need FP64, and this GPU's FP64 pipe retires two lanes per
// SM and clock: with every entry decided there, the 64 x 64 grid (n = m = 4096)
// took 158 us (argmax) and 192 us (support), and clouds of n = m = 8192 in
// d = 64 took 34 ms each. Almost every entry is decided by a wide margin, so the
// kernels below form each exponent in FP32 with a bound on its error, and only
// the entries that the bound leaves open are formed again in FP64, by the same
// sequence of rounded operations as before: the same results bit for bit.
//
// With tf the FP32 value of t = v_j - gC_ij and V a bound on |v_j|,
//     |tf - t| <= c (V + |tf|),
// c = 2^-22 for FP32 costs (v cut to FP32: 2^-23 |v|; gamma rounded: 2^-24 gC; the
// FMA: 2^-24 |tf|; gC <= |v| + |t|), 2^-21 for FP64 costs (C cut to FP32 as well)
// and (d + 12) 2^-24 for points (D from d differences, squares and sums: (d + 3)
// 2^-24 D). x -> x +- c |x| is increasing, so an entry below
//     M - 3 c (V + |M|) - slack        (M: the largest tf met so far)
// is below the entry that gave M in FP64 too, and no later entry changes that;
// likewise tf decides against a threshold outside 3 c (V + |threshold|) + slack. A NaN
// (gamma = 0 with a cost beyond FP32's range, whose exponent is v_j) decides nothing.
// `slack` covers FP32 underflow. The bound holds for 1e-30 <= gamma (s_C) <= 1e30
// or 0 and for |V|, |M| and thresholds up to 1e8 (an exponent that overflows FP32
// is then below every one that matters); rows outside, or with a NaN or +inf, are
// decided by the all-FP64 scan of the row. So is a row whose maximum only came within
// 1e8 after entries were passed over that the margin at the final maximum does not
// rule out.

constexpr float kScreenMax = 1.0e8f;

__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
// |v_j| as it enters V: -inf (a column without mass: never the answer) counts 0; NaN,
// +inf and what lies beyond FP32's range make V infinite
__device__ __forceinline__ float bound_of(float vf, double v) {
  const float a = fabsf(vf);
  if (a <= 3.4e38f) return a;
  return __double2hiint(v) == (int)0xfff00000 && __double2loint(v) == 0 ? 0.f : INFINITY;
}
struct Screen {
  float g;      // gamma (dense) or gamma s_C (points), rounded to FP32
  float c3;     // 3 c
  float slack;
};
__device__ __forceinline__ float screen_margin(const Screen& sc, float V, float at) {
  return fmaf(sc.c3, V + fabsf(at), sc.slack);
}
// support thresholds of a row: tf > hi counts, tf < lo does not; between: FP64.
// Returns false when the row needs the all-FP64 scan.
__device__ __forceinline__ bool support_bounds(const Screen& sc, float V, double ui, double log_tau, float& lo,
                                               float& hi) {
  if (ui == -INFINITY) {  // a row without mass counts nothing
    lo = hi = INFINITY;
    return true;
  }
  const double thr = log_tau - ui;
  if (!(V <= kScreenMax) || !(fabs(thr) <= (double)kScreenMax)) return false;
  const float tf = (float)thr;
  // 2^-50 (|u| + |log tau|): the FP64 roundings of (u + v) and of thr
  const float dlt = screen_margin(sc, V, tf) + (float)((fabs(ui) + fabs(log_tau)) * 8.9e-16);
  lo = tf - dlt;
  hi = tf + dlt;
  return dlt <= kScreenMax;
}

// Dense cost: one warp per row, 8 rows per CTA. Column potentials are cut to FP32
// into a shared tile by the CTA (shared by its rows); a lane streams its part of
// the row in batches of 16 entries (4 x 16 bytes when the rows are aligned), the
// next batch's loads in flight while one is tested. Bound by the read of C:
// n = m = 4096, FP32 (67 MB), argmax and support together: 349 -> 56 us on one GB300 (60
// to 86 us on others); with three CTAs per SM (512 CTAs, the second wave nearly empty) 78
// us where it took 56.
constexpr int kScreenTile = 4096;
template <class T, int V, int MODE>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 && V > 1 ? 4 : 2) plan_screen_dense_kernel(int64_t n, int64_t m, const T* C, int64_t ldc,
                                                                     const double* u, const double* v,
                                                                     double gamma, double log_tau, Screen sc,
                                                                     int64_t* idx_out, int64_t* counts,
                                                                     unsigned long long* total) {
  constexpr int U = 16 / V;
  __shared__ __align__(16) float vt[kScreenTile];
  __shared__ float vmax[kWarps];
  __shared__ float skipped[kWarps];  // argmax: the row's largest entry passed over because the maximum was out of reach
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) skipped[warp] = -INFINITY;
  const int64_t i = (int64_t)blockIdx.x * kWarps + warp;
  const bool rv = i < n;
  const T* crow = C + (rv ? i : 0) * ldc;
  const double ui = MODE == 1 && rv ? u[i] : 0.0;
  const uint64_t pol = cost_policy(0);
  float Vb = 0.f, M = -INFINITY, lo = 0.f, hi = 0.f;
  bool ok = true;
  Acc<MODE> acc;
  for (int64_t t0 = 0; t0 < m; t0 += kScreenTile) {
    const int tw = (int)min((int64_t)kScreenTile, m - t0);
    T cA[U][V], cB[U][V];
    auto load = [&](int j0, T (&c)[U][V]) {
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const int j = j0 + q * 32 * V;
        if (j < tw) ld_stream(crow + t0 + j, c[q], pol);
      }
    };
    if (rv) load(lane * V, cA);
    if (t0 > 0) __syncthreads();  // every warp is done with the previous tile
    float vb = 0.f;
    for (int q = threadIdx.x; q < tw; q += kThreads) {
      const float vf = cut_f32(__ldg(v + t0 + q));
      vt[q] = vf;
      vb = fmaxf(vb, bound_of(vf, __ldg(v + t0 + q)));
    }
    vb = warp_max_f(vb);
    if (lane == 0) vmax[warp] = vb;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kWarps; ++q) Vb = fmaxf(Vb, vmax[q]);
    if constexpr (MODE == 1) ok = ok && support_bounds(sc, Vb, ui, log_tau, lo, hi);
    else ok = ok && Vb <= kScreenMax;
    if (!rv || !ok) continue;  // (uniform in the warp)
    // the exact decision on one entry of this lane
    auto exact = [&](T cij, int64_t j) {
      const double gC = __dmul_rn(gamma, (double)cij);
      const double vj = __ldg(v + j);
      if constexpr (MODE == 0) argmax_merge(acc.best, acc.idx, __dsub_rn(vj, gC), j);
      else acc.cnt += (__dsub_rn(__dadd_rn(ui, vj), gC) > log_tau) ? 1 : 0;
    };
    auto test = [&](int j0, const T (&c)[U][V]) {
      float tf[U][V];
      float mx = -INFINITY;
      int above = 0, not_below = 0;
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const int j = j0 + q * 32 * V;
        float b[V];
        if (j < tw) {
          ld_vec_smem<V>(&vt[j], b);
        } else {
#pragma unroll
          for (int e = 0; e < V; ++e) b[e] = -INFINITY;
        }
#pragma unroll
        for (int e = 0; e < V; ++e) {
          tf[q][e] = j < tw ? fmaf(-sc.g, cut_f32(c[q][e]), b[e]) : -INFINITY;
          if constexpr (MODE == 0) mx = max_nan(mx, tf[q][e]);
          else {
            above += tf[q][e] > hi ? 1 : 0;
            // (a NaN is open; of an FP32 cost it is a NaN in FP64 too, which counts nowhere)
            if constexpr (sizeof(T) == 8) not_below += tf[q][e] < lo ? 0 : 1;
            else not_below += tf[q][e] >= lo ? 1 : 0;
          }
        }
      }
      if constexpr (MODE == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        M = max_nan(M, mx);
        const float thr = M - screen_margin(sc, Vb, M);
        if (!(fabsf(M) <= kScreenMax)) {
          if (lane == 0) skipped[warp] = M;
        } else if (mx >= thr) {  // (uniform) the batch holds a contender
#pragma unroll
          for (int q = 0; q < U; ++q)
#pragma unroll
            for (int e = 0; e < V; ++e)
              if (tf[q][e] >= thr) exact(c[q][e], t0 + j0 + q * 32 * V + e);
        }
      } else {
        acc.cnt += above;
        if (not_below != above) {
#pragma unroll
          for (int q = 0; q < U; ++q)
#pragma unroll
            for (int e = 0; e < V; ++e)
              if (!(tf[q][e] < lo) && !(tf[q][e] > hi)) exact(c[q][e], t0 + j0 + q * 32 * V + e);
        }
      }
    };
    constexpr int STEP = 32 * V * U;
    // warp-uniform loop (the batch maximum is taken over the warp)
    for (int b0 = 0; b0 < tw; b0 += 2 * STEP) {
      const int j0 = b0 + lane * V;
      load(j0 + STEP, cB);
      test(j0, cA);
      if (b0 + STEP >= tw) break;
      load(j0 + 2 * STEP, cA);
      test(j0 + STEP, cB);
    }
  }
  if (!rv) return;
  // (a maximum that came into reach late: what was skipped before must lie below it for sure)
  if constexpr (MODE == 0) {
    __syncwarp();
    ok = ok && fabsf(M) <= kScreenMax && skipped[warp] < M - screen_margin(sc, Vb, M);
  }
  if (!ok) {  // outside the bound's reach: every entry in FP64
    acc = Acc<MODE>();
    for (int64_t j = lane; j < m; j += 32) {
      const double gC = __dmul_rn(gamma, (double)__ldg(crow + j));
      acc.add(ui, __ldg(v + j), gC, j, log_tau);
    }
  }
  acc.finish(i, lane, idx_out, counts, total);
}

// Point costs: a CTA decides kSR rows against its chunk of the columns, the CTAs
// of a cluster (up to 8 along the columns, so that few rows still fill the GPU)
// share the rows and rank 0 merges their results through distributed shared
// memory: no global scratch, so calls stay asynchronous and independent. FP32
// bound (a subtraction and an FMA per entry and coordinate, packed in pairs so that
// the issue slots left take the rest): each thread forms a 4 x 8 tile of squared
// distances in registers from coordinate-major tiles in shared memory, three
// 16-byte shared loads per 32 entries and coordinate.
// n = m = 8192, d = 64, argmax and support together: 68.5 ms -> 0.95 ms (0.43 ms
// would be the FP32 pipe's time; the rest is staging, the FP64 decisions and tails).
constexpr int kSR = 64;          // rows per CTA
constexpr int kSC = 128;         // columns per tile
constexpr int kSK = 32;          // coordinates per staged chunk
constexpr int kSPad = kSC + 4;   // staged row stride: 16-byte rows, staggered banks
constexpr int kCand = 16;        // argmax: contenders kept per row
constexpr int kOpen = 1024;      // support: undecided entries kept per CTA

struct ScreenSmem {
  float xs[kMaxD][kSR];                     // the rows' coordinates
  union {
    float ys[kSK][kSPad];                   // a chunk of the tile's coordinates
    double cand_t[kSR][kCand];              // (after the sweep) FP64 exponents of the contenders
    struct {                                // (at the end) this CTA's part of the all-FP64 scans
      double best[kSR];
      long long idx[kSR];
      long long cnt[kSR];
    } part;
  };
  float vt[kSC];
  float red[kWarps];
  union {
    struct {
      float tf[kSR][kCand];
      int32_t j[kSR][kCand];
    } cand;
    int32_t open[kOpen][2];                 // (row of the CTA, column)
  };
  int ncand[kSR];
  float skipped[kSR];                       // argmax: the largest entry passed over, see the dense kernel
  int nopen;
  double best[kSR];                         // results of this CTA's chunk, read by rank 0
  long long idx[kSR];
  long long cnt[kSR];
  int scan[kSR];                            // the row needs the all-FP64 scan, says this CTA's chunk
  int any[kSR];                             // ... says any chunk
};

// The exact exponent pieces of one entry, as plan_int_points_kernel forms them.
__device__ __forceinline__ double exact_gC(const float* x, int xstride, const float* y, int d, double sC,
                                           double gamma) {
  double D = 0.0;
  for (int k = 0; k < d; ++k) {
    const double df = __dsub_rn(widen(x[k * xstride]), widen(__ldg(y + k)));
    D = __dadd_rn(D, __dmul_rn(df, df));
  }
  return __dmul_rn(gamma, __dmul_rn(sC, D));
}

template <class V>
__device__ __forceinline__ V ld_cluster(const V* p, uint32_t rank) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  if constexpr (sizeof(V) == 8) {
    unsigned long long q;
    asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(q) : "r"(ra) : "memory");
    return *reinterpret_cast<V*>(&q);
  } else {
    uint32_t q;
    asm volatile("ld.shared::cluster.b32 %0, [%1];" : "=r"(q) : "r"(ra) : "memory");
    return *reinterpret_cast<V*>(&q);
  }
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, 2) plan_screen_points_kernel(int64_t n, int64_t m, int d, const float* X,
                                                                         const float* Y, double sC, const double* u,
                                                                         const double* v, double gamma,
                                                                         double log_tau, Screen sc, int64_t chunk,
                                                                         int64_t* idx_out, int64_t* counts,
                                                                         unsigned long long* total) {
  __shared__ __align__(16) ScreenSmem s;
  pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rg = tid >> 4, cg = tid & 15;  // this thread's rows 4 rg .. 4 rg + 3; 16 threads per row
  const int64_t i0 = (int64_t)blockIdx.x * kSR;
  const int64_t c0 = min(m, (int64_t)blockIdx.y * chunk), c1 = min(m, c0 + chunk);
  for (int q = tid; q < kSR * d; q += kThreads) {
    const int r = q / d, k = q - r * d;
    s.xs[k][r] = i0 + r < n ? X[(i0 + r) * d + k] : 0.f;
  }
  // V of the chunk
  float Vb = 0.f;
  for (int64_t j = c0 + tid; j < c1; j += kThreads) {
    const double vj = __ldg(v + j);
    Vb = fmaxf(Vb, bound_of(cut_f32(vj), vj));
  }
  Vb = warp_max_f(Vb);
  if (lane == 0) s.red[warp] = Vb;
  if (tid < kSR) {
    s.ncand[tid] = 0;
    s.skipped[tid] = -INFINITY;
    s.best[tid] = 0.0;
    s.idx[tid] = -1;
    s.cnt[tid] = 0;
    s.scan[tid] = 0;
  }
  if (tid == 0) s.nopen = 0;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kWarps; ++q) Vb = fmaxf(Vb, s.red[q]);
  float M[4], lo[4], hi[4];
  int above_r[4];
  bool rok[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    M[r] = -INFINITY;
    lo[r] = hi[r] = 0.f;
    above_r[r] = 0;
    const int64_t i = i0 + 4 * rg + r;
    if constexpr (MODE == 1) rok[r] = i < n && support_bounds(sc, Vb, u[i], log_tau, lo[r], hi[r]);
    else rok[r] = i < n && Vb <= kScreenMax;
    if (i < n && !rok[r]) s.scan[4 * rg + r] = 1;  // (the same value from each of the row's threads)
  }

  // The staged pieces (tile, chunk of coordinates) in order; a piece is loaded into
  // registers while the one before it is worked on. Wide chunks: a lane owns a
  // coordinate (coalesced along the point), 4 columns per store; narrow ones: a
  // thread owns a column.
  float pre[16];
  float pre_v = 0.f;
  auto fetch = [&](int64_t jt, int k0) {
    const int kn = min(kSK, d - k0);
    const int tn = (int)min((int64_t)kSC, c1 - jt);
    const float* yt = Y + jt * d + k0;
    if (kn > 8) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int jj = 4 * (warp + 8 * q) + e;
          pre[4 * q + e] = lane < kn && jj < tn ? __ldg(yt + jj * d + lane) : 0.f;
        }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = (tid >> 7) + 2 * q, jj = tid & (kSC - 1);
        pre[q] = k < kn && jj < tn ? __ldg(yt + jj * d + k) : 0.f;
      }
    }
    if (k0 == 0 && tid < kSC) pre_v = tid < tn ? cut_f32(__ldg(v + jt + tid)) : -INFINITY;
  };
  auto store = [&](int k0) {
    const int kn = min(kSK, d - k0);
    if (kn > 8) {
      if (lane < kn) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<float4*>(&s.ys[lane][4 * (warp + 8 * q)]) =
              make_float4(pre[4 * q], pre[4 * q + 1], pre[4 * q + 2], pre[4 * q + 3]);
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = (tid >> 7) + 2 * q;
        if (k < kn) s.ys[k][tid & (kSC - 1)] = pre[q];
      }
    }
    if (k0 == 0 && tid < kSC) s.vt[tid] = pre_v;
  };
  fetch(c0, 0);
  for (int64_t jt = c0; jt < c1; jt += kSC) {
    unsigned long long a2[4][4];  // pairs of columns (e, e + 1) of the squared distances
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int e = 0; e < 4; ++e) a2[r][e] = 0ull;
    for (int k0 = 0; k0 < d; k0 += kSK) {
      const int kn = min(kSK, d - k0);
      __syncthreads();  // every thread is done with the previous piece
      store(k0);
      __syncthreads();
      if (k0 + kSK < d) fetch(jt, k0 + kSK);
      else if (jt + kSC < c1) fetch(jt + kSC, 0);
#pragma unroll 4
      for (int k = 0; k < kn; ++k) {
        const float4 x4 = *reinterpret_cast<const float4*>(&s.xs[k0 + k][4 * rg]);
        const ulonglong2 ya = *reinterpret_cast<const ulonglong2*>(&s.ys[k][4 * cg]);
        const ulonglong2 yb = *reinterpret_cast<const ulonglong2*>(&s.ys[k][64 + 4 * cg]);
        const float x[4] = {x4.x, x4.y, x4.z, x4.w};
        const unsigned long long y[4] = {ya.x, ya.y, yb.x, yb.y};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          unsigned long long nx;  // (-x, -x)
          asm("mov.b64 %0, {%1, %1};" : "=l"(nx) : "f"(-x[r]));
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            unsigned long long df;
            asm("add.rn.f32x2 %0, %1, %2;" : "=l"(df) : "l"(y[e]), "l"(nx));
            asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(a2[r][e]) : "l"(df));
          }
        }
      }
    }
    float acc[4][8];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[r][2 * e]), "=f"(acc[r][2 * e + 1]) : "l"(a2[r][e]));
    // entry e of this thread: column jt + 4 cg + e, or jt + 64 + 4 cg + (e - 4)
    float h[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) h[e] = s.vt[(e < 4 ? 0 : 60) + 4 * cg + e];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int row = 4 * rg + r;
      if constexpr (MODE == 0) {
        float mx = -INFINITY;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          acc[r][e] = fmaf(-sc.g, acc[r][e], h[e]);
          mx = max_nan(mx, acc[r][e]);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        M[r] = max_nan(M[r], mx);
        const float thr = M[r] - screen_margin(sc, Vb, M[r]);
        const bool in = fabsf(M[r]) <= kScreenMax, hit = rok[r] && mx >= thr && in;  // (the same in the row's 16 threads)
        if (!in && cg == 0) s.skipped[row] = M[r];
        if (__any_sync(0xffffffffu, hit)) {
          if (hit) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
              if (acc[r][e] >= thr) {
                const int at = atomicAdd(&s.ncand[row], 1);
                if (at < kCand) {
                  s.cand.tf[row][at] = acc[r][e];
                  s.cand.j[row][at] = (int32_t)(jt + (e < 4 ? 0 : 60) + 4 * cg + e);
                } else {
                  s.scan[row] = 1;  // too many near ties: the row is scanned in FP64
                }
              }
          }
          __syncwarp();
          // drop what the new maximum rules out: one held contender per thread
          const unsigned half = 0xffffu << (lane & 16);
          const int have = min(s.ncand[row], kCand);
          const float f = cg < have ? s.cand.tf[row][cg] : 0.f;
          const int32_t fj = cg < have ? s.cand.j[row][cg] : 0;
          const bool keep = hit && cg < have && f >= thr;
          const unsigned kept = __ballot_sync(0xffffffffu, keep) & half;
          __syncwarp();
          if (hit) {
            if (keep) {
              const int at = __popc(kept & ((1u << lane) - 1u));
              s.cand.tf[row][at] = f;
              s.cand.j[row][at] = fj;
            }
            if (cg == 0) s.ncand[row] = __popc(kept);
          }
          __syncwarp();
        }
      } else {
        int above = 0, below = 0;  // the rest, NaNs among it, is open
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          acc[r][e] = fmaf(-sc.g, acc[r][e], h[e]);
          above += acc[r][e] > hi[r] ? 1 : 0;
          below += acc[r][e] < lo[r] ? 1 : 0;
        }
        above_r[r] += above;
        if (above + below != 8 && rok[r]) {
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (!(acc[r][e] < lo[r]) && !(acc[r][e] > hi[r])) {
              const int at = atomicAdd(&s.nopen, 1);
              if (at < kOpen) {
                s.open[at][0] = row;
                s.open[at][1] = (int32_t)(jt + (e < 4 ? 0 : 60) + 4 * cg + e);
              } else {
                s.scan[row] = 1;
              }
            }
        }
      }
    }
  }
  __syncthreads();
  if constexpr (MODE == 0) {
    // (a chunk whose exponents are all -inf has nothing to offer; a maximum that came
    // into reach late: what was skipped before must lie below it for sure)
    if (cg == 0) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const bool done = fabsf(M[r]) <= kScreenMax ? s.skipped[4 * rg + r] < M[r] - screen_margin(sc, Vb, M[r])
                                                    : M[r] == -INFINITY;
        if (rok[r] && !done) s.scan[4 * rg + r] = 1;
      }
    }
    // the contenders' exact exponents; every thread takes (row, slot) pairs
    for (int q = tid; q < kSR * kCand; q += kThreads) {
      const int row = q & (kSR - 1), k = q / kSR;
      if (k < s.ncand[row]) {
        const int64_t j = s.cand.j[row][k];
        s.cand_t[row][k] =
            __dsub_rn(__ldg(v + j), exact_gC(&s.xs[0][row], kSR, Y + j * d, d, sC, gamma));
      }
    }
    __syncthreads();
    if (tid < kSR) {
      double bv = 0.0;
      int64_t bi = -1;
      for (int k = 0; k < s.ncand[tid]; ++k) argmax_merge(bv, bi, s.cand_t[tid][k], (int64_t)s.cand.j[tid][k]);
      s.best[tid] = bv;
      s.idx[tid] = bi;
    }
  } else {
    const int no = min(s.nopen, kOpen);
    for (int q = tid; q < no; q += kThreads) {
      const int row = s.open[q][0];
      const int64_t j = s.open[q][1];
      const double gC = exact_gC(&s.xs[0][row], kSR, Y + j * d, d, sC, gamma);
      if (__dsub_rn(__dadd_rn(u[i0 + row], __ldg(v + j)), gC) > log_tau)
        atomicAdd((unsigned long long*)&s.cnt[row], 1ull);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int c = above_r[r];
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
      if (cg == 0 && rok[r]) atomicAdd((unsigned long long*)&s.cnt[4 * rg + r], (unsigned long long)c);
    }
  }
  cluster_sync();  // every chunk's results are visible to the cluster
  const uint32_t ranks = gridDim.y;
  // Rows that need the all-FP64 scan: every CTA scans its own chunk of them, one warp per
  // row (a cloud with repeated points, say 8-bit colours, has most of its rows here).
  int need = 0;
  if (tid < kSR) {
    bool none = MODE == 0;
    for (uint32_t q = 0; q < ranks; ++q) {
      need |= ld_cluster(&s.scan[tid], q);
      if constexpr (MODE == 0) none = none && ld_cluster(&s.idx[tid], q) < 0;
    }
    need = i0 + tid < n && (need || none) ? 1 : 0;
    s.any[tid] = need;
  }
  if (__syncthreads_or(need)) {  // (the same in every CTA of the cluster)
    for (int r = warp; r < kSR; r += kWarps) {
      if (!s.any[r]) continue;
      Acc<MODE> acc;
      const double ui = MODE == 1 ? u[i0 + r] : 0.0;
      for (int64_t j = c0 + lane; j < c1; j += 32)
        acc.add(ui, __ldg(v + j), exact_gC(&s.xs[0][r], kSR, Y + j * d, d, sC, gamma), j, log_tau);
      acc.reduce();
      if (lane == 0) {
        if constexpr (MODE == 0) {
          s.part.best[r] = acc.best;
          s.part.idx[r] = acc.idx;
        } else {
          s.part.cnt[r] = acc.cnt;
        }
      }
    }
    cluster_sync();  // the parts are visible to rank 0
  }
  if (cluster_rank() == 0) {
    long long c = 0;
    if (tid < kSR && i0 + tid < n) {
      const bool f = s.any[tid];
      if constexpr (MODE == 0) {
        double bv = 0.0;
        int64_t bi = -1;
        for (uint32_t q = 0; q < ranks; ++q)
          argmax_merge(bv, bi, ld_cluster(f ? &s.part.best[tid] : &s.best[tid], q),
                       (int64_t)ld_cluster(f ? &s.part.idx[tid] : &s.idx[tid], q));
        idx_out[i0 + tid] = bi < 0 ? 0 : bi;
      } else {
        for (uint32_t q = 0; q < ranks; ++q) c += ld_cluster(f ? &s.part.cnt[tid] : &s.cnt[tid], q);
        if (counts) counts[i0 + tid] = c;
      }
    }
    if constexpr (MODE == 1) {
      if (total && warp < kSR / 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (lane == 0 && c) atomicAdd(total, (unsigned long long)c);
      }
    }
  }
  cluster_sync();  // no CTA leaves while rank 0 reads its shared memory
}
}  // namespace pint
}  // namespace eot
