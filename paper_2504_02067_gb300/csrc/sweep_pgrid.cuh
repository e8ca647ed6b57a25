// Mixed-precision sweeps of low-dimensional point clouds (d <= 16) from split
// coordinates. As pts_sweep_kernel (sweep_pts.cuh) they form the cost
// C_ij = s_C |x_i - y_j|^2 on the fly; the exponent is kept in base 2,
//     t2_ij = (Ah_i + Bh_j) log2 e - |x'_i - y'_j|^2,   x' = sqrt(gamma s_C log2 e) (x - x_0),
// so that no scaling is left per entry and ex2 takes t2 as it is. Every scaled
// coordinate is split where it is staged, x' = xh + xl with xh on a grid of step s (a
// power of two) and |xl| <= s / 2, and
//     |x' - y'|^2 = sum dh^2 + sum dl (2 dh + dl),   dh = xh - yh, dl = xl - yl.
// s = 2^ceil(log2(sqrt(D')) - 11.5) for D' >= max |x' - y'|^2 makes dh and dh^2 exact
// in FP32 and keeps the running sum of Ah + Bh (on the 1/8 grid, s^2 <= 1/8) and the
// -dh^2 exact while below 2 D'. What is rounded is dl and the second sum, at 2^-25 of
// dh s: up to sqrt(D') s where every pair is far apart (translated clouds), so this
// serves D' <= 2^11. Beyond, up to 2^15, a third part xm on the grid 2^-11 s takes
// the products dh dm, exact as well, out of the second sum:
//     sum dh^2 + 2 sum dh dm + sum dm (dm + 2 dl) + 2 sum dh dl.
// Relative error of the plan's entries (rms over the mass, FP32 emulated against 64
// bits, Sinkhorn potentials; uniform clouds in the unit cube, then one of them moved
// by 5; the general sweeps / these):
//     D'      parts  d = 2                             d = 16
//     739     2      5.5e-8 / 2.7e-8, 6.1e-8 / 3.2e-8  3.4e-8 / 2.0e-8, 6.7e-8 / 3.9e-8
//     2047    2      4.7e-8 / 2.3e-8, 6.5e-8 / 3.8e-8  3.1e-8 / 2.1e-8, 4.3e-8 / 3.8e-8
//     2955    3      4.1e-8 / 2.2e-8, 6.4e-8 / 3.1e-8  3.2e-8 / 1.6e-8, 4.0e-8 / 2.0e-8
//     31740   3      2.8e-8 / 1.6e-8, 5.2e-8 / 2.5e-8  2.9e-8 / 1.5e-8, 3.0e-8 / 1.6e-8
// (two parts at 31740, one cloud moved: 3.0e-7 and 5.4e-7). t2 is rounded once; the
// scheme of sweep_pts.cuh (TwoSum differences, compensated squares, a two-term
// gamma s_C) rounds four times. Five FP32 instructions per coordinate (eight with
// three parts) against eighteen.
//
// Work split: FP32-issue-bound for large clouds (each thread owns RO elements, the
// other side's records are broadcast from shared memory), latency-bound for small
// ones, where a CTA's warps split the other side `ws` ways for the same own
// elements and a cluster of up to 8 CTAs splits it further. All partial sums meet in
// shared memory, then through distributed shared memory in rank order: no global
// partials, no ticket, a fixed order. Measured (general sweeps -> these): gradients of
// n = m = 65536, d = 3 (four sweeps) 62.4 -> 18.5 ms; training step of n = 1000,
// m = 700, d = 2 36.8 -> 13.3 ms.
#pragma once
#include "sweep_pts.cuh"

namespace eot {
namespace pg {

constexpr int kMaxD = 16;
// The split's range of gamma s_C log2(e) max |x - y|^2 (base-2 exponent units), tested at
// every temperature; the general sweeps serve the rest (below, the scale of the
// coordinates runs out of FP32: a gamma that FP32 rounds to 0, coinciding points).
constexpr double kMinBound = 0x1p-40;
constexpr double kMaxTwo = 2048.0;     // two parts per coordinate
constexpr double kMaxBound = 32768.0;  // three
__host__ __device__ inline int parts_of(double bound) {  // 0: the general sweeps
  return !(bound >= kMinBound && bound <= kMaxBound) ? 0 : bound <= kMaxTwo ? 2 : 3;
}
// The online max of an LSE moves in whole units of the base-2 exponent, so that every
// rescaling (here and where partial sums meet) is by an exact power of two.
constexpr float kThetaB2 = 12.0f;      // lazy-rescale threshold
constexpr float kLowest = -2097152.0f; // an LSE's start: below every exponent of the split range
constexpr double kLog2eD = 1.4426950408889634074;
constexpr double kLn2D = 0.69314718055994530942;

struct Args {
  const double* dmax;  // device: >= max |x_i - y_j|^2
  int ws;              // warps of a CTA that share own elements (1, 2, 4 or 8)
};

struct Geo {
  int64_t B, S, chunk;
  int ro, ws;
};
// Fewest waves x per-thread entries. A CTA's fixed cost (prologue, combine, epilogue:
// about 2 us) is worth about 48 entries per thread at two CTAs per SM; staging an
// other-side record costs a thread about 3.5 entries.
// grad: the gradient sweeps, with a sum per coordinate in registers; parts: of a coordinate.
inline Geo geo_of(int sms, int64_t n_own, int64_t n_oth, int d, bool grad, int parts) {
  Geo best{};
  double bc = -1.0;
  for (int ro : {1, 2, 4}) {
    const bool built = parts == 3 ? (ro == 1 || (d <= 4 && ro == 2))
                       : grad     ? (ro == 1 || (d <= 4 && ro == 2))
                                  : (d <= 4 ? ro != 2 : ro == 2);
    if (!built) continue;
    for (int ws : {1, 2, 4, 8}) {
      const int64_t own = (int64_t)(kThreads / ws) * ro, B = (n_own + own - 1) / own;
      for (int64_t S = 1; S <= 8; ++S) {
        const int64_t chunk = ((n_oth + S - 1) / S + 7) / 8 * 8, Sr = (n_oth + chunk - 1) / chunk;
        if (Sr != S) continue;
        const int64_t waves = (B * S + 2 * sms - 1) / (2 * sms);
        const double c = (double)waves * (48.0 + (double)((chunk + ws - 1) / ws) * ro + 3.5 * (double)((chunk + kThreads - 1) / kThreads));
        if (bc < 0.0 || c < bc) {
          bc = c;
          best = Geo{B, S, chunk, ro, ws};
        }
      }
    }
  }
  return best;
}

// dX, dY: out_e,k = scale ownfac_e sum_o P-weights (x_e - x_o)_k, the sum in scaled
// coordinates (1 / sigma undoes the scaling)
struct GradEpi {
  static constexpr int kDot = 0;
  double scale;
  const double* ownfac;
  float* out;
  int d;
  template <int D>
  __device__ void grad(int64_t e, const double (&v)[D], double inv_sigma) {
    const double f = scale * ownfac[e] * inv_sigma;
#pragma unroll
    for (int k = 0; k < D; ++k)
      if (k < d) out[e * d + k] = (float)(f * v[k]);
  }
  __device__ void finish(const double*) {}
};

struct Scale {
  float sh, sl;   // sigma = sqrt(gamma s_C log2 e) as an FP32 pair
  float magic;    // 1.5 x 2^23 s: adding and subtracting it rounds to the grid
  double sigma;
};

// (x - c) sigma as a grid part, (P = 3) a part on the grid 2^-11 s, and a remainder
template <int P>
__device__ __forceinline__ void split_coord(float x, float c, const Scale& sc, float& xh, float& xm, float& xl) {
  const float t = sub_rn(x, c);  // TwoSum: x - c = t + e
  const float bv = sub_rn(t, x);
  const float e = sub_rn(sub_rn(x, sub_rn(t, bv)), add_rn(c, bv));
  const float p = mul_rn(t, sc.sh);
  const float pe = fmaf(t, sc.sh, -p) + fmaf(t, sc.sl, e * sc.sh);
  xh = sub_rn(add_rn(p, sc.magic), sc.magic);
  const float r = sub_rn(p, xh);
  if constexpr (P == 3) {
    const float magic = sc.magic * 0x1p-11f;
    xm = sub_rn(add_rn(r, magic), magic);
    xl = add_rn(sub_rn(r, xm), pe);
  } else {
    xl = add_rn(r, pe);
  }
}
// A log2 e (A on the 1/8 grid, |A| < 2^19) as a part on the 1/8 grid and a remainder
__device__ __forceinline__ void split_offset(float A, float& ph, float& pr) {
  constexpr float L = 1.44269502f, Ll = 1.92596299e-8f;  // log2 e = L + Ll
  const float p = mul_rn(A, L);
  const float pe = fmaf(A, L, -p) + A * Ll;
  ph = rintf(p * 8.0f) * 0.125f;
  pr = sub_rn(p, ph) + pe;
}

template <class V>
__device__ __forceinline__ float ld_cluster_f(const V* p, uint32_t rank) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(ra) : "memory");
  return v;
}

// What one thread does with its RO own elements and a tile of the other side's
// records; shared by the sweep kernel below and the batched solver's sweeps.
template <int D, int RO, int NR, bool LSE, int SQM, bool GRAD, int P = 2>
struct Core {
  static constexpr int NA = GRAD ? D : (LSE ? 1 : NR);  // sums per own element
  static constexpr int NW = GRAD || LSE ? 1 : NR;       // weights per other element
  static constexpr int OFF = P * D;                     // a record's offsets, then its weights
  static constexpr int REC = (OFF + 2 + NW + 3) / 4 * 4;
  float xh[RO][D], xl[RO][D], xm[RO][P == 3 ? D : 1], ph[RO], pr[RO];
  float S[RO][NA], Cc[RO][NA], mx[RO], hm[RO];

  __device__ __forceinline__ void own(int r, bool ev, const float* x, int d, const float (&ctr)[D], const Scale& sc,
                                      float A) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      float m = 0.f;
      if (ev && k < d) split_coord<P>(__ldg(x + k), ctr[k], sc, xh[r][k], m, xl[r][k]);
      else xh[r][k] = xl[r][k] = 0.f;
      if constexpr (P == 3) xm[r][k] = m;
    }
    split_offset(ev ? A : 0.f, ph[r], pr[r]);
    mx[r] = kLowest;
    hm[r] = LSE ? ph[r] - kLowest : ph[r];
#pragma unroll
    for (int k = 0; k < NA; ++k) S[r][k] = Cc[r][k] = 0.f;
  }
  // one record: [yh (D), yl (D), ym (P = 3: D), high offset, low offset, weights]
  static __device__ __forceinline__ void stage(float (&rec)[REC], const float* y, int d, const float (&ctr)[D],
                                               const Scale& sc, float B, const float (&w)[NW]) {
    float v[REC];
#pragma unroll
    for (int k = 0; k < REC; ++k) v[k] = 0.f;
#pragma unroll
    for (int k = 0; k < D; ++k)
      if (k < d) {
        float m = 0.f;
        split_coord<P>(__ldg(y + k), ctr[k], sc, v[k], m, v[D + k]);
        if constexpr (P == 3) v[2 * D + k] = m;
      }
    split_offset(B, v[OFF], v[OFF + 1]);
#pragma unroll
    for (int k = 0; k < NW; ++k) v[OFF + 2 + k] = w[k];
#pragma unroll
    for (int k = 0; k < REC; k += 4)
      *reinterpret_cast<float4*>(&rec[k]) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
  }
  static __device__ __forceinline__ void load(const float (&rec)[REC], float (&v)[REC]) {
#pragma unroll
    for (int k = 0; k < REC; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(&rec[k]);
      v[k] = x.x;
      v[k + 1] = x.y;
      v[k + 2] = x.z;
      v[k + 3] = x.w;
    }
  }
  // t2 of own element r and the record v (h: the own side's high offset)
  __device__ __forceinline__ float expo2(int r, float h, const float (&v)[REC]) const {
    float acc = h + v[OFF];
    float lo = pr[r] + v[OFF + 1];
    if constexpr (P == 2) {
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const float dh = xh[r][k] - v[k], dl = xl[r][k] - v[D + k];
        acc = fmaf(-dh, dh, acc);
        lo = fmaf(-dl, fmaf(2.0f, dh, dl), lo);
      }
    } else {
      float mid = 0.f, low = 0.f;  // sum dh dm (exact), sum dh dl
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const float dh = xh[r][k] - v[k], dl = xl[r][k] - v[D + k], dm = xm[r][k] - v[2 * D + k];
        acc = fmaf(-dh, dh, acc);
        mid = fmaf(dh, dm, mid);
        lo = fmaf(-dm, fmaf(2.0f, dl, dm), lo);
        low = fmaf(dh, dl, low);
      }
      acc = fmaf(-2.0f, mid, acc);
      lo = fmaf(-2.0f, low, lo);
    }
    return acc + lo;
  }
  // the records q0 <= q < q1 of a tile
  __device__ __forceinline__ void tile(const float (*rec)[REC], int q0, int q1) {
    for (int qb = q0; qb < q1; qb += kPtsFlush) {
      const int qe = min(q1, qb + kPtsFlush);
      float acc[RO][NA];
#pragma unroll
      for (int r = 0; r < RO; ++r)
#pragma unroll
        for (int k = 0; k < NA; ++k) acc[r][k] = 0.f;
      if constexpr (LSE) {
        constexpr int G = RO == 1 ? 4 : (D <= 4 ? 2 : 1);  // entries per test of the running max
        for (int q = qb; q < qe; q += G) {
          float t[RO][G], w[G], tm[RO];
          bool up = false;
#pragma unroll
          for (int u = 0; u < G; ++u) {
            float v[REC];
            load(rec[min(q + u, qe - 1)], v);
            w[u] = q + u < qe ? v[OFF + 2] : 0.f;
#pragma unroll
            for (int r = 0; r < RO; ++r) t[r][u] = expo2(r, hm[r], v);
          }
#pragma unroll
          for (int r = 0; r < RO; ++r) {
            tm[r] = t[r][0];
#pragma unroll
            for (int u = 1; u < G; ++u) tm[r] = fmaxf(tm[r], t[r][u]);
            up |= tm[r] > kThetaB2;
          }
          for (int k = 0; k < 4 && up; ++k) {  // raise the max, form the group again
            up = false;
#pragma unroll
            for (int r = 0; r < RO; ++r) {
              if (!(tm[r] > kThetaB2)) continue;
              const float dlt = ceilf(tm[r]);
              mx[r] += dlt;
              hm[r] = ph[r] - mx[r];
              const float f = ex2_approx(-dlt);
              acc[r][0] *= f;
              S[r][0] *= f;
              Cc[r][0] *= f;
#pragma unroll
              for (int u = 0; u < G; ++u) {
                float v[REC];
                load(rec[min(q + u, qe - 1)], v);
                t[r][u] = expo2(r, hm[r], v);
                tm[r] = u == 0 ? t[r][0] : fmaxf(tm[r], t[r][u]);
              }
              up |= tm[r] > kThetaB2;
            }
          }
#pragma unroll
          for (int r = 0; r < RO; ++r)
#pragma unroll
            for (int u = 0; u < G; ++u) acc[r][0] = fmaf(ex2_approx(t[r][u]), w[u], acc[r][0]);
        }
      } else {
#pragma unroll 2
        for (int q = qb; q < qe; ++q) {
          float v[REC];
          load(rec[q], v);
#pragma unroll
          for (int r = 0; r < RO; ++r) {
            const float ex = ex2_approx(expo2(r, ph[r], v));
            if constexpr (GRAD) {
              const float pw = ex * v[OFF + 2];
#pragma unroll
              for (int k = 0; k < D; ++k) {
                float low = xl[r][k] - v[D + k];
                if constexpr (P == 3) low += xm[r][k] - v[2 * D + k];
                acc[r][k] = fmaf(pw, (xh[r][k] - v[k]) + low, acc[r][k]);
              }
            } else {
#pragma unroll
              for (int k = 0; k < NR; ++k) {
                if ((SQM >> k) & 1) acc[r][k] = fmaf(ex * ex, v[OFF + 2 + k], acc[r][k]);
                else acc[r][k] = fmaf(ex, v[OFF + 2 + k], acc[r][k]);
              }
            }
          }
        }
      }
#pragma unroll
      for (int r = 0; r < RO; ++r)
#pragma unroll
        for (int k = 0; k < NA; ++k) kadd(S[r][k], Cc[r][k], acc[r][k]);
    }
  }
};

// sigma and the grid of one temperature: kap = gamma s_C log2 e, dmax >= max |x - y|^2,
// parts_of(kap dmax) > 0
__device__ __forceinline__ Scale make_scale(double gamma, double sC, double dmax) {
  const double kap = gamma * sC * kLog2eD;
  Scale s;
  s.sigma = sqrt(kap);
  s.sh = (float)s.sigma;
  s.sl = (float)(s.sigma - (double)s.sh);
  // s = 2^ceil(log2(sqrt(kap dmax)) - 11.5) (twice that at some powers of two), at least 2^-30
  const int ex = max((ilogb(kap * dmax) - 21) >> 1, -30);
  s.magic = 1.5f * __int_as_float((127 + 23 + ex) << 23);
  return s;
}

// Adds the sums of the `ws` warp groups that share own elements (slots w * OWN + o of
// red and rmx, o < OWN) into slot o, in order; all threads, between barriers.
template <int NA, bool LSE, int L>
__device__ __forceinline__ void combine_groups(float2 (*red)[L], float* rmx, int OWN, int ws) {
  for (int o = threadIdx.x; o < OWN; o += kThreads) {
    float M = kLowest;
    if constexpr (LSE) {
      for (int w = 0; w < ws; ++w) M = fmaxf(M, rmx[w * OWN + o]);
    }
#pragma unroll
    for (int k = 0; k < NA; ++k) {
      float s0 = 0.f, c0 = 0.f;
      for (int w = 0; w < ws; ++w) {
        const float2 q = red[k][w * OWN + o];
        const float f = LSE ? ex2_approx(rmx[w * OWN + o] - M) : 1.0f;
        kadd(s0, c0, q.x * f);
        c0 += q.y * f;
      }
      red[k][o] = make_float2(s0, c0);
    }
    if constexpr (LSE) rmx[o] = M;
  }
}

template <int D, int RO, int NR, bool LSE, int SQM, bool ROWS, bool GRAD, int P, class Epi>
__global__ void __launch_bounds__(kThreads, 2) sweep_kernel(SweepArgs<float> a, Args g, Epi epi) {
  using C = Core<D, RO, NR, LSE, SQM, GRAD, P>;
  constexpr int NA = C::NA, NW = C::NW, REC = C::REC;
  constexpr int TO = D <= 4 ? 256 : 128;
  constexpr int ND = Epi::kDot;
  constexpr int kRec = REC * TO * 4, kRed = NA * kThreads * RO * 8;
  __shared__ __align__(16) unsigned char buf[kRec > kRed ? kRec : kRed];
  __shared__ float rmx[LSE ? kThreads * RO : 1];
  __shared__ Scale sc_s;
  __shared__ double beta_s;
  __shared__ int first_s;
  float(*rec)[REC] = reinterpret_cast<float(*)[REC]>(buf);
  float2(*red)[kThreads * RO] = reinterpret_cast<float2(*)[kThreads * RO]>(buf);  // (after the sweep)

  const int64_t n_own = ROWS ? a.n : a.m, n_oth = ROWS ? a.m : a.n;
  const float* xo = ROWS ? a.X : a.Y;
  const float* xt = ROWS ? a.Y : a.X;
  const float* ho = ROWS ? a.Ah : a.Bh;
  const float* ht = ROWS ? a.Bh : a.Ah;
  const int d = a.d;
  const int64_t blk = blockIdx.x;
  const int64_t j0 = (int64_t)blockIdx.y * a.chunk, j1 = min(n_oth, j0 + a.chunk);
  float ctr[D];  // the common centre: the first point of X
#pragma unroll
  for (int k = 0; k < D; ++k) ctr[k] = k < d ? __ldg(a.X + k) : 0.f;
  pdl_wait();
  if (a.active && *a.active == 0.0) return;  // (no CTA changes it before all have read it: the cluster stays whole)
  if (threadIdx.x == 0) sc_s = make_scale(a.gamma_dev ? *a.gamma_dev : (double)a.gamma, a.sC, *g.dmax);
  if constexpr (HasPrepare<Epi>::value) {
    if (threadIdx.x >= 32 && threadIdx.x < 64) epi.prepare(blk == 0 && blockIdx.y == 0, beta_s, first_s);
  }
  __syncthreads();
  const Scale sc = sc_s;
  if constexpr (HasPrepare<Epi>::value) {
    epi.beta = beta_s;
    epi.first = first_s != 0;
  }

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ow = kWarps / g.ws, grp = warp / ow;  // warps across own elements; this warp's share of the others
  const int OWN = ow * 32 * RO, ol = (warp - grp * ow) * 32 + lane;
  C c;
#pragma unroll
  for (int r = 0; r < RO; ++r) {
    const int64_t e = blk * OWN + r * (ow * 32) + ol;
    const bool ev = e < n_own;
    c.own(r, ev, xo + e * d, d, ctr, sc, ev ? ho[e] : 0.f);
  }
  for (int64_t jt = j0; jt < j1; jt += TO) {
    const int tn = (int)min((int64_t)TO, j1 - jt);
    __syncthreads();
    for (int q = threadIdx.x; q < tn; q += kThreads) {
      const int64_t j = jt + q;
      float w[NW];
#pragma unroll
      for (int k = 0; k < NW; ++k) w[k] = ROWS ? a.wc[k][j] : a.wr[k][j];
      C::stage(rec[q], xt + j * d, d, ctr, sc, ht[j], w);
    }
    __syncthreads();
    const int seg = (tn + g.ws - 1) / g.ws;
    c.tile(rec, grp * seg, min(tn, (grp + 1) * seg));
  }
  pdl_trigger();

  // ---- the CTA's warp groups, then the cluster's CTAs, in order ----
  __syncthreads();  // (the records are done with)
#pragma unroll
  for (int r = 0; r < RO; ++r) {
    const int at = grp * OWN + r * (ow * 32) + ol;
#pragma unroll
    for (int k = 0; k < NA; ++k) red[k][at] = make_float2(c.S[r][k], c.Cc[r][k]);
    if constexpr (LSE) rmx[at] = c.mx[r];
  }
  __syncthreads();
  if (g.ws > 1) combine_groups<NA, LSE>(red, rmx, OWN, g.ws);
  cluster_sync();  // every CTA's sums are visible to the cluster
  const uint32_t rank = cluster_rank(), ranks = gridDim.y;
  const int per = (OWN + (int)ranks - 1) / (int)ranks;
  const int o0 = (int)rank * per, o1 = min(OWN, o0 + per);
  double wd[ND > 0 ? ND : 1];
#pragma unroll
  for (int k = 0; k < (ND > 0 ? ND : 1); ++k) wd[k] = 0.0;
  for (int o = o0 + threadIdx.x; o < o1; o += kThreads) {
    const int64_t e = blk * OWN + o;
    if (e >= n_own) continue;
    float M = kLowest;
    if constexpr (LSE) {
      for (uint32_t q = 0; q < ranks; ++q) M = fmaxf(M, ld_cluster_f(&rmx[o], q));
    }
    double tot[NA];
#pragma unroll
    for (int k = 0; k < NA; ++k) {
      float s0 = 0.f, c0 = 0.f;
      for (uint32_t q = 0; q < ranks; ++q) {
        const float2 x = ld_cluster_f2(&red[k][o], q);
        const float f = LSE ? ex2_approx(ld_cluster_f(&rmx[o], q) - M) : 1.0f;
        kadd(s0, c0, x.x * f);
        c0 += x.y * f;
      }
      tot[k] = (double)s0 + (double)c0;
    }
    DotArr<ND> dd;
    if constexpr (GRAD) epi.template grad<D>(e, tot, 1.0 / sc.sigma);
    else if constexpr (LSE && ROWS) epi.row_lse(e, (double)M * kLn2D, tot[0], dd.v);
    else if constexpr (LSE) epi.col_lse(e, (double)M * kLn2D, tot[0], dd.v);
    else if constexpr (ROWS) epi.row(e, tot, dd.v);
    else epi.col(e, tot, dd.v);
#pragma unroll
    for (int k = 0; k < ND; ++k) wd[k] += dd.v[k];
  }
  if constexpr (ND > 0) {
#pragma unroll
    for (int k = 0; k < ND; ++k) wd[k] = warp_sum(wd[k]);
    cta_dot_finish<ND>(wd, blk * ranks + rank, (int64_t)gridDim.x * ranks, a.dotpart, a.cnt_dot, epi);
  }
  cluster_sync();  // no CTA leaves while another reads its shared memory
}

// Gradients of higher-dimensional clouds (16 < d <= 64) from the same split
// coordinates: out_e,k = scale ownfac_e sum_o P_eo (x_e - x_o)_k for every k in one
// pass (the general kernel, sweep_pts.cuh, keeps sixteen sums per thread and forms
// every distance again for each sixteen coordinates, eighteen instructions each).
// FP32-pipe bound: 5 d instructions per entry for the exponent and 2 d for the
// products. A CTA owns kGR elements and walks the other side in tiles of kGC: (1) a
// 4 x 8 block of exponents per thread from coordinate-major tiles (packed FP32 pairs,
// six 16-byte shared loads per 160 packed operations), the weighted plan entries to
// shared memory; (2) a 4 x 4 block (elements x coordinates) per thread over those
// entries. Two CTAs per SM; a cluster of up to 8 CTAs splits the other side.
// A training step of
// n = m = 16384, d = 64: 339 -> 236 ms.
// Three parts (P = 3): 8 d for the exponent, chunks half as long, one CTA per SM.
constexpr int kGR = 64, kGC = 128, kGD = 64;
template <int P>
struct GradSmem {
  static constexpr int kGK = P == 3 ? 16 : 32;
  float xs[P][kGD][kGR];  // the own side's xh, xl (, xm), coordinate-major; at the end the sums as pairs
  union {
    float ys[P][kGK][kGC + 4];  // a chunk of the tile's yh, yl (, ym)
    float p[kGC][kGR + 4];      // weighted plan entries of the tile
  };
  float yr[kGC][kGD];           // the tile's coordinates (zeros beyond d)
  float qh[kGC], qr[kGC], w[kGC];
  Scale sc;
};

template <bool ROWS, int P>
__global__ void __launch_bounds__(kThreads, P == 3 ? 1 : 2) grad_tile_kernel(SweepArgs<float> a, Args g, double scale,
                                                                             const double* ownfac, float* out) {
  constexpr int kGK = GradSmem<P>::kGK;
  extern __shared__ __align__(16) unsigned char raw[];
  GradSmem<P>& s = *reinterpret_cast<GradSmem<P>*>(raw);
  const int64_t n_own = ROWS ? a.n : a.m, n_oth = ROWS ? a.m : a.n;
  const float* xo = ROWS ? a.X : a.Y;
  const float* xt = ROWS ? a.Y : a.X;
  const float* ho = ROWS ? a.Ah : a.Bh;
  const float* ht = ROWS ? a.Bh : a.Ah;
  const float* wt = ROWS ? a.wc[0] : a.wr[0];
  const int d = a.d, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t e0 = (int64_t)blockIdx.x * kGR;
  const int64_t j0 = min(n_oth, (int64_t)blockIdx.y * a.chunk), j1 = min(n_oth, j0 + a.chunk);
  pdl_wait();
  if (tid == 0) s.sc = make_scale(a.gamma_dev ? *a.gamma_dev : (double)a.gamma, a.sC, *g.dmax);
  for (int q = tid; q < kGC * kGD; q += kThreads) s.yr[q / kGD][q % kGD] = 0.f;
  __syncthreads();
  const Scale sc = s.sc;
  for (int q = tid; q < kGR * kGD; q += kThreads) {
    const int r = q / kGD, k = q % kGD;
    float xh = 0.f, xm = 0.f, xl = 0.f;
    if (e0 + r < n_own && k < d) split_coord<P>(__ldg(xo + (e0 + r) * d + k), __ldg(a.X + k), sc, xh, xm, xl);
    s.xs[0][k][r] = xh;
    s.xs[1][k][r] = xl;
    if constexpr (P == 3) s.xs[2][k][r] = xm;
  }
  const int rg = tid >> 4, cg = tid & 15;  // elements 4 rg .. + 3; columns 4 cg .. + 3 and 64 + 4 cg .. + 3
  float ph[4], pr[4];
  unsigned long long x2[4][2];  // phase 2: coordinates 4 cg .. 4 cg + 3 of the own elements
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int64_t e = e0 + 4 * rg + r;
    const bool ev = e < n_own;
    split_offset(ev ? ho[e] : 0.f, ph[r], pr[r]);
    float x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = ev && 4 * cg + k < d ? __ldg(xo + e * d + 4 * cg + k) : 0.f;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x2[r][0]) : "f"(x[0]), "f"(x[1]));
    asm("mov.b64 %0, {%1, %2};" : "=l"(x2[r][1]) : "f"(x[2]), "f"(x[3]));
  }
  float S[4][4], Cc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int k = 0; k < 4; ++k) S[r][k] = Cc[r][k] = 0.f;
  unsigned long long two2;
  asm("mov.b64 %0, {%1, %1};" : "=l"(two2) : "f"(2.0f));

  for (int64_t jt = j0; jt < j1; jt += kGC) {
    const int tn = (int)min((int64_t)kGC, j1 - jt);
    // pairs of columns: sum dh^2, sum dl (2 dh + dl); P = 3: the latter is sum dm (dm + 2 dl),
    // and sum dh dm, sum dh dl
    unsigned long long q2[4][4], l2[4][4], mid2[4][P == 3 ? 4 : 1], low2[4][P == 3 ? 4 : 1];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        q2[r][e] = l2[r][e] = 0ull;
        if constexpr (P == 3) mid2[r][e] = low2[r][e] = 0ull;
      }
    for (int k0 = 0; k0 < d; k0 += kGK) {
      const int kn = min(kGK, d - k0);
      __syncthreads();  // the previous chunk (or the previous tile's entries) is done with
      if (k0 == 0) {
        for (int q = tid; q < tn * d; q += kThreads) {
          const int jj = q / d, k = q - jj * d;
          s.yr[jj][k] = __ldg(xt + jt * d + q);
        }
        if (tid < kGC) {
          const bool jv = tid < tn;
          split_offset(jv ? ht[jt + tid] : 0.f, s.qh[tid], s.qr[tid]);
          s.w[tid] = jv ? wt[jt + tid] : 0.f;
        }
      }
      if (lane < kn) {
        const float c = __ldg(a.X + k0 + lane);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float h[4], l[4], md[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int jj = 4 * (warp + 8 * q) + e;
            h[e] = l[e] = md[e] = 0.f;
            if (jj < tn) split_coord<P>(__ldg(xt + (jt + jj) * d + k0 + lane), c, sc, h[e], md[e], l[e]);
          }
          *reinterpret_cast<float4*>(&s.ys[0][lane][4 * (warp + 8 * q)]) = make_float4(h[0], h[1], h[2], h[3]);
          *reinterpret_cast<float4*>(&s.ys[1][lane][4 * (warp + 8 * q)]) = make_float4(l[0], l[1], l[2], l[3]);
          if constexpr (P == 3)
            *reinterpret_cast<float4*>(&s.ys[2][lane][4 * (warp + 8 * q)]) = make_float4(md[0], md[1], md[2], md[3]);
        }
      }
      __syncthreads();
#pragma unroll 2
      for (int k = 0; k < kn; ++k) {
        const float4 xh4 = *reinterpret_cast<const float4*>(&s.xs[0][k0 + k][4 * rg]);
        const float4 xl4 = *reinterpret_cast<const float4*>(&s.xs[1][k0 + k][4 * rg]);
        const ulonglong2 ha = *reinterpret_cast<const ulonglong2*>(&s.ys[0][k][4 * cg]);
        const ulonglong2 hb = *reinterpret_cast<const ulonglong2*>(&s.ys[0][k][64 + 4 * cg]);
        const ulonglong2 la = *reinterpret_cast<const ulonglong2*>(&s.ys[1][k][4 * cg]);
        const ulonglong2 lb = *reinterpret_cast<const ulonglong2*>(&s.ys[1][k][64 + 4 * cg]);
        const float xh[4] = {xh4.x, xh4.y, xh4.z, xh4.w}, xl[4] = {xl4.x, xl4.y, xl4.z, xl4.w};
        const unsigned long long yh[4] = {ha.x, ha.y, hb.x, hb.y}, yl[4] = {la.x, la.y, lb.x, lb.y};
        float xm[4];
        unsigned long long ym[4];
        if constexpr (P == 3) {
          const float4 xm4 = *reinterpret_cast<const float4*>(&s.xs[2][k0 + k][4 * rg]);
          const ulonglong2 ma = *reinterpret_cast<const ulonglong2*>(&s.ys[2][k][4 * cg]);
          const ulonglong2 mb = *reinterpret_cast<const ulonglong2*>(&s.ys[2][k][64 + 4 * cg]);
          xm[0] = xm4.x, xm[1] = xm4.y, xm[2] = xm4.z, xm[3] = xm4.w;
          ym[0] = ma.x, ym[1] = ma.y, ym[2] = mb.x, ym[3] = mb.y;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          unsigned long long nh, nl;
          asm("mov.b64 %0, {%1, %1};" : "=l"(nh) : "f"(-xh[r]));
          asm("mov.b64 %0, {%1, %1};" : "=l"(nl) : "f"(-xl[r]));
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            unsigned long long dh, dl, t;
            asm("add.rn.f32x2 %0, %1, %2;" : "=l"(dh) : "l"(yh[e]), "l"(nh));
            asm("add.rn.f32x2 %0, %1, %2;" : "=l"(dl) : "l"(yl[e]), "l"(nl));
            asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(q2[r][e]) : "l"(dh));
            if constexpr (P == 3) {
              unsigned long long nm, dm;
              asm("mov.b64 %0, {%1, %1};" : "=l"(nm) : "f"(-xm[r]));
              asm("add.rn.f32x2 %0, %1, %2;" : "=l"(dm) : "l"(ym[e]), "l"(nm));
              asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(mid2[r][e]) : "l"(dh), "l"(dm));
              asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(t) : "l"(two2), "l"(dl), "l"(dm));
              asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(l2[r][e]) : "l"(dm), "l"(t));
              asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(low2[r][e]) : "l"(dh), "l"(dl));
            } else {
              asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(t) : "l"(two2), "l"(dh), "l"(dl));
              asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(l2[r][e]) : "l"(dl), "l"(t));
            }
          }
        }
      }
    }
    __syncthreads();  // the last chunk of ys is done with: the entries take its place
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int col = (e < 2 ? 0 : 60) + 4 * cg + 2 * e;  // columns col, col + 1
      float pa[4], pb[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float qa, qb, la, lb;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(qa), "=f"(qb) : "l"(q2[r][e]));
        asm("mov.b64 {%0, %1}, %2;" : "=f"(la), "=f"(lb) : "l"(l2[r][e]));
        float ta = (ph[r] + s.qh[col]) - qa, tb = (ph[r] + s.qh[col + 1]) - qb;
        float ua = (pr[r] + s.qr[col]) - la, ub = (pr[r] + s.qr[col + 1]) - lb;
        if constexpr (P == 3) {
          float ma, mb, wa, wb;
          asm("mov.b64 {%0, %1}, %2;" : "=f"(ma), "=f"(mb) : "l"(mid2[r][e]));
          asm("mov.b64 {%0, %1}, %2;" : "=f"(wa), "=f"(wb) : "l"(low2[r][e]));
          ta = fmaf(-2.0f, ma, ta);
          tb = fmaf(-2.0f, mb, tb);
          ua = fmaf(-2.0f, wa, ua);
          ub = fmaf(-2.0f, wb, ub);
        }
        ta += ua;
        tb += ub;
        pa[r] = ex2_approx(ta) * s.w[col];
        pb[r] = ex2_approx(tb) * s.w[col + 1];
      }
      *reinterpret_cast<float4*>(&s.p[col][4 * rg]) = make_float4(pa[0], pa[1], pa[2], pa[3]);
      *reinterpret_cast<float4*>(&s.p[col + 1][4 * rg]) = make_float4(pb[0], pb[1], pb[2], pb[3]);
    }
    __syncthreads();
    // elements 4 rg .. + 3, coordinates 4 cg .. + 3
    for (int b = 0; b < tn; b += kPtsFlush) {
      const int be = min(tn, b + kPtsFlush);
      unsigned long long acc[4][2];
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = 0ull;
#pragma unroll 4
      for (int j = b; j < be; ++j) {
        const float4 p4 = *reinterpret_cast<const float4*>(&s.p[j][4 * rg]);
        const float4 y4 = *reinterpret_cast<const float4*>(&s.yr[j][4 * cg]);
        const float p[4] = {p4.x, p4.y, p4.z, p4.w};
        unsigned long long ny[2];
        asm("mov.b64 %0, {%1, %2};" : "=l"(ny[0]) : "f"(-y4.x), "f"(-y4.y));
        asm("mov.b64 %0, {%1, %2};" : "=l"(ny[1]) : "f"(-y4.z), "f"(-y4.w));
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          unsigned long long pp, df;
          asm("mov.b64 %0, {%1, %1};" : "=l"(pp) : "f"(p[r]));
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            asm("add.rn.f32x2 %0, %1, %2;" : "=l"(df) : "l"(x2[r][k]), "l"(ny[k]));
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[r][k]) : "l"(pp), "l"(df));
          }
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          float u, v;
          asm("mov.b64 {%0, %1}, %2;" : "=f"(u), "=f"(v) : "l"(acc[r][k]));
          kadd(S[r][2 * k], Cc[r][2 * k], u);
          kadd(S[r][2 * k + 1], Cc[r][2 * k + 1], v);
        }
    }
  }
  pdl_trigger();
  __syncthreads();
  float2(*red)[kGD] = reinterpret_cast<float2(*)[kGD]>(&s.xs[0][0][0]);  // [kGR][kGD]
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int k = 0; k < 4; ++k) red[4 * rg + r][4 * cg + k] = make_float2(S[r][k], Cc[r][k]);
  cluster_sync();  // every CTA's sums are visible to the cluster
  const uint32_t rank = cluster_rank(), ranks = gridDim.y;
  const int per = (kGR + (int)ranks - 1) / (int)ranks;
  const int r0 = (int)rank * per, r1 = min(kGR, r0 + per);
  for (int q = r0 * kGD + tid; q < r1 * kGD; q += kThreads) {
    const int r = q / kGD, k = q % kGD;
    const int64_t e = e0 + r;
    if (e >= n_own || k >= d) continue;
    float s0 = 0.f, c0 = 0.f;
    for (uint32_t c = 0; c < ranks; ++c) {  // in rank order
      const float2 x = ld_cluster_f2(&red[r][k], c);
      kadd(s0, c0, x.x);
      c0 += x.y;
    }
    out[e * d + k] = (float)(scale * ownfac[e] * ((double)s0 + (double)c0));
  }
  cluster_sync();  // no CTA leaves while another reads its shared memory
}

// Chunks of the other side: the fewest waves x (tiles per CTA + 1); per_sm CTAs per SM.
inline Geo grad_geo(int sms, int64_t n_own, int64_t n_oth, int per_sm) {
  Geo best{};
  int64_t bc = -1;
  const int64_t B = (n_own + kGR - 1) / kGR, tiles = (n_oth + kGC - 1) / kGC, slots = (int64_t)per_sm * sms;
  for (int64_t k = 1; k <= 8 && k <= tiles; ++k) {
    const int64_t tk = (tiles + k - 1) / k, S = (tiles + tk - 1) / tk;
    const int64_t c = (B * S + slots - 1) / slots * (tk + 1);
    if (bc >= 0 && c >= bc) continue;
    bc = c;
    best = Geo{B, S, tk * kGC, 0, 0};
  }
  return best;
}

// Two bounds on max |x_i - y_j|^2 for a caller's s_C. ext[0], ext[1]: max |x - x_0|^2 and
// max |y - x_0|^2 (FP32, rounded up by a part in 10^5), since |x_i - y_j| <= |x_i - x_0| +
// |y_j - x_0|; up to kBoxD dimensions, where it is the tighter one, ext[2 + k] and
// ext[2 + kBoxD + k]: the largest x_k and -x_k of either cloud, the box whose squared
// diagonal bounds it too. All of them as ordered integers, zeroed before; a NaN makes them
// infinite. The grid's threads are a multiple of d in the second loop, so that each stays
// with one coordinate.
__host__ __device__ inline uint32_t ordered_bits(uint32_t b) { return b >> 31 ? ~b : b | 0x80000000u; }
__host__ __device__ inline uint32_t unordered_bits(uint32_t b) { return b >> 31 ? b & 0x7fffffffu : ~b; }
constexpr int kBoxD = 8, kExtents = 2 + 2 * kBoxD;
static __global__ void __launch_bounds__(kThreads) extent_kernel(const float* X, const float* Y, int64_t n, int64_t m,
                                                                 int d, uint32_t* ext) {
  __shared__ uint32_t box[kExtents];
  for (int q = threadIdx.x; q < kExtents; q += kThreads) box[q] = 0u;
  __syncthreads();
  pdl_wait();
  auto up = [](float x) { return ordered_bits(__float_as_uint(x == x ? x : INFINITY)); };
  const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x, T = (int64_t)gridDim.x * kThreads;
  float r[2] = {0.f, 0.f};
  for (int64_t q = t; q < n + m; q += T) {
    const float* p = q < n ? X + q * d : Y + (q - n) * d;
    float s = 0.f;
#pragma unroll 8
    for (int k = 0; k < d; ++k) {
      const float e = __ldg(p + k) - __ldg(X + k);
      s = fmaf(e, e, s);
    }
    s = s == s ? s * 1.00001f : INFINITY;
    r[q < n ? 0 : 1] = fmaxf(r[q < n ? 0 : 1], s);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const float w = warp_max_f(r[c]);
    if ((threadIdx.x & 31) == 0) atomicMax(&box[c], up(w));
  }
  const int64_t Td = T / d * d;
  if (d <= kBoxD && t < Td) {
    float hi = -INFINITY, lo = -INFINITY;
    for (int64_t q = t; q < (n + m) * d; q += Td) {
      const float x = __ldg(q < n * d ? X + q : Y + (q - n * d));
      hi = fmaxf(hi, x == x ? x : INFINITY);
      lo = fmaxf(lo, x == x ? -x : INFINITY);
    }
    const int k = (int)(t % d);
    atomicMax(&box[2 + k], up(hi));
    atomicMax(&box[2 + kBoxD + k], up(lo));
  }
  __syncthreads();
  for (int q = threadIdx.x; q < kExtents; q += kThreads)
    if (box[q]) atomicMax(ext + q, box[q]);
}

}  // namespace pg
}  // namespace eot
