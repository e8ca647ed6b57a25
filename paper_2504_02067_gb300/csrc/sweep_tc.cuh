// Point-cloud sweeps whose cross term x_i . y_j runs on the tensor cores
// (tcgen05, kind::f16 on FP16, FP32 accumulation in TMEM), for the mixed path at
// larger d (up to 64 coordinates).
//
// Exactness (an exact-slice / Ozaki-style splitting). Both point sets are moved
// by one common centre c (the first point of X; exact in FP64, distances do not
// change). Each cloud gets one exponent E (every centred coordinate |x_k| < 2^E)
// and every coordinate is rounded to 2^(E-b) and cut into four balanced digits of
// radix 1024,
//     x_k = 2^(E-b+30) sum_s d_sk 2^-10s,   |d_0| <= 2^(b-30), -512 <= d_s < 512,
// integers that FP16 holds exactly. The 10 slice pairs (s, t) with s + t <= 3 are
// added into four "level" accumulators S_L = sum_{s+t=L} D_s D_t^T, and
//     x . y = 2^(Ex + Ey - 2b + 60) G,   G = S_0 + 2^-10 S_1 + 2^-20 S_2 + 2^-30 S_3.
// b = 38 keeps S_0 and S_1 exact in the FP32 accumulator whatever the data (over 64
// coordinates |S_0| <= 2^22, |S_1| <= 2^24). S_1 is at most 512 times the sum of two
// points' |d_0|, so b is 39 or 40 where the largest points' sums of |x_k| allow it
// (tc_scale; |S_0| stays within 2^24 then), which they do unless points lie near the
// corners of the clouds' cube: each bit makes what is dropped four times smaller. S_2
// and S_3 are exact while below 2^24 (one unit off, 2^-20 and less of a level-0 unit,
// beyond). What is dropped, the pairs s + t >= 4, is 2^-23.6 sqrt(3 d) (rms) of a
// level-0 unit 2^(Ex + Ey - 2b + 60), in scaled coordinates (below) of an exponent
// unit. Where that exceeds 2^-27 the three pairs s + t = 4 are issued too: into level
// 3's accumulator, whose first MMA scales it by 2^-10 (scale-input-d). The rest is
// the coordinates' rounding. Row sums off (L1 over the mass; emulated, 300 Sinkhorn-
// balanced points, uniform d = 17 / eight Gaussians d = 64), FP32 rounding included:
//     gamma    five 8-bit digits,   these             (b = 37, ten pairs always)
//              fifteen pairs
//     2^10     4.4e-9 / 6.8e-9      3.8e-9 / 5.5e-9   1.8e-8 / 3.0e-8
//     2^12     6.6e-9 / 1.6e-8      3.5e-9 / 4.9e-9   7.1e-8 / 1.3e-7
//     2^14     2.3e-8 / 5.9e-8      4.0e-9 / 4.6e-9   2.9e-7 / 5.3e-7
//     2^18     3.7e-7 / 9.7e-7      5.6e-8 / 5.7e-8   4.7e-6 / 8.7e-6
// A CG column sweep of n = m = 16384, d = 64: 0.263 ms with ten pairs, 0.34 with thirteen
// (0.36 with fifteen pairs of BF16 digits). Coordinates beyond d are zero: only ceil(d / 16) of the four K = 16 steps
// of a pair are issued.
//
// Exponent algebra. In base-2 units (t2 = t log2 e) the exponent of the plan is
//     t2_ij = P_i + Q_j + x'_i . y'_j,   P_i = (A_i - K |x_i|^2) log2 e,
//     Q_j = (B_j - K |y_j|^2) log2 e,   x' = sqrt(2 K log2 e) (x - c) in FP64,
// with K = gamma s_C and A, B the high parts of the potentials. The digits are those
// of the scaled coordinates, made anew whenever gamma changes (tc_prep_kernel: 8 MB of
// digits per 16384 points, once per stage), so that x' . y' = 2^a G with a power of
// two. A small kernel before each sweep (tc_sweep_prep_kernel) forms P and Q in FP64
// and splits each into a high part on the 1/8 grid and a low part below 1/16: the
// other side's low part is folded into its weights (w_j 2^ql_j, one record per point:
// {Qh, w0} in 8 bytes for one weight, {Qh, w0, w1, w2} in 16) and the own side's into
// one FP64 factor 2^pl_i that the finishing CTA applies to the row's total. Per entry
// the epilogue then needs
//     t2 = (Ph + Qh) + 2^a S_0 + 2^(a-10) S_1 + 2^(a-20) S_2 + 2^(a-30) S_3,
// an addition and four FMAs in this order: Ph + Qh is exact on the grid, every product
// is exact (a power of two), the first sums cancel exactly, and what is rounded is
// rounded at the size of t2. (Scaling by an FP32 pair kappa after folding the levels
// into an FP32 pair takes ten instructions: a CG sweep of n = m = 16384, d = 64 took
// 0.299 ms, this way 0.262 ms; the digits with a whole training step 230 -> 215 ms.)
//
// Tile width and operands. With both operands in shared memory a tcgen05.mma of
// M = 128, K = 16 costs about 55 cycles whatever its N up to 96 (measured on GB300:
// 55 cycles at N = 32, 48 and 96; 96 at N = 192, the tensor unit's own rate): the A
// operand's 4 KB, read again by every MMA, bound it, and the epilogue's record reads
// and the tile copies compete for the same bandwidth. The tile is 96 points wide: the
// four level accumulators take 384 of the 512 TMEM columns, handed over level pair by
// level pair, and the own points' four digit slices (128 lanes x 32 columns each)
// fill the other 128, so the MMAs read A from TMEM and only B from shared memory.
// (By itself that changed nothing while the epilogue was the longer side: a CG sweep of
// n = m = 16384, d = 64 took 0.301 ms with A in shared memory and 0.299 ms so.)
//
// CTA roles (480 threads, one CTA per SM: about 155 KB of shared memory):
//   warp 0, lane 0 and warp 14, lane 0: the (up to) 40 MMAs of each tile, twenty
//     each (levels 0, 3 and levels 1, 2), with a commit per level. A
//     tcgen05.mma blocks its thread while the tensor unit's short queue is
//     full, so these threads do nothing else: any other work in them, or a
//     lost issue slot, leaves the tensor unit idle;
//   warp 1: TMEM allocation (512 columns) and release; lane 0 issues the bulk
//     copies (the other side's 96-point tiles into three slice buffers and their
//     records into five record slots);
//   warps 2-13: epilogue. Warp w reads TMEM lanes 32 (w mod 4) .. +31 (one own
//     point per thread) and a third (32) of the tile's 96 columns; before the
//     first tile they store the own points' slices to TMEM.
// Hand-offs are mbarriers: full[sb] (the slices of buffer sb landed), sfree[sb][i]
// (issuer i's MMAs reading buffer sb are done), rec[s] (records landed), lvl[g] (the
// MMAs of levels {0,1}, {2,3} are done, one arrival per issuer: accumulators readable),
// lfree[g] (the 12 epilogue warps have loaded those levels into registers; the next
// tile's MMAs may overwrite them). Every wait is bounded (tc.cuh).
#pragma once
#include <cuda_fp16.h>

#include "sweep_pts.cuh"
#include "tc.cuh"

namespace eot {
namespace tc {

constexpr int kM = 128;     // own points per CTA = TMEM lanes = MMA M
constexpr int kN = 96;      // other-side points per tile = MMA N
constexpr int kSlices = 4;  // radix-1024 digits per coordinate
constexpr int kLevels = 4;  // s + t = 0 .. 3
constexpr int kMinBits = 38, kMaxBits = 40;  // |x_k| 2^-E in units of 2^-b
constexpr int kEpiWarps = 12;                  // 3 per TMEM lane quarter
constexpr int kParts = kEpiWarps / 4;          // column parts of a tile
constexpr int kPartCols = kN / kParts;         // 32 columns per epilogue warp and tile
constexpr int kGroups = kPartCols / 8;         // groups of 8 columns in the arithmetic
constexpr int kMmaWarpB = 2 + kEpiWarps;      // the second MMA-issuing warp (after the epilogue warps)
constexpr int kTcThreads = 32 * (3 + kEpiWarps);
constexpr int kTcWarps = kTcThreads / 32;
constexpr uint32_t kRowB = 128;    // bytes per point and slice: 64 FP16 digits
constexpr uint32_t kOthSlice = kN * kRowB;                          // 12 KB
constexpr uint32_t kOffOth = 0;
constexpr int kSliceBufs = 3;                                       // tile tt: slice buffer tt % 3
constexpr int kRecSlots = kSliceBufs + 2;                           // tile tt: record slot tt % 5
constexpr uint32_t kRecBytes = kN * 16;                             // 1.5 KB: a slot at the widest record
constexpr uint32_t kOffRec = kOffOth + kSliceBufs * kSlices * kOthSlice;  // 144 KB
constexpr uint32_t kOffBar = kOffRec + kRecSlots * kRecBytes;            // + 7.5 KB
constexpr uint32_t kSmemBytes = kOffBar + 256 + 1024;               // barriers, TMEM slot; 1024-byte alignment slack
constexpr uint32_t kTmemCols = 512;                                 // 4 levels x 96, then the own slices
constexpr uint32_t kOwnCol = kLevels * kN;                          // 4 slices x 32 columns
constexpr int64_t kPadRows = 384;                                   // lcm(kM, kN)
constexpr uint32_t kIdesc = idesc_f16_f32(kM, kN);
static_assert(kLevels * kN + kSlices * 32 <= (int)kTmemCols, "level accumulators and own slices exceed TMEM");
constexpr int kMinD = 17;  // the tensor-core path serves d >= kMinD
constexpr double kLog2eD = 1.4426950408889634;
constexpr double kLn2D = 0.6931471805599453;
constexpr float kTheta2 = 12.0f;       // lazy-rescale threshold of the online max (base 2)
constexpr float kPadQ = -8388608.0f;   // -2^23: Qh of padded points (weights 0), and the LSE max's start
constexpr double kQLimit = 1048576.0;  // |P|, |Q| < 2^20: sums of grid values stay exact in FP32

// Per-sweep data of an own point (written by tc_sweep_prep_kernel).
struct OwnRec {
  float ph;   // high part of P on the 1/8 grid
  float pad;
  double pl;  // P - ph, |pl| <= 1/16
  double f1;  // 2^pl
  double f2;  // 2^(2 pl): sums of squared entries
};

// Per point set: the fixed digit slices and |x - c|^2 (per problem), and the
// per-sweep records of the point set in either role.
struct Side {
  const __half* slices;  // [kSlices][npad][64], 128-byte swizzle per 8-row atom
  const double* nx;             // [npad] |x - c|^2 (0 for padding)
  float* rec;                   // [npad][rec_floats(NR)] as the other side: {Qh, w0 2^ql[, w1 2^ql, w2 2^ql]}
  OwnRec* own;                  // [npad] as the own side
  int64_t npad;
};
struct TcArgs {
  Side X, Y;
  const unsigned long long* emax;  // [4] bits of the FP64 max |x_k - c_k| and max sum_k |x_k - c_k| of X, then of Y
  float* kappa;                    // [2] 2^a, 1 where the pairs s + t = 4 are needed (per sweep)
  int* err;                        // status word: kStatTimeout on a wait that ran out, kStatRange
};

__host__ __device__ inline int64_t pad_rows(int64_t n) { return (n + kPadRows - 1) / kPadRows * kPadRows; }
// Floats per record: sweeps with one weight (the CG halves, the LSE sweeps)
// read 8 bytes per column, so one 16-byte shared load serves two columns.
__host__ __device__ constexpr int rec_floats(int nr) { return nr == 1 ? 2 : 4; }

// sqrt(2 K log2 e), K = gamma s_C, and E with every scaled centred coordinate
// |x'_k| < 2^E (0 for a cloud of one point; rounding is monotone, so the largest
// coordinate's scaled value bounds every other).
__device__ __forceinline__ double tc_sigma(double gamma, double sC) { return sqrt(2.0 * gamma * sC * kLog2eD); }
__device__ __forceinline__ int cloud_exp(unsigned long long bits, double sigma) {
  const double mx = __longlong_as_double((long long)bits) * sigma;
  int e = 0;
  if (mx > 0.0) frexp(mx, &e);  // mx = f 2^e, f in [0.5, 1)
  return e;
}

// The digits of one temperature: sigma, the clouds' exponents and the bits b.
struct TcScale {
  double sigma;
  int ex, ey, bits;
  __device__ __forceinline__ int a() const { return ex + ey - 2 * (bits - 30); }  // x' . y' = 2^a G
};
__device__ __forceinline__ TcScale tc_scale(const TcArgs& ta, double gamma, double sC) {
  TcScale s;
  s.sigma = tc_sigma(gamma, sC);
  s.ex = cloud_exp(ta.emax[0], s.sigma);
  s.ey = cloud_exp(ta.emax[2], s.sigma);
  // the largest points' sums of |x'_k| 2^-E: with b bits sum |d_0| <= 2^(b-30) that + 33
  const double sum = s.sigma * (ldexp(__longlong_as_double((long long)ta.emax[1]), -s.ex) +
                                ldexp(__longlong_as_double((long long)ta.emax[3]), -s.ey));
  s.bits = kMaxBits;
  while (s.bits > kMinBits && !(ldexp(sum, s.bits - 30) + 66.0 <= 32768.0)) --s.bits;
  return s;
}

// max_{i,k} |x_ik - c_k| (FP64, exact differences) and a bound on max_i sum_k |x_ik - c_k|
// (FP32, rounded up) of one cloud, one warp per point, into emax[0] and emax[1] as the bits
// of non-negative doubles (ordered like the values: compared as integers, off the FP64
// pipe), which start at 0.
static __global__ void tc_extent_kernel(const float* X, int64_t n, int d, const float* centre,
                                        unsigned long long* emax) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const float c0 = lane < d ? centre[lane] : 0.f, c1 = lane + 32 < d ? centre[lane + 32] : 0.f;
  const double w0 = widen(c0), w1 = widen(c1);
  unsigned long long mx = 0ull;
  float ms = 0.f;
  auto far = [&](float x, double w) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(widen(x) - w) & 0x7fffffffffffffffull;
    mx = mx > b ? mx : b;
  };
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < n;
       i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const float a = lane < d ? X[i * d + lane] : c0, b = lane + 32 < d ? X[i * d + lane + 32] : c1;
    far(a, w0);
    far(b, w1);
    float s = fabsf(a - c0) + fabsf(b - c1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    ms = fmaxf(ms, s == s ? s : INFINITY);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = mx > b ? mx : b;
  }
  if (lane == 0 && mx > 0ull) {
    atomicMax(emax, mx);
    atomicMax(emax + 1, (unsigned long long)__double_as_longlong((double)ms * 1.00001));
  }
}

// One warp per point of either cloud (rows >= n and coordinates >= d are zero): the
// four digit slices of the scaled coordinates in the swizzled K-major layout and
// |x - c|^2 in FP64. Centring keeps |x|^2, |y|^2 and x.y bounded by the data's extent,
// so the expansion |x|^2 + |y|^2 - 2 x.y keeps its accuracy however far the clouds lie
// from the origin. gamma_dev (nullable): gamma is read on the device.
static __global__ void tc_prep_kernel(SweepArgs<float> a, TcArgs ta) {
  __shared__ TcScale scale;  // (its FP64 operations once per CTA)
  pdl_wait();
  if (threadIdx.x == 0) scale = tc_scale(ta, (double)(a.gamma_dev ? (float)*a.gamma_dev : a.gamma), a.sC);
  __syncthreads();
  const int64_t grow = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, d = a.d;
  const bool isx = grow < ta.X.npad;
  const Side& sd = isx ? ta.X : ta.Y;
  const int64_t row = isx ? grow : grow - ta.X.npad, n = isx ? a.n : a.m, npad = sd.npad;
  if (row >= npad) return;
  const float* X = isx ? a.X : a.Y;
  const float* centre = a.X;
  __half* sl = const_cast<__half*>(sd.slices);
  double xv[2] = {0.0, 0.0};
  if (row < n) {
    if (lane < d) xv[0] = (double)X[row * d + lane] - (double)centre[lane];
    if (lane + 32 < d) xv[1] = (double)X[row * d + lane + 32] - (double)centre[lane + 32];
  }
  double q = xv[0] * xv[0] + xv[1] * xv[1];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  const TcScale sc = scale;
  const int e = isx ? sc.ex : sc.ey;
  if (lane == 0) const_cast<double*>(sd.nx)[row] = q;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int k = lane + 32 * c;
    long long Q = (long long)rint(ldexp(xv[c] * sc.sigma, sc.bits - e));  // |Q| <= 2^b
    const int64_t idx = row * 64 + (((k >> 3) ^ (int)(row & 7)) << 3) + (k & 7);
#pragma unroll
    for (int s = kSlices - 1; s > 0; --s) {  // balanced digits from the lowest up
      const long long dig = ((Q + 512) & 1023) - 512;
      sl[(int64_t)s * npad * 64 + idx] = __float2half_rn((float)dig);
      Q = (Q - dig) >> 10;
    }
    sl[idx] = __float2half_rn((float)Q);  // |Q| <= 2^(b - 30)
  }
}

// Before each sweep: 2^a and the choice of pairs, the other side's records (all npad of them; padded
// points get Qh = -2^23 and weights 0, so no tile needs a mask) and the own
// side's P split. The same gamma as the sweep: (float) of the device value.
template <int NR, int SQM, bool ROWS>
__global__ void tc_sweep_prep_kernel(SweepArgs<float> a, TcArgs ta) {
  pdl_wait();
  if (a.active && *a.active == 0.0) return;
  const Side so = ROWS ? ta.X : ta.Y;
  const Side sq = ROWS ? ta.Y : ta.X;
  const int64_t n_own = ROWS ? a.n : a.m, n_oth = ROWS ? a.m : a.n;
  const float g = a.gamma_dev ? (float)*a.gamma_dev : a.gamma;
  const double K = (double)g * a.sC;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i == 0) {
    const double k0 = ldexp(1.0, tc_scale(ta, (double)g, a.sC).a());
    ta.kappa[0] = (float)k0;
    // 2^-23.6 sqrt(3 d) 2^a > 2^-27
    ta.kappa[1] = k0 * k0 * (3.0 * a.d) > 0x1p-7 ? 1.f : 0.f;
  }
  if (i < sq.npad) {
    constexpr int RW = rec_floats(NR);
    float4 r = make_float4(kPadQ, 0.f, 0.f, 0.f);
    if (i < n_oth) {
      const float* hq = ROWS ? a.Bh : a.Ah;
      const double Q = ((double)hq[i] - K * sq.nx[i]) * kLog2eD;
      if (!(fabs(Q) < kQLimit)) atomicOr(ta.err, kStatRange);
      const double qh = rint(Q * 8.0) * kGrid;
      const double ql = Q - qh;
      const double f1 = exp2(ql);
      const double f2 = SQM ? exp2(2.0 * ql) : 0.0;
      const float* const* wt = ROWS ? a.wc : a.wr;
      r.x = (float)qh;
      r.y = (float)((double)wt[0][i] * ((SQM & 1) ? f2 : f1));
      if constexpr (NR > 1) r.z = (float)((double)wt[1][i] * ((SQM & 2) ? f2 : f1));
      if constexpr (NR > 2) r.w = (float)((double)wt[2][i] * ((SQM & 4) ? f2 : f1));
    }
    if constexpr (RW == 2) reinterpret_cast<float2*>(sq.rec)[i] = make_float2(r.x, r.y);
    else reinterpret_cast<float4*>(sq.rec)[i] = r;
  } else if (i < sq.npad + so.npad) {
    const int64_t e = i - sq.npad;
    OwnRec o{0.f, 0.f, 0.0, 1.0, 1.0};
    if (e < n_own) {
      const float* ho = ROWS ? a.Ah : a.Bh;
      const double P = ((double)ho[e] - K * so.nx[e]) * kLog2eD;
      if (!(fabs(P) < kQLimit)) atomicOr(ta.err, kStatRange);
      const double ph = rint(P * 8.0) * kGrid;
      o.ph = (float)ph;
      o.pl = P - ph;
      o.f1 = exp2(o.pl);
      o.f2 = SQM ? exp2(2.0 * o.pl) : 1.0;
    }
    so.own[e] = o;
  }
}

// Base-2 log-sum-exp pairs (m in whole units, s >= 0; s == 0: empty): the factors are
// exact powers of two (a running max on the 1/8 grid cost the rounding of ex2.approx per
// move: row sums of clustered points in d = 64 6.7e-8 off).
__device__ __forceinline__ void lse2_add(double& M, double& s, double qm, double qs) {
  if (!(qs > 0.0)) return;
  if (!(s > 0.0)) {
    M = qm;
    s = qs;
    return;
  }
  const double Mn = fmax(M, qm);
  s = s * (double)ex2_approx((float)(M - Mn)) + qs * (double)ex2_approx((float)(qm - Mn));
  M = Mn;
}

// Waits by lane 0 only, result broadcast: keeps the warp converged before the
// .sync.aligned TMEM loads.
// Each poll may sleep up to kEpiSleepNs, so that waiting epilogue warps leave
// the issue slots of their SM sub-partition to the MMA-issuing thread.
constexpr uint32_t kEpiSleepNs = 200;
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, int* err) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity, err, kStatTimeout, kTcWaitNs, kEpiSleepNs) ? 1 : 0;
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

template <int V>
using I = std::integral_constant<int, V>;

template <int NR, bool LSE, int SQM, bool ROWS, class Epi>
__global__ void __launch_bounds__(kTcThreads, 1) tc_sweep_kernel(SweepArgs<float> a, TcArgs ta, Epi epi) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(sm + kOffBar);  // [kSliceBufs] the slices of the slice buffer landed
  uint64_t* sfree = full + kSliceBufs;         // [kSliceBufs][2] per issuer: its MMAs reading the slice buffer done
  uint64_t* lvl = sfree + 2 * kSliceBufs;      // [2] MMAs of levels {0,1}, {2,3} done (one arrival per issuer)
  uint64_t* lfree = lvl + 2;                   // [2] those levels loaded by all epilogue warps
  uint64_t* recf = lfree + 2;                  // [kRecSlots] records of the slot landed
  uint64_t* ownf = recf + kRecSlots;           // the own slices are in TMEM (one arrival per epilogue warp)
  uint32_t* tslot = (uint32_t*)(ownf + 1);
  static_assert(3 * kSliceBufs + 4 + kRecSlots + 2 <= 32, "barrier area");
  constexpr int NA = LSE ? 1 : NR;
  constexpr int ND = Epi::kDot;
  constexpr int RW = rec_floats(NR);
  constexpr uint32_t kTileRec = kN * RW * 4;  // record bytes of a tile
  __shared__ float hsum[kParts - 1][NA][kM], hcmp[kParts - 1][NA][kM], hmax[kParts - 1][kM];
  __shared__ int last_blk;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_own = ROWS ? a.n : a.m, n_oth = ROWS ? a.m : a.n;
  const Side so = ROWS ? ta.X : ta.Y;
  const Side sq = ROWS ? ta.Y : ta.X;
  const int64_t blk = blockIdx.x, sidx = blockIdx.y, S = gridDim.y;
  const int64_t j0 = sidx * a.chunk, j1 = min(n_oth, j0 + a.chunk);
  const int T = (int)((j1 - j0 + kN - 1) / kN);

  if (threadIdx.x == 0) {
    for (int k = 0; k < kSliceBufs; ++k) {
      mbar_init(&full[k], 1);
      mbar_init(&sfree[2 * k], 1);
      mbar_init(&sfree[2 * k + 1], 1);
    }
    for (int g = 0; g < 2; ++g) mbar_init(&lvl[g], 2);
    for (int g = 0; g < 2; ++g) mbar_init(&lfree[g], kEpiWarps);
    for (int k = 0; k < kRecSlots; ++k) mbar_init(&recf[k], 1);
    mbar_init(ownf, kEpiWarps);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(tslot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *(volatile uint32_t*)tslot;
  pdl_wait();
  if (a.active && *a.active == 0.0) {  // CG stopped: nothing to do (uniform over the grid)
    __syncthreads();
    if (warp == 1) tmem_free(tbase, kTmemCols);
    return;
  }

  // per-thread results of the epilogue (own point r of this CTA, one column part)
  const bool epi_warp = warp >= 2 && warp < 2 + kEpiWarps;
  const int q = warp & 3, part = epi_warp ? (warp - 2) >> 2 : 0;
  const int r = 32 * q + lane;
  const int64_t e = blk * kM + r;
  const bool ev = epi_warp && e < n_own;
  float Sa[NA], Ca[NA], mx = kPadQ;
#pragma unroll
  for (int k = 0; k < NA; ++k) {
    Sa[k] = 0.f;
    Ca[k] = 0.f;
  }

  if (warp == 1) {
    // ---------------- bulk copies (one thread) ----------------
    // Tile tt's slices into buffer tt % 3 and its records into slot tt % 5. Tiles 0-2
    // go at once; tile tt >= 3 once the MMAs of tile tt - 3 are done (sfree), by when
    // the epilogue had loaded tile tt - 4 and so finished tile tt - 5, the previous
    // user of the record slot.
    if (lane == 0) {
      const unsigned char* oth_src = (const unsigned char*)sq.slices;
      int issued = 0;
      for (int tt = 0; tt < T; ++tt) {
        const int sb = tt % kSliceBufs, rs = tt % kRecSlots;
        const uint32_t opar = (uint32_t)((tt - kSliceBufs) / kSliceBufs) & 1u;  // tile tt - kSliceBufs' phase
        if (tt >= kSliceBufs &&
            (!mbar_wait(&sfree[2 * sb], opar, ta.err, kStatTimeout, kTcWaitNs, kEpiSleepNs) ||
             !mbar_wait(&sfree[2 * sb + 1], opar, ta.err, kStatTimeout, kTcWaitNs, kEpiSleepNs)))
          break;
        const int64_t jt = j0 + (int64_t)tt * kN;
        const unsigned char* src = oth_src + jt * kRowB;
        mbar_arrive_expect_tx(&full[sb], kSlices * kOthSlice);
        for (int s = 0; s < kSlices; ++s)
          bulk_g2s(sm + kOffOth + (sb * kSlices + s) * kOthSlice, src + (int64_t)s * sq.npad * kRowB, kOthSlice,
                   &full[sb]);
        mbar_arrive_expect_tx(&recf[rs], kTileRec);
        bulk_g2s(sm + kOffRec + rs * kRecBytes, sq.rec + jt * RW, kTileRec, &recf[rs]);
        issued = tt + 1;
      }
      // leave no copy in flight (bounded waits that ignore the error flag): the
      // slices of the last tiles issued (a buffer was reused only after the MMAs had
      // read its previous tile) and their records
      for (int tt = (issued > kSliceBufs ? issued - kSliceBufs : 0); tt < issued; ++tt)
        mbar_wait(&full[tt % kSliceBufs], (tt / kSliceBufs) & 1, ta.err, 0, kTcDrainNs);
      for (int tt = (issued > kRecSlots ? issued - kRecSlots : 0); tt < issued; ++tt)
        mbar_wait(&recf[tt % kRecSlots], (tt / kRecSlots) & 1, ta.err, 0, kTcDrainNs);
    }
    __syncwarp();
  } else if (warp == 0 || warp == kMmaWarpB) {
    // ---------------- MMAs (two threads) ----------------
    // Issuer A (warp 0) owns levels 0 and 3, issuer B (the last warp) levels 1
    // and 2 (five slice pairs each): each level's accumulation chain stays in one
    // thread, and with the issuers on two SM sub-partitions the tensor unit's short
    // queue stays fed while the epilogue warps compete for issue slots (one issuer
    // loses ~25 % of the MMA rate to them). Per tile each waits for the slices, then
    // for the epilogue to have loaded levels {0,1} and {2,3} of the previous tile,
    // issues and commits its level of either pair (A, where they are needed, the three
    // pairs of level 4 before level 3), and commits its use of the slice buffer
    // (sfree[buffer][issuer]).
    if (lane == 0) {
      const int who = warp == 0 ? 0 : 1;
      const int ksteps = (a.d + 15) / 16;
      const bool own_ok = mbar_wait(ownf, 0, ta.err, kStatTimeout);
      tc_fence_after();
      // the own slices' columns and the descriptor of the first other-side slice;
      // every MMA adds a compile-time offset (all unrolled)
      const uint32_t acol = tbase + kOwnCol;
      const uint64_t bdesc0 = desc_sw128(smem_u32(sm + kOffOth));
      const uint32_t four = ta.kappa[1] != 0.f ? 1u : 0u;
      auto level = [&](uint64_t bdesc, auto Lc) {
        constexpr int L = Lc.value;
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) {
          if (k4 >= ksteps) break;  // coordinates beyond d are zero
#pragma unroll
          for (int s = 0; s < kSlices; ++s) {
            const int t = L - s;
            if (t < 0 || t >= kSlices) continue;
            const uint32_t at = tbase + (uint32_t)(L * kN), am = acol + (uint32_t)(s * 32 + k4 * 8);
            const uint64_t bm = bdesc + (uint64_t)((t * kOthSlice + k4 * 32) >> 4);
            if (L == 3 && k4 == 0 && s == 0) mma_f16_scaled10(at, am, bm, kIdesc, four);
            else mma_f16(at, am, bm, kIdesc, (k4 == 0 && s == 0) ? 0u : 1u);
          }
        }
      };
      // the pairs s + t = 4 into level 3's accumulator (which then starts from 2^-10 of it);
      // rolled: the loop over the tiles stays short where they are not needed
      auto level4 = [&](uint64_t bdesc) {
#pragma unroll 1
        for (int k4 = 0; k4 < ksteps; ++k4) {
#pragma unroll
          for (int s = 1; s < kSlices; ++s)
            mma_f16(tbase + (uint32_t)(3 * kN), acol + (uint32_t)(s * 32 + k4 * 8),
                    bdesc + (uint64_t)(((4 - s) * kOthSlice + k4 * 32) >> 4), kIdesc, (k4 == 0 && s == 1) ? 0u : 1u);
        }
      };
      int committed = 0;
      bool ok = own_ok;
      for (int tt = 0; ok && tt < T; ++tt) {
        const int sb = tt % kSliceBufs;
        const uint32_t fpar = (uint32_t)(tt / kSliceBufs) & 1u;
        const uint32_t ppar = (uint32_t)(tt - 1) & 1u;
        const uint64_t bdesc = bdesc0 + (uint64_t)((sb * kSlices * kOthSlice) >> 4);
        if (!mbar_wait(&full[sb], fpar, ta.err, kStatTimeout) ||
            (tt >= 1 && !mbar_wait(&lfree[0], ppar, ta.err, kStatTimeout))) {
          ok = false;
        } else {
          tc_fence_after();
          if (who == 0) level(bdesc, I<0>());
          else level(bdesc, I<1>());
          mma_commit(&lvl[0]);
          if (tt >= 1 && !mbar_wait(&lfree[1], ppar, ta.err, kStatTimeout)) {
            ok = false;
          } else {
            tc_fence_after();
            if (who == 0) {
              if (four) level4(bdesc);
              level(bdesc, I<3>());
            } else {
              level(bdesc, I<2>());
            }
            mma_commit(&lvl[1]);
          }
        }
        uint64_t* sf = &sfree[2 * sb + who];
        mma_commit(sf);  // also after a partly issued tile: its MMAs end before the CTA does
        if (ok) {
          committed = tt + 1;
        } else {  // that commit covers every MMA this thread issued: wait for it alone
          mbar_wait(sf, fpar, ta.err, 0, kTcDrainNs);
          committed = 0;
        }
      }
      // this issuer's MMAs of the last two committed tiles (earlier ones were
      // seen done by the copy thread before it reused their buffer)
      for (int tt = (committed > kSliceBufs ? committed - kSliceBufs : 0); tt < committed; ++tt)
        mbar_wait(&sfree[2 * (tt % kSliceBufs) + who], (tt / kSliceBufs) & 1, ta.err, 0, kTcDrainNs);
    }
    __syncwarp();
  } else if (epi_warp) {
    // ---------------- epilogue ----------------
    // the own point's digit slices to TMEM: part p stores slice p, part 0 also slice 3
    // (global layout: 128-byte swizzled rows, chunk c of a row at position c ^ (row & 7))
    for (int sl = part; sl < kSlices; sl += kParts) {
      const uint4* src = reinterpret_cast<const uint4*>(so.slices + ((int64_t)sl * so.npad + e) * 64);
      uint32_t v[32];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint4 x = __ldg(src + (c ^ (r & 7)));
        v[4 * c] = x.x;
        v[4 * c + 1] = x.y;
        v[4 * c + 2] = x.z;
        v[4 * c + 3] = x.w;
      }
      tmem_st32(tbase + ((uint32_t)(32 * q) << 16) + kOwnCol + (uint32_t)(sl * 32), v);
    }
    tmem_st_wait();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(ownf);
    const float ph = so.own[e].ph;  // e < npad: padded rows have records
    const float k0 = ta.kappa[0], k1 = k0 * 0x1p-10f, k2 = k0 * 0x1p-20f, k3 = k0 * 0x1p-30f;
    // LSE: hm = ph - mx. The max starts at -2^23, far below every entry, so the
    // first group of columns raises it to its own maximum (the one inexact step, it
    // only chooses the shift); from then on ph and mx are on the grid and hm is exact.
    // A raise forms the group's exponents again (a difference of rounded exponents
    // would not be exact), for which the LSE sweeps keep G as an FP32 pair instead of
    // adding the levels to the exponent as they come (three instructions more per
    // entry; holding the tile's levels in TMEM until its max is settled keeps the next
    // tile's MMAs waiting: 0.434 ms per LSE sweep at n = m = 16384, d = 64, this way
    // 0.317).
    float hm = LSE ? ph - mx : ph;
    const uint32_t tcol = tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(part * kPartCols);
    const float* recs = (const float*)(sm + kOffRec);
    auto release = [&](int g) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&lfree[g]);
    };
    for (int tt = 0; tt < T; ++tt) {
      const uint32_t par = (uint32_t)tt & 1u;
      const int rs = tt % kRecSlots;
      if (!warp_wait(&recf[rs], (uint32_t)(tt / kRecSlots) & 1u, ta.err)) break;
      const float* rt = recs + rs * (kRecBytes / 4) + part * kPartCols * RW;
      if (!warp_wait(&lvl[0], par, ta.err)) break;  // levels 0 and 1
      tc_fence_after();
      uint32_t u0[kPartCols], u1[kPartCols];
      tmem_ld32(tcol, u0);
      tmem_ld32(tcol + (uint32_t)kN, u1);
      tmem_ld_wait();
      release(0);
      if constexpr (!LSE) {
        float t[kPartCols];
#pragma unroll
        for (int c = 0; c < kPartCols; c += 2) {
          float qa, qb;
          if constexpr (RW == 2) {
            const float4 R = *reinterpret_cast<const float4*>(rt + c * 2);
            qa = R.x;
            qb = R.z;
          } else {
            qa = rt[c * 4];
            qb = rt[c * 4 + 4];
          }
          t[c] = fmaf(__uint_as_float(u1[c]), k1, fmaf(__uint_as_float(u0[c]), k0, __fadd_rn(hm, qa)));
          t[c + 1] = fmaf(__uint_as_float(u1[c + 1]), k1, fmaf(__uint_as_float(u0[c + 1]), k0, __fadd_rn(hm, qb)));
        }
        if (!warp_wait(&lvl[1], par, ta.err)) break;  // levels 2 and 3
        tc_fence_after();
        tmem_ld32(tcol + (uint32_t)(2 * kN), u0);
        tmem_ld32(tcol + (uint32_t)(3 * kN), u1);
        tmem_ld_wait();
        release(1);
#pragma unroll
        for (int c = 0; c < kPartCols; ++c)
          t[c] = fmaf(__uint_as_float(u1[c]), k3, fmaf(__uint_as_float(u0[c]), k2, t[c]));
#pragma unroll
        for (int c = 0; c < kGroups; ++c) {
          float acc[NA];
#pragma unroll
          for (int k = 0; k < NA; ++k) acc[k] = 0.f;
          // the group's weights, 8 columns
          float w[NA][8];
          if constexpr (RW == 2) {
#pragma unroll
            for (int jj = 0; jj < 8; jj += 2) {
              const float4 R = *reinterpret_cast<const float4*>(rt + (c * 8 + jj) * 2);
              w[0][jj] = R.y;
              w[0][jj + 1] = R.w;
            }
          } else {
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
              const float4 R = *reinterpret_cast<const float4*>(rt + (c * 8 + jj) * 4);
              const float ws[3] = {R.y, R.z, R.w};
#pragma unroll
              for (int k = 0; k < NA; ++k) w[k][jj] = ws[k];
            }
          }
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            const float ex = ex2_approx(t[c * 8 + jj]);
#pragma unroll
            for (int k = 0; k < NA; ++k) acc[k] = fmaf(((SQM >> k) & 1) ? ex * ex : ex, w[k][jj], acc[k]);
          }
#pragma unroll
          for (int k = 0; k < NA; ++k) kadd(Sa[k], Ca[k], acc[k]);
        }
      } else {
        // G = S_0 + 2^-10 S_1 + ... as an FP32 pair (gh, gl) in (u0, u1). S_0 is an
        // integer up to 2^24 and 2^-10 S_1 a multiple of 2^-10 up to 2^14: where
        // |S_0| >= |2^-10 S_1| Fast2Sum is exact, and otherwise the sum stays within
        // 2^15 and h - S_0 is a multiple of 2^-9 or 2^-10 that FP32 holds, so z and the
        // error are exact as well.
#pragma unroll
        for (int c = 0; c < kPartCols; ++c) {
          const float s0 = __uint_as_float(u0[c]), s1 = __uint_as_float(u1[c]);
          const float h = fmaf(s1, 0x1p-10f, s0);
          const float z = __fsub_rn(h, s0);
          u0[c] = __float_as_uint(h);
          u1[c] = __float_as_uint(fmaf(s1, 0x1p-10f, -z));
        }
        if (!warp_wait(&lvl[1], par, ta.err)) break;  // levels 2 and 3
        tc_fence_after();
#pragma unroll
        for (int L = 2; L < kLevels; ++L) {
          uint32_t u[kPartCols];
          tmem_ld32(tcol + (uint32_t)(L * kN), u);
          tmem_ld_wait();
          if (L == 3) release(1);
          const float sc = L == 2 ? 0x1p-20f : 0x1p-30f;
#pragma unroll
          for (int c = 0; c < kPartCols; ++c)
            u1[c] = __float_as_uint(fmaf(__uint_as_float(u[c]), sc, __uint_as_float(u1[c])));
        }
#pragma unroll
        for (int c = 0; c < kGroups; ++c) {
          float qh[8], w[8], t[8], tmax;
#pragma unroll
          for (int jj = 0; jj < 8; jj += 2) {
            const float4 R = *reinterpret_cast<const float4*>(rt + (c * 8 + jj) * 2);
            qh[jj] = R.x;
            w[jj] = R.y;
            qh[jj + 1] = R.z;
            w[jj + 1] = R.w;
          }
          auto form = [&] {
            tmax = -3.0e38f;
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
              t[jj] = fmaf(__uint_as_float(u1[c * 8 + jj]), k0,
                           fmaf(__uint_as_float(u0[c * 8 + jj]), k0, __fadd_rn(hm, qh[jj])));
              tmax = fmaxf(tmax, t[jj]);
            }
          };
          form();
          for (int k = 0; k < 4 && tmax > kTheta2; ++k) {  // raise the max (rare after the first group)
            const float dlt = ceilf(tmax);  // whole units: exact factors here and where partial sums meet
            mx += dlt;
            hm = ph - mx;
            const float f = ex2_approx(-dlt);
            Sa[0] *= f;
            Ca[0] *= f;
            form();
          }
          float acc = 0.f;
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) acc = fmaf(ex2_approx(t[jj]), w[jj], acc);
          kadd(Sa[0], Ca[0], acc);
        }
      }
    }
    if (part > 0) {  // parts 1 and 2 hand their sums to part 0
#pragma unroll
      for (int k = 0; k < NA; ++k) {
        hsum[part - 1][k][r] = Sa[k];
        hcmp[part - 1][k][r] = Ca[k];
      }
      hmax[part - 1][r] = mx;
    }
  }
  pdl_trigger();
  tc_fence_before();
  __syncthreads();  // every TMEM read and MMA is done; the parts are in shared memory
  if (warp == 1) {
    tc_fence_after();
    tmem_free(tbase, kTmemCols);
  }
  if (epi_warp && part == 0 && ev) {
    if constexpr (!LSE) {
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        double v = (double)Sa[k] + (double)Ca[k];
#pragma unroll
        for (int pp = 0; pp < kParts - 1; ++pp) v += (double)hsum[pp][k][r] + (double)hcmp[pp][k][r];
        a.rowpart[((int64_t)k * S + sidx) * n_own + e] = v;
      }
    } else {
      double M = 0.0, s = 0.0;
      lse2_add(M, s, (double)mx, (double)Sa[0] + (double)Ca[0]);
#pragma unroll
      for (int pp = 0; pp < kParts - 1; ++pp)
        lse2_add(M, s, (double)hmax[pp][r], (double)hsum[pp][0][r] + (double)hcmp[pp][0][r]);
      a.rowpart[((int64_t)0 * S + sidx) * n_own + e] = M;
      a.rowpart[((int64_t)1 * S + sidx) * n_own + e] = s;
    }
  }
  __syncthreads();

  // ---- the last CTA of this own block adds the S partials in fixed order ----
  if (threadIdx.x == 0) {
    __threadfence();
    last_blk = (atomicAdd(a.cnt_rowblk + blk, 1) == (int)S - 1);
  }
  __syncthreads();
  if (!last_blk) return;
  __threadfence();
  double wd[ND > 0 ? ND : 1];
#pragma unroll
  for (int k = 0; k < (ND > 0 ? ND : 1); ++k) wd[k] = 0.0;
  if (threadIdx.x < kM) {
    const int64_t ee = blk * kM + threadIdx.x;
    if (ee < n_own) {
      const OwnRec o = so.own[ee];
      DotArr<ND> dd;
      if constexpr (!LSE) {
        double tot[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) {
          double v = 0.0;
          ordered_loads(a.rowpart + (int64_t)k * S * n_own + ee, n_own, S, [&](double qv) { v += qv; });
          tot[k] = v * (((SQM >> k) & 1) ? o.f2 : o.f1);
        }
        if constexpr (ROWS) epi.row(ee, tot, dd.v);
        else epi.col(ee, tot, dd.v);
      } else {
        double M = 0.0, s = 0.0;
        ordered_loads2(a.rowpart + ee, a.rowpart + S * n_own + ee, n_own, S,
                       [&](double qm, double qs) { lse2_add(M, s, qm, qs); });
        const double m_nat = s > 0.0 ? (M + o.pl) * kLn2D : 0.0;
        if constexpr (ROWS) epi.row_lse(ee, m_nat, s, dd.v);
        else epi.col_lse(ee, m_nat, s, dd.v);
      }
#pragma unroll
      for (int k = 0; k < ND; ++k) wd[k] = dd.v[k];
    }
  }
  if (threadIdx.x == 0) a.cnt_rowblk[blk] = 0;
  if constexpr (ND > 0) {
#pragma unroll
    for (int k = 0; k < ND; ++k) wd[k] = warp_sum(wd[k]);
    cta_dot_finish<ND, Epi, kTcWarps>(wd, blk, gridDim.x, a.dotpart, a.cnt_dot, epi);
  }
}

}  // namespace tc
}  // namespace eot
