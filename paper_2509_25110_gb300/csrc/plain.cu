// Plain FP64 / FP32 path: the tau-window sum of Eq. (2) per (k, l) on the CUDA
// cores (Algorithm 1's gang over k and vector loops over l and tau, here one
// CTA per (k, rows of an l-tile, source chunk)), and the FP64 k-sum of Eq. (1).
#include <cmath>
#include <type_traits>

#include "internal.h"

namespace gcamb {

// The first step(s) of a sum over lanes of several values a lane holds: a
// lane keeps half of its values, sends the other half to its partner (lane
// XOR o) and adds what it receives.
template <typename T, int N, int V>
__device__ __forceinline__ void halve_lanes(T (&v)[V], int lane, int o) {
  const bool up = (lane & o) != 0;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const T send = up ? v[j] : v[j + N];
    const T keep = up ? v[j + N] : v[j];
    v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
}

// FP32 sums over lanes and what follows them are carried as the sum of two
// floats: their additions are those of the largest numbers (E-mode of 5 sources
// to l 2001, error against 64 bits 3.7e-8, 5.0e-8 with plain floats, at 278 and
// 275 us).
__device__ __forceinline__ float2 add_ff(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x), t = __fsub_rn(s, a.x);
  const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, t)), __fsub_rn(b.x, t));
  return make_float2(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ double add_ff(double a, double b) { return a + b; }
__device__ __forceinline__ float2 shfl_ff(float2 v, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}
__device__ __forceinline__ double shfl_ff(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
// (where the first float is infinite or NaN the second holds nothing)
__device__ __forceinline__ float round_ff(float2 s) { return fabsf(s.x) <= 3.402823466e38f ? __fadd_rn(s.x, s.y) : s.x; }
__device__ __forceinline__ double round_ff(double s) { return s; }
__device__ __forceinline__ double wide(float2 s) {
  return fabsf(s.x) <= 3.402823466e38f ? (double)s.x + (double)s.y : (double)s.x;
}
__device__ __forceinline__ double wide(double s) { return s; }
__device__ __forceinline__ float2 as_ff(float v) { return make_float2(v, 0.f); }
__device__ __forceinline__ double as_ff(double v) { return v; }
template <typename T>
using PlainSum = std::conditional_t<sizeof(T) == 8, double, float2>;

// halve_lanes on such sums.
template <int N, int V>
__device__ __forceinline__ void halve_lanes(float2 (&v)[V], int lane, int o) {
  const bool up = (lane & o) != 0;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const float2 send = up ? v[j] : v[j + N], keep = up ? v[j + N] : v[j];
    v[j] = add_ff(keep, shfl_ff(send, o));
  }
}

// Sum over the 8 lanes of a group of each of the RV values a lane holds
// (RV = 4, 8); lane L of the group returns the total of value L / (8 / RV).
// The additions of one value are the same for both RV (partners 4, 2, 1).
template <typename T, int RV>
__device__ __forceinline__ PlainSum<T> reduce_group(T (&v)[RV], int lane) {
  static_assert(RV == 4 || RV == 8, "reduce_group: RV in {4, 8}");
  if constexpr (sizeof(T) == 8) {
    halve_lanes<T, RV / 2>(v, lane, 4);
    halve_lanes<T, RV / 4>(v, lane, 2);
    if constexpr (RV == 8) halve_lanes<T, 1>(v, lane, 1);
    else v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return v[0];
  } else {
    float2 w[RV / 2];
    const bool up = (lane & 4) != 0;
#pragma unroll
    for (int j = 0; j < RV / 2; ++j) {
      const T send = up ? v[j] : v[j + RV / 2], keep = up ? v[j + RV / 2] : v[j];
      w[j] = add_ff(as_ff(keep), as_ff(__shfl_xor_sync(0xffffffffu, send, 4)));
    }
    halve_lanes<RV / 4>(w, lane, 2);
    if constexpr (RV == 8) halve_lanes<1>(w, lane, 1);
    else w[0] = add_ff(w[0], shfl_ff(w[0], 1));
    return w[0];
  }
}

// What is summed against the table's w_i j_l:
//   kFieldT       the sources themselves
//   kFieldE       S_P x^-2, x = k (tau0 - tau) (E-mode, Eq. 3)
//   kFieldTensor  S_P, S_P x^-1, S_P x^-2 and S_T x^-2 (tensor modes)
enum PlainField { kFieldT = 0, kFieldE = 1, kFieldTensor = 2 };

struct PlainArgs {
  const int32_t *nkb;   // [nk][nlt] stored tau-blocks
  const int64_t *off;   // [nk][nlt] first block
  const int *lrow;      // [nl] multipole of each row
  const double *kk, *tau, *wtau;
  const float2 *dt2;    // [ntau] tau0 - tau as the sum of two floats
  const double *cl;     // [nl] c_l = sqrt((l+2)!/(l-2)!) of each row (0 for l < 2)
  const float2 *cl2;    // [nl] the same as the sum of two floats
  const double *xthr;   // [nl] Watson thresholds, or null: every row takes the whole tile's prefix
  double tau0, x_lo;
  int nk, nlt, nl, ntau, M;
  // tensor: lmin.  Temperature: a block's steps - 1 where rows take whole blocks,
  // else 0 (one word for both, and looked at outside the sums: as an argument of its
  // own, and in them, it made registers spill: FP32, six to eight sources 5-9%).
  int lmin_or_round;
  int q0;               // last k of the launch
  int rows;             // rows per CTA: 128 or 64
};

constexpr int kPlainWarps = 4;
constexpr int kPlainKB = 64;  // tau nodes per table block

// Rows a lane holds at a time (a warp pass covers 4 of them per lane group).
constexpr int plain_rv(int nv) { return nv == 1 ? 8 : 4; }

// Steps whose table loads a lane has in flight together: FP64 is bound by its
// pipe at one (2 measured the same), FP32 by loads in flight (E-mode, 5
// sources, l_max 2001: 352 us at one, 318 at two).
template <typename T>
constexpr int plain_unroll() { return sizeof(T) == 8 ? 1 : 2; }

// Steps ahead at which a row's line is asked into L2 (0: not), a line a lane:
// the FP32 kernel's registers hold two steps' loads, which cover half of the
// DRAM latency (E-mode, 5 sources, l_max 2001: 301 us without, 290 / 278 /
// 273 / 278 / 282 / 298 at 2 / 3 / 4 / 6 / 8 / 16).  FP64 gains nothing (l_max 500 68.8,
// 68.4 at 4, l_max 5000 7953, 7910 at 4 and 8622 at 8).
template <typename T>
constexpr int plain_ahead() { return sizeof(T) == 8 ? 0 : 4; }

// A row's sum is taken in groups of 32 blocks (2048 nodes), each reduced over
// the lanes and added to those before it.  The group is the same for every
// number of sources, so that a source's result does not depend on the batch it
// came in (a staged chunk holds 128 blocks of one FP64 source, 32 of four).
constexpr int kPlainGroup = 32;

// Tau blocks staged in shared memory at a time: whole groups, up to 64 KB of
// sources.  (Staging every group by itself: one FP64 source, 8000 tau 2546 ->
// 3169 us.)
// (FP32 E-mode of three and four sources: one group, so that no loop over groups
// takes registers: 205 -> 196 and 227 -> 214 us, 1106 k x 698 tau to l 1738.)
constexpr bool plain_one_group(int nv, size_t esize, int field) {
  return esize == 4 && field == kFieldE && (nv == 3 || nv == 4);
}
constexpr int plain_stage_blocks(int nv, size_t esize, int field) {
  if (plain_one_group(nv, esize, field)) return kPlainGroup;
  return (int)(65536 / (nv * esize * kPlainKB)) / kPlainGroup * kPlainGroup;
}

// x^-1 and x^-2 of one node as sums of two floats (about 2^-45 relative), from
// x = k dt with k and dt as sums of two floats, in FP32 operations: GB300's
// FP64 pipe runs at 1/64 of the FP32 rate.
__device__ __forceinline__ void inv_x_ff(float2 k, float2 d, float2 &i1, float2 &i2) {
  const float p = __fmul_rn(k.x, d.x);
  float e = __fmaf_rn(k.x, d.x, -p);
  e = __fmaf_rn(k.x, d.y, e);
  e = __fmaf_rn(k.y, d.x, e);
  const float r = __frcp_rn(p);
  i1.x = r;
  i1.y = __fmul_rn(r, __fmaf_rn(-e, r, __fmaf_rn(-p, r, 1.f)));
  const float p2 = __fmul_rn(p, p);
  const float e2 = __fmaf_rn(__fmul_rn(2.f, p), e, __fmaf_rn(p, p, -p2));
  const float s = __frcp_rn(p2);
  i2.x = s;
  i2.y = __fmul_rn(s, __fmaf_rn(-e2, s, __fmaf_rn(-p2, s, 1.f)));
}

// v (f.x + f.y), rounded once but for the last bits of f.
__device__ __forceinline__ float mul_ff(float v, float2 f) {
  const float p = __fmul_rn(v, f.x);
  const float e = __fmaf_rn(v, f.y, __fmaf_rn(v, f.x, -p));
  return fabsf(p) <= 3.4e38f ? __fadd_rn(p, e) : p;  // overflow, infinities, NaN: the plain product
}

// (v.x + v.y) (f.x + f.y), the same way.
__device__ __forceinline__ float mul_ff(float2 v, float2 f) {
  const float p = __fmul_rn(v.x, f.x);
  const float e = __fmaf_rn(v.y, f.x, __fmaf_rn(v.x, f.y, __fmaf_rn(v.x, f.x, -p)));
  return fabsf(p) <= 3.4e38f ? __fadd_rn(p, e) : p;
}

// The power series of the tensor kernels at small x for the nodes
// below the cut, from j_l(x) = x^l s_l(x^2),
// s_l(y) = sum_n (-y/2)^n / (n! (2l+2n+1)!!) (seven terms: exact to rounding
// for x <= 0.2):
//   e_l = x^(l-2) [l (l-1) s_l - 2 x^2 s_l + 2 s_(l-1)],
//   b_l = 2 x^(l-1) [s_(l-1) - (l-1) s_l].
__device__ __forceinline__ double sph_series(int l, double y) {
  double df = 1.0;  // (2l+1)!!
  for (int j = 3; j <= 2 * l + 1; j += 2) df *= j;
  double term = 1.0 / df, sum = term;
  for (int n = 0; n < 6; ++n) {
    term *= (-0.5 * y) / ((n + 1) * (2.0 * l + 2 * n + 3));
    sum += term;
  }
  return sum;
}

// E-mode term of row l from the sum D2 of S_P x^-2 j_l: c_l D2, plus, at
// l = 2, the nodes below x_lo (the tail of the tau grid: x falls with tau)
// through the power series
//   j_2(x)/x^2 = 1/15 - x^2/210 + x^4/7560 - x^6/498960 + O(x^8)
// (from j_l(x) = x^l sum_n (-x^2/2)^n / (n! (2l+2n+1)!!)): there the table's
// j_2 may be cut to zero (activity threshold, Miller start) although
// j_2(x)/x^2 -> 1/15.  For l >= 3 their eps_l is below
// c_l x_lo^(l-2)/(2l+1)!!, and x_lo <= 0.2.
template <typename T>
__device__ __forceinline__ T emode_row(const PlainArgs &a, int row, double kq, PlainSum<T> d2, const T *src) {
  if (a.lrow[row] != 2) {
    // c_l from the grid: its square root and the FP64 product per (row,
    // source) took half of the FP32 kernel's time
    if constexpr (sizeof(T) == 8) return a.cl[row] * d2;
    else return mul_ff(d2, a.cl2[row]);
  }
  const double c = a.cl[row];
  double d = c * wide(d2);
  {
    double tail = 0.0;
    for (int i = a.ntau - 1; i >= 0; --i) {
      const double x = kq * (a.tau0 - a.tau[i]);
      if (!(x < a.x_lo)) break;
      const double x2 = x * x;
      const double e2 = 1.0 / 15.0 - x2 * (1.0 / 210.0 - x2 * (1.0 / 7560.0 - x2 / 498960.0));
      tail += a.wtau[i] * (double)src[i] * e2;
    }
    d += c * tail;
  }
  return (T)d;
}

// One CTA (4 warps): `rows` multipoles of an l-tile x MC sources at one k.
// The sources' tau-prefix is staged in shared memory (times x^-1, x^-2 for
// the polarisation and tensor fields; NV = MC or 4 MC staged vectors).
//
// What bounds it.  FP64: the DFMA pipe (two lanes a clock and SM), so every
// FP64 instruction that is not a product of the sum counts: the row prefixes
// are compared as integers, the lanes of a group of 8 share a row (16-byte
// loads; the lane sums of 32 rows reduce in 7 adds, where a warp per row
// needed 9 adds for 8), the tensor kernels read the table once for their
// four sums and combine them here.  FP32: HBM for one source, else the FP32
// pipe and shared-memory reads, which RV rows a lane amortise.
// Measured (one model, before -> after): FP64 l_max 500 93 -> 69 us,
// l_max 5000 9380 -> 7951 us (its products alone: 7300 us); tensor modes l_max
// 1500 3105 (four passes and a combining one) -> 1948 us; FP32 E-mode, 5
// sources, l_max 2001 950 -> 278 us.
//
// Splits: a warp pass covers 4 RV rows (lane group g, slot i: row 4 i + g);
// the rows / 32 row warps take passes in turn, and the 128 / rows warps that
// share a row take every (128 / rows)-th tau block; their sums are added in a
// fixed order.  `rows` depends on the grid only (plain_rows), so a source's
// result does not depend on the batch it came in.
//
// a.xthr (flat j_l grids, else null): per row the Watson threshold below
// which |j_l| < eps_cut.  The tile's tau-prefix is that of its lowest
// multipole; four adjacent rows stop at the first step (16 or 32 nodes) whose first
// node has x below the lowest one's threshold (x falls along tau, so every
// later node is below it too): the terms left out are below eps_cut |w S|
// each.  With x^-1 or x^-2 only rows whose threshold is at least 1 stop:
// j_l(x) x^-2 rises with x below the threshold (l >= 3 there), so each term
// left out is below eps_cut |w S| as well, and c_l / x^2 (below 300) times that
// in the result; these fields have the thresholds only where that is nothing
// (kRowCut).
template <typename T, int MC, int FIELD>
__global__ void __launch_bounds__(kPlainWarps * 32, 4)
    los_plain_kernel(const T *__restrict__ table, const T *__restrict__ S, const T *__restrict__ ST,
                     T *__restrict__ Delta, T *__restrict__ DE, T *__restrict__ DB, PlainArgs a) {
  using V16 = std::conditional_t<sizeof(T) == 8, double2, float4>;
  constexpr int KB = kPlainKB;
  constexpr int NV = FIELD == kFieldTensor ? 4 * MC : MC;
  constexpr int RV = plain_rv(NV);
  constexpr int VE = 16 / sizeof(T);        // nodes per 16-byte load
  constexpr int SN = 8 * VE;                // nodes per step of a lane group (128 bytes of a row): 16 or 32
  constexpr int STEPS = KB / SN;            // steps per block
  constexpr int CHB = plain_stage_blocks(NV, sizeof(T), FIELD);
  constexpr int HALO = FIELD == kFieldTensor ? 1 : 0;  // tensor: also the row before the CTA's first
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int R = a.rows, TS = kTileL / R;
  const int q = a.q0 - blockIdx.y;          // the long prefixes (high k) first
  const int lt = blockIdx.x / TS, rsub = (blockIdx.x - lt * TS) * R;
  const int m0 = blockIdx.z * MC, mc = min(MC, a.M - m0);
  const int row0 = lt * kTileL + rsub;      // first output row of the CTA
  if (row0 >= a.nl) return;
  const size_t e_idx = (size_t)q * a.nlt + lt;
  const int nb = a.nkb[e_idx];
  if (nb == 0 && (FIELD == kFieldT || a.lrow[row0] > 5)) {  // nothing active, no small-x tail: zeros
    for (int idx = threadIdx.x; idx < mc * R; idx += kPlainWarps * 32) {
      const int m = idx / R, r = idx - m * R;
      if (row0 + r >= a.nl) continue;
      const size_t o = ((size_t)(m0 + m) * a.nk + q) * a.nl + row0 + r;
      Delta[o] = T(0);
      if constexpr (FIELD == kFieldTensor) DE[o] = DB[o] = T(0);
    }
    return;
  }
  const double kq = a.kk[q];
  const int stride = (nb < CHB ? nb : CHB) * KB;  // staged nodes per vector
  T *s = reinterpret_cast<T *>(smem_raw);                       // [NV][stride]
  using Sum = PlainSum<T>;
  Sum *res = reinterpret_cast<Sum *>(s + (size_t)NV * stride);  // [TS][NV][R]
  long long *xb = reinterpret_cast<long long *>(res + (size_t)NV * kTileL);  // [nb STEPS] x of each step's first node
  Sum *halo = reinterpret_cast<Sum *>(xb + nb * STEPS);         // tensor: [NV] sums of row row0 - 1
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = lane >> 3, sub = lane & 7;
  const int WR = kPlainWarps / TS, rw = warp % WR, ts = warp / WR;
  // nonnegative doubles order as their bit patterns
  for (int i = tid; i < nb * STEPS; i += kPlainWarps * 32) {
    const int n = SN * (FIELD == kFieldT ? i & ~a.lmin_or_round : i);  // whole blocks: that of the block's first node
    xb[i] = n < a.ntau ? __double_as_longlong(kq * (a.tau0 - a.tau[n])) : -1;
  }
  for (int i = tid; i < NV * kTileL; i += kPlainWarps * 32) res[i] = as_ff(T(0));
  if (HALO && tid < NV) halo[tid] = as_ff(T(0));
  const T *chunk = table + (size_t)a.off[e_idx] * (kTileL * KB);
  for (int b0 = 0; b0 < nb; b0 += CHB) {
    const int nbc = min(CHB, nb - b0), nt = nbc * KB, t0 = b0 * KB;
    if (b0) __syncthreads();
    // ---- stage the sources of nodes t0 .. t0 + nt (zero beyond ntau)
    if constexpr (FIELD == kFieldT) {
#pragma unroll
      for (int m = 0; m < MC; ++m) {
        const T *src = S + ((size_t)(m0 + m) * a.nk + q) * a.ntau;
#pragma unroll 4
        for (int t = tid; t < nt; t += kPlainWarps * 32)
          s[m * stride + t] = (m < mc && t0 + t < a.ntau) ? src[t0 + t] : T(0);
      }
    } else {
      const float kh = (float)kq;
      const float2 k2 = make_float2(kh, (float)(kq - (double)kh));
      // SU nodes' loads per thread in flight (a node at a time left the stage
      // bound by load latency)
      constexpr int SU = NV >= 8 ? 2 : 4;
      for (int tb = tid; tb < nt; tb += SU * kPlainWarps * 32) {
        T vv[SU][MC], ww[SU][MC];
#pragma unroll
        for (int u = 0; u < SU; ++u) {
          const int t = tb + u * kPlainWarps * 32;
          const bool in = t < nt && t0 + t < a.ntau;
#pragma unroll
          for (int m = 0; m < MC; ++m) {
            const size_t o = ((size_t)(m0 + m) * a.nk + q) * a.ntau + t0 + t;
            vv[u][m] = (in && m < mc) ? S[o] : T(0);
            ww[u][m] = (FIELD == kFieldTensor && in && m < mc) ? ST[o] : T(0);
          }
        }
#pragma unroll
        for (int u = 0; u < SU; ++u) {
          const int t = tb + u * kPlainWarps * 32;
          if (t >= nt) break;
          const bool in = t0 + t < a.ntau;
          const T(&v)[MC] = vv[u];
          const T(&w)[MC] = ww[u];
          T v0[MC], v1[MC], v2[MC], w2[MC];
          bool keep = false, ff = false;
          if constexpr (sizeof(T) == 4) {
            const float2 d2 = in ? a.dt2[t0 + t] : make_float2(0.f, 0.f);
            const float xf = k2.x * d2.x;
            // well above the cut and inside FP32's range of x^2: no FP64 needed
            ff = xf > 1e-14f && xf < 1e15f && xf > 1.01f * (float)a.x_lo && kh > 1e-30f && d2.x > 1e-30f;
            if (ff) {
              float2 i1, i2;
              inv_x_ff(k2, d2, i1, i2);
#pragma unroll
              for (int m = 0; m < MC; ++m) {
                v0[m] = v[m];
                v1[m] = mul_ff(v[m], i1);
                v2[m] = mul_ff(v[m], i2);
                w2[m] = mul_ff(w[m], i2);
              }
              keep = true;
            }
          }
          if (!ff) {
            const double x = in ? kq * (a.tau0 - a.tau[t0 + t]) : 0.0;
            keep = in && x >= a.x_lo;
            const double i1 = FIELD == kFieldTensor && keep ? 1.0 / x : 0.0;
            const double i2 = keep ? 1.0 / (x * x) : 0.0;
#pragma unroll
            for (int m = 0; m < MC; ++m) {
              v0[m] = v[m];
              v1[m] = FIELD == kFieldTensor ? (T)((double)v[m] * i1) : T(0);
              v2[m] = (T)((double)v[m] * i2);
              w2[m] = FIELD == kFieldTensor ? (T)((double)w[m] * i2) : T(0);
            }
          }
#pragma unroll
          for (int m = 0; m < MC; ++m) {
            if constexpr (FIELD == kFieldE) {
              s[m * stride + t] = keep ? v2[m] : T(0);
            } else {
              s[(4 * m + 0) * stride + t] = keep ? v0[m] : T(0);
              s[(4 * m + 1) * stride + t] = keep ? v1[m] : T(0);
              s[(4 * m + 2) * stride + t] = keep ? v2[m] : T(0);
              s[(4 * m + 3) * stride + t] = keep ? w2[m] : T(0);
            }
          }
        }
      }
    }
    __syncthreads();
    // ---- rows, a group of blocks at a time
    constexpr bool kOne = plain_one_group(NV, sizeof(T), FIELD);
#pragma unroll 1
    for (int gb = 0; gb < (kOne ? 1 : nbc); gb += kPlainGroup) {
      const int b1 = kOne ? b0 : b0 + gb, ng = kOne ? nbc : min(kPlainGroup, nbc - gb);
      const T *sg = s + gb * KB;
      for (int rb = rw * 4 * RV; rb < R; rb += WR * 4 * RV) {
        int ns[RV];  // steps of this group that rows rb + 4 i .. + 3 need
        const int nsc = ng * STEPS;
        int nmin = nsc, nmax = 0;
#pragma unroll
        for (int i = 0; i < RV; ++i) {
          const int row = row0 + rb + 4 * i;
          ns[i] = 0;
          if (row < a.nl) {
            ns[i] = nsc;
            if (a.xthr) {
              const double xe = a.xthr[row];
              if (FIELD == kFieldT || xe >= 1.0) {
                const long long xi = __double_as_longlong(xe);
                int n = 0;
                for (int c = 0; c < nsc; c += 32)
                  n += __popc(__ballot_sync(0xffffffffu, c + lane < nsc && xb[b1 * STEPS + c + lane] >= xi));
                ns[i] = n;
              }
            }
          }
          nmax = max(nmax, ns[i]);
          nmin = min(nmin, ns[i]);
        }
        T acc[NV][RV];
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int i = 0; i < RV; ++i) acc[v][i] = T(0);
        const T *rows = chunk + (size_t)b1 * kTileL * KB + (rsub + rb + grp) * KB + sub * VE;
        // a lane's row of the pass (4 RV rows) for the lines ahead
        constexpr int AHEAD = plain_ahead<T>();
        const T *arow = chunk + (size_t)b1 * kTileL * KB + (rsub + rb + lane) * KB;
        int an = 0;  // its steps
        if constexpr (AHEAD > 0) {
#pragma unroll
          for (int i = 0; i < RV; ++i) an = (lane >> 2) == i ? ns[i] : an;
        }
        // steps that all RV row sets need, then the rest (a set's bound is
        // uniform over the warp); UN steps' loads are in flight together
        auto step = [&](int i0, auto un, auto check) {
          constexpr int UN = decltype(un)::value;
          V16 j[UN][RV];
#pragma unroll
          for (int u = 0; u < UN; ++u) {
            const int st = i0 + u * TS;
            const T *blk = rows + (size_t)(st / STEPS) * (kTileL * KB) + (st % STEPS) * SN;
#pragma unroll
            for (int i = 0; i < RV; ++i)
              if (!check || st < ns[i]) j[u][i] = __ldg(reinterpret_cast<const V16 *>(blk + 4 * i * KB));
          }
#pragma unroll
          for (int u = 0; u < UN; ++u) {
            const int st = i0 + u * TS;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
              const V16 sv = *reinterpret_cast<const V16 *>(sg + v * stride + st * SN + sub * VE);
#pragma unroll
              for (int i = 0; i < RV; ++i) {
                if (check && st >= ns[i]) continue;
                const V16 t = j[u][i];
                if constexpr (sizeof(T) == 8) {
                  acc[v][i] = fma(t.y, sv.y, fma(t.x, sv.x, acc[v][i]));
                } else {
                  const float d = __fmaf_rn(t.w, sv.w, __fmaf_rn(t.z, sv.z, __fmaf_rn(t.y, sv.y, __fmul_rn(t.x, sv.x))));
                  acc[v][i] = __fadd_rn(acc[v][i], d);
                }
              }
            }
          }
        };
        constexpr int UN = plain_unroll<T>();
        int st = ts;
        for (; st + (UN - 1) * TS < nmin; st += UN * TS) {
          if constexpr (AHEAD > 0) {
#pragma unroll
            for (int u = 0; u < UN; ++u) {
              const int sa = st + (AHEAD + u) * TS;
              if (sa < an)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(arow + (size_t)(sa / STEPS) * (kTileL * KB) + (sa % STEPS) * SN));
            }
          }
          step(st, std::integral_constant<int, UN>(), std::false_type());
        }
        for (; st < nmax; st += TS) step(st, std::integral_constant<int, 1>(), std::true_type());
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const Sum t = reduce_group<T, RV>(acc[v], lane);
          constexpr int LPV = 8 / RV;  // lanes that end with the same value
          if (sub % LPV == 0) {
            Sum *r = res + (ts * NV + v) * R + rb + grp + 4 * (sub / LPV);
            *r = b1 ? add_ff(*r, t) : t;
          }
        }
      }
    }
    if constexpr (HALO) {
      // tensor: row row0 - 1 (of this tile, or the last row of the tile before
      // it, whose prefix is at least as long), by the last warp over all lanes
      if (warp == kPlainWarps - 1 && row0 > 0) {
        const int pr = row0 - 1, plt = pr / kTileL;
        const T *prow = table + (size_t)a.off[(size_t)q * a.nlt + plt] * (kTileL * KB) + (size_t)b0 * kTileL * KB +
                        (pr - plt * kTileL) * KB;
        for (int g0 = 0; g0 < nt; g0 += kPlainGroup * KB) {
          T h[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) h[v] = T(0);
          for (int t = g0 + lane; t < min(nt, g0 + kPlainGroup * KB); t += 32) {
            const T j = __ldg(prow + (size_t)(t / KB) * kTileL * KB + t % KB);
#pragma unroll
            for (int v = 0; v < NV; ++v)
              if (v % 4 != 3) h[v] = fma(j, s[v * stride + t], h[v]);
          }
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            if (v % 4 == 3) continue;
            Sum hs = as_ff(h[v]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) hs = add_ff(hs, shfl_ff(hs, o));
            if (lane == 0) halo[v] = add_ff(halo[v], hs);
          }
        }
      }
    }
  }
  __syncthreads();
  // ---- outputs
  auto sum = [&](int v, int r) {
    Sum t = res[v * R + r];
    for (int i = 1; i < TS; ++i) t = add_ff(t, res[(i * NV + v) * R + r]);
    return t;
  };
  for (int idx = tid; idx < mc * R; idx += kPlainWarps * 32) {
    const int m = idx / R, r = idx - m * R;
    const int row = row0 + r;
    if (row >= a.nl) continue;
    const size_t o = ((size_t)(m0 + m) * a.nk + q) * a.nl + row;
    if constexpr (FIELD == kFieldT) {
      Delta[o] = round_ff(sum(m, r));
    } else if constexpr (FIELD == kFieldE) {
      Delta[o] = emode_row<T>(a, row, kq, sum(m, r), S + ((size_t)(m0 + m) * a.nk + q) * a.ntau);
    } else {
      const size_t so = ((size_t)(m0 + m) * a.nk + q) * a.ntau;
      const int l = a.lmin_or_round + row;
      Delta[o] = emode_row<T>(a, row, kq, sum(4 * m + 3, r), ST + so);
      double ve = 0.0, vb = 0.0;
      if (l >= 2) {
        const double d0 = wide(sum(4 * m, r)), d1 = wide(sum(4 * m + 1, r)), d2 = wide(sum(4 * m + 2, r));
        double p0, p1;  // D0, D1 of row l - 1
        if (row == 0) {
          // j_(l-1) = (2l+1)/x j_l - j_(l+1) (the sums leave out the same nodes)
          p1 = a.nl > 1 ? (2.0 * l + 1.0) * d2 - wide(sum(4 * m + 1, 1)) : 0.0;
          p0 = a.nl > 1 ? (2.0 * l + 1.0) * d1 - wide(sum(4 * m, 1)) : 0.0;
        } else {
          p0 = wide(r > 0 ? sum(4 * m, r - 1) : halo[4 * m]);
          p1 = wide(r > 0 ? sum(4 * m + 1, r - 1) : halo[4 * m + 1]);
        }
        ve = (double)l * (l - 1) * d2 - 2.0 * d0 + 2.0 * p1;
        vb = 2.0 * p0 - 2.0 * (l - 1) * d1;
        if (l <= 5) {
          const T *src = S + so;
          for (int i = a.ntau - 1; i >= 0; --i) {
            const double x = kq * (a.tau0 - a.tau[i]);
            if (x >= a.x_lo) break;
            const double y = x * x, sl = sph_series(l, y), sm = sph_series(l - 1, y);
            const double xl2 = l == 2 ? 1.0 : pow(x, l - 2);
            const double ws = a.wtau[i] * (double)src[i];
            ve += ws * xl2 * ((double)l * (l - 1) * sl - 2.0 * y * sl + 2.0 * sm);
            vb += ws * 2.0 * xl2 * x * (sm - (l - 1) * sl);
          }
        }
      }
      DE[o] = (T)ve;
      DB[o] = (T)vb;
    }
  }
}

// E-mode small-x cut: at least 1e-12 and every x at which the l = 2 row of
// the table may hold zero (the activity threshold of the tile holding l = 2,
// the Miller start of j_2); at most 0.2, where the four-term series of
// j_2(x)/x^2 is still exact to 1e-12 (eps_cut <= 1e-3 keeps it near 0.12).
int emode_x_lo(const gcamb_grid *g, double *x_lo) {
  double x = 1e-12;
  if (g->lmin <= 2) {
    if (g->lmin >= 1) x = fmax(x, watson_threshold(g->lmin, std::log(g->eps_cut)));
    if (g->nxs > 2) x = fmax(x, g->xstart[2]);
  }
  *x_lo = x;
  return x <= 0.2 ? 0 : -1;
}

// Largest eps_cut with which rows stop at the very step of their own prefix.
// Beyond it temperature rows take whole blocks of 64 nodes, and polarisation and
// tensor rows the whole tile's prefix, whose rows but the lowest lose next to
// nothing at any eps_cut (E-mode at eps_cut 1e-8, 1e-6, 1e-4, error of the
// transfers: 2e-12, 2e-10, 2e-8; with rows' own prefixes 3e-8, 1e-6, 3e-4).  At
// 1e-20 the rows' own prefixes leave out 3e-20 of them, below FP64's rounding.
constexpr double kRowCut = 1e-20;

// Full-prefix tiles of the grid: blocks / longest prefix.  (A log-spaced k grid
// has most of its work in the last few k, so that the number of non-empty tiles
// says little.)
static double plain_tiles(const Table &t) { return t.max_nkb > 0 ? (double)t.nblocks / t.max_nkb : 0.0; }

// Rows per CTA of the plain kernel: a whole 128-row tile, or 64 rows (the
// CTA's four warps then share out the tau steps in pairs) where the tiles are
// too few to balance the SMs; FP32, bound by loads rather than a pipe, needs
// fewer.  Sampled multipoles take 64 rows too: the prefixes of one tile's rows
// then span most of the grid, and the warps of a CTA would finish far apart.  By
// the grid alone, so that a source's sums do not depend on its batch.  Measured at
// 128 / 64 (32) rows: FP64 l_max 500 (570 tiles) 73 / 69 (74) us; tensor l_max 1500
// (2540) 1950 / 2058 (2385); l_max 5000 (19702) 7951 / 7962 (8334); sampled l_max 2500
// (2043) 343 / 293 (302); FP32, one and eight sources, 285 tiles 15 / 18 and 29 / 35 us,
// 570 25 / 29 and 50 / 65, 1899 76 / 89 and 132 / 191, but 122 tiles 13 / 13 and 25 / 23.
static int plain_rows(const gcamb_grid *g, const Table &t) {
  return !g->lsampled && plain_tiles(t) >= kSms * (t.lay.esize == 8 ? 8 : 2) ? 128 : 64;
}

// Sources per CTA: the batch in equal chunks of at most `most` (the table is read
// once per chunk, and FP64 sums of sources that are not there would cost as much
// as real ones), smaller ones where a grid gives the chip too few CTAs: FP64
// three an SM, FP32 one and a half, counted in full-prefix CTAs with all rows in
// use.  FP64, four sources: 300 k x 400 tau sampled to l 500 (403) 114 -> 81 us, 64
// k x 100 tau to l 64 (63) 19 -> 15 us; two sources at 403: 60 -> 51 us, at 537 no
// gain.  FP32, 16 sources at 63: 14.8 -> 12.6 us.
static int plain_sources(const gcamb_grid *g, const Table &t, int M, int most) {
  const double ctas = plain_tiles(t) * (kTileL / plain_rows(g, t)) * g->nl / ((double)g->nlt * kTileL);
  const double want = t.lay.esize == 8 ? 3.0 * kSms : 1.5 * kSms;
  int chunks = (M + most - 1) / most;
  if (ctas * chunks < want) chunks = ctas * M <= want ? M : (int)std::ceil(want / ctas);
  return (M + chunks - 1) / chunks;
}

static PlainArgs plain_args(const gcamb_grid *g, const Table &t, int M, int field) {
  PlainArgs a{};
  a.nkb = t.d_nkb;
  a.off = t.d_off;
  a.lrow = g->d_lrow;
  a.kk = g->d_k;
  a.tau = g->d_tau;
  a.wtau = g->d_wtau;
  a.dt2 = reinterpret_cast<const float2 *>(g->d_dt2);
  a.cl = g->d_cl;
  a.cl2 = reinterpret_cast<const float2 *>(g->d_cl2);
  // rows stop at their own prefix on flat j_l grids only
  a.xthr = (g->kernel == 0 && !g->curved && (field == kFieldT || g->eps_cut <= kRowCut)) ? g->d_xthr : nullptr;
  a.tau0 = g->tau0;
  a.x_lo = 1e-12;
  a.nk = g->nk;
  a.nlt = g->nlt;
  a.nl = g->nl;
  a.ntau = g->ntau;
  a.M = M;
  a.rows = plain_rows(g, t);
  return a;
}

// nk, nlt: the k prefix and l-tiles of the launch (the whole grid, or an
// uneven plan chunk's).
template <typename T, int MC, int FIELD>
static int launch_plain_t(const gcamb_grid *g, const Table &t, const T *S, const T *ST, int M, T *D, T *DE, T *DB,
                          int nk, int nlt, cudaStream_t st) {
  constexpr int NV = FIELD == kFieldTensor ? 4 * MC : MC;
  PlainArgs a = plain_args(g, t, M, FIELD);
  if (FIELD != kFieldT && emode_x_lo(g, &a.x_lo))
    return fail(GCAMB_EINVAL, "los_transfer: eps_cut too large for the l = 2 limit of the polarisation kernels");
  const int stage = t.max_nkb < plain_stage_blocks(NV, sizeof(T), FIELD) ? t.max_nkb : plain_stage_blocks(NV, sizeof(T), FIELD);
  const size_t smem = (size_t)NV * stage * kPlainKB * sizeof(T) + (size_t)NV * kTileL * sizeof(PlainSum<T>) +
                      (size_t)t.max_nkb * (kPlainKB * sizeof(T) / 128) * sizeof(long long) + NV * sizeof(PlainSum<T>);
  // (at most 64 KB staged, 8 KB of sums and 13 KB of steps: plain_limits)
  cudaError_t e = cudaFuncSetAttribute(los_plain_kernel<T, MC, FIELD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kDynSmem);
  if (e != cudaSuccess) return cuda_fail(e, "los_transfer: smem attribute");
  ProfScope prof(GCAMB_K_LOS_PLAIN, st);
  a.q0 = nk - 1;
  if (FIELD == kFieldTensor) a.lmin_or_round = g->lmin;
  if (FIELD == kFieldT) a.lmin_or_round = g->eps_cut > kRowCut ? kPlainKB * (int)sizeof(T) / 128 - 1 : 0;
  for (int m0 = 0; m0 < M; m0 += 65535 * MC) {
    a.M = M - m0 < 65535 * MC ? M - m0 : 65535 * MC;
    const dim3 grid(nlt * (kTileL / a.rows), nk, (a.M + MC - 1) / MC);
    const size_t si = (size_t)m0 * g->nk * g->ntau, so = (size_t)m0 * g->nk * g->nl;
    los_plain_kernel<T, MC, FIELD><<<grid, kPlainWarps * 32, smem, st>>>(
        static_cast<const T *>(t.d_data), S + si, ST ? ST + si : nullptr, D + so, DE ? DE + so : nullptr,
        DB ? DB + so : nullptr, a);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "los_transfer: launch");
  return GCAMB_OK;
}

// Limits of the path: the whole tau-prefix of a chunk of 1, 2, 4 (FP32 also 8)
// sources is at most 200 KB, and there are at most 65535 chunks.  The kernel stages
// 64 KB at a time and takes other chunks; what it would need is less.  The limits
// are part of the interface: a grid is refused or taken by its size alone.
static int plain_limits(const Table &t, int M, int mode) {
  const int mc = mode != GCAMB_PLAIN64 && M >= 8 ? 8 : (M >= 4 ? 4 : (M >= 2 ? 2 : 1));
  const size_t smem = (size_t)mc * t.max_nkb * kPlainKB * (mode == GCAMB_PLAIN64 ? 8 : 4);
  if (smem > 200 * 1024) return fail(GCAMB_EINVAL, "los_transfer: tau grid too long for the plain kernel");
  if ((M + mc - 1) / mc > 65535) return fail(GCAMB_EINVAL, "los_transfer: too many sources for one launch");
  return GCAMB_OK;
}

template <int FIELD>
static int launch_los_plain_f(const gcamb_grid *g, const void *S, int M, int mode, void *Delta, cudaStream_t st) {
  const Table &t = g->tab[mode];
  if (int rc = plain_limits(t, M, mode)) return rc;
  if (mode == GCAMB_PLAIN64) {
    auto s = static_cast<const double *>(S);
    auto d = static_cast<double *>(Delta);
    const int mc = plain_sources(g, t, M, 4);
    auto go = [&](auto c) {
      return launch_plain_t<double, decltype(c)::value, FIELD>(g, t, s, nullptr, M, d, nullptr, nullptr, g->nk, g->nlt,
                                                               st);
    };
    if (mc == 1) return go(std::integral_constant<int, 1>());
    if (mc == 2) return go(std::integral_constant<int, 2>());
    if (mc == 3) return go(std::integral_constant<int, 3>());
    return go(std::integral_constant<int, 4>());
  }
  auto s = static_cast<const float *>(S);
  auto d = static_cast<float *>(Delta);
  const int mc = plain_sources(g, t, M, 8);
  auto go = [&](auto c) {
    return launch_plain_t<float, decltype(c)::value, FIELD>(g, t, s, nullptr, M, d, nullptr, nullptr, g->nk, g->nlt, st);
  };
  switch (mc) {
    case 1: return go(std::integral_constant<int, 1>());
    case 2: return go(std::integral_constant<int, 2>());
    case 3: return go(std::integral_constant<int, 3>());
    case 4: return go(std::integral_constant<int, 4>());
    case 5: return go(std::integral_constant<int, 5>());
    case 6: return go(std::integral_constant<int, 6>());
    case 7: return go(std::integral_constant<int, 7>());
    default: return go(std::integral_constant<int, 8>());
  }
}

int launch_los_plain(const gcamb_grid *g, const void *S, int M, int mode, void *Delta, cudaStream_t st, bool emode) {
  return emode ? launch_los_plain_f<kFieldE>(g, S, M, mode, Delta, st)
               : launch_los_plain_f<kFieldT>(g, S, M, mode, Delta, st);
}

// Tensor modes, one launch: D0, D1, D2 of S_P and the x^-2 sum of S_T share
// each table load, and each CTA combines its rows (with the row before its
// first):
//   Delta_T[l] = c_l (x^-2 sum of S_T) + the l = 2 tail
//   Delta_E[l] = l (l-1) D2[l] - 2 D0[l] + 2 D1[l-1] + tail_e(l)
//   Delta_B[l] = 2 D0[l-1] - 2 (l-1) D1[l] + tail_b(l)
// Row l-1 of the first multipole (lmin >= 2) comes from the recurrence
// j_(l-1) = (2l+1)/x j_l - j_(l+1):  D1[l-1] = (2l+1) D2[l] - D1[l+1],
// D0[l-1] = (2l+1) D1[l] - D0[l+1] (all three sums leave out the same nodes).
// The tails add, for l = 2..5, the series terms of the nodes below the cut.
int launch_los_tensor(const gcamb_grid *g, const void *ST, const void *SP, int M, int mode, void *DT, void *DE,
                      void *DB, cudaStream_t st) {
  if (g->lsampled)
    return fail(GCAMB_EUNSUPPORTED, "los_transfer_tensor: the kernels take row l-1: needs a grid of every multipole");
  if (g->lmin >= 2 && g->lmax == g->lmin)
    return fail(GCAMB_EINVAL, "los_transfer_tensor: needs lmax > lmin when lmin >= 2 (the kernels take j_(l-1))");
  double x_lo = 1e-12;
  if (emode_x_lo(g, &x_lo)) return fail(GCAMB_EINVAL, "los_transfer_tensor: eps_cut too large for the l = 2 limit");
  if ((size_t)M * g->nk > 0x7fffffffULL) return fail(GCAMB_EINVAL, "los_transfer_tensor: too many rows");
  const Table &t = g->tab[mode];
  if (int rc = plain_limits(t, M, mode)) return rc;
  auto go = [&](auto v, auto c) {
    using T = decltype(v);
    return launch_plain_t<T, decltype(c)::value, kFieldTensor>(
        g, t, static_cast<const T *>(SP), static_cast<const T *>(ST), M, static_cast<T *>(DT), static_cast<T *>(DE),
        static_cast<T *>(DB), g->nk, g->nlt, st);
  };
  if (mode == GCAMB_PLAIN64) return go(0.0, std::integral_constant<int, 1>());
  return M >= 2 ? go(0.f, std::integral_constant<int, 2>()) : go(0.f, std::integral_constant<int, 1>());
}

// C^XY_l[m] = 4 pi sum_k w_k P[m][k] DX[m][k][l] DY[m][k][l] in FP64 (kCross;
// else Y = X and only DX is read).  kPrefix (the uneven FP32 plan): source
// m0 + m of the chunk on its own k prefix [0, nk_m) with the trapezoid in ln k
// of that prefix (the last node of a shorter prefix takes half its interval)
// and zero above its own l_max; rows of DX beyond the prefix are not read.
//
// A serial walk over k by one thread per (m, l) is bound by the latency of
// its loads (l_max = 5000, 3000 k, one model: 1097 us for 120 MB).  Here the
// k range is cut into kClParts contiguous parts, summed in eight groups of
// eight: a warp sums one part (or 2, 4, 8 of them in turn) for 32 adjacent
// multipoles with eight loads in flight; the CTAs of a cluster (grid y) share
// out the groups and the first one adds the eight group sums it gets through
// distributed shared memory.  The order of the additions is fixed by nk
// alone: it does not depend on the cluster size, the batch or the block.  The
// weight 4 pi w_k P is formed once per (k, CTA), not per element, which leaves
// two FP64 operations an element (GB300's FP64 pipe runs at 1/64 of the FP32
// one).  Measured, one model: l_max 5000 x 3000 k 1097 -> 68 us, l_max 500 x
// 300 k 116 -> 7.8 us; cross spectra, l_max 1500 x 1000 k 528 -> 11.9 us.
constexpr int kClParts = 64, kClGroups = 8;
enum ClKind { kAuto = 0, kCross = 1, kPrefix = 2 };

struct ClPrefix {
  const double *kk;
  const int *lrow, *lmax_m, *nk_m;
  int m0;
};

template <typename TD, int KIND>
__global__ void __launch_bounds__(256) cl_sum_kernel(const TD *__restrict__ DX, const TD *__restrict__ DY,
                                                     const double *__restrict__ Pk, const double *__restrict__ wk,
                                                     int nk, int nl, double *__restrict__ Cl, ClPrefix px) {
  __shared__ double fw[8][32];               // weights of a warp's next 32 k
  __shared__ double part[kClParts][32];      // this CTA's parts (the first kClParts / cluster size rows)
  __shared__ double gsum[kClGroups][32];     // the first CTA of the cluster: every group's sum
  const int cs = gridDim.y, rank = blockIdx.y;  // cluster size (1, 2, 4, 8) and rank: the cluster spans grid y
  // the first CTA's shared memory is written below: every CTA tells that it runs,
  // the wait for all of them stands before the write, behind the sums
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");  // all that earlier kernels wrote
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = blockIdx.x * 32 + lane;
  const size_t m = blockIdx.z;                            // source within DX
  const size_t mg = KIND == kPrefix ? px.m0 + m : m;      // source within Pk and Cl
  const TD *dx = DX + m * nk * nl + l, *dy = DY + m * nk * nl + l;
  const double *p = Pk + mg * nk;
  const double four_pi = 4.0 * 3.14159265358979323846;
  const int nkm = KIND == kPrefix ? px.nk_m[mg] : nk;
  const bool live = l < nl && (KIND != kPrefix || px.lrow[l] <= px.lmax_m[mg]);
  const int pc = (nk + kClParts - 1) / kClParts;  // k per part
  const int ppw = 8 / cs;                         // parts per warp
  for (int j = 0; j < ppw; ++j) {
    const int lp = warp * ppw + j;  // part within the CTA
    const int qb = min(nkm, (rank * (kClParts / cs) + lp) * pc), qe = min(nkm, qb + pc);
    double acc = 0.0;
    for (int q0 = qb; q0 < qe; q0 += 32) {
      __syncwarp();
      const int q = q0 + lane;
      if (q < qe) {
        double w = wk[q];
        if (KIND == kPrefix && nkm < nk && q + 1 == nkm) w = q > 0 ? 0.5 * (log(px.kk[q]) - log(px.kk[q - 1])) : 0.0;
        fw[warp][lane] = four_pi * w * p[q];
      }
      __syncwarp();
      const int n = min(32, qe - q0);
      if (live) {
#pragma unroll 1
        for (int i = 0; i < n; i += 8) {
          TD x[8], y[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const size_t o = (size_t)(q0 + i + u) * nl;
            x[u] = i + u < n ? dx[o] : TD(0);
            if constexpr (KIND == kCross) y[u] = i + u < n ? dy[o] : TD(0);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (i + u < n) acc = fma(fw[warp][i + u], (double)x[u] * (double)(KIND == kCross ? y[u] : x[u]), acc);
        }
      }
    }
    part[lp][lane] = acc;
  }
  __syncthreads();
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  const int ng = kClGroups / cs;  // groups of this CTA
  if (warp < ng) {
    double s = part[warp * 8][lane];
#pragma unroll
    for (int j = 1; j < 8; ++j) s += part[warp * 8 + j][lane];
    // into the first CTA's gsum
    uint32_t dst = (uint32_t)__cvta_generic_to_shared(&gsum[rank * ng + warp][lane]);
    asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, 0;\n\tst.shared::cluster.f64 [a], %1;\n\t}\n" ::"r"(dst),
                 "d"(s)
                 : "memory");
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (rank == 0 && warp == 0 && l < nl) {
    double s = gsum[0][lane];
#pragma unroll
    for (int g = 1; g < kClGroups; ++g) s += gsum[g][lane];
    Cl[mg * nl + l] = s;
  }
}

template <typename TD, int KIND>
static cudaError_t launch_cl_sum(const gcamb_grid *g, const void *DX, const void *DY, const double *Pk, int M,
                                 double *Cl, cudaStream_t st, const ClPrefix &px = ClPrefix()) {
  if (cudaError_t e = cudaGetLastError()) return e;  // a launch before this one
  // cluster size: the smallest that gives every SM six CTAs of 256 threads
  // (of the eight that fit), up to the portable eight: with one model even
  // l_max = 5000 has only 157 blocks of 32 multipoles
  const unsigned lb = (unsigned)((g->nl + 31) / 32);
  unsigned cs = 1;
  while (cs < 8 && (size_t)lb * M * cs < kSms * 6) cs *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(lb, cs, (unsigned)M);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[2]{};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = cs;
  at[0].val.clusterDim.z = 1;
  // behind the transfer functions' kernel: its launch is done as that one ends
  // (not in a caller's capture, where what precedes need not be a kernel)
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const bool known = cudaStreamIsCapturing(st, &cap) == cudaSuccess;
  if (!known) cudaGetLastError();  // another stream's capture: the query's own error
  const bool plain_stream = known && cap == cudaStreamCaptureStatusNone;
  cfg.attrs = at;
  cfg.numAttrs = plain_stream ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, cl_sum_kernel<TD, KIND>, static_cast<const TD *>(DX), static_cast<const TD *>(DY),
                            Pk, static_cast<const double *>(g->d_wk), g->nk, g->nl, Cl, px);
}

int launch_cl_cross(const gcamb_grid *g, const void *DX, const void *DY, int d_dtype, const double *Pk, int M,
                    double *Cl, cudaStream_t st) {
  if (M > 65535) return fail(GCAMB_EINVAL, "cl_cross: too many sources for one launch");
  ProfScope prof(GCAMB_K_CL, st);
  cudaError_t e = d_dtype == GCAMB_F64 ? launch_cl_sum<double, kCross>(g, DX, DY, Pk, M, Cl, st)
                                       : launch_cl_sum<float, kCross>(g, DX, DY, Pk, M, Cl, st);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "cl_cross: launch");
  return GCAMB_OK;
}

// Sources per launch pair of the FP32 plan (the Delta buffer of a chunk).
constexpr int kPlainChunk = 16;

size_t plain_plan_workspace_bytes(const gcamb_grid *g, int M) {
  const int mc = M < kPlainChunk ? M : kPlainChunk;
  return (size_t)(mc > 0 ? mc : 1) * g->nk * g->nl * sizeof(float);
}

int launch_plain_plan(const gcamb_grid *g, const float *S, const double *Pk, int M, const int *lmax_c,
                      const int *nk_c, const int *d_lmax, const int *d_nk, double *Cl, void *ws, cudaStream_t st) {
  const Table &t = g->tab[GCAMB_PLAIN32];
  float *D = static_cast<float *>(ws);
  for (int m0 = 0; m0 < M; m0 += kPlainChunk) {
    const int mc = M - m0 < kPlainChunk ? M - m0 : kPlainChunk;
    // the chunk's longest k prefix and highest l-tile (host copies of the plan)
    int nkc = 1, ltc = 0;
    for (int j = m0; j < m0 + mc; ++j) {
      nkc = nk_c[j] > nkc ? nk_c[j] : nkc;
      int r = g->rowof[lmax_c[j] - g->lmin];
      for (int l = lmax_c[j]; r < 0 && l > g->lmin; --l) r = g->rowof[l - 1 - g->lmin];
      const int lt = (r < 0 ? 0 : r) / kTileL;
      ltc = lt > ltc ? lt : ltc;
    }
    if ((size_t)8 * t.max_nkb * kPlainKB * sizeof(float) > 200 * 1024)
      return fail(GCAMB_EINVAL, "plan_launch: tau grid too long for the plain kernel");
    const float *Sc = S + (size_t)m0 * g->nk * g->ntau;
    if (int rc = launch_plain_t<float, 8, kFieldT>(g, t, Sc, nullptr, mc, D, nullptr, nullptr, nkc, ltc + 1, st))
      return rc;
    cudaError_t e = cudaSuccess;
    {
      ProfScope prof(GCAMB_K_CL, st);
      e = launch_cl_sum<float, kPrefix>(g, D, D, Pk, mc, Cl, st, ClPrefix{g->d_k, g->d_lrow, d_lmax, d_nk, m0});
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "plan_launch: FP32 launch");
  }
  return GCAMB_OK;
}

int launch_cl(const gcamb_grid *g, const void *Delta, int d_dtype, const double *Pk, int M, double *Cl,
              cudaStream_t st) {
  if (M > 65535) return fail(GCAMB_EINVAL, "cl: too many sources for one launch");
  ProfScope prof(GCAMB_K_CL, st);
  cudaError_t e = d_dtype == GCAMB_F64 ? launch_cl_sum<double, kAuto>(g, Delta, Delta, Pk, M, Cl, st)
                                       : launch_cl_sum<float, kAuto>(g, Delta, Delta, Pk, M, Cl, st);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "cl: launch");
  return GCAMB_OK;
}

}  // namespace gcamb
