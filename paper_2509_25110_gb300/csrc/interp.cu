// Source interpolation onto the transfer k grid (the step that prepares the
// sources before the projection, Sec. 3.3): the natural cubic spline in k of
// every (source, tau) column.  On nodes k_0 < ... < k_(n-1), h_j = k_(j+1) - k_j,
// the second derivatives solve the tridiagonal system
//   h_(j-1) M_(j-1) + 2 (h_(j-1) + h_j) M_j + h_j M_(j+1)
//       = 6 [(y_(j+1) - y_j)/h_j - (y_j - y_(j-1))/h_(j-1)],   0 < j < n-1,
// with M_0 = M_(n-1) = 0; on [k_j, k_(j+1)], t = (k - k_j)/h_j,
//   y = (1-t) y_j + t y_(j+1) + h_j^2/6 [((1-t)^3 - (1-t)) M_j + (t^3 - t) M_(j+1)]
// (the cubic factors are evaluated in their factored forms, which do not
// cancel next to a node).
// The elimination coefficients and 1/h depend on the k nodes only and are
// formed on the host.  The arithmetic is that of the sources: FP64 for FP64
// sources, FP32 for FP32 sources (the GPU's FP64 rate would make the FP32 case
// ALU-bound).
//
// FP32: one kernel solves and evaluates, marching up the nodes
// (spline_march_kernel).  FP64, and FP32 nodes so uneven that a segment's
// neighbourhood does not decide its second derivatives (seg_halo_ok): one
// thread per (source, tau) column runs the forward sweep and the back
// substitution over all nodes (reads along k are coalesced across tau), then
// one thread per output element evaluates the spline.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "internal.h"

namespace gcamb {

namespace {

// Node coefficients of one precision: h, 1/h, c', 1/den (each [n]).
template <typename A>
struct NodeCoef {
  const A *h, *ih, *cp, *inv;
};

// Per column: d'_j = (r_j - h_(j-1) d'_(j-1)) / den_j, M_j = d'_j - c'_j M_(j+1).
template <typename T, typename A>
__global__ void __launch_bounds__(256) spline_solve_kernel(const T *__restrict__ y, NodeCoef<A> c, int n, int ntau,
                                                           int M, A *__restrict__ Md) {
  const size_t col = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // m * ntau + tau
  if (col >= (size_t)M * ntau) return;
  const size_t m = col / ntau, t = col - m * ntau;
  const T *yc = y + m * (size_t)n * ntau + t;
  A *mc = Md + m * (size_t)n * ntau + t;
  mc[0] = A(0);
  mc[(size_t)(n - 1) * ntau] = A(0);
  if (n < 3) return;
  A y0 = (A)yc[0], y1 = (A)yc[ntau];
  A s0 = (y1 - y0) * c.ih[0];  // slope of the previous interval
  A dprev = A(0);
#pragma unroll 8
  for (int j = 1; j < n - 1; ++j) {
    const A y2 = (A)yc[(size_t)(j + 1) * ntau];
    const A s1 = (y2 - y1) * c.ih[j];
    const A r = A(6) * (s1 - s0);
    const A d = (r - (j > 1 ? c.h[j - 1] * dprev : A(0))) * c.inv[j];
    mc[(size_t)j * ntau] = d;
    dprev = d;
    y1 = y2;
    s0 = s1;
  }
  A next = A(0);  // M_(n-1)
#pragma unroll 8
  for (int j = n - 2; j >= 1; --j) {
    const A v = mc[(size_t)j * ntau] - c.cp[j] * next;
    mc[(size_t)j * ntau] = v;
    next = v;
  }
}

// Blocks: x = (block of kQB output nodes) * ntc + (tau chunk of 256),
// y = source; tau is the fastest index, so loads and stores are coalesced.
// Each thread walks kQB consecutive output nodes of its column and reloads
// the interval's y and M only when the interval changes.
constexpr int kQB = 64;

// An output node's factors: y = u y_j + s y_(j+1) + a M_j + b M_(j+1),
// s = (k - k_j)/h, u = 1 - s, a = -h^2/6 s u (1 + u), b = -h^2/6 s u (1 + s)
// (u^3 - u = -s u (1 + u) and s^3 - s = -s u (1 + s): no cancellation near the
// nodes), each rounded once from FP64.
template <typename A>
struct __align__(4 * sizeof(A)) OutCoef {
  A s, u, a, b;
};

// V adjacent columns of a thread, loaded and stored together.
template <int V, typename T = float>
struct __align__(sizeof(T) * V) FV {
  T e[V];
};

template <typename T, int V>
__global__ void __launch_bounds__(256) spline_eval_kernel(const T *__restrict__ y, const T *__restrict__ Md,
                                                          const int *__restrict__ jq,
                                                          const OutCoef<T> *__restrict__ qc, int n, int nq, int ntau,
                                                          int ntc, T *__restrict__ out) {
  const int qb = (int)(blockIdx.x / (unsigned)ntc);
  const int t = ((int)(blockIdx.x - (unsigned)qb * ntc) * 256 + threadIdx.x) * V;
  if (t >= ntau) return;
  const size_t m = blockIdx.y;
  const int q0 = qb * kQB, q1 = min(nq, q0 + kQB);
  int jc = -1;
  FV<V, T> y0{}, y1{}, m0{}, m1{};
  for (int q = q0; q < q1; ++q) {
    const int j = jq[q];
    if (j != jc) {
      const size_t i0 = (m * (size_t)n + j) * ntau + t, i1 = i0 + ntau;
      y0 = *reinterpret_cast<const FV<V, T> *>(y + i0);
      y1 = *reinterpret_cast<const FV<V, T> *>(y + i1);
      m0 = *reinterpret_cast<const FV<V, T> *>(Md + i0);
      m1 = *reinterpret_cast<const FV<V, T> *>(Md + i1);
      jc = j;
    }
    const OutCoef<T> c = qc[q];
    FV<V, T> r;
#pragma unroll
    for (int v = 0; v < V; ++v)  // small terms first
      r.e[v] = fma(c.u, y0.e[v], fma(c.s, y1.e[v], fma(c.a, m0.e[v], c.b * m1.e[v])));
    *reinterpret_cast<FV<V, T> *>(out + (m * nq + q) * (size_t)ntau + t) = r;
  }
}

// FP32 sources: solve and evaluate in one pass.  A thread marches up the k
// nodes of its tau columns in segments of kSegT intervals: the forward sweep
// runs kSegH nodes ahead; the back substitution starts there, from zero,
// reaches the segment, and each interval's outputs follow as its two second
// derivatives are known.
//
// A value r_i changes d'_j of the forward sweep by the product of the factors
// h_(k-1)/den_k between them, and d'_i changes M_j of the back substitution by
// the product of the c'_k (0.27 a node on even nodes, at most 2/3 and 1/2 on
// any).  So kSegH nodes decide a second derivative: what is left out is below
// 2^-40 (2^-45 on even nodes) of the second derivative at that distance (the
// host checks the products, seg_halo_ok), that is below FP32's rounding of the
// values here unless those are less than 2^-16 of the ones 24 nodes away.  The k
// range is also cut into parts whose forward sweeps start kSegH nodes early, in
// the same way.  (32 nodes and 2^-54: 1512 -> 1596 us, small shapes up to 40%
// slower.)
//
// Bound by HBM: the sources are read once (1 GB of 256 x 1000 x 1000), the
// outputs written once (8.2 GB on 8000 nodes).  The columns' values arrive by
// asynchronous copies into a ring two segments ahead, the nodes' coefficients
// and the outputs' factors likewise (read from global memory where they are
// used, they missed the little L1 the rings leave: 2850 us).  The sweep over whole columns that this
// replaces wrote and read the second derivatives and was one serial chain of
// loads a column: 1099 us and 1585 us for the evaluation, now 1488 us (DRAM at
// 80% of its peak cycles).  (Segments
// solved by themselves, with both neighbourhoods loaded and swept for each:
// 1927 us at best.)
constexpr int kSegT = 8, kSegA = 3, kSegH = kSegA * kSegT;  // segment, segments ahead
constexpr int kYSlots = kSegA + 3, kDSlots = kSegA + 1;     // rings of segments: values, d'
constexpr int kSegPad = 2 * kSegH + 2 * kSegT;              // zero coefficients before and after the nodes'
constexpr int kCSlots = kYSlots + 1, kQSlots = 3;           // rings shared by the block: coefficients, output factors
constexpr int kSegQ = 96;                                   // output nodes staged per segment (more: read from global)
constexpr int kSegSmem = (kYSlots + kDSlots) * kSegT * 128 * 4 + kQSlots * kSegQ * 16 + kCSlots * kSegT * 16 +
                         kQSlots * (kSegT + 1) * 4;

struct __align__(16) SegCoef {
  float ih, hm, inv, cp;  // 1/h_j, h_(j-1), 1/den_j, c'_j (0 where the node has no equation)
};

// coef and qs start at node 0 (kSegPad zero coefficients before it; qs[j] = nq
// from the last node on, for kSegPad nodes).
template <int V>
__global__ void __launch_bounds__(128 / V) spline_march_kernel(const float *__restrict__ y,
                                                               const SegCoef *__restrict__ coef,
                                                               const int *__restrict__ qs,
                                                               const OutCoef<float> *__restrict__ qc,
                                                               const int4 *__restrict__ parts, int n, int nq,
                                                               int ntau, int ntc, float *__restrict__ out) {
  constexpr int NT = 128 / V, T = kSegT, A = kSegA;
  extern __shared__ __align__(16) float ring[];
  FV<V> *yr = reinterpret_cast<FV<V> *>(ring) + threadIdx.x;  // [slot][row]: stride NT
  FV<V> *dr = yr + kYSlots * T * NT;
  OutCoef<float> *qring = reinterpret_cast<OutCoef<float> *>(ring + (kYSlots + kDSlots) * T * 128);
  float4 *cring = reinterpret_cast<float4 *>(qring + kQSlots * kSegQ);      // ih, hm, inv, cp
  int *nring = reinterpret_cast<int *>(cring + kCSlots * T);                // first outputs of a segment's intervals
  const int part = (int)(blockIdx.x / (unsigned)ntc);
  const int t = (int)(blockIdx.x - (unsigned)part * ntc) * 128 + threadIdx.x * V;
  const bool live = t < ntau;
  const size_t m = blockIdx.y;
  const int4 pt = parts[part];  // segments [x, y), of their outputs [z, w)
  const int sa = pt.x, sb = pt.y;
  const float *src = y + m * (size_t)n * ntau + t;
  float *oc = out + m * (size_t)nq * ntau + t;
  auto yslot = [&](int seg) { return yr + (seg + kYSlots * 4) % kYSlots * (T * NT); };
  auto dslot = [&](int seg) { return dr + (seg + kDSlots * 4) % kDSlots * (T * NT); };
  auto cslot = [&](int seg) { return cring + (seg + kCSlots * 4) % kCSlots * T; };
  auto copy16 = [](void *to, const void *from) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from)
                 : "memory");
  };
  // values and coefficients of a segment
  auto load = [&](int seg) {
    if (live) {
      FV<V> *to = yslot(seg);
#pragma unroll
      for (int r = 0; r < T; ++r) {
        const float *p = src + (size_t)min(max(seg * T + r, 0), n - 1) * ntau;
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to + r * NT)),
                     "l"(p), "n"(4 * V)
                     : "memory");
      }
    }
    if (threadIdx.x < T) copy16(cslot(seg) + threadIdx.x, coef + seg * T + threadIdx.x);
  };
  const int s_first = sa - 2 * A;
  load(s_first + A);
  load(s_first + A + 1);
  asm volatile("cp.async.commit_group;" ::: "memory");
  int qa = 0, qb = 0;  // outputs of segment s + 1: [qa, qb)
  int qs1 = qs[max(s_first + 1, sa) * T];
  FV<V> s0{}, dp{};
  for (int s = s_first; s < sb; ++s) {
    // this iteration's copies: values two segments past the sweep, factors of the next segment's
    // outputs.  A slot was last read before the barrier of the iteration before.
    load(s + A + 2);
    const int qs0 = qs1;  // first output of segment s + 1 (from the part's first segment on)
    qs1 = __ldg(qs + max(s + 2, sa) * T);
    const int na = qa, nb = qb;  // this segment's
    qa = max(qs0, pt.z);
    qb = s + 1 >= sa ? max(qa, min(qs1, pt.w)) : qa;
    if (s + 1 >= sa) {
      OutCoef<float> *to = qring + (s + 1 + kQSlots) % kQSlots * kSegQ;
      if (qb - qa <= kSegQ)
        for (int i = threadIdx.x; i < qb - qa; i += NT) copy16(to + i, qc + qa + i);
      if (threadIdx.x <= T)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(
                         nring + (s + 1 + kQSlots) % kQSlots * (T + 1) + threadIdx.x)),
                     "l"(qs + (s + 1) * T + threadIdx.x)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 1;" ::: "memory");
    __syncthreads();  // the copies of the iteration before, all threads' (segments up to s + A + 1)
    if (!live) continue;
    {
      // forward sweep of segment s + A; nodes without an equation have zero coefficients, hence d' = 0
      const int f = s + A;
      const FV<V> *ya = yslot(f), *yb = yslot(f + 1);
      const float4 *cf = cslot(f);
      FV<V> *d = dslot(f);
      FV<V> y1 = ya[0];
#pragma unroll
      for (int r = 0; r < T; ++r) {
        const FV<V> y2 = r + 1 < T ? ya[(r + 1) * NT] : yb[0];
        const float4 k = cf[r];
        // the part's first node: the slope before it is not known, its equation is left out
        const bool lead = s == s_first && r == 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const float s1 = (y2.e[v] - y1.e[v]) * k.x;
          dp.e[v] = lead ? 0.f : (6.f * (s1 - s0.e[v]) - k.y * dp.e[v]) * k.z;
          s0.e[v] = s1;
        }
        d[r * NT] = dp;
        y1 = y2;
      }
    }
    if (s < sa) continue;
    // back substitution down to the segment
    FV<V> next{};
#pragma unroll
    for (int g = A; g >= 1; --g) {
      const FV<V> *d = dslot(s + g);
      const float4 *cf = cslot(s + g);
#pragma unroll
      for (int r = T - 1; r >= 0; --r) {
        const FV<V> x = d[r * NT];
#pragma unroll
        for (int v = 0; v < V; ++v) next.e[v] = x.e[v] - cf[r].w * next.e[v];
      }
    }
    const FV<V> *d = dslot(s), *ya = yslot(s);
    const float4 *cf = cslot(s);
    const OutCoef<float> *qst = qring + (s + kQSlots) % kQSlots * kSegQ;
    const int *nst = nring + (s + kQSlots) % kQSlots * (T + 1);
    const bool staged = nb - na <= kSegQ;
    FV<V> yn = yslot(s + 1)[0];
#pragma unroll
    for (int r = T - 1; r >= 0; --r) {
      const FV<V> x = d[r * NT], y0 = ya[r * NT];
      FV<V> cur;
#pragma unroll
      for (int v = 0; v < V; ++v) cur.e[v] = x.e[v] - cf[r].w * next.e[v];
      int q = max(nst[r], pt.z);
      const int q1 = min(nst[r + 1], pt.w);
      float *o = oc + (size_t)q * ntau;
      auto put = [&](const OutCoef<float> &w, float *op) {
        FV<V> z;
#pragma unroll
        for (int v = 0; v < V; ++v)
          z.e[v] = fmaf(w.u, y0.e[v], fmaf(w.s, yn.e[v], fmaf(w.a, cur.e[v], w.b * next.e[v])));  // small terms first
        if constexpr (V == 2) __stcs(reinterpret_cast<float2 *>(op), make_float2(z.e[0], z.e[1]));
        else __stcs(op, z.e[0]);
      };
      if (staged) {
        for (; q + 4 <= q1; q += 4) {
#pragma unroll
          for (int u = 0; u < 4; ++u) put(qst[q + u - na], o + (size_t)u * ntau);
          o += (size_t)4 * ntau;
        }
        for (; q < q1; ++q, o += ntau) put(qst[q - na], o);
      } else {
        for (; q + 4 <= q1; q += 4) {
          OutCoef<float> w[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) w[u] = qc[q + u];
#pragma unroll
          for (int u = 0; u < 4; ++u) put(w[u], o + (size_t)u * ntau);
          o += (size_t)4 * ntau;
        }
        for (; q < q1; ++q, o += ntau) put(qc[q], o);
      }
      next = cur;
      yn = y0;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

// Workspace regions (each 256-byte aligned): node coefficients [4][n], each
// output node's factors [nq][4], its interval [nq] (int), the intervals' first
// outputs [n] (int): sized for FP64; the second derivatives [M][n][ntau] in the
// arithmetic's precision (sized for FP64).  One upload fills the regions
// before the derivatives.  The kernels read the regions by 16- and 32-byte
// loads, a workspace may have any alignment: the regions start at its first
// multiple of kInterpAlign, within the kInterpAlign bytes of slack in total.
constexpr size_t kInterpAlign = 256;

struct InterpLayout {
  size_t coef, q, qj, qs, md, total;
  InterpLayout(int M, int n, int ntau, int nq) {
    coef = 0;
    q = coef + a256(((size_t)n + kSegPad) * 4 * sizeof(double));
    qj = q + a256((size_t)nq * 4 * sizeof(double));
    qs = qj + a256((size_t)nq * sizeof(int));
    md = qs + a256(((size_t)n + kSegPad) * sizeof(int));
    total = md + a256((size_t)M * n * ntau * sizeof(double)) + kInterpAlign;
  }
};

// The regions up to the derivatives on the host, aligned as on the device.
struct alignas(kInterpAlign) HostBlock {
  char b[kInterpAlign];
};

template <typename T>
void launch_interp_columns(const InterpLayout &L, char *w, int n, int nq, int ntau, int M, const T *S_in, T *S_out,
                           cudaStream_t st) {
  const T *c = reinterpret_cast<const T *>(w + L.coef);
  NodeCoef<T> nc{c, c + n, c + 2 * n, c + 3 * n};
  T *Md = reinterpret_cast<T *>(w + L.md);
  const size_t cols = (size_t)M * ntau;
  const int nqb = (nq + kQB - 1) / kQB;
  spline_solve_kernel<T, T><<<(unsigned)((cols + 255) / 256), 256, 0, st>>>(S_in, nc, n, ntau, M, Md);
  auto eval = [&](auto v) {
    constexpr int V = decltype(v)::value;
    const int ntc = (ntau / V + 255) / 256;
    spline_eval_kernel<T, V><<<dim3((unsigned)((size_t)nqb * ntc), (unsigned)M), 256, 0, st>>>(
        S_in, Md, reinterpret_cast<const int *>(w + L.qj), reinterpret_cast<const OutCoef<T> *>(w + L.q), n, nq, ntau,
        ntc, S_out);
  };
  // FP32: four columns a thread in 16-byte loads and stores where the rows are aligned (Md's are)
  if (sizeof(T) == 4 && ntau % 4 == 0 &&
      (reinterpret_cast<uintptr_t>(S_in) | reinterpret_cast<uintptr_t>(S_out)) % 16 == 0)
    eval(std::integral_constant<int, sizeof(T) == 4 ? 4 : 1>());
  else
    eval(std::integral_constant<int, 1>());
}

// Whether kSegH nodes decide a second derivative: every product of kSegH - 1
// consecutive factors of either sweep is below 2^-40.  (The host
// needs logarithms of n factors; sums over the window slide.)
bool seg_halo_ok(const double *h, const double *cp, const double *inv, int n) {
  const double bound = -40.0 * 0.69314718055994530942;
  double fw = 0.0, bw = 0.0;
  std::vector<double> lf(n, -1e30), lb(n, -1e30);  // ends of the system: a factor of zero
  for (int j = 2; j < n - 1; ++j) lf[j] = std::log(h[j - 1] * inv[j]);
  for (int j = 1; j < n - 2; ++j) lb[j] = std::log(cp[j]);
  const int w = kSegH - 1;
  for (int j = 0; j < n; ++j) {
    double a = 0.0, b = 0.0;
    if (j + w > n) break;  // a shorter window reaches the system's end
    if (j == 0 || lf[j - 1] < -1e29 || lb[j - 1] < -1e29) {
      for (int i = j; i < j + w; ++i) {
        a += lf[i];
        b += lb[i];
      }
      fw = a;
      bw = b;
    } else {
      fw += lf[j + w - 1] - lf[j - 1];
      bw += lb[j + w - 1] - lb[j - 1];
    }
    if (fw > bound || bw > bound) return false;
  }
  return true;
}

// Parts of the march, {first segment, one past the last, first output, one past
// the last}, of about equal work t, counted in segments: kPartOuts outputs take
// about as long as a segment's sweep and back substitution.  A part's sweep
// starts 2 kSegA segments early, so `blocks` columns' parts take (2 kSegA + t)
// (1 + W / t) one after the other on the chip's places, W = all work / places;
// t = sqrt(2 kSegA W) is its least, and at least kPartMin.  Four blocks fit an
// SM, but W is reckoned with kPartPlaces = 5: parts a little finer leave fewer
// places idle at the end (four: 1512 -> 1533 us, 21 shapes 0.85 .. 1.17 of the
// speed, most of them below 1).  A segment with many outputs (nodes that are sparse where the grid
// is dense) is shared out by outputs; segments without any are left out where
// a part can start behind them.  Kernel time, parts of at least 16 whole
// segments -> these (nodes -> grid, tau, sources): 200 -> 8000, 300, 8: 582 ->
// 50 us; 395 -> 6075, 498, 15: 267 -> 67; 200 -> 1000, 300, 8: 59 -> 16;
// 518 -> 4312, 499, 155: 439 -> 415; 1000 -> 8000, 1000, 256: 1509 -> 1488.
constexpr int kPartOuts = 64, kPartMin = 4, kPartPlaces = 5;

std::vector<int4> march_parts(const int *qs, int n, int nq, size_t blocks) {
  const int nseg = (n - 2) / kSegT + 1;
  const double work = (nseg + (double)nq / kPartOuts) * (double)blocks / (kSms * kPartPlaces);
  const double target = std::max((double)kPartMin, std::sqrt(2.0 * kSegA * work));
  std::vector<int4> parts;
  int4 p{-1, 0, 0, 0};
  double c = 0.0;
  for (int s = 0, q = 0; s < nseg;) {
    const int q1 = s + 1 < nseg ? qs[(s + 1) * kSegT] : nq;
    if (p.x < 0) {
      if (q1 == q) {  // no outputs yet
        ++s;
        continue;
      }
      p = int4{s, 0, q, 0};
      c = 0.0;
    }
    const double room = (target - c - 1.0) * kPartOuts, segc = 1.0 + (double)(q1 - q) / kPartOuts;
    const bool last = s + 1 == nseg;
    // the whole segment (a small one is not split)
    if (q1 - q <= room || 4.0 * segc <= target || (c == 0.0 && q1 - q <= kPartOuts)) {
      c += segc;
      q = q1;
      ++s;
      if (!last && c < target) continue;
      p.y = s;
    } else if (room >= kPartOuts || c == 0.0) {  // as many of its outputs as fit
      q += std::max(kPartOuts, (int)room);
      p.y = s + 1;
    } else {  // up to the segment before
      p.y = s;
    }
    p.w = q;
    if (p.w > p.z) parts.push_back(p);
    p.x = -1;
  }
  return parts;
}

}  // namespace

size_t interp_workspace_bytes(int M, int nk_in, int ntau, int nk_out) {
  return InterpLayout(M, nk_in, ntau, nk_out).total;
}

int launch_interp_sources(const double *k_in, int nk_in, const void *S_in, int M, int ntau, int dtype,
                          const gcamb_grid *g, void *S_out, void *ws, size_t ws_bytes, cudaStream_t st) {
  const int n = nk_in, nq = g->nk;
  const InterpLayout L(M, n, ntau, nq);
  if (ws_bytes < L.total) return fail(GCAMB_EINVAL, "interp_sources: workspace too small");
  if ((size_t)nq * ((ntau + 255) / 256) > 0x7fffffffULL || M > 65535 || (size_t)M * ntau / 256 > 0x7fffffffULL)
    return fail(GCAMB_EINVAL, "interp_sources: too many sources or nodes for one launch");
  // elimination coefficients (nodes only) and each output node's interval
  std::vector<double> c64(4 * (size_t)n, 0.0);
  std::vector<OutCoef<double>> q64(nq);
  std::vector<HostBlock> blocks(L.md / kInterpAlign);  // zeros
  char *up = reinterpret_cast<char *>(blocks.data());
  int *qj = reinterpret_cast<int *>(up + L.qj), *qs = reinterpret_cast<int *>(up + L.qs);
  double *h = c64.data(), *ih = h + n, *cp = ih + n, *inv = cp + n;
  for (int j = 0; j + 1 < n; ++j) {
    h[j] = k_in[j + 1] - k_in[j];
    ih[j] = 1.0 / h[j];
  }
  for (int j = 1; j < n - 1; ++j) {
    const double b = 2.0 * (h[j - 1] + h[j]);
    const double den = b - (j > 1 ? h[j - 1] * cp[j - 1] : 0.0);
    inv[j] = 1.0 / den;
    cp[j] = (j < n - 2 ? h[j] : 0.0) * inv[j];
  }
  for (int q = 0, jn = 0; q < nq; ++q) {
    const double k = g->k[q];
    int j = (int)(std::upper_bound(k_in, k_in + n, k) - k_in) - 1;
    j = j < 0 ? 0 : (j > n - 2 ? n - 2 : j);
    qj[q] = j;
    // The weights of y_j and y_(j+1) add up to one in FP64, where u is no more exact
    // by itself (rounded by itself: error of random columns 7 .. 17% larger); rounded
    // to FP32 and in the cubic factors u is that of the upper node, exact near it.
    const double s = (k - k_in[j]) / h[j], u = (k_in[j + 1] - k) / h[j], f = -h[j] * h[j] / 6.0 * s * u;
    q64[q] = {s, dtype == GCAMB_F64 ? 1.0 - s : u, f * (1.0 + u), f * (1.0 + s)};
    for (; jn <= j; ++jn) qs[jn] = q;  // the grid's k rise: first output of interval jn
    if (q == nq - 1)
      for (; jn < n + kSegPad; ++jn) qs[jn] = nq;
  }
  // segments of intervals, and the parts of the k range
  const size_t nchunk = ((size_t)ntau + 127) / 128;
  std::vector<int4> parts;
  if (dtype == GCAMB_F32) parts = march_parts(qs, n, nq, nchunk * M);
  const bool seg = dtype == GCAMB_F32 && parts.size() * nchunk <= 0x7fffffffULL && seg_halo_ok(h, cp, inv, n);
  if (dtype == GCAMB_F64) {
    std::copy(c64.begin(), c64.end(), reinterpret_cast<double *>(up + L.coef));
    std::copy(q64.begin(), q64.end(), reinterpret_cast<OutCoef<double> *>(up + L.q));
  } else {
    if (seg) {
      SegCoef *sc = reinterpret_cast<SegCoef *>(up + L.coef) + kSegPad;  // zeros around
      for (int j = 0; j < n; ++j)
        sc[j] = SegCoef{(float)ih[j], j > 0 ? (float)h[j - 1] : 0.f, (float)inv[j], (float)cp[j]};
    } else {
      std::copy(c64.begin(), c64.end(), reinterpret_cast<float *>(up + L.coef));
    }
    OutCoef<float> *qc = reinterpret_cast<OutCoef<float> *>(up + L.q);
    for (int q = 0; q < nq; ++q) qc[q] = {(float)q64[q].s, (float)q64[q].u, (float)q64[q].a, (float)q64[q].b};
    // the parts (at most nq) behind the factors, whose region is sized for FP64's
    if (seg) std::copy(parts.begin(), parts.end(), reinterpret_cast<int4 *>(qc + nq));
  }
  char *w = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(ws) + kInterpAlign - 1) & ~(uintptr_t)(kInterpAlign - 1));
  // a pageable copy returns once the host data is staged
  cudaError_t e = cudaMemcpyAsync(w, up, L.md, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_fail(e, "interp_sources: coefficient upload");
  ProfScope prof(GCAMB_K_INTERP, st);
  if (dtype == GCAMB_F64)
    launch_interp_columns<double>(L, w, n, nq, ntau, M, static_cast<const double *>(S_in), static_cast<double *>(S_out),
                                  st);
  else if (seg) {
    auto go = [&](auto v) {
      constexpr int V = decltype(v)::value;
      const auto *qc = reinterpret_cast<const OutCoef<float> *>(w + L.q);
      spline_march_kernel<V><<<dim3((unsigned)(parts.size() * nchunk), (unsigned)M), 128 / V, kSegSmem, st>>>(
          static_cast<const float *>(S_in), reinterpret_cast<const SegCoef *>(w + L.coef) + kSegPad,
          reinterpret_cast<const int *>(w + L.qs), qc, reinterpret_cast<const int4 *>(qc + nq), n, nq, ntau, (int)nchunk,
          static_cast<float *>(S_out));
    };
    if (ntau % 2 == 0 && (reinterpret_cast<uintptr_t>(S_in) | reinterpret_cast<uintptr_t>(S_out)) % 8 == 0)
      go(std::integral_constant<int, 2>());
    else
      go(std::integral_constant<int, 1>());
  } else
    launch_interp_columns<float>(L, w, n, nq, ntau, M, static_cast<const float *>(S_in), static_cast<float *>(S_out),
                                 st);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "interp_sources: launch");
  return GCAMB_OK;
}

namespace {

// C_l on every multipole from a grid of sampled multipoles: the natural cubic
// spline in l of D_l = l (l+1) C_l through the sampled rows; sampled
// multipoles are copied.  The elimination coefficients depend on the sampled
// multipoles only and come from the host (no divisions on the device); one
// thread per model runs the FP64 sweep over the nl samples ...
__global__ void cl_spline_solve_kernel(const double *__restrict__ Cs, const int *__restrict__ lrow,
                                       const double *__restrict__ h, const double *__restrict__ ih,
                                       const double *__restrict__ cp, const double *__restrict__ inv, int nl, int M,
                                       double *__restrict__ Md) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M) return;
  const double *c = Cs + (size_t)m * nl;
  double *mm = Md + (size_t)m * nl;
  mm[0] = 0.0;
  mm[nl - 1] = 0.0;
  if (nl < 3) return;
  auto D = [&](int j) { const double l = __ldg(lrow + j); return l * (l + 1.0) * __ldg(c + j); };
  double y1 = D(1);
  double s0 = (y1 - D(0)) * ih[0];
  double dprev = 0.0;
#pragma unroll 8
  for (int j = 1; j < nl - 1; ++j) {
    const double y2 = D(j + 1);
    const double s1 = (y2 - y1) * ih[j];
    const double d = (6.0 * (s1 - s0) - (j > 1 ? h[j - 1] * dprev : 0.0)) * inv[j];
    mm[j] = d;
    dprev = d;
    y1 = y2;
    s0 = s1;
  }
  double next = 0.0;
#pragma unroll 8
  for (int j = nl - 2; j >= 1; --j) {
    const double v = mm[j] - cp[j] * next;
    mm[j] = v;
    next = v;
  }
}

// ... and one thread per (model, l) evaluates, with each output multipole's
// bracketing samples (lo, lo+1) and position s from the host.
__global__ void cl_spline_eval_kernel(const double *__restrict__ Cs, const double *__restrict__ Md,
                                      const int *__restrict__ lrow, const int *__restrict__ rowof,
                                      const int *__restrict__ jl, const double *__restrict__ sl, int nl, int lmin,
                                      int nout, int M, double *__restrict__ out) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (size_t)M * nout) return;
  const int m = (int)(e / nout), i = (int)(e - (size_t)m * nout);
  const int l = lmin + i;
  const double *c = Cs + (size_t)m * nl;
  const int own = rowof[i];
  if (own >= 0) {
    out[e] = c[own];
    return;
  }
  const int lo = jl[i];
  const double l0 = lrow[lo], l1 = lrow[lo + 1], h = l1 - l0;
  const double s = sl[i], u = 1.0 - s, su = s * u;
  const double y0 = l0 * (l0 + 1.0) * c[lo], y1 = l1 * (l1 + 1.0) * c[lo + 1];
  const double *mm = Md + (size_t)m * nl;
  const double d = u * y0 + s * y1 - h * h / 6.0 * su * ((1.0 + u) * mm[lo] + (1.0 + s) * mm[lo + 1]);
  out[e] = d / ((double)l * (l + 1.0));
}

// The same in one block per model for up to kSmemSamples samples: the
// model's D_l and the coefficients are staged in shared memory, thread 0
// sweeps there (no global-memory latency in the chain), then the block
// evaluates the model's multipoles.
constexpr int kSmemSamples = 4000;

__global__ void __launch_bounds__(256) cl_spline_block_kernel(const double *__restrict__ Cs,
                                                              const int *__restrict__ lrow,
                                                              const int *__restrict__ rowof,
                                                              const double *__restrict__ coef,
                                                              const int *__restrict__ jl,
                                                              const double *__restrict__ sl, int nl, int lmin,
                                                              int nout, double *__restrict__ out) {
  extern __shared__ double sh[];
  double *y = sh, *mm = y + nl, *h = mm + nl, *ih = h + nl, *cp = ih + nl, *inv = cp + nl;
  const int m = blockIdx.x;
  const double *c = Cs + (size_t)m * nl;
  for (int j = threadIdx.x; j < nl; j += blockDim.x) {
    const double l = lrow[j];
    y[j] = l * (l + 1.0) * c[j];
    h[j] = coef[j];
    ih[j] = coef[nl + j];
    cp[j] = coef[2 * nl + j];
    inv[j] = coef[3 * nl + j];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    mm[0] = 0.0;
    mm[nl - 1] = 0.0;
    if (nl >= 3) {
      double s0 = (y[1] - y[0]) * ih[0], dprev = 0.0;
      for (int j = 1; j < nl - 1; ++j) {
        const double s1 = (y[j + 1] - y[j]) * ih[j];
        const double d = (6.0 * (s1 - s0) - (j > 1 ? h[j - 1] * dprev : 0.0)) * inv[j];
        mm[j] = d;
        dprev = d;
        s0 = s1;
      }
      double next = 0.0;
      for (int j = nl - 2; j >= 1; --j) {
        next = mm[j] - cp[j] * next;
        mm[j] = next;
      }
    }
  }
  __syncthreads();
  double *o = out + (size_t)m * nout;
  for (int i = threadIdx.x; i < nout; i += blockDim.x) {
    const int own = rowof[i];
    if (own >= 0) {
      o[i] = c[own];
      continue;
    }
    const int l = lmin + i, lo = jl[i];
    const double hh = h[lo], s = sl[i], u = 1.0 - s, su = s * u;
    const double d = u * y[lo] + s * y[lo + 1] - hh * hh / 6.0 * su * ((1.0 + u) * mm[lo] + (1.0 + s) * mm[lo + 1]);
    o[i] = d / ((double)l * (l + 1.0));
  }
}

// Up to kPcrSamples samples: the second derivatives by parallel cyclic
// reduction.  Stage s adds multiples of the equations s = 1, 2, 4, ... away that
// cancel the neighbours, the factors (of the nodes alone) from the host:
//   d_j <- d_j + alpha_j d_(j-s) + gamma_j d_(j+s),  M_j = d_j / b_j at the end.
// log2(nl) steps of two FP64 multiply-adds a thread instead of a serial sweep
// of 2 nl steps, each several dependent FP64 operations long: 130 samples, one
// model 64 -> 11 us (cold caches).
constexpr int kPcrSamples = 1024;

int pcr_stages(int nl) {
  int k = 0;
  while ((1 << k) < nl - 2) ++k;
  return k;
}

__global__ void __launch_bounds__(256) cl_spline_pcr_kernel(const double *__restrict__ Cs, const int *__restrict__ lrow,
                                                            const int *__restrict__ rowof,
                                                            const double *__restrict__ ih,
                                                            const double *__restrict__ fac, int stages,
                                                            const int *__restrict__ jl, const double *__restrict__ sl,
                                                            int nl, int lmin, int nout, double *__restrict__ out) {
  __shared__ double y[kPcrSamples], da[kPcrSamples], db[kPcrSamples];
  const int m = blockIdx.x;
  const double *c = Cs + (size_t)m * nl;
  for (int j = threadIdx.x; j < nl; j += blockDim.x) {
    const double l = lrow[j];
    y[j] = l * (l + 1.0) * c[j];
  }
  __syncthreads();
  for (int j = threadIdx.x; j < nl; j += blockDim.x)
    da[j] = j > 0 && j < nl - 1 ? 6.0 * ((y[j + 1] - y[j]) * ih[j] - (y[j] - y[j - 1]) * ih[j - 1]) : 0.0;
  double *d = da, *dn = db;
  for (int s = 0; s < stages; ++s) {
    __syncthreads();
    const double *al = fac + (size_t)2 * s * nl, *ga = al + nl;
    for (int j = threadIdx.x; j < nl; j += blockDim.x) {
      double v = d[j];
      if (j >= (1 << s)) v = fma(al[j], d[j - (1 << s)], v);
      if (j + (1 << s) < nl) v = fma(ga[j], d[j + (1 << s)], v);
      dn[j] = v;
    }
    double *t = d;
    d = dn;
    dn = t;
  }
  __syncthreads();
  const double *ib = fac + (size_t)2 * stages * nl;  // 1 / b, zero at both ends
  for (int j = threadIdx.x; j < nl; j += blockDim.x) d[j] *= ib[j];
  __syncthreads();
  double *o = out + (size_t)m * nout;
  // grid y shares out the outputs (each block repeats the reduction, which is
  // small against them: FP64 on one SM took most of the time)
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < nout; i += gridDim.y * blockDim.x) {
    const int own = rowof[i];
    if (own >= 0) {
      o[i] = c[own];
      continue;
    }
    const int l = lmin + i, lo = jl[i];
    const double hh = (double)(lrow[lo + 1] - lrow[lo]), s = sl[i], u = 1.0 - s, su = s * u;
    const double v = u * y[lo] + s * y[lo + 1] - hh * hh / 6.0 * su * ((1.0 + u) * d[lo] + (1.0 + s) * d[lo + 1]);
    o[i] = v / ((double)l * (l + 1.0));
  }
}

size_t al(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

// Coefficients: [h, 1/h, c', 1/den], or (up to kPcrSamples samples) [h, 1/h]
// and the reduction's factors.
static size_t cl_interp_coefs(int nl) {
  return (nl <= kPcrSamples ? 2 + 2 * (size_t)pcr_stages(nl) + 1 : 4) * (size_t)nl;
}

// Workspace: coefficients (doubles) | [s] (nout doubles) | [lo] (nout ints) |
// second derivatives [M][nl] (doubles).
size_t cl_interp_workspace_bytes(const gcamb_grid *g, int M) {
  const size_t nout = (size_t)(g->lmax - g->lmin + 1);
  return al(cl_interp_coefs(g->nl) * sizeof(double)) + al(nout * sizeof(double)) + al(nout * sizeof(int)) +
         al((size_t)M * g->nl * sizeof(double));
}

}  // namespace gcamb

using namespace gcamb;

extern "C" {

int gcamb_cl_interp_workspace(const gcamb_grid *g, int M, size_t *bytes) {
  if (!g || !bytes || M < 0) return fail(GCAMB_EINVAL, "cl_interp_workspace: bad argument");
  *bytes = cl_interp_workspace_bytes(g, M);
  return GCAMB_OK;
}

int gcamb_cl_interp(const gcamb_grid *g, const double *Cl_s, int M, double *Cl, void *ws, size_t ws_bytes,
                    void *stream) {
  if (!g) return fail(GCAMB_EINVAL, "cl_interp: NULL grid");
  if (M < 0) return fail(GCAMB_EINVAL, "cl_interp: M < 0");
  if (M == 0) return GCAMB_OK;
  if (!Cl_s || !Cl || !ws) return fail(GCAMB_EINVAL, "cl_interp: NULL pointer");
  if (ws_bytes < cl_interp_workspace_bytes(g, M)) return fail(GCAMB_EINVAL, "cl_interp: workspace too small");
  if (int rc = ensure_device_grid(const_cast<gcamb_grid *>(g))) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const int nl = g->nl, nout = g->lmax - g->lmin + 1;
  const bool pcr = nl <= kPcrSamples;
  const size_t ncoef = cl_interp_coefs(nl);
  const size_t o1 = al(ncoef * sizeof(double)), o2 = o1 + al((size_t)nout * sizeof(double));
  const size_t o3 = o2 + al((size_t)nout * sizeof(int));
  std::vector<char> up(o3, 0);  // coefficients, s, lo in one upload
  double *coef = reinterpret_cast<double *>(up.data()), *sv = reinterpret_cast<double *>(up.data() + o1);
  int *jv = reinterpret_cast<int *>(up.data() + o2);
  double *h = coef, *ih = h + nl;
  for (int j = 0; j + 1 < nl; ++j) {
    h[j] = (double)(g->lrow[j + 1] - g->lrow[j]);
    ih[j] = 1.0 / h[j];
  }
  const int stages = pcr ? pcr_stages(nl) : 0;
  if (pcr) {
    std::vector<double> A(nl, 0.0), B(nl, 1.0), C(nl, 0.0), An(nl), Bn(nl), Cn(nl);
    for (int j = 1; j < nl - 1; ++j) {
      A[j] = j > 1 ? h[j - 1] : 0.0;
      B[j] = 2.0 * (h[j - 1] + h[j]);
      C[j] = j < nl - 2 ? h[j] : 0.0;
    }
    for (int s = 0; s < stages; ++s) {
      double *fa = coef + (2 + 2 * (size_t)s) * nl, *fg = fa + nl;
      const int w = 1 << s;
      for (int j = 0; j < nl; ++j) {
        const double al_ = j >= w ? -A[j] / B[j - w] : 0.0, ga_ = j + w < nl ? -C[j] / B[j + w] : 0.0;
        fa[j] = al_;
        fg[j] = ga_;
        An[j] = j >= w ? al_ * A[j - w] : 0.0;
        Cn[j] = j + w < nl ? ga_ * C[j + w] : 0.0;
        Bn[j] = B[j] + (j >= w ? al_ * C[j - w] : 0.0) + (j + w < nl ? ga_ * A[j + w] : 0.0);
      }
      A.swap(An);
      B.swap(Bn);
      C.swap(Cn);
    }
    double *ib = coef + (2 + 2 * (size_t)stages) * nl;
    for (int j = 1; j < nl - 1; ++j) ib[j] = 1.0 / B[j];
  } else {
    double *cp = ih + nl, *inv = cp + nl;
    for (int j = 1; j < nl - 1; ++j) {
      const double den = 2.0 * (h[j - 1] + h[j]) - (j > 1 ? h[j - 1] * cp[j - 1] : 0.0);
      inv[j] = 1.0 / den;
      cp[j] = (j < nl - 2 ? h[j] : 0.0) * inv[j];
    }
  }
  for (int i = 0, j = 0; i < nout && nl > 1; ++i) {
    const int l = g->lmin + i;
    while (j + 2 < nl && g->lrow[j + 1] <= l) ++j;
    jv[i] = j;
    sv[i] = (l - g->lrow[j]) * ih[j];
  }
  char *w = static_cast<char *>(ws);
  double *d_coef = reinterpret_cast<double *>(w);
  double *d_s = reinterpret_cast<double *>(w + o1);
  int *d_j = reinterpret_cast<int *>(w + o2);
  double *Md = reinterpret_cast<double *>(w + o3);
  // a pageable copy returns once the host data is staged
  cudaError_t e = cudaMemcpyAsync(w, up.data(), o3, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_fail(e, "cl_interp: coefficient upload");
  ProfScope prof(GCAMB_K_INTERP, st);
  if (pcr) {
    const unsigned ny = (unsigned)std::max(1, std::min((nout + 255) / 256, 304 / std::min(M, 304)));
    cl_spline_pcr_kernel<<<dim3((unsigned)M, ny), 256, 0, st>>>(Cl_s, g->d_lrow, g->d_rowof, d_coef + nl, d_coef + 2 * (size_t)nl, stages, d_j,
                                            d_s, nl, g->lmin, nout, Cl);
  } else if (nl <= kSmemSamples) {
    static_assert(6 * kSmemSamples * sizeof(double) <= kDynSmem, "samples in shared memory");
    const size_t smem = (size_t)6 * nl * sizeof(double);
    e = cudaFuncSetAttribute(cl_spline_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmem);
    if (e != cudaSuccess) return cuda_fail(e, "cl_interp: smem attribute");
    cl_spline_block_kernel<<<M, 256, smem, st>>>(Cl_s, g->d_lrow, g->d_rowof, d_coef, d_j, d_s, nl, g->lmin, nout, Cl);
  } else {
    cl_spline_solve_kernel<<<(M + 127) / 128, 128, 0, st>>>(Cl_s, g->d_lrow, d_coef, d_coef + nl, d_coef + 2 * nl,
                                                            d_coef + 3 * nl, nl, M, Md);
    const size_t n = (size_t)M * nout;
    cl_spline_eval_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(Cl_s, Md, g->d_lrow, g->d_rowof, d_j, d_s, nl,
                                                                       g->lmin, nout, M, Cl);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "cl_interp: launch");
  return GCAMB_OK;
}

int gcamb_interp_sources_workspace(const gcamb_grid *g, int M, int nk_in, size_t *bytes) {
  if (!g || !bytes) return fail(GCAMB_EINVAL, "interp_sources_workspace: NULL argument");
  if (M < 0 || nk_in < 2) return fail(GCAMB_EINVAL, "interp_sources_workspace: need M >= 0 and nk_in >= 2");
  *bytes = interp_workspace_bytes(M, nk_in, g->ntau, g->nk);
  return GCAMB_OK;
}

int gcamb_interp_sources(const gcamb_grid *g, const double *k_in, int nk_in, const void *S_in, int M, int dtype,
                         void *S_out, void *ws, size_t ws_bytes, void *stream) {
  if (!g) return fail(GCAMB_EINVAL, "interp_sources: NULL grid");
  if (dtype != GCAMB_F64 && dtype != GCAMB_F32) return fail(GCAMB_EINVAL, "interp_sources: dtype must be F64 or F32");
  if (M < 0 || nk_in < 2) return fail(GCAMB_EINVAL, "interp_sources: need M >= 0 and nk_in >= 2");
  if (!k_in) return fail(GCAMB_EINVAL, "interp_sources: NULL k_in");
  for (int j = 0; j < nk_in; ++j) {
    if (!std::isfinite(k_in[j])) return fail(GCAMB_EINVAL, "interp_sources: k_in not finite");
    if (j && !(k_in[j] > k_in[j - 1])) return fail(GCAMB_EINVAL, "interp_sources: k_in must be strictly increasing");
  }
  if (g->k.front() < k_in[0] || g->k.back() > k_in[nk_in - 1])
    return fail(GCAMB_EINVAL, "interp_sources: the grid's k range must lie inside [k_in[0], k_in[nk_in-1]]");
  if (M == 0) return GCAMB_OK;
  if (!S_in || !S_out || !ws) return fail(GCAMB_EINVAL, "interp_sources: NULL pointer");
  return launch_interp_sources(k_in, nk_in, S_in, M, g->ntau, dtype, g, S_out, ws, ws_bytes, (cudaStream_t)stream);
}

}  // extern "C"
