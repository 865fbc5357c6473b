// tcgen05 GEMMs of the emulator network.
//
//   C[M][N] = A[M][K] . B[N][K]^T   (bf16 operands, FP32 accumulation, fused epilogue)
//
// Both operands are bf16 tensors in global memory, copied by TMA into the
// 128-byte swizzled layout the tensor cores read.  An operand may be stored
// with the contraction index contiguous (K-major: [rows][K]) or with its rows
// contiguous (MN-major: [K][rows]), so that the weight gradients (contraction
// over the batch) and the input gradients (over W's output index) read the
// same activations, gradients and weights as the forward pass: no transposed
// copies exist.  Whoever produces an operand rounds it to bf16 once.
//
// 128 x 128 tiles, K in chunks of 64 through a ring of 32 KB stages: warp 0
// issues the copies, warp 1 the MMAs (M = 128, N = 128, K = 16 into a TMEM
// accumulator, in increasing k), warps 2-17 the epilogue, 32 x 32 values each,
// turned through shared memory so that every global access is along a row.
// Sixteen epilogue warps: eight left the latency of erff, the exp of C_l and
// the global loads bare.
//
// Up to 152 tiles: one tile a CTA, six stages (a stage's copy takes about 1.2
// us from issue to use, and three in flight give an SM 80 GB/s; the last
// layer's input gradient 38 -> 22 us with six), the epilogue's tiles over the
// ring.  More tiles: 152 persistent CTAs with four stages (three beside the exp
// table), two TMEM accumulators and the epilogue's tiles beside the ring, so
// that a tile's loads and MMAs run under the epilogue of the one before.  640 tiles of the loss layer (batch 4096,
// n_out 2499) took 46 us with one tile a CTA, two CTAs an SM, whose 2.1 waves
// ran as three; now 34 us.
//
// What bounds it: at the emulator's sizes (4096 x 512 x 512 .. 4096 x 2499 x
// 512) one tile's operands take longer from L2 than its MMAs; the GEMMs it
// replaces converted FP32 operands in the loading threads, a row a thread,
// without a copy in flight beside the MMAs.  Measured, batch 4096, width 512,
// n_out 2499: forward 412 -> 47 us, input gradients 554 -> 44 us, weight
// gradients 350 -> 28 us, a whole training step 1600 -> 150 us, bit for bit the
// same parameters; 4096 served spectra 907 -> 107 us.
//
// Every wait is bounded; a timeout sets the error word and the CTA drains its
// copies and MMAs and frees its TMEM.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include <cstdint>
#include <type_traits>

#include "mbar.cuh"

namespace gcamb {
namespace emu {

// kGelu: Z = acc + bias (FP32, if C), bf16(GELU(Z)) -> Cb;  kBias: FP32 acc +
// bias -> C;  kExp: exp(acc + bias de-standardised, plus the amplitude term)
// -> CD;  kDGelu: acc GELU'(Z) -> C (FP32) and Cb (bf16);  kSliced: K in slices of
// kSliceK, each its own accumulation from zero, added in FP32 in increasing
// order -> C (the weight gradients, whose batch sum would otherwise be one
// long truncating tensor-core chain).
// kLoss (training, last layer): the gradient g = scale (acc + bias - Y) of the
// mean squared error -> C (FP32) and Cb (bf16), and the warps' sums of (acc +
// bias - Y)^2.
enum Epi { kGelu = 0, kBias = 1, kExp = 2, kDGelu = 3, kSliced = 4, kLoss = 5 };

constexpr int kChunkK = 64;
constexpr int kSliceChunks = 4;  // chunks per slice (kSliced)
constexpr int kStageG = 32768;
constexpr int kEpiWarpsG = 16;
constexpr int kGemmThreads = 64 + 32 * kEpiWarpsG;
constexpr int kPitch = 34;       // floats per row of the epilogue's tiles (32 x 32 a warp)
constexpr int gemm_stages(int epi, bool ps) { return ps ? (epi == kExp ? 3 : 4) : 6; }
constexpr int gemm_smem(int epi, bool ps) {
  return gemm_stages(epi, ps) * kStageG + 1024 /*align*/ + 256 /*barriers*/ + (epi == kExp ? 4096 * 8 : 0) /*exp table*/ +
         (ps ? kEpiWarpsG * 32 * kPitch * 4 : 0);
}

struct Prob {
  CUtensorMap ta, tb;
  int M, N, K;
  int tiles_n;          // tiles along N
  int tile_end;         // grouped launches: first tile of the next problem
  float *C;
  long long ldc;
  __nv_bfloat16 *Cb;
  long long ldb;
  const float *bias;    // [N]
  const float *Z;       // kDGelu: [M][ldc]
};

// kExp: C_l = exp(y sd + mu + (x_amp - mu_amp)).
struct ExpArgs {
  double *CD;           // [M][N]
  const float *mu, *sd; // [N]
  const float *X, *mu_x;
  int n_in, amp;        // amplitude column of X, or -1
  const unsigned long long *tab;  // exp2 table (see exp_q53)
};

struct LossArgs {
  const float *Y;       // [rows][N]
  const int *idx;       // target row of each batch row, or null
  float scale;
  float *part;          // [tiles][kEpiWarpsG]
};

template <int NP>
struct GemmArgs {
  Prob p[NP];
  ExpArgs ex;
  LossArgs ls;
  int np;
  int *err;
};

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }

__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// exp(y) for |y| < 690, q = (y + 1024 ln 2) 2^53, in integers: GB300's FP64
// pipe runs at 1/64 of the FP32 rate, so an FP64 exp of every C_l costs more
// than the network (4096 x 2499: 444 us).  k = the steps of ln 2 / 4096 below y
// (at most 0.006 too few from the rounded factor and q's high half: never
// above, so that the rest z is no less than 0 and below 2^-12.5); the result is the
// table's 2^(k mod 4096 / 4096) times 1 + z + z^2 (1/2 + z (1/6 + z/24)), in
// 32 x 32-bit products, each as wide as its term needs.  Within 0.92 units in
// the last place over the range (3.9e6 arguments against 113-bit arithmetic).
// A 64-bit high product for each of y log2(e), two table factors, the rest and
// the last product made 118 instructions of an exp (and 2.0 units): the served
// layer 74 us, now 52.
constexpr int kExpTab = 4096;                                 // 2^(j / 4096), Q2.62
constexpr unsigned long long kExpLn2 = 0x58B90BFBE8E7BCD6ull;  // ln 2 / 4096 in Q.75 = 1024 ln 2 in Q.53
constexpr unsigned int kExpLo = 41502639u, kExpSpan = 2893859389u;  // y + 1024 ln 2 in Q.21: 19.79, + 1379.9

__device__ __forceinline__ double exp_q53(unsigned long long q, const unsigned long long *__restrict__ tab) {
  const unsigned int k = __umulhi((unsigned int)(q >> 32), 3098164009u) >> 8;  // 4096 log2(e) 2^19
  const unsigned long long t = tab[k & (kExpTab - 1)];
  const unsigned long long z = (q << 22) - (unsigned long long)k * kExpLn2;  // Q.75
  const unsigned int zh = (unsigned int)(z >> 32);                           // Q.43
  const unsigned int w = __umulhi(zh, 87381u) + 0x2AAAAAABu;                 // 1/6 + z/24: Q.32
  const unsigned int u = (__umulhi(zh, w) >> 11) + 0x80000000u;              // 1/2 + z w: Q.32
  const unsigned int z2 = (unsigned int)(((unsigned long long)zh * zh) >> 30);  // Q.56
  const unsigned long long p = z + ((unsigned long long)__umulhi(z2, u) << 19);
  const unsigned int th = (unsigned int)(t >> 32), tl = (unsigned int)t, ph = (unsigned int)(p >> 32),
                     pl = (unsigned int)p;
  const unsigned long long r =
      t + (((unsigned long long)th * ph + __umulhi(th, pl) + __umulhi(tl, ph)) >> 11);  // Q2.62, below 2^63 (1 + 2^-19)
  const unsigned int ov = (unsigned int)(r >> 63);
  const unsigned long long m = (r + (512ull << ov)) >> (10 + ov);  // 53 bits; a carry moves to the exponent
  return __longlong_as_double((long long)(((unsigned long long)((k >> 12) - 2 + ov) << 52) + m));
}

// A float below 512 in Q.53 (truncated below 2^-53); any value above: nothing that is used.
__device__ __forceinline__ long long fix53(float v) {
  const unsigned int b = __float_as_uint(v);
  const int e = (int)((b >> 23) & 255u) - 97;
  const unsigned long long m = e > -97 ? (b & 0x7fffffu) | 0x800000u : 0;
  const long long q = (long long)(e >= 0 ? m << min(e, 63) : m >> min(-e, 63));
  return (int)b < 0 ? -q : q;
}

// Programmatic dependent launch: a kernel of the emulator's chain starts while
// the one before it drains (barriers, TMEM, tables) and waits here before it
// touches anything an earlier kernel wrote.  Every kernel of the chain waits
// (the bias sums at their end), so what it reads or overwrites is complete through the whole chain.
__device__ __forceinline__ void pdl_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// Shared-memory descriptor, 128-byte swizzle, version 1.  K-major: 8-row
// groups 1024 bytes apart.  MN-major: 64-row groups (one TMA box of 64 k)
// 8192 bytes apart (leading offset), 8-k groups 1024 bytes apart (stride).
template <bool MN>
__device__ __forceinline__ uint64_t g_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(MN ? 8192 >> 4 : 1) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

template <int EPI, bool AMN, bool BMN, int NP, bool PS>
__global__ void __launch_bounds__(kGemmThreads, 1) gemm_kernel(const __grid_constant__ GemmArgs<NP> a) {
  constexpr bool kSl = EPI == kSliced;
  constexpr int kStagesG = gemm_stages(EPI, PS);
  constexpr uint32_t kCols = kSl || PS ? 256 : 128;  // TMEM columns: two accumulators, or one
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kStagesG * kStageG);
  // full[ST], empty[ST], tfull[2], tempty[2], drain, slot, abort
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kStagesG), tfull0 = smem_u32(bars + 2 * kStagesG),
                 tempty0 = smem_u32(bars + 2 * kStagesG + 2), drain = smem_u32(bars + 2 * kStagesG + 4);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kStagesG + 5);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 2 * kStagesG + 6);
  unsigned long long *tab = reinterpret_cast<unsigned long long *>(bars + 32);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // tiles blockIdx.x, + gridDim.x, .. (PS; else one)
  const int ntiles = a.p[NP > 1 ? a.np - 1 : 0].tile_end;
  // The exp layer's last, partial round: a tile's rows (of each warp's 32) shared
  // out over up to four CTAs, which all compute the tile, cheap beside its exps
  // (640 tiles on 152 CTAs are 4.2 rounds: 58 -> 52 us).
  constexpr bool kShare = PS && EPI == kExp;
  const int full = kShare ? ntiles / (int)gridDim.x * (int)gridDim.x : ntiles, rest = ntiles - full;
  const int share = rest * 4 <= (int)gridDim.x ? 4 : (rest * 2 <= (int)gridDim.x ? 2 : 1);
  const int nunits = full + rest * share;
  struct Tile {
    const Prob *p;
    int tile, i0, n0, nkc, per, nsl;  // per: chunks per accumulation, nsl: accumulations
    int ra, rb;                       // rows [ra, rb) of a warp's 32
  };
  auto get_tile = [&](int t) {
    Tile r;
    int pi = 0;
    r.ra = 0;
    r.rb = 32;
    if (kShare && t >= full) {
      const int u = t - full;
      r.ra = 32 / share * (u % share);
      r.rb = r.ra + 32 / share;
      t = full + u / share;
    }
    if constexpr (NP > 1)
      while (pi + 1 < a.np && t >= a.p[pi].tile_end) ++pi;
    r.p = &a.p[pi];
    r.tile = t - (NP > 1 && pi > 0 ? a.p[pi - 1].tile_end : 0);
    r.i0 = r.tile / r.p->tiles_n * 128;
    r.n0 = r.tile % r.p->tiles_n * 128;
    r.nkc = (r.p->K + kChunkK - 1) / kChunkK;
    r.per = kSl ? kSliceChunks : r.nkc;
    r.nsl = kSl ? (r.nkc + r.per - 1) / r.per : 1;
    return r;
  };
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStagesG; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      mbar_init(tempty0 + 8 * b, kEpiWarpsG);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if constexpr (EPI == kExp)
    for (int i = threadIdx.x; i < kExpTab; i += kGemmThreads) tab[i] = a.ex.tab[i];
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  pdl_wait();
  // what follows the weight gradients runs beside them (the bias sums, which
  // read nothing later than this kernel's own inputs)
  if constexpr (kSl) pdl_start();

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0, last[kStagesG];
      uint32_t ph = 0;
#pragma unroll
      for (int s = 0; s < kStagesG; ++s) last[s] = -1;
      bool ok = true;
      for (int t = blockIdx.x; t < nunits && ok; t += gridDim.x) {
        const Tile tl = get_tile(t);
        const CUtensorMap *ta = &tl.p->ta, *tb = &tl.p->tb;
        for (int kc = 0; kc < tl.nkc; ++kc) {
          if (!mbar_wait(empty0 + 8 * stage, ph ^ 1u, abort_flag, a.err)) {
            ok = false;
            break;
          }
          const uint32_t sa = smem_u32(smem + stage * kStageG), sb = sa + 16384, bar = full0 + 8 * stage;
          const int k0 = kc * kChunkK;
          mbar_expect_tx(bar, kStageG);
          last[stage] = (int)ph;
          if constexpr (AMN) {
            tma_load_2d(sa, ta, tl.i0, k0, bar);
            tma_load_2d(sa + 8192, ta, tl.i0 + 64, k0, bar);
          } else {
            tma_load_2d(sa, ta, k0, tl.i0, bar);
          }
          if constexpr (BMN) {
            tma_load_2d(sb, tb, tl.n0, k0, bar);
            tma_load_2d(sb + 8192, tb, tl.n0 + 64, k0, bar);
          } else {
            tma_load_2d(sb, tb, k0, tl.n0, bar);
          }
          if (++stage == kStagesG) {
            stage = 0;
            ph ^= 1u;
          }
        }
      }
      // no copy may still be landing when the CTA exits
#pragma unroll
      for (int s = 0; s < kStagesG; ++s)
        if (last[s] >= 0) mbar_wait(full0 + 8 * s, (uint32_t)last[s], nullptr, a.err);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((AMN ? 1u : 0u) << 15) | ((BMN ? 1u : 0u) << 16) |
                                 ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      int stage = 0, un = 0;  // un: accumulations so far, in buffers 0, 1, 0, ..
      uint32_t ph = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < nunits && ok; t += gridDim.x) {
        const Tile tl = get_tile(t);
        int first = 0;
        for (int kc = 0; kc < tl.nkc; ++kc) {
          const int buf = un & 1;
          if ((first == 0 && !mbar_wait(tempty0 + 8 * buf, ((uint32_t)(un >> 1) & 1u) ^ 1u, abort_flag, a.err)) ||
              !mbar_wait(full0 + 8 * stage, ph, abort_flag, a.err)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sa = smem_u32(smem + stage * kStageG), sb = sa + 16384;
          const uint32_t d = tmem + (uint32_t)(buf * 128);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const uint64_t da = g_desc<AMN>(sa + kk * (AMN ? 2048 : 32)), db = g_desc<BMN>(sb + kk * (BMN ? 2048 : 32));
            const uint32_t acc = (first | kk) ? 1u : 0u;
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
                "l"(da), "l"(db), "r"(idesc), "r"(acc));
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(empty0 +
                                                                                                         8 * stage)
                       : "memory");
          if (++first == tl.per || kc == tl.nkc - 1) {
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tfull0 +
                                                                                                           8 * buf)
                         : "memory");
            first = 0;
            ++un;
          }
          if (++stage == kStagesG) {
            stage = 0;
            ph ^= 1u;
          }
        }
      }
      // every MMA this thread issued has completed before TMEM is freed
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(drain) : "memory");
      mbar_wait(drain, 0, nullptr, a.err);
    }
  } else {
    // ---- epilogue: warp w has TMEM lanes 32 (w % 4) .., columns 32 quarter ..
    const int sp = warp & 3, cq = (warp - 2) >> 2;
    const uint32_t taddr = tmem + ((uint32_t)(sp * 32) << 16) + (uint32_t)(cq * 32);
    // its 32 x 32 tile in shared memory (one tile a CTA: over the ring, which all MMAs have read)
    float *st = reinterpret_cast<float *>(PS ? reinterpret_cast<unsigned char *>(tab + (EPI == kExp ? kExpTab : 0)) : smem) +
                (warp - 2) * 32 * kPitch;
    const int c2 = 2 * (lane & 15), rp = lane >> 4;  // two adjacent columns of rows rp, rp + 2, ..
    int un = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < nunits; t += gridDim.x) {
      const Tile tl = get_tile(t);
      const Prob &p = *tl.p;
      const int ib = tl.i0 + sp * 32, nr = min(32, p.M - ib), nb = tl.n0 + cq * 32;
      float acc[32];
      float2 gz[EPI == kDGelu ? 16 : 1];
      float yt[EPI == kLoss ? 32 : 1];
      // kExp: the lane's column's scale, mean and bias; row `lane`'s amplitude and its mean
      float xsd = 1.f, xmu = 0.f, xbs = 0.f, xa = 0.f, xm = 0.f;
      if constexpr (EPI == kExp) {
        const ExpArgs &x = a.ex;
        const int n = nb + lane;
        if (n < p.N) {
          xsd = x.sd[n];
          xmu = x.mu[n];
          xbs = p.bias[n];
        }
        if (x.amp >= 0) {
          xm = x.mu_x[x.amp];
          xa = lane < nr ? x.X[(size_t)(ib + lane) * x.n_in + x.amp] : xm;
        }
      }
      auto load32 = [&](uint32_t ad, uint32_t(&r)[32]) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
            "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
              "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
              "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
            : "r"(ad));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      };
      if constexpr (EPI == kDGelu) {
        // GELU' of the tile's pre-activations while the MMAs run, all loads in flight
        const int n = nb + c2;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int r = ib + 2 * i + rp;
          gz[i] = (r < p.M && n < p.N) ? *reinterpret_cast<const float2 *>(p.Z + (long long)r * p.ldc + n)
                                       : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) gz[i] = make_float2(gelu_grad_f(gz[i].x), gelu_grad_f(gz[i].y));
      }
      if constexpr (EPI == kLoss) {
        // the targets of the tile while the MMAs run (lane's column)
        const int n = nb + lane;
        const int tr = ib + lane < p.M ? (a.ls.idx ? a.ls.idx[ib + lane] : ib + lane) : 0;
#pragma unroll
        for (int r = 0; r < 32; ++r) {
          const float *y = a.ls.Y + (size_t)__shfl_sync(0xffffffffu, tr, r) * p.N;
          yt[r] = n < p.N ? __ldg(y + n) : 0.f;
        }
      }
#pragma unroll
      for (int j = 0; j < 32; ++j) acc[j] = 0.f;
      for (int sl = 0; sl < tl.nsl; ++sl, ++un) {
        const int buf = un & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(tfull0 + 8 * buf, (uint32_t)(un >> 1) & 1u, abort_flag, a.err))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t r[32];
        load32(taddr + (uint32_t)(buf * 128), r);
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = kSl ? acc[j] + __uint_as_float(r[j]) : __uint_as_float(r[j]);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty0 + 8 * buf);
      }
      if (!ok) break;
      {
        float2 *row = reinterpret_cast<float2 *>(st + lane * kPitch);
#pragma unroll
        for (int j = 0; j < 16; ++j) row[j] = make_float2(acc[2 * j], acc[2 * j + 1]);
      }
      __syncwarp();
      // body(r) for the lane's rows: first, + step, ..  A full tile has no exit in
      // the loop, so that the rows' chains (erff, the exp of C_l) interleave.
      auto rows = [&](auto step, auto body) {
        constexpr int S = decltype(step)::value;
        if (nr == 32) {
#pragma unroll 8
          for (int i = 0; i < 32 / S; ++i) body(i * S + (S == 2 ? rp : 0));
        } else {
#pragma unroll 1
          for (int i = 0; i < 32 / S; ++i)
            if (i * S + (S == 2 ? rp : 0) < nr) body(i * S + (S == 2 ? rp : 0));
        }
      };
      if constexpr (EPI == kGelu) {
        const int n = nb + c2;  // ldc, ldb even
        const float2 b = make_float2(n < p.N ? p.bias[n] : 0.f, n + 1 < p.N ? p.bias[n + 1] : 0.f);
        if (n < p.N)
          rows(std::integral_constant<int, 2>(), [&](int r) {
            float2 v = *reinterpret_cast<const float2 *>(st + r * kPitch + c2);
            v.x += b.x;
            v.y += b.y;
            if (p.C)  // the padding column holds nothing that is read
              *reinterpret_cast<float2 *>(p.C + (long long)(ib + r) * p.ldc + n) = v;
            *reinterpret_cast<__nv_bfloat162 *>(p.Cb + (long long)(ib + r) * p.ldb + n) =
                __floats2bfloat162_rn(gelu_f(v.x), gelu_f(v.y));
          });
      } else if constexpr (EPI == kDGelu) {
        const int n = nb + c2;
        if (n < p.N) {
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int r = 2 * i + rp;
            if (r < nr) {
              float2 v = *reinterpret_cast<const float2 *>(st + r * kPitch + c2);
              v.x *= gz[i].x;
              v.y *= gz[i].y;
              *reinterpret_cast<float2 *>(p.C + (long long)(ib + r) * p.ldc + n) = v;
              *reinterpret_cast<__nv_bfloat162 *>(p.Cb + (long long)(ib + r) * p.ldb + n) = __floats2bfloat162_rn(v.x, v.y);
            }
          }
        }
      } else if constexpr (EPI == kExp) {
        // lane's column nb + lane; y sd + mu + sh in Q.53 from integers: y's and
        // sd's mantissas (31 bits) multiply exactly, shifted right by a positive
        // count where |y sd| < 100
        const ExpArgs &x = a.ex;
        const int n = nb + lane;
        const bool cin = n < p.N;
        const float sd = xsd > 0.f ? xsd : 1.f;
        const unsigned long long qmu = (unsigned long long)fix53(xmu) + kExpLn2;
        const unsigned int sbits = __float_as_uint(sd);
        const int ms = (int)((sbits & 0x7fffffu) | 0x800000u) << 7, es = 261 - (int)(sbits >> 23);
        // Elements out of the fixed-point range take the FP64 exp, each by itself: a
        // spectrum is the same bits alone and among any others of a batch.
        const bool badc = !(fabsf(xmu) < 300.f) || !(fabsf(xm) < 300.f) || (sbits >> 23) == 0;  // the column (or a subnormal sd)
        const unsigned int badr = __ballot_sync(0xffffffffu, !(fabsf(xa) < 300.f));             // rows
        const bool badt = __any_sync(0xffffffffu, badc) || badr;
        *reinterpret_cast<long long *>(st + lane * kPitch + 32) = fix53(xa) - fix53(xm);
        __syncwarp();
        // row r's argument in Q.53, and whether it is out of the range
        auto arg = [&](int r, bool &out) {
          const float *sr = st + r * kPitch;
          const float y = sr[lane] + xbs;
          const unsigned int yb = __float_as_uint(y);
          const int sg = (int)yb >> 31;
          const int my = ((int)(((yb << 7) & 0x3fffffffu) | 0x40000000u) ^ sg) - sg;  // a subnormal y: 0 or -2^-53
          const int rs = min(es - (int)((yb >> 23) & 255u), 63);
          const unsigned long long q =
              (unsigned long long)(((long long)my * ms) >> (rs & 63)) + qmu + *reinterpret_cast<const unsigned long long *>(sr + 32);
          out = !(fabsf(y * sd) < 100.f) || (unsigned int)(q >> 32) - kExpLo > kExpSpan;
          return q;
        };
        constexpr int RU = 8;  // rows whose chains interleave
        for (int r0 = tl.ra; r0 < min(nr, tl.rb); r0 += RU) {
          double c[RU];
          bool bad = badt;
#pragma unroll
          for (int i = 0; i < RU; ++i) {
            bool out;
            c[i] = exp_q53(arg(r0 + i, out), tab);
            bad |= out;
          }
          if (__any_sync(0xffffffffu, bad)) {
#pragma unroll
            for (int i = 0; i < RU; ++i) {
              const double shd = (double)__shfl_sync(0xffffffffu, xa, r0 + i) - (double)xm;
              bool out;
              arg(r0 + i, out);
              const float y = st[(r0 + i) * kPitch + lane] + xbs;
              if (out || badc || (badr >> (r0 + i) & 1u)) c[i] = exp((double)y * (double)sd + (double)xmu + shd);
            }
          }
#pragma unroll
          for (int i = 0; i < RU; ++i)
            if (r0 + i < nr && cin) x.CD[(long long)(ib + r0 + i) * p.N + n] = c[i];
        }
      } else if constexpr (EPI == kLoss) {
        float sq = 0.f;
        const int n = nb + lane;
        if (n < p.N) {
          const float b = p.bias[n];
#pragma unroll
          for (int r = 0; r < 32; ++r) {
            if (r < nr) {
              const float o = st[r * kPitch + lane] + b;
              const float d = o - yt[r];
              const float g = a.ls.scale * d;
              p.C[(long long)(ib + r) * p.ldc + n] = g;
              p.Cb[(long long)(ib + r) * p.ldb + n] = __float2bfloat16_rn(g);
              sq += d * d;
            }
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0) a.ls.part[(size_t)tl.tile * kEpiWarpsG + warp - 2] = sq;
      } else {
        // rows of any length and alignment
        const int n = nb + lane;
        if (n < p.N) {
          const float b = EPI == kBias ? p.bias[n] : 0.f;
          rows(std::integral_constant<int, 1>(), [&](int r) {
            const float v = st[r * kPitch + lane];
            p.C[(long long)(ib + r) * p.ldc + n] = EPI == kBias ? v + b : v;
          });
        }
      }
      __syncwarp();  // the tile is read before the next one overwrites it
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
  }
}

}  // namespace emu
}  // namespace gcamb
