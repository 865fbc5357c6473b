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
// One CTA per 128 x 128 tile, K in chunks of 64 through a ring of 32 KB
// stages: three where the tiles are more than the SMs (two CTAs fit an SM,
// one's epilogue beside the other's main loop), six where one CTA has the SM
// to itself (a stage's copy takes about 1.2 us from issue to use, and three
// in flight give an SM 80 GB/s; the last layer's input gradient 38 -> 21 us, the
// weight gradients 32 -> 28 us): warp 0 issues the copies, warp 1 the MMAs (M = 128, N = 128, K = 16 into one
// TMEM accumulator, in increasing k), warps 2-9 the epilogue, which turns the
// tile through shared memory so that every global access is along a row.
//
// What bounds it: at the emulator's sizes (4096 x 512 x 512 .. 4096 x 2499 x
// 512) one tile's operands take longer from L2 than its MMAs; the GEMMs it
// replaces converted FP32 operands in the loading threads, a row a thread,
// without a copy in flight beside the MMAs.  Measured, batch 4096, width 512,
// n_out 2499: forward
// 412 -> 57 us, input gradients 554 -> 47 us, weight gradients 350 -> 28 us, a
// whole training step 1600 -> 181 us, bit for bit the same parameters; 4096
// served spectra 907 -> 129 us.
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
constexpr int kGemmThreads = 320;
constexpr int kPitch = 66;       // floats per row of the epilogue's tiles
constexpr int gemm_smem(int stages) { return stages * kStageG + 1024 /*align*/ + 256 /*barriers*/ + 192 * 8 /*exp tables*/; }

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
  const unsigned long long *tab;  // exp2 tables (see exp_q53)
};

struct LossArgs {
  const float *Y;       // [rows][N]
  const int *idx;       // target row of each batch row, or null
  float scale;
  float *part;          // [tiles][8]
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

// exp(y) for y = q 2^-53, |y| < 690, in 64-bit integers: GB300's FP64 pipe
// runs at 1/64 of the FP32 rate, so an FP64 exp of every C_l costs more than
// the network (4096 x 2499: 444 us).  t = y log2(e); exp2 of its fraction is
// the product of two table entries (2^(i/64), 2^(j/8192), Q1.63) and
// 1 + z + z^2/2 + z^3/6 of the rest (z < 2^-13.5; the next term is below
// 2^-58).  Every step keeps at least 2^-52 relative, so the result is within
// about one unit in the last place of the FP64 one.
__device__ __forceinline__ double exp_q53(long long q, const unsigned long long *__restrict__ tab) {
  const unsigned long long kLog2e = 0xB8AA3B295C17F0BCull;                 // log2(e), Q1.63
  const unsigned long long yu = (unsigned long long)q + (1ull << 63);      // y + 1024, Q11.53
  // (y + 1024) log2 e in Q.52 less 1024 log2 e
  const long long t = (long long)(__umul64hi(yu, kLog2e) - (kLog2e >> 1));
  const int e = (int)(t >> 52);
  const unsigned long long f = (unsigned long long)t & ((1ull << 52) - 1);
  const unsigned long long r0 = __umul64hi(tab[f >> 46], tab[64 + ((f >> 39) & 127)]);  // Q2.62
  const unsigned long long g = (f & ((1ull << 39) - 1)) << 25;             // the rest, Q.77
  const unsigned long long z = __umul64hi(g, 0xB17217F7D1CF79ACull);       // times ln 2: Q.77
  const unsigned int zh = (unsigned int)(z >> 32);                         // Q.45
  const unsigned int z2 = __umulhi(zh, zh);                                // z^2: Q.58; z^2 / 2: Q.59
  const unsigned int z3 = __umulhi(__umulhi(z2, zh), 0x55555556u);         // z^3 / 6: Q.(59 + 45 - 32) = Q.72
  const unsigned long long p = z + ((unsigned long long)z2 << 18) + ((unsigned long long)z3 << 5);
  const unsigned long long r = r0 + (__umul64hi(r0, p) >> 13);             // Q2.62
  // r in [2^62, 2^63]: round to 53 bits; a carry to 2^63 moves to the exponent
  const unsigned long long m = (r + (1ull << 9)) >> 10;
  return __longlong_as_double((long long)(((unsigned long long)(e + 1022) << 52) + m));
}

// Programmatic dependent launch: a kernel of the emulator's chain starts while
// the one before it drains (barriers, TMEM, tables) and waits here before it
// touches anything an earlier kernel wrote.  Every kernel of the chain waits,
// so what it reads or overwrites is complete through the whole chain.
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

template <int EPI, bool AMN, bool BMN, int NP, int ST>
__global__ void __launch_bounds__(kGemmThreads, ST == 3 ? 2 : 1) gemm_kernel(const __grid_constant__ GemmArgs<NP> a) {
  constexpr bool kSl = EPI == kSliced;
  constexpr int kStagesG = ST;
  constexpr uint32_t kCols = kSl ? 256 : 128;  // TMEM columns: one accumulator, sliced: two
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kStagesG * kStageG);
  // full[ST], empty[ST], tfull[2], tempty[2], drain, slot, abort
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + ST), tfull0 = smem_u32(bars + 2 * ST),
                 tempty0 = smem_u32(bars + 2 * ST + 2), drain = smem_u32(bars + 2 * ST + 4);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * ST + 5);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 2 * ST + 6);
  unsigned long long *tab = reinterpret_cast<unsigned long long *>(bars + 32);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int pi = 0;
  if constexpr (NP > 1)
    while (pi + 1 < a.np && (int)blockIdx.x >= a.p[pi].tile_end) ++pi;
  const Prob &p = a.p[pi];
  const int tile = (int)blockIdx.x - (NP > 1 && pi > 0 ? a.p[pi - 1].tile_end : 0);
  const int i0 = tile / p.tiles_n * 128, n0 = tile % p.tiles_n * 128;
  const int nkc = (p.K + kChunkK - 1) / kChunkK;
  const int per = kSl ? kSliceChunks : nkc;                  // chunks per accumulation
  const int nsl = kSl ? (nkc + per - 1) / per : 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStagesG; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      mbar_init(tempty0 + 8 * b, 8);
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
    for (int i = threadIdx.x; i < 192; i += kGemmThreads) tab[i] = a.ex.tab[i];
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0, last[kStagesG];
      uint32_t ph = 0;
#pragma unroll
      for (int s = 0; s < kStagesG; ++s) last[s] = -1;
      for (int kc = 0; kc < nkc; ++kc) {
        if (!mbar_wait(empty0 + 8 * stage, ph ^ 1u, abort_flag, a.err)) break;
        const uint32_t sa = smem_u32(smem + stage * kStageG), sb = sa + 16384, bar = full0 + 8 * stage;
        const int k0 = kc * kChunkK;
        mbar_expect_tx(bar, kStageG);
        last[stage] = (int)ph;
        if constexpr (AMN) {
          tma_load_2d(sa, &p.ta, i0, k0, bar);
          tma_load_2d(sa + 8192, &p.ta, i0 + 64, k0, bar);
        } else {
          tma_load_2d(sa, &p.ta, k0, i0, bar);
        }
        if constexpr (BMN) {
          tma_load_2d(sb, &p.tb, n0, k0, bar);
          tma_load_2d(sb + 8192, &p.tb, n0 + 64, k0, bar);
        } else {
          tma_load_2d(sb, &p.tb, k0, n0, bar);
        }
        if (++stage == kStagesG) {
          stage = 0;
          ph ^= 1u;
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
      int stage = 0;
      uint32_t ph = 0;
      for (int kc = 0; kc < nkc; ++kc) {
        const int sl = kc / per, buf = kSl ? sl & 1 : 0, first = kc - sl * per;
        if (kSl && first == 0 && !mbar_wait(tempty0 + 8 * buf, ((uint32_t)(sl >> 1) & 1u) ^ 1u, abort_flag, a.err)) break;
        if (!mbar_wait(full0 + 8 * stage, ph, abort_flag, a.err)) break;
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
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(empty0 + 8 * stage)
                     : "memory");
        if (first == per - 1 || kc == nkc - 1)
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tfull0 + 8 * buf)
                       : "memory");
        if (++stage == kStagesG) {
          stage = 0;
          ph ^= 1u;
        }
      }
      // every MMA this thread issued has completed before TMEM is freed
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(drain) : "memory");
      mbar_wait(drain, 0, nullptr, a.err);
    }
  } else {
    // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .., columns 64 half ..
    const int sp = warp & 3, half = (warp - 2) >> 2;
    const uint32_t taddr = tmem + ((uint32_t)(sp * 32) << 16) + (uint32_t)(half * 64);
    float acc[kSl ? 64 : 1];
    float2 gz[EPI == kDGelu || EPI == kLoss ? 32 : 1];
    bool ok = true;
    auto load32 = [&](uint32_t ad, uint32_t(&r)[32]) {
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
          "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
            "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
            "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
            "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
          : "r"(ad));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    };
    if constexpr (kSl) {
#pragma unroll
      for (int j = 0; j < 64; ++j) acc[j] = 0.f;
      for (int sl = 0; sl < nsl; ++sl) {
        const int buf = sl & 1;
        if (!mbar_wait(tfull0 + 8 * buf, (uint32_t)(sl >> 1) & 1u, abort_flag, a.err)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int h = 0; h < 4; ++h) {  // 16 columns at a time (registers)
          uint32_t r[16];
          const uint32_t ad = taddr + (uint32_t)(buf * 128 + h * 16);
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
              : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
              : "r"(ad));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[h * 16 + j] += __uint_as_float(r[j]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty0 + 8 * buf);
      }
    } else {
      if constexpr (EPI == kDGelu) {
        // GELU' of the tile's pre-activations while the MMAs run: all 32 rows'
        // loads in flight, two adjacent columns a lane
        const int ib = i0 + sp * 32, n = n0 + half * 64 + 2 * lane;
#pragma unroll
        for (int r = 0; r < 32; ++r)
          gz[r] = (ib + r < p.M && n < p.N) ? *reinterpret_cast<const float2 *>(p.Z + (long long)(ib + r) * p.ldc + n)
                                            : make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < 32; ++r) gz[r] = make_float2(gelu_grad_f(gz[r].x), gelu_grad_f(gz[r].y));
      }
      if constexpr (EPI == kLoss) {
        // the targets of the tile while the MMAs run (lane's columns n, n + 32)
        const int ib = i0 + sp * 32, n = n0 + half * 64 + lane;
        const int tr = ib + lane < p.M ? (a.ls.idx ? a.ls.idx[ib + lane] : ib + lane) : 0;
#pragma unroll
        for (int r = 0; r < 32; ++r) {
          const float *y = a.ls.Y + (size_t)__shfl_sync(0xffffffffu, tr, r) * p.N;
          gz[r].x = n < p.N ? __ldg(y + n) : 0.f;
          gz[r].y = n + 32 < p.N ? __ldg(y + n + 32) : 0.f;
        }
      }
      ok = mbar_wait(tfull0, 0, abort_flag, a.err);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    // all MMAs have read the ring: it now holds the epilogue's tiles
    float *st = reinterpret_cast<float *>(smem) + (warp - 2) * 32 * kPitch;
    if (__all_sync(0xffffffffu, ok)) {
      float2 *row = reinterpret_cast<float2 *>(st + lane * kPitch);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if constexpr (kSl) {
#pragma unroll
          for (int j = 0; j < 16; ++j) row[h * 16 + j] = make_float2(acc[h * 32 + 2 * j], acc[h * 32 + 2 * j + 1]);
        } else {
          uint32_t r[32];
          load32(taddr + (uint32_t)(h * 32), r);
#pragma unroll
          for (int j = 0; j < 16; ++j)
            row[h * 16 + j] = make_float2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
        }
      }
      __syncwarp();
      const int ib = i0 + sp * 32, nr = min(32, p.M - ib), nb = n0 + half * 64;
      // body(r) for the warp's rows.  A full tile has no exit in the loop, so that
      // the rows' chains (erff, expf, the exp of C_l) interleave: eight warps
      // alone leave their latency bare.
      auto rows = [&](auto un, auto body) {
        if (nr == 32) {
#pragma unroll decltype(un)::value
          for (int r = 0; r < 32; ++r) body(r);
        } else {
#pragma unroll 1
          for (int r = 0; r < nr; ++r) body(r);
        }
      };
      if constexpr (EPI == kGelu) {
        const int n = nb + 2 * lane;  // two adjacent columns a lane; ldc, ldb even
        const float2 b = make_float2(n < p.N ? p.bias[n] : 0.f, n + 1 < p.N ? p.bias[n + 1] : 0.f);
        if (n < p.N)
          rows(std::integral_constant<int, 8>(), [&](int r) {
            float2 v = *reinterpret_cast<const float2 *>(st + r * kPitch + 2 * lane);
            v.x += b.x;
            v.y += b.y;
            if (p.C)  // the padding column holds nothing that is read
              *reinterpret_cast<float2 *>(p.C + (long long)(ib + r) * p.ldc + n) = v;
            *reinterpret_cast<__nv_bfloat162 *>(p.Cb + (long long)(ib + r) * p.ldb + n) =
                __floats2bfloat162_rn(gelu_f(v.x), gelu_f(v.y));
          });
      } else if constexpr (EPI == kDGelu) {
        const int n = nb + 2 * lane;
        if (n < p.N) {
#pragma unroll
          for (int r = 0; r < 32; ++r) {
            if (r < nr) {
              float2 v = *reinterpret_cast<const float2 *>(st + r * kPitch + 2 * lane);
              v.x *= gz[r].x;
              v.y *= gz[r].y;
              *reinterpret_cast<float2 *>(p.C + (long long)(ib + r) * p.ldc + n) = v;
              *reinterpret_cast<__nv_bfloat162 *>(p.Cb + (long long)(ib + r) * p.ldb + n) = __floats2bfloat162_rn(v.x, v.y);
            }
          }
        }
      } else if constexpr (EPI == kExp) {
        // lane's columns nb + lane, + 32; the amplitude term of row `lane`
        const ExpArgs &x = a.ex;
        float sd[2], mu[2], bs[2];
        long long qmu[2];
        int ms[2], es[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int n = nb + lane + 32 * u;
          const bool c = n < p.N;
          sd[u] = c ? x.sd[n] : 1.f;
          sd[u] = sd[u] > 0.f ? sd[u] : 1.f;
          mu[u] = c ? x.mu[n] : 0.f;
          bs[u] = c ? p.bias[n] : 0.f;
          qmu[u] = __double2ll_rn((double)mu[u] * 9007199254740992.0);
          const unsigned int sbits = __float_as_uint(sd[u]);
          ms[u] = (int)((sbits & 0x7fffffu) | 0x800000u);
          es[u] = (int)(sbits >> 23) - 150;
          if ((sbits >> 23) == 0) mu[u] = __int_as_float(0x7f800000);  // subnormal sd: take the FP64 path
        }
        double sh = 0.0;
        if (x.amp >= 0 && lane < nr) sh = (double)x.X[(size_t)(ib + lane) * x.n_in + x.amp] - (double)x.mu_x[x.amp];
        const float shf_l = (float)sh;
        const long long qsh_l = __double2ll_rn(sh * 9007199254740992.0);
        constexpr int RU = 4;  // rows whose chains interleave
        for (int r0 = 0; r0 < nr; r0 += RU) {
          double c[RU][2];
          bool bad = false;
#pragma unroll
          for (int i = 0; i < RU; ++i) {
            const int r = r0 + i;
            const float shf = __shfl_sync(0xffffffffu, shf_l, r);
            const long long qsh = __shfl_sync(0xffffffffu, qsh_l, r);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const float y = st[r * kPitch + lane + 32 * u] + bs[u];
              const float fa = y * sd[u];
              bad |= !(fabsf(fa) < 900.f && fabsf(mu[u]) < 900.f && fabsf(shf) < 900.f &&
                       fabsf(fa + mu[u] + shf) < 690.f);
              const unsigned int yb = __float_as_uint(y);
              const int ye = (int)((yb >> 23) & 255u);
              int my = ye ? (int)((yb & 0x7fffffu) | 0x800000u) : 0;  // a subnormal y adds less than 2^-53
              my = (yb >> 31) ? -my : my;
              const long long m = (long long)my * (long long)ms[u];
              const int s = ye + es[u] - 97;  // y sd 2^53 = m 2^s
              const unsigned long long q =
                  s >= 0 ? (unsigned long long)m << min(s, 63) : (unsigned long long)(m >> min(-s, 63));
              c[i][u] = exp_q53((long long)(q + (unsigned long long)qmu[u] + (unsigned long long)qsh), tab);
            }
          }
          if (__any_sync(0xffffffffu, bad)) {  // out of the fixed-point range: FP64
#pragma unroll
            for (int i = 0; i < RU; ++i) {
              const double shd = __shfl_sync(0xffffffffu, sh, r0 + i);
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const int n = nb + lane + 32 * u;
                const float y = st[(r0 + i) * kPitch + lane + 32 * u] + bs[u];
                c[i][u] = exp((double)y * (double)sd[u] + (double)(n < p.N ? x.mu[n] : 0.f) + shd);
              }
            }
          }
#pragma unroll
          for (int i = 0; i < RU; ++i)
#pragma unroll
            for (int u = 0; u < 2; ++u)
              if (r0 + i < nr && nb + lane + 32 * u < p.N)
                x.CD[(long long)(ib + r0 + i) * p.N + nb + lane + 32 * u] = c[i][u];
        }
      } else if constexpr (EPI == kLoss) {
        float sq = 0.f;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int n = nb + lane + 32 * u;
          if (n >= p.N) continue;
          const float b = p.bias[n];
#pragma unroll
          for (int r = 0; r < 32; ++r) {
            if (r < nr) {
              const float o = st[r * kPitch + lane + 32 * u] + b;
              const float d = o - (u ? gz[r].y : gz[r].x);
              const float g = a.ls.scale * d;
              p.C[(long long)(ib + r) * p.ldc + n] = g;
              p.Cb[(long long)(ib + r) * p.ldb + n] = __float2bfloat16_rn(g);
              sq += d * d;
            }
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0) a.ls.part[(size_t)tile * 8 + warp - 2] = sq;
      } else {
        // lane's columns nb + lane, + 32: rows of any length and alignment
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int n = nb + lane + 32 * u;
          if (n >= p.N) continue;
          const float b = EPI == kBias ? p.bias[n] : 0.f;
          rows(std::integral_constant<int, 8>(), [&](int r) {
            const float v = st[r * kPitch + lane + 32 * u];
            p.C[(long long)(ib + r) * p.ldc + n] = EPI == kBias ? v + b : v;
          });
        }
      }
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
