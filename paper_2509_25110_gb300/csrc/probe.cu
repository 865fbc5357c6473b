// Throughput probes for the plain arithmetic pipes (the roofline of the FP64
// and FP32 CUDA-core kernels).  Eight independent FMA chains per thread keep
// the pipe busy; the grid covers every SM several times over.
#include <cuda_bf16.h>

#include "internal.h"
#include "mbar.cuh"

namespace gcamb {

namespace {

__device__ __forceinline__ uint64_t e_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// One 128 x 64 bf16 tile of an FP32 matrix [128][K] (columns k0 .., zero
// beyond K), one row per thread, in the swizzled K-major layout.
__device__ __forceinline__ void load_tile(const float *p, int K, int k0, unsigned char *tile) {
  const int tid = threadIdx.x;
  const float *src = p + (long long)tid * K;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    uint32_t w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = k0 + c * 8 + 2 * u;
      const __nv_bfloat162 h = __floats2bfloat162_rn(k < K ? __ldg(src + k) : 0.f, k + 1 < K ? __ldg(src + k + 1) : 0.f);
      w[u] = *reinterpret_cast<const uint32_t *>(&h);
    }
    const uint32_t o = (uint32_t)tid * 128u + ((uint32_t)(c ^ (tid & 7)) << 4);
    *reinterpret_cast<uint4 *>(tile + o) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// C[128][128] = A[128][K] . B[128][K]^T in one TMEM accumulator, K in steps
// of 16: the accumulation self-test (two buffers; the threads fill one while
// the MMAs drain the other).
__global__ void __launch_bounds__(128, 1) mma_probe_kernel(const float *A, const float *B, int K, float *C, int *err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // [buf0: A 16 KB | B 16 KB][buf1: A | B][barriers]
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + 65536);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 3);
  const uint32_t done0 = smem_u32(bars), fin = smem_u32(bars + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(done0) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(done0 + 8) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(fin) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) |
                             ((uint32_t)(128 >> 4) << 24);
  const int nkc = (K + 63) / 64;
  bool ok = true;
  for (int kc = 0; kc < nkc && ok; ++kc) {
    const int buf = kc & 1;
    bool w = true;
    if (kc >= 2) w = mbar_wait(done0 + 8 * buf, (uint32_t)((kc - 2) >> 1) & 1u, nullptr, err);
    // every thread takes the same branch (no thread may be left at a barrier)
    if (!__syncthreads_and(w)) {
      ok = false;
      break;
    }
    unsigned char *ta = smem + buf * 32768, *tb = ta + 16384;
    load_tile(A, K, kc * 64, ta);
    load_tile(B, K, kc * 64, tb);
    // generic-proxy stores -> visible to the tensor cores (async proxy)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sa = smem_u32(ta), sb = smem_u32(tb);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const uint64_t da = e_desc(sa + kk * 32), db = e_desc(sb + kk * 32);
        const uint32_t acc = (kc | kk) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
            "l"(da), "l"(db), "r"(idesc), "r"(acc));
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(done0 + 8 * buf)
                   : "memory");
    }
  }
  // all MMAs done (also on the error path, before TMEM is freed)
  if (threadIdx.x == 0)
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(fin) : "memory");
  const bool fin_ok = mbar_wait(fin, 0, nullptr, err);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (ok && fin_ok) {
    const int i = warp * 32 + lane;
#pragma unroll 1
    for (int c = 0; c < 8; ++c) {
      uint32_t r[16];
      const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(c * 16);
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
            "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
          : "r"(taddr));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int j = 0; j < 16; ++j) C[(long long)i * 128 + c * 16 + j] = __uint_as_float(r[j]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem) : "memory");
  }
}

constexpr int kProbeSmem = 65536 + 1024 + 256;

}  // namespace

int run_probe_mma(const float *A, const float *B, int K, float *C, cudaStream_t st) {
  int *err = device_error_flag();
  if (!err) return fail(GCAMB_ECUDA, "probe_mma: error flag allocation");
  cudaError_t e = cudaFuncSetAttribute(mma_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kProbeSmem);
  if (e != cudaSuccess) return cuda_fail(e, "probe_mma: smem attribute");
  mma_probe_kernel<<<1, 128, kProbeSmem, st>>>(A, B, K, C, err);
  e = cudaGetLastError();
  return e == cudaSuccess ? GCAMB_OK : cuda_fail(e, "probe_mma: launch");
}

template <typename T>
__global__ void __launch_bounds__(256) fma_probe_kernel(T a, T b, int iters, T *out) {
  T c[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) c[u] = (T)(threadIdx.x + u);
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int u = 0; u < 8; ++u) c[u] = fma(c[u], a, b);
  }
  T s = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u) s += c[u];
  if (s == (T)-12345.678) out[0] = s;  // keeps the chains live; never true for these inputs
}

template <typename T>
static int probe_t(double *flops) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  T *out = nullptr;
  cudaError_t e = cudaMalloc(&out, sizeof(T));
  if (e != cudaSuccess) return cuda_fail(e, "probe: cudaMalloc");
  const int blocks = sms * 8, threads = 256;
  const int iters = sizeof(T) == 8 ? 2048 : 65536;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  fma_probe_kernel<T><<<blocks, threads>>>((T)0.999999, (T)1e-7, iters / 8, out);  // warm-up
  float best = 1e30f;
  for (int rep = 0; rep < 3; ++rep) {
    cudaEventRecord(e0);
    fma_probe_kernel<T><<<blocks, threads>>>((T)0.999999, (T)1e-7, iters, out);
    cudaEventRecord(e1);
    cudaEventSynchronize(e1);
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    best = ms < best ? ms : best;
  }
  e = cudaGetLastError();
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(out);
  if (e != cudaSuccess) return cuda_fail(e, "probe: kernel");
  *flops = 2.0 * 8.0 * (double)iters * blocks * threads / (best * 1e-3);
  return GCAMB_OK;
}

int run_probe_flops(int what, double *flops) {
  return what == 0 ? probe_t<double>(flops) : probe_t<float>(flops);
}

// One thread waits, with the kernels' bounded wait, on an mbarrier that no
// one arrives on: after the wait limit it writes GCAMB_ETIMEOUT to *err and
// the kernel ends.
__global__ void wait_selftest_kernel(int *err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_wait(smem_u32(&bar), 0, nullptr, err);
  }
}

int run_wait_selftest(int *status, cudaStream_t st) {
  int *err = status ? status : device_error_flag();
  if (!err) return fail(GCAMB_ECUDA, "selftest_wait: error flag allocation");
  wait_selftest_kernel<<<1, 32, 0, st>>>(err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "selftest_wait: launch");
  return GCAMB_OK;
}

}  // namespace gcamb
