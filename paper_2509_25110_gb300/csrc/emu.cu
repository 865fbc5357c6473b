// Emulator of log C_l with a projection fallback.
//
// An MLP maps the 9 source-generator features to standardised log C_l
// (l = lmin..lmax of a grid).  It is trained on the device by the library's
// own kernels: tcgen05 GEMMs with bf16 operands and FP32 accumulation
// (emu_gemm.cuh) for the forward pass, the input and weight gradients, and
// small kernels for the loss, bias gradients and Adam.  Parameters and Adam
// moments are FP32, as are pre-activations and gradients; every matrix-product
// operand is rounded to bf16 once, by the kernel that produces it (Adam writes
// the weights' bf16 copies beside the FP32 ones).  A held-out check (spectra from the projection path) marks cells
// of parameter space as trusted; gcamb_emulate answers trusted requests from
// the network and the rest from the batched projection (gcamb_los_cl) on
// sources regenerated from the features.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "emu_gemm.cuh"
#include "internal.h"

using namespace gcamb;
using namespace gcamb::emu;

struct gcamb_emu {
  gcamb_grid *g = nullptr;
  int n_in = 0, width = 0, depth = 0, n_out = 0, max_batch = 0;
  std::vector<int> sizes;                // n_in, width x depth, n_out
  std::vector<size_t> w_off, b_off;      // offsets of W_l [out][in] and b_l [out] in theta
  size_t n_params = 0;
  float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
  float *mu_x = nullptr, *isd_x = nullptr, *mu_y = nullptr, *sd_y = nullptr;
  float *loss_part = nullptr;             // the last layer's warps' sums of squared errors
  // bf16 operands, rows padded to 8 elements (the copies' 16-byte strides):
  // weights [out][in], standardised features and activations [B][in] (act[l]
  // is the input of layer l), gradients wrt the pre-activations [B][out]
  std::vector<__nv_bfloat16 *> W, act, dB;
  std::vector<float *> Z, dF;            // FP32 [B][padded width]: hidden pre-activations, gradients wrt the pre-activations
  unsigned long long *exp_tab = nullptr; // exp2 tables of exp_q53
  int *flags_host = nullptr, *flags_dev = nullptr;  // mapped host copy of emulate's fallback flags
  // tensor maps of those buffers for the last batch size
  struct Maps {
    CUtensorMap act_k, act_mn, d_k, d_mn, w_k, w_mn;
  };
  std::vector<Maps> maps;
  int maps_B = 0;
  int64_t step = 0;
  int *err = nullptr;
  // trust cells: bit d of a cell is (x[cell_dim[d]] > cell_mid[d])
  std::vector<int> cell_dim;
  std::vector<float> cell_mid;
  std::vector<unsigned char> trusted;
  int *d_cell_dim = nullptr;
  float *d_cell_mid = nullptr;
  unsigned char *d_trusted = nullptr;
  double check_max_err = -1.0, check_tol = 0.0;
  // fallback buffers
  int fb_cap = 0, fb_mode = GCAMB_F16X3;
  float *fb_x = nullptr, *fb_S = nullptr;
  double *fb_P = nullptr, *fb_C = nullptr;
  int *fb_idx = nullptr;
  void *fb_ws = nullptr;
  size_t fb_ws_bytes = 0;
};

// Column of the amplitude feature ln(1e10 A_s) in the 9-feature layout.
static int amp_col(const gcamb_emu *e) { return e->n_in == 9 ? 8 : -1; }

namespace {

constexpr uint32_t kEmuMagic = 0x47454D55u;  // "GEMU"

int ck(cudaError_t e, const char *what) { return e == cudaSuccess ? GCAMB_OK : cuda_fail(e, what); }

template <typename T>
int dalloc(T **p, size_t n) {
  cudaError_t e = cudaMalloc(p, std::max<size_t>(1, n) * sizeof(T));
  if (e != cudaSuccess) {
    *p = nullptr;
    return e == cudaErrorMemoryAllocation ? fail(GCAMB_ENOMEM, "emu: device allocation") : cuda_fail(e, "emu: cudaMalloc");
  }
  return GCAMB_OK;
}

// ---------------------------------------------------------------- kernels

__device__ __forceinline__ uint64_t sm64(uint64_t c) {
  uint64_t z = c + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// U(-bound, bound) from SplitMix64 on (seed, parameter index)
__global__ void init_uniform_kernel(float *p, size_t n, float bound, uint64_t seed, uint64_t base) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double u = (double)(sm64((seed << 40) ^ (base + i)) >> 11) * (1.0 / 9007199254740992.0);
    p[i] = (float)((2.0 * u - 1.0) * bound);
  }
}

// Standardised features, rounded to the bf16 operand of the first layer.
__global__ void standardize_kernel(const float *__restrict__ X, const int *__restrict__ idx, int B, int n,
                                   const float *__restrict__ mu, const float *__restrict__ isd,
                                   __nv_bfloat16 *__restrict__ xs, int ld) {
  pdl_start();
  pdl_wait();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * n) return;
  const int b = e / n, j = e - b * n;
  const int r = idx ? idx[b] : b;
  xs[(size_t)b * ld + j] = __float2bfloat16_rn((X[(size_t)r * n + j] - mu[j]) * isd[j]);
}

constexpr int kSumCols = 16;    // columns of a block of bias_kernel
constexpr int kSumClasses = 32;

// Column sums by rows mod 32: thread (column c, class r) holds the sum of its
// rows b = r, r + 32, ... in increasing order; the classes are added as a
// balanced tree (16, 8, 4, 2, 1 apart).  Fixed order: deterministic.
__device__ __forceinline__ void class_sum(float (*s)[kSumCols + 1], int c, int r, float v, float *out) {
  s[r][c] = v;
  __syncthreads();
#pragma unroll
  for (int o = kSumClasses / 2; o > 0; o >>= 1) {
    if (r < o) s[r][c] += s[r + o][c];
    __syncthreads();
  }
  if (r == 0 && out) *out = s[0][c];
}

// Bias gradients of every layer (grid y): column sums of d [B][ld], all of a
// thread's next 32 rows in flight.  The grid's last block adds up the loss
// from the warps' partial sums, in order.
constexpr int kMaxLayers = 9;
struct BiasSums {
  const float *d[kMaxLayers];
  float *db[kMaxLayers];
  int N[kMaxLayers], ld[kMaxLayers];
  const float *part;
  int nparts;
  float inv_total;
  float *loss;
};

__global__ void __launch_bounds__(kSumCols *kSumClasses) bias_kernel(const __grid_constant__ BiasSums a, int B, int L) {
  __shared__ float s[kSumClasses][kSumCols + 1];
  __shared__ double red[kSumCols * kSumClasses / 32];
  const int c = threadIdx.x % kSumCols, r = threadIdx.x / kSumCols, l = blockIdx.y;
  // Runs beside the weight gradients, whose CTAs let it start once everything
  // read here was complete (20 us of column sums under 28 us of GEMM: training
  // step 164 -> 150 us).  Only the block of the loss waits, at its end, so that
  // what waits for this kernel finds the weight gradients complete too.
  pdl_start();
  if (l == L) {
    if (blockIdx.x > 0) return;
    if (!a.loss) {
      pdl_wait();
      return;
    }
    double t = 0.0;
    for (int i = threadIdx.x; i < a.nparts; i += kSumCols * kSumClasses) t += (double)a.part[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int i = 1; i < kSumCols * kSumClasses / 32; ++i) t += red[i];
      *a.loss = (float)(t * a.inv_total);
    }
    pdl_wait();
    return;
  }
  const int n = blockIdx.x * kSumCols + c, N = a.N[l];
  if (blockIdx.x * kSumCols >= (unsigned)N) return;  // the whole block
  const float *d = a.d[l];
  const size_t ld = a.ld[l];
  float sum = 0.f;
  if (n < N) {
    int b = r;
    for (; b + 31 * kSumClasses < B; b += 32 * kSumClasses) {
      float v[32];
#pragma unroll
      for (int u = 0; u < 32; ++u) v[u] = __ldcg(d + (size_t)(b + u * kSumClasses) * ld + n);
#pragma unroll
      for (int u = 0; u < 32; ++u) sum += v[u];
    }
    for (; b < B; b += kSumClasses) sum += d[(size_t)b * ld + n];
  }
  class_sum(s, c, r, sum, n < N ? a.db[l] + n : nullptr);
}

// Adam on the flat parameters; layer grid y writes its weights' bf16 copy too.
struct AdamLayers {
  size_t w_off[kMaxLayers], end[kMaxLayers];  // the layer's first weight, one past its last bias
  unsigned int nw[kMaxLayers];                // weights
  int nin[kMaxLayers], ld[kMaxLayers];
  __nv_bfloat16 *Wb[kMaxLayers];
};

// bf16 copies of every layer's weights (grid y) from the FP32 parameters.
__global__ void weights_bf16_kernel(const float *__restrict__ p, const __grid_constant__ AdamLayers L) {
  const int l = blockIdx.y;
  const float *W = p + L.w_off[l];
  const unsigned int n = L.nw[l], nin = L.nin[l];
  for (unsigned int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const unsigned int o = e / nin;
    L.Wb[l][(size_t)o * L.ld[l] + (e - o * nin)] = __float2bfloat16_rn(W[e]);
  }
}

__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, AdamLayers L, float lr, float b1, float b2, float eps, float bc1,
                            float bc2) {
  constexpr int U = 4;  // parameters a thread, all loads in flight
  pdl_start();
  const int l = blockIdx.y;
  const size_t base = L.w_off[l];
  const unsigned int n = (unsigned int)(L.end[l] - base), nw = L.nw[l], nin = L.nin[l];
  pdl_wait();
  for (unsigned int e0 = blockIdx.x * (blockDim.x * U) + threadIdx.x; e0 < n; e0 += gridDim.x * (blockDim.x * U)) {
    float gi[U], mo[U], vo[U], po[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned int e = e0 + u * blockDim.x;
      if (e < n) {
        gi[u] = g[base + e];
        mo[u] = m[base + e];
        vo[u] = v[base + e];
        po[u] = p[base + e];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned int e = e0 + u * blockDim.x;
      if (e >= n) break;
      // one rounding order, whatever the compiler contracts
      const float mi = __fmaf_rn(1.f - b1, gi[u], __fmul_rn(b1, mo[u]));
      const float vi = __fmaf_rn(__fmul_rn(1.f - b2, gi[u]), gi[u], __fmul_rn(b2, vo[u]));
      m[base + e] = mi;
      v[base + e] = vi;
      const float pi = po[u] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
      p[base + e] = pi;
      if (e < nw) {
        const unsigned int o = e / nin;
        L.Wb[l][(size_t)o * L.ld[l] + (e - o * nin)] = __float2bfloat16_rn(pi);
      }
    }
  }
}

// column mean and standard deviation (two passes, FP64), thread per column
__global__ void colstats_kernel(const float *__restrict__ X, int N, int n, float *__restrict__ mu,
                                float *__restrict__ sd) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  double s = 0.0;
  for (int i = 0; i < N; ++i) s += X[(size_t)i * n + j];
  const double mean = s / N;
  double q = 0.0;
  for (int i = 0; i < N; ++i) {
    const double d = X[(size_t)i * n + j] - mean;
    q += d * d;
  }
  mu[j] = (float)mean;
  sd[j] = (float)sqrt(q / N);
}

// C_l is proportional to A_s (Eq. 1 is linear in P), so the amplitude
// feature ln(1e10 A_s) (column amp of X, or none if amp < 0) enters log C_l
// exactly as an additive term, relative to its training mean: the network
// learns log C_l - (x_amp - mu_amp), and that term is added back on output.
__device__ __forceinline__ double amp_shift(const float *__restrict__ X, int n_in, int amp,
                                            const float *__restrict__ mu_x, size_t s) {
  return amp < 0 ? 0.0 : (double)X[s * n_in + amp] - (double)mu_x[amp];
}

__global__ void log_kernel(const double *__restrict__ C, size_t N, int n, const float *__restrict__ X, int n_in,
                           int amp, const float *__restrict__ mu_x, float *__restrict__ Y) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N * n; i += (size_t)gridDim.x * blockDim.x)
    Y[i] = (float)(log(C[i]) - amp_shift(X, n_in, amp, mu_x, i / n));
}

__global__ void standardize_y_kernel(float *__restrict__ Y, size_t N, int n, const float *__restrict__ mu,
                                     const float *__restrict__ sd) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N * n; i += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(i % n);
    Y[i] = (Y[i] - mu[j]) / (sd[j] > 0.f ? sd[j] : 1.f);
  }
}

__global__ void inv_sd_kernel(const float *__restrict__ sd, int n, float *__restrict__ isd) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) isd[j] = sd[j] > 1e-12f ? 1.f / sd[j] : 0.f;
}

__global__ void cell_kernel(const float *__restrict__ X, int B, int n_in, const int *__restrict__ dims,
                            const float *__restrict__ mids, int nd, const unsigned char *__restrict__ trusted,
                            int *__restrict__ fallback, int *__restrict__ fallback_host) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  int c = 0;
  for (int d = 0; d < nd; ++d)
    if (X[(size_t)b * n_in + dims[d]] > mids[d]) c |= 1 << d;
  const int f = trusted ? (trusted[c] ? 0 : 1) : 1;
  fallback[b] = f;
  fallback_host[b] = f;
}

// per-sample max |C_emu / C_ref - 1|
__global__ void __launch_bounds__(256) maxrel_kernel(const double *__restrict__ Ce, const double *__restrict__ Cr,
                                                     int n, double *__restrict__ err) {
  __shared__ double red[256];
  const size_t b = blockIdx.x;
  double mx = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double r = Cr[b * n + j];
    const double e = r != 0.0 ? fabs(Ce[b * n + j] / r - 1.0) : fabs(Ce[b * n + j]);
    mx = e > mx ? e : mx;
  }
  red[threadIdx.x] = mx;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) err[b] = red[0];
}

__global__ void gather_rows_kernel(const float *__restrict__ X, const int *__restrict__ idx, int B, int n,
                                   float *__restrict__ out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < B * n) out[e] = X[(size_t)idx[e / n] * n + (e % n)];
}

__global__ void scatter_rows_kernel(const double *__restrict__ src, const int *__restrict__ idx, int B, int n,
                                    double *__restrict__ dst) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)B * n; e += (size_t)gridDim.x * blockDim.x)
    dst[(size_t)idx[e / n] * n + (e % n)] = src[e];
}

// Synthetic sources of one generator family from its 9 features
// (tau*, sigma, r_s, cos phi, sin phi, k_D, b, n_s, ln(1e10 A_s)):
// S(k, tau) = N(tau; tau*, sigma) cos(k r_s + phi) exp(-(k/k_D)^2)
//           + b exp(-(tau - 11000)^2 / (2 2000^2)) exp(-k / 0.01),
// P(k) = A_s (k / 0.05)^(n_s - 1).  S separates into tau and k factors: one
// block per (source, 256 k nodes) evaluates them once in FP64 (shared memory)
// and combines them with two multiply-adds per element; stored FP32 (S) and
// FP64 (P).
__global__ void __launch_bounds__(256) synth_kernel(const float *__restrict__ X, const double *__restrict__ k,
                                                    const double *__restrict__ tau, int nk, int ntau,
                                                    float *__restrict__ S, double *__restrict__ P) {
  extern __shared__ double sh[];  // g[ntau], late[ntau], a[256], e[256]
  double *gt = sh, *lt = sh + ntau, *ak = sh + 2 * ntau, *ek = ak + 256;
  const int m = blockIdx.y, q0 = blockIdx.x * 256;
  const float *f = X + (size_t)m * 9;
  const double ts = f[0], sg = f[1], rs = f[2], phi = atan2((double)f[4], (double)f[3]), kd = f[5], bb = f[6];
  const double inv_norm = 1.0 / (sg * sqrt(2.0 * 3.14159265358979323846));
  for (int i = threadIdx.x; i < ntau; i += blockDim.x) {
    const double t = tau[i];
    gt[i] = exp(-(t - ts) * (t - ts) / (2.0 * sg * sg)) * inv_norm;
    lt[i] = bb * exp(-(t - 11000.0) * (t - 11000.0) / (2.0 * 2000.0 * 2000.0));
  }
  {
    const int q = q0 + threadIdx.x;
    if (q < nk) {
      const double kk = k[q];
      ak[threadIdx.x] = cos(kk * rs + phi) * exp(-(kk / kd) * (kk / kd));
      ek[threadIdx.x] = exp(-kk / 0.01);
      P[(size_t)m * nk + q] = exp((double)f[8]) * 1e-10 * pow(kk / 0.05, (double)f[7] - 1.0);
    }
  }
  __syncthreads();
  const int nq = min(256, nk - q0);
  for (int qq = 0; qq < nq; ++qq) {
    const double a = ak[qq], b = ek[qq];
    float *row = S + ((size_t)m * nk + q0 + qq) * ntau;
    for (int i = threadIdx.x; i < ntau; i += blockDim.x) row[i] = (float)fma(gt[i], a, lt[i] * b);
  }
}

// ---------------------------------------------------------------- GEMM launcher

// Launch of a kernel of the chain behind the one before it (see pdl_wait); what
// that one's launch may have left as an error is returned too.
template <typename... P, typename... A>
cudaError_t chain_launch(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  if (cudaError_t e = cudaGetLastError()) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

template <int EPI, bool AMN, bool BMN, int NP, bool PS>
int gemm_ps(const GemmArgs<NP> &a, int grid, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(gemm_kernel<EPI, AMN, BMN, NP, PS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       gemm_smem(EPI, PS));
  if (e != cudaSuccess) return cuda_fail(e, "emu: gemm smem attribute");
  return ck(chain_launch(gemm_kernel<EPI, AMN, BMN, NP, PS>, dim3(grid), dim3(kGemmThreads), gemm_smem(EPI, PS), st, a),
            "emu: gemm launch");
}

// One tile a CTA where every tile has an SM to itself, else persistent CTAs
// (see emu_gemm.cuh).
template <int EPI, bool AMN, bool BMN, int NP>
int gemm(const GemmArgs<NP> &a, int tiles, cudaStream_t st) {
  return tiles <= kSms ? gemm_ps<EPI, AMN, BMN, NP, false>(a, tiles, st)
                       : gemm_ps<EPI, AMN, BMN, NP, true>(a, kSms, st);
}

// Rows and tiles of a problem: C[M][N] over K.
int set_prob(Prob &p, int M, int N, int K, int first_tile) {
  p.M = M;
  p.N = N;
  p.K = K;
  p.tiles_n = (N + 127) / 128;
  p.tile_end = first_tile + (M + 127) / 128 * p.tiles_n;
  return p.tile_end;
}

int pad8(int n) { return (n + 7) & ~7; }

// Tensor map of a bf16 matrix [rows][cols] with padded rows of ld elements:
// boxes of 64 columns by `box` rows, 128-byte swizzle, zero beyond its extents.
int encode_bf16(CUtensorMap *tm, const __nv_bfloat16 *p, int rows, int cols, int ld, int box) {
  auto fn = reinterpret_cast<CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                          const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                          CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                          CUtensorMapFloatOOBfill)>(tensor_map_encoder());
  if (!fn) return fail(GCAMB_ECUDA, "emu: cuTensorMapEncodeTiled is not available from the driver");
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t boxes[2] = {64, (cuuint32_t)box};
  const cuuint32_t es[2] = {1, 1};
  const CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(p), dims, strides, boxes, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(GCAMB_ECUDA, "emu: tensor map rejected (" + std::to_string((int)r) + ")");
  return GCAMB_OK;
}

// The handle's tensor maps for batch size B.  K-major operands are copied in
// boxes of 128 rows x 64 k, MN-major ones in boxes of 64 k x 64 rows.
int ensure_maps(gcamb_emu *e, int B) {
  if (e->maps_B == B) return GCAMB_OK;
  const int L = e->depth + 1;
  e->maps.resize(L);
  e->maps_B = 0;
  for (int l = 0; l < L; ++l) {
    auto &m = e->maps[l];
    const int nin = e->sizes[l], nout = e->sizes[l + 1];
    int rc;
    if ((rc = encode_bf16(&m.act_k, e->act[l], B, nin, pad8(nin), 128)) ||
        (rc = encode_bf16(&m.act_mn, e->act[l], B, nin, pad8(nin), 64)) ||
        (rc = encode_bf16(&m.d_k, e->dB[l], B, nout, pad8(nout), 128)) ||
        (rc = encode_bf16(&m.d_mn, e->dB[l], B, nout, pad8(nout), 64)) ||
        (rc = encode_bf16(&m.w_k, e->W[l], nout, nin, pad8(nin), 128)) ||
        (rc = encode_bf16(&m.w_mn, e->W[l], nout, nin, pad8(nin), 64)))
      return rc;
  }
  e->maps_B = B;
  return GCAMB_OK;
}

AdamLayers layers_of(const gcamb_emu *e) {
  AdamLayers al{};
  for (int l = 0; l <= e->depth; ++l) {
    al.w_off[l] = e->w_off[l];
    al.end[l] = e->b_off[l] + e->sizes[l + 1];
    al.nw[l] = (unsigned)((size_t)e->sizes[l + 1] * e->sizes[l]);
    al.nin[l] = e->sizes[l];
    al.ld[l] = pad8(e->sizes[l]);
    al.Wb[l] = e->W[l];
  }
  return al;
}

// bf16 copies of all weights (after the parameters were written as a whole), in
// one launch: one a layer took a caller that sets the parameters of nine layers
// from 31 to 74 us, now 44.
int refresh_weights(gcamb_emu *e, cudaStream_t st) {
  const AdamLayers al = layers_of(e);
  unsigned most = 0;
  for (int l = 0; l <= e->depth; ++l) most = std::max(most, al.nw[l]);
  weights_bf16_kernel<<<dim3(std::min(512u, (most + 255) / 256), e->depth + 1), 256, 0, st>>>(e->theta, al);
  return ck(cudaGetLastError(), "emu: weight copies");
}

// Forward pass of B rows, the output as FP32 to out [B][n_out], as C_l to CD
// [B][n_out], or (Y: training) as the loss gradient and its partial sums, with
// the hidden pre-activations kept.
int forward_pass(gcamb_emu *e, const float *X, const int *idx, int B, const float *Y, float *out, double *CD,
                 cudaStream_t st) {
  const int L = e->depth + 1;
  if (int rc = ensure_maps(e, B)) return rc;
  {
    const int n = B * e->n_in;
    standardize_kernel<<<(n + 255) / 256, 256, 0, st>>>(X, idx, B, e->n_in, e->mu_x, e->isd_x, e->act[0],
                                                        pad8(e->n_in));
  }
  for (int l = 0; l < L; ++l) {
    const int nin = e->sizes[l], nout = e->sizes[l + 1];
    GemmArgs<1> a{};
    Prob &p = a.p[0];
    p.ta = e->maps[l].act_k;
    p.tb = e->maps[l].w_k;
    const int tiles = set_prob(p, B, nout, nin, 0);
    a.np = 1;
    p.bias = e->theta + e->b_off[l];
    a.err = e->err;
    int rc;
    if (l < L - 1) {
      p.C = Y ? e->Z[l] : nullptr;
      p.ldc = pad8(nout);
      p.Cb = e->act[l + 1];
      p.ldb = pad8(nout);
      rc = gemm<kGelu, false, false, 1>(a, tiles, st);
    } else if (CD) {
      a.ex = ExpArgs{CD, e->mu_y, e->sd_y, X, e->mu_x, e->n_in, amp_col(e), e->exp_tab};
      rc = gemm<kExp, false, false, 1>(a, tiles, st);
    } else if (Y) {
      p.C = e->dF[l];
      p.ldc = p.ldb = pad8(nout);
      p.Cb = e->dB[l];
      a.ls = LossArgs{Y, idx, 2.f / (float)((size_t)B * nout), e->loss_part};
      rc = gemm<kLoss, false, false, 1>(a, tiles, st);
    } else {
      p.C = out;
      p.ldc = nout;
      rc = gemm<kBias, false, false, 1>(a, tiles, st);
    }
    if (rc) return rc;
  }
  return GCAMB_OK;
}

// 2^(j / kExpTab) as Q2.62, from the series of exp(x ln 2) in double-double
// arithmetic (products by fused multiply-add).
void exp2_table(unsigned long long *tab) {
  const double ln2h = 0x1.62e42fefa39efp-1, ln2l = 0x1.abc9e3b39803fp-56;
  for (int i = 0; i < kExpTab; ++i) {
    const double f = i / (double)kExpTab;  // exact
    const double xh = f * ln2h, xl = std::fma(f, ln2h, -xh) + f * ln2l;
    double sh = 1.0, sl = 0.0;  // Horner: s = 1 + x/n s
    for (int n = 26; n >= 1; --n) {
      // t = x s
      const double th = xh * sh, tl = std::fma(xh, sh, -th) + (xh * sl + xl * sh);
      // t / n
      const double qh = th / n, ql = (std::fma(-qh, (double)n, th) + tl) / n;
      // 1 + q
      const double uh = 1.0 + qh, ul = (1.0 - uh) + qh + ql;
      sh = uh + ul;
      sl = ul - (sh - uh);
    }
    const double scale = 4611686018427387904.0;  // 2^62: sh in [1, 2) is an integer there
    tab[i] = (unsigned long long)(sh * scale) + (unsigned long long)(long long)std::nearbyint(sl * scale);
  }
}

int check_emu(const gcamb_emu *e, int B) {
  if (!e) return fail(GCAMB_EINVAL, "emu: NULL handle");
  if (B < 1 || B > e->max_batch) return fail(GCAMB_EINVAL, "emu: batch must be in [1, max_batch]");
  return GCAMB_OK;
}

}  // namespace

extern "C" {

int gcamb_emu_create(gcamb_grid *g, int n_in, int width, int depth, int max_batch, uint64_t seed, gcamb_emu **out) {
  if (!out) return fail(GCAMB_EINVAL, "emu_create: out is NULL");
  *out = nullptr;
  if (!g) return fail(GCAMB_EINVAL, "emu_create: NULL grid");
  if (n_in != 9) return fail(GCAMB_EINVAL, "emu_create: the source generator has 9 features");
  if (width < 16 || width > 4096 || depth < 1 || depth > 8) return fail(GCAMB_EINVAL, "emu_create: width/depth");
  if (max_batch < 1 || max_batch > (1 << 20)) return fail(GCAMB_EINVAL, "emu_create: max_batch");
  int rc = ensure_device_grid(g);
  if (rc) return rc;
  gcamb_emu *e = new (std::nothrow) gcamb_emu();
  if (!e) return fail(GCAMB_ENOMEM, "emu_create: host allocation");
  e->g = g;
  e->n_in = n_in;
  e->width = width;
  e->depth = depth;
  e->n_out = g->nl;
  e->max_batch = max_batch;
  e->sizes.push_back(n_in);
  for (int d = 0; d < depth; ++d) e->sizes.push_back(width);
  e->sizes.push_back(e->n_out);
  size_t o = 0;
  for (size_t l = 0; l + 1 < e->sizes.size(); ++l) {
    e->w_off.push_back(o);
    o += (size_t)e->sizes[l + 1] * e->sizes[l];
    e->b_off.push_back(o);
    o += e->sizes[l + 1];
  }
  e->n_params = o;
  const size_t mb = (size_t)max_batch;
  rc = GCAMB_OK;
  auto bf16_buf = [&](std::vector<__nv_bfloat16 *> &v, size_t n) {
    __nv_bfloat16 *q = nullptr;
    if (!rc) rc = dalloc(&q, n);
    v.push_back(q);
  };
  auto f32_buf = [&](std::vector<float *> &v, size_t n) {
    float *q = nullptr;
    if (!rc) rc = dalloc(&q, n);
    v.push_back(q);
  };
  for (int l = 0; l <= depth; ++l) {
    const int nin = e->sizes[l], nout = e->sizes[l + 1];
    bf16_buf(e->W, (size_t)nout * pad8(nin));
    bf16_buf(e->act, mb * pad8(nin));
    bf16_buf(e->dB, mb * pad8(nout));
    f32_buf(e->dF, mb * pad8(nout));
    if (l < depth) f32_buf(e->Z, mb * pad8(nout));
  }
  if (rc || (rc = dalloc(&e->theta, o)) || (rc = dalloc(&e->grad, o)) || (rc = dalloc(&e->m, o)) ||
      (rc = dalloc(&e->v, o)) || (rc = dalloc(&e->mu_x, n_in)) || (rc = dalloc(&e->isd_x, n_in)) ||
      (rc = dalloc(&e->mu_y, e->n_out)) || (rc = dalloc(&e->sd_y, e->n_out)) ||
      (rc = dalloc(&e->loss_part, ((mb + 127) / 128) * ((e->n_out + 127) / 128) * kEpiWarpsG)) ||
      (rc = dalloc(&e->err, 1)) || (rc = dalloc(&e->exp_tab, kExpTab))) {
    gcamb_emu_destroy(e);
    return rc;
  }
  if (cudaHostAlloc(reinterpret_cast<void **>(&e->flags_host), mb * sizeof(int), cudaHostAllocMapped) != cudaSuccess ||
      cudaHostGetDevicePointer(reinterpret_cast<void **>(&e->flags_dev), e->flags_host, 0) != cudaSuccess) {
    cudaGetLastError();
    gcamb_emu_destroy(e);
    return fail(GCAMB_ENOMEM, "emu_create: mapped flags");
  }
  {
    std::vector<unsigned long long> tab(kExpTab);
    exp2_table(tab.data());
    if ((rc = ck(cudaMemcpy(e->exp_tab, tab.data(), kExpTab * sizeof(unsigned long long), cudaMemcpyHostToDevice), "emu_create: tables"))) {
      gcamb_emu_destroy(e);
      return rc;
    }
  }
  // parameters U(-1/sqrt(fan_in), 1/sqrt(fan_in)); identity normalisation
  for (size_t l = 0; l + 1 < e->sizes.size(); ++l) {
    const float bound = 1.f / sqrtf((float)e->sizes[l]);
    const size_t nw = (size_t)e->sizes[l + 1] * e->sizes[l];
    init_uniform_kernel<<<256, 256>>>(e->theta + e->w_off[l], nw, bound, seed, e->w_off[l]);
    init_uniform_kernel<<<64, 256>>>(e->theta + e->b_off[l], e->sizes[l + 1], bound, seed, e->b_off[l]);
  }
  if ((rc = refresh_weights(e, nullptr))) {
    gcamb_emu_destroy(e);
    return rc;
  }
  cudaMemset(e->m, 0, o * sizeof(float));
  cudaMemset(e->v, 0, o * sizeof(float));
  cudaMemset(e->err, 0, sizeof(int));
  std::vector<float> zeros(std::max(n_in, e->n_out), 0.f), ones(std::max(n_in, e->n_out), 1.f);
  cudaMemcpy(e->mu_x, zeros.data(), n_in * sizeof(float), cudaMemcpyHostToDevice);
  cudaMemcpy(e->isd_x, ones.data(), n_in * sizeof(float), cudaMemcpyHostToDevice);
  cudaMemcpy(e->mu_y, zeros.data(), e->n_out * sizeof(float), cudaMemcpyHostToDevice);
  rc = ck(cudaMemcpy(e->sd_y, ones.data(), e->n_out * sizeof(float), cudaMemcpyHostToDevice), "emu_create: init");
  if (rc) {
    gcamb_emu_destroy(e);
    return rc;
  }
  *out = e;
  return GCAMB_OK;
}

int gcamb_emu_destroy(gcamb_emu *e) {
  if (!e) return GCAMB_OK;
  for (void *p : {(void *)e->theta, (void *)e->grad, (void *)e->m, (void *)e->v, (void *)e->mu_x, (void *)e->isd_x,
                  (void *)e->mu_y, (void *)e->sd_y, (void *)e->loss_part,
                  (void *)e->err, (void *)e->exp_tab, (void *)e->d_cell_dim, (void *)e->d_cell_mid,
                  (void *)e->d_trusted, (void *)e->fb_x, (void *)e->fb_S, (void *)e->fb_P, (void *)e->fb_C,
                  (void *)e->fb_idx, e->fb_ws})
    cudaFree(p);
  for (auto *v : {&e->W, &e->act, &e->dB})
    for (__nv_bfloat16 *p : *v) cudaFree(p);
  for (auto *v : {&e->Z, &e->dF})
    for (float *p : *v) cudaFree(p);
  if (e->flags_host) cudaFreeHost(e->flags_host);
  delete e;
  return GCAMB_OK;
}

int gcamb_emu_num_params(const gcamb_emu *e, size_t *n) {
  if (!e || !n) return fail(GCAMB_EINVAL, "emu_num_params: NULL argument");
  *n = e->n_params;
  return GCAMB_OK;
}

int gcamb_emu_params(gcamb_emu *e, float *host_out, const float *host_in) {
  if (!e) return fail(GCAMB_EINVAL, "emu_params: NULL handle");
  const size_t bytes = e->n_params * sizeof(float);
  if (host_in) {
    int rc = ck(cudaMemcpy(e->theta, host_in, bytes, cudaMemcpyHostToDevice), "emu_params: upload");
    if (!rc) rc = refresh_weights(e, nullptr);
    if (!rc) rc = ck(cudaStreamSynchronize(nullptr), "emu_params: weight copies");
    if (rc) return rc;
  }
  if (host_out) return ck(cudaMemcpy(host_out, e->theta, bytes, cudaMemcpyDeviceToHost), "emu_params: download");
  return GCAMB_OK;
}

int gcamb_emu_grads(gcamb_emu *e, float *host_out) {
  if (!e || !host_out) return fail(GCAMB_EINVAL, "emu_grads: NULL argument");
  return ck(cudaMemcpy(host_out, e->grad, e->n_params * sizeof(float), cudaMemcpyDeviceToHost), "emu_grads");
}

int gcamb_emu_norm(gcamb_emu *e, float *mu_x, float *sd_x, float *mu_y, float *sd_y, int set) {
  if (!e) return fail(GCAMB_EINVAL, "emu_norm: NULL handle");
  if (set) {
    if (!mu_x || !sd_x || !mu_y || !sd_y) return fail(GCAMB_EINVAL, "emu_norm: NULL array");
    std::vector<float> isd(e->n_in);
    for (int j = 0; j < e->n_in; ++j) isd[j] = sd_x[j] > 1e-12f ? 1.f / sd_x[j] : 0.f;
    cudaMemcpy(e->mu_x, mu_x, e->n_in * sizeof(float), cudaMemcpyHostToDevice);
    cudaMemcpy(e->isd_x, isd.data(), e->n_in * sizeof(float), cudaMemcpyHostToDevice);
    cudaMemcpy(e->mu_y, mu_y, e->n_out * sizeof(float), cudaMemcpyHostToDevice);
    return ck(cudaMemcpy(e->sd_y, sd_y, e->n_out * sizeof(float), cudaMemcpyHostToDevice), "emu_norm: upload");
  }
  std::vector<float> isd(e->n_in);
  if (mu_x) cudaMemcpy(mu_x, e->mu_x, e->n_in * sizeof(float), cudaMemcpyDeviceToHost);
  if (sd_x) {
    cudaMemcpy(isd.data(), e->isd_x, e->n_in * sizeof(float), cudaMemcpyDeviceToHost);
    for (int j = 0; j < e->n_in; ++j) sd_x[j] = isd[j] > 0.f ? 1.f / isd[j] : 0.f;
  }
  if (mu_y) cudaMemcpy(mu_y, e->mu_y, e->n_out * sizeof(float), cudaMemcpyDeviceToHost);
  if (sd_y) cudaMemcpy(sd_y, e->sd_y, e->n_out * sizeof(float), cudaMemcpyDeviceToHost);
  return ck(cudaGetLastError(), "emu_norm: download");
}

// Replaces every sd_y[j] by the root mean square of the per-l deviations, so
// that the loss weighs each multipole's error in nats (log C_l) equally.
__global__ void global_scale_kernel(float *__restrict__ sd, int n) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double s = 0.0;
    for (int j = 0; j < n; ++j) s += (double)sd[j] * sd[j];
    const float r = (float)sqrt(s / n);
    for (int j = 0; j < n; ++j) sd[j] = r;
  }
}

int gcamb_emu_fit_norm(gcamb_emu *e, const float *X, const double *Cl, int N, int per_l, float *Y, void *stream) {
  if (!e || !X || !Cl || !Y) return fail(GCAMB_EINVAL, "emu_fit_norm: NULL argument");
  if (N < 2) return fail(GCAMB_EINVAL, "emu_fit_norm: need at least 2 samples");
  cudaStream_t st = (cudaStream_t)stream;
  float *sdx = nullptr;
  int rc = dalloc(&sdx, e->n_in);
  if (rc) return rc;
  colstats_kernel<<<1, 32, 0, st>>>(X, N, e->n_in, e->mu_x, sdx);
  inv_sd_kernel<<<1, 32, 0, st>>>(sdx, e->n_in, e->isd_x);
  log_kernel<<<1024, 256, 0, st>>>(Cl, (size_t)N, e->n_out, X, e->n_in, amp_col(e), e->mu_x, Y);
  colstats_kernel<<<(e->n_out + 127) / 128, 128, 0, st>>>(Y, N, e->n_out, e->mu_y, e->sd_y);
  if (!per_l) global_scale_kernel<<<1, 32, 0, st>>>(e->sd_y, e->n_out);
  standardize_y_kernel<<<1024, 256, 0, st>>>(Y, N, e->n_out, e->mu_y, e->sd_y);
  rc = ck(cudaGetLastError(), "emu_fit_norm: launch");
  cudaStreamSynchronize(st);
  cudaFree(sdx);
  return rc;
}

int gcamb_emu_forward(gcamb_emu *e, const float *X, int B, float *Y, void *stream) {
  int rc = check_emu(e, B);
  if (rc) return rc;
  if (!X || !Y) return fail(GCAMB_EINVAL, "emu_forward: NULL pointer");
  cudaStream_t st = (cudaStream_t)stream;
  return forward_pass(e, X, nullptr, B, nullptr, Y, nullptr, st);
}

int gcamb_emu_train_step(gcamb_emu *e, const float *X, const float *Y, const int *idx, int B, float lr, float *loss,
                         void *stream) {
  int rc = check_emu(e, B);
  if (rc) return rc;
  if (!X || !Y) return fail(GCAMB_EINVAL, "emu_train_step: NULL pointer");
  cudaStream_t st = (cudaStream_t)stream;
  const int L = e->depth + 1;
  if ((rc = forward_pass(e, X, idx, B, Y, nullptr, nullptr, st))) return rc;
  // d of layer l-1 [b][i] = (sum_o d_l[b][o] W_l[o][i]) GELU'(Z_{l-1}[b][i])
  for (int l = L - 1; l >= 1; --l) {
    const int nin = e->sizes[l], nout = e->sizes[l + 1];
    GemmArgs<1> a{};
    Prob &p = a.p[0];
    p.ta = e->maps[l].d_k;
    p.tb = e->maps[l].w_mn;
    const int tiles = set_prob(p, B, nin, nout, 0);
    a.np = 1;
    p.C = e->dF[l - 1];
    p.ldc = pad8(nin);
    p.Cb = e->dB[l - 1];
    p.ldb = pad8(nin);
    p.Z = e->Z[l - 1];
    a.err = e->err;
    if ((rc = gemm<kDGelu, false, true, 1>(a, tiles, st))) return rc;
  }
  // dW_l[o][i] = sum_b d_l[b][o] h_l[b][i], every layer in one launch
  {
    GemmArgs<kMaxLayers> a{};
    int tiles = 0;
    for (int l = L - 1; l >= 0; --l) {
      const int nin = e->sizes[l], nout = e->sizes[l + 1];
      Prob &p = a.p[a.np++];
      p.ta = e->maps[l].d_mn;
      p.tb = e->maps[l].act_mn;
      tiles = set_prob(p, nout, nin, B, tiles);
      p.C = e->grad + e->w_off[l];
      p.ldc = nin;
    }
    a.err = e->err;
    if ((rc = gemm<kSliced, true, true, kMaxLayers>(a, tiles, st))) return rc;
  }
  {
    BiasSums bs{};
    int nmax = 0;
    for (int l = 0; l < L; ++l) {
      bs.d[l] = e->dF[l];
      bs.db[l] = e->grad + e->b_off[l];
      bs.N[l] = e->sizes[l + 1];
      bs.ld[l] = pad8(e->sizes[l + 1]);
      nmax = std::max(nmax, bs.N[l]);
    }
    bs.part = e->loss_part;
    bs.nparts = ((B + 127) / 128) * ((e->n_out + 127) / 128) * kEpiWarpsG;
    bs.inv_total = 1.f / ((float)B * e->n_out);
    bs.loss = loss;
    if ((rc = ck(chain_launch(bias_kernel, dim3((nmax + kSumCols - 1) / kSumCols, L + 1), dim3(kSumCols * kSumClasses),
                              0, st, bs, B, L),
                 "emu_train_step: bias gradients")))
      return rc;
  }
  ++e->step;
  const float b1 = 0.9f, b2 = 0.999f;
  const float bc1 = 1.f - powf(b1, (float)e->step), bc2 = 1.f - powf(b2, (float)e->step);
  const AdamLayers al = layers_of(e);
  size_t most = 0;
  for (int l = 0; l < L; ++l) most = std::max(most, al.end[l] - al.w_off[l]);
  const unsigned blocks = (unsigned)std::min<size_t>(4096, (most + 1023) / 1024);
  return ck(chain_launch(adam_kernel, dim3(blocks, L), dim3(256), 0, st, e->theta, e->grad, e->m, e->v, al, lr, b1, b2,
                         1e-8f, bc1, bc2),
            "emu_train_step: Adam");
}

int gcamb_synth_sources(const gcamb_grid *g, const float *X, int M, float *S, double *Pk, void *stream) {
  if (!g || (M > 0 && (!X || !S || !Pk))) return fail(GCAMB_EINVAL, "synth_sources: NULL argument");
  if (M < 0 || M > 65535) return fail(GCAMB_EINVAL, "synth_sources: M out of range");
  if (M == 0) return GCAMB_OK;
  int rc = ensure_device_grid(const_cast<gcamb_grid *>(g));
  if (rc) return rc;
  const size_t smem = (2 * (size_t)g->ntau + 512) * sizeof(double);
  if (smem > (size_t)kDynSmem) return fail(GCAMB_EINVAL, "synth_sources: tau grid too long");
  cudaError_t ea = cudaFuncSetAttribute(synth_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmem);
  if (ea != cudaSuccess) return cuda_fail(ea, "synth_sources: smem attribute");
  dim3 grid((g->nk + 255) / 256, M);
  synth_kernel<<<grid, 256, smem, (cudaStream_t)stream>>>(X, g->d_k, g->d_tau, g->nk, g->ntau, S, Pk);
  return ck(cudaGetLastError(), "synth_sources: launch");
}

int gcamb_emu_check(gcamb_emu *e, const float *X, const double *Cl_ref, int N, double tol, int min_count,
                    double *report, void *stream) {
  if (!e || !X || !Cl_ref || !report) return fail(GCAMB_EINVAL, "emu_check: NULL argument");
  if (N < 1 || N > e->max_batch) return fail(GCAMB_EINVAL, "emu_check: N must be in [1, max_batch]");
  cudaStream_t st = (cudaStream_t)stream;
  std::vector<float> hx((size_t)N * e->n_in);
  int rc = ck(cudaMemcpy(hx.data(), X, hx.size() * sizeof(float), cudaMemcpyDeviceToHost), "emu_check: features");
  if (rc) return rc;
  // per-spectrum errors first
  std::vector<double> he(N);
  {
    double *d_err = nullptr, *d_ce = nullptr;
    if ((rc = dalloc(&d_err, N)) || (rc = dalloc(&d_ce, (size_t)N * e->n_out))) {
      cudaFree(d_err);
      return rc;
    }
    if (!(rc = forward_pass(e, X, nullptr, N, nullptr, nullptr, d_ce, st))) {
      maxrel_kernel<<<N, 256, 0, st>>>(d_ce, Cl_ref, e->n_out, d_err);
      rc = ck(cudaStreamSynchronize(st), "emu_check: kernels");
      if (!rc) rc = ck(cudaMemcpy(he.data(), d_err, N * sizeof(double), cudaMemcpyDeviceToHost), "emu_check: errors");
    }
    cudaFree(d_err);
    cudaFree(d_ce);
    if (rc) return rc;
  }
  // cells: split the (at most 4) features whose two halves at the held-out
  // median differ most in mean log error
  struct Cand {
    double score;
    int j;
    float med;
  };
  std::vector<Cand> cands;
  for (int j = 0; j < e->n_in; ++j) {
    std::vector<float> col(N);
    for (int i = 0; i < N; ++i) col[i] = hx[(size_t)i * e->n_in + j];
    std::vector<float> srt(col);
    std::nth_element(srt.begin(), srt.begin() + N / 2, srt.end());
    const float med = srt[N / 2];
    double s0 = 0, s1 = 0;
    int n0 = 0, n1 = 0;
    for (int i = 0; i < N; ++i) {
      const double le = std::log(std::max(he[i], 1e-300));
      if (col[i] > med) {
        s1 += le;
        ++n1;
      } else {
        s0 += le;
        ++n0;
      }
    }
    if (n0 && n1) cands.push_back({std::fabs(s1 / n1 - s0 / n0), j, med});
  }
  std::stable_sort(cands.begin(), cands.end(), [](const Cand &a, const Cand &b) { return a.score > b.score; });
  e->cell_dim.clear();
  e->cell_mid.clear();
  for (size_t c = 0; c < cands.size() && c < 4; ++c) {
    e->cell_dim.push_back(cands[c].j);
    e->cell_mid.push_back(cands[c].med);
  }
  const int nd = (int)e->cell_dim.size(), ncell = 1 << nd;
  cudaFree(e->d_cell_dim);
  cudaFree(e->d_cell_mid);
  cudaFree(e->d_trusted);
  e->d_cell_dim = nullptr;
  e->d_cell_mid = nullptr;
  e->d_trusted = nullptr;
  if ((rc = dalloc(&e->d_cell_dim, std::max(1, nd))) || (rc = dalloc(&e->d_cell_mid, std::max(1, nd))) ||
      (rc = dalloc(&e->d_trusted, ncell)))
    return rc;
  cudaMemcpy(e->d_cell_dim, e->cell_dim.data(), nd * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(e->d_cell_mid, e->cell_mid.data(), nd * sizeof(float), cudaMemcpyHostToDevice);
  std::vector<int> hc(N, 0);
  for (int i = 0; i < N; ++i)
    for (int d = 0; d < nd; ++d)
      if (hx[(size_t)i * e->n_in + e->cell_dim[d]] > e->cell_mid[d]) hc[i] |= 1 << d;
  std::vector<double> cmax(ncell, 0.0);
  std::vector<int> cnt(ncell, 0);
  double emax = 0.0, esum = 0.0;
  int within = 0;
  for (int i = 0; i < N; ++i) {
    cmax[hc[i]] = std::max(cmax[hc[i]], he[i]);
    cnt[hc[i]]++;
    emax = std::max(emax, he[i]);
    esum += he[i];
    within += he[i] <= tol;
  }
  e->trusted.assign(ncell, 0);
  int ntr = 0;
  double served = 0.0;
  for (int c = 0; c < ncell; ++c) {
    e->trusted[c] = (cnt[c] >= std::max(1, min_count) && cmax[c] <= tol) ? 1 : 0;
    ntr += e->trusted[c];
    if (e->trusted[c]) served += cnt[c];
  }
  cudaMemcpy(e->d_trusted, e->trusted.data(), ncell, cudaMemcpyHostToDevice);
  e->check_max_err = emax;
  e->check_tol = tol;
  report[0] = emax;                     // max rel err over all held-out spectra
  report[1] = esum / N;                 // mean of the per-spectrum max rel err
  report[2] = (double)within / N;       // fraction of held-out spectra within tol
  report[3] = (double)ntr / ncell;      // fraction of cells trusted
  report[4] = served / N;               // fraction of held-out spectra in trusted cells
  report[5] = ncell;
  return GCAMB_OK;
}

int gcamb_emulate(gcamb_emu *e, const float *X, int B, double *Cl, int *used_fallback, void *stream) {
  int rc = check_emu(e, B);
  if (rc) return rc;
  if (!X || !Cl || !used_fallback) return fail(GCAMB_EINVAL, "emulate: NULL pointer");
  cudaStream_t st = (cudaStream_t)stream;
  // the cell of every request first: its flags land in mapped host memory while the network runs
  const int nd = (int)e->cell_dim.size();
  cell_kernel<<<(B + 255) / 256, 256, 0, st>>>(X, B, e->n_in, e->d_cell_dim, e->d_cell_mid, nd, e->d_trusted,
                                               used_fallback, e->flags_dev);
  if ((rc = forward_pass(e, X, nullptr, B, nullptr, nullptr, Cl, st))) return rc;
  if ((rc = ck(cudaStreamSynchronize(st), "emulate: sync"))) return rc;
  // requests outside the trusted cells: the batched projection on regenerated sources
  const volatile int *hf = e->flags_host;
  std::vector<int> idx;
  for (int b = 0; b < B; ++b)
    if (hf[b]) idx.push_back(b);
  if (idx.empty()) return GCAMB_OK;
  const int Mf = (int)idx.size();
  gcamb_grid *g = e->g;
  const int mode = e->fb_mode;
  if (!g->tab[mode].built && (rc = gcamb_bessel_table(g, mode, stream))) return rc;
  if (Mf > e->fb_cap) {
    for (void *p : {(void *)e->fb_x, (void *)e->fb_S, (void *)e->fb_P, (void *)e->fb_C, (void *)e->fb_idx}) cudaFree(p);
    e->fb_x = nullptr;
    e->fb_S = nullptr;
    e->fb_P = nullptr;
    e->fb_C = nullptr;
    e->fb_idx = nullptr;
    e->fb_cap = 0;
    if ((rc = dalloc(&e->fb_x, (size_t)Mf * 9)) || (rc = dalloc(&e->fb_S, (size_t)Mf * g->nk * g->ntau)) ||
        (rc = dalloc(&e->fb_P, (size_t)Mf * g->nk)) || (rc = dalloc(&e->fb_C, (size_t)Mf * g->nl)) ||
        (rc = dalloc(&e->fb_idx, Mf)))
      return rc;
    e->fb_cap = Mf;
  }
  size_t need = 0;
  if ((rc = gcamb_los_cl_workspace(g, Mf, mode, &need))) return rc;
  if (need > e->fb_ws_bytes) {
    cudaFree(e->fb_ws);
    e->fb_ws = nullptr;
    e->fb_ws_bytes = 0;
    if (cudaMalloc(&e->fb_ws, need) != cudaSuccess) {
      e->fb_ws = nullptr;
      return fail(GCAMB_ENOMEM, "emulate: fallback workspace");
    }
    e->fb_ws_bytes = need;
  }
  cudaMemcpyAsync(e->fb_idx, idx.data(), Mf * sizeof(int), cudaMemcpyHostToDevice, st);
  gather_rows_kernel<<<(Mf * 9 + 255) / 256, 256, 0, st>>>(X, e->fb_idx, Mf, 9, e->fb_x);
  if ((rc = gcamb_synth_sources(g, e->fb_x, Mf, e->fb_S, e->fb_P, stream))) return rc;
  if ((rc = gcamb_los_cl(g, e->fb_S, e->fb_P, Mf, mode, e->fb_C, e->fb_ws, e->fb_ws_bytes, stream))) return rc;
  scatter_rows_kernel<<<256, 256, 0, st>>>(e->fb_C, e->fb_idx, Mf, g->nl, Cl);
  return ck(cudaGetLastError(), "emulate: fallback");
}

int gcamb_emu_info(const gcamb_emu *e, double *info) {
  if (!e || !info) return fail(GCAMB_EINVAL, "emu_info: NULL argument");
  info[0] = (double)e->n_params;
  info[1] = (double)e->step;
  info[2] = e->check_max_err;
  info[3] = e->check_tol;
  int ntr = 0;
  for (unsigned char t : e->trusted) ntr += t;
  info[4] = e->trusted.empty() ? 0.0 : (double)ntr / e->trusted.size();
  info[5] = (double)e->n_out;
  int herr = 0;
  cudaMemcpy(&herr, e->err, sizeof(int), cudaMemcpyDeviceToHost);
  info[6] = herr;
  info[7] = (double)e->width;
  return GCAMB_OK;
}

// Checkpoint: magic, version, architecture, step, parameters, Adam moments,
// normalisation, trust cells, then a 64-bit FNV-1a checksum of all of it.
int gcamb_emu_save(const gcamb_emu *e, const char *path) {
  if (!e || !path) return fail(GCAMB_EINVAL, "emu_save: NULL argument");
  std::vector<unsigned char> buf;
  auto put = [&](const void *p, size_t n) {
    const unsigned char *c = static_cast<const unsigned char *>(p);
    buf.insert(buf.end(), c, c + n);
  };
  const uint32_t hdr[6] = {kEmuMagic, 1u, (uint32_t)e->n_in, (uint32_t)e->width, (uint32_t)e->depth,
                           (uint32_t)e->n_out};
  put(hdr, sizeof hdr);
  put(&e->step, sizeof e->step);
  std::vector<float> h(e->n_params);
  for (float *src : {e->theta, e->m, e->v}) {
    cudaMemcpy(h.data(), src, e->n_params * sizeof(float), cudaMemcpyDeviceToHost);
    put(h.data(), h.size() * sizeof(float));
  }
  std::vector<float> nx(e->n_in), ny(e->n_out);
  for (float *src : {e->mu_x, e->isd_x}) {
    cudaMemcpy(nx.data(), src, e->n_in * sizeof(float), cudaMemcpyDeviceToHost);
    put(nx.data(), nx.size() * sizeof(float));
  }
  for (float *src : {e->mu_y, e->sd_y}) {
    cudaMemcpy(ny.data(), src, e->n_out * sizeof(float), cudaMemcpyDeviceToHost);
    put(ny.data(), ny.size() * sizeof(float));
  }
  const int32_t nd = (int32_t)e->cell_dim.size();
  put(&nd, sizeof nd);
  put(e->cell_dim.data(), nd * sizeof(int));
  put(e->cell_mid.data(), nd * sizeof(float));
  const int32_t nt = (int32_t)e->trusted.size();
  put(&nt, sizeof nt);
  put(e->trusted.data(), nt);
  put(&e->check_max_err, sizeof(double));
  put(&e->check_tol, sizeof(double));
  if (cudaGetLastError() != cudaSuccess) return fail(GCAMB_ECUDA, "emu_save: download");
  uint64_t hsum = 1469598103934665603ull;
  for (unsigned char c : buf) {
    hsum ^= c;
    hsum *= 1099511628211ull;
  }
  FILE *f = fopen(path, "wb");
  if (!f) return fail(GCAMB_EINVAL, std::string("emu_save: cannot open ") + path);
  const bool ok = fwrite(buf.data(), 1, buf.size(), f) == buf.size() && fwrite(&hsum, 1, 8, f) == 8;
  fclose(f);
  return ok ? GCAMB_OK : fail(GCAMB_EINVAL, "emu_save: write failed");
}

int gcamb_emu_load(gcamb_emu *e, const char *path) {
  if (!e || !path) return fail(GCAMB_EINVAL, "emu_load: NULL argument");
  FILE *f = fopen(path, "rb");
  if (!f) return fail(GCAMB_EINVAL, std::string("emu_load: cannot open ") + path);
  std::vector<unsigned char> buf;
  unsigned char tmp[65536];
  size_t r;
  while ((r = fread(tmp, 1, sizeof tmp, f)) > 0) buf.insert(buf.end(), tmp, tmp + r);
  fclose(f);
  if (buf.size() < 8) return fail(GCAMB_EINVAL, "emu_load: truncated file");
  uint64_t hsum = 1469598103934665603ull, stored;
  for (size_t i = 0; i < buf.size() - 8; ++i) {
    hsum ^= buf[i];
    hsum *= 1099511628211ull;
  }
  std::memcpy(&stored, buf.data() + buf.size() - 8, 8);
  if (hsum != stored) return fail(GCAMB_EINVAL, "emu_load: checksum mismatch");
  size_t pos = 0;
  auto get = [&](void *p, size_t n) -> bool {
    if (pos + n > buf.size() - 8) return false;
    std::memcpy(p, buf.data() + pos, n);
    pos += n;
    return true;
  };
  uint32_t hdr[6];
  if (!get(hdr, sizeof hdr) || hdr[0] != kEmuMagic || hdr[1] != 1u) return fail(GCAMB_EINVAL, "emu_load: not a checkpoint");
  if ((int)hdr[2] != e->n_in || (int)hdr[3] != e->width || (int)hdr[4] != e->depth || (int)hdr[5] != e->n_out)
    return fail(GCAMB_EINVAL, "emu_load: architecture differs from this emulator");
  int64_t step;
  if (!get(&step, sizeof step)) return fail(GCAMB_EINVAL, "emu_load: truncated");
  std::vector<float> h(e->n_params);
  for (float *dst : {e->theta, e->m, e->v}) {
    if (!get(h.data(), h.size() * sizeof(float))) return fail(GCAMB_EINVAL, "emu_load: truncated");
    cudaMemcpy(dst, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice);
  }
  if (int rc = refresh_weights(e, nullptr)) return rc;
  std::vector<float> nx(e->n_in), ny(e->n_out);
  for (float *dst : {e->mu_x, e->isd_x}) {
    if (!get(nx.data(), nx.size() * sizeof(float))) return fail(GCAMB_EINVAL, "emu_load: truncated");
    cudaMemcpy(dst, nx.data(), nx.size() * sizeof(float), cudaMemcpyHostToDevice);
  }
  for (float *dst : {e->mu_y, e->sd_y}) {
    if (!get(ny.data(), ny.size() * sizeof(float))) return fail(GCAMB_EINVAL, "emu_load: truncated");
    cudaMemcpy(dst, ny.data(), ny.size() * sizeof(float), cudaMemcpyHostToDevice);
  }
  int32_t nd = 0, nt = 0;
  if (!get(&nd, sizeof nd) || nd < 0 || nd > 16) return fail(GCAMB_EINVAL, "emu_load: bad cells");
  std::vector<int> cd(nd);
  std::vector<float> cm(nd);
  if (!get(cd.data(), nd * sizeof(int)) || !get(cm.data(), nd * sizeof(float)) || !get(&nt, sizeof nt) ||
      !(nt == (1 << nd) || (nd == 0 && nt == 0)))
    return fail(GCAMB_EINVAL, "emu_load: bad cells");
  std::vector<unsigned char> tr(nt);
  double cmax = 0, ctol = 0;
  if (!get(tr.data(), nt) || !get(&cmax, sizeof cmax) || !get(&ctol, sizeof ctol))
    return fail(GCAMB_EINVAL, "emu_load: truncated");
  e->step = step;
  e->cell_dim = cd;
  e->cell_mid = cm;
  e->trusted = tr;
  e->check_max_err = cmax;
  e->check_tol = ctol;
  cudaFree(e->d_cell_dim);
  cudaFree(e->d_cell_mid);
  cudaFree(e->d_trusted);
  e->d_cell_dim = nullptr;
  e->d_cell_mid = nullptr;
  e->d_trusted = nullptr;
  int rc;
  if ((rc = dalloc(&e->d_cell_dim, std::max(1, nd))) || (rc = dalloc(&e->d_cell_mid, std::max(1, nd))) ||
      (rc = dalloc(&e->d_trusted, std::max(1, nt))))
    return rc;
  cudaMemcpy(e->d_cell_dim, cd.data(), nd * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(e->d_cell_mid, cm.data(), nd * sizeof(float), cudaMemcpyHostToDevice);
  return ck(cudaMemcpy(e->d_trusted, tr.data(), nt, cudaMemcpyHostToDevice), "emu_load: upload");
}

}  // extern "C"
