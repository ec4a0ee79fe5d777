// Row-wise, element-wise and coder kernels of the EDPC step.
//
// Every reduction runs in a fixed order (warp xor-butterflies, then shared
// memory in warp order), and nothing is accumulated with floating-point
// atomics. So the encoder and the decoder, which launch the same kernels on
// the same values, compute bit-identical probabilities and CDFs.
#include <cuda_fp8.h>

#include <algorithm>

#include "kernels.cuh"
#include "launch.cuh"

namespace edpc {

// ============================================================================================
// Initial values: SplitMix64 counter streams (Steele, Lea, Flood, OOPSLA 2014).
// Value idx of tensor tid is output idx+1 of the stream seeded with
// seed + G * tid * 2^32; its top 24 bits k give w = (2k + 1 - 2^24) / 2^24 in
// (-1, 1), exact in FP32, and the value is the FP32 product bound * w.
// ============================================================================================
__device__ __forceinline__ unsigned long long sm64_mix(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void init_values_kernel(float* dst, size_t n, unsigned long long seed, int tid, float bound,
                                   size_t start, float fill) {
  pdl_wait();
  pdl_launch();
  const unsigned long long G = 0x9E3779B97F4A7C15ull;
  const unsigned long long base = seed + G * ((unsigned long long)tid << 32);
  for (size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x; j < n; j += (size_t)gridDim.x * blockDim.x) {
    if (bound < 0.f) {
      dst[j] = fill;
      continue;
    }
    unsigned long long z = sm64_mix(base + G * (start + j + 1));
    int k = (int)(z >> 40);
    float w = (float)(2 * k + 1 - (1 << 24)) * (1.0f / 16777216.0f);
    dst[j] = __fmul_rn(bound, w);
  }
}

cudaError_t launch_init_values(float* dst, size_t n, uint64_t seed, int tid, float bound, size_t start,
                               float fill, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  int grid = (int)((n + 255) / 256);
  if (grid > 152 * 32) grid = 152 * 32;
  return launch_k(init_values_kernel, dim3(grid), dim3(256), 0, st, dst, n, seed, tid, bound, start, fill);
}

// ============================================================================================
// Warp helpers
// ============================================================================================
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ============================================================================================
// Embedding: h0 = concat_k E[x_{i-K+k}] (the model input of Algorithm 1's Model()).
// ============================================================================================
__global__ void embed_kernel(const uint8_t* __restrict__ data, Split sp, const StepCtl* __restrict__ ctl,
                             const float* __restrict__ E, int K, int D, float* __restrict__ X,
                             uint8_t* __restrict__ ctx, const int* __restrict__ rg, size_t gs) {
  pdl_wait();
  pdl_launch();
  const int s = blockIdx.x;
  if (rg) E += (size_t)rg[s] * gs;  // grouped mode: the row's own model
  const int F = K * D;
  // A stream past its end (inactive) keeps its last context: its bytes
  // [i - K, i) would run beyond the stream, and its outputs are masked.
  if (data && ctl->i <= sp.len(s)) {
    const long long base = sp.off(s) + ctl->i - K;
    for (int k = threadIdx.x; k < K; k += blockDim.x) ctx[(size_t)s * K + k] = data[base + k];
    __syncthreads();
  }
  for (int idx = threadIdx.x; idx < F; idx += blockDim.x) {
    int k = idx / D, d = idx - k * D;
    int c = ctx[(size_t)s * K + k];
    X[(size_t)s * F + idx] = E[c * D + d];
  }
}

cudaError_t launch_embed(const uint8_t* data, Split sp, const StepCtl* ctl, const float* E, int b, int K,
                         int D, float* X, uint8_t* ctx, cudaStream_t st, const int* rg, size_t gs) {
  return launch_k(embed_kernel, dim3(b), dim3(128), 0, st, data, sp, ctl, E, K, D, X, ctx, rg, gs);
}

// ============================================================================================
// LayerNorm forward (Eq. 9), one warp per row, two-pass statistics.
// ============================================================================================
__global__ void ln_fwd_kernel(const float* __restrict__ X, const float* __restrict__ g,
                              const float* __restrict__ be, float* __restrict__ xhat,
                              float* __restrict__ rstd, float* __restrict__ X0, int b, int F) {
  pdl_wait();
  pdl_launch();
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= b) return;
  const float* x = X + (size_t)row * F;
  float s = 0.f;
  for (int c = lane; c < F; c += 32) s += x[c];
  const float mean = warp_sum(s) / (float)F;
  float q = 0.f;
  for (int c = lane; c < F; c += 32) {
    float d = x[c] - mean;
    q += d * d;
  }
  const float var = warp_sum(q) / (float)F;
  const float r = 1.0f / sqrtf(var + kLnEps);
  for (int c = lane; c < F; c += 32) {
    float h = (x[c] - mean) * r;
    xhat[(size_t)row * F + c] = h;
    X0[(size_t)row * F + c] = h * g[c] + be[c];
  }
  if (lane == 0) rstd[row] = r;
}

cudaError_t launch_ln_fwd(const float* X, const float* g, const float* be, float* xhat, float* rstd,
                          float* X0, int b, int F, cudaStream_t st) {
  return launch_k(ln_fwd_kernel, dim3(div_up(b, 8)), dim3(256), 0, st, X, g, be, xhat, rstd, X0, b, F);
}

// ============================================================================================
// Column sums over rows of the FP32 path (bias and LN-affine gradients), all of
// a block's tensors in one launch, fixed order: warp w sums rows w, w+8, ...
// for 32 columns; then warps are added in order.
// ============================================================================================
__global__ void __launch_bounds__(256) colsum_kernel(ColsumJobs jobs) {
  pdl_wait();
  pdl_launch();
  __shared__ float part[8][33];
  int t = blockIdx.x, j = 0;
  while (j < jobs.n - 1 && t >= (jobs.job[j].cols + 31) / 32) {
    t -= (jobs.job[j].cols + 31) / 32;
    ++j;
  }
  const ColsumJob jb = jobs.job[j];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = t * 32 + lane;
  float s = 0.f;
  if (c < jb.cols) {
    // the rows' loads go out sixteen at a time; the adds keep their order
    constexpr int U = 16;
    const size_t ld = (size_t)jb.ld;
    const float* x = jb.X + (size_t)w * ld + c;
    const float* y = jb.Y ? jb.Y + (size_t)w * ld + c : nullptr;
    for (int r = w; r < jb.rows; r += 8 * U) {
      const size_t o = (size_t)(r - w) * ld;
      float vx[U], vy[U];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const bool in = r + 8 * q < jb.rows;
        vx[q] = in ? x[o + 8 * q * ld] : 0.f;
        vy[q] = in && y ? y[o + 8 * q * ld] : 0.f;
      }
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (r + 8 * q < jb.rows) s = y ? fmaf(vx[q], vy[q], s) : s + vx[q];
    }
  }
  part[w][lane] = s;
  __syncthreads();
  if (w == 0 && c < jb.cols) {
    float v = part[0][lane];
#pragma unroll
    for (int i = 1; i < 8; ++i) v += part[i][lane];
    jb.out[c] = v;
  }
}

cudaError_t launch_colsum(const ColsumJobs& jobs, cudaStream_t st) {
  int tiles = 0;
  for (int j = 0; j < jobs.n; ++j) tiles += div_up(jobs.job[j].cols, 32);
  return launch_k(colsum_kernel, dim3(tiles), dim3(256), 0, st, jobs);
}

// ============================================================================================
// LayerNorm backward: dX = dRes + rstd * (dxh - mean(dxh) - xhat * mean(dxh * xhat)),
// dxh = dX0 * g; one warp per row.
// ============================================================================================
__global__ void ln_bwd_kernel(const float* __restrict__ dX0, const float* __restrict__ xhat,
                              const float* __restrict__ rstd, const float* __restrict__ g,
                              const float* __restrict__ dRes, float* __restrict__ dX, int b, int F) {
  pdl_wait();
  pdl_launch();
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= b) return;
  const size_t o = (size_t)row * F;
  float s1 = 0.f, s2 = 0.f;
  for (int c = lane; c < F; c += 32) {
    float d = dX0[o + c] * g[c];
    s1 += d;
    s2 += d * xhat[o + c];
  }
  const float m1 = warp_sum(s1) / (float)F;
  const float m2 = warp_sum(s2) / (float)F;
  const float r = rstd[row];
  for (int c = lane; c < F; c += 32) {
    float d = dX0[o + c] * g[c];
    dX[o + c] = dRes[o + c] + r * (d - m1 - xhat[o + c] * m2);
  }
}

cudaError_t launch_ln_bwd(const float* dX0, const float* xhat, const float* rstd, const float* g,
                          const float* dRes, float* dX, int b, int F, cudaStream_t st) {
  return launch_k(ln_bwd_kernel, dim3(div_up(b, 8)), dim3(256), 0, st, dX0, xhat, rstd, g, dRes, dX, b, F);
}

// ============================================================================================
// FDM forward (Eq. 15): y_s[j] = sum_i x'_s[i] U_s[i][j]. One CTA per stream;
// threads own 4 consecutive columns and a row group; row groups are added in order.
// ============================================================================================
// A stream that is past its end (or masked in the model API) has no
// prediction to make: its y is written as zeros and its U_s is not read.
__device__ __forceinline__ bool fdm_row_active(const FdmAct& a, int s) {
  if (!a.ctl) return true;
  return a.active ? a.active[s] != 0 : (long long)a.ctl->i < a.sp.len(s);
}

__device__ __forceinline__ void fdm_zero_row(float* Y, __nv_bfloat16* Yb, __nv_bfloat16* YbT, int ldT, int s,
                                             int Fp) {
  for (int j = threadIdx.x; j < Fp; j += blockDim.x) {
    Y[(size_t)s * Fp + j] = 0.f;
    if (Yb) Yb[(size_t)s * Fp + j] = __float2bfloat16_rn(0.f);
    if (YbT) YbT[(size_t)j * ldT + s] = __float2bfloat16_rn(0.f);
  }
}

__global__ void __launch_bounds__(256) fdm_fwd_kernel(const float* __restrict__ Xp, const float* __restrict__ U,
                                                      float* __restrict__ Y, int Fp, __nv_bfloat16* Yb,
                                                      __nv_bfloat16* YbT, int ldT, FdmAct act) {
  pdl_wait();
  pdl_launch();
  extern __shared__ float sm[];
  float* xs = sm;              // Fp
  float* part = sm + Fp;       // groups x Fp
  const int s = blockIdx.x;
  if (!fdm_row_active(act, s)) {
    fdm_zero_row(Y, Yb, YbT, ldT, s, Fp);
    return;
  }
  const int cols4 = Fp >> 2;
  const int groups = blockDim.x / cols4;
  const int cg = threadIdx.x % cols4, rg = threadIdx.x / cols4;
  for (int i = threadIdx.x; i < Fp; i += blockDim.x) xs[i] = Xp[(size_t)s * Fp + i];
  __syncthreads();
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (rg < groups) {
    const float4* u = reinterpret_cast<const float4*>(U + (size_t)s * Fp * Fp) + cg;
    int i = rg;
#pragma unroll 4
    for (; i < Fp; i += groups) {
      float4 v = __ldcs(u + (size_t)i * cols4);
      float x = xs[i];
      acc.x += x * v.x;
      acc.y += x * v.y;
      acc.z += x * v.z;
      acc.w += x * v.w;
    }
    float* p = part + (size_t)rg * Fp + cg * 4;
    p[0] = acc.x; p[1] = acc.y; p[2] = acc.z; p[3] = acc.w;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < Fp; j += blockDim.x) {
    float t = part[j];
    for (int g = 1; g < groups; ++g) t += part[(size_t)g * Fp + j];
    Y[(size_t)s * Fp + j] = t;
    if (Yb) Yb[(size_t)s * Fp + j] = __float2bfloat16_rn(t);
    if (YbT) YbT[(size_t)j * ldT + s] = __float2bfloat16_rn(t);
  }
}

// Streamed FDM forward helpers (F' in {128, 256, 512, 1024}): TMA bulk copies
// of 16 KB (consecutive rows of U_s are contiguous) into a ring of shared
// memory slots, each with an mbarrier; every wait is bounded.
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void bar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)));
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t parity) {
  for (uint32_t it = 0; it < (1u << 26); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

template <int FP>
struct FdmRing {
  static constexpr int NT = FP < 256 ? FP : 256;     // threads
  static constexpr int CPT = FP / NT;                 // columns per thread
  static constexpr int SROWS = 4096 / FP;             // rows per 16 KB stage
  static constexpr int NST = FP / SROWS;              // stages per stream
  static constexpr int RING = NST < 3 ? NST : 3;
  static constexpr size_t kSmem = (size_t)RING * 16384 + (size_t)FP * 4 + 64;
};

// Persistent FDM forward: kFdmPersistPerSm CTAs per SM walk the streams s =
// blockIdx.x, blockIdx.x + gridDim.x, ...; thread 0 keeps kFdmPersistRing
// 16 KB copies in flight across stream boundaries (no drain between streams,
// no partial last wave). Thread t owns columns t, t + NT, ... of the stream's
// y and sums its rows in increasing i (deterministic, no cross-thread
// reduction).
constexpr int kFdmPersistRing = 6;
constexpr int kFdmPersistPerSm = 2;

template <int FP>
__global__ void __launch_bounds__(FdmRing<FP>::NT)
    fdm_fwd_persist_kernel(const float* __restrict__ Xp, const float* __restrict__ U, float* __restrict__ Y,
                           __nv_bfloat16* Yb, __nv_bfloat16* YbT, int ldT, int* err, FdmAct act, int b) {
  using R = FdmRing<FP>;
  constexpr int RING = kFdmPersistRing;
  extern __shared__ __align__(128) float smf[];
  float* buf = smf;                         // RING x 16 KB
  float* xs = smf + (size_t)RING * 4096;    // FP
  uint64_t* bars = reinterpret_cast<uint64_t*>(xs + FP);
  const int t = threadIdx.x;
  if (t == 0) {
    for (int q = 0; q < RING; ++q) bar_init(&bars[q]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // producer cursor (thread 0): next stream and stage to copy, copies issued
  int ps = blockIdx.x, pst = 0;
  uint32_t issued = 0;
  auto next_active = [&](int s0) {
    int s1 = s0;
    while (s1 < b && !fdm_row_active(act, s1)) s1 += gridDim.x;
    return s1;
  };
  auto issue_one = [&]() {
    if (ps >= b) return;
    const float* src = U + (size_t)ps * FP * FP + (size_t)pst * 4096;
    bulk_load(buf + (size_t)(issued % RING) * 4096, src, 16384u, &bars[issued % RING]);
    ++issued;
    if (++pst == R::NST) {
      pst = 0;
      ps = next_active(ps + gridDim.x);
    }
  };
  // The first copies go out before the dependent-launch wait: U and the step
  // control were written by launches that completed before the preceding
  // launch (whose own wait this one follows) could start; only x' comes from
  // the preceding launch, and every thread reads it after the wait below.
  if (t == 0) {
    ps = next_active(ps);
    for (int q = 0; q < RING; ++q) issue_one();
  }
  pdl_wait();
  pdl_launch();
  uint32_t used = 0;  // copies consumed (same sequence as issued)
  bool ok = true;
  for (int s = blockIdx.x; s < b; s += gridDim.x) {
    if (!fdm_row_active(act, s)) {  // CTA-uniform
      fdm_zero_row(Y, Yb, YbT, ldT, s, FP);
      continue;
    }
    __syncthreads();  // the previous stream's readers are done with xs
    for (int i = t; i < FP; i += R::NT) xs[i] = Xp[(size_t)s * FP + i];
    __syncthreads();
    float acc[R::CPT];
#pragma unroll
    for (int j = 0; j < R::CPT; ++j) acc[j] = 0.f;
    for (int st = 0; st < R::NST; ++st, ++used) {
      const int q = (int)(used % RING);
      ok = bar_wait(&bars[q], (used / RING) & 1u) && ok;
      const float* u = buf + (size_t)q * 4096;
      const float* xv = xs + st * R::SROWS;
#pragma unroll
      for (int r = 0; r < R::SROWS; ++r) {
        const float xr = xv[r];
#pragma unroll
        for (int j = 0; j < R::CPT; ++j) acc[j] += xr * u[r * FP + t + j * R::NT];
      }
      __syncthreads();  // slot q consumed by every thread
      if (t == 0) issue_one();
    }
#pragma unroll
    for (int j = 0; j < R::CPT; ++j) {
      const int c = t + j * R::NT;
      Y[(size_t)s * FP + c] = acc[j];
      if (Yb) Yb[(size_t)s * FP + c] = __float2bfloat16_rn(acc[j]);
      if (YbT) YbT[(size_t)c * ldT + s] = __float2bfloat16_rn(acc[j]);
    }
  }
  if (!ok && t == 0 && err) atomicOr(err, 8);
}

template <int FP>
cudaError_t launch_fdm_fwd_persist(const float* Xp, const float* U, float* Y, int b, __nv_bfloat16* Yb,
                                   __nv_bfloat16* YbT, int ldT, int* err, const FdmAct& act, cudaStream_t st) {
  const size_t smem = (size_t)kFdmPersistRing * 16384 + (size_t)FP * 4 + 64 + 64;
  static OncePerDevice once;
  cudaError_t attr = once_on_device(once, [&] {
    return cudaFuncSetAttribute(fdm_fwd_persist_kernel<FP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  int sms = 0;
  if (attr == cudaSuccess) attr = sm_count(&sms);
  if (attr != cudaSuccess) return attr;
  const int grid = sms * kFdmPersistPerSm;
  const int g = b < grid ? b : grid;
  return launch_k(fdm_fwd_persist_kernel<FP>, dim3(g), dim3(FdmRing<FP>::NT), smem, st, Xp, U, Y, Yb, YbT, ldT, err,
                  act, b);
}

cudaError_t launch_fdm_fwd(const float* Xp, const float* U, float* Y, int b, int Fp, cudaStream_t st,
                           __nv_bfloat16* Yb, __nv_bfloat16* YbT, int ldT, int* err, FdmAct act) {
  switch (Fp) {
    case 128: return launch_fdm_fwd_persist<128>(Xp, U, Y, b, Yb, YbT, ldT, err, act, st);
    case 256: return launch_fdm_fwd_persist<256>(Xp, U, Y, b, Yb, YbT, ldT, err, act, st);
    case 512: return launch_fdm_fwd_persist<512>(Xp, U, Y, b, Yb, YbT, ldT, err, act, st);
    case 1024: return launch_fdm_fwd_persist<1024>(Xp, U, Y, b, Yb, YbT, ldT, err, act, st);
    default: break;
  }
  const int cols4 = Fp / 4;
  const int threads = cols4 >= 256 ? cols4 : (256 / cols4) * cols4;
  const int groups = threads / cols4;
  size_t smem = (size_t)(Fp + groups * Fp) * sizeof(float);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(fdm_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return launch_k(fdm_fwd_kernel, dim3(b), dim3(threads), smem, st, Xp, U, Y, Fp, Yb, YbT, ldT, act);
}

// ============================================================================================
// FDM adjoint + Adam (the per-stream HBM-bound update). One warp per FDM row i;
// lanes own float4 column chunks. For row i of stream s:
//   dx'_s[i] = sum_j U[i][j] dy[j]   (pre-update U, warp reduction in fixed order)
//   g[i][j]  = x'_s[i] dy[j]         (rank-1 gradient of Eq. 15)
//   m, v, U  <- Adam(g)              (bias-corrected, lr from the step control)
// ============================================================================================
constexpr int kFdmRowsPerCta = 32;

__device__ __forceinline__ void adam1(float& p, float& m, float& v, float g, float lr, float bc1, float bc2) {
  m = kB1 * m + (1.0f - kB1) * g;
  v = kB2 * v + (1.0f - kB2) * g * g;
  float mh = m / bc1;
  float vh = v / bc2;
  p = p - lr * mh / (sqrtf(vh) + kAdamEps);
}

// adam1 with the contractions spelled out as the compiler chooses them in the fused
// adjoint (fdm_bwd_kernel<1> and the generic one: G; the wider ones: not G). The
// update that runs on its own stream instead (EDPC_FLAG_OVERLAP_FDM) must give the
// same bits, since the container is decoded by the fused one; left to the compiler
// its kernels contracted other products than the fused ones at most widths.
template <bool G>
__device__ __forceinline__ void adam1_fused(float& p, float& m, float& v, float g, float lr, float bc1, float bc2) {
  m = G ? __fmaf_rn(1.0f - kB1, g, __fmul_rn(kB1, m)) : __fmaf_rn(kB1, m, __fmul_rn(1.0f - kB1, g));
  v = __fmaf_rn(__fmul_rn(1.0f - kB2, g), g, __fmul_rn(kB2, v));
  p = p - lr * (m / bc1) / (sqrtf(v / bc2) + kAdamEps);
}

__device__ __forceinline__ void store_dxp(const FdmBwdArgs& a, int s, int i, float v) {
  a.dXp[(size_t)s * a.Fp + i] = v;
  if (a.dXpb) a.dXpb[(size_t)s * a.Fp + i] = __float2bfloat16_rn(v);
  if (a.dXpbT) a.dXpbT[(size_t)i * a.ldT + s] = __float2bfloat16_rn(v);
}

template <int NCH>  // float4 chunks per lane per row: Fp = 128 * NCH
__global__ void __launch_bounds__(256) fdm_bwd_kernel(FdmBwdArgs a) {
  pdl_wait();
  pdl_launch();
  const int s = blockIdx.y;
  const int Fp = a.Fp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const StepCtl c = *a.ctl;
  bool act = a.active ? (a.active[s] != 0) : ((long long)c.i < a.sp.len(s));
  const int row0 = blockIdx.x * kFdmRowsPerCta;
  if (!act) {
    // dy is zero for an inactive stream, so dx' = 0 and its FDM state is left as is.
    for (int r = warp; r < kFdmRowsPerCta; r += 8)
      if (lane == 0 && row0 + r < Fp) store_dxp(a, s, row0 + r, 0.f);
    if (!a.update) {
      for (int r = warp; r < kFdmRowsPerCta; r += 8) {
        int i = row0 + r;
        if (i >= Fp) break;
        float4* gu = reinterpret_cast<float4*>(a.gU + ((size_t)s * Fp + i) * Fp);
#pragma unroll
        for (int q = 0; q < NCH; ++q) gu[lane + 32 * q] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    return;
  }
  float4 dy[NCH];
#pragma unroll
  for (int q = 0; q < NCH; ++q) dy[q] = reinterpret_cast<const float4*>(a.dY + (size_t)s * Fp)[lane + 32 * q];
  for (int r = warp; r < kFdmRowsPerCta; r += 8) {
    const int i = row0 + r;
    if (i >= Fp) break;
    const float xi = a.Xp[(size_t)s * Fp + i];
    const size_t ro = ((size_t)s * Fp + i) * Fp;
    float4* U4 = reinterpret_cast<float4*>(a.U + ro);
    float dot = 0.f;
    if (a.update) {
      float4* M4 = reinterpret_cast<float4*>(a.Um + ro);
      float4* V4 = reinterpret_cast<float4*>(a.Uv + ro);
      float4 u[NCH], m[NCH], v[NCH];
#pragma unroll
      for (int q = 0; q < NCH; ++q) {
        u[q] = __ldcs(U4 + lane + 32 * q);
        m[q] = __ldcs(M4 + lane + 32 * q);
        v[q] = __ldcs(V4 + lane + 32 * q);
      }
#pragma unroll
      for (int q = 0; q < NCH; ++q) {
        dot += u[q].x * dy[q].x;
        dot += u[q].y * dy[q].y;
        dot += u[q].z * dy[q].z;
        dot += u[q].w * dy[q].w;
        adam1(u[q].x, m[q].x, v[q].x, xi * dy[q].x, c.lr, c.bc1, c.bc2);
        adam1(u[q].y, m[q].y, v[q].y, xi * dy[q].y, c.lr, c.bc1, c.bc2);
        adam1(u[q].z, m[q].z, v[q].z, xi * dy[q].z, c.lr, c.bc1, c.bc2);
        adam1(u[q].w, m[q].w, v[q].w, xi * dy[q].w, c.lr, c.bc1, c.bc2);
        __stcs(U4 + lane + 32 * q, u[q]);
        __stcs(M4 + lane + 32 * q, m[q]);
        __stcs(V4 + lane + 32 * q, v[q]);
      }
    } else {
      float4* G4 = reinterpret_cast<float4*>(a.gU + ro);
#pragma unroll
      for (int q = 0; q < NCH; ++q) {
        float4 u = U4[lane + 32 * q];
        dot += u.x * dy[q].x;
        dot += u.y * dy[q].y;
        dot += u.z * dy[q].z;
        dot += u.w * dy[q].w;
        G4[lane + 32 * q] = make_float4(xi * dy[q].x, xi * dy[q].y, xi * dy[q].z, xi * dy[q].w);
      }
    }
    dot = warp_sum(dot);
    if (lane == 0) store_dxp(a, s, i, dot);
  }
}

// ---- split form: dx' on the critical path, the update on a side stream ------------------------
__device__ __forceinline__ bool fdm_split_active(const FdmSplitArgs& a, int s, long long i) {
  return a.active ? (a.active[s] != 0) : (i < a.sp.len(s));
}

template <int NCH>
__global__ void __launch_bounds__(256) fdm_dx_kernel(FdmSplitArgs a) {
  pdl_wait();
  pdl_launch();
  const int s = blockIdx.y;
  const int Fp = a.Fp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const StepCtl c = *a.ctl;
  const int row0 = blockIdx.x * kFdmRowsPerCta;
  if (blockIdx.x == 0 && s == 0 && threadIdx.x == 0) *a.pend = FdmPend{c.i, c.lr, c.bc1, c.bc2};
  const bool act = fdm_split_active(a, s, c.i);
  if (blockIdx.x == 0 && act) {  // the update's inputs, kept past this step's x' and dy
    for (int j = threadIdx.x; j < Fp; j += blockDim.x) {
      a.xp_pend[(size_t)s * Fp + j] = a.Xp[(size_t)s * Fp + j];
      a.dy_pend[(size_t)s * Fp + j] = a.dY[(size_t)s * Fp + j];
    }
  }
  FdmBwdArgs o{};
  o.dXp = a.dXp;
  o.dXpb = a.dXpb;
  o.dXpbT = a.dXpbT;
  o.ldT = a.ldT;
  o.Fp = Fp;
  if (!act) {
    for (int r = warp; r < kFdmRowsPerCta; r += 8)
      if (lane == 0 && row0 + r < Fp) store_dxp(o, s, row0 + r, 0.f);
    return;
  }
  float4 dy[NCH];
#pragma unroll
  for (int q = 0; q < NCH; ++q) dy[q] = reinterpret_cast<const float4*>(a.dY + (size_t)s * Fp)[lane + 32 * q];
  for (int r = warp; r < kFdmRowsPerCta; r += 8) {
    const int i = row0 + r;
    if (i >= Fp) break;
    const float4* U4 = reinterpret_cast<const float4*>(a.U + ((size_t)s * Fp + i) * Fp);
    float4 u[NCH];
#pragma unroll
    for (int q = 0; q < NCH; ++q) u[q] = __ldcs(U4 + lane + 32 * q);
    float dot = 0.f;
#pragma unroll
    for (int q = 0; q < NCH; ++q) {
      dot += u[q].x * dy[q].x;
      dot += u[q].y * dy[q].y;
      dot += u[q].z * dy[q].z;
      dot += u[q].w * dy[q].w;
    }
    dot = warp_sum(dot);
    if (lane == 0) store_dxp(o, s, i, dot);
  }
}

template <int NCH>
__global__ void __launch_bounds__(256) fdm_adam_kernel(FdmSplitArgs a) {
  pdl_wait();
  pdl_launch();
  const int s = blockIdx.y;
  const int Fp = a.Fp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const FdmPend pd = *a.pend;
  if (!fdm_split_active(a, s, pd.i)) return;  // a finished stream's FDM is left as is
  const int row0 = blockIdx.x * kFdmRowsPerCta;
  float4 dy[NCH];
#pragma unroll
  for (int q = 0; q < NCH; ++q) dy[q] = reinterpret_cast<const float4*>(a.dy_pend + (size_t)s * Fp)[lane + 32 * q];
  for (int r = warp; r < kFdmRowsPerCta; r += 8) {
    const int i = row0 + r;
    if (i >= Fp) break;
    const float xi = a.xp_pend[(size_t)s * Fp + i];
    const size_t ro = ((size_t)s * Fp + i) * Fp;
    float4* U4 = reinterpret_cast<float4*>(a.U + ro);
    const float4* B4 = reinterpret_cast<const float4*>((a.Ub ? a.Ub : a.U) + ro);
    float4* M4 = reinterpret_cast<float4*>(a.Um + ro);
    float4* V4 = reinterpret_cast<float4*>(a.Uv + ro);
    float4 u[NCH], m[NCH], v[NCH];
#pragma unroll
    for (int q = 0; q < NCH; ++q) {
      u[q] = __ldcs(B4 + lane + 32 * q);
      m[q] = __ldcs(M4 + lane + 32 * q);
      v[q] = __ldcs(V4 + lane + 32 * q);
    }
#pragma unroll
    for (int q = 0; q < NCH; ++q) {
      adam1(u[q].x, m[q].x, v[q].x, xi * dy[q].x, pd.lr, pd.bc1, pd.bc2);
      adam1(u[q].y, m[q].y, v[q].y, xi * dy[q].y, pd.lr, pd.bc1, pd.bc2);
      adam1(u[q].z, m[q].z, v[q].z, xi * dy[q].z, pd.lr, pd.bc1, pd.bc2);
      adam1(u[q].w, m[q].w, v[q].w, xi * dy[q].w, pd.lr, pd.bc1, pd.bc2);
      __stcs(U4 + lane + 32 * q, u[q]);
      __stcs(M4 + lane + 32 * q, m[q]);
      __stcs(V4 + lane + 32 * q, v[q]);
    }
  }
}

// Persistent form of the update, built to run beside the step's other kernels:
// one CTA of 512 threads per SM, at most 80 registers a thread and no shared
// memory, so the step's tensor-core GEMM CTAs still fit on every SM. The FDM
// rows are cut into units of 32 lanes x NU float4 (2, or 1 for odd NCH); warp w of
// CTA c owns units u = c * 16 + w, u + W, u + 2W, ... (W = 16 * grid) and
// updates two units per iteration, so every lane has 6 NU independent
// 16-byte loads in flight. Warps never synchronise.
constexpr int kAdamWarps = 16;

template <int NCH>
__global__ void __maxnreg__(80) fdm_adam_persist_kernel(FdmSplitArgs a) {
  constexpr int FP = 128 * NCH;
  constexpr int NU = NCH % 2 ? 1 : 2;    // float4 per lane per unit
  constexpr int UPR = NCH / NU;          // units per FDM row
  pdl_wait();
  pdl_launch();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const FdmPend pd = *a.pend;
  const float* src = a.Ub ? a.Ub : a.U;  // Adam base (the delayed update reads the other parity)
  const int units = a.b * FP * UPR;      // < 2^31: at most 65535 x 1024 x 4
  const int W = gridDim.x * kAdamWarps;
  for (int u0 = blockIdx.x * kAdamWarps + warp; u0 < units; u0 += 2 * W) {
    const int un[2] = {u0, u0 + W};
    bool act[2];
    float xi[2];
    size_t base[2];
    int dyo[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int g = un[h] / UPR;  // global FDM row: stream g / F', row g % F'
      const int part = un[h] % UPR;
      const int s = g / FP;
      act[h] = un[h] < units && fdm_split_active(a, s, pd.i);
      xi[h] = act[h] ? a.xp_pend[g] : 0.f;
      base[h] = (size_t)g * FP + (size_t)part * 128 * NU;
      dyo[h] = s * FP + part * 128 * NU;
    }
    float4 u[2][NU], m[2][NU], v[2][NU];
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (act[h]) {
#pragma unroll
        for (int q = 0; q < NU; ++q) {
          u[h][q] = __ldcs(reinterpret_cast<const float4*>(src + base[h]) + lane + 32 * q);
          m[h][q] = __ldcs(reinterpret_cast<const float4*>(a.Um + base[h]) + lane + 32 * q);
          v[h][q] = __ldcs(reinterpret_cast<const float4*>(a.Uv + base[h]) + lane + 32 * q);
        }
      }
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (act[h]) {
#pragma unroll
        for (int q = 0; q < NU; ++q) {
          const float4 dy = reinterpret_cast<const float4*>(a.dy_pend + dyo[h])[lane + 32 * q];
          adam1_fused<NCH == 1>(u[h][q].x, m[h][q].x, v[h][q].x, xi[h] * dy.x, pd.lr, pd.bc1, pd.bc2);
          adam1_fused<NCH == 1>(u[h][q].y, m[h][q].y, v[h][q].y, xi[h] * dy.y, pd.lr, pd.bc1, pd.bc2);
          adam1_fused<NCH == 1>(u[h][q].z, m[h][q].z, v[h][q].z, xi[h] * dy.z, pd.lr, pd.bc1, pd.bc2);
          adam1_fused<NCH == 1>(u[h][q].w, m[h][q].w, v[h][q].w, xi[h] * dy.w, pd.lr, pd.bc1, pd.bc2);
          __stcs(reinterpret_cast<float4*>(a.U + base[h]) + lane + 32 * q, u[h][q]);
          __stcs(reinterpret_cast<float4*>(a.Um + base[h]) + lane + 32 * q, m[h][q]);
          __stcs(reinterpret_cast<float4*>(a.Uv + base[h]) + lane + 32 * q, v[h][q]);
        }
      }
  }
}

// Generic fallback for F' not a multiple of 128: one element per lane step.
__global__ void __launch_bounds__(256) fdm_bwd_generic_kernel(FdmBwdArgs a) {
  pdl_wait();
  pdl_launch();
  const int s = blockIdx.y;
  const int Fp = a.Fp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const StepCtl c = *a.ctl;
  bool act = a.active ? (a.active[s] != 0) : ((long long)c.i < a.sp.len(s));
  const int row0 = blockIdx.x * kFdmRowsPerCta;
  for (int r = warp; r < kFdmRowsPerCta; r += 8) {
    const int i = row0 + r;
    if (i >= Fp) break;
    const size_t ro = ((size_t)s * Fp + i) * Fp;
    if (!act) {
      if (lane == 0) store_dxp(a, s, i, 0.f);
      if (!a.update)
        for (int j = lane; j < Fp; j += 32) a.gU[ro + j] = 0.f;
      continue;
    }
    const float xi = a.Xp[(size_t)s * Fp + i];
    float dot = 0.f;
    for (int j = lane; j < Fp; j += 32) {
      float dyj = a.dY[(size_t)s * Fp + j];
      float u = a.U[ro + j];
      dot += u * dyj;
      if (a.update) {
        float m = a.Um[ro + j], v = a.Uv[ro + j];
        adam1(u, m, v, xi * dyj, c.lr, c.bc1, c.bc2);
        a.U[ro + j] = u;
        a.Um[ro + j] = m;
        a.Uv[ro + j] = v;
      } else {
        a.gU[ro + j] = xi * dyj;
      }
    }
    dot = warp_sum(dot);
    if (lane == 0) store_dxp(a, s, i, dot);
  }
}

cudaError_t launch_fdm_bwd(const FdmBwdArgs& a, cudaStream_t st) {
  dim3 grid(div_up(a.Fp, kFdmRowsPerCta), a.b);
  cudaError_t e = cudaSuccess;
  switch (a.Fp) {
    case 128: e = launch_k(fdm_bwd_kernel<1>, dim3(grid), dim3(256), 0, st, a); break;
    case 256: e = launch_k(fdm_bwd_kernel<2>, dim3(grid), dim3(256), 0, st, a); break;
    case 384: e = launch_k(fdm_bwd_kernel<3>, dim3(grid), dim3(256), 0, st, a); break;
    case 512: e = launch_k(fdm_bwd_kernel<4>, dim3(grid), dim3(256), 0, st, a); break;
    case 1024: e = launch_k(fdm_bwd_kernel<8>, dim3(grid), dim3(256), 0, st, a); break;
    default: e = launch_k(fdm_bwd_generic_kernel, dim3(grid), dim3(256), 0, st, a); break;
  }
  return e;
}

__global__ void __launch_bounds__(256) fdm_dx_generic_kernel(FdmSplitArgs a) {
  pdl_wait();
  pdl_launch();
  const int s = blockIdx.y;
  const int Fp = a.Fp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const StepCtl c = *a.ctl;
  if (blockIdx.x == 0 && s == 0 && threadIdx.x == 0) *a.pend = FdmPend{c.i, c.lr, c.bc1, c.bc2};
  const bool act = fdm_split_active(a, s, c.i);
  if (blockIdx.x == 0 && act)
    for (int j = threadIdx.x; j < Fp; j += blockDim.x) {
      a.xp_pend[(size_t)s * Fp + j] = a.Xp[(size_t)s * Fp + j];
      a.dy_pend[(size_t)s * Fp + j] = a.dY[(size_t)s * Fp + j];
    }
  FdmBwdArgs o{};
  o.dXp = a.dXp;
  o.dXpb = a.dXpb;
  o.dXpbT = a.dXpbT;
  o.ldT = a.ldT;
  o.Fp = Fp;
  const int row0 = blockIdx.x * kFdmRowsPerCta;
  for (int r = warp; r < kFdmRowsPerCta; r += 8) {
    const int i = row0 + r;
    if (i >= Fp) break;
    float dot = 0.f;
    if (act)
      for (int j = lane; j < Fp; j += 32) dot += a.U[((size_t)s * Fp + i) * Fp + j] * a.dY[(size_t)s * Fp + j];
    dot = warp_sum(dot);
    if (lane == 0) store_dxp(o, s, i, act ? dot : 0.f);
  }
}

// FUSED: the overlapped update of Algorithm 1's schedule; else the delayed update's.
template <bool FUSED>
__global__ void __launch_bounds__(256) fdm_adam_generic_kernel(FdmSplitArgs a) {
  pdl_wait();
  pdl_launch();
  const int s = blockIdx.y;
  const int Fp = a.Fp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const FdmPend pd = *a.pend;
  if (!fdm_split_active(a, s, pd.i)) return;
  const int row0 = blockIdx.x * kFdmRowsPerCta;
  for (int r = warp; r < kFdmRowsPerCta; r += 8) {
    const int i = row0 + r;
    if (i >= Fp) break;
    const size_t ro = ((size_t)s * Fp + i) * Fp;
    const float xi = a.xp_pend[(size_t)s * Fp + i];
    const float* src = a.Ub ? a.Ub : a.U;
    for (int j = lane; j < Fp; j += 32) {
      float u = src[ro + j], m = a.Um[ro + j], v = a.Uv[ro + j];
      const float g = xi * a.dy_pend[(size_t)s * Fp + j];
      if (FUSED)
        adam1_fused<true>(u, m, v, g, pd.lr, pd.bc1, pd.bc2);
      else
        adam1(u, m, v, g, pd.lr, pd.bc1, pd.bc2);
      a.U[ro + j] = u;
      a.Um[ro + j] = m;
      a.Uv[ro + j] = v;
    }
  }
}

cudaError_t launch_fdm_dx(const FdmSplitArgs& a, cudaStream_t st) {
  dim3 grid(div_up(a.Fp, kFdmRowsPerCta), a.b);
  switch (a.Fp) {
    case 128: return launch_k(fdm_dx_kernel<1>, grid, dim3(256), 0, st, a);
    case 256: return launch_k(fdm_dx_kernel<2>, grid, dim3(256), 0, st, a);
    case 384: return launch_k(fdm_dx_kernel<3>, grid, dim3(256), 0, st, a);
    case 512: return launch_k(fdm_dx_kernel<4>, grid, dim3(256), 0, st, a);
    case 1024: return launch_k(fdm_dx_kernel<8>, grid, dim3(256), 0, st, a);
    default: return launch_k(fdm_dx_generic_kernel, grid, dim3(256), 0, st, a);
  }
}

template <int NCH>
cudaError_t launch_adam_persist(const FdmSplitArgs& a, cudaStream_t st) {
  // The CTA stays resident for the whole update: keep its SM configured for
  // the largest shared-memory carveout, so GEMM CTAs still fit beside it.
  static OncePerDevice once;
  cudaError_t e = once_on_device(once, [] {
    return cudaFuncSetAttribute(fdm_adam_persist_kernel<NCH>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                cudaSharedmemCarveoutMaxShared);
  });
  int sms = 0;
  if (e == cudaSuccess) e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  return launch_k(fdm_adam_persist_kernel<NCH>, dim3(sms), dim3(32 * kAdamWarps), 0, st, a);
}

cudaError_t launch_fdm_adam(const FdmSplitArgs& a, cudaStream_t st, bool persistent) {
  if (persistent) switch (a.Fp) {
      case 128: return launch_adam_persist<1>(a, st);
      case 256: return launch_adam_persist<2>(a, st);
      case 384: return launch_adam_persist<3>(a, st);
      case 512: return launch_adam_persist<4>(a, st);
      case 1024: return launch_adam_persist<8>(a, st);
      default: break;
    }
  dim3 grid(div_up(a.Fp, kFdmRowsPerCta), a.b);
  switch (a.Fp) {
    case 128: return launch_k(fdm_adam_kernel<1>, grid, dim3(256), 0, st, a);
    case 256: return launch_k(fdm_adam_kernel<2>, grid, dim3(256), 0, st, a);
    case 384: return launch_k(fdm_adam_kernel<3>, grid, dim3(256), 0, st, a);
    case 512: return launch_k(fdm_adam_kernel<4>, grid, dim3(256), 0, st, a);
    case 1024: return launch_k(fdm_adam_kernel<8>, grid, dim3(256), 0, st, a);
    default:
      return launch_k(persistent ? fdm_adam_generic_kernel<true> : fdm_adam_generic_kernel<false>, grid, dim3(256), 0,
                      st, a);
  }
}

__device__ __forceinline__ void advance_in_place(const Advance& a);

// One value of dE, and Adam on its parameter (u.P == nullptr: the gradient only).
__device__ __forceinline__ void emb_out(float* __restrict__ dE, const EmbAdam& u, size_t o, float g) {
  dE[o] = g;
  if (!u.P) return;
  float p = u.P[o], m = u.M[o], v = u.V[o];
  // adam1 with the contractions spelled out as the other parameters' Adam has
  // them: beside the sums above the compiler contracted the other products
  m = __fmaf_rn(kB1, m, __fmul_rn(1.0f - kB1, g));
  v = __fmaf_rn(kB2, v, __fmul_rn(__fmul_rn(1.0f - kB2, g), g));
  p = p - u.ctl->a_lr * (m / u.ctl->a_bc1) / (sqrtf(v / u.ctl->a_bc2) + kAdamEps);
  u.P[o] = p;
  u.M[o] = m;
  u.V[o] = v;
  if (u.Pb) u.Pb[o] = __float2bfloat16_rn(p);
}

// ============================================================================================
// Embedding backward: scatter-add of dh0 into E's rows, owner computes.
// CTA (c, q) owns byte value c and chunk q of kEmbChunkPos consecutive
// positions; warp w of 8 sums a contiguous eighth of the chunk in increasing
// position (emb_range_sum). The 8 warp sums are added in warp order. With one
// chunk that is dE[c]; with several, each CTA writes its partial and the last
// CTA of c to arrive adds the chunks' partials in chunk order (a fence
// precedes the arrival counter), so the result does not depend on timing.
// Position p = s*K + k has its D gradient values at dX[p*D ..).
// ============================================================================================
// Per-warp scratch of emb_range_sum: a ring of four stages of FL floats and the
// matching positions of one block, relative to its start.
constexpr int kEmbBlock = 2048;  // 64 consecutive positions a lane
template <int FL>
struct __align__(16) EmbScratch {
  static constexpr int kStages = 4, kFloats = FL;
  float ring[kStages][FL];
  uint16_t list[kEmbBlock];
};
using EmbDeep = EmbScratch<512>;  // two CTAs an SM: long chains, few CTAs
using EmbWide = EmbScratch<256>;  // three CTAs an SM: many CTAs

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One warp's sum of the rows dX[p*D ..) over the positions p in [p_lo, p_hi)
// with ctx[p] == c, in increasing p: lane d gets dimension d in a0 and d + 32 in a1.
// The adds must stay in order, so a frequent byte's warp is bound by the
// dependent add of its rows; all else is latency. Blocks of 2048 positions: a
// lane compares its 64 consecutive ones at once (one load latency a block), a
// prefix sum of the lanes' counts places their hits in the list, and the rows
// come through a ring of asynchronous copies, up to 128 rows of 16 floats ahead
// of the adds. Walking 256 positions at a time with ballots paid a load latency
// each: 13.8 us for 512 streams of 32 positions (59 us with the rows loaded
// eight at a time); now 5.7, most of it gained by loading a stage's rows into
// registers before the serial adds (59 cycles a row as one load and add each).
template <int DT, class Scratch>
__device__ __forceinline__ void emb_range_sum(const uint8_t* __restrict__ ctx, const float* __restrict__ dX, int Drt,
                                              uint32_t c, int p_lo, int p_hi, Scratch& s, float& a0, float& a1) {
  constexpr int ST = Scratch::kStages, FL = Scratch::kFloats;
  const int lane = threadIdx.x & 31;
  const int D = DT > 0 ? DT : Drt;
  const int R = FL / D, C4 = D / 4;  // rows of a stage, 16-byte pieces of a row
  const int l0 = min(lane, D - 1), l1 = min(lane + 32, D - 1);
  const uint32_t cc = c * 0x01010101u;
  a0 = a1 = 0.f;
  for (int pb = p_lo; pb < p_hi; pb += kEmbBlock) {
    // hits of positions [q0, q0 + 64): bit k of m is q0 + k
    const int q0 = pb + lane * 64;
    unsigned long long m = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = q0 + 16 * u;
      uint32_t w[4];
      if (q + 16 <= p_hi && ((reinterpret_cast<uintptr_t>(ctx) + q) & 15) == 0) {
        const uint4 x = *reinterpret_cast<const uint4*>(ctx + q);
        w[0] = x.x;
        w[1] = x.y;
        w[2] = x.z;
        w[3] = x.w;
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          w[k] = ~cc;  // never matches
          for (int t = 0; t < 4; ++t)
            if (q + 4 * k + t < p_hi) w[k] = (w[k] & ~(0xFFu << (8 * t))) | (uint32_t)ctx[q + 4 * k + t] << (8 * t);
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        // 0xFF bytes where equal -> one bit each, in byte order
        const uint32_t eq = __vcmpeq4(w[k], cc) & 0x08040201u;
        m |= (unsigned long long)((eq | eq >> 8 | eq >> 16 | eq >> 24) & 15u) << (16 * u + 4 * k);
      }
    }
    const int cnt = __popcll(m);
    int at = cnt;  // inclusive prefix sum over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += v;
    }
    const int n = __shfl_sync(0xffffffffu, at, 31);
    if (n == 0) continue;  // warp-uniform
    at -= cnt;
    while (m) {
      s.list[at++] = (uint16_t)(lane * 64 + __ffsll((long long)m) - 1);
      m &= m - 1;
    }
    __syncwarp();
    const float* rows = dX + (size_t)pb * D;
    const int stages = (n + R - 1) / R;
    auto issue = [&](int k) {
      if (k < stages) {
        float* st = s.ring[k % ST];
        const int r_n = min(R, n - k * R);
#pragma unroll
        for (int u = 0; u < FL / 128; ++u) {
          const int r = (lane + 32 * u) / C4, q = (lane + 32 * u - r * C4) * 4;
          if (r < r_n) cp_async16(st + r * D + q, rows + (size_t)s.list[k * R + r] * D + q);
        }
      }
      cp_async_commit();
    };
    for (int k = 0; k < ST; ++k) issue(k);
    for (int k = 0; k < stages; ++k) {
      cp_async_wait<ST - 1>();
      __syncwarp();
      const float* st = s.ring[k % ST];
      const int r_n = min(R, n - k * R);
      // (lanes beyond D add some other dimension's values, which nothing reads)
      if (DT > 0 && DT <= 32 && r_n == R) {
        constexpr int RR = DT > 0 ? FL / (DT > 0 ? DT : 1) : 1;
        float v[RR];  // the loads first: only the adds are serial
#pragma unroll
        for (int r = 0; r < RR; ++r) v[r] = st[r * D + l0];
#pragma unroll
        for (int r = 0; r < RR; ++r) a0 += v[r];
      } else {
#pragma unroll 4
        for (int r = 0; r < r_n; ++r) {
          a0 += st[r * D + l0];
          if (D > 32) a1 += st[r * D + l1];
        }
      }
      __syncwarp();  // the stage is read before its next copies
      issue(k + ST);
    }
    cp_async_wait<0>();
    __syncwarp();
  }
}

template <int DT, class Scratch>
__global__ void __launch_bounds__(256) embed_bwd_owner_kernel(const uint8_t* __restrict__ ctx,
                                                              const float* __restrict__ dX, int P, int D,
                                                              float* __restrict__ dE, float* __restrict__ part,
                                                              unsigned* __restrict__ cnt, Advance adv,
                                                              EmbAdam upd) {
  pdl_wait();
  pdl_launch();
  if (adv.ctl && blockIdx.x == 255 && blockIdx.y == 0 && threadIdx.x == 255) advance_in_place(adv);
  extern __shared__ __align__(16) unsigned char emb_smem[];
  Scratch* scratch = reinterpret_cast<Scratch*>(emb_smem);
  __shared__ float wsum[8][64];
  __shared__ int is_last;
  const uint32_t c = blockIdx.x;
  const int nq = gridDim.y, q = blockIdx.y;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c_lo = min(P, q * kEmbChunkPos), c_hi = min(P, c_lo + kEmbChunkPos);
  const int per = ((c_hi - c_lo + 8 * 128 - 1) / (8 * 128)) * 128;  // positions per warp, a multiple of 128
  const int p_lo = min(c_hi, c_lo + w * per), p_hi = min(c_hi, p_lo + per);
  float a0, a1;  // dims lane and lane + 32
  emb_range_sum<DT>(ctx, dX, D, c, p_lo, p_hi, scratch[w], a0, a1);
  wsum[w][lane] = a0;
  wsum[w][lane + 32] = a1;
  __syncthreads();
  const int t = threadIdx.x;
  float sum = 0.f;
  if (t < D) {
    sum = wsum[0][t];
#pragma unroll
    for (int ww = 1; ww < 8; ++ww) sum += wsum[ww][t];
  }
  if (nq == 1) {
    if (t < D) emb_out(dE, upd, (size_t)c * D + t, sum);
    return;
  }
  if (t < D) {
    part[((size_t)c * nq + q) * D + t] = sum;
    __threadfence();
  }
  __syncthreads();
  if (t == 0) is_last = (atomicAdd(&cnt[c], 1u) == (unsigned)(nq - 1));
  __syncthreads();
  if (is_last && t < D) {
    __threadfence();
    const float* src = part + (size_t)c * nq * D + t;
    float acc = 0.f;
    for (int k = 0; k < nq; ++k) acc += __ldcg(src + (size_t)k * D);
    emb_out(dE, upd, (size_t)c * D + t, acc);
    if (t == 0) cnt[c] = 0u;
  }
}

int embed_bwd_chunks(int b, int K) { return (b * K + kEmbChunkPos - 1) / kEmbChunkPos; }

template <int DT, class Scratch, class... A>
static cudaError_t launch_emb_owner(dim3 grid, cudaStream_t st, A... args) {
  constexpr size_t smem = 8 * sizeof(Scratch);
  auto k = embed_bwd_owner_kernel<DT, Scratch>;
  static OncePerDevice once;
  const cudaError_t attr = once_on_device(
      once, [&] { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); });
  if (attr != cudaSuccess) return attr;
  return launch_k(k, grid, dim3(256), smem, st, args...);
}

template <int DT>
static cudaError_t launch_emb(dim3 grid, cudaStream_t st, const uint8_t* ctx, const float* dX, int P, int D, float* dE,
                              float* part, unsigned* cnt, const Advance& adv, const EmbAdam& upd) {
  // 256 CTAs (one chunk) are resident at once with the deep ring; with several chunks more CTAs an SM count more
  if (grid.y == 1) return launch_emb_owner<DT, EmbDeep>(grid, st, ctx, dX, P, D, dE, part, cnt, adv, upd);
  return launch_emb_owner<DT, EmbWide>(grid, st, ctx, dX, P, D, dE, part, cnt, adv, upd);
}

cudaError_t launch_embed_bwd(const uint8_t* ctx, const float* dX, int b, int K, int D, float* dE, float* part,
                             unsigned* cnt, const Advance& adv, const EmbAdam& upd, cudaStream_t st) {
  if (D > 64) return cudaErrorInvalidValue;
  const int nq = embed_bwd_chunks(b, K);
  if (nq > 1 && (!part || !cnt)) return cudaErrorInvalidValue;
  const dim3 grid(256, nq < 1 ? 1 : nq);
  switch (D) {  // the configurations' widths have their loops unrolled
    case 8: return launch_emb<8>(grid, st, ctx, dX, b * K, D, dE, part, cnt, adv, upd);
    case 16: return launch_emb<16>(grid, st, ctx, dX, b * K, D, dE, part, cnt, adv, upd);
    default: return launch_emb<0>(grid, st, ctx, dX, b * K, D, dE, part, cnt, adv, upd);
  }
}

// Grouped embedding adjoint: CTA (group g, pair of byte values); warps 4v to
// 4v + 3 own byte value 2 cb + v, each one quarter of the group's context
// positions (in blocks of 512), summed in increasing position
// (emb_range_sum); the four quarter sums are then added in order. So each
// dE[g][c] is a fixed-order sum that depends on the group alone.
template <int DT>
__global__ void __launch_bounds__(256) embed_bwd_groups_kernel(const uint8_t* __restrict__ ctx,
                                                               const float* __restrict__ dX, int K, int D,
                                                               float* __restrict__ dE,
                                                               const GroupInfo* __restrict__ gi, size_t gs,
                                                              Advance adv, EmbAdam upd) {
  pdl_wait();
  pdl_launch();
  if (adv.ctl && blockIdx.x == 0 && blockIdx.y == 127 && threadIdx.x == 255) advance_in_place(adv);
  extern __shared__ __align__(16) unsigned char emb_smem[];
  EmbWide* scratch = reinterpret_cast<EmbWide*>(emb_smem);
  __shared__ float part[8][64];
  const GroupInfo g = gi[blockIdx.x];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t c = blockIdx.y * 2 + (w >> 2);
  // the group's streams only: its padding rows never hold a byte (their
  // gradient is zero) and their all-zero contexts would all match byte 0
  const int g_lo = g.r0 * K, g_hi = (g.r0 + g.s) * K;
  const int per = ((g_hi - g_lo + 4 * 512 - 1) / (4 * 512)) * 512;  // a quarter, whole 512-position blocks
  const int p_lo = min(g_hi, g_lo + (w & 3) * per), p_hi = min(g_hi, p_lo + per);
  float a0, a1;
  emb_range_sum<DT>(ctx, dX, D, c, p_lo, p_hi, scratch[w], a0, a1);
  part[w][lane] = a0;
  part[w][lane + 32] = a1;
  __syncthreads();
  if ((w & 3) == 0) {
    const size_t o = (size_t)blockIdx.x * gs + (size_t)c * D;
    for (int d = lane; d < D; d += 32)
      emb_out(dE, upd, o + d, ((part[w][d] + part[w + 1][d]) + part[w + 2][d]) + part[w + 3][d]);
  }
}

template <int DT, class... A>
static cudaError_t launch_emb_groups(dim3 grid, cudaStream_t st, A... args) {
  constexpr size_t smem = 8 * sizeof(EmbWide);
  static OncePerDevice once;
  const cudaError_t attr = once_on_device(once, [] {
    return cudaFuncSetAttribute(embed_bwd_groups_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (attr != cudaSuccess) return attr;
  return launch_k(embed_bwd_groups_kernel<DT>, grid, dim3(256), smem, st, args...);
}

cudaError_t launch_embed_bwd_groups(const uint8_t* ctx, const float* dX, int K, int D, float* dE,
                                    const GroupInfo* gi, int ngroups, size_t gs, const Advance& adv, const EmbAdam& upd,
                                    cudaStream_t st) {
  if (D > 64 || ngroups < 1 || ngroups > 65535 || !gi || (reinterpret_cast<uintptr_t>(ctx) & 3))
    return cudaErrorInvalidValue;
  const dim3 grid(ngroups, 128);
  switch (D) {
    case 8: return launch_emb_groups<8>(grid, st, ctx, dX, K, D, dE, gi, gs, adv, upd);
    case 16: return launch_emb_groups<16>(grid, st, ctx, dX, K, D, dE, gi, gs, adv, upd);
    default: return launch_emb_groups<0>(grid, st, ctx, dX, K, D, dE, gi, gs, adv, upd);
  }
}

// ============================================================================================
// Adam on the shared parameters (Sec. 4.1: lr 1e-3; beta, eps as documented).
// ============================================================================================
// P is read from Pin and written to P (Pin == P: in place; the delayed-update
// schedule writes the next parameters beside the current ones). Pb: the BF16
// copy, refreshed in the same pass. Four parameters a thread (tensor sizes are
// multiples of 8): bound by loads in flight; with one parameter a thread the
// 64 MiB mix's 2.0 M took 11.0 us, now 9.3. The whole set at once is the
// delayed update's form; Algorithm 1's runs layer by layer (adam_layer_kernel).
__global__ void __launch_bounds__(256) adam_kernel(float4* P, const float4* Pin, const float4* __restrict__ G,
                                                   float4* __restrict__ M, float4* __restrict__ V,
                                                   uint2* __restrict__ Pb, size_t n4, const StepCtl* __restrict__ ctl) {
  pdl_wait();
  pdl_launch();
  const float lr = ctl->a_lr, bc1 = ctl->a_bc1, bc2 = ctl->a_bc2;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n4; e += (size_t)gridDim.x * blockDim.x) {
    float4 p = Pin[e], m = M[e], v = V[e];
    const float4 g = G[e];
    adam1(p.x, m.x, v.x, g.x, lr, bc1, bc2);
    adam1(p.y, m.y, v.y, g.y, lr, bc1, bc2);
    adam1(p.z, m.z, v.z, g.z, lr, bc1, bc2);
    adam1(p.w, m.w, v.w, g.w, lr, bc1, bc2);
    P[e] = p;
    M[e] = m;
    V[e] = v;
    if (Pb) {
      __align__(8) __nv_bfloat162 h[2] = {__floats2bfloat162_rn(p.x, p.y), __floats2bfloat162_rn(p.z, p.w)};
      Pb[e] = *reinterpret_cast<const uint2*>(h);
    }
  }
}

cudaError_t launch_adam(float* P, const float* G, float* M, float* V, __nv_bfloat16* Pb, size_t n, const StepCtl* ctl,
                        cudaStream_t st, const float* Pin) {
  if (n & 3) return cudaErrorInvalidValue;
  const size_t n4 = n / 4;
  const int grid = (int)std::min<size_t>((n4 + 255) / 256, 152 * 8);
  return launch_k(adam_kernel, dim3(grid), dim3(256), 0, st, reinterpret_cast<float4*>(P),
                  reinterpret_cast<const float4*>(Pin ? Pin : P), reinterpret_cast<const float4*>(G),
                  reinterpret_cast<float4*>(M), reinterpret_cast<float4*>(V), reinterpret_cast<uint2*>(Pb), n4, ctl);
}

// ============================================================================================
// Step control: advance to the next time index and derive its scalars.
// ============================================================================================
// Reads the step control of the current step from `src` and writes the next
// step's to `dst` (the same record, or the other of the delayed-update
// schedule's two, whose sticky error bits are kept).
// The control record of the next step (i + 1) from that of the current one.
__device__ __forceinline__ StepCtl advance_ctl(StepCtl c, int dst_err, Split sp, int K, int ring_slots, int b) {
  c.err |= dst_err;
  c.i += 1;
  c.t += 1;
  long long i = c.i;
  int bact;
  if (sp.cp) {
    // uneven split: the count changes only at the table's time indices
    bact = c.bact;
    while (c.cpi < sp.ncp && sp.cp[c.cpi].i <= i) bact = sp.cp[c.cpi++].bact;
  } else {
    bact = (i < sp.q) ? b : (i == sp.q ? sp.rem : 0);
  }
  c.bact = bact;
  c.inv_bact = bact > 0 ? 1.0f / (float)bact : 0.f;
  c.bc1 = 1.0f - powf(kB1, (float)c.t);
  c.bc2 = 1.0f - powf(kB2, (float)c.t);
  c.slot = (int)((i - K) % ring_slots);
  return c;
}

// In place, by one thread of a launch that no reader of the record overlaps but
// Adam, which reads its own copy of the scalars (a_*), and kernels that set
// error bits (which are left alone).
__device__ __forceinline__ void advance_in_place(const Advance& a) {
  const StepCtl c = advance_ctl(*a.ctl, 0, a.sp, a.K, a.ring_slots, a.b);
  a.ctl->i = c.i;
  a.ctl->t = c.t;
  a.ctl->bact = c.bact;
  a.ctl->slot = c.slot;
  a.ctl->inv_bact = c.inv_bact;
  a.ctl->bc1 = c.bc1;
  a.ctl->bc2 = c.bc2;
  a.ctl->cpi = c.cpi;
}

__global__ void step_advance_kernel(const StepCtl* src, StepCtl* dst, Split sp, int K, int ring_slots, int b) {
  pdl_wait();
  pdl_launch();
  *dst = advance_ctl(*src, dst->err, sp, K, ring_slots, b);
}
cudaError_t launch_step_advance(StepCtl* ctl, Split sp, int K, int ring_slots, int b, cudaStream_t st,
                                StepCtl* dst) {
  return launch_k(step_advance_kernel, dim3(1), dim3(1), 0, st, (const StepCtl*)ctl, dst ? dst : ctl, sp, K,
                  ring_slots, b);
}

// ============================================================================================
// Range coder (32-bit, carry-propagating). See the oracle's coder for the
// same rule: r = R >> 16; low += r*cum; R = r*f (or R - r*cum for the last
// symbol); renormalise bytewise below 2^24.
//
// One thread codes a stream, so a symbol's dependent chain is what a launch
// takes. The last 2 to 7 code bytes stay in a register pair (pend): a carry out
// of low is an addition there, a renormalisation (r >= 2^8 and f >= 1, so at
// most two bytes) is three shifts without a loop or a branch, and the bytes go
// out four at a time. A carry out of pend's own bytes (all 0xFF) stays as the
// bit above them until they leave; it is then added to the bytes already in
// the window. 1024 symbols of 4096 streams take 94 us (92 ns a symbol). With a
// byte of cache, a count of pending 0xFF bytes and a loop of byte stores, plus
// three allocations and three launches, the call took 597 us; now 113.
// ============================================================================================
struct EncIO {
  uint8_t* out;
  uint32_t cap;
  bool aligned;  // the window starts on a 4-byte boundary (every position is a multiple of 4 until the flush)
  __device__ EncIO(uint8_t* o, uint32_t c) : out(o), cap(c), aligned((reinterpret_cast<uintptr_t>(o) & 3) == 0) {}
};

// n bytes of v into the window from pos on, after a carry into the bytes before
// them. Returns the new position, and err in the upper half: bytes beyond the
// capacity are lost and set it, to kLostFF while every lost byte is 0xFF (a carry
// goes through those into the window, once), else to kLost. By value, so that the
// state stays in registers.
constexpr uint32_t kLost = 1, kLostFF = 2;
__device__ __noinline__ unsigned long long enc_put_slow(uint8_t* out, uint32_t cap, uint32_t pos, uint32_t err, uint32_t v,
                                                        uint32_t n, bool carry) {
  if (carry && err != kLost) {
    for (uint32_t p = pos; p-- > 0;)
      if (++out[p] != 0) break;
    if (err) err = kLost;
  }
  for (uint32_t k = n; k-- > 0;) {
    const uint8_t byte = (uint8_t)(v >> (8 * k));
    if (pos < cap)
      out[pos++] = byte;
    else
      err = err != kLost && byte == 0xFF ? kLostFF : kLost;
  }
  return (unsigned long long)err << 32 | pos;
}

__device__ __forceinline__ void enc_put(EncState& s, const EncIO& io, uint32_t v, uint32_t n, bool carry) {
  const unsigned long long r = enc_put_slow(io.out, io.cap, s.pos, s.err, v, n, carry);
  s.pos = (uint32_t)r;
  s.err = (uint32_t)(r >> 32);
}

// Codes a ring slot's symbol w (cum in the low half, f - 1 in the high one; kSkip: none).
__device__ __forceinline__ void enc_symbol(EncState& s, const EncIO& io, uint32_t w) {
  const bool skip = w == kSkip;
  const uint32_t cum = w & 0xFFFFu, f = (w >> 16) + 1u;
  const uint32_t r = s.range >> kTBits, d = skip ? 0u : r * cum;
  s.low += d;
  uint32_t plo = (uint32_t)s.pend, phi = (uint32_t)(s.pend >> 32);
  const uint32_t carry = s.low < d ? 1u : 0u;
  plo += carry;
  phi += plo < carry ? 1u : 0u;
  const uint32_t nr = (skip || cum + f == (uint32_t)kT) ? s.range - d : r * f;
  const uint32_t n8 = nr < kTop ? (nr < (kTop >> 8) ? 16u : 8u) : 0u;  // bits that leave low
  phi = __funnelshift_l(plo, phi, n8);
  plo = (plo << n8) | __funnelshift_l(s.low, 0u, n8);
  s.low <<= n8;
  s.range = nr << n8;
  s.npend += n8 >> 3;
  // 6 or 7 bytes (and the bit above them): the first four leave. The common
  // case is one predicated store; the branch is taken for unaligned windows,
  // at a window's end and for carries only.
  const bool put = s.npend >= 6;
  const uint32_t sh = put ? 8 * (s.npend - 4) : 0;
  const uint32_t v = __funnelshift_r(plo, phi, sh);
  const bool fast = put && (phi >> sh) == 0 && s.pos + 4 <= io.cap && io.aligned;
  if (fast) *reinterpret_cast<uint32_t*>(io.out + s.pos) = __byte_perm(v, 0, 0x0123);
  if (put && !fast) enc_put(s, io, v, 4, (phi >> sh) != 0);
  s.pos += fast ? 4u : 0u;
  s.npend -= put ? 4u : 0u;
  plo = put ? plo & ((1u << sh) - 1u) : plo;
  phi = put ? 0u : phi;
  s.pend = ((unsigned long long)phi << 32) | plo;
}

__device__ __forceinline__ void enc_init(EncState& s) {
  s.pend = 0;
  s.low = 0;
  s.range = 0xFFFFFFFFu;
  s.npend = 0;
  s.pos = 0;
  s.err = 0;
  s.pad = 0;
}

// The last byte and everything pending; returns the length without trailing
// zero bytes (which the decoder reads past the end), or 0xFFFFFFFF on overflow.
__device__ __forceinline__ uint32_t enc_finish(EncState& s, const EncIO& io) {
  // The value low rounded up to a multiple of 2^24 lies in [low, low + R).
  const uint32_t low = s.low + (kTop - 1);
  s.pend += low < s.low ? 1u : 0u;
  s.pend = (s.pend << 8) | (low >> 24);  // at most 6 bytes
  const uint32_t n = s.npend + 1, n1 = n > 4 ? n - 4 : 0;  // first n1, then the last (up to four)
  const bool carried = (s.pend >> (8 * n)) != 0;
  if (n1) enc_put(s, io, (uint32_t)(s.pend >> 32), n1, carried);
  enc_put(s, io, (uint32_t)s.pend, n - n1, carried && !n1);
  s.low = 0;
  s.pend = 0;
  s.npend = 0;
  uint32_t len = s.pos;
  while (len > 0 && io.out[len - 1] == 0) --len;
  return s.err ? 0xFFFFFFFFu : len;
}

// Codes nsteps ring slots of stream s from slot0 on, the symbols of the next
// kAhead slots in flight meanwhile (coalesced across the streams of a warp; 32
// ahead, unrolled, outgrew the instruction cache: 134 us against 114).
__device__ __forceinline__ void enc_slots(EncState& st, const EncIO& io, const uint32_t* __restrict__ ring,
                                          int ring_slots, int slot0, int nsteps, int b, int s) {
  constexpr int kAhead = 8;
  uint32_t nx[kAhead];
  int slot = slot0, t = 0;
  auto fetch = [&]() {
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      nx[q] = t + q < nsteps ? ring[(size_t)slot * b + s] : kSkip;
      if (++slot == ring_slots) slot = 0;
    }
    t += kAhead;
  };
  fetch();
  while (t < nsteps + kAhead) {
    uint32_t w[kAhead];
#pragma unroll
    for (int q = 0; q < kAhead; ++q) w[q] = nx[q];
    fetch();
#pragma unroll
    for (int q = 0; q < kAhead; ++q) enc_symbol(st, io, w[q]);
  }
}

__global__ void prefix_encode_kernel(EncState* es, const uint8_t* __restrict__ data, Split sp, int K, int b,
                                     uint8_t* out, const unsigned long long* out_off, const uint32_t* out_cap) {
  pdl_wait();
  pdl_launch();
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= b) return;
  EncState st;
  enc_init(st);
  const EncIO io(out + out_off[s], out_cap[s]);
  long long n = sp.len(s) < K ? sp.len(s) : K;
  const uint8_t* x = data + sp.off(s);
  for (long long i = 0; i < n; ++i) enc_symbol(st, io, 256u * x[i] | 255u << 16);
  es[s] = st;
}

cudaError_t launch_prefix_encode(EncState* es, const uint8_t* data, Split sp, int K, int b, uint8_t* out,
                                 const unsigned long long* out_off, const uint32_t* out_cap, cudaStream_t st) {
  return launch_k(prefix_encode_kernel, dim3(div_up(b, 128)), dim3(128), 0, st, es, data, sp, K, b, out, out_off, out_cap);
}

// One thread per stream, one warp per CTA: the streams' chains spread over the SMs.
constexpr int kEncThreads = 32;

__global__ void __launch_bounds__(kEncThreads) range_encode_kernel(EncState* es, const uint32_t* __restrict__ ring,
                                                                   int ring_slots, int slot0, int nsteps, int b,
                                                                   uint8_t* out, const unsigned long long* out_off,
                                                                   const uint32_t* out_cap) {
  pdl_wait();
  pdl_launch();
  const int s = blockIdx.x * kEncThreads + threadIdx.x;
  if (s >= b) return;
  EncState st = es[s];
  const EncIO io(out + out_off[s], out_cap[s]);
  enc_slots(st, io, ring, ring_slots, slot0, nsteps, b, s);
  es[s] = st;
}

cudaError_t launch_range_encode(EncState* es, const uint32_t* ring, int ring_slots, int slot0, int nsteps, int b,
                                uint8_t* out, const unsigned long long* out_off, const uint32_t* out_cap,
                                cudaStream_t st) {
  if (nsteps <= 0) return cudaSuccess;
  return launch_k(range_encode_kernel, dim3(div_up(b, kEncThreads)), dim3(kEncThreads), 0, st, es, ring, ring_slots,
                  slot0, nsteps, b, out, out_off, out_cap);
}

// Whole streams in one launch: nsteps symbols each into windows of cap bytes.
__global__ void __launch_bounds__(kEncThreads) range_encode_whole_kernel(const uint32_t* __restrict__ sym, int nsteps,
                                                                         int b, uint8_t* out, uint32_t cap,
                                                                         uint32_t* out_len) {
  const int s = blockIdx.x * kEncThreads + threadIdx.x;
  if (s >= b) return;
  EncState st;
  enc_init(st);
  const EncIO io(out + (size_t)s * cap, cap);
  enc_slots(st, io, sym, nsteps, 0, nsteps, b, s);
  out_len[s] = enc_finish(st, io);
}

cudaError_t launch_range_encode_whole(const uint32_t* sym, int nsteps, int b, uint8_t* out, uint32_t cap,
                                      uint32_t* out_len, cudaStream_t st) {
  NoPdl scope;
  return launch_k(range_encode_whole_kernel, dim3(div_up(b, kEncThreads)), dim3(kEncThreads), 0, st, sym, nsteps, b,
                  out, cap, out_len);
}

__global__ void encode_flush_kernel(EncState* es, int b, uint8_t* out, const unsigned long long* out_off,
                                    const uint32_t* out_cap, uint32_t* out_len) {
  pdl_wait();
  pdl_launch();
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= b) return;
  EncState st = es[s];
  const EncIO io(out + out_off[s], out_cap[s]);
  out_len[s] = enc_finish(st, io);
  es[s] = st;
}

cudaError_t launch_encode_flush(EncState* es, int b, uint8_t* out, const unsigned long long* out_off,
                                const uint32_t* out_cap, uint32_t* out_len, cudaStream_t st) {
  return launch_k(encode_flush_kernel, dim3(div_up(b, 128)), dim3(128), 0, st, es, b, out, out_off, out_cap, out_len);
}

__device__ __forceinline__ uint32_t dec_byte(const uint8_t* in, uint32_t len, uint32_t& pos) {
  uint32_t v = pos < len ? in[pos] : 0u;
  ++pos;
  return v;
}

__device__ __forceinline__ void dec_update(DecState& d, const uint8_t* in, uint32_t len, uint32_t r, uint32_t c,
                                           uint32_t f) {
  d.code -= r * c;
  d.range = (c + f == (uint32_t)kT) ? d.range - r * c : r * f;
  while (d.range < kTop) {
    d.code = (d.code << 8) | dec_byte(in, len, d.pos);
    d.range <<= 8;
  }
}

__global__ void dec_init_kernel(DecState* ds, const uint8_t* bits, const unsigned long long* off,
                                const uint32_t* len, int b) {
  pdl_wait();
  pdl_launch();
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= b) return;
  DecState d;
  d.pos = 0;
  d.range = 0xFFFFFFFFu;
  d.code = 0;
  d.err = 0;
  const uint8_t* in = bits + off[s];
  for (int k = 0; k < 4; ++k) d.code = (d.code << 8) | dec_byte(in, len[s], d.pos);
  ds[s] = d;
}

cudaError_t launch_dec_init(DecState* ds, const uint8_t* bits, const unsigned long long* off, const uint32_t* len,
                            int b, cudaStream_t st) {
  return launch_k(dec_init_kernel, dim3(div_up(b, 128)), dim3(128), 0, st, ds, bits, off, len, b);
}

__global__ void prefix_decode_kernel(DecState* ds, const uint8_t* bits, const unsigned long long* off,
                                     const uint32_t* len, Split sp, int K, int b, uint8_t* data) {
  pdl_wait();
  pdl_launch();
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= b) return;
  DecState d = ds[s];
  const uint8_t* in = bits + off[s];
  const uint32_t L = len[s];
  long long n = sp.len(s) < K ? sp.len(s) : K;
  uint8_t* x = data + sp.off(s);
  for (long long i = 0; i < n; ++i) {
    uint32_t r = d.range >> kTBits;
    uint32_t target = d.code / r;
    if (target > (uint32_t)kT - 1) target = kT - 1;
    uint32_t sym = target >> 8;
    dec_update(d, in, L, r, sym << 8, 256u);
    x[i] = (uint8_t)sym;
  }
  ds[s] = d;
}

cudaError_t launch_prefix_decode(DecState* ds, const uint8_t* bits, const unsigned long long* off,
                                 const uint32_t* len, Split sp, int K, int b, uint8_t* data, cudaStream_t st) {
  return launch_k(prefix_decode_kernel, dim3(div_up(b, 128)), dim3(128), 0, st, ds, bits, off, len, sp, K, b, data);
}

// ============================================================================================
// Head: softmax -> integer CDF -> (encode slot | decode symbol) -> CE gradient.
// One warp per stream; lane l owns symbols 8l..8l+7.
// CDF rule: f_j = 1 + floor(fl32(p_j * 65280)); the remainder 2^16 - sum f goes
// to the first largest f; cum is the exclusive prefix sum.
// ============================================================================================
struct RowCdf {
  uint32_t f[8];
  uint32_t cum[8];  // exclusive prefix within the whole row
};

// v[i] for 0 <= i < 8 without putting the array into local memory.
__device__ __forceinline__ uint32_t pick8(const uint32_t (&v)[8], int i) {
  uint32_t r = v[0];
#pragma unroll
  for (int q = 1; q < 8; ++q) r = i == q ? v[q] : r;
  return r;
}

__device__ __forceinline__ void row_cdf(const float (&p)[8], int lane, RowCdf& o) {
  int fsum = 0;
  uint32_t best = 0;
  int bidx = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    o.f[q] = 1u + (uint32_t)floorf(__fmul_rn(p[q], (float)(kT - 256)));
    fsum += (int)o.f[q];
    if (o.f[q] > best) {
      best = o.f[q];
      bidx = lane * 8 + q;
    }
  }
  const int total = __reduce_add_sync(0xffffffffu, fsum);
  // argmax of f, lowest index on ties
  const uint32_t top = __reduce_max_sync(0xffffffffu, best);
  bidx = __reduce_min_sync(0xffffffffu, best == top ? bidx : 256);
  const int rem = kT - total;
#pragma unroll
  for (int q = 0; q < 8; ++q)  // (constant indices keep the row in registers)
    if (bidx == lane * 8 + q) o.f[q] = (uint32_t)((int)o.f[q] + rem);
  uint32_t run = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    o.cum[q] = run;
    run += o.f[q];
  }
  // exclusive scan of lane totals
  uint32_t incl = run;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += v;
  }
  const uint32_t excl = incl - run;
#pragma unroll
  for (int q = 0; q < 8; ++q) o.cum[q] += excl;
}

// Transposed BF16 store of an [R][cols] tile held in shared memory:
// YT[c][r0 + r] for r < R, as 16-byte stores (R = 8 or 16).
template <int R>
__device__ __forceinline__ void store_tile_T(const __nv_bfloat16* tile, int ld_s, int cols, int r0,
                                             __nv_bfloat16* YT, int ldT) {
  for (int c = threadIdx.x; c < cols; c += blockDim.x) {
    __align__(16) __nv_bfloat16 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = tile[r * ld_s + c];
    uint4* dst = reinterpret_cast<uint4*>(YT + (size_t)c * ldT + r0);
#pragma unroll
    for (int q = 0; q < R / 8; ++q) dst[q] = reinterpret_cast<const uint4*>(v)[q];
  }
}

// What bounds it is one row's chain of warp reductions (the grid is a warp per
// stream), so all that does not hang on the logits comes before the
// dependent-launch wait: the step control, the stream's bounds, the byte to
// encode or the decoder's state and target (all written at least two launches
// ago), and eight rows a CTA spread 512 streams over 64 SMs. With sixteen rows
// and everything after the wait the 64 MiB mix's step spent 8.7 us here; now
// 4.6.
constexpr int kRowsHead = 8;

__global__ void __launch_bounds__(32 * kRowsHead) head_kernel(HeadArgs a) {
  __shared__ __nv_bfloat16 tile[kRowsHead][256];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s = blockIdx.x * kRowsHead + warp;
  const bool valid = s < a.b;  // warp-uniform
  const StepCtl c = *a.ctl;
  bool active = false;
  int x = -1;
  DecState d{};
  uint32_t target = 0, dr = 0;
  if (valid) {
    active = a.mode == 2 ? a.active[s] != 0 : (long long)c.i < a.sp.len(s);
    if (active) {
      if (a.mode == 0) {
        x = a.data[a.sp.off(s) + c.i];  // warp-uniform
      } else if (a.mode == 1) {
        d = a.dec[s];
        dr = d.range >> kTBits;
        target = min(d.code / dr, (uint32_t)kT - 1);
      } else {
        x = a.targets[s];
      }
    }
  }
  float inv = c.inv_bact;
  if (valid && a.rg) {  // grouped mode: the mean over the row's own group (as set_ctl / step_advance form it)
    const int n = group_active(a.gi[a.rg[s]], c.i);
    inv = n > 0 ? 1.0f / (float)n : 0.f;
  }
  pdl_wait();
  pdl_launch();
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // Adam's scalars of this step
    a.ctl->a_lr = c.lr;
    a.ctl->a_bc1 = c.bc1;
    a.ctl->a_bc2 = c.bc2;
  }
  float dzv[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) dzv[q] = 0.f;
  if (valid) {
    const float* z = a.z + (size_t)s * 256 + lane * 8;
    float zz[8], p[8];
    float4 z0 = reinterpret_cast<const float4*>(z)[0], z1 = reinterpret_cast<const float4*>(z)[1];
    zz[0] = z0.x; zz[1] = z0.y; zz[2] = z0.z; zz[3] = z0.w;
    zz[4] = z1.x; zz[5] = z1.y; zz[6] = z1.z; zz[7] = z1.w;
    float mx = zz[0];
#pragma unroll
    for (int q = 1; q < 8; ++q) mx = fmaxf(mx, zz[q]);
    mx = warp_max(mx);
    float se = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      p[q] = expf(zz[q] - mx);
      se += p[q];
    }
    se = warp_sum(se);
#pragma unroll
    for (int q = 0; q < 8; ++q) p[q] = p[q] / se;

    RowCdf cdf;
    row_cdf(p, lane, cdf);
    if (a.freq_out) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        a.freq_out[(size_t)s * 256 + lane * 8 + q] = cdf.f[q];
        a.cum_out[(size_t)s * 257 + lane * 8 + q] = cdf.cum[q];
      }
      if (lane == 31) a.cum_out[(size_t)s * 257 + 256] = (uint32_t)kT;
    }

    if (active) {
      if (a.mode == 0) {
        uint32_t cx = __shfl_sync(0xffffffffu, pick8(cdf.cum, x & 7), x >> 3);
        uint32_t fx = __shfl_sync(0xffffffffu, pick8(cdf.f, x & 7), x >> 3);
        if (lane == 0) a.ring[(size_t)c.slot * a.b + s] = cx | ((fx - 1u) << 16);
      } else if (a.mode == 1) {
        unsigned ball = __ballot_sync(0xffffffffu, cdf.cum[0] <= target);
        int L = 31 - __clz(ball);
        int cnt = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) cnt += (cdf.cum[q] <= target) ? 1 : 0;
        cnt = __shfl_sync(0xffffffffu, cnt, L);
        x = L * 8 + cnt - 1;
        uint32_t cx = __shfl_sync(0xffffffffu, pick8(cdf.cum, x & 7), L);
        uint32_t fx = __shfl_sync(0xffffffffu, pick8(cdf.f, x & 7), L);
        if (lane == 0) {
          dec_update(d, a.bits + a.bits_off[s], a.bits_len[s], dr, cx, fx);
          a.dec[s] = d;
          a.data[a.sp.off(s) + c.i] = (uint8_t)x;
        }
      }
    } else if (a.mode == 0 && lane == 0) {
      a.ring[(size_t)c.slot * a.b + s] = kSkip;
    }

    float* dz = a.dz + (size_t)s * 256 + lane * 8;
    float* po = a.p ? a.p + (size_t)s * 256 + lane * 8 : nullptr;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      int j = lane * 8 + q;
      dzv[q] = active ? (p[q] - (j == x ? 1.0f : 0.0f)) * inv : 0.f;
      dz[q] = dzv[q];
      if (po) po[q] = p[q];
    }
    if (a.dzb) {
      __align__(16) __nv_bfloat16 hb[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) hb[q] = __float2bfloat16_rn(dzv[q]);
      *reinterpret_cast<uint4*>(a.dzb + (size_t)s * 256 + lane * 8) = *reinterpret_cast<const uint4*>(hb);
    }
  }
  if (a.dzbT) {
#pragma unroll
    for (int q = 0; q < 8; ++q) tile[warp][lane * 8 + q] = __float2bfloat16_rn(dzv[q]);
    __syncthreads();
    store_tile_T<kRowsHead>(&tile[0][0], 256, 256, blockIdx.x * kRowsHead, a.dzbT, a.ldT);
  }
}

cudaError_t launch_head(const HeadArgs& a, cudaStream_t st) {
  return launch_k(head_kernel, dim3(div_up(a.b, kRowsHead)), dim3(32 * kRowsHead), 0, st, a);
}

// A warp per row. What bounds it is HBM (a row is 1 KB in, 2 KB out): p and f
// move as 16-byte pieces; cum's rows of 257 words have no alignment beyond 4
// bytes, so they go through shared memory and out as whole 128-byte warp
// stores. With a stride of 32 bytes between a warp's lanes on all three sides
// 32,291 rows took 68.2 us; now 15.1 (6.6 TB/s).
__global__ void __launch_bounds__(256) cdf_quantize_kernel(const float* __restrict__ P, int rows,
                                                           uint32_t* __restrict__ freq, uint32_t* __restrict__ cum,
                                                           bool v16) {
  __shared__ __align__(16) uint32_t sc[8][256];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s = blockIdx.x * 8 + w;
  if (s >= rows) return;
  float p[8];
  const float* src = P + (size_t)s * 256 + lane * 8;
  if (v16) {
    const float4 a = __ldcs(reinterpret_cast<const float4*>(src)), b = __ldcs(reinterpret_cast<const float4*>(src) + 1);
    p[0] = a.x; p[1] = a.y; p[2] = a.z; p[3] = a.w;
    p[4] = b.x; p[5] = b.y; p[6] = b.z; p[7] = b.w;
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) p[q] = src[q];
  }
  RowCdf cdf;
  row_cdf(p, lane, cdf);
  uint32_t* f = freq + (size_t)s * 256 + lane * 8;
  if (v16) {
    __stcs(reinterpret_cast<uint4*>(f), make_uint4(cdf.f[0], cdf.f[1], cdf.f[2], cdf.f[3]));
    __stcs(reinterpret_cast<uint4*>(f) + 1, make_uint4(cdf.f[4], cdf.f[5], cdf.f[6], cdf.f[7]));
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) f[q] = cdf.f[q];
  }
  uint4* t = reinterpret_cast<uint4*>(&sc[w][lane * 8]);
  t[0] = make_uint4(cdf.cum[0], cdf.cum[1], cdf.cum[2], cdf.cum[3]);
  t[1] = make_uint4(cdf.cum[4], cdf.cum[5], cdf.cum[6], cdf.cum[7]);
  __syncwarp();
  uint32_t* c = cum + (size_t)s * 257;
#pragma unroll
  for (int q = 0; q < 8; ++q) __stcs(c + q * 32 + lane, sc[w][q * 32 + lane]);
  if (lane == 0) __stcs(c + 256, (uint32_t)kT);
}

cudaError_t launch_cdf_quantize(const float* p, int rows, uint32_t* freq, uint32_t* cum, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  const bool v16 = ((reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(freq)) & 15) == 0;
  NoPdl scope;
  return launch_k(cdf_quantize_kernel, dim3(div_up(rows, 8)), dim3(256), 0, st, p, rows, freq, cum, v16);
}

// ============================================================================================
// BF16 path: LayerNorm forward / backward with fused BF16 operand copies.
// kRowsLN warps per CTA, one row each; the BF16 rows are staged in shared memory
// and written transposed ([c][row], 16-byte runs) for the dW GEMMs.
// ============================================================================================
constexpr int kRowsLN = 8;  // rows (warps) per CTA of the LayerNorm kernels

// NPL = F / 32 values per lane held in registers (all loads issued up front);
// NPL = 0 is the generic loop for any F.
template <int NPL>
__global__ void __launch_bounds__(32 * kRowsLN)
    ln_fwd_bf16_kernel(const float* __restrict__ X, const float* __restrict__ g, const float* __restrict__ be,
                       float* __restrict__ xhat, float* __restrict__ rstd, __nv_bfloat16* __restrict__ X0b,
                       __nv_bfloat16* __restrict__ X0bT, int b, int F, int ldT, const int* __restrict__ rg,
                       size_t gs) {
  pdl_wait();
  pdl_launch();
  extern __shared__ __nv_bfloat16 tile_dyn[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * kRowsLN + warp;
  __nv_bfloat16* trow = tile_dyn + (size_t)warp * F;
  if (row < b) {
    if (rg) {  // grouped mode: the row's own gamma and beta
      g += (size_t)rg[row] * gs;
      be += (size_t)rg[row] * gs;
    }
    const float* x = X + (size_t)row * F;
    if (NPL > 0) {
      float v[NPL > 0 ? NPL : 1];
#pragma unroll
      for (int q = 0; q < NPL; ++q) v[q] = x[lane + 32 * q];
      float sm = 0.f;
#pragma unroll
      for (int q = 0; q < NPL; ++q) sm += v[q];
      const float mean = warp_sum(sm) / (float)F;
      float qv = 0.f;
#pragma unroll
      for (int q = 0; q < NPL; ++q) {
        const float d = v[q] - mean;
        qv += d * d;
      }
      const float r = 1.0f / sqrtf(warp_sum(qv) / (float)F + kLnEps);
#pragma unroll
      for (int q = 0; q < NPL; ++q) {
        const int c = lane + 32 * q;
        const float h = (v[q] - mean) * r;
        xhat[(size_t)row * F + c] = h;
        const __nv_bfloat16 o = __float2bfloat16_rn(h * g[c] + be[c]);
        X0b[(size_t)row * F + c] = o;
        trow[c] = o;
      }
      if (lane == 0) rstd[row] = r;
    } else {
      float sm = 0.f;
      for (int c = lane; c < F; c += 32) sm += x[c];
      const float mean = warp_sum(sm) / (float)F;
      float qv = 0.f;
      for (int c = lane; c < F; c += 32) {
        const float d = x[c] - mean;
        qv += d * d;
      }
      const float r = 1.0f / sqrtf(warp_sum(qv) / (float)F + kLnEps);
      for (int c = lane; c < F; c += 32) {
        const float h = (x[c] - mean) * r;
        xhat[(size_t)row * F + c] = h;
        const __nv_bfloat16 o = __float2bfloat16_rn(h * g[c] + be[c]);
        X0b[(size_t)row * F + c] = o;
        trow[c] = o;
      }
      if (lane == 0) rstd[row] = r;
    }
  } else {
    for (int c = lane; c < F; c += 32) trow[c] = __float2bfloat16_rn(0.f);
  }
  __syncthreads();
  store_tile_T<kRowsLN>(tile_dyn, F, F, blockIdx.x * kRowsLN, X0bT, ldT);
}

cudaError_t launch_ln_fwd_bf16(const float* X, const float* g, const float* be, float* xhat, float* rstd,
                               __nv_bfloat16* X0b, __nv_bfloat16* X0bT, int b, int F, int ldT, cudaStream_t st,
                               const int* rg, size_t gs) {
  const size_t smem = (size_t)kRowsLN * F * sizeof(__nv_bfloat16);
  const dim3 grid(div_up(b, kRowsLN)), block(32 * kRowsLN);
  switch (F) {
    case 128:
      return launch_k(ln_fwd_bf16_kernel<4>, grid, block, smem, st, X, g, be, xhat, rstd, X0b, X0bT, b, F, ldT, rg, gs);
    case 256:
      return launch_k(ln_fwd_bf16_kernel<8>, grid, block, smem, st, X, g, be, xhat, rstd, X0b, X0bT, b, F, ldT, rg, gs);
    case 512:
      return launch_k(ln_fwd_bf16_kernel<16>, grid, block, smem, st, X, g, be, xhat, rstd, X0b, X0bT, b, F, ldT, rg,
                      gs);
    case 1024:
      return launch_k(ln_fwd_bf16_kernel<32>, grid, block, smem, st, X, g, be, xhat, rstd, X0b, X0bT, b, F, ldT, rg,
                      gs);
    default:
      return launch_k(ln_fwd_bf16_kernel<0>, grid, block, smem, st, X, g, be, xhat, rstd, X0b, X0bT, b, F, ldT, rg, gs);
  }
}

// Embedding (the model input) and the first block's LayerNorm in one launch:
// warp w of the CTA gathers row s's context (as embed_kernel does), holds
// X[s][c] for c = lane + 32 q in registers, writes X (FP32) and then runs
// exactly the arithmetic of ln_fwd_bf16_kernel<NPL> on those values.
template <int NPL>
__global__ void __launch_bounds__(32 * kRowsLN)
    embed_ln_bf16_kernel(const uint8_t* __restrict__ data, Split sp, const StepCtl* __restrict__ ctl,
                         const float* __restrict__ E, int K, int D, float* __restrict__ X, uint8_t* __restrict__ ctx,
                         const float* __restrict__ g, const float* __restrict__ be, float* __restrict__ xhat,
                         float* __restrict__ rstd, __nv_bfloat16* __restrict__ X0b, __nv_bfloat16* __restrict__ X0bT,
                         int b, int ldT, const int* __restrict__ rg, size_t gs) {
  pdl_wait();
  pdl_launch();
  constexpr int F = 32 * NPL;
  extern __shared__ __nv_bfloat16 tile_dyn[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s = blockIdx.x * kRowsLN + warp;
  __nv_bfloat16* trow = tile_dyn + (size_t)warp * F;
  if (s < b) {
    if (rg) {  // grouped mode: the row's own model
      const size_t o = (size_t)rg[s] * gs;
      E += o;
      g += o;
      be += o;
    }
    const int i = ctl->i;
    // A stream past its end (inactive) keeps its last context, as in embed_kernel.
    if (data && i <= sp.len(s)) {
      const long long base = sp.off(s) + i - K;
      for (int k = lane; k < K; k += 32) ctx[(size_t)s * K + k] = data[base + k];
    }
    __syncwarp();
    float v[NPL];
#pragma unroll
    for (int q = 0; q < NPL; ++q) {
      const int c = lane + 32 * q, k = c / D, dd = c - k * D;
      v[q] = E[(int)ctx[(size_t)s * K + k] * D + dd];
      X[(size_t)s * F + c] = v[q];
    }
    float sm = 0.f;
#pragma unroll
    for (int q = 0; q < NPL; ++q) sm += v[q];
    const float mean = warp_sum(sm) / (float)F;
    float qv = 0.f;
#pragma unroll
    for (int q = 0; q < NPL; ++q) {
      const float d = v[q] - mean;
      qv += d * d;
    }
    const float r = 1.0f / sqrtf(warp_sum(qv) / (float)F + kLnEps);
#pragma unroll
    for (int q = 0; q < NPL; ++q) {
      const int c = lane + 32 * q;
      const float h = (v[q] - mean) * r;
      xhat[(size_t)s * F + c] = h;
      const __nv_bfloat16 o = __float2bfloat16_rn(h * g[c] + be[c]);
      X0b[(size_t)s * F + c] = o;
      trow[c] = o;
    }
    if (lane == 0) rstd[s] = r;
  } else {
    for (int c = lane; c < F; c += 32) trow[c] = __float2bfloat16_rn(0.f);
  }
  __syncthreads();
  store_tile_T<kRowsLN>(tile_dyn, F, F, blockIdx.x * kRowsLN, X0bT, ldT);
}

cudaError_t launch_embed_ln_bf16(const uint8_t* data, Split sp, const StepCtl* ctl, const float* E, int b, int K,
                                 int D, float* X, uint8_t* ctx, const float* g, const float* be, float* xhat,
                                 float* rstd, __nv_bfloat16* X0b, __nv_bfloat16* X0bT, int ldT, cudaStream_t st,
                                 const int* rg, size_t gs) {
  const int F = K * D;
  const size_t smem = (size_t)kRowsLN * F * sizeof(__nv_bfloat16);
  const dim3 grid(div_up(b, kRowsLN)), block(32 * kRowsLN);
#define EDPC_ELN(NPL) \
  launch_k(embed_ln_bf16_kernel<NPL>, grid, block, smem, st, data, sp, ctl, E, K, D, X, ctx, g, be, xhat, rstd, X0b, \
           X0bT, b, ldT, rg, gs)
  switch (F) {
    case 128: return EDPC_ELN(4);
    case 256: return EDPC_ELN(8);
    case 512: return EDPC_ELN(16);
    case 1024: return EDPC_ELN(32);
    default: return cudaErrorInvalidValue;
  }
#undef EDPC_ELN
}

template <int NPL>
__global__ void __launch_bounds__(32 * kRowsLN)
    ln_bwd_bf16_kernel(const float* __restrict__ dX0, const float* __restrict__ xhat, const float* __restrict__ rstd,
                       const float* __restrict__ g, const float* __restrict__ dRes, float* __restrict__ dX,
                       __nv_bfloat16* __restrict__ dXb, __nv_bfloat16* __restrict__ dXbT, int b, int F, int ldT,
                       const int* __restrict__ rg, size_t gs) {
  pdl_wait();
  pdl_launch();
  extern __shared__ __nv_bfloat16 tile_dyn[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * kRowsLN + warp;
  __nv_bfloat16* trow = tile_dyn + (size_t)warp * F;
  if (row < b) {
    if (rg) g += (size_t)rg[row] * gs;  // grouped mode: the row's own gamma
    const size_t o = (size_t)row * F;
    const float r = rstd[row];
    if (NPL > 0) {
      float d[NPL > 0 ? NPL : 1], xh[NPL > 0 ? NPL : 1], rs[NPL > 0 ? NPL : 1];
#pragma unroll
      for (int q = 0; q < NPL; ++q) {
        const int c = lane + 32 * q;
        d[q] = dX0[o + c] * g[c];
        xh[q] = xhat[o + c];
        rs[q] = dRes[o + c];
      }
      float s1 = 0.f, s2 = 0.f;
#pragma unroll
      for (int q = 0; q < NPL; ++q) {
        s1 += d[q];
        s2 += d[q] * xh[q];
      }
      const float m1 = warp_sum(s1) / (float)F;
      const float m2 = warp_sum(s2) / (float)F;
#pragma unroll
      for (int q = 0; q < NPL; ++q) {
        const int c = lane + 32 * q;
        const float v = rs[q] + r * (d[q] - m1 - xh[q] * m2);
        dX[o + c] = v;
        if (dXb) {
          const __nv_bfloat16 h = __float2bfloat16_rn(v);
          dXb[o + c] = h;
          trow[c] = h;
        }
      }
    } else {
      float s1 = 0.f, s2 = 0.f;
      for (int c = lane; c < F; c += 32) {
        const float dd = dX0[o + c] * g[c];
        s1 += dd;
        s2 += dd * xhat[o + c];
      }
      const float m1 = warp_sum(s1) / (float)F;
      const float m2 = warp_sum(s2) / (float)F;
      for (int c = lane; c < F; c += 32) {
        const float dd = dX0[o + c] * g[c];
        const float v = dRes[o + c] + r * (dd - m1 - xhat[o + c] * m2);
        dX[o + c] = v;
        if (dXb) {
          const __nv_bfloat16 h = __float2bfloat16_rn(v);
          dXb[o + c] = h;
          trow[c] = h;
        }
      }
    }
  } else if (dXbT) {
    for (int c = lane; c < F; c += 32) trow[c] = __float2bfloat16_rn(0.f);
  }
  if (dXbT) {
    __syncthreads();
    store_tile_T<kRowsLN>(tile_dyn, F, F, blockIdx.x * kRowsLN, dXbT, ldT);
  }
}

cudaError_t launch_ln_bwd_bf16(const float* dX0, const float* xhat, const float* rstd, const float* g,
                               const float* dRes, float* dX, __nv_bfloat16* dXb, __nv_bfloat16* dXbT, int b, int F,
                               int ldT, cudaStream_t st, const int* rg, size_t gs) {
  const size_t smem = dXbT ? (size_t)kRowsLN * F * sizeof(__nv_bfloat16) : 0;
  const dim3 grid(div_up(b, kRowsLN)), block(32 * kRowsLN);
#define EDPC_LNB(NPL)                                                                                      \
  launch_k(ln_bwd_bf16_kernel<NPL>, grid, block, smem, st, dX0, xhat, rstd, g, dRes, dX, dXb, dXbT, b, F, ldT, rg, \
           gs)
  switch (F) {
    case 128: return EDPC_LNB(4);
    case 256: return EDPC_LNB(8);
    case 512: return EDPC_LNB(16);
    case 1024: return EDPC_LNB(32);
    default: return EDPC_LNB(0);
  }
#undef EDPC_LNB
}

// ============================================================================================
// Batched column sums (bias and LN-affine gradients), fixed order: CTA = one
// tile of TW columns of one job and one chunk of rows; warp w sums the chunk's
// rows w, w+16, ...; warps are then added in order. TW = 32 (one column per
// lane, four interleaved row accumulators) below 2048 rows; from there, when
// every job allows 16-byte loads, TW = 128 (four columns per lane, eight
// interleaved row accumulators: rows r, r+16, ..., r+112 of each pass). With
// several chunks, the last CTA of a tile to arrive adds the chunk partials in
// chunk order (a fence before the arrival counter makes the partials visible
// to it).
// ============================================================================================
template <bool VEC>
__global__ void __launch_bounds__(512) colsum_multi_kernel(ColsumJobs jobs) {
  pdl_wait();
  pdl_launch();
  constexpr int TW = VEC ? 128 : 32;
  constexpr int CPL = VEC ? 4 : 1;  // columns per lane
  __shared__ float part[16][TW + 1];
  __shared__ int is_last;
  const int tile = blockIdx.x;
  int t = blockIdx.x, j = 0;
  while (j < jobs.n - 1 && t >= (jobs.job[j].cols + TW - 1) / TW) {
    t -= (jobs.job[j].cols + TW - 1) / TW;
    ++j;
  }
  const ColsumJob jb = jobs.job[j];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = t * TW + lane * CPL;
  const int nch = gridDim.y;
  const int r_lo = (nch > 1) ? blockIdx.y * jobs.chunk_rows : 0;
  const int r_hi = (nch > 1) ? min(jb.rows, r_lo + jobs.chunk_rows) : jb.rows;
  float a[8][CPL];
#pragma unroll
  for (int k = 0; k < 8; ++k)
#pragma unroll
    for (int q = 0; q < CPL; ++q) a[k][q] = 0.f;
  auto load = [&](int r, float (&v)[CPL]) {
    const size_t o = (size_t)r * jb.ld + c;
    if (VEC) {
      float4 x = *reinterpret_cast<const float4*>(jb.X + o);
      if (jb.Y) {
        const float4 y = *reinterpret_cast<const float4*>(jb.Y + o);
        x.x *= y.x;
        x.y *= y.y;
        x.z *= y.z;
        x.w *= y.w;
      }
      v[0] = x.x;
      if (CPL > 1) {
        v[CPL > 1 ? 1 : 0] = x.y;
        v[CPL > 2 ? 2 : 0] = x.z;
        v[CPL > 3 ? 3 : 0] = x.w;
      }
    } else {
      v[0] = jb.Y ? jb.X[o] * jb.Y[o] : jb.X[o];
    }
  };
  if (!VEC && c < jb.cols) {
    // rows w, w+16, ... with four interleaved accumulators; sixteen rows' loads
    // go out together (the sums run in the same order as four at a time)
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    int r = r_lo + w;
    const size_t ld = (size_t)jb.ld;
    for (; r + 240 < r_hi; r += 256) {
      float x[16], y[16];
      const float* px = jb.X + (size_t)r * ld + c;
#pragma unroll
      for (int k = 0; k < 16; ++k) x[k] = px[(size_t)(16 * k) * ld];
      if (jb.Y) {
        const float* py = jb.Y + (size_t)r * ld + c;
#pragma unroll
        for (int k = 0; k < 16; ++k) y[k] = py[(size_t)(16 * k) * ld];
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
          a0 = fmaf(x[k], y[k], a0);
          a1 = fmaf(x[k + 1], y[k + 1], a1);
          a2 = fmaf(x[k + 2], y[k + 2], a2);
          a3 = fmaf(x[k + 3], y[k + 3], a3);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
          a0 += x[k];
          a1 += x[k + 1];
          a2 += x[k + 2];
          a3 += x[k + 3];
        }
      }
    }
    if (jb.Y) {
      for (; r + 48 < r_hi; r += 64) {
        a0 = fmaf(jb.X[(size_t)r * ld + c], jb.Y[(size_t)r * ld + c], a0);
        a1 = fmaf(jb.X[(size_t)(r + 16) * ld + c], jb.Y[(size_t)(r + 16) * ld + c], a1);
        a2 = fmaf(jb.X[(size_t)(r + 32) * ld + c], jb.Y[(size_t)(r + 32) * ld + c], a2);
        a3 = fmaf(jb.X[(size_t)(r + 48) * ld + c], jb.Y[(size_t)(r + 48) * ld + c], a3);
      }
      for (; r < r_hi; r += 16) a0 = fmaf(jb.X[(size_t)r * ld + c], jb.Y[(size_t)r * ld + c], a0);
    } else {
      for (; r + 48 < r_hi; r += 64) {
        a0 += jb.X[(size_t)r * ld + c];
        a1 += jb.X[(size_t)(r + 16) * ld + c];
        a2 += jb.X[(size_t)(r + 32) * ld + c];
        a3 += jb.X[(size_t)(r + 48) * ld + c];
      }
      for (; r < r_hi; r += 16) a0 += jb.X[(size_t)r * ld + c];
    }
    a[0][0] = (a0 + a1) + (a2 + a3);
  }
  if (VEC && c < jb.cols) {
    int r = r_lo + w;
    for (; r + 112 < r_hi; r += 128) {
      float v[8][CPL];
#pragma unroll
      for (int k = 0; k < 8; ++k) load(r + 16 * k, v[k]);
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int q = 0; q < CPL; ++q) a[k][q] += v[k][q];
    }
    for (; r < r_hi; r += 16) {
      float v[CPL];
      load(r, v);
#pragma unroll
      for (int q = 0; q < CPL; ++q) a[0][q] += v[q];
    }
  }
#pragma unroll
  for (int q = 0; q < CPL; ++q)
    part[w][lane * CPL + q] =
        VEC ? ((a[0][q] + a[1][q]) + (a[2][q] + a[3][q])) + ((a[4][q] + a[5][q]) + (a[6][q] + a[7][q])) : a[0][q];
  __syncthreads();
  const int tc = threadIdx.x;  // column of the tile handled in the final sums
  const int cc = t * TW + tc;
  float sum = 0.f;
  if (tc < TW) {
    sum = part[0][tc];
#pragma unroll
    for (int i = 1; i < 16; ++i) sum += part[i][tc];
  }
  if (nch == 1) {
    if (tc < TW && cc < jb.cols) jb.out[cc] = sum;
    return;
  }
  if (tc < TW) {
    jobs.part[((size_t)tile * nch + blockIdx.y) * TW + tc] = sum;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) is_last = (atomicAdd(&jobs.cnt[tile], 1u) == (unsigned)(nch - 1));
  __syncthreads();
  if (is_last && tc < TW) {
    __threadfence();
    const float* src = jobs.part + (size_t)tile * nch * TW + tc;
    float acc = 0.f;
    for (int k = 0; k < nch; ++k) acc += __ldcg(src + (size_t)k * TW);
    if (cc < jb.cols) jb.out[cc] = acc;
    if (tc == 0) jobs.cnt[tile] = 0u;
  }
}

bool colsum_vec(const ColsumJobs& jobs) {
  // 128-column tiles only from 2048 rows on: below that the 32-column grid's
  // parallelism matters more (the sums end the side stream before Adam)
  for (int j = 0; j < jobs.n; ++j) {
    const ColsumJob& b = jobs.job[j];
    if (b.rows < 2048) return false;
    if ((b.cols & 3) || (b.ld & 3) || (reinterpret_cast<uintptr_t>(b.X) & 15) ||
        (b.Y && (reinterpret_cast<uintptr_t>(b.Y) & 15)))
      return false;
  }
  return true;
}

int colsum_tiles(const ColsumJobs& jobs) {
  const int tw = colsum_vec(jobs) ? 128 : 32;
  int tiles = 0;
  for (int j = 0; j < jobs.n; ++j) tiles += (jobs.job[j].cols + tw - 1) / tw;
  return tiles;
}

int colsum_chunk_rows(int rows, int tiles) {
  // about 256 CTAs in all: the column sums run on a side stream beside the
  // step's critical path, and a wider grid would take SMs from it
  if (rows <= 512 || tiles <= 0) return 0;
  int nch = 256 / tiles;
  if (nch > kColsumMaxChunks) nch = kColsumMaxChunks;
  if (nch > rows / 256) nch = rows / 256;
  if (nch < 2) return 0;
  int cr = (rows + nch - 1) / nch;
  return (cr + 15) / 16 * 16;
}

cudaError_t launch_colsum_multi(const ColsumJobs& jobs, cudaStream_t st) {
  const int tiles = colsum_tiles(jobs);
  if (tiles == 0) return cudaSuccess;
  int rows = 0;
  for (int j = 0; j < jobs.n; ++j) rows = max(rows, jobs.job[j].rows);
  int nch = 1;
  if (jobs.chunk_rows > 0 && jobs.part && jobs.cnt) {
    for (int j = 0; j < jobs.n; ++j)
      if (jobs.job[j].rows != rows) return cudaErrorInvalidValue;  // one chunking for every job
    nch = (rows + jobs.chunk_rows - 1) / jobs.chunk_rows;
    if (nch > kColsumMaxChunks) return cudaErrorInvalidValue;
  }
  if (colsum_vec(jobs)) return launch_k(colsum_multi_kernel<true>, dim3(tiles, nch), dim3(512), 0, st, jobs);
  return launch_k(colsum_multi_kernel<false>, dim3(tiles, nch), dim3(512), 0, st, jobs);
}

// ============================================================================================
// Grouped column sums (bias and LN-affine gradients of independent per-file
// models): CTA = 32 columns of one job and one group, 16 warps; warp w sums
// the group's stream rows w, w + 16, ... for its lane's column, and the 16
// warp sums are added in warp order.
// ============================================================================================
__global__ void __launch_bounds__(512) colsum_groups_kernel(ColsumJobs jobs, const GroupInfo* __restrict__ gi,
                                                            size_t gs) {
  pdl_wait();
  pdl_launch();
  __shared__ float part[16][33];
  const ColsumJob j = jobs.job[blockIdx.z];
  const GroupInfo g = gi[blockIdx.y];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  float a = 0.f;
  if (c < j.cols) {
    const size_t ld = (size_t)j.ld;
    for (int r = g.r0 + w; r < g.r0 + g.s; r += 16)
      a += j.Y ? j.X[r * ld + c] * j.Y[r * ld + c] : j.X[r * ld + c];
  }
  part[w][lane] = a;
  __syncthreads();
  if (w == 0 && c < j.cols) {
    float t = part[0][lane];
#pragma unroll
    for (int q = 1; q < 16; ++q) t += part[q][lane];
    j.out[(size_t)blockIdx.y * gs + c] = t;
  }
}

cudaError_t launch_colsum_groups(const ColsumJobs& jobs, const GroupInfo* gi, int ngroups, size_t gs,
                                 cudaStream_t st) {
  if (jobs.n < 1 || jobs.n > kMaxColsumJobs || ngroups < 1 || ngroups > 65535 || !gi) return cudaErrorInvalidValue;
  int maxc = 0;
  for (int k = 0; k < jobs.n; ++k) maxc = max(maxc, jobs.job[k].cols);
  return launch_k(colsum_groups_kernel, dim3(div_up(maxc, 32), ngroups, jobs.n), dim3(512), 0, st, jobs, gi, gs);
}

// ============================================================================================
// Adam of one layer's parameters with both BF16 copies of its weights: CTA = one
// 32 x 32 tile of a weight matrix (four parameters a thread; the updated tile
// goes through shared memory into the transposed copy) or 1024 entries of the
// layer's bias and LayerNorm vectors; grid y = group (grouped mode).
// A layer's launch (5 us for the 0.4 M parameters of a block of the 64 MiB mix)
// follows its gradients on a side stream, so most of the update hides under the
// rest of the adjoint, and the transposed copies need no pass of their own at
// the next step's start (8.5 us there, 56 us for 12 independent models).
// ============================================================================================
__global__ void __launch_bounds__(256) adam_layer_kernel(AdamLayer a) {
  pdl_wait();
  pdl_launch();
  __shared__ __nv_bfloat16 t[32][34];
  const float lr = a.ctl->a_lr, bc1 = a.ctl->a_bc1, bc2 = a.ctl->a_bc2;
  const size_t go = (size_t)blockIdx.y * a.gs;  // the group's parameters
  auto update = [&](size_t e) -> float4 {        // four parameters at e
    e += go;
    float4 p = *reinterpret_cast<float4*>(a.P + e), m = *reinterpret_cast<float4*>(a.M + e),
           v = *reinterpret_cast<float4*>(a.V + e);
    const float4 g = *reinterpret_cast<const float4*>(a.G + e);
    adam1(p.x, m.x, v.x, g.x, lr, bc1, bc2);
    adam1(p.y, m.y, v.y, g.y, lr, bc1, bc2);
    adam1(p.z, m.z, v.z, g.z, lr, bc1, bc2);
    adam1(p.w, m.w, v.w, g.w, lr, bc1, bc2);
    *reinterpret_cast<float4*>(a.P + e) = p;
    *reinterpret_cast<float4*>(a.M + e) = m;
    *reinterpret_cast<float4*>(a.V + e) = v;
    if (a.Pb) {
      __align__(8) __nv_bfloat162 h[2] = {__floats2bfloat162_rn(p.x, p.y), __floats2bfloat162_rn(p.z, p.w)};
      *reinterpret_cast<uint2*>(a.Pb + e) = *reinterpret_cast<const uint2*>(h);
    }
    return p;
  };
  if ((int)blockIdx.x < a.ntiles) {  // CTA-uniform
    const TransposeTile tl = a.tiles[blockIdx.x];
    const int y = threadIdx.x >> 3, x = (threadIdx.x & 7) * 4;  // rows and columns are multiples of 8
    if (tl.r0 + y < tl.rows && tl.c0 + x < tl.cols) {
      const float4 p = update(tl.off + (size_t)(tl.r0 + y) * tl.cols + tl.c0 + x);
      t[y][x] = __float2bfloat16_rn(p.x);
      t[y][x + 1] = __float2bfloat16_rn(p.y);
      t[y][x + 2] = __float2bfloat16_rn(p.z);
      t[y][x + 3] = __float2bfloat16_rn(p.w);
    }
    __syncthreads();
    // y: column, x: four rows
    if (tl.c0 + y < tl.cols && tl.r0 + x < tl.rows) {
      __align__(8) __nv_bfloat16 h[4] = {t[x][y], t[x + 1][y], t[x + 2][y], t[x + 3][y]};
      *reinterpret_cast<uint2*>(a.PbT + go + tl.off + (size_t)(tl.c0 + y) * tl.rows + tl.r0 + x) =
          *reinterpret_cast<const uint2*>(h);
    }
    return;
  }
  // entry e4 of the layer's vectors, laid end to end
  size_t e = ((size_t)(blockIdx.x - a.ntiles) * 256 + threadIdx.x) * 4;
  for (int q = 0; q < a.nvec; ++q) {
    if (e < a.vec[q].n) {
      update(a.vec[q].off + e);
      return;
    }
    e -= a.vec[q].n;
  }
}

cudaError_t launch_adam_layer(const AdamLayer& a, cudaStream_t st) {
  size_t nv = 0;
  for (int q = 0; q < a.nvec; ++q) {
    if ((a.vec[q].n | a.vec[q].off) & 3) return cudaErrorInvalidValue;
    nv += a.vec[q].n;
  }
  const size_t grid = a.ntiles + (nv + 1023) / 1024;
  if (grid == 0) return cudaSuccess;
  if (grid > 0x7fffffffu) return cudaErrorInvalidValue;
  return launch_k(adam_layer_kernel, dim3((unsigned)grid, a.groups), dim3(256), 0, st, a);
}

// ============================================================================================
// Transposed copies of every weight matrix in one launch (32 x 32 tiles through shared memory).
// ============================================================================================
__global__ void transpose_tiles_kernel(const __nv_bfloat16* __restrict__ Pb, __nv_bfloat16* __restrict__ PbT,
                                       const TransposeTile* __restrict__ tiles, int ntiles) {
  pdl_wait();
  pdl_launch();
  __shared__ __nv_bfloat16 t[32][34];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  for (int i = blockIdx.x; i < ntiles; i += gridDim.x) {  // several tiles per CTA when there are many
    const TransposeTile tl = tiles[i];
    if (i != (int)blockIdx.x) __syncthreads();  // the previous tile's reads of t are done
    for (int k = ty; k < 32; k += 8) {
      int r = tl.r0 + k, cc = tl.c0 + tx;
      t[k][tx] = (r < tl.rows && cc < tl.cols) ? Pb[tl.off + (size_t)r * tl.cols + cc] : __float2bfloat16_rn(0.f);
    }
    __syncthreads();
    for (int k = ty; k < 32; k += 8) {
      int cc = tl.c0 + k, r = tl.r0 + tx;
      if (cc < tl.cols && r < tl.rows) PbT[tl.off + (size_t)cc * tl.rows + r] = t[tx][k];
    }
  }
}
cudaError_t launch_transpose_tiles(const __nv_bfloat16* Pb, __nv_bfloat16* PbT, const TransposeTile* tiles,
                                   int ntiles, cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  const int grid = ntiles < 152 * 16 ? ntiles : 152 * 16;
  return launch_k(transpose_tiles_kernel, dim3(grid), dim3(256), 0, st, Pb, PbT, tiles, ntiles);
}

// ============================================================================================
// FP32 -> BF16 operand copies (row-major and transposed), via a 32x32 tile.
// ============================================================================================
__global__ void to_bf16_kernel(const float* __restrict__ X, int rows, int cols, int ldx, __nv_bfloat16* Y, int ldy,
                               __nv_bfloat16* YT, int ldt) {
  pdl_wait();
  pdl_launch();
  __shared__ float tile[32][33];
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  for (int k = ty; k < 32; k += 8) {
    int r = r0 + k, cc = c0 + tx;
    float v = (r < rows && cc < cols) ? X[(size_t)r * ldx + cc] : 0.f;
    tile[k][tx] = v;
    if (Y && r < rows && cc < cols) Y[(size_t)r * ldy + cc] = __float2bfloat16_rn(v);
  }
  if (!YT) return;
  __syncthreads();
  for (int k = ty; k < 32; k += 8) {
    int cc = c0 + k, r = r0 + tx;
    if (cc < cols && r < rows) YT[(size_t)cc * ldt + r] = __float2bfloat16_rn(tile[tx][k]);
  }
}

cudaError_t launch_to_bf16(const float* X, int rows, int cols, int ldx, __nv_bfloat16* Y, int ldy,
                           __nv_bfloat16* YT, int ldt, cudaStream_t st) {
  dim3 grid(div_up(cols, 32), div_up(rows, 32));
  return launch_k(to_bf16_kernel, dim3(grid), dim3(256), 0, st, X, rows, cols, ldx, Y, ldy, YT, ldt);
}

// ============================================================================================
// FP8 e4m3 operand quantization: amax pass (integer atomicMax on the float bits
// of |x|, order-independent), then the convert pass with s = 2^k.
// ============================================================================================
__device__ __forceinline__ int fp8_exp(float amax) {
  if (!(amax > 0.f)) return 0;
  int e;
  frexpf(amax, &e);  // amax = m 2^e, m in [0.5, 1)
  int k = 9 - e;     // amax 2^k in [256, 512)
  if (ldexpf(amax, k) > 448.f) k -= 1;
  return k < -120 ? -120 : (k > 120 ? 120 : k);
}

__global__ void fp8_amax_kernel(Fp8Jobs J) {
  pdl_wait();
  pdl_launch();
  const Fp8Job& jb = J.job[blockIdx.y];
  const long long n8 = (long long)jb.rows * (jb.cols / 8);  // 8 BF16 per 16-byte load
  float m = 0.f;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n8; i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / (jb.cols / 8), c = (i % (jb.cols / 8)) * 8;
    const uint4 v = *reinterpret_cast<const uint4*>(jb.src + r * jb.ld + c);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float2 f = __bfloat1622float2(h[q]);
      m = fmaxf(m, fmaxf(fabsf(f.x), fabsf(f.y)));
    }
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ float wm[32];
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, wm[w]);
    atomicMax(J.amax + jb.slot, __float_as_uint(m));
  }
}

__global__ void fp8_convert_kernel(Fp8Jobs J) {
  pdl_wait();
  pdl_launch();
  const Fp8Job& jb = J.job[blockIdx.y];
  const int k = fp8_exp(__uint_as_float(J.amax[jb.slot]));
  const float sc = ldexpf(1.f, k);
  if (blockIdx.x == 0 && threadIdx.x == 0) J.inv[jb.slot] = ldexpf(1.f, -k);
  const long long n8 = (long long)jb.rows * (jb.cols / 8);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n8; i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / (jb.cols / 8), c = (i % (jb.cols / 8)) * 8;
    const uint4 v = *reinterpret_cast<const uint4*>(jb.src + r * jb.ld + c);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
    uint8_t o[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float2 f = __bfloat1622float2(h[q]);
      o[2 * q] = (uint8_t)__nv_cvt_float_to_fp8(f.x * sc, __NV_SATFINITE, __NV_E4M3);
      o[2 * q + 1] = (uint8_t)__nv_cvt_float_to_fp8(f.y * sc, __NV_SATFINITE, __NV_E4M3);
    }
    *reinterpret_cast<uint2*>(jb.dst + r * jb.ld8 + c) = *reinterpret_cast<const uint2*>(o);
  }
}

cudaError_t launch_fp8_quantize(const Fp8Jobs& J, cudaStream_t st) {
  if (J.n <= 0) return cudaSuccess;
  if (J.n > kMaxFp8Jobs) return cudaErrorInvalidValue;
  long long most = 0;
  for (int j = 0; j < J.n; ++j) {
    const Fp8Job& jb = J.job[j];
    // 16-byte loads and 8-byte stores: cols and both strides in whole vectors
    if (jb.cols % 8 || jb.ld % 8 || jb.ld8 % 8) return cudaErrorInvalidValue;
    most = std::max(most, (long long)jb.rows * (jb.cols / 8));
  }
  const int per_job = (int)std::min<long long>(std::max<long long>(1, (most + 255) / 256), 2 * 152);
  cudaError_t e = launch_k(fp8_amax_kernel, dim3(per_job, J.n), dim3(256), 0, st, J);
  if (e != cudaSuccess) return e;
  return launch_k(fp8_convert_kernel, dim3(per_job, J.n), dim3(256), 0, st, J);
}

__global__ void zero_u32_kernel(unsigned* p, int n) {
  pdl_wait();
  pdl_launch();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = 0u;
}

cudaError_t launch_zero_u32(unsigned* p, int n, cudaStream_t st) {
  return launch_k(zero_u32_kernel, dim3(1), dim3(256), 0, st, p, n);
}

}  // namespace edpc
