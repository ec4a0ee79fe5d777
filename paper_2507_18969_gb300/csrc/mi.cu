// Mutual information of Sec. 3.1.1 (Information Flow Refinement): Kraskov's
// k-nearest-neighbour estimate of I(Z; Y) between an MBRB's skip input and
// its fused output.
//
// ksg_dist_kernel computes the FP32 max-norm distances of every pair, tile by
// tile over the upper triangle, into an N x N matrix for Z and one for Y;
// ksg_select_kernel (a warp per sample i) takes eps(i) = the k-th smallest
// joint distance max(dz, dy) over j != i and counts c_z(i) = #{j != i:
// dz(i, j) < eps(i)} and c_y(i) likewise. |a - b| and max are exact in FP32 up
// to the one rounding of a - b (the same for b - a), so the counts are fixed
// by the FP32 samples, whatever the order.
// What bounds it is the FP32 pipe: a subtraction and a maximum per coordinate
// and pair, halved by the symmetry and by packed subtractions (two per
// instruction). With a CTA per sample that reads every other sample from L2 and
// selects over all N values with CTA-wide barriers, 2048 samples of 512 + 512
// coordinates took 1525 us a call; now 205 (distances 139, selection 19). That
// form (ksg_row_kernel) remains for few samples, where it is the faster one.
// The host then forms
// psi(k) + psi(N) - mean(psi(c_z + 1) + psi(c_y + 1)) in FP64.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "launch.cuh"

namespace edpc {

namespace {

constexpr int kTile = 64;  // samples of a distance tile's side
constexpr int kChunk = 32; // coordinates staged at a time
constexpr int kLd = kChunk + 4;  // padded: eight consecutive rows start on distinct banks
constexpr int kStages = 3;

__device__ __forceinline__ void cp_async(float* dst, const float* src, int bytes, bool v16) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  if (v16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

// Rows [r0, r0 + 64) and coordinates [q0, q0 + 32) of X (zeros beyond either
// end: a zero difference never raises a maximum of absolute values).
template <bool V16>
__device__ __forceinline__ void load_rows(float* s, const float* __restrict__ X, int N, int d, int r0, int q0) {
  constexpr int W = V16 ? 4 : 1;  // coordinates per copy
#pragma unroll 4
  for (int e = threadIdx.x; e < kTile * kChunk / W; e += 256) {
    const int r = e / (kChunk / W), q = (e % (kChunk / W)) * W;
    const bool in = r0 + r < N && q0 + q < d;  // (V16: d is a multiple of 4)
    cp_async(s + r * kLd + q, in ? X + (size_t)(r0 + r) * d + q0 + q : X, in ? 4 * W : 0, V16);
  }
}

// max(m, |a.x - b.x|, |a.y - b.y|), NaN differences ignored (as fmaxf does)
__device__ __forceinline__ float max_diff(float m, unsigned long long a, unsigned long long b) {
  unsigned long long x;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(x) : "l"(a), "l"(b));
  const float lo = __uint_as_float((unsigned)x), hi = __uint_as_float((unsigned)(x >> 32));
  return fmaxf(fmaxf(m, fabsf(lo)), fabsf(hi));
}

// D[z][i - r0][j] = max-norm distance of samples i and j of Z (z = 0) or Y
// (z = 1) for the rows r0 <= i < r0 + R of a panel, +infinity for j = i and for
// the columns N <= j < ld that pad a row. CTA (t, z) computes one 64 x 64 tile:
// of the upper triangle, stored both ways, when the panel holds every row;
// else of the panel's R x ld rectangle. 256 threads, 4 x 4 pairs each (rows
// ty + 16 a, columns tx + 16 b).
template <bool V16>
__global__ void __launch_bounds__(256) ksg_dist_kernel(const float* __restrict__ Z, const float* __restrict__ Y, int N,
                                                       int dz, int dy, float* __restrict__ D, int ld, int r0, int R) {
  extern __shared__ __align__(16) float sm[];  // kStages x (64 rows of i, 64 rows of j)
  const float* X = blockIdx.y ? Y : Z;
  const int d = blockIdx.y ? dy : dz;
  D += (size_t)blockIdx.y * R * ld;
  const int nt = ld / kTile;
  const bool sym = R == N;
  int ti = 0, t = blockIdx.x;
  if (sym) {  // row block ti holds the column blocks ti .. nt - 1
    while (t >= nt - ti) t -= nt - ti++;
    t += ti;
  } else {
    ti = t / nt;
    t -= ti * nt;
  }
  const int i0 = r0 + ti * kTile, j0 = t * kTile;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);
  const int nq = (d + kChunk - 1) / kChunk;
  auto load = [&](int c) {
    float* s = sm + (c % kStages) * (2 * kTile * kLd);
    load_rows<V16>(s, X, N, d, i0, c * kChunk);
    load_rows<V16>(s + kTile * kLd, X, N, d, j0, c * kChunk);
  };
  for (int c = 0; c < kStages - 1; ++c) {
    if (c < nq) load(c);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float m[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) m[a][b] = 0.f;
  for (int c = 0; c < nq; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();
    if (c + kStages - 1 < nq) load(c + kStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* si = sm + (c % kStages) * (2 * kTile * kLd);
    const float* sj = si + kTile * kLd;
    const int qe = min(kChunk, d - c * kChunk);
#pragma unroll 8
    for (int q = 0; q < qe; q += 4) {
      ulonglong2 vi[4], vj[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        vi[a] = *reinterpret_cast<const ulonglong2*>(si + (ty + 16 * a) * kLd + q);
        vj[a] = *reinterpret_cast<const ulonglong2*>(sj + (tx + 16 * a) * kLd + q);
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) m[a][b] = max_diff(max_diff(m[a][b], vi[a].x, vj[b].x), vi[a].y, vj[b].y);
    }
  }
  const float inf = __int_as_float(0x7f800000);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int i = i0 + ty + 16 * a;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int j = j0 + tx + 16 * b;
      const float v = (i == j || i >= N || j >= N) ? inf : m[a][b];
      if (i < r0 + R) D[(size_t)(i - r0) * ld + j] = v;
      if (sym && j0 > i0 && j < N) D[(size_t)j * ld + i] = v;  // the other triangle
    }
  }
}

// Counts of one sample per warp. The k-th smallest joint distance is at most
// the k-th smallest of the 32 lanes' minima (k <= 32), so only the values up
// to that bound go into the warp's list (N floats of shared memory, enough for
// all of them), where an exact radix select on the bits of the non-negative
// floats (31 passes of warp-wide counts) finds it.
__global__ void ksg_select_kernel(const float* __restrict__ D, int R, int ld, int k, unsigned* __restrict__ cz,
                                  unsigned* __restrict__ cy) {
  extern __shared__ __align__(16) float sm[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * (blockDim.x >> 5) + w;
  if (i >= R) return;
  float* list = sm + (size_t)w * ld;
  const float4* rz = reinterpret_cast<const float4*>(D + (size_t)i * ld);
  const float4* ry = reinterpret_cast<const float4*>(D + (size_t)(R + i) * ld);
  const int n4 = ld / 4;
  const float inf = __int_as_float(0x7f800000);
  float mn = inf;
#pragma unroll 4
  for (int e = lane; e < n4; e += 32) {
    const float4 a = rz[e], b = ry[e];
    mn = fminf(mn, fminf(fminf(fmaxf(a.x, b.x), fmaxf(a.y, b.y)), fminf(fmaxf(a.z, b.z), fmaxf(a.w, b.w))));
  }
  float bound = inf;
  if (k <= 32) {
    // rank of this lane's minimum among the 32 (ties by lane); rank k - 1 holds the bound
    int rank = 0;
    for (int l = 0; l < 32; ++l) {
      const float o = __shfl_sync(0xffffffffu, mn, l);
      rank += (o < mn || (o == mn && l < lane)) ? 1 : 0;
    }
    const unsigned at = __ballot_sync(0xffffffffu, rank == k - 1);
    bound = __shfl_sync(0xffffffffu, mn, __ffs(at) - 1);
  }
  int m = 0;  // values in the list
  for (int e0 = 0; e0 < n4; e0 += 32) {
    const int e = e0 + lane;
    float u[4] = {inf, inf, inf, inf};
    if (e < n4) {
      const float4 a = rz[e], b = ry[e];
      u[0] = fmaxf(a.x, b.x);
      u[1] = fmaxf(a.y, b.y);
      u[2] = fmaxf(a.z, b.z);
      u[3] = fmaxf(a.w, b.w);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bool in = e < n4 && u[q] <= bound;
      const unsigned hit = __ballot_sync(0xffffffffu, in);
      if (in) list[m + __popc(hit & ((1u << lane) - 1u))] = u[q];
      m += __popc(hit);
    }
  }
  __syncwarp();
  unsigned prefix = 0, mask = 0;
  int kk = k;
  for (int bit = 30; bit >= 0; --bit) {
    int c = 0;
    for (int j = lane; j < m; j += 32) {
      const unsigned u = __float_as_uint(list[j]);
      c += ((u & mask) == prefix && ((u >> bit) & 1u) == 0u) ? 1 : 0;
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (c < kk) {
      kk -= c;
      prefix |= 1u << bit;
    }
    mask |= 1u << bit;
  }
  const float eps = __uint_as_float(prefix);
  int nz = 0, ny = 0;
#pragma unroll 4
  for (int e = lane; e < n4; e += 32) {
    const float4 a = rz[e], b = ry[e];
    nz += (a.x < eps) + (a.y < eps) + (a.z < eps) + (a.w < eps);
    ny += (b.x < eps) + (b.y < eps) + (b.z < eps) + (b.w < eps);
  }
  nz = __reduce_add_sync(0xffffffffu, nz);
  ny = __reduce_add_sync(0xffffffffu, ny);
  if (lane == 0) {
    cz[i] = (unsigned)nz;
    cy[i] = (unsigned)ny;
  }
}

// Few samples: CTA i computes the distances of sample i to every sample j (a warp
// per j, lanes over the coordinates, a butterfly maximum) into shared memory,
// selects eps(i) with CTA-wide counts and counts c_z and c_y. One launch, no
// workspace, a CTA per sample: the tiles above are too few CTAs by then, and each
// runs through all the coordinates alone. The same exact differences and maxima,
// so the same counts.
constexpr int kRowThreads = 256;

__device__ __forceinline__ int block_sum(int v, int* red) {
  v = __reduce_add_sync(0xffffffffu, v);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  int s = 0;
#pragma unroll
  for (int q = 0; q < kRowThreads / 32; ++q) s += red[q];
  return s;
}

__global__ void __launch_bounds__(kRowThreads) ksg_row_kernel(const float* __restrict__ Z, const float* __restrict__ Y,
                                                              int N, int dz, int dy, int k, unsigned* __restrict__ cz,
                                                              unsigned* __restrict__ cy) {
  extern __shared__ __align__(16) float sm[];
  float* zi = sm;        // dz
  float* yi = zi + dz;   // dy
  float* sdz = yi + dy;  // N
  float* sdy = sdz + N;  // N
  __shared__ int red[kRowThreads / 32];
  const int i = blockIdx.x, t = threadIdx.x;
  const int w = t >> 5, lane = t & 31;
  for (int q = t; q < dz; q += kRowThreads) zi[q] = Z[(size_t)i * dz + q];
  for (int q = t; q < dy; q += kRowThreads) yi[q] = Y[(size_t)i * dy + q];
  __syncthreads();
  for (int j = w; j < N; j += kRowThreads / 32) {
    float a = 0.f, b = 0.f;
    for (int q = lane; q < dz; q += 32) a = fmaxf(a, fabsf(Z[(size_t)j * dz + q] - zi[q]));
    for (int q = lane; q < dy; q += 32) b = fmaxf(b, fabsf(Y[(size_t)j * dy + q] - yi[q]));
    for (int o = 16; o > 0; o >>= 1) {
      a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
      b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
    if (lane == 0) {
      sdz[j] = a;
      sdy[j] = b;
    }
  }
  __syncthreads();
  unsigned prefix = 0, mask = 0;
  int kk = k;
  for (int bit = 30; bit >= 0; --bit) {
    int c = 0;
    for (int j = t; j < N; j += kRowThreads) {
      if (j == i) continue;
      const unsigned u = __float_as_uint(fmaxf(sdz[j], sdy[j]));
      c += ((u & mask) == prefix && ((u >> bit) & 1u) == 0u) ? 1 : 0;
    }
    c = block_sum(c, red);
    if (c < kk) {
      kk -= c;
      prefix |= 1u << bit;
    }
    mask |= 1u << bit;
  }
  const float eps = __uint_as_float(prefix);
  int nz = 0, ny = 0;
  for (int j = t; j < N; j += kRowThreads) {
    if (j == i) continue;
    nz += sdz[j] < eps ? 1 : 0;
    ny += sdy[j] < eps ? 1 : 0;
  }
  nz = block_sum(nz, red);
  ny = block_sum(ny, red);
  if (t == 0) {
    cz[i] = (unsigned)nz;
    cy[i] = (unsigned)ny;
  }
}

// Which of the two: a tile's chain over max(dz, dy) coordinates against the row
// kernel's N / 8 samples a warp. Calls in us, rows / tiles, dz = dy:
//   32 samples: 39 / 41 (1 coordinate), 49 / 66 (512)     64: 42 / 41 (33), 42 / 44 (128), 49 / 66 (512)
//   96: 50 / 43 (128), 50 / 52 (256), 62 / 65 (512)        128: 52 / 45 (128), 51 / 54 (256), 64 / 66 (512)
//   160: 51 / 45 (128), 56 / 54 (256), 78 / 65 (512)
// Rows that are not 16-byte aligned cost the row kernel more: 128: 76 / 68 (511).
bool use_rows(int N, int dz, int dy, bool v16) {
  return N < 64 || (N <= (v16 ? 128 : 96) && std::max(dz, dy) >= 2 * N);
}
static_assert(sizeof(float) * (8192 + 2 * 128) <= 48 * 1024, "the row kernel needs no attribute");

// The distance workspace comes from a memory pool of the library's own, one per
// device, that keeps at most kWorkspace bytes between calls (stream-ordered, so
// concurrent calls on any threads and streams get buffers of their own; what
// they hold beyond that goes back to the device when they synchronize). A pool
// lives as long as its device's context: nothing destroys it at process exit,
// when the driver may be gone already, and a process that resets a device with
// cudaDeviceReset must not call this entry point on it again.
constexpr size_t kWorkspace = (size_t)64 << 20;
cudaMemPool_t g_pool[OncePerDevice::kDevices] = {};

cudaError_t workspace_alloc(float** p, size_t bytes, cudaStream_t st) {
  static OncePerDevice once;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= OncePerDevice::kDevices)  // the device's default pool, which keeps nothing unless it is told to
    return cudaMallocAsync(reinterpret_cast<void**>(p), bytes, st);
  e = once.run(dev, [&] {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    cudaError_t r = cudaMemPoolCreate(&pool, &props);
    if (r != cudaSuccess) return r;
    uint64_t keep = kWorkspace;
    r = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (r != cudaSuccess)
      cudaMemPoolDestroy(pool);
    else
      g_pool[dev] = pool;
    return r;
  });
  return e != cudaSuccess ? e : cudaMallocFromPoolAsync(reinterpret_cast<void**>(p), bytes, g_pool[dev], st);
}

// The tiled form: the distances into the workspace, then the counts.
int launch_tiles(const float* Z, const float* Y, int N, int dz, int dy, int k, bool v16, uint32_t* cz, uint32_t* cy,
                 cudaStream_t st) {
  constexpr size_t kDistSmem = (size_t)kStages * 2 * kTile * kLd * sizeof(float);
  constexpr size_t kListSmem = 128 * 1024;
  static OncePerDevice once;
  const cudaError_t attr = once_on_device(once, [] {
    cudaError_t r =
        cudaFuncSetAttribute(ksg_dist_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDistSmem);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(ksg_dist_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDistSmem);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(ksg_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kListSmem);
    return r;
  });
  if (attr != cudaSuccess) return fail(EDPC_ECUDA, std::string("ksg attribute: ") + cudaGetErrorString(attr));
  // The distances of all rows at once where they fit kWorkspace; else panels of rows.
  const int ld = (int)round_up(N, kTile);
  const size_t row = 2 * sizeof(float) * (size_t)ld;
  int R = N;
  if (row * N > kWorkspace) R = (int)(kWorkspace / row / kTile * kTile);
  float* D = nullptr;
  cudaError_t e = workspace_alloc(&D, row * R, st);
  while (e == cudaErrorMemoryAllocation && R > kTile) {  // a smaller panel when memory is short
    cudaGetLastError();
    R = (int)round_up(R / 2, kTile);
    e = workspace_alloc(&D, row * R, st);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(e == cudaErrorMemoryAllocation ? EDPC_ENOMEM : EDPC_ECUDA,
                std::string("ksg workspace: ") + cudaGetErrorString(e));
  }
  const int warps = (int)std::min<size_t>(8, kListSmem / (sizeof(float) * ld));
  const unsigned nt = ld / kTile;
  for (int r0 = 0; r0 < N && e == cudaSuccess; r0 += R) {
    const int rows = std::min(R, N - r0);
    const unsigned tiles = rows == N ? nt * (nt + 1) / 2 : nt * div_up(rows, kTile);
    auto k1 = v16 ? ksg_dist_kernel<true> : ksg_dist_kernel<false>;
    e = launch_k(k1, dim3(tiles, 2), dim3(256), kDistSmem, st, Z, Y, N, dz, dy, D, ld, r0, rows);
    if (e == cudaSuccess)
      e = launch_k(ksg_select_kernel, dim3(div_up(rows, warps)), dim3(32 * warps), sizeof(float) * ld * warps, st,
                   (const float*)D, rows, ld, k, (unsigned*)cz + r0, (unsigned*)cy + r0);
  }
  {
    const cudaError_t f = cudaFreeAsync(D, st);
    if (e == cudaSuccess) e = f;
  }
  return e == cudaSuccess ? EDPC_OK : fail(EDPC_ECUDA, std::string("ksg: ") + cudaGetErrorString(e));
}

// psi(x) for x >= 1: recurrence up to x >= 10, then the asymptotic series
// ln x - 1/(2x) - sum_n B_2n / (2n x^2n) (Abramowitz & Stegun 6.3.6, 6.3.18).
double digamma_ge1(double x) {
  double r = 0;
  while (x < 10.0) {
    r -= 1.0 / x;
    x += 1.0;
  }
  const double x2 = 1.0 / (x * x);
  const double series =
      x2 * (1.0 / 12 - x2 * (1.0 / 120 - x2 * (1.0 / 252 - x2 * (1.0 / 240 - x2 * (1.0 / 132 - x2 * 691.0 / 32760)))));
  return r + std::log(x) - 0.5 / x - series;
}

}  // namespace

}  // namespace edpc

using namespace edpc;

extern "C" int edpc_ksg_mi(const float* Z, const float* Y, uint32_t N, uint32_t dz, uint32_t dy, uint32_t k,
                           uint32_t* cz, uint32_t* cy, double* mi, void* cuda_stream) {
  if (!Z || !Y || !cz || !cy || !mi) return fail(EDPC_EINVAL, "NULL argument");
  if (N < 2 || N > 8192) return fail(EDPC_EINVAL, "N must be in [2, 8192]");
  if (k < 1 || k >= N || k > 64) return fail(EDPC_EINVAL, "k must be in [1, min(64, N - 1)]");
  if (dz < 1 || dy < 1 || dz + dy > 8192) return fail(EDPC_EINVAL, "dz, dy >= 1 and dz + dy <= 8192");
  const bool v16 = dz % 4 == 0 && dy % 4 == 0 &&
                   ((reinterpret_cast<uintptr_t>(Z) | reinterpret_cast<uintptr_t>(Y)) & 15) == 0;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  NoPdl scope;
  cudaError_t e = cudaSuccess;
  if (use_rows((int)N, (int)dz, (int)dy, v16))
    e = launch_k(ksg_row_kernel, dim3(N), dim3(kRowThreads), sizeof(float) * ((size_t)dz + dy + 2 * (size_t)N), st, Z, Y,
                 (int)N, (int)dz, (int)dy, (int)k, (unsigned*)cz, (unsigned*)cy);
  else
    EDPC_TRY(launch_tiles(Z, Y, (int)N, (int)dz, (int)dy, (int)k, v16, cz, cy, st));
  std::vector<uint32_t> hz(N), hy(N);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hz.data(), cz, 4 * (size_t)N, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hy.data(), cy, 4 * (size_t)N, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return fail(EDPC_ECUDA, std::string("ksg: ") + cudaGetErrorString(e));
  // counts repeat: each psi(c + 1) is formed once (0 marks one not formed yet; psi has no integer root)
  std::vector<double> psi(N, 0.0);
  auto psi1 = [&](uint32_t c) {
    if (psi[c] == 0.0) psi[c] = digamma_ge1(c + 1.0);
    return psi[c];
  };
  double s = 0;
  for (uint32_t q = 0; q < N; ++q) {
    const double pz = psi1(hz[q]);
    s += pz + psi1(hy[q]);
  }
  *mi = digamma_ge1((double)k) + digamma_ge1((double)N) - s / N;
  return EDPC_OK;
}
