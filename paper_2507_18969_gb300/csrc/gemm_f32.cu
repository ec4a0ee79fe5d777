// Plain FP32 SIMT GEMM with a fused bias / residual epilogue.
//
// This is the "plain FP32" arithmetic of the model's Linear layers
// (Eqs. 10, 13, 14, 16, the head, and their adjoints). Each output element
// sums its K products in increasing k order by fused multiply-adds, so results
// are deterministic and the same for every tile.
//
// Operands arrive by 16-byte asynchronous copies in STAGES stages of BKT = 32
// values of k, in the layout they have in memory: an operand whose k is
// contiguous as [m][k] rows of BKT + 4 floats (the padding puts eight
// consecutive rows on distinct banks), one whose m is contiguous as [k][m]
// rows. Either way a thread's TM (or TN) values of four consecutive k are TM
// (TN) 16-byte shared-memory loads, and four k are TM * TN * 4 FMAs.
#include "kernels.cuh"
#include "launch.cuh"

namespace edpc {

namespace {

constexpr int BKT = 32;

// Exact erf GELU and its derivative (Eqs. 11-12 and their adjoint).
__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

__device__ __forceinline__ void cp16(float* dst, const float* src, int bytes) {  // bytes < 16: zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src), "r"(bytes)
               : "memory");
}

// One operand of a tile: ROWS rows (m or n) by BKT values of k.
//   KC: k contiguous in memory; thread values r = t + i * T (T threads along the side)
//   else: the rows are contiguous; thread values come in runs of V = min(4, TR):
//         r = (i / V) * V * T + t * V + i % V
template <bool KC, int ROWS, int TR>
struct Operand {
  static constexpr int T = ROWS / TR;
  static constexpr int V = TR < 4 ? TR : 4;
  static constexpr int LD = KC ? BKT + 4 : ROWS;
  static constexpr int FLOATS = KC ? ROWS * LD : BKT * LD;
  static constexpr int PIECES = ROWS * BKT / 4;  // 16-byte pieces of a stage
  static_assert(KC || ROWS % 4 == 0, "rows are copied four at a time");

  static __device__ __forceinline__ int row(int t, int i) {
    return KC ? t + i * T : (i / V) * (V * T) + t * V + i % V;
  }
  template <int NT>
  static __device__ __forceinline__ void load(float* s, const float* __restrict__ X, int ld, int r0, int rows, int k0,
                                              int K, int tid) {
#pragma unroll
    for (int p = 0; p < (PIECES + NT - 1) / NT; ++p) {
      const int e = tid + p * NT;
      if (PIECES % NT && e >= PIECES) break;
      if (KC) {
        const int r = e / (BKT / 4), k = (e % (BKT / 4)) * 4;
        const int left = (r0 + r < rows) ? K - (k0 + k) : 0;
        const int n = left >= 4 ? 16 : (left > 0 ? left * 4 : 0);
        cp16(s + r * LD + k, n ? X + (size_t)(r0 + r) * ld + k0 + k : X, n);
      } else {
        const int k = e / (ROWS / 4), r = (e % (ROWS / 4)) * 4;
        const int left = (k0 + k < K) ? rows - (r0 + r) : 0;
        const int n = left >= 4 ? 16 : (left > 0 ? left * 4 : 0);
        cp16(s + k * LD + r, n ? X + (size_t)(k0 + k) * ld + r0 + r : X, n);
      }
    }
  }
  // f[q][i] = value of row(t, i) at k + q
  static __device__ __forceinline__ void frag(const float* s, int t, int k, float (&f)[4][TR]) {
    if (KC) {
#pragma unroll
      for (int i = 0; i < TR; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(s + row(t, i) * LD + k);
        f[0][i] = v.x;
        f[1][i] = v.y;
        f[2][i] = v.z;
        f[3][i] = v.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float* p = s + (k + q) * LD;
        if (V == 4) {
#pragma unroll
          for (int i = 0; i < TR; i += 4) {
            const float4 v = *reinterpret_cast<const float4*>(p + row(t, i));
            f[q][i] = v.x;
            f[q][i + (V > 1 ? 1 : 0)] = v.y;
            f[q][i + (V > 2 ? 2 : 0)] = v.z;
            f[q][i + (V > 3 ? 3 : 0)] = v.w;
          }
        } else {
#pragma unroll
          for (int i = 0; i < TR; ++i) f[q][i] = p[row(t, i)];
        }
      }
    }
  }
};

template <int BM, int BN, int TM, int TN, int STAGES, bool AK, bool BK, int KB>
struct Tile {
  using A = Operand<AK, BM, TM>;
  using B = Operand<BK, BN, TN>;
  static constexpr int TX = BN / TN, TY = BM / TM, NT = TX * TY;
  static constexpr int WX = TX < 8 ? TX : 8, WY = 32 / WX;  // threads of a warp along n and m
  static_assert(NT % 32 == 0 && TX % WX == 0 && TY % WY == 0, "whole warps");
  static constexpr int STAGE = A::FLOATS + KB * B::FLOATS;  // KB: sections of B (branches)
  static constexpr size_t kSmem = (size_t)STAGES * STAGE * sizeof(float);
};

// EPI_BRANCH: KB sections of B (rows i * H + n), one accumulator set each, so
// that the branches of a hidden unit meet in one thread; EPI_BRANCH_BWD: KB
// branches in the epilogue only.
template <int BM, int BN, int TM, int TN, int STAGES, bool AK, bool BK, int EPI, int KB>
__global__ void __launch_bounds__(Tile<BM, BN, TM, TN, STAGES, AK, BK, EPI == EPI_BRANCH ? KB : 1>::NT)
    gemm_f32_kernel(const GemmF32 g) {
  constexpr int SEC = EPI == EPI_BRANCH ? KB : 1;
  using S = Tile<BM, BN, TM, TN, STAGES, AK, BK, SEC>;
  extern __shared__ __align__(16) float smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tx = (warp % (S::TX / S::WX)) * S::WX + lane % S::WX;
  const int ty = (warp / (S::TX / S::WX)) * S::WY + lane / S::WX;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int nk = (g.K + BKT - 1) / BKT;
  auto load_a = [&](int kb) {
    S::A::template load<S::NT>(smem + (kb % STAGES) * S::STAGE, g.A, g.lda, m0, g.M, kb * BKT, g.K, tid);
  };
  auto load_b = [&](int kb) {
#pragma unroll
    for (int i = 0; i < SEC; ++i)
      S::B::template load<S::NT>(smem + (kb % STAGES) * S::STAGE + S::A::FLOATS + i * S::B::FLOATS,
                                 g.B + (size_t)i * g.N * g.ldb, g.ldb, n0, g.N, kb * BKT, g.K, tid);
  };
  // Weights (b_early) were written at least two launches earlier, so their
  // first stages are fetched before the dependent-launch wait.
  if (g.b_early)
    for (int q = 0; q < STAGES - 1 && q < nk; ++q) load_b(q);
  pdl_wait();
  pdl_launch();
  for (int q = 0; q < STAGES - 1; ++q) {
    if (q < nk) {
      if (!g.b_early) load_b(q);
      load_a(q);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float acc[SEC][TM][TN];
#pragma unroll
  for (int x = 0; x < SEC; ++x)
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[x][i][j] = 0.f;

  for (int kb = 0; kb < nk; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();  // stage kb has landed for every thread, and stage kb - 1 has been read
    if (kb + STAGES - 1 < nk) {
      load_b(kb + STAGES - 1);
      load_a(kb + STAGES - 1);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* sa = smem + (kb % STAGES) * S::STAGE;
    const float* sb = sa + S::A::FLOATS;
#pragma unroll
    for (int k = 0; k < BKT; k += 4) {
      float a[4][TM];
      S::A::frag(sa, ty, k, a);
#pragma unroll
      for (int x = 0; x < SEC; ++x) {
        float b[4][TN];
        S::B::frag(sb + x * S::B::FLOATS, tx, k, b);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[x][i][j] = fmaf(a[q][i], b[q][j], acc[x][i][j]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + S::A::row(ty, i);
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int n = n0 + S::B::row(tx, j);
      if (n >= g.N) continue;
      if (EPI == EPI_BRANCH) {  // X_i + c_i -> C, GELU of their product -> G2
        float* c = g.C + (size_t)m * g.ldc + n;
        float f = 1.f;
#pragma unroll
        for (int x = 0; x < SEC; ++x) {
          const float v = acc[x][i][j] + g.bias[x * g.N + n];
          c[(size_t)x * g.N] = v;
          f = x ? f * v : v;
        }
        g.G2[(size_t)m * g.N + n] = gelu_f(f);
      } else if (EPI == EPI_BRANCH_BWD) {  // the accumulator is dG; X_i are in R
        const float* a = g.R + (size_t)m * g.ldr + n;
        float xs[KB], f = 1.f;
#pragma unroll
        for (int x = 0; x < KB; ++x) {
          xs[x] = a[(size_t)x * g.N];
          f = x ? f * xs[x] : xs[x];
        }
        const float df = acc[0][i][j] * gelu_grad_f(f);
#pragma unroll
        for (int x = 0; x < KB; ++x) {
          float o = 1.f;
#pragma unroll
          for (int l = 0; l < KB; ++l)
            if (l != x) o *= xs[l];
          g.C[(size_t)m * g.ldc + (size_t)x * g.N + n] = df * o;
        }
      } else {
        float v = acc[0][i][j];
        if (EPI >= EPI_BIAS) v += g.bias[n];
        if (EPI == EPI_BIAS_RESID) v += g.R[(size_t)m * g.ldr + n];
        g.C[(size_t)m * g.ldc + n] = v;
      }
    }
  }
}

template <int BM, int BN, int TM, int TN, int STAGES, bool AK, bool BK, int EPI, int KB = 1>
cudaError_t launch_one(const GemmF32& g, cudaStream_t st) {
  using S = Tile<BM, BN, TM, TN, STAGES, AK, BK, EPI == EPI_BRANCH ? KB : 1>;
  auto k = gemm_f32_kernel<BM, BN, TM, TN, STAGES, AK, BK, EPI, KB>;
  static OncePerDevice once;
  const cudaError_t attr = once_on_device(
      once, [&] { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem); });
  if (attr != cudaSuccess) return attr;
  return launch_k(k, dim3(div_up(g.N, BN), div_up(g.M, BM)), dim3(S::NT), S::kSmem, st, g);
}

template <int BM, int BN, int TM, int TN, int STAGES>
cudaError_t launch_tile(const GemmF32& g, cudaStream_t st) {
  // the layouts the model uses: forward (A, B k-contiguous, with bias), input
  // gradient (A only) and weight gradient (neither)
  if (g.a_kcont && g.b_kcont) {
    if (g.epi == EPI_BIAS) return launch_one<BM, BN, TM, TN, STAGES, true, true, EPI_BIAS>(g, st);
    if (g.epi == EPI_BIAS_RESID) return launch_one<BM, BN, TM, TN, STAGES, true, true, EPI_BIAS_RESID>(g, st);
  }
  if (g.epi == EPI_BRANCH_BWD && g.a_kcont && !g.b_kcont) {
    if (g.k == 1) return launch_one<BM, BN, TM, TN, STAGES, true, false, EPI_BRANCH_BWD, 1>(g, st);
    if (g.k == 2) return launch_one<BM, BN, TM, TN, STAGES, true, false, EPI_BRANCH_BWD, 2>(g, st);
    if (g.k == 3) return launch_one<BM, BN, TM, TN, STAGES, true, false, EPI_BRANCH_BWD, 3>(g, st);
  }
  if (g.epi != EPI_STORE || g.b_kcont) return cudaErrorInvalidValue;
  if (g.a_kcont) return launch_one<BM, BN, TM, TN, STAGES, true, false, EPI_STORE>(g, st);
  return launch_one<BM, BN, TM, TN, STAGES, false, false, EPI_STORE>(g, st);
}

template <int BM, int BN, int TM, int TN, int STAGES>
cudaError_t launch_branch(const GemmF32& g, cudaStream_t st) {
  if (g.k == 1) return launch_one<BM, BN, TM, TN, STAGES, true, true, EPI_BRANCH, 1>(g, st);
  if (g.k == 2) return launch_one<BM, BN, TM, TN, STAGES, true, true, EPI_BRANCH, 2>(g, st);
  if (g.k == 3) return launch_one<BM, BN, TM, TN, STAGES, true, true, EPI_BRANCH, 3>(g, st);
  return cudaErrorInvalidValue;
}

bool vec16(const float* p, int ld) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && ld % 4 == 0; }

}  // namespace

cudaError_t launch_gemm_f32(const GemmF32& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  // every width is a multiple of 8 and every tensor 16-byte aligned (checked, for the 16-byte copies)
  if (!vec16(g.A, g.lda) || !vec16(g.B, g.ldb)) return cudaErrorInvalidValue;
  // Tile by the number of outputs: the largest that still gives the 152 SMs
  // work. A tile's chain over K is what the small ones wait for, so they take
  // more CTAs of fewer values each; the large ones are bound by the shared
  // memory's 128 bytes a cycle (TM + TN values in for TM * TN FMAs). Times in
  // us with the tiles on either side (and of the former 64 x 64 tile with
  // synchronous 4-byte loads), forward layout, M x N x K:
  //   64 x 512 x 512     8x8 5.1, 8x16 6.4 (32.9)      128 x 512 x 512   8x8 9.3, 8x16 7.1, 16x32 8.8 (33.0)
  //   512 x 256 x 512    8x16 10.0, 16x32 9.8 (33.3)   512 x 512 x 512   16x32 16.1, 32x64 14.7 (33.6)
  //   1024 x 512 x 512   32x64 20.1, 64x64 22.1 (33.7) 1024 x 1024 x 2048 (weight gradient) 32x64 127.8,
  //   64x64 106.1 (189.7)
  const long long outs = (long long)g.M * g.N;
  if (g.epi == EPI_BRANCH) {
    // k accumulator sets a thread: smaller tiles of hidden units. 16 x 32 for the
    // 64 MiB mix's 512 x 256 units (96 steps 63.0 ms; 32 x 32 tiles of 64 threads
    // 65.1, separate GEMM and GELU launches 63.3); at four streams the fused
    // launches take a small model's 512 steps from 38.1 to 36.2 ms.
    if (!g.a_kcont || !g.b_kcont) return cudaErrorInvalidValue;
    if (outs >= 512 << 10) return launch_branch<64, 32, 8, 4, 3>(g, st);
    if (outs >= 24 << 10) return launch_branch<16, 32, 4, 2, 5>(g, st);
    if (outs >= 12 << 10) return launch_branch<8, 16, 2, 2, 8>(g, st);
    return launch_branch<8, 8, 2, 1, 8>(g, st);
  }
  if (outs >= 1 << 20) return launch_tile<64, 64, 8, 4, 3>(g, st);
  if (outs >= 192 << 10) return launch_tile<32, 64, 4, 4, 4>(g, st);
  if (outs >= 96 << 10) return launch_tile<16, 32, 4, 2, 6>(g, st);
  if (outs >= 48 << 10) return launch_tile<8, 16, 2, 2, 8>(g, st);
  return launch_tile<8, 8, 2, 1, 8>(g, st);
}

}  // namespace edpc
