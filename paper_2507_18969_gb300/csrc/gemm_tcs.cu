// BF16 GEMM of a Linear layer over few streams, with the streams on the MMA's
// N side: D^T = W X^T on the 5th-generation tensor cores.
//
// The forward and input-gradient GEMMs of a step of some hundred streams are a
// chain of launches of a few microseconds each, so what counts is the time
// from the predecessor's end to this launch's last store. With the 128 rows of
// the MMA taken from the weights, the part of the operands that comes from the
// predecessor is NS (32 or 64) rows instead of 128: 32 KB instead of 128 KB at
// K = 512, into an SM that takes about 146 GB/s. The weights' 128 rows were
// written launches ago and are in shared memory (or on their way) before the
// dependent-launch wait. The accumulator then holds a feature per TMEM lane and
// a stream per column: row-major outputs are stores of 32 consecutive features
// a warp, the transposed BF16 copies are runs of a lane's own streams, the bias
// is one value a lane, and no output passes through shared memory.
//
// At 512 streams, F = 512, H = 256, in the step (one-tile kernel before): branch
// GEMM 5.7 -> 5.2 us, its adjoint 6.1 -> 4.8, out GEMM 3.7 -> 3.2, head 5.4 -> 4.3;
// and, back to back, branch GEMM 5.8 -> 4.8, adjoint 6.6 -> 5.7, a plain K = 512
// 4.9 -> 4.0 once the issuing warps ran as whole warps (elect_one). What is left
// is the chain: 0.35 us until the first stage lands, 0.22 us a K block of 64 for
// its four MMAs, 0.4 to 1.3 us of epilogue, and the hand-over between launches.
//
// Per element the products, their order over K and the epilogue's operations
// are those of gemm_tc_kernel, and so are the results, bit for bit.
//
//   warp 8 (a lane)    TMA loads into an 8-stage ring: 128 rows of W (in the
//                      branch GEMM 128 / k rows of each branch's section, 32
//                      for k = 3) and NS rows of X, 64 BF16 of K a stage;
//   warp 9 (a lane)    tcgen05.mma (M = 128, N = NS), TMEM allocation;
//   warps 0-7          epilogue: warp w reads lanes 32 (w & 3) .. of the columns
//                      of half w >> 2; loads that do not depend on the
//                      accumulator, and GELU's derivative, come before.
// Waits are bounded as in gemm_tc_kernel.
#include "gemm_tc.cuh"
#include "gemm_tc_dev.cuh"
#include "kernels.cuh"
#include "launch.cuh"

namespace edpc {

namespace {

using namespace tc;

constexpr int kStagesS = 8;
constexpr int kThreadsS = kEpiThreads + 64;

// Stages of a launch of nk K blocks: no more than those, since the side streams'
// GEMMs share the SMs; at least two, whose space the branch GEMM's exchange takes.
__host__ __device__ constexpr int stages_s(int nk) { return nk < 2 ? 2 : (nk < kStagesS ? nk : kStagesS); }

// Rows of W a section takes: all 128 but in the branch GEMM.
template <int MODE, int KB>
constexpr int section_rows() { return MODE != TC_BRANCH ? 128 : (KB == 1 ? 128 : (KB == 2 ? 64 : 32)); }

template <int NS>
constexpr size_t smem_bytes_s(int stages) { return 1024 + (size_t)stages * (BM * BKB + NS * BKB) + 256; }

// 8 consecutive streams of a lane into the transposed copy (16-byte aligned run).
__device__ __forceinline__ void put_run8(const TcEpi& e, int col, int s, const float* v) {
  if (s + 8 <= e.ldct) *reinterpret_cast<uint4*>(e.CbT + (size_t)col * e.ldct + s) = pack8(v);
}

template <int NS, int MODE, int KB>
__global__ void __launch_bounds__(kThreadsS, 1)
    gemm_tcs_kernel(const __grid_constant__ CUtensorMap tw, const __grid_constant__ CUtensorMap tx, const TcEpi e) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  constexpr int SECTIONS = (MODE == TC_BRANCH) ? KB : 1;
  constexpr int SR = section_rows<MODE, KB>();
  constexpr uint32_t W_BYTES = BM * BKB, X_BYTES = NS * BKB;
  constexpr uint32_t TX_BYTES = SECTIONS * SR * BKB + X_BYTES;
  constexpr int NC = NS / 2;  // columns (streams) of an epilogue thread
  uint8_t* sW = smem;
  const int nk = (e.K + 63) / 64;
  const int nst = stages_s(nk);  // stages of this launch
  uint8_t* sX = smem + nst * W_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(sX + nst * X_BYTES);
  uint64_t* empty = full + kStagesS;
  uint64_t* done = empty + kStagesS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * SR;  // first feature (of every section: hidden unit)
  const int m0 = blockIdx.y * NS;  // first stream

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStagesS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tw)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tx)) : "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)tmem_cols<NS>()));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  auto load_w = [&](int kb, int s) {
    mbar_expect_tx(&full[s], TX_BYTES);
#pragma unroll
    for (int i = 0; i < SECTIONS; ++i)
      tma_load_2d(sW + s * W_BYTES + i * (SR * BKB), &tw, kb * 64, (MODE == TC_BRANCH ? i * e.H : 0) + n0, &full[s]);
  };
  if (warp == 8) {
    for (int kb = 0; kb < nk && kb < nst; ++kb) {
      if (elect_one()) load_w(kb, kb);
      __syncwarp();
    }
  }

  // The epilogue's inputs besides the accumulator (written two or more
  // launches ago): the lane's bias, the residual or the saved branch outputs.
  const int r = (warp & 3) * 32 + lane;          // TMEM lane
  const int sec = r / SR, u = r - sec * SR;      // section and feature within it
  const int width = MODE == TC_PLAIN ? e.N : e.H;
  const int col = n0 + u;                        // feature / hidden unit
  const bool cok = col < width && sec < SECTIONS;
  const int s0 = m0 + (warp >> 2) * NC;          // the thread's first stream
  float bias = 0.f;
  float pre[MODE == TC_BRANCH ? 1 : (MODE == TC_BRANCH_BWD ? KB : 1)][NC];
  if (warp < 8 && cok) {
    if (MODE != TC_BRANCH_BWD && e.bias) bias = e.bias[(MODE == TC_BRANCH ? sec * e.H : 0) + col];
    if (MODE == TC_PLAIN && e.R) {
#pragma unroll
      for (int j = 0; j < NC; ++j) pre[0][j] = s0 + j < e.M ? e.R[(size_t)(s0 + j) * e.ldr + col] : 0.f;
    }
  }
  if (MODE == TC_BRANCH_BWD && warp < 8) {
#pragma unroll
    for (int i = 0; i < KB; ++i)
#pragma unroll
      for (int j = 0; j < NC; ++j)
        pre[MODE == TC_BRANCH_BWD ? i : 0][j] =
            cok && s0 + j < e.M ? e.Aux[(size_t)(s0 + j) * e.ldaux + i * e.H + col] : 0.f;
  }
  pdl_wait();
  pdl_launch();

  if (warp == 8) {
    int s = 0;
    uint32_t ph = 1;
    for (int kb = 0; kb < nk; ++kb) {
      if (kb >= nst && !warp_wait(&empty[s], ph, abort_flag)) break;
      if (elect_one()) {
        if (kb >= nst) load_w(kb, s);
        tma_load_2d(sX + s * X_BYTES, &tx, kb * 64, m0, &full[s]);
      }
      __syncwarp();
      if (++s == nst) {
        s = 0;
        ph ^= 1u;
      }
    }
  } else if (warp == 9) {
    constexpr uint32_t idesc = idesc_bf16(NS);
    const uint32_t ad = desc_lo(sW), bd = desc_lo(sX);
    int s = 0;
    uint32_t ph = 0;
    for (int kb = 0; kb < nk; ++kb) {
      if (!warp_wait(&full[s], ph, abort_flag)) break;
      tc_fence_after();
      if (elect_one()) {
        mma_stage<false>(tmem, ad + s * (W_BYTES >> 4), bd + s * (X_BYTES >> 4), idesc, kb == 0);
        if (kb + nst < nk) mma_commit(&empty[s]);  // (else nothing waits for the stage)
      }
      __syncwarp();
      if (++s == nst) {
        s = 0;
        ph ^= 1u;
      }
    }
    __syncwarp();
    if (elect_one()) mma_commit(done);
  }
  __syncwarp();

  float gg[MODE == TC_BRANCH_BWD ? NC : 1];
  if (MODE == TC_BRANCH_BWD && warp < 8) {
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      float xf = 1.f;
#pragma unroll
      for (int i = 0; i < KB; ++i) xf *= pre[MODE == TC_BRANCH_BWD ? i : 0][j];
      gg[MODE == TC_BRANCH_BWD ? j : 0] = gelu_grad_f(xf);
    }
  }
  // The TMEM loads are warp-collective, so the wait result is made CTA-uniform first.
  const bool ok = __syncthreads_and(mbar_wait(done, 0, abort_flag) ? 1 : 0) != 0;
  tc_fence_after();
  if (ok && warp < 8) {
    float v[NC];
    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * NC);
#pragma unroll
    for (int c = 0; c < NC; c += 16) {
      float t[16];
      tmem_ld16(taddr + (uint32_t)c, t);
#pragma unroll
      for (int j = 0; j < 16; ++j) v[c + j] = t[j];
    }
    if (MODE == TC_PLAIN) {
      if (cok) {
        if (e.bias) {
#pragma unroll
          for (int j = 0; j < NC; ++j) v[j] += bias;
        }
        if (e.R) {
#pragma unroll
          for (int j = 0; j < NC; ++j) v[j] += pre[0][j];
        }
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          if (s0 + j >= e.M) break;
          if (e.C) e.C[(size_t)(s0 + j) * e.ldc + col] = v[j];
          if (e.Cb) e.Cb[(size_t)(s0 + j) * e.ldcb + col] = __float2bfloat16_rn(v[j]);
        }
        if (e.CbT) {
#pragma unroll
          for (int j = 0; j < NC; j += 8) put_run8(e, col, s0 + j, v + j);
        }
      }
    } else if (MODE == TC_BRANCH) {
      // X_i -> C (kept for the adjoint) and to shared memory, where a unit's branches meet
      static_assert((size_t)SECTIONS * NS * SR * 4 <= 2 * (W_BYTES + X_BYTES), "the exchange fits two stages");
      float* xs = reinterpret_cast<float*>(sW);  // [section][stream][unit]; the stages are idle
      if (sec < SECTIONS) {
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          if (cok) v[j] += bias;
          if (KB > 1) xs[((size_t)sec * NS + (warp >> 2) * NC + j) * SR + u] = v[j];
          if (cok && s0 + j < e.M) e.C[(size_t)(s0 + j) * e.ldc + sec * e.H + col] = v[j];
        }
      }
      // thread -> (unit, RUN consecutive streams)
      constexpr int RUN = NS * SR / kEpiThreads;
      const int uu = KB > 1 ? (int)threadIdx.x % SR : u;
      const int so = KB > 1 ? (int)threadIdx.x / SR * RUN : (warp >> 2) * NC;
      float g[RUN];
      if (KB > 1) {
        epi_sync8();
#pragma unroll
        for (int j = 0; j < RUN; ++j) {
          float f = 1.f;
#pragma unroll
          for (int i = 0; i < SECTIONS; ++i) f *= xs[((size_t)i * NS + so + j) * SR + uu];
          g[j] = gelu_f(f);
        }
      } else {
#pragma unroll
        for (int j = 0; j < RUN; ++j) g[j] = gelu_f(v[j]);
      }
      const int h = n0 + uu, sg = m0 + so;
      if (h < e.H) {
#pragma unroll
        for (int j = 0; j < RUN; ++j)
          if (sg + j < e.M) e.Cb[(size_t)(sg + j) * e.ldcb + h] = __float2bfloat16_rn(g[j]);
        if constexpr (RUN >= 8) {
#pragma unroll
          for (int j = 0; j < RUN; j += 8) put_run8(e, h, sg + j, g + j);
        } else {
          static_assert(RUN == 4, "a thread's run");
          if (sg + 4 <= e.ldct) {
            __align__(8) __nv_bfloat162 q[2] = {__floats2bfloat162_rn(g[0], g[1]), __floats2bfloat162_rn(g[2], g[3])};
            *reinterpret_cast<uint2*>(e.CbT + (size_t)h * e.ldct + sg) = *reinterpret_cast<const uint2*>(q);
          }
        }
      }
    } else {
      if (cok) {
#pragma unroll
        for (int j = 0; j < NC; ++j) v[j] *= gg[MODE == TC_BRANCH_BWD ? j : 0];
#pragma unroll
        for (int i = 0; i < KB; ++i) {
          float dd[NC];
#pragma unroll
          for (int j = 0; j < NC; ++j) {
            float prod = 1.f;
#pragma unroll
            for (int l = 0; l < KB; ++l)
              if (l != i) prod *= pre[MODE == TC_BRANCH_BWD ? l : 0][j];
            dd[j] = v[j] * prod;
          }
          const int c = i * e.H + col;
#pragma unroll
          for (int j = 0; j < NC; ++j) {
            if (s0 + j >= e.M) break;
            e.C[(size_t)(s0 + j) * e.ldc + c] = dd[j];
            e.Cb[(size_t)(s0 + j) * e.ldcb + c] = __float2bfloat16_rn(dd[j]);
          }
#pragma unroll
          for (int j = 0; j < NC; j += 8) put_run8(e, c, s0 + j, dd + j);
        }
      }
    }
  }
  if (!ok && threadIdx.x == 0 && e.err) atomicOr(e.err, kErrTcTimeout);
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) {
    // Let any TMA copies still in flight land before the CTA exits.
    for (int s = 0; s < nst && s < nk; ++s) {
      for (uint32_t it = 0; it < (1u << 20); ++it)
        if (mbar_try_wait(&full[s], 0) || mbar_try_wait(&full[s], 1)) break;
    }
  }
  if (warp == 9) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)tmem_cols<NS>()));
  }
}

template <int NS, int MODE, int KB>
cudaError_t launch_s(const TcGemm& g, cudaStream_t st) {
  auto k = gemm_tcs_kernel<NS, MODE, KB>;
  static OncePerDevice once;
  const cudaError_t attr_err = once_on_device(once, [&] {
    const cudaError_t r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)smem_bytes_s<NS>(kStagesS));
    return r != cudaSuccess
               ? r
               : cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  });
  if (attr_err != cudaSuccess) return attr_err;
  TcEpi e{};
  e.M = g.M;
  e.N = g.N;
  e.K = g.K;
  e.H = g.H;
  e.k = g.k;
  e.C = g.C;
  e.ldc = g.ldc;
  e.Cb = g.Cb;
  e.ldcb = g.ldcb;
  e.CbT = g.CbT;
  e.ldct = g.ldct;
  e.bias = g.bias;
  e.R = g.R;
  e.ldr = g.ldr;
  e.Aux = g.Aux;
  e.ldaux = g.ldaux;
  e.err = g.err;
  const int width = MODE == TC_PLAIN ? g.N : g.H;
  constexpr int SR = section_rows<MODE, KB>();
  const dim3 grid((width + SR - 1) / SR, (g.M + NS - 1) / NS);
  return launch_k(k, grid, dim3(kThreadsS), smem_bytes_s<NS>(stages_s((g.K + 63) / 64)), st, g.ta, g.tb, e);
}

template <int NS>
cudaError_t launch_ns(const TcGemm& g, cudaStream_t st) {
  switch (g.mode * 10 + (g.mode == TC_PLAIN ? 0 : g.k)) {
    case TC_PLAIN * 10: return launch_s<NS, TC_PLAIN, 1>(g, st);
    case TC_BRANCH * 10 + 1: return launch_s<NS, TC_BRANCH, 1>(g, st);
    case TC_BRANCH * 10 + 2: return launch_s<NS, TC_BRANCH, 2>(g, st);
    case TC_BRANCH * 10 + 3: return launch_s<NS, TC_BRANCH, 3>(g, st);
    case TC_BRANCH_BWD * 10 + 1: return launch_s<NS, TC_BRANCH_BWD, 1>(g, st);
    case TC_BRANCH_BWD * 10 + 2: return launch_s<NS, TC_BRANCH_BWD, 2>(g, st);
    case TC_BRANCH_BWD * 10 + 3: return launch_s<NS, TC_BRANCH_BWD, 3>(g, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

int tcs_section_rows(int mode, int k) {
  if (mode != TC_BRANCH) return 128;
  return k == 1 ? 128 : (k == 2 ? 64 : 32);
}

int tcs_streams(int mode, int k, int M, int N, int H) {
  const int sr = tcs_section_rows(mode, k), width = mode == TC_PLAIN ? N : H;
  for (int ns : {32, 64})
    if ((long long)((width + sr - 1) / sr) * ((M + ns - 1) / ns) <= 152) return ns;
  return 0;
}

cudaError_t launch_gemm_tcs(const TcGemm& g, cudaStream_t st) {
  if (g.fp8 || g.mt || g.gk || g.splitk > 1 || g.k < 1 || g.k > 3 || (g.CbT && (g.ldct & 7)) ||
      g.box_b != tcs_section_rows(g.mode, g.k))
    return cudaErrorInvalidValue;
  switch (g.ns) {  // the rows of tb's box
    case 32: return launch_ns<32>(g, st);
    case 64: return launch_ns<64>(g, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace edpc
