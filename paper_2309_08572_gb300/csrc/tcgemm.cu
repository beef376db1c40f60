// Tensor-core GEMM for sm_103a: tcgen05.mma with TMEM accumulators, operands staged in
// shared memory by TMA (cp.async.bulk.tensor) through an mbarrier pipeline.
//
// Core product (real):  D[b][i][j] = sum_k A[b][i][k] * B[b][j][k]
// with A (M x K) and B (N x K) both K-major (K contiguous), elements TF32 (stored as FP32)
// or BF16, accumulated in FP32 in tensor memory.  One CTA computes a 128 x BN tile:
//   warp 0 lane 0   issues the TMA loads of A and B k-blocks into a STAGES-deep ring,
//   warp 1 lane 0   issues the tcgen05.mma instructions (4 per 128-byte k-block) and
//                   commits them to the ring's "empty" barriers and, at the end, to the
//                   accumulator barrier,
//   all 4 warps     read the accumulator back with tcgen05.ld (warp w owns TMEM lanes
//                   32w..32w+31, i.e. tile rows 32w..32w+31) and write the output.
// Every wait on an mbarrier is bounded (kWaitNs); a wait that gives up sets the caller's
// error flag and the kernel winds down without touching the output.
//
// Complex products ride on the real core (the paper's contractions, Sec. III.A, are
// complex):  with op(A) = X (m x k) and op(B) = Y (k x n) complex,
//   Ar[i][2p] = Re X_ip, Ar[i][2p+1] = Im X_ip                                   (m x 2k)
//   Br[2q][2p] = Re Y_pq, Br[2q][2p+1] = -Im Y_pq,
//   Br[2q+1][2p] = Im Y_pq, Br[2q+1][2p+1] = Re Y_pq                              (2n x 2k)
// gives Ar Br^T = the interleaved (re, im) m x n result, i.e. one real GEMM of the same
// 8mnk flops as a complex one, written straight into complex64 storage.  Split precision
// (TF32x3 / BF16x3): x = hi(x) + lo(x) with hi, lo in the MMA type; the packed operands
// carry three K-segments, A as [hi | hi | lo] and B as [hi | lo | hi], so one GEMM over
// 3 x 2k sums hi*hi + hi*lo + lo*hi (the lo*lo term is below FP32 rounding for TF32).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "exactplan.h"
#include "internal.h"
#include "tcgemm.h"

namespace mpdo {
std::atomic<long long> g_tc_launches{0};
namespace tc {

constexpr int BM = 128;
constexpr int kThreads = 128;
constexpr unsigned long long kWaitNs = 2000000000ull;   // 2 s per wait, then give up

__device__ __forceinline__ uint32_t su32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long gtime() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(su32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for the phase with the given parity; false when it gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_test(bar, parity)) return true;
  const unsigned long long t0 = gtime();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (mbar_test(bar, parity)) return true;
    if (gtime() - t0 > kWaitNs) return false;
  }
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%3, %4, %5}], [%2];" ::"r"(su32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(su32(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Shared-memory matrix descriptor of a K-major tile written by TMA with 128-byte swizzle:
// rows of 128 bytes, 8-row groups 1024 bytes apart (stride byte offset), version 1
// (tcgen05), layout SWIZZLE_128B.  The leading byte offset is not used by this layout.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// Instruction descriptor, dense kind::tf32 / kind::f16: D format F32 (bits 4-5 = 1), A and
// B formats (bits 7-9, 10-12: TF32 = 2, BF16 = 1), both K-major, N >> 3 at bit 17,
// M >> 4 at bit 24.
template <int ELT>
__host__ __device__ constexpr uint32_t idesc(int n) {
  return (1u << 4) | ((ELT == 4 ? 2u : 1u) << 7) | ((ELT == 4 ? 2u : 1u) << 10) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}
template <int ELT>
__device__ __forceinline__ void umma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t id,
                                     uint32_t accum) {
  if constexpr (ELT == 4) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(id), "r"(accum));
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(id), "r"(accum));
  }
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          su32(bar))
      : "memory");
}
// 32 consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

struct Epi {
  float* d;       // output, real view: row i of batch b at d + b*sd + i*ldd (floats)
  long ldd, sd;
  double* d64;    // FP64 accumulation target (mode 1), same strides
  float ar, ai;   // complex alpha (pairs of columns are (re, im)); mode 0
  float br, bi;   // complex beta; use_beta = 0 skips reading d
  int use_beta;
  double scale;   // mode 1: d64 += scale * acc
  int mode;       // 0: FP32 (complex alpha/beta), 1: FP64 accumulate
};

// One output tile of the real product: A rows from m0, B rows from n0, batch entry bz.  epi(row,
// column, v) takes each thread's 32 columns of its row; all lanes call it, also beyond the matrix.
// DEP: the launch may begin before its predecessor in the stream has ended, and waits for it here.
template <int ELT, int BN, int STAGES, bool DEP, typename F>
__device__ __forceinline__ void tc_tile(const CUtensorMap* ma, const CUtensorMap* mb, int m0, int n0,
                                        int bz, int K, int* err, F&& epi) {
  constexpr int BK = 128 / ELT;                      // elements per 128-byte k-block row
  constexpr uint32_t A_BYTES = BM * 128, B_BYTES = BN * 128;
  constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  constexpr uint32_t TMEM_COLS = BN <= 32 ? 32 : BN <= 64 ? 64 : BN <= 128 ? 128 : 256;
  extern __shared__ uint8_t smem_raw[];
  // tiles on a 1024-byte boundary (the 128-byte swizzle pattern repeats every 8 rows)
  uint8_t* smem = smem_raw + ((1024 - (su32(smem_raw) & 1023)) & 1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* accb = empty + STAGES;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(accb + 1);
  int* abort_flag = reinterpret_cast<int*>(tslot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk = (K + BK - 1) / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accb, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tslot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  if constexpr (DEP) asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp == 0) {
    if (lane == 0) {
      // producer: k-block kb goes to stage kb % STAGES once the MMAs of kb - STAGES are done
      for (int kb = 0; kb < nk; ++kb) {
        const int s = kb % STAGES;
        if (kb >= STAGES && !mbar_wait(&empty[s], ((kb / STAGES) - 1) & 1)) {
          atomicExch(abort_flag, 1);
          atomicExch(err, 1);
          break;
        }
        if (*(volatile int*)abort_flag) break;
        uint8_t* sa = smem + s * STAGE_BYTES;
        mbar_expect_tx(&full[s], STAGE_BYTES);
        tma_load_3d(sa, ma, &full[s], kb * BK, m0, bz);
        tma_load_3d(sa + A_BYTES, mb, &full[s], kb * BK, n0, bz);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t id = idesc<ELT>(BN);
      bool ok = true;
      for (int kb = 0; kb < nk; ++kb) {
        const int s = kb % STAGES;
        if (!mbar_wait(&full[s], (kb / STAGES) & 1)) {
          atomicExch(abort_flag, 1);
          atomicExch(err, 2);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = su32(smem + s * STAGE_BYTES);
        const uint64_t ad = sdesc(sa), bd = sdesc(sa + A_BYTES);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)   // 32 bytes of K per instruction
          umma<ELT>(tmem, ad + 2 * kk, bd + 2 * kk, id, (kb | kk) != 0);
        umma_commit(&empty[s]);
      }
      // the accumulator barrier fires when every MMA issued above has completed
      umma_commit(accb);
      (void)ok;
    }
    __syncwarp();
  }

  // epilogue: TMEM -> registers -> global
  bool ready = true;
  if (lane == 0) ready = mbar_wait(accb, 0);
  ready = __shfl_sync(0xffffffffu, ready ? 1 : 0, 0) != 0;
  if (!ready) {
    if (lane == 0) atomicExch(err, 3);
  } else if (!*(volatile int*)abort_flag) {
    tc_fence_after();
    const int row = m0 + warp * 32 + lane;
    const uint32_t tw = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int c = 0; c < BN; c += 32) {
      float v[32];
      tmem_ld32(tw + c, v);
      epi(row, n0 + c, v);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS)
                 : "memory");
  }
}

template <int ELT, int BN, int STAGES>
__global__ void __launch_bounds__(kThreads, 1)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb,
                   int M, int N, int K, Epi ep, int* err) {
  const int bz = blockIdx.z;
  auto epi = [&](int row, int col0, const float* v) {
    if (row < M) {
      if (ep.mode == 0) {
        float* dp = ep.d + (long)bz * ep.sd + (long)row * ep.ldd + col0;
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          if (col0 + j >= N) break;
          const float xr = v[j], xi = v[j + 1];
          float yr = ep.ar * xr - ep.ai * xi, yi = ep.ar * xi + ep.ai * xr;
          if (ep.use_beta) {
            const float cr = dp[j], ci = (col0 + j + 1 < N) ? dp[j + 1] : 0.f;
            yr += ep.br * cr - ep.bi * ci;
            yi += ep.br * ci + ep.bi * cr;
          }
          dp[j] = yr;
          if (col0 + j + 1 < N) dp[j + 1] = yi;
        }
      } else {
        double* dp = ep.d64 + (long)bz * ep.sd + (long)row * ep.ldd + col0;
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (col0 + j < N) dp[j] += ep.scale * (double)v[j];
      }
    }
  };
  tc_tile<ELT, BN, STAGES, false>(&ma, &mb, blockIdx.y * BM, blockIdx.x * BN, bz, K, err, epi);
}

// ------------------------------------------------------------------ surrogate's products
// Products of the fully connected network in BF16 with the elementwise work around them in the
// epilogue: bias and tanh going forward, the loss, tanh' going back, the operands of the products
// that follow (BF16, K-major in both orientations) and the column sums of the biases' gradients.
// The network is small (256 wide, a batch of 512: 2 us of products), so a pass is bound by its
// launches, each with its drain and fill: packing, bias, tanh and sums of their own made 52 of
// them a training step, now it takes 10.  A launch runs a group of products (all weight gradients
// at once, with the sums of the parts in blocks behind the tiles), and its set-up (barriers, TMEM,
// descriptors) overlaps the end of the launch before it (programmatic dependent launch).
// A training step at batch 512 (24-256-256-256-2): 363 -> 99 us (136 without the overlap and with
// tiles of 64 columns at least), an input gradient at batch 64: 193 -> 54 us (82).
__device__ __forceinline__ void mlp_epilogue(const MlpEpi& e, int M, int N, int row, int col0,
                                             float* v, int tiles_n) {
  if (col0 >= N) return;
  const int lane = threadIdx.x & 31;
  const bool in = row < M;
  if (e.bias) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (col0 + j < N) v[j] += e.bias[col0 + j];
  }
  if (e.act) {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = tanhf(v[j]);
  }
  if (e.t) {
    double s = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (in && col0 + j < N) {
        const float d = v[j] - e.t[(long)row * N + col0 + j];
        v[j] = 2.f * d * e.scale;
        s += (double)d * d;
      }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) e.loss[(long)(row / 32) * tiles_n + col0 / 32] = s;
  }
  if (e.a && in) {
    const float* ap = e.a + (long)row * e.lda + col0;
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (col0 + j < N) {
        const float x = ap[j];
        v[j] *= (1.f - x * x);
      }
  }
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (!in || col0 + j >= N) v[j] = 0.f;
  if (in && e.d) {
    float* dp = e.d + (long)row * e.ldd + col0;
    if (col0 + 32 <= N && e.ldd % 4 == 0 && (reinterpret_cast<uintptr_t>(e.d) & 15) == 0) {
#pragma unroll
      for (int j = 0; j < 32; j += 4)
        *reinterpret_cast<float4*>(dp + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (col0 + j < N) dp[j] = v[j];
    }
  }
  if (in && e.row) {   // rows of ldr % 8 == 0, zeros behind the last column
    __nv_bfloat162* rp = reinterpret_cast<__nv_bfloat162*>(e.row + (long)row * e.ldr + col0);
#pragma unroll
    for (int j = 0; j < 32; j += 8)
      if (col0 + j < e.ldr) {
        __nv_bfloat162 q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = __floats2bfloat162_rn(v[j + 2 * i], v[j + 2 * i + 1]);
        *reinterpret_cast<uint4*>(rp + j / 2) = *reinterpret_cast<const uint4*>(q);
      }
  }
  if (in && e.col) {   // neighbouring lanes, neighbouring rows
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (col0 + j < N) e.col[(long)(col0 + j) * e.ldc + row] = __float2bfloat16_rn(v[j]);
  }
  if (e.csum) {
    // sums over the warp's rows: each exchange hands half of the remaining columns over, and lane
    // l ends with column l
    float x[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) x[j] = v[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int j = 0; j < o; ++j) {
        const float give = up ? x[j] : x[j + o], keep = up ? x[j + o] : x[j];
        x[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
    if (col0 + lane < N) e.csum[(long)(row / 32) * N + col0 + lane] = x[0];
  }
}

template <int BN, int STAGES, int CAP>
__global__ void __launch_bounds__(kThreads, 1)
    mlp_gemm_kernel(const __grid_constant__ MlpGroup<CAP> g, int* err) {
  const int b = blockIdx.x;
  // the next launch may be set up while this one runs; its own wait stands before its first read
  // or write of memory
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (b >= g.tiles) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // sums of the parts: 128 bias gradients a block, and the loss in the last
    if (b == (int)gridDim.x - 1) {
      __shared__ double red[kThreads];
      double s = 0;
      for (long i = threadIdx.x; i < g.loss_n; i += kThreads) s += g.loss[i];
      red[threadIdx.x] = s;
      __syncthreads();
      for (int k = kThreads / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
      }
      if (threadIdx.x == 0) *g.loss_sum = red[0];
      return;
    }
    int q = b - g.tiles, p = 0;
    while (p < g.count - 1 && q >= (g.p[p].N + kThreads - 1) / kThreads)
      q -= (g.p[p++].N + kThreads - 1) / kThreads;
    const int c = q * kThreads + threadIdx.x, N = g.p[p].N;
    if (c < N) {
      float s = 0.f;
      for (int i = 0; i < g.parts; ++i) s += g.p[p].sum_in[(long)i * N + c];
      g.p[p].sum_out[c] = s;
    }
    return;
  }
  int p = 0;
  while (p + 1 < g.count && b >= g.p[p + 1].tile0) ++p;
  const MlpProd& q = g.p[p];
  const int t = b - q.tile0, tn = (q.N + BN - 1) / BN, M = q.M, N = q.N;
  auto epi = [&](int row, int col0, float* v) {
    mlp_epilogue(q.e, M, N, row, col0, v, (N + 31) / 32);
  };
  tc_tile<2, BN, STAGES, true>(&q.a, &q.b, t / tn * BM, t % tn * BN, 0, q.K, err, epi);
}

// ------------------------------------------------------------------ operand packing
__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}
template <typename TO>
__device__ __forceinline__ void split3(float x, TO& hi, TO& lo);
template <>
__device__ __forceinline__ void split3<float>(float x, float& hi, float& lo) {
  hi = tf32_rna(x);
  lo = tf32_rna(x - hi);
}
template <>
__device__ __forceinline__ void split3<__nv_bfloat16>(float x, __nv_bfloat16& hi,
                                                      __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}
template <typename TO>
__device__ __forceinline__ TO to_elt(float x);
template <>
__device__ __forceinline__ float to_elt<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 to_elt<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}

// X[r][c] = src[b*sb + r*s_r + c*s_c] (conjugated when conj), r < rows, c < kc.
// side 0 (A operand): out[b][r][t*2kc + 2c + {0,1}] = parts of (Re, Im)
// side 1 (B operand): out[b][2r][t*2kc + 2c + {0,1}] = parts of (Re, -Im),
//                     out[b][2r+1][...]             = parts of (Im, Re)
// parts t: nparts = 1 -> the value; nparts = 3 -> A [hi, hi, lo], B [hi, lo, hi].
constexpr int PT = 32;
template <typename TIN, typename TO>
__global__ void __launch_bounds__(PT * 8)
    pack_kernel(int rows, int kc, const TIN* __restrict__ src, long s_r, long s_c, long sb,
                int conj, int side, int nparts, TO* __restrict__ out, long ldo, long so) {
  __shared__ float2 tile[PT][PT + 1];   // [r][c]
  const int r0 = blockIdx.y * PT, c0 = blockIdx.x * PT, b = blockIdx.z;
  const int tx = threadIdx.x, ty = threadIdx.y;
  src += (long)b * sb;
  const bool c_fast = (s_c == 1);
  for (int q = ty; q < PT; q += 8) {
    // coalesced along whichever index is contiguous in the source
    const int r = c_fast ? r0 + q : r0 + tx;
    const int c = c_fast ? c0 + tx : c0 + q;
    float2 v = make_float2(0.f, 0.f);
    if (r < rows && c < kc) {
      const TIN t = src[(long)r * s_r + (long)c * s_c];
      v = make_float2((float)t.x, conj ? -(float)t.y : (float)t.y);
    }
    if (c_fast) tile[q][tx] = v; else tile[tx][q] = v;
  }
  __syncthreads();
  const long kseg = 2L * kc;
  for (int q = ty; q < PT; q += 8) {
    const int r = r0 + q, c = c0 + tx;
    if (r >= rows || c >= kc) continue;
    const float2 v = tile[q][tx];
    if (side == 0) {
      TO* o = out + (long)b * so + (long)r * ldo + 2L * c;
      if (nparts == 1) {
        o[0] = to_elt<TO>(v.x);
        o[1] = to_elt<TO>(v.y);
      } else {
        TO hr, lr, hi, li;
        split3<TO>(v.x, hr, lr);
        split3<TO>(v.y, hi, li);
        o[0] = hr; o[1] = hi;
        o[kseg] = hr; o[kseg + 1] = hi;
        o[2 * kseg] = lr; o[2 * kseg + 1] = li;
      }
    } else {
      TO* o0 = out + (long)b * so + (2L * r) * ldo + 2L * c;
      TO* o1 = o0 + ldo;
      if (nparts == 1) {
        o0[0] = to_elt<TO>(v.x); o0[1] = to_elt<TO>(-v.y);
        o1[0] = to_elt<TO>(v.y); o1[1] = to_elt<TO>(v.x);
      } else {
        TO hr, lr, hi, li, hm, lm;
        split3<TO>(v.x, hr, lr);
        split3<TO>(v.y, hi, li);
        split3<TO>(-v.y, hm, lm);
        o0[0] = hr; o0[1] = hm; o1[0] = hi; o1[1] = hr;
        o0[kseg] = lr; o0[kseg + 1] = lm; o1[kseg] = li; o1[kseg + 1] = lr;
        o0[2 * kseg] = hr; o0[2 * kseg + 1] = hm; o1[2 * kseg] = hi; o1[2 * kseg + 1] = hr;
      }
    }
  }
}

// ------------------------------------------------------------------ exact products
// FP64-accurate product of FP32 operands on the BF16 tensor cores, by error-free slicing
// (the splitting scheme of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59, 2012).  Every row r of the A operand (and of the
// B operand) is scaled by 2^-e_r, e_r the exponent of its largest |Re|, |Im|, and written as
// six slices of integers in [-128, 128] (exact in BF16):
//   x 2^-e_r = 2^-7 (q_1 + 2^-8 q_2 + ... + 2^-40 q_6) + O(2^-48).
// The product of slice t of A and slice u of B is a sum of integer products of at most
// 2^14 each; 1024 of them stay below 2^24 and are therefore exact in the FP32 accumulator.  The
// accumulators are taken out in time and added with the weight 2^-(14 + 8(t+u)) (t, u from 0),
// and the sum is scaled by 2^(e_r + e_q).  The slice pairs with t + u <= 5 are computed (21 of
// 36): a dropped pair contributes terms below 2^-48 of the two rows' largest entries.  The result carries the FP32 inputs' product to
// ~2^-48 of the rows' largest entries, enough for the eigenvalues of a Gram matrix of FP32
// data down to ~1e-14 of the largest (the floor of FP64 sums of the same products).
//
// The kernel's tile is 128 rows by 64 real columns.  A stage holds 32 K terms of all six slices
// of both operands (72 KB, three stages), so the 21 pairs run on operands that were loaded once:
// 27 bytes per clock and SM from L2, where loading every pair's operands took 128.  The pairs
// (t, u) of one weight t + u add into one accumulator, six of 64 TMEM columns; a sum stays
// below 2^24 for 1024 / (t + u + 1) terms.  Slice t of A meets the slices 0 .. 5 - t of B in
// products of up to 256 columns -- those slices, and the accumulators of the weights t .. 5, lie
// one behind the other -- because a product of 64 columns took 88 clocks, more than twice its share
// of the tensor pipe's rate (3600 -> 2700 clocks a stage with the wide ones).  The sums' limit
// means that every XDRAIN = 5 stages (at most 6 x 160 terms) eight warps take the accumulators
// out, weight after weight, while the products of the other weights run.  They add them as
// integers -- weights 0..2 and 3..5 shifted into two 64-bit sums, exact -- since the FP64 pipe, at
// 2 operations per clock and SM, bound an FP64 drain to an eighth of the MMA rate.
//
// The stages of all tiles, one tile after another, are dealt to at most one CTA per SM in equal
// ranges (a launch of a tile and K slice per CTA left the last wave nearly empty and paid the fill
// of the ring, the TMEM allocation and the output for every slice, 17 us each); the ring runs on
// from tile to tile.  A range's first and last tile may be another CTA's as well: their integer
// sums (exact, so in any order) are added by exact_finish_kernel.  Gram matrices compute the tiles
// that reach the upper half, from one packed operand: the rows of A are the even rows of the packed
// B.  Bound by the tensor pipe and the accumulators' turn-around.  768 x 768 x 4096 Gram, this
// kernel: 1150 us with every pair's operands loaded anew and an FP64 drain, 367 us with slices of K
// and 64-column products, 313 us in equal ranges, 201 us with wide products.
constexpr int XS = kExactSlices;
constexpr int XBN = kExactCols;   // output tile width (real columns)
constexpr int XKB = kExactK;      // K terms of a stage
static_assert(BM == kExactRows && kSms == kExactSms, "the plan's tile and device");
constexpr int XSTAGES = 3;
constexpr int XDRAIN = 5;      // stages between drains
constexpr int XTHREADS = 320;  // warp 0 TMA, warp 1 MMA, warps 2-9 drain
constexpr int XA_SLICE = BM * XKB * 2, XB_SLICE = XBN * XKB * 2;
constexpr int XSTAGE_BYTES = XS * (XA_SLICE + XB_SLICE);
constexpr long XPART = kExactPart;   // a CTA's part of a tile: [column of 32][half, row]
static_assert(kExactPartBytes == XPART * (long)sizeof(longlong2), "the plan's parts");
constexpr int kNonFinite = 0x7fffffff;   // exponent of a row with a non-finite entry
constexpr int kZeroRow = -1000000;       // and of a zero row (any smaller value)

// As sdesc, for rows of 64 bytes with 64-byte swizzle (8-row groups 512 bytes apart).
__device__ __forceinline__ uint64_t sdesc64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

// 2^(e_r + e_q) (2^-30 hi + 2^-54 lo), NaN when either row had a non-finite entry.  The power of
// two goes straight into the exponent field where the result stays normal: three FP64
// operations an element, where ldexp's multiplications took a third of a short product's time.
__device__ __forceinline__ double exact_value(long long hi, long long lo, int er, int eq) {
  if (er == kNonFinite || eq == kNonFinite) return NAN;
  if (er <= kZeroRow || eq <= kZeroRow || (hi | lo) == 0) return 0.0;
  const double v = fma((double)lo, 0x1p-24, (double)hi);
  const int s = er + eq - 30, h = __double2hiint(v), ex = ((h >> 20) & 2047) + s;
  if (v == 0.0 || ex <= 0 || ex >= 2047) return ldexp(v, s);
  return __hiloint2double(h + (s << 20), __double2loint(v));
}

// Output of one complex element (i, q), with its mirror image for a Gram matrix.
__device__ __forceinline__ void exact_store(double2* C, long ldc, int i, int q, double re, double im,
                                            int gram, int accumulate) {
  if (gram && q < i) return;
  if (gram && q == i) im = 0.0;
  double2* p = C + (long)i * ldc + q;
  double2 v = make_double2(re, im);
  if (accumulate) v = cadd(v, *p);
  *p = v;
  if (gram && q > i) C[(long)q * ldc + i] = cconj(v);
}

// tile index -> (row tile, column tile); a Gram's row tile mt starts at column tile mt * 128 / 32
__device__ __forceinline__ void exact_tile(int tile, int nt, int gram, int& mt, int& ct) {
  mt = 0;
  if (!gram) {
    mt = tile / nt;
    ct = tile - mt * nt;
    return;
  }
  constexpr int step = BM / (XBN / 2);
  while (tile >= nt - mt * step) {
    tile -= nt - mt * step;
    ++mt;
  }
  ct = mt * step + tile;
}

__global__ void __launch_bounds__(XTHREADS, 1)
    tc_exact_kernel(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb,
                    int M, int N, int ldk, int nst, int tiles, long per, long total, int gram,
                    const int* __restrict__ ea,
                    const int* __restrict__ eb, double2* C, long ldc, long sc, int accumulate,
                    longlong2* part, int* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024 - (su32(smem_raw) & 1023)) & 1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + XSTAGES * XSTAGE_BYTES);
  uint64_t* empty = full + XSTAGES;
  uint64_t* gfull = empty + XSTAGES;   // [XS] accumulator of a weight ready for the drain
  uint64_t* gempty = gfull + XS;       // [XS] drained
  uint32_t* tslot = reinterpret_cast<uint32_t*>(gempty + XS);
  int* abort_flag = reinterpret_cast<int*>(tslot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nt = (N + XBN - 1) / XBN;
  // this CTA's stages: `left` of them from stage s0 of a tile (over the batch)
  int s0 = (int)(blockIdx.x * per % nst), tile = (int)(blockIdx.x * per / nst);
  int left = (int)min(per, total - blockIdx.x * per), len, m0, n0, bz;
  auto locate = [&]() {
    len = min(nst - s0, left);
    bz = tile / tiles;
    int mt, ct;
    exact_tile(tile - bz * tiles, nt, gram, mt, ct);
    m0 = mt * BM;
    n0 = ct * XBN;
  };
  auto next = [&]() {
    left -= len;
    s0 = 0;
    ++tile;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < XSTAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int g = 0; g < XS; ++g) {
      mbar_init(&gfull[g], 1);
      mbar_init(&gempty[g], 8);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tslot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (; left > 0 && ok; next()) {
        locate();
        for (int j = 0; j < len && ok; ++j, ++it) {
          const int s = it % XSTAGES;
          if (it >= XSTAGES && !mbar_wait(&empty[s], ((it / XSTAGES) - 1) & 1)) {
            atomicExch(abort_flag, 1);
            atomicExch(err, 11);
            ok = false;
          }
          if (*(volatile int*)abort_flag) ok = false;
          if (!ok) break;
          uint8_t* sa = smem + s * XSTAGE_BYTES;
          mbar_expect_tx(&full[s], XSTAGE_BYTES);
          const int c0 = (s0 + j) * XKB;
          for (int t = 0; t < XS; ++t) {
            tma_load_3d(sa + t * XA_SLICE, &ma, &full[s], t * ldk + c0, m0, bz);
            tma_load_3d(sa + XS * XA_SLICE + t * XB_SLICE, &mb, &full[s], t * ldk + c0, n0, bz);
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      bool ok = true;
      int it = 0, d = -1;   // stages and drain periods so far
      for (; left > 0 && ok; next()) {
        locate();
        for (int j = 0; j < len && ok; ++j, ++it) {
          const int s = it % XSTAGES;
          const bool first = j % XDRAIN == 0, last = j % XDRAIN == XDRAIN - 1 || j == len - 1;
          if (first) ++d;
          if (!mbar_wait(&full[s], (it / XSTAGES) & 1)) {
            atomicExch(abort_flag, 1);
            atomicExch(err, 12);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = su32(smem + s * XSTAGE_BYTES);
          // slice t of A against the slices 0 .. 5 - t of B, which lie one behind the other like the
          // accumulators of the weights t .. 5: products of up to 256 columns
#pragma unroll
          for (int t = 0; t < XS; ++t) {
#pragma unroll
            for (int u = 0; u < XS - t; u += 4) {
              constexpr int kMax = 4;
              const int nu = XS - t - u < kMax ? XS - t - u : kMax;
              if (first && t == 0 && d > 0) {
                // the drain of the period before must have emptied these accumulators
                for (int g = u; g < u + nu && ok; ++g) ok = mbar_wait(&gempty[g], (d - 1) & 1);
                if (!ok) {
                  atomicExch(abort_flag, 1);
                  atomicExch(err, 13);
                  break;
                }
                tc_fence_after();
              }
              const uint64_t ad = sdesc64(sa + t * XA_SLICE),
                             bd = sdesc64(sa + XS * XA_SLICE + u * XB_SLICE);
#pragma unroll
              for (int kk = 0; kk < 2; ++kk)
                umma<2>(tmem + (t + u) * XBN, ad + 2 * kk, bd + 2 * kk, idesc<2>(nu * XBN),
                        (first && t == 0 && kk == 0) ? 0u : 1u);
            }
            if (!ok) break;
            if (last) umma_commit(&gfull[t]);   // weight t has its last pair
          }
          if (ok) umma_commit(&empty[s]);
        }
      }
    }
    __syncwarp();
  } else {
    // drain warps: TMEM lanes 32 (warp % 4) .. +31 are tile rows, columns 32 hf .. +31
    const int q = warp & 3, hf = (warp - 2) >> 2;
    bool ok = true;
    int d = 0, first = 0;   // periods so far; 0: the range's first tile
    for (; left > 0 && ok; next(), first = 1) {
      locate();
      const int row = m0 + q * 32 + lane;
      long long hi[32], lo[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) hi[j] = lo[j] = 0;
      const int end = d + (len + XDRAIN - 1) / XDRAIN;
      for (; d < end && ok; ++d) {
#pragma unroll
        for (int g = 0; g < XS; ++g) {
          bool ready = true;
          if (lane == 0) ready = mbar_wait(&gfull[g], d & 1);
          ready = __shfl_sync(0xffffffffu, ready ? 1 : 0, 0) != 0;
          if (!ready || *(volatile int*)abort_flag) {
            if (lane == 0 && !ready) atomicExch(err, 14);
            ok = false;
            break;
          }
          tc_fence_after();
          float v[32];
          tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + g * XBN + hf * 32, v);
          tc_fence_before();
          __syncwarp();
          if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(&gempty[g])) : "memory");
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const long long x = (long long)__float2int_rn(v[j]) * (1 << (8 * (2 - g % 3)));
            if (g < 3) hi[j] += x; else lo[j] += x;
          }
        }
      }
      if (!ok) break;
      if (len < nst) {
        longlong2* pp = part + (long)(2 * blockIdx.x + first) * XPART +
                        (hf * 4 + q) * 32 + lane;
#pragma unroll
        for (int j = 0; j < 32; ++j) pp[j * 256] = make_longlong2(hi[j], lo[j]);
      } else if (row < M) {
        const int c0 = n0 + hf * 32, er = ea[(long)bz * M + row];
        double2* cp = C + (long)bz * sc;
#pragma unroll
        for (int j = 0; j < 32; j += 2)
          if (c0 + j < N) {
            const int qc = (c0 + j) >> 1, eq = eb[(long)bz * (N / 2) + qc];
            exact_store(cp, ldc, row, qc, exact_value(hi[j], lo[j], er, eq),
                        exact_value(hi[j + 1], lo[j + 1], er, eq), gram, accumulate);
          }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
  }
}

// The tiles that belong to more than one CTA's range: the sum of their integer parts and the
// output.  Eight columns of a tile a block, a thread to a row and half as in the drain.
__global__ void __launch_bounds__(256) exact_finish_kernel(int M, int N, int nst, int tiles, long per,
                                                           int gram, const longlong2* part,
                                                           const int* __restrict__ ea,
                                                           const int* __restrict__ eb, double2* C,
                                                           long ldc, long sc, int accumulate) {
  const long tile = blockIdx.x;
  const long c0 = tile * nst / per, c1 = ((tile + 1) * nst - 1) / per;
  if (c0 == c1) return;
  const int j0 = blockIdx.y * 8, bz = (int)(tile / tiles), nt = (N + XBN - 1) / XBN;
  int mt, ct;
  exact_tile((int)(tile - (long)bz * tiles), nt, gram, mt, ct);
  const int row = mt * BM + (threadIdx.x & 127), col = ct * XBN + (threadIdx.x >> 7) * 32 + j0;
  long long hi[8] = {}, lo[8] = {};
  for (long c = c0; c <= c1; ++c) {
    const longlong2* p = part + (2 * c + (c * per / nst == tile ? 0 : 1)) * XPART + j0 * 256 + threadIdx.x;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const longlong2 x = p[j * 256];
      hi[j] += x.x;
      lo[j] += x.y;
    }
  }
  if (row >= M) return;
  const int er = ea[(long)bz * M + row];
#pragma unroll
  for (int j = 0; j < 8; j += 2)
    if (col + j < N) {
      const int qc = (col + j) >> 1, eq = eb[(long)bz * (N / 2) + qc];
      exact_store(C + (long)bz * sc, ldc, row, qc, exact_value(hi[j], lo[j], er, eq),
                  exact_value(hi[j + 1], lo[j + 1], er, eq), gram, accumulate);
    }
}

// e[b][r] = exponent of the largest |Re|, |Im| of row r of X (X[r][c] = src[b*sb + r*s_r +
// c*s_c], c < kc): max = f 2^e with f in [0.5, 1); kNonFinite for a row with an infinity or a NaN.
// e is set to a value below kZeroRow before.  Reads are coalesced whichever index is
// contiguous: a warp per row (8 rows of a CTA), or the 32 rows of a CTA across the lanes; the
// columns are shared out over grid.y.
template <typename TIN>
__global__ void __launch_bounds__(256) row_exp_kernel(int rows, int kc, const TIN* __restrict__ src,
                                                     long s_r, long s_c, long sb, int cols, int* e) {
  using F = decltype(TIN().x);
  __shared__ F red[8][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool c_fast = s_c == 1;
  const int c0 = blockIdx.y * cols, c1 = min(kc, c0 + cols);
  const int r = c_fast ? blockIdx.x * 8 + warp : blockIdx.x * 32 + lane;
  F mx = 0, bad = 0;
  if (r < rows) {
    const TIN* x = src + (long)blockIdx.z * sb + (long)r * s_r;
    for (int c = c0 + (c_fast ? lane : warp); c < c1; c += c_fast ? 32 : 8) {
      const TIN v = x[(long)c * s_c];
      bad += (v.x - v.x) + (v.y - v.y);     // 0, or NaN for a non-finite entry
      const F a = fabs(v.x), b = fabs(v.y);
      mx = a > mx ? a : mx;
      mx = b > mx ? b : mx;
    }
  }
  if (!(bad == 0)) mx = INFINITY;
  if (c_fast) {
    for (int o = 16; o > 0; o >>= 1) {
      const F y = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = y > mx ? y : mx;
    }
    if (lane > 0) return;
  } else {
    red[warp][lane] = mx;
    __syncthreads();
    if (warp > 0) return;
    for (int k = 1; k < 8; ++k) mx = red[k][lane] > mx ? red[k][lane] : mx;
  }
  if (r < rows && mx > 0) {
    int ex = kNonFinite;
    if (!isinf(mx)) frexp(mx, &ex);
    atomicMax(&e[(long)blockIdx.z * rows + r], ex);
  }
}

// x 2^(47 - e) rounded to an integer, for |x| < 2^e: shifts of the significand.
__device__ __forceinline__ long long shift_round(long long m, int s) {
  return s >= 0 ? m << s : s < -62 ? 0 : (m + (1LL << (-s - 1))) >> -s;
}
__device__ __forceinline__ long long to_fixed(float x, int e) {
  const int b = __float_as_int(x), ex = (b >> 23) & 255;
  const long long q = shift_round((b & 0x7fffff) | (ex ? 0x800000 : 0), (ex ? ex : 1) - 150 + 47 - e);
  return b < 0 ? -q : q;
}
__device__ __forceinline__ long long to_fixed(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 2047);
  const long long q = shift_round((b & 0xfffffffffffffLL) | (ex ? 1LL << 52 : 0),
                                  (ex ? ex : 1) - 1075 + 47 - e);
  return b < 0 ? -q : q;
}
// The XS slices of x: q = sum_t 2^(8 (XS - 1 - t)) d[t], |d[t]| <= 128, so x = 2^-7 sum_t 2^-8t d[t]
// 2^e to 2^-48 2^e.  Halves go to the even neighbour: the digits of -x are those of x negated, and
// what the dropped pairs leave out has no preferred sign (digits in [-128, 127], of mean -1/2, made
// the error of a Gram of 500 rows 9 % larger).
__device__ __forceinline__ void slice_all(long long q, float* d) {
#pragma unroll
  for (int t = XS - 1; t > 0; --t) {
    const long long r = (q + 127 + ((q >> 8) & 1)) >> 8;
    d[t] = (float)(int)(q - r * 256);
    q = r;
  }
  d[0] = (float)(int)q;
}

// Sliced packing (layout as pack_kernel, with XS K-segments of ldk elements, one per slice;
// the segment tails up to ldk are zeros): row scale 2^-e[b][r] (A side) or the column scale of
// the complex column (B side, rows 2r and 2r+1).
template <typename TIN>
__global__ void __launch_bounds__(PT * 8)
    pack_exact_kernel(int rows, int kc, const TIN* __restrict__ src, long s_r, long s_c, long sb,
                      int conj, int side, const int* __restrict__ e, __nv_bfloat16* __restrict__ out,
                      long ldo, long so, int ldk) {
  __shared__ TIN tile[PT][PT + 1];
  const int r0 = blockIdx.y * PT, c0 = blockIdx.x * PT, b = blockIdx.z;
  const int tx = threadIdx.x, ty = threadIdx.y;
  src += (long)b * sb;
  const bool c_fast = (s_c == 1);
  for (int qq = ty; qq < PT; qq += 8) {
    const int r = c_fast ? r0 + qq : r0 + tx;
    const int c = c_fast ? c0 + tx : c0 + qq;
    TIN v;
    v.x = 0;
    v.y = 0;
    if (r < rows && c < kc) {
      v = src[(long)r * s_r + (long)c * s_c];
      if (conj) v.y = -v.y;
    }
    if (c_fast) tile[qq][tx] = v; else tile[tx][qq] = v;
  }
  __syncthreads();
  for (int qq = ty; qq < PT; qq += 8) {
    const int r = r0 + qq, c = c0 + tx;
    if (r >= rows || 2 * c >= ldk) continue;
    const int er = e[(long)b * rows + r];
    const TIN v = tile[qq][tx];
    float qr[XS], qi[XS];
    const bool live = er != kNonFinite && er > kZeroRow;
    slice_all(live ? to_fixed(v.x, er) : 0, qr);
    slice_all(live ? to_fixed(v.y, er) : 0, qi);
    __nv_bfloat162* o0 = reinterpret_cast<__nv_bfloat162*>(
        out + (long)b * so + (side == 0 ? (long)r : 2L * r) * ldo + 2L * c);
    __nv_bfloat162* o1 = o0 + ldo / 2;
#pragma unroll
    for (int t = 0; t < XS; ++t) {
      if (side == 0) {
        o0[t * (ldk / 2)] = __floats2bfloat162_rn(qr[t], qi[t]);
      } else {
        o0[t * (ldk / 2)] = __floats2bfloat162_rn(qr[t], -qi[t]);
        o1[t * (ldk / 2)] = __floats2bfloat162_rn(qi[t], qr[t]);
      }
    }
  }
}

// Exponents and sliced packing of both operands of a product in one launch (blockIdx.z = operand
// x batch + b), for K short enough that one CTA takes PR rows whole: a pass for the exponents,
// then PW columns at a time through shared memory.  Two launches each, row_exp_kernel and
// pack_exact_kernel share long rows out over more CTAs.
constexpr int PR = 16, PW = 128;
constexpr int kFusedPackK = kExactFusedPackK;
struct PackOp {
  const void* src;
  __nv_bfloat16* out;
  int* e;
  long s_r, s_c, sb, so;
  int rows, conj, side;
};
template <typename TIN>
__device__ void pack_rows(const PackOp& op, int b, int kc, int ldk, unsigned char* raw) {
  using F = decltype(TIN().x);
  TIN(*tile)[PW + 1] = reinterpret_cast<TIN(*)[PW + 1]>(raw);
  __shared__ F red[16][PR];
  __shared__ int s_e[PR];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = blockIdx.x * PR;
  if (r0 >= op.rows) return;
  const TIN* src = static_cast<const TIN*>(op.src) + (long)b * op.sb;
  const bool c_fast = op.s_c == 1;
  // largest |Re|, |Im| of a row, INFINITY for one with a non-finite entry
  auto take = [](const TIN v, F& mx, F& bad) {
    bad += (v.x - v.x) + (v.y - v.y);
    const F a = fabs(v.x), c = fabs(v.y);
    mx = a > mx ? a : mx;
    mx = c > mx ? c : mx;
  };
  if (c_fast) {
#pragma unroll
    for (int k = 0; k < PR / 8; ++k) {
      const int r = r0 + warp + 8 * k;
      F mx = 0, bad = 0;
      if (r < op.rows) {
        const TIN* x = src + (long)r * op.s_r;
#pragma unroll 4
        for (int c = lane; c < kc; c += 32) take(x[c], mx, bad);
      }
      if (!(bad == 0)) mx = INFINITY;
      for (int o = 16; o > 0; o >>= 1) {
        const F y = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = y > mx ? y : mx;
      }
      if (lane == 0) red[0][warp + 8 * k] = mx;
    }
    __syncthreads();
  } else {
    const int r = r0 + tid % PR;
    F mx = 0, bad = 0;
    if (r < op.rows) {
#pragma unroll 4
      for (int c = tid / PR; c < kc; c += 16) take(src[(long)r * op.s_r + (long)c * op.s_c], mx, bad);
    }
    if (!(bad == 0)) mx = INFINITY;
    red[tid / PR][tid % PR] = mx;
    __syncthreads();
    if (tid < PR) {
      for (int k = 1; k < 16; ++k) mx = red[k][tid] > mx ? red[k][tid] : mx;
      red[0][tid] = mx;
    }
    __syncthreads();
  }
  if (tid < PR && r0 + tid < op.rows) {
    const F mx = red[0][tid];
    int ex = 2 * kZeroRow;
    if (isinf(mx)) ex = kNonFinite;
    else if (mx > 0) frexp(mx, &ex);
    s_e[tid] = ex;
    op.e[(long)b * op.rows + r0 + tid] = ex;
  }
  for (int c0 = 0; 2 * c0 < ldk; c0 += PW) {
    __syncthreads();
    for (int i = tid; i < PR * PW; i += 256) {
      const int r = c_fast ? i / PW : i % PR, c = c_fast ? i % PW : i / PR;
      TIN v;
      v.x = 0;
      v.y = 0;
      if (r0 + r < op.rows && c0 + c < kc) {
        v = src[(long)(r0 + r) * op.s_r + (long)(c0 + c) * op.s_c];
        if (op.conj) v.y = -v.y;
      }
      tile[r][c] = v;
    }
    __syncthreads();
    for (int i = tid; i < PR * PW; i += 256) {
      const int r = i / PW, c = c0 + i % PW;
      if (r0 + r >= op.rows || 2 * c >= ldk) continue;
      const int er = s_e[r];
      const TIN v = tile[r][i % PW];
      float qr[XS], qi[XS];
      const bool live = er != kNonFinite && er > kZeroRow;
      slice_all(live ? to_fixed(v.x, er) : 0, qr);
      slice_all(live ? to_fixed(v.y, er) : 0, qi);
      const long ldo = (long)XS * ldk;
      __nv_bfloat162* o0 = reinterpret_cast<__nv_bfloat162*>(
          op.out + (long)b * op.so + (long)(r0 + r) * (op.side ? 2 : 1) * ldo + 2L * c);
      __nv_bfloat162* o1 = o0 + ldo / 2;
#pragma unroll
      for (int t = 0; t < XS; ++t) {
        o0[t * (ldk / 2)] = __floats2bfloat162_rn(qr[t], op.side ? -qi[t] : qi[t]);
        if (op.side) o1[t * (ldk / 2)] = __floats2bfloat162_rn(qi[t], qr[t]);
      }
    }
  }
}
template <typename TA, typename TB>
__global__ void __launch_bounds__(256) pack_both_kernel(const PackOp a, const PackOp b, int batch,
                                                        int kc, int ldk) {
  __shared__ __align__(16) unsigned char raw[PR * (PW + 1) * sizeof(double2)];
  if ((int)blockIdx.z < batch) pack_rows<TB>(b, blockIdx.z, kc, ldk, raw);
  else pack_rows<TA>(a, blockIdx.z - batch, kc, ldk, raw);
}

// BF16 copies of FP32 matrices (job: src[r*s_r + c], r < rows, c < cols), as they are and/or
// transposed, all of a pass in one launch; tiled through shared memory so that reads and both
// writes are coalesced.
__global__ void __launch_bounds__(PT * 8) mlp_pack_kernel(const __grid_constant__ MlpPack g) {
  __shared__ float tile[PT][PT + 1];
  int p = 0;
  while (p + 1 < g.count && (int)blockIdx.x >= g.job[p + 1].tile0) ++p;
  const MlpPackJob& j = g.job[p];
  const int t = blockIdx.x - j.tile0, tc = (j.cols + PT - 1) / PT;
  const int r0 = t / tc * PT, c0 = t % tc * PT, tx = threadIdx.x, ty = threadIdx.y;
  for (int q = ty; q < PT; q += 8) {
    const int r = r0 + q, c = c0 + tx;
    const float v = r < j.rows && c < j.cols ? j.src[(long)r * j.s_r + c] : 0.f;
    tile[q][tx] = v;
    if (j.row && r < j.rows && c < j.cols) j.row[(long)r * j.ldr + c] = __float2bfloat16_rn(v);
  }
  __syncthreads();
  if (j.col)
    for (int q = ty; q < PT; q += 8) {
      const int c = c0 + q, r = r0 + tx;
      if (r < j.rows && c < j.cols) j.col[(long)c * j.ldc + r] = __float2bfloat16_rn(tile[tx][q]);
    }
}

// ------------------------------------------------------------------ host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    else
      cudaGetLastError();
  });
  return fn;
}

// 3-D K-major map: dims {K, rows, batch}, box {row_bytes of K, box_rows, 1}, swizzled over the
// row's 128 or 64 bytes.
bool make_map(CUtensorMap* map, int elt, const void* base, long k, long rows, long ld, long sb,
              int batch, int box_rows, int row_bytes = 128) {
  auto fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)k, (cuuint64_t)rows, (cuuint64_t)batch};
  const cuuint64_t strides[2] = {(cuuint64_t)ld * elt,
                                 (cuuint64_t)(batch > 1 ? sb : rows * ld) * elt};
  const cuuint32_t box[3] = {(cuuint32_t)(row_bytes / elt), (cuuint32_t)box_rows, 1};
  const cuuint32_t es[3] = {1, 1, 1};
  CUresult r = fn(map, elt == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                  3, const_cast<void*>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE,
                  row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <int ELT, int BN, int STAGES>
constexpr size_t smem_bytes() {
  return (size_t)STAGES * (BM + BN) * 128 + 1024 + 2 * STAGES * 8 + 64;
}

template <int ELT, int BN, int STAGES>
cudaError_t launch_bn(cudaStream_t st, const CUtensorMap& ma, const CUtensorMap& mb, int M, int N,
                      int K, int batch, const Epi& ep, int* err) {
  constexpr size_t sm = smem_bytes<ELT, BN, STAGES>();
  static const cudaError_t attr = cudaFuncSetAttribute(
      tc_gemm_kernel<ELT, BN, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (attr != cudaSuccess) return attr;
  dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, batch);
  tc_gemm_kernel<ELT, BN, STAGES><<<grid, kThreads, sm, st>>>(ma, mb, M, N, K, ep, err);
  count_launch();
  g_tc_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

}  // namespace tc

using namespace tc;

// The tile width with the least time on the busiest SM: waves of tiles times a tile's time, which
// is its columns and a fixed part (fill, narrow products' lower rate, epilogue) worth 64 of them;
// the narrower of equals.  2304 x 4608 x 4608 (TF32x3 of a bond's new centre): 324 tiles of 256
// columns need three waves of 152, and so do 432 of 192, each a quarter
// shorter: the call takes 242 us instead of 290; 1500 x 1500 x 500 104 instead of 118, 297 x 1600 x
// 200 54 instead of 66; sizes whose width stays take the same.
int tc_pick_bn(long M, long N, int batch) {
  const long mt = (M + BM - 1) / BM;
  int best = 64;
  long cost = -1;
  for (int bn : {64, 128, 192, 256}) {
    if (bn > 64 && N <= bn / 2) break;
    const long c = (mt * ((N + bn - 1) / bn) * batch + kSms - 1) / kSms * (bn + 64);
    if (cost < 0 || c < cost) {
      cost = c;
      best = bn;
    }
  }
  return best;
}

cudaError_t tc_gemm_real(cudaStream_t st, int elt, int M, int N, int K, const void* A, long lda,
                         long sa, const void* B, long ldb, long sb, int batch, const TcEpilogue& e,
                         int* err, int bn) {
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  if (K <= 0) return cudaErrorInvalidValue;
  if ((lda * elt) % 16 || (ldb * elt) % 16 || (batch > 1 && ((sa * elt) % 16 || (sb * elt) % 16)) ||
      (reinterpret_cast<uintptr_t>(A) & 15) || (reinterpret_cast<uintptr_t>(B) & 15))
    return cudaErrorInvalidValue;
  if (bn <= 0) bn = tc_pick_bn(M, N, batch);
  CUtensorMap ma, mb;
  if (!make_map(&ma, elt, A, K, M, lda, sa, batch, BM) ||
      !make_map(&mb, elt, B, K, N, ldb, sb, batch, bn))
    return cudaErrorInvalidValue;
  Epi ep;
  ep.d = e.d;
  ep.d64 = e.d64;
  ep.ldd = e.ldd;
  ep.sd = e.sd;
  ep.ar = e.ar; ep.ai = e.ai; ep.br = e.br; ep.bi = e.bi;
  ep.use_beta = e.use_beta;
  ep.scale = e.scale;
  ep.mode = e.d64 ? 1 : 0;
  if (elt == 4) {
    if (bn == 256) return launch_bn<4, 256, 4>(st, ma, mb, M, N, K, batch, ep, err);
    if (bn == 192) return launch_bn<4, 192, 5>(st, ma, mb, M, N, K, batch, ep, err);
    if (bn == 128) return launch_bn<4, 128, 6>(st, ma, mb, M, N, K, batch, ep, err);
    return launch_bn<4, 64, 8>(st, ma, mb, M, N, K, batch, ep, err);
  }
  if (bn == 256) return launch_bn<2, 256, 4>(st, ma, mb, M, N, K, batch, ep, err);
  if (bn == 192) return launch_bn<2, 192, 5>(st, ma, mb, M, N, K, batch, ep, err);
  if (bn == 128) return launch_bn<2, 128, 6>(st, ma, mb, M, N, K, batch, ep, err);
  return launch_bn<2, 64, 8>(st, ma, mb, M, N, K, batch, ep, err);
}

cudaError_t mlp_pack(cudaStream_t st, MlpPack& g) {
  int tiles = 0;
  for (int i = 0; i < g.count; ++i) {
    g.job[i].tile0 = tiles;
    tiles += ((g.job[i].rows + PT - 1) / PT) * ((g.job[i].cols + PT - 1) / PT);
  }
  count_launch();
  mlp_pack_kernel<<<tiles, dim3(PT, 8), 0, st>>>(g);
  return cudaGetLastError();
}

namespace {
template <int BN, int STAGES, int CAP>
cudaError_t mlp_launch(cudaStream_t st, MlpGroup<CAP>& g, int* err) {
  constexpr size_t sm = smem_bytes<2, BN, STAGES>();
  static const cudaError_t attr =
      cudaFuncSetAttribute(mlp_gemm_kernel<BN, STAGES, CAP>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (attr != cudaSuccess) return attr;
  g.tiles = 0;
  int extra = 0;
  for (int i = 0; i < g.count; ++i) {
    MlpProd& q = g.p[i];
    if (!make_map(&q.a, 2, q.A, q.K, q.M, q.lda, 0, 1, BM) ||
        !make_map(&q.b, 2, q.B, q.K, q.N, q.ldb, 0, 1, BN))
      return cudaErrorInvalidValue;
    q.tile0 = g.tiles;
    g.tiles += ((q.M + BM - 1) / BM) * ((q.N + BN - 1) / BN);
    extra += (q.N + kThreads - 1) / kThreads;
  }
  if (!g.loss_sum) extra = -1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g.tiles + extra + 1);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  MPDO_CUDA_TRY(cudaLaunchKernelEx(&cfg, mlp_gemm_kernel<BN, STAGES, CAP>, g, err));
  count_launch();
  g_tc_launches.fetch_add(g.count, std::memory_order_relaxed);
  return cudaGetLastError();
}
}  // namespace
// A pass's products are short, and their epilogues, which grow with the tile, are most of their time:
// 256 columns only where nearly every SM has such a tile, 128 and 64 where half of them have, else 32.
template <int CAP>
cudaError_t mlp_products(cudaStream_t st, MlpGroup<CAP>& g, int* err) {
  int maxn = 0;
  long t256 = 0, t128 = 0, t64 = 0;
  for (int i = 0; i < g.count; ++i) {
    const long mt = (g.p[i].M + BM - 1) / BM;
    maxn = std::max(maxn, g.p[i].N);
    t256 += mt * ((g.p[i].N + 255) / 256);
    t128 += mt * ((g.p[i].N + 127) / 128);
    t64 += mt * ((g.p[i].N + 63) / 64);
  }
  if (maxn > 128 && t256 >= 148) return mlp_launch<256, 4, CAP>(st, g, err);
  if (maxn > 64 && t128 >= 74) return mlp_launch<128, 6, CAP>(st, g, err);
  if (t64 >= 74) return mlp_launch<64, 8, CAP>(st, g, err);
  return mlp_launch<32, 8, CAP>(st, g, err);   // half the epilogue per thread
}
template cudaError_t mlp_products<1>(cudaStream_t, MlpGroup<1>&, int*);
template cudaError_t mlp_products<kMlpMaxLayers>(cudaStream_t, MlpGroup<kMlpMaxLayers>&, int*);

size_t tc_pack_bytes(int mode, long rows, long k, int batch) {
  const int elt = tc_mode_elt(mode);
  const long kr = (long)tc_mode_parts(mode) * 2 * k;
  const long ld = tc_pack_ld(mode, k);
  (void)kr;
  return (size_t)batch * rows * ld * elt + 256;
}

template <typename TIN>
cudaError_t tc_pack(cudaStream_t st, int mode, int side, int rows, int kc, const cx<TIN>* src,
                    long s_r, long s_c, long sb, int conj, int batch, void* out) {
  const long ld = tc_pack_ld(mode, kc);
  const long so = (long)(side == 0 ? rows : 2 * rows) * ld;
  dim3 grid((kc + PT - 1) / PT, (rows + PT - 1) / PT, batch), block(PT, 8);
  const int np = tc_mode_parts(mode);
  if (tc_mode_elt(mode) == 4)
    pack_kernel<cx<TIN>, float><<<grid, block, 0, st>>>(rows, kc, src, s_r, s_c, sb, conj, side,
                                                       np, static_cast<float*>(out), ld, so);
  else
    pack_kernel<cx<TIN>, __nv_bfloat16><<<grid, block, 0, st>>>(
        rows, kc, src, s_r, s_c, sb, conj, side, np, static_cast<__nv_bfloat16*>(out), ld, so);
  count_launch();
  return cudaGetLastError();
}

// Source strides of op(X) as an (rows x kc) matrix indexed [r][c] from a row-major matrix
// with leading dimension ld: for the A operand rows = m, c = k; for B rows = n, c = k.
static void op_strides(int side, int op, long ld, long* s_r, long* s_c, int* conj) {
  // A: op(A)[i][p]; N: A[i][p], T/C: A[p][i], R: conj A[i][p]
  // B: X[q][p] = op(B)[p][q]; N/R: B[p][q] -> s_r = 1, s_c = ld; T/C: B[q][p]
  const bool trans = (op == OP_T || op == OP_C);
  *conj = (op == OP_C || op == OP_R) ? 1 : 0;
  const bool rowmajor_rc = side == 0 ? !trans : trans;
  if (rowmajor_rc) { *s_r = ld; *s_c = 1; } else { *s_r = 1; *s_c = ld; }
}

template <typename TIN>
cudaError_t tc_cgemm(cudaStream_t st, int mode, int opa, int opb, int m, int n, int k,
                     const cx<TIN>* A, long lda, long sa, const cx<TIN>* B, long ldb, long sb,
                     float2* C, long ldc, long sc, int batch, float2 alpha, float2 beta,
                     void* ws, size_t ws_bytes, int* err) {
  if (m <= 0 || n <= 0 || batch <= 0) return cudaSuccess;
  const int elt = tc_mode_elt(mode);
  // K is processed in chunks whose packed operands fit the workspace; later chunks add to
  // the output (beta = 1)
  long kc = k;
  while (kc > 32 && tc_cgemm_ws_bytes(mode, m, n, kc, batch) > ws_bytes) kc = (kc + 1) / 2;
  if (kc < k) kc = std::max(32L, kc / 32 * 32);
  if (tc_cgemm_ws_bytes(mode, m, n, kc, batch) > ws_bytes) return cudaErrorMemoryAllocation;
  long sra, sca, srb, scb;
  int cja, cjb;
  op_strides(0, opa, lda, &sra, &sca, &cja);
  op_strides(1, opb, ldb, &srb, &scb, &cjb);
  for (long k0 = 0; k0 < k; k0 += kc) {
    const int kn = (int)std::min<long>(kc, k - k0);
    const long ld = tc_pack_ld(mode, kn);
    const size_t abytes = ((size_t)batch * m * ld * elt + 255) & ~(size_t)255;
    char* pa = static_cast<char*>(ws);
    char* pb = pa + abytes;
    MPDO_CUDA_TRY(tc_pack<TIN>(st, mode, 0, m, kn, A + k0 * sca, sra, sca, sa, cja, batch, pa));
    MPDO_CUDA_TRY(tc_pack<TIN>(st, mode, 1, n, kn, B + k0 * scb, srb, scb, sb, cjb, batch, pb));
    TcEpilogue e;
    e.d = reinterpret_cast<float*>(C);
    e.ldd = 2 * ldc;
    e.sd = 2 * sc;
    e.ar = alpha.x; e.ai = alpha.y;
    if (k0 == 0) {
      e.br = beta.x; e.bi = beta.y;
    } else {
      e.br = 1.f; e.bi = 0.f;
    }
    e.use_beta = (e.br != 0.f || e.bi != 0.f);
    const long kr = (long)tc_mode_parts(mode) * 2 * kn;
    MPDO_CUDA_TRY(tc_gemm_real(st, elt, m, 2 * n, (int)kr, pa, ld, (long)m * ld, pb, ld,
                               2L * n * ld, batch, e, err, 0));
  }
  return cudaSuccess;
}

// ---- exact products: C (complex FP64) = op(A) op(B), FP32 or FP64 complex A and B
namespace {
// op(B) = op(A)^+ of the same data: the product is Hermitian
template <typename TA, typename TB>
bool is_gram(int opa, int opb, int m, int n, const TA* A, long lda, long sa, const TB* B, long ldb,
             long sb) {
  return std::is_same<TA, TB>::value && (const void*)A == (const void*)B && lda == ldb && sa == sb &&
         m == n && ((opa == OP_C && opb == OP_N) || (opa == OP_N && opb == OP_C));
}
}  // namespace

cudaError_t tc_exact_init() {
  static const cudaError_t attr =
      cudaFuncSetAttribute(tc_exact_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(XSTAGES * XSTAGE_BYTES + 1024 + 256));
  return attr;
}

template <typename TA, typename TB>
cudaError_t tc_cgemm_exact(cudaStream_t st, int opa, int opb, int m, int n, int k, const TA* A,
                           long lda, long sa, const TB* B, long ldb, long sb, double2* C, long ldc,
                           long sc, int batch, void* ws, size_t ws_bytes, int* err) {
  const bool gram = is_gram(opa, opb, m, n, A, lda, sa, B, ldb, sb);
  if (m <= 0 || n <= 0 || batch <= 0) return cudaSuccess;
  if (k <= 0) return cudaErrorInvalidValue;
  const long kc = exact_piece(m, n, k, batch, gram, ws_bytes);
  if (kc == 0) return cudaErrorMemoryAllocation;
  long sra, sca, srb, scb;
  int cja, cjb;
  op_strides(0, opa, lda, &sra, &sca, &cja);
  op_strides(1, opb, ldb, &srb, &scb, &cjb);
  MPDO_CUDA_TRY(tc_exact_init());
  for (long k0 = 0; k0 < k; k0 += kc) {
    const int kn = (int)std::min<long>(kc, k - k0);
    const ExactPlan pl = exact_piece_plan(m, n, kn, batch, gram, ws_bytes);
    const int ldk = (int)exact_ldk(kn);
    const long ldo = (long)XS * ldk;
    char* p = static_cast<char*>(ws);
    __nv_bfloat16* pa = reinterpret_cast<__nv_bfloat16*>(p);
    if (!gram) p += ((size_t)batch * m * ldo * 2 + 255) & ~(size_t)255;
    __nv_bfloat16* pb = reinterpret_cast<__nv_bfloat16*>(p);
    p += ((size_t)batch * 2 * n * ldo * 2 + 255) & ~(size_t)255;
    int* eb = reinterpret_cast<int*>(p);
    int* ea = gram ? eb : eb + (size_t)batch * n;
    p += ((size_t)batch * (m + n) * sizeof(int) + 255) & ~(size_t)255;
    longlong2* part = pl.parts ? reinterpret_cast<longlong2*>(p) : nullptr;
    auto exps = [&](auto* x, int rows, long sr, long s_c, long s_b, int* e) {
      const int rb = s_c == 1 ? (rows + 7) / 8 : (rows + 31) / 32;
      // enough column slices for about two CTAs per SM, at least 64 columns each
      int sl = std::max(1, std::min((kn + 63) / 64, 304 / std::max(1, rb * batch)));
      const int cols = (kn + sl - 1) / sl;
      sl = (kn + cols - 1) / cols;
      row_exp_kernel<<<dim3(rb, sl, batch), 256, 0, st>>>(rows, kn, x, sr, s_c, s_b, cols, e);
    };
    // exponents and packing as launches of their own, over column slices and tiles
    auto pack = [&](auto* x, int rows, long sr, long s_c, long s_b, int cj, int side, const int* e,
                    __nv_bfloat16* o) {
      pack_exact_kernel<<<dim3((ldk / 2 + PT - 1) / PT, (rows + PT - 1) / PT, batch), dim3(PT, 8), 0,
                          st>>>(rows, kn, x, sr, s_c, s_b, cj, side, e, o, ldo,
                                (side ? 2L : 1L) * rows * ldo, ldk);
    };
    const TA* a0 = A + k0 * sca;
    const TB* b0 = B + k0 * scb;
    if (kn <= kFusedPackK && 2L * batch <= 65535) {   // the grid's z extent
      const PackOp ob{b0, pb, eb, srb, scb, sb, 2L * n * ldo, n, cjb, 1};
      const PackOp oa{a0, pa, ea, sra, sca, sa, (long)m * ldo, m, cja, 0};
      pack_both_kernel<TA, TB><<<dim3((std::max(gram ? 0 : m, n) + PR - 1) / PR, 1, gram ? batch : 2 * batch),
                                 256, 0, st>>>(oa, ob, batch, kn, ldk);
      count_launch();
    } else {
      // exponents below kZeroRow until a row's entries raise them
      MPDO_CUDA_TRY(cudaMemsetAsync(eb, 0x80, (size_t)batch * (gram ? n : m + n) * sizeof(int), st));
      exps(b0, n, srb, scb, sb, eb);
      pack(b0, n, srb, scb, sb, cjb, 1, eb, pb);
      if (!gram) {
        exps(a0, m, sra, sca, sa, ea);
        pack(a0, m, sra, sca, sa, cja, 0, ea, pa);
      }
      count_launch(gram ? 2 : 4);
    }
    MPDO_CUDA_TRY(cudaGetLastError());
    CUtensorMap ma, mb;
    if (!make_map(&ma, 2, pa, ldo, m, gram ? 2 * ldo : ldo, (gram ? 2L * n : m) * ldo, batch, BM,
                  XKB * 2) ||
        !make_map(&mb, 2, pb, ldo, 2L * n, ldo, 2L * n * ldo, batch, XBN, XKB * 2))
      return cudaErrorInvalidValue;
    const size_t smem = XSTAGES * XSTAGE_BYTES + 1024 + 256;
    const int acc = k0 > 0 ? 1 : 0;
    tc_exact_kernel<<<pl.ctas, XTHREADS, smem, st>>>(ma, mb, m, 2 * n, ldk, pl.nst, pl.tiles, pl.per,
                                                     pl.total, gram ? 1 : 0, ea, eb, C, ldc, sc, acc,
                                                     part, err);
    count_launch();
    g_tc_launches.fetch_add(1, std::memory_order_relaxed);
    MPDO_CUDA_TRY(cudaGetLastError());
    if (part) {
      exact_finish_kernel<<<dim3((unsigned)((long)pl.tiles * batch), 4), 256, 0, st>>>(
          m, 2 * n, pl.nst, pl.tiles, pl.per, gram ? 1 : 0, part, ea, eb, C, ldc, sc, acc);
      count_launch();
      MPDO_CUDA_TRY(cudaGetLastError());
    }
  }
  return cudaSuccess;
}

template cudaError_t tc_cgemm_exact<float2, float2>(cudaStream_t, int, int, int, int, int,
                                                    const float2*, long, long, const float2*,
                                                    long, long, double2*, long, long, int, void*,
                                                    size_t, int*);
template cudaError_t tc_cgemm_exact<float2, double2>(cudaStream_t, int, int, int, int, int,
                                                     const float2*, long, long, const double2*,
                                                     long, long, double2*, long, long, int, void*,
                                                     size_t, int*);
template cudaError_t tc_cgemm_exact<double2, float2>(cudaStream_t, int, int, int, int, int,
                                                     const double2*, long, long, const float2*,
                                                     long, long, double2*, long, long, int, void*,
                                                     size_t, int*);
template cudaError_t tc_cgemm_exact<double2, double2>(cudaStream_t, int, int, int, int, int,
                                                      const double2*, long, long, const double2*,
                                                      long, long, double2*, long, long, int, void*,
                                                      size_t, int*);

size_t tc_cgemm_ws_bytes(int mode, long m, long n, long k, int batch) {
  const int elt = tc_mode_elt(mode);
  const long ld = tc_pack_ld(mode, k);
  return (((size_t)batch * m * ld * elt + 255) & ~(size_t)255) + (size_t)batch * 2 * n * ld * elt;
}

template cudaError_t tc_pack<float>(cudaStream_t, int, int, int, int, const cx<float>*, long, long,
                                    long, int, int, void*);
template cudaError_t tc_pack<double>(cudaStream_t, int, int, int, int, const cx<double>*, long,
                                     long, long, int, int, void*);
template cudaError_t tc_cgemm<float>(cudaStream_t, int, int, int, int, int, int, const cx<float>*,
                                     long, long, const cx<float>*, long, long, float2*, long, long,
                                     int, float2, float2, void*, size_t, int*);

}  // namespace mpdo

// ------------------------------------------------------------------ C ABI (tests)
#include "../../include/mpdo.h"

namespace mpdo {
void set_global_error(const char* msg);
}

namespace {
// Scratch of the entry points below, stream-ordered from a memory pool of the library's own per
// device.  cudaMalloc and cudaFree of some 100 MB a call took 273 of a product's 568 us (2304 x
// 2304 x 768) and 283 of a Gram's 772 us; a pool allocation that finds its memory takes about one.
// At a synchronisation the pool keeps at most kPoolKeep and returns the rest to the device;
// scratch_trim() returns all that is not in use, and the library's other allocations call it before
// they give up.  The driver orders reuse between streams and threads.
constexpr uint64_t kPoolKeep = 512ull << 20;
constexpr int kPoolDevs = 16;
std::mutex g_pool_mu;
cudaMemPool_t g_pool[kPoolDevs] = {};
cudaMemPool_t scratch_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= kPoolDevs) return nullptr;
  std::lock_guard<std::mutex> lock(g_pool_mu);
  if (!g_pool[dev]) {
    cudaMemPoolProps pr = {};
    pr.allocType = cudaMemAllocationTypePinned;
    pr.location.type = cudaMemLocationTypeDevice;
    pr.location.id = dev;
    uint64_t keep = kPoolKeep;
    cudaMemPool_t p;
    if (cudaMemPoolCreate(&p, &pr) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    g_pool[dev] = p;
  }
  return g_pool[dev];
}
// The flag is zeroed and behind the scratch; without a pool, plain allocations as they come.
struct Scratch {
  void* p = nullptr;
  int* err = nullptr;
  cudaStream_t st;
  bool pooled = false;
  explicit Scratch(cudaStream_t s) : st(s) {}
  bool alloc(size_t bytes) {
    bytes = (bytes + 255) / 256 * 256;
    if (cudaMemPool_t pool = scratch_pool())
      pooled = cudaMallocFromPoolAsync(&p, bytes + 256, pool, st) == cudaSuccess;
    if (!pooled && (cudaGetLastError(), mpdo::dev_malloc(&p, bytes + 256) != cudaSuccess)) {
      p = nullptr;
      return false;
    }
    err = reinterpret_cast<int*>(static_cast<char*>(p) + bytes);
    cudaMemsetAsync(err, 0, sizeof(int), st);
    return true;
  }
  ~Scratch() {
    if (!p) return;
    if (pooled) cudaFreeAsync(p, st);
    else cudaFree(p);
  }
};
int tc_fail(int code, const char* msg) {
  mpdo::set_global_error(msg);
  return code;
}
}  // namespace

namespace mpdo {
void scratch_trim() {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  for (cudaMemPool_t p : g_pool)
    if (p) cudaMemPoolTrimTo(p, 0);
}
cudaError_t dev_malloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    scratch_trim();
    e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) cudaGetLastError();
  }
  return e;
}
}  // namespace mpdo

extern "C" {

void mpdo_kernel_trim(void) { mpdo::scratch_trim(); }

long long mpdo_tc_gemm_launches(void) { return mpdo::g_tc_launches.load(); }

int mpdo_kernel_tcgemm_real(int elt, int m, int n, int k, const void* a, long lda, const void* b,
                            long ldb, float* d, long ldd, void* stream) {
  if ((elt != 2 && elt != 4) || m < 0 || n < 0 || k < 1 || !a || !b || !d)
    return tc_fail(MPDO_ERR_ARG, "bad tcgemm_real arguments");
  if ((lda * elt) % 16 || (ldb * elt) % 16 || lda < k || ldb < k || ldd < n)
    return tc_fail(MPDO_ERR_ARG, "tcgemm_real: leading dimensions must cover k (n) and be "
                                 "multiples of 16 bytes");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Scratch w(st);
  if (!w.alloc(0)) return tc_fail(MPDO_ERR_OOM, "tcgemm_real: error flag");
  mpdo::TcEpilogue e;
  e.d = d;
  e.ldd = ldd;
  cudaError_t ce = mpdo::tc_gemm_real(st, elt, m, n, k, a, lda, 0, b, ldb, 0, 1, e,
                                      w.err, 0);
  int herr = 0;
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(&herr, w.err, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess) return tc_fail(MPDO_ERR_CUDA, cudaGetErrorString(ce));
  if (herr) return tc_fail(MPDO_ERR_TIMEOUT, "tcgemm_real: a pipeline wait gave up");
  return MPDO_OK;
}

int mpdo_kernel_tcgemm(int mode, int opa, int opb, int m, int n, int k, const void* a, long lda,
                       long sa, const void* b, long ldb, long sb, void* c, long ldc, long sc,
                       int batch, void* stream) {
  if (mode < 0 || mode > 3 || opa < 0 || opa > 3 || opb < 0 || opb > 3 || m < 0 || n < 0 ||
      k < 1 || batch < 0 || !a || !b || !c)
    return tc_fail(MPDO_ERR_ARG, "bad tcgemm arguments");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t ws = mpdo::tc_cgemm_ws_bytes(mode, m, n, k, batch);
  Scratch w(st);
  if (!w.alloc(ws)) return tc_fail(MPDO_ERR_OOM, "tcgemm workspace");
  cudaError_t ce = mpdo::tc_cgemm<float>(
      st, mode, opa, opb, m, n, k, static_cast<const float2*>(a), lda, sa,
      static_cast<const float2*>(b), ldb, sb, static_cast<float2*>(c), ldc, sc, batch,
      make_float2(1.f, 0.f), make_float2(0.f, 0.f), w.p, ws, w.err);
  int herr = 0;
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(&herr, w.err, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess) return tc_fail(MPDO_ERR_CUDA, cudaGetErrorString(ce));
  if (herr) return tc_fail(MPDO_ERR_TIMEOUT, "tcgemm: a pipeline wait gave up");
  return MPDO_OK;
}

int mpdo_kernel_tcgemm_exact(int opa, int opb, int m, int n, int k, const void* a, long lda,
                             long sa, const void* b, long ldb, long sb, void* c, long ldc,
                             long sc, int batch, void* stream) {
  if (opa < 0 || opa > 3 || opb < 0 || opb > 3 || m < 0 || n < 0 || k < 1 || batch < 0 || !a ||
      !b || !c)
    return tc_fail(MPDO_ERR_ARG, "bad tcgemm_exact arguments");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const bool gram = mpdo::is_gram(opa, opb, m, n, a, lda, sa, b, ldb, sb);
  const size_t ws = mpdo::exact_ws_bytes(m, n, k, batch, gram);
  Scratch w(st);
  if (!w.alloc(ws)) return tc_fail(MPDO_ERR_OOM, "tcgemm_exact workspace");
  cudaError_t ce = mpdo::tc_cgemm_exact<float2, float2>(
      st, opa, opb, m, n, k, static_cast<const float2*>(a), lda, sa, static_cast<const float2*>(b),
      ldb, sb, static_cast<double2*>(c), ldc, sc, batch, w.p, ws, w.err);
  int herr = 0;
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(&herr, w.err, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess) return tc_fail(MPDO_ERR_CUDA, cudaGetErrorString(ce));
  if (herr) return tc_fail(MPDO_ERR_TIMEOUT, "tcgemm_exact: a pipeline wait gave up");
  return MPDO_OK;
}

}  // extern "C"
