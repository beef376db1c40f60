// Parallel two-sided block Jacobi eigensolver for Hermitian matrices (FP64 / FP32).
//
// The columns are split into blocks of JW = 8; every round pairs the blocks by a
// round-robin tournament.  One CTA per pair diagonalises its 16 x 16 principal sub-matrix
// with scalar cyclic Jacobi rotations in shared memory (GVL sym.schur2 with the complex
// phase factored out) and publishes the accumulated 16 x 16 unitary; after a grid-wide
// barrier the warps of all CTAs apply the unitaries, A[p, q] <- U_p^+ A[p, q] U_q for the 16 x 16
// tiles of the upper half (mirrored into the lower) and V[:, q] <- V[:, q] U_q, and a second
// barrier ends the round.  A tile needs no other tile, so A is read and written once a round, and
// V is kept transposed, so that its rows are contiguous.  A sweep in which no pair rotated ends
// the iteration.  Cost per sweep ~4 n^3 complex MACs; the matrix stays in L2 (29 MB
// with V at n = 1350).  A round there is bound by FP32 issue in the tiles (~12 us
// of FMAs) and, before them, the serial chain of 15 rotation steps and the grid barriers; rows and
// columns in two passes of 16 x np by the pairs' own CTAs, each waiting for its loads, took 92 us.
// In the late sweeps few pairs have anything left to rotate: a sub-problem looks first, and a round
// in which none had leaves out its tiles and second barrier.  The mixed solver's six levels at n =
// 1350 (FP32 solves of 1350 down to 464): 1240 ms with the passes, 250 ms with tiles, ~190 ms with the
// look ahead and items from a counter; FP64 at n = 400: 277 -> 92 ms.
#include <cooperative_groups.h>
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include "../../include/mpdo.h"

#include "common.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

namespace mpdo {
namespace {

constexpr int JW = 8;          // block width
constexpr int JS = 2 * JW;     // sub-problem size
constexpr int JT = 256;        // threads per CTA: one per entry of the sub-problem
constexpr int JV = 32;         // columns of V^T in a warp's item
constexpr int kMaxPairs = 1024;   // n <= 16384
// Sweeps of the 16x16 sub-problem per block-pair visit.  One sweep per visit is the
// classic one-sided-update choice: the outer rounds keep rotating the pair, so a fully
// converged sub-problem buys little and costs 15 warp rounds per extra sweep.
constexpr int kInnerSweeps = 1;


template <typename R> struct Tol;
template <> struct Tol<double> { static constexpr double rel = 1e-15, abs = 2.2e-16; };
// FP32: absolute threshold only.  Eigenvalues below ~eps |A| are not resolved in FP32
// whatever the rotations do (every FP32 cut sits above 10 eps, and the mixed solver
// resolves the small ones in its next level), so pairs whose coupling is below eps |A|
// are left alone; this saves the sweeps a relative threshold spends on them.
template <> struct Tol<float> { static constexpr float rel = 0.f, abs = 6e-8f; };

template <typename R>
__global__ void pad_copy_kernel(int n, int np, const cx<R>* __restrict__ a, long lda,
                                cx<R>* __restrict__ ap, cx<R>* __restrict__ vp, int* counters) {
  long total = (long)np * np;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    int i = (int)(e / np), j = (int)(e % np);
    cx<R> v = mkc<R>(0, 0);
    if (i < n && j < n) v = a[(long)i * lda + j];
    ap[e] = v;
    vp[e] = mkc<R>(i == j ? 1 : 0, 0);
  }
  if (blockIdx.x == 0 && threadIdx.x < 4) counters[threadIdx.x] = 0;
}

// Warp-private products of 16 x 16 tiles: lane (r = lane / 2, h = lane % 2) has the entries
// (r, 8 h .. 8 h + 7).  Operands read along a row of 16 are aligned vectors that half of the lanes
// share; a tile read down its rows has a stride of 17.
template <typename T>
__device__ __forceinline__ void tile_zero(T* acc) {
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i].x = acc[i].y = 0;
}
// acc += sum_k x(k) y[k][8 h + i], x(k) from left(k)
template <typename T, typename F>
__device__ __forceinline__ void tile_mul(T* acc, const T* y, int h, F&& left) {
#pragma unroll 4
  for (int k = 0; k < JS; ++k) {
    const T x = left(k);
    T q[8];
    const float4* p = reinterpret_cast<const float4*>(y + k * JS + 8 * h);
#pragma unroll
    for (int i = 0; i < (int)sizeof(T) / 2; ++i) reinterpret_cast<float4*>(q)[i] = p[i];
#pragma unroll
    for (int i = 0; i < 8; ++i) cfma(acc[i], x, q[i]);
  }
}
template <typename T>
__device__ __forceinline__ void copy8(T* dst, const T* src) {
#pragma unroll
  for (int i = 0; i < (int)sizeof(T) / 2; ++i)
    reinterpret_cast<float4*>(dst)[i] = reinterpret_cast<const float4*>(src)[i];
}

// Rotation of the pair (al, be) with coupling g of modulus ag: cosine and s e of the two columns,
// from rounded roots and quotients.  In FP32 approximate ones (rsqrtf, __fdividef) shorten the chain
// of a step from ~600 clocks to ~150 (n = 1350, mixed: 211 ms instead of 224), but their errors are
// one-sided: over the ~1000 rounds of a solve the spectrum shrinks by 1e-5 (n = 400; 1.5e-6 here),
// which the polar step after the sub-problem, itself rounded to FP32, does not see.
template <typename R>
__device__ __forceinline__ R modulus(cx<R> g) { return sqrt(cabs2(g)); }
template <typename R>
__device__ __forceinline__ void rotation(cx<R> g, R ag, R al, R be, R& c, cx<R>& o) {
  const R tau = (be - al) / (2 * ag);
  const R t = (tau >= 0 ? R(1) : R(-1)) / (fabs(tau) + sqrt(R(1) + tau * tau));
  c = R(1) / sqrt(R(1) + t * t);
  o = cscale(mkc<R>(g.x / ag, g.y / ag), t * c);
}

template <typename R>
constexpr size_t coop_smem() {   // per warp: U_p, U_q, a tile of stride 17
  return (size_t)(JT / 32) * (2 * JS * JS + JS * (JS + 1)) * sizeof(cx<R>);
}

template <typename R>
__global__ void __launch_bounds__(JT, 2) jacobi_coop_kernel(int np, int nblk, cx<R>* ap, cx<R>* vt,
                                                            cx<R>* ug, int* act, int* next,
                                                            int* counters, int max_sweeps) {
  using T = cx<R>;
  cg::grid_group grid = cg::this_grid();
  extern __shared__ __align__(16) unsigned char jc_raw[];
  __shared__ T S[2][JS][JS + 1];
  __shared__ T U[2][JS][JS + 1];
  __shared__ R rc[JS];             // per index: cosine, partner's coefficient, partner
  __shared__ T ro[JS];
  __shared__ int rp[JS];
  __shared__ unsigned char s_act[kMaxPairs];
  __shared__ unsigned char sa[JS - 1][JS / 2], sb[JS - 1][JS / 2];   // pairs of a step, a < b
  __shared__ R s_anorm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pairs = nblk / 2;
  if (tid < (JS - 1) * (JS / 2)) {
    int a, b;
    tourney(tid / (JS / 2), tid % (JS / 2), JS, a, b);
    sa[tid / (JS / 2)][tid % (JS / 2)] = (unsigned char)min(a, b);
    sb[tid / (JS / 2)][tid % (JS / 2)] = (unsigned char)max(a, b);
  }

  // |A| scale for the absolute rotation floor: sum of |diag|, reduced in a fixed order so
  // that every CTA (and every run) uses the same threshold
  {
    __shared__ R wpart[JT / 32];
    R part = 0;
    for (int i = tid; i < np; i += JT) part += fabs(ap[(long)i * np + i].x);
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0) wpart[tid >> 5] = part;
    __syncthreads();
    if (tid == 0) {
      R t = 0;
      for (int k = 0; k < JT / 32; ++k) t += wpart[k];
      s_anorm = t;
    }
  }
  __syncthreads();
  const R atol = Tol<R>::abs * s_anorm;
  const int i = tid / JS, j = tid % JS;
  // the warp's buffers and its place among all warps
  T* Up = reinterpret_cast<T*>(jc_raw) + (size_t)warp * (2 * JS * JS + JS * (JS + 1));
  T* Uq = Up + JS * JS;
  T* X = Uq + JS * JS;
  const int r = lane >> 1, h = lane & 1;
  const int vcols = (np + JV - 1) / JV, vitems = pairs * vcols;
  const int items = vitems + pairs * (pairs + 1) / 2;
  if (blockIdx.x == 0 && tid == 0) next[0] = gridDim.x * (JT / 32);
  int sweep = 0, tick = 0;   // tick: rounds so far
  for (; sweep < max_sweeps; ++sweep) {
    for (int round = 0; round < nblk - 1; ++round, ++tick) {
      int* flags = act + (tick & 1) * pairs;
      // ---- the pairs' sub-problems: cyclic Jacobi, one entry of S and U a thread
      for (int pr = blockIdx.x; pr < pairs; pr += gridDim.x) {
        int bi, bj;
        tourney(round, pr, nblk, bi, bj);
        auto at = [&](int x) { return x < JW ? bi * JW + x : bj * JW + x - JW; };
        auto couples = [&](R ag, R al, R be) {
          return (ag > Tol<R>::rel * sqrt(fabs(al * be))) && (ag > atol);
        };
        int cur = 0, active = 0;
        S[0][i][j] = ap[(long)at(i) * np + at(j)];
        U[0][i][j] = mkc<R>(i == j ? 1 : 0, 0);
        __syncthreads();
        // nothing to rotate, as in most pairs of the late sweeps: one look instead of 15 steps
        const int live = __syncthreads_or(i < j && couples(modulus<R>(S[0][i][j]), S[0][i][i].x, S[0][j][j].x));
        for (int inner = 0; inner < (live ? kInnerSweeps : 0); ++inner) {
          int any_inner = 0;
          for (int st = 0; st < JS - 1; ++st) {
            int f = 0;
            if (tid < JS / 2) {
              const int a = sa[st][tid], b = sb[st][tid];
              const T g = S[cur][a][b];
              const R ag = modulus<R>(g), al = S[cur][a][a].x, be = S[cur][b][b].x;
              f = couples(ag, al, be);
              R c = 1;
              T o = mkc<R>(0, 0);
              if (f) rotation<R>(g, ag, al, be, c, o);
              // columns: x_a <- c x_a - s conj(e) x_b, x_b <- s e x_a + c x_b
              rc[a] = rc[b] = c;
              ro[a] = mkc<R>(-o.x, o.y);
              ro[b] = o;
              rp[a] = b;
              rp[b] = a;
            }
            if (!__syncthreads_or(f)) continue;
            any_inner = 1;
            const int oi = rp[i], oj = rp[j];
            const R ci = rc[i], cj = rc[j];
            const T xi = cconj(ro[i]), xj = ro[j];
            auto col = [&](T u, T v) {
              T t = cscale(u, cj);
              cfma(t, v, xj);
              return t;
            };
            T ns = cscale(col(S[cur][i][j], S[cur][i][oj]), ci);
            cfma(ns, xi, col(S[cur][oi][j], S[cur][oi][oj]));
            const T nu = col(U[cur][i][j], U[cur][i][oj]);
            S[cur ^ 1][i][j] = ns;
            U[cur ^ 1][i][j] = nu;
            cur ^= 1;
            __syncthreads();
          }
          active |= any_inner;
          if (!any_inner) break;
        }
        // One Newton-Schulz polar step U <- U (3I - U^+U)/2 removes the drift of the
        // accumulated rotations from unitarity (quadratic in the drift), so repeated
        // applications do not scale the spectrum.
        T nu = U[cur][i][j];
        if (active) {
          T acc = mkc<R>(0, 0);
          for (int k = 0; k < JS; ++k) cfma(acc, cconj(U[cur][k][i]), U[cur][k][j]);
          U[cur ^ 1][i][j] = acc;               // G = U^+ U
          __syncthreads();
          nu = cscale(nu, R(1.5));
          for (int k = 0; k < JS; ++k) cfma(nu, cscale(U[cur][i][k], R(-0.5)), U[cur ^ 1][k][j]);
        }
        ug[(long)pr * JS * JS + tid] = nu;
        if (tid == 0) {
          flags[pr] = active;
          if (active) {
            atomicAdd(&counters[sweep & 1], 1);
            atomicAdd(&counters[3], 1);  // active pair-rounds, for the flop count
          }
        }
        __syncthreads();
      }
      grid.sync();
      // ---- the tiles, an item a warp: 16 x JV of V^T, or a 16 x 16 tile of A's upper half; the
      // first ones by place, further ones from a counter, asked for an item ahead
      if (blockIdx.x == 0 && tid == 0) {
        next[(tick + 1) & 1] = gridDim.x * (JT / 32);
        if (round == 0) counters[(sweep + 1) & 1] = 0;
      }
      int any = 0;
      for (int p = tid; p < pairs; p += JT) any |= s_act[p] = (unsigned char)flags[p];
      // no pair rotated: every CTA sees that, and the flags of the next round lie elsewhere
      if (!__syncthreads_or(any)) continue;
      int ahead = 0;
      for (int it = blockIdx.x * (JT / 32) + warp; it < items; it = ahead) {
        if (lane == 0) ahead = atomicAdd(&next[tick & 1], 1);
        ahead = __shfl_sync(0xffffffffu, ahead, 0);
        T acc[8];
        if (it < vitems) {
          const int q = it / vcols, c0 = (it - q * vcols) * JV;
          if (!s_act[q]) continue;
          int bi, bj;
          tourney(round, q, nblk, bi, bj);
          static_assert(JV == 2 * JS, "two tiles an item");
          T* row = vt + (long)(r < JW ? bi * JW + r : bj * JW + r - JW) * np + c0 + 8 * h;
          const bool two = c0 + JS < np;          // np is a multiple of 16
          T x0[8], x1[8], u[8];
          copy8(x0, row);
          if (two) copy8(x1, row + JS);
          copy8(u, ug + (long)q * JS * JS + lane * 8);
          copy8(Uq + lane * 8, u);
          copy8(X + r * JS + 8 * h, x0);
          if (two) copy8(Up + r * JS + 8 * h, x1);
          __syncwarp();
          tile_zero(acc);
          tile_mul(acc, X, h, [&](int k) { return Uq[k * JS + r]; });
          copy8(row, acc);
          if (two) {
            tile_zero(acc);
            tile_mul(acc, Up, h, [&](int k) { return Uq[k * JS + r]; });
            copy8(row + JS, acc);
          }
          __syncwarp();
        } else {
          const int t = it - vitems;
          int q = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
          while (q * (q + 1) / 2 > t) --q;
          while ((q + 1) * (q + 2) / 2 <= t) ++q;
          const int p = t - q * (q + 1) / 2;
          if (!s_act[p] && !s_act[q]) continue;
          int pi, pj, qi, qj;
          tourney(round, p, nblk, pi, pj);
          tourney(round, q, nblk, qi, qj);
          const int prow = r < JW ? pi * JW + r : pj * JW + r - JW;
          const int qrow = r < JW ? qi * JW + r : qj * JW + r - JW;
          T* dst = ap + (long)prow * np + (h ? qj : qi) * JW;
          T u[8], w[8];
          copy8(acc, dst);
          copy8(u, ug + (long)p * JS * JS + lane * 8);
          copy8(w, ug + (long)q * JS * JS + lane * 8);
#pragma unroll
          for (int c = 0; c < 8; ++c) X[r * (JS + 1) + 8 * h + c] = acc[c];
          copy8(Up + lane * 8, u);
          copy8(Uq + lane * 8, w);
          __syncwarp();
          tile_zero(acc);
          tile_mul(acc, Uq, h, [&](int k) { return X[r * (JS + 1) + k]; });
          __syncwarp();
          copy8(X + r * JS + 8 * h, acc);
          __syncwarp();
          tile_zero(acc);
          tile_mul(acc, X, h, [&](int k) { return cconj(Up[k * JS + r]); });
          __syncwarp();
#pragma unroll
          for (int c = 0; c < 8; ++c) X[r * (JS + 1) + 8 * h + c] = acc[c];
          __syncwarp();
          T mir[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) mir[c] = cconj(X[(8 * h + c) * (JS + 1) + r]);
          if (p == q) {
            // its own mirror image: the upper half decides
#pragma unroll
            for (int c = 0; c < 8; ++c)
              if (8 * h + c < r) acc[c] = mir[c];
          } else {
            copy8(ap + (long)qrow * np + (h ? pj : pi) * JW, mir);
          }
          copy8(dst, acc);
          __syncwarp();
        }
      }
      grid.sync();
    }
    int done = (atomicAdd(&counters[sweep & 1], 0) == 0);
    if (done) { ++sweep; break; }
  }
  if (blockIdx.x == 0 && tid == 0) counters[2] = sweep;
}

// Sort the eigenvalues (diagonal of the converged matrix, positions < n) descending into w, their
// positions into perm, which may be ap's own memory.  One CTA, bitonic sort on a power of two.
template <typename R>
__global__ void eig_sort_kernel(int n, int np, const cx<R>* ap, int* perm, double* w) {
  extern __shared__ unsigned char smem_raw[];
  int P = 1;
  while (P < n) P <<= 1;
  double* key = reinterpret_cast<double*>(smem_raw);
  int* val = reinterpret_cast<int*>(key + P);
  __shared__ int s_nan;
  if (threadIdx.x == 0) s_nan = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    double kv = -INFINITY;
    if (i < n) {
      kv = (double)ap[(long)i * np + i].x;
      if (!isfinite(kv)) { s_nan = 1; kv = -INFINITY; }
    }
    key[i] = kv;
    val[i] = i;
  }
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < P; i += blockDim.x) {
        int l = i ^ j;
        if (l > i) {
          bool desc = ((i & k) == 0);
          double ki = key[i], kl = key[l];
          bool sw = desc ? (ki < kl) : (ki > kl);
          if (sw) {
            key[i] = kl; key[l] = ki;
            int t = val[i]; val[i] = val[l]; val[l] = t;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) w[i] = (s_nan && i == 0) ? NAN : key[i];
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const int col = val[k];
    perm[k] = (col >= 0 && col < n) ? col : k;
  }
}

// v[i][k] = vt[perm[k]][i], through shared memory (one CTA gathering single entries took 650 us at
// n = 1350).
template <typename R>
__global__ void __launch_bounds__(256) eig_gather_kernel(int n, int np, const int* __restrict__ perm,
                                                         const cx<R>* __restrict__ vt, cx<R>* v,
                                                         long ldv) {
  __shared__ cx<R> tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, k0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
  for (int q = ty; q < 32; q += 8)
    if (k0 + q < n && i0 + tx < n) tile[q][tx] = vt[(long)perm[k0 + q] * np + i0 + tx];
  __syncthreads();
  for (int q = ty; q < 32; q += 8)
    if (i0 + q < n && k0 + tx < n) v[(long)(i0 + q) * ldv + k0 + tx] = tile[tx][q];
}

// ---------------------------------------------------------------------------------------
// Single-CTA cyclic Jacobi with the whole problem resident in shared memory: the Hermitian
// matrix A and the accumulator V live in shared memory; each round of the round-robin
// ordering rotates np/2 disjoint index pairs at once (GVL sym.schur2 with the complex
// phase factored out): rotation parameters, then one pass over the 2x2 blocks of A (row
// and column rotation together) and the columns of V, with a block barrier after each.  Rotations act on A itself (two-sided),
// so eigenvectors are accurate to eps |A| / gap.  Used for n <= smem_jacobi_max<R>().
// The input (precision RI) is rounded to R on load and the eigenvectors are written in
// precision RO, so a solve of an FP64 matrix in FP32 sweeps needs no conversion launches.
constexpr int SJ_THREADS = 1024;

template <typename R, typename RI, typename RO>
__global__ void __launch_bounds__(SJ_THREADS) jacobi_smem_kernel(int n, int np,
                                                                 const cx<RI>* __restrict__ a,
                                                                 long lda, cx<RO>* v, long ldv,
                                                                 double* w, int* counters,
                                                                 int max_sweeps) {
  using T = cx<R>;
  extern __shared__ unsigned char sj_raw[];
  T* A = reinterpret_cast<T*>(sj_raw);       // row-major np x np
  T* V = A + (size_t)np * np;
  __shared__ R s_anorm;
  __shared__ int s_rot;
  __shared__ double s_key[128];
  __shared__ int s_val[128];
  __shared__ R pc[64], ps[64];
  __shared__ T pe[64];
  __shared__ int pp[64], pq[64], pf[64];
  const int tid = threadIdx.x, lane = tid & 31;
  const int nthr = blockDim.x;
  const int half = np / 2;
  for (int e = tid; e < np * np; e += nthr) {
    int i = e / np, j = e % np;
    T z = mkc<R>(0, 0);
    if (i < n && j < n) {
      const cx<RI> t = a[(long)i * lda + j];
      z = mkc<R>((R)t.x, (R)t.y);
    }
    A[e] = z;
    V[e] = mkc<R>(i == j ? 1 : 0, 0);
  }
  if (tid == 0) s_anorm = 0;
  __syncthreads();
  if (tid < 32) {
    R part = 0;
    for (int i = lane; i < n; i += 32) part += fabs(A[(size_t)i * np + i].x);
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) s_anorm = part;
  }
  __syncthreads();
  const R atol = Tol<R>::abs * s_anorm;
  int sweep = 0;
  int total_rot = 0;   // thread 0: rotations applied (pair-rounds with an active pair)
  for (; sweep < max_sweeps; ++sweep) {
    if (tid == 0) s_rot = 0;
    __syncthreads();
    for (int r = 0; r < np - 1; ++r) {
      for (int k = tid; k < half; k += nthr) {
        int p, q;
        tourney(r, k, np, p, q);
        if (p > q) { int t = p; p = q; q = t; }
        T g = A[(size_t)p * np + q];
        R ag = sqrt(cabs2(g));
        R al = A[(size_t)p * np + p].x, be = A[(size_t)q * np + q].x;
        int f = (ag > Tol<R>::rel * sqrt(fabs(al * be))) && (ag > atol);
        pp[k] = p; pq[k] = q; pf[k] = f;
        if (f) {
          R tau = (be - al) / (2 * ag);
          R t = (tau >= 0 ? R(1) : R(-1)) / (fabs(tau) + sqrt(R(1) + tau * tau));
          R c = R(1) / sqrt(R(1) + t * t);
          pc[k] = c; ps[k] = t * c;
          pe[k] = mkc<R>(g.x / ag, g.y / ag);
          atomicAdd(&s_rot, 1);
        }
      }
      __syncthreads();
      // The disjoint pairs partition the indices, so A' = J^+ A J splits into independent
      // 2x2 blocks: block (a, b) holds rows {p_a, q_a} x columns {p_b, q_b} and needs only
      // the rotations of pairs a and b.  One pass updates every block (and the columns of
      // V), with no barrier between the row and the column rotation.
      for (int e = tid; e < half * half; e += nthr) {
        const int ka = e / half, kb = e - ka * half;
        const int fa = pf[ka], fb = pf[kb];
        if (!fa && !fb) continue;
        const int pa = pp[ka], qa = pq[ka], pb = pp[kb], qb = pq[kb];
        const R ca = fa ? pc[ka] : R(1), sa = fa ? ps[ka] : R(0);
        const R cb = fb ? pc[kb] : R(1), sb = fb ? ps[kb] : R(0);
        const T ea = fa ? pe[ka] : mkc<R>(1, 0), eb = fb ? pe[kb] : mkc<R>(1, 0);
        T* rp = A + (size_t)pa * np;
        T* rq = A + (size_t)qa * np;
        const T x0 = rp[pb], x1 = rp[qb], y0 = rq[pb], y1 = rq[qb];
        // rows (pair a): p' = c x - s e y, q' = s x conj(e) + c y
        const T u0 = csub(cscale(x0, ca), cscale(cmul(ea, y0), sa));
        const T u1 = csub(cscale(x1, ca), cscale(cmul(ea, y1), sa));
        const T w0 = cadd(cscale(cmulc(x0, ea), sa), cscale(y0, ca));
        const T w1 = cadd(cscale(cmulc(x1, ea), sa), cscale(y1, ca));
        // columns (pair b): p' = c x - s y conj(e), q' = s x e + c y
        rp[pb] = csub(cscale(u0, cb), cscale(cmulc(u1, eb), sb));
        rp[qb] = cadd(cscale(cmul(u0, eb), sb), cscale(u1, cb));
        rq[pb] = csub(cscale(w0, cb), cscale(cmulc(w1, eb), sb));
        rq[qb] = cadd(cscale(cmul(w0, eb), sb), cscale(w1, cb));
      }
      for (int e = tid; e < np * half; e += nthr) {
        const int row = e / half, kb = e - row * half;
        if (!pf[kb]) continue;
        const int p = pp[kb], q = pq[kb];
        const R c = pc[kb], sn = ps[kb];
        const T ee = pe[kb];
        T* vr = V + (size_t)row * np;
        const T x = vr[p], y = vr[q];
        vr[p] = csub(cscale(x, c), cscale(cmulc(y, ee), sn));
        vr[q] = cadd(cscale(cmul(x, ee), sn), cscale(y, c));
      }
      __syncthreads();
    }
    if (tid == 0) total_rot += s_rot;
    // every thread reads the count before thread 0 resets it for the next sweep (a thread
    // that read the reset value would leave the loop alone and break the block barriers)
    const int rotated = s_rot;
    __syncthreads();
    if (rotated == 0) { ++sweep; break; }
  }
  // eigenvalues = diagonal; sort descending (n <= 128)
  __shared__ int s_nan;
  if (tid == 0) s_nan = 0;
  __syncthreads();
  int P = 2;
  while (P < n) P <<= 1;                       // n <= 118 -> P <= 128
  for (int c = tid; c < P; c += nthr) {
    double key = -INFINITY;
    if (c < n) {
      key = (double)A[(size_t)c * np + c].x;
      if (!isfinite(key)) { s_nan = 1; key = -INFINITY; }
    }
    s_key[c] = key;
    s_val[c] = c;
  }
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int c = tid; c < P; c += nthr) {
        int l = c ^ j;
        if (l > c) {
          bool desc = ((c & k) == 0);
          double ki = s_key[c], kl = s_key[l];
          if (desc ? (ki < kl) : (ki > kl)) {
            s_key[c] = kl; s_key[l] = ki;
            int t = s_val[c]; s_val[c] = s_val[l]; s_val[l] = t;
          }
        }
      }
      __syncthreads();
    }
  }
  // a non-finite input is reported as a NaN leading eigenvalue (callers flag it); the
  // gather index is clamped so a broken permutation can never leave the arrays
  for (int i = tid; i < n; i += nthr) w[i] = (s_nan && i == 0) ? NAN : s_key[i];
  for (int e = tid; e < n * n; e += nthr) {
    int i = e / n, k = e % n;
    int col = s_val[k];
    col = (col >= 0 && col < n) ? col : k;
    const T t = V[(size_t)i * np + col];
    v[(long)i * ldv + k] = mkc<RO>((RO)t.x, (RO)t.y);
  }
  if (tid == 0 && counters) {
    counters[2] = sweep;
    counters[3] = total_rot;   // each rotates 2 rows and 2 columns of A and 2 columns of V
  }
}

// ---------------------------------------------------------------------------------------
// FP32 sweeps of a graded Hermitian PSD matrix A = D C D (C of unit diagonal and moderate
// condition, D spanning decades), as L^+ L of a pivoted Cholesky factor L is.  Rotations are
// taken while |a_pq| > kGradedRel sqrt(a_pp a_qq), whatever the size of the pair, so every
// eigenpair is resolved relative to its own size (Demmel and Veselic, "Jacobi's method is
// more accurate than QR", 1992): one solve covers the whole spectrum, where an absolute
// threshold covers two decades of it.  The sweeps stop after one whose largest
// |a_pq| / sqrt(a_pp a_qq) was below kGradedStop: convergence is quadratic, so about its
// square is left, which the FP64 refinement removes (L^+ L of the update's Grams, r = 13..73:
// 3 to 5 sweeps, mixing angles of 1e-6 to 5e-5 left, 1e-10 after one refinement pass).
//
// One CTA; a round touches every 2 x 2 block, so it is bound by shared-memory traffic and issue
// slots of one SM, and below ~60 rows by the latency of its two phases.  Hence:
//  - only the blocks above the diagonal exist;
//  - the matrix is stored by the seats of the round-robin tournament, not by index: pair k sits
//    on seats T_k and B_k, block (a, b) is the same four words in every round, and after a
//    rotation each entry is written to its seats of the next round (players move one seat).  A
//    thread keeps its blocks, whose addresses it computes once; four planes (T or B row, T or B
//    column) make every access contiguous across lanes;
//  - the eigenvectors are not accumulated here: the rotations go to a log, which
//    rot_apply_kernel replays on the rows of the identity on other SMs.  Without the
//    accumulator a matrix of 168 fits the shared memory of an SM (118 with it).
// By index, with looked-up pairs and mirrored writes, a round of n = 118 took 1.2 us.  The pairs
// have warps of their own: a warp with blocks as well made all others wait for its rotations.
// In place of one-sided FP64 sweeps on the factor (3.6 ms a Gram on one SM's FP64 pipe) and of
// the levels of the mixed solver (5 rounds of ~9 launches): 40 atoms, two layers in FP64 719 ->
// 84 ms, 100 atoms, three layers in the mixed tensor-core form 1488 -> 791 ms.
constexpr float kGradedRel = 2e-6f;
constexpr float kGradedStop = 1e-3f;
constexpr int kGradedHalf = kGradedMax / 2;
constexpr int kGradedThreads = 512;      // block threads, besides the warps of the pairs ...
constexpr int kGradedFew = 416;          // ... and with more than 4 blocks each (128 registers)

// Seats: T_k = (0, k), B_k = (1, k).  T_0 stays; T_k moves to T_{k-1}, T_1 to B_0, B_k to
// B_{k+1} and the last B to the last T.
__device__ __forceinline__ void next_seat(int half, int& t, int& k) {
  if (half == 1 || (t == 0 && k == 0)) return;
  if (t == 0) {
    if (k == 1) { t = 1; k = 0; } else { --k; }
  } else {
    if (k == half - 1) t = 0; else ++k;
  }
}
// Player on a seat at the start of a sweep (m = 2 half - 1 moving players, player m on T_0).
__device__ __forceinline__ int seat_player(int m, int t, int k) {
  return t == 0 ? (k == 0 ? m : k) : (k == 0 ? 0 : m - k);
}
// Where the entry of seats (ta, ka), (tb, kb) goes after a round: its word (below 2^15), with bit
// 15 set when it is stored conjugated.  Words: plane (row seat type, column seat type) of half x
// half, then the pairs' own entries g_k = (T_k, B_k).
__device__ __forceinline__ unsigned seat_target(int half, int ta, int ka, int tb, int kb) {
  next_seat(half, ta, ka);
  next_seat(half, tb, kb);
  const unsigned conj = 0x8000u;
  const int P = half * half;
  if (ka == kb) return (4 * P + ka) | (ta == 0 ? 0u : conj);
  if (ka < kb) return (ta * 2 + tb) * P + ka * half + kb;
  return ((tb * 2 + ta) * P + kb * half + ka) | conj;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void seat_store(float2* A, unsigned target, float2 z) {
  z.y = __uint_as_float(__float_as_uint(z.y) ^ ((target << 16) & 0x80000000u));
  A[target & 0x7fffu] = z;
}

// log: (c, Re s e, Im s e, rotated) of pair k of round i < *rounds at log[i * np / 2 + k];
// perm[i]: column of the i-th largest diagonal entry.  A diagonal that is not finite is left
// for the caller to find in the refined eigenvalues.
template <int IT>   // blocks of a thread
__global__ void __launch_bounds__(IT > 4 ? kGradedFew + 96 : kGradedThreads + 96) jacobi_graded_kernel(
    int n, int np, const double2* __restrict__ a, long lda, float4* log, int* rounds, int* perm,
    int max_sweeps) {
  extern __shared__ float2 gj_a[];   // four planes, then g
  __shared__ float4 s_rot[kGradedHalf];
  __shared__ float s_d[2][kGradedHalf];   // diagonal of T_k, B_k
  __shared__ double s_red[kGradedThreads / 32 + 3];
  __shared__ unsigned s_max;
  __shared__ float s_key[kGradedMax];
  const int tid = threadIdx.x, lane = tid & 31, nthr = blockDim.x;
  const int half = np / 2, m = np - 1, P = half * half;
  // a power of two brings the largest diagonal entry near 2^30: FP32 then holds the squares
  // of entries 16 decades below it
  double dm = 0.0;
  for (int i = tid; i < n; i += nthr) dm = fmax(dm, a[(long)i * lda + i].x);
  for (int o = 16; o > 0; o >>= 1) dm = fmax(dm, __shfl_xor_sync(0xffffffffu, dm, o));
  if (lane == 0) s_red[tid >> 5] = dm;
  __syncthreads();
  for (int k = 0; k < (nthr >> 5); ++k) dm = fmax(dm, s_red[k]);
  const double sc = (dm > 0.0 && isfinite(dm)) ? ldexp(1.0, 30 - ilogb(dm)) : 1.0;
  auto entry = [&](int i, int j) {
    if (i >= n || j >= n) return make_float2(0.f, 0.f);
    const double2 t = a[(long)i * lda + j];
    return make_float2((float)(t.x * sc), (float)(t.y * sc));
  };
  for (int e = tid; e < 4 * P; e += nthr) {
    const int pl = e / P, ka = (e % P) / half, kb = e % half;
    if (ka < kb) gj_a[e] = entry(seat_player(m, pl >> 1, ka), seat_player(m, pl & 1, kb));
  }
  // the first warps take a pair a lane and nothing else: the others wait for their rotations
  const int pt = (half + 31) / 32 * 32;
  unsigned own_to = 0;                        // where the pair's own entry goes
  float *al_to = nullptr, *be_to = nullptr;   // and its diagonal entries
  if (tid < half) {
    const int p = seat_player(m, 0, tid), q = seat_player(m, 1, tid);
    gj_a[4 * P + tid] = entry(p, q);
    s_d[0][tid] = entry(p, p).x;
    s_d[1][tid] = entry(q, q).x;
    own_to = seat_target(half, 0, tid, 1, tid);
    int t = 0, k = tid;
    next_seat(half, t, k);
    al_to = &s_d[t][k];
    t = 1;
    k = tid;
    next_seat(half, t, k);
    be_to = &s_d[t][k];
  }
  // the blocks (ka < kb) of this thread: row i of the folded triangle holds the blocks of pair
  // i and then those of pair half - 1 - i
  const int nb = half * (half - 1) / 2;
  int ab[IT];          // ka | kb << 8, -1 for none; word ka half + kb in every plane
  unsigned to[IT][2];  // targets of the four words, 16 bits each
#pragma unroll
  for (int t = 0; t < IT; ++t) {
    const int e = tid - pt + t * (nthr - pt);
    ab[t] = -1;
    if (tid >= pt && e < nb) {
      const int i = e / (half - 1), j = e - i * (half - 1);
      const bool lo = j < half - 1 - i;
      const int ka = lo ? i : half - 1 - i, kb = lo ? i + 1 + j : half - i + (j - (half - 1 - i));
      ab[t] = ka | (kb << 8);
      for (int q = 0; q < 2; ++q)
        to[t][q] = seat_target(half, q, ka, 0, kb) | (seat_target(half, q, ka, 1, kb) << 16);
    }
  }
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    float worst = 0.f;   // the sweep's largest |g|^2 / (al be) of this thread's pair
    if (tid == 0) s_max = 0u;
    __syncthreads();
    for (int r = 0; r < m; ++r) {
      // phase 1: the rotation of every pair; the other warps fetch their blocks meanwhile
      float2 x[IT][4];
      float4 rot = make_float4(1.f, 0.f, 0.f, 0.f);
      float al = 0.f, be = 0.f, g2 = 0.f;
      float2 g = make_float2(0.f, 0.f);
      if (tid < pt) {
        if (tid < half) {
          g = gj_a[4 * P + tid];
          al = s_d[0][tid];
          be = s_d[1][tid];
          g2 = cabs2(g);
          if (g2 > kGradedRel * kGradedRel * al * be && g2 > 0.f) {
            // with d = be - al and s = sqrt(d^2 + 4 |g|^2): c^2 = (|d| + s) / 2s and
            // s e = sign(d) g / (s c).  Approximate roots (a few ulp): their error is that of
            // the accumulated rotations' rounding, which the refinement removes.
            const float d = be - al, s2 = fmaf(d, d, 4.f * g2);
            const float rs = rsqrt_approx(s2), w = fmaf(s2, rs, fabsf(d)), c2 = 0.5f * w * rs;
            const float ic = rsqrt_approx(c2), k = copysignf(rs * ic, d);
            rot = make_float4(c2 * ic, k * g.x, k * g.y, 1.f);
          }
          s_rot[tid] = rot;
        }
      } else {
#pragma unroll
        for (int t = 0; t < IT; ++t)
          if (ab[t] >= 0) {
            const float2* w = gj_a + (ab[t] & 255) * half + (ab[t] >> 8);
#pragma unroll
            for (int q = 0; q < 4; ++q) x[t][q] = w[q * P];
          }
      }
      __syncthreads();
      // phase 2: rotate, and everything to its next seat
      if (tid < half) {
        if (rot.w != 0.f) {
          const float d = be - al, s2 = fmaf(d, d, 4.f * g2);
          const float dt = copysignf(__fdividef(2.f * g2, fmaf(s2, rsqrt_approx(s2), fabsf(d))), d);
          const float pr = al * be;
          worst = fmaxf(worst, pr > 0.f ? __fdividef(g2, pr) : 1.f);
          al -= dt;
          be += dt;
          g = make_float2(0.f, 0.f);
        }
        *al_to = al;
        *be_to = be;
        seat_store(gj_a, own_to, g);
        log[(long)(sweep * m + r) * half + tid] = rot;
      }
#pragma unroll
      for (int t = 0; t < IT; ++t) {
        if (ab[t] < 0) continue;
        const float4 ra = s_rot[ab[t] & 255], rb = s_rot[ab[t] >> 8];
        if (ra.w != 0.f || rb.w != 0.f) {
          const float2 sa = make_float2(ra.y, ra.z), sb = make_float2(rb.y, rb.z);
          // rows (pair a): T' = c T - s e B, B' = s conj(e) T + c B
          const float2 u0 = csub(cscale(x[t][0], ra.x), cmul(sa, x[t][2]));
          const float2 u1 = csub(cscale(x[t][1], ra.x), cmul(sa, x[t][3]));
          const float2 w0 = cadd(cmulc(x[t][0], sa), cscale(x[t][2], ra.x));
          const float2 w1 = cadd(cmulc(x[t][1], sa), cscale(x[t][3], ra.x));
          // columns (pair b): T' = c T - s conj(e) B, B' = s e T + c B
          x[t][0] = csub(cscale(u0, rb.x), cmulc(u1, sb));
          x[t][1] = cadd(cmul(u0, sb), cscale(u1, rb.x));
          x[t][2] = csub(cscale(w0, rb.x), cmulc(w1, sb));
          x[t][3] = cadd(cmul(w0, sb), cscale(w1, rb.x));
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) seat_store(gj_a, to[t][q >> 1] >> (16 * (q & 1)), x[t][q]);
      }
      __syncthreads();
    }
    if (worst > 0.f) atomicMax(&s_max, __float_as_uint(worst));   // positive floats order as integers
    __syncthreads();
    const float mx = __uint_as_float(s_max);
    __syncthreads();
    if (!(mx > kGradedStop * kGradedStop)) { ++sweep; break; }
  }
  // whole sweeps bring every player back to its first seat
  if (tid < half) {
    const int p = seat_player(m, 0, tid), q = seat_player(m, 1, tid);
    if (p < n) s_key[p] = s_d[0][tid];
    if (q < n) s_key[q] = s_d[1][tid];
  }
  for (int i = tid; i < n; i += nthr) perm[i] = i;   // valid whatever the keys (NaN: ranks collide)
  __syncthreads();
  for (int i = tid; i < n; i += nthr) {
    const float key = s_key[i];
    int rank = 0;
    for (int k = 0; k < n; ++k) rank += s_key[k] > key || (!(s_key[k] < key) && k < i);
    perm[rank < n ? rank : n - 1] = i;
  }
  if (tid == 0) *rounds = sweep * m;
}

// Rows of the accumulated rotations, V = J_1 J_2 ... : the log replayed on rows of the identity
// (V's rows are independent), one warp per row, kRotWarps rows of a CTA sharing the log, which
// comes into shared memory kRotChunk rounds at a time, the next chunk in flight while the
// present one is applied.  Bound by the latency of a round (two columns read, rotated and
// written back): 37 us at n = 60, where fetching each round's rotations one round ahead from L2
// took 96 us.  Columns are written in the order of perm, widened to FP64.
constexpr int kRotWarps = 4;
constexpr int kRotChunk = 16;
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
template <int KP>   // pairs of a lane
__global__ void __launch_bounds__(32 * kRotWarps) rot_apply_kernel(int n, int np,
                                                                   const float4* __restrict__ log,
                                                                   const int* __restrict__ nrounds,
                                                                   const int* __restrict__ perm,
                                                                   double2* z, long ldz) {
  __shared__ float2 rows[kRotWarps][kGradedMax];
  __shared__ __align__(16) float4 buf[2][kRotChunk][32 * KP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = blockIdx.x * kRotWarps + warp;
  const bool live = row < n;
  float2* v = rows[warp];
  const int half = np / 2, m = np - 1, rounds = *nrounds;
  for (int c = lane; c < np; c += 32) v[c] = make_float2(c == row ? 1.f : 0.f, 0.f);
  auto fetch = [&](int i0, int b) {
    const int cnt = min(kRotChunk, rounds - i0);
    for (int e = threadIdx.x; e < cnt * half; e += 32 * kRotWarps) {
      const int i = e / half, k = e - i * half;
      cp_async16(&buf[b][i][k], &log[(long)(i0 + i) * half + k]);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (rounds > 0) fetch(0, 0);
  for (int i0 = 0, b = 0; i0 < rounds; i0 += kRotChunk, b ^= 1) {
    if (i0 + kRotChunk < rounds) {
      fetch(i0 + kRotChunk, b ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const int cnt = min(kRotChunk, rounds - i0);
    int r = i0 % m;
    for (int i = 0; live && i < cnt; ++i, r = r + 1 == m ? 0 : r + 1) {
#pragma unroll
      for (int t = 0; t < KP; ++t) {
        const int k = lane + 32 * t;
        if (k >= half) continue;
        const float4 rot = buf[b][i][k];
        if (rot.w == 0.f) continue;
        int p = k == 0 ? m : r + k, q = k == 0 ? r : r - k;   // the players of T_k and B_k
        if (k && p >= m) p -= m;
        if (q < 0) q += m;
        const float2 x = v[p], y = v[q], se = make_float2(rot.y, rot.z);
        v[p] = csub(cscale(x, rot.x), cmulc(y, se));
        v[q] = cadd(cmul(x, se), cscale(y, rot.x));
      }
      __syncwarp();
    }
    __syncthreads();   // the chunk is free for the fetch after the next
  }
  if (!live) return;
  for (int c = lane; c < n; c += 32) {
    const float2 x = v[perm[c]];
    z[(long)row * ldz + c] = make_double2((double)x.x, (double)x.y);
  }
}

template <typename R>
constexpr int smem_jacobi_max() { return sizeof(R) == 8 ? 84 : 118; }

inline int padded_n(int n) {
  int nblk = (n + JW - 1) / JW;
  if (nblk < 2) nblk = 2;
  if (nblk & 1) ++nblk;
  return nblk * JW;
}

template <typename R, typename RI, typename RO>
cudaError_t smem_jacobi_launch(cudaStream_t st, int n, const cx<RI>* a, long lda, cx<RO>* v,
                               long ldv, double* w, int* counters, int max_sweeps) {
  const int np2 = n + (n & 1);
  const size_t sm = 2ull * np2 * np2 * sizeof(cx<R>);
  const int smax = smem_jacobi_max<R>() + (smem_jacobi_max<R>() & 1);
  // once per instantiation (a thread-safe static initialiser)
  static const cudaError_t attr = cudaFuncSetAttribute(
      jacobi_smem_kernel<R, RI, RO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
      (int)(2ull * smax * smax * sizeof(cx<R>)));
  MPDO_CUDA_TRY(attr);
  count_launch();
  const int thr = std::min(SJ_THREADS, std::max(64, ((np2 / 2) * np2 + 31) / 32 * 32));
  jacobi_smem_kernel<R, RI, RO><<<1, thr, sm, st>>>(n, np2, a, lda, v, ldv, w, counters,
                                                    max_sweeps);
  return cudaGetLastError();
}

}  // namespace

template <typename RI, typename RO>
cudaError_t heig_smem_f32(cudaStream_t st, int n, const cx<RI>* a, long lda, cx<RO>* v, long ldv,
                          double* w, int* counters, int max_sweeps) {
  if (n <= 0) return cudaSuccess;
  if (n > kSmemJacobiMaxF32) return cudaErrorInvalidValue;
  return smem_jacobi_launch<float, RI, RO>(st, n, a, lda, v, ldv, w, counters, max_sweeps);
}
template cudaError_t heig_smem_f32<double, double>(cudaStream_t, int, const double2*, long,
                                                   double2*, long, double*, int*, int);
template cudaError_t heig_smem_f32<double, float>(cudaStream_t, int, const double2*, long,
                                                  float2*, long, double*, int*, int);

size_t graded_log_bytes(int n) {
  const size_t np = n + (n & 1);
  return kGradedSweeps * (np - 1) * (np / 2) * sizeof(float4) + 256 + (np + 8) * sizeof(int);
}

cudaError_t heig_graded_f32(cudaStream_t st, int n, const double2* a, long lda, double2* z,
                            long ldz, void* mem) {
  if (n < 1 || n > kGradedMax) return cudaErrorInvalidValue;
  const int np = n + (n & 1), half = np / 2, rounds = kGradedSweeps * (np - 1);
  float4* log = static_cast<float4*>(mem);
  int* perm = reinterpret_cast<int*>(log + (size_t)rounds * half);
  int* nrounds = perm + np;
  const size_t sm = ((size_t)np * np + half) * sizeof(float2);
  const int nb = half * (half - 1) / 2;
  const int bthr = nb > 4 * kGradedThreads ? kGradedFew
                                           : std::min(kGradedThreads, std::max(32, (nb + 31) / 32 * 32));
  const int it = (nb + bthr - 1) / bthr;   // at most 9 (nb <= 3486)
  const int thr = bthr + (half + 31) / 32 * 32;
  auto launch = [&](auto kern) -> cudaError_t {
    kern<<<1, thr, sm, st>>>(n, np, a, lda, log, nrounds, perm, kGradedSweeps);
    return cudaGetLastError();
  };
  // opt in to the largest size, once per instantiation
  static const cudaError_t attr = [] {
    constexpr int kMaxSmem = (kGradedMax * kGradedMax + kGradedHalf) * (int)sizeof(float2);
    auto set = [](auto kern) {
      return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    };
    cudaError_t e = set(jacobi_graded_kernel<1>);
    if (e == cudaSuccess) e = set(jacobi_graded_kernel<2>);
    if (e == cudaSuccess) e = set(jacobi_graded_kernel<4>);
    if (e == cudaSuccess) e = set(jacobi_graded_kernel<9>);
    return e;
  }();
  MPDO_CUDA_TRY(attr);
  count_launch(2);
  MPDO_CUDA_TRY(it <= 1   ? launch(jacobi_graded_kernel<1>)
                : it <= 2 ? launch(jacobi_graded_kernel<2>)
                : it <= 4 ? launch(jacobi_graded_kernel<4>)
                          : launch(jacobi_graded_kernel<9>));
  auto apply = [&](auto kern) {
    kern<<<(n + kRotWarps - 1) / kRotWarps, 32 * kRotWarps, 0, st>>>(n, np, log, nrounds, perm, z, ldz);
  };
  if (half <= 32) apply(rot_apply_kernel<1>);
  else if (half <= 64) apply(rot_apply_kernel<2>);
  else apply(rot_apply_kernel<3>);
  return cudaGetLastError();
}

int eig_padded_n(int n) { return padded_n(n); }

// Executed rotation flops per unit of counters[3] (8 real flops per complex element update):
// the one-CTA kernel counts applied rotations (each updates 2 rows and 2 columns of A and 2
// columns of V, n elements each: 6 n updates); the block kernel counts active pair-rounds
// (2 x 16 x 16 x n_pad complex multiply-adds: both sides of half of A, and V).
double eig_flops_per_count(int n, bool fp64) {
  const int smax = fp64 ? 84 : 118;
  if (n <= smax) return 8.0 * 6.0 * (double)(n + (n & 1));
  return 8.0 * 2 * 256 * (double)padded_n(n);
}

template <typename R>
size_t eig_work_bytes(int n_cap) {
  size_t np = padded_n(n_cap);
  return (2 * np * np + np * JS) * sizeof(cx<R>) + 256 + np * sizeof(int);
}

template <typename R>
void eig_work_bind(EigWork<R>& w, void* base, int n_cap) {
  size_t np = padded_n(n_cap);
  w.n_cap = n_cap;
  w.ap = reinterpret_cast<cx<R>*>(base);
  w.vp = w.ap + np * np;
  w.ug = w.vp + np * np;
  w.counters = reinterpret_cast<int*>(w.ug + np * JS);
  w.act = w.counters + 64;
}

template <typename R>
cudaError_t heig(cudaStream_t st, int n, const cx<R>* a, long lda, cx<R>* v, long ldv,
                 double* w, EigWork<R>& work, int max_sweeps) {
  if (n <= 0) return cudaSuccess;
  if (n > work.n_cap) return cudaErrorInvalidValue;
  if (n <= smem_jacobi_max<R>())
    return smem_jacobi_launch<R, R, R>(st, n, a, lda, v, ldv, w, work.counters, max_sweeps);
  int np = padded_n(n);
  int nblk = np / JW;
  long total = (long)np * np;
  int blocks = (int)((total + 255) / 256);
  if (blocks > 4096) blocks = 4096;
  count_launch(4);
  pad_copy_kernel<R><<<blocks, 256, 0, st>>>(n, np, a, lda, work.ap, work.vp, work.counters);
  MPDO_CUDA_TRY(cudaGetLastError());
  // as many CTAs as the device holds at once, or as there are items for their warps
  static const int resident = [] {
    int dev = 0, sms = 0, per = 0;
    if (cudaFuncSetAttribute(jacobi_coop_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)coop_smem<R>()) != cudaSuccess ||
        cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, jacobi_coop_kernel<R>, JT,
                                                      coop_smem<R>()) != cudaSuccess)
      return 0;
    return sms * per;
  }();
  const int pairs = nblk / 2;
  if (resident < 1 || pairs > kMaxPairs) return cudaErrorInvalidConfiguration;
  const long items = (long)pairs * ((np + JV - 1) / JV) + (long)pairs * (pairs + 1) / 2;
  const int grid = (int)std::min<long>(resident, std::max<long>(pairs, (items + JT / 32 - 1) / (JT / 32)));
  int* next = work.counters + 8;   // items handed out in even and odd rounds
  void* args[] = {&np, &nblk, &work.ap, &work.vp, &work.ug, &work.act, &next, &work.counters,
                  &max_sweeps};
  MPDO_CUDA_TRY(cudaLaunchCooperativeKernel((void*)jacobi_coop_kernel<R>, dim3(grid), dim3(JT), args,
                                            coop_smem<R>(), st));
  int P = 1;
  while (P < n) P <<= 1;
  size_t sm = (size_t)P * (sizeof(double) + sizeof(int));
  // sort keys beyond n = 2048 exceed the default 48 KB of shared memory (with the kernel's
  // static flag): opt in up to n = 16384, 192 KB (once per instantiation)
  static const cudaError_t fattr = cudaFuncSetAttribute(
      eig_sort_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
      (int)(16384 * (sizeof(double) + sizeof(int))));
  MPDO_CUDA_TRY(fattr);
  if (P > 16384) return cudaErrorInvalidValue;
  int* perm = reinterpret_cast<int*>(work.ap);   // the matrix is read before its memory is written
  eig_sort_kernel<R><<<1, 1024, sm, st>>>(n, np, work.ap, perm, w);
  MPDO_CUDA_TRY(cudaGetLastError());
  eig_gather_kernel<R><<<dim3((n + 31) / 32, (n + 31) / 32), 256, 0, st>>>(n, np, perm, work.vp, v,
                                                                          ldv);
  return cudaGetLastError();
}

template size_t eig_work_bytes<double>(int);
template size_t eig_work_bytes<float>(int);
template void eig_work_bind<double>(EigWork<double>&, void*, int);
template void eig_work_bind<float>(EigWork<float>&, void*, int);
template cudaError_t heig<double>(cudaStream_t, int, const double2*, long, double2*, long,
                                  double*, EigWork<double>&, int);
template cudaError_t heig<float>(cudaStream_t, int, const float2*, long, float2*, long,
                                 double*, EigWork<float>&, int);

}  // namespace mpdo

// ---------------------------------------------------------------------------------------
// Allocation-free eigensolver entry point (mpdo_heig_noalloc, declared in mpdo.h).
// Its scratch -- the padded working matrix, the eigenvector accumulator and the sweep
// counters -- is one file-scope device array sized for n <= MPDO_HEIG_NOALLOC_NMAX, so a
// call performs no device allocation.  Host code cannot use the array's name as a device
// address; the address is looked up with cudaGetSymbolAddress once per device (first call
// with that device current) and passed to the kernels.
namespace {
constexpr int kNoAllocNMax = MPDO_HEIG_NOALLOC_NMAX;
constexpr size_t kNoAllocBytes =
    (2ull * kNoAllocNMax + 16) * kNoAllocNMax * sizeof(double2) + 256 + kNoAllocNMax * sizeof(int);
static_assert(kNoAllocNMax % (2 * mpdo::JW) == 0, "maximum must be a whole number of block pairs");
static __device__ __align__(256) unsigned char g_heig_scratch[kNoAllocBytes];
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
// per device: the CUDA context the address was looked up in, and the address.  A device
// reset (or a primary context destroyed and created again) loads the module anew, possibly
// elsewhere, so the address is looked up again whenever the current context changes.
void* g_scratch_ctx[kMaxDevices] = {};
void* g_scratch_addr[kMaxDevices] = {};
using CtxGetCurrentFn = CUresult (*)(CUcontext*);
void* current_context() {
  static CtxGetCurrentFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return static_cast<CtxGetCurrentFn>(nullptr);
    }
    return reinterpret_cast<CtxGetCurrentFn>(p);
  }();
  CUcontext c = nullptr;
  if (fn) fn(&c);
  return c;
}
}  // namespace

namespace mpdo {
void set_global_error(const char* msg);
}

extern "C" int mpdo_heig_noalloc(int prec, int n, void* a, void* v, double* w, int* sweeps,
                                 void* stream) {
  using namespace mpdo;
  if (prec != 0 && prec != 1) {
    set_global_error("mpdo_heig_noalloc: prec must be 0 (complex128) or 1 (complex64)");
    return MPDO_ERR_ARG;
  }
  if (n < 1 || n > kNoAllocNMax) {
    set_global_error("mpdo_heig_noalloc: n must be in 1..MPDO_HEIG_NOALLOC_NMAX (192)");
    return MPDO_ERR_ARG;
  }
  if (!a || !v || !w) {
    set_global_error("mpdo_heig_noalloc: null matrix, vector or eigenvalue pointer");
    return MPDO_ERR_ARG;
  }
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    set_global_error("mpdo_heig_noalloc: no usable current CUDA device");
    return MPDO_ERR_CUDA;
  }
  void* base = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    void* ctx = current_context();
    if (!g_scratch_addr[dev] || ctx != g_scratch_ctx[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_heig_scratch);
      if (e != cudaSuccess || !p) {
        set_global_error("mpdo_heig_noalloc: cudaGetSymbolAddress of the scratch array failed");
        return MPDO_ERR_CUDA;
      }
      g_scratch_addr[dev] = p;
      g_scratch_ctx[dev] = current_context();
    }
    base = g_scratch_addr[dev];
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int* counters;
  if (prec == 0) {
    EigWork<double> wk;
    eig_work_bind<double>(wk, base, kNoAllocNMax);
    counters = wk.counters;
    e = heig<double>(st, n, static_cast<const double2*>(a), n, static_cast<double2*>(v), n, w,
                     wk, 30);
  } else {
    EigWork<float> wk;
    eig_work_bind<float>(wk, base, kNoAllocNMax);
    counters = wk.counters;
    e = heig<float>(st, n, static_cast<const float2*>(a), n, static_cast<float2*>(v), n, w, wk,
                    20);
  }
  if (e == cudaSuccess && sweeps) {
    e = cudaMemcpyAsync(sweeps, counters + 2, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e != cudaSuccess) {
    set_global_error(cudaGetErrorString(e));
    return MPDO_ERR_CUDA;
  }
  return MPDO_OK;
}
