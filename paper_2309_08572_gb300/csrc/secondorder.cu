// Two-copy environments of the second-order observables in a real basis.
//
// A site of rho, X[(s,s')][(a,b)][(r,r')] = sum_k A[a,s,k,r] conj(A[b,s',k,r']), turns into its
// conjugate when the members of all three pairs are exchanged.  In the orthonormal Hermitian basis
// of each pair -- e_pp; (e_pq + e_qp)/sqrt2 at (p < q); i (e_pq - e_qp)/sqrt2 at (p > q), its
// conjugate on the pair (r,r') -- X is therefore real: nine real dl^2 x dr^2 matrices M_mu.  A
// contracted bond is a plain real dot product; two crossed copies (tr rho^2) are
// sum_mu M_mu (x) M_mu, the diagonal ones (collision) the three mu with s = s', the trace is the
// sum of these three, and the environment E of two copies is real and symmetric.  One site then
// takes 9 (l^2 r + l r^2 / 2) real multiply-adds with l = dl^2, r = dr^2 (and a third of that for
// the collision), against 9 (l^2 r + l r^2) complex ones, four times as many, in the matrices' own
// basis; it needs no reordering passes between the products.
#include "common.cuh"
#include "internal.h"
#include "kernels.h"

namespace mpdo {
namespace {

// M[mu][alpha][beta] from the site operator rf[(a,s,r)][(b,s',r')]: the sum over the exchanges of
// the pairs whose members differ, one pair's exchange taken as twice the real part.  Bound by the
// reads of rf from L2 (up to four per output).
template <typename R>
__global__ void herm_site_kernel(int dl, int dr, const cx<R>* __restrict__ rf, R* __restrict__ m) {
  const long l2 = (long)dl * dl, r2 = (long)dr * dr, rows = 3L * dl * dr;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < 9 * l2 * r2;
       e += (long)gridDim.x * blockDim.x) {
    const int be = (int)(e % r2), al = (int)(e / r2 % l2), mu = (int)(e / (r2 * l2));
    const int x[3] = {mu / 3, al / dl, be / dr}, y[3] = {mu % 3, al % dl, be % dr};
    int bits[3], nd = 0, q = 0;   // pairs whose members differ; of these, antisymmetric ones
    R sc = R(1);
    int sgn = 1;
    for (int i = 0; i < 3; ++i) {
      bits[i] = -1;
      if (x[i] != y[i]) {
        bits[i] = nd - 1;         // its bit in the sum; -1 of the first: not exchanged
        nd++;
        sc *= R(0.70710678118654752440);
        if (x[i] > y[i]) {
          ++q;
          if (i == 2) sgn = -sgn;
        }
      }
    }
    if (nd > 0) sc *= R(2);
    R sum = R(0);
    for (int w = 0; w < (nd > 1 ? 1 << (nd - 1) : 1); ++w) {
      int u[3], v[3], s = sgn;
      for (int i = 0; i < 3; ++i) {
        const bool ex = bits[i] >= 0 && (w >> bits[i] & 1);
        u[i] = ex ? y[i] : x[i];
        v[i] = ex ? x[i] : y[i];
        if (ex && x[i] > y[i]) s = -s;
      }
      const cx<R> t = rf[(((long)u[1] * 3 + u[0]) * dr + u[2]) * rows +
                         ((long)v[1] * 3 + v[0]) * dr + v[2]];
      const R c = (q & 1) ? t.y : t.x;                 // Re(i^q t) up to its sign
      sum += (s < 0) != (q == 1 || q == 2) ? -c : c;
    }
    m[e] = sum * sc;
  }
}

// Real product C[b] = A[b] B[b] of the sweeps, b < 12: the nine M_mu with the crossed environment
// and the three of the diagonal with the diagonal one.  Entry (i, k) of A[b] is at i ai + k ak,
// (k, j) of B[b] at k bk + j bj, C row-major; offsets of a batch entry: its matrix M (mb), the
// environment (eb: crossed or diagonal) or a workspace (wb).  sym: C[b] is symmetric and its tiles
// below the diagonal are left out.
//
// Bound by the FP64 pipe (half an FMA per clock and SM quarter): a tile of 32 x 32 on four warps
// keeps a warp on every quarter with six shared loads for eight FMAs (512 clocks) and gives each
// SM several tiles at D = 16 (192 tiles of a 64 x 64 split would leave 40 of 152 SMs two of them
// and the rest one).  FP32 has the rate to want 64 x 64.
constexpr int kSoK = 16, kSoThreads = 128;
struct SoSide {
  const void *m, *cross, *diag;   // M, and per batch entry the other operand
  long mstride, wstride;          // entries of one M_mu; of one workspace matrix (0: environments)
};
template <typename R, int TM, int TN>
__global__ void __launch_bounds__(kSoThreads) so_product_kernel(int m, int n, int k, SoSide a,
                                                                long ai, long ak, SoSide b,
                                                                long bk, long bj, R* c, int sym) {
  constexpr int BM = 16 * TM, BN = 8 * TN;
  const int i0 = blockIdx.y * BM, j0 = blockIdx.x * BN, z = blockIdx.z;
  if (sym && j0 + BN <= i0) return;
  const int mu = z < 9 ? z : 4 * (z - 9);
  auto base = [&](const SoSide& s) {
    if (s.m) return static_cast<const R*>(s.m) + mu * s.mstride;
    return static_cast<const R*>(z < 9 ? s.cross : s.diag) + z * s.wstride;
  };
  const R *A = base(a), *B = base(b);
  __shared__ R As[2][kSoK][BM + 1], Bs[2][kSoK][BN + 1];
  const int tid = threadIdx.x, tx = tid % 8, ty = tid / 8;
  constexpr int NA = BM * kSoK / kSoThreads, NB = BN * kSoK / kSoThreads;
  R ra[NA], rb[NB];
  // neighbouring threads along the operand's contiguous axis
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = tid + q * kSoThreads, kk = ak == 1 ? e % kSoK : e / BM,
                i = ak == 1 ? e / kSoK : e % BM;
      ra[q] = i0 + i < m && k0 + kk < k ? A[(long)(i0 + i) * ai + (long)(k0 + kk) * ak] : R(0);
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = tid + q * kSoThreads, kk = bk == 1 ? e % kSoK : e / BN,
                j = bk == 1 ? e / kSoK : e % BN;
      rb[q] = j0 + j < n && k0 + kk < k ? B[(long)(k0 + kk) * bk + (long)(j0 + j) * bj] : R(0);
    }
  };
  auto store = [&](int s) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = tid + q * kSoThreads;
      As[s][ak == 1 ? e % kSoK : e / BM][ak == 1 ? e / kSoK : e % BM] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = tid + q * kSoThreads;
      Bs[s][bk == 1 ? e % kSoK : e / BN][bk == 1 ? e / kSoK : e % BN] = rb[q];
    }
  };
  R acc[TM][TN] = {};
  load(0);
  store(0);
  __syncthreads();
  int s = 0;
  for (int k0 = 0; k0 < k; k0 += kSoK, s ^= 1) {
    if (k0 + kSoK < k) load(k0 + kSoK);
#pragma unroll
    for (int kk = 0; kk < kSoK; ++kk) {
      R x[TM], y[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) x[i] = As[s][kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) y[j] = Bs[s][kk][tx + 8 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(x[i], y[j], acc[i][j]);
    }
    if (k0 + kSoK < k) store(s ^ 1);
    __syncthreads();
  }
  R* C = c + (long)z * m * n;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int r = i0 + ty + 16 * i, q = j0 + tx + 8 * j;
      if (r < m && q < n) C[(long)r * n + q] = acc[i][j];
    }
}

// The new environments from the products' upper halves: nine terms of the crossed one, three of
// the diagonal one, in order.
template <typename R>
__global__ void so_finish_kernel(long n, const R* __restrict__ p, R* cross, R* diag) {
  const long n2 = n * n;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < 2 * n2;
       e += (long)gridDim.x * blockDim.x) {
    const bool d = e >= n2;
    const long f = d ? e - n2 : e, i = f / n, j = f % n, q = i <= j ? f : j * n + i;
    R t = R(0);
    for (int z = d ? 9 : 0; z < (d ? 12 : 9); ++z) t += p[z * n2 + q];
    (d ? diag : cross)[f] = t;
  }
}

// The traced environment through a site: out[beta] = sum_alpha e[alpha] Tr[alpha][beta] (left) or
// out[alpha] = sum_beta Tr[alpha][beta] e[beta], Tr = M_0 + M_4 + M_8.  32 outputs a CTA, each
// sum over eight warps (left) or the lanes of a warp (right), added in a fixed order: one thread a
// sum would be a chain of up to 3 dl^2 FP64 operations.
template <typename R>
__global__ void __launch_bounds__(256) so_trace_kernel(int left, int l2, int r2,
                                                       const R* __restrict__ m,
                                                       const R* __restrict__ e, R* out) {
  __shared__ R part[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, o0 = blockIdx.x * 32;
  if (left) {
    R t = R(0);
    if (o0 + lane < r2)
      for (int mu = 0; mu < 9; mu += 4)
        for (int a = warp; a < l2; a += 8)
          t = fma(e[a], m[((long)mu * l2 + a) * r2 + o0 + lane], t);
    part[warp][lane] = t;
    __syncthreads();
    if (warp == 0 && o0 + lane < r2) {
      for (int w = 1; w < 8; ++w) t += part[w][lane];
      out[o0 + lane] = t;
    }
  } else {
    for (int o = o0 + warp; o < min(o0 + 32, l2); o += 8) {
      R t = R(0);
      for (int mu = 0; mu < 9; mu += 4)
        for (int b = lane; b < r2; b += 32) t = fma(m[((long)mu * l2 + o) * r2 + b], e[b], t);
      for (int s = 16; s > 0; s >>= 1) t += __shfl_xor_sync(0xffffffffu, t, s);
      if (lane == 0) out[o] = t;
    }
  }
}

// tr rho^2, tr rho_L^2, tr rho_R^2, the collision sum and tr rho from the environments at the
// cut, in FP64: parts of a fixed set of entries per thread, added in a fixed order.
constexpr int kSoDotBlocks = 64;
template <typename R>
__global__ void __launch_bounds__(256) so_dot_kernel(int n, const R* __restrict__ cl,
                                                     const R* __restrict__ cr,
                                                     const R* __restrict__ dl,
                                                     const R* __restrict__ dr,
                                                     const R* __restrict__ el,
                                                     const R* __restrict__ er, double* parts) {
  __shared__ double red[8][5];
  double t[5] = {};
  const long n2 = (long)n * n;
  for (long e = blockIdx.x * 256L + threadIdx.x; e < n2; e += 256L * gridDim.x) {
    const long i = e / n, j = e % n;
    const double x = (double)cl[e], y = (double)cr[e];
    t[0] += x * y;
    t[1] += x * ((double)er[i] * er[j]);
    t[2] += y * ((double)el[i] * el[j]);
    t[3] += (double)dl[e] * dr[e];
    if (i == j) t[4] += (double)el[i] * er[i];
  }
  for (int q = 0; q < 5; ++q)
    for (int o = 16; o > 0; o >>= 1) t[q] += __shfl_xor_sync(0xffffffffu, t[q], o);
  if ((threadIdx.x & 31) == 0)
    for (int q = 0; q < 5; ++q) red[threadIdx.x >> 5][q] = t[q];
  __syncthreads();
  if (threadIdx.x < 5) {
    double s = 0;
    for (int w = 0; w < 8; ++w) s += red[w][threadIdx.x];
    parts[blockIdx.x * 5 + threadIdx.x] = s;
  }
}
// one warp per result
__global__ void so_dot_sum_kernel(const double* __restrict__ parts, double* out) {
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  double t = 0;
  for (int b = lane; b < kSoDotBlocks; b += 32) t += parts[b * 5 + q];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) out[q] = t;
}

template <typename R>
cudaError_t so_product(cudaStream_t st, int m, int n, int k, const SoSide& a, long ai, long ak,
                       const SoSide& b, long bk, long bj, R* c, int sym) {
  constexpr int TM = sizeof(R) == 8 ? 2 : 4, TN = sizeof(R) == 8 ? 4 : 8;
  const dim3 grid((n + 8 * TN - 1) / (8 * TN), (m + 16 * TM - 1) / (16 * TM), 12);
  count_launch();
  so_product_kernel<R, TM, TN><<<grid, kSoThreads, 0, st>>>(m, n, k, a, ai, ak, b, bk, bj, c, sym);
  return cudaGetLastError();
}

}  // namespace

template <typename R>
cudaError_t so_site(cudaStream_t st, int dl, int dr, const cx<R>* rf, R* m) {
  const long total = 9L * dl * dl * dr * dr;
  count_launch();
  herm_site_kernel<R><<<(int)std::min<long>((total + 255) / 256, 16384), 256, 0, st>>>(dl, dr, rf, m);
  return cudaGetLastError();
}

template <typename R>
cudaError_t so_step(cudaStream_t st, bool left, int dl, int dr, const R* m, R* cross, R* diag,
                    const R* e, R* eout, R* w, R* p) {
  const int l2 = dl * dl, r2 = dr * dr;
  const long ms = (long)l2 * r2;
  const SoSide M{m, nullptr, nullptr, ms, 0}, E{nullptr, cross, diag, 0, 0};
  const SoSide W{nullptr, w, w, 0, ms};
  if (left) {
    // W_mu = M_mu^T E (r2 x l2), then E' += W_mu M_mu
    MPDO_CUDA_TRY(so_product<R>(st, r2, l2, l2, M, 1, r2, E, l2, 1, w, 0));
    MPDO_CUDA_TRY(so_product<R>(st, r2, r2, l2, W, l2, 1, M, r2, 1, p, 1));
  } else {
    // W_mu = M_mu E (l2 x r2), then E' += W_mu M_mu^T
    MPDO_CUDA_TRY(so_product<R>(st, l2, r2, r2, M, r2, 1, E, r2, 1, w, 0));
    MPDO_CUDA_TRY(so_product<R>(st, l2, l2, r2, W, r2, 1, M, 1, r2, p, 1));
  }
  const long n = left ? r2 : l2;
  count_launch(2);
  so_finish_kernel<R><<<(int)std::min<long>((2 * n * n + 255) / 256, 16384), 256, 0, st>>>(
      n, p, cross, diag);
  so_trace_kernel<R><<<(int)((n + 31) / 32), 256, 0, st>>>(left ? 1 : 0, l2, r2, m, e, eout);
  return cudaGetLastError();
}

template <typename R>
cudaError_t so_dots(cudaStream_t st, int n, const R* cl, const R* cr, const R* dl, const R* dr,
                    const R* el, const R* er, double* parts, double* out) {
  count_launch(2);
  so_dot_kernel<R><<<kSoDotBlocks, 256, 0, st>>>(n, cl, cr, dl, dr, el, er, parts);
  so_dot_sum_kernel<<<1, 32 * 5, 0, st>>>(parts, out);
  return cudaGetLastError();
}

#define SO_INST(R)                                                                              \
  template cudaError_t so_site<R>(cudaStream_t, int, int, const cx<R>*, R*);                    \
  template cudaError_t so_step<R>(cudaStream_t, bool, int, int, const R*, R*, R*, const R*, R*, \
                                  R*, R*);                                                      \
  template cudaError_t so_dots<R>(cudaStream_t, int, const R*, const R*, const R*, const R*,    \
                                  const R*, const R*, double*, double*);
SO_INST(float)
SO_INST(double)
}  // namespace mpdo
