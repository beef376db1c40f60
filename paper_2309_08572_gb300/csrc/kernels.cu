// Elementwise and small kernels of the MPDO update, observables and sampling.
// Every kernel here is memory- or latency-bound; the contractions are in gemm.cu.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace mpdo {
namespace {

inline int nblocks(long total, int threads = 256, int cap = 16384) {
  long b = (total + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (int)b;
}

// out[i0][i2][i1][i3] = in[i0][i1][i2][i3]
template <typename T>
__global__ void swap12_kernel(long n0, long n1, long n2, long n3, const T* __restrict__ in,
                              T* __restrict__ out) {
  long total = n0 * n1 * n2 * n3;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    long i3 = e % n3;
    long r = e / n3;
    long i1 = r % n1;
    r /= n1;
    long i2 = r % n2;
    long i0 = r / n2;
    // e enumerates the OUTPUT [i0][i2][i1][i3]
    out[e] = in[((i0 * n1 + i1) * n2 + i2) * n3 + i3];
  }
}

// site [l][s][k][r] -> [r][s][k][l]
template <typename T>
__global__ void reverse_site_kernel(int dl, int d, int k, int dr, const T* __restrict__ in,
                                    T* __restrict__ out) {
  long total = (long)dl * d * k * dr;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    // output index [r][s][k][l]
    long l = e % dl;
    long t = e / dl;
    long kk = t % k;
    t /= k;
    long s = t % d;
    long r = t / d;
    out[e] = in[((l * d + s) * k + kk) * dr + r];
  }
}

// A[l][s][k][r] <- sum_s' U[s][s'] A[l][s'][k][r]
template <typename R>
__global__ void one_site_kernel(int dl, int k, int dr, const cx<R>* __restrict__ u,
                                cx<R>* a) {
  long plane = (long)k * dr;
  long total = (long)dl * plane;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    long l = e / plane, q = e % plane;
    cx<R>* base = a + l * 3 * plane + q;
    cx<R> x0 = base[0], x1 = base[plane], x2 = base[2 * plane];
    for (int s = 0; s < 3; ++s) {
      cx<R> acc = mkc<R>(0, 0);
      cfma(acc, u[s * 3 + 0], x0);
      cfma(acc, u[s * 3 + 1], x1);
      cfma(acc, u[s * 3 + 2], x2);
      base[s * plane] = acc;
    }
  }
}

template <typename R>
__global__ void product_state_kernel(cx<R> v0, cx<R> v1, cx<R> v2, cx<R>* base, long stride,
                                     int n) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    base[i * stride + 0] = v0;
    base[i * stride + 1] = v1;
    base[i * stride + 2] = v2;
  }
}

// rs/irs from the left-Gram spectrum sigma (descending): numerical rank cut.
template <typename R>
__global__ void gram_mask_kernel(int n, const double* __restrict__ sig, double gtol,
                                 R* rs, R* irs, StepScalars* sc) {
  double s0 = sig[0];
  bool bad = !(s0 > 0.0) || !isfinite(s0);
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    double s = sig[c];
    if (!bad && s > gtol * s0) {
      rs[c] = (R)sqrt(s);
      irs[c] = (R)(1.0 / sqrt(s));
    } else {
      rs[c] = 0;
      irs[c] = 0;
    }
  }
  if (threadIdx.x == 0 && bad) sc->flags |= 1;
}

// R[c][x] = rs[c] conj(V[x][c]); Vs[x][c] = V[x][c] irs[c]; Vr[x][c] = V[x][c] rs[c]
template <typename R>
__global__ void gram_factor_kernel(int n, const cx<R>* __restrict__ v, const R* __restrict__ rs,
                                   const R* __restrict__ irs, cx<R>* rmat, cx<R>* vs, cx<R>* vr) {
  long total = (long)n * n;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    int x = (int)(e / n), c = (int)(e % n);
    cx<R> val = v[e];
    vs[e] = cscale(val, irs[c]);
    vr[e] = cscale(val, rs[c]);
    rmat[(long)c * n + x] = cscale(cconj(val), rs[c]);
  }
}

// Phi[(S,s,b),(S2,s2,b2)] = sum_{t,t2} C[(S,s,t),(S2,s2,t2)] Gj[(b,t),(b2,t2)]
template <typename R>
__global__ void build_phi_kernel(int dm, const cx<R>* __restrict__ ct,
                                 const cx<R>* __restrict__ gj, cx<R>* phi) {
  long n = 9L * dm;
  long total = n * n;
  long ldg = 3L * dm;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    long row = e / n, col = e % n;
    int ss = (int)(row / dm), b = (int)(row % dm);     // ss = S*3 + s
    int ss2 = (int)(col / dm), b2 = (int)(col % dm);
    cx<R> acc = mkc<R>(0, 0);
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
      for (int t2 = 0; t2 < 3; ++t2)
        cfma(acc, ct[(ss * 3 + t) * 27 + ss2 * 3 + t2], gj[(b * 3 + t) * ldg + b2 * 3 + t2]);
    phi[e] = acc;
  }
}

// Sum over the CTA of 256 threads in a fixed order; every thread gets it.  red: 8 doubles.
__device__ __forceinline__ double block_sum(double x, double* red) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  return ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
}
// Length of the leading run of x[0..n) above thr (n if all are); all threads of the CTA.
__device__ __forceinline__ int leading_run(const double* x, int n, double thr, int* s_min) {
  __syncthreads();
  if (threadIdx.x == 0) *s_min = n;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    if (!(x[i] > thr)) {
      atomicMin(s_min, i);
      break;
    }
  __syncthreads();
  return *s_min;
}

// Bond cut on the spectrum lam (descending, n): keep <= chi values above htol*lam0.
// The total weight is the trace of the matrix itself (noise-free in expectation), not
// the sum of the positive computed eigenvalues, which is biased upward by the noise floor.
template <typename R>
__global__ void __launch_bounds__(256) bond_select_kernel(int n, const double* __restrict__ lam,
                                                          const cx<R>* __restrict__ hm, long ldh,
                                                          double htol, int chi, StepScalars* sc,
                                                          DevStats* st) {
  __shared__ double red[8];
  __shared__ int s_keep;
  const double l0 = lam[0];
  const bool bad = !(l0 > 0.0) || !isfinite(l0);
  int keep = bad ? 1 : leading_run(lam, min(n, chi), htol * l0, &s_keep);
  if (keep < 1) keep = 1;
  double t = 0, kp = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    t += (double)hm[(long)i * ldh + i].x;
    if (i < keep) kp += lam[i] > 0 ? lam[i] : 0.0;
  }
  const double tot = block_sum(t, red), kept = block_sum(kp, red);
  if (threadIdx.x == 0) {
    sc->keep = keep;
    sc->tot = tot;
    sc->kept = kept;
    sc->renorm = (kept > 0) ? sqrt(tot / kept) : 0.0;
    if (bad || !(kept > 0) || !isfinite(tot)) sc->flags |= 1;
    st->disc_bond_w += (tot > 0) ? (tot - kept) / tot : 0.0;
    if (keep > st->chi_used_max) st->chi_used_max = keep;
    st->n_updates += 1;
  }
}

// Q[(b',T,m),(b,t)] = renorm * sum_{S,s} conj(W[(S,s,b)][b']) E[m][(S,T),(s,t)]
template <typename R>
__global__ void make_q_kernel(int dm, int keep, int m_ops, const cx<R>* __restrict__ w,
                              const cx<R>* __restrict__ e, const StepScalars* sc, cx<R>* q) {
  long cols = 3L * dm;
  long rows = (long)keep * 3 * m_ops;
  long total = rows * cols;
  R ren = (R)sc->renorm;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total;
       idx += (long)gridDim.x * blockDim.x) {
    long row = idx / cols, col = idx % cols;
    int m = (int)(row % m_ops);
    long r2 = row / m_ops;
    int T = (int)(r2 % 3);
    int bp = (int)(r2 / 3);
    int b = (int)(col / 3), t = (int)(col % 3);
    const cx<R>* em = e + (long)m * 81;
    cx<R> acc = mkc<R>(0, 0);
#pragma unroll
    for (int S = 0; S < 3; ++S)
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        cx<R> wv = w[((long)(S * 3 + s) * dm + b) * keep + bp];
        cfma(acc, cconj(wv), em[(S * 3 + T) * 9 + s * 3 + t]);
      }
    q[idx] = cscale(acc, ren);
  }
}

// Inner-index cut + purity-preserving truncation (Sec. III.D Eqs. xiformula / ppt with
// T = 1, P = identity; theta = 0 when infeasible; clamp negatives; keep the trace).
// Writes f[k] = sqrt(Lambda~_k / w_k) for k < kk.
// The CTAs of a fixed grid (kNormBlocks) form partial sums of tr W (diagonal real parts) and
// ||W||_F^2 over the ntr x ntr matrix wm (= sum w^2 for the Hermitian W, whatever part of its
// spectrum was resolved); the one that finishes last (a ticket; nobody waits) adds them in a
// fixed order and selects, its lanes sharing the weights.  FP64 operations take ~64 clocks each
// here: one thread walking through the weights, with two tangents of arc cosines, took 28 us
// (K = 8) where this takes about a third; tan(acos c) is sqrt(1 - c^2) / c.
constexpr int kNormBlocks = 64;
template <typename R>
__global__ void __launch_bounds__(256) kraus_select_kernel(
    int n, const double* __restrict__ w, const cx<R>* __restrict__ wm, int ntr, double* parts,
    unsigned int* ticket, double kcut, int kmax, int use_ppt, double* f, StepScalars* sc,
    DevStats* st, double* trace) {
  __shared__ double red[8];
  __shared__ int s_kk, s_last;
  const int tid = threadIdx.x, lane = tid & 31;
  {
    double t = 0, f2 = 0;
    const long total = (long)ntr * ntr;
    for (long e = blockIdx.x * 256L + tid; e < total; e += 256L * kNormBlocks) {
      const cx<R> v = wm[e];
      f2 += (double)v.x * v.x + (double)v.y * v.y;
      if (e / ntr == e % ntr) t += (double)v.x;
    }
    t = block_sum(t, red);
    f2 = block_sum(f2, red);
    if (tid == 0) {
      parts[2 * blockIdx.x] = t;
      parts[2 * blockIdx.x + 1] = f2;
      __threadfence();
      s_last = atomicAdd(ticket, 1u) == kNormBlocks - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) *ticket = 0u;
  }
  const double w0 = w[0] > 0 ? w[0] : 0.0;
  const bool bad = !(w0 > 0.0) || !isfinite(w0);
  int kk = bad ? 1 : leading_run(w, min(n, kmax), kcut * kcut * w0, &s_kk);
  if (kk < 1) kk = 1;
  if (tid >= 32) return;
  auto warp_sum = [](double x) {
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  };
  const double sum = warp_sum(__ldcg(&parts[2 * lane]) + __ldcg(&parts[2 * lane + 64]));
  const double sq = warp_sum(__ldcg(&parts[2 * lane + 1]) + __ldcg(&parts[2 * lane + 65]));
  double sumk = 0, sqk = 0;
  for (int i = lane; i < kk; i += 32) {
    const double v = w[i] > 0 ? w[i] : 0.0;
    sumk += v;
    sqk += v * v;
  }
  sumk = warp_sum(sumk);
  sqk = warp_sum(sqk);
  // The trace the truncation keeps (reading A2) is carried in FP64 across updates: the
  // channel multiplies it by tr(theta')/tr(theta) of this block (bond total sc->tot over
  // sc->trpre, both FP64 sums of the same stored tensors), so rounding of the stored
  // tensors and of the products that form the new centre does not accumulate in the norm.
  const bool carried = trace && sc->trpre > 0 && sc->tot > 0 && isfinite(*trace);
  const double target = carried ? *trace * (sc->tot / sc->trpre) : sum;
  __syncwarp();
  if (carried && lane == 0) *trace = target;

  double theta = 0.0, x = 0.0, shift = 0.0;
  int infeas = 0, clamped = 0;
  const bool ppt = use_ppt && !bad;
  if (ppt) {
    const double nl = sqrt(sq), nlp = sqrt(sqk), ntp = sqrt((double)kk);
    const double cos_sig = fmin(1.0, sumk / (nlp * ntp));
    double c = sum / (nl * ntp);   // cos theta = |T| cos phi / |T'|
    if (c > 1.0) { infeas = 1; c = 1.0; }
    theta = acos(c);
    if (cos_sig < 1.0)
      x = sqrt((1.0 - c) * (1.0 + c)) / c * (cos_sig / sqrt((1.0 - cos_sig) * (1.0 + cos_sig))) - 1.0;
    shift = nlp * cos_sig / ntp;
  }
  // Lambda~ before its scale
  auto value = [&](int i) {
    const double lp = w[i] > 0 ? w[i] : 0.0;
    return ppt ? lp + x * (lp - shift) : lp;
  };
  double lsum = 0;
  for (int i = lane; i < kk; i += 32) {
    const double v = value(i);
    if (v < 0) ++clamped; else lsum += v;
  }
  lsum = warp_sum(lsum);
  clamped = (int)__reduce_add_sync(0xffffffffu, (unsigned)clamped);
  const double scale = lsum > 0 ? target / lsum : 0.0;
  for (int i = lane; i < kk; i += 32) {
    const double wi = w[i], v = value(i);
    f[i] = wi > 0 && v > 0 ? sqrt(v * scale / wi) : 0.0;
  }
  if (lane > 0) return;
  sc->kkeep = kk;
  sc->ktot = sum;
  sc->theta = theta;
  sc->infeasible = infeas;
  sc->clamped = clamped;
  if (bad) sc->flags |= 1;
  st->disc_kraus_w += (sum > 0) ? (sum - sumk) / sum : 0.0;
  if (use_ppt && theta < st->ppt_theta_min) st->ppt_theta_min = theta;
  st->ppt_infeasible += infeas;
  st->ppt_clamped += clamped;
  if (kk > st->k_used_max) st->k_used_max = kk;
}

// ||theta||^2 of the two-site block before the channel, from the two Gram matrices:
// sum_{s,b,b'} G_i[(s,b'),(s,b)] sum_t G_j[(b,t),(b',t)]  (G_i, G_j: 3D x 3D, index s*D+b
// resp. b*3+t), accumulated in FP64 into sc->trpre.  One CTA.
template <typename R>
__global__ void trace_pre_kernel(int dm, const cx<R>* __restrict__ gi, const cx<R>* __restrict__ gj,
                                 StepScalars* sc) {
  __shared__ double red[256];
  const long n3 = 3L * dm;
  double t = 0;
  for (long e = threadIdx.x; e < (long)dm * dm; e += blockDim.x) {
    const int b = (int)(e / dm), bp = (int)(e % dm);
    double gtr = 0, gti = 0;
    for (int q = 0; q < 3; ++q) {
      const cx<R> v = gj[(long)(b * 3 + q) * n3 + bp * 3 + q];
      gtr += (double)v.x;
      gti += (double)v.y;
    }
    for (int s = 0; s < 3; ++s) {
      const cx<R> v = gi[(long)(s * dm + bp) * n3 + s * dm + b];
      t += (double)v.x * gtr - (double)v.y * gti;
    }
  }
  red[threadIdx.x] = t;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    sc->trpre = red[0];
    sc->flags = 0;   // the update's flags start afresh
  }
}

// out = sum |a_e|^2 over n complex entries, in FP64 (one CTA; the norm of the centre site).
template <typename R>
__global__ void sumsq_kernel(long n, const cx<R>* __restrict__ a, double* out) {
  __shared__ double red[256];
  double t = 0;
  for (long e = threadIdx.x; e < n; e += blockDim.x) {
    const cx<R> v = a[e];
    t += (double)v.x * v.x + (double)v.y * v.y;
  }
  red[threadIdx.x] = t;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

// out = in with its 6 axes reordered: out axis i is in axis perm[i] (dims of in: d[0..5]).
template <typename T>
__global__ void permute6_kernel(const T* __restrict__ in, T* __restrict__ out, int d0, int d1,
                                int d2, int d3, int d4, int d5, int p0, int p1, int p2, int p3,
                                int p4, int p5) {
  const int d[6] = {d0, d1, d2, d3, d4, d5};
  const int p[6] = {p0, p1, p2, p3, p4, p5};
  long st[6];
  st[5] = 1;
  for (int i = 4; i >= 0; --i) st[i] = st[i + 1] * d[i + 1];
  const long total = st[0] * d[0];
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    long rem = e, off = 0;
    for (int i = 5; i >= 0; --i) {
      const int od = d[p[i]];
      const long idx = rem % od;
      rem /= od;
      off += idx * st[p[i]];
    }
    out[e] = in[off];
  }
}

// R[(a,b)][s][s'][(r,r')] (a, b < dl; s, s' < 3; r, r' < dr): mode 0 keeps it, mode 1 zeroes
// the blocks s != s' (the diagonal transfer of the collision probability), mode 2 writes the
// trace over s into tr[(a,b)][(r,r')] instead.
template <typename T>
__global__ void rho_site_kernel(long dl2, long dr2, T* r, T* tr, int mode) {
  const long total = dl2 * 9 * dr2;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const long q = e % dr2, ss = (e / dr2) % 9, ab = e / (9 * dr2);
    const int s = (int)(ss / 3), s2 = (int)(ss % 3);
    if (mode == 1) {
      if (s != s2) { r[e].x = 0; r[e].y = 0; }
    } else if (mode == 2 && s == 0 && s2 == 0) {
      T v = r[e];
      const T v1 = r[e + 4 * dr2], v2 = r[e + 8 * dr2];
      v.x += v1.x + v2.x;
      v.y += v1.y + v2.y;
      tr[ab * dr2 + q] = v;
    }
  }
}

// Deterministic FP64 contractions of environments into parts[blockIdx]: mode 0:
// sum_e Re(x[e] y[e]); mode 1: sum_{(ab),(cd)} Re(c[(ab),(cd)] u[ab] u[cd]) with n2 = dim of
// (ab).  A second pass (one CTA) adds the parts in order.
template <typename T>
__global__ void __launch_bounds__(256) env_dot_kernel(long n2, const T* __restrict__ x,
                                                      const T* __restrict__ y, int mode,
                                                      double* parts) {
  __shared__ double red[256];
  double t = 0;
  const long total = mode == 0 ? n2 : n2 * n2;
  for (long e = blockIdx.x * 256L + threadIdx.x; e < total; e += 256L * gridDim.x) {
    if (mode == 0) {
      t += (double)x[e].x * y[e].x - (double)x[e].y * y[e].y;
    } else {
      const long i = e / n2, j = e % n2;
      // c[(ab),(cd)] u[ab] u[cd]
      const double ur = (double)y[i].x * y[j].x - (double)y[i].y * y[j].y;
      const double ui = (double)y[i].x * y[j].y + (double)y[i].y * y[j].x;
      t += (double)x[e].x * ur - (double)x[e].y * ui;
    }
  }
  red[threadIdx.x] = t;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) parts[blockIdx.x] = red[0];
}
__global__ void sum_parts_kernel(int n, const double* parts, double* out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double s = 0;
    for (int i = 0; i < n; ++i) s += parts[i];
    *out = s;
  }
}

// Vks[kappa][k] = V[kappa][k] * f[k], k < kk (V has leading dimension ldv)
template <typename R, typename RO>
__global__ void scale_vk_kernel(int n, int kk, const cx<R>* __restrict__ v, long ldv,
                                const double* __restrict__ f, cx<RO>* out) {
  long total = (long)n * kk;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    int r = (int)(e / kk), c = (int)(e % kk);
    cx<R> t = cscale(v[(long)r * ldv + c], (R)f[c]);
    out[e] = mkc<RO>((RO)t.x, (RO)t.y);
  }
}

// Energy automaton, one-site step: from F0, FZ, F1 (= env^T A for the three states)
// form G0 = P F0, GZ = Z F0, G1 = P F1 + (-h X - bJ Z) F0 - J Z FZ on the s index.
// Layout of F*: [l'][s][k][r] with plane = k*dr; proj = 1 uses P = |0><0|+|1><1|,
// proj = 0 uses the identity.  Six automata are stacked: [0..2] projected, [3..5] raw.
template <typename R>
__global__ void energy_mix_kernel(int dl, int plane, const cx<R>* __restrict__ f, long fstride,
                                  cx<R>* g, long gstride, double J, double hx, double bz) {
  long total = (long)dl * plane;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    long l = e / plane, q = e % plane;
    long off = l * 3 * plane + q;
    for (int proj = 1; proj >= 0; --proj) {
      int base = proj ? 0 : 3;
      const cx<R>* f0 = f + (base + 0) * fstride + off;
      const cx<R>* fz = f + (base + 1) * fstride + off;
      const cx<R>* f1 = f + (base + 2) * fstride + off;
      cx<R>* g0 = g + (base + 0) * gstride + off;
      cx<R>* gz = g + (base + 1) * gstride + off;
      cx<R>* g1 = g + (base + 2) * gstride + off;
      cx<R> a0 = f0[0], a1 = f0[plane], a2 = f0[2 * plane];
      cx<R> z0 = fz[0], z1 = fz[plane];
      cx<R> b0 = f1[0], b1 = f1[plane], b2 = f1[2 * plane];
      // G0
      g0[0] = a0;
      g0[plane] = a1;
      g0[2 * plane] = proj ? mkc<R>(0, 0) : a2;
      // GZ: Z = diag(1, -1, 0)
      gz[0] = a0;
      gz[plane] = cscale(a1, R(-1));
      gz[2 * plane] = mkc<R>(0, 0);
      // G1 = P F1 + (-h X - bJ Z) F0 - J Z FZ  (X swaps s' <- s on the qubit levels)
      R h = (R)hx, bj = (R)(bz * J), jj = (R)J;
      cx<R> o0 = cadd(b0, cadd(cscale(a1, -h), cscale(a0, -bj)));
      o0 = cadd(o0, cscale(z0, -jj));
      cx<R> o1 = cadd(b1, cadd(cscale(a0, -h), cscale(a1, bj)));
      o1 = cadd(o1, cscale(z1, jj));
      g1[0] = o0;
      g1[plane] = o1;
      g1[2 * plane] = proj ? mkc<R>(0, 0) : b2;
    }
  }
}

__global__ void energy_init_kernel(long env, double2* e) {
  const int a = threadIdx.x;
  if (a < 6) e[a * env] = make_double2(a % 3 == 0 ? 1.0 : 0.0, 0.0);
}
__global__ void energy_result_kernel(long env, const double2* __restrict__ e,
                                     const double* __restrict__ trace, double* res) {
  const int a = threadIdx.x;
  if (a < 6) res[a] = e[a * env].x;
  if (a == 6) res[6] = *trace;
}

// ----------------------------------------------------------------- sampling
__device__ __forceinline__ void philox_round(uint32_t& c0, uint32_t& c1, uint32_t& c2,
                                             uint32_t& c3, uint32_t k0, uint32_t k1) {
  const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
  uint32_t hi0 = __umulhi(M0, c0), lo0 = M0 * c0;
  uint32_t hi1 = __umulhi(M1, c2), lo1 = M1 * c2;
  uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
  c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
}

// Philox4x32-10 (Salmon et al., SC'11) on counter (site, sample, 0, 0), key = seed.
__device__ double philox_uniform(uint64_t seed, uint32_t sample, uint32_t site) {
  uint32_t c0 = site, c1 = sample, c2 = 0, c3 = 0;
  uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  for (int r = 0; r < 10; ++r) {
    if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    philox_round(c0, c1, c2, c3, k0, k1);
  }
  uint64_t v = ((uint64_t)c0 << 21) | (uint64_t)(c1 >> 11);
  return (double)v * 0x1.0p-53;
}

// q[smp][v] = sum_{r,r'} Ev[smp][v][r][r'] Rt[r][r'] ; pick v; copy chosen env.
template <typename R>
__global__ void sample_pick_kernel(int dr, const cx<R>* __restrict__ ev, const cx<R>* __restrict__ rt,
                                   uint64_t seed, int site, int site_user, int n_sites,
                                   cx<R>* env_out, uint8_t* bits, double* probs, int last) {
  int smp = blockIdx.x;
  long plane = (long)dr * dr;
  const cx<R>* base = ev + (long)smp * 3 * plane;
  __shared__ double red[3][256];
  double q[3] = {0, 0, 0};
  for (long e = threadIdx.x; e < plane; e += blockDim.x) {
    cx<R> rv = rt[e];
    for (int v = 0; v < 3; ++v) {
      cx<R> x = base[v * plane + e];
      q[v] += (double)x.x * rv.x - (double)x.y * rv.y;
    }
  }
  for (int v = 0; v < 3; ++v) red[v][threadIdx.x] = q[v];
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int v = 0; v < 3; ++v) red[v][threadIdx.x] += red[v][threadIdx.x + s];
    __syncthreads();
  }
  __shared__ int pick;
  if (threadIdx.x == 0) {
    double q0 = red[0][0] > 0 ? red[0][0] : 0, q1 = red[1][0] > 0 ? red[1][0] : 0,
           q2 = red[2][0] > 0 ? red[2][0] : 0;
    double tot = q0 + q1 + q2;
    double u = philox_uniform(seed, (uint32_t)smp, (uint32_t)site_user);
    int v = 2;
    if (u < q0 / tot) v = 0;
    else if (u < (q0 + q1) / tot) v = 1;
    pick = v;
    bits[(long)smp * n_sites + site_user] = (uint8_t)v;
    if (last) {
      double pv = (v == 0) ? red[0][0] : (v == 1 ? red[1][0] : red[2][0]);
      probs[smp] = pv;
    }
  }
  __syncthreads();
  const cx<R>* src = base + pick * plane;
  for (long e = threadIdx.x; e < plane; e += blockDim.x) env_out[(long)smp * plane + e] = src[e];
}

// Newton-Schulz polar step for a near-isometry A with Gram G = A^+A (n x n):
// P = (3I - G)/2 (applied to A) and Q = (I + G)/2 (applied to the other factor), so that
// A P has unit Gram to second order and (A P)(Q B) = A B - A E^2 B / 4 with E = G - I.
template <typename R>
__global__ void polar_factors_kernel(int n, const cx<R>* __restrict__ g, cx<R>* pm, cx<R>* qm) {
  long total = (long)n * n;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    int i = (int)(e / n), j = (int)(e % n);
    cx<R> v = g[e];
    R d = (i == j) ? R(1) : R(0);
    pm[e] = mkc<R>((R)1.5 * d - (R)0.5 * v.x, (R)(-0.5) * v.y);
    qm[e] = mkc<R>((R)0.5 * d + (R)0.5 * v.x, (R)0.5 * v.y);
  }
}

// Inner-index truncation through the dual Gram W' = B^+B (used when B has fewer columns
// than rows): with W' y_k = w_k y_k, the kept rows of the new centre are
// f_k x_k^+ B = f_k sqrt(w_k) y_k^+  (x_k = B y_k / sqrt(w_k)), so no product with B is needed.
template <typename R, typename RO>
__global__ void dual_rows_kernel(int kk, int cols, const cx<R>* __restrict__ y, long ldy,
                                 const double* __restrict__ f, const double* __restrict__ w,
                                 cx<RO>* out) {
  long total = (long)kk * cols;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    int k = (int)(e / cols), c = (int)(e % cols);
    double wk = w[k] > 0 ? w[k] : 0.0;
    R sc = (R)(f[k] * sqrt(wk));
    cx<R> t = cscale(cconj(y[(long)c * ldy + k]), sc);
    out[e] = mkc<RO>((RO)t.x, (RO)t.y);
  }
}

// Pivoted Cholesky of the Hermitian PSD n x n matrix w (precision R, n <= 1024): W ~ L L^+
// with L n x r (row-major, row stride lr), greedy diagonal pivoting, stopping once the
// largest remaining diagonal is <= tol * tr W or after rmax (<= kGradedMax) columns.
// *rout = r, or kPcholGaveUp when a wait for another CTA gave up; *resid = largest remaining diagonal
// / tr W.
//
// The columns depend on one another, so the factor is bound by the latency of a column.  An FP64
// warp instruction occupies its quarter of the SM for 64 clocks whatever its active lanes, so a
// row's dot product is split over four or eight lanes such that the row warps of a CTA, and one
// further warp for the pivot's square root, find a quarter each; the lanes' sums part into real
// and imaginary halves with the first exchange, which leaves one operation a step.  Rows beyond 32
// go to the CTAs of a thread-block cluster (row i belongs to rank i mod S), each row's part of L --
// and of W, where it fits -- in its CTA's shared memory.  Per column every CTA sends its best
// remaining diagonal, a remote store, and that row of L, a bulk copy, to every CTA; both count
// their bytes at the receiver's mbarrier (a remote store for every entry of the row kept the
// barriers counting for 1200 clocks): one hop, after which all hold the pivot and its row, against a cluster
// barrier (1200 clocks) and a fetch of the row (1400) before.  Where the slots of all candidates'
// rows do not fit (n > 832 at 168 columns) the owner sends the pivot's row in a second hop.  The
// remaining diagonals follow from the unscaled column, beside its scaling.  Slots alternate by
// column parity: a CTA sends for column j + 2 only after every CTA has sent for j + 1, which each
// does when its threads are done with column j.  Candidates are compared as integers
// (non-negative doubles order alike), which keeps the FP64 pipe to the dot products.  Sums and the
// pivot choice follow a fixed order, so the factor does not depend on scheduling.
// n 156, rank 52: 225 -> 122 us; n 400, rank 55: 258 -> 151; n 64, rank 45: 170 -> 88; n 32, rank
// 24: 54 -> 41 us.
constexpr int kPcWarps = 8;              // row warps of a CTA
constexpr int kPcCtas = 16;
constexpr unsigned long long kPcWaitNs = 1000000000ull;
// largest key of the warp (bits of a non-negative double, or -1) and the smallest index with it
__device__ __forceinline__ void warp_best(long long& key, int& idx) {
  const int hi = (int)(key >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned lo = hi == mh ? (unsigned)key : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
  const int x = hi == mh && lo == ml ? idx : 0x7fffffff;
  idx = __reduce_min_sync(0xffffffffu, x);
  key = ((long long)mh << 32) | ml;
}
__device__ __forceinline__ uint32_t pc_su32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// address of x (of this CTA's shared memory) in the cluster's CTA of that rank
__device__ __forceinline__ uint32_t pc_map(uint32_t x, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(rank));
  return r;
}
// one remote store that counts its bytes at the receiver's barrier
__device__ __forceinline__ void pc_send(uint32_t dst, uint32_t bar, long long a, long long b) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%2, %3}, [%1];"
               ::"r"(dst), "r"(bar), "l"(a), "l"(b)
               : "memory");
}
// bytes (a multiple of 16) from this CTA's shared memory, as one count at the receiver's barrier
__device__ __forceinline__ void pc_copy(uint32_t dst, uint32_t bar, const void* src, int bytes) {
  asm volatile(
      "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%2], %3, [%1];" ::"r"(
          dst),
      "r"(bar), "r"(pc_su32(src)), "r"(bytes)
      : "memory");
}
__device__ __forceinline__ void pc_send(uint32_t dst, uint32_t bar, float2 v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%2, %3}, [%1];"
               ::"r"(dst), "r"(bar), "r"(__float_as_int(v.x)), "r"(__float_as_int(v.y))
               : "memory");
}
__device__ __forceinline__ bool pc_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool pc_wait(uint32_t bar, uint32_t parity) {
  if (pc_test(bar, parity)) return true;
  unsigned long long t0, t1;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (pc_test(bar, parity)) return true;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
    if (t1 - t0 > kPcWaitNs) return false;
  }
}
template <typename R, bool CLUSTER, int LANES>
__global__ void __launch_bounds__(32 * (kPcWarps + 1)) pchol_kernel(
    int n, const cx<R>* __restrict__ w, int rmax, double tol, cx<R>* L, int lr, int* rout,
    double* resid, int* piv, int w_rows, int all_rows) {
  using T = cx<R>;
  cg::cluster_group cluster = cg::this_cluster();
  const int S = CLUSTER ? (int)cluster.num_blocks() : 1, c = CLUSTER ? (int)cluster.block_rank() : 0;
  extern __shared__ __align__(16) unsigned char pc_raw[];
  T* Ls = reinterpret_cast<T*>(pc_raw);          // own rows of L, stride rmax
  const int nlm = (n + S - 1) / S;
  // the candidates' rows of L, [2][S][rmax] (all_rows), or the pivot's, [2][rmax]
  T* rows = Ls + (size_t)nlm * rmax;
  const int nslot = all_rows ? S : 1;
  T* Ws = rows + (CLUSTER ? (size_t)2 * nslot * rmax : 0);   // own rows of W, stride n (w_rows)
  __shared__ __align__(16) longlong2 post[2][kPcCtas];   // best remaining diagonals: bits, index
  __shared__ __align__(8) unsigned long long bars[4];
  __shared__ long long s_v[2][kPcWarps];
  __shared__ int s_i[2][kPcWarps], s_late;
  __shared__ double s_tr[kPcWarps], post_tr, s_inv, s_inv2, s_dp;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = (blockDim.x >> 5) - 1;
  const int lgS = 31 - __clz(S);                 // S is a power of two
  const int lr_ = lane & (LANES - 1), li = tid / LANES, i = c + li * S;
  const int part = lr_ >= LANES / 2;             // lanes of the upper half end with the imaginary part
  const bool own = warp < nw && li < nlm && i < n;
  if (w_rows)
    for (int e = tid; e < nlm * n; e += blockDim.x) {
      const int row = c + (e / n) * S;
      if (row < n) Ws[e] = w[(long)row * n + e % n];
    }
  double d = 0.0;
  if (own) {
    d = (double)w[(long)i * n + i].x;
    if (!(d > 0.0)) d = 0.0;
  }
  double tp = lr_ == 0 ? d : 0.0;
  for (int o = 16; o > 0; o >>= 1) tp += __shfl_xor_sync(0xffffffffu, tp, o);
  if (lane == 0 && warp < nw) s_tr[warp] = tp;
  if (tid == 0) s_late = 0;
  if (CLUSTER && tid < 4) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(pc_su32(&bars[tid])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  double tr = 0.0;
  for (int k = 0; k < nw; ++k) tr += s_tr[k];
  if constexpr (CLUSTER) {
    if (tid == 0) post_tr = tr;
    cluster.sync();
    tr = 0.0;
    for (int q = 0; q < S; ++q) tr += *cluster.map_shared_rank(&post_tr, q);
  }
  const double thr = tol * tr;
  auto expect = [&](uint32_t bar, int bytes) {
    if (tid == 0)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                   : "memory");
  };
  // the first j entries of row i of L (this CTA's) into a slot of every CTA
  auto send_row = [&](int j, int i, const T* slot, uint32_t bar) {
    const T* mine = Ls + (size_t)(i >> lgS) * rmax;
    const uint32_t s0 = pc_su32(slot);
    if constexpr (sizeof(R) == 8) {
      // one copy a receiver: FP64 entries are 16 bytes
      if (j > 0 && warp == nw && lane < S)
        pc_copy(pc_map(s0, lane), pc_map(bar, lane), mine, j * (int)sizeof(T));
    } else {
      for (int q = warp; q < S; q += nw + 1) {
        const uint32_t rb = pc_map(bar, q), rs = pc_map(s0, q);
        for (int k = lane; k < j; k += 32) pc_send(rs + k * (int)sizeof(T), rb, mine[k]);
      }
    }
  };
  // The best remaining diagonal of all rows, as bits: this CTA's (all_rows: with that row of L, up
  // to column j) into every CTA's slots, and the best of the posts.  A wait that gave up is noted
  // in s_late, which the CTA's threads look at together, after their next barrier.
  auto pivot = [&](int j, long long& bv, int& p) {
    const int par = j & 1;
    bv = own ? __double_as_longlong(d) : -1;
    int bi = own ? i : 0x7fffffff;
    warp_best(bv, bi);
    if (lane == 0 && warp < nw) {
      s_v[par][warp] = bv;
      s_i[par][warp] = bi;
    }
    __syncthreads();
    bv = lane < nw ? s_v[par][lane] : -1;
    bi = lane < nw ? s_i[par][lane] : 0x7fffffff;
    warp_best(bv, bi);
    if constexpr (CLUSTER) {
      const uint32_t bar = pc_su32(&bars[par]);
      expect(bar, S * (16 + (all_rows ? j * (int)sizeof(T) : 0)));
      if (all_rows) send_row(j, bi, rows + ((size_t)par * S + c) * rmax, bar);
      if (warp == 0 && lane < S)
        pc_send(pc_map(pc_su32(&post[par][c]), lane), pc_map(bar, lane), bv, (long long)bi);
      if (!pc_wait(bar, (uint32_t)(j >> 1) & 1)) s_late = 1;
      const longlong2 v = post[par][lane & (kPcCtas - 1)];
      bv = lane < S ? v.x : -1;
      bi = lane < S ? (int)v.y : 0x7fffffff;
      warp_best(bv, bi);
    }
    p = bi;
  };
  const long long thrb = __double_as_longlong(thr);
  constexpr long long kInf = 0x7ff0000000000000ll;   // above: not a number
  int r = 0, p = -1;
  long long last = 0;
  for (int j = 0; j < rmax; ++j) {
    pivot(j, last, p);
    if (!(last > thrb && last <= kInf)) {
      __syncthreads();
      break;
    }
    if (piv && c == 0 && tid == 0) piv[j] = p;
    const T* prow = Ls + (size_t)p * rmax;
    if constexpr (CLUSTER) {
      prow = rows + ((size_t)(j & 1) * nslot + (all_rows ? p & (S - 1) : 0)) * rmax;
      if (!all_rows) {
        const uint32_t bar = pc_su32(&bars[2 + (j & 1)]);
        expect(bar, j * (int)sizeof(T));
        if ((p & (S - 1)) == c) send_row(j, p, prow, bar);
        if (!pc_wait(bar, (uint32_t)(j >> 1) & 1)) s_late = 1;
      }
    }
    R wip = R(0), v = R(0);
    if (own) {
      const T* wr = w_rows ? Ws + (size_t)li * n : w + (long)i * n;
      wip = reinterpret_cast<const R*>(wr + p)[part];
    }
    if (warp < nw) {
      T acc = mkc<R>(0, 0), acc2 = mkc<R>(0, 0);
      if (own) {
        const T* lrow = Ls + (size_t)li * rmax;
        for (int k = lr_; k < j; k += LANES) {
          const T a = lrow[k], b = prow[k];
          // acc + acc2 += a * conj(b)
          acc.x = fma(a.x, b.x, acc.x);
          acc.y = fma(a.y, b.x, acc.y);
          acc2.x = fma(a.y, b.y, acc2.x);
          acc2.y = fma(-a.x, b.y, acc2.y);
        }
      }
      acc = cadd(acc, acc2);
      // the first exchange leaves one half of the lanes the real part and the other the imaginary
      const R give = part ? acc.x : acc.y;
      v = (part ? acc.y : acc.x) + __shfl_xor_sync(0xffffffffu, give, LANES / 2);
      for (int o = LANES / 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      v = wip - v;
    } else {
      const double dp = __longlong_as_double(last), inv = rsqrt(dp);
      if (lane == 0) {
        s_dp = dp * inv;
        s_inv = inv;
        s_inv2 = inv * inv;
      }
    }
    double sq = (double)v * v;
    sq += __shfl_xor_sync(0xffffffffu, sq, LANES / 2);
    __syncthreads();
    if (CLUSTER && s_late) break;
    if (own) {
      const double nd = fma(-sq, s_inv2, d);
      d = (i == p || __double2hiint(nd) < 0) ? 0.0 : nd;
      R lij = v * (R)s_inv;
      if (i == p) lij = part ? R(0) : (R)s_dp;
      if ((lr_ & (LANES / 2 - 1)) == 0) reinterpret_cast<R*>(Ls + (size_t)li * rmax + j)[part] = lij;
      // the row may go out as a copy, which reads through the asynchronous proxy
      if constexpr (CLUSTER && sizeof(R) == 8) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    r = j + 1;
    last = 0;
  }
  if (r == rmax) {                          // the largest remaining diagonal
    pivot(rmax, last, p);
    __syncthreads();
  }
  if (c == 0 && tid == 0) {
    const double ld = __longlong_as_double(last);
    *rout = r;
    *resid = !s_late && tr > 0 && ld > 0.0 ? ld / tr : 0.0;
  }
  // L to global memory only now: a store before an exchange holds it up until the store has landed
  for (int e = tid; e < nlm * r; e += blockDim.x) {
    const int row = e / r, k = e - row * r;
    if (c + row * S < n) L[(long)(c + row * S) * lr + k] = Ls[(size_t)row * rmax + k];
  }
  if constexpr (CLUSTER) {
    cluster.sync();   // no CTA leaves before what was sent to it has landed
    if (s_late && tid == 0) *rout = kPcholGaveUp;   // whichever CTA's wait it was
  }
}

// x = L1^-1 (r x r, lower triangular, row-major), L1[a][b] = L[piv[a]][b] the pivot rows of a
// pivoted Cholesky factor.  A warp per column of x, by columns of L1: once x_b is known every
// lane takes L1[a][b] x_b off its rows a > b.  Bound by the latency of the r dependent steps, so
// L1 comes through shared memory kInvChunk columns at a time (a step that waited for its
// entries from L2 took three times as long: 45 us at r = 52).
constexpr int kInvWarps = 4, kInvChunk = 16;
template <int RL>   // rows of a lane: a = lane + 32 t
__global__ void __launch_bounds__(32 * kInvWarps) pchol_inverse_kernel(int r,
                                                                      const double2* __restrict__ L,
                                                                      int lr,
                                                                      const int* __restrict__ piv,
                                                                      double2* x) {
  __shared__ double2 col[kInvChunk][32 * RL];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j0 = blockIdx.x * kInvWarps, j = j0 + warp;
  double inv[RL];
  double2 s[RL];
#pragma unroll
  for (int t = 0; t < RL; ++t) {
    const int a = lane + 32 * t;
    inv[t] = a < r ? 1.0 / L[(long)piv[a] * lr + a].x : 0.0;
    s[t] = make_double2(a == j ? 1.0 : 0.0, 0.0);
  }
  for (int b0 = j0 / kInvChunk * kInvChunk; b0 < r; b0 += kInvChunk) {
    __syncthreads();
    for (int e = threadIdx.x; e < kInvChunk * r; e += 32 * kInvWarps) {
      const int a = e / kInvChunk, b = e % kInvChunk;
      col[b][a] = b0 + b < r ? L[(long)piv[a] * lr + b0 + b] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const int b1 = min(r, b0 + kInvChunk);
    for (int b = max(b0, j); b < b1; ++b) {
      // x_b from its lane: every lane selects its own candidate, the broadcast takes the right one
      double2 xb = make_double2(0.0, 0.0);
#pragma unroll
      for (int t = 0; t < RL; ++t)
        if (t == b >> 5) xb = cscale(s[t], inv[t]);
      xb.x = __shfl_sync(0xffffffffu, xb.x, b & 31);
      xb.y = __shfl_sync(0xffffffffu, xb.y, b & 31);
#pragma unroll
      for (int t = 0; t < RL; ++t) {
        const int a = lane + 32 * t;
        if (a == b) s[t] = xb;
        else if (a > b && a < r) s[t] = csub(s[t], cmul(col[b - b0][a], xb));
      }
    }
  }
  if (j >= r) return;
#pragma unroll
  for (int t = 0; t < RL; ++t) {
    const int a = lane + 32 * t;
    if (a < r) x[(long)a * r + j] = a >= j ? s[t] : make_double2(0.0, 0.0);
  }
}

// out (rows x r) = the columns piv[0..r) of in (row stride ldi)
template <typename T>
__global__ void gather_cols_kernel(long rows, int r, const T* __restrict__ in, long ldi,
                                   const int* __restrict__ piv, T* __restrict__ out) {
  const long total = rows * r;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x)
    out[e] = in[(e / r) * ldi + piv[e % r]];
}

// zs[i][c] = z[i][c] / sqrt(s_c) (0 where s_c <= 0): eigenvectors of L L^+ from those of L^+ L
template <typename R>
__global__ void lift_kernel(int r, const cx<R>* __restrict__ z, const double* __restrict__ s,
                            cx<R>* zs) {
  long total = (long)r * r;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    int c = (int)(e % r);
    double sc = s[c] > 0 ? 1.0 / sqrt(s[c]) : 0.0;
    zs[e] = cscale(z[e], (R)sc);
  }
}

}  // namespace

// ------------------------------------------------------------- launchers
// Rows x cols complex matrix copied between precisions (strided rows on both sides).
template <typename Ri, typename Ro>
__global__ void convert_kernel(int rows, int cols, const cx<Ri>* __restrict__ in, long ldi,
                               cx<Ro>* __restrict__ out, long ldo) {
  long total = (long)rows * cols;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    long r = e / cols, c = e % cols;
    cx<Ri> v = in[r * ldi + c];
    out[r * ldo + c] = mkc<Ro>((Ro)v.x, (Ro)v.y);
  }
}

template <typename Ri, typename Ro>
cudaError_t convert(cudaStream_t st, int rows, int cols, const cx<Ri>* in, long ldi, cx<Ro>* out,
                    long ldo) {
  long total = (long)rows * cols;
  if (total <= 0) return cudaSuccess;
  count_launch();
  convert_kernel<Ri, Ro><<<nblocks(total), 256, 0, st>>>(rows, cols, in, ldi, out, ldo);
  return cudaGetLastError();
}
template cudaError_t convert<float, double>(cudaStream_t, int, int, const cx<float>*, long,
                                            cx<double>*, long);
template cudaError_t convert<double, float>(cudaStream_t, int, int, const cx<double>*, long,
                                            cx<float>*, long);

template <typename T>
cudaError_t swap12(cudaStream_t st, long n0, long n1, long n2, long n3, const T* in, T* out) {
  long total = n0 * n1 * n2 * n3;
  if (total <= 0) return cudaSuccess;
  count_launch();
  swap12_kernel<T><<<nblocks(total), 256, 0, st>>>(n0, n1, n2, n3, in, out);
  return cudaGetLastError();
}
template <typename T>
cudaError_t reverse_site(cudaStream_t st, int dl, int d, int k, int dr, const T* in, T* out) {
  long total = (long)dl * d * k * dr;
  count_launch();
  reverse_site_kernel<T><<<nblocks(total), 256, 0, st>>>(dl, d, k, dr, in, out);
  return cudaGetLastError();
}
template <typename R>
cudaError_t one_site(cudaStream_t st, int dl, int k, int dr, const cx<R>* u, cx<R>* a) {
  long total = (long)dl * k * dr;
  count_launch();
  one_site_kernel<R><<<nblocks(total), 256, 0, st>>>(dl, k, dr, u, a);
  return cudaGetLastError();
}
template <typename R>
cudaError_t product_state(cudaStream_t st, const double* v, cx<R>* base, long stride, int n) {
  count_launch();
  product_state_kernel<R><<<(n + 127) / 128, 128, 0, st>>>(
      mkc<R>((R)v[0], (R)v[1]), mkc<R>((R)v[2], (R)v[3]), mkc<R>((R)v[4], (R)v[5]), base, stride,
      n);
  return cudaGetLastError();
}
template <typename R>
cudaError_t gram_mask(cudaStream_t st, int n, const double* sig, double gtol, R* rs, R* irs,
                      StepScalars* sc) {
  count_launch();
  gram_mask_kernel<R><<<1, 256, 0, st>>>(n, sig, gtol, rs, irs, sc);
  return cudaGetLastError();
}
template <typename R>
cudaError_t gram_factor(cudaStream_t st, int n, const cx<R>* v, const R* rs, const R* irs,
                        cx<R>* rmat, cx<R>* vs, cx<R>* vr) {
  count_launch();
  gram_factor_kernel<R><<<nblocks((long)n * n), 256, 0, st>>>(n, v, rs, irs, rmat, vs, vr);
  return cudaGetLastError();
}
template <typename R>
cudaError_t build_phi(cudaStream_t st, int dm, const cx<R>* ct, const cx<R>* gj, cx<R>* phi) {
  long n = 9L * dm;
  count_launch();
  build_phi_kernel<R><<<nblocks(n * n), 256, 0, st>>>(dm, ct, gj, phi);
  return cudaGetLastError();
}
template <typename R>
cudaError_t bond_select(cudaStream_t st, int n, const double* lam, const cx<R>* hm, long ldh,
                        double htol, int chi, StepScalars* sc, DevStats* ds) {
  count_launch();
  bond_select_kernel<R><<<1, 256, 0, st>>>(n, lam, hm, ldh, htol, chi, sc, ds);
  return cudaGetLastError();
}
template <typename R>
cudaError_t make_q(cudaStream_t st, int dm, int keep, int m_ops, const cx<R>* w, const cx<R>* e,
                   const StepScalars* sc, cx<R>* q) {
  long total = (long)keep * 3 * m_ops * 3 * dm;
  count_launch();
  make_q_kernel<R><<<nblocks(total), 256, 0, st>>>(dm, keep, m_ops, w, e, sc, q);
  return cudaGetLastError();
}
template <typename R>
cudaError_t kraus_select(cudaStream_t st, int n, const double* w, const cx<R>* wm, int ntr,
                         double kcut, int kmax, int use_ppt, double* f, StepScalars* sc,
                         DevStats* ds, double* trace) {
  // the partial sums and the ticket live after the kept scale factors f (at most 1024 of them)
  double* parts = f + 1024;
  count_launch();
  kraus_select_kernel<R><<<kNormBlocks, 256, 0, st>>>(
      n, w, wm, ntr, parts, reinterpret_cast<unsigned int*>(parts + 2 * kNormBlocks), kcut, kmax,
      use_ppt, f, sc, ds, trace);
  return cudaGetLastError();
}
template <typename R>
cudaError_t trace_pre(cudaStream_t st, int dm, const cx<R>* gi, const cx<R>* gj, StepScalars* sc) {
  count_launch();
  trace_pre_kernel<R><<<1, 256, 0, st>>>(dm, gi, gj, sc);
  return cudaGetLastError();
}
template <typename T>
cudaError_t permute6(cudaStream_t st, const int* d, const int* p, const T* in, T* out) {
  long total = 1;
  for (int i = 0; i < 6; ++i) total *= d[i];
  count_launch();
  permute6_kernel<T><<<nblocks(total), 256, 0, st>>>(in, out, d[0], d[1], d[2], d[3], d[4], d[5],
                                                     p[0], p[1], p[2], p[3], p[4], p[5]);
  return cudaGetLastError();
}
template <typename R>
cudaError_t rho_site(cudaStream_t st, long dl2, long dr2, cx<R>* r, cx<R>* tr, int mode) {
  count_launch();
  rho_site_kernel<cx<R>><<<nblocks(dl2 * 9 * dr2), 256, 0, st>>>(dl2, dr2, r, tr, mode);
  return cudaGetLastError();
}
constexpr int kDotBlocks = 64;
template <typename R>
cudaError_t env_dot(cudaStream_t st, long n2, const cx<R>* x, const cx<R>* y, int mode,
                    double* parts, double* out) {
  count_launch(2);
  env_dot_kernel<cx<R>><<<kDotBlocks, 256, 0, st>>>(n2, x, y, mode, parts);
  sum_parts_kernel<<<1, 32, 0, st>>>(kDotBlocks, parts, out);
  return cudaGetLastError();
}

template <typename R>
cudaError_t sumsq(cudaStream_t st, long n, const cx<R>* a, double* out) {
  count_launch();
  sumsq_kernel<R><<<1, 256, 0, st>>>(n, a, out);
  return cudaGetLastError();
}
template <typename R, typename RO>
cudaError_t scale_vk(cudaStream_t st, int n, int kk, const cx<R>* v, long ldv, const double* f,
                     cx<RO>* out) {
  count_launch();
  scale_vk_kernel<R, RO><<<nblocks((long)n * kk), 256, 0, st>>>(n, kk, v, ldv, f, out);
  return cudaGetLastError();
}
template <typename R>
cudaError_t energy_mix(cudaStream_t st, int dl, int plane, const cx<R>* f, long fstride,
                       cx<R>* g, long gstride, double J, double hx, double bz) {
  count_launch();
  energy_mix_kernel<R><<<nblocks((long)dl * plane), 256, 0, st>>>(dl, plane, f, fstride, g,
                                                                    gstride, J, hx, bz);
  return cudaGetLastError();
}
cudaError_t energy_init(cudaStream_t st, long env, double2* e) {
  count_launch();
  energy_init_kernel<<<1, 32, 0, st>>>(env, e);
  return cudaGetLastError();
}
cudaError_t energy_result(cudaStream_t st, long env, const double2* e, const double* trace,
                          double* res) {
  count_launch();
  energy_result_kernel<<<1, 32, 0, st>>>(env, e, trace, res);
  return cudaGetLastError();
}
template <typename R>
cudaError_t sample_pick(cudaStream_t st, int n_samples, int dr, const cx<R>* ev, const cx<R>* rt,
                        uint64_t seed, int site, int site_user, int n_sites, cx<R>* env_out,
                        uint8_t* bits, double* probs, int last) {
  count_launch();
  sample_pick_kernel<R><<<n_samples, 256, 0, st>>>(dr, ev, rt, seed, site, site_user, n_sites,
                                                   env_out, bits, probs, last);
  return cudaGetLastError();
}

template <typename R>
cudaError_t polar_factors(cudaStream_t st, int n, const cx<R>* g, cx<R>* pm, cx<R>* qm) {
  count_launch();
  polar_factors_kernel<R><<<nblocks((long)n * n), 256, 0, st>>>(n, g, pm, qm);
  return cudaGetLastError();
}

template <typename R, typename RO>
cudaError_t dual_rows(cudaStream_t st, int kk, int cols, const cx<R>* y, long ldy, const double* f,
                      const double* w, cx<RO>* out) {
  count_launch();
  dual_rows_kernel<R, RO><<<nblocks((long)kk * cols), 256, 0, st>>>(kk, cols, y, ldy, f, w, out);
  return cudaGetLastError();
}

template <typename R>
cudaError_t pchol(cudaStream_t st, int n, const cx<R>* w, int rmax, double tol, cx<R>* L, int lr,
                  int* rout, double* resid, int* piv) {
  if (n < 1 || n > 1024 || rmax < 1 || rmax > kGradedMax) return cudaErrorInvalidValue;
  // One CTA needs no exchange, which is worth more than other CTAs' FP64 pipes up to 32 rows (rank
  // 24: 41 us against 49 us on four); then up to 20 rows a CTA with eight lanes each (n 64, rank 45:
  // four CTAs 88 us, two 104; n 200, rank 52: sixteen 119, eight 144; 20 rows: 2.35 us a column with
  // eight lanes, 2.47 with four), beyond 16 CTAs more rows with four lanes (n 400, rank 55: 151 us,
  // eight lanes 162).  FP32 keeps four lanes: its sums keep their order.
  const int S = n > 160 ? kPcCtas : n > 64 ? 8 : n > 32 ? 4 : 1;
  const int rows = (n + S - 1) / S;
  const int lanes = S > 1 && rows <= 20 && sizeof(R) == 8 ? 8 : 4;
  const int threads = (rows * lanes + 31) / 32 * 32 + 32;   // and the warp of the root
  rmax = std::min(rmax, n);
  const size_t wb = (size_t)rows * n * sizeof(cx<R>);
  constexpr size_t kMax = 222 * 1024;   // leaves the static arrays their place
  auto l_bytes = [&](int slots) { return ((size_t)rows + slots) * rmax * sizeof(cx<R>); };
  const int all_rows = S > 1 && l_bytes(2 * S) <= kMax ? 1 : 0;
  const size_t lb = l_bytes(S == 1 ? 0 : all_rows ? 2 * S : 2);
  const int w_rows = lb + wb <= kMax ? 1 : 0;
  auto* kern = S == 1 ? pchol_kernel<R, false, 4>
                      : lanes == 8 ? pchol_kernel<R, true, 8> : pchol_kernel<R, true, 4>;
  static const cudaError_t attr = [] {
    cudaError_t e = cudaSuccess;
    for (auto* f : {pchol_kernel<R, false, 4>, pchol_kernel<R, true, 4>, pchol_kernel<R, true, 8>}) {
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMax);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    }
    return e;
  }();
  MPDO_CUDA_TRY(attr);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(S);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = w_rows ? lb + wb : lb;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = S;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = S > 1 ? 1 : 0;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kern, n, w, rmax, tol, L, lr, rout, resid, piv, w_rows, all_rows);
}
template cudaError_t pchol<float>(cudaStream_t, int, const float2*, int, double, float2*, int,
                                  int*, double*, int*);
template cudaError_t pchol<double>(cudaStream_t, int, const double2*, int, double, double2*, int,
                                   int*, double*, int*);
cudaError_t pchol_inverse(cudaStream_t st, int r, const double2* L, int lr, const int* piv,
                          double2* x) {
  if (r < 1 || r > kGradedMax) return cudaErrorInvalidValue;
  count_launch();
  auto run = [&](auto kern) {
    kern<<<(r + kInvWarps - 1) / kInvWarps, 32 * kInvWarps, 0, st>>>(r, L, lr, piv, x);
  };
  if (r <= 32) run(pchol_inverse_kernel<1>);
  else if (r <= 64) run(pchol_inverse_kernel<2>);
  else run(pchol_inverse_kernel<(kGradedMax + 31) / 32>);
  return cudaGetLastError();
}
template <typename T>
cudaError_t gather_cols(cudaStream_t st, long rows, int r, const T* in, long ldi, const int* piv,
                        T* out) {
  count_launch();
  gather_cols_kernel<T><<<nblocks(rows * r), 256, 0, st>>>(rows, r, in, ldi, piv, out);
  return cudaGetLastError();
}
template cudaError_t gather_cols<float2>(cudaStream_t, long, int, const float2*, long, const int*,
                                         float2*);
template cudaError_t gather_cols<double2>(cudaStream_t, long, int, const double2*, long, const int*,
                                          double2*);
template <typename R>
cudaError_t lift(cudaStream_t st, int r, const cx<R>* z, const double* s, cx<R>* zs) {
  count_launch();
  lift_kernel<R><<<nblocks((long)r * r), 256, 0, st>>>(r, z, s, zs);
  return cudaGetLastError();
}
template cudaError_t lift<float>(cudaStream_t, int, const float2*, const double*, float2*);

#define INST(R)                                                                               \
  template cudaError_t swap12<cx<R>>(cudaStream_t, long, long, long, long, const cx<R>*,     \
                                     cx<R>*);                                               \
  template cudaError_t reverse_site<cx<R>>(cudaStream_t, int, int, int, int, const cx<R>*,   \
                                           cx<R>*);                                         \
  template cudaError_t one_site<R>(cudaStream_t, int, int, int, const cx<R>*, cx<R>*);      \
  template cudaError_t product_state<R>(cudaStream_t, const double*, cx<R>*, long, int);     \
  template cudaError_t gram_mask<R>(cudaStream_t, int, const double*, double, R*, R*,       \
                                    StepScalars*);                                          \
  template cudaError_t gram_factor<R>(cudaStream_t, int, const cx<R>*, const R*, const R*,  \
                                      cx<R>*, cx<R>*, cx<R>*);                              \
  template cudaError_t build_phi<R>(cudaStream_t, int, const cx<R>*, const cx<R>*, cx<R>*); \
  template cudaError_t make_q<R>(cudaStream_t, int, int, int, const cx<R>*, const cx<R>*,   \
                                 const StepScalars*, cx<R>*);                               \
  template cudaError_t energy_mix<R>(cudaStream_t, int, int, const cx<R>*, long, cx<R>*,    \
                                     long, double, double, double);                         \
  template cudaError_t bond_select<R>(cudaStream_t, int, const double*, const cx<R>*, long,  \
                                      double, int, StepScalars*, DevStats*);                 \
  template cudaError_t kraus_select<R>(cudaStream_t, int, const double*, const cx<R>*, int,   \
                                       double, int, int, double*, StepScalars*, DevStats*,   \
                                       double*);                                             \
  template cudaError_t trace_pre<R>(cudaStream_t, int, const cx<R>*, const cx<R>*,           \
                                    StepScalars*);                                           \
  template cudaError_t polar_factors<R>(cudaStream_t, int, const cx<R>*, cx<R>*, cx<R>*);   \
  template cudaError_t sumsq<R>(cudaStream_t, long, const cx<R>*, double*);                 \
  template cudaError_t permute6<cx<R>>(cudaStream_t, const int*, const int*, const cx<R>*,    \
                                       cx<R>*);                                              \
  template cudaError_t rho_site<R>(cudaStream_t, long, long, cx<R>*, cx<R>*, int);           \
  template cudaError_t env_dot<R>(cudaStream_t, long, const cx<R>*, const cx<R>*, int,       \
                                  double*, double*);                                          \
  template cudaError_t sample_pick<R>(cudaStream_t, int, int, const cx<R>*, const cx<R>*,   \
                                      uint64_t, int, int, int, cx<R>*, uint8_t*, double*, int);
INST(double)
INST(float)
#undef INST

#define INST2(R, RO)                                                                          \
  template cudaError_t scale_vk<R, RO>(cudaStream_t, int, int, const cx<R>*, long,           \
                                       const double*, cx<RO>*);                              \
  template cudaError_t dual_rows<R, RO>(cudaStream_t, int, int, const cx<R>*, long,          \
                                        const double*, const double*, cx<RO>*);
INST2(double, double)
INST2(float, float)
INST2(double, float)
#undef INST2

}  // namespace mpdo
