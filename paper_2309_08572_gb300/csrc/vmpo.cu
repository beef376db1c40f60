// Vectorized MPO engine with purity-preserving truncation on the bond (the paper's main
// engine: Sec. III.A "vectorized MPO", Sec. III.D Eqs. xiformula and ppt, App. B).
//
// rho is an MPS over the doubled index eta = (s, s') (d^2 = 9 per site), site tensors
// A_n[l][eta][r] in complex128, kept in mixed-canonical form for the Frobenius inner product.
// A two-site op acts on the pair (eta_i, eta_j) as its superoperator (built on the host from
// the op's Kraus set).  One update, centre at i (right-to-left updates run on the mirrored
// chain, as in the MPDO engine):
//   theta  = A_i A_j                       ((9 D_l) x (9 D_r), [l][eta_i][eta_j][r])
//   theta' = S theta on (eta_i, eta_j)     (81 x 81 superoperator, batched over l)
//   theta' = U Lambda V^+                  (eigenpairs of theta' theta'^+;
//                                           Lambda = sqrt of the eigenvalues above the cut,
//                                           V^+ = Lambda^-1 U^+ theta')
//   T_k    = (L (x) tau)^T U[:, k] * V^+[k, :] (tau (x) R)   (trace environment: L, R the
//            contractions of the sites left of i / right of j with tau[(s,s')] = delta_ss')
//   keep the chi largest: naive (unchanged) or PPT's values with this T (trace and
//   xi = tr rho^2 / tr rho^2 of the bond kept);  A_i <- U_keep, A_j <- diag(Lambda~) V^+_keep.
// The left trace environment of the new centre is updated from the new A_i; the right ones
// are recomputed after every change of direction.  Observables: tr(O rho) contracts each
// site with o[(s,s')] = O[s', s]; the TFIM energies run as a three-state automaton per
// projector (identity / qubit projector), one kernel per site.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <complex>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "../../include/mpdo.h"
#include "common.cuh"
#include "exactplan.h"
#include "internal.h"
#include "kernels.h"
#include "tcgemm.h"

namespace mpdo {
void set_global_error(const char* msg);
}

using namespace mpdo;

namespace {

using zc = std::complex<double>;

// Scalars of one vMPO update read by the host.
struct VScalars {
  int nz;        // Schmidt values above the cut
  int keep;      // kept
  int infeasible;
  int clamped;
  int flags;     // bit 0: numeric problem
  double theta;  // PPT angle
  double disc;   // discarded weight fraction (sum of Lambda^2)
};

// Cut and truncation of the Schmidt values (eigenvalues lam of theta' theta'^+, descending):
// nz = count above cut^2 lam_0, keep = min(nz, chi); mode 1 = PPT with the trace environment
// T_k = Re(tl_k trw_k) / Lambda_k (trw carries the factor Lambda_k of U^+ theta'; Eqs.
// xiformula, ppt; theta = 0 when infeasible, negative values clamped, rescaled so that
// T'.Lambda~ = T.Lambda); out[k] = Lambda~_k (k < keep), sv[k] = sqrt(lam_k) for k < nz.
// One warp, its lanes sharing the values (FP64 operations take ~64 clocks each here); tan(acos c)
// is sqrt(1 - c^2) / c.
__global__ void __launch_bounds__(32) vmpo_cut_kernel(int n, const double* __restrict__ lam,
                                                      const double2* __restrict__ tl,
                                                      const double2* __restrict__ tr, double cut2,
                                                      int chi, int mode, double* sv, double* out,
                                                      VScalars* sc) {
  const int lane = threadIdx.x;
  const double l0 = lam[0];
  VScalars s{};
  if (!(l0 > 0.0) || !isfinite(l0)) {
    s.flags = 1;
    s.nz = s.keep = 1;
    if (lane == 0) *sc = s;
    return;
  }
  auto warp_sum = [](double x) {
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  };
  int nz = n;
  for (int k0 = 0; k0 < n; k0 += 32) {   // the leading run above the cut
    const bool in = k0 + lane < n && lam[k0 + lane] > cut2 * l0;
    const unsigned miss = ~__ballot_sync(0xffffffffu, in);
    if (miss) {
      nz = min(n, k0 + __ffs(miss) - 1);
      break;
    }
  }
  if (nz < 1) nz = 1;
  const int keep = nz < chi ? nz : chi;
  double tot = 0, kept = 0;
  for (int k = lane; k < nz; k += 32) {
    sv[k] = sqrt(fmax(lam[k], 0.0));
    tot += lam[k];
    if (k < keep) kept += lam[k];
  }
  tot = warp_sum(tot);
  kept = warp_sum(kept);
  s.nz = nz;
  s.keep = keep;
  s.disc = tot > 0 ? (tot - kept) / tot : 0.0;
  if (mode == 0) {
    for (int k = lane; k < keep; k += 32) out[k] = sv[k];
  } else {
    // T_k = Re(tl_k tr_k) (real for a Hermitian rho up to near-degeneracies)
    auto trace_env = [&](int k) { return (tl[k].x * tr[k].x - tl[k].y * tr[k].y) / sv[k]; };
    double lt = 0, nl = 0, lpt = 0, nlp = 0, ntp = 0;
    for (int k = lane; k < nz; k += 32) {
      const double t = trace_env(k), a = sv[k] * t, b = sv[k] * sv[k];
      lt += a;
      nl += b;
      if (k < keep) {
        lpt += a;
        nlp += b;
        ntp += t * t;
      }
    }
    lt = warp_sum(lt);
    nl = sqrt(warp_sum(nl));
    lpt = warp_sum(lpt);
    nlp = sqrt(warp_sum(nlp));
    ntp = sqrt(warp_sum(ntp));
    const double cos_sig = fmin(1.0, lpt / (nlp * ntp));
    double c = lt / (nl * ntp);   // cos theta = |T| cos phi / |T'|
    if (c > 1.0 || !(ntp > 0)) {
      s.infeasible = 1;
      c = 1.0;
    }
    s.theta = acos(c);
    double x = 0.0;
    if (cos_sig < 1.0)
      x = sqrt((1.0 - c) * (1.0 + c)) / c * (cos_sig / sqrt((1.0 - cos_sig) * (1.0 + cos_sig))) - 1.0;
    double dot = 0;
    int clamped = 0;
    for (int k = lane; k < keep; k += 32) {
      const double t = trace_env(k);
      double v = cos_sig < 1.0 ? sv[k] + x * (sv[k] - nlp * cos_sig * t / ntp) : sv[k];
      if (v < 0) {
        v = 0;
        ++clamped;
      }
      out[k] = v;
      dot += v * t;
    }
    dot = warp_sum(dot);
    s.clamped = (int)__reduce_add_sync(0xffffffffu, (unsigned)clamped);
    const double scale = (dot != 0.0) ? lt / dot : 0.0;
    for (int k = lane; k < keep; k += 32) out[k] *= scale;
  }
  if (lane == 0) *sc = s;
}

// x[(l, eta)] = env[l] tau[eta] (side 0) or x[(eta, r)] = tau[eta] env[r] (side 1)
__global__ void trace_vec_kernel(int d, const double2* __restrict__ env, int side, double2* x) {
  const int total = 9 * d;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int eta = side == 0 ? e % 9 : e / d;
    const int b = side == 0 ? e / 9 : e % d;
    const bool diag = (eta == 0 || eta == 4 || eta == 8);
    x[e] = diag ? env[b] : make_double2(0.0, 0.0);
  }
}

// rows k < keep of vh (ld ldv) scaled by f[k] / sv[k] (f = Lambda~ or 1 for the isometry)
__global__ void scale_rows_kernel(int keep, int cols, const double2* __restrict__ in, long ldi,
                                  const double* __restrict__ num, const double* __restrict__ den,
                                  double2* out, long ldo) {
  const long total = (long)keep * cols;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const int k = (int)(e / cols), c = (int)(e % cols);
    const double f = (num ? num[k] : 1.0) / den[k];
    const double2 v = in[(long)k * ldi + c];
    out[(long)k * ldo + c] = make_double2(v.x * f, v.y * f);
  }
}

// The energy automaton on one site: for projector p (0: identity, 1: qubit projector),
// states s = 0 (no term yet), 1 (a Z waiting for its partner), 2 (term complete):
//   E0' = E0 T[P], E1' = E0 T[PZP], E2' = E2 T[P] - J E1 T[PZP] + E0 T[P H1 P]
// with T[O](E)[r] = sum_{l,eta} E[l] o[eta] A[l,eta,r], o[(s,s')] = O[s',s] and H1 = -hx X - b J Z:
// only the entries of A with eta in {00, 01, 10, 11, 22} meet a non-zero o.  env in/out:
// [2 projectors][3 states][dl | dr].  A CTA takes 32 columns r of one projector, its eight warps
// sharing the rows l (one thread per column took 177 us at D = 16).
__global__ void __launch_bounds__(256) vmpo_energy_kernel(int dl, int dr,
                                                          const double2* __restrict__ a,
                                                          const double2* __restrict__ ein,
                                                          double2* eout, double J, double hx,
                                                          double bz) {
  __shared__ double2 part[8][3][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, p = blockIdx.y;
  const int r = blockIdx.x * 32 + lane;
  const double2* e0 = ein + (p * 3 + 0) * dl;
  const double2* e1 = ein + (p * 3 + 1) * dl;
  const double2* e2 = ein + (p * 3 + 2) * dl;
  double2 n0 = make_double2(0, 0), n1 = n0, n2 = n0;
  if (r < dr)
    for (int l = warp; l < dl; l += 8) {
      const double2* al = a + (long)l * 9 * dr + r;
      const double2 a0 = al[0], a1 = al[dr], a3 = al[3L * dr], a4 = al[4L * dr];
      double2 t0 = cadd(a0, a4);
      const double2 t1 = csub(a0, a4);
      if (p == 0) t0 = cadd(t0, al[8L * dr]);
      const double2 t2 = csub(cscale(cadd(a1, a3), -hx), cscale(t1, bz * J));
      cfma(n0, e0[l], t0);
      cfma(n1, e0[l], t1);
      cfma(n2, e2[l], t0);
      cfma(n2, cscale(e1[l], -J), t1);
      cfma(n2, e0[l], t2);
    }
  part[warp][0][lane] = n0;
  part[warp][1][lane] = n1;
  part[warp][2][lane] = n2;
  __syncthreads();
  if (warp < 3 && r < dr) {
    double2 x = part[0][warp][lane];
    for (int k = 1; k < 8; ++k) x = cadd(x, part[k][warp][lane]);
    eout[(p * 3 + warp) * dr + r] = x;
  }
}

// product state: site s, eta = (t, t') -> v_t conj(v_t') (v host-side complex128 in device copy)
__global__ void vmpo_product_kernel(const double* v, double2* base, long stride, int n) {
  const int s = blockIdx.x, eta = threadIdx.x;
  if (s >= n || eta >= 9) return;
  const int si = eta / 3, sp = eta % 3;
  const double re = v[2 * si] * v[2 * sp] + v[2 * si + 1] * v[2 * sp + 1];
  const double im = v[2 * si + 1] * v[2 * sp] - v[2 * si] * v[2 * sp + 1];
  base[(long)s * stride + eta] = make_double2(re, im);
}

// mirrored site: [l][eta][r] -> [r][eta][l]
__global__ void vmpo_reverse_kernel(int dl, int dr, const double2* __restrict__ in, double2* out) {
  const long total = (long)dl * 9 * dr;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const int r = (int)(e % dr), eta = (int)((e / dr) % 9), l = (int)(e / (9L * dr));
    out[((long)r * 9 + eta) * dl + l] = in[e];
  }
}

inline int nblk(long n) { return (int)std::min<long>((n + 255) / 256, 4096); }

}  // namespace

struct VOp {
  int site = 0;
  std::vector<zc> s, sm;   // pair superoperator and its mirror (sites swapped), 81 x 81
};

struct mpdo_vmpo_s {
  int n = 0, chi = 0, mode = 1;
  double cut2 = 0;
  cudaStream_t st = nullptr;
  bool own_stream = false;
  bool rev = false;
  int centre = 0;                 // user coordinates
  std::vector<int> bond;          // storage coordinates, size n + 1
  size_t site_cap = 0;
  double2* sites = nullptr;
  double2 *th = nullptr, *th2 = nullptr, *H = nullptr, *U = nullptr, *Vh = nullptr;
  double2 *S = nullptr, *x = nullptr, *tl = nullptr, *tr = nullptr;
  double2 *Lenv = nullptr, *Renv = nullptr, *etmp = nullptr, *ebuf = nullptr;
  double *lam = nullptr, *sv = nullptr, *lt = nullptr;
  EigWork<double> eig;
  void* eigmem = nullptr;
  // tensor-core form (mpdo_vmpo_set_precision 1): exact-slice products and the mixed solver
  int tc = 0;
  // factor of the Gram and the graded solver's workspace (see split)
  double2 *L = nullptr, *Gs = nullptr, *Zs = nullptr;
  MixWork gradw;
  void* gradmem = nullptr;
  PcholOut* dpc = nullptr;
  PcholOut* hpc = nullptr;   // pinned
  MixWork mixw;
  void* mixmem = nullptr;
  void* tcws = nullptr;
  size_t tcws_bytes = 0;
  int* tcerr = nullptr;
  int* htcerr = nullptr;   // pinned
  double sv_req = 0;       // requested cut (Schmidt values, relative)
  VScalars* dsc = nullptr;
  VScalars* hsc = nullptr;
  std::vector<void*> allocs;
  std::string err;
  double2* site(int s) const { return sites + (size_t)s * site_cap; }
};

namespace {

int vfail(mpdo_vmpo h, int code, const std::string& msg) {
  if (h) h->err = msg;
  set_global_error(msg.c_str());
  return code;
}
#define VK(expr)                                                                     \
  do {                                                                               \
    cudaError_t _e = (expr);                                                         \
    if (_e != cudaSuccess)                                                           \
      return vfail(h, MPDO_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(_e)); \
  } while (0)

int valloc(mpdo_vmpo h, void** p, size_t bytes) {
  if (dev_malloc(p, bytes ? bytes : 16) != cudaSuccess) {
    cudaGetLastError();
    return vfail(h, MPDO_ERR_OOM, "vmpo: device allocation of " + std::to_string(bytes) + " bytes");
  }
  h->allocs.push_back(*p);
  if (cudaMemsetAsync(*p, 0, bytes ? bytes : 16, h->st) != cudaSuccess) {
    cudaGetLastError();
    return vfail(h, MPDO_ERR_CUDA, "vmpo: clearing a new buffer");
  }
  return MPDO_OK;
}

cudaError_t g64(cudaStream_t st, int opa, int opb, int m, int n, int k, const double2* A, long lda,
                long sa, const double2* B, long ldb, long sb, double2* C, long ldc, long sc,
                int batch) {
  return cgemm<double>(st, opa, opb, m, n, k, A, lda, sa, B, ldb, sb, C, ldc, sc, batch,
                       make_double2(1, 0), make_double2(0, 0));
}

// Products of the update: in the tensor-core form, those of at least 2^21 complex
// multiply-adds (both output sides >= 16) as error-free BF16 slice products summed in FP64
// (carried to ~2^-48 of each operand row's largest entry); FP64 CUDA cores otherwise.
cudaError_t u64(mpdo_vmpo h, int opa, int opb, int m, int n, int k, const double2* A, long lda,
                long sa, const double2* B, long ldb, long sb, double2* C, long ldc, long sc,
                int batch) {
  if (h->tc && ExactRoute{(double)(1 << 21), false}.takes(m, n, k, batch, A == B))
    return tc_cgemm_exact<double2, double2>(h->st, opa, opb, m, n, k, A, lda, sa, B, ldb, sb, C,
                                            ldc, sc, batch, h->tcws, h->tcws_bytes, h->tcerr);
  return g64(h->st, opa, opb, m, n, k, A, lda, sa, B, ldb, sb, C, ldc, sc, batch);
}

// right trace environments Renv[n] (right of site n, storage coords) for all n
int right_envs(mpdo_vmpo h) {
  const long cap = h->chi;
  double2 one = make_double2(1, 0);
  VK(cudaMemcpyAsync(h->Renv + (long)(h->n - 1) * cap, &one, sizeof(double2), cudaMemcpyHostToDevice,
                     h->st));
  for (int s = h->n - 1; s >= 1; --s) {
    const int dl = h->bond[s], dr = h->bond[s + 1];
    // x[(eta, r)] = tau[eta] R[r];  Renv[s-1][l] = sum A[l, (eta, r)] x[(eta, r)]
    count_launch();
    trace_vec_kernel<<<nblk(9L * dr), 256, 0, h->st>>>(dr, h->Renv + (long)s * cap, 1, h->x);
    VK(cudaGetLastError());
    VK(g64(h->st, OP_N, OP_N, dl, 1, 9 * dr, h->site(s), 9L * dr, 0, h->x, 1, 0,
           h->Renv + (long)(s - 1) * cap, 1, 0, 1));
  }
  return MPDO_OK;
}

// left trace environment of site s+1 from that of site s and site s's tensor
int left_env_step(mpdo_vmpo h, int s) {
  const long cap = h->chi;
  const int dl = h->bond[s], dr = h->bond[s + 1];
  count_launch();
  trace_vec_kernel<<<nblk(9L * dl), 256, 0, h->st>>>(dl, h->Lenv + (long)s * cap, 0, h->x);
  VK(cudaGetLastError());
  VK(g64(h->st, OP_N, OP_N, 1, dr, 9 * dl, h->x, 9L * dl, 0, h->site(s), dr, 0,
         h->Lenv + (long)(s + 1) * cap, dr, 0, 1));
  return MPDO_OK;
}

int left_envs_to(mpdo_vmpo h, int upto) {
  double2 one = make_double2(1, 0);
  VK(cudaMemcpyAsync(h->Lenv, &one, sizeof(double2), cudaMemcpyHostToDevice, h->st));
  for (int s = 0; s < upto; ++s) {
    int rc = left_env_step(h, s);
    if (rc) return rc;
  }
  return MPDO_OK;
}

int reverse(mpdo_vmpo h) {
  for (int s = 0; s <= (h->n - 1) / 2; ++s) {
    const int t = h->n - 1 - s;
    const size_t ns = (size_t)h->bond[s] * 9 * h->bond[s + 1];
    const size_t nt = (size_t)h->bond[t] * 9 * h->bond[t + 1];
    count_launch();
    vmpo_reverse_kernel<<<nblk(ns), 256, 0, h->st>>>(h->bond[s], h->bond[s + 1], h->site(s), h->th);
    if (t != s) {
      count_launch();
      vmpo_reverse_kernel<<<nblk(nt), 256, 0, h->st>>>(h->bond[t], h->bond[t + 1], h->site(t),
                                                      h->th2);
    }
    VK(cudaGetLastError());
    VK(cudaMemcpyAsync(h->site(t), h->th, ns * sizeof(double2), cudaMemcpyDeviceToDevice, h->st));
    if (t != s)
      VK(cudaMemcpyAsync(h->site(s), h->th2, nt * sizeof(double2), cudaMemcpyDeviceToDevice, h->st));
  }
  std::reverse(h->bond.begin(), h->bond.end());
  h->rev = !h->rev;
  return MPDO_OK;
}

// Eigenpairs of the Gram in h->H (n x n): *nval eigenvalues in h->lam, descending, and *nvec
// eigenvectors in the columns of h->U (row stride *nvec).  Through the pivoted Cholesky factor
// H ~ L L^+ and the graded solver on L^+ L, as in the MPDO update; a rank beyond the solver's size
// takes the full solve: FP64 Jacobi, or in the tensor-core form the mixed solver, resolved below a
// tenth of the cut.  (Eight sites at chi 16, n = 144: the FP64 Jacobi took 28 ms a solve.)  The factor
// goes down to the rounding of H whatever the cut: what it leaves below its last pivot sums over up to
// n rows and turns the kept pairs, whose values and T_k enter the result one by one (stopping at a
// hundredth of the cut: energies off by 3e-4 at a cut of 1e-2, 1e-8 at 1e-4).  One host
// synchronisation.
int split(mpdo_vmpo h, int n, int* nval, int* nvec) {
  cudaStream_t st = h->st;
  if (n <= 1024) {
    const int rmax = std::min(n, kGradedMax);
    const double tol = h->tc ? 1e-15 : 1e-16;
    VK(pchol<double>(st, n, h->H, rmax, tol, h->L, kGradedMax, &h->dpc->r, &h->dpc->resid));
    VK(cudaMemcpyAsync(h->hpc, h->dpc, sizeof(*h->hpc), cudaMemcpyDeviceToHost, st));
    VK(cudaStreamSynchronize(st));
    const int r = h->hpc->r;
    const PcholFit fit = pchol_fit(*h->hpc, n, rmax, tol);
    if (fit == PcholFit::zero) return vfail(h, MPDO_ERR_NUMERIC, "vmpo: zero or non-finite state");
    if (fit == PcholFit::fits) {
      *nval = r;
      *nvec = h->mode == 1 ? r : std::min(r, h->chi);
      VK(cgemm_gram<double>(st, 0, r, n, h->L, kGradedMax, h->Zs, r));
      VK(heig_graded(st, r, h->Zs, r, h->Gs, r, h->lam, h->gradw, true));
      VK(u64(h, OP_N, OP_N, n, *nvec, r, h->L, kGradedMax, 0, h->Gs, r, 0, h->U, *nvec, 0, 1));
      return MPDO_OK;
    }
  }
  *nval = *nvec = n;
  if (h->tc)
    VK(heig_mixed(st, n, h->H, n, h->U, n, h->lam, 0.1 * h->cut2, h->mixw, nullptr, nullptr,
                  h->mode == 1 ? 0 : h->chi + 1));
  else
    VK(heig<double>(st, n, h->H, n, h->U, n, h->lam, h->eig, 30));
  return MPDO_OK;
}

// one update on storage bond (i, i+1), centre at i; the centre moves to i+1
int update(mpdo_vmpo h, int i, const VOp& op, mpdo_trunc_stats* acc) {
  cudaStream_t st = h->st;
  const int dl = h->bond[i], dm = h->bond[i + 1], dr = h->bond[i + 2];
  const int rows = 9 * dl, cols = 9 * dr;
  const std::vector<zc>& S = h->rev ? op.sm : op.s;
  VK(cudaMemcpyAsync(h->S, S.data(), 81 * 81 * sizeof(double2), cudaMemcpyHostToDevice, st));
  // theta = A_i A_j ; theta' = S on (eta_i, eta_j), batched over l
  VK(u64(h, OP_N, OP_N, rows, cols, dm, h->site(i), dm, 0, h->site(i + 1), cols, 0, h->th, cols,
         0, 1));
  VK(u64(h, OP_N, OP_N, 81, dr, 81, h->S, 81, 0, h->th, dr, 81L * dr, h->th2, dr, 81L * dr, dl));
  // Schmidt decomposition through the Gram theta' theta'^+.  PPT needs T and Lambda of every
  // Schmidt pair, naive mode those that can be kept.
  int nval = 0, nvec = 0;
  if (h->tc) {
    VK(u64(h, OP_N, OP_C, rows, rows, cols, h->th2, cols, 0, h->th2, cols, 0, h->H, rows, 0, 1));
  } else {
    VK(cgemm_gram<double>(st, 1, rows, cols, h->th2, cols, h->H, rows));
  }
  int rc = split(h, rows, &nval, &nvec);
  if (rc) return rc;
  const int ldu = nvec;
  // trace environment: tl = (L (x) tau)^T U ; W = U^+ theta' (row k = Lambda_k V^+_k) ;
  // trw = W (tau (x) R)
  VK(u64(h, OP_C, OP_N, nvec, cols, rows, h->U, ldu, 0, h->th2, cols, 0, h->th, cols, 0, 1));
  if (h->mode == 1) {
    count_launch();
    trace_vec_kernel<<<nblk(rows), 256, 0, st>>>(dl, h->Lenv + (long)i * h->chi, 0, h->x);
    VK(cudaGetLastError());
    VK(g64(st, OP_N, OP_N, 1, nvec, rows, h->x, rows, 0, h->U, ldu, 0, h->tl, nvec, 0, 1));
    count_launch();
    trace_vec_kernel<<<nblk(cols), 256, 0, st>>>(dr, h->Renv + (long)(i + 1) * h->chi, 1,
                                                  h->x + rows);
    VK(cudaGetLastError());
    VK(g64(st, OP_N, OP_N, nvec, 1, cols, h->th, cols, 0, h->x + rows, 1, 0, h->tr, 1, 0, 1));
  }
  count_launch();
  vmpo_cut_kernel<<<1, 32, 0, st>>>(nval, h->lam, h->tl, h->tr, h->cut2, h->chi, h->mode, h->sv,
                                    h->lt, h->dsc);
  VK(cudaGetLastError());
  VK(cudaMemcpyAsync(h->hsc, h->dsc, sizeof(VScalars), cudaMemcpyDeviceToHost, st));
  if (h->tc) VK(cudaMemcpyAsync(h->htcerr, h->tcerr, sizeof(int), cudaMemcpyDeviceToHost, st));
  VK(cudaStreamSynchronize(st));
  if (h->tc && *h->htcerr) return vfail(h, MPDO_ERR_TIMEOUT, "vmpo: a tensor-core pipeline wait gave up");
  if (h->hsc->flags & 1) return vfail(h, MPDO_ERR_NUMERIC, "vmpo: zero or non-finite state");
  const int keep = h->hsc->keep;
  // A_i <- U_keep ; A_{i+1} <- diag(Lambda~ / Lambda) W_keep
  VK(cudaMemcpy2DAsync(h->site(i), keep * sizeof(double2), h->U, ldu * sizeof(double2),
                       keep * sizeof(double2), rows, cudaMemcpyDeviceToDevice, st));
  count_launch();
  scale_rows_kernel<<<nblk((long)keep * cols), 256, 0, st>>>(keep, cols, h->th, cols, h->lt, h->sv,
                                                             h->site(i + 1), cols);
  VK(cudaGetLastError());
  h->bond[i + 1] = keep;
  rc = left_env_step(h, i);
  if (rc) return rc;
  if (acc) {
    acc->disc_bond_w += h->hsc->disc;
    acc->ppt_infeasible += h->hsc->infeasible;
    acc->ppt_clamped += h->hsc->clamped;
    if (h->mode == 1 && h->hsc->theta < acc->ppt_theta_min) acc->ppt_theta_min = h->hsc->theta;
    acc->chi_used_max = std::max(acc->chi_used_max, keep);
    acc->n_updates += 1;
  }
  return MPDO_OK;
}

// host: the pair superoperator of a Kraus set (81 x 81 complex), re-indexed from the
// two-site row-major vec ((s_i,s_j),(s'_i,s'_j)) to the MPO pair ((s_i,s'_i),(s_j,s'_j));
// mirrored: the two sites swapped
void pair_superop(const double* ops, int m, bool mirror, std::vector<zc>& out) {
  out.assign(81 * 81, zc(0, 0));
  for (int q = 0; q < m; ++q) {
    const double* e = ops + 2 * 81 * q;
    auto E = [&](int r, int c) { return zc(e[2 * (r * 9 + c)], e[2 * (r * 9 + c) + 1]); };
    // S[(a,b),(c,d)] = E[a][c] conj(E[b][d]) on two-site indices a = (si,sj) etc.
    for (int si = 0; si < 3; ++si)
      for (int sj = 0; sj < 3; ++sj)
        for (int pi = 0; pi < 3; ++pi)
          for (int pj = 0; pj < 3; ++pj)
            for (int ti = 0; ti < 3; ++ti)
              for (int tj = 0; tj < 3; ++tj)
                for (int ui = 0; ui < 3; ++ui)
                  for (int uj = 0; uj < 3; ++uj) {
                    // ket (si,sj) <- (ti,tj), bra (pi,pj) <- (ui,uj)
                    const zc v = E(si * 3 + sj, ti * 3 + tj) * std::conj(E(pi * 3 + pj, ui * 3 + uj));
                    int etai = si * 3 + pi, etaj = sj * 3 + pj;    // output MPO pair
                    int mui = ti * 3 + ui, muj = tj * 3 + uj;      // input MPO pair
                    if (mirror) {
                      std::swap(etai, etaj);
                      std::swap(mui, muj);
                    }
                    out[(etai * 9 + etaj) * 81 + mui * 9 + muj] += v;
                  }
  }
}

}  // namespace

extern "C" {

int mpdo_vmpo_create(int n_sites, int chi_max, int use_ppt, double sv_cutoff,
                     const double* init_site_vec, void* cuda_stream, mpdo_vmpo* out) {
  if (n_sites < 2 || chi_max < 1 || chi_max > 256 || !out)
    return vfail(nullptr, MPDO_ERR_ARG, "vmpo: n_sites >= 2 and chi_max in 1..256 required");
  std::unique_ptr<mpdo_vmpo_s> hp(new (std::nothrow) mpdo_vmpo_s());
  if (!hp) return vfail(nullptr, MPDO_ERR_OOM, "vmpo: host allocation");
  mpdo_vmpo h = hp.get();
  h->n = n_sites;
  h->chi = chi_max;
  h->mode = use_ppt ? 1 : 0;
  // Gram eigenvalues resolve to ~1e-16 of the largest: Schmidt values below sqrt(1e-15) of
  // the largest are numerical zeros whatever cut is asked for
  const double sv = sv_cutoff > 0 ? sv_cutoff : 1e-14;
  h->sv_req = sv;
  h->cut2 = std::max(sv * sv, 1e-15);
  if (cuda_stream) {
    h->st = static_cast<cudaStream_t>(cuda_stream);
  } else {
    if (cudaStreamCreateWithFlags(&h->st, cudaStreamNonBlocking) != cudaSuccess) {
      cudaGetLastError();
      return vfail(nullptr, MPDO_ERR_CUDA, "vmpo: stream creation");
    }
    h->own_stream = true;
  }
  h->bond.assign(n_sites + 1, 1);
  const long D = chi_max, n9 = 9 * D;
  h->site_cap = (size_t)D * 9 * D;
  auto A = [&](void** p, size_t count) { return valloc(h, p, count * sizeof(double2)); };
  int rc;
  if ((rc = A((void**)&h->sites, h->site_cap * n_sites)) || (rc = A((void**)&h->th, n9 * n9)) ||
      (rc = A((void**)&h->th2, n9 * n9)) || (rc = A((void**)&h->H, n9 * n9)) ||
      (rc = A((void**)&h->U, n9 * n9)) || (rc = A((void**)&h->S, 81 * 81)) ||
      (rc = A((void**)&h->x, 2 * n9)) || (rc = A((void**)&h->tl, n9)) ||
      (rc = A((void**)&h->tr, n9)) ||
      (rc = A((void**)&h->Lenv, (size_t)(n_sites + 1) * D)) ||
      (rc = A((void**)&h->Renv, (size_t)(n_sites + 1) * D)) ||
      (rc = A((void**)&h->ebuf, 12 * D)) ||
      (rc = valloc(h, (void**)&h->lam, n9 * sizeof(double))) ||
      (rc = valloc(h, (void**)&h->sv, n9 * sizeof(double))) ||
      (rc = valloc(h, (void**)&h->lt, n9 * sizeof(double))) ||
      (rc = valloc(h, (void**)&h->dsc, sizeof(VScalars))) ||
      (rc = A((void**)&h->L, (size_t)n9 * kGradedMax)) ||
      (rc = A((void**)&h->Gs, (size_t)kGradedMax * kGradedMax)) ||
      (rc = A((void**)&h->Zs, (size_t)kGradedMax * kGradedMax)) ||
      (rc = valloc(h, (void**)&h->dpc, sizeof(*h->dpc))) ||
      (rc = valloc(h, &h->gradmem, mix_work_bytes((int)std::min<long>(n9, kGradedMax)))) ||
      (rc = valloc(h, &h->eigmem, eig_work_bytes<double>((int)n9)))) {
    mpdo_vmpo_destroy(hp.release());
    return rc;
  }
  eig_work_bind<double>(h->eig, h->eigmem, (int)n9);
  mix_work_bind(h->gradw, h->gradmem, (int)std::min<long>(n9, kGradedMax));
  if (cudaMallocHost((void**)&h->hsc, sizeof(VScalars)) != cudaSuccess ||
      cudaMallocHost((void**)&h->hpc, sizeof(*h->hpc)) != cudaSuccess) {
    cudaGetLastError();
    mpdo_vmpo_destroy(hp.release());
    return vfail(nullptr, MPDO_ERR_OOM, "vmpo: pinned host allocation");
  }
  double pl[6] = {1.0 / std::sqrt(2.0), 0, 1.0 / std::sqrt(2.0), 0, 0, 0};
  const double* v = init_site_vec ? init_site_vec : pl;
  double* dv = nullptr;
  if ((rc = valloc(h, (void**)&dv, 6 * sizeof(double)))) {
    mpdo_vmpo_destroy(hp.release());
    return rc;
  }
  cudaMemcpyAsync(dv, v, 6 * sizeof(double), cudaMemcpyHostToDevice, h->st);
  count_launch();
  vmpo_product_kernel<<<n_sites, 32, 0, h->st>>>(dv, h->sites, (long)h->site_cap, n_sites);
  if (cudaGetLastError() != cudaSuccess || (rc = right_envs(h)) || (rc = left_envs_to(h, 0)) ||
      cudaStreamSynchronize(h->st) != cudaSuccess) {
    mpdo_vmpo_destroy(hp.release());
    return rc ? rc : vfail(nullptr, MPDO_ERR_CUDA, "vmpo: initial state");
  }
  *out = hp.release();
  return MPDO_OK;
}

int mpdo_vmpo_apply_layer(mpdo_vmpo h, const mpdo_layer* layer, mpdo_trunc_stats* stats) {
  if (!h || !layer || layer->n_ops < 0 || (layer->n_ops > 0 && !layer->ops))
    return vfail(h, MPDO_ERR_ARG, "vmpo: bad layer");
  std::vector<VOp> ops(layer->n_ops);
  for (int k = 0; k < layer->n_ops; ++k) {
    const mpdo_op& op = layer->ops[k];
    if (op.kind != 2 || op.site < 0 || op.site > h->n - 2 || op.n_kraus < 1 || !op.ops)
      return vfail(h, MPDO_ERR_ARG, "vmpo: ops must be two-site channels within the chain");
    for (int a = 0; a < 2 * 81 * op.n_kraus; ++a)
      if (!std::isfinite(op.ops[a])) return vfail(h, MPDO_ERR_NUMERIC, "vmpo: non-finite op");
    ops[k].site = op.site;
    pair_superop(op.ops, op.n_kraus, false, ops[k].s);
    pair_superop(op.ops, op.n_kraus, true, ops[k].sm);
  }
  mpdo_trunc_stats acc{};
  acc.ppt_theta_min = 1e300;
  for (const VOp& op : ops) {
    const int i = op.site;
    bool ltr;
    if (h->centre == i) ltr = true;
    else if (h->centre == i + 1) ltr = false;
    else return vfail(h, MPDO_ERR_STATE, "vmpo: two-site op does not touch the centre");
    int rc;
    if (ltr == h->rev) {
      // the storage runs along the update direction: mirror, then rebuild the environments
      if ((rc = reverse(h)) || (rc = right_envs(h))) return rc;
      const int cs = h->rev ? h->n - 1 - h->centre : h->centre;
      if ((rc = left_envs_to(h, cs))) return rc;
    }
    const int is = h->rev ? h->n - 2 - i : i;
    if ((rc = update(h, is, op, &acc))) return rc;
    h->centre = ltr ? i + 1 : i;
  }
  if (stats) *stats = acc;
  return MPDO_OK;
}

int mpdo_vmpo_expect_energy(mpdo_vmpo h, double J, double hx, double b, double* e_raw,
                            double* e_success, double* success_prob, double* trace) {
  if (!h) return vfail(nullptr, MPDO_ERR_ARG, "vmpo: null handle");
  // env [2][3][D]: start E0 = 1, E1 = E2 = 0 for both projectors
  const long D = h->chi;
  double2* ein = h->ebuf;
  double2* eout = h->ebuf + 6 * D;
  // packed [projector][state][bond] with the bond dimension 1 of the chain's left end
  std::vector<double2> init(6 * D, make_double2(0, 0));
  init[0] = make_double2(1, 0);
  init[3] = make_double2(1, 0);
  VK(cudaMemcpyAsync(ein, init.data(), sizeof(double2) * 6 * D, cudaMemcpyHostToDevice, h->st));
  for (int s = 0; s < h->n; ++s) {
    const int dl = h->bond[s], dr = h->bond[s + 1];
    count_launch();
    vmpo_energy_kernel<<<dim3((dr + 31) / 32, 2), 256, 0, h->st>>>(dl, dr, h->site(s), ein, eout, J,
                                                                  hx, b);
    VK(cudaGetLastError());
    std::swap(ein, eout);
  }
  double2 res[6];
  VK(cudaMemcpyAsync(res, ein, sizeof(res), cudaMemcpyDeviceToHost, h->st));
  VK(cudaStreamSynchronize(h->st));
  // the final bond dimension is 1: state q of projector p sits at ein[(p*3+q)*1]
  const double norm = res[0].x, tot = res[2].x, ps = res[3].x, tots = res[5].x;
  if (!(norm != 0) || !std::isfinite(norm)) return vfail(h, MPDO_ERR_NUMERIC, "vmpo: zero trace");
  if (e_raw) *e_raw = tot / norm;
  if (e_success) *e_success = ps != 0 ? tots / ps : NAN;
  if (success_prob) *success_prob = ps;
  if (trace) *trace = norm;
  return MPDO_OK;
}

int mpdo_vmpo_purity(mpdo_vmpo h, double* purity) {
  if (!h || !purity) return vfail(h, MPDO_ERR_ARG, "vmpo: null argument");
  // canonical gauge: <<rho|rho>> is the centre's squared Frobenius norm
  const int c = h->rev ? h->n - 1 - h->centre : h->centre;
  const long cnt = (long)h->bond[c] * 9 * h->bond[c + 1];
  double* d = h->lam;
  VK(sumsq<double>(h->st, cnt, h->site(c), d));
  VK(cudaMemcpyAsync(purity, d, sizeof(double), cudaMemcpyDeviceToHost, h->st));
  VK(cudaStreamSynchronize(h->st));
  return MPDO_OK;
}

int mpdo_vmpo_collision(mpdo_vmpo h, double* collision) {
  if (!h || !collision) return vfail(h, MPDO_ERR_ARG, "vmpo: null argument");
  // rho_xx = prod_n A_n[., (s_n, s_n), .]: E <- sum_s A_s^T E A_s (D x D, the pair of copies)
  // and t <- sum_s t A_s (the trace), with A_s = A_n[:, (s, s), :] (rows of stride 9 D_r);
  // the site order of the storage does not matter for a sum over all x
  const long D = h->chi;
  double2* E = h->th;              // D x D
  double2* En = E + D * D;         // D x D
  double2* T = En + D * D;         // 3 x D x D
  double2* t = T + 3 * D * D;      // D
  double2* tn = t + D;             // D
  const double2 one = make_double2(1, 0), zero = make_double2(0, 0);
  VK(cudaMemcpyAsync(E, &one, sizeof(double2), cudaMemcpyHostToDevice, h->st));
  VK(cudaMemcpyAsync(t, &one, sizeof(double2), cudaMemcpyHostToDevice, h->st));
  for (int s = 0; s < h->n; ++s) {
    const int dl = h->bond[s], dr = h->bond[s + 1];
    const double2* A = h->site(s);
    const long la = 9L * dr, sd = 4L * dr;   // diagonal eta = 0, 4, 8
    // T_s = E A_s, batched over the three diagonal entries
    VK(cgemm<double>(h->st, OP_N, OP_N, dl, dr, dl, E, dl, 0, A, la, sd, T, dr, (long)dl * dr, 3,
                     one, zero));
    for (int q = 0; q < 3; ++q) {
      VK(cgemm<double>(h->st, OP_T, OP_N, dr, dr, dl, A + q * sd, la, 0, T + (long)q * dl * dr, dr,
                       0, En, dr, 0, 1, one, q ? one : zero));
      VK(cgemm<double>(h->st, OP_N, OP_N, 1, dr, dl, t, dl, 0, A + q * sd, la, 0, tn, dr, 0, 1,
                       one, q ? one : zero));
    }
    std::swap(E, En);
    std::swap(t, tn);
  }
  double2 r[2];
  VK(cudaMemcpyAsync(&r[0], E, sizeof(double2), cudaMemcpyDeviceToHost, h->st));
  VK(cudaMemcpyAsync(&r[1], t, sizeof(double2), cudaMemcpyDeviceToHost, h->st));
  VK(cudaStreamSynchronize(h->st));
  if (!(r[1].x != 0) || !std::isfinite(r[1].x)) return vfail(h, MPDO_ERR_NUMERIC, "vmpo: zero trace");
  *collision = r[0].x / (r[1].x * r[1].x);
  return MPDO_OK;
}

int mpdo_vmpo_get_dims(mpdo_vmpo h, int* bond_dims, int* centre) {
  if (!h) return vfail(nullptr, MPDO_ERR_ARG, "vmpo: null handle");
  for (int u = 0; u < h->n - 1; ++u) {
    const int s = h->rev ? h->n - 1 - u : u;
    if (bond_dims) bond_dims[u] = h->rev ? h->bond[s] : h->bond[s + 1];
  }
  if (centre) *centre = h->centre;
  return MPDO_OK;
}

int mpdo_vmpo_set_precision(mpdo_vmpo h, int mode) {
  if (!h || (mode != 0 && mode != 1)) return vfail(h, MPDO_ERR_ARG, "vmpo: mode must be 0 or 1");
  if (mode == 1 && !h->mixmem) {
    const int n9 = 9 * h->chi;
    const size_t tw = (size_t)256 << 20;
    int rc;
    if ((rc = valloc(h, &h->mixmem, mix_work_bytes(n9))) || (rc = valloc(h, &h->tcws, tw)) ||
        (rc = valloc(h, (void**)&h->tcerr, sizeof(int)))) {
      h->mixmem = nullptr;
      return rc;
    }
    if (cudaMallocHost((void**)&h->htcerr, sizeof(int)) != cudaSuccess) {
      cudaGetLastError();
      h->htcerr = nullptr;
      h->mixmem = nullptr;
      return vfail(h, MPDO_ERR_OOM, "vmpo: pinned host allocation");
    }
    *h->htcerr = 0;
    mix_work_bind(h->mixw, h->mixmem, n9);
    h->mixw.tcws = h->tcws;
    h->mixw.tcws_bytes = tw;
    h->mixw.tcerr = h->tcerr;
    h->mixw.tc_min_macs = (double)(1 << 21);
    h->tcws_bytes = tw;
  }
  h->tc = mode;
  // the mixed solver resolves eigenvalues to ~1e-14 of the largest: numerical zeros below
  // 10 x that in the tensor-core form, below 1e-15 in FP64
  h->cut2 = std::max(h->sv_req * h->sv_req, mode ? 1e-13 : 1e-15);
  VK(cudaStreamSynchronize(h->st));
  return MPDO_OK;
}

int mpdo_vmpo_destroy(mpdo_vmpo h) {
  if (!h) return MPDO_OK;
  if (h->st) cudaStreamSynchronize(h->st);
  mix_work_release(h->mixw);
  for (void* p : h->allocs) cudaFree(p);
  if (h->hsc) cudaFreeHost(h->hsc);
  if (h->hpc) cudaFreeHost(h->hpc);
  if (h->htcerr) cudaFreeHost(h->htcerr);
  if (h->own_stream) cudaStreamDestroy(h->st);
  delete h;
  return MPDO_OK;
}

}  // extern "C"
