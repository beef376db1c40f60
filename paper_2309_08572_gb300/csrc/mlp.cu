// MLP surrogate on the GPU: forward, backward and Adam kernels (FP32), behind the C ABI.
//
// Not a method of the paper: a small fully connected network (tanh hidden layers, linear
// output) learns (energy per site, success probability) of noisy QAOA circuits from
// samples the MPDO engine produced, and its input gradient proposes angles that the
// engine then re-scores.
//   forward   z_l = a_{l-1} W_l + b_l, a_l = tanh(z_l) (hidden), a_L = z_L
//   loss      mean over batch and outputs of (a_L - t)^2
//   backward  dz_L = 2 (a_L - t) / (B n_out), dz_l = da_l (1 - a_l^2),
//             dW_l = a_{l-1}^T dz_l, db_l = column sums of dz_l, da_{l-1} = dz_l W_l^T
//   Adam      (Kingma & Ba) with bias correction.
// Weights are stored [fan_in][fan_out] row-major, one flat FP32 array W_0 b_0 W_1 b_1 ...
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "../../include/mpdo.h"
#include "common.cuh"
#include "tcgemm.h"

namespace mpdo {
void set_global_error(const char* msg);
}

namespace {

constexpr int SBM = 64, SBN = 64, SBK = 16, SNT = 256;

// C = op(A) op(B), A is M x K after op, B is K x N after op (row-major storage); then, where given,
// + bias per column, tanh (act), and times 1 - a^2 (a like C): passes of their own over the small
// matrices would each cost a launch.
__global__ void __launch_bounds__(SNT) sgemm_kernel(int M, int N, int K, const float* __restrict__ A,
                                                    long sam, long sak, const float* __restrict__ B,
                                                    long sbk, long sbn, float* C, long ldc,
                                                    const float* __restrict__ bias, int act,
                                                    const float* __restrict__ a2) {
  __shared__ float As[SBK][SBM + 4];
  __shared__ float Bs[SBK][SBN + 4];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * SBM, n0 = blockIdx.x * SBN;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += SBK) {
    for (int e = tid; e < SBM * SBK; e += SNT) {
      int mi, ki;
      if (sak == 1) { mi = e / SBK; ki = e % SBK; } else { ki = e / SBM; mi = e % SBM; }
      int gm = m0 + mi, gk = k0 + ki;
      As[ki][mi] = (gm < M && gk < K) ? A[gm * sam + gk * sak] : 0.f;
    }
    for (int e = tid; e < SBN * SBK; e += SNT) {
      int ni, ki;
      if (sbn == 1) { ki = e / SBN; ni = e % SBN; } else { ni = e / SBK; ki = e % SBK; }
      int gn = n0 + ni, gk = k0 + ki;
      Bs[ki][ni] = (gn < N && gk < K) ? B[gk * sbk + gn * sbn] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < SBK; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int gm = m0 + ty + 16 * i;
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int gn = n0 + tx + 16 * j;
      if (gn >= N) continue;
      float v = acc[i][j] + (bias ? bias[gn] : 0.f);
      if (act) v = tanhf(v);
      if (a2) {
        const float x = a2[gm * ldc + gn];
        v *= (1.f - x * x);
      }
      C[gm * ldc + gn] = v;
    }
  }
}

// dz = 2 (y - t) / (B n_out); per-block partial sums of (y - t)^2 into part[]
__global__ void mse_grad_kernel(long n, float scale, const float* __restrict__ y,
                                const float* __restrict__ t, float* dz, double* part) {
  __shared__ double red[256];
  double s = 0;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
    float d = y[e] - t[e];
    dz[e] = 2.f * d * scale;
    s += (double)d * d;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// db[j] = sum_i dz[i][j]: 32 columns a block, the rows over eight warps (one thread a column took
// 31 us at 512 rows), added in a fixed order.
__global__ void __launch_bounds__(256) colsum_kernel(int rows, int cols, const float* __restrict__ dz,
                                                     float* db) {
  __shared__ float part[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (j < cols)
    for (int i = warp; i < rows; i += 8) s += dz[(long)i * cols + j];
  part[warp][lane] = s;
  __syncthreads();
  if (warp || j >= cols) return;
  for (int w = 1; w < 8; ++w) s += part[w][lane];
  db[j] = s;
}

__global__ void fill_rows_kernel(int rows, int cols, const float* __restrict__ v, float* out) {
  long n = (long)rows * cols;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
    out[e] = v[e % cols];
}

__global__ void adam_kernel(long n, float lr, float b1, float b2, float eps, float c1, float c2,
                            const float* __restrict__ g, float* m, float* v, float* p) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
    float gi = g[e];
    float mi = b1 * m[e] + (1.f - b1) * gi;
    float vi = b2 * v[e] + (1.f - b2) * gi * gi;
    m[e] = mi;
    v[e] = vi;
    p[e] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

inline int nb(long n) {
  long b = (n + 255) / 256;
  return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

}  // namespace

struct mpdo_mlp_s {
  cudaStream_t st = nullptr;
  bool own_stream = false;
  std::vector<int> w;       // widths, size L+1
  int max_batch = 0;
  long n_params = 0;
  std::vector<long> woff, boff;
  float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
  std::vector<float*> acts;  // L+1 buffers, [max_batch][w_l]
  float *da = nullptr, *db2 = nullptr;  // two scratch [max_batch][max width]
  double* part = nullptr;
  double* hpart = nullptr;   // pinned
  int t = 0;
  int maxw = 0;
  std::string err;
  // BF16 tensor-core products (mpdo_mlp_set_precision): the operands of every layer, the parts of
  // the bias gradients and the loss, and the pipeline's error flag in one allocation; the
  // parameters, gradients and Adam moments stay FP32
  int tc = 0;
  void* tcmem = nullptr;
  std::vector<__nv_bfloat16*> xr, xc, zr, zc;   // activations and dz (index: layer's units), K-major
  std::vector<__nv_bfloat16*> wr, wt;           // weights as they are and transposed
  std::vector<float*> csum;
  double* lpart = nullptr;
  struct TcOut { double loss; int err, pad; };
  TcOut* tcout = nullptr;
  long ldb = 0;                                 // row stride of xc and zc
};

namespace {

int mlp_fail(mpdo_mlp m, int code, const std::string& msg) {
  if (m) m->err = msg;
  mpdo::set_global_error(msg.c_str());
  return code;
}

#define MK(expr)                                                                      \
  do {                                                                                \
    cudaError_t _e = (expr);                                                          \
    if (_e != cudaSuccess) return mlp_fail(m, MPDO_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(_e)); \
  } while (0)

// C = op(A) op(B), A is M x K after op, B is K x N after op, in FP32 on the CUDA cores, with
// sgemm_kernel's elementwise work.
cudaError_t sgemm(mpdo_mlp m, bool ta, bool tb, int M, int N, int K, const float* A, long lda,
                  const float* B, long ldb, float* C, long ldc, const float* bias, int act,
                  const float* a2) {
  long sam = ta ? 1 : lda, sak = ta ? lda : 1;
  long sbk = tb ? 1 : ldb, sbn = tb ? ldb : 1;
  dim3 grid((N + SBN - 1) / SBN, (M + SBM - 1) / SBM);
  mpdo::count_launch();
  sgemm_kernel<<<grid, SNT, 0, m->st>>>(M, N, K, A, sam, sak, B, sbk, sbn, C, ldc, bias, act, a2);
  return cudaGetLastError();
}

// layers [0, n) of the forward pass into m->acts; y: where the output goes if n is all of them
int run_forward(mpdo_mlp m, int batch, int n, const float* x, float* y) {
  const int L = (int)m->w.size() - 1;
  for (int l = 0; l < n; ++l)
    MK(sgemm(m, false, false, batch, m->w[l + 1], m->w[l], l ? m->acts[l] : x, m->w[l],
             m->params + m->woff[l], m->w[l + 1], l == L - 1 ? y : m->acts[l + 1], m->w[l + 1],
             m->params + m->boff[l], l < L - 1, nullptr));
  return MPDO_OK;
}

// backward from d(output) in m->da: the gradients of the parameters (x) or of the input (gx)
int run_backward(mpdo_mlp m, int batch, const float* x, float* gx) {
  const int L = (int)m->w.size() - 1;
  float* cur = m->da;
  float* nxt = m->db2;
  for (int l = L - 1; l >= 0; --l) {
    const int fi = m->w[l], fo = m->w[l + 1];
    if (!gx) {
      // dW = a_{l-1}^T dz  (fi x fo), db = colsum(dz)
      MK(sgemm(m, true, false, fi, fo, batch, l ? m->acts[l] : x, fi, cur, fo,
               m->grads + m->woff[l], fo, nullptr, 0, nullptr));
      mpdo::count_launch();
      colsum_kernel<<<(fo + 31) / 32, 256, 0, m->st>>>(batch, fo, cur, m->grads + m->boff[l]);
      MK(cudaGetLastError());
      if (l == 0) break;
    }
    // dz_l = (dz_{l+1} W^T) (1 - a_l^2)  (batch x fi)
    MK(sgemm(m, false, true, batch, fi, fo, cur, fo, m->params + m->woff[l], fo, l ? nxt : gx, fi,
             nullptr, 0, l ? m->acts[l] : nullptr));
    std::swap(cur, nxt);
  }
  return MPDO_OK;
}

// ---- the same on the tensor cores (mpdo_mlp_set_precision)
inline long r8(long x) { return (x + 7) / 8 * 8; }   // 16-byte rows

// BF16 operands of the pass: the weights (tr: transposed, for the forward pass; pl: as they are,
// for the backward one), x, and wout on every row of the output's dz
int tc_operands(mpdo_mlp m, int batch, const float* x, bool pl, bool xcol, const float* wout) {
  const int L = (int)m->w.size() - 1;
  mpdo::MlpPack g;
  g.count = 0;
  g.job[g.count++] = {x, m->w[0], batch, m->w[0], 0, m->xr[0], xcol ? m->xc[0] : nullptr,
                      r8(m->w[0]), m->ldb};
  for (int l = 0; l < L; ++l)
    g.job[g.count++] = {m->params + m->woff[l], m->w[l + 1], m->w[l], m->w[l + 1], 0,
                        pl ? m->wr[l] : nullptr, m->wt[l], r8(m->w[l + 1]), r8(m->w[l])};
  if (wout)
    g.job[g.count++] = {wout, 0, batch, m->w[L], 0, m->zr[L], nullptr, r8(m->w[L]), 0};
  MK(mpdo::mlp_pack(m->st, g));
  return MPDO_OK;
}

int tc_product(mpdo_mlp m, const __nv_bfloat16* A, const __nv_bfloat16* B, int M, int N, int K,
               const mpdo::MlpEpi& e) {
  mpdo::MlpGroup<1> g = {};
  mpdo::MlpProd& p = g.p[0];
  p.A = A; p.B = B; p.lda = p.ldb = r8(K);
  p.M = M; p.N = N; p.K = K;
  p.e = e;
  g.count = 1;
  MK(mpdo::mlp_products<1>(m->st, g, &m->tcout->err));
  return MPDO_OK;
}

// layers [0, n): hidden ones into m->acts and the operands of the next product (and, train, of the
// weight gradients); the output layer by `out`
int tc_forward(mpdo_mlp m, int batch, int n, bool train, const mpdo::MlpEpi& out) {
  const int L = (int)m->w.size() - 1;
  for (int l = 0; l < n; ++l) {
    const int fo = m->w[l + 1];
    mpdo::MlpEpi e = {};
    if (l < L - 1) {
      e.act = 1;
      e.d = m->acts[l + 1]; e.ldd = fo;
      e.row = m->xr[l + 1]; e.ldr = r8(fo);
      if (train) { e.col = m->xc[l + 1]; e.ldc = m->ldb; }
    } else {
      e = out;
    }
    e.bias = m->params + m->boff[l];
    int rc = tc_product(m, m->xr[l], m->wt[l], batch, fo, m->w[l], e);
    if (rc) return rc;
  }
  return MPDO_OK;
}

// from the output's dz (zr[L], zc[L], csum[L]): the gradients of the parameters and the loss, or
// of the input
int tc_backward(mpdo_mlp m, int batch, float* gx) {
  const int L = (int)m->w.size() - 1;
  for (int l = L - 1; l >= (gx ? 0 : 1); --l) {
    const int fi = m->w[l], fo = m->w[l + 1];
    mpdo::MlpEpi e = {};
    if (l) {
      e.a = m->acts[l]; e.lda = fi;
      e.row = m->zr[l]; e.ldr = r8(fi);
      if (!gx) { e.col = m->zc[l]; e.ldc = m->ldb; e.csum = m->csum[l]; }
    } else {
      e.d = gx; e.ldd = fi;
    }
    int rc = tc_product(m, m->zr[l + 1], m->wr[l], batch, fi, fo, e);
    if (rc) return rc;
  }
  if (gx) return MPDO_OK;
  mpdo::MlpGroup<mpdo::kMlpMaxLayers> g = {};
  for (int l = 0; l < L; ++l) {
    mpdo::MlpProd& p = g.p[l];
    p.A = m->xc[l]; p.B = m->zc[l + 1]; p.lda = p.ldb = m->ldb;
    p.M = m->w[l]; p.N = m->w[l + 1]; p.K = batch;
    p.e.d = m->grads + m->woff[l]; p.e.ldd = m->w[l + 1];
    p.sum_in = m->csum[l + 1]; p.sum_out = m->grads + m->boff[l];
  }
  g.count = L;
  g.parts = (batch + 31) / 32;
  g.loss = m->lpart;
  g.loss_n = (long)g.parts * ((m->w[L] + 31) / 32);
  g.loss_sum = &m->tcout->loss;
  MK(mpdo::mlp_products<mpdo::kMlpMaxLayers>(m->st, g, &m->tcout->err));
  return MPDO_OK;
}

}  // namespace

extern "C" {

int mpdo_mlp_create(int n_layers, const int* widths, int max_batch, void* stream, mpdo_mlp* out) {
  if (n_layers < 1 || n_layers > 16 || !widths || max_batch < 1 || !out)
    return mlp_fail(nullptr, MPDO_ERR_ARG, "mlp: bad create arguments");
  for (int l = 0; l <= n_layers; ++l)
    if (widths[l] < 1 || widths[l] > 4096) return mlp_fail(nullptr, MPDO_ERR_ARG, "mlp: width out of 1..4096");
  mpdo_mlp m = new (std::nothrow) mpdo_mlp_s();
  if (!m) return mlp_fail(nullptr, MPDO_ERR_OOM, "mlp: host allocation");
  m->w.assign(widths, widths + n_layers + 1);
  m->max_batch = max_batch;
  long off = 0;
  for (int l = 0; l < n_layers; ++l) {
    m->woff.push_back(off);
    off += (long)m->w[l] * m->w[l + 1];
    m->boff.push_back(off);
    off += m->w[l + 1];
  }
  m->n_params = off;
  for (int x : m->w) m->maxw = std::max(m->maxw, x);
  if (stream) {
    m->st = static_cast<cudaStream_t>(stream);
  } else {
    if (cudaStreamCreateWithFlags(&m->st, cudaStreamNonBlocking) != cudaSuccess) {
      delete m;
      return mlp_fail(nullptr, MPDO_ERR_CUDA, "mlp: stream creation");
    }
    m->own_stream = true;
  }
  bool ok = mpdo::dev_malloc(&m->params, sizeof(float) * off) == cudaSuccess &&
            mpdo::dev_malloc(&m->grads, sizeof(float) * off) == cudaSuccess &&
            mpdo::dev_malloc(&m->m, sizeof(float) * off) == cudaSuccess &&
            mpdo::dev_malloc(&m->v, sizeof(float) * off) == cudaSuccess &&
            mpdo::dev_malloc(&m->da, sizeof(float) * (size_t)max_batch * m->maxw) == cudaSuccess &&
            mpdo::dev_malloc(&m->db2, sizeof(float) * (size_t)max_batch * m->maxw) == cudaSuccess &&
            mpdo::dev_malloc(&m->part, sizeof(double) * 4096) == cudaSuccess &&
            cudaMallocHost(&m->hpart, sizeof(double) * 4096) == cudaSuccess;
  for (int l = 0; ok && l <= n_layers; ++l) {
    float* p = nullptr;
    ok = mpdo::dev_malloc(&p, sizeof(float) * (size_t)max_batch * m->w[l]) == cudaSuccess;
    m->acts.push_back(p);
  }
  if (!ok) {
    cudaGetLastError();
    mpdo_mlp_destroy(m);
    return mlp_fail(nullptr, MPDO_ERR_OOM, "mlp: device allocation");
  }
  cudaMemsetAsync(m->params, 0, sizeof(float) * off, m->st);
  cudaMemsetAsync(m->m, 0, sizeof(float) * off, m->st);
  cudaMemsetAsync(m->v, 0, sizeof(float) * off, m->st);
  cudaStreamSynchronize(m->st);
  *out = m;
  return MPDO_OK;
}

long long mpdo_mlp_n_params(mpdo_mlp m) { return m ? m->n_params : -1; }

int mpdo_mlp_set_params(mpdo_mlp m, const float* host) {
  if (!m || !host) return mlp_fail(m, MPDO_ERR_ARG, "mlp: null argument");
  for (long i = 0; i < m->n_params; ++i)
    if (!std::isfinite(host[i])) return mlp_fail(m, MPDO_ERR_NUMERIC, "mlp: non-finite parameter");
  MK(cudaMemcpyAsync(m->params, host, sizeof(float) * m->n_params, cudaMemcpyHostToDevice, m->st));
  MK(cudaMemsetAsync(m->m, 0, sizeof(float) * m->n_params, m->st));
  MK(cudaMemsetAsync(m->v, 0, sizeof(float) * m->n_params, m->st));
  MK(cudaStreamSynchronize(m->st));
  m->t = 0;
  return MPDO_OK;
}

int mpdo_mlp_get_params(mpdo_mlp m, float* host) {
  if (!m || !host) return mlp_fail(m, MPDO_ERR_ARG, "mlp: null argument");
  MK(cudaMemcpyAsync(host, m->params, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost, m->st));
  MK(cudaStreamSynchronize(m->st));
  return MPDO_OK;
}

int mpdo_mlp_forward(mpdo_mlp m, int batch, const float* x, float* y) {
  if (!m || !x || !y || batch < 1 || batch > m->max_batch) return mlp_fail(m, MPDO_ERR_ARG, "mlp: bad forward arguments");
  const int L = (int)m->w.size() - 1;
  if (!m->tc) {
    if (L == 1) {   // the one product reads x while it writes y, which may be the same memory
      MK(cudaMemcpyAsync(m->acts[0], x, sizeof(float) * (size_t)batch * m->w[0],
                         cudaMemcpyDeviceToDevice, m->st));
      x = m->acts[0];
    }
    return run_forward(m, batch, L, x, y);
  }
  int rc = tc_operands(m, batch, x, false, false, nullptr);
  if (rc) return rc;
  mpdo::MlpEpi e = {};
  e.d = y; e.ldd = m->w[L];
  return tc_forward(m, batch, L, false, e);
}

int mpdo_mlp_loss_grad(mpdo_mlp m, int batch, const float* x, const float* t, float* loss,
                       float* grad_host) {
  if (!m || !x || !t || batch < 1 || batch > m->max_batch) return mlp_fail(m, MPDO_ERR_ARG, "mlp: bad loss_grad arguments");
  const int L = (int)m->w.size() - 1;
  const long n = (long)batch * m->w[L];
  int rc, blocks = 0;
  if (m->tc) {
    if ((rc = tc_operands(m, batch, x, true, true, nullptr))) return rc;
    mpdo::MlpEpi e = {};
    e.t = t; e.scale = 1.f / (float)n; e.loss = m->lpart;
    e.row = m->zr[L]; e.ldr = r8(m->w[L]);
    e.col = m->zc[L]; e.ldc = m->ldb;
    e.csum = m->csum[L];
    if ((rc = tc_forward(m, batch, L, true, e))) return rc;
    if ((rc = tc_backward(m, batch, nullptr))) return rc;
    MK(cudaMemcpyAsync(m->hpart, m->tcout, sizeof(mpdo_mlp_s::TcOut), cudaMemcpyDeviceToHost, m->st));
  } else {
    if ((rc = run_forward(m, batch, L, x, m->acts[L]))) return rc;
    blocks = nb(n);
    mpdo::count_launch();
    mse_grad_kernel<<<blocks, 256, 0, m->st>>>(n, 1.f / (float)n, m->acts[L], t, m->da, m->part);
    MK(cudaGetLastError());
    if ((rc = run_backward(m, batch, x, nullptr))) return rc;
    MK(cudaMemcpyAsync(m->hpart, m->part, sizeof(double) * blocks, cudaMemcpyDeviceToHost, m->st));
  }
  if (grad_host) MK(cudaMemcpyAsync(grad_host, m->grads, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost, m->st));
  MK(cudaStreamSynchronize(m->st));
  double s = 0;
  if (m->tc) {
    const mpdo_mlp_s::TcOut& o = *reinterpret_cast<const mpdo_mlp_s::TcOut*>(m->hpart);
    if (o.err) return mlp_fail(m, MPDO_ERR_TIMEOUT, "mlp: a tensor-core pipeline wait gave up");
    s = o.loss;
  }
  for (int b = 0; b < blocks; ++b) s += m->hpart[b];
  if (loss) *loss = (float)(s / (double)n);
  return MPDO_OK;
}

int mpdo_mlp_adam_step(mpdo_mlp m, float lr) {
  if (!m || !(lr > 0)) return mlp_fail(m, MPDO_ERR_ARG, "mlp: bad learning rate");
  m->t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)m->t), c2 = 1.f - powf(b2, (float)m->t);
  mpdo::count_launch();
  adam_kernel<<<nb(m->n_params), 256, 0, m->st>>>(m->n_params, lr, b1, b2, 1e-8f, c1, c2, m->grads,
                                                  m->m, m->v, m->params);
  MK(cudaGetLastError());
  return MPDO_OK;
}

int mpdo_mlp_input_grad(mpdo_mlp m, int batch, const float* x, const float* wout_host, float* gx) {
  if (!m || !x || !wout_host || !gx || batch < 1 || batch > m->max_batch)
    return mlp_fail(m, MPDO_ERR_ARG, "mlp: bad input_grad arguments");
  const int L = (int)m->w.size() - 1;
  // d(output) = wout broadcast over rows; the output itself is not needed
  MK(cudaMemcpyAsync(m->db2, wout_host, sizeof(float) * m->w[L], cudaMemcpyHostToDevice, m->st));
  int rc;
  if (m->tc) {
    if ((rc = tc_operands(m, batch, x, true, false, m->db2))) return rc;
    if ((rc = tc_forward(m, batch, L - 1, false, {}))) return rc;
    if ((rc = tc_backward(m, batch, gx))) return rc;
  } else {
    if ((rc = run_forward(m, batch, L - 1, x, nullptr))) return rc;
    mpdo::count_launch();
    fill_rows_kernel<<<nb((long)batch * m->w[L]), 256, 0, m->st>>>(batch, m->w[L], m->db2, m->da);
    MK(cudaGetLastError());
    if ((rc = run_backward(m, batch, x, gx))) return rc;
  }
  MK(cudaStreamSynchronize(m->st));
  return MPDO_OK;
}

int mpdo_mlp_set_precision(mpdo_mlp m, int mode) {
  if (!m || (mode != 0 && mode != 1)) return mlp_fail(m, MPDO_ERR_ARG, "mlp: precision mode must be 0 or 1");
  MK(cudaStreamSynchronize(m->st));
  if (mode == 1 && !m->tcmem) {
    const int L = (int)m->w.size() - 1;
    const long ldb = r8(m->max_batch), groups = (m->max_batch + 127) / 128 * 4;
    // twice: the sizes, then the addresses
    uintptr_t base = 0;
    for (int pass = 0; pass < 2; ++pass) {
      size_t off = 0;
      auto take = [&](size_t bytes) {
        void* p = reinterpret_cast<void*>(base + off);
        off += (bytes + 255) / 256 * 256;
        return p;
      };
      m->xr.assign(L + 1, nullptr);
      m->xc = m->zr = m->zc = m->wr = m->wt = m->xr;
      m->csum.assign(L + 1, nullptr);
      auto bf = [&](long rows, long ld) { return static_cast<__nv_bfloat16*>(take(2 * rows * ld)); };
      for (int l = 0; l <= L; ++l) {
        const long w = m->w[l];
        if (l < L) {
          m->xr[l] = bf(m->max_batch, r8(w));
          m->xc[l] = bf(w, ldb);
          m->wr[l] = bf(w, r8(m->w[l + 1]));
          m->wt[l] = bf(m->w[l + 1], r8(w));
        }
        if (l > 0) {
          m->zr[l] = bf(m->max_batch, r8(w));
          m->zc[l] = bf(w, ldb);
          m->csum[l] = static_cast<float*>(take(sizeof(float) * groups * w));
        }
      }
      m->lpart = static_cast<double*>(take(sizeof(double) * groups * ((m->w[L] + 31) / 32)));
      m->tcout = static_cast<mpdo_mlp_s::TcOut*>(take(sizeof(mpdo_mlp_s::TcOut)));
      if (pass == 0) {
        if (mpdo::dev_malloc(&m->tcmem, off) != cudaSuccess) {
          cudaGetLastError();
          m->tcmem = nullptr;
          return mlp_fail(m, MPDO_ERR_OOM, "mlp: tensor-core operand buffers");
        }
        base = reinterpret_cast<uintptr_t>(m->tcmem);
      }
    }
    m->ldb = ldb;
    MK(cudaMemsetAsync(m->tcout, 0, sizeof(mpdo_mlp_s::TcOut), m->st));
  }
  m->tc = mode;
  return MPDO_OK;
}

int mpdo_mlp_destroy(mpdo_mlp m) {
  if (!m) return MPDO_OK;
  if (m->st) cudaStreamSynchronize(m->st);
  if (m->tcmem) cudaFree(m->tcmem);
  for (float* p : m->acts) if (p) cudaFree(p);
  if (m->params) cudaFree(m->params);
  if (m->grads) cudaFree(m->grads);
  if (m->m) cudaFree(m->m);
  if (m->v) cudaFree(m->v);
  if (m->da) cudaFree(m->da);
  if (m->db2) cudaFree(m->db2);
  if (m->part) cudaFree(m->part);
  if (m->hpart) cudaFreeHost(m->hpart);
  if (m->own_stream) cudaStreamDestroy(m->st);
  delete m;
  return MPDO_OK;
}

}  // extern "C"
