// Learned beta-ladder predictor: an fp32 MLP 259 -> 256 -> 256 -> 256 -> 32
// with a monotone head, trained with Adam on the squared ladder error plus an
// optional relative-gap term.  The paper has no learned
// component; the predictor replaces the adaptive-ladder preprocessing of
// Algorithm S2 by a network reading cheap instance features and short pilot
// histograms, on the grounds that ladders of one size are nearly identical
// across instances (Fig. S12).  These are tiny dense layers, so they run as
// plain SIMT kernels: a 32x32-tiled product with bias / ReLU / ReLU-mask
// epilogues and row sums for bias gradients, a warp-per-sample head (scan and
// reverse scan over the 32 outputs), and an elementwise Adam step.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "ctx.h"
#include "internal.h"

namespace {

constexpr int kIn = 259, kHid = 256, kOut = 32, kLayers = 4;
constexpr int kDims[kLayers + 1] = {kIn, kHid, kHid, kHid, kOut};

// The kernels of a pass are short and each needs all of the one before it, so
// the gaps between them count.  They are launched so that a kernel's blocks may
// be set up once every block of the one before has called let_next
// (launch_next); wait_previous then waits until that kernel has finished and
// its writes are visible, so that order and results are those of plain
// launches.  The products call let_next after their main loop: called at the
// start, the waiting blocks crowded onto few SMs (1024 samples, 12 steps: 2.53
// ms plain, 3.98 early, 2.53 late; 256 samples, 10 steps: 1.15, 1.15, 0.95 ms;
// 64 samples, 5 steps: 0.59, 0.46, 0.46 ms; called again on the same
// minibatches, host work and the weights' readback included).
__device__ __forceinline__ void let_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One product C[m][n] = epi( sum_k A(m,k) B(k,n) ) with A(m,k) = A[m*sam +
// k*sak], B(k,n) = B[k*sbk + n*sbn].  Epilogue: + bias[n]; ReLU; times
// (mask[m*ldc + n] > 0).  `rowsum`, if given, receives sum_k A(m,k) (the
// bias gradient) as one more column, B(k, N) = 1.
struct Product {
  int M, N, K;
  const float *A, *B;
  int sam, sak, sbk, sbn;
  float *C;
  int ldc, relu;
  const float *bias, *mask;
  float *rowsum;
  int tn, tiles;    // tiles along n, and in all (0: no product)
};

// A layer's independent products (dW and dZ of the layer below) and, in one
// more block, the loss sum go out in one launch.
struct Products {
  Product p[2];
  int loss_n;              // samples of the loss sum (0: none)
  const float *loss_s;
  float *loss;
};

// A 32 x 32 tile per block of 128 threads, 2 x 4 outputs per thread, K in
// steps of 32 whose global loads are issued one step ahead.  What bounds
// these layers (256 x 256 x 259 and below) is not arithmetic but how many
// SMs take part and the latency of each K step: a 64 x 64 tile put 256 x 256
// on 16 SMs and waited for every load (48 us per product).  With 64 blocks,
// the loads ahead and 10 instead of 19 launches a training step of 256
// samples went from 0.40 to 0.11 ms (0.09 with the launches of launch_next).
// Every output is one fmaf chain over k in order.
constexpr int kTile = 32, kGemmThreads = 128;

__device__ __forceinline__ void loss_sum(int B, const float *loss_s, float *loss, float *part) {
  // 256 partial sums in fixed order, two per thread
  for (int t = threadIdx.x; t < 256; t += kGemmThreads) {
    float s = 0.f;
    for (int i = t; i < B; i += 256) s += loss_s[i];
    part[t] = s;
  }
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = part[0] / (float)(B * kOut);
}

__global__ void __launch_bounds__(kGemmThreads) gemm_kernel(const __grid_constant__ Products P) {
  __shared__ __align__(16) float As[kTile][kTile + 2];   // rows 8-byte aligned (float2 reads)
  __shared__ __align__(16) float Bs[kTile][kTile + 4];   // rows 16-byte aligned (float4 reads)
  wait_previous();
  int tile = (int)blockIdx.x;
  if (P.loss_n) {
    if (tile == 0) {
      loss_sum(P.loss_n, P.loss_s, P.loss, &As[0][0]);
      return;
    }
    --tile;
  }
  const bool second = tile >= P.p[0].tiles;
  const Product &g = P.p[second ? 1 : 0];
  if (second) tile -= P.p[0].tiles;
  const int M = g.M, N = g.N, K = g.K;
  const int m0 = (tile / g.tn) * kTile, n0 = (tile % g.tn) * kTile;
  const int tid = threadIdx.x, r = tid & 31, w = tid >> 5;
  // element e = w + 4 q of a tile: lanes run along the contiguous index
  const bool ak = g.sak == 1, bk = g.sbk == 1;
  float ra[8], rb[8];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = w + 4 * q;
      const int ma = m0 + (ak ? e : r), ka = k0 + (ak ? r : e);
      ra[q] = (ma < M && ka < K) ? g.A[(size_t)ma * g.sam + (size_t)ka * g.sak] : 0.f;
      const int nb = n0 + (bk ? e : r), kb = k0 + (bk ? r : e);
      rb[q] = (nb < N && kb < K) ? g.B[(size_t)kb * g.sbk + (size_t)nb * g.sbn] : (nb == N && kb < K ? 1.f : 0.f);
    }
  };
  const int tx = tid & 7, ty = tid >> 3;   // outputs m0 + 2 ty + i, n0 + 4 tx + j
  float acc[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  load(0);
  for (int k0 = 0; k0 < K; k0 += kTile) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = w + 4 * q;
      if (ak) As[r][e] = ra[q]; else As[e][r] = ra[q];
      if (bk) Bs[r][e] = rb[q]; else Bs[e][r] = rb[q];
    }
    __syncthreads();
    if (k0 + kTile < K) load(k0 + kTile);
#pragma unroll
    for (int kk = 0; kk < kTile; ++kk) {
      const float2 a = *reinterpret_cast<const float2 *>(&As[kk][2 * ty]);
      const float4 b = *reinterpret_cast<const float4 *>(&Bs[kk][4 * tx]);
      const float av[2] = {a.x, a.y}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
  }
  let_next();
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int m = m0 + 2 * ty + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      float v = acc[i][j];
      if (n < N) {
        if (g.bias) v += g.bias[n];
        if (g.relu) v = fmaxf(v, 0.f);
        if (g.mask) v = (g.mask[(size_t)m * g.ldc + n] > 0.f) ? v : 0.f;
        g.C[(size_t)m * g.ldc + n] = v;
      } else if (n == N && g.rowsum) {
        g.rowsum[m] = v;
      }
    }
  }
}

__device__ __forceinline__ float softplus_f(float x) {
  return fmaxf(x, 0.f) + log1pf(expf(-fabsf(x)));
}

// One warp per sample: beta_k = beta_min + sum_{m<=k} softplus(o_m);
// loss_s = sum_k (beta_k - y_k)^2 + gw (32/31) sum_{k>=1} r_k^2 with the
// relative gap error r_k = (softplus(o_k) - d_k) / d_k, d_k = y_k - y_{k-1},
// so that sum_s loss_s / (B * 32) is the mean squared ladder error plus gw
// times the mean squared relative gap error; dO_m = sigmoid(o_m) (sum_{k>=m}
// dL/dbeta_k + [m >= 1] 2 gw r_m / (d_m B * 31)) with dL/dbeta_k =
// 2 (beta_k - y_k) / (B * 32).
__global__ void head_kernel(int B, const float *O, const float *Y, float beta_min, float gw, float *beta_out,
                            float *dO, float *loss_s) {
  let_next();
  wait_previous();
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= B) return;
  const float o = O[(size_t)warp * kOut + lane];
  const float sp = softplus_f(o);
  float c = sp;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const float v = __shfl_up_sync(0xFFFFFFFFu, c, d);
    if (lane >= d) c += v;
  }
  const float beta = beta_min + c;
  if (beta_out) beta_out[(size_t)warp * kOut + lane] = beta;
  if (!Y) return;
  const float y = Y[(size_t)warp * kOut + lane];
  const float yprev = __shfl_up_sync(0xFFFFFFFFu, y, 1);
  const float diff = beta - y;
  float l = diff * diff;
  float r = 0.f, dgap = 1.f;
  if (gw != 0.f && lane >= 1) {
    dgap = y - yprev;
    r = (sp - dgap) / dgap;
    l += gw * (32.f / 31.f) * r * r;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, d);
  if (lane == 0) loss_s[warp] = l;
  float g = 2.f * diff / (float)(B * kOut);
  // suffix sum over k >= m
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const float v = __shfl_down_sync(0xFFFFFFFFu, g, d);
    if (lane + d < 32) g += v;
  }
  const float sig = 1.f / (1.f + expf(-o));
  float dov = sig * g;
  if (gw != 0.f && lane >= 1) dov += sig * (2.f * gw * r / dgap / (float)(B * (kOut - 1)));
  dO[(size_t)warp * kOut + lane] = dov;
}

// Adam (Kingma & Ba): m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2;
// p -= lr * (m / c1) / (sqrt(v / c2) + eps) with c1 = 1 - b1^t, c2 = 1 - b2^t.
// The pass's last kernel also hands out the loss (loss_out may be NULL): all
// reads of the minibatch are done by then, so the caller may have the loss in
// the minibatch's own memory.
__global__ void adam_kernel(int n, float *p, const float *g, float *m, float *v, float lr, float b1,
                            float b2, float c1, float c2, float eps, const float *loss, float *loss_out) {
  let_next();
  wait_previous();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0 && loss_out) *loss_out = *loss;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace

namespace pc {

size_t mlp_param_count() {
  size_t n = 0;
  for (int l = 0; l < kLayers; ++l) n += (size_t)kDims[l + 1] * kDims[l] + kDims[l + 1];
  return n;
}

}  // namespace pc

struct pc_mlp {
  pc_ctx *ctx = nullptr;
  int device = 0;    // the context's device, kept for pc_mlp_destroy
  float beta_min = 0.f;
  float gap_weight = 0.f;   // weight of the relative-gap term of the loss
  int64_t t = 0;
  size_t n_params = 0;
  size_t w_off[kLayers], b_off[kLayers];
  pc::DevBuf<float> params, grads, m, v;
  int cap = 0;   // batch capacity of the activation buffers
  pc::DevBuf<float> X, H[3], O, dO, dH[3], Y, beta, loss_s, loss;
  pc::PinnedBuf<float> host_loss;
};

using namespace pc;

namespace {

template <typename... P, typename... A>
int launch_next(void (*kern)(P...), int blocks, int threads, cudaStream_t st, A... args) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  PC_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;   // a captured pass keeps plain edges
  PC_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...));
  PC_CUDA_TRY(cudaGetLastError());
  return PC_OK;
}

Product product(int M, int N, int K, const float *A, int sam, int sak, const float *B, int sbk, int sbn, float *C,
                int ldc, const float *bias, int relu, const float *mask, float *rowsum) {
  const int tn = (N + (rowsum ? 1 : 0) + kTile - 1) / kTile;
  return {M, N, K, A, B, sam, sak, sbk, sbn, C, ldc, relu, bias, mask, rowsum, tn, tn * ((M + kTile - 1) / kTile)};
}

int gemm(cudaStream_t st, const Products &P) {
  const int blocks = P.p[0].tiles + P.p[1].tiles + (P.loss_n ? 1 : 0);
  return launch_next(gemm_kernel, blocks, kGemmThreads, st, P);
}

int ensure_batch(pc_mlp *mm, int batch) {
  if (batch <= mm->cap) return PC_OK;
  int rc;
  const size_t b = (size_t)batch;
  if ((rc = mm->X.alloc(b * kIn)) || (rc = mm->O.alloc(b * kOut)) || (rc = mm->dO.alloc(b * kOut)) ||
      (rc = mm->Y.alloc(b * kOut)) || (rc = mm->beta.alloc(b * kOut)) || (rc = mm->loss_s.alloc(b)) ||
      (rc = mm->loss.alloc(1)))
    return rc;
  for (int l = 0; l < 3; ++l)
    if ((rc = mm->H[l].alloc(b * kHid)) || (rc = mm->dH[l].alloc(b * kHid))) return rc;
  if ((rc = mm->host_loss.reserve(1))) return rc;
  mm->cap = batch;
  return PC_OK;
}

// Forward pass from X (device, [batch][259]) to O; beta if requested.
int forward(pc_mlp *mm, int batch, const float *X, float *beta_dev) {
  cudaStream_t st = mm->ctx->stream;
  const float *p = mm->params.p;
  const float *in = X;
  int rc;
  for (int l = 0; l < kLayers; ++l) {
    Products P = {};
    float *out = l < 3 ? mm->H[l].p : mm->O.p;
    P.p[0] = product(batch, kDims[l + 1], kDims[l], in, kDims[l], 1, p + mm->w_off[l], 1, kDims[l], out, kDims[l + 1],
                     p + mm->b_off[l], l < 3, nullptr, nullptr);
    if ((rc = gemm(st, P))) return rc;
    in = out;
  }
  if (beta_dev)
    return launch_next(head_kernel, (batch * 32 + 255) / 256, 256, st, batch, mm->O.p, nullptr, mm->beta_min, 0.f,
                       beta_dev, nullptr, nullptr);
  return PC_OK;
}

// Loss and gradients into mm->loss and mm->grads for X, Y on the device.
int backward(pc_mlp *mm, int batch, const float *X, const float *Y) {
  cudaStream_t st = mm->ctx->stream;
  int rc = forward(mm, batch, X, nullptr);
  if (rc) return rc;
  if ((rc = launch_next(head_kernel, (batch * 32 + 255) / 256, 256, st, batch, mm->O.p, Y, mm->beta_min,
                        mm->gap_weight, mm->beta.p, mm->dO.p, mm->loss_s.p)))
    return rc;
  const float *p = mm->params.p;
  float *g = mm->grads.p;
  const float *dZ = mm->dO.p;
  for (int l = kLayers - 1; l >= 0; --l) {
    const int out = kDims[l + 1], in = kDims[l];
    const float *Hin = (l == 0) ? X : mm->H[l - 1].p;
    Products P = {};
    // dW[out][in] = sum_b dZ[b][out] Hin[b][in], db[out] = sum_b dZ[b][out]
    P.p[0] = product(out, in, batch, dZ, 1, out, Hin, in, 1, g + mm->w_off[l], in, nullptr, 0, nullptr,
                     g + mm->b_off[l]);
    // dZ_{l-1}[b][in] = (sum_o dZ[b][o] W[o][in]) * (H_{l-1} > 0)
    if (l > 0)
      P.p[1] = product(batch, in, out, dZ, out, 1, p + mm->w_off[l], in, 1, mm->dH[l - 1].p, in, nullptr, 0,
                       mm->H[l - 1].p, nullptr);
    if (l == kLayers - 1) {
      P.loss_n = batch;
      P.loss_s = mm->loss_s.p;
      P.loss = mm->loss.p;
    }
    if ((rc = gemm(st, P))) return rc;
    if (l > 0) dZ = mm->dH[l - 1].p;
  }
  return PC_OK;
}

// loss_out: where the kernel stores the loss as well, or NULL.
int adam(pc_mlp *mm, float lr, float *loss_out = nullptr) {
  mm->t += 1;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = (float)(1.0 - std::pow(0.9, (double)mm->t));
  const float c2 = (float)(1.0 - std::pow(0.999, (double)mm->t));
  const int n = (int)mm->n_params;
  return launch_next(adam_kernel, (n + 255) / 256, 256, mm->ctx->stream, n, mm->params.p, mm->grads.p, mm->m.p,
                     mm->v.p, lr, b1, b2, c1, c2, eps, mm->loss.p, loss_out);
}

// Whether a kernel on `device` may store a float at p: aligned memory of that
// device.  Anything else a copy can reach (another device, a byte offset).
bool stores_directly(const float *p, int device) {
  cudaPointerAttributes at = {};
  if (reinterpret_cast<uintptr_t>(p) % sizeof(float)) return false;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice && at.device == device;
}

}  // namespace

namespace pc {

pc_ctx *mlp_context(pc_mlp *mm) { return mm->ctx; }

int mlp_input(pc_mlp *mm, int batch, float **X_dev) {
  int rc = ensure_batch(mm, batch);
  if (rc) return rc;
  *X_dev = mm->X.p;
  return PC_OK;
}

int mlp_forward_input(pc_mlp *mm, int batch, const float **beta_dev) {
  int rc = ensure_batch(mm, batch);
  if (rc) return rc;
  if ((rc = forward(mm, batch, mm->X.p, mm->beta.p))) return rc;
  *beta_dev = mm->beta.p;
  return PC_OK;
}

}  // namespace pc

namespace {

// Weights file: magic, the five layer widths, beta_min, then W[l] ([out][in]
// row-major) and b[l] of every layer as little-endian fp32.
constexpr char kMlpMagic[8] = {'P', 'C', 'M', 'L', 'P', '0', '0', '1'};

}  // namespace

extern "C" {

int pc_mlp_create(pc_ctx *c, pc_mlp **out, const float *const *W, const float *const *b, float beta_min) try {
  if (!c || !out || !W || !b) return fail(PC_EINVAL, "NULL argument");
  *out = nullptr;
  PC_CUDA_TRY(cudaSetDevice(c->device));
  pc_mlp *mm = new pc_mlp();
  mm->ctx = c;
  mm->device = c->device;
  mm->beta_min = beta_min;
  size_t off = 0;
  for (int l = 0; l < kLayers; ++l) {
    mm->w_off[l] = off;
    off += (size_t)kDims[l + 1] * kDims[l];
    mm->b_off[l] = off;
    off += (size_t)kDims[l + 1];
  }
  mm->n_params = off;
  std::vector<float> h(off);
  for (int l = 0; l < kLayers; ++l) {
    if (!W[l] || !b[l]) {
      delete mm;
      return fail(PC_EINVAL, "NULL weight");
    }
    std::memcpy(h.data() + mm->w_off[l], W[l], sizeof(float) * kDims[l + 1] * kDims[l]);
    std::memcpy(h.data() + mm->b_off[l], b[l], sizeof(float) * kDims[l + 1]);
  }
  int rc;
  if ((rc = mm->params.alloc(off)) || (rc = mm->grads.alloc(off)) || (rc = mm->m.alloc(off)) ||
      (rc = mm->v.alloc(off)) || (rc = mm->m.zero(c->stream)) || (rc = mm->v.zero(c->stream))) {
    delete mm;
    return rc;
  }
  cudaError_t e = cudaMemcpyAsync(mm->params.p, h.data(), off * 4, cudaMemcpyHostToDevice, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) {
    delete mm;
    return fail(PC_ECUDA, cudaGetErrorString(e));
  }
  *out = mm;
  return PC_OK;
} catch (...) {
  return pc::fail_exception();
}

void pc_mlp_destroy(pc_mlp *mm) try {
  if (!mm) return;
  // the context may already be gone: use only the device recorded at
  // creation (cudaFree waits for the device's work on these buffers)
  cudaSetDevice(mm->device);
  delete mm;
} catch (...) {
}

int pc_mlp_forward(pc_mlp *mm, int batch, const float *X, float *beta) try {
  if (!mm || !X || !beta || batch < 1) return fail(PC_EINVAL, "bad arguments");
  PC_CUDA_TRY(cudaSetDevice(mm->ctx->device));
  cudaStream_t st = mm->ctx->stream;
  int rc = ensure_batch(mm, batch);
  if (rc) return rc;
  PC_CUDA_TRY(cudaMemcpyAsync(mm->X.p, X, (size_t)batch * kIn * 4, cudaMemcpyHostToDevice, st));
  if ((rc = forward(mm, batch, mm->X.p, mm->beta.p))) return rc;
  PC_CUDA_TRY(cudaMemcpyAsync(beta, mm->beta.p, (size_t)batch * kOut * 4, cudaMemcpyDeviceToHost, st));
  PC_CUDA_TRY(cudaStreamSynchronize(st));
  return PC_OK;
} catch (...) {
  return pc::fail_exception();
}

int pc_mlp_grads(pc_mlp *mm, int batch, const float *X, const float *Y, float *loss, float *const *gW,
                 float *const *gb) try {
  if (!mm || !X || !Y || batch < 1) return fail(PC_EINVAL, "bad arguments");
  PC_CUDA_TRY(cudaSetDevice(mm->ctx->device));
  cudaStream_t st = mm->ctx->stream;
  int rc = ensure_batch(mm, batch);
  if (rc) return rc;
  PC_CUDA_TRY(cudaMemcpyAsync(mm->X.p, X, (size_t)batch * kIn * 4, cudaMemcpyHostToDevice, st));
  PC_CUDA_TRY(cudaMemcpyAsync(mm->Y.p, Y, (size_t)batch * kOut * 4, cudaMemcpyHostToDevice, st));
  if ((rc = backward(mm, batch, mm->X.p, mm->Y.p))) return rc;
  std::vector<float> h(mm->n_params);
  PC_CUDA_TRY(cudaMemcpyAsync(h.data(), mm->grads.p, h.size() * 4, cudaMemcpyDeviceToHost, st));
  float l = 0.f;
  PC_CUDA_TRY(cudaMemcpyAsync(&l, mm->loss.p, 4, cudaMemcpyDeviceToHost, st));
  PC_CUDA_TRY(cudaStreamSynchronize(st));
  if (loss) *loss = l;
  for (int k = 0; k < kLayers; ++k) {
    if (gW && gW[k]) std::memcpy(gW[k], h.data() + mm->w_off[k], sizeof(float) * kDims[k + 1] * kDims[k]);
    if (gb && gb[k]) std::memcpy(gb[k], h.data() + mm->b_off[k], sizeof(float) * kDims[k + 1]);
  }
  return PC_OK;
} catch (...) {
  return pc::fail_exception();
}

int pc_mlp_train_step_dev(pc_mlp *mm, int batch, const float *X_dev, const float *Y_dev, float lr,
                          float *loss_dev) try {
  if (!mm || !X_dev || !Y_dev || batch < 1) return fail(PC_EINVAL, "bad arguments");
  PC_CUDA_TRY(cudaSetDevice(mm->ctx->device));
  int rc = ensure_batch(mm, batch);
  if (rc) return rc;
  if ((rc = backward(mm, batch, X_dev, Y_dev))) return rc;
  // a copy is a node of its own between two kernels: the update stores the
  // loss itself where it can
  const bool direct = loss_dev && stores_directly(loss_dev, mm->device);
  if (loss_dev && !direct)
    PC_CUDA_TRY(cudaMemcpyAsync(loss_dev, mm->loss.p, 4, cudaMemcpyDeviceToDevice, mm->ctx->stream));
  return adam(mm, lr, direct ? loss_dev : nullptr);
} catch (...) {
  return pc::fail_exception();
}

int pc_mlp_train_step(pc_mlp *mm, int batch, const float *X, const float *Y, float lr, float *loss) try {
  if (!mm || !X || !Y || batch < 1) return fail(PC_EINVAL, "bad arguments");
  PC_CUDA_TRY(cudaSetDevice(mm->ctx->device));
  cudaStream_t st = mm->ctx->stream;
  int rc = ensure_batch(mm, batch);
  if (rc) return rc;
  PC_CUDA_TRY(cudaMemcpyAsync(mm->X.p, X, (size_t)batch * kIn * 4, cudaMemcpyHostToDevice, st));
  PC_CUDA_TRY(cudaMemcpyAsync(mm->Y.p, Y, (size_t)batch * kOut * 4, cudaMemcpyHostToDevice, st));
  if ((rc = backward(mm, batch, mm->X.p, mm->Y.p))) return rc;
  if ((rc = adam(mm, lr))) return rc;
  if (loss) {
    PC_CUDA_TRY(cudaMemcpyAsync(mm->host_loss.p, mm->loss.p, 4, cudaMemcpyDeviceToHost, st));
    PC_CUDA_TRY(cudaStreamSynchronize(st));
    *loss = mm->host_loss.p[0];
  }
  return PC_OK;
} catch (...) {
  return pc::fail_exception();
}

int pc_mlp_get_params(pc_mlp *mm, float *const *W, float *const *b) try {
  if (!mm) return fail(PC_EINVAL, "NULL argument");
  PC_CUDA_TRY(cudaSetDevice(mm->ctx->device));
  std::vector<float> h(mm->n_params);
  PC_CUDA_TRY(cudaMemcpyAsync(h.data(), mm->params.p, h.size() * 4, cudaMemcpyDeviceToHost, mm->ctx->stream));
  PC_CUDA_TRY(cudaStreamSynchronize(mm->ctx->stream));
  for (int k = 0; k < kLayers; ++k) {
    if (W && W[k]) std::memcpy(W[k], h.data() + mm->w_off[k], sizeof(float) * kDims[k + 1] * kDims[k]);
    if (b && b[k]) std::memcpy(b[k], h.data() + mm->b_off[k], sizeof(float) * kDims[k + 1]);
  }
  return PC_OK;
} catch (...) {
  return pc::fail_exception();
}

int pc_mlp_set_gap_weight(pc_mlp *mm, float w) try {
  if (!mm || !std::isfinite(w) || w < 0.f) return fail(PC_EINVAL, "gap weight must be finite and >= 0");
  mm->gap_weight = w;
  return PC_OK;
} catch (...) {
  return pc::fail_exception();
}

int pc_mlp_save(pc_mlp *mm, const char *path) try {
  if (!mm || !path) return fail(PC_EINVAL, "NULL argument");
  PC_CUDA_TRY(cudaSetDevice(mm->ctx->device));
  std::vector<float> h(mm->n_params);
  PC_CUDA_TRY(cudaMemcpyAsync(h.data(), mm->params.p, h.size() * 4, cudaMemcpyDeviceToHost, mm->ctx->stream));
  PC_CUDA_TRY(cudaStreamSynchronize(mm->ctx->stream));
  FILE *f = fopen(path, "wb");
  if (!f) return fail(PC_EINVAL, std::string("cannot open ") + path);
  int32_t dims[kLayers + 1];
  for (int l = 0; l <= kLayers; ++l) dims[l] = kDims[l];
  bool ok = fwrite(kMlpMagic, 1, 8, f) == 8 && fwrite(dims, 4, kLayers + 1, f) == (size_t)kLayers + 1 &&
            fwrite(&mm->beta_min, 4, 1, f) == 1;
  for (int l = 0; ok && l < kLayers; ++l) {
    const size_t nw = (size_t)kDims[l + 1] * kDims[l], nb = (size_t)kDims[l + 1];
    ok = fwrite(h.data() + mm->w_off[l], 4, nw, f) == nw && fwrite(h.data() + mm->b_off[l], 4, nb, f) == nb;
  }
  if (fclose(f) != 0) ok = false;
  return ok ? PC_OK : fail(PC_EINVAL, std::string("write failed: ") + path);
} catch (...) {
  return pc::fail_exception();
}

int pc_mlp_load(pc_ctx *c, const char *path, pc_mlp **out) try {
  if (!c || !path || !out) return fail(PC_EINVAL, "NULL argument");
  *out = nullptr;
  FILE *f = fopen(path, "rb");
  if (!f) return fail(PC_EINVAL, std::string("cannot open ") + path);
  char magic[8];
  int32_t dims[kLayers + 1];
  float beta_min = 0.f;
  bool ok = fread(magic, 1, 8, f) == 8 && std::memcmp(magic, kMlpMagic, 8) == 0 &&
            fread(dims, 4, kLayers + 1, f) == (size_t)kLayers + 1 && fread(&beta_min, 4, 1, f) == 1;
  for (int l = 0; ok && l <= kLayers; ++l) ok = dims[l] == kDims[l];
  std::vector<std::vector<float>> W(kLayers), b(kLayers);
  for (int l = 0; ok && l < kLayers; ++l) {
    W[l].resize((size_t)kDims[l + 1] * kDims[l]);
    b[l].resize((size_t)kDims[l + 1]);
    ok = fread(W[l].data(), 4, W[l].size(), f) == W[l].size() && fread(b[l].data(), 4, b[l].size(), f) == b[l].size();
  }
  fclose(f);
  if (!ok) return fail(PC_EINVAL, std::string("not a ladder-MLP weights file of this network: ") + path);
  const float *Wp[kLayers], *bp[kLayers];
  for (int l = 0; l < kLayers; ++l) {
    Wp[l] = W[l].data();
    bp[l] = b[l].data();
  }
  return pc_mlp_create(c, out, Wp, bp, beta_min);
} catch (...) {
  return pc::fail_exception();
}

}  // extern "C"
