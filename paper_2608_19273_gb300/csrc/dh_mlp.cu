// Training and inference kernels of the FP32 MLP pressure seed (layout and
// inputs in dh_mlp.cuh).  Loss: mean squared error on y = ln(p/E).
//
// Gradients are deterministic: each CTA takes 64 samples, sums every one of the 1217 gradient
// entries over them in a fixed order into one row of a partial-gradient table, and a second
// kernel sums the rows in a fixed order.  No floating-point atomics anywhere.
//
// A batch of 4096 is 28 MFLOP, half a microsecond of the FP32 pipe: a training step is bound by the
// chain of latencies within a CTA and by its launches.  The gradient kernel therefore spreads a CTA's
// 64 samples over 256 threads (two samples x four neurons each in the layers, four weights each in
// the weight gradient, operands by 16-byte shared-memory loads) where one thread per sample walked
// through all 32 neurons, and a training step is two launches: the sum of the rows also does the
// Adam update and writes the loss.
// 20 steps of batch 4096: 577 us with one thread per sample and four operations a step, 251 now.
#include <cmath>

#include "dh_internal.cuh"
#include "dh_mlp.cuh"

namespace dh {

constexpr int GB = 64;  // samples per gradient CTA

// Raw invariants x (n x 3, row-major) and, if p is given, targets y = ln(p/E)
// from conserved states in SoA layout with the given stride.
__global__ void k_mlp_features(const double* __restrict__ cons, const double* __restrict__ p, int64_t n,
                               int64_t stride, float* __restrict__ x, float* __restrict__ y) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double q[5], xd[3];
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = cons[v * stride + i];
    srhd_invariants(q, xd);
#pragma unroll
    for (int j = 0; j < 3; ++j) x[3 * i + j] = (float)xd[j];
    if (y) y[i] = (float)log(p[i] / (q[4] + q[0]));
  }
}

// Mean and standard deviation of the three inputs, in two deterministic passes:
// per-CTA FP64 partial sums (fixed order), then one CTA sums the partial rows.
__global__ void k_mlp_stats_partial(const float* __restrict__ x, int64_t n, double* __restrict__ part) {
  __shared__ double s[256][6];
  double a[6] = {0, 0, 0, 0, 0, 0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double v = x[3 * i + j];
      a[j] += v;
      a[3 + j] = fma(v, v, a[3 + j]);
    }
  }
#pragma unroll
  for (int j = 0; j < 6; ++j) s[threadIdx.x][j] = a[j];
  __syncthreads();
  if (threadIdx.x < 6) {
    double t = 0.0;
    for (int i = 0; i < (int)blockDim.x; ++i) t += s[i][threadIdx.x];
    part[blockIdx.x * 6 + threadIdx.x] = t;
  }
}

__global__ void k_mlp_stats_final(const double* __restrict__ part, int nb, int64_t n, float* __restrict__ w) {
  if (threadIdx.x < 3) {
    const int j = threadIdx.x;
    double s1 = 0.0, s2 = 0.0;
    for (int b = 0; b < nb; ++b) { s1 += part[b * 6 + j]; s2 += part[b * 6 + 3 + j]; }
    const double mean = s1 / (double)n;
    double var = s2 / (double)n - mean * mean;
    if (!(var > 1e-30)) var = 1.0;
    w[MLP_MEAN + j] = (float)mean;
    w[MLP_STD + j] = (float)sqrt(var);
  }
}

// Forward pass on raw inputs (z-scored with the statistics in w).
__global__ void k_mlp_forward(const float* __restrict__ wg, const float* __restrict__ x, int64_t n,
                              float* __restrict__ y) {
  __shared__ __align__(16) float w[MLP_LEN];
  for (int i = threadIdx.x; i < MLP_LEN; i += blockDim.x) w[i] = wg[i];
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double xd[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
    float xn[3], h1[32], h2[32];
    mlp_normalize(w, xd, xn);
    y[i] = mlp_forward(w, xn, h1, h2);
  }
}

constexpr int GT = 256;   // threads of a gradient CTA
constexpr int GP = 36;    // pitch of the per-sample rows (16-byte aligned, four banks further per sample)
constexpr size_t GRAD_SMEM = sizeof(float) * (MLP_LEN + 32 * GP + 4 * GB * GP + 6 * GB);
static_assert(GRAD_SMEM <= 48 * 1024, "within the default shared memory of a CTA");

// Per-CTA partial gradient of (1/B) sum (y_i - t_i)^2 over samples [off, off + B).
// part row layout: 1217 gradient entries, then the partial sum of squared residuals.
__global__ void __launch_bounds__(GT) k_mlp_grad(const float* __restrict__ wg, const float* __restrict__ x,
                                                 const float* __restrict__ t, int64_t off, int B,
                                                 float* __restrict__ part) {
  extern __shared__ __align__(16) float gsm[];
  float* w = gsm;                 // the weights
  float* w2t = w + MLP_LEN;       // W2 transposed: [j][i], pitch GP
  float* sh1 = w2t + 32 * GP;     // per sample: hidden activations and back-propagated errors
  float* sh2 = sh1 + GB * GP;
  float* sg1 = sh2 + GB * GP;
  float* sg2 = sg1 + GB * GP;
  float* sx = sg2 + GB * GP;      // [j][sample]: z-scored inputs
  float* sgy = sx + 3 * GB;
  float* sr2 = sgy + GB;
  const int tid = threadIdx.x;
  for (int i = tid; i < MLP_LEN; i += GT) {
    const float v = wg[i];
    w[i] = v;
    if (i >= MLP_W2 && i < MLP_B2) w2t[((i - MLP_W2) & 31) * GP + ((i - MLP_W2) >> 5)] = v;
  }
  const int64_t s0 = (int64_t)blockIdx.x * GB;
  if (tid < 3 * GB) {  // one input of one sample per thread, z-scored as in mlp_normalize
    const int j = tid / GB, k = tid % GB;
    const bool valid = s0 + k < B;
    const double xd = valid ? x[3 * (off + s0 + k) + j] : 0.0;
    sx[j * GB + k] = valid ? (float)((xd - (double)wg[MLP_MEAN + j]) / (double)wg[MLP_STD + j]) : 0.0f;
  } else {
    const int k = tid - 3 * GB;
    sr2[k] = s0 + k < B ? t[off + s0 + k] : 0.0f;  // the target, replaced by the squared residual below
  }
  __syncthreads();
  // two samples x four neurons per thread; the eight threads of a sample are neighbouring lanes
  const int n4 = 4 * (tid & 7), ka = 2 * (tid >> 3);
  float h1[2][4], h2[2][4], g2[2][4];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float s = w[MLP_B1 + n4 + i];
#pragma unroll
      for (int j = 0; j < 3; ++j) s = fmaf(w[MLP_W1 + 3 * (n4 + i) + j], sx[j * GB + ka + q], s);
      h1[q][i] = tanhf(s);
    }
#pragma unroll
  for (int q = 0; q < 2; ++q)
    *reinterpret_cast<float4*>(sh1 + (ka + q) * GP + n4) = make_float4(h1[q][0], h1[q][1], h1[q][2], h1[q][3]);
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int i = 0; i < 4; ++i) h2[q][i] = w[MLP_B2 + n4 + i];
#pragma unroll 8
  for (int j = 0; j < 32; ++j) {
    const float4 r = *reinterpret_cast<const float4*>(w2t + j * GP + n4);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float h = sh1[(ka + q) * GP + j];
      h2[q][0] = fmaf(r.x, h, h2[q][0]);
      h2[q][1] = fmaf(r.y, h, h2[q][1]);
      h2[q][2] = fmaf(r.z, h, h2[q][2]);
      h2[q][3] = fmaf(r.w, h, h2[q][3]);
    }
  }
  const float w3[4] = {w[MLP_W3 + n4], w[MLP_W3 + n4 + 1], w[MLP_W3 + n4 + 2], w[MLP_W3 + n4 + 3]};
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    float y = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      h2[q][i] = tanhf(h2[q][i]);
      y = fmaf(w3[i], h2[q][i], y);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) y += __shfl_xor_sync(0xffffffffu, y, o);  // the same value in all eight lanes
    const int k = ka + q;
    const bool valid = s0 + k < B;
    const float r = valid ? y + w[MLP_B3] - sr2[k] : 0.0f;
    const float gy = 2.0f * r / (float)B;
    __syncwarp();  // every lane has read the target
    if ((tid & 7) == 0) {
      sr2[k] = r * r;
      sgy[k] = gy;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) g2[q][i] = gy * w3[i] * (1.0f - h2[q][i] * h2[q][i]);
    *reinterpret_cast<float4*>(sh2 + k * GP + n4) = make_float4(h2[q][0], h2[q][1], h2[q][2], h2[q][3]);
    *reinterpret_cast<float4*>(sg2 + k * GP + n4) = make_float4(g2[q][0], g2[q][1], g2[q][2], g2[q][3]);
  }
  __syncwarp();
  // back-propagation to the first layer
  float g1[2][4] = {};
#pragma unroll 8
  for (int a = 0; a < 32; ++a) {
    const float4 r = *reinterpret_cast<const float4*>(w + MLP_W2 + 32 * a + n4);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float g = sg2[(ka + q) * GP + a];
      g1[q][0] = fmaf(r.x, g, g1[q][0]);
      g1[q][1] = fmaf(r.y, g, g1[q][1]);
      g1[q][2] = fmaf(r.z, g, g1[q][2]);
      g1[q][3] = fmaf(r.w, g, g1[q][3]);
    }
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
#pragma unroll
    for (int i = 0; i < 4; ++i) g1[q][i] *= 1.0f - h1[q][i] * h1[q][i];
    *reinterpret_cast<float4*>(sg1 + (ka + q) * GP + n4) = make_float4(g1[q][0], g1[q][1], g1[q][2], g1[q][3]);
  }
  __syncthreads();
  // gradient entries, each summed over the CTA's samples in order
  float* row = part + (int64_t)blockIdx.x * MLP_LEN;
  {
    const int a = tid >> 3;  // W2[a][n4 .. n4+3] += g2[a] h1[n4 .. n4+3]
    float s[4] = {};
#pragma unroll 8
    for (int m = 0; m < GB; ++m) {
      const float g = sg2[m * GP + a];
      const float4 h = *reinterpret_cast<const float4*>(sh1 + m * GP + n4);
      s[0] = fmaf(g, h.x, s[0]);
      s[1] = fmaf(g, h.y, s[1]);
      s[2] = fmaf(g, h.z, s[2]);
      s[3] = fmaf(g, h.w, s[3]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) row[MLP_W2 + 32 * a + n4 + i] = s[i];  // (the caller's table need not be 16-byte aligned)
  }
  if (tid < 194) {  // the other entries, one per thread (each kind in warps of its own)
    const int l = tid & 31, kind = tid >> 5;
    int e;
    float s = 0.0f;
    if (kind < 3) {         // W1[a][j] += g1[a] x[j]
      const int a = tid / 3, j = tid % 3;
      e = MLP_W1 + tid;
#pragma unroll 8
      for (int m = 0; m < GB; ++m) s = fmaf(sg1[m * GP + a], sx[j * GB + m], s);
    } else if (kind == 3) {  // b1[a] += g1[a]
      e = MLP_B1 + l;
#pragma unroll 8
      for (int m = 0; m < GB; ++m) s += sg1[m * GP + l];
    } else if (kind == 4) {  // b2[a] += g2[a]
      e = MLP_B2 + l;
#pragma unroll 8
      for (int m = 0; m < GB; ++m) s += sg2[m * GP + l];
    } else if (kind == 5) {  // W3[a] += gy h2[a]
      e = MLP_W3 + l;
#pragma unroll 8
      for (int m = 0; m < GB; ++m) s = fmaf(sgy[m], sh2[m * GP + l], s);
    } else {                 // b3 += gy; squared residuals
      e = l == 0 ? MLP_B3 : MLP_NW;
      const float* src = l == 0 ? sgy : sr2;
#pragma unroll 8
      for (int m = 0; m < GB; ++m) s += src[m];
    }
    row[e] = s;
  }
}

// Adam (Kingma & Ba 2015): m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2;
// w -= lr (m / c1) / (sqrt(v / c2) + eps), c1 = 1 - b1^t, c2 = 1 - b2^t.
struct AdamArgs {
  float *w, *m, *v;
  float lr, b1, b2, eps, c1, c2;
};
__device__ __forceinline__ void adam_entry(const AdamArgs& A, int e, float ge) {
  const float me = fmaf(A.b1, A.m[e], (1.0f - A.b1) * ge);
  const float ve = fmaf(A.b2, A.v[e], (1.0f - A.b2) * ge * ge);
  A.m[e] = me;
  A.v[e] = ve;
  A.w[e] -= A.lr * (me / A.c1) / (sqrtf(ve / A.c2) + A.eps);
}

// grad[e] = sum_b part[b][e], grad[1217] = loss.  A CTA takes 32 entries: warp r sums the rows r, r + 8, ..
// in order, then the eight sums are added in order.  With A.w the entries' Adam update follows, and
// the loss also goes to loss_out (if not NULL).
constexpr int RED_T = 256;
__global__ void __launch_bounds__(RED_T) k_mlp_reduce(const float* __restrict__ part, int nb, int B,
                                                      float* __restrict__ grad, const AdamArgs A, float* loss_out) {
  __shared__ float sums[8][33];
  const int lane = threadIdx.x & 31, r = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (e <= MLP_NW) {
#pragma unroll 8
    for (int b = r; b < nb; b += 8) s += part[(int64_t)b * MLP_LEN + e];
  }
  sums[r][lane] = s;
  __syncthreads();
  if (r != 0 || e > MLP_NW) return;
  s = sums[0][lane];
#pragma unroll
  for (int k = 1; k < 8; ++k) s += sums[k][lane];
  if (e == MLP_NW) {
    s /= (float)B;
    if (loss_out) *loss_out = s;
  }
  grad[e] = s;
  if (A.w && e < MLP_NW) adam_entry(A, e, s);
}

__global__ void k_mlp_adam(const float* __restrict__ g, const AdamArgs A) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < MLP_NW) adam_entry(A, e, g[e]);
}

static AdamArgs adam_args(float* w, float* m, float* v, int32_t t, float lr, float b1, float b2, float eps) {
  const float c1 = (float)(1.0 - std::pow((double)b1, t)), c2 = (float)(1.0 - std::pow((double)b2, t));
  return AdamArgs{w, m, v, lr, b1, b2, eps, c1, c2};
}

// One gradient over samples [offset, offset + B): partial rows, then their sum (and, with A.w, the Adam
// update and the loss).
static dh_status grad_launch(const float* w, const float* x, const float* t, int64_t offset, int32_t B, float* partials,
                             float* grad, const AdamArgs& A, float* loss_out, cudaStream_t s) {
  const int nb = (B + GB - 1) / GB;
  k_mlp_grad<<<nb, GT, GRAD_SMEM, s>>>(w, x, t, offset, B, partials);
  k_mlp_reduce<<<(MLP_NW + 1 + 31) / 32, RED_T, 0, s>>>(partials, nb, B, grad, A, loss_out);
  return cuda_error(cudaGetLastError(), "dh_mlp_grad launch");
}

static int grid_for(int64_t n) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (n + 255) / 256;
  return (int)std::min<int64_t>(std::max<int64_t>(want, 1), (int64_t)sms * 8);
}

}  // namespace dh

using namespace dh;

extern "C" {

dh_status dh_mlp_features(const double* cons, const double* p, int64_t n, int64_t stride, float* x, float* y,
                          void* stream) {
  if (!cons || !x || n <= 0 || stride < n || (y && !p)) { set_error("dh_mlp_features: bad arguments"); return DH_EINVAL; }
  k_mlp_features<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(cons, p, n, stride, x, y);
  return cuda_error(cudaGetLastError(), "dh_mlp_features launch");
}

dh_status dh_mlp_standardize(const float* x, int64_t n, float* w, double* scratch, int32_t scratch_len,
                             void* stream) {
  if (!x || !w || !scratch || n <= 1) { set_error("dh_mlp_standardize: bad arguments"); return DH_EINVAL; }
  const int nb = std::min(grid_for(n), scratch_len / 6);
  if (nb < 1) { set_error("dh_mlp_standardize: scratch must hold at least 6 doubles"); return DH_EINVAL; }
  cudaStream_t s = (cudaStream_t)stream;
  k_mlp_stats_partial<<<nb, 256, 0, s>>>(x, n, scratch);
  k_mlp_stats_final<<<1, 32, 0, s>>>(scratch, nb, n, w);
  return cuda_error(cudaGetLastError(), "dh_mlp_standardize launch");
}

dh_status dh_mlp_forward(const float* w, const float* x, int64_t n, float* y, void* stream) {
  if (!w || !x || !y || n <= 0) { set_error("dh_mlp_forward: bad arguments"); return DH_EINVAL; }
  k_mlp_forward<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(w, x, n, y);
  return cuda_error(cudaGetLastError(), "dh_mlp_forward launch");
}

dh_status dh_mlp_grad(const float* w, const float* x, const float* t, int64_t offset, int32_t B, float* partials,
                      float* grad, void* stream) {
  if (!w || !x || !t || !partials || !grad || B <= 0 || offset < 0) { set_error("dh_mlp_grad: bad arguments"); return DH_EINVAL; }
  return grad_launch(w, x, t, offset, B, partials, grad, AdamArgs{}, nullptr, (cudaStream_t)stream);
}

dh_status dh_mlp_adam(float* w, float* m, float* v, const float* g, int32_t t, float lr, float b1, float b2,
                      float eps, void* stream) {
  if (!w || !m || !v || !g || t < 1) { set_error("dh_mlp_adam: bad arguments"); return DH_EINVAL; }
  k_mlp_adam<<<(MLP_NW + 255) / 256, 256, 0, (cudaStream_t)stream>>>(g, adam_args(w, m, v, t, lr, b1, b2, eps));
  return cuda_error(cudaGetLastError(), "dh_mlp_adam launch");
}

dh_status dh_mlp_train(float* w, float* m, float* v, const float* x, const float* t, int64_t n, int32_t batch,
                       int32_t steps, int32_t t0, float lr, float* partials, float* grad, float* loss_log,
                       void* stream) {
  if (!w || !m || !v || !x || !t || !partials || !grad || n <= 0 || batch <= 0 || batch > n || steps < 0 || t0 < 0) {
    set_error("dh_mlp_train: bad arguments");
    return DH_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t nbatch = n / batch;
  for (int k = 0; k < steps; ++k) {
    const int64_t off = (int64_t)(k % nbatch) * batch;
    const dh_status st = grad_launch(w, x, t, off, batch, partials, grad,
                                     adam_args(w, m, v, t0 + k + 1, lr, 0.9f, 0.999f, 1e-8f),
                                     loss_log ? loss_log + k : nullptr, s);
    if (st != DH_OK) return st;
  }
  return DH_OK;
}

}  // extern "C"
