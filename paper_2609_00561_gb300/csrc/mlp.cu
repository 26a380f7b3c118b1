// MLP of the learned blocking: forward pass, loss gradient and Adam step as
// plain CUDA kernels (FP32; the network has ~6k parameters and batches of a
// few hundred matrices: bound by launches and latency, no tensor cores).  Weights
// that fit a CTA's shared memory: a CTA per sample through all layers (mlp_fused);
// wider networks, and the forward pass of large batches: a launch per layer, a
// thread per output element.  Layout of the flat parameter array:
//   W1 [nf][h], b1 [h], W2 [h][h], b2 [h], W3 [h][c+1], b3 [c+1]
// (c = ncls; the last output is the regression head).  Every sum runs in a
// fixed order, so results do not depend on the launch shape.
#include <algorithm>
#include <cmath>

#include "iccg_internal.h"

namespace iccg {
namespace {

constexpr int kMlpThreads = 128;

struct MlpOff {
  int64_t w1, b1, w2, b2, w3, b3, total;
};

MlpOff mlp_off(int nf, int h, int c) {
  MlpOff o;
  o.w1 = 0;
  o.b1 = o.w1 + int64_t(nf) * h;
  o.w2 = o.b1 + h;
  o.b2 = o.w2 + int64_t(h) * h;
  o.w3 = o.b2 + h;
  o.b3 = o.w3 + int64_t(h) * (c + 1);
  o.total = o.b3 + (c + 1);
  return o;
}

int blocks_for(int64_t n) { return int((n + kMlpThreads - 1) / kMlpThreads); }

// out[b][o] = act(sum_i in[b][i] W[i][o] + bias[o]), i ascending
__global__ void dense_fwd(const float *in, int nin, const float *W, const float *bias, int nout, int batch,
                          float *out, int relu) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= batch * nout) return;
  const int b = idx / nout, o = idx % nout;
  float s = bias[o];
  for (int i = 0; i < nin; ++i) s = fmaf(in[b * nin + i], W[i * nout + o], s);
  out[idx] = relu ? fmaxf(s, 0.0f) : s;
}

// per sample: softmax cross entropy of z[b][0:c] against y[b] plus
// wreg (z[b][c] - yreg[b])^2; dz = d(loss / batch) / dz; lb[b] = sample loss
__global__ void head_grad(const float *z, int c, const int32_t *y, const float *yreg, float wreg, int batch,
                          float *dz, float *lb) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= batch) return;
  const float *zb = z + b * (c + 1);
  float *db = dz + b * (c + 1);
  float mx = zb[0];
  for (int k = 1; k < c; ++k) mx = fmaxf(mx, zb[k]);
  float se = 0.0f;
  for (int k = 0; k < c; ++k) se += expf(zb[k] - mx);
  const float inv_b = 1.0f / float(batch);
  const int yb = y[b];
  for (int k = 0; k < c; ++k) {
    const float p = expf(zb[k] - mx) / se;
    db[k] = (p - (k == yb ? 1.0f : 0.0f)) * inv_b;
  }
  const float err = zb[c] - yreg[b];
  db[c] = 2.0f * wreg * err * inv_b;
  lb[b] = (logf(se) + mx - zb[yb]) + wreg * err * err;
}

// Every weight and bias gradient of the three layers in one launch, a thread
// per parameter in the flat order, and the mean loss:
//   gW[i][o] = sum_b in[b][i] d[b][o],  gb[o] = sum_b d[b][o]  (b ascending).
// Latency bound (a few thousand threads, one sum over the batch each): the
// loads of kMlpBatch samples are issued together ahead of their multiply-adds.
constexpr int kMlpBatch = 16;

struct MlpLayer {
  const float *in, *d;   // [batch][nin], [batch][nout]
  int nin, nout;
  int64_t off;           // first parameter
};
struct MlpLayers {
  MlpLayer l[3];
};

__global__ void mlp_wgrad(MlpLayers L, int batch, int64_t np, const float *lb, float *grad, float *loss) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx < np) {
    const MlpLayer m = idx >= L.l[2].off ? L.l[2] : (idx >= L.l[1].off ? L.l[1] : L.l[0]);
    const int64_t k = idx - m.off;
    const int i = int(k / m.nout), o = int(k % m.nout);   // i = nin: the bias
    float s = 0.0f;
    for (int b0 = 0; b0 < batch; b0 += kMlpBatch) {
      float x[kMlpBatch], d[kMlpBatch];
#pragma unroll
      for (int u = 0; u < kMlpBatch; ++u) {
        const size_t b = size_t(b0 + u);
        const bool ok = b0 + u < batch;
        x[u] = ok && i < m.nin ? __ldcg(m.in + b * m.nin + i) : 1.0f;
        d[u] = ok ? __ldcg(m.d + b * m.nout + o) : 0.0f;
      }
#pragma unroll
      for (int u = 0; u < kMlpBatch; ++u)
        if (b0 + u < batch) s = fmaf(x[u], d[u], s);
    }
    grad[idx] = s;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
    float s = 0.0f;
    for (int b0 = 0; b0 < batch; b0 += kMlpBatch) {
      float x[kMlpBatch];
#pragma unroll
      for (int u = 0; u < kMlpBatch; ++u) x[u] = b0 + u < batch ? __ldcg(lb + b0 + u) : 0.0f;
#pragma unroll
      for (int u = 0; u < kMlpBatch; ++u)
        if (b0 + u < batch) s += x[u];
    }
    *loss = s / float(batch);
  }
}

// Forward pass and, with GRAD, the sample losses and the activations'
// gradients of a small network, a CTA per sample (grid-stride), a thread per
// unit, the weights staged once per CTA (rows padded to an odd stride, so that
// both W x and W^T d read shared memory without bank conflicts).
//
// Bound by launch and load latency: as one launch per layer and direction the
// step ran 8 dependent launches of 3-6 us each on a few thousand threads
// reading their weights from L2; here the layers follow one another inside a
// CTA behind barriers.  What an earlier kernel of the step writes is read from
// L2 (this kernel may have started before that one ended).  Every sum has the
// order of the launches per layer (the same bits).
struct MlpFused {
  const float *P, *X;
  int nf, h, c, batch;
  float *h1, *h2, *z;          // outputs: [batch][h] (may be null), [batch][c + 1] (null with GRAD)
  const int32_t *y;
  const float *yreg;
  float wreg;
  float *d1, *d2, *dz, *lb;
};

__host__ __device__ inline int mlp_odd(int k) { return k | 1; }
__host__ __device__ inline int64_t mlp_fused_floats(int64_t nf, int64_t h, int64_t c) {
  return (nf + h) * (h | 1) + h * ((c + 1) | 1) + nf + 3 * h + 3 * (c + 1);
}

template <bool GRAD>
__global__ void mlp_fused(MlpFused a, MlpOff o) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  extern __shared__ float sm[];
  const int nf = a.nf, h = a.h, c1 = a.c + 1, hs = mlp_odd(h), cs = mlp_odd(c1), t = threadIdx.x, T = blockDim.x;
  float *W1 = sm, *W2 = W1 + nf * hs, *W3 = W2 + h * hs, *x = W3 + h * cs, *v1 = x + nf, *v2 = v1 + h, *e2 = v2 + h;
  float *zs = e2 + h, *ds = zs + c1, *es = ds + c1;
  for (int k = t; k < nf * h; k += T) W1[(k / h) * hs + k % h] = __ldcg(a.P + o.w1 + k);
  for (int k = t; k < h * h; k += T) W2[(k / h) * hs + k % h] = __ldcg(a.P + o.w2 + k);
  for (int k = t; k < h * c1; k += T) W3[(k / c1) * cs + k % c1] = __ldcg(a.P + o.w3 + k);
  for (int b = blockIdx.x; b < a.batch; b += gridDim.x) {
    for (int k = t; k < nf; k += T) x[k] = __ldg(a.X + size_t(b) * nf + k);
    __syncthreads();
    for (int u = t; u < h; u += T) {
      float s = __ldcg(a.P + o.b1 + u);
      for (int i = 0; i < nf; ++i) s = fmaf(x[i], W1[i * hs + u], s);
      s = fmaxf(s, 0.0f);
      v1[u] = s;
      if (a.h1) a.h1[size_t(b) * h + u] = s;
    }
    __syncthreads();
    for (int u = t; u < h; u += T) {
      float s = __ldcg(a.P + o.b2 + u);
#pragma unroll 8
      for (int i = 0; i < h; ++i) s = fmaf(v1[i], W2[i * hs + u], s);
      s = fmaxf(s, 0.0f);
      v2[u] = s;
      if (a.h2) a.h2[size_t(b) * h + u] = s;
    }
    __syncthreads();
    for (int u = t; u < c1; u += T) {
      float s = __ldcg(a.P + o.b3 + u);
#pragma unroll 8
      for (int i = 0; i < h; ++i) s = fmaf(v2[i], W3[i * cs + u], s);
      zs[u] = s;
      if (!GRAD) a.z[size_t(b) * c1 + u] = s;
    }
    if (GRAD) {
      __syncthreads();
      const int c = a.c, yb = __ldg(a.y + b);
      float mx = zs[0];
      for (int k = 1; k < c; ++k) mx = fmaxf(mx, zs[k]);
      for (int k = t; k < c; k += T) es[k] = expf(zs[k] - mx);
      __syncthreads();
      float se = 0.0f;
      for (int k = 0; k < c; ++k) se += es[k];
      const float inv_b = 1.0f / float(a.batch);
      for (int k = t; k < c1; k += T) {
        float v;
        if (k < c) {
          const float p = es[k] / se;
          v = (p - (k == yb ? 1.0f : 0.0f)) * inv_b;
        } else {
          const float err = zs[c] - __ldg(a.yreg + b);
          v = 2.0f * a.wreg * err * inv_b;
          a.lb[b] = (logf(se) + mx - zs[yb]) + a.wreg * err * err;
        }
        ds[k] = v;
        a.dz[size_t(b) * c1 + k] = v;
      }
      __syncthreads();
      for (int u = t; u < h; u += T) {
        float s = 0.0f;
        for (int k = 0; k < c1; ++k) s = fmaf(ds[k], W3[u * cs + k], s);
        s = v2[u] > 0.0f ? s : 0.0f;
        e2[u] = s;
        a.d2[size_t(b) * h + u] = s;
      }
      __syncthreads();
      for (int u = t; u < h; u += T) {
        float s = 0.0f;
#pragma unroll 8
        for (int k = 0; k < h; ++k) s = fmaf(e2[k], W2[u * hs + k], s);
        a.d1[size_t(b) * h + u] = v1[u] > 0.0f ? s : 0.0f;
      }
    }
    __syncthreads();   // x, v1, v2 are reused by the next sample
  }
}

// dx[b][i] = (sum_o d[b][o] W[i][o]) * (act[b][i] > 0), o ascending
__global__ void dense_bwd_in(const float *d, const float *W, int nin, int nout, const float *act, int batch,
                             float *dx) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= batch * nin) return;
  const int b = idx / nin, i = idx % nin;
  float s = 0.0f;
  for (int o = 0; o < nout; ++o) s = fmaf(d[b * nout + o], W[i * nout + o], s);
  dx[idx] = act[idx] > 0.0f ? s : 0.0f;
}

__global__ void adam_step(float *p, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                          float eps, float c1, float c2) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float gk = g[k];
  const float mk = b1 * m[k] + (1.0f - b1) * gk;
  const float vk = b2 * v[k] + (1.0f - b2) * gk * gk;
  m[k] = mk;
  v[k] = vk;
  p[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

bool shape_ok(int nf, int h, int c, int batch) {
  return nf >= 1 && h >= 1 && c >= 1 && batch >= 1 && nf <= 4096 && h <= 4096 && c <= 4096 &&
         int64_t(batch) * std::max(std::max(nf, h), c + 1) < (int64_t(1) << 31);
}

// a launch whose start overlaps the end of the previous kernel (it waits for
// that kernel's results itself, griddepcontrol.wait)
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), int grid, int threads, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// One fused launch (mlp_fused) for networks whose weights fit the 48 KB of
// shared memory every CTA can have (hidden width up to about 95); a launch per
// layer for wider ones.  On a GB300 at 20-64-64-7, batch 160, a training step
// (gradient and Adam) took 73 us with a launch per layer.
bool mlp_small(int nf, int h, int c) { return mlp_fused_floats(nf, h, c) * 4 <= 48 * 1024; }

// The forward pass alone is fused for small batches only: its CTAs each stage the
// weights for one sample or a few, one barrier-separated layer after another,
// while the launches per layer have a thread per output.  us a call, per layer /
// fused: 20-64-64-6 16.6 / 14.3 at batch 1216 (29 MB of weights staged), 16.6 / 17.3
// at 2000 (47 MB); 20-95-95-6 18.7 / 14.9 at 608 (28 MB), 18.7 / 24.6 at 1000 (46
// MB); 20-8-8-3 12.5 / 9.3 at 5000, 12.5 / 14.5 at 10000.  (The gradient's fused
// kernel saves five launches and stays ahead at every batch up to 1,000,000.)
bool mlp_forward_fused(int nf, int h, int c, int batch) {
  return mlp_small(nf, h, c) && batch <= 5000 && mlp_fused_floats(nf, h, c) * 4 * batch <= 30000000;
}

template <bool GRAD>
cudaError_t launch_fused(const MlpFused &a, cudaStream_t s) {
  const int threads = std::min(256, std::max(64, (a.h + 31) / 32 * 32));
  return launch_pdl(mlp_fused<GRAD>, std::min(a.batch, 1216), threads, size_t(mlp_fused_floats(a.nf, a.h, a.c)) * 4, s,
                    a, mlp_off(a.nf, a.h, a.c));
}

iccg_status launched(cudaError_t e) { return e == cudaSuccess ? ICCG_OK : ICCG_ERR_CUDA; }

void forward(const float *P, int nf, int h, int c, const float *X, int batch, float *h1, float *h2, float *z,
             cudaStream_t s) {
  const MlpOff o = mlp_off(nf, h, c);
  dense_fwd<<<blocks_for(int64_t(batch) * h), kMlpThreads, 0, s>>>(X, nf, P + o.w1, P + o.b1, h, batch, h1, 1);
  dense_fwd<<<blocks_for(int64_t(batch) * h), kMlpThreads, 0, s>>>(h1, h, P + o.w2, P + o.b2, h, batch, h2, 1);
  dense_fwd<<<blocks_for(int64_t(batch) * (c + 1)), kMlpThreads, 0, s>>>(h2, h, P + o.w3, P + o.b3, c + 1, batch, z,
                                                                          0);
}

}  // namespace
}  // namespace iccg

using namespace iccg;

extern "C" {

int64_t iccg_mlp_nparams(int32_t nf, int32_t hidden, int32_t ncls) {
  if (nf < 1 || hidden < 1 || ncls < 1) return -1;
  return mlp_off(nf, hidden, ncls).total;
}

iccg_status iccg_mlp_forward(const float *params, int32_t nf, int32_t hidden, int32_t ncls, const float *X,
                             int32_t batch, float *out, float *act, iccg_stream_t stream) {
  if (!params || !X || !out || !shape_ok(nf, hidden, ncls, batch)) return ICCG_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (mlp_forward_fused(nf, hidden, ncls, batch)) {
    MlpFused a{};
    a.P = params; a.X = X; a.nf = nf; a.h = hidden; a.c = ncls; a.batch = batch; a.z = out;
    a.h1 = act;
    a.h2 = act ? act + size_t(batch) * hidden : nullptr;
    return launched(launch_fused<false>(a, s));
  }
  float *h1 = act, *tmp = nullptr;
  if (!h1) {
    if (cudaMallocAsync(reinterpret_cast<void **>(&tmp), sizeof(float) * 2 * size_t(batch) * hidden, s) != cudaSuccess)
      return ICCG_ERR_CUDA;
    h1 = tmp;
  }
  forward(params, nf, hidden, ncls, X, batch, h1, h1 + size_t(batch) * hidden, out, s);
  cudaError_t e = cudaGetLastError();
  if (tmp) cudaFreeAsync(tmp, s);
  return launched(e);
}

iccg_status iccg_mlp_grad(const float *params, int32_t nf, int32_t hidden, int32_t ncls, const float *X,
                          const int32_t *ycls, const float *yreg, float wreg, int32_t batch, float *grad,
                          float *loss, float *work, iccg_stream_t stream) {
  if (!params || !X || !ycls || !yreg || !grad || !loss || !work || !shape_ok(nf, hidden, ncls, batch))
    return ICCG_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int h = hidden, c = ncls;
  const size_t B = size_t(batch);
  float *h1 = work, *h2 = h1 + B * h, *d1 = h2 + B * h, *d2 = d1 + B * h, *z = d2 + B * h, *lb = z + B * (c + 1);
  float *dz = lb + B;
  // work layout: h1, h2, dh1, dh2 [batch][h]; z [batch][c+1]; sample losses
  // [batch]; dz [batch][c+1]
  const MlpOff o = mlp_off(nf, h, c);
  if (mlp_small(nf, h, c)) {
    MlpFused a{};
    a.P = params; a.X = X; a.nf = nf; a.h = h; a.c = c; a.batch = batch; a.h1 = h1; a.h2 = h2;
    a.y = ycls; a.yreg = yreg; a.wreg = wreg; a.d1 = d1; a.d2 = d2; a.dz = dz; a.lb = lb;
    const cudaError_t e = launch_fused<true>(a, s);
    if (e != cudaSuccess) return ICCG_ERR_CUDA;
  } else {
    forward(params, nf, h, c, X, batch, h1, h2, z, s);
    head_grad<<<blocks_for(batch), kMlpThreads, 0, s>>>(z, c, ycls, yreg, wreg, batch, dz, lb);
    dense_bwd_in<<<blocks_for(int64_t(batch) * h), kMlpThreads, 0, s>>>(dz, params + o.w3, h, c + 1, h2, batch, d2);
    dense_bwd_in<<<blocks_for(int64_t(batch) * h), kMlpThreads, 0, s>>>(d2, params + o.w2, h, h, h1, batch, d1);
    if (cudaGetLastError() != cudaSuccess) return ICCG_ERR_CUDA;
  }
  const MlpLayers L{{{X, d1, nf, h, o.w1}, {h1, d2, h, h, o.w2}, {h2, dz, h, c + 1, o.w3}}};
  return launched(launch_pdl(mlp_wgrad, blocks_for(o.total), kMlpThreads, 0, s, L, batch, o.total,
                             static_cast<const float *>(lb), grad, loss));
}

iccg_status iccg_mlp_adam(float *params, const float *grad, float *m, float *v, int64_t nparams, float lr,
                          float beta1, float beta2, float eps, int32_t step, iccg_stream_t stream) {
  if (!params || !grad || !m || !v || nparams < 1 || step < 1 || !(beta1 >= 0.f && beta1 < 1.f) ||
      !(beta2 >= 0.f && beta2 < 1.f))
    return ICCG_ERR_ARG;
  const float c1 = 1.0f - std::pow(beta1, float(step)), c2 = 1.0f - std::pow(beta2, float(step));
  return launched(launch_pdl(adam_step, blocks_for(nparams), kMlpThreads, 0, static_cast<cudaStream_t>(stream), params,
                             grad, m, v, nparams, lr, beta1, beta2, eps, c1, c2));
}

}  // extern "C"
