// Training of the MLP Q-function (an extension: the paper uses tables and names deep RL
// as future work, Section 7): fitted-Q regression on transitions the solver generated.
//
// Network 16 -> H -> H -> 4 * nprec (ReLU), fp32, parameters in the layout
// W1[H][16], b1[H], W2[H][H], b2[H], W3[4 nprec][H], b3[4 nprec].
// Loss over a batch of B transitions: (1 / (4 B)) sum_b sum_j 1/2 (Q(f_b)[j, a_bj] - y_bj)^2
// with targets y_bj = r_b + gamma (1 - done_b) max_p Q_target(f'_b)[j, p] (or given targets).
//
// Each CTA takes 32 samples of the batch, one per lane: the layers are evaluated for all of them at
// once (a warp takes eight neurons, the weights broadcast from shared memory, the activations kept
// sample-contiguous), then the gradient of every parameter is summed over the samples in sample
// order in registers. What bounded the step was latency: one sample after the other, one thread per
// neuron with its weights' loads in series, some 24 us a sample and 780 us a step at batch 1024 and
// H = 64. No atomics: the result is deterministic. A second kernel sums the CTA partials in CTA
// order and applies Adam (Kingma and Ba, ICLR 2015).
#include "internal.h"

namespace mpcg {

namespace {

constexpr int kMlpThreads = 256;

struct MlpShape {
  int H, nout, nprec;
  long long np;
  long long oW1, ob1, oW2, ob2, oW3, ob3;
};

__host__ __device__ MlpShape mlp_shape(int H, int nprec) {
  MlpShape s;
  s.H = H;
  s.nprec = nprec;
  s.nout = 4 * nprec;
  s.oW1 = 0;
  s.ob1 = s.oW1 + (long long)H * kNFeat;
  s.oW2 = s.ob1 + H;
  s.ob2 = s.oW2 + (long long)H * H;
  s.oW3 = s.ob2 + H;
  s.ob3 = s.oW3 + (long long)s.nout * H;
  s.np = s.ob3 + s.nout;
  return s;
}

constexpr int kRow = 36;  // floats between two rows of 32 samples (rows start four banks apart)
constexpr int kNeurons = 8;  // neurons of a warp at a time

// Shared memory of a CTA: the weights of one network, then rows of 32 samples.
struct MlpTile {
  float* w;                        // [np]
  float *f, *h1, *h2, *out;        // [16], [H], [H], [nout] rows
  float *dout, *dh2, *dh1;         // [nout], [H], [H] rows
};
__host__ __device__ inline long long mlp_rows(const MlpShape& s, bool grad) {
  return kNFeat + 2LL * s.H + s.nout + (grad ? s.nout + 2LL * s.H : 0);
}
__host__ __device__ inline long long mlp_wpad(const MlpShape& s) { return (s.np + 3) / 4 * 4; }
__device__ __forceinline__ MlpTile mlp_tile(float* sh, const MlpShape& s) {
  MlpTile t;
  t.w = sh;
  t.f = t.w + mlp_wpad(s);
  t.h1 = t.f + kNFeat * kRow;
  t.h2 = t.h1 + s.H * kRow;
  t.out = t.h2 + s.H * kRow;
  t.dout = t.out + s.nout * kRow;
  t.dh2 = t.dout + s.nout * kRow;
  t.dh1 = t.dh2 + s.H * kRow;
  return t;
}

__device__ __forceinline__ void load_weights(float* dst, const float* __restrict__ w, const MlpShape& s) {
  for (int i = threadIdx.x; i < (int)s.np; i += kMlpThreads) dst[i] = __ldg(w + i);
}

// y_i = act(b_i + sum_j W[i][j] x_j) over j in order, for rows i of n (x: m rows of 32 samples), and 0
// for lanes without a sample: they then pass nothing back and add nothing to a gradient, even where a
// weight is not finite.
template <bool RELU>
__device__ __forceinline__ void layer(const float* W, const float* b, int n, int m, const float* x, float* y,
                                      int samples) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i0 = w * kNeurons; i0 < n; i0 += kMlpThreads / 32 * kNeurons) {
    const int cnt = min(kNeurons, n - i0);
    float a[kNeurons];
#pragma unroll
    for (int u = 0; u < kNeurons; ++u) a[u] = u < cnt ? b[i0 + u] : 0.f;
#pragma unroll 4
    for (int j = 0; j < m; ++j) {
      const float xv = x[j * kRow + lane];
#pragma unroll
      for (int u = 0; u < kNeurons; ++u)
        if (u < cnt) a[u] = fmaf(W[(i0 + u) * m + j], xv, a[u]);
    }
#pragma unroll
    for (int u = 0; u < kNeurons; ++u)
      if (u < cnt) y[(i0 + u) * kRow + lane] = lane < samples && (!RELU || a[u] > 0.f) ? a[u] : 0.f;
  }
  __syncthreads();
}

// dx_k = sum_i W[i][k] dy_i over i in order where x_k > 0, else 0, for the m rows of x.
__device__ __forceinline__ void layer_back(const float* W, int n, int m, const float* dy, const float* x, float* dx) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int k0 = w * kNeurons; k0 < m; k0 += kMlpThreads / 32 * kNeurons) {
    const int cnt = min(kNeurons, m - k0);
    float a[kNeurons];
#pragma unroll
    for (int u = 0; u < kNeurons; ++u) a[u] = 0.f;
#pragma unroll 4
    for (int i = 0; i < n; ++i) {
      const float d = dy[i * kRow + lane];
#pragma unroll
      for (int u = 0; u < kNeurons; ++u)
        if (u < cnt) a[u] = fmaf(W[i * m + k0 + u], d, a[u]);
    }
#pragma unroll
    for (int u = 0; u < kNeurons; ++u)
      if (u < cnt) dx[(k0 + u) * kRow + lane] = x[(k0 + u) * kRow + lane] > 0.f ? a[u] : 0.f;
  }
  __syncthreads();
}

// g[i][j] = sum over the 32 samples, in order, of dy_i x_j (n by m), and gb[i] = the sum of dy_i.
// A thread takes four by four entries (rows i0, i0 + 4, ... would share banks: it takes rows a
// quarter of the tile apart), reading four samples of a row at a time.
__device__ __forceinline__ void layer_grad(const float* dy, int n, const float* x, int m, float* g, float* gb) {
  const int tj = (m + 3) / 4, ti = (n + 3) / 4;  // tile entries i0 + u ti, j0 + v tj
  for (int e = threadIdx.x; e < ti * tj; e += kMlpThreads) {
    const int i0 = e / tj, j0 = e - i0 * tj;
    float a[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) a[u][v] = 0.f;
    for (int q = 0; q < 8; ++q) {
      float4 y4[4], x4[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * ti, j = j0 + u * tj;
        y4[u] = *reinterpret_cast<const float4*>(dy + (i < n ? i : 0) * kRow + 4 * q);
        x4[u] = *reinterpret_cast<const float4*>(x + (j < m ? j : 0) * kRow + 4 * q);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          a[u][v] = fmaf(y4[u].x, x4[v].x, a[u][v]);
          a[u][v] = fmaf(y4[u].y, x4[v].y, a[u][v]);
          a[u][v] = fmaf(y4[u].z, x4[v].z, a[u][v]);
          a[u][v] = fmaf(y4[u].w, x4[v].w, a[u][v]);
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int i = i0 + u * ti, j = j0 + v * tj;
        if (i < n && j < m) g[(long long)i * m + j] = a[u][v];
      }
  }
  for (int i = threadIdx.x; i < n; i += kMlpThreads) {
    float a = 0.f;
    for (int q = 0; q < 32; ++q) a += dy[i * kRow + q];
    gb[i] = a;
  }
}

// The network on the `samples` samples in t.f (t.w: its weights): t.h1, t.h2, t.out.
__device__ __forceinline__ void net(const MlpTile& t, const MlpShape& s, int samples) {
  layer<true>(t.w + s.oW1, t.w + s.ob1, s.H, kNFeat, t.f, t.h1, samples);
  layer<true>(t.w + s.oW2, t.w + s.ob2, s.H, s.H, t.h1, t.h2, samples);
  layer<false>(t.w + s.oW3, t.w + s.ob3, s.nout, s.H, t.h2, t.out, samples);
}

// The features of the CTA's samples (row src of `feats` for lane t; zeros for lanes without one).
__device__ __forceinline__ void load_feats(float* f, const float* __restrict__ feats, const long long* src, int cnt) {
  for (int e = threadIdx.x; e < 32 * kNFeat; e += kMlpThreads) {
    const int smp = e / kNFeat, j = e - smp * kNFeat;
    f[j * kRow + smp] = smp < cnt ? __ldg(feats + src[smp] * kNFeat + j) : 0.f;
  }
  __syncthreads();
}

// r + gamma (1 - done) max over the entries p allowed for operation j of out[(j nprec + p) kRow]
// (the one-step Bellman backup of Section 4.1 with Q given by the network).
__device__ __forceinline__ float target_of(const float* out, int nprec, int j, const OpMask& mask, float r, int done,
                                           float gamma) {
  float m = -INFINITY;
  for (int p = 0; p < nprec; ++p)
    if ((mask.m[j] >> p) & 1u) m = fmaxf(m, out[(j * nprec + p) * kRow]);
  return r + (done ? 0.f : gamma * m);
}

// Fitted-Q targets y[b][4] from the target network wt on feats_next[b], 32 samples per CTA.
__global__ void __launch_bounds__(kMlpThreads) mlp_targets_kernel(const float* __restrict__ wt, int H, int nprec,
                                                                  const float* __restrict__ feats_next,
                                                                  const float* __restrict__ rew,
                                                                  const int* __restrict__ done, int B, float gamma,
                                                                  OpMask mask, float* y) {
  extern __shared__ __align__(16) float sh[];
  __shared__ long long src[32];
  const MlpShape s = mlp_shape(H, nprec);
  const MlpTile t = mlp_tile(sh, s);
  load_weights(t.w, wt, s);
  for (long long b0 = 32LL * blockIdx.x; b0 < B; b0 += 32LL * gridDim.x) {
    const int cnt = (int)min(32LL, B - b0);
    if (threadIdx.x < 32) src[threadIdx.x] = b0 + threadIdx.x;
    __syncthreads();
    load_feats(t.f, feats_next, src, cnt);
    net(t, s, cnt);
    const int smp = threadIdx.x >> 2, j = threadIdx.x & 3;
    if (smp < cnt) y[(b0 + smp) * 4 + j] = target_of(t.out + smp, nprec, j, mask, rew[b0 + smp], done[b0 + smp], gamma);
    __syncthreads();
  }
}

// 32 samples of the batch per CTA: gradient partials of the CTA -> part[blockIdx.x][np], loss
// partial -> lpart[blockIdx.x]. With y == nullptr the targets come from the target network on the
// next features (fitted Q); otherwise y[b][4] are the targets. With count > 0 sample b of the
// minibatch is transition Philox4x64-10(key (seed, 0x6d6c7030), counter (t, b, 0, 0)) word 0 mod
// count, otherwise transition b.
__global__ void __launch_bounds__(kMlpThreads) mlp_grad_kernel(
    const float* __restrict__ w, const float* __restrict__ wt, int H, int nprec, const float* __restrict__ feats,
    const float* __restrict__ feats_next, const int* __restrict__ acts, const float* __restrict__ rew,
    const int* __restrict__ done, const float* __restrict__ y, long long count, unsigned long long seed,
    unsigned long long step, int B, float gamma, OpMask mask, float* part, double* lpart) {
  extern __shared__ __align__(16) float sh[];
  __shared__ long long src[32];
  __shared__ float yt[32][4];
  const MlpShape s = mlp_shape(H, nprec);
  const MlpTile t = mlp_tile(sh, s);
  const int b0 = blockIdx.x * 32, cnt = min(32, B - b0);
  const float scale = 1.f / (4.f * (float)B);
  if (threadIdx.x < 32) {
    long long at = b0 + (threadIdx.x < cnt ? (int)threadIdx.x : 0);
    if (count > 0) {
      U64x4 c;
      c.v[0] = step;
      c.v[1] = (unsigned long long)at;
      c.v[2] = 0;
      c.v[3] = 0;
      at = (long long)(philox4x64_10(c, seed, 0x6d6c7030ull).v[0] % (unsigned long long)count);
    }
    src[threadIdx.x] = at;
  }
  __syncthreads();
  const int smp = threadIdx.x >> 2, op = threadIdx.x & 3;  // (the first 128 threads: a sample's operation each)
  if (y) {
    if (smp < cnt) yt[smp][op] = y[(b0 + smp) * 4 + op];
  } else {
    load_weights(t.w, wt, s);
    load_feats(t.f, feats_next, src, cnt);
    net(t, s, cnt);
    if (smp < cnt) yt[smp][op] = target_of(t.out + smp, nprec, op, mask, rew[src[smp]], done[src[smp]], gamma);
    __syncthreads();
  }
  load_weights(t.w, w, s);
  load_feats(t.f, feats, src, cnt);
  net(t, s, cnt);
  // output error: only the taken action of each operation carries gradient
  for (int e = threadIdx.x; e < s.nout * 32; e += kMlpThreads) t.dout[(e >> 5) * kRow + (e & 31)] = 0.f;
  __syncthreads();
  double l = 0.0;
  if (smp < cnt) {
    const int o = op * nprec + acts[src[smp] * 4 + op];
    const float d = t.out[o * kRow + smp] - yt[smp][op];
    t.dout[o * kRow + smp] = d * scale;
    l = 0.5 * (double)d * (double)d * (double)scale;
  }
  __syncthreads();
  // the loss: the first four warps' terms
  __shared__ double lw[4];
  if (threadIdx.x < 128) {
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) l += __shfl_xor_sync(0xffffffffu, l, q);
    if ((threadIdx.x & 31) == 0) lw[threadIdx.x >> 5] = l;
  }
  layer_back(t.w + s.oW3, s.nout, s.H, t.dout, t.h2, t.dh2);
  layer_back(t.w + s.oW2, s.H, s.H, t.dh2, t.h1, t.dh1);
  float* dst = part + (long long)blockIdx.x * s.np;
  layer_grad(t.dh1, s.H, t.f, kNFeat, dst + s.oW1, dst + s.ob1);
  layer_grad(t.dh2, s.H, t.h1, s.H, dst + s.oW2, dst + s.ob2);
  layer_grad(t.dout, s.nout, t.h2, s.H, dst + s.oW3, dst + s.ob3);
  if (threadIdx.x == 0) lpart[blockIdx.x] = lw[0] + lw[1] + lw[2] + lw[3];
}

// Sums the CTA partials (CTA order) into grad; optionally applies Adam step t to w.
__global__ void mlp_reduce_adam_kernel(const float* __restrict__ part, int nparts, long long np, float* grad, float* w,
                                       float* m, float* v, int t, float lr, float b1, float b2, float eps,
                                       const double* lpart, double* loss) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < np; i += (long long)gridDim.x * blockDim.x) {
    float gi = 0.f;
    for (int c = 0; c < nparts; ++c) gi += part[(long long)c * np + i];
    if (grad) grad[i] = gi;
    if (w) {
      const float mi = b1 * m[i] + (1.f - b1) * gi;
      const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
      m[i] = mi;
      v[i] = vi;
      const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
      w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
  }
  if (loss && blockIdx.x == 0 && threadIdx.x == 0) {
    double l = 0.0;
    for (int c = 0; c < nparts; ++c) l += lpart[c];
    *loss = l;
  }
}

}  // namespace

long long mlp_nparams_dev(int H, int nprec) { return mlp_shape(H, nprec).np; }

size_t mlp_grad_smem(int H, int nprec) {
  const MlpShape s = mlp_shape(H, nprec);
  return sizeof(float) * (size_t)(mlp_wpad(s) + kRow * mlp_rows(s, true));
}

cudaError_t mlp_set_smem_limit(size_t bytes) {
  const cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(mlp_targets_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t launch_mlp_grad(const float* w, const float* wt, int H, int nprec, const float* feats,
                            const float* feats_next, const int* acts, const float* rew, const int* done, const float* y,
                            long long count, unsigned long long seed, unsigned long long t, int B, float gamma,
                            OpMask mask, float* part, double* lpart, cudaStream_t s) {
  cudaGetLastError();
  mlp_grad_kernel<<<(B + kMlpChunk - 1) / kMlpChunk, kMlpThreads, mlp_grad_smem(H, nprec), s>>>(
      w, wt, H, nprec, feats, feats_next, acts, rew, done, y, count, seed, t, B, gamma, mask, part, lpart);
  return cudaGetLastError();
}

cudaError_t launch_mlp_targets(const float* wt, int H, int nprec, const float* feats_next, const float* rew,
                               const int* done, int B, float gamma, OpMask mask, float* y, cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  const MlpShape sh = mlp_shape(H, nprec);
  const size_t smem = sizeof(float) * (size_t)(mlp_wpad(sh) + kRow * mlp_rows(sh, false));
  const int grid = (int)((B + 31LL) / 32);
  cudaGetLastError();
  mlp_targets_kernel<<<grid < 608 ? grid : 608, kMlpThreads, smem, s>>>(wt, H, nprec, feats_next, rew, done, B, gamma,
                                                                         mask, y);
  return cudaGetLastError();
}

cudaError_t launch_mlp_reduce_adam(const float* part, int nparts, long long np, float* grad, float* w, float* m,
                                   float* v, int t, float lr, const double* lpart, double* loss, cudaStream_t s) {
  cudaGetLastError();
  mlp_reduce_adam_kernel<<<(int)((np + 255) / 256), 256, 0, s>>>(part, nparts, np, grad, w, m, v, t, lr, 0.9f, 0.999f,
                                                                  1e-8f, lpart, loss);
  return cudaGetLastError();
}

}  // namespace mpcg
