// Training of the learned blending coefficient on the GPU: the network maps
// an element's normalised modal energies (encoded, nin inputs) through two
// hidden layers of 32 ReLU units to a sigmoid output; the loss is the
// cross-entropy against the smoothness indicator's alpha (in [0, 1], taken as
// a probability), whose gradient in the output logit is (y - t) / n.  Forward and
// backward passes, Adam, and the epoch loop are this file's kernels.
#include <cooperative_groups.h>

#include <cstdint>
#include <cstring>
#include <vector>

#include "../../include/cr.h"
#include "cr_common.cuh"

namespace {

constexpr int kH = 32;
constexpr int kChunk = 64;    // samples cached in shared memory per pass
constexpr int kThreads = 128;

__host__ __device__ constexpr int param_count(int nin) {
  return kH * nin + kH + kH * kH + kH + kH + 1;
}

// Gradient of the cross-entropy over samples [0, n) (indices through idx
// when given) and the loss (t softplus(-z) + (1 - t) softplus(z)) * inv_n.
// One block handles chunks of 64 samples: threads 0..63 run forward and
// backward for one sample each into shared memory, then all threads reduce
// their share of the gradient entries.  Block b writes its partial sums to
// part[b][0..P) and its loss to part[b][P]; k_mlp_reduce adds the blocks in a
// fixed order, so the result does not depend on block scheduling.
template <int NIN>
__global__ void __launch_bounds__(kThreads) k_mlp_grad(const float* __restrict__ prm,
                                                        const float* __restrict__ X,
                                                        const float* __restrict__ T,
                                                        const int* __restrict__ idx, int n,
                                                        float inv_n, float* __restrict__ part) {
  constexpr int P = param_count(NIN);
  constexpr int PER = (P + kThreads - 1) / kThreads;
  constexpr int REC = NIN + 4 * kH + 1;  // x, h1, da1, h2, da2, dz per sample
  extern __shared__ float sm[];
  float* sp = sm;                // parameters [P]
  float* sr = sm + P;            // sample records [kChunk][REC]
  const int tid = threadIdx.x;
  for (int g = tid; g < P; g += kThreads) sp[g] = prm[g];
  const float* W1 = sp;
  const float* B1 = W1 + kH * NIN;
  const float* W2 = B1 + kH;
  const float* B2 = W2 + kH * kH;
  const float* W3 = B2 + kH;
  float acc[PER];
#pragma unroll
  for (int r = 0; r < PER; ++r) acc[r] = 0.0f;
  float lsum = 0.0f;
  __syncthreads();
  const float B3 = W3[kH];  // read only after every thread's copy is visible
  for (int base = blockIdx.x * kChunk; base < n; base += gridDim.x * kChunk) {
    const int cnt = min(kChunk, n - base);
    if (tid < cnt) {
      const int s = idx ? idx[base + tid] : base + tid;
      float* R = sr + tid * REC;
      float* x = R;
      float* h1 = x + NIN;
      float* d1 = h1 + kH;
      float* h2 = d1 + kH;
      float* d2 = h2 + kH;
#pragma unroll
      for (int i = 0; i < NIN; ++i) x[i] = X[(size_t)s * NIN + i];
      for (int j = 0; j < kH; ++j) {
        float a = B1[j];
#pragma unroll
        for (int i = 0; i < NIN; ++i) a += W1[j * NIN + i] * x[i];
        h1[j] = a;  // pre-activation kept until the backward pass
      }
      float z = B3;
      for (int j = 0; j < kH; ++j) {
        float a = B2[j];
        for (int i = 0; i < kH; ++i) a += W2[j * kH + i] * fmaxf(h1[i], 0.0f);
        h2[j] = a;
        z += W3[j] * fmaxf(a, 0.0f);
      }
      const float y = 1.0f / (1.0f + expf(-z));
      const float t = T[s];
      const float sp = log1pf(expf(-fabsf(z)));  // softplus(z) = max(z, 0) + sp
      lsum += (t * (fmaxf(-z, 0.0f) + sp) + (1.0f - t) * (fmaxf(z, 0.0f) + sp)) * inv_n;
      const float dz = (y - t) * inv_n;
      R[REC - 1] = dz;
      for (int j = 0; j < kH; ++j) d2[j] = h2[j] > 0.0f ? dz * W3[j] : 0.0f;
      for (int i = 0; i < kH; ++i) {
        float a = 0.0f;
        for (int j = 0; j < kH; ++j) a += W2[j * kH + i] * d2[j];
        d1[i] = h1[i] > 0.0f ? a : 0.0f;
      }
      for (int j = 0; j < kH; ++j) {
        h1[j] = fmaxf(h1[j], 0.0f);
        h2[j] = fmaxf(h2[j], 0.0f);
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const int g = tid + r * kThreads;
      if (g >= P) break;
      float a = 0.0f;
      if (g < kH * NIN) {  // W1[j][i] += d1[j] x[i]
        const int j = g / NIN, i = g - j * NIN;
        for (int s = 0; s < cnt; ++s) a += sr[s * REC + NIN + kH + j] * sr[s * REC + i];
      } else if (g < kH * NIN + kH) {  // b1
        const int j = g - kH * NIN;
        for (int s = 0; s < cnt; ++s) a += sr[s * REC + NIN + kH + j];
      } else if (g < kH * NIN + kH + kH * kH) {  // W2[j][i] += d2[j] h1[i]
        const int gg = g - kH * NIN - kH, j = gg / kH, i = gg - j * kH;
        for (int s = 0; s < cnt; ++s) a += sr[s * REC + NIN + 3 * kH + j] * sr[s * REC + NIN + i];
      } else if (g < kH * NIN + 2 * kH + kH * kH) {  // b2
        const int j = g - kH * NIN - kH - kH * kH;
        for (int s = 0; s < cnt; ++s) a += sr[s * REC + NIN + 3 * kH + j];
      } else if (g < P - 1) {  // w3[j] += dz h2[j]
        const int j = g - kH * NIN - 2 * kH - kH * kH;
        for (int s = 0; s < cnt; ++s) a += sr[s * REC + REC - 1] * sr[s * REC + NIN + 2 * kH + j];
      } else {  // b3
        for (int s = 0; s < cnt; ++s) a += sr[s * REC + REC - 1];
      }
      acc[r] += a;
    }
    __syncthreads();
  }
  float* out = part + (size_t)blockIdx.x * (P + 1);
#pragma unroll
  for (int r = 0; r < PER; ++r) {
    const int g = tid + r * kThreads;
    if (g < P) out[g] = acc[r];
  }
  // block sum of the per-sample losses (threads >= 64 hold 0), fixed order
  __syncthreads();
  sr[tid] = lsum;
  __syncthreads();
  if (tid == 0) {
    float l = 0.0f;
    for (int i = 0; i < kThreads; ++i) l += sr[i];
    out[P] = l;
  }
}

// grad[g] = sum over blocks b = 0, 1, ... of part[b][g]; loss likewise (g = P).
__global__ void k_mlp_reduce(const float* __restrict__ part, int nblocks, int P,
                             float* __restrict__ grad, float* __restrict__ loss) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g > P) return;
  float a = 0.0f;
  for (int b = 0; b < nblocks; ++b) a += part[(size_t)b * (P + 1) + g];
  if (g < P) grad[g] = a;
  else *loss = a;
}

__global__ void k_mlp_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, int n, float lr, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float b1 = 0.9f, b2 = 0.999f;
  const float mi = b1 * m[i] + (1.0f - b1) * g[i];
  const float vi = b2 * v[i] + (1.0f - b2) * g[i] * g[i];
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

__global__ void k_accumulate(float* dst, const float* src) { *dst += *src; }

constexpr int kMaxGradBlocks = 304;  // two blocks per SM

int grad_blocks(int n) {
  int blocks = (n + kChunk - 1) / kChunk;
  if (blocks > kMaxGradBlocks) blocks = kMaxGradBlocks;
  return blocks < 1 ? 1 : blocks;
}

// Loss and gradient of samples [0, n) into grad and loss (overwritten); part
// is scratch of grad_blocks(n) * (P + 1) floats.
template <int NIN>
cudaError_t launch_grad(const float* prm, const float* X, const float* T, const int* idx, int n,
                        float* part, float* grad, float* loss, cudaStream_t s) {
  constexpr int P = param_count(NIN);
  const size_t smem = (size_t)(P + kChunk * (NIN + 4 * kH + 1)) * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(k_mlp_grad<NIN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  const int blocks = grad_blocks(n);
  k_mlp_grad<NIN><<<blocks, kThreads, smem, s>>>(prm, X, T, idx, n, 1.0f / float(n), part);
  k_mlp_reduce<<<(P + 1 + 255) / 256, 256, 0, s>>>(part, blocks, P, grad, loss);
  return cudaGetLastError();
}

cudaError_t dispatch_grad(int nin, const float* prm, const float* X, const float* T, const int* idx,
                          int n, float* part, float* grad, float* loss, cudaStream_t s) {
  switch (nin) {
    case 2: return launch_grad<2>(prm, X, T, idx, n, part, grad, loss, s);
    case 3: return launch_grad<3>(prm, X, T, idx, n, part, grad, loss, s);
    case 4: return launch_grad<4>(prm, X, T, idx, n, part, grad, loss, s);
    case 5: return launch_grad<5>(prm, X, T, idx, n, part, grad, loss, s);
    case 9: return launch_grad<9>(prm, X, T, idx, n, part, grad, loss, s);
    case 16: return launch_grad<16>(prm, X, T, idx, n, part, grad, loss, s);
    case 25: return launch_grad<25>(prm, X, T, idx, n, part, grad, loss, s);
  }
  return cudaErrorInvalidValue;
}

bool nin_supported(int nin) {
  return nin == 2 || nin == 3 || nin == 4 || nin == 5 || nin == 9 || nin == 16 || nin == 25;
}

// ---------------------------------------------------------------------------
// One epoch of Adam in one launch (minibatches of up to kEpochBlocks chunks of
// kChunk samples).  A minibatch is little work (512 samples of 16 inputs: 6
// MFLOP) behind a chain of dependent steps, and as four kernels per minibatch
// it took 40 us: launches, one thread per sample walking through both layers,
// parameters and moments through memory.  Here a cluster of up to 8 CTAs keeps
// the parameters in shared memory for the whole epoch; CTA r takes chunks r, r +
// C, ... of each minibatch with four hidden units of two samples per thread, then
// the chunks' partial gradients are exchanged through distributed shared memory
// and each CTA updates its share of the parameters in every CTA (two cluster
// barriers per minibatch).  The next chunk's samples are fetched meanwhile.
// Every sum runs in the order of k_mlp_grad and k_mlp_reduce (units and samples
// ascending, chunk by chunk).
// Measured (50,000 samples of 16 inputs, batch 512, two epochs, whole call):
// 7.93 -> 1.82 ms.  Up to 48 chunks (3,072 samples): past that one cluster falls behind
// the grid of one launch per step (16 inputs, ms per epoch, this kernel and that: 3,073
// samples 0.63 and 0.75, 6,000 0.59 and 0.50).
constexpr int kEpochThreads = 352;                       // 11 warps: one gradient item per thread
constexpr int kMaxCluster = 8, kEpochBlocks = 48;        // chunks per minibatch the kernel takes
constexpr int kHS = kH + 4;                              // row stride of the hidden arrays (128-bit reads
                                                         // of 8 rows hit all banks: 4 x odd)
constexpr int x_stride(int nin) { return 4 * (((nin + 3) / 4) | 1); }

// Samples of chunk c of minibatch k (k batch < n; batch and c kChunk stay in the int
// range, (k + 1) batch need not).
__host__ __device__ constexpr int chunk_samples(int n, int batch, int k, int c) {
  const int total = batch < n - k * batch ? batch : n - k * batch;
  return total - c * kChunk < kChunk ? total - c * kChunk : kChunk;
}
static_assert(chunk_samples(2147483647, 3072, 699050, 0) == kChunk && chunk_samples(2147483647, 3072, 699050, 31) == 63 &&
                  chunk_samples(700, 512, 1, 2) == 60,
              "the last minibatch of the largest sample count");

template <int NIN> struct EpochShape {
  static constexpr int P = param_count(NIN), XS = x_stride(NIN);
  static constexpr int PER = (kChunk * NIN + kEpochThreads - 1) / kEpochThreads;
  static size_t smem(int per_cta) {
    return sizeof(float) * ((P + 3) / 4 * 4 + kChunk * (XS + 4 * kHS + 4) + (size_t)per_cta * (P + 1));
  }
};

template <int NIN>
__global__ void __launch_bounds__(kEpochThreads, 1)
    k_mlp_epoch(float* __restrict__ prm, float* __restrict__ mom, float* __restrict__ var, const float* __restrict__ X,
                const float* __restrict__ T, const int* __restrict__ idx, int n, int batch,
                const float2* __restrict__ corr, float lr, float* __restrict__ epoch_loss) {
  namespace cg = cooperative_groups;
  using Sh = EpochShape<NIN>;
  constexpr int P = Sh::P, XS = Sh::XS, PER = Sh::PER;
  cg::cluster_group cl = cg::this_cluster();
  const int C = int(cl.num_blocks()), rank = int(cl.block_rank()), tid = threadIdx.x;
  extern __shared__ __align__(16) float sm[];
  float* sp = sm;                          // parameters [P]
  float* xs = sp + (P + 3) / 4 * 4;        // inputs [kChunk][XS]
  float* h1 = xs + kChunk * XS;            // [kChunk][kHS]: relu of layer 1
  float* h2 = h1 + kChunk * kHS;           // relu of layer 2
  float* d1 = h2 + kChunk * kHS;           // gradients at the pre-activations
  float* d2 = d1 + kChunk * kHS;
  float* dz = d2 + kChunk * kHS;           // [kChunk]
  float* ls = dz + kChunk;                 // [kChunk] losses
  float* ts = ls + kChunk;                 // [kChunk] targets
  float* part = ts + 2 * kChunk;           // [chunks of this CTA][P + 1]
  const float* W1 = sp;
  const float* B1 = W1 + kH * NIN;
  const float* W2 = B1 + kH;
  const float* B2 = W2 + kH * kH;
  const float* W3 = B2 + kH;
  // this CTA's share of the parameters, one per thread and pass, moments in registers
  const int share = (P + C - 1) / C, first = rank * share;
  constexpr int OWN = (P + kEpochThreads - 1) / kEpochThreads;  // C = 1: all of them
  float rm[OWN], rv[OWN];
#pragma unroll
  for (int o = 0; o < OWN; ++o) {
    const int g = first + tid + o * kEpochThreads;
    const bool own = tid + o * kEpochThreads < share && g < P;
    rm[o] = own ? mom[g] : 0.0f;
    rv[o] = own ? var[g] : 0.0f;
  }
  for (int g = tid; g < P; g += kEpochThreads) sp[g] = prm[g];
  for (int t = tid; t < kChunk * XS; t += kEpochThreads) xs[t] = 0.0f;  // padding columns stay 0
  const int nb = (n - 1) / batch + 1;
  float el = 0.0f;

  // the chunk (minibatch k, chunk c) of this CTA's sequence into registers
  float rx[PER], rt = 0.0f;
  auto fetch = [&](int k, int c) {
    const int base = k * batch + c * kChunk;
    const int cnt = chunk_samples(n, batch, k, c);
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const int t = tid + r * kEpochThreads, s = t / NIN;
      rx[r] = s < cnt ? X[(size_t)idx[base + s] * NIN + (t - s * NIN)] : 0.0f;
    }
    if (tid < kChunk) rt = tid < cnt ? T[idx[base + tid]] : 0.0f;
  };
  auto chunks_of = [&](int k) { return (min(batch, n - k * batch) + kChunk - 1) / kChunk; };
  if (rank < chunks_of(0)) fetch(0, rank);
  cl.sync();

  for (int k = 0; k < nb; ++k) {
    const int total = min(batch, n - k * batch), nc = chunks_of(k);
    const float inv_n = 1.0f / float(total);
    int slot = 0;
    for (int c = rank; c < nc; c += C, ++slot) {
      const int cnt = min(kChunk, total - c * kChunk);
#pragma unroll
      for (int r = 0; r < PER; ++r) {
        const int t = tid + r * kEpochThreads, s = t / NIN;
        if (s < kChunk) xs[s * XS + (t - s * NIN)] = rx[r];
      }
      if (tid < kChunk) ts[tid] = rt;
      __syncthreads();
      // the next chunk of this CTA (in this minibatch or the next one it has work in)
      if (c + C < nc) fetch(k, c + C);
      else if (k + 1 < nb && rank < chunks_of(k + 1)) fetch(k + 1, rank);
      // threads 0..255: samples s0, s0 + 32 and hidden units j0 .. j0 + 3
      const int s0 = tid & 31, j0 = (tid >> 5) * 4;
      const bool work = tid < 256;
      float pre[2][4];
      if (work) {  // layer 1
#pragma unroll
        for (int u = 0; u < 4; ++u) pre[0][u] = pre[1][u] = B1[j0 + u];
#pragma unroll
        for (int i0 = 0; i0 < NIN; i0 += 4) {
          const float4 xa = *reinterpret_cast<const float4*>(xs + s0 * XS + i0);
          const float4 xb = *reinterpret_cast<const float4*>(xs + (s0 + 32) * XS + i0);
          const float va[4] = {xa.x, xa.y, xa.z, xa.w}, vb[4] = {xb.x, xb.y, xb.z, xb.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (i0 + i >= NIN) break;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float w = W1[(j0 + u) * NIN + i0 + i];
              pre[0][u] = fmaf(w, va[i], pre[0][u]);
              pre[1][u] = fmaf(w, vb[i], pre[1][u]);
            }
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<float4*>(h1 + (s0 + 32 * h) * kHS + j0) =
              make_float4(fmaxf(pre[h][0], 0.0f), fmaxf(pre[h][1], 0.0f), fmaxf(pre[h][2], 0.0f), fmaxf(pre[h][3], 0.0f));
      }
      __syncthreads();
      if (work) {  // layer 2
#pragma unroll
        for (int u = 0; u < 4; ++u) pre[0][u] = pre[1][u] = B2[j0 + u];
#pragma unroll
        for (int i0 = 0; i0 < kH; i0 += 4) {
          const float4 xa = *reinterpret_cast<const float4*>(h1 + s0 * kHS + i0);
          const float4 xb = *reinterpret_cast<const float4*>(h1 + (s0 + 32) * kHS + i0);
          const float va[4] = {xa.x, xa.y, xa.z, xa.w}, vb[4] = {xb.x, xb.y, xb.z, xb.w};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 w4 = *reinterpret_cast<const float4*>(W2 + (j0 + u) * kH + i0);
            const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              pre[0][u] = fmaf(w[i], va[i], pre[0][u]);
              pre[1][u] = fmaf(w[i], vb[i], pre[1][u]);
            }
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<float4*>(h2 + (s0 + 32 * h) * kHS + j0) =
              make_float4(fmaxf(pre[h][0], 0.0f), fmaxf(pre[h][1], 0.0f), fmaxf(pre[h][2], 0.0f), fmaxf(pre[h][3], 0.0f));
      }
      __syncthreads();
      if (tid < kChunk) {  // output, loss and its gradient in the logit; samples past the end count as 0
        float z = W3[kH];
#pragma unroll
        for (int j = 0; j < kH; ++j) z = fmaf(W3[j], h2[tid * kHS + j], z);
        const float y = 1.0f / (1.0f + expf(-z));
        const float t = ts[tid];
        const float sp1 = log1pf(expf(-fabsf(z)));
        const float l = (t * (fmaxf(-z, 0.0f) + sp1) + (1.0f - t) * (fmaxf(z, 0.0f) + sp1)) * inv_n;
        ls[tid] = tid < cnt ? l : 0.0f;
        dz[tid] = tid < cnt ? (y - t) * inv_n : 0.0f;
      }
      __syncthreads();
      if (work) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int s = s0 + 32 * h;
          float v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = pre[h][u] > 0.0f ? dz[s] * W3[j0 + u] : 0.0f;
          *reinterpret_cast<float4*>(d2 + s * kHS + j0) = make_float4(v[0], v[1], v[2], v[3]);
        }
      }
      __syncthreads();
      if (work) {  // d1[i] = sum_j W2[j][i] d2[j] for i = j0 .. j0 + 3
        float a[2][4] = {};
#pragma unroll
        for (int j1 = 0; j1 < kH; j1 += 4) {
          const float4 xa = *reinterpret_cast<const float4*>(d2 + s0 * kHS + j1);
          const float4 xb = *reinterpret_cast<const float4*>(d2 + (s0 + 32) * kHS + j1);
          const float va[4] = {xa.x, xa.y, xa.z, xa.w}, vb[4] = {xb.x, xb.y, xb.z, xb.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 w4 = *reinterpret_cast<const float4*>(W2 + (j1 + j) * kH + j0);
            const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              a[0][u] = fmaf(w[u], va[j], a[0][u]);
              a[1][u] = fmaf(w[u], vb[j], a[1][u]);
            }
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int s = s0 + 32 * h;
          const float4 p4 = *reinterpret_cast<const float4*>(h1 + s * kHS + j0);
          *reinterpret_cast<float4*>(d1 + s * kHS + j0) =
              make_float4(p4.x > 0.0f ? a[h][0] : 0.0f, p4.y > 0.0f ? a[h][1] : 0.0f, p4.z > 0.0f ? a[h][2] : 0.0f,
                          p4.w > 0.0f ? a[h][3] : 0.0f);
        }
      }
      __syncthreads();
      // gradient of this chunk, samples in order: tiles of 2 x 4 of W2 and W1,
      // single entries of the rest
      float* out = part + (size_t)slot * (P + 1);
      constexpr int TW2 = kH / 2 * (kH / 4), QN = (NIN + 3) / 4, TW1 = kH / 2 * QN;
      for (int it = tid; it < TW2 + TW1 + 3 * kH + 2; it += kEpochThreads) {
        if (it < TW2 + TW1) {
          const bool second = it < TW2;
          const int r = second ? it : it - TW2, q = second ? kH / 4 : QN;
          const int j = r / q * 2, i = r % q * 4;
          const float* A = (second ? d2 : d1) + j;
          const float* B = (second ? h1 : xs) + i;
          const int bs = second ? kHS : XS;
          float a[2][4] = {};
#pragma unroll 8
          for (int s = 0; s < cnt; ++s) {
            const float2 d = *reinterpret_cast<const float2*>(A + s * kHS);
            const float4 v = *reinterpret_cast<const float4*>(B + s * bs);
            a[0][0] = fmaf(d.x, v.x, a[0][0]);
            a[0][1] = fmaf(d.x, v.y, a[0][1]);
            a[0][2] = fmaf(d.x, v.z, a[0][2]);
            a[0][3] = fmaf(d.x, v.w, a[0][3]);
            a[1][0] = fmaf(d.y, v.x, a[1][0]);
            a[1][1] = fmaf(d.y, v.y, a[1][1]);
            a[1][2] = fmaf(d.y, v.z, a[1][2]);
            a[1][3] = fmaf(d.y, v.w, a[1][3]);
          }
          float* o = second ? out + kH * NIN + kH : out;
          const int row = second ? kH : NIN;
#pragma unroll
          for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int w = 0; w < 4; ++w)
              if (i + w < row) o[(j + u) * row + i + w] = a[u][w];
        } else {
          const int r = it - TW2 - TW1, kind = r / kH, j = r - kind * kH;
          float a = 0.0f;
          if (kind == 0) {  // b1
            for (int s = 0; s < cnt; ++s) a += d1[s * kHS + j];
            out[kH * NIN + j] = a;
          } else if (kind == 1) {  // b2
            for (int s = 0; s < cnt; ++s) a += d2[s * kHS + j];
            out[kH * NIN + kH + kH * kH + j] = a;
          } else if (kind == 2) {  // w3
            for (int s = 0; s < cnt; ++s) a = fmaf(dz[s], h2[s * kHS + j], a);
            out[kH * NIN + 2 * kH + kH * kH + j] = a;
          } else {  // b3 and the loss
            const float* v = j == 0 ? dz : ls;
            for (int s = 0; s < cnt; ++s) a += v[s];
            out[P - 1 + j] = a;
          }
        }
      }
      __syncthreads();
    }
    cl.sync();  // every chunk's partial gradient is there
    const float2 cc = corr[k];
#pragma unroll
    for (int o = 0; o < OWN; ++o) {
      const int l = tid + o * kEpochThreads, g = first + l;
      if (l < share && g < P) {
        float gr = 0.0f;
        for (int c = 0; c < nc; ++c) gr += cl.map_shared_rank(part, c % C)[(size_t)(c / C) * (P + 1) + g];
        const float b1 = 0.9f, b2 = 0.999f;
        const float mi = b1 * rm[o] + (1.0f - b1) * gr;
        const float vi = b2 * rv[o] + (1.0f - b2) * gr * gr;
        rm[o] = mi;
        rv[o] = vi;
        float p = sp[g];
        p -= lr * (mi / cc.x) / (sqrtf(vi / cc.y) + 1e-8f);
        for (int c = 0; c < C; ++c) cl.map_shared_rank(sp, c)[g] = p;
      }
    }
    if (rank == 0 && tid == kEpochThreads - 1) {
      float l = 0.0f;
      for (int c = 0; c < nc; ++c) l += cl.map_shared_rank(part, c % C)[(size_t)(c / C) * (P + 1) + P];
      el += l;
    }
    cl.sync();  // every CTA has the new parameters, and nobody reads the partial sums any more
  }
#pragma unroll
  for (int o = 0; o < OWN; ++o) {
    const int l = tid + o * kEpochThreads, g = first + l;
    if (l < share && g < P) {
      mom[g] = rm[o];
      var[g] = rv[o];
      prm[g] = sp[g];
    }
  }
  if (rank == 0 && tid == kEpochThreads - 1) *epoch_loss = el;
}

template <int NIN>
cudaError_t launch_epoch(float* prm, float* mom, float* var, const float* X, const float* T, const int* idx, int n,
                         int batch, const float2* corr, float lr, float* epoch_loss, cudaStream_t s) {
  const int chunks = (batch + kChunk - 1) / kChunk;  // batch <= n
  int C = 1;
  while (C < kMaxCluster && C < chunks) C *= 2;
  const size_t smem = EpochShape<NIN>::smem((chunks + C - 1) / C);
  // the limit belongs to the kernel, not to the call: every call sets the one of the
  // largest minibatch, so that calls of several threads do not lower each other's
  constexpr int kMost = (kEpochBlocks + kMaxCluster - 1) / kMaxCluster;
  cudaError_t e = cudaFuncSetAttribute(k_mlp_epoch<NIN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)EpochShape<NIN>::smem(kMost));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(kEpochThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mlp_epoch<NIN>, prm, mom, var, X, T, idx, n, batch, corr, lr, epoch_loss);
}

cudaError_t dispatch_epoch(int nin, float* prm, float* mom, float* var, const float* X, const float* T, const int* idx,
                           int n, int batch, const float2* corr, float lr, float* epoch_loss, cudaStream_t s) {
  switch (nin) {
    case 2: return launch_epoch<2>(prm, mom, var, X, T, idx, n, batch, corr, lr, epoch_loss, s);
    case 3: return launch_epoch<3>(prm, mom, var, X, T, idx, n, batch, corr, lr, epoch_loss, s);
    case 4: return launch_epoch<4>(prm, mom, var, X, T, idx, n, batch, corr, lr, epoch_loss, s);
    case 5: return launch_epoch<5>(prm, mom, var, X, T, idx, n, batch, corr, lr, epoch_loss, s);
    case 9: return launch_epoch<9>(prm, mom, var, X, T, idx, n, batch, corr, lr, epoch_loss, s);
    case 16: return launch_epoch<16>(prm, mom, var, X, T, idx, n, batch, corr, lr, epoch_loss, s);
    case 25: return launch_epoch<25>(prm, mom, var, X, T, idx, n, batch, corr, lr, epoch_loss, s);
  }
  return cudaErrorInvalidValue;
}

uint64_t splitmix64(uint64_t* s) {
  uint64_t z = (*s += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

}  // namespace

extern "C" {

int cr_mlp_param_count(int nin) { return nin_supported(nin) ? param_count(nin) : -1; }

cr_status cr_mlp_grad(int nin, const float* params, const float* X, const float* t, int n,
                      float* grad, float* loss, void* stream) {
  if (!nin_supported(nin) || !params || !X || !t || !grad || !loss || n < 1) return CR_E_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float* part = nullptr;  // per-block partial sums, stream-ordered allocation
  const size_t bytes = sizeof(float) * (size_t)grad_blocks(n) * (param_count(nin) + 1);
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&part), bytes, s);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? CR_E_NOMEM : CR_E_CUDA;
  e = dispatch_grad(nin, params, X, t, nullptr, n, part, grad, loss, s);
  const cudaError_t e2 = cudaFreeAsync(part, s);
  return (e == cudaSuccess && e2 == cudaSuccess) ? CR_OK : CR_E_CUDA;
}

cr_status cr_mlp_train(int nin, float* params, const float* X, const float* t, int n, int batch,
                       int epochs, float lr, unsigned long long seed, float* epoch_loss,
                       void* stream) {
  if (!nin_supported(nin) || !params || !X || !t || n < 1 || batch < 1 || epochs < 0 || !(lr > 0.0f))
    return CR_E_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int P = param_count(nin);
  const int most = batch < n ? batch : n;        // samples of the largest minibatch
  const int nb = (n - 1) / batch + 1;            // minibatches per epoch
  const bool by_epoch = (most + kChunk - 1) / kChunk <= kEpochBlocks;
  // one device allocation: moments, losses, the epoch's sample order, and the
  // bias corrections (epoch kernel) or gradient and partial sums (per minibatch)
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) & ~size_t(255);
    return o;
  };
  const size_t o_mom = take(sizeof(float) * P), o_var = take(sizeof(float) * P), o_el = take(sizeof(float)),
               o_bl = take(sizeof(float)), o_idx = take(sizeof(int) * (size_t)n),
               o_corr = take(by_epoch ? sizeof(float2) * (size_t)nb : 0), o_grad = take(by_epoch ? 0 : sizeof(float) * P),
               o_part = take(by_epoch ? 0 : sizeof(float) * (size_t)grad_blocks(most) * (P + 1));
  unsigned char* mem = nullptr;
  cr_status st = CR_OK;
  auto ok = [&](cudaError_t e) {
    if (e != cudaSuccess && st == CR_OK) st = (e == cudaErrorMemoryAllocation) ? CR_E_NOMEM : CR_E_CUDA;
    return st == CR_OK;
  };
  ok(cudaMalloc(&mem, off));
  auto at = [&](size_t o) { return reinterpret_cast<float*>(mem + o); };
  float *mom = at(o_mom), *var = at(o_var), *el = at(o_el), *bl = at(o_bl);
  int* idx = reinterpret_cast<int*>(mem + o_idx);
  if (st == CR_OK) {
    ok(cudaMemsetAsync(mom, 0, sizeof(float) * P, s));
    ok(cudaMemsetAsync(var, 0, sizeof(float) * P, s));
  }
  // The host arrays of an epoch (sample order, bias corrections) are read by copies
  // that may still be queued behind earlier epochs' kernels when the call returns to
  // the host, so an epoch writes the pair that the last one did not use, once the
  // event behind that pair's own copies has passed.  The next order is drawn while
  // the device runs, and no epoch waits for the one before it.
  struct HostEpoch {
    std::vector<int> perm;
    std::vector<float2> corr;
    cudaEvent_t copied = nullptr;
    ~HostEpoch() {
      if (copied) cudaEventDestroy(copied);
    }
  } host[2];
  try {
    for (HostEpoch& h : host) {
      h.perm.resize(n);
      if (by_epoch) h.corr.resize(nb);
    }
  } catch (const std::bad_alloc&) {
    st = CR_E_NOMEM;
  }
  for (HostEpoch& h : host)
    if (st == CR_OK) ok(cudaEventCreateWithFlags(&h.copied, cudaEventDisableTiming));
  uint64_t rs = seed;
  int step = 0;
  for (int ep = 0; ep < epochs && st == CR_OK; ++ep) {
    HostEpoch& h = host[ep & 1];
    if (ep >= 2 && !ok(cudaEventSynchronize(h.copied))) break;
    int* perm = h.perm.data();
    for (int i = 0; i < n; ++i) perm[i] = i;
    for (int i = n - 1; i > 0; --i) {  // Fisher-Yates with a seeded splitmix64
      const int j = int(splitmix64(&rs) % uint64_t(i + 1));
      const int tmp = perm[i];
      perm[i] = perm[j];
      perm[j] = tmp;
    }
    ok(cudaMemcpyAsync(idx, perm, sizeof(int) * n, cudaMemcpyHostToDevice, s));
    if (by_epoch) {
      float2* corr = h.corr.data();
      for (int k = 0; k < nb; ++k) {
        ++step;
        corr[k].x = 1.0f - powf(0.9f, float(step));
        corr[k].y = 1.0f - powf(0.999f, float(step));
      }
      float2* dcorr = reinterpret_cast<float2*>(mem + o_corr);
      ok(cudaMemcpyAsync(dcorr, corr, sizeof(float2) * nb, cudaMemcpyHostToDevice, s));
      if (st == CR_OK) ok(cudaEventRecord(h.copied, s));
      if (st == CR_OK) ok(dispatch_epoch(nin, params, mom, var, X, t, idx, n, most, dcorr, lr, el, s));
      continue;
    }
    if (st == CR_OK) ok(cudaEventRecord(h.copied, s));
    ok(cudaMemsetAsync(el, 0, sizeof(float), s));
    float* grad = at(o_grad);
    for (int b0 = 0; b0 < n && st == CR_OK; b0 += batch) {
      const int cnt = n - b0 < batch ? n - b0 : batch;
      ok(dispatch_grad(nin, params, X, t, idx + b0, cnt, at(o_part), grad, bl, s));
      ++step;
      const float c1 = 1.0f - powf(0.9f, float(step)), c2 = 1.0f - powf(0.999f, float(step));
      k_mlp_adam<<<(P + 255) / 256, 256, 0, s>>>(params, grad, mom, var, P, lr, c1, c2);
      ok(cudaGetLastError());
      k_accumulate<<<1, 1, 0, s>>>(el, bl);
      ok(cudaGetLastError());
      if (n - b0 <= batch) break;  // (b0 + batch may pass the int range)
    }
  }
  float sum = 0.0f;
  if (st == CR_OK && epochs > 0) ok(cudaMemcpyAsync(&sum, el, sizeof(float), cudaMemcpyDeviceToHost, s));
  ok(cudaStreamSynchronize(s));
  if (epoch_loss) *epoch_loss = st == CR_OK && epochs > 0 ? sum / nb : 0.0f;
  if (mem) cudaFree(mem);
  return st;
}

}  // extern "C"
