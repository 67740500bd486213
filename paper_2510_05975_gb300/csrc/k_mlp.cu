// k_mlp.cu -- training of the learned early-stop network (not part of the paper's method; the
// paper's search stops only by Alg. 1's rule).
//
// Network: 16 -> 64 -> 64 -> 1, ReLU, logit z; loss = mean binary cross-entropy with logits
//   l(z, y) = max(z, 0) - z y + log(1 + exp(-|z|)).
// Parameters (FP32 master copy), flat: W1[64][16] b1[64] W2[64][64] b2[64] w3[64] b3[1].
// Samples: one per (training query, hop t <= max_trace) of a traced plain search; features as
// in the search kernel, label y = (t >= last hop at which the query's top-k list changed).
// Inputs are standardised with the training set's per-feature mean and standard deviation.
// Optimiser: Adam (beta 0.9 / 0.999, eps 1e-8); minibatch rows drawn with replacement by a
// counter-based hash of (seed, step, slot).  Gradients: one partial per group of 128 samples, each
// entry one sum over the group's samples in order; partials are summed in group order, so training
// is deterministic.
//
// A step is three launches: activations and their gradients (32 samples a CTA, one sample per lane,
// 8 outputs per warp), the groups' parameter gradients (eight CTAs a group), and the sum over the
// groups with Adam's update.  Each sum keeps its order; what is parallel is the outputs.  Bound by the
// dependent FMA chains, load latency and launches: a step of 4,096 samples took 90 us with one CTA of
// 128 threads doing all of a group's work (32 CTAs in all), now 25 us (10.6 + 10 + 5); fitting on
// 10,000 traces (384 steps) 35.8 -> 11.4 ms.
#include "launch_count.h"
#include "cng_internal.h"
#include "device_common.cuh"
#include "mlp_internal.h"
#include "search_internal.h"

namespace cng {

constexpr int MT = 128;  // samples per group (one partial gradient)
constexpr int MA = 32;   // samples per CTA of the forward / backward kernel
constexpr int MF = 256;  // its threads
constexpr int MO = 64 / (MF / 32);  // outputs of a layer per warp
constexpr int MG = 8;    // CTAs per group of the gradient kernel
constexpr int MC = 1024; // groups whose activations are held at once (144 MB)

CNG_DEV uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

// ---- samples from traces ---------------------------------------------------------------------
// counts[q] = min(hops[q], T); offsets by an exclusive scan in one CTA (sequential chunks).
__global__ void trace_offsets_kernel(const int32_t* __restrict__ hops, int64_t nq, int T,
                                     int64_t* __restrict__ off) {
  __shared__ int64_t carry;
  __shared__ int64_t ws[32];
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t b = 0; b < nq; b += blockDim.x) {
    int64_t i = b + threadIdx.x;
    int64_t v = i < nq ? min(hops[i], T) : 0;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int64_t t = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += t;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
      int64_t w = lane < (int)(blockDim.x >> 5) ? ws[lane] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int64_t t = __shfl_up_sync(FULL, w, o);
        if (lane >= o) w += t;
      }
      ws[lane] = w;
    }
    __syncthreads();
    int64_t incl = x + (warp > 0 ? ws[warp - 1] : 0) + carry;
    if (i < nq) off[i] = incl - v;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) off[nq] = carry;
}

__global__ void flatten_kernel(const float* __restrict__ feats, const int32_t* __restrict__ hops,
                               const int32_t* __restrict__ tlc, const int64_t* __restrict__ off,
                               int64_t nq, int T, float* __restrict__ X, float* __restrict__ y) {
  int64_t q = blockIdx.x;
  if (q >= nq) return;
  const int c = min(hops[q], T);
  const int64_t o = off[q];
  for (int e = threadIdx.x; e < c * 16; e += blockDim.x) {
    int t = e >> 4, j = e & 15;
    X[(o + t) * 16 + j] = feats[((int64_t)q * T + t) * 16 + j];
    if (j == 0) y[o + t] = (t + 1 >= tlc[q]) ? 1.f : 0.f;
  }
}

// per-feature sum and sum of squares in double (one partial per CTA, then one CTA sums them)
__global__ void __launch_bounds__(256) feat_stats_kernel(const float* __restrict__ X, int64_t N,
                                                         double* __restrict__ part) {
  __shared__ double ws[8][32];
  double a[16], b[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) a[j] = b[j] = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      double v = X[i * 16 + j];
      a[j] += v;
      b[j] += v * v;
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a[j] += __shfl_xor_sync(FULL, a[j], o);
      b[j] += __shfl_xor_sync(FULL, b[j], o);
    }
  }
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      ws[warp][j] = a[j];
      ws[warp][16 + j] = b[j];
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double x = 0;
    for (int w = 0; w < 8; ++w) x += ws[w][threadIdx.x];
    part[blockIdx.x * 32 + threadIdx.x] = x;
  }
}

__global__ void feat_norm_kernel(const double* __restrict__ part, int nparts, int64_t N,
                                 float* __restrict__ mu, float* __restrict__ sg) {
  int j = threadIdx.x;
  if (j >= 16) return;
  double x = 0, z = 0;
  for (int p = 0; p < nparts; ++p) {
    x += part[p * 32 + j];
    z += part[p * 32 + 16 + j];
  }
  double m = x / (double)N;
  double v = z / (double)N - m * m;
  mu[j] = (float)m;
  sg[j] = (float)sqrt(v > 1e-12 ? v : 1e-12);
}

__global__ void standardise_kernel(float* __restrict__ X, int64_t N, const float* __restrict__ mu,
                                   const float* __restrict__ sg) {
  int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= N * 16) return;
  int j = (int)(e & 15);
  X[e] = (X[e] - mu[j]) / sg[j];
}

// ---- forward + backward --------------------------------------------------------------------------
// Activations and gradients of up to MC groups, [samples rounded up to MT][..]: x 16, h1, h2, g1 (dL/da1) and
// g2 (dL/da2) 64 each, dz and the loss 1 each.
struct MlpActs {
  float *x, *h1, *h2, *g1, *g2, *dz, *ls;
};
CNG_DEV void put4(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
static MlpActs acts_of(float* p, int groups) {
  const size_t n = (size_t)groups * MT;
  MlpActs a;
  a.x = p;
  a.h1 = a.x + n * 16;
  a.h2 = a.h1 + n * 64;
  a.g1 = a.h2 + n * 64;
  a.g2 = a.g1 + n * 64;
  a.dz = a.g2 + n * 64;
  a.ls = a.dz + n;
  return a;
}

// Samples s0 .. of the batch: rows drawn by hash of (seed, step, slot), or 0..B-1 (seed 0).  Lane = sample; warp w computes
// outputs MO w .. + MO - 1 of each layer and keeps them in registers for the backward pass.
__global__ void __launch_bounds__(MF)
mlp_fwd_bwd_kernel(const float* __restrict__ P, const float* __restrict__ X, const float* __restrict__ Y,
                   int64_t N, int B, int s0, uint64_t seed, int64_t step, float inv_scale, MlpActs A) {
  __shared__ __align__(16) float w[MLP_NPARAMS_PAD];
  __shared__ float h1[MA * 65];  // [sample][65] (pad: conflict-free columns)
  __shared__ float h2[MA * 65];  // later dL/da2
  __shared__ float dzs[MA];
  const int t = threadIdx.x, lane = t & 31, o0 = (t >> 5) * MO;
  const int s = (int)blockIdx.x * MA + lane, slot = s0 + s;
  const bool live = slot < B;
  int64_t row = 0;
  if (live) {
    row = seed ? (int64_t)(splitmix64(seed ^ ((uint64_t)step * 0x100000001B3ull + (uint64_t)slot)) %
                           (uint64_t)N)
               : slot;
  }
  float x[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) x[j] = live ? X[row * 16 + j] : 0.f;
  const float y = live ? Y[row] : 0.f;
  // every load of the weights in flight at once: a loop of dependent batches costs more than a layer
#pragma unroll
  for (int k = 0; k < (MLP_NPARAMS + MF - 1) / MF; ++k)
    if (k * MF + t < MLP_NPARAMS) w[k * MF + t] = P[k * MF + t];
  const float* W1 = w;
  const float* b1 = W1 + 64 * 16;
  const float* W2 = b1 + 64;
  const float* b2 = W2 + 64 * 64;
  const float* w3 = b2 + 64;
  const float* b3 = w3 + 64;
  if (o0 == 0) {
#pragma unroll
    for (int j = 0; j < 16; j += 4) put4(A.x + s * 16 + j, x + j);
  }
  __syncthreads();
  float r1[MO], a[MO];
#pragma unroll
  for (int k = 0; k < MO; ++k) {
    r1[k] = b1[o0 + k];
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
      const float4 v = *reinterpret_cast<const float4*>(W1 + (o0 + k) * 16 + i);
      r1[k] = fmaf(v.x, x[i], r1[k]);
      r1[k] = fmaf(v.y, x[i + 1], r1[k]);
      r1[k] = fmaf(v.z, x[i + 2], r1[k]);
      r1[k] = fmaf(v.w, x[i + 3], r1[k]);
    }
    r1[k] = fmaxf(r1[k], 0.f);
    h1[lane * 65 + o0 + k] = r1[k];
    a[k] = b2[o0 + k];
  }
#pragma unroll
  for (int k = 0; k < MO; k += 4) put4(A.h1 + s * 64 + o0 + k, r1 + k);
  __syncthreads();
#pragma unroll 4
  for (int i = 0; i < 64; i += 4) {
    const float* h = h1 + lane * 65 + i;
    const float ha = h[0], hb = h[1], hc = h[2], hd = h[3];
#pragma unroll
    for (int k = 0; k < MO; ++k) {
      const float4 v = *reinterpret_cast<const float4*>(W2 + (o0 + k) * 64 + i);
      a[k] = fmaf(v.x, ha, a[k]);
      a[k] = fmaf(v.y, hb, a[k]);
      a[k] = fmaf(v.z, hc, a[k]);
      a[k] = fmaf(v.w, hd, a[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < MO; ++k) {
    a[k] = fmaxf(a[k], 0.f);
    h2[lane * 65 + o0 + k] = a[k];
  }
#pragma unroll
  for (int k = 0; k < MO; k += 4) put4(A.h2 + s * 64 + o0 + k, a + k);
  __syncthreads();
  if (o0 == 0) {
    float z = b3[0];
#pragma unroll 16
    for (int o = 0; o < 64; ++o) z = fmaf(w3[o], h2[lane * 65 + o], z);
    const float sig = 1.f / (1.f + expf(-z));
    const float dz = live ? (sig - y) * inv_scale : 0.f;
    dzs[lane] = dz;
    A.dz[s] = dz;
    A.ls[s] = live ? fmaxf(z, 0.f) - z * y + log1pf(expf(-fabsf(z))) : 0.f;
  }
  __syncthreads();
  const float dz = dzs[lane];
#pragma unroll
  for (int k = 0; k < MO; ++k) {
    a[k] = a[k] > 0.f ? dz * w3[o0 + k] : 0.f;
    h2[lane * 65 + o0 + k] = a[k];
  }
#pragma unroll
  for (int k = 0; k < MO; k += 4) put4(A.g2 + s * 64 + o0 + k, a + k);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < MO; ++k) a[k] = 0.f;
#pragma unroll 8
  for (int o = 0; o < 64; ++o) {
    const float gv = h2[lane * 65 + o];
#pragma unroll
    for (int k = 0; k < MO; k += 4) {
      const float4 v = *reinterpret_cast<const float4*>(W2 + o * 64 + o0 + k);
      a[k] = fmaf(v.x, gv, a[k]);
      a[k + 1] = fmaf(v.y, gv, a[k + 1]);
      a[k + 2] = fmaf(v.z, gv, a[k + 2]);
      a[k + 3] = fmaf(v.w, gv, a[k + 3]);
    }
  }
#pragma unroll
  for (int k = 0; k < MO; ++k) a[k] = r1[k] > 0.f ? a[k] : 0.f;
#pragma unroll
  for (int k = 0; k < MO; k += 4) put4(A.g1 + s * 64 + o0 + k, a + k);
}

// Parameter gradients of one group of MT samples (blockIdx.x), each entry a sum over the samples in
// order.  blockIdx.y < 4: rows 16 y .. +15 of W2; 4: W1; 5: b1; 6: b2; 7: w3, b3 and the loss.  The
// operands go to shared memory first: from global memory each step of the 128-step sums waited for a
// load (49 us a launch for 32 groups, against 10).
__global__ void __launch_bounds__(256) mlp_group_grad_kernel(MlpActs A, float* __restrict__ part,
                                                             float* __restrict__ part_loss) {
  __shared__ __align__(16) float wide[MT * 64];
  __shared__ __align__(16) float slim[MT * 16];
  const int t = threadIdx.x, y = blockIdx.y;
  const int64_t s0 = (int64_t)blockIdx.x * MT;
  float* out = part + (size_t)blockIdx.x * MLP_NPARAMS;
  const float* src[4] = {A.g1, A.g1, A.g2, A.h2};
  const float4* pw = reinterpret_cast<const float4*>((y < 4 ? A.h1 : src[y - 4]) + s0 * 64);
#pragma unroll
  for (int k = 0; k < MT * 16 / 256; ++k) reinterpret_cast<float4*>(wide)[k * 256 + t] = pw[k * 256 + t];
  if (y < 5) {
    // 16 floats a sample: the tile's columns of g2, or the sample's inputs
    const float* ps = y < 4 ? A.g2 + s0 * 64 + 16 * y : A.x + s0 * 16;
    const int ld = y < 4 ? 64 : 16;
#pragma unroll
    for (int k = 0; k < MT * 4 / 256; ++k) {
      const int e = k * 256 + t;
      reinterpret_cast<float4*>(slim)[e] = *reinterpret_cast<const float4*>(ps + (e >> 2) * ld + (e & 3) * 4);
    }
  } else if (y == 7) {
    slim[t] = t < MT ? A.dz[s0 + t] : A.ls[s0 + t - MT];
  }
  __syncthreads();
  if (y < 5) {  // thread = one of the 64 wide columns and 4 of the 16 slim ones
    const int c = t & 63, f = (t >> 6) * 4;
    float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 16
    for (int q = 0; q < MT; ++q) {
      const float v = wide[q * 64 + c];
      const float4 g = *reinterpret_cast<const float4*>(slim + q * 16 + f);
      a[0] = fmaf(g.x, v, a[0]);
      a[1] = fmaf(g.y, v, a[1]);
      a[2] = fmaf(g.z, v, a[2]);
      a[3] = fmaf(g.w, v, a[3]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      out[y < 4 ? 64 * 16 + 64 + (16 * y + f + k) * 64 + c : c * 16 + f + k] = a[k];
  } else if (t < 64) {
    float a = 0.f;
    if (y < 7) {
#pragma unroll 16
      for (int q = 0; q < MT; ++q) a += wide[q * 64 + t];
      out[y == 5 ? 64 * 16 + t : 64 * 16 + 64 + 64 * 64 + t] = a;
    } else {
#pragma unroll 16
      for (int q = 0; q < MT; ++q) a = fmaf(slim[q], wide[q * 64 + t], a);
      out[64 * 16 + 64 + 64 * 64 + 64 + t] = a;
    }
  } else if (y == 7 && (t == 64 || t == 96)) {
    const float* v = t == 64 ? slim : slim + MT;
    float a = 0.f;
#pragma unroll 16
    for (int q = 0; q < MT; ++q) a += v[q];
    if (t == 64)
      out[MLP_NPARAMS - 1] = a;
    else
      part_loss[blockIdx.x] = a;
  }
}

// The gradient from the groups' partials, summed in group order, and the mean loss.
CNG_DEV float sum_parts(const float* __restrict__ part, int nparts, int p) {
  float a = 0.f;
#pragma unroll 32
  for (int c = 0; c < nparts; ++c) a += part[(size_t)c * MLP_NPARAMS + p];
  return a;
}
CNG_DEV void mean_loss(const float* __restrict__ part_loss, int nparts, float scale, float* loss) {
  float l = 0.f;
  for (int c = 0; c < nparts; ++c) l += part_loss[c];
  *loss = l * scale;
}

__global__ void reduce_grad_kernel(const float* __restrict__ part, int nparts,
                                   const float* __restrict__ part_loss, float loss_scale,
                                   float* __restrict__ grad, float* __restrict__ loss) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < MLP_NPARAMS) grad[p] = sum_parts(part, nparts, p);
  if (p == 0 && loss) mean_loss(part_loss, nparts, loss_scale, loss);
}

CNG_DEV void adam_update(float* __restrict__ P, float* __restrict__ m, float* __restrict__ v, int p,
                         float gi, int64_t t, float lr) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  float mi = b1 * m[p] + (1.f - b1) * gi;
  float vi = b2 * v[p] + (1.f - b2) * gi * gi;
  m[p] = mi;
  v[p] = vi;
  float mh = mi / (1.f - powf(b1, (float)t));
  float vh = vi / (1.f - powf(b2, (float)t));
  P[p] -= lr * mh / (sqrtf(vh) + eps);
}

__global__ void adam_kernel(float* __restrict__ P, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, int64_t t, float lr) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= MLP_NPARAMS) return;
  adam_update(P, m, v, p, g[p], t, lr);
}

// The last launch of a training step: gradient, loss (if wanted) and Adam's update.
__global__ void reduce_adam_kernel(const float* __restrict__ part, int nparts,
                                   const float* __restrict__ part_loss, float loss_scale,
                                   float* __restrict__ loss, float* __restrict__ P, float* __restrict__ m,
                                   float* __restrict__ v, int64_t t, float lr) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p == 0 && loss) mean_loss(part_loss, nparts, loss_scale, loss);
  if (p >= MLP_NPARAMS) return;
  adam_update(P, m, v, p, sum_parts(part, nparts, p), t, lr);
}

// Kaiming-uniform weights, zero biases, from the counter-based generator.
__global__ void mlp_init_kernel(float* __restrict__ P, uint64_t seed) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= MLP_NPARAMS) return;
  float bound = 0.f;
  if (p < 64 * 16) bound = sqrtf(6.f / 16.f);
  else if (p >= 64 * 16 + 64 && p < 64 * 16 + 64 + 64 * 64) bound = sqrtf(6.f / 64.f);
  else if (p >= 64 * 16 + 64 + 64 * 64 + 64 && p < MLP_NPARAMS - 1) bound = sqrtf(6.f / 64.f);
  uint64_t r = splitmix64(seed * 0x9E3779B97F4A7C15ull + (uint64_t)p);
  float u = (float)(r >> 40) * (1.f / 16777216.f);  // [0, 1)
  P[p] = bound * (2.f * u - 1.f);
}

// FP32 master parameters + normalisation -> packed inference block (BF16 weights).
__global__ void pack_model_kernel(const float* __restrict__ P, const float* __restrict__ mu,
                                  const float* __restrict__ sg, unsigned char* __restrict__ blk) {
  // output-major rows padded to 24 and 72 elements (the pads are zero)
  __nv_bfloat16* W1b = reinterpret_cast<__nv_bfloat16*>(blk);
  __nv_bfloat16* W2b = W1b + 64 * 24;
  float* f = reinterpret_cast<float*>(W2b + 64 * 72);
  const float* W1 = P;
  const float* b1 = W1 + 64 * 16;
  const float* W2 = b1 + 64;
  const float* b2 = W2 + 64 * 64;
  const float* w3 = b2 + 64;
  const float* b3 = w3 + 64;
  for (int e = threadIdx.x; e < 64 * 24; e += blockDim.x) {
    const int o = e / 24, i = e % 24;
    W1b[e] = __float2bfloat16_rn(i < 16 ? W1[o * 16 + i] : 0.f);
  }
  for (int e = threadIdx.x; e < 64 * 72; e += blockDim.x) {
    const int o = e / 72, i = e % 72;
    W2b[e] = __float2bfloat16_rn(i < 64 ? W2[o * 64 + i] : 0.f);
  }
  for (int e = threadIdx.x; e < 64; e += blockDim.x) {
    f[e] = b1[e];
    f[64 + e] = b2[e];
    f[128 + e] = w3[e];
  }
  if (threadIdx.x < 4) f[192 + threadIdx.x] = threadIdx.x == 0 ? b3[0] : 0.f;
  if (threadIdx.x < 16) {
    f[196 + threadIdx.x] = mu[threadIdx.x];
    f[212 + threadIdx.x] = sg[threadIdx.x];
  }
}

// ---- host-side launchers ---------------------------------------------------------------------------
int mlp_parts(int B) { return (B + MT - 1) / MT; }
size_t mlp_scratch_floats(int B) {
  const size_t n = (size_t)std::min(mlp_parts(B), MC) * MT;
  return (size_t)mlp_parts(B) * (MLP_NPARAMS + 1) + 4 + n * (16 + 4 * 64 + 2);
}

// scratch: the groups' losses, their partial gradients, the activations of MC groups (16-byte aligned)
static cudaError_t launch_partials(const float* P, const float* X, const float* Y, int64_t N, int B,
                                   uint64_t seed, int64_t step, float* scratch, float** part,
                                   float** part_loss, cudaStream_t s) {
  const int parts = mlp_parts(B);
  *part_loss = scratch;
  *part = scratch + parts;
  const MlpActs A = acts_of(scratch + ((size_t)parts * (MLP_NPARAMS + 1) + 3) / 4 * 4, std::min(parts, MC));
  for (int g0 = 0; g0 < parts; g0 += MC) {
    const int groups = std::min(parts - g0, MC);
    count_launch();
    mlp_fwd_bwd_kernel<<<groups * (MT / MA), MF, 0, s>>>(P, X, Y, N, B, g0 * MT, seed, step,
                                                         1.f / (float)B, A);
    count_launch();
    mlp_group_grad_kernel<<<dim3(groups, MG), 256, 0, s>>>(A, *part + (size_t)g0 * MLP_NPARAMS, *part_loss + g0);
  }
  return cudaGetLastError();
}

cudaError_t launch_mlp_grad(const float* P, const float* X, const float* Y, int64_t N, int B,
                            float* scratch, float* grad, float* loss, cudaStream_t s) {
  float *part, *part_loss;
  cudaError_t e = launch_partials(P, X, Y, N, B, 0, 0, scratch, &part, &part_loss, s);
  if (e != cudaSuccess) return e;
  count_launch();
  reduce_grad_kernel<<<(MLP_NPARAMS + 255) / 256, 256, 0, s>>>(part, mlp_parts(B), part_loss,
                                                               1.f / (float)B, grad, loss);
  return cudaGetLastError();
}

cudaError_t launch_mlp_step(float* P, const float* X, const float* Y, int64_t N, int B, uint64_t seed,
                            int64_t t, float lr, float* m, float* v, float* scratch, float* loss,
                            cudaStream_t s) {
  float *part, *part_loss;
  cudaError_t e = launch_partials(P, X, Y, N, B, seed, t, scratch, &part, &part_loss, s);
  if (e != cudaSuccess) return e;
  count_launch();
  reduce_adam_kernel<<<(MLP_NPARAMS + 127) / 128, 128, 0, s>>>(part, mlp_parts(B), part_loss,
                                                               1.f / (float)B, loss, P, m, v, t, lr);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* P, float* m, float* v, const float* g, int64_t t, float lr, cudaStream_t s) {
  count_launch();
  adam_kernel<<<(MLP_NPARAMS + 255) / 256, 256, 0, s>>>(P, m, v, g, t, lr);
  return cudaGetLastError();
}

cudaError_t launch_mlp_init(float* P, uint64_t seed, cudaStream_t s) {
  count_launch();
  mlp_init_kernel<<<(MLP_NPARAMS + 255) / 256, 256, 0, s>>>(P, seed);
  return cudaGetLastError();
}

cudaError_t launch_pack_model(const float* P, const float* mu, const float* sg, void* blk, cudaStream_t s) {
  count_launch();
  pack_model_kernel<<<1, 256, 0, s>>>(P, mu, sg, (unsigned char*)blk);
  return cudaGetLastError();
}

cudaError_t launch_samples(const float* feats, const int32_t* hops, const int32_t* tlc, int64_t nq, int T,
                           int64_t* off, float* X, float* y, cudaStream_t s) {
  count_launch();
  flatten_kernel<<<(unsigned)nq, 128, 0, s>>>(feats, hops, tlc, off, nq, T, X, y);
  return cudaGetLastError();
}

cudaError_t launch_offsets(const int32_t* hops, int64_t nq, int T, int64_t* off, cudaStream_t s) {
  count_launch();
  trace_offsets_kernel<<<1, 1024, 0, s>>>(hops, nq, T, off);
  return cudaGetLastError();
}

cudaError_t launch_standardise(float* X, int64_t N, double* part, float* mu, float* sg, cudaStream_t s) {
  const int nparts = 64;
  count_launch();
  feat_stats_kernel<<<nparts, 256, 0, s>>>(X, N, part);
  count_launch();
  feat_norm_kernel<<<1, 32, 0, s>>>(part, nparts, N, mu, sg);
  count_launch();
  standardise_kernel<<<(unsigned)((N * 16 + 255) / 256), 256, 0, s>>>(X, N, mu, sg);
  return cudaGetLastError();
}

}  // namespace cng
